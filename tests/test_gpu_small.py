"""One-launch steps of small meshes (esdc_small.cuh) against the oracle: the
solves they contain (dense cosine products, the Chebyshev semi-iteration on
every operator), block edges and remainders, lines that do and do not divide a
block, every role split, the rule's border, and the failure path."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
import paper_2405_19994_gb300 as P  # noqa: E402
from paper_2405_19994_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    P.lib()


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


def smooth_state(wl):
    """Rest plus a smooth potential bump, gates at their values there (from the oracle's rest states)."""
    V = wl.V0 + 60.0 * np.exp(-((np.arange(wl.n_nodes) % wl.nx) / max(wl.nx, 8) - 0.3) ** 2 / 0.05)
    V += np.random.default_rng(2).normal(0.0, 0.3, wl.n_nodes)
    lv = np.linspace(V.min(), V.max(), 40)
    tab = np.array([O.ionic_rest(wl.model, wl.params, float(v)) for v in lv])
    return np.stack([V] + [np.interp(V, lv, tab[:, s]) for s in range(1, wl.n_state)])


def step_both(wl, M, K, solver="auto", t=0.3, **kw):
    """One step on the GPU and by the oracle; the kernels the GPU step launched per class."""
    s = P.Solver.from_workload(wl, M_max=M, solver=solver, **kw)
    y0 = smooth_state(wl)
    y = s.new_state()
    y[:, : wl.n_nodes] = torch.from_numpy(y0)
    s.profile(True)
    s.sweep(y, t, wl.dt, M, K)
    launches = {k: v[1] for k, v in s.profile_read().items()}
    rc, res, ymax, per_state = s.residual()
    assert rc == 0
    want, _, _, wres = O.Monodomain(wl).step(y0, t, wl.dt, M, K, want_resid=True)
    got = y[:, : wl.n_nodes].cpu().numpy()
    wr = np.abs(wres).max(axis=(0, 2))
    # the residual is a difference of numbers of the state's size
    assert np.all(np.abs(per_state - wr) <= 1e-9 * wr + 1e-13 * np.abs(want).max(axis=1) + 1e-15)
    return got, want, launches, s


ONE = {"setup": 0, "node": 1, "cg": 0, "residual": 0}

SHAPES = [
    # model, mesh, order, conductivity, solver: Chebyshev unless the DCT is named or automatic
    ("hh", (33, 1, 1), 2, "scalar", "auto"),        # one line, one node in the second block
    ("hh", (64, 1, 1), 2, "scalar", "auto"),        # DCT on one line over two blocks
    ("hh", (1, 32, 1), 2, "scalar", "auto"),        # DCT along y only
    ("hh", (500, 1, 1), 2, "scalar", "auto"),
    ("hh", (13, 11, 1), 2, "scalar", "auto"),       # dense odd axes, lines across blocks
    ("hh", (32, 24, 1), 2, "scalar", "auto"),
    ("hh", (16, 8, 4), 2, "scalar", "auto"),        # 3D DCT, lines inside blocks
    ("hh", (7, 5, 6), 2, "scalar", "dct"),          # 3D DCT, odd lines across blocks
    ("hh", (1, 9, 5), 2, "scalar", "dct"),          # y and z only
    ("hh", (128, 16, 1), 2, "scalar", "auto"),
    ("hh", (31, 9, 4), 2, "scalar", "auto"),
    ("hh", (101, 75, 1), 2, "scalar", "auto"),      # 64 nodes per block
    ("hh", (97, 101, 1), 2, "field", "auto"),       # 128 nodes per block, four roles
    ("hh", (30, 20, 6), 2, "layers", "auto"),
    ("hh", (24, 13, 1), 4, "scalar", "cheb"),
    ("hh", (3, 2, 2), 4, "scalar", "cheb"),         # axes shorter than the stencil
    ("hh", (16, 12, 5), 4, "scalar", "dct"),
    ("syn19", (17, 9, 3), 2, "scalar", "auto"),
    ("syn19", (16, 16, 4), 2, "scalar", "auto"),
    ("syn19", (150, 140, 1), 2, "scalar", "auto"),  # 256 nodes per block, two roles
]


def workload(model, mesh, order, cond):
    wl = (I.hh_sheet_32() if model == "hh" else I.syn19_slab()).with_mesh(*mesh)
    wl.boxes = np.array([[0, 3, 0, 2, 0, 2]], np.int32)
    wl.order = order
    if cond == "field":
        wl.sigma_field = I.lognormal_field(*mesh, seed=3)
    if cond == "layers":
        wl.layers = I.fibre_layers(mesh[2])
    return wl


@pytest.mark.parametrize("model,mesh,order,cond,solver", SHAPES)
@pytest.mark.parametrize("M,K", [(3, 3), (1, 2)])
def test_one_launch_step_matches_the_oracle(model, mesh, order, cond, solver, M, K):
    wl = workload(model, mesh, order, cond)
    got, want, launches, _ = step_both(wl, M, K, solver=solver)
    assert launches == ONE
    # V: the solves stop at 1e-14 of the right-hand side or are direct; K M of them and the stiff
    # gates' rounding stay two orders below 1e-11
    assert rel(got[0], want[0]) < 1e-11
    assert np.abs(got[1:] - want[1:]).max() < 1e-11


def test_rule_border_and_other_routes():
    # 152 x 256 nodes and below take one launch (a field: 152 x 512); the sequence otherwise
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wl = I.hh_sheet_32().with_mesh(sms, 256, 1)
    assert step_both(wl, 2, 1, solver="cheb")[2] == ONE
    wl = I.hh_sheet_32().with_mesh(sms, 257, 1)
    assert step_both(wl, 2, 1, solver="cheb")[2]["cg"] == 2
    wl = workload("hh", (sms, 257, 1), 2, "field")
    assert step_both(wl, 2, 1)[2] == ONE
    wl = I.hh_sheet_32().with_mesh(12, 10, 1)
    assert step_both(wl, 2, 1, solver="cg")[2]["cg"] == 2
    assert step_both(wl, 2, 1, fuse_node1=False)[2] == ONE


def test_failure_paths():
    wl = I.hh_sheet_32().with_mesh(40, 32, 1)
    y0 = smooth_state(wl)
    # an iteration cap of 1 is reported, and a NaN in the state
    s = P.Solver.from_workload(wl, M_max=3, solver="cheb", cg_maxit=1)
    y = s.new_state()
    y[:, : wl.n_nodes] = torch.from_numpy(y0)
    s.sweep(y, 0.3, wl.dt, 3, 2)
    assert s.residual()[0] == -3
    for solver in ("cheb", "auto"):
        w = I.hh_sheet_32().with_mesh(32, 32, 1) if solver == "auto" else wl
        s = P.Solver.from_workload(w, M_max=3, solver=solver)
        y0w = smooth_state(w)
        for bad in (True, False):                           # the handle steps normally afterwards
            y = s.new_state()
            y[:, : w.n_nodes] = torch.from_numpy(y0w)
            if bad:
                y[0, 77] = float("nan")
            s.sweep(y, 0.3, w.dt, 3, 2)
            assert s.residual()[0] == (-4 if bad else 0)
        # one block does not arrive at the barrier: every wait gives up, the handle recovers
        s.debug_barrier(0, 2000)
        s.sweep(y, 0.3, w.dt, 3, 2)
        assert s.residual()[0] == -5
        s.debug_barrier(-1)
        y[:, : w.n_nodes] = torch.from_numpy(y0w)
        s.sweep(y, 0.3, w.dt, 3, 2)
        assert s.residual()[0] == 0
        want = O.Monodomain(w).step(y0w, 0.3, w.dt, 3, 2)[0]
        assert rel(y[0, : w.n_nodes].cpu().numpy(), want[0]) < 1e-11
