"""One-launch steps with a single collocation node, where node 1 of a sweep writes the row that the evaluation
before it reads: several sweeps on every split of a node over warps, against the oracle and bit for bit from
run to run."""
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


def smooth_state(wl):
    """Rest plus a smooth potential bump, gates at their values there (from the oracle's rest states)."""
    V = wl.V0 + 60.0 * np.exp(-((np.arange(wl.n_nodes) % wl.nx) / max(wl.nx, 8) - 0.3) ** 2 / 0.05)
    V += np.random.default_rng(4).normal(0.0, 0.3, wl.n_nodes)
    lv = np.linspace(V.min(), V.max(), 40)
    tab = np.array([O.ionic_rest(wl.model, wl.params, float(v)) for v in lv])
    return np.stack([V] + [np.interp(V, lv, tab[:, s]) for s in range(1, wl.n_state)])


# four roles per node (32 and 128 nodes per block), two roles (256), DCT and Chebyshev
MESHES = [(37, 29, 1), (32, 32, 1), (139, 139, 1), (150, 140, 1)]


@pytest.mark.parametrize("model", ["hh", "syn19"])
@pytest.mark.parametrize("mesh", MESHES)
@pytest.mark.parametrize("K", [2, 5])
@pytest.mark.parametrize("fuse", [True, False])
def test_single_node_sweeps(model, mesh, K, fuse):
    wl = (I.hh_sheet_32() if model == "hh" else I.syn19_slab()).with_mesh(*mesh)
    wl.boxes = np.array([[0, 3, 0, 2, 0, 1]], np.int32)
    s = P.Solver.from_workload(wl, M_max=1, fuse_node1=fuse)
    y0 = smooth_state(wl)
    start = s.new_state()
    start[:, : wl.n_nodes] = torch.from_numpy(y0)
    y, first = s.new_state(), None
    s.profile(True)
    for _ in range(8):
        y.copy_(start)
        s.sweep(y, 0.3, wl.dt, 1, K)
        got = y[:, : wl.n_nodes].cpu().numpy()
        if first is None:
            first = got
        assert np.array_equal(got, first)
    assert {k: v[1] for k, v in s.profile_read().items()} == {"setup": 0, "node": 8, "cg": 0, "residual": 0}
    assert s.residual()[0] == 0
    want = O.Monodomain(wl).step(y0, 0.3, wl.dt, 1, K)[0]
    # the bound of the one-launch steps' oracle tests: solves to 1e-14 and the stiff gates' rounding stay
    # two orders below it
    assert np.abs(first[0] - want[0]).max() < 1e-11 * np.abs(want[0]).max()
    assert np.abs(first[1:] - want[1:]).max() < 1e-11
