"""Single Chebyshev solves of small meshes through exchange cells (up to 512 nodes per SM) against
the oracle's operator: every kind of conductivity and stencil, meshes of two nodes, of one warp, with
empty lanes and on both sides of the border, solves after one another and between steps, zero and
non-finite right-hand sides, the iteration cap."""
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


def workload(kind, shape):
    if kind == "layers":
        wl = I.hh_aniso_slab().with_mesh(*shape)
    else:
        wl = I.hh_sheet_32().with_mesh(*shape)
        if kind == "field":
            wl.sigma_field = I.lognormal_field(*shape, seed=4)
        if kind == "order4":
            wl.order = 4
    return wl


def operator(wl, kind):
    m = O.Monodomain(wl)
    if kind in ("layers", "field"):
        return 0.05 * 0.3 / (wl.chi * wl.Cm), m.conductivity
    return 0.05 * 0.3 / (wl.chi * wl.Cm) * wl.sigma, m.laplacian


@pytest.mark.parametrize("kind,shape", [(k, s) for k in ("scalar", "field", "order4", "layers")
                                        for s in ((2, 1, 1), (32, 1, 1), (37, 29, 1), (13, 11, 9), (200, 194, 1), (278, 279, 1),
                                                  (280, 279, 1))
                                        if k != "layers" or s[2] > 1 or s[0] > 100])
def test_solves(kind, shape):
    wl = workload(kind, shape)
    s = P.Solver.from_workload(wl, M_max=3, solver="cheb")
    g, A = operator(wl, kind)
    rng = np.random.default_rng(6)
    y = s.new_state()
    s.init_state(y, -75.0)
    for n in range(3):
        want = rng.normal(size=wl.n_nodes)
        b = want - g * A(want)
        x = torch.from_numpy(want + [1.0, 1e-5, 1e-10][n] * rng.normal(size=wl.n_nodes)).cuda()
        it = s.diffusion_solve(g, torch.from_numpy(b).cuda(), x)
        got = x.cpu().numpy()
        assert 1 <= it < 60
        # stop test 1e-14 ||b||, the smallest eigenvalue is 1; b's own rounding and the residual's come on top
        assert np.linalg.norm(b - (got - g * A(got))) <= 1.5e-14 * np.linalg.norm(b)
        assert np.linalg.norm(got - want) <= 1.5e-14 * np.linalg.norm(b)
        s.sweep(y, 0.0, 0.025, 3, 2)                    # a step between the solves shares their cells
    assert s.residual()[0] == 0


@pytest.mark.parametrize("kind", ["scalar", "field"])
def test_zero_cap_and_non_finite(kind):
    wl = workload(kind, (61, 43, 1))
    g, _ = operator(wl, kind)
    s = P.Solver.from_workload(wl, solver="cheb", cg_maxit=2)
    z = torch.zeros(wl.n_nodes, dtype=torch.float64, device="cuda")
    assert s.diffusion_solve(g, z, torch.zeros_like(z)) == 0
    b = torch.randn(wl.n_nodes, dtype=torch.float64, device="cuda")
    with pytest.raises(P.EsdcError) as e:
        s.diffusion_solve(g, b, torch.zeros_like(b))
    assert e.value.code == -3
    b[77] = float("nan")
    with pytest.raises(P.EsdcError) as e:
        s.diffusion_solve(g, b, torch.zeros_like(b))
    assert e.value.code == -4
    assert s.diffusion_solve(g, z, torch.zeros_like(z)) == 0
