"""The FP64 Chebyshev solve by FP32 corrections (large meshes with nx a multiple of 4)
against the conjugate gradients of the same library and the operator's own residual:
warm and cold starts, right-hand sides at and beyond FP32's range (which the FP64
iterations finish), the iteration cap, non-finite input."""
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


def workload(layers):
    wl = I.hh_aniso_slab().with_mesh(100, 80, 51)          # 408,000 nodes: above the refinement's border
    if not layers:
        wl.layers = None
    return wl


@pytest.mark.parametrize("layers", [True, False])
@pytest.mark.parametrize("scale", [1.0, 1e-11, 1e-60, 1e60])
@pytest.mark.parametrize("warm", [False, True])
def test_solve_reaches_the_stop_test(layers, scale, warm):
    wl = workload(layers)
    s = P.Solver.from_workload(wl, solver="cheb")
    m = O.Monodomain(wl)
    rng = np.random.default_rng(5)
    want = rng.normal(size=wl.n_nodes) * scale
    g = 0.05 * 0.3 / (wl.chi * wl.Cm) * (1.0 if layers else wl.sigma)
    apply = (lambda v: v - g * m.conductivity(v)) if layers else (lambda v: v - g * m.laplacian(v))
    b = apply(want)
    x0 = want + (1e-4 * scale * rng.normal(size=wl.n_nodes) if warm else -want)
    x = torch.from_numpy(x0).cuda()
    it = s.diffusion_solve(g, torch.from_numpy(b).cuda(), x)
    got = x.cpu().numpy()
    assert 1 <= it < 60
    # the stop test of every solve is 1e-14 of ||b||; evaluating the residual in FP64 adds its own rounding
    assert np.linalg.norm(b - apply(got)) <= 1.3e-14 * np.linalg.norm(b)
    # the smallest eigenvalue is 1: the error is at most the residual
    assert np.linalg.norm(got - want) <= 1.3e-14 * np.linalg.norm(b)


def test_caps_and_non_finite_input():
    wl = workload(True)
    s = P.Solver.from_workload(wl, solver="cheb", cg_maxit=3)
    b = torch.randn(wl.n_nodes, dtype=torch.float64, device="cuda")
    with pytest.raises(P.EsdcError) as e:
        s.diffusion_solve(0.01, b, torch.zeros_like(b))
    assert e.value.code == -3
    b[123] = float("inf")
    with pytest.raises(P.EsdcError) as e:
        s.diffusion_solve(0.01, b, torch.zeros_like(b))
    assert e.value.code == -4
    # a right-hand side of zero takes no iteration
    z = torch.zeros_like(b)
    assert s.diffusion_solve(0.01, z, torch.zeros_like(b)) == 0
