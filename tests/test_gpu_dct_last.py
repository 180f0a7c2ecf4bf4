"""The direct solve's last transformed axis in one kernel (forward, spectral division, inverse) against the
oracle's own operator: both stencils, one to three axes, the shortest and longest FFT lines, odd numbers of
lines, meshes whose tiles are fewer than the SMs, a right-hand side solved in place, a non-finite one."""
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


@pytest.mark.parametrize("shape", [(2, 1, 1), (4096, 1, 1), (1, 64, 1), (7, 2, 1), (3, 256, 1), (31, 64, 1), (256, 256, 1),
                                   (512, 1024, 1), (5, 3, 2), (9, 7, 32), (1, 1, 8)])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("inplace", [False, True])
def test_solve(shape, order, inplace):
    wl = I.hh_sheet_32().with_mesh(*shape)
    wl.order = order
    s = P.Solver.from_workload(wl, solver="dct")
    m = O.Monodomain(wl)
    b = np.random.default_rng(31).normal(size=wl.n_nodes)
    g = 0.05
    bd = torch.from_numpy(b).cuda()
    x = bd if inplace else torch.full_like(bd, float("nan"))           # the guess plays no part
    for _ in range(1 if inplace else 2):
        assert s.diffusion_solve(g, bd, x) == 1
    got = x.cpu().numpy()
    # an exact solve: rounding of log2 n butterfly stages a transform, and of the residual's own stencil
    assert np.abs(got - g * m.laplacian(got) - b).max() < 1e-14 * (1 + 16 * 3 * g / wl.h**2) * np.abs(b).max()


@pytest.mark.parametrize("order", [2, 4])
def test_non_finite(order):
    wl = I.hh_sheet_32().with_mesh(33, 64, 1)
    wl.order = order
    s = P.Solver.from_workload(wl, solver="dct")
    b = torch.randn(wl.n_nodes, dtype=torch.float64, device="cuda")
    b[100] = float("inf")
    with pytest.raises(P.EsdcError) as e:
        s.diffusion_solve(0.05, b, torch.zeros_like(b))
    assert e.value.code == -4
