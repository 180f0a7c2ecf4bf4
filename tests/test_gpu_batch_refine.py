"""Batched Chebyshev solves by FP32 corrections (tissues above 16384 nodes) against the
batched conjugate gradients: tissues on both sides of the border, odd, thin and three-dimensional
ones, spectra beyond what FP32 refines, potentials at and beyond FP32's range, each alone and in the batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2405_19994_gb300 as P  # noqa: E402
from paper_2405_19994_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    P.lib()


MESHES = [(128, 128, 1), (129, 128, 1), (37, 29, 1), (20001, 1, 1), (3, 7001, 1), (33, 31, 17), (1, 127, 131), (257, 200, 1)]


def tissues(stiff=1.0):
    """Pure diffusion (no ionic currents, no stimulus): the step is linear in V."""
    wls = []
    for k, (nx, ny, nz) in enumerate(MESHES):
        w = I.hh_batch(n=1, seed=20 + k, side=(48, 48), sigma=(0.05 * stiff, 0.3 * stiff))[0].with_mesh(nx, ny, nz)
        w.params = np.array(w.params, dtype=np.float64)
        w.params[:3] = 0.0
        w.amp = np.zeros_like(w.amp)
        wls.append(w)
    return wls


def step(wls, scale, seed=3, persistent=None, **kw):
    b = P.Batch.from_workloads(wls, M_max=3, **kw)
    if persistent:
        b.set_persistent(True, *persistent)
    y = b.new_state()
    b.init_state(y, -75.0)
    for k, w in enumerate(wls):
        v = np.random.default_rng([seed, w.nx, w.ny, w.nz]).uniform(4.0, 6.0, size=w.n_nodes)
        b.tissue(y, k)[0] = torch.from_numpy(scale * v).cuda()
    b.sweep(y, 0.0, wls[0].dt, 3, 4)
    rc, _, _ = b.residual()
    out = [b.tissue(y, k).cpu().numpy().copy() for k in range(len(wls))]
    it = b.stats(4, 3).copy()
    b.close()
    return rc, out, it


@pytest.mark.parametrize("stiff", [1.0, 280.0])
@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e-11, 1e17])
def test_tissues_match_cg_and_stay_alone(stiff, scale):
    wls = tissues(stiff)
    rc, got, it = step(wls, scale)
    rc_cg, want, _ = step(wls, scale, solver="cg")
    assert rc == 0 and rc_cg == 0 and it.max() < 200
    for k, w in enumerate(wls):
        # Each of the 12 solves leaves 1e-14 ||b|| at most in either run (smallest eigenvalue 1); the
        # explicit terms of later nodes see it through dt D L, whose norm is below kappa - 1.
        kappa = 1.0 + 8.0 * w.dt * w.sigma / (w.chi * w.Cm) / w.h**2 * (1.5 if w.nz > 1 else 1.0)
        tol = 12 * 2e-14 * kappa
        err = np.linalg.norm(got[k][0] - want[k][0]) / np.linalg.norm(want[k][0])
        assert err <= tol, (MESHES[k], err, tol)
        if scale == 1.0:
            _, alone, _ = step([w], scale)
            assert np.array_equal(alone[0], got[k]), MESHES[k]
    if scale == 1.0:
        rc, pers, it_p = step(wls, scale, persistent=(256, 96))
        assert rc == 0 and np.array_equal(it, it_p)
        assert all(np.array_equal(a, b) for a, b in zip(pers, got))


@pytest.mark.parametrize("cap", [1, 5])
def test_iteration_cap(cap):
    rc, _, it = step(tissues(), 1.0, cg_maxit=cap)
    assert rc == -3 and it.max() <= cap


def test_non_finite_tissue_is_reported():
    wls = tissues()[:2]
    b = P.Batch.from_workloads(wls, M_max=3)
    y = b.new_state()
    b.init_state(y, -75.0)
    b.tissue(y, 1)[0, 777] = float("inf")
    b.sweep(y, 0.0, wls[0].dt, 3, 4)
    rc, _, _ = b.residual()
    b.close()
    assert rc == -4
