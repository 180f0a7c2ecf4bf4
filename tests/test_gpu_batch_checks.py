"""Batched Chebyshev solves whose residual checks follow one another pass by pass: with a spectrum of
1 + 1e-5 a correction is one FP32 iteration that checks, its defect checks in the next pass, and so does
the next correction.  The partial sums of one check must not meet those of the next, so every launch
shape and every repetition gives the same bits, a tissue's own alone as well, and the CG's result."""
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


MESHES = [(512, 509, 1), (129, 128, 1), (40, 41, 30), (300, 217, 1), (64, 64, 1)]


def tissues(stiff):
    """Pure diffusion: no ionic currents, no stimulus."""
    wls = []
    for k, mesh in enumerate(MESHES):
        w = I.hh_batch(n=1, seed=50 + k, side=(48, 48), sigma=(0.05 * stiff, 0.3 * stiff))[0].with_mesh(*mesh)
        w.params = np.array(w.params, dtype=np.float64)
        w.params[:3] = 0.0
        w.amp = np.zeros_like(w.amp)
        wls.append(w)
    return wls


def run(wls, shape=None, persistent=None, reps=1, **kw):
    b = P.Batch.from_workloads(wls, M_max=3, **kw)
    if shape:
        b.set_shape(*shape)
    if persistent:
        b.set_persistent(True, *persistent)
    y, y0 = b.new_state(), b.new_state()
    b.init_state(y0, -75.0)
    for k, w in enumerate(wls):
        v = np.random.default_rng([9, w.nx, w.ny, w.nz]).uniform(4.0, 6.0, size=w.n_nodes)
        b.tissue(y0, k)[0] = torch.from_numpy(v).cuda()
    out = []
    for _ in range(reps):
        y.copy_(y0)
        b.sweep(y, 0.0, wls[0].dt, 3, 4)
        rc, _, _ = b.residual()
        assert rc == 0
        out.append(([b.tissue(y, k).cpu().numpy().copy() for k in range(len(wls))], b.stats(4, 3).copy()))
    b.close()
    return out


@pytest.mark.parametrize("stiff", [1e-5, 1e-4, 1e-2])
def test_consecutive_checks(stiff):
    wls = tissues(stiff)
    runs = run(wls, reps=6)
    for shape in ((1, 512, 1), (1, 256, 4), (2, 256, 1)):
        runs += run(wls, shape=shape, reps=3)
    for pers in ((512, 128), (256, 96)):
        runs += run(wls, persistent=pers, reps=3)
    first, it = runs[0]
    for got, it_n in runs[1:]:
        assert np.array_equal(it, it_n)
        assert all(np.array_equal(a, b) for a, b in zip(got, first))
    for k in range(len(wls)):
        alone, _ = run([wls[k]])[0]
        assert np.array_equal(alone[0], first[k]), MESHES[k]
    want, _ = run(wls, solver="cg")[0]
    for k in range(len(wls)):
        # 12 solves to 1e-14 ||b|| in either run; the explicit terms' factor kappa - 1 is below 1 here
        err = np.linalg.norm(first[k][0] - want[k][0]) / np.linalg.norm(want[k][0])
        assert err <= 12 * 2e-14 * 2.0, (MESHES[k], err)


@pytest.mark.parametrize("cap", [2**31 - 1, 2**31 - 9])
def test_largest_iteration_caps(cap):
    # cg_maxit is any int from 1 on: the largest ones change nothing
    wls = tissues(1.0)
    want, it = run(wls)[0]
    for persistent in (None, (512, 128)):
        got, it_n = run(wls, persistent=persistent, cg_maxit=cap)[0]
        assert it.min() >= 1 and np.array_equal(it, it_n)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))


def test_most_tissues_of_every_launch_shape():
    # 128 single-tile tissues per block of one 512-thread block per SM, but for the last: a block whose warps take
    # quarters of tiles touches 129
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = I.hh_sheet_32().with_mesh(3, 2, 1)
    w.boxes = np.array([[0, 1, 0, 1, 0, 1]], np.int32)
    b = P.Batch.from_workloads([w] * (128 * sms - 1), M_max=1)
    y0, y = b.new_state(), b.new_state()
    b.init_state(y0, -70.0)
    y0[0] += torch.rand(y0.shape[1], dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    y.copy_(y0)
    b.sweep(y, 0.0, w.dt, 1, 2)
    assert b.residual()[0] == 0
    want = y.clone()
    for shape in ((1, 512, 1), (1, 256, 1)):
        b.set_shape(*shape)
        y.copy_(y0)
        b.sweep(y, 0.0, w.dt, 1, 2)
        assert b.residual()[0] == 0 and torch.equal(y, want)
    for threads in (512, 256):
        b.set_persistent(True, threads, 128)
        y.copy_(y0)
        b.sweep(y, 0.0, w.dt, 1, 2)
        assert b.residual()[0] == 0 and torch.equal(y, want)
    b.close()
    # a batch that one of the shapes cannot take is refused
    with pytest.raises(P.EsdcError) as e:
        P.Batch.from_workloads([w] * (256 * sms), M_max=1)
    assert e.value.code == -6
