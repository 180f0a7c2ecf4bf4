"""The FP32 corrections' acceptance test: a correction's residual is kept by recursion in FP32, and the solve accepts
it with an allowance for what that misses of r - B e.  Here the same iteration in numpy's float32 on the spectra that
are refined (kappa up to 64): the allowance covers what it misses.  On the GPU: whatever the iteration cap cuts off,
a solve that reports success has met its stop test."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def constant(name):
    src = open(os.path.join(ROOT, "paper_2405_19994_gb300", "csrc", "esdc_internal.h")).read()
    return float(re.search(r"#define %s (\S+)" % name, src).group(1))


def op(v, g):
    """(I - g L) v, mirrored faces, in v's precision."""
    s, c = np.zeros_like(v), np.zeros(v.shape, v.dtype)
    for ax in range(v.ndim):
        lo, hi = [slice(None)] * v.ndim, [slice(None)] * v.ndim
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        s[tuple(lo)] += v[tuple(hi)]
        s[tuple(hi)] += v[tuple(lo)]
        c[tuple(lo)] += 1
        c[tuple(hi)] += 1
    g = v.dtype.type(g)
    return (v.dtype.type(1) + g * c) * v - g * s


def correction(r0, g, kappa, f):
    F = np.float32
    theta, delta = 0.5 * (kappa + 1.0), 0.5 * (kappa - 1.0)
    s1 = theta / delta
    rho, q = 1.0 / s1, (np.sqrt(kappa) - 1.0) / (np.sqrt(kappa) + 1.0)
    r = r0.astype(F)
    d, e = r * F(1.0 / theta), np.zeros(r.shape, F)
    for _ in range(int(np.ceil(np.log(0.5 * f) / np.log(q)))):
        bd = op(d, g)
        e, r = e + d, r - bd
        rn = 1.0 / (2.0 * s1 - rho)
        d = F(rn * rho) * d + F(2.0 * rn / delta) * r
        rho = rn
    return e.astype(np.float64), r.astype(np.float64)


@pytest.mark.parametrize("kappa", [4.0, 16.0, 33.0, 48.0, 63.9])
@pytest.mark.parametrize("shape", [(300, 300), (48, 48, 48), (60000,)])
def test_allowance_covers_the_recursion(kappa, shape):
    allow = max(constant("ESDC_REF_ALLOW_MIN"), constant("ESDC_REF_ALLOW_KAPPA") * kappa)
    x = np.meshgrid(*[np.linspace(0.0, 1.0, n) for n in shape], indexing="ij")
    smooth = sum(np.cos(np.pi * (i + 2) * c) for i, c in enumerate(x))
    rough = np.random.default_rng(1).normal(size=shape)
    spike = np.zeros(shape)
    spike[tuple(n // 3 for n in shape)] = 1.0
    front = 1.0 / (1.0 + np.exp((x[-1] - 0.4) * 200.0))
    g = (kappa - 1.0) / (4.0 * len(shape))
    for r0 in (smooth, rough, spike, front, 1.0 + 1e-3 * smooth):
        e, r = correction(r0, g, kappa, 3.2e-6)
        miss = np.linalg.norm(r0 - op(e, g) - r) / np.linalg.norm(r0)
        assert miss <= allow, (miss, allow)


@pytest.mark.gpu
@pytest.mark.parametrize("kappa", [20.0, 60.0])
@pytest.mark.parametrize("tol", [4e-5, 1e-6])
def test_reported_success_meets_the_stop_test(kappa, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_19994_gb300 as P
    from paper_2405_19994_gb300 import inputs as I
    wl = I.hh_aniso_slab().with_mesh(100, 80, 51)          # 408,000 nodes: above the refinement's border
    wl.layers = None
    x = np.meshgrid(*[np.linspace(0.0, 1.0, n) for n in (wl.nz, wl.ny, wl.nx)], indexing="ij")
    b = (np.cos(2.0 * np.pi * x[0]) + np.cos(3.0 * np.pi * x[1]) + np.cos(4.0 * np.pi * x[2])).reshape(-1)
    g = (kappa - 1.0) / 12.0 * wl.h**2
    bt, done = torch.from_numpy(b).cuda(), 0
    for cap in range(1, 70):
        s = P.Solver.from_workload(wl, solver="cheb", tol_cg=tol, cg_maxit=cap)
        v = torch.zeros_like(bt)
        try:
            s.diffusion_solve(g, bt, v)
        except P.EsdcError as e:
            assert e.code == -3
            continue
        done += 1
        r = b - op(v.cpu().numpy().reshape(wl.nz, wl.ny, wl.nx), g / wl.h**2).reshape(-1)
        # this residual's own rounding is 1e-14 of ||b||
        assert np.linalg.norm(r) <= (1.0 + 1e-6) * tol * np.linalg.norm(b), cap
    assert done > 0
