"""The first work of a process on a handle recorded into a CUDA graph: a step of a small mesh of either model, in
a process of its own (what a kernel needs on the device beforehand is uploaded once per process).  On torch's
streams and on a stream that waits for the legacy stream, where a synchronous copy inside the capture is an error."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes, types
import numpy as np, torch
import paper_2405_19994_gb300 as P
from paper_2405_19994_gb300 import inputs as I
from oracle import oracle as O
model, nx, ny, blocking = %r, %d, %d, %r
wl = (I.hh_sheet_32() if model == "hh" else I.syn19_slab()).with_mesh(nx, ny, 1)
wl.boxes = np.array([[0, 3, 0, 2, 0, 1]], np.int32)
s = P.Solver.from_workload(wl, M_max=3)
rest = np.array(O.ionic_rest(wl.model, wl.params, wl.V0))
y0 = np.repeat(rest[:, None], wl.n_nodes, axis=1)
y0[0] += 30.0 * np.exp(-(((np.arange(wl.n_nodes) %% nx) / nx - 0.3) ** 2) / 0.05)
start = s.new_state()
start[:, : wl.n_nodes] = torch.from_numpy(y0)
y = start.clone()
torch.cuda.synchronize()
if blocking:
    cu = ctypes.CDLL("libcuda.so.1")
    st, graph, ex = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    def ok(rc):
        assert rc == 0, rc
    ok(cu.cuStreamCreate(ctypes.byref(st), 0))
    ok(cu.cuStreamBeginCapture_v2(st, 0))
    s.sweep(y, 0.3, wl.dt, 3, 3, stream=types.SimpleNamespace(cuda_stream=st.value))
    ok(cu.cuStreamEndCapture(st, ctypes.byref(graph)))
    ok(cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)))
    replay = lambda: ok(cu.cuGraphLaunch(ex, st))
else:
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        s.sweep(y, 0.3, wl.dt, 3, 3)
    replay = g.replay
want = O.Monodomain(wl).step(y0, 0.3, wl.dt, 3, 3)[0]
got = []
for _ in range(3):
    y.copy_(start)
    torch.cuda.synchronize()
    replay()
    torch.cuda.synchronize()
    assert s.residual()[0] == 0
    got.append(y[:, : wl.n_nodes].cpu().numpy())
assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
# the bound of the one-launch steps' oracle tests
assert np.abs(got[0][0] - want[0]).max() < 1e-11 * np.abs(want[0]).max()
assert np.abs(got[0][1:] - want[1:]).max() < 1e-11
y.copy_(start)
s.sweep(y, 0.3, wl.dt, 3, 3)                       # outside a graph: from the set-up's table
plain = y[:, : wl.n_nodes].cpu().numpy()
assert np.abs(plain[0] - got[0][0]).max() < 1e-11 * np.abs(want[0]).max()
print("captured")
"""


@pytest.mark.parametrize("blocking", [False, True])
@pytest.mark.parametrize("model,nx,ny", [("hh", 37, 29), ("syn19", 37, 29), ("syn19", 32, 16)])
def test_first_step_in_a_graph(model, nx, ny, blocking):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", SCRIPT % (model, nx, ny, blocking)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]
