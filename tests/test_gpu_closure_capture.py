"""The scratch of lbm_closure_loss_grad, in processes of their own: calls of several threads, the
first call of the process among them, while another thread captures a CUDA graph; and a call after
the device's context was reset, whose memory nothing may be kept of."""
import subprocess
import sys

import pytest

from tests.conftest import ROOT

pytestmark = pytest.mark.gpu

CAPTURE = """
import ctypes, threading
import torch
from paper_2305_09910_gb300 import lbm
n, threads = 4096, 8
g = torch.Generator(device="cuda").manual_seed(3)
p = torch.randn(1345, device="cuda", generator=g) * 0.1
x = torch.randn(n, 7, device="cuda", generator=g)
s, t, w = (torch.rand(n, device="cuda", generator=g) for _ in range(3))
grads = [torch.zeros(1345, device="cuda") for _ in range(threads)]
streams = [torch.cuda.Stream() for _ in range(threads)]
a = torch.zeros(8, device="cuda")
torch.cuda.synchronize()
losses, errors = [None] * threads, []
def call(k):
    try:
        for _ in range(20):
            losses[k] = lbm.lbm_closure_loss_grad(p, x, t, s, w, n, 0, 1, 0.1, grads[k],
                                                  stream=ctypes.c_void_p(streams[k].cuda_stream))
    except Exception as e:
        errors.append(e)
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, capture_error_mode="thread_local"):
    a.add_(1.0)
    work = [threading.Thread(target=call, args=(k,)) for k in range(threads)]
    [th.start() for th in work]
    [th.join() for th in work]
    a.add_(1.0)
graph.replay()
torch.cuda.synchronize()
assert not errors, errors
assert a.eq(2.0).all()
want = torch.zeros(1345, device="cuda")
loss = lbm.lbm_closure_loss_grad(p, x, t, s, w, n, 0, 1, 0.1, want)
for k in range(threads):
    assert abs(losses[k] - loss) <= 1e-12 * loss, (k, losses[k], loss)  # float64 sums, another order
    # float32 sums and atomics in another order: 4e-6 of the magnitudes summed, which are a few times
    # the largest component here
    assert (grads[k] - want).abs().max().item() <= 4e-5 * want.abs().max().item(), k
print("ok")
"""

RESET = """
import ctypes
import numpy as np
from paper_2305_09910_gb300 import lbm
cu = ctypes.CDLL("libcuda.so.1")
def ok(r):
    assert r == 0, r
def upload(a):
    d = ctypes.c_uint64(0)
    ok(cu.cuMemAlloc_v2(ctypes.byref(d), ctypes.c_size_t(a.nbytes)))
    ok(cu.cuMemcpyHtoD_v2(d, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes)))
    return ctypes.c_void_p(d.value)
rng = np.random.default_rng(5)
n = 1000
host = [a.astype(np.float32) for a in (rng.normal(0, 0.1, 1345), rng.normal(0, 1, 7 * n), rng.random(n), rng.random(n),
                                       rng.random(n), np.zeros(1345))]
ok(cu.cuInit(0))
def call():
    ctx = ctypes.c_void_p(0)
    ok(cu.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), 0))
    ok(cu.cuCtxSetCurrent(ctx))
    p, x, t, s, w, g = (upload(a) for a in host)
    loss = ctypes.c_double(0.0)
    st = lbm.load().lbm_closure_loss_grad(p, x, t, s, w, n, 0, 1, 0.1, g, ctypes.byref(loss), None)
    assert st == 0, lbm.load().lbm_last_error(None)
    return loss.value
first = call()
ok(cu.cuDevicePrimaryCtxReset_v2(0))
assert abs(call() - first) <= 1e-12 * first
print("ok")
"""


@pytest.mark.parametrize("program", [CAPTURE, RESET], ids=["capture", "reset"])
def test_scratch_of_the_loss_gradient(program):
    r = subprocess.run([sys.executable, "-c", program], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), (r.returncode, r.stdout[-500:], r.stderr[-2000:])


def test_scratch_slots_are_left_as_they_were_found():
    """Calls in a row, of different sizes and of no sample, and with all weights zero between: a slot holds
    nothing of the call before."""
    import torch

    from paper_2305_09910_gb300 import lbm

    g = torch.Generator(device="cuda").manual_seed(9)
    n = 5000
    p = torch.randn(1345, device="cuda", generator=g) * 0.1
    x = torch.randn(n, 7, device="cuda", generator=g)
    s, t, w = (torch.rand(n, device="cuda", generator=g) for _ in range(3))
    grad, dev = torch.zeros(1345, device="cuda"), torch.zeros(1, device="cuda", dtype=torch.float64)
    first = {}
    for k in range(3):
        for m in (5000, 1, 0, 33, 640):
            loss = lbm.lbm_closure_loss_grad(p, x, t, s, w, m, 0, 1, 0.1, grad)
            assert abs(loss - first.setdefault(m, loss)) <= 1e-12 * first[m]  # float64 sums in another order
            assert lbm.lbm_closure_loss_grad(p, x, t, s, 0 * w, m, 0, 1, 0.1, grad) == 0.0
    assert first[0] == 0.0 and first[5000] > 0.0
