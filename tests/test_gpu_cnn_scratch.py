"""Buffers of the learned post-equaliser.  Where the device has room for two gradient buffers
but not for one per layer, the handle is created all the same and its gradients are those of a
handle with all of them (the same BF16 values; the FP32 sums differ in the order of their
atomics).  A caller's gradient buffer that is not on a 16-byte boundary is filled like any
other, and nothing beside it is written."""
import pytest

from chain_helpers import ensure_built, rel_rms
from test_gpu_cnn import _data, _dev
from test_gpu_cnn_edges import _net

pytestmark = pytest.mark.gpu

LAYERS, K_MAX = 8, 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("K", [131, 5000])
def test_two_gradient_buffers(K):
    import torch
    z, t = _data(K, 41)
    z, t = _dev(z), _dev(t)
    roomy = _net(K_MAX, LAYERS)
    want = {}
    for tc in (1, 0):
        roomy.set_option("TCGEN05", tc)
        loss, g = roomy.grads(z, t)
        want[tc] = loss, roomy.unflatten(g.cpu().numpy())
    roomy.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # rows of 128 bytes: 7 activations, 2 gradients, 32 bytes twice; a handle with 5 more does not fit
    need = K_MAX * (9 * 128 + 64)
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - need - (256 << 20), dtype=torch.uint8, device="cuda")
    try:
        left, _ = torch.cuda.mem_get_info()
        assert need < left < need + K_MAX * 4 * 128
        net = _net(K_MAX, LAYERS)
    finally:
        del hold
        torch.cuda.empty_cache()
    for tc in (1, 0):
        net.set_option("TCGEN05", tc)
        loss, g = net.grads(z, t)
        g = net.unflatten(g.cpu().numpy())
        assert abs(loss - want[tc][0]) < 1e-9 * want[tc][0]
        for (dW, db), (rW, rb) in zip(g, want[tc][1]):
            assert rel_rms(dW, rW) < 1e-5 and rel_rms(db, rb) < 1e-5
    net.close()


@pytest.mark.parametrize("layers,offset", [(2, 1), (4, 1), (4, 2), (4, 3)])
def test_gradient_buffer_off_the_16_byte_boundary(layers, offset):
    import ctypes as ct
    import torch
    z, t = _data(777, 43)
    z, t = _dev(z), _dev(t)
    net = _net(1000, layers)
    want_loss, want = net.grads(z, t)
    buf = torch.full((net.n_params + 8,), 7.5, device="cuda")
    assert buf.data_ptr() % 16 == 0
    loss = ct.c_double()
    torch.cuda.synchronize()
    st = net.lib.rx_cnn_grads(net.h, z.data_ptr(), z.stride(0), t.data_ptr(), t.stride(0), 777,
                              buf.data_ptr() + 4 * offset, ct.byref(loss))
    assert st == 0 and abs(loss.value - want_loss) < 1e-9 * want_loss
    g, w = net.unflatten(buf[offset:offset + net.n_params].cpu().numpy()), net.unflatten(want.cpu().numpy())
    for (dW, db), (rW, rb) in zip(g, w):           # (FP32 atomics in another order)
        assert rel_rms(dW, rW) < 1e-5 and rel_rms(db, rb) < 1e-5
    assert torch.all(buf[:offset] == 7.5) and torch.all(buf[offset + net.n_params:] == 7.5)
    net.close()


def test_first_use_by_several_threads():
    # every convolution needs the driver's tensor-map entry point, looked up at the first use, and a
    # context, which a new thread has not bound: in a process of its own, so that this is the first
    import subprocess
    import sys
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = """
import sys, threading
sys.path[:0] = [%r, %r]
import torch
from test_gpu_cnn import _data, _dev
from test_gpu_cnn_edges import _net
z = _dev(_data(5000, 47)[0])
n = 8
nets = [_net(5000, 4) for _ in range(n)]
torch.cuda.synchronize()
gate, out, bad = threading.Barrier(n), [None] * n, []
def work(i):
    try:
        gate.wait()
        out[i] = nets[i].apply(z)
    except Exception as e:
        bad.append(repr(e))
ts = [threading.Thread(target=work, args=(i,)) for i in range(n)]
[t.start() for t in ts]
[t.join() for t in ts]
torch.cuda.synchronize()
assert not bad, bad
assert all(torch.equal(o, out[0]) for o in out)
""" % (root, os.path.join(root, "tests"))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
