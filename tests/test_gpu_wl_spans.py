"""Segments and pretraining far longer than the buffers (both are accepted up to 2^30):
outputs against the FP64 reference (oracle/wl.py), and a call's time follows what the
buffer holds, not the lengths that were set."""
import numpy as np
import pytest

from oracle import wl as W
from test_gpu_wl import _built, _check, _run_both  # noqa: F401  (_built: module fixture)
from test_gpu_wl_edges import _samples

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mod", ["qpsk", "16qam"])
@pytest.mark.parametrize("seg,pre,acq,bufs", [
    (1 << 16, 0, 0, [40, 17]),
    (1 << 20, 1 << 20, 32, [40, 300, 33]),
    (16, 1 << 20, 0, [300, 555]),
    (64, 4096, 16, [1000, 47]),
])
def test_lengths_above_the_buffer(mod, seg, pre, acq, bufs):
    cuts = [0] + [2 * int(c) for c in np.cumsum(bufs)]
    x = _samples(mod, sum(bufs), 2104063177 + seg % 1000 + pre % 999)
    p = W.WLParams(mod=mod, mu=2e-3, seg_len=seg, pretrain=pre, acq=acq)
    _check(_run_both(x, cuts, p, 2 if mod == "qpsk" else 4), mod)


@pytest.mark.parametrize("seg,pre", [(1 << 20, 0), (16, 1 << 20), (1 << 20, 1 << 20)])
def test_time_follows_the_buffer(seg, pre):
    # 40 symbols take some 10 us; half a million symbols of empty chunks would take over 10 ms
    import torch
    from paper_2104_06311_gb300 import WLEqualiser
    eq = WLEqualiser(4, 40, seg_len=seg, pretrain=pre, acq=0)
    x = torch.from_numpy(_samples("16qam", 40, 5).astype(np.complex64)).cuda()
    ms = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        eq.process(x)
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    eq.close()
    assert min(ms) < 2.0, ms
