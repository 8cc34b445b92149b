"""A reset on one stream, the next recording on another: the new stream's work comes behind
the reset, ordered on the device (binding a stream does not wait on the host), also when
the earlier stream is still busy."""
import time

import numpy as np
import pytest

from chain_helpers import ensure_built
from test_gpu_wl_edges import _samples

pytestmark = pytest.mark.gpu

BUSY = 400_000_000      # clock cycles that the earlier stream spins: about 0.2 s


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_widely_linear():
    import torch
    from paper_2104_06311_gb300 import WLEqualiser
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    eq = WLEqualiser(4, 4000, stream=s1, acq=1024)
    bind = lambda s: eq.lib.rx_wl_set_cuda_stream(eq.h, s.cuda_stream)
    x = torch.from_numpy(_samples("16qam", 4000, 11).astype(np.complex64)).cuda()
    other = torch.from_numpy(_samples("16qam", 3000, 12).astype(np.complex64)).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        want, want_z = (t.clone() for t in eq.process(x, want_z=True))
        eq.process(other)                       # other taps and other carried samples
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(BUSY)
        eq.reset()
    t0 = time.perf_counter()
    assert bind(s2) == 0
    took = time.perf_counter() - t0
    busy = not s1.query()
    with torch.cuda.stream(s2):
        got, got_z = eq.process(x, want_z=True)
    torch.cuda.synchronize()
    assert busy and took < 0.05, (busy, took)
    assert torch.equal(got, want) and torch.equal(got_z, want_z)
    eq.close()


@pytest.mark.parametrize("chunk", [None, 60_000])
def test_receiver(chunk):
    import torch
    import linksim as L
    from chain_helpers import make_receiver, rx_params
    lk = L.Link(n_sym=60_000, L_km=500.0, snr_db=12.0, seed=2104063181)
    g = L.generate(lk)
    rx = make_receiver(rx_params(lk, g.in_scale), SYM_OUT=1)
    x = torch.from_numpy(g.samples).cuda()
    rx.reserve(x.shape[0])
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()

    def calls():
        out = rx.alloc_out(lk.n_sym + 64, sym=True)
        pos = 0
        step = chunk or x.shape[0]
        for a in list(range(0, x.shape[0], step)) + [None]:
            _, n, _, _ = rx.process(None if a is None else x[a:a + step], out, sym_offset=pos)
            pos += n
        return out, pos

    rx.set_cuda_stream(s1)
    with torch.cuda.stream(s1):
        want, n = calls()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(BUSY)
        rx.reset()
    t0 = time.perf_counter()
    rx.set_cuda_stream(s2)
    took = time.perf_counter() - t0
    busy = not s1.query()
    with torch.cuda.stream(s2):
        got, m = calls()
    torch.cuda.synchronize()
    assert busy and took < 0.05, (busy, took)
    assert m == n == lk.n_sym
    assert torch.equal(got["bits"], want["bits"]) and torch.equal(got["sym"][:, :n], want["sym"][:, :n])
    rx.close()
