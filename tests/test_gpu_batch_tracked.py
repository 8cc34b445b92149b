"""A batch of uneven channels with frequency tracking on (the default) and teams of different
sizes: every channel's bits, symbols and LLRs are those of a receiver of its own, bit for bit."""
import numpy as np
import pytest

import linksim as L
from chain_helpers import ensure_built, make_receiver, rx_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_channels_equal_their_own_receivers():
    import torch
    from paper_2104_06311_gb300 import Batch
    lens = [1 << 15, 150_000, 40_007, 1 << 17, 20_000, 90_003, 33_000, 65_536 + 16_384, 50_001, 120_000]
    links = [L.Link(mod="16qam" if i % 3 == 1 else "qpsk", baud=10e9 + 2e9 * i, n_sym=n, L_km=300.0 + 400.0 * i,
                    snr_db=19.0 if i % 3 == 1 else 12.0, adc="int8", fo_hz=0.0 if i % 3 == 1 else 60e6, seed=2104063220 + i)
             for i, n in enumerate(lens)]
    gens = [L.generate(lk) for lk in links]
    xs = [torch.from_numpy(np.ascontiguousarray(g.samples)).cuda() for g in gens]
    b = Batch([dict(baud=lk.baud, L_km=lk.L_km, in_scale=g.in_scale, max_samples=x.shape[0],
                    mod_bits=4 if lk.mod == "16qam" else 2) for lk, g, x in zip(links, gens, xs)])
    teams = [int(b.get_param(i, "EQ_TEAM")) for i in range(len(lens))]
    assert len(set(teams)) > 1 and max(teams) > 2, teams
    outs = b.alloc_outs(xs, llr=True, sym=True)
    b.process(xs, outs)
    b.sync()
    for i, (lk, g, x, o) in enumerate(zip(links, gens, xs, outs)):
        p = rx_params(lk, g.in_scale, fft_n=int(b.get_param(i, "FFT_N")), overlap=int(b.get_param(i, "OVERLAP")))
        rx = make_receiver(p, LLR_OUT=1, SYM_OUT=1, EQ_WARPS=4)
        r = rx.run_stream(x, llr=True, sym=True)
        K, m = r["n"], p.bits
        assert K == o["n"] == lk.n_sym
        assert torch.equal(r["bits"][:, :K * m // 32], o["bits"][:, :K * m // 32]), i
        assert torch.equal(r["sym"][:, :K], o["sym"][:, :K]), i
        assert torch.equal(r["llr"][:, :K * m], o["llr"][:, :K * m]), i
        rx.close()
    b.close()
