"""A recording gives the same bits, symbols and LLRs however its calls are cut into
pipeline pieces and phase-search chunks: one call in 1 and 12 pieces and in the number
that the call's length chooses, and calls short enough for the finest chunks.  The noise
variance is a sum over chunks of FP32 partial sums of at most 256 terms: 256 x 2^-24
bounds either sum, twice that and a few roundings the LLRs' relative difference."""
import numpy as np
import pytest

import linksim as L
from chain_helpers import ensure_built, make_receiver, rx_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("mod,nb", [("qpsk", 16), ("16qam", 64), ("qpsk", 7)])
def test_pieces_and_chunks(mod, nb):
    import torch
    lk = L.Link(mod=mod, n_sym=600_000, L_km=500.0, snr_db=13.0 if mod == "qpsk" else 20.0, seed=2104063161)
    g = L.generate(lk)
    p = rx_params(lk, g.in_scale, fo_track=mod == "qpsk")
    x = torch.from_numpy(g.samples).cuda()
    outs = []
    for chunk, kw in ((None, {}), (None, dict(PIPELINE=1)), (None, dict(PIPELINE=12)), (150_000, {})):
        rx = make_receiver(p, LLR_OUT=1, SYM_OUT=1, BPS_HALFWIN=nb, **kw)
        o = rx.run_stream(x, chunk=chunk, llr=True, sym=True)
        outs.append({k: (v.cpu().numpy() if k != "n" else v) for k, v in o.items() if k in ("bits", "llr", "sym", "n")})
        rx.close()
    a = outs[0]
    K, m = a["n"], 2 if mod == "qpsk" else 4
    assert K == lk.n_sym
    for b in outs[1:]:
        assert b["n"] == K
        assert np.array_equal(a["bits"][:, :K * m // 32], b["bits"][:, :K * m // 32])
        assert np.array_equal(a["sym"][:, :K], b["sym"][:, :K])
        la, lb = a["llr"][:, :K * m], b["llr"][:, :K * m]
        assert np.max(np.abs(la - lb) / (np.abs(la) + 1e-30)) <= (2 * 256 + 4) * 2.0 ** -24


@pytest.mark.parametrize("mod,nb,seed", [("16qam", 7, 1), ("16qam", 24, 2), ("qpsk", 7, 3), ("qpsk", 50, 4), ("16qam", 41, 5),
                                         ("qpsk", 0, 6), ("16qam", 32, 7)])
def test_near_ties_fall_alike(mod, nb, seed):
    # half windows of the sliding pass (and one of the register blocks), at a noise that makes
    # near ties of two angles common: every angle the same, so every symbol
    import torch
    lk = L.Link(mod=mod, n_sym=600_000, L_km=200.0, snr_db=11.0 if mod == "qpsk" else 17.0, seed=2104063190 + seed)
    g = L.generate(lk)
    p = rx_params(lk, g.in_scale, fo_track=mod == "qpsk")
    x = torch.from_numpy(g.samples).cuda()
    want = None
    for chunk, kw in ((None, dict(PIPELINE=1)), (None, {}), (None, dict(PIPELINE=12)), (150_000, {}), (400_002, {})):
        rx = make_receiver(p, SYM_OUT=1, BPS_HALFWIN=nb, **kw)
        o = rx.run_stream(x, chunk=chunk, sym=True)
        got = (o["bits"].cpu().numpy(), o["sym"][:, :o["n"]].cpu().numpy())
        rx.close()
        if want is None:
            want = got
        assert np.array_equal(got[1], want[1]), (chunk, kw, int((got[1] != want[1]).sum()))
        assert np.array_equal(got[0], want[0])


@pytest.mark.parametrize("mod,nb,form", [("qpsk", 16, 1), ("16qam", 64, 1), ("16qam", 16, 2), ("qpsk", 24, 1), ("16qam", 7, 1)])
def test_llrs_do_not_depend_on_the_cut(mod, nb, form):
    # the noise variance is summed over fixed spans of symbols, so the LLRs are the same to the
    # last bit in one call, in any number of pieces and in calls
    import torch
    lk = L.Link(mod=mod, n_sym=600_000, L_km=300.0, snr_db=13.0 if mod == "qpsk" else 20.0, seed=2104063200 + nb)
    g = L.generate(lk)
    p = rx_params(lk, g.in_scale, fo_track=mod == "qpsk")
    x = torch.from_numpy(g.samples).cuda()
    m = 2 if mod == "qpsk" else 4
    want = None
    for chunk, kw in ((None, dict(PIPELINE=1)), (None, {}), (None, dict(PIPELINE=12)), (150_000, {}), (700_002, {})):
        rx = make_receiver(p, LLR_OUT=form, BPS_HALFWIN=nb, **kw)
        o = rx.run_stream(x, chunk=chunk, llr=True)
        got = o["llr"][:, :o["n"] * m].clone()
        rx.close()
        want = got if want is None else want
        assert torch.equal(got, want), (chunk, kw)
