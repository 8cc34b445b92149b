"""Widely-linear DD-LMS at the edges of its schedule against the FP64 reference
(oracle/wl.py): single symbols, ragged ends, segments shorter than the pretraining, a
first segment without any, more and fewer segments than a warp holds."""
import numpy as np
import pytest

from oracle import wl as W
from test_gpu_wl import _built, _check, _run_both  # noqa: F401  (_built: module fixture)

pytestmark = pytest.mark.gpu


def _samples(mod, n_sym, seed):
    rng = np.random.default_rng(seed)
    lv = np.array([-1.0, 1.0]) / np.sqrt(2) if mod == "qpsk" else np.array([-3.0, -1.0, 1.0, 3.0]) / np.sqrt(10)
    s = rng.choice(lv, n_sym) + 1j * rng.choice(lv, n_sym)
    x = np.zeros(2 * n_sym, complex)
    x[0::2] = s
    x[1::2] = 0.5 * (s + np.roll(s, -1))
    x += 0.05 * np.conj(x) + 0.02 * (rng.standard_normal(2 * n_sym) + 1j * rng.standard_normal(2 * n_sym))
    return x


@pytest.mark.parametrize("mod,seg,pre,acq,bufs", [
    ("qpsk", 16, 0, 0, [1, 17, 33]),
    ("16qam", 16, 48, 32, [40, 47, 512]),
    ("qpsk", 64, 128, 16, [16, 1, 300, 2000]),
    ("16qam", 256, 16, 0, [256 * 17 + 5, 31]),
    ("16qam", 32, 32, 1600, [1000, 1, 1030]),
    ("qpsk", 1024, 96, 48, [63, 1024 * 2 + 47, 64]),
])
def test_schedule_edges(mod, seg, pre, acq, bufs):
    cuts = [0] + [2 * int(c) for c in np.cumsum(bufs)]
    x = _samples(mod, sum(bufs), 2104063141 + seg)
    p = W.WLParams(mod=mod, mu=2e-3, seg_len=seg, pretrain=pre, acq=acq)
    _check(_run_both(x, cuts, p, 2 if mod == "qpsk" else 4), mod)
