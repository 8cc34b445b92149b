"""Kramers-Kronig front end with the shortest buffers (odd and even window counts, buffers
inside the look-ahead and the history) against the FP64 reference (oracle/kk.py), for the
table-driven 8-bit form and the float one."""
import pytest

import linksim.kk as LK
from oracle import kk as K
from chain_helpers import rel_rms
from test_gpu_kk import TOL, _built, _stream  # noqa: F401  (_built: module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adc", ["int8", "f32"])
@pytest.mark.parametrize("bufs", [[1], [2], [1, 1, 1, 2, 3, 5], [7, 1, 2], [6, 4, 11]])
def test_short_buffers(adc, bufs):
    from paper_2104_06311_gb300 import KKFrontEnd
    n = 512 * sum(bufs)
    lk = LK.KKLink(n_sym=n // 4, adc=adc, L_km=1500.0, cspr_db=12.0, snr_db=24.0, seed=2104063151 + n)
    g = LK.generate(lk)
    cuts = [0]
    for b in bufs:
        cuts.append(cuts[-1] + 512 * b)
    fe = KKFrontEnd(lk.baud, lk.carrier_hz, lk.L_km, 512 * max(bufs))
    yg, fg = _stream(fe, g.samples, cuts, g)
    yo, Eo, _ = K.kk_frontend(g.samples, g.in_scale, g.in_offset, lk.baud, lk.sps, lk.carrier_hz, lk.L_km)
    assert rel_rms(fg, Eo) < TOL and rel_rms(yg, yo) < TOL


@pytest.mark.parametrize("at", [0, 100, 255])
def test_field_outside_the_stream_is_zero(at):
    # an infinite intensity takes the phase of its window from the samples around it; in front of the
    # stream there is no field all the same
    import torch
    from paper_2104_06311_gb300 import KKFrontEnd
    fe = KKFrontEnd(1e9, 0.516e9, 1000.0, 4096)
    x = torch.ones(4096, device="cuda")
    x[at] = float("inf")
    _, field = fe.process(x, field=True)
    assert torch.all(field[:fe.delay] == 0)


@pytest.mark.parametrize("carrier", [0.516321e9, 1.2345e9, 1.9990001e9])
@pytest.mark.parametrize("pos", [0, 512 * 123457])
def test_carrier_phase_off_the_recording_grid(carrier, pos):
    # intensity 1 everywhere: amplitude 1, phase 0, so the field is the carrier's turn alone.  Its
    # error: 24 significant bits of the half turn (pi 2^-25), one unit in the last place of the
    # sine and of the cosine (2^-24 each near 1) and of the product with the amplitude
    import math
    import numpy as np
    import torch
    from paper_2104_06311_gb300 import KKFrontEnd
    n = 8192
    fe = KKFrontEnd(1e9, carrier, 1000.0, n)
    fe.set_position(pos)
    _, field = fe.process(torch.ones(n, device="cuda"), field=True)
    f = field.cpu().numpy().astype(np.complex128)[fe.delay:]
    inc = int(carrier / 4e9 % 1.0 * 2.0 ** 64)                 # exact: a double's 53 bits
    turn = np.array([((pos + i) * inc % (1 << 64)) / 2.0 ** 64 for i in range(f.shape[0])])
    err = np.abs(f - np.exp(2j * np.pi * turn))
    print(f"carrier {carrier:.6g} from {pos}: max {err.max():.2e}")
    assert err.max() < math.pi * 2.0 ** -25 + math.sqrt(2) * 2 * 2.0 ** -24
