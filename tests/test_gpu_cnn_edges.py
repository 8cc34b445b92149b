"""The tcgen05 path of the learned post-equaliser against its mma.sync path at the edges
of its tiles (128 symbols; 114 in the last layer; a halo of 7) and at the shortest
sequences, for every depth of network, after a longer call has left values behind the
sequence's end.

Both paths multiply the same BF16 values and add in FP32; they differ in the order of the
sums (1e-6), which moves a stored BF16 activation to its neighbour (2^-8) about once in
2000, one of the 960 terms of the next sum: 1e-4 of an output.  The bounds leave a factor
of ten; a gradient also meets a ReLU mask that such a value flips."""
import numpy as np
import pytest

from chain_helpers import ensure_built, rel_rms
from test_gpu_cnn import _data, _dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _net(K_max, layers, seed=3):
    from paper_2104_06311_gb300 import CNN
    rng = np.random.default_rng(seed)
    dims = [4] + [64] * (layers - 1) + [4]
    p = [(rng.standard_normal((15, a, b)) * np.sqrt(2.0 / (15 * a)), 0.05 * rng.standard_normal(b))
         for a, b in zip(dims[:-1], dims[1:])]
    net = CNN(K_max, layers=layers)
    net.set_params(p)
    return net


@pytest.mark.parametrize("layers", [2, 3, 4, 5])
@pytest.mark.parametrize("K", [1, 7, 15, 113, 114, 115, 127, 128, 129, 142, 143, 257, 699])
def test_tile_edges(K, layers):
    net = _net(1000, layers)
    zl, tl = _data(1000, 23)
    z, t = _data(K, 29)
    net.apply(_dev(zl))
    net.grads(_dev(zl), _dev(tl))
    y = net.apply(_dev(z)).cpu().numpy()
    loss, g = net.grads(_dev(z), _dev(t))
    g = net.unflatten(g.cpu().numpy())
    net.set_option("TCGEN05", 0)
    yr = net.apply(_dev(z)).cpu().numpy()
    lr, gr = net.grads(_dev(z), _dev(t))
    gr = net.unflatten(gr.cpu().numpy())
    z32 = z.astype(np.complex64)
    assert rel_rms(y - z32, yr - z32) < 1e-3
    assert abs(loss - lr) < 1e-3 * lr
    for (dW, db), (rW, rb) in zip(g, gr):
        assert rel_rms(dW, rW) < 1e-2 and rel_rms(db, rb) < 1e-2


def test_output_may_be_the_input():
    net = _net(3000, 4)
    z, _ = _data(3000, 31)
    y = net.apply(_dev(z))
    x = _dev(z)
    net.apply(x, out=x)
    assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
