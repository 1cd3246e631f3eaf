"""The warm-start network's tiles against the oracle: grids whose tiles hold
one, two and four MMA blocks of 128 slots, staged as three runs per tile or
(long lines) as nine, with ragged last tiles."""
import numpy as np
import pytest

from oracle import cnn_oracle as C
import tfde_inputs as inp
from gpu_helpers import relerr, to_dev, to_host
from test_gpu_cnn import bf16_backward, bf16_forward, pad_channels, random_net

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2511_21198_gb300 import build
    build.build()
    from paper_2511_21198_gb300 import tfde
    tfde.load()
    return tfde


# slots from the first to the last interior point: 1 block per tile up to
# 38912 (152 SMs x 256), 2 up to 77824, 4 above; nine runs when a line and its
# neighbours do not fit twice in shared memory
@pytest.mark.parametrize("n", [(1, 1, 1), (3, 2, 41), (38, 30, 32), (61, 33, 40), (600, 3, 2), (1100, 8, 5)])
def test_tiles_match_oracle(T, n):
    from paper_2511_21198_gb300 import warmstart as W
    flat = random_net(W, 5)
    layers = W.flat_to_layers(flat)
    shape = tuple(reversed(n))
    u = inp.uniform_vector(shape, 15) - 0.3
    un = u + 0.05 * (inp.uniform_vector(shape, 16) - 0.5)
    coef = [0.3, 0.6, 0.8, 1.0, 1.5, 0.7, 0.5, 2.0, 1.2]
    net = T.tfde_cnn_create(n)
    try:
        T.tfde_cnn_set_params(net, flat)
        x0 = to_dev(np.zeros(shape))
        T.tfde_cnn_predict(net, to_dev(u), None, coef, x0)
        loss = T.tfde_cnn_accumulate(net, to_dev(u), None, coef, to_dev(un))
        g = W.flat_to_layers(T.tfde_cnn_get_grads(net))
    finally:
        T.tfde_cnn_destroy(net)
    x, s = C.input_channels(u, None, coef[0:3], coef[3:6], coef[6:9])
    x = pad_channels(x, W.CHANNELS[0])
    ref = bf16_forward(layers, x)[0]
    got = (to_host(x0) - u) / s
    # activations stored in BF16 (2^-9) on both sides: rounding-boundary flips only
    assert relerr(got, ref) < 1e-2
    L, gref = bf16_backward(layers, x, (un - u)[None] / s)
    assert abs(loss - L) <= 1e-3 * L
    for k in range(4):
        for a, b in ((g[k][0], gref[k][0]), (g[k][1], gref[k][1])):
            assert relerr(a, b) < 1e-2, k
