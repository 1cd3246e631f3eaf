"""The weight gradient's sums over the grid carry at least 53 bits.  An input of
ones through layers that pass it on, and a last layer of zeros, make the last
layer's gradient the plain sum of the output gradients, which the targets set:
five single points whose largest and smallest are 52 binary places apart and
whose large ones cancel.  In 53 bits the sum is exact in any order; every
chunk that is summed in FP32 holds one of them."""
import itertools

import numpy as np
import pytest

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2511_21198_gb300 import build
    build.build()
    from paper_2511_21198_gb300 import tfde
    tfde.load()
    return tfde


# 145 tiles of one block on as many CTAs; 545 tiles of four, up to four per CTA
@pytest.mark.parametrize("n", [(32, 32, 16), (64, 64, 64)])
@pytest.mark.parametrize("order", list(itertools.permutations(range(5)))[::17])
def test_sums_keep_53_bits(T, n, order):
    from paper_2511_21198_gb300 import warmstart as W
    flat = np.zeros(4 * W.PSZ, dtype=np.float32)
    for l in range(3):   # channel 0 passed on
        flat[l * W.PSZ:l * W.PSZ + W.WSZ].reshape(16, 16, 27)[0, 0, 13] = 1.0
    N = n[0] * n[1] * n[2]   # a power of two: the scale 2 / N is exact
    values = [2.0**30, 2.0**4, 2.0**-22, -2.0**4, -2.0**30]
    un = np.ones((n[2], n[1], n[0]))
    step = n[2] // 6
    for k, z in zip(order, range(2, n[2] - 2, step)):
        un[z, n[1] // 2, n[0] // 2] = 1.0 - values[k] * N / 2   # dZ = 2 (0 - (un - u) / max |u|) / N
    net = T.tfde_cnn_create(n)
    try:
        T.tfde_cnn_set_params(net, flat)
        T.tfde_cnn_accumulate(net, to_dev(np.ones_like(un)), None, [0.0] * 9, to_dev(un))
        g = T.tfde_cnn_get_grads(net)
    finally:
        T.tfde_cnn_destroy(net)
    last = g[3 * W.PSZ:]
    assert np.all(last[:W.WSZ].reshape(16, 16, 27)[0, 0] == 2.0**-22), last[:27]
    assert last[W.WSZ] == 2.0**-22
