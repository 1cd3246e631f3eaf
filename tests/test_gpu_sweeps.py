"""Gram-Schmidt sweeps whose last block sums the partial results and closes the
Arnoldi step: the tensor-core path's device-side GMRES cycle against its
host-driven one for restart lengths below, at and above eight vectors per
sweep, and batches at each chunk width of the vector kernels (one block per
problem up to 128 per problem) against the problems solved alone."""
import pytest
import torch

import tfde_inputs as inp
from gpu_helpers import relerr, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2511_21198_gb300 import build
    build.build()
    from paper_2511_21198_gb300 import tfde
    tfde.load()
    yield tfde
    tfde.tfde_stats_reset(False)


@pytest.mark.parametrize("n", [(8, 8, 8), (24, 40, 16), (128, 64, 72)])
@pytest.mark.parametrize("restart", [3, 8, 9, 64])
def test_device_cycle_matches_host_cycle(T, n, restart):
    h = T.tfde_assemble(T.make_params(n, (0.3, 0.6, 0.8), (1.0,) * 3, (0.2, 0.5, 0.8), 0.1), T.TFDE_MIXED)
    try:
        b = to_dev(inp.uniform_vector((n[2], n[1], n[0]), 12))
        out = []
        for timed in (True, False, False):   # the second device-side solve repeats the first
            T.tfde_stats_reset(timed)
            x = torch.zeros_like(b)
            info = T.tfde_pgmres(h, b, x, restart, 1e-11, 2000)
            assert info.relres <= 1e-11
            out.append((info.iters, to_host(x)))
        # sums in another order: a step at most per cycle
        assert abs(out[0][0] - out[1][0]) <= 1 + out[0][0] // restart
        assert abs(out[1][0] - out[2][0]) <= 1
        for _, x in out[1:]:   # all meet 1e-11 on a well-conditioned system
            assert relerr(x, out[0][1]) < 1e-9
    finally:
        T.tfde_stats_reset(False)
        T.tfde_destroy(h)


@pytest.mark.parametrize("sizes", [(8, 8), (8, 16, 64), (128, 128, 128, 128, 128, 32), (128,) * 10 + (8,)])
def test_batch_chunks_match_single_problems(T, sizes):
    prm, us = [], []
    for i, n in enumerate(sizes):
        km = (1.0, 1.2, 0.8) if i % 3 == 2 else (0.5, 0.6, 0.7)
        prm.append(T.make_params((n,) * 3, (0.3, 0.5, 0.7), (1.0, 1.2, 0.8), km, 0.05))
        us.append(to_dev(inp.smoothed_uniform((n,) * 3, i % 4)))
    ref = [u.clone() for u in us]
    B = T.tfde_batch_create(prm, 20)
    try:
        for m in range(2):
            T.tfde_batch_cn_advance(B, us, None, m == 0, 1e-11)
    finally:
        T.tfde_batch_destroy(B)
    for p, u, w in zip(prm, us, ref):
        h = T.tfde_assemble(p, T.TFDE_MIXED)
        try:
            for m in range(2):
                T.tfde_cn_advance(h, w, None, m == 0, 1e-11)
        finally:
            T.tfde_destroy(h)
        assert float(torch.linalg.norm(u - w) / torch.linalg.norm(w)) < 1e-9
