"""The device-side iteration loops of the FP64 and ragged-grid solves against
the host-driven iterations (taken while per-launch timing is on): same
iteration counts and solutions, iteration limits, restart lengths that change
between solves, and different iterates and streams on one problem."""
import numpy as np
import pytest
import torch

from oracle import tfde_oracle as o
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


def problem(T, n, sym, mixed):
    d, kp = (0.4, 0.55, 0.7), (1.0, 1.3, 0.8)
    km = kp if sym else (0.5, 0.7, 1.4)
    op = o.Problem(n=(n[0], n[1], max(1, n[2])), delta=d, kp=kp, km=km, dt=0.02, dim=3 if n[2] else 2)
    return op, T.tfde_assemble(T.make_params(n, d, kp, km, 0.02), T.TFDE_MIXED if mixed else T.TFDE_FP64)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n", [(16, 16, 16), (13, 9, 21), (1, 3, 2), (37, 45, 0), (97, 20, 11)])
def test_pcg_loop_matches_host_iterations(T, n, mixed):
    if mixed and n == (16, 16, 16):
        n = (15, 16, 17)   # a grid of the ragged path
    op, h = problem(T, n, True, mixed)
    try:
        b = to_dev(inp.uniform_vector(op.shape, 3))
        out = []
        for timed in (True, False, False):   # the last one on another stream and iterate
            T.tfde_stats_reset(timed)
            x = torch.zeros_like(b)
            s = torch.cuda.Stream() if len(out) == 2 else torch.cuda.current_stream()
            s.wait_stream(torch.cuda.current_stream())
            info = T.tfde_pcg(h, b, x, 1e-11, 500, s)
            torch.cuda.synchronize()
            assert info.relres <= 1e-11
            out.append((info.iters, to_host(x)))
        assert out[0][0] == out[1][0] == out[2][0]
        # both solutions meet 1e-11; the well-conditioned system keeps them that close
        assert relerr(out[1][1], out[0][1]) < 1e-9 and relerr(out[2][1], out[1][1]) < 1e-12
        info = T.tfde_pcg(h, b, torch.zeros_like(b), 1e-14, 2, check=False)
        assert info.iters <= 2 and (info.status == T.TFDE_ENOCONV or info.relres <= 1e-14)
        zero = torch.zeros_like(b)
        assert T.tfde_pcg(h, zero, x, 1e-11, 500).iters == 0 and float(x.abs().max()) == 0.0
        bad = b.clone()
        bad.view(-1)[0] = float("inf")
        assert T.tfde_pcg(h, bad, torch.zeros_like(b), 1e-11, 500, check=False).status == T.TFDE_ENAN
    finally:
        T.tfde_stats_reset(False)
        T.tfde_destroy(h)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n", [(13, 9, 21), (37, 45, 0), (97, 20, 11)])
def test_gmres_loop_matches_host_iterations(T, n, mixed):
    op, h = problem(T, n, False, mixed)
    try:
        b = to_dev(inp.uniform_vector(op.shape, 4))
        for restart in (20, 5, 64):   # shorter, then longer than the first: the basis grows
            out = []
            for timed in (True, False):
                T.tfde_stats_reset(timed)
                x = torch.zeros_like(b)
                info = T.tfde_pgmres(h, b, x, restart, 1e-11, 2000)
                assert info.relres <= 1e-11
                out.append((info.iters, to_host(x)))
            # the two Gram-Schmidt variants round differently: a step at most per cycle
            assert abs(out[0][0] - out[1][0]) <= 1 + out[0][0] // restart
            assert relerr(out[1][1], out[0][1]) < 1e-9
        info = T.tfde_pgmres(h, b, torch.zeros_like(b), 20, 1e-14, 3, check=False)
        assert info.iters <= 3
    finally:
        T.tfde_stats_reset(False)
        T.tfde_destroy(h)
