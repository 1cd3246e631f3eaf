"""Tile widths of the split contraction (256, 128 or 64 lines by the number of
tiles): operator and preconditioner in the inner arithmetic, and chained steps,
against the oracle on grids that take each width along each axis, with ragged
last tiles, per-block and merged input boxes, and one or several row blocks."""
import numpy as np
import pytest

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
    return tfde


GRIDS = [(8, 8, 8), (40, 32, 24), (64, 64, 64), (72, 200, 16), (136, 104, 88), (128, 128, 128), (448, 40, 24),
         (16, 448, 56)]


@pytest.mark.parametrize("n", GRIDS)
def test_widths_match_oracle(T, n):
    d, kp, km = (0.4, 0.55, 0.7), (1.0, 1.3, 0.8), (0.5, 0.7, 1.4)
    op = o.Problem(n=n, delta=d, kp=kp, km=km, dt=0.02)
    v = inp.uniform_vector(op.shape, 41)
    h = T.tfde_assemble(T.make_params(n, d, kp, km, 0.02), T.TFDE_MIXED)
    try:
        y = to_dev(np.zeros_like(v))
        # split BF16: 2^-16 per operand, three axis terms
        T.tfde_matvec(h, T.TFDE_OP_A | T.TFDE_OP_FAST, to_dev(v), y)
        assert relerr(to_host(y), o.apply_A(op, v)) < 1e-4
        # one BF16 operator term (2^-9) in each of the six sine transforms
        T.tfde_precond(h, to_dev(v), y)
        assert relerr(to_host(y), o.apply_Pinv(o.build_tau(op), v)) < 2e-2
        u = to_dev(v)
        for m in range(2):
            info = T.tfde_cn_advance(h, u, None, m == 0, 1e-11)
            assert info.relres <= 1e-11 and not info.fallback
    finally:
        T.tfde_destroy(h)
    h = T.tfde_assemble(T.make_params(n, d, kp, km, 0.02), T.TFDE_FP64)
    try:
        w = to_dev(v)
        for m in range(2):
            T.tfde_cn_advance(h, w, None, m == 0, 1e-12)
        assert relerr(to_host(u), to_host(w)) < 1e-9
    finally:
        T.tfde_destroy(h)


@pytest.mark.parametrize("sizes", [(8, 16), (32, 48, 64), (128, 128, 96, 64)])
def test_batch_widths_match_single_problems(T, sizes):
    import torch
    prm, us = [], []
    for i, n in enumerate(sizes):
        km = (1.0, 1.2, 0.8) if i % 2 else (0.5, 0.6, 0.7)
        prm.append(T.make_params((n,) * 3, (0.3, 0.5, 0.7), (1.0, 1.2, 0.8), km, 0.05))
        us.append(to_dev(inp.smoothed_uniform((n,) * 3, i)))
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
