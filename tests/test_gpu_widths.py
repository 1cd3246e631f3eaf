"""Every tile width of the split contraction against the oracle's preconditioner
and the FP64 path: grids on which the three rules (split input planes, the inner
PCG's hi-only passes in the grid basis, two contractions per launch) choose 256,
128 and 64 lines, apart from one another, with whole and ragged last tiles.
test_host_state_cpu.py holds the widths below against the library's rule."""
import numpy as np
import pytest

import tfde_inputs as inp
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

# grid: lines per tile along (x, y, z) of the split, hi-only and paired passes
WIDTHS = {
    (96, 96, 96): ((64, 128, 64), (64, 128, 64), (64, 128, 64)),
    (152, 152, 152): ((64, 128, 64), (128, 128, 128), (256, 256, 256)),
    (184, 184, 184): ((256, 256, 256), (256, 256, 256), (256, 256, 256)),   # ragged last tiles on x and z
    (192, 192, 192): ((256, 256, 256), (256, 256, 256), (256, 256, 256)),
    (200, 200, 200): ((128, 256, 128), (256, 256, 256), (256, 256, 256)),
}


@pytest.fixture(scope="module")
def T():
    from paper_2511_21198_gb300 import build
    build.build()
    from paper_2511_21198_gb300 import tfde
    tfde.load()
    return tfde


def rel(a, b):
    import torch
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n", list(WIDTHS))
def test_widths_match_fp64(T, n, sym):
    import torch
    d, kp = (0.4, 0.55, 0.7), (1.0, 1.3, 0.8)
    prm = T.make_params(n, d, kp, kp if sym else (0.5, 0.7, 1.4), 0.02)
    b = to_dev(inp.uniform_vector((n[2], n[1], n[0]), 51))

    def solve(h, x):
        return T.tfde_pcg(h, b, x, 1e-12, 500) if sym else T.tfde_pgmres(h, b, x, 20, 1e-12, 500)

    h = T.tfde_assemble(prm, T.TFDE_FP64)
    try:
        y, z, ref = torch.zeros_like(b), torch.zeros_like(b), torch.zeros_like(b)
        T.tfde_matvec(h, T.TFDE_OP_A, b, y)
        T.tfde_precond(h, b, z)
        solve(h, ref)
    finally:
        T.tfde_destroy(h)
    h = T.tfde_assemble(prm, T.TFDE_MIXED)
    try:
        v = torch.zeros_like(b)
        # split BF16: 2^-16 per operand, three axis terms
        T.tfde_matvec(h, T.TFDE_OP_A | T.TFDE_OP_FAST, b, v)
        assert rel(v, y) < 1e-4
        # one BF16 operator term (2^-9) in each of the six sine transforms
        T.tfde_precond(h, b, v)
        assert rel(v, z) < 2e-2
        for spectral in (1, 0):
            T.tfde_set_spectral_inner(h, spectral)
            x = torch.zeros_like(b)
            info = solve(h, x)
            # both meet 1e-12 on a well-conditioned system
            assert info.relres <= 1e-12 and not info.fallback and rel(x, ref) < 1e-10
    finally:
        T.tfde_destroy(h)


def test_batch_of_256_line_tiles(T):
    """Four 128^3 problems: 256 wide tiles per axis, for which the rule takes 256 lines."""
    import torch
    prm, us = [], []
    for i in range(4):
        km = (1.0, 1.2, 0.8) if i % 2 else (0.5, 0.6, 0.7)
        prm.append(T.make_params((128,) * 3, (0.3, 0.5, 0.7), (1.0, 1.2, 0.8), km, 0.05))
        us.append(to_dev(inp.smoothed_uniform((128,) * 3, i)))
    ref = [u.clone() for u in us]
    B = T.tfde_batch_create(prm, 20)
    try:
        for spectral in (1, 0):   # eigenbasis, then the grouped operator and preconditioner
            T.tfde_batch_set_spectral_inner(B, spectral)
            for u, w in zip(us, ref):
                u.copy_(w)
            for m in range(2):
                infos = T.tfde_batch_cn_advance(B, us, None, m == 0, 1e-11)
                assert all(i.relres <= 1e-11 and not i.fallback for i in infos)
            for i, p in enumerate(prm):
                h = T.tfde_assemble(p, T.TFDE_FP64)
                try:
                    w = ref[i].clone()
                    for m in range(2):
                        T.tfde_cn_advance(h, w, None, m == 0, 1e-12)
                finally:
                    T.tfde_destroy(h)
                assert rel(us[i], w) < 1e-9
    finally:
        T.tfde_batch_destroy(B)
