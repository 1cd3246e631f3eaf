"""The line passes at the lengths they are taken for: every tile width (FP64 8
lines, FP32 32 and 64) with many matrix chunks, one and two row blocks, the
second operand and all three strides; and device pointers aligned to their
element only, which give the aligned ones' results."""
import numpy as np
import pytest
import torch

import test_gpu_line as line
import tfde_inputs as inp
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu
T = line.T


# 127^3: FP64 8 lines, the DST pair in one pass of 127 rows, FP32 32 lines; 128
# rows exactly; 150 x 140 x 135: FP32 64 lines, two row blocks on every axis
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n", [(127, 127, 127), (128, 127, 126), (150, 140, 135)])
def test_wide_tiles_match_oracle(T, n, sym):
    line.test_line_passes_match_oracle(T, n, sym)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n", [(15, 17, 33), (61, 90, 0), (127, 20, 21)])
def test_element_aligned_pointers(T, n, sym, mixed):
    kp = (1.0, 1.3, 0.8)
    km = kp if sym else (0.5, 0.7, 1.4)
    h = T.tfde_assemble(T.make_params(n, (0.4, 0.55, 0.7), kp, km, 0.02), T.TFDE_MIXED if mixed else T.TFDE_FP64)
    v = to_dev(inp.uniform_vector((max(1, n[2]), n[1], n[0]), 9))

    def off():   # 8 bytes past a 256-byte boundary
        return torch.zeros(v.numel() + 1, dtype=v.dtype, device=v.device)[1:].view(v.shape)

    def results(new):
        b, out = new(), []
        b.copy_(v)
        for op in (T.TFDE_OP_A, T.TFDE_OP_RHS) + ((T.TFDE_OP_A | T.TFDE_OP_FAST,) if mixed else ()):
            out.append(new())
            T.tfde_matvec(h, op, b, out[-1])
        out.append(new())
        T.tfde_precond(h, b, out[-1])
        out.append(new())
        if sym:
            T.tfde_pcg(h, b, out[-1], 1e-10, 200)
        else:
            T.tfde_pgmres(h, b, out[-1], 20, 1e-10, 200)
        u = new()
        u.copy_(v)
        for m in range(2):
            T.tfde_cn_advance(h, u, b, m == 0, 1e-10)
        return out + [u]

    try:
        for a, b in zip(results(lambda: torch.zeros_like(v)), results(off)):
            assert a.data_ptr() % 16 == 0 and b.data_ptr() % 16 == 8
            assert torch.equal(a, b)
    finally:
        T.tfde_destroy(h)
