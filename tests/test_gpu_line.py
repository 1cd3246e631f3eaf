"""The dense line passes (FP64 and FP32) at the edges of their tiles and of
their range: operator, right-hand-side operator and preconditioner against the
oracle, symmetric (folded Toeplitz lines) and not, odd and even lengths, matrix
rows in one and in several blocks, and lengths on both sides of the limits
beyond which the FFT passes take over."""
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


GRIDS = [(1, 2, 3), (8, 9, 17), (15, 16, 33), (63, 64, 65), (88, 89, 7), (127, 129, 4), (3, 130, 168), (169, 5, 6),
         (2, 3, 231), (232, 4, 3), (233, 3, 2), (3, 288, 5), (289, 2, 4), (640, 3, 2), (2, 641, 3), (45, 130, 0),
         (511, 300, 0), (130, 641, 0)]


@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n", GRIDS)
def test_line_passes_match_oracle(T, n, sym):
    d, kp = (0.4, 0.55, 0.7), (1.0, 1.3, 0.8)
    km = kp if sym else (0.5, 0.7, 1.4)
    op = o.Problem(n=(n[0], n[1], max(1, n[2])), delta=d, kp=kp, km=km, dt=0.02, dim=3 if n[2] else 2)
    v = inp.uniform_vector(op.shape, 41).astype(np.float32).astype(np.float64)
    refs = {T.TFDE_OP_A: o.apply_A(op, v), T.TFDE_OP_RHS: o.rhs(op, v, None)}
    pref = o.apply_Pinv(o.build_tau(op), v)
    # FP64 as the FFT passes' own tests; FP32: unit roundoff 6e-8, three (six)
    # products whose sums err by a few roundoffs each, the operator's terms
    # cancelling in the right-hand side
    for prec, fast, tol in ((T.TFDE_FP64, 0, 1e-13), (T.TFDE_MIXED, T.TFDE_OP_FAST, 2e-6)):
        h = T.tfde_assemble(T.make_params(n, d, kp, km, 0.02), prec)
        try:
            y = to_dev(np.zeros_like(v))
            for which, ref in refs.items():
                T.tfde_matvec(h, which | fast, to_dev(v), y)
                assert relerr(to_host(y), ref) < tol, (prec, which)
            T.tfde_precond(h, to_dev(v), y)
            assert relerr(to_host(y), pref) < tol, prec
        finally:
            T.tfde_destroy(h)
