"""Which loop drives a solve on the FFT and line passes.  The passes of a
device-side loop are captured once and launched as a graph, so the library's
per-kind launch counter sees only a solve's own set-up; a host-driven loop's
passes are all counted.  The device-side loops run by default, are given up
while per-launch timing is on, and on TFDE_MIXED problems by
tfde_set_device_loop(.., 0), with the same results."""
import pytest
import torch

import tfde_inputs as inp
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2511_21198_gb300 import build
    build.build()
    from paper_2511_21198_gb300 import tfde
    tfde.load()
    yield tfde
    tfde.tfde_stats_reset(False)


def solver(T, n, sym, mixed):
    km = (1.0, 1.3, 0.8) if sym else (0.5, 0.7, 1.4)
    h = T.tfde_assemble(T.make_params(n, (0.4, 0.55, 0.7), (1.0, 1.3, 0.8), km, 0.02),
                        T.TFDE_MIXED if mixed else T.TFDE_FP64)
    b = to_dev(inp.uniform_vector((max(1, n[2]), n[1], n[0]), 3))

    def solve(timed):
        """(launches of this kind, iterations, solution)"""
        T.tfde_stats_reset(timed)
        x = torch.zeros_like(b)
        info = T.tfde_pcg(h, b, x, 1e-11, 500) if sym else T.tfde_pgmres(h, b, x, 20, 1e-11, 500)
        assert info.relres <= 1e-11
        return T.tfde_stats_get().kind[3].launches, info.iters, x

    return h, solve


@pytest.mark.parametrize("mixed,sym", [(False, True), (True, True), (True, False)])
@pytest.mark.parametrize("n", [(15, 16, 17), (37, 45, 0)])
def test_loop_by_default_and_by_switch(T, n, sym, mixed):
    h, solve = solver(T, n, sym, mixed)
    passes = 2 if n[2] == 0 else 3   # the operator's; a sweep's last iteration ends before the preconditioner
    try:
        solve(False)   # builds the graph
        dev, it, x = solve(False)
        host, _, xh = solve(True)
        assert it >= 4 and host >= dev + passes * it
        T.tfde_set_device_loop(h, False)
        off, _, xo = solve(False)
        if mixed:
            assert off == host and torch.equal(xo, xh)
        else:   # no effect on FP64 problems
            assert off == dev and torch.equal(xo, x)
        T.tfde_set_device_loop(h, True)
        again, _, xa = solve(False)
        assert again == dev and torch.equal(xa, x)
        assert float(torch.linalg.norm(x - xh) / torch.linalg.norm(xh)) < 1e-9
    finally:
        T.tfde_stats_reset(False)
        T.tfde_destroy(h)


def test_tensor_core_cycle_runs_on_the_device(T):
    """The GMRES cycle that test_gpu_sweeps compares with the host-driven one."""
    n = (24, 40, 16)
    h, solve = solver(T, n, False, True)
    try:
        before = T.tfde_device_loop_launches(h)
        solve(False)
        ran = T.tfde_device_loop_launches(h)
        solve(True)
        assert before == 0 and ran > 0 and T.tfde_device_loop_launches(h) == ran
    finally:
        T.tfde_stats_reset(False)
        T.tfde_destroy(h)
