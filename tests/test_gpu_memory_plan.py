"""What a run holds against its plan: the device memory that a context takes for a run stays within
mctrg_footprint beside the shared prefix, and so within the caller's budget."""
import numpy as np
import pytest

from paper_1710_03757_gb300 import build, mctrg

pytestmark = pytest.mark.gpu

# allocations are rounded up to 2 MiB each; a context has fewer than 48
ROUNDING = 48 * (2 << 20)


@pytest.fixture(scope="module")
def torch():
    build.build()
    mctrg.lib()
    return pytest.importorskip("torch")


def _context(opts, L, chi, imp):
    ctx = mctrg.mctrg_create(opts)
    if imp:
        assert mctrg.mctrg_init_impurity(ctx, 0.44, 0.0, L, chi, imp) == 0
    else:
        assert mctrg.mctrg_init_lattice(ctx, 0.44, 0.0, L, chi) == 0
    return ctx


@pytest.mark.parametrize("L,chi,n,precision,imp,budget", [
    (16, 8, 2560, mctrg.MCTRG_FP64, 0, 32 << 30),      # a low-rank level of K = 16 below full levels of n = 64
    (16, 24, 100, mctrg.MCTRG_FP64, 0, 24 << 30),      # K = 256 below n = 576
    (16, 17, 200, mctrg.MCTRG_FP64TC, 0, 24 << 30),    # a low-rank level larger than the full ones
    (16, 16, 400, mctrg.MCTRG_TF32X3, 0, 16 << 30),    # rounded operands beside the matrices
    (16, 8, 600, mctrg.MCTRG_FP64, 2, 8 << 30),        # every level per item
])
def test_a_run_holds_what_it_planned(torch, L, chi, n, precision, imp, budget):
    opts = mctrg.make_options(precision=precision, hbm_budget_bytes=budget)
    for warm in (True, False):                         # the first pass loads the kernels
        ctx = _context(opts, L, chi, imp)
        plan = mctrg.mctrg_footprint(ctx, n)
        assert plan <= budget
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ln, sg, fl = np.zeros(n), np.zeros(n, np.int8), np.zeros(n, np.uint8)
        status, _ = mctrg.mctrg_run(ctx, n, 3, 0, ln, sg, fl)
        held = before - torch.cuda.mem_get_info()[0]
        mctrg.mctrg_destroy(ctx)
        assert status in (mctrg.MCTRG_OK, mctrg.MCTRG_EDOMAIN)
    print("planned %.3f GB, held %.3f GB" % (plan / 1e9, held / 1e9))
    assert held <= plan + ROUNDING
