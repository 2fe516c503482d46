"""The digit-slice GEMM gives the same bits every time: the digit sums of levels
0 .. 4 are exact integers, and the order in which the others are summed is fixed,
so 25 repeats of H_eff psi agree bit for bit if every MMA that touches a common
accumulator runs in the order of issue.  K of one block up to K chunks of 768
and several of them, tiles on every SM; and the value itself against the FP64
GEMM form, as in the other digit tests (1e-13 of the largest element)."""
import numpy as np
import pytest

from workloads import build_mpo, yc4_j1j2_bonds

from gpu_helpers import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,steps", [(12, 4), (700, 10)])
def test_digit_form_repeats_bit_for_bit(m, steps):
    import torch
    ctx = context(build_mpo(yc4_j1j2_bonds(1.0, 0.5), 8), m, prec="tf32x3")
    for _ in range(steps):
        ctx.unit_cell_step()
    rng = np.random.default_rng(m)
    N = sum(ctx.psi_layout(p)[1] for p in range(ctx.P))
    x = torch.tensor(rng.standard_normal(N) * 10.0 ** rng.uniform(-8, 0, N), device="cuda", dtype=torch.float64)
    y0, first, y = (torch.zeros_like(x) for _ in range(3))
    ctx.heff_apply_fp64(-1, x, y0, 0)
    ctx.heff_apply_fp64(-1, x, first, 1)
    torch.cuda.synchronize()
    assert (first - y0).abs().max().item() < 1e-13 * y0.abs().max().item()
    for _ in range(25):
        y.zero_()
        ctx.heff_apply_fp64(-1, x, y, 1)
        torch.cuda.synchronize()
        assert torch.equal(y, first)
    ctx.close()
