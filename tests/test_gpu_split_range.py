"""The hi + lo split of FP64 values around the exponents where it changes from
integer to FP64 arithmetic (below 2^-74, above 2^100): a whole psi of entries of
one size, on either side of each line and straddling it, so that every entry
counts.  Element by element against the FP64 oracle, with the relative bounds of
test_gpu_split_edges.py (products 3 * 2^-17 and 3 * 2^-21, FP32 sums) and nothing
absolute: the smallest rests, 2^-12 2^-90 of their input, and the largest sums,
some 2^20 times theirs, are normal FP32 numbers."""
import numpy as np
import pytest

from oracle.idmrg import Block, heff_apply, sector_mask
from workloads import build_mpo, random_chain_bonds

from gpu_helpers import context, gpu_heff, superblock_from_gpu

pytestmark = pytest.mark.gpu

BOUND = {"tf32x3": 2.0**-14, "bf16x3": 2.0**-13}


@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("m,steps", [(2, 3), (7, 4), (33, 6)])
def test_split_over_the_exponent_range(m, steps, prec):
    mpo = build_mpo(random_chain_bonds(8, 0.5, 1.5, 3), 8)
    ctx = context(mpo, m, prec=prec)
    for _ in range(steps):
        ctx.unit_cell_step()
    rng = np.random.default_rng(m)
    for p in range(ctx.P):
        L, W1, W2, R = superblock_from_gpu(ctx, mpo, p)
        mask = sector_mask(L.q, mpo.phys_charge, R.q)
        u = np.where(mask, rng.uniform(0.5, 2.0, mask.shape) * rng.choice([-1.0, 1.0], mask.shape), 0.0)
        yr = heff_apply(L, W1, W2, R, u)
        ya = heff_apply(Block(abs(L.op), L.q), abs(W1), abs(W2), Block(abs(R.op), R.q), abs(u))
        for e in (0, -72, -74, -75, -80, -90, 98, 100, 101):
            got = gpu_heff(ctx, p, u * 2.0**e) * 2.0**-e
            assert np.all(np.abs(got - yr) <= BOUND[prec] * ya), (p, e)
    ctx.close()
