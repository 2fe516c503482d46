"""Packing of split (hi + lo) operands at the edges of its windows: sectors of 1
to about 60 states, so that the 32-row, 64-column windows, the 16-byte groups and
the K blocks end inside, at and just past a segment, and psi entries from 1 down
to 1e-30 with zeros between them (below 2^-74 the split is formed another way).
Element by element against the FP64 oracle.  A product's relative error is at
most 3 * 2^-17 for BF16 pairs (each operand's rest 2^-18, lo * lo 2^-18, doubled)
and 3 * 2^-21 for TF32 pairs, and FP32 accumulation adds at most 2^-23 per term
of the few hundred in a sum; two such stages stay below 2^-13 and 2^-14 of the
same sums over absolute values."""
import numpy as np
import pytest

from oracle.idmrg import Block, heff_apply, sector_mask
from workloads import build_mpo, random_chain_bonds, yc4_j1j2_bonds

from gpu_helpers import context, gpu_heff, superblock_from_gpu

pytestmark = pytest.mark.gpu

BOUND = {"tf32x3": 2.0**-14, "bf16x3": 2.0**-13}


@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("bonds,m,steps", [
    (random_chain_bonds(8, 0.5, 1.5, 3), m, n) for m, n in ((2, 3), (7, 4), (33, 6), (128, 8), (190, 9))
] + [(yc4_j1j2_bonds(1.0, 0.5), 24, 5)])
def test_split_heff_at_window_edges(bonds, m, steps, prec):
    mpo = build_mpo(bonds, 8)
    ctx = context(mpo, m, prec=prec)
    for _ in range(steps):
        ctx.unit_cell_step()
    rng = np.random.default_rng(m)
    for p in range(ctx.P):
        L, W1, W2, R = superblock_from_gpu(ctx, mpo, p)
        mask = sector_mask(L.q, mpo.phys_charge, R.q)
        x = np.where(mask, rng.standard_normal(mask.shape) * 10.0 ** rng.uniform(-30, 0, mask.shape), 0.0)
        x[rng.random(mask.shape) < 0.1] = 0.0
        yr = heff_apply(L, W1, W2, R, x)
        ya = heff_apply(Block(abs(L.op), L.q), abs(W1), abs(W2), Block(abs(R.op), R.q), abs(x))
        assert np.all(np.abs(gpu_heff(ctx, p, x) - yr) <= BOUND[prec] * ya + 1e-34), p
    ctx.close()
