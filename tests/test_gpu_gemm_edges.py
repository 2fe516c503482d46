"""FP64 and digit-slice grouped GEMMs at the edges of their tiles: sectors of 1
to 40 states, so that output blocks end inside, at and just past the 8 x 8
quadrants, 16 x 16 CTA tiles and 32 x 32 list tiles of the FP64 kernel and the
16- and 32-column groups of the digit-slice kernel's read-out, and K runs from
1 past several 16-deep steps.  H_eff psi against the FP64 oracle, within 1e-13
of max|H psi|: sums of at most a few hundred products of O(1) operands, each
rounded at 2^-53 (the digit form: cut at 2^-56 of its row's largest element)."""
import numpy as np
import pytest

from oracle.idmrg import heff_apply, sector_mask
from workloads import build_mpo, random_chain_bonds, yc4_j1j2_bonds

from gpu_helpers import context, gpu_heff, superblock_from_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp64tc"])
@pytest.mark.parametrize("bonds,m,steps", [
    (random_chain_bonds(8, 0.5, 1.5, 3), m, n) for m, n in ((2, 3), (7, 4), (16, 5), (33, 6), (61, 7), (128, 8))
] + [(yc4_j1j2_bonds(1.0, 0.5), 24, 5)])
def test_heff_at_tile_edges(bonds, m, steps, prec):
    mpo = build_mpo(bonds, 8)
    ctx = context(mpo, m, prec=prec)
    for _ in range(steps):
        ctx.unit_cell_step()
    rng = np.random.default_rng(m)
    for p in range(ctx.P):
        L, W1, W2, R = superblock_from_gpu(ctx, mpo, p)
        mask = sector_mask(L.q, mpo.phys_charge, R.q)
        x = np.where(mask, rng.standard_normal(mask.shape), 0.0)
        yr = heff_apply(L, W1, W2, R, x)
        assert np.max(np.abs(gpu_heff(ctx, p, x) - yr)) < 1e-13 * np.max(np.abs(yr)), p
