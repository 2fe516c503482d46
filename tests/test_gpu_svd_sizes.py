"""Sector SVDs beyond the block kernels at the sizes where the FP32 tournament
changes its register blocking (columns of up to 384, 640, 896, 1280 rows, and
longer): singular values of the GPU's own ground state against numpy's SVD of
the same sector matrices, within 1e-10 (the bound of the other SVD tests: both
are backward stable in 64 bits, the sums of squares are 1), and the kept
weight."""
import numpy as np
import pytest

from workloads import build_mpo, random_chain_bonds, yc4_j1j2_bonds

from gpu_helpers import context, gpu_psi_dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bonds,ell,m,steps,rows", [
    (yc4_j1j2_bonds(1.0, 0.5), 8, 700, 10, (321, 384)),
    (yc4_j1j2_bonds(1.0, 0.5), 8, 1000, 11, (385, 640)),
    (yc4_j1j2_bonds(1.0, 0.5), 8, 1500, 11, (641, 896)),
    (yc4_j1j2_bonds(1.0, 0.5), 8, 2048, 12, (897, 1280)),
    (yc4_j1j2_bonds(1.0, 0.5), 8, 2800, 13, (1281, 2048)),
])
def test_large_sector_singular_values(bonds, ell, m, steps, rows):
    mpo = build_mpo(bonds, ell)
    ctx = context(mpo, m, prec="bf16x3", lanczos_tol=1e-9)
    for _ in range(steps - 1):
        ctx.unit_cell_step()
    ctx.predict_wavefunction(-1)
    ctx.lanczos_solve(-1)
    eps, _, kept = ctx.truncate(-1)
    assert rows[0] <= ctx.svd_stats()["max_cols"] <= rows[1]
    qL, _ = ctx.block_basis(0, 0)
    qR, _ = ctx.block_basis(0, 1)
    qp = np.asarray(mpo.phys_charge)
    M = gpu_psi_dense(ctx, 0, (len(qL), 2, 2, len(qR))).reshape(2 * len(qL), 2 * len(qR))
    ql = (qL[:, None] + qp[None, :]).ravel()
    qr = (qp[:, None] + qR[None, :]).ravel()
    s = []
    for Q in np.unique(ql):
        a, b = np.nonzero(ql == Q)[0], np.nonzero(qr == -Q)[0]
        if len(a) and len(b):
            s.append(np.linalg.svd(M[np.ix_(a, b)], compute_uv=False))
    s = np.sort(np.concatenate(s))[::-1]
    lam = ctx.get_lambda(0)
    assert len(lam) == len(s)
    assert np.max(np.abs(lam - s)) < 1e-10
    assert abs((1.0 - eps[0]) - np.sum(s[:kept[0]] ** 2)) < 1e-10


@pytest.mark.parametrize("bonds,m,steps,prec", [
    (yc4_j1j2_bonds(1.0, 0.5), 130, 8, "fp64"),      # sectors around 64 columns: some refined, some not
    (yc4_j1j2_bonds(1.0, 0.5), 300, 9, "tf32x3"),    # block kernels
    (yc4_j1j2_bonds(1.0, 0.5), 300, 9, "fp64"),
    (random_chain_bonds(8, 0.5, 1.5, 5), 300, 9, "fp64tc"),  # ranks below the sector sizes
    (yc4_j1j2_bonds(1.0, 0.5), 1000, 11, "bf16x3"),  # large-sector kernels
])
def test_kept_bases_orthonormal(bonds, m, steps, prec):
    """The identity channels of the new blocks are U^T U and V V^T: the kept
    singular vectors are orthonormal to rounding, whichever of the refinement
    and the final Jacobi's sweeps finished a sector.  (1e-12: a product of up to
    2 m terms of rounding 2^-53 per step, over a dozen steps.)"""
    mpo = build_mpo(bonds, 8)
    ctx = context(mpo, m, prec=prec)
    for _ in range(steps):
        ctx.unit_cell_step()
    for p in range(ctx.P):
        for side, channel in ((0, -1), (1, 0)):
            op = ctx.block_to_host(p, side)[channel]
            assert np.max(np.abs(op - np.eye(len(op)))) < 1e-12, (p, side)
