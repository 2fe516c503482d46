"""Sector SVDs of wavefunctions with dense and nearly degenerate spectra (lattice
symmetries give such multiplets; ground states of short clusters do not): the
start vector of a solve that stops at once has sector matrices of planted
singular values.  All states are kept, so U, the singular values and V must give
the wavefunction back, and both bases must be orthonormal.

Bounds.  64-bit arithmetic: about ten products of n <= 462 terms, each rounding
to sqrt(n) 2^-52 at most, 20 sqrt(462) 2^-52 < 1e-13.  FP32-pair sweeps of the
large sectors (mixed precisions): up to 3 sweeps of n rotations with 2^-48 each,
sqrt(3 n) 2^-48 = 1.4e-13, and as much again in every other factor: 1e-12."""
import numpy as np
import pytest

from oracle.checkpoint import read_checkpoint
from workloads import build_mpo, chain_bonds

from gpu_helpers import context
import paper_1606_06790_gb300 as pkg

pytestmark = pytest.mark.gpu

SPECTRA = {
    "graded": lambda rng, n: 10.0 ** -np.sort(rng.uniform(0, 9, n)),
    "two_percent": lambda rng, n: rng.uniform(0.98, 1.0, n),
    "quartets": lambda rng, n: np.repeat(10.0 ** -rng.uniform(0, 6, -(-n // 4)), 4)[:n] * (1 + 1e-4 * rng.random(n)),
    "groups": lambda rng, n: np.repeat(10.0 ** -rng.uniform(0, 6, -(-n // 30)), 30)[:n] * (1 + 1e-3 * rng.random(n)),
    "equal": lambda rng, n: np.ones(n),
}


def _planted(ctx, mpo, p, spectrum, rng):
    """(D_L, d, d, D_R) wavefunction of unit norm with the given singular values."""
    qL, _ = ctx.block_basis(p, 0)
    qR, _ = ctx.block_basis(p, 1)
    qp = np.asarray(mpo.phys_charge)
    ql, qr = (qL[:, None] + qp[None, :]).ravel(), (qp[:, None] + qR[None, :]).ravel()
    M = np.zeros((len(ql), len(qr)))
    for Q in np.unique(ql):
        a, b = np.nonzero(ql == Q)[0], np.nonzero(qr == -Q)[0]
        k = min(len(a), len(b))
        if k:
            u = np.linalg.qr(rng.standard_normal((len(a), k)))[0]
            v = np.linalg.qr(rng.standard_normal((len(b), k)))[0]
            M[np.ix_(a, b)] = (u * SPECTRA[spectrum](rng, k)) @ v.T
    return (M / np.linalg.norm(M)).reshape(len(qL), 2, 2, len(qR))


@pytest.mark.parametrize("spectrum", list(SPECTRA))
@pytest.mark.parametrize("prec,sites,bound", [("fp64", 8, 1e-13), ("fp64", 10, 1e-13), ("fp64tc", 11, 1e-13), ("bf16x3", 11, 1e-12)])
def test_dense_spectra(prec, sites, bound, spectrum, tmp_path):
    import torch
    rng = np.random.default_rng(sites)
    mpo = build_mpo(chain_bonds(4), 4)
    ctx = context(mpo, 2**sites, prec=prec, lanczos_tol=1e30)  # every residual is small enough
    while ctx.iteration < sites:  # blocks of n sites become blocks of n + 1
        n = ctx.iteration
        psi = [_planted(ctx, mpo, p, spectrum if n == sites - 1 else "two_percent", rng) for p in range(ctx.P)]
        x = np.concatenate([pkg.layout_pack(*ctx.psi_layout(p), psi[p]) for p in range(ctx.P)])
        ctx.set_start_vector(-1, torch.tensor(x, device="cuda", dtype=torch.float64))
        ctx.lanczos_solve(-1)
        ctx.truncate(-1)
        ctx.update_environments(-1)
        ctx.advance()
    path = str(tmp_path / "state")
    ctx.save(path)
    for p, t in enumerate(read_checkpoint(path)["prev"]):
        u, v = t.U.reshape(-1, t.U.shape[2]), t.V.reshape(-1, t.V.shape[2])
        assert u.shape[1] == 2**sites
        eye = np.eye(u.shape[1])
        back = np.linalg.norm((u * t.lam) @ v.T - psi[p].reshape(len(u), len(v)))
        errs = [np.max(np.abs(u.T @ u - eye)), np.max(np.abs(v.T @ v - eye)), back]
        print(prec, sites, spectrum, p, "%.1e %.1e %.1e" % tuple(errs), ctx.svd_stats())
        assert max(errs) < bound, errs
    ctx.close()
