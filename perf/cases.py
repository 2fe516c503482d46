"""The workloads that performance work on this library is measured on.

A case is one call (or one short sequence of calls) of the public API on a
problem of a stated size:

* ``step``: one parallel iteration (``Context.unit_cell_step``) of a run that
  continues from a saved state: prediction, Lanczos, sector SVDs, cut, new
  environments.  The state moves on with every pass, as in a run.
* ``heff``: H_eff psi of one superblock or of all of them, in the context's own
  arithmetic or in one of the FP64-accurate forms, as an eigensolver of the
  caller's would ask for it.
* ``batch``: one step of a context over several disorder realisations.
* ``observe``: one step and the bond strengths and spin correlations of the
  unit it leaves behind (what a production run records per iteration).

The state a run continues from is a checkpoint written here from the couplings
alone, so that it is the same whatever the library computes: the state of the
paper's first iterations, in which blocks of n sites still hold all (or, cut
here to m, nearly all) of their 2^n states.  The ground states of the clusters
of iterations n - 1 and n - 2 come from a short Lanczos run on the clusters'
spins; their singular vectors are the bases of the blocks and their singular
values what the prediction reads; the blocks' operators come from the recursion
of Eqs. L, R.  Couplings come from the case's seed: those of the configured
model times 1 +- 5 %, for the batch i.i.d. in [0.8, 1.2] (wider draws leave
clusters with nearly free end spins, whose ground state no solver tolerance
pins down).
"""
import math
import os
import struct
import tempfile

import numpy as np
import torch

import paper_1606_06790_gb300 as pkg
from workloads import build_mpo, chain_bonds, j1j2_chain_bonds, kagome_yc8_bonds, open_chain_bonds, random_chain_bonds, yc4_j1j2_bonds

ELL = {"chain": 4, "j1j2": 4, "randchain": 16, "yc4": 8, "kagome": 12}
MPO_DIM = {"chain": 5, "j1j2": 8, "randchain": 5, "yc4": 17, "kagome": 20}  # about; for work()


def listed():
    return [
        # the smallest call: H_eff psi of one superblock of the uniform chain at m = 32, inside a caller's own solver
        dict(name="heff_chain_m32", kind="heff", lattice="chain", m=32, prec="fp64", p=1, form=-1),
        # the small end of the m scan on the uniform chain, plain FP64: launches and host work between them
        dict(name="step_chain_m32", kind="step", lattice="chain", m=32, prec="fp64"),
        # the random-bond chain at its configured size (l = 16, m = 256), tensor-core precision
        dict(name="step_randchain_m256", kind="step", lattice="randchain", m=256, prec="tf32x3"),
        # the same chain in plain FP64 at an odd m of a scan
        dict(name="step_randchain_m181_fp64", kind="step", lattice="randchain", m=181, prec="fp64"),
        # J1-J2 cylinder (l = 8), FP64-accurate tensor-core mode, a middle m of a scan
        dict(name="step_yc4_m500_fp64tc", kind="step", lattice="yc4", m=500, prec="fp64tc"),
        # J1-J2 cylinder at its configured size
        dict(name="step_yc4_m1024", kind="step", lattice="yc4", m=1024, prec="bf16x3"),
        # kagome cylinder (l = 12, six superblocks) at the small end of the paper's production range (m = 1000 .. 2800)
        dict(name="step_kagome_m1000", kind="step", lattice="kagome", m=1000, prec="bf16x3"),
        # matvecs of the kagome cylinder at its configured size, all superblocks: the reduced-precision inner matvec ...
        dict(name="heff_kagome_m2048", kind="heff", lattice="kagome", m=2048, prec="bf16x3", p=-1, form=-1),
        # ... and the FP64-accurate one on the tensor cores that starts every restart
        dict(name="heff_kagome_m1500_digits", kind="heff", lattice="kagome", m=1500, prec="bf16x3", p=-1, form=1),
        # a disorder average: twelve realisations of uneven unit cells and m in one context
        dict(name="batch_12", kind="batch", count=12, m=64, prec="tf32x3"),
        # what a production run records per iteration: a step, then bond strengths and correlations of the unit
        dict(name="observe_j1j2_m64", kind="observe", lattice="j1j2", m=64, prec="fp64"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "heff", "heff", "batch", "observe"])
    if kind == "step":
        lattice, lo, hi = rng.choice([("chain", 16, 128), ("randchain", 32, 400), ("yc4", 64, 1000), ("kagome", 64, 1000)])
        m = _logint(rng, lo, hi)
        precs = ["tf32x3", "bf16x3"] + (["fp64tc"] if m <= 500 else []) + (["fp64", "fp64"] if m <= 200 else [])
        return dict(kind=kind, lattice=lattice, m=m, prec=rng.choice(precs))
    if kind == "heff":
        lattice, lo, hi = rng.choice([("chain", 16, 256), ("randchain", 32, 512), ("yc4", 64, 1024), ("kagome", 64, 2048)])
        m = _logint(rng, lo, hi)
        prec, form = rng.choice([("bf16x3", -1), ("tf32x3", -1), ("tf32x3", 1), ("fp64tc", -1)] + ([("fp64", -1), ("bf16x3", 0)] if m <= 700 else []))
        return dict(kind=kind, lattice=lattice, m=m, prec=prec, p=rng.choice([-1, -1, 0]), form=form)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 12), m=_logint(rng, 16, 64), prec=rng.choice(["fp64", "tf32x3", "bf16x3"]))
    return dict(kind=kind, lattice=rng.choice(["chain", "j1j2"]), m=_logint(rng, 16, 96), prec=rng.choice(["fp64", "tf32x3"]))


# ---------------------------------------------------------------- inputs
def _mpo(lattice, seed):
    g = np.random.default_rng([seed, 1606])
    ell = ELL[lattice]
    bonds = {"chain": lambda: chain_bonds(ell), "randchain": lambda: random_chain_bonds(ell, 0.5, 1.5, 1606),
             # dimerised, so that the ground state is unique and its unit has one fixed point
             "j1j2": lambda: [b._replace(jxy=b.jxy * x, jz=b.jz * x) for b, x in zip(j1j2_chain_bonds(ell, 1.0, 0.3), [1.25, 0.75] * 2 + [1.0] * 4)],
             "yc4": lambda: yc4_j1j2_bonds(1.0, 0.5), "kagome": lambda: kagome_yc8_bonds(1.0)}[lattice]()
    f = g.uniform(0.95, 1.05, len(bonds))
    return build_mpo([b._replace(jxy=b.jxy * x, jz=b.jz * x) for b, x in zip(bonds, f)], ell)


class _Basis:
    """Product basis of a block of spins ordered by charge sectors: ``q`` and
    ``dim`` per sector, ``place[k]`` the position of product state k (first site
    most significant), ``groups`` the (old sector, site state, first row) runs
    that make up each sector.  Left blocks grow to the right and list sectors by
    ascending charge, (old sector, site state) inside; right blocks grow to the
    left, descending, (site state, old sector) inside."""

    def __init__(self, side, old=None):
        self.side = side
        oq, od = (old.q, old.dim) if old else ([0], [1])
        off = np.concatenate([[0], np.cumsum(od)])
        self.q, self.dim, self.groups, at = [], [], [], 0
        self.pos = [np.zeros(off[-1], np.int64) for _ in range(2)]  # old state, site state -> new state
        for Q in sorted({c + s for c in oq for s in (1, -1)}, reverse=side == "R"):
            order = [(i, s) for i in range(len(oq)) for s in range(2)] if side == "L" else [(i, s) for s in range(2) for i in range(len(oq))]
            rows, here = 0, []
            for i, s in order:
                if oq[i] + (1, -1)[s] == Q:
                    self.pos[s][off[i]:off[i + 1]] = at + rows + np.arange(od[i])
                    here.append((i, s, rows))
                    rows += od[i]
            self.q.append(Q)
            self.dim.append(rows)
            self.groups.append(here)
            at += rows
        p = old.place if old else np.zeros(1, np.int64)
        self.place = np.stack([self.pos[0][p], self.pos[1][p]], 1 if side == "L" else 0).reshape(-1)
        off = np.concatenate([[0], np.cumsum(self.dim)])
        self.sl = [slice(int(x), int(y)) for x, y in zip(off, off[1:])]


def _bases(side, n):
    out = []
    for _ in range(n):
        out.append(_Basis(side, out[-1] if out else None))
    return out


def _cluster_ground(bonds, N, seed):
    """Approximate ground state (2^N amplitudes) of sum J s_i.s_j over the bonds
    of an open cluster of N spins with total S^z = 0: 60 Lanczos steps."""
    dev = torch.device("cuda")
    up = torch.arange(2 ** N, device=dev)
    pop = torch.zeros(2 ** N, dtype=torch.int64, device=dev)
    for k in range(N):
        pop += (up >> k) & 1
    x = torch.where(pop == N // 2, _psi(2 ** N, seed), 0.0)
    const = -sum(b.jz for b in bonds) / 4.0

    def apply(v):  # s_i.s_j = (swap of i and j) / 2 - 1/4
        y = const * v
        for b in bonds:
            shape = (2 ** b.i, 2, 2 ** (b.j - b.i - 1), 2, 2 ** (N - 1 - b.j))
            y.view(shape).add_(v.view(shape).transpose(1, 3), alpha=b.jz / 2.0)
        return y

    V, al, be = [x / x.norm()], [], []
    for k in range(60):
        w = apply(V[k])
        a = torch.dot(w, V[k])
        w = w - a * V[k]
        if k:
            w = w - be[-1] * V[k - 1]
        al.append(a)
        be.append(w.norm())
        V.append(w / be[-1])
    al, be = torch.stack(al).cpu().numpy(), torch.stack(be).cpu().numpy()[:-1]
    y = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))[1][:, 0]
    x = torch.zeros_like(x)
    for c, v in zip(y, V):
        x += float(c) * v
    return x / x.norm()


def _operators(mpo, sites, side, bases, dev):
    """The block's operators, one dense matrix per MPO channel, and the charges
    of the channels (Eqs. L, R with nothing cut)."""
    order = sites if side == "L" else sites[::-1]
    op = torch.zeros(mpo.W[order[0]].shape[0 if side == "L" else 1], 1, 1, dtype=torch.float64, device=dev)
    op[-1 if side == "L" else 0] = 1.0
    for k, basis in zip(order, bases):
        w = mpo.W[k]
        at = [torch.from_numpy(x).to(dev) for x in basis.pos]
        new = torch.zeros(w.shape[1 if side == "L" else 0], sum(basis.dim), sum(basis.dim), dtype=torch.float64, device=dev)
        for a, b, s, t in zip(*np.nonzero(w)):
            src, dst = (a, b) if side == "L" else (b, a)
            new[dst][at[s][:, None], at[t][None, :]] += float(w[a, b, s, t]) * op[src]
        op = new
    bond = (sites[-1] + 1 if side == "L" else sites[0]) % mpo.ell
    return op, [int(c) * (1 if side == "L" else -1) for c in mpo.bond_charge[bond]]


class _Block:
    """A block in its kept basis: sectors, and per channel and in-sector the
    block to the out-sector (None where there is none)."""

    def __init__(self, mpo, sites, side, bases, rot, live, dev):
        full = bases[-1]
        op, self.chq = _operators(mpo, sites, side, bases, dev)
        where = {c: g for g, c in enumerate(full.q)}
        self.q, self.dim = [full.q[i] for i in live], [rot[i].shape[1] for i in live]
        self.ops = []
        for a, ch in enumerate(self.chq):
            row = []
            for i in live:
                o = where.get(full.q[i] + ch, -1)
                row.append(rot[o].T @ op[a][full.sl[o], full.sl[i]] @ rot[i] if o in live else None)
            self.ops.append(row)


def _sites(m):
    """Sites of the smallest block with at least m states."""
    return max(3, math.ceil(math.log2(m)))


def _sector_sizes(n, m):
    """States kept in the n + 1 charge sectors of n spins: m (or all 2^n) in the
    sectors' own proportions, the same for +q and -q; whatever rounding leaves
    over goes to the middle."""
    full = [math.comb(n, j) for j in range(n + 1)]
    k = [min(f, int(f * m / 2 ** n)) for f in full]
    for j in sorted(range(n + 1), key=lambda j: abs(2 * j - n)) * 8:
        other = n - j
        more = 1 if other == j else 2
        if sum(k) + more <= min(m, 2 ** n) and k[j] < full[j] and j <= other:
            k[j] += 1
            k[other] += other != j
    return k


class _State:
    """A run's state before iteration n: blocks of n sites for every pair (or
    those that superblocks `pairs` need) and the truncations at n - 1 and n - 2."""

    def __init__(self, case, seed, pairs=None):
        dev = self.dev = torch.device("cuda")
        self.mpo = _mpo(case["lattice"], seed)
        self.m, self.ell = case["m"], self.mpo.ell
        self.P, self.n = self.ell // 2, _sites(case["m"])
        n, ell = self.n, self.ell
        self.bL, self.bR = _bases("L", n), _bases("R", n)
        k = _sector_sizes(n, self.m)
        self.live = [i for i in range(n + 1) if k[i]]
        self.L, self.R, self.cut1, self.cut2 = {}, {}, {}, {}
        for p in range(self.P) if pairs is None else sorted({q % self.P for p in pairs for q in (p, p + 1)}):
            for back in (1, 2):
                # superblock p at n - back: the sites from 2p on, split in the middle
                N = n + 1 - back
                psi = _cluster_ground(open_chain_bonds(self.mpo.bonds, ell, 2 * p, 2 * p + 2 * N - 1), 2 * N, seed + p)
                M = torch.empty(2 ** N, 2 ** N, dtype=torch.float64, device=dev)
                left, right = self.bL[N - 1], self.bR[N - 1]
                M[torch.from_numpy(left.place).to(dev)[:, None], torch.from_numpy(right.place).to(dev)[None, :]] = psi.view(2 ** N, 2 ** N)
                M = M.cpu().numpy()
                svd = [np.linalg.svd(M[a, b]) for a, b in zip(left.sl, right.sl)]
                keep = k if back == 1 else left.dim
                U, lam, V = ([torch.from_numpy(np.ascontiguousarray(x)) for x in y] for y in zip(*((u[:, :c], s[:c], v[:c].T) for (u, s, v), c in zip(svd, keep))))
                (self.cut1 if back == 1 else self.cut2)[p] = ([u.to(dev) for u in U], lam, [v.to(dev) for v in V])
            U, _, V = self.cut1[p]
            self.L[p] = _Block(self.mpo, [(2 * p + j) % ell for j in range(n)], "L", self.bL, U, self.live, dev)
            self.R[p] = _Block(self.mpo, [(2 * p + n + j) % ell for j in range(n)], "R", self.bR, V, self.live, dev)

    # -- H_eff psi in 64 bits, sector by sector
    def layout(self, p):
        """Sub-blocks {(left sector, s, t): (right sector, column)}, row offsets and widths, length."""
        L, R = self.L[p], self.R[(p + 1) % self.P]
        where = {c: j for j, c in enumerate(R.q)}
        sub, roff, C, N = {}, [], [], 0
        for i, c in enumerate(L.q):
            col = 0
            for s in range(2):
                for t in range(2):
                    j = where.get(-c - (1, -1)[s] - (1, -1)[t])
                    if j is not None:
                        sub[i, s, t] = (j, col)
                        col += R.dim[j]
            roff.append(N)
            C.append(col)
            N += L.dim[i] * col
        return sub, roff, C, N

    def two_site(self, p):
        c1, c2 = (2 * p + self.n) % self.ell, (2 * p + self.n + 1) % self.ell
        W = np.einsum("abse,bctf->acstef", self.mpo.W[c1], self.mpo.W[c2])
        terms = {}
        for a, c, s, t, e, f in zip(*np.nonzero(W)):
            terms.setdefault((a, e, f), []).append((c, s, t, float(W[a, c, s, t, e, f])))
        return terms

    def apply(self, p, x):
        L, R = self.L[p], self.R[(p + 1) % self.P]
        sub, roff, C, N = self.layout(p)
        terms, out = self.two_site(p), torch.zeros_like(x)
        lq = {c: i for i, c in enumerate(L.q)}
        T3 = {}
        for i in range(len(L.q)):
            rows = x[roff[i]:roff[i] + L.dim[i] * C[i]].view(L.dim[i], C[i])
            for a, ch in enumerate(L.chq):
                so = lq.get(L.q[i] + ch)
                if so is None or L.ops[a][i] is None:
                    continue
                T1 = L.ops[a][i] @ rows
                for e in range(2):
                    for f in range(2):
                        if (i, e, f) not in sub:
                            continue
                        j, col = sub[i, e, f]
                        for c, s, t, v in terms.get((a, e, f), ()):
                            key, part = (so, s, t, c, j), v * T1[:, col:col + R.dim[j]]
                            T3[key] = T3[key] + part if key in T3 else part
        rq = {c: j for j, c in enumerate(R.q)}
        for (so, s, t, c, j), y in T3.items():
            jo = rq.get(R.q[j] + R.chq[c])
            if jo is None or (so, s, t) not in sub or sub[so, s, t][0] != jo or R.ops[c][j] is None:
                continue
            col = sub[so, s, t][1]
            out[roff[so]:roff[so] + L.dim[so] * C[so]].view(L.dim[so], C[so])[:, col:col + R.dim[jo]] += y @ R.ops[c][j].T
        return out

    # -- checkpoint
    def write(self, path):
        with open(path, "wb") as f:
            f.write(b"IDMRGCK1" + struct.pack("<iiiiii", self.ell, 2, self.P, self.m, 0, 0))
            f.write(_vec([w.shape[0] for w in self.mpo.W] + [self.mpo.W[0].shape[0]], "i4"))
            f.write(struct.pack("<iid", self.n, -1, 0.0))
            hist = list(range(-1, self.n))
            f.write(_vec(hist, "i4") + _vec([-0.45 * (2 * k + 2) for k in hist], "f8") + _vec([], "i4") + _vec([], "f8"))
            for p in range(self.P):
                for b in (self.L[p], self.R[p]):
                    f.write(_vec(b.q, "i4") + _vec(b.dim, "i4") + _vec(b.chq, "i4"))
                    _write_all(f, [x for row in b.ops for x in row if x is not None])
                self._truncation(f, p, 1)
                self._truncation(f, p, 2)

    def _truncation(self, f, p, back):
        """The truncation of superblock p at n - back, from blocks of n - back
        sites to blocks of one site more."""
        N = self.n - back
        U, lam, V = self.cut1[p] if back == 1 else self.cut2[p]
        live = self.live if back == 1 else list(range(N + 2))
        U, lam, V = [U[i] for i in live], torch.cat([lam[i] for i in live]).numpy(), [V[i] for i in live]
        old, new = (self.bL[N - 1], self.bR[N - 1]), (self.bL[N], self.bR[N])
        if back == 1:  # the blocks it starts from are in the basis of the truncation before
            inner = self.cut2[p][0], self.cut2[(p + 1) % self.P][2]
            U = [torch.cat([inner[0][i].T @ u[r:r + old[0].dim[i]] for i, _, r in new[0].groups[g]]) for g, u in zip(live, U)]
            V = [torch.cat([inner[1][j].T @ v[r:r + old[1].dim[j]] for j, _, r in new[1].groups[g]]) for g, v in zip(live, V)]
        k = [u.shape[1] for u in U]
        f.write(struct.pack("<i", 1))
        for b in old:
            f.write(_vec(b.q, "i4") + _vec(b.dim, "i4"))
        for b in new:
            f.write(_vec([b.q[i] for i in live], "i4") + _vec(k, "i4"))
        f.write(struct.pack("<q", len(live)))
        uo = vo = lo = 0
        for g, i in enumerate(live):
            r, c = new[0].dim[i], new[1].dim[i]
            f.write(struct.pack("<iiiiiqqi", new[0].q[i], k[g], r, c, g, uo, vo, lo))
            f.write(_vec([x for j, s, first in new[0].groups[i] for x in (j, s, first)], "i4", 3))
            f.write(_vec([x for j, s, first in new[1].groups[i] for x in (s, j, first)], "i4", 3))
            uo, vo, lo = uo + r * k[g], vo + c * k[g], lo + k[g]
        f.write(_vec(lam, "f8") + _vec(np.sort(lam)[::-1], "f8") + struct.pack("<ddqq", 0.0, 0.0, uo, vo))
        _write_all(f, U)
        _write_all(f, V)


def _vec(a, code, width=1):
    a = np.asarray(a, dtype="<" + code)
    return struct.pack("<q", a.size // width) + a.tobytes()


def _write_all(f, blocks):
    flat = torch.cat([b.reshape(-1) for b in blocks]) if blocks else torch.zeros(0, dtype=torch.float64)
    f.write(struct.pack("<q", flat.numel()))
    f.write(memoryview(flat.cpu().numpy()))


def _context(mpo, case, **kw):
    return pkg.Context(mpo.W, mpo.phys_charge, mpo.bond_charge, m=case["m"], prec=case["prec"], **kw)


def _restored(case, seed):
    state = _State(case, seed)
    ctx = _context(state.mpo, case)
    fd, path = tempfile.mkstemp(suffix=".ck", dir="/dev/shm" if os.path.isdir("/dev/shm") else None)
    os.close(fd)
    try:
        state.write(path)
        ctx.load(path)
    finally:
        os.unlink(path)
    return state, ctx


def _psi(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    return x / x.norm()


def _pairs(ell):
    """Nearest and next-nearest bonds of a unit, and correlations over four units."""
    return [(i, i + r) for i in range(ell) for r in (1, 2)] + [(0, r) for r in range(3, 4 * ell + 1)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        return dict(kind=kind, ctx=_restored(case, seed)[1])
    if kind == "heff":
        state, ctx = _restored(case, seed)
        ps = range(state.P) if case["p"] < 0 else [case["p"]]
        psi = _psi(sum(state.layout(p)[3] for p in ps), seed)
        return dict(kind=kind, ctx=ctx, p=case["p"], form=case["form"], psi=psi, out=torch.zeros_like(psi))
    if kind == "batch":
        # realisations as in the disorder workload: l = 8, 12, 16, 24 by turns, m in three sizes
        probs, ms = [], []
        for r in range(case["count"]):
            ell = (8, 12, 16, 24)[r % 4]
            mpo = build_mpo(random_chain_bonds(ell, 0.8, 1.2, 1000 * seed + r), ell)
            probs.append((mpo.W, mpo.phys_charge, mpo.bond_charge))
            ms.append(max(4, case["m"] * (4, 6, 8)[r // 4 % 3] // 8))
        ctx = pkg.Context.batch(probs, ms, prec=case["prec"])
        for _ in range(7):
            ctx.unit_cell_step()
        return dict(kind=kind, ctx=ctx)
    ctx = _context(_mpo(case["lattice"], seed), case)
    for _ in range(14):
        ctx.unit_cell_step()
    return dict(kind=kind, ctx=ctx, pairs=_pairs(ELL[case["lattice"]]))


def run(state):
    ctx = state["ctx"]
    if state["kind"] == "heff":
        if state["form"] < 0:
            ctx.heff_apply(state["p"], state["psi"], state["out"])
        else:
            ctx.heff_apply_fp64(state["p"], state["psi"], state["out"], state["form"])
        return state["out"]
    r = ctx.unit_cell_step()
    # what the step computes: energies, centre bonds, the weight that the cut
    # keeps and every singular value.  Matvec counts say how the solver got
    # there; the number of states kept depends on rounding where a spectrum
    # runs into the zero threshold (1e-12), and with it the spectrum's length at
    # the next step: zeros fill it up
    lam = np.zeros((ctx.P, 2 * ctx.opts.m))
    for p in range(ctx.P):
        x = ctx.get_lambda(p)
        lam[p, :len(x)] = x
    out = dict(energy=r["energy"], bond=r["bond"], weight=1.0 - r["eps"], lam=lam)
    if state["kind"] == "observe":
        out["corr"] = ctx.spin_dot(state["pairs"])
    return out


# ---------------------------------------------------------------- work
def _heff_work(w, m, P):
    """Flops and bytes of one H_eff psi over P superblocks: sectors of m states
    in the proportions of free spins."""
    k = _sites(m)
    D = {k - 2 * j: m * math.comb(k, j) / 2 ** k for j in range(k + 1)}
    N = sum(D[q] * D.get(-q - s - t, 0.0) for q in D for s in (1, -1) for t in (1, -1))
    # channels by charge 0, +2, -2 in about equal shares
    env = w * (sum(D[q] * D.get(q + c, 0.0) for q in D for c in (0, 2, -2)) / 3)
    gemm = 2.0 * w * sum(D[q] * D.get(q + c, 0.0) * D.get(-q - s - t, 0.0) for q in D for c in (0, 2, -2) for s in (1, -1) for t in (1, -1)) / 3
    return P * 2 * gemm, P * 8.0 * (2 * env + 2 * N), P * N


def _step_work(w, m, P):
    """The least a step can do: 40 matvecs (the count reported for a predicted
    start), the singular value decompositions of the sector matrices, new
    environments; every environment, wavefunction and basis once."""
    f, b, N = _heff_work(w, m, P)
    k = _sites(m) + 1
    svd = P * sum(26.0 * (2 * m * math.comb(k, j) / 2 ** k) ** 3 for j in range(k + 1))
    env = f / 2
    return 40 * f + svd + env, 2 * b + 8.0 * 2 * N


def work(case):
    if case["kind"] == "heff":
        P = ELL[case["lattice"]] // 2 if case["p"] < 0 else 1
        f, b, _ = _heff_work(MPO_DIM[case["lattice"]], case["m"], P)
        return {"bytes": b, "flops": f}
    if case["kind"] == "batch":
        f = b = 0.0
        for r in range(case["count"]):
            x = _step_work(5, max(4, case["m"] * (4, 6, 8)[r // 4 % 3] // 8), (4, 6, 8, 12)[r % 4])
            f, b = f + x[0], b + x[1]
        return {"bytes": b, "flops": f}
    f, b = _step_work(MPO_DIM[case["lattice"]], case["m"], ELL[case["lattice"]] // 2)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- 64-bit values
def _ground(apply, x):
    """Lowest eigenpair: Lanczos with full re-orthogonalisation, restarted from
    its Ritz vector until a restart changes nothing."""
    x = x / x.norm()
    for _ in range(4):
        V, al, be = [x], [], []
        for _ in range(120):
            w = apply(V[-1])
            al.append(float(w @ V[-1]))
            B = torch.stack(V)
            for _ in range(2):
                w = w - B.T @ (B @ w)
            b = float(w.norm())
            e, y = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
            if b * abs(y[-1, 0]) < 2e-15 * abs(e[0]) or b < 1e-13:
                break
            be.append(b)
            V.append(w / b)
        x = torch.tensor(y[:, 0], device=x.device) @ torch.stack(V[:len(al)])
        x = x / x.norm()
        if len(al) < 4:
            break
    return float(x @ apply(x)), x


def _exact_step(case, seed):
    S = _State(case, seed)
    energy, bond, weight, lam = [], [], [], np.zeros((S.P, 2 * S.m))
    for p in range(S.P):
        L, R = S.L[p], S.R[(p + 1) % S.P]
        sub, roff, C, N = S.layout(p)
        e, psi = _ground(lambda v: S.apply(p, v), _psi(N, seed + p))
        c1, c2 = (2 * p + S.n) % S.ell, (2 * p + S.n + 1) % S.ell
        W1, W2 = S.mpo.W[c1], S.mpo.W[c2]
        h = np.einsum("bse,btf->stef", W1[-1, 1:-1], W2[1:-1, 0])
        blk = {(i, s, t): psi[roff[i]:roff[i] + L.dim[i] * C[i]].view(L.dim[i], C[i])[:, col:col + R.dim[j]]
               for (i, s, t), (j, col) in sub.items()}
        b = 0.0
        for (i, s, t), x in blk.items():
            for e1 in range(2):
                for f1 in range(2):
                    y = blk.get((i, e1, f1))
                    if h[s, t, e1, f1] != 0.0 and y is not None and y.shape == x.shape:
                        b += float(h[s, t, e1, f1]) * float((x * y).sum())
        sv = []
        for Q in sorted({c + s for c in L.q for s in (1, -1)}):
            rows = [(i, s) for i in range(len(L.q)) for s in range(2) if L.q[i] + (1, -1)[s] == Q]
            cols = [(t, j) for t in range(2) for j in range(len(R.q)) if R.q[j] + (1, -1)[t] == -Q]
            if rows and cols:
                sv.append(torch.linalg.svdvals(torch.cat([torch.cat([blk[i, s, t] for t, _ in cols], 1) for i, s in rows], 0)))
        s = np.sort(torch.cat(sv).cpu().numpy())[::-1]
        D = top = min(S.m, int(np.sum(s > 1e-12 * s[0])))
        while 0 < D < len(s) and not s[D] < s[D - 1] * (1 - 1e-7):
            D -= 1
        lam[p, :len(s)] = s
        weight.append(float(np.sum(s[:D or top] ** 2)))
        energy.append(e)
        bond.append(b)
    return dict(energy=np.array(energy), bond=np.array(bond), weight=np.array(weight), lam=lam)


def exact(case, seed):
    if case["kind"] == "heff":
        P = ELL[case["lattice"]] // 2
        ps = list(range(P)) if case["p"] < 0 else [case["p"]]
        S = _State(case, seed, pairs=ps)
        N = [S.layout(p)[3] for p in ps]
        return torch.cat([S.apply(p, x) for p, x in zip(ps, _psi(sum(N), seed).split(N))])
    if case["kind"] == "step" and case["lattice"] in ("chain", "randchain"):
        return _exact_step(case, seed)
    return None  # a batch and a measured run start from the library's own steps; the cylinders take a minute and more
