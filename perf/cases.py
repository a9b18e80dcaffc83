"""What a user of the two-site DMRG engine has it do, as cases that can be timed and compared.

A case is an operation at one two-site step of a seeded synthetic system: N orbitals, n electrons, 2*S_z, bond
dimension D, the step's left site, and how the bond dimension is spread (`sectors` = 0: over every reachable
(particles, 2*S_z) sector in proportion to its Schmidt-rank bound, which gives many small blocks; k > 0: over the k
largest sectors of each bond, the few large blocks that sweeps arrive at).  Sizes are those of the repository's
workloads and tests: 8, 13 and 24 orbitals, D = 256 to 512, and what lies between.

Operations, each through the package's public entry points:
  heff      Y = H_eff X for nvec vectors in one of the three precisions (the Davidson product, where sweep time goes)
  adjoint   the autograd function: Y = H_eff X, then the gradients for X and for both operator arenas
  davidson  the lowest eigenpair from a given start vector, with a cap on the products as in warm-up sweeps
  step      one whole two-site step on host buffers: Davidson, truncation to D, renormalisation
  rdm       the 1- and 2-particle reduced density matrices (integral gradients)
"""
import itertools
import math

import numpy as np
import torch

from paper_2305_05581_gb300 import Context, TNS_BF16X3, TNS_FP64, TNS_TF32
from paper_2305_05581_gb300.autograd import arena_tensor, heff

PRECISION = {"fp64": TNS_FP64, "tf32": TNS_TF32, "bf16x3": TNS_BF16X3}
SITE_QN = ((0, 0), (1, 1), (1, -1), (2, 0))  # (particles, 2*S_z) of |0>, |up>, |dn>, |updn>


def _case(name, op, N, n, s2, D, site, sectors, precision="fp64", nvec=1, cap=0):
    return dict(name=name, op=op, N=N, n_elec=n, two_sz=s2, D=D, site=site, sectors=sectors, precision=precision,
                nvec=nvec, cap=cap)


def listed():
    return [
        # the smallest system: 8 orbitals with an exact bond dimension, blocks of 1 to 36 states; launches and latency
        _case("heff_fp64_n8", "heff", 8, 8, 0, 256, 3, 0),
        # a few large, ragged sectors (up to about 100 states) in an open-shell system: the sizes of the full-size tests
        _case("heff_fp64_n13_few", "heff", 13, 13, 1, 260, 6, 3),
        # the 24-orbital workload on every sector: millions of products on blocks of at most 26 states
        _case("heff_fp64_n24", "heff", 24, 24, 0, 512, 11, 0),
        # the same bond dimension in the few sectors a sweep concentrates it in: FP64 products and refreshes
        _case("heff_fp64_n24_few", "heff", 24, 24, 0, 512, 11, 9),
        # the reduced-precision product that the precision form's Davidson runs some forty times a step
        _case("heff_bf16_n24", "heff", 24, 24, 0, 512, 11, 0, "bf16x3"),
        _case("heff_bf16_n24_few", "heff", 24, 24, 0, 512, 11, 9, "bf16x3"),
        # a block of four Davidson vectors, an off-centre bond, an odd bond dimension
        _case("heff_bf16_n16_x4", "heff", 16, 15, 1, 333, 5, 6, "bf16x3", nvec=4),
        # the TF32 form at a bond whose blocks are wide rather than tall
        _case("heff_tf32_n13_few", "heff", 13, 13, 1, 260, 4, 3, "tf32"),
        # the differentiation form: product and gradients
        _case("adjoint_n13", "adjoint", 13, 12, 0, 160, 6, 5),
        # Davidson in FP64, capped as in a warm-up sweep
        _case("davidson_fp64_n16", "davidson", 16, 16, 0, 200, 7, 8, cap=14),
        # a whole two-site step in the precision form, start vector and result in host memory
        _case("step_bf16_n16", "step", 16, 16, 0, 256, 7, 6, "bf16x3", cap=16),
        # density matrices of a 10-orbital state
        _case("rdm_n10", "rdm", 10, 10, 0, 96, 4, 0),
    ]


def draw(rng):
    """One more case of the same ranges: 8 to 22 orbitals (fewer for the whole calls), D up to 448."""
    op = rng.choice(["heff"] * 6 + ["adjoint", "davidson", "step", "rdm"])
    hi = {"heff": 22, "adjoint": 14, "davidson": 17, "step": 17, "rdm": 11}[op]
    dmax = {"heff": 448, "adjoint": 180, "davidson": 224, "step": 256, "rdm": 120}[op]
    while True:
        N = rng.randint(8, hi)
        n = N + rng.choice([-2, -1, 0, 0, 1])
        s2 = rng.choice([0, 2]) if n % 2 == 0 else rng.choice([-1, 1, 3])
        D = int(round(math.exp(rng.uniform(math.log(32), math.log(dmax)))))
        site = rng.randint(N // 3, (2 * N) // 3 - 1)
        sectors = rng.choice([0, 3, 4, 5, 6, 8, 10, 12])
        precision = "fp64" if op in ("adjoint", "rdm") else rng.choice(["fp64", "fp64", "bf16x3", "bf16x3", "tf32"])
        nvec = rng.choice([1, 1, 1, 2, 3, 4]) if op == "heff" else 1
        cap = rng.randint(8, 16) if op in ("davidson", "step") else 0
        c = dict(op=op, N=N, n_elec=n, two_sz=s2, D=D, site=site, sectors=sectors, precision=precision, nvec=nvec, cap=cap)
        if all(_bonds(c)):
            return c


# ----------------------------------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------------------------------
def _determinants(sites, n, s2):
    if (n + s2) % 2:
        return 0
    nu, nd = (n + s2) // 2, (n - s2) // 2
    return math.comb(sites, nu) * math.comb(sites, nd) if nu >= 0 and nd >= 0 else 0


def _bonds(case):
    """[(sector, dim)] of every bond: dims in proportion to the Schmidt-rank bound, D in all, and such that every site
    tensor can be an isometry from either side."""
    N, n, s2, D = case["N"], case["n_elec"], case["two_sz"], case["D"]
    dims = []
    for b in range(N + 1):
        full = {}
        for q in itertools.product(range(2 * b + 1), range(-b, b + 1)):
            d = min(_determinants(b, *q), _determinants(N - b, n - q[0], s2 - q[1]))
            if d > 0:
                full[q] = d
        if case["sectors"]:
            full = {q: full[q] for q in sorted(full, key=lambda q: (-full[q], q))[:case["sectors"]]}
        total = sum(full.values())
        if total > D:
            share = {q: D * f / total for q, f in full.items()}
            full = {q: int(s) for q, s in share.items()}
            for q in sorted(share, key=lambda q: (full[q] - share[q], q))[:D - sum(full.values())]:
                full[q] += 1
        dims.append({q: d for q, d in full.items() if d > 0})
    changed = True
    while changed:
        changed = False
        for b, step in [(b, -1) for b in range(1, N + 1)] + [(b, 1) for b in range(N - 1, -1, -1)]:
            for q in list(dims[b]):
                room = sum(dims[b + step].get((q[0] + step * a, q[1] + step * c), 0) for a, c in SITE_QN)
                if dims[b][q] > room:
                    changed = True
                    dims[b][q] = room
                    if not room:
                        del dims[b][q]
    return [sorted(d.items()) for d in dims]


def _system(case, seed):
    """Integrals with the symmetry and decay of molecular ones, and an MPS canonical around the step."""
    N, site = case["N"], case["site"]
    rng = np.random.default_rng([seed, N, case["D"]])
    lam = 3.0 if N <= 13 else 5.0
    dist = np.abs(np.subtract.outer(np.arange(N), np.arange(N)))
    h = rng.standard_normal((N, N)) * np.exp(-dist / lam)
    h = np.tril(h) + np.tril(h, -1).T
    i, j = np.tril_indices(N)
    pair = np.zeros((N, N), dtype=np.int64)
    pair[i, j] = pair[j, i] = np.arange(len(i))
    g = 0.5 * rng.standard_normal((len(i), len(i))) * np.exp(-np.add.outer(dist[i, j], dist[i, j]) / lam)
    g = np.tril(g) + np.tril(g, -1).T
    v = g[pair[:, :, None, None], pair[None, None]]
    v[np.arange(N), np.arange(N), np.arange(N), np.arange(N)] += 1.0
    bonds = _bonds(case)
    sites = []
    for b in range(N):
        left, right, blocks = dict(bonds[b]), dict(bonds[b + 1]), {}
        if b <= site:
            for qr, dr in bonds[b + 1]:
                keys = [((qr[0] - a, qr[1] - c), s) for s, (a, c) in enumerate(SITE_QN)]
                keys = [k for k in keys if k[0] in left]
                q = np.linalg.qr(rng.standard_normal((sum(left[k[0]] for k in keys), dr)))[0]
                at = 0
                for k in keys:
                    blocks[k] = np.ascontiguousarray(q[at:at + left[k[0]]])
                    at += left[k[0]]
        else:
            for ql, dl in bonds[b]:
                keys = [((ql[0] + a, ql[1] + c), s) for s, (a, c) in enumerate(SITE_QN)]
                keys = [k for k in keys if k[0] in right]
                q = np.linalg.qr(rng.standard_normal((sum(right[k[0]] for k in keys), dl)))[0].T
                at = 0
                for qr, s in keys:
                    blocks[(ql, s)] = np.ascontiguousarray(q[:, at:at + right[qr]])
                    at += right[qr]
        sites.append(blocks)
    return h, v, bonds, sites


def _psi_blocks(case, bonds):
    """(q_l, s1, s2, q_r) and shape of every block of the two-site vector, in the engine's order."""
    n, s2, k = case["n_elec"], case["two_sz"], case["site"]
    right = sorted(((n - q[0], s2 - q[1]), d) for q, d in bonds[k + 2])
    out = []
    for ql, dl in bonds[k]:
        for a, b in itertools.product(range(4), range(4)):
            need = (n - ql[0] - SITE_QN[a][0] - SITE_QN[b][0], s2 - ql[1] - SITE_QN[a][1] - SITE_QN[b][1])
            out += [((ql, a, b, qr), (dl, dr)) for qr, dr in right if qr == need]
    return out


def _vector(case, bonds, rng):
    """A unit two-site vector in the basis of the bonds, its entries graded over the states as Schmidt weights are."""
    k = case["site"]
    wl = {q: 10.0 ** (-3.0 * rng.random(d)) for q, d in bonds[k]}
    wr = {(case["n_elec"] - q[0], case["two_sz"] - q[1]): 10.0 ** (-3.0 * rng.random(d)) for q, d in bonds[k + 2]}
    x = np.concatenate([(rng.standard_normal(shape) * wl[ql][:, None] * wr[qr]).ravel()
                        for (ql, a, b, qr), shape in _psi_blocks(case, bonds)])
    return x / np.linalg.norm(x)


def _vectors(case, seed, bonds):
    rng = np.random.default_rng([seed, 77])
    return np.stack([_vector(case, bonds, rng) for _ in range(2 if case["op"] == "adjoint" else case["nvec"])])


def _prepare(case, seed):
    h, v, bonds, sites = _system(case, seed)
    ctx = Context(device=0, stream=torch.cuda.current_stream().cuda_stream)
    ctx.load_integrals(h, v)
    ctx.mps_import(case["N"], case["n_elec"], case["two_sz"], case["D"], bonds, sites)
    ctx.build_env(case["site"])
    return ctx, _vectors(case, seed, bonds)


def prepare(case, seed):
    ctx, x = _prepare(case, seed)
    s = dict(case=case, ctx=ctx, site=case["site"], precision=PRECISION[case["precision"]])
    if case["op"] == "step":
        s["x"] = torch.from_numpy(x[0]).pin_memory()
        s["psi"] = torch.empty_like(s["x"]).pin_memory()
        s["kept"] = torch.empty_like(s["x"]).pin_memory()
        return s
    s["x"] = torch.from_numpy(x).cuda()
    s["y"] = torch.empty_like(s["x"])
    if case["op"] == "adjoint":
        s["arenas"] = [arena_tensor(ctx, case["site"], side).requires_grad_() for side in (0, 1)]
        s["x"], s["yb"] = s["x"][0].clone().requires_grad_(), s["x"][1].clone()
    return s


# ----------------------------------------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------------------------------------
def run(s):
    c, ctx, site = s["case"], s["ctx"], s["site"]
    if c["op"] == "heff":
        ctx.heff_apply_ptr(site, s["x"].data_ptr(), s["y"].data_ptr(), c["nvec"], s["precision"])
        return s["y"]
    if c["op"] == "adjoint":
        y = heff(s["x"], *s["arenas"], ctx, site)
        return (y, *torch.autograd.grad(y, [s["x"], *s["arenas"]], s["yb"]))
    if c["op"] == "davidson":
        s["y"].copy_(s["x"])
        energy, _, _ = ctx.davidson_ptr(site, s["y"].data_ptr(), tol=1e-8, max_iter=c["cap"], precision=s["precision"])
        return s["y"], energy
    if c["op"] == "step":
        st = ctx.step(site, True, c["D"], tol=1e-8, max_iter=c["cap"], precision=s["precision"],
                      x0_host_ptr=s["x"].data_ptr(), psi_host_ptr=s["psi"].data_ptr())
        ctx.psi_guess(site, s["kept"].data_ptr())  # the truncated wavefunction, from the step's new site tensors
        return s["psi"], s["kept"], st.energy
    return ctx.rdm_ptr(site, s["x"].data_ptr(), c["N"])


_COST = {}


def work(case):
    """Flops: Eq. (2) with the cheaper chain order, as the library counts them for these tables; bytes: both blocks'
    operators once, each vector read and written once."""
    key = tuple(sorted((k, v) for k, v in case.items() if k in ("N", "n_elec", "two_sz", "D", "site", "sectors")))
    if key not in _COST:
        ctx, x = _prepare(case, 0)
        flops, _ = ctx.heff_flops(case["site"])
        _COST[key] = flops, sum(ctx.env_arena(case["site"], side)[1] for side in (0, 1)), x.shape[1]
        ctx.close()
    flops, arena, length = _COST[key]
    if case["op"] == "adjoint":  # the product, H_eff Ybar, and alpha Ybar R X^T and alpha Ybar^T L X of every product
        return {"bytes": 8.0 * (2 * arena + 4 * length), "flops": 4.0 * flops}
    if case["op"] == "rdm":
        return {"bytes": 8.0 * (2 * arena + length + case["N"] ** 2 + case["N"] ** 4), "flops": 3.0 * flops}
    products = case["cap"] if case["op"] in ("davidson", "step") else case["nvec"]
    return {"bytes": 8.0 * (arena + 2 * length * case["nvec"]), "flops": float(flops) * products}


# ----------------------------------------------------------------------------------------------------------------------
# the same numbers from the determinant expansion, in 64 bits (up to 13 orbitals)
# ----------------------------------------------------------------------------------------------------------------------
class _Expansion:
    """The two-site space of a case inside the space of all determinants (occupation strings of up and down spins)."""

    def __init__(self, case, seed):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.N, n, s2 = case["N"], case["n_elec"], case["two_sz"]
        self.h, self.v, bonds, sites = _system(case, seed)
        self.x, k, N = _vectors(case, seed, bonds), case["site"], self.N
        strings = [[sum(1 << p for p in c) for c in itertools.combinations(range(N), e)]
                   for e in ((n + s2) // 2, (n - s2) // 2)]
        self.strings = strings
        at = [np.full(1 << N, -1, dtype=np.int64) for _ in range(2)]
        for a, s in zip(at, strings):
            a[s] = np.arange(len(s))
        left = self._grow(bonds, sites, range(k))
        right = self._grow(bonds, sites, range(N - 1, k + 1, -1), (n, s2))
        self.blocks = []
        for (ql, s1, s2_, qr), shape in _psi_blocks(case, bonds):
            ul, dl, ml = left[ql]
            ur, dr, mr = right[(n - qr[0], s2 - qr[1])]
            up = ul[:, None] + ur[None] + ((s1 in (1, 3)) << k) + ((s2_ in (1, 3)) << (k + 1))
            dn = dl[:, None] + dr[None] + ((s1 in (2, 3)) << k) + ((s2_ in (2, 3)) << (k + 1))
            # creation operators run orbital by orbital, up before down: the sign of moving every up to the front
            odd = np.zeros(up.shape, dtype=np.int64)
            for p in range(N):
                odd += ((dn >> p) & 1) * sum((up >> q) & 1 for q in range(p + 1, N))
            where = at[0][up] * len(strings[1]) + at[1][dn]
            self.blocks.append((self._t(ml), self._t(mr), self._t(1.0 - 2.0 * (odd % 2)), self._t(where), shape))
        self.moves = [[self._move(p, q, s, a) for p in range(N) for q in range(N)] for s, a in zip(strings, at)]

    def _t(self, a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(self.dev)

    @staticmethod
    def _grow(bonds, sites, order, target=None):
        """{bond sector: (up strings, down strings, states as determinants x dim or dim x determinants)} of a block."""
        one = np.zeros(1, dtype=np.int64)
        at = {((0, 0) if target is None else target): (one, one, np.ones((1, 1)))}
        for b in order:
            new = {}
            for (ql, s), t in sites[b].items():
                qr = (ql[0] + SITE_QN[s][0], ql[1] + SITE_QN[s][1])
                src, dst = (ql, qr) if target is None else (qr, ql)
                if src in at:
                    u, d, m = at[src]
                    new.setdefault(dst, []).append((u + ((s in (1, 3)) << b), d + ((s in (2, 3)) << b),
                                                    m @ t if target is None else t @ m))
            at = {q: (np.concatenate([p[0] for p in ps]), np.concatenate([p[1] for p in ps]),
                      np.concatenate([p[2] for p in ps], axis=0 if target is None else 1)) for q, ps in new.items()}
        return at

    def _move(self, p, q, strings, at):
        """a+_p a_q on the strings of one spin: source rows, target rows, signs."""
        s = np.array(strings, dtype=np.int64)
        ok = ((s >> q) & 1 == 1) & ((p == q) | ((s >> p) & 1 == 0))
        src = np.nonzero(ok)[0]
        t = s[src] - (1 << q) + (1 << p)
        odd = sum(((s[src] >> r) & 1 for r in range(min(p, q) + 1, max(p, q))), np.zeros(len(src), dtype=np.int64))
        return self._t(src), self._t(at[t]), self._t(1.0 - 2.0 * (odd % 2))

    def full(self, x):
        out = torch.zeros(len(self.strings[0]) * len(self.strings[1]), dtype=torch.float64, device=self.dev)
        o = 0
        for ml, mr, sign, where, (m, n) in self.blocks:
            blk = self._t(x[o:o + m * n].reshape(m, n))
            out[where.reshape(-1)] = (sign * (ml @ blk @ mr)).reshape(-1)
            o += m * n
        return out.reshape(len(self.strings[0]), len(self.strings[1]))

    def project(self, c):
        c = c.reshape(-1)
        return torch.cat([(ml.T @ (sign * c[where]) @ mr.T).reshape(-1) for ml, mr, sign, where, _ in self.blocks])

    def excite(self, c, pq, add=None):
        """sum over spins of a+_p a_q on c (added to `add`)."""
        out = torch.zeros_like(c) if add is None else add
        src, dst, sg = self.moves[0][pq]
        out.index_add_(0, dst, c[src] * sg[:, None])
        src, dst, sg = self.moves[1][pq]
        out.index_add_(1, dst, c[:, src] * sg)
        return out

    def hamiltonian(self, c):
        N = self.N
        d = torch.stack([self.excite(c, pq) for pq in range(N * N)]).reshape(N * N, -1)
        one = self.h - 0.5 * np.einsum("prrq->pq", self.v)
        g = 0.5 * self._t(self.v.reshape(N * N, N * N)) @ d
        del d
        g += self._t(one.reshape(-1, 1)) * c.reshape(1, -1)
        out = torch.zeros_like(c)
        for pq in range(N * N):
            self.excite(g[pq].reshape(c.shape), pq, out)
        return out

    def heff(self, x):
        return self.project(self.hamiltonian(self.full(x)))


def exact(case, seed):
    if case["N"] > 13 or case["op"] in ("davidson", "step") or (case["op"] == "rdm" and case["N"] > 11):
        return None
    e = _Expansion(case, seed)
    if case["op"] == "heff":
        return torch.stack([e.heff(x) for x in e.x])
    if case["op"] == "adjoint":
        return e.heff(e.x[0]), e.heff(e.x[1]), None, None
    N, c = case["N"], e.full(e.x[0])
    d = torch.stack([e.excite(c, pq) for pq in range(N * N)]).reshape(N * N, -1)
    norm = float((c * c).sum())
    gamma = (d @ c.reshape(-1) / norm).reshape(N, N).cpu().numpy()
    two = (d @ d.T / norm).reshape(N, N, N, N).cpu().numpy().transpose(1, 0, 2, 3)  # <E_ij E_kl> = <E_ji psi, E_kl psi>
    for j in range(N):
        two[:, j, j, :] -= gamma
    two = (two + two.transpose(1, 0, 2, 3)) / 2
    two = (two + two.transpose(0, 1, 3, 2)) / 2
    two = (two + two.transpose(2, 3, 0, 1)) / 2
    return (gamma + gamma.T) / 2, two
