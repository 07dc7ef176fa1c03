"""Timing cases of the two-site DMRG library: what its users have it do.

A program of this library holds a context (integrals, block bases, a position) and
asks for H psi at that position over and over with new vectors (a Davidson run is
nothing else), in FP64 or in one of the two mixed working precisions, for one problem
or for a batch of them; between Davidson runs it moves one block on.  So the contexts
here are the handle that a program keeps (one per case, grown once from seeded bases),
and the inputs that change from pass to pass are the wave functions.

Entry points ("do"):
  hpsi      DMRG.hpsi on a CUDA tensor
  batch     Batch.hpsi: the H psi of several problems in one call
  davidson  DMRG.davidson to convergence from a start vector (energy, wave function)
  lowp      DMRG.davidson_lowp: a fixed number of working-precision iterations
  move      DMRG.renormalize with given bases, then H psi at the next position (which
            reads every operator of the new block)

A product in a mixed working precision is accurate to 32 bits at best, so its outputs
are handed on in float32.
"""
import math

import numpy as np
import torch

from paper_2001_04890_gb300 import binding

PREC = {"fp64": binding.PREC_FP64, "fp32": binding.PREC_FP32, "bf16x3": binding.PREC_BF16X3}
SITE = ((0, 0), (1, 0), (0, 1), (1, 1))  # (n_up, n_dn) of the states 0, up, dn, updn


def listed():
    def case(name, do, prec, L, M, N=None, two_sz=0, M_right=None, tc_min=33, by_work=0, count=1, iters=0):
        return dict(name=name, do=do, prec=prec, L=L, N=N if N is not None else L, two_sz=two_sz, M=M,
                    M_right=M_right or M, tc_min=tc_min, by_work=by_work, count=count, iters=iters)

    return [
        # the smallest problem of the benchmark and tests: launches and latency
        case("hpsi_fp64_L8_M64", "hpsi", "fp64", 8, 64),
        # a small active space with an odd electron number and unequal bond dimensions
        case("hpsi_fp64_L11_odd", "hpsi", "fp64", 11, 150, N=9, two_sz=1, M_right=117),
        # few sectors of many states (up to 88): the large blocks of an FP64 run
        case("hpsi_fp64_L12_M800", "hpsi", "fp64", 12, 800),
        # the FP64 benchmark: middle bond of 24 orbitals
        case("hpsi_fp64_L24_M512", "hpsi", "fp64", 24, 512),
        # the FP32 working precision, at the benchmark's size and with large blocks
        case("hpsi_fp32_L24_M512", "hpsi", "fp32", 24, 512),
        case("hpsi_fp32_L12_M800", "hpsi", "fp32", 12, 800),
        # split-BF16 x3 with the launch shape that a context starts with (small blocks in FP64)
        case("hpsi_bf16x3_L24_M1024", "hpsi", "bf16x3", 24, 1024),
        # split-BF16 x3 with every block on the tensor cores: the mixed workload of the benchmark
        case("hpsi_bf16x3_all_L40_M2000", "hpsi", "bf16x3", 40, 2000, tc_min=1, by_work=1),
        # many small problems in one call (10 to 20 orbitals, M 64 to 256)
        case("batch_bf16x3_16", "batch", "bf16x3", 20, 256, tc_min=1, count=16),
        # the benchmark's step: working-precision Davidson iterations from a fixed vector
        case("lowp_bf16x3_all_L24_M1024", "lowp", "bf16x3", 24, 1024, tc_min=1, by_work=1, iters=4),
        # a whole FP64 Davidson run of a small problem
        case("davidson_fp64_L10_M128", "davidson", "fp64", 10, 128),
        # one block move of a sweep
        case("move_fp64_L16_M256", "move", "fp64", 16, 256),
    ]


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    do = rng.choice(["hpsi", "hpsi", "hpsi", "batch", "lowp", "davidson", "move"])
    prec = rng.choice(["fp64", "fp64", "fp32", "bf16x3", "bf16x3"])
    L = rng.randint(8, 24)
    M = between(64, 512 if prec == "fp64" else 1024)
    tc_min = rng.choice([1, 33])
    count, iters = 1, 0
    if do == "batch":
        L, M, count = 20, 256, rng.randint(3, 16)
    elif do == "lowp":
        prec, iters = rng.choice(["fp32", "bf16x3"]), rng.randint(2, 6)
    elif do == "davidson":
        prec, L, M = "fp64", rng.randint(8, 10), between(64, 256)
    elif do == "move":
        prec, L, M = "fp64", rng.randint(8, 16), between(64, 256)
    N = L + rng.randint(-2, 2)
    return dict(do=do, prec=prec, L=L, N=N, two_sz=N % 2, M=M, M_right=max(48, int(M * rng.uniform(0.6, 1.0))),
                tc_min=tc_min, by_work=rng.choice([0, 1]), count=count, iters=iters)

# --------------------------------------------------------------------------- problems


def integrals(L, rng):
    """Seeded one- and two-electron integrals with the locality of an orbital ordering."""
    h = np.diag(-2.0 + 4.0 * np.arange(L) / L)
    i, j = np.triu_indices(L, k=1)
    h[i, j] = h[j, i] = rng.normal(0.0, 0.1, i.size) * np.exp(-np.abs(i - j) / 4.0)
    i, j = np.triu_indices(L)
    B = np.zeros((2 * L, L, L))
    B[:, i, j] = rng.normal(0.0, 0.15, (2 * L, i.size))
    B[:, j, i] = B[:, i, j]
    B = B.reshape(2 * L, L * L)
    return h, (B.T @ B).reshape(L, L, L, L)


def filling(case):
    return (case["N"] + case["two_sz"]) // 2, (case["N"] - case["two_sz"]) // 2


def middle(case):
    return (case["L"] - 2) // 2


def enlarged(sec, left):
    """Sectors of block (x) site (left) or site (x) block, sorted: {(nu, nd): [(block sector, site state), ...]}."""
    out = {}
    for key in sorted(sec):
        for s, (u, d) in enumerate(SITE):
            out.setdefault((key[0] + u, key[1] + d), []).append((key, s))
    for subs in out.values():
        subs.sort(key=None if left else lambda x: (x[1], x[0]))
    return {E: out[E] for E in sorted(out)}


def kept_states(dims, sites, case, M):
    """States kept per sector: a Gaussian around the mean filling, at most what is there, M in all."""
    d = np.array(list(dims.values()))
    if d.sum() <= M:
        return dict(dims)
    mean = np.array(filling(case)) * sites / case["L"]
    w = -((np.array(list(dims)) - mean) ** 2).sum(1) / (sites / 2.0)  # logarithm of the weight
    lo, hi = -50.0, 400.0
    for _ in range(60):
        mid = (lo + hi) / 2
        lo, hi = (mid, hi) if np.minimum(d, np.floor(np.exp(np.minimum(w + mid, 30.0)) + 0.5)).sum() < M else (lo, mid)
    kept = np.minimum(d, np.floor(np.exp(np.minimum(w + hi, 30.0)) + 0.5)).astype(int)
    for n in np.argsort(-kept, kind="stable")[: kept.sum() - M]:
        kept[n] -= 1
    return {E: int(m) for E, m in zip(dims, kept)}


def one_site_more(sec, direction, sites, case, rng):
    """A renormalization with random orthonormal bases: (direction, kept, O by enlarged sector, sectors after)."""
    lay = enlarged(sec, direction > 0)
    dims = {E: sum(sec[a] for a, _ in subs) for E, subs in lay.items()}
    kept = kept_states(dims, sites, case, case["M"] if direction > 0 else case["M_right"])
    O = {E: np.linalg.qr(rng.standard_normal((dims[E], kept[E])))[0] for E in lay}
    return direction, kept, O, {E: m for E, m in kept.items() if m > 0}


def bases(case, k, rng):
    """The renormalizations that build the left blocks of 1..k and the right blocks of 1..L-2-k sites."""
    sides = []
    for direction, sites in ((1, k), (-1, case["L"] - 2 - k)):
        sec, steps = {(0, 0): 1}, []
        for n in range(1, sites + 1):
            steps.append(one_site_more(sec, direction, n, case, rng))
            sec = steps[-1][3]
        sides.append(steps)
    return sides


def problem(case, seed=0):
    """(h, v, left steps, right steps) of a context at its middle bond."""
    rng = np.random.default_rng(seed)
    h, v = integrals(case["L"], rng)
    return (h, v, *bases(case, middle(case), rng))


def flat(O):
    return np.concatenate([o.ravel() for o in O.values()])


def grow(case, seed):
    """A context at its middle bond."""
    h, v, left, right = problem(case, seed)
    c = binding.DMRG(h, v, case["N"], case["two_sz"], case["M"], PREC[case["prec"]])
    c.set_tune(tc_min=case["tc_min"], by_work=case["by_work"])
    c.set_renorm_precision(binding.PREC_FP64 if case["prec"] == "fp64" else binding.PREC_FP32)
    for at, steps in ((0, left), (case["L"] - 2, right)):
        c.set_position(at, 1 if at == 0 else -1)
        for direction, kept, O, _ in steps:
            c.renormalize(direction, flat(O), list(kept.values()))
    c.set_renorm_precision(binding.PREC_FP64)
    c.set_position(middle(case), 1)
    return c


def instances(case):
    """The problems of a batch: sizes up to the case's, every one with its own integrals and bases."""
    rng = np.random.default_rng(77)
    sizes = [(int(rng.integers(10, case["L"] + 1)), int(rng.integers(64, case["M"] + 1))) for _ in range(case["count"])]
    return [dict(case, L=L, N=L, two_sz=L % 2, M=M, M_right=M) for L, M in sizes]


_kept = {}  # the handle of the case at hand: the program that the case stands for keeps it


def handle(case):
    """(context or batch, length of psi)."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _kept:
        _kept.clear()
        if case["do"] == "batch":
            b = binding.Batch([grow(one, n) for n, one in enumerate(instances(case))])
            _kept[key] = b, b.offsets[-1]
        else:
            c = grow(case, 0)
            c.hpsi_flops()  # plans the position, as the first call there does
            _kept[key] = c, c.psi_layout()[1]
    return _kept[key]


def psi_blocks(left, right, case):
    """The blocks (a, b, c, d) of psi in their order."""
    nu, nd = filling(case)
    for a in sorted(left):
        for b, (bu, bd) in enumerate(SITE):
            for c, (cu, cd) in enumerate(SITE):
                d = (nu - a[0] - bu - cu, nd - a[1] - bd - cd)
                if d in right:
                    yield a, b, c, d


def sectors(steps):
    return steps[-1][3] if steps else {(0, 0): 1}


# --------------------------------------------------------------------------- what is measured


def move_basis(left, case, seed):
    """The basis of a block move: the left block one site longer."""
    return one_site_more(sectors(left), 1, middle(case) + 1, case, np.random.default_rng(seed + 500))


def start_vector(dim, seed):
    x = np.random.default_rng(seed + 1000).standard_normal(dim)
    return x / np.linalg.norm(x)


def prepare(case, seed):
    h, dim = handle(case)
    s = dict(case=case, h=h)
    if case["do"] == "move":
        _, _, left, right = problem(case)
        _, kept, O, sec = move_basis(left, case, seed)
        after = sectors(right[:-1])
        dim = sum(sec[a] * after[d] for a, _, _, d in psi_blocks(sec, after, case))
        s.update(kept=list(kept.values()), O=flat(O))
    s["psi"] = torch.from_numpy(start_vector(dim, seed)).cuda()
    return s


def run(s):
    case, h, psi = s["case"], s["h"], s["psi"]
    if case["do"] in ("hpsi", "batch"):
        sigma = h.hpsi(psi)
        return sigma if case["prec"] == "fp64" else sigma.float()
    if case["do"] == "move":
        h.set_position(middle(case), 1)
        h.renormalize(1, s["O"], s["kept"])
        return h.hpsi(psi)
    h.set_psi(psi)
    out = torch.empty_like(psi)
    if case["do"] == "lowp":
        energy, _ = h.davidson_lowp(tol=1e-300, max_iter=case["iters"], allow_noconv=True)
        return torch.tensor(energy, dtype=torch.float32), h.get_psi(out).float()
    energy, _ = h.davidson(tol=1e-11, max_iter=400, allow_noconv=True)
    h.get_psi(out)
    return energy, out * torch.sign(torch.dot(out, psi))  # an eigenvector has no sign of its own


def block_ops(sec, sites, L):
    """Stored operators of a block by the change of (n_up, n_dn): [(change, how many)]."""
    k = sites
    return [((0, 0), 1 + k * (k + 1)), ((1, 0), L), ((0, 1), L), ((2, 0), k * (k - 1) // 2),
            ((0, 2), k * (k - 1) // 2), ((1, 1), k * k), ((1, -1), k * k)]


def work(case):
    if case["do"] == "batch":
        each = [work(dict(one, do="hpsi")) for one in instances(case)]
        return {key: sum(w[key] for w in each) for key in ("bytes", "flops")}
    h, v, left, right = problem(case)
    k, L = middle(case), case["L"]
    a, b, n_left, n_right = sectors(left), sectors(right), k, L - 2 - k
    flops = bytes_ = 0.0
    size = 8 if case["prec"] == "fp64" else 4
    if case["do"] == "move":  # every new operator O^T (block (x) site) O, each old one read, each new one written
        _, _, _, new = move_basis(left, case, 0)
        lay = enlarged(a, True)
        for (du, dd), n in block_ops(new, k + 1, L):
            for E, m in new.items():
                F = new.get((E[0] + du, E[1] + dd), 0)
                bytes_ += 8 * n * m * F
                for x, _ in lay[E]:
                    y = a.get((x[0] + du, x[1] + dd), 0)
                    flops += 2.0 * n * (F * y * a[x] + F * a[x] * m)
        for (du, dd), n in block_ops(a, k, L):
            bytes_ += 8 * n * sum(m * a.get((x[0] + du, x[1] + dd), 0) for x, m in a.items())
        a, b, k, n_left, n_right = new, sectors(right[:-1]), k + 1, k + 1, n_right - 1
    table = [[(*E, m) for E, m in sorted(sec.items())] for sec in (a, b)]
    one, _ = binding.plan_hpsi_flops(h, v, case["N"], case["two_sz"], k, *table)
    # matrix-vector products: the start vector's too; a run to convergence takes 40 or more
    times = {"lowp": case["iters"] + 1, "davidson": 40}.get(case["do"], 1)
    for sec, sites in ((a, n_left), (b, n_right)):
        for (du, dd), n in block_ops(sec, sites, L):
            bytes_ += size * n * sum(m * sec.get((x[0] + du, x[1] + dd), 0) for x, m in sec.items())
    dim = sum(a[x] * b[y] for x, _, _, y in psi_blocks(a, b, case))
    return {"bytes": bytes_ + 16.0 * dim, "flops": flops + times * one}


# --------------------------------------------------------------------------- in 64 bits, from the definition


class FullCI:
    """H on the determinants of all L orbitals, and the block bases as vectors of them."""

    def __init__(self, case, h, v, left, right):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        L, (nu, nd) = case["L"], filling(case)
        self.L = L
        up, dn = ([m for m in range(1 << L) if bin(m).count("1") == n] for n in (nu, nd))
        bit = lambda m, i: m >> (L - 1 - i) & 1  # noqa: E731  orbital 0 is the leftmost site
        U = np.array([[bit(m, i) for i in range(L)] for m in up])
        D = np.array([[bit(m, i) for i in range(L)] for m in dn])
        four = 4 ** np.arange(L - 1, -1, -1)
        self.at = self.put((U @ four)[:, None] + (2 * D @ four)[None, :])
        before = np.cumsum(D, 1) - D  # each up electron passes the down electrons of the sites before it
        self.sign = self.put(1.0 - 2.0 * ((U @ before.T) & 1))
        self.Eu, self.Ed = self.moves(up, L, bit), self.moves(dn, L, bit)
        hp = h - 0.5 * np.einsum("ijjl->il", v)
        self.h, self.v = self.put(hp.reshape(-1)), self.put(0.5 * v.reshape(L * L, L * L))
        self.VL, self.VR = self.vectors(left, True), self.vectors(right, False)
        self.blocks = list(psi_blocks(sectors(left), sectors(right), case))

    def put(self, x):
        return torch.from_numpy(np.ascontiguousarray(x)).to(self.dev)

    def moves(self, strings, L, bit):
        """E_ij = a+_i a_j on the strings of one spin: (L*L, n, n)."""
        row = {m: n for n, m in enumerate(strings)}
        E = np.zeros((L * L, len(strings), len(strings)))
        for m, col in row.items():
            for j in range(L):
                if not bit(m, j):
                    continue
                low = m ^ 1 << (L - 1 - j)
                for i in range(L):
                    if not bit(low, i):
                        between = sum(bit(low, x) for x in range(min(i, j) + 1, max(i, j)))
                        E[i * L + j, row[low | 1 << (L - 1 - i)], col] = (-1.0) ** between
        return self.put(E)

    def vectors(self, steps, left):
        """Basis vectors of a block by sector, in the product basis of its sites."""
        V = {(0, 0): torch.ones(1, 1, dtype=torch.float64, device=self.dev)}
        for n, (_, kept, O, sec) in enumerate(steps):
            new = {}
            for E, subs in enlarged({x: y.shape[1] for x, y in V.items()}, left).items():
                if kept[E] == 0:
                    continue
                size, at = 4 ** n, 0
                X = torch.zeros(size, 4, kept[E], dtype=torch.float64, device=self.dev)
                Y = X if left else X.view(4, size, kept[E])
                o = self.put(O[E])
                for a, s in subs:
                    m = V[a].shape[1]
                    (Y[:, s] if left else Y[s]).add_(V[a] @ o[at:at + m])
                    at += m
                new[E] = Y.reshape(4 * size, kept[E])
            V = new
        return V

    def apply(self, psi):
        nl, nr = (next(iter(V.values())).shape[0] for V in (self.VL, self.VR))
        full = torch.zeros(nl, 4, 4, nr, dtype=torch.float64, device=self.dev)
        at = 0
        for a, b, c, d in self.blocks:
            m, n = self.VL[a].shape[1], self.VR[d].shape[1]
            full[:, b, c] += self.VL[a] @ psi[at:at + m * n].view(m, n) @ self.VR[d].T
            at += m * n
        C = full.view(-1)[self.at] * self.sign
        D = self.Eu @ C + C @ self.Ed.transpose(1, 2)
        G = (self.v @ D.view(D.shape[0], -1)).view(D.shape) + self.h[:, None, None] * C
        S = torch.einsum("xab,xbc->ac", self.Eu, G) + torch.einsum("xab,xcb->ac", G, self.Ed)
        full.zero_().view(-1)[self.at.view(-1)] = (S * self.sign).view(-1)
        return torch.cat([(self.VL[a].T @ full[:, b, c] @ self.VR[d]).reshape(-1) for a, b, c, d in self.blocks])


def lowest(H, x, steps=250):
    """Lowest eigenpair by Lanczos with every vector kept orthogonal."""
    V, alpha, beta = [x / x.norm()], [], []
    for _ in range(min(steps, x.numel())):
        w = H(V[-1])
        alpha.append(torch.dot(w, V[-1]))
        Q = torch.stack(V)
        for _ in range(2):
            w = w - Q.T @ (Q @ w)
        beta.append(w.norm())
        if beta[-1] < 1e-10:
            break
        V.append(w / beta[-1])
    n = len(alpha)
    T = torch.diag(torch.stack(alpha))
    for i in range(n - 1):
        T[i, i + 1] = T[i + 1, i] = beta[i]
    e, y = torch.linalg.eigh(T)
    z = torch.stack(V[:n]).T @ y[:, 0]
    return e[0].item(), z * torch.sign(torch.dot(z, x))


def exact(case, seed):
    if case["L"] > 12 or case["do"] in ("batch", "lowp") or case["do"] == "davidson" and case["L"] > 10:
        return None
    h, v, left, right = problem(case)
    if case["do"] == "move":
        left, right = left + [move_basis(left, case, seed)], right[:-1]
    H = FullCI(case, h, v, left, right)
    dim = sum(H.VL[a].shape[1] * H.VR[d].shape[1] for a, _, _, d in H.blocks)
    psi = H.put(start_vector(dim, seed))
    return lowest(H.apply, psi) if case["do"] == "davidson" else H.apply(psi)
