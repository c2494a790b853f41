"""Workloads of the quaternion AO->MO integral transformation, as a program calls it.

A case is one call (or one iteration) of a user's program: a chain or a cluster of atoms with a
contracted basis, molecular-orbital coefficients in hand, the transformed integrals wanted.  The sizes
are those of this repository's input recipes (`synth`: `tiny_dc`, `medium_dc`, `dcb_cluster`,
`large_dcb`, `serving_requests`, the unrestricted and the kinetic-balance chains), scaled down where the
whole system does not fit a pass of two seconds.

Keys of a case:
  kind    "transform": one `Context.transform`, basis and coefficients resident;
          "scf": new coefficients from the host each pass, the result back on the host
          (`set_coefficients` or its variant, then `transform`), as an orbital-optimisation loop does;
          "unpack": `transform`, then `unpack` of the Coulomb block to all complex (pq|rs);
          "batch": `transform_batch` over `n` requests; "serve": `n` requests through a `Server`
  geom    "chain" (n centres in d0) or "cluster" (d0 x d1 x d2 centres)
  shells  "ss" (two s), "sp" (s and p), "spd" (s, p on every 2nd, d on every 4th centre)
  nprim   primitives per shell;  nK  active Kramers pairs (spinors for input "ku")
  blocks  "c" Coulomb, "cg" + Gaunt, "cgb" + gauge;  tau  Schwarz threshold;  form  "split" or "fp64"
  input   "quaternion", "ku" (Kramers-unrestricted spinors) or "rkb" (restricted kinetic balance)
"""
import math

import numpy as np
import torch

from paper_2606_04316_gb300 import qdt, synth

BLOCKS = {"c": ("coulomb",), "cg": ("coulomb", "gaunt"), "cgb": ("coulomb", "gaunt", "gauge")}
FORM = {"split": qdt.SPLIT, "fp64": qdt.FP64}


def _case(name, kind, geom, d, shells, nprim, nK, blocks, tau, form, inp="quaternion", n=1):
    return {"name": name, "kind": kind, "geom": geom, "d0": d[0], "d1": d[1], "d2": d[2], "shells": shells, "nprim": nprim,
            "nK": nK, "blocks": blocks, "tau": tau, "form": form, "input": inp, "n": n}


def listed():
    return [
        # the smallest call: two atoms, all blocks; launches and host work count
        _case("pair-dcb", "transform", "chain", (2, 1, 1), "sp", 2, 2, "cgb", 0.0, "split"),
        # the uncontracted 6-centre model system in the all-FP64 form, nothing screened
        _case("tiny-dc-fp64", "transform", "chain", (6, 1, 1), "ss", 1, 8, "c", 0.0, "fp64"),
        # an iteration of a kinetic-balance SCF: host coefficients in, host integrals out
        _case("rkb9-dcb-scf", "scf", "chain", (9, 1, 1), "sp", 3, 11, "cgb", 1e-12, "split", "rkb"),
        # Kramers-unrestricted spinors, Coulomb and Gaunt, an odd size
        _case("ku13-cg-scf", "scf", "chain", (13, 1, 1), "sp", 3, 27, "cg", 1e-12, "split", "ku"),
        # the reference form of a small molecule: all FP64, all blocks
        _case("chain7-dcb-fp64", "transform", "chain", (7, 1, 1), "sp", 3, 7, "cgb", 1e-12, "fp64"),
        # a small basis with a wide active space: the contractions dominate
        _case("chain9-c-wide", "unpack", "chain", (9, 1, 1), "sp", 3, 20, "c", 1e-11, "split"),
        # s/p/d shells with wide exponent ranges, the large cluster's recipe at 12 centres
        _case("spd12-dcb", "transform", "cluster", (3, 2, 2), "spd", 3, 12, "cgb", 1e-12, "split"),
        # a compact cluster: nearly every shell quartet is kept
        _case("cluster18-dcb", "transform", "cluster", (3, 3, 2), "sp", 3, 17, "cgb", 1e-12, "split"),
        # the screened chain, Dirac-Coulomb, at its full size
        _case("chain40-dc", "transform", "chain", (40, 1, 1), "sp", 3, 40, "c", 1e-12, "split"),
        # the screened chain with all Dirac-Coulomb-Breit blocks
        _case("chain24-dcb", "transform", "chain", (24, 1, 1), "sp", 3, 24, "cgb", 1e-12, "split"),
        # small requests of several users fused into one call
        _case("batch12-dcb", "batch", "chain", (6, 1, 1), "sp", 3, 8, "cgb", 1e-11, "split", n=12),
        # requests with their own geometry arriving at a server
        _case("serve6-dcb", "serve", "cluster", (3, 2, 1), "sp", 3, 8, "cgb", 1e-11, "split", n=6),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["transform", "transform", "transform", "scf", "unpack", "batch", "serve"])
    blocks = rng.choice(["c", "cg", "cgb", "cgb"])
    tau = rng.choice([0.0, 1e-11, 1e-12, 1e-12])
    form = rng.choice(["split", "split", "split", "fp64"])
    inp = rng.choice(["quaternion", "quaternion", "quaternion", "ku", "rkb"])
    geom = rng.choice(["chain", "chain", "cluster"])
    shells = rng.choice(["sp", "sp", "sp", "ss", "spd"])
    nprim = rng.choice([1, 2, 3, 3])
    n = 1
    if kind in ("batch", "serve"):
        n, form, inp, shells, tau = rng.randint(2, 8), "split", "quaternion", "sp", 1e-11
        d = (logint(2, 7), 1, 1) if geom == "chain" else (2, rng.randint(1, 2), rng.randint(1, 2))
        nK = rng.randint(4, 12)
    elif form == "fp64":
        d = (logint(2, 7), 1, 1) if geom == "chain" else (2, rng.randint(1, 2), 1)
        nK = rng.randint(2, 7)
        shells = "sp" if shells == "spd" else shells
    elif geom == "chain":
        shells = "sp" if shells == "spd" else shells
        d = (logint(2, 32 if blocks == "c" and kind == "transform" else 22), 1, 1)
        nK = rng.randint(2, max(4, min(32, 2 * d[0])))
    else:
        d = rng.choice([(2, 2, 1), (2, 2, 2), (3, 2, 1), (3, 2, 2), (3, 3, 1), (4, 2, 2)])
        d = (2, 2, rng.randint(1, 2)) if shells == "spd" else d
        nK = rng.randint(2, 16)
    if kind == "unpack":
        nK = min(nK, 16)
    if tau == 0.0 and geom == "chain":
        d = (min(d[0], 10), 1, 1)
    if inp == "ku":
        geom, d, nK = "chain", (d[0], 1, 1), min(2 * nK, 30)
    if inp == "rkb":
        geom, d = "chain", (d[0], 1, 1)
    if inp != "quaternion":
        shells = "sp"
    if shells == "spd":
        geom, nprim = "cluster", 3
    c = _case("", kind, geom, d, shells, nprim, nK, blocks, tau, form, inp, n)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _problem(case, seed):
    blocks, tau, nK = BLOCKS[case["blocks"]], case["tau"], case["nK"]
    shells = {"ss": (0, 0), "sp": (0, 1), "spd": None}[case["shells"]]
    d = (case["d0"], case["d1"], case["d2"])
    seed = int(seed) % (1 << 31)
    if case["shells"] == "spd":
        p = synth.large_dcb(seed=seed, dims=d, nK=nK)
        p.blocks, p.tau = blocks, tau
        return p
    if case["input"] == "ku":
        return synth.ku_chain_problem(d[0], nK, seed=seed, shells=shells, nprim=case["nprim"], blocks=blocks, tau=tau)
    if case["input"] == "rkb":
        return synth.rkb_chain_problem(d[0], nK, seed=seed, shells=shells, nprim=case["nprim"], blocks=blocks, tau=tau)
    if case["geom"] == "chain":
        return synth.chain_problem(d[0], nK, seed=seed, shells=shells, nprim=case["nprim"], blocks=blocks, tau=tau)
    return synth.cluster_problem(d, nK, seed=seed, shells_fn=lambda i: shells, nprim=case["nprim"], blocks=blocks, tau=tau)


def _problems(case, seed):
    """The requests of a batch or a server: every other one a little larger or smaller."""
    out = []
    for i in range(case["n"]):
        c = dict(case)
        if case["kind"] in ("batch", "serve"):
            c["d0"] = max(1, case["d0"] + (i % 3) - 1)
            c["nK"] = max(1, case["nK"] - (i % 4))
            c["blocks"] = case["blocks"] if i % 2 == 0 else "c"
        out.append(_problem(c, seed * 64 + i))
    return out


def _set(ctx, p, CL, CS):
    if p.rkb:
        ctx.set_rkb_coefficients(CL, CS, synth.C_LIGHT_GEN, spinors=not p.kramers)
    elif p.kramers:
        ctx.set_coefficients(CL, CS)
    else:
        ctx.set_spinor_coefficients(CL, CS)


def prepare(case, seed):
    problems = _problems(case, seed)
    st = {"case": case, "problems": problems, "prec": FORM[case["form"]]}
    if case["kind"] == "serve":
        st["server"] = qdt.Server(0, n_slots=4)
        st["outs"] = [np.zeros(len(p.blocks) * _packed(p)) for p in problems]
        return st
    st["ctx"], st["outs"] = [], []
    for p in problems:
        ctx = qdt.Context(0)
        ctx.set_basis(p.basis)
        if case["kind"] == "scf":       # pinned host buffers, as such a loop keeps them
            st["host"] = [torch.from_numpy(a).pin_memory() for a in (p.CL, p.CS)]
            st["outs"].append(torch.zeros(len(p.blocks) * _packed(p), dtype=torch.float64).pin_memory())
        else:
            _set(ctx, p, torch.from_numpy(p.CL).cuda(), torch.from_numpy(p.CS).cuda())
            st["outs"].append(torch.zeros(len(p.blocks) * _packed(p), dtype=torch.float64, device="cuda"))
        st["ctx"].append(ctx)
    if case["kind"] == "unpack":
        n = (2 if problems[0].kramers else 1) * problems[0].nK
        st["full"] = torch.zeros(2 * n ** 4, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return st


def _packed(p):
    """Doubles of one packed block."""
    nP = p.nK * (p.nK + 1) // 2
    return nP * (nP + 1) // 2 * (16 if p.kramers else 4)


def run(st):
    kind, problems, outs, prec = st["case"]["kind"], st["problems"], st["outs"], st["prec"]
    if kind == "batch":
        qdt.transform_batch([(c, p.blocks, 0, p.nK, p.tau, prec, o) for c, p, o in zip(st["ctx"], problems, outs)])
        return outs
    if kind == "serve":
        srv, handles = st["server"], []
        for p, o in zip(problems, outs):
            req, keep = srv.make_request(p, p.blocks, 0, p.nK, p.tau, prec, o)
            handles.append(srv.submit(req, keep))
        for h in handles:
            srv.wait(h)
        return outs
    ctx, p, out = st["ctx"][0], problems[0], outs[0]
    if kind == "scf":
        _set(ctx, p, st["host"][0], st["host"][1])
    ctx.transform(p.blocks, 0, p.nK, p.tau, prec, out)
    if kind == "unpack":
        ctx.unpack(out[: _packed(p)], p.nK, "coulomb", st["full"])
        return [out, st["full"]]
    return [out]


# -------------------------------------------------------------------- work

def work(case):
    """Coefficients read and integrals written once; the two half-transforms and the Hermite
    contractions of the integrals as multiply-adds, with the share of pair products that a chain's
    screening leaves (pairs further apart than about 14 centres are below the threshold)."""
    total_b = total_f = 0.0
    for i in range(case["n"]):
        d0, nK, blocks = case["d0"], case["nK"], case["blocks"]
        if case["kind"] in ("batch", "serve"):
            d0, nK = max(1, d0 + (i % 3) - 1), max(1, nK - (i % 4))
            blocks = blocks if i % 2 == 0 else "c"
        nc = d0 * case["d1"] * case["d2"]
        keep = min(1.0, (14.0 / nc) ** 2) if case["geom"] == "chain" and case["tau"] > 0 else 1.0
        nL = {"ss": 2 * nc, "sp": 4 * nc, "spd": nc + 3 * ((nc + 1) // 2) + 6 * ((nc + 3) // 4)}[case["shells"]]
        nS = 3 * nL if case["shells"] == "ss" else int(2.25 * nL)         # p shells: 6 distinct derivative functions
        parts = 2 if case["input"] == "ku" else 4
        nP = nK * (nK + 1) // 2
        cols, packed = parts * nP, nP * (nP + 1) // 2 * parts * parts
        M0, M1 = nL * (nL + 1) // 2 + nS * (nS + 1) // 2, nL * nS
        nb = {"c": 1, "cg": 2, "cgb": 3}[blocks]
        total_b += 8.0 * (4 * nL * nK * (2 if case["input"] == "rkb" else 4) + nb * packed)
        if case["kind"] == "unpack":
            total_b += 16.0 * ((2 if parts == 4 else 1) * nK) ** 4 + 8.0 * packed
        prim = float(case["nprim"]) ** 4
        f = 2.0 * M0 * M0 * keep * cols + M0 * cols * cols + 20.0 * prim * M0 * M0 * keep / 2
        if nb > 1:
            f += 3 * (2.0 * M1 * M1 * keep * cols + M1 * cols * cols) + 20.0 * prim * M1 * M1 * keep / 2
        if nb > 2:
            f += 2.0 * 9 * M1 * M1 * keep * cols + 3 * M1 * cols * cols + 80.0 * prim * M1 * M1 * keep / 2
        total_f += f
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------- the same in 64 bits, unscreened

def _herm(L):
    """Hermite triples of order <= L and their index."""
    tri = [(t, u, s - t - u) for s in range(L + 1) for t in range(s, -1, -1) for u in range(s - t, -1, -1)]
    return tri, {h: i for i, h in enumerate(tri)}


def _boys(T, nmax):
    """F_0..F_nmax of a tensor T: the series of the top order and the downward recursion, or the
    asymptotic F_0 and the upward recursion where erf(sqrt T) is 1 in 64 bits."""
    big = T > 40.0
    t = torch.where(big, torch.ones_like(T), T)
    term = torch.full_like(t, 1.0 / (2 * nmax + 1))
    total = term.clone()
    for k in range(1, 180):
        term = term * (2 * t) / (2 * nmax + 2 * k + 1)
        total = total + term
    e = torch.exp(-t)
    lo = [None] * (nmax + 1)
    lo[nmax] = e * total
    for n in range(nmax - 1, -1, -1):
        lo[n] = (2 * t * lo[n + 1] + e) / (2 * n + 1)
    b = torch.where(big, T, torch.full_like(T, 50.0))
    eb = torch.exp(-b)
    hi = 0.5 * torch.sqrt(math.pi / b)
    out = []
    for n in range(nmax + 1):
        out.append(torch.where(big, hi, lo[n]))
        hi = ((2 * n + 1) * hi - eb) / (2 * b)
    return out


def _hermite_tensor(base, X, L):
    """R_{tuv} of order <= L from the R^n_{000} in `base`, X the three distances; a list over triples."""
    tri, _ = _herm(L)
    cur = {}
    for m in range(L, -1, -1):
        new = {(0, 0, 0): base[m]}
        for h in tri[1:]:
            if sum(h) > L - m:
                break
            ax = 0 if h[0] else 1 if h[1] else 2
            d = [0, 0, 0]
            d[ax] = 1
            h1 = tuple(a - b for a, b in zip(h, d))
            v = X[ax] * cur[h1]
            if h[ax] > 1:
                h2 = tuple(a - 2 * b for a, b in zip(h, d))
                v = v + (h[ax] - 1) * cur[h2]
            new[h] = v
        cur = new
    return [cur[h] for h in tri]


class _Shells:
    """Contracted Cartesian shells and their derivative functions as sums of primitive terms."""

    def __init__(self, basis):
        self.n = basis.n_shells
        self.l = [int(x) for x in basis.shell_l]
        self.A = [np.asarray(basis.xyz[c], float) for c in basis.shell_center]
        off = np.concatenate([[0], np.cumsum(basis.shell_nprim)])
        self.ex = [np.asarray(basis.exps[off[s]:off[s + 1]], float) for s in range(self.n)]
        self.co = [np.asarray(basis.coefs[off[s]:off[s + 1]], float) for s in range(self.n)]
        self.first = np.concatenate([[0], np.cumsum([(x + 1) * (x + 2) // 2 for x in self.l])])

    def functions(self, s, small):
        """Per function of a shell: a list of (powers, weight per primitive)."""
        l, a, d = self.l[s], self.ex[s], self.co[s]
        out = []
        for c in [(i, j, l - i - j) for i in range(l, -1, -1) for j in range(l - i, -1, -1)]:
            g = a[:, None] + a[None, :]
            ov = d[:, None] * d[None, :] * (math.pi / g) ** 1.5
            for k in c:
                ov = ov * math.prod(range(2 * k - 1, 0, -2)) / (2 * g) ** k
            w = d / math.sqrt(ov.sum())
            if not small:
                out.append([(c, w)])
                continue
            for K in range(3):
                up = tuple(x + (i == K) for i, x in enumerate(c))
                terms = [(up, -2.0 * a * w)]
                if c[K]:
                    terms.append((tuple(x - (i == K) for i, x in enumerate(c)), c[K] * w))
                out.append(terms)
        return out


def _pair(sh, A, sa, B, sb):
    """One shell pair: exponents p [n], centres P [n, 3] and E [n, herm, function pairs] of its primitives."""
    a, b = np.meshgrid(sh.ex[A], sh.ex[B], indexing="ij")
    a, b = a.ravel(), b.ravel()
    p = a + b
    la, lb = sh.l[A] + sa, sh.l[B] + sb
    P = (a[:, None] * sh.A[A] + b[:, None] * sh.A[B]) / p[:, None]
    E1 = []
    for x in range(3):
        ab = sh.A[A][x] - sh.A[B][x]
        t = np.zeros((la + 1, lb + 1, la + lb + 2, p.size))
        t[0, 0, 0] = np.exp(-a * b / p * ab * ab)
        for i in range(la + 1):
            for j in range(lb + 1):
                if i == j == 0:
                    continue
                src, dist = (t[i - 1, j], P[:, x] - sh.A[A][x]) if j == 0 else (t[i, j - 1], P[:, x] - sh.A[B][x])
                for k in range(i + j + 1):
                    t[i, j, k] = dist * src[k] + (k + 1) * src[k + 1] + (src[k - 1] / (2 * p) if k else 0.0)
        E1.append(t)
    tri, _ = _herm(la + lb)
    fa, fb = sh.functions(A, sa), sh.functions(B, sb)
    na, nb = len(sh.ex[A]), len(sh.ex[B])
    E = np.zeros((p.size, len(tri), len(fa) * len(fb)))
    for i, f in enumerate(fa):
        for j, g in enumerate(fb):
            for pa, wa in f:
                for pb, wb in g:
                    w = np.repeat(wa, nb) * np.tile(wb, na)
                    for h, (t, u, v) in enumerate(tri):
                        if t <= pa[0] + pb[0] and u <= pa[1] + pb[1] and v <= pa[2] + pb[2]:
                            E[:, h, i * len(fb) + j] += w * E1[0][pa[0], pb[0], t] * E1[1][pa[1], pb[1], u] * E1[2][pa[2], pb[2], v]
    return p, P, E


def _groups(sh, cls, dev):
    """Shell pairs of a class grouped by kind: stacked p, P, E, the first row of each pair and its functions."""
    kinds, rows, row = {}, [], 0
    if cls == 0:
        todo = [(A, s, B, s) for s in (0, 1) for A in range(sh.n) for B in range(A, sh.n)]
    else:
        todo = [(A, 0, B, 1) for A in range(sh.n) for B in range(sh.n)]
    for A, sa, B, sb in todo:
        p, P, E = _pair(sh, A, sa, B, sb)
        kinds.setdefault((sh.l[A] + sa + sh.l[B] + sb, sa, E.shape), []).append((p, P, E, row))
        na, nb = E.shape[2] // _nf(sh, B, sb), _nf(sh, B, sb)
        fa = _f0(sh, A, sa) + np.repeat(np.arange(na), nb)
        fb = _f0(sh, B, sb) + np.tile(np.arange(nb), na)
        rows.append((fa, fb, A == B and sa == sb))
        row += E.shape[2]
    g = []
    for (L, _, _), v in kinds.items():
        p, P, E = (torch.from_numpy(np.stack([x[i] for x in v])).to(dev) for i in range(3))
        idx = torch.tensor(np.stack([x[3] + np.arange(x[2].shape[2]) for x in v]), device=dev)
        g.append((L, p, P, E, idx))
    return g, rows, row


def _nf(sh, s, small):
    return (sh.l[s] + 1) * (sh.l[s] + 2) // 2 * (3 if small else 1)


def _f0(sh, s, small):
    return int(sh.first[-1]) + 3 * int(sh.first[s]) if small else int(sh.first[s])


def _integrals(groups, M, gauge, dev):
    """(ab|cd) over a class, and for the gauge kernel the six (ab|r_I r_J/r^3|cd)."""
    G = torch.zeros(7 if gauge else 1, M, M, dtype=torch.float64, device=dev)
    IJ = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
    for L1, p1, P1, E1, i1 in groups:
        tri1, _ = _herm(L1)
        for L2, p2, P2, E2, i2 in groups:
            tri2, _ = _herm(L2)
            sgn = torch.tensor([(-1.0) ** sum(h) for h in tri2], dtype=torch.float64, device=dev)
            E2s = (E2 * sgn[None, None, :, None]).reshape(E2.shape[0], -1, E2.shape[3])
            L = L1 + L2 + (2 if gauge else 0)
            _, ih = _herm(L)
            per = p1.shape[1] * p2.numel() * (len(ih) * (2 if gauge else 1) * 3 + 7 * len(tri1) * len(tri2)) * 8
            step = max(1, int(6e9 // per))
            for c in range(0, p1.shape[0], step):
                p, P, E = p1[c:c + step], P1[c:c + step], E1[c:c + step]
                a = p[:, :, None, None]
                q = p2[None, None]
                X = [P[:, :, None, None, x] - P2[None, None, :, :, x] for x in range(3)]
                rho = a * q / (a + q)
                T = rho * (X[0] ** 2 + X[1] ** 2 + X[2] ** 2)
                F = _boys(T, L)
                pre = 2 * math.pi ** 2.5 / (a * q * torch.sqrt(a + q))
                base = [F[n] * pre * (-2 * rho) ** n for n in range(L1 + L2 + 1)]
                RC = torch.stack(_hermite_tensor(base, X, L1 + L2))

                def contract(R, shift):
                    at = torch.tensor([[ih[tuple(x + y + z for x, y, z in zip(h, k, shift))] for k in tri2] for h in tri1], device=dev)
                    m = R[at]                                    # [h, k, c, ij, G, kl]
                    m = m.permute(4, 2, 3, 0, 5, 1).reshape(m.shape[4], -1, m.shape[5] * m.shape[1])
                    t = torch.bmm(m, E2s).reshape(m.shape[0], p.shape[0], p.shape[1] * len(tri1), -1)
                    e = E.reshape(E.shape[0], -1, E.shape[3])
                    return torch.einsum("gcky,ckx->cxgy", t, e)

                r, s = i1[c:c + step][:, :, None, None], i2[None, None]
                G[0][r, s] = contract(RC, (0, 0, 0))
                if gauge:
                    pr = math.pi ** 2.5 * torch.sqrt(a + q) / (a * q) ** 2
                    Fm = [-(2 * T * F[0] + torch.exp(-T))] + F
                    RR = torch.stack(_hermite_tensor([(F[n] - Fm[n]) * pr * (-2 * rho) ** n for n in range(L + 1)], X, L))
                    for k, (I, J) in enumerate(IJ):
                        sh = [0, 0, 0]
                        sh[I] += 1
                        sh[J] += 1
                        v = -contract(RR, tuple(sh))
                        G[1 + k][r, s] = v + (G[0][r, s] if I == J else 0.0)
    return G


def _spinors(C, kramers):
    """Complex [rows, 2, n]: every spinor (both members of a Kramers pair)."""
    al, be = C[..., 0] + 1j * C[..., 1], C[..., 2] + 1j * C[..., 3]
    if not kramers:
        return np.stack([al, be], 1)
    out = np.zeros((C.shape[0], 2, 2 * C.shape[1]), complex)
    out[:, 0, 0::2], out[:, 1, 0::2], out[:, 0, 1::2], out[:, 1, 1::2] = al, be, -be.conj(), al.conj()
    return out


SIGMA = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], complex)


def _exact_problem(p, full):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    sh = _Shells(p.basis)
    CL, CS = _spinors(p.CL, p.kramers), _spinors(p.CS, p.kramers)
    if p.rkb:                                            # (1/2c) sigma.p over the derivative functions
        C = np.einsum("Kuv,mvp->mKup", SIGMA, CS) * (-0.5j / synth.C_LIGHT_GEN)
        CS = C.reshape(-1, 2, C.shape[3])
    C = torch.from_numpy(np.concatenate([CL, CS])).to(dev)
    n = p.nK
    P, Q = np.triu_indices(n)
    nP = P.size
    done, whole = [], None
    cache = {}
    for b in p.blocks:
        cls = 0 if b == "coulomb" else 1
        if cls not in cache:
            cache.clear()
            g, rows, M = _groups(sh, cls, dev)
            fa = torch.tensor(np.concatenate([r[0] for r in rows]), device=dev)
            fb = torch.tensor(np.concatenate([r[1] for r in rows]), device=dev)
            once = torch.tensor(np.concatenate([np.full(r[0].size, r[2]) for r in rows]), device=dev)
            cache[cls] = (_integrals(g, M, cls == 1 and "gauge" in p.blocks, dev), fa, fb, once)
        G, fa, fb, once = cache[cls]
        ops = [torch.eye(2, dtype=torch.complex128, device=dev)] if cls == 0 else [torch.from_numpy(s).to(dev) for s in SIGMA]

        def density(x, y, op):
            d = torch.zeros(fa.numel(), len(x), dtype=torch.complex128, device=dev)
            for t in range(2):
                for u in range(2):
                    if op[t, u] != 0:
                        d += op[t, u] * C[fa][:, t, x].conj() * C[fb][:, u, y]
                        d += torch.where(once[:, None], 0.0, op[t, u] * C[fb][:, t, x].conj() * C[fa][:, u, y])
            return d

        pairs = [(2 * P, 2 * Q), (2 * P + 1, 2 * Q)] if p.kramers else [(P, Q)]
        D = []
        for op in ops:
            cols = []
            for x, y in pairs:
                d = density(x, y, op)
                cols += [d.real, d.imag]
            D.append(torch.stack(cols, 2).reshape(fa.numel(), -1))
        if b != "gauge":
            O = sum(d.T @ (G[0] @ d) for d in D)
        else:
            at = [[1, 2, 3], [2, 4, 5], [3, 5, 6]]
            O = sum(D[i].T @ (G[at[i][j]] @ D[j]) for i in range(3) for j in range(3))
        parts = 2 * len(pairs)
        iu, ju = (torch.from_numpy(v).to(dev) for v in np.triu_indices(nP))
        done.append(O.reshape(nP, parts, nP, parts)[iu, :, ju, :].reshape(-1))
        if full and b == "coulomb":
            m = (2 if p.kramers else 1) * n
            x, y = np.divmod(np.arange(m * m), m)
            d = density(x, y, ops[0])
            re, im = G[0] @ d.real, G[0] @ d.imag
            whole = torch.stack([d.real.T @ re - d.imag.T @ im, d.real.T @ im + d.imag.T @ re], -1).reshape(-1)
    return torch.cat(done).cpu(), (None if whole is None else whole.cpu())


def exact(case, seed):
    cost = 0.0
    for i in range(case["n"]):
        nc = (case["d0"] + 1) * case["d1"] * case["d2"] if case["n"] > 1 else case["d0"] * case["d1"] * case["d2"]
        per = {"ss": 30.0, "sp": 3500.0, "spd": 12000.0}[case["shells"]]
        cost += nc ** 4 * (case["nprim"] / 3.0) ** 4 * per * (4 if case["blocks"] == "cgb" else 1)
    if cost > 4.5e8:                 # longer than several seconds
        return None
    got = [_exact_problem(p, case["kind"] == "unpack") for p in _problems(case, seed)]
    if case["kind"] == "unpack":
        return [got[0][0], got[0][1]]
    return [g[0] for g in got]
