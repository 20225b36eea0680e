"""The work this library is timed on: contractions, their gradients, transforms and factorizations.

Every case is one pass of what a tensor-network program does with the
library, through its public entry points.  Legs follow the recipes of
``synthetic``; sizes run from the parity tests' to the benchmark's.

kinds
  pair        one contraction of two rank-4 U(1) tensors with its gradients
  mps         the one-site effective Hamiltonian ((L.A).W).R of an MPS chain
              (U(1), fermion parity or SU(2) x U(1) legs), with or without
              the gradients of L, A, W and R
  recouple    the SU(2) recoupling contraction of two rank-4 tensors with its gradients
  su2_move    permute (recoupled), fuse and split of a rank-4 SU(2) tensor
  u1_move     permute, fuse and split of a rank-4 U(1) tensor
  batch       many independent two-site effective Hamiltonians in batch plans, with gradients
  mera        energy of a ternary-MERA patch and its gradient in w and u
  svd, eig    blockwise factorization of a two-site tensor or of its density
              matrix, and the product of the factors
"""
import functools
import itertools
import json
import math

import numpy as np
import torch

import paper_1203_2222_gb300 as P
from paper_1203_2222_gb300 import networks, synthetic

GROUPS = {"u1": P.U1, "z2f": P.Z2F, "su2u1": P.SU2U1}
DTYPES = {"float32": torch.float32, "float64": torch.float64}


# --------------------------------------------------------------------- cases --
def listed():
    return [
        # a small operator product, as in a test or in a small simulation: launches and host time
        {"name": "u1_pair_small", "kind": "pair", "labels": 5, "degen": 4, "seed": 1234, "dtype": "float32"},
        # a matrix-vector product of a double-precision eigensolver (no gradient)
        {"name": "u1_mps_apply_f64", "kind": "mps", "group": "u1", "D": 768, "dtype": "float64", "grad": False},
        # gradient-based optimisation of an MPS at an ordinary bond: many small sectors
        {"name": "u1_mps_grad", "kind": "mps", "group": "u1", "D": 2048, "dtype": "float32", "grad": True},
        # fermionic chain: two large sectors a leg
        {"name": "z2f_mps_grad", "kind": "mps", "group": "z2f", "D": 2048, "dtype": "float32", "grad": True},
        # spinful electrons: composite labels, small recoupled sectors
        {"name": "su2u1_mps_grad", "kind": "mps", "group": "su2u1", "D": 1024, "dtype": "float32", "grad": True},
        # large-sector recoupling contraction, forward and backward: the largest call
        {"name": "su2_recouple_grad", "kind": "recouple", "dmax": 32, "jmax2": 8, "dtype": "float32"},
        # index manipulation of an SU(2) tensor between contractions
        {"name": "su2_move_f64", "kind": "su2_move", "spins": 3, "degen": 20, "dtype": "float64"},
        # index manipulation of a large abelian tensor with ragged degeneracies
        {"name": "u1_move", "kind": "u1_move", "labels": 5, "degen": 31, "dtype": "float32"},
        # many chains at once (parallel two-site updates)
        {"name": "u1_batch_grad", "kind": "batch", "n": 128, "dmin": 64, "dmax": 1024},
        # a MERA patch: a network of rank-4 tensors with tiny sectors
        {"name": "u1_mera_grad", "kind": "mera", "deg": 5, "qmax": 4},
        # truncation step of a two-site update: the bond keeps the chain's own degeneracies
        {"name": "u1_svd", "kind": "svd", "D": 2048, "full": False},
        # spectrum of the two-site density matrix, nothing truncated
        {"name": "u1_eig", "kind": "eig", "D": 2048, "full": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "mps", "mps", "mps", "recouple", "su2_move", "u1_move", "batch", "mera", "svd", "eig"])
    dtype = rng.choice(["float32", "float32", "float64"])
    if kind == "pair":
        return {"kind": kind, "labels": rng.randint(2, 7), "degen": rng.randint(2, 8), "seed": rng.randint(1, 9999),
                "dtype": dtype}
    if kind == "mps":
        group = rng.choice(["u1", "z2f", "su2u1"])
        if dtype == "float64":
            D = _log(rng, 48, {"u1": 1500, "z2f": 400, "su2u1": 700}[group])
        else:
            D = _log(rng, 48, {"u1": 4096, "z2f": 3072, "su2u1": 2048}[group])
        return {"kind": kind, "group": group, "D": D, "dtype": dtype, "grad": rng.random() < 0.6}
    if kind == "recouple":
        if dtype == "float64":
            return {"kind": kind, "dmax": rng.randint(2, 6), "jmax2": rng.randint(3, 7), "dtype": dtype}
        return {"kind": kind, "dmax": _log(rng, 3, 26), "jmax2": rng.randint(4, 8), "dtype": dtype}
    if kind == "su2_move":
        return {"kind": kind, "spins": rng.randint(2, 5), "degen": _log(rng, 3, 16), "dtype": dtype}
    if kind == "u1_move":
        return {"kind": kind, "labels": rng.randint(1, 7), "degen": _log(rng, 3, 30), "dtype": dtype}
    if kind == "batch":
        dmin = _log(rng, 32, 256)
        return {"kind": kind, "n": _log(rng, 4, 128), "dmin": dmin, "dmax": _log(rng, dmin, 1024)}
    if kind == "mera":
        return {"kind": kind, "deg": rng.randint(2, 6), "qmax": rng.randint(2, 4)}
    return {"kind": kind, "D": _log(rng, 48, 2048), "full": rng.random() < 0.5}


# ---------------------------------------------------------------------- legs --
def _ragged(degen, n, stream):
    """n degeneracies around ``degen`` (at most ``degen`` + 2, at least 1)."""
    r = synthetic.uniform_int(1234 + degen, max(1, degen - 5), degen + 2, n, stream=stream)
    return [int(x) for x in r]


def _reversed(legs):
    return [(l, d, -s) for l, d, s in legs]


@functools.lru_cache(maxsize=None)
def _spec(key):
    """Legs and contraction order of a case (plain tuples; nothing on the GPU)."""
    c = json.loads(key)
    k = c["kind"]
    if k == "pair":
        qs = list(range(-(c["labels"] // 2), c["labels"] - c["labels"] // 2))
        dl = [synthetic.uniform_int(c["seed"], 1, c["degen"], len(qs), stream=i) for i in range(6)]
        A = [(qs, dl[0], 1), (qs, dl[1], 1), (qs, dl[2], -1), (qs, dl[3], -1)]
        B = [(qs, dl[2], 1), (qs, dl[3], 1), (qs, dl[4], -1), (qs, dl[5], -1)]
        return {"A": A, "B": B, "pairs": ([2, 3], [0, 1])}
    if k == "mps":
        if c["group"] == "u1":
            q = max(2, min(20, c["D"] // 24))
            return synthetic.u1_mps_heff(D=c["D"], qmax=q, sigma=max(1.0, 0.3 * q))
        if c["group"] == "z2f":
            return synthetic.z2f_mps_heff(D=c["D"])
        return synthetic.su2u1_mps_heff(D=c["D"])
    if k == "recouple":
        r = synthetic.su2_recouple(dmax=c["dmax"], jmax2=c["jmax2"])
        return {"A": r["A"], "B": r["B"], "pairs": (r["pairsA"], r["pairsB"])}
    if k == "su2_move":
        spins = [2 * i for i in range(c["spins"])]
        return {"T": [(spins, [c["degen"]] * len(spins), 1)] * 4, "perm": [0, 2, 1, 3]}
    if k == "u1_move":
        qs = list(range(-(c["labels"] // 2), c["labels"] - c["labels"] // 2))
        legs = [(qs, _ragged(c["degen"], len(qs), i), s) for i, s in enumerate((1, -1, 1, -1))]
        return {"T": legs, "perm": [2, 0, 3, 1]}
    if k == "batch":
        return synthetic.u1_two_site_batch(n=c["n"], dmin=c["dmin"], dmax=c["dmax"])
    if k == "mera":
        return synthetic.u1_mera(qmax=c["qmax"], deg=c["deg"])
    q = max(2, min(20, c["D"] // 24))
    return synthetic.u1_two_site_svd(D=c["D"], qmax=q, sigma=max(1.0, 0.3 * q))


def _key(case):
    return json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)


def _dtype(case):
    return DTYPES[case.get("dtype", "float64" if case["kind"] in ("svd", "eig") else "float32")]


# ------------------------------------------------------ structures and inputs --
@functools.lru_cache(maxsize=None)
def _handles(key):
    """Structures (and constants) a program builds once and keeps; its plans hang on them."""
    c, s = json.loads(key), _spec(key)
    k, H = c["kind"], {}
    if k in ("pair", "recouple"):
        g = P.U1 if k == "pair" else P.SU2
        H = {n: P.Structure(g, s[n]) for n in "AB"}
    elif k == "mps":
        H = {n: P.Structure(GROUPS[c["group"]], s[n]) for n in "LAWR"}
    elif k in ("su2_move", "u1_move"):
        H["T"] = P.Structure(P.SU2 if k == "su2_move" else P.U1, s["T"])
    elif k == "batch":
        S = {n: [P.Structure(P.U1, p[n]) for p in s["problems"]] for n in ("L", "theta", "W", "R")}
        plans, cur = [], S["L"]
        for an, bn, pa, pb in s["steps"]:
            plans.append(P.contract_batch_plan(cur if an is None else S[an], S[bn], pa, pb, P.BF16X3))
            cur = plans[-1].outs
        H = {"plans": plans, "numel": {"L": plans[0].off_a[-1], "theta": plans[0].off_b[-1], "W": plans[1].off_b[-1],
                                       "R": plans[3].off_b[-1]}}
    elif k == "mera":
        S = networks.mera_structures(s)
        h, one = networks.mera_h_and_identity(S, s)
        H = {"S": S, "h": torch.as_tensor(h).float().cuda(), "one": torch.as_tensor(one).float().cuda()}
    else:
        if k == "eig":
            H["T"] = P.Structure(P.U1, s["theta"][:2] + _reversed(s["theta"][:2]))
        else:
            H["T"] = P.Structure(P.U1, s["theta"])
        plan = P.svd_plan(H["T"], 2) if k == "svd" else P.eig_plan(H["T"], 2)
        H["plan"], H["keep"] = plan, _kept(key, plan.labels, plan.full)
    return H


def _kept(key, labels, full):
    """Vectors kept per block: all, or what the chain's own bond leg holds of that charge
    (theta's row legs are incoming, so block x meets the bond's charge -x)."""
    if json.loads(key)["full"]:
        return list(full)
    q, d, _ = _spec(key)["theta"][0]
    bond = dict(zip(q, d))
    return [min(f, bond.get(-x, 0)) for x, f in zip(labels, full)]


def _randn(gen, n, dtype, scale=1.0):
    return torch.randn(n, device="cuda", generator=gen, dtype=dtype).mul_(scale)


def _numel(key):
    """Elements of every random input, in the order they are drawn."""
    H, k = _handles(key), json.loads(key)["kind"]
    if k in ("pair", "recouple"):
        return {n: H[n].numel for n in "AB"}
    if k == "mps":
        return {n: H[n].numel for n in "LAWR"}
    if k == "batch":
        return H["numel"]
    if k == "mera":
        return {n: H["S"][n].numel for n in "twu"}
    return {"T": H["T"].numel}


def _inputs(case, seed):
    key, k = _key(case), case["kind"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = _dtype(case)
    if k == "eig":
        return {"T": _density(_spec(key)["theta"], gen)}
    scale = 1.0 / math.sqrt(_spec(key)["chi"]) if k == "mera" else 1.0
    return {n: _randn(gen, m, dtype, scale) for n, m in _numel(key).items()}


def _density(theta, gen):
    """rho = M M^T of a random two-site matrix M, block by block, as block data (row legs, row legs reversed)."""
    legs = theta[:2] + _reversed(theta[:2])
    lay, n = _layout("u1", legs)
    (qa, da, _), (qs, ds, _), (qt, dt, _), (qb, db, _) = theta
    rows = {}
    for (i, j) in itertools.product(range(len(qa)), range(len(qs))):
        rows.setdefault(-qa[i] - qs[j], []).append((i, j))
    cols = {}
    for (i, j) in itertools.product(range(len(qt)), range(len(qb))):
        x = qt[i] - qb[j]
        cols[x] = cols.get(x, 0) + dt[i] * db[j]
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    where = {(p[0], p[1], p[2], p[3]): (o, sh) for p, _, o, sh in lay}
    for x, rt in sorted(rows.items()):
        d = [da[i] * ds[j] for i, j in rt]
        M = torch.randn(sum(d), max(1, cols.get(x, 0)), dtype=torch.float64, device="cuda", generator=gen)
        R = M @ M.T
        R = 0.5 * (R + R.T)
        r0 = np.concatenate([[0], np.cumsum(d)])
        for a, (i, j) in enumerate(rt):
            for b, (i2, j2) in enumerate(rt):
                o, sh = where[(i, j, i2, j2)]
                out[o:o + d[a] * d[b]] = R[r0[a]:r0[a + 1], r0[b]:r0[b + 1]].reshape(-1)
    return out


def prepare(case, seed):
    key, k = _key(case), case["kind"]
    H, x = _handles(key), _inputs(case, seed)
    st = {"kind": k, "case": case, "H": H, "x": x, "spec": _spec(key)}
    grad = k in ("pair", "recouple", "batch") or (k == "mps" and case["grad"])
    if grad:
        for v in x.values():
            v.requires_grad_(True)
    if k == "mera":
        x["w"].requires_grad_(True)
        x["u"].requires_grad_(True)
        return st
    if grad:  # the cotangent of the result, as the rest of a network hands it back
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed) + 77)
        st["G"] = _randn(gen, _result_numel(key), _dtype(case))
    return st


@functools.lru_cache(maxsize=None)
def _result_numel(key):
    c, H, s = json.loads(key), _handles(key), _spec(key)
    prec = P.FP64 if _dtype(c) == torch.float64 else P.BF16X3
    if c["kind"] in ("pair", "recouple"):
        return P.contract_plan(H["A"], H["B"], *s["pairs"], prec).out.numel
    if c["kind"] == "batch":
        return H["plans"][3].off_c[-1]
    t1 = P.contract_plan(H["L"], H["A"], [2], [0], prec).out
    t2 = P.contract_plan(t1, H["W"], *map(list, s["steps"][0]), prec).out
    return P.contract_plan(t2, H["R"], *map(list, s["steps"][1]), prec).out.numel


# ---------------------------------------------------------------------- pass --
def run(st):
    k, H, x, s = st["kind"], st["H"], st["x"], st["spec"]
    if k in ("pair", "recouple"):
        C = P.contract(P.SymTensor(H["A"], x["A"]), P.SymTensor(H["B"], x["B"]), *s["pairs"]).data
        dA, dB = torch.autograd.grad(C, [x["A"], x["B"]], grad_outputs=st["G"])
        return {"C": C, "dA": dA, "dB": dB}
    if k == "mps":
        T = {n: P.SymTensor(H[n], x[n]) for n in "LAWR"}
        T1 = P.contract(T["L"], T["A"], [2], [0])
        T2 = P.contract(T1, T["W"], *s["steps"][0])
        Y = P.contract(T2, T["R"], *s["steps"][1]).data
        if not st["case"]["grad"]:
            return {"Y": Y}
        g = torch.autograd.grad(Y, [x[n] for n in "LAWR"], grad_outputs=st["G"])
        return dict(zip(("Y", "dL", "dA", "dW", "dR"), (Y,) + g))
    if k in ("su2_move", "u1_move"):
        M = P.permute(P.SymTensor(H["T"], x["T"]), s["perm"])
        F = P.fuse(M, 0)
        B = P.split(F, 0, [M.legs[0], M.legs[1]])
        return {"permuted": M.data, "fused": F.data, "split": B.data}
    if k == "batch":
        p = H["plans"]
        t = P.contract_batch(p[0], x["L"], x["theta"])
        t = P.contract_batch(p[1], t, x["W"])
        t = P.contract_batch(p[2], t, x["W"])
        Y = P.contract_batch(p[3], t, x["R"])
        g = torch.autograd.grad(Y, [x[n] for n in ("L", "theta", "W", "R")], grad_outputs=st["G"])
        return dict(zip(("Y", "dL", "dtheta", "dW", "dR"), (Y,) + g))
    if k == "mera":
        E = networks.mera_energy(H["S"], x["t"], x["w"], x["u"], H["h"], H["one"], checkpoint=True)
        dw, du = torch.autograd.grad(E, [x["w"], x["u"]])
        return {"E": E, "dw": dw, "du": du}
    # svd, eig: the factors are fixed up to the sign of every vector pair, the values and the product are not
    plan = H["plan"]
    values = plan.execute(x["T"])
    Us, Vs = plan.bond(H["keep"])
    U, V, kept = plan.factors(2)
    M = P.contract(P.SymTensor(Us, U), P.SymTensor(Vs, V), [2], [0]).data
    return {"values": values, "kept": kept, "product": M}


# ---------------------------------------------------------------------- work --
def _fused(legs, idx, sign):
    """{charge: dimension} of legs ``idx`` fused (U(1))."""
    out = {0: 1}
    for l in idx:
        q, d, s = legs[l]
        nxt = {}
        for x, n in out.items():
            for a, m in zip(q, d):
                y = x + sign * s * a
                nxt[y] = nxt.get(y, 0) + n * m
        out = nxt
    return out


def _spin_fused(legs, idx):
    """{spin: number of degenerate copies} of legs ``idx`` fused (SU(2))."""
    out = {0: 1}
    for l in idx:
        q, d, _ = legs[l]
        nxt = {}
        for x, n in out.items():
            for a, m in zip(q, d):
                for y in range(abs(x - a), x + a + 1, 2):
                    nxt[y] = nxt.get(y, 0) + n * m
        out = nxt
    return out


def _parity_fused(legs, idx):
    e, o = 1, 0
    for l in idx:
        a, b = legs[l][1]
        e, o = e * a + o * b, e * b + o * a
    return {0: e, 1: o}


def _pair_fused(legs, idx, sign):
    out = {(0, 0): 1}
    for l in idx:
        q, d, s = legs[l]
        nxt = {}
        for (x, j), n in out.items():
            for (a, i), m in zip(q, d):
                for y in range(abs(j - i), j + i + 1, 2):
                    z = (x + sign * s * a, y)
                    nxt[z] = nxt.get(z, 0) + n * m
        out = nxt
    return out


def _mnk(group, A, B, pa, pb):
    """Multiply-adds of one contraction, and the legs of its result."""
    fa = [l for l in range(len(A)) if l not in pa]
    fb = [l for l in range(len(B)) if l not in pb]
    if group == "u1":
        m, k, n = _fused(A, fa, -1), _fused(A, pa, 1), _fused(B, fb, 1)
    elif group == "z2f":
        m, k, n = _parity_fused(A, fa), _parity_fused(A, pa), _parity_fused(B, fb)
    elif group == "su2":
        m, k, n = _spin_fused(A, fa), _spin_fused(A, pa), _spin_fused(B, fb)
    else:
        m, k, n = _pair_fused(A, fa, -1), _pair_fused(A, pa, 1), _pair_fused(B, fb, 1)
    return sum(m[x] * k[x] * n[x] for x in k if x in m and x in n), [A[l] for l in fa] + [B[l] for l in fb]


@functools.lru_cache(maxsize=None)
def _work(key):
    c, s = json.loads(key), _spec(key)
    k, es = c["kind"], 8 if _dtype(c) == torch.float64 else 4
    ne = sum(_numel(key).values())
    if k in ("pair", "recouple"):
        f, _ = _mnk("u1" if k == "pair" else "su2", s["A"], s["B"], *s["pairs"])
        return {"bytes": es * (2 * ne + 2 * _result_numel(key)), "flops": 6.0 * f}
    if k == "mps":
        f1, t = _mnk(c["group"], s["L"], s["A"], [2], [0])
        f2, t = _mnk(c["group"], t, s["W"], *map(list, s["steps"][0]))
        f3, _ = _mnk(c["group"], t, s["R"], *map(list, s["steps"][1]))
        two = 2 if c["grad"] else 1
        return {"bytes": es * two * (ne + _result_numel(key)), "flops": (6.0 if c["grad"] else 2.0) * (f1 + f2 + f3)}
    if k in ("su2_move", "u1_move"):
        return {"bytes": es * 6 * ne, "flops": 0.0}
    if k == "batch":
        f = 0
        for p in s["problems"]:
            t = p["L"]
            for _, bn, pa, pb in s["steps"]:
                g, t = _mnk("u1", t, p[bn], pa, pb)
                f += g
        return {"bytes": es * 2 * (ne + _result_numel(key)), "flops": 6.0 * f}
    if k == "mera":
        t, w, u, h = s["t"], s["w"], s["u"], s["h"]
        f1, r = _mnk("u1", t, _reversed(t), [], [])
        f2, a = _mnk("u1", w, _reversed(w), [1, 2], [1, 2])
        f3, b = _mnk("u1", w, _reversed(w), [2, 3], [2, 3])
        f4, r = _mnk("u1", r, a, [0, 2], [0, 2])
        f5, r = _mnk("u1", r, b, [0, 1], [0, 2])
        f6, r = _mnk("u1", u, r, [2, 3], [0, 2])
        f7, r = _mnk("u1", r, _reversed(u), [2, 3], [2, 3])
        f8, _ = _mnk("u1", r, _reversed(h), [0, 1, 2, 3], [0, 1, 2, 3])
        return {"bytes": es * (2 * ne + 2 * _handles(key)["h"].numel()),
                "flops": 2.0 * f1 + 4.0 * f4 + 6.0 * (f2 + f3 + f5 + f6 + f7) + 8.0 * f8}
    plan = _handles(key)["plan"]
    f = 0.0
    for m, n, r in zip(plan.m, plan.n, _handles(key)["keep"]):
        a, b = max(m, n), min(m, n)
        # values and both sets of vectors (Golub and Van Loan's counts), then the product
        f += (9.0 * b ** 3 if k == "eig" else min(14.0 * a * b * b + 8.0 * b ** 3, 6.0 * a * b * b + 20.0 * b ** 3))
        f += 2.0 * m * n * r
    return {"bytes": es * (2 * ne + plan.nsv + sum(_handles(key)["keep"])), "flops": f}


def work(case):
    return dict(_work(_key(case)))


# --------------------------------------------- 64-bit values, in plain torch --
@functools.lru_cache(maxsize=None)
def _cg(ja, jb, jc):
    """Clebsch-Gordan coefficients [ma, mb, mc] of doubled spins, m ascending (Racah's sum)."""
    f = math.factorial
    out = np.zeros((ja + 1, jb + 1, jc + 1))
    pre = math.sqrt((jc + 1) * f((ja + jb - jc) // 2) * f((ja - jb + jc) // 2) * f((-ja + jb + jc) // 2)
                    / f((ja + jb + jc) // 2 + 1))
    for a, b in itertools.product(range(ja + 1), range(jb + 1)):
        ma, mb = 2 * a - ja, 2 * b - jb
        mc = ma + mb
        if abs(mc) > jc:
            continue
        r = math.sqrt(f((ja + ma) // 2) * f((ja - ma) // 2) * f((jb + mb) // 2) * f((jb - mb) // 2)
                      * f((jc + mc) // 2) * f((jc - mc) // 2))
        t = 0.0
        for i in range((ja + jb - jc) // 2 + 1):
            d = [i, (ja + jb - jc) // 2 - i, (ja - ma) // 2 - i, (jb + mb) // 2 - i, (jc - jb + ma) // 2 + i,
                 (jc - ja - mb) // 2 + i]
            if min(d) >= 0:
                t += (-1) ** i / math.prod(f(v) for v in d)
        out[a, b, (mc + jc) // 2] = pre * r * t
    return out


def _triangle(a, b, c):
    return abs(a - b) <= c <= a + b and (a + b + c) % 2 == 0


def _spin(group, label):
    return label if group == "su2" else label[1]


def _combs(spins):
    """Node spins (below the root) of the left comb over ``spins`` coupled to zero, lexicographic."""
    if len(spins) < 2:
        return [()] if not spins or spins[0] == 0 else []
    out = []

    def rec(top, i, lab):
        if i == len(spins) - 1:
            if top == spins[i]:
                out.append(lab)
            return
        for y in range(abs(top - spins[i]), top + spins[i] + 1, 2):
            rec(y, i + 1, lab + (y,))

    rec(spins[0], 1, ())
    return out


def _layout(group, legs, total=0):
    """Blocks of a tensor: (label positions, comb node spins, offset, shape), and their total size."""
    out, off = [], 0
    for pos in itertools.product(*[range(len(l[0])) for l in legs]):
        labs = [l[0][p] for l, p in zip(legs, pos)]
        if group in ("u1", "su2u1"):
            if sum(l[2] * (x if group == "u1" else x[0]) for l, x in zip(legs, labs)) != total:
                continue
        elif group == "z2f" and sum(labs) % 2 != total:
            continue
        inner = _combs([_spin(group, x) for x in labs]) if group in ("su2", "su2u1") else [()]
        shape = tuple(l[1][p] for l, p in zip(legs, pos))
        for i in inner:
            out.append((pos, i, off, shape))
            off += math.prod(shape)
    return out, off


@functools.lru_cache(maxsize=None)
def _structural(spins, dirs, inner):
    """Components of one comb labelling over all m, with the cup (-1)^(j-m) on incoming legs."""
    if len(spins) == 1:
        q = np.ones((1,))
    else:
        tops = (spins[0],) + tuple(inner) + (0,)
        q = np.eye(spins[0] + 1)
        for i in range(1, len(spins)):
            q = np.tensordot(q, _cg(tops[i - 1], spins[i], tops[i]), axes=([q.ndim - 1], [0]))
        q = q[..., 0]
    for i, (j, s) in enumerate(zip(spins, dirs)):
        if s == -1:
            cup = np.zeros((j + 1, j + 1))
            for m in range(j + 1):
                cup[m, j - m] = (-1) ** (j - m)
            q = np.moveaxis(np.tensordot(cup, q, axes=([1], [i])), 0, i)
    return q


def _offsets(group, leg):
    w = [(1 if group in ("u1", "z2f") else _spin(group, x) + 1) * d for x, d in zip(leg[0], leg[1])]
    return np.concatenate([[0], np.cumsum(w)]).astype(int)


def _dense(group, legs, data):
    """The tensor of block data ``data`` with every symmetry written out."""
    lay, _ = _layout(group, legs)
    offs = [_offsets(group, l) for l in legs]
    out = torch.zeros([int(o[-1]) for o in offs], dtype=torch.float64, device=data.device)
    for pos, inner, o, sh in lay:
        blk = data[o:o + math.prod(sh)].double().reshape(sh)
        sl = tuple(slice(int(f[p]), int(f[p + 1])) for f, p in zip(offs, pos))
        out[sl] += blk if group in ("u1", "z2f") else _spread(group, legs, pos, inner, blk)
    return out


def _q_of(group, legs, pos, inner, device):
    q = _structural(tuple(_spin(group, l[0][p]) for l, p in zip(legs, pos)), tuple(l[2] for l in legs), inner)
    return torch.as_tensor(np.ascontiguousarray(q), device=device)


def _spread(group, legs, pos, inner, blk):
    q = _q_of(group, legs, pos, inner, blk.device)
    k = blk.dim()
    a = blk.reshape([v for d in blk.shape for v in (d, 1)])
    b = q.reshape([v for d in q.shape for v in (1, d)])
    return (a * b).reshape([blk.shape[i] * q.shape[i] for i in range(k)])


def _blocks(group, legs, dense):
    """Block data of a dense symmetric tensor (or of a cotangent: the adjoint of _dense)."""
    lay, n = _layout(group, legs)
    offs = [_offsets(group, l) for l in legs]
    out = torch.zeros(n, dtype=torch.float64, device=dense.device)
    for pos, inner, o, sh in lay:
        sub = dense[tuple(slice(int(f[p]), int(f[p + 1])) for f, p in zip(offs, pos))]
        if group in ("su2", "su2u1"):
            q = _q_of(group, legs, pos, inner, dense.device)
            sub = sub.reshape([v for d, m in zip(sh, q.shape) for v in (d, m)])
            b = q.reshape([v for d in q.shape for v in (1, d)])
            sub = (sub * b).sum(dim=tuple(range(1, 2 * len(sh), 2)))
        out[o:o + math.prod(sh)] = sub.reshape(-1)
    return out


def _ordered(group, x, legs, perm):
    """x with its legs in the order ``perm``; fermionic legs gain -1 for every exchanged pair of odd ones."""
    if group == "z2f":
        par = []
        for i, l in enumerate(legs):
            p = torch.cat([torch.full((d,), float(q)) for q, d in zip(l[0], l[1])]).to(x)
            par.append(p.reshape([-1 if j == i else 1 for j in range(len(legs))]))
        for a in range(len(perm)):
            for b in range(a + 1, len(perm)):
                if perm[a] > perm[b]:
                    x = x * (1.0 - 2.0 * par[perm[a]] * par[perm[b]])
    return x.permute(list(perm))


def _join(group, x, A, y, B, pa, pb):
    fa = [l for l in range(len(A)) if l not in pa]
    fb = [l for l in range(len(B)) if l not in pb]
    n = len(pa)
    x = _ordered(group, x, A, fa + list(pa))
    y = _ordered(group, y, B, list(pb) + fb)
    return torch.tensordot(x, y, dims=(list(range(len(fa), len(A))), list(range(n)))), \
        [A[l] for l in fa] + [B[l] for l in fb]


def _chain(group, tensors, legs, steps):
    x, l = tensors[0], legs[0]
    for (t, b), (pa, pb) in zip(zip(tensors[1:], legs[1:]), steps):
        x, l = _join(group, x, l, t, b, list(pa), list(pb))
    return x, l


def _chain_exact(group, data, legs, steps, G, names):
    """Result and gradients of a chain of contractions, through dense tensors."""
    leaf = {}
    for n in names:
        if n not in leaf:
            leaf[n] = _dense(group, legs[n], data[n].detach()).requires_grad_(G is not None)
    Y, l = _chain(group, [leaf[n] for n in names], [legs[n] for n in names], steps)
    out = [_blocks(group, l, Y.detach())]
    if G is not None:
        uniq = list(dict.fromkeys(names))
        g = torch.autograd.grad(Y, [leaf[n] for n in uniq], grad_outputs=_dense(group, l, G))
        out += [_blocks(group, legs[n], v) for n, v in zip(uniq, g)]
    return out


@functools.lru_cache(maxsize=None)
def _overlap(spins, perm, pairs):
    """R[out, in]: comb labellings of ``spins`` against those of the permuted legs (a comb, or two
    pairs joined at the root), as overlaps of their components (all legs outgoing)."""
    ps = [spins[p] for p in perm]
    up = (1,) * 4
    ket = np.stack([_structural(spins, up, e) for e in _combs(list(spins))])
    if pairs:
        outs = [x for x in range(max(abs(ps[0] - ps[1]), abs(ps[2] - ps[3])), min(ps[0] + ps[1], ps[2] + ps[3]) + 1)
                if _triangle(ps[0], ps[1], x) and _triangle(ps[2], ps[3], x)]
        bra = [np.tensordot(_cg(ps[0], ps[1], x) @ _cg(x, x, 0)[..., 0], _cg(ps[2], ps[3], x), axes=([2], [2]))
               for x in outs]
    else:
        outs = _combs(ps)
        bra = [_structural(tuple(ps), up, e) for e in outs]
    ket = ket.transpose([0] + [1 + p for p in perm])
    R = np.stack(bra).reshape(len(outs), -1) @ ket.reshape(len(ket), -1).T
    return outs, R


def _groups4(legs):
    """Blocks of a rank-4 SU(2) tensor by label positions: {positions: (offset, comb labellings, shape)}."""
    out = {}
    for pos, inner, o, sh in _layout("su2", legs)[0]:
        out.setdefault(pos, [o, [], sh])[1].append(inner)
    return out


def _matrix_places(legs, perm):
    """{x: (rows, cols, {positions of legs perm[:2]: first row}, {positions of legs perm[2:]: first column})}."""
    def side(ls):
        at = {}
        for i, j in itertools.product(range(len(legs[ls[0]][0])), range(len(legs[ls[1]][0]))):
            a, b = legs[ls[0]][0][i], legs[ls[1]][0][j]
            for x in range(abs(a - b), a + b + 1, 2):
                d = at.setdefault(x, [0, {}])
                d[1][(i, j)] = d[0]
                d[0] += legs[ls[0]][1][i] * legs[ls[1]][1][j]
        return at

    r, c = side(perm[:2]), side(perm[2:])
    return {x: (r[x][0], c[x][0], r[x][1], c[x][1]) for x in r if x in c}


def _to_matrix(legs, perm, data, back=None):
    """Matrices M_x (two pairs of legs) of comb block data; with ``back``, the adjoint: block data from matrices."""
    places = _matrix_places(legs, perm)
    if back is None:
        M = {x: torch.zeros(p[0], p[1], dtype=torch.float64, device=data.device) for x, p in places.items()}
    else:
        M, out = back, torch.zeros(_layout("su2", legs)[1], dtype=torch.float64, device=data.device)
    for pos, (o, inner, sh) in _groups4(legs).items():
        spins = tuple(l[0][p] for l, p in zip(legs, pos))
        xs, R = _overlap(spins, tuple(perm), True)
        Rt = torch.as_tensor(R, device=data.device)
        n = math.prod(sh)
        psh = [sh[p] for p in perm]
        rc = (psh[0] * psh[1], psh[2] * psh[3])
        at = [(places[x][2][(pos[perm[0]], pos[perm[1]])], places[x][3][(pos[perm[2]], pos[perm[3]])]) for x in xs]
        if back is None:
            v = (Rt @ data[o:o + n * len(inner)].double().reshape(len(inner), n)).reshape([len(xs)] + list(sh))
            v = v.permute([0] + [1 + p for p in perm]).reshape([len(xs)] + list(rc))
            for i, x in enumerate(xs):
                M[x][at[i][0]:at[i][0] + rc[0], at[i][1]:at[i][1] + rc[1]] = v[i]
        else:
            v = torch.stack([M[x][a:a + rc[0], b:b + rc[1]] for x, (a, b) in zip(xs, at)]).reshape([len(xs)] + psh)
            inv = [perm.index(p) for p in range(4)]
            v = v.permute([0] + [1 + p for p in inv]).reshape(len(xs), n)
            out[o:o + n * len(inner)] = (Rt.T @ v).reshape(-1)
    return M if back is None else out


def _from_pairs(legs, M, data=None):
    """Block data of a tensor whose tree is two pairs joined at the root, from its matrices (or, with data, back)."""
    places = _matrix_places(legs, [0, 1, 2, 3])
    blocks, off = [], 0
    for pos in itertools.product(*[range(len(l[0])) for l in legs]):
        sp = [l[0][p] for l, p in zip(legs, pos)]
        sh = [l[1][p] for l, p in zip(legs, pos)]
        for x in range(abs(sp[0] - sp[1]), sp[0] + sp[1] + 1, 2):
            if _triangle(sp[2], sp[3], x):
                blocks.append((x, pos, off, sh))
                off += math.prod(sh)
    if data is None:
        out = torch.zeros(off, dtype=torch.float64, device="cuda")
    else:
        out = {x: torch.zeros(p[0], p[1], dtype=torch.float64, device=data.device) for x, p in places.items()}
    for x, pos, o, sh in blocks:
        r, c = places[x][2][pos[:2]], places[x][3][pos[2:]]
        m, n = sh[0] * sh[1], sh[2] * sh[3]
        if data is None:
            if x in M:
                out[o:o + m * n] = M[x][r:r + m, c:c + n].reshape(-1)
        else:
            out[x][r:r + m, c:c + n] = data[o:o + m * n].double().reshape(m, n)
    return out


def _recouple_exact(case, x, G):
    s = _spec(_key(case))
    A, B = s["A"], s["B"]
    pa, pb = [0, 2, 1, 3], [0, 1, 2, 3]
    MA, MB = _to_matrix(A, pa, x["A"].detach()), _to_matrix(B, pb, x["B"].detach())
    legs = [A[0], A[2], B[2], B[3]]
    # contracting a pair of trees over the same coupled spin x leaves (-1)^(2x) / sqrt(2x + 1)
    fac = {q: (-1.0) ** q / math.sqrt(q + 1.0) for q in MA if q in MB}
    C = _from_pairs(legs, {q: f * (MA[q] @ MB[q]) for q, f in fac.items()})
    dC = _from_pairs(legs, None, G)
    zero = lambda M: torch.zeros_like(M)  # noqa: E731
    dMA = {q: fac[q] * (dC[q] @ MB[q].T) if q in fac and q in dC else zero(MA[q]) for q in MA}
    dMB = {q: fac[q] * (MA[q].T @ dC[q]) if q in fac and q in dC else zero(MB[q]) for q in MB}
    return {"C": C, "dA": _to_matrix(A, pa, x["A"].detach(), dMA), "dB": _to_matrix(B, pb, x["B"].detach(), dMB)}


def _pair_rows(group, a, b):
    """{fused label: (size, {(ia, ib): first row})} of two outgoing legs fused."""
    at = {}
    for i, j in itertools.product(range(len(a[0])), range(len(b[0]))):
        p, q = a[0][i], b[0][j]
        for x in ([p + q] if group == "u1" else range(abs(p - q), p + q + 1, 2)):
            d = at.setdefault(x, [0, {}])
            d[1][(i, j)] = d[0]
            d[0] += a[1][i] * b[1][j]
    return at


def _move_exact(group, legs, perm, data):
    plegs = [legs[p] for p in perm]
    lay, n = _layout(group, plegs)
    out = torch.zeros(n, dtype=torch.float64, device=data.device)
    if group == "u1":
        src = {pos: (o, sh) for pos, _, o, sh in _layout(group, legs)[0]}
        for pos, _, o, sh in lay:
            ipos = [0] * 4
            for i, p in enumerate(perm):
                ipos[p] = pos[i]
            so, ssh = src[tuple(ipos)]
            out[o:o + math.prod(sh)] = data[so:so + math.prod(sh)].double().reshape(ssh).permute(perm).reshape(-1)
    else:
        dst = _groups4(plegs)
        for pos, (o, inner, sh) in _groups4(legs).items():
            labs, R = _overlap(tuple(l[0][p] for l, p in zip(legs, pos)), tuple(perm), False)
            n1 = math.prod(sh)
            v = torch.as_tensor(R, device=data.device) @ data[o:o + n1 * len(inner)].double().reshape(len(inner), n1)
            v = v.reshape([len(labs)] + list(sh)).permute([0] + [1 + p for p in perm])
            do, dlabs, _ = dst[tuple(pos[p] for p in perm)]
            for i, lab in enumerate(labs):
                at = do + dlabs.index(lab) * n1
                out[at:at + n1] = v[i].reshape(-1)
    rows = _pair_rows(group, plegs[0], plegs[1])
    xs = sorted(rows)
    fl = [(xs, [rows[x][0] for x in xs], plegs[0][2])] + plegs[2:]
    flay, fn = _layout(group, fl)
    fsrc = {(pos, inner): (o, sh) for pos, inner, o, sh in flay}
    fused = torch.zeros(fn, dtype=torch.float64, device=data.device)
    for pos, inner, o, sh in lay:
        x = inner[0] if inner else sum(plegs[i][0][pos[i]] for i in (0, 1))
        fo, fsh = fsrc[((xs.index(x),) + pos[2:], inner[1:] if inner else ())]
        r = rows[x][1][pos[:2]]
        m = sh[0] * sh[1]
        fused[fo:fo + math.prod(fsh)].view(fsh)[r:r + m] = out[o:o + math.prod(sh)].reshape((m,) + tuple(sh[2:]))
    return {"permuted": out, "fused": fused, "split": out}


def _factor_exact(case, T):
    """Values per block (label ascending, largest first), the kept ones and the product of the kept factors."""
    key = _key(case)
    theta = _spec(key)["theta"]
    legs = theta if case["kind"] == "svd" else theta[:2] + _reversed(theta[:2])
    lay, n = _layout("u1", legs)
    rows, cols, blocks = {}, {}, {}
    for idx, at, sign in (((0, 1), rows, 1), ((2, 3), cols, -1)):
        for i, j in itertools.product(*[range(len(legs[l][0])) for l in idx]):
            x = sign * (legs[idx[0]][2] * legs[idx[0]][0][i] + legs[idx[1]][2] * legs[idx[1]][0][j])
            d = at.setdefault(x, [0, {}])
            d[1][(i, j)] = d[0]
            d[0] += legs[idx[0]][1][i] * legs[idx[1]][1][j]
    xs = sorted(x for x in rows if x in cols)
    M = {x: torch.zeros(rows[x][0], cols[x][0], dtype=torch.float64) for x in xs}
    host = T.cpu()
    for pos, _, o, sh in lay:
        x = legs[0][2] * legs[0][0][pos[0]] + legs[1][2] * legs[1][0][pos[1]]
        r, c = rows[x][1][pos[:2]], cols[x][1][pos[2:]]
        m, k = sh[0] * sh[1], sh[2] * sh[3]
        blocks[pos] = (x, r, c, m, k, o)
        M[x][r:r + m, c:c + k] = host[o:o + m * k].reshape(m, k)
    full = [min(M[x].shape) for x in xs]
    keep = _kept(key, xs, full)
    values, kept, prod = [], [], {}
    for x, k in zip(xs, keep):
        if case["kind"] == "svd":
            u, s, v = torch.linalg.svd(M[x], full_matrices=False)
        else:
            s, u = torch.linalg.eigh(M[x])
            o = torch.argsort(s.abs(), descending=True, stable=True)
            s, u = s[o], u[:, o]
            v = u.T
        values.append(s)
        kept.append(s[:k])
        prod[x] = (u[:, :k] * s[:k]) @ v[:k]
    out = torch.zeros(n, dtype=torch.float64)
    for x, r, c, m, k, o in blocks.values():
        out[o:o + m * k] = prod[x][r:r + m, c:c + k].reshape(-1)
    return {"values": torch.cat(values), "kept": torch.cat(kept), "product": out}


def _mera_exact(case, x):
    key = _key(case)
    s, H = _spec(key), _handles(key)
    d = {n: _dense("u1", s[n], x[n].detach()).requires_grad_(n != "t") for n in "twu"}
    h = _dense("u1", _reversed(s["h"]), H["h"])
    one = _dense("u1", _reversed(s["h"]), H["one"])
    top = torch.einsum("st,uv->stuv", d["t"], d["t"])
    w1 = torch.einsum("sxya,txyb->satb", d["w"], d["w"])
    w2 = torch.einsum("saxy,tbxy->satb", d["w"], d["w"])
    rho = torch.einsum("stuv,saub,tcvd->abcd", top, w1, w2)  # (a3, a3', b1, b1')
    y = torch.einsum("cdpq,prqt->cdrt", d["u"], rho)
    rp = torch.einsum("cdrt,efrt->cdef", y, d["u"])
    E = (rp * h).sum() / (rp * one).sum()
    gw, gu = torch.autograd.grad(E, [d["w"], d["u"]])
    return {"E": E.detach(), "dw": _blocks("u1", s["w"], gw), "du": _blocks("u1", s["u"], gu)}


def exact(case, seed):
    k, key = case["kind"], _key(case)
    s = _spec(key)
    if k == "recouple" and case["dmax"] > 20:
        return None  # over 20 seconds in 64 bits
    if k == "mps" and case["D"] > {"u1": 3000, "z2f": 2600, "su2u1": 1200}[case["group"]]:
        return None
    st = prepare(case, seed)
    x, G = st["x"], st.get("G")
    if k == "pair":
        r = _chain_exact("u1", x, s, [s["pairs"]], G, ["A", "B"])
        return dict(zip(("C", "dA", "dB"), r))
    if k == "recouple":
        return _recouple_exact(case, x, G)
    if k == "mps":
        r = _chain_exact(case["group"], x, s, [([2], [0])] + list(s["steps"]), G, list("LAWR"))
        return dict(zip(("Y", "dL", "dA", "dW", "dR"), r))
    if k == "su2_move":
        return _move_exact("su2", s["T"], s["perm"], x["T"])
    if k == "u1_move":
        return _move_exact("u1", s["T"], s["perm"], x["T"])
    if k == "batch":
        names = ["L", "theta", "W", "W", "R"]
        steps = [(pa, pb) for _, _, pa, pb in s["steps"]]
        H = _handles(key)
        off = {"L": H["plans"][0].off_a, "theta": H["plans"][0].off_b, "W": H["plans"][1].off_b,
               "R": H["plans"][3].off_b}
        oc, parts = H["plans"][3].off_c, []
        for i, p in enumerate(s["problems"]):
            data = {n: x[n].detach()[off[n][i]:off[n][i + 1]] for n in off}
            parts.append(_chain_exact("u1", data, p, steps, G[oc[i]:oc[i + 1]], names))
        return dict(zip(("Y", "dL", "dtheta", "dW", "dR"), [torch.cat([p[j] for p in parts]) for j in range(5)]))
    if k == "mera":
        return _mera_exact(case, x)
    return _factor_exact(case, x["T"])
