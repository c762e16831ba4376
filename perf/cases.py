"""The work users of this library have it do, as timed cases.

A case is one call (or one batch call) through the package's public entry
points on device data: sign(T) by every variant in earnest use, over small,
ordinary and large orders, the batched call, the Schur routes, complex T and
a general function of T.  Inputs follow paper_1607_06303_gb300/inputs.py's
recipe, drawn on the device: |t_ii| ~ U[0.5, 2] with a given share of
negative signs, strictly upper t_ij ~ N(0, 1/n).
"""
import math

import torch

import paper_1607_06303_gb300 as p

DEV = "cuda:0"

# fields each kind of case carries, beside its name
#   tri      n, neg (share of negative eigenvalues), order, variant
#   batch    count, n_min, n_max
#   pair     n, neg, variant      (S = Q sign(T) Q^T from a real Schur pair)
#   complex  n, neg               (complex triangular T)
#   funm     n, phi               (phi(T) on separated eigenvalues)
#   general  n                    (sign(A), Schur decomposition included)


def listed():
    return [
        # the smallest solve of everyday use (a control step, one system): latency
        {"name": "tri_256", "kind": "tri", "n": 256, "neg": 0.5, "order": "random", "variant": "AUTO"},
        # an ordinary float64 solve of odd order, unbalanced inertia
        {"name": "tri_1001", "kind": "tri", "n": 1001, "neg": 0.3, "order": "random", "variant": "AUTO"},
        # a large float64 solve (the recursive Parlett-Higham workload)
        {"name": "tri_8192", "kind": "tri", "n": 8192, "neg": 0.25, "order": "random", "variant": "AUTO"},
        # eigenvalues already grouped by sign, as an ordered Schur form gives them
        {"name": "sorted_8192", "kind": "tri", "n": 8192, "neg": 0.25, "order": "sorted", "variant": "AUTO"},
        # Parlett-Sylvester with its reordering, odd order
        {"name": "reorder_3001", "kind": "tri", "n": 3001, "neg": 0.1, "order": "random", "variant": "PS_FP64"},
        # the headline: mixed precision with refinement at full size
        {"name": "mixed_16384", "kind": "tri", "n": 16384, "neg": 0.5, "order": "random", "variant": "PH_MIXED_FP16"},
        # the same at an ordinary ragged order
        {"name": "mixed_3001", "kind": "tri", "n": 3001, "neg": 0.4, "order": "random", "variant": "PH_MIXED_FP16"},
        # many independent problems in one call
        {"name": "batch_300", "kind": "batch", "count": 300, "n_min": 32, "n_max": 2048},
        # sign(A) from a caller's real Schur pair
        {"name": "pair_2000", "kind": "pair", "n": 2000, "neg": 0.5, "variant": "AUTO"},
        # a complex Schur form
        {"name": "complex_1000", "kind": "complex", "n": 1000, "neg": 0.5},
        # another function of T on the same partition
        {"name": "funm_1500", "kind": "funm", "n": 1500, "phi": "EXP"},
        # sign(A) of a general matrix, decomposition and all
        {"name": "general_200", "kind": "general", "n": 200},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tri", "tri", "mixed", "batch", "pair", "complex", "funm", "general"])
    neg = round(rng.uniform(0.05, 0.95), 3)
    if kind == "tri":
        variant = rng.choice(["AUTO", "PH_FP64", "PH_FP64_EFFICIENT", "PS_FP64"])
        n = _log_int(rng, 33, {"AUTO": 8192, "PH_FP64": 5000, "PH_FP64_EFFICIENT": 8000, "PS_FP64": 6000}[variant])
        return {"kind": "tri", "n": n, "neg": neg, "order": rng.choice(["random", "random", "sorted"]),
                "variant": variant}
    if kind == "mixed":
        variant = rng.choice(["PH_MIXED_FP16", "PH_MIXED_FP16", "PH_MIXED_TF32", "PH_MIXED_BF16"])
        n = _log_int(rng, 400, {"PH_MIXED_FP16": 16384, "PH_MIXED_TF32": 12000, "PH_MIXED_BF16": 6000}[variant])
        return {"kind": "tri", "n": n, "neg": neg, "order": "random", "variant": variant}
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 20, 300), "n_min": 32, "n_max": _log_int(rng, 64, 2048)}
    if kind == "pair":
        return {"kind": "pair", "n": _log_int(rng, 100, 4000), "neg": neg,
                "variant": rng.choice(["AUTO", "PH_MIXED_FP16"])}
    if kind == "complex":
        return {"kind": "complex", "n": _log_int(rng, 50, 2000), "neg": neg}
    if kind == "funm":
        return {"kind": "funm", "n": _log_int(rng, 50, 4000), "phi": rng.choice(["EXP", "SQRT"])}
    return {"kind": "general", "n": _log_int(rng, 32, 256)}


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _signs(n, neg, order, g):
    s = torch.ones(n, dtype=torch.float64, device=DEV)
    k = int(math.floor(neg * n + 0.5))
    if order == "sorted":
        s[n - k:] = -1.0
    else:
        s[torch.randperm(n, generator=g, device=DEV)[:k]] = -1.0
    return s


def _normal(shape, g):
    # full float64 mantissas; two float32 draws, because drawing n^2 float64
    # normals takes longer than the solves
    x = torch.randn(shape, generator=g, device=DEV).double()
    x.add_(torch.randn(shape, generator=g, device=DEV), alpha=2.0 ** -24)
    return x


def _triangular(n, neg, order, g):
    """T in the package's layout: row j of the tensor is column j of T."""
    t = _normal((n, n), g).mul_(1.0 / math.sqrt(n)).tril_(-1)
    mags = 0.5 + 1.5 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    t.diagonal().copy_(_signs(n, neg, order, g) * mags)
    return t


def _batch_shape(case):
    # sizes log-uniform, shares of negatives uniform, the same for every seed
    # of a case (its work is then a fixed amount)
    g = torch.Generator().manual_seed(12345 + case["count"])
    u = torch.rand(2, case["count"], generator=g, dtype=torch.float64)
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    return [int(round(math.exp(lo + (hi - lo) * float(x)))) for x in u[0]], [float(x) for x in u[1]]


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "tri":
        t = _triangular(case["n"], case["neg"], case["order"], g)
        return {"kind": kind, "T": t, "U": torch.empty_like(t), "variant": p.Variant[case["variant"]]}
    if kind == "batch":
        ns, negs = _batch_shape(case)
        total = sum(n * n for n in ns)
        T = torch.empty(total, dtype=torch.float64, device=DEV)
        U = torch.empty(total, dtype=torch.float64, device=DEV)
        Tp, Up, at = [], [], 0
        for n, neg in zip(ns, negs):
            T[at:at + n * n].view(n, n).copy_(_triangular(n, neg, "random", g))
            Tp.append(T.data_ptr() + 8 * at)
            Up.append(U.data_ptr() + 8 * at)
            at += n * n
        return {"kind": kind, "T": T, "U": U, "n": ns, "Tp": Tp, "Up": Up}
    if kind == "pair":
        t = _triangular(case["n"], case["neg"], "random", g)
        q, r = torch.linalg.qr(_normal((case["n"], case["n"]), g))
        q = (q * torch.sign(r.diagonal())).contiguous()
        return {"kind": kind, "T": t, "Q": q, "U": torch.empty_like(t), "variant": p.Variant[case["variant"]]}
    if kind == "complex":
        n = case["n"]
        z = torch.complex(_normal((n, n), g), _normal((n, n), g)).mul_(1.0 / math.sqrt(2.0 * n)).tril_(-1)
        mags = 0.5 + 1.5 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
        z.diagonal().copy_(torch.complex(_signs(n, case["neg"], "random", g) * mags, _normal((n,), g)))
        return {"kind": kind, "T": z, "U": torch.empty_like(z)}
    if kind == "funm":
        n = case["n"]
        t = _normal((n, n), g).mul_(1.0 / math.sqrt(n)).tril_(-1)
        # separated eigenvalues 1 .. 1 + n / 50, as Parlett's substitution wants;
        # scaled down for exp, which would overflow
        d = torch.linspace(1.0, 1.0 + 0.02 * n, n, dtype=torch.float64, device=DEV)
        t.diagonal().copy_(d[torch.randperm(n, generator=g, device=DEV)])
        if case["phi"] == "EXP":
            t.mul_(4.0 / (1.0 + 0.02 * n))
        return {"kind": kind, "T": t, "U": torch.empty_like(t), "phi": p.Phi[case["phi"]]}
    a = 100.0 * torch.rand(case["n"], case["n"], generator=g, device=DEV, dtype=torch.float64) - 50.0
    return {"kind": kind, "T": a, "U": torch.empty_like(a)}


def run(s):
    kind = s["kind"]
    if kind == "tri":
        return p.sign(s["T"], s["variant"], out=s["U"])
    if kind == "batch":
        stream = torch.cuda.current_stream().cuda_stream
        status, info = p.sign_tri_batched(s["n"], s["Tp"], s["n"], s["Up"], s["n"], p.Variant.AUTO, stream)
        if status != 0:
            raise p.SignTriError(status, "sign_tri_batched")
        return {"U": s["U"], "info": torch.tensor(info)}
    if kind == "pair":
        return p.sign_schur(s["Q"], s["T"], s["variant"], out=s["U"])
    if kind == "complex":
        return p.sign_complex(s["T"], out=s["U"])
    if kind == "funm":
        return p.funm(s["T"], s["phi"], out=s["U"])
    return p.sign_general(s["T"], out=s["U"])


def _terms(n):
    return math.comb(n, 3) if n >= 3 else 0


def _sign_flops(n, neg):
    # the substitution's own sums: 2 flops a term where the signs agree, 4 where they differ
    same = neg * neg + (1.0 - neg) * (1.0 - neg)
    return _terms(n) * (2.0 * same + 4.0 * (1.0 - same))


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    read_upper_write_all = 8.0 * (n * (n + 1) / 2 + n * n)
    if kind == "tri":
        return {"bytes": read_upper_write_all, "flops": _sign_flops(n, case["neg"])}
    if kind == "batch":
        ns, negs = _batch_shape(case)
        return {"bytes": sum(8.0 * (m * (m + 1) / 2 + m * m) for m in ns),
                "flops": sum(_sign_flops(m, q) for m, q in zip(ns, negs))}
    if kind == "pair":
        return {"bytes": read_upper_write_all + 8.0 * n * n, "flops": _sign_flops(n, case["neg"]) + 3.0 * n ** 3}
    if kind == "complex":
        return {"bytes": 2 * read_upper_write_all, "flops": 4.0 * _sign_flops(n, case["neg"])}
    if kind == "funm":
        return {"bytes": read_upper_write_all, "flops": 4.0 * _terms(n)}
    # Hessenberg reduction with Q (14/3 n^3), QR sweeps in complex arithmetic
    # (about 25 n^3 complex), sign of T and the two products
    return {"bytes": 16.0 * n * n, "flops": (14.0 / 3.0 + 100.0 + 12.0) * n ** 3}


# ---- what the calls should return, in plain float64 torch ------------------

def _sign_tri64(Tt):
    """sign(T) for a stack (B, n, n) of upper triangular T given by their
    transposes, entry by entry over anti-diagonals: TU = UT where the signs
    of t_ii and t_jj differ, U^2 = I where they agree."""
    B, n, _ = Tt.shape
    Tt = Tt.contiguous()
    T = Tt.transpose(1, 2).contiguous()
    t = torch.diagonal(T, dim1=1, dim2=2)
    real = t.real if t.is_complex() else t
    s = torch.where(real > 0, 1.0, -1.0).to(T.dtype)
    U = torch.diag_embed(s).contiguous()
    Ut = U.clone()
    for d in range(1, n):
        m = n - d
        rows = lambda M: M.as_strided((B, m, d - 1), (n * n, n + 1, 1), 1)            # noqa: E731
        cols = lambda M: M.as_strided((B, m, d - 1), (n * n, n + 1, 1), d * n + 1)    # noqa: E731
        si, sj = s[:, :m], s[:, d:]
        opposite = (si + sj).abs() == 0
        x = (rows(U) * cols(Tt)).sub_(rows(T) * cols(Ut)).sum(-1) if d > 1 else 0.0
        y = (rows(U) * cols(Ut)).sum(-1) if d > 1 else torch.zeros_like(si)
        tij = torch.diagonal(T, d, 1, 2)
        gap = torch.where(opposite, t[:, :m] - t[:, d:], torch.ones_like(si))
        u = torch.where(opposite, (tij * (si - sj) + x) / gap, -y / torch.where(opposite, torch.ones_like(si), si + sj))
        torch.diagonal(U, d, 1, 2).copy_(u)
        torch.diagonal(Ut, -d, 1, 2).copy_(u)
    return Ut


def _sqrt_tri64(Tt):
    n = Tt.shape[0]
    T = Tt.t().contiguous()
    U, Ut = torch.diag(T.diagonal().sqrt()), torch.diag(T.diagonal().sqrt())
    r = T.diagonal().sqrt()
    for d in range(1, n):
        m = n - d
        rows = U.as_strided((m, d - 1), (n + 1, 1), 1)
        cols = Ut.as_strided((m, d - 1), (n + 1, 1), d * n + 1)
        u = (T.diagonal(d) - (rows * cols).sum(-1)) / (r[:m] + r[d:])
        U.diagonal(d).copy_(u)
        Ut.diagonal(-d).copy_(u)
    return Ut


def exact(case, seed):
    kind = case["kind"]
    if kind == "tri" and case["n"] > 8192:
        return None  # the plain recurrence takes too long
    s = prepare(case, seed)
    if kind in ("tri", "complex"):
        return _sign_tri64(s["T"][None])[0]
    if kind == "batch":
        order = sorted(range(len(s["n"])), key=lambda i: s["n"][i])
        start = [0]
        for n in s["n"]:
            start.append(start[-1] + n * n)
        out = torch.empty_like(s["T"])
        for k in range(0, len(order), 32):
            group = order[k:k + 32]
            top = max(s["n"][i] for i in group)
            # shorter problems get unit diagonals behind them, which touch nothing
            T = torch.eye(top, dtype=torch.float64, device=DEV).repeat(len(group), 1, 1)
            for a, i in enumerate(group):
                n = s["n"][i]
                T[a, :n, :n] = s["T"][start[i]:start[i + 1]].view(n, n)
            U = _sign_tri64(T)
            for a, i in enumerate(group):
                n = s["n"][i]
                out[start[i]:start[i + 1]].view(n, n).copy_(U[a, :n, :n])
        return {"U": out, "info": None}
    if kind == "pair":
        Ut = _sign_tri64(s["T"][None])[0]
        return s["Q"].t() @ Ut @ s["Q"]
    if kind == "funm":
        if case["phi"] == "EXP":
            return torch.linalg.matrix_exp(s["T"])
        return _sqrt_tri64(s["T"])
    # sign(A): Newton's iteration with determinant scaling, then unscaled
    X = s["T"].clone()
    for k in range(60):
        Y = torch.linalg.inv(X)
        mu = 1.0
        if k < 12:
            mu = float(torch.exp(-torch.linalg.slogdet(X)[1] / X.shape[0]))
        Z = 0.5 * (mu * X + Y / mu)
        done = k >= 12 and float((Z - X).norm()) <= 1e-15 * float(Z.norm())
        X = Z
        if done:
            break
    return X
