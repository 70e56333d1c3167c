"""Timed cases of the library: what a user's program has it do, through its public entry points.

Five kinds of case:

- "sketch":   the two products of a pair of passes, Y = A X and Z = A^H W, on operands in hand (a caller who
              drives the passes), in each arithmetic that is used in earnest;
- "orth":     the orthonormal basis of a tall thin matrix (the "QR" after a pass);
- "lowrank":  the rank-k approximation of a matrix by Algorithm 2 or Algorithm 4, written out;
- "complete": matrix completion by alternating updates;
- "batch":    Algorithm 2 over many small uneven matrices through a batch plan.

The singular vectors of a rank-k approximation are defined only up to a right unit quaternion per pair, so
"lowrank" and "complete" return the approximation itself, U diag(S) V^H, which is also what an image program
is after.  S comes as FP64 whatever the storage; beside FP32 planes it is kept in FP32, and the batch's factors
are kept in the type of the patches that they stand for.
"""
import math

import torch

from paper_2507_13731_gb300 import qlr

_COMPUTE = {"auto": qlr.COMPUTE_AUTO, "tf32": qlr.COMPUTE_TF32, "tf32_rn": qlr.COMPUTE_TF32_RN,
            "mixed": qlr.COMPUTE_TF32_MIXED}
_DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_DEV = "cuda"


def listed():
    return [
        # one patch of odd size: launches and latency
        {"name": "sketch patch 517x389", "kind": "sketch", "m": 517, "n": 389, "l": 23, "dtype": "f32",
         "compute": "auto", "pure": True},
        # the pass sweep's matrix (4096 square, k = 100, p = 10) in FP32-accurate arithmetic
        {"name": "sketch 3xtf32 4096", "kind": "sketch", "m": 4096, "n": 4096, "l": 110, "dtype": "f32",
         "compute": "auto", "pure": False},
        # the Krylov views of the large colour field (block of 60)
        {"name": "sketch tf32 20000x10000", "kind": "sketch", "m": 20000, "n": 10000, "l": 60, "dtype": "f32",
         "compute": "tf32", "pure": True},
        # the same field's final pass over the stacked basis (3 blocks of 60)
        {"name": "sketch tf32rn 20000x10000", "kind": "sketch", "m": 20000, "n": 10000, "l": 180, "dtype": "f32",
         "compute": "tf32_rn", "pure": True},
        # the mixed-precision workload: BF16 planes, k = 200, p = 20
        {"name": "sketch bf16 16384x8192", "kind": "sketch", "m": 16384, "n": 8192, "l": 220, "dtype": "bf16",
         "compute": "auto", "pure": False},
        # the QR after a view of the large field, and that of its stacked basis
        {"name": "orth 20000x60", "kind": "orth", "m": 20000, "l": 60},
        {"name": "orth 20000x180", "kind": "orth", "m": 20000, "l": 180},
        # a small image in FP64
        {"name": "lowrank f64 256x192", "kind": "lowrank", "m": 256, "n": 192, "k": 10, "p": 5, "v": 2, "algo": 2,
         "dtype": "f64", "compute": "auto", "pure": False},
        # the pass sweep, three passes, one column short of square
        {"name": "lowrank f32 4096x4095", "kind": "lowrank", "m": 4096, "n": 4095, "k": 100, "p": 10, "v": 3,
         "algo": 2, "dtype": "f32", "compute": "auto", "pure": False},
        # the large pure quaternion field: block Krylov, six views, TF32 with a rounded final pass
        {"name": "krylov 20000x10000", "kind": "lowrank", "m": 20000, "n": 10000, "k": 50, "p": 10, "v": 6,
         "algo": 4, "dtype": "f32", "compute": "tf32_rn", "pure": True},
        # completion of a 4096 square image with 70 % of its pixels missing
        {"name": "complete 4096", "kind": "complete", "m": 4096, "n": 4096, "k": 30, "p": 10, "v": 2, "iters": 3},
        # 512 patches of uneven size and rank
        {"name": "batch 512", "kind": "batch", "count": 512, "mmin": 64, "mmax": 1024, "nmin": 64, "nmax": 768,
         "rmin": 8, "rmax": 64, "p": 8, "v": 3, "sizes": 1238},
    ]


def _logint(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sketch", "sketch", "sketch", "orth", "lowrank", "lowrank", "complete", "batch"])
    if kind == "sketch":
        dtype, compute = rng.choice([("f32", "auto"), ("f32", "tf32"), ("f32", "tf32_rn"), ("bf16", "auto")])
        return {"kind": kind, "m": _logint(rng, 256, 20000), "n": _logint(rng, 192, 10000),
                "l": _logint(rng, 15, 180), "dtype": dtype, "compute": compute, "pure": rng.random() < 0.5}
    if kind == "orth":
        l = _logint(rng, 15, 220)
        return {"kind": kind, "m": _logint(rng, max(256, 2 * l), 20000), "l": l}
    if kind == "lowrank":
        if rng.random() < 0.25:
            return {"kind": kind, "m": _logint(rng, 128, 512), "n": _logint(rng, 128, 512), "k": rng.randint(5, 20),
                    "p": rng.randint(5, 10), "v": rng.randint(2, 4), "algo": 2, "dtype": "f64", "compute": "auto",
                    "pure": rng.random() < 0.5}
        algo = rng.choice([2, 2, 4])
        return {"kind": kind, "m": _logint(rng, 500, 10000), "n": _logint(rng, 500, 5000),
                "k": _logint(rng, 10, 100 if algo == 2 else 50), "p": 10, "v": rng.randint(2, 4) if algo == 2 else
                rng.randint(4, 6), "algo": algo, "dtype": "f32",
                "compute": rng.choice(["auto", "mixed"] if algo == 2 else ["mixed", "tf32_rn"]),
                "pure": rng.random() < 0.5}
    if kind == "complete":
        return {"kind": kind, "m": _logint(rng, 256, 4096), "n": _logint(rng, 256, 4096), "k": _logint(rng, 8, 30),
                "p": 10, "v": rng.choice([2, 4]), "iters": rng.randint(1, 3)}
    return {"kind": kind, "count": _logint(rng, 16, 512), "mmin": 64, "mmax": _logint(rng, 256, 1024), "nmin": 64,
            "nmax": _logint(rng, 256, 768), "rmin": 8, "rmax": _logint(rng, 16, 64), "p": 8,
            "v": rng.choice([2, 3, 4]), "sizes": rng.randrange(1 << 20)}


# ---------------------------------------------------------------------------------------- inputs
def _gen(seed, tag=0):
    g = torch.Generator(device=_DEV)
    g.manual_seed(1000003 * (seed % (1 << 40)) + tag)
    return g


def _gauss(g, *shape):
    return torch.randn(*shape, generator=g, device=_DEV, dtype=torch.float32)


def _rows(m, n, planes, dtype):
    return qlr.empty_rowmajor(m, n, planes, dtype)


def _colour(g, m, n, planes, dtype):
    """An image-like field: 64 random 2-D cosines per plane, scaled to [0, 1], plus noise of +-0.05."""
    out = _rows(m, n, planes, dtype)
    y = torch.arange(m, device=_DEV, dtype=torch.float32)[:, None] * (2 * math.pi / m)
    x = torch.arange(n, device=_DEV, dtype=torch.float32)[None, :] * (2 * math.pi / n)
    for c in range(planes):
        f = torch.randint(0, 9, (2, 64), generator=g, device=_DEV).float()
        amp, ph = _gauss(g, 64), torch.rand(64, generator=g, device=_DEV) * (2 * math.pi)
        left, right = y * f[0][None, :], f[1][:, None] * x + ph[:, None]
        P = torch.cat([left.cos() * amp, -left.sin() * amp], 1) @ torch.cat([right.cos(), right.sin()], 0)
        lo, hi = P.min(), P.max()
        P = (P - lo) / (hi - lo) + (torch.rand(m, n, generator=g, device=_DEV) - 0.5) * 0.1
        out[c].copy_(P)
    return out


def _decaying(g, m, n, planes, dtype, sigma):
    """A matrix whose singular values are close to sigma: B diag(sigma) C, B real Gaussian, C quaternion Gaussian."""
    r = len(sigma)
    s = torch.tensor(sigma, device=_DEV, dtype=torch.float32)
    out = _rows(m, n, planes, dtype)
    wide = torch.float64 if dtype == torch.float64 else torch.float32
    B = (_gauss(g, m, r) * (s / math.sqrt(m))).to(wide)
    for c in range(planes):
        out[c].copy_(B @ (_gauss(g, r, n) / math.sqrt(planes * n)).to(wide))
    return out


def _lowrank_noise(g, m, n, r, noise, dtype):
    """A pure matrix of rank r (real times pure), unit RMS over its planes, plus Gaussian noise."""
    B, C = _gauss(g, m, r), _gauss(g, 3, r, n)
    A = torch.matmul(B, C)
    A *= A.square().mean().rsqrt()
    A += noise * _gauss(g, 3, m, n)
    out = _rows(m, n, 3, dtype)
    out.copy_(A)
    return out


def _thin(g, rows, cols, dtype=torch.float32, scale=1.0):
    t = qlr.empty_thin(rows, cols, dtype)
    t.copy_((_gauss(g, 4, cols, rows) * scale).transpose(1, 2))
    return t


def _spectrum(case):
    m, n, k, p = case["m"], case["n"], case["k"], case["p"]
    r = min(m, n, 256 if case["algo"] == 4 else max(2 * (k + p), 128))
    if case["dtype"] == "f64":
        return [0.5 ** i if i < 12 else 0.5 ** 12 / (i - 10) for i in range(r)]   # a fast decay and a floor
    if case["algo"] == 4:
        return [math.exp(-i / 50.0) for i in range(r)]
    return [1.0 / (i + 1) for i in range(r)]                                     # the slow decay


def _side_h(case):
    return case["v"] % 2 == 0 and case["n"] > case["m"]


def _batch_sizes(case):
    g = torch.Generator()
    g.manual_seed(case["sizes"])
    u = torch.rand(3, case["count"], generator=g, dtype=torch.float64)
    pick = lambda t, lo, hi: (lo + (t * (hi - lo + 1)).floor()).long().tolist()  # noqa: E731
    ms, ns, rs = (pick(u[0], case["mmin"], case["mmax"]), pick(u[1], case["nmin"], case["nmax"]),
                  pick(u[2], case["rmin"], case["rmax"]))
    out = []
    for m, n, r in zip(ms, ns, rs):
        l = min(r + case["p"], m, n)
        k = min(r, l)
        out.append((m, n, k, l - k, r))
    return out


def _inputs(case, seed):
    """The seeded inputs of a case (what exact() reads too)."""
    kind = case["kind"]
    g = _gen(seed)
    if kind == "sketch":
        m, n, l = case["m"], case["n"], case["l"]
        A = _colour(g, m, n, 3 if case["pure"] else 4, _DTYPE[case["dtype"]])
        return {"A": A, "X": _thin(g, n, l), "W": _thin(g, m, l, scale=1 / math.sqrt(m))}
    if kind == "orth":
        m, l = case["m"], case["l"]
        # a view of a matrix of slow decay: a condition number near l, its directions mixed by the test matrix
        s = torch.tensor([1.0 / (1 + i) for i in range(l)], device=_DEV)
        Y = qlr.empty_thin(m, l)
        mix = torch.linalg.qr(_gauss(g, l, l))[0]
        Y.copy_(torch.matmul(_gauss(g, 4, m, l) * s, mix))
        return {"Y": Y}
    if kind == "lowrank":
        m, n, dt = case["m"], case["n"], _DTYPE[case["dtype"]]
        A = _decaying(g, m, n, 3 if case["pure"] else 4, dt, _spectrum(case))
        return {"A": A, "omega": _thin(g, m if _side_h(case) else n, case["k"] + case["p"], dt)}
    if kind == "complete":
        m, n = case["m"], case["n"]
        M = _lowrank_noise(g, m, n, case["k"], 1e-2, torch.float32)
        mask = (torch.rand(m, n, generator=g, device=_DEV) >= 0.7).to(torch.uint8)
        return {"M": M, "mask": mask, "omega": _thin(g, m if _side_h(case) else n, case["k"] + case["p"])}
    As, oms = [], []
    for m, n, k, p, r in _batch_sizes(case):
        As.append(_lowrank_noise(g, m, n, r, 1e-3, torch.bfloat16))
        oms.append(_thin(g, n, k + p))
    return {"As": As, "omegas": oms}


def prepare(case, seed):
    kind = case["kind"]
    ctx = qlr.Context(torch.cuda.current_device())
    s = {"case": case, "ctx": ctx, **_inputs(case, seed)}
    if kind == "sketch":
        m, n, l = case["m"], case["n"], case["l"]
        s["Y"], s["Z"] = qlr.empty_thin(m, l), qlr.empty_thin(n, l)
        ctx.reserve(qlr.workspace_size(m, n, l, 0, 2))
    elif kind == "orth":
        s["Q"] = qlr.empty_thin(case["m"], case["l"])
        ctx.reserve(qlr.workspace_size(case["m"], case["l"], case["l"], 0, 2))
    elif kind in ("lowrank", "complete"):
        m, n, k = case["m"], case["n"], case["k"]
        dt = _DTYPE[case.get("dtype", "f32")]
        algo = case.get("algo", 2)
        compute = qlr.COMPUTE_F64 if dt == torch.float64 else _COMPUTE[case.get("compute", "auto")]
        s["U"], s["V"] = qlr.empty_thin(m, k, dt), qlr.empty_thin(n, k, dt)
        s["S"] = torch.empty(k, dtype=torch.float64, device=_DEV)
        s["C"] = _rows(m, n, 4, dt)
        if kind == "lowrank":
            s["mask"] = torch.zeros(m, n, dtype=torch.uint8, device=_DEV)   # nothing kept: all of U diag(S) V^H
        ctx.reserve(qlr.workspace_size(m, n, k, case["p"], case["v"], algo, compute))
    else:
        sizes = _batch_sizes(case)
        s["Uf"], s["Vf"] = (torch.empty(sum(4 * z[i] * z[2] for z in sizes), device=_DEV) for i in (0, 1))
        s["Sf"] = torch.empty(sum(z[2] for z in sizes), dtype=torch.float64, device=_DEV)
        Us, Ss, Vs, u, v, w = [], [], [], 0, 0, 0
        for m, n, k, p, r in sizes:
            Us.append(s["Uf"][u:u + 4 * m * k].view(4, k, m).transpose(1, 2))
            Vs.append(s["Vf"][v:v + 4 * n * k].view(4, k, n).transpose(1, 2))
            Ss.append(s["Sf"][w:w + k])
            u, v, w = u + 4 * m * k, v + 4 * n * k, w + k
        s["plan"] = qlr.Batch(ctx, s["As"], [z[2] for z in sizes], [z[3] for z in sizes], case["v"], s["omegas"],
                              Us, Ss, Vs, compute=qlr.COMPUTE_BF16)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "sketch":
        compute = _COMPUTE[case["compute"]]
        qlr.qsketch(ctx, qlr.OP_N, s["A"], s["X"], s["Y"], compute)
        qlr.qsketch(ctx, qlr.OP_H, s["A"], s["W"], s["Z"], compute)
        return {"Y": s["Y"], "Z": s["Z"]}
    if kind == "orth":
        qlr.cholqr(ctx, s["Y"], s["Q"])
        return {"Q": s["Q"]}
    if kind == "lowrank":
        f64 = case["dtype"] == "f64"
        qlr.qsvd_lowrank(ctx, s["A"], case["k"], case["p"], case["v"], s["omega"], s["U"], s["S"], s["V"],
                         algo=case["algo"], compute=_COMPUTE[case["compute"]])
        qlr.complete_update(ctx, s["C"], s["mask"], s["C"], s["U"], s["S"], s["V"], case["k"])
        return {"approx": s["C"], "S": s["S"] if f64 else s["S"].float()}
    if kind == "complete":
        qlr.complete(ctx, s["M"], s["mask"], case["k"], case["p"], case["v"], case["iters"], s["omega"], s["C"],
                     s["U"], s["S"], s["V"])
        return {"C": s["C"], "S": s["S"].float()}
    s["plan"].run()
    return {"U": s["Uf"].bfloat16(), "S": s["Sf"].float(), "V": s["Vf"].bfloat16()}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for m, n, k, p, r in _batch_sizes(case):
            b += 3 * 2 * m * n * case["v"] + 16 * n * (k + p) + 24 * k * (m + n) + 12 * k
            f += 24 * m * n * (k + p) * case["v"]
        return {"bytes": b, "flops": f}
    m, l = case["m"], case.get("l", 0)
    if kind == "orth":
        return {"bytes": 32 * m * l, "flops": 32 * m * l * l}      # Gram and triangular product, half of 32 each
    n = case["n"]
    es = {"f64": 8, "f32": 4, "bf16": 2}[case.get("dtype", "f32")]
    pl = 3 if case.get("pure") else 4
    if kind == "sketch":
        return {"bytes": 2 * pl * m * n * es + 32 * l * (m + n), "flops": 2 * 8 * pl * m * n * l}
    k, v = case["k"], case["v"]
    l = k + case["p"]
    if kind == "lowrank":
        cols = v * l
        if case["algo"] == 4:
            cols = (v - 1) * l + ((v // 2) if v % 2 == 0 else (v - 1) // 2) * l
        return {"bytes": v * pl * m * n * es + 4 * m * n * es + m * n, "flops": 8 * pl * m * n * cols + 32 * m * n * k}
    it = case["iters"]
    return {"bytes": it * (v * 4 * m * n * es + m * n + 3 * m * n * es + 4 * m * n * es),
            "flops": it * (32 * m * n * l * v + 32 * m * n * k)}


# ------------------------------------------------------------------------- the same in 64 bits, by plain torch
_TERMS = [[(0, 0, 1), (1, 1, -1), (2, 2, -1), (3, 3, -1)], [(0, 1, 1), (1, 0, 1), (2, 3, 1), (3, 2, -1)],
          [(0, 2, 1), (1, 3, -1), (2, 0, 1), (3, 1, 1)], [(0, 3, 1), (1, 2, 1), (2, 1, -1), (3, 0, 1)]]


def _planes(A):
    A = A.double()
    return [None, *A] if A.shape[0] == 3 else list(A)


def _mul(A, B):
    """Quaternion matrix product of plane lists (None: a zero plane)."""
    out = []
    for terms in _TERMS:
        t = None
        for a, b, sg in terms:
            if A[a] is None or B[b] is None:
                continue
            t = sg * (A[a] @ B[b]) if t is None else t.add_(A[a] @ B[b], alpha=sg)
        out.append(t)
    return out


def _ct(A):
    return [None if a is None else (a.T if c == 0 else -a.T) for c, a in enumerate(A)]


def _adjoint(Y):
    """The complex adjoint, each quaternion a 2 x 2 block."""
    a, b = torch.complex(Y[0], Y[1]), torch.complex(Y[2], Y[3])
    m, n = a.shape
    X = torch.stack([torch.stack([a, b], -1), torch.stack([-b.conj(), a.conj()], -1)], 1)   # m, 2, n, 2
    return X.reshape(2 * m, 2 * n)


def _unadjoint(X):
    a, b = X[0::2, 0::2], X[0::2, 1::2]
    return [a.real.contiguous(), a.imag.contiguous(), b.real.contiguous(), b.imag.contiguous()]


def _qr(Y):
    """Thin QR with a positive real diagonal: the adjoint's is unique, so it is the adjoint of the quaternion one."""
    Q, R = torch.linalg.qr(_adjoint(Y))
    d = torch.diagonal(R)
    ph = d / d.abs()
    return _unadjoint(Q * ph[None, :]), R * ph.conj()[:, None]


def _exact_svd(A, k, p, v, omega, algo):
    """(approximation of rank k, S) by Algorithm 2 or 4 as the paper prints them."""
    q2, K1, K2 = omega, [], []
    if algo == 4 and v >= 4:
        views = v - 1
    else:
        views, algo = v, 2
    for i in range(1, views + 1):
        if i % 2:
            q1, R = _qr(_mul(A, q2))
            K1.append(q1)
        else:
            q2, R = _qr(_mul(_ct(A), q1))
            K2.append(q2)
    if algo == 4:
        if v % 2 == 0:
            q1, _ = _qr([torch.cat([b[c] for b in K1], 1) for c in range(4)])
            q2, R = _qr(_mul(_ct(A), q1))
        else:
            q2, _ = _qr([torch.cat([b[c] for b in K2], 1) for c in range(4)])
            q1, R = _qr(_mul(A, q2))
    u, s, vh = torch.linalg.svd(R)
    Rk = (u[:, :2 * k] * s[:2 * k]) @ vh[:2 * k]
    mid = _unadjoint(Rk if v % 2 else Rk.conj().T)       # odd: A ~ Q1 R Q2^H; even: A ~ Q1 R^H Q2^H
    return _mul(_mul(q1, mid), _ct(q2)), s[0:2 * k:2]


def _exact_lowrank(A, case, omega, algo):
    if _side_h(case):
        C, S = _exact_svd(_ct(A), case["k"], case["p"], case["v"], omega, algo)
        return _ct(C), S
    return _exact_svd(A, case["k"], case["p"], case["v"], omega, algo)


def _exact_sigma(A, k, v, omega):
    """The singular values that Algorithm 2 finds, by Cholesky factors of well conditioned Grams."""
    q = omega
    for i in range(1, v + 1):
        y = _mul(A if i % 2 else _ct(A), q)
        X = _adjoint(y)
        G = X.conj().T @ X
        if i == v:
            return torch.linalg.eigvalsh(G).flip(0).clamp_min(0).sqrt()[0:2 * k:2]
        L = torch.linalg.cholesky(G)
        q = _unadjoint(torch.linalg.solve_triangular(L, X.conj().T, upper=False).conj().T)


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "sketch":
        A = _planes(x["A"])
        wide = lambda t: list((t.bfloat16() if case["dtype"] == "bf16" else t).double())  # noqa: E731
        return {"Y": torch.stack(_mul(A, wide(x["X"]))), "Z": torch.stack(_mul(_ct(A), wide(x["W"])))}
    if kind == "orth":
        return {"Q": torch.stack(_qr(_planes(x["Y"]))[0])}
    if kind == "lowrank":
        C, S = _exact_lowrank(_planes(x["A"]), case, list(x["omega"].double()), case["algo"])
        return {"approx": torch.stack(C), "S": S}
    if kind == "complete":
        M, seen = [torch.zeros_like(x["mask"], dtype=torch.float64), *x["M"].double()], x["mask"].bool()
        C = [t * seen for t in M]
        for _ in range(case["iters"]):
            X, S = _exact_lowrank(C, case, list(x["omega"].double()), 2)
            C = [torch.where(seen, a, b) for a, b in zip(M, X)]
        return {"C": torch.stack(C), "S": S}
    S = [_exact_sigma(_planes(a), z[2], case["v"], list(o.double()))
         for a, o, z in zip(x["As"], x["omegas"], _batch_sizes(case))]
    return {"U": None, "S": torch.cat(S), "V": None}       # U and V: a unit quaternion per pair is free
