"""The work that users of the library have it do, as timed cases.

Every case goes through the public entry points (the C ABI's binding,
paper_2509_02840_gb300/bdu.py).  Sizes are those of the benchmark
configurations (256 x 128, 4096 x 4096, the 16384-node network, the serving
mix of 64..2048), of the problems the paper's table lists, and odd ones
between them.

Kinds:
  stream  -- one resident factorization takes `updates` calls of rank r and is
             then read back whole (Q, d, e, P);
  inplace -- the allocation-free rank-1 update of device buffers;
  batch   -- one batched update of `sessions` resident factorizations of uneven
             sizes and ranks 1..4; every session's d, e is read afterwards and
             the first four are read whole, as an eviction does;
  thin    -- one rank-k tracking step and the read of the thin factors;
  bhu     -- `steps` iterations of the Householder update's compact form;
  tri     -- the symmetric variant, in place on device buffers;
  query   -- singular values and the truncated factors of a resident
             factorization.
Mixed-form factors are held in FP32 and returned in that type.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2509_02840_gb300 import bdu


def listed():
    return [
        # a small dense problem of the size of the paper's table, updated in a
        # caller's own buffers: latency of one tiny update
        {"name": "inplace_608x188", "kind": "inplace", "m": 608, "n": 188},
        # the benchmark's first configuration: host vectors, FP64, read back
        {"name": "fp64_256x128", "kind": "stream", "form": "fp64", "m": 256, "n": 128, "r": 1, "updates": 1,
         "overlap": False, "data": "dense", "host": True},
        # more columns than rows (held as the transposed problem), rank 2, odd sizes
        {"name": "fp64_701x1493_r2", "kind": "stream", "form": "fp64", "m": 701, "n": 1493, "r": 2, "updates": 1,
         "overlap": False, "data": "dense", "host": True},
        # the recommender stream in FP64: one ratings column set
        {"name": "fp64_4096", "kind": "stream", "form": "fp64", "m": 4096, "n": 4096, "r": 1, "updates": 1,
         "overlap": False, "data": "ratings", "host": False},
        # the headline: a burst of four ratings columns in the overlapped mixed form
        {"name": "mixed_4096_burst4", "kind": "stream", "form": "mixed", "m": 4096, "n": 4096, "r": 1, "updates": 4,
         "overlap": True, "data": "ratings", "host": False},
        # a block update (rank 8, tall), mixed form
        {"name": "mixed_3001x1003_r8", "kind": "stream", "form": "mixed", "m": 3001, "n": 1003, "r": 8, "updates": 1,
         "overlap": False, "data": "block", "host": False},
        # continuous serving: one batch of uneven sessions, both forms
        {"name": "batch_mixed_32", "kind": "batch", "form": "mixed", "sessions": 32, "lo": 64, "hi": 2048, "mix": 1},
        {"name": "batch_fp64_16", "kind": "batch", "form": "fp64", "sessions": 16, "lo": 64, "hi": 1024, "mix": 2},
        # rank-256 tracking of a 16384-node network, one edge column at a time
        {"name": "thin_mixed_16384_k256", "kind": "thin", "form": "mixed", "m": 16384, "n": 16384, "k": 256},
        # a partial Householder update (n much smaller than m), rank 8 in one sweep
        {"name": "bhu_4472x936_s96", "kind": "bhu", "m": 4472, "n": 936, "r": 8, "steps": 96},
        # the symmetric variant on a small graph
        {"name": "tri_600", "kind": "tri", "n": 600},
        # what a user asks of a factorization: leading singular values, truncated factors
        {"name": "query_2048", "kind": "query", "form": "fp64", "m": 2048, "n": 2048, "sv": 64, "keep": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stream", "stream", "stream", "stream", "inplace", "batch", "thin", "bhu", "tri", "query"])
    if kind == "stream":
        form = rng.choice(["fp64", "mixed"])
        top = 2400 if form == "fp64" else 3600
        a, b = _log(rng, 48, top), _log(rng, 48, top)
        r = rng.choice([1, 1, 2, 3, 4, 8])
        if form == "fp64" and a + b > 2400:
            r = min(r, 2)
        overlap = form == "mixed" and r == 1 and rng.random() < 0.7
        return {"kind": kind, "form": form, "m": a, "n": b, "r": r,
                "updates": rng.choice([2, 3, 4]) if overlap else 1, "overlap": overlap,
                "data": rng.choice(["dense", "ratings", "block"]) if r > 1 else rng.choice(["dense", "ratings"]),
                "host": rng.random() < 0.5}
    if kind == "inplace":
        n = _log(rng, 8, 256)
        return {"kind": kind, "m": max(n, _log(rng, 16, 1024)), "n": n}
    if kind == "batch":
        form = rng.choice(["fp64", "mixed"])
        return {"kind": kind, "form": form, "sessions": rng.randint(5, 32 if form == "mixed" else 16), "lo": 64,
                "hi": _log(rng, 256, 2048 if form == "mixed" else 1024), "mix": rng.randint(3, 10 ** 6)}
    if kind == "thin":
        m, n = _log(rng, 1000, 16384), _log(rng, 1000, 16384)
        return {"kind": kind, "form": rng.choice(["fp64", "mixed"]), "m": m, "n": n, "k": _log(rng, 16, 400)}
    if kind == "bhu":
        n = _log(rng, 64, 1200)
        return {"kind": kind, "m": n + _log(rng, 1, 4000), "n": n, "r": rng.choice([1, 2, 8]),
                "steps": min(n, rng.randint(8, 120))}
    if kind == "tri":
        return {"kind": kind, "n": _log(rng, 40, 900)}
    n = _log(rng, 100, 2048)
    return {"kind": kind, "form": rng.choice(["fp64", "mixed"]), "m": n + rng.choice([0, rng.randint(1, 500)]), "n": n,
            "sv": min(n, rng.randint(1, 100)), "keep": min(n, rng.randint(1, 100))}


# ---------------------------------------------------------------- inputs

def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _orthogonal(n, g):
    """A product of 8 Householder reflectors with N(0, 1) vectors (FP64, on the GPU; symmetric storage does not
    matter: the returned tensor is read column by column)."""
    X = torch.eye(n, dtype=torch.float64, device="cuda")
    for _ in range(8):
        v = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
        X -= torch.outer(X @ v, v) * (2.0 / torch.dot(v, v))
    return X


def _host_cols(X):
    """Column-major host copy."""
    return X.t().contiguous().cpu().numpy().T


def _band(k, g):
    d = 1.0 + 9.0 * torch.rand(k, dtype=torch.float64, device="cuda", generator=g)
    e = torch.randn(max(k - 1, 0), dtype=torch.float64, device="cuda", generator=g)
    return d, e


def _factors(m, n, g):
    Q, P = _orthogonal(m, g), _orthogonal(n, g)
    d, e = _band(min(m, n), g)
    return Q, d, e, P


def _update(m, n, r, data, g):
    """(B, C) as (r, m) and (r, n) device tensors: their rows are the update's columns."""
    if data == "ratings":  # 2 % of the rows rated 1..5; c picks one item
        B = torch.zeros(r, m, dtype=torch.float64, device="cuda")
        C = torch.zeros(r, n, dtype=torch.float64, device="cuda")
        k = max(1, round(0.02 * m))
        for t in range(r):
            rows = torch.randperm(m, device="cuda", generator=g)[:k]
            B[t, rows] = torch.randint(1, 6, (k,), device="cuda", generator=g).double()
            C[t, torch.randint(0, n, (1,), device="cuda", generator=g)] = 1.0
        return B, C
    B = torch.randn(r, m, dtype=torch.float64, device="cuda", generator=g)
    C = torch.randn(r, n, dtype=torch.float64, device="cuda", generator=g)
    return B, C / math.sqrt(n) if data == "block" else C


def _prec(case):
    return bdu.FP64 if case["form"] == "fp64" else bdu.MIXED


def _handle(Q, d, e, P, case, **more):
    return bdu.Factorization(_host_cols(Q), d.cpu().numpy(), e.cpu().numpy(), _host_cols(P), precision=_prec(case),
                             stream=torch.cuda.current_stream().cuda_stream or None, **more)


def _sizes(case):
    """The sessions of a batch: (m, n, r), m and n log-uniform."""
    import random
    rng = random.Random(case["mix"])
    return [(_log(rng, case["lo"], case["hi"]), _log(rng, case["lo"], case["hi"]), rng.randint(1, 4))
            for _ in range(case["sessions"])]


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "stream":
        m, n, r = case["m"], case["n"], case["r"]
        Q, d, e, P = _factors(m, n, g)
        ups = [_update(m, n, r, case["data"], g) for _ in range(case["updates"])]
        if case["host"]:
            ups = [(B.cpu().numpy().T, C.cpu().numpy().T) for B, C in ups]
        return {"case": case, "F": _handle(Q, d, e, P, case, overlap=case["overlap"]), "ups": ups}
    if kind == "inplace":
        m, n = case["m"], case["n"]
        Q, d, e, P = _factors(m, n, g)
        B, C = _update(m, n, 1, "dense", g)
        bufs = [Q.t().contiguous(), d, e if n > 1 else torch.zeros(1, dtype=torch.float64, device="cuda"),
                P.t().contiguous(), B, C]
        fn = bdu.load().bdu_update_rank1_noalloc
        fn.argtypes = [ctypes.c_int64] * 2 + [ctypes.c_void_p] * 7
        fn.restype = ctypes.c_int
        return {"case": case, "bufs": bufs, "fn": fn}
    if kind == "batch":
        fs, ups = [], []
        for m, n, r in _sizes(case):
            fs.append(_handle(*_factors(m, n, g), case))
            ups.append(_update(m, n, r, "dense", g))
        return {"case": case, "F": fs, "ups": ups}
    if kind == "thin":
        m, n, k = case["m"], case["n"], case["k"]
        Q1 = torch.linalg.qr(torch.randn(m, k, dtype=torch.float64, device="cuda", generator=g))[0]
        P1 = torch.linalg.qr(torch.randn(n, k, dtype=torch.float64, device="cuda", generator=g))[0]
        d, e = _band(k, g)
        b = torch.zeros(m, dtype=torch.float64, device="cuda")
        c = torch.zeros(n, dtype=torch.float64, device="cuda")
        b[torch.randint(0, m, (1,), device="cuda", generator=g)] = 0.5 + torch.rand(1, dtype=torch.float64,
                                                                                   device="cuda", generator=g)
        c[torch.randint(0, n, (1,), device="cuda", generator=g)] = 1.0
        T = bdu.ThinTracker(_host_cols(Q1), d.cpu().numpy(), e.cpu().numpy(), _host_cols(P1), precision=_prec(case))
        return {"case": case, "T": T, "b": b, "c": c}
    if kind == "bhu":
        m, n, r, steps = case["m"], case["n"], case["r"], case["steps"]
        d, e = _band(n, g)
        U, V = _update(m, n, r, "dense", g)
        kl, kr, wb = bdu.bhu_sizes(m, n, steps)
        z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")  # noqa: E731
        out = {"alpha": z(steps), "beta": z(max(1, min(steps, n - 1))), "Y": z(kl, m), "W": z(max(kr, 1), n),
               "SL": z(kl, kl), "SR": z(max(kr, 1), max(kr, 1))}
        return {"case": case, "d": d, "e": e, "U": U, "V": V, "out": out,
                "ws": torch.zeros(wb // 8 + 2, dtype=torch.float64, device="cuda")}
    if kind == "tri":
        n = case["n"]
        Q = _orthogonal(n, g).t().contiguous()
        a, b = _band(n, g)
        c = torch.randn(n, dtype=torch.float64, device="cuda", generator=g) / math.sqrt(n)
        ub = bdu.tri_sizes(n, n)[2]
        return {"case": case, "Q": Q, "a": a, "b": b, "c": c,
                "ws": torch.zeros(ub // 8 + 2, dtype=torch.float64, device="cuda")}
    Q, d, e, P = _factors(case["m"], case["n"], g)
    return {"case": case, "F": _handle(Q, d, e, P, case)}


# ---------------------------------------------------------------- one pass

def _whole(F, case):
    Q, d, e, P = F.read()
    if case["form"] == "mixed":
        Q, P = Q.astype(np.float32), P.astype(np.float32)
    return [Q, d, e, P]


def run(state):
    case = state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "stream":
        F = state["F"]
        for B, C in state["ups"]:
            if case["host"]:
                F.update(B, C)
            else:
                F.update_dev(B.data_ptr(), C.data_ptr(), case["r"])
        return _whole(F, case)
    if kind == "inplace":
        Q, d, e, P, b, c = state["bufs"]
        code = state["fn"](case["m"], case["n"], Q.data_ptr(), d.data_ptr(), e.data_ptr(), P.data_ptr(),
                           b.data_ptr(), c.data_ptr(), stream)
        if code != 0:
            raise RuntimeError("bdu_update_rank1_noalloc: status %d" % code)
        return [Q, d, e, P]
    if kind == "batch":
        fs, ups = state["F"], state["ups"]
        bdu.update_batch(fs, [B.data_ptr() for B, _ in ups], [C.data_ptr() for _, C in ups],
                         [B.shape[0] for B, _ in ups])
        bands = [F.read_bidiagonal() for F in fs]
        return {"d": np.concatenate([d for d, _ in bands]), "e": np.concatenate([e for _, e in bands]),
                "evicted": [_whole(F, case) for F in fs[:4]]}
    if kind == "thin":
        T = state["T"]
        dropped, err2 = T.update_dev(state["b"].data_ptr(), state["c"].data_ptr())
        Q1, d, e, P1 = T.read()
        if case["form"] == "mixed":
            Q1, P1 = Q1.astype(np.float32), P1.astype(np.float32)
        return {"dropped": dropped, "err2": err2, "Q1": Q1, "d": d, "e": e, "P1": P1}
    if kind == "bhu":
        o = state["out"]
        bdu.bhu_factor(case["m"], case["n"], case["steps"], state["d"].data_ptr(), state["e"].data_ptr(),
                       state["U"].data_ptr(), state["V"].data_ptr(), o["alpha"].data_ptr(), o["beta"].data_ptr(),
                       o["Y"].data_ptr(), o["W"].data_ptr(), o["SL"].data_ptr(), o["SR"].data_ptr(),
                       state["ws"].data_ptr(), stream=stream, r=case["r"])
        return o
    if kind == "tri":
        bdu.tri_update_dev(case["n"], state["Q"].data_ptr(), state["a"].data_ptr(), state["b"].data_ptr(), 0.75,
                           state["c"].data_ptr(), state["ws"].data_ptr(), stream=stream)
        return [state["Q"], state["a"], state["b"]]
    F = state["F"]
    L, R, idx, err2 = F.read_truncated(case["keep"])
    return {"sv": F.singular_values(case["sv"]), "L": L, "R": R, "idx": idx, "err2": err2}


# ---------------------------------------------------------------- work

def _column(m, n, es):
    """Bytes and operations of one rank-1 column: Q, P read and written once; about 0.75 k^2 rotations a side (and
    the spike's m - n), each 6 operations on every row of Q or P and about 26 to generate."""
    if m < n:
        m, n = n, m
    rot = 0.75 * n * n
    flops = 6.0 * (rot + (m - n)) * m + 6.0 * rot * n + 26.0 * (2 * rot + m - n)
    return 2.0 * es * (m * m + n * n) + 8.0 * (m + n) + 32.0 * n, flops


def work(case):
    kind = case["kind"]
    if kind in ("stream", "inplace"):
        es = 4 if case.get("form") == "mixed" else 8
        b, f = _column(case["m"], case["n"], es)
        k = case.get("r", 1) * case.get("updates", 1)
        m, n = case["m"], case["n"]
        return {"bytes": b + 8.0 * (k - 1) * (m + n), "flops": f * k + 2.0 * k * (m * m + n * n)}
    if kind == "batch":
        es = 4 if case["form"] == "mixed" else 8
        by = fl = 0.0
        for m, n, r in _sizes(case):
            b, f = _column(m, n, es)
            by += b + 8.0 * (r - 1) * (m + n)
            fl += f * r + 2.0 * r * (m * m + n * n)
        return {"bytes": by, "flops": fl}
    if kind == "thin":
        es = 4 if case["form"] == "mixed" else 8
        m, n, k = case["m"], case["n"], case["k"]
        rot = 0.75 * (k + 1) ** 2
        return {"bytes": 2.0 * es * (m + n) * k + 8.0 * (m + n) + 32.0 * k,
                "flops": 8.0 * (m + n) * k + 2.0 * (m + n) * k * (k + 1) + 12.0 * rot * (k + 1) + 52.0 * rot}
    if kind == "bhu":
        m, n, s, r = case["m"], case["n"], case["steps"], case["r"]
        # the factored products of step j: about four passes over Y and W of width j and the rank-r terms
        return {"bytes": 8.0 * ((m + n) * (s + r) + 2 * s * s + 2 * n),
                "flops": sum(8.0 * (m + n) * j + 4.0 * (m + n) * r for j in range(1, s + 1))}
    if kind == "tri":
        n = case["n"]
        return {"bytes": 16.0 * n * n + 40.0 * n, "flops": sum(8.0 * n * j for j in range(1, n)) + 4.0 * n ** 3}
    m, n, k, sv = case["m"], case["n"], case["keep"], case["sv"]
    es = 4 if case["form"] == "mixed" else 8
    # Sturm counts: about 50 bits of each value, one division a pivot
    return {"bytes": es * (2 * m + n) * k + 8.0 * (m + n) * k + 16.0 * n, "flops": 3.0 * 50 * 2 * n * sv + 3.0 * m * k}


# ---------------------------------------------------------------- in 64 bits

def exact(case, seed):
    """The bidiagonal a Givens or full Householder update ends with is fixed only up to signs, and its trailing
    entries (and the factors' columns) are ill-conditioned functions of A, so there is no value to hold them to;
    the queries and the first steps of the Householder process have one."""
    kind = case["kind"]
    if kind == "query":
        g = _gen(seed)
        m, n = case["m"], case["n"]
        Q, d, e, P = _factors(m, n, g)
        B = torch.diag(d) + torch.diag(e, 1)
        sv = torch.linalg.svdvals(B)[:case["sv"]]
        low = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), e])
        w = d * d + low * low
        idx = torch.sort(torch.sort(w, descending=True, stable=True)[1][:case["keep"]])[0]
        prev = torch.where(idx > 0, idx - 1, idx)
        L = Q[:, idx] * d[idx] + Q[:, prev] * low[idx]
        kept = torch.zeros(n, dtype=torch.bool, device="cuda")
        kept[idx] = True
        return {"sv": sv, "L": L, "R": P[:, idx], "idx": idx + 1, "err2": float(w[~kept].sum())}
    if kind == "bhu":
        g = _gen(seed)
        m, n, r, steps = case["m"], case["n"], case["r"], case["steps"]
        d, e = _band(n, g)
        U, V = _update(m, n, r, "dense", g)
        A = torch.zeros(m, n, dtype=torch.float64, device="cuda")
        A[:n] = torch.diag(d) + torch.diag(e, 1)
        A += U.t() @ V
        kl, kr = min(steps, n if m > n else n - 1), max(0, min(steps, n - 2))
        alpha = torch.zeros(steps, dtype=torch.float64, device="cuda")
        beta = torch.zeros(max(1, min(steps, n - 1)), dtype=torch.float64, device="cuda")
        Y = torch.zeros(kl, m, dtype=torch.float64, device="cuda")
        W = torch.zeros(max(kr, 1), n, dtype=torch.float64, device="cuda")

        def house(x):
            y = x.clone()
            s = 1.0 - 2.0 * torch.signbit(x[0]).double()
            norm = torch.linalg.norm(x)
            y[0] += s * norm
            return y / torch.linalg.norm(y), -s * norm

        for k in range(steps):
            if k < kl:
                y, alpha[k] = house(A[k:, k])
                A[k:] -= 2.0 * torch.outer(y, y @ A[k:])
                Y[k, k:] = y
            else:
                alpha[k] = A[k, k]
            if k < kr:
                w, beta[k] = house(A[k, k + 1:])
                A[:, k + 1:] -= 2.0 * torch.outer(A[:, k + 1:] @ w, w)
                W[k, k + 1:] = w
            elif k < n - 1:
                beta[k] = A[k, k + 1]

        def upper(Z, k):  # the products' upper triangular factor: I - Z' S Z
            S = torch.zeros(k, k, dtype=torch.float64, device="cuda")
            for j in range(k):
                S[j, j] = 2.0
                if j:
                    S[:j, j] = -2.0 * (S[:j, :j] @ (Z[:j] @ Z[j]))
            return S.t().contiguous()  # column by column

        return {"alpha": alpha, "beta": beta, "Y": Y, "W": W, "SL": upper(Y, kl),
                "SR": upper(W, kr) if kr else None}
    return None
