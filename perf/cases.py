"""Performance cases of the library: what its users have it do, through the public entry points.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from a seed, ``run`` does one pass, ``exact``
computes the same outputs in 64 bits with plain torch (pairwise products, sorted or indexed sums).  The families:

* ``total``    polynomials holding (nearly) all monomials up to a total degree: the moderately sparse products, on the
               dense path, from the smallest calls to powers of a full size; int64 or float64, whole or truncated by degree
* ``weighted`` the weighted exponent structure of the highly sparse benchmark (one factor weighted 1 1 2 3 5, the other
               5 3 2 1 1), int64, hash path
* ``laurent``  random Laurent polynomials in a wide box, nearly every pair a term of its own
* ``poisson``  Poisson series: narrow boxes (many pairs per output term) or the wide boxes of celestial mechanics
* ``batch``    products of uneven sizes and both kinds in one call
* ``graph``    small products prepared once and replayed
* ``codec``    exponent vectors to codes and back
"""
from __future__ import annotations

import math
import zlib
from collections import deque
from types import SimpleNamespace

import numpy as np
import torch

import paper_1004_4548_gb300 as kron


def listed():
    return [
        # smallest calls of interactive use: 1001 x 1001 terms, latency and launches count
        {"name": "total_d10", "family": "total", "v": 4, "df": 10, "dg": 10, "keep": 1.0, "coef": "i64", "cmax": 1 << 20, "trunc": -1},
        # the headline product: 10626 x 10626 terms
        {"name": "total_d20", "family": "total", "v": 4, "df": 20, "dg": 20, "keep": 1.0, "coef": "i64", "cmax": 1 << 20, "trunc": -1},
        # Fateman's benchmark at full size, (1+x+y+z+t)^30 times itself plus one: coefficients of the whole 64-bit range
        {"name": "power_d30", "family": "total", "v": 4, "df": 30, "dg": 30, "keep": 1.0, "coef": "power", "cmax": 0, "trunc": -1},
        # the same structure with float64 coefficients, operands of different sizes and with holes
        {"name": "total_f64", "family": "total", "v": 4, "df": 16, "dg": 13, "keep": 0.9, "coef": "f64", "cmax": 0, "trunc": -1},
        # multiplication of truncated power series: only the terms up to the operands' own degree
        {"name": "total_trunc", "family": "total", "v": 4, "df": 22, "dg": 22, "keep": 1.0, "coef": "i64", "cmax": 1 << 31, "trunc": 22},
        # the highly sparse benchmark: 6188 x 6188 terms, 5.8 million output terms, hash path
        {"name": "weighted_d12", "family": "weighted", "d": 12, "cmax": 1 << 20},
        # random float64 Laurent polynomials, the output nearly as long as the number of pairs
        {"name": "laurent_f64", "family": "laurent", "v": 6, "nf": 2311, "ng": 1507, "half": 20, "coef": "f64"},
        # Poisson series whose products fall on few keys (perturbation theory to low order)
        {"name": "poisson_narrow", "family": "poisson", "npoly": 2, "ntrig": 2, "nf": 3001, "ng": 2203, "prange": 4, "trange": 8},
        # Poisson series of the planetary kind: 3 polynomial and 4 trigonometric variables, nearly every key its own
        {"name": "poisson_wide", "family": "poisson", "npoly": 3, "ntrig": 4, "nf": 5003, "ng": 3989, "prange": 4, "trange": 8},
        # a batch of uneven products, half polynomials, half Poisson series
        {"name": "batch_mix", "family": "batch", "count": 16, "most": 3000},
        # a prepared batch of small products, replayed
        {"name": "graph_small", "family": "graph", "count": 16, "most": 200},
        # exponents to codes and back, 3 million terms in 5 variables
        {"name": "codec", "family": "codec", "v": 5, "n": 3000017, "width": 41},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["total", "total", "total", "weighted", "laurent", "poisson", "poisson", "batch", "graph", "codec"])
    if family == "total":
        v = rng.randint(2, 5)
        coef = rng.choice(["i64", "i64", "f64", "power"])
        top = {"f64": 6000, "i64": 15000, "power": 46376}[coef]

        def degree(n):
            d = 2
            while d < 60 and math.comb(v + d + 1, v) <= n:
                d += 1
            return d
        df = degree(_log(rng, 50, top))
        dg = df if coef == "power" else degree(_log(rng, 50, top))
        keep = 1.0 if coef == "power" else rng.choice([1.0, 0.9, 0.5])
        trunc = rng.choice([-1, -1, max(df, dg)])
        return {"family": family, "v": v, "df": df, "dg": dg, "keep": keep, "coef": coef,
                "cmax": rng.choice([1 << 20, 1 << 30, 1 << 40]) if coef == "i64" else 0, "trunc": trunc}
    if family == "weighted":
        return {"family": family, "d": rng.randint(5, 12), "cmax": rng.choice([1 << 20, 1 << 40])}
    if family == "laurent":
        return {"family": family, "v": rng.randint(4, 6), "nf": _log(rng, 60, 2311), "ng": _log(rng, 60, 1507), "half": rng.randint(12, 20),
                "coef": rng.choice(["i64", "f64"])}
    if family == "poisson":
        wide = rng.random() < 0.5
        return {"family": family, "npoly": 3 if wide else 2, "ntrig": rng.randint(3, 4) if wide else 2, "nf": _log(rng, 60, 5003 if wide else 3001),
                "ng": _log(rng, 60, 3989 if wide else 2203), "prange": rng.randint(3, 5), "trange": rng.randint(6, 10)}
    if family in ("batch", "graph"):
        return {"family": family, "count": rng.randint(3, 16), "most": _log(rng, 200, 3000) if family == "batch" else rng.randint(60, 200)}
    return {"family": family, "v": rng.randint(2, 6), "n": _log(rng, 1000, 3000017), "width": rng.randint(9, 41)}


# ---------------------------------------------------------------------------- inputs (numpy, from the seed alone)

def _simplex(v, d):
    """All nonnegative v-tuples of sum at most d, [v, count] int32."""
    rows = np.zeros((1, 0), np.int32)
    for _ in range(v):
        room = d - rows.sum(axis=1) + 1
        starts = np.repeat(np.cumsum(room) - room, room)
        col = (np.arange(int(room.sum())) - starts).astype(np.int32)
        rows = np.concatenate([np.repeat(rows, room, axis=0), col[:, None]], axis=1)
    return rows.T


def _integers(rng, n, cmax):
    """Nonzero and of random sign, from a range in which sums hardly ever cancel."""
    c = rng.integers(-cmax, cmax, n)
    return np.where(c >= 0, c + 1, c).astype(np.int64)


def _floats(rng, n):
    return np.where(rng.random(n) < 0.5, -1.0, 1.0) * (0.25 + rng.random(n))


def _poly(rng, exps, coef):
    """The terms in an order of the seed's."""
    p = rng.permutation(exps.shape[1])
    return SimpleNamespace(exps=np.ascontiguousarray(exps[:, p]).astype(np.int32), coef=coef[p])


def _total(shape, rng, v, d, keep, coef, cmax):
    e = _simplex(v, d)
    if keep < 1.0:
        e = e[:, shape.random(e.shape[1]) < keep]
    return _poly(rng, e, _floats(rng, e.shape[1]) if coef == "f64" else _integers(rng, e.shape[1], cmax))


def _power(rng, weight, d, plus):
    """(1 + sum_k weight_k x_k)^d + plus, coefficients modulo 2^64."""
    e = _simplex(len(weight), d)
    fact = [math.factorial(k) for k in range(d + 1)]
    c = []
    for r in e.T.tolist():
        m = fact[d] // math.prod([fact[x] for x in r] + [fact[d - sum(r)]])
        c.append((m * math.prod(int(a) ** x for a, x in zip(weight, r)) + (0 if any(r) else plus)) % (1 << 64))
    return _poly(rng, e, np.array(c, dtype=np.uint64).view(np.int64))


def _distinct(n, draw_rows):
    rows = np.zeros((0, 0), np.int64)
    while rows.shape[0] < n:
        more = draw_rows(2 * n + 64)
        rows = np.concatenate([rows, more]) if rows.size else more
        _, first = np.unique(rows, axis=0, return_index=True)
        rows = rows[np.sort(first)]
    return rows[:n]


def _laurent(shape, rng, v, n, half, coef):
    rows = _distinct(n, lambda m: shape.integers(-half, half + 1, (m, v)))
    return _poly(rng, rows.T, _floats(rng, n) if coef == "f64" else _integers(rng, n, 1 << 20))


def _canonical(t, kind):
    """Valid terms: the highest-index nonzero multiplier positive, no sine of the zero vector."""
    nz = t != 0
    some = nz.any(axis=1)
    last = t.shape[1] - 1 - np.argmax(nz[:, ::-1], axis=1)
    return (some & (t[np.arange(t.shape[0]), last] > 0)) | (~some & (kind == 0))


def _pseries(rng, p, t, k, coef):
    q = rng.permutation(k.size)
    return SimpleNamespace(exps=np.ascontiguousarray(p[:, q].astype(np.int32)), trig=np.ascontiguousarray(t[:, q].astype(np.int32)),
                           kind=k[q].astype(np.uint8), coef=coef[q])


def _series(shape, rng, n, npoly, ntrig, prange, trange):
    def rows(m):
        p = shape.integers(-prange, prange + 1, (4 * m, npoly))
        t = shape.integers(-trange, trange + 1, (4 * m, ntrig))
        k = shape.integers(0, 2, 4 * m)
        r = np.concatenate([p, t, k[:, None]], axis=1)[_canonical(t, k)]
        return r[:m]
    box = (2 * prange + 1) ** npoly * (2 * trange + 1) ** ntrig
    r = _distinct(min(n, box // 3), rows)
    p, t, k = r[:, :npoly], r[:, npoly:npoly + ntrig], r[:, -1]
    c = np.where(rng.random(len(r)) < 0.5, -1.0, 1.0) * 10.0 ** (rng.random(len(r)) - np.abs(p).sum(1) - np.abs(t).sum(1))
    return _pseries(rng, p.T, t.T, k, c)


def _uneven(shape, rng, v, poisson, most):
    """An operand of the uneven batch: log-uniform size, a subset of a simplex, weighted in half the draws."""
    n = int(round(math.exp(shape.uniform(math.log(50), math.log(most)))))
    d = next((d for d in range(4, 20) if math.comb(v + d, v) >= n), 20)
    e = _simplex(v, d)
    e = e[:, shape.permutation(e.shape[1])[:n]]
    top = np.full(v, d)
    if shape.random() < 0.5:
        w = np.array([1, 2, 3, 5])[shape.integers(0, 4, v)]
        e, top = e * w[:, None], d * w
    n = e.shape[1]
    if not poisson:
        return _poly(rng, e, _integers(rng, n, 1 << 20))
    npoly = v - v // 2
    p, t = e[:npoly] - (top[:npoly] // 2)[:, None], e[npoly:].copy()
    nz = t != 0
    last = t.shape[0] - 1 - np.argmax(nz[::-1], axis=0)
    sign = np.where(shape.random(t.shape) < 0.5, -1, 1)
    sign[last, np.arange(n)] = 1
    k = np.where(nz.any(axis=0), shape.integers(0, 2, n), 0)
    l1 = np.abs(p).sum(0) + np.abs(t).sum(0)
    c = np.where(rng.random(n) < 0.5, -1.0, 1.0) * 10.0 ** (rng.random(n) - l1 / d)
    return _pseries(rng, p, t * sign, k, c)


def _host(case, seed):
    """The operands of a case, in host memory: a list of (f, g).  The exponents belong to the case, as the supports of
    a user's problem do; the coefficients and the order of the terms to the seed."""
    values = sorted((k, x) for k, x in case.items() if k != "name")
    shape, rng = np.random.default_rng(zlib.crc32(repr(values).encode())), np.random.default_rng([int(seed), 1004, 4548])
    fam = case["family"]
    if fam == "total":
        if case["coef"] == "power":
            weight = 2 * rng.integers(0, 5, case["v"]) + 1
            return [(_power(rng, weight, case["df"], 0), _power(rng, weight, case["dg"], 1))]
        return [tuple(_total(shape, rng, case["v"], case[d], case["keep"], case["coef"], case["cmax"]) for d in ("df", "dg"))]
    if fam == "weighted":
        e = _simplex(5, case["d"])
        return [tuple(_poly(rng, e * np.array(w)[:, None], _integers(rng, e.shape[1], case["cmax"]))
                      for w in ((1, 1, 2, 3, 5), (5, 3, 2, 1, 1)))]
    if fam == "laurent":
        return [tuple(_laurent(shape, rng, case["v"], case[n], case["half"], case["coef"]) for n in ("nf", "ng"))]
    if fam == "poisson":
        return [tuple(_series(shape, rng, case[n], case["npoly"], case["ntrig"], case["prange"], case["trange"]) for n in ("nf", "ng"))]
    return [tuple(_uneven(shape, rng, v, k % 2 == 1, case["most"]) for _ in "fg")
            for k, v in enumerate(shape.integers(2, 7, case["count"]).tolist())]


def _codec_box(case):
    lo = np.array([-(case["width"] // 2) + k for k in range(case["v"])], np.int32)
    return lo, lo + case["width"] - 1


def _codec_exps(case, seed):
    lo, hi = _codec_box(case)
    rng = np.random.default_rng([int(seed), 77])
    return np.stack([rng.integers(a, b + 1, case["n"]) for a, b in zip(lo, hi)]).astype(np.int32)


def _gpu(p):
    return SimpleNamespace(**{k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in vars(p).items()})


# A prepared batch owns its results: the newest ones are kept, so that outputs stay readable after their state is gone.
_prepared = deque(maxlen=16)


def prepare(case, seed):
    fam = case["family"]
    if fam == "codec":
        lo, hi = _codec_box(case)
        return {"family": fam, "exps": torch.from_numpy(_codec_exps(case, seed)).cuda(), "lo": lo, "hi": hi}
    pairs = [(_gpu(f), _gpu(g)) for f, g in _host(case, seed)]
    if fam == "batch":
        return {"family": fam, "pairs": pairs}   # the results live in the library's context, until its next batch
    if fam == "graph":
        batch = kron.PreparedBatch(pairs)
        _prepared.append(batch)
        return {"family": fam, "batch": batch}
    opts = {"trunc_degree": case["trunc"]} if case.get("trunc", -1) >= 0 else {}
    return {"family": fam, "f": pairs[0][0], "g": pairs[0][1], "opts": opts}


def run(state):
    fam = state["family"]
    if fam == "codec":
        codes = kron.kron_encode(state["exps"], state["lo"], state["hi"])
        return [codes, kron.kron_decode(codes, state["lo"], state["hi"])]
    if fam in ("batch", "graph"):
        if fam == "batch":
            res = kron.kron_mul_batch(state["pairs"])
        else:
            state["batch"].launch()
            torch.cuda.current_stream().synchronize()   # the results' statuses are read after the launch's stream is done
            res = state["batch"].results()
        return [np.array([(r["status"], r["path"], r["nterms"]) for r in res])] + \
            [[r[k] for k in ("exps", "trig", "kind", "coef") if k in r] for r in res]
    f, g = state["f"], state["g"]
    if fam == "poisson":
        return list(kron.poisson_mul(f, g)[:4])
    exps, coef, _, (lo, hi) = kron.poly_mul(f.exps, f.coef, g.exps, g.coef, **state["opts"])
    return [exps, coef, lo, hi]


# ---------------------------------------------------------------------------- the same in 64 bits, plainly

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _sum_by_key(batches, krange):
    """Sorted distinct keys and the sums of their values, from batches of (keys, values)."""
    if krange <= 1 << 28:
        acc = live = None
        for k, v in batches():
            if acc is None:
                acc = torch.zeros(krange, dtype=v.dtype, device=k.device)
            acc.index_add_(0, k, v)
        live = (acc != 0).nonzero().flatten()
        return live, acc[live]
    got = list(batches())
    keys, vals = torch.cat([k for k, _ in got]), torch.cat([v for _, v in got])
    keys, at = torch.unique(keys, return_inverse=True)
    acc = torch.zeros(keys.numel(), dtype=vals.dtype, device=keys.device).index_add_(0, at, vals)
    live = acc != 0
    return keys[live], acc[live]


def _weights(w):
    c = [1]
    for x in w:
        c.append(c[-1] * int(x))
    return c[:-1], c[-1]


def _digits(key, c, w, lo):
    return torch.stack([(key // a) % int(b) + int(o) for a, b, o in zip(c, w, lo)]).to(torch.int32)


def _exact_poly(f, g, trunc=-1):
    dev = _device()
    fe, ge = (torch.from_numpy(p.exps).to(dev).long() for p in (f, g))
    fc, gc = (torch.from_numpy(np.ascontiguousarray(p.coef)).to(dev) for p in (f, g))
    flo, glo = fe.amin(1), ge.amin(1)
    lo, hi = (flo + glo).tolist(), (fe.amax(1) + ge.amax(1)).tolist()
    if trunc >= 0:   # degree in the place of the last variable, as the most significant digit
        fe, ge = (torch.cat([e[:-1], e.sum(0, keepdim=True)]) for e in (fe, ge))
        flo, glo = fe.amin(1), ge.amin(1)
    low, high = (flo + glo).tolist(), (fe.amax(1) + ge.amax(1)).tolist()
    w = [b - a + 1 for a, b in zip(low, high)]
    if trunc >= 0:
        w[-1] = min(w[-1], trunc - low[-1] + 1)
    c, krange = _weights(w)
    ct = torch.tensor(c, device=dev)[:, None]
    fk, gk = ((fe - flo[:, None]) * ct).sum(0), ((ge - glo[:, None]) * ct).sum(0)
    step = max(1, (1 << 24) // gk.numel())

    def batches():
        for a in range(0, fk.numel(), step):
            k = (fk[a:a + step, None] + gk[None, :]).flatten()
            v = (fc[a:a + step, None] * gc[None, :]).flatten()
            yield (k, v) if trunc < 0 else (k[k < krange], v[k < krange])
    key, val = _sum_by_key(batches, krange)
    e = _digits(key, c, w, low)
    if trunc >= 0:
        e[-1] -= e[:-1].sum(0).to(torch.int32)
    return [e, val, np.array(lo, np.int32), np.array(hi, np.int32)]


def _exact_poisson(f, g):
    dev = _device()
    t = {n: [torch.from_numpy(np.ascontiguousarray(getattr(p, n))).to(dev) for p in (f, g)] for n in ("exps", "trig", "kind", "coef")}
    fe, ge = (x.long() for x in t["exps"])
    ft, gt = (x.long() for x in t["trig"])
    fk, gk = (x.long() for x in t["kind"])
    fc, gc = t["coef"]
    plo = (fe.amin(1) + ge.amin(1)).tolist()
    pw = (fe.amax(1) + ge.amax(1) - fe.amin(1) - ge.amin(1) + 1).tolist()
    r = (ft.abs().amax(1) + gt.abs().amax(1)).tolist()
    pc, wp = _weights(pw)
    tc, wt = _weights([2 * x + 1 for x in r])
    half = (wt - 1) // 2 + 1
    col = lambda c: torch.tensor(c, device=dev)[:, None]  # noqa: E731
    fp, gp = ((e - e.amin(1, keepdim=True)).mul(col(pc)).sum(0) for e in (fe, ge))
    fu, gu = ((x * col(tc)).sum(0) for x in (ft, gt))
    step = max(1, (1 << 23) // gp.numel())

    def batches():
        for a in range(0, fp.numel(), step):
            s = slice(a, a + step)
            kf, kg = fk[s, None], gk[None, :]
            kd, p = kf ^ kg, fp[s, None] + gp[None, :]
            v = fc[s, None] * 0.5 * gc[None, :]
            for tt, neg in ((fu[s, None] + gu[None, :], (kf & kg) == 1), (fu[s, None] - gu[None, :], (kf == 0) & (kg == 1))):
                x = torch.where(neg ^ ((tt < 0) & (kd == 1)), -v, v)
                ok = ~((tt == 0) & (kd == 1))
                yield (((kd * half + tt.abs()) * wp + p)[ok], x[ok])
    key, val = _sum_by_key(batches, 2 * half * wp)
    kind, rest = key // (half * wp), key % (half * wp)
    trig = _digits(rest // wp + (half - 1), tc, [2 * x + 1 for x in r], [-x for x in r])
    return [_digits(rest % wp, pc, pw, plo), trig, kind.to(torch.uint8), val]


def exact(case, seed):
    if case["family"] == "codec":
        e = _codec_exps(case, seed)
        lo, hi = _codec_box(case)
        c, _ = _weights(hi - lo + 1)
        return [((e.astype(np.int64) - lo[:, None]) * np.array(c)[:, None]).sum(0), e]
    pairs = _host(case, seed)
    if case["family"] in ("batch", "graph"):
        return [None] + [_exact_poisson(f, g) if hasattr(f, "trig") else _exact_poly(f, g)[:2] for f, g in pairs]
    f, g = pairs[0]
    return _exact_poisson(f, g) if case["family"] == "poisson" else _exact_poly(f, g, case.get("trunc", -1))


# ---------------------------------------------------------------------------- what a pass cannot do without

def _expected(cells, hits):
    """Expected number of distinct cells that `hits` uniform draws reach."""
    return cells * -math.expm1(-hits / cells)


def _product_work(nf, ng, np_, nt, nout, pairs=None):
    term = 4 * (np_ + nt) + 8 + (1 if nt else 0)
    return {"bytes": int(term * (nf + ng + nout)), "flops": int((3 if nt else 2) * (nf * ng if pairs is None else pairs))}


def work(case):
    fam = case["family"]
    if fam == "codec":   # exponents read, codes written and read, exponents written
        return {"bytes": case["n"] * (8 * case["v"] + 16), "flops": 4 * case["n"] * case["v"]}
    if fam == "total":
        v, df, dg, keep, n = case["v"], case["df"], case["dg"], case["keep"], case["trunc"]
        by = lambda d: math.comb(v + d - 1, v - 1) * keep  # noqa: E731  (terms of degree d)
        kept = sum(by(a) * by(b) for a in range(df + 1) for b in range(dg + 1) if n < 0 or a + b <= n)
        return _product_work(math.comb(v + df, v) * keep, math.comb(v + dg, v) * keep, v, 0,
                             math.comb(v + (df + dg if n < 0 else min(n, df + dg)), v), kept)
    if fam == "weighted":
        n = math.comb(5 + case["d"], 5)   # output terms: about 0.15 a pair at degree 12, more at lower degrees
        return _product_work(n, n, 5, 0, n * n * min(1.0, 0.152 * (12 / case["d"]) ** 1.5))
    if fam == "laurent":
        return _product_work(case["nf"], case["ng"], case["v"], 0, case["nf"] * case["ng"])
    if fam == "poisson":
        box = (4 * case["prange"] + 1) ** case["npoly"] * (4 * case["trange"] + 1) ** case["ntrig"]
        cells = box * 0.4   # sums of two uniform draws reach the edges of the box rarely
        return _product_work(case["nf"], case["ng"], case["npoly"], case["ntrig"], _expected(cells, 2 * case["nf"] * case["ng"]))
    b = f = 0
    for x, y in _host(case, 1):
        nt = x.trig.shape[0] if hasattr(x, "trig") else 0
        w = _product_work(x.coef.size, y.coef.size, x.exps.shape[0], nt, min(x.coef.size * y.coef.size, 20 * (x.coef.size + y.coef.size)))
        b, f = b + w["bytes"], f + w["flops"]
    return {"bytes": b, "flops": f}
