"""Windowed accumulation of highly sparse products, at the sizes where it can go
wrong: single terms, windows addressed directly, offsets of 64 bits, keys that
cluster, tables that fill up and are halved, runs of windows formed in one walk,
series without a polynomial part, with a zero multiplier or of one kind only.
Small products against the oracle; large ones against the table in device memory
(asked for by its size), bit for bit for int64."""
import numpy as np
import pytest

import oracle
from tests.gpu_compare import assert_poly_close, assert_poly_equal, assert_pseries_close, to_np
from workloads import Poly, PSeries, Rng, dense_total_degree, mp_sparse, poisson_random, random_poly, random_pseries

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kron():
    import paper_1004_4548_gb300 as k
    k.load()
    return k


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def poly(k, f, g, **opts):
    return k.poly_mul(dev(f.exps), dev(f.coef), dev(g.exps), dev(g.coef), path=k.KR_PATH_HASH, **opts)


def pseries(k, f, g, **opts):
    up = [PSeries(*(dev(getattr(s, n)) for n in ("exps", "trig", "kind", "coef"))) for s in (f, g)]
    return k.poisson_mul(*up, path=k.KR_PATH_HASH, **opts)


def clustered(n, seed, step):
    """Clusters of consecutive exponents, far apart: x in [0, 24) + step * (0 .. 9), and one more variable."""
    rng = Rng(seed)
    grid = np.stack(np.meshgrid(np.arange(24), np.arange(10), np.arange(3), indexing="ij"), -1).reshape(-1, 3)
    rows = grid[rng.perm(grid.shape[0])[:n]]
    e = np.stack([rows[:, 0] + step * rows[:, 1], rows[:, 2]]).astype(np.int32)
    return Poly(np.ascontiguousarray(e), rng.nonzero_ints(-1000, 1000, n))


POLY = {
    "one_by_one": lambda: (random_poly(3, 1, -5, 5, 1), random_poly(3, 1, -5, 5, 2)),
    "one_by_many": lambda: (random_poly(4, 1, -50, 50, 3), random_poly(4, 33, -50, 50, 4)),
    "warp_edge": lambda: (random_poly(4, 32, -50, 50, 5), random_poly(4, 31, -50, 50, 6)),
    "swapped": lambda: (random_poly(5, 301, -30, 30, 7), random_poly(5, 97, -30, 30, 8)),
    "offsets_64": lambda: (random_poly(3, 260, -100000, 100000, 9), random_poly(3, 307, -100000, 100000, 10)),
    "clustered": lambda: (clustered(700, 11, 1 << 14), clustered(650, 12, 1 << 18)),
    "clustered_64": lambda: (clustered(700, 13, 1 << 26), clustered(650, 14, 1 << 20)),
    "direct": lambda: (dense_total_degree(3, 13, -100, 100, 15), dense_total_degree(3, 12, -100, 100, 16)),
    "shared_keys": lambda: (mp_sparse("f", 6, -1000, 1000, 17), mp_sparse("g", 6, -1000, 1000, 18)),
    "cancelling": lambda: (Poly(np.array([[0, 90000], [90000, 0]], np.int32), np.array([1, -1], np.int64)),
                           Poly(np.array([[0, 90000], [90000, 0]], np.int32), np.array([1, 1], np.int64))),
}


@pytest.mark.parametrize("case", sorted(POLY))
def test_polynomials(kron, case):
    f, g = POLY[case]()
    ex, cf, _, _ = poly(kron, f, g)
    assert_poly_equal(ex, cf, oracle.poly_mul(f, g), case)
    ff, gf = Poly(f.exps, f.coef.astype(np.float64)), Poly(g.exps, g.coef.astype(np.float64))
    ex, cf, _, _ = poly(kron, ff, gf)
    assert_poly_close(ex, cf, oracle.poly_mul(ff, gf, keep_zero=True), 1e-12, case)


def one_kind(p, kind):
    """The series with every term of one kind (terms that would repeat or vanish dropped)."""
    keep = p.kind == 0 if kind == 0 else p.kind == 1
    return PSeries(np.ascontiguousarray(p.exps[:, keep]), np.ascontiguousarray(p.trig[:, keep]), p.kind[keep], p.coef[keep])


def with_zero_multipliers(p):
    """Polynomial terms (zero multiplier vector) beside the series' own."""
    m = 40
    e = random_poly(p.npoly, m, -4, 4, 99).exps
    e = e[:, :m]
    t = np.zeros((p.ntrig, e.shape[1]), np.int32)
    keep = (p.trig != 0).any(axis=0)
    return PSeries(np.ascontiguousarray(np.concatenate([p.exps[:, keep], e], axis=1)),
                   np.ascontiguousarray(np.concatenate([p.trig[:, keep], t], axis=1)),
                   np.concatenate([p.kind[keep], np.zeros(e.shape[1], np.uint8)]),
                   np.concatenate([p.coef[keep], np.linspace(0.5, 1.5, e.shape[1])]))


PSER = {
    "one_by_one": lambda: (random_pseries(2, 2, 1, 3, 4, 1), random_pseries(2, 2, 1, 3, 4, 2)),
    "no_polynomial": lambda: (random_pseries(0, 4, 150, 0, 8, 3), random_pseries(0, 4, 210, 0, 8, 4)),
    "one_multiplier": lambda: (random_pseries(2, 1, 300, 9, 40, 5), random_pseries(2, 1, 170, 9, 40, 6)),
    "cosines": lambda: (one_kind(random_pseries(2, 3, 200, 4, 6, 7), 0), one_kind(random_pseries(2, 3, 150, 4, 6, 8), 0)),
    "sines": lambda: (one_kind(random_pseries(2, 3, 200, 4, 6, 9), 1), one_kind(random_pseries(2, 3, 150, 4, 6, 10), 1)),
    "sine_cosine": lambda: (one_kind(random_pseries(2, 3, 200, 4, 6, 9), 1), one_kind(random_pseries(2, 3, 150, 4, 6, 8), 0)),
    "zero_multipliers": lambda: (with_zero_multipliers(random_pseries(2, 2, 120, 4, 6, 11)),
                                 with_zero_multipliers(random_pseries(2, 2, 160, 4, 6, 12))),
    "same_operand": lambda: (random_pseries(2, 3, 140, 4, 6, 13),) * 2,
    "offsets_64": lambda: (random_pseries(2, 4, 200, 500, 100, 14), random_pseries(2, 4, 130, 500, 100, 15)),
}


@pytest.mark.parametrize("case", sorted(PSER))
def test_series(kron, case):
    f, g = PSER[case]()
    assert_pseries_close(pseries(kron, f, g), oracle.poisson_mul(f, g, keep_zero=True), 1e-12, case)


def test_key_windows_join_up(kron):
    f, g = random_poly(4, 200, -40, 40, 21), random_poly(4, 310, -40, 40, 22)
    ex, cf, codes, _ = (to_np(x) if i < 3 else x for i, x in enumerate(poly(kron, f, g, want_codes=True)))
    cuts = [0, int(codes[1]), int(codes[cf.size // 3]), int(codes[-1]), 0]
    parts = [poly(kron, f, g, code_lo=a, code_hi=b) for a, b in zip(cuts[:-1], cuts[1:])]
    assert np.array_equal(np.concatenate([to_np(p[0]) for p in parts], axis=1), ex)
    assert np.array_equal(np.concatenate([to_np(p[1]) for p in parts]), cf)


def test_batch_of_every_form(kron):
    """Dense, 32-bit and 64-bit windows, table and Poisson products, and a failing one, in one call."""
    jobs = [(random_poly(2, 50, 0, 12, 31), random_poly(2, 60, 0, 12, 32)),
            POLY["offsets_64"](), POLY["swapped"](), POLY["clustered"](),
            (random_poly(3, 40, -9, 9, 33), random_poly(3, 40, -9, 9, 34)), POLY["shared_keys"]()]
    dup = random_poly(3, 40, -90, 90, 35)
    dup.exps[:, 1] = dup.exps[:, 0]
    jobs.append((dup, random_poly(3, 40, -90, 90, 36)))
    opts = [{}] * len(jobs)
    opts[4] = {"path": kron.KR_PATH_HASH, "table_slots": 1 << 14}
    series = [PSER["no_polynomial"](), PSER["zero_multipliers"]()]
    up = lambda p: type(p)(*(dev(x) for x in vars(p).values()))  # noqa: E731
    res = kron.kron_mul_batch([(up(f), up(g)) for f, g in jobs + series], opts=opts + [{}, {"path": kron.KR_PATH_HASH}])
    assert res[6]["status"] == kron.KR_ERR_DUP
    for i, (f, g) in enumerate(jobs):
        if i != 6:
            assert res[i]["status"] == 0
            assert_poly_equal(res[i]["exps"], res[i]["coef"], oracle.poly_mul(f, g), f"job {i}")
    for r, (f, g) in zip(res[len(jobs):], series):
        assert_pseries_close([r[k] for k in ("exps", "trig", "kind", "coef")], oracle.poisson_mul(f, g, keep_zero=True))


def test_host_outputs_and_capacity(kron):
    f, g = random_poly(4, 120, -40, 40, 41), random_poly(4, 90, -40, 40, 42)
    r = oracle.poly_mul(f, g)
    for cap in (1, r.coef.shape[0] - 1, r.coef.shape[0], 2 * r.coef.shape[0]):
        for host in (False, True):
            ex, cf, _, _ = poly(kron, f, g, capacity=cap, host_out=host)
            assert_poly_equal(ex, cf, r, f"capacity {cap}, host {host}")


@pytest.mark.parametrize("case", ["shared_keys", "own_keys"])
def test_large_polynomials_equal_the_table(kron, case):
    """Runs of several windows (keys shared), and runs formed in one walk."""
    if case == "shared_keys":
        f, g = mp_sparse("f", 10, -1000, 1000, 51), mp_sparse("g", 10, -1000, 1000, 52)
    else:
        f, g = random_poly(5, 5200, -30, 30, 53), random_poly(5, 4100, -30, 30, 54)
    a = [to_np(x) for x in poly(kron, f, g)[:2]]
    b = [to_np(x) for x in poly(kron, f, g, table_slots=1 << 25)[:2]]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def test_large_series_equal_the_table(kron):
    """Positive and equal coefficients: sums of signed equal values are exact in
    float64 whatever their order, so both ways must agree to the last bit."""
    f, g = poisson_random(3800, 3, 4, 4, 8, 55, mag="unit"), poisson_random(2900, 3, 4, 4, 8, 56, mag="unit")
    f.coef[:] = 2.0
    g.coef[:] = 3.0
    a = [to_np(x) for x in pseries(kron, f, g)[:4]]
    b = [to_np(x) for x in pseries(kron, f, g, table_slots=1 << 26)[:4]]
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


BOXES = {   # widths: least significant first
    "ones": [1, 1, 1],
    "one_inside": [7, 1, 5],
    "powers_of_two": [1 << 16, 2, 1 << 15, 1 << 16, 1 << 15],           # codes up to 2^63 - 1 (less one value of the last)
    "whole_int": [(1 << 31) - 1],
    "whole_ints": [(1 << 31) - 1, (1 << 31) - 1, 2],
    "narrow_wide": [3, (1 << 31) - 1, (1 << 30) - 1],
    "at_32_bits": [65537, 65535, 3],
    "many": [2, 3, 5, 7, 11, 13, 17, 19],
}


@pytest.mark.parametrize("box", sorted(BOXES))
def test_codes_to_digits(kron, box):
    """Division by the reciprocal: the ends of each digit, codes either side of
    2^32, the last code of the box.  Whole numbers: every digit is exact."""
    w = BOXES[box]
    if box == "powers_of_two":
        w = w[:-1] + [(1 << 15) - 1]
    lo = [-(x // 2) for x in w]
    hi = [a + x - 1 for a, x in zip(lo, w)]
    rng = np.random.default_rng(71)
    W = 1
    codes = {0}
    for x in w:
        codes |= {W - 1, W, W * (x - 1), W * x - 1}
        W *= x
    assert W < 1 << 63
    codes |= {W - 1, (1 << 32) - 1, 1 << 32, (1 << 32) + 1} | {int(c) for c in rng.integers(0, W, 500)}
    codes = sorted(c for c in codes if c < W)
    want = np.zeros((len(w), len(codes)), np.int32)
    for i, c in enumerate(codes):
        for k, x in enumerate(w):
            want[k, i] = c % x + lo[k]
            c //= x
    assert np.array_equal(to_np(kron.kron_decode(dev(np.array(codes, np.int64)), lo, hi)), want)
    assert np.array_equal(to_np(kron.kron_encode(dev(want), lo, hi)), np.array(codes, np.int64))
    # and as the digits of a product: one term by every other, the box moved
    one = Poly(np.zeros((len(w), 1), np.int32), np.array([3], np.int64))
    ex, cf, _, _ = poly(kron, one, Poly(want, np.arange(1, len(codes) + 1, dtype=np.int64)))
    assert np.array_equal(to_np(ex), want) and np.array_equal(to_np(cf), 3 * np.arange(1, len(codes) + 1))


@pytest.mark.parametrize("n", [2, 3, 31, 33, 63, 65, 129, 511, 512, 513, 514, 1025, 4095, 4097, 6188, 9001, 16383, 16384])
def test_terms_in_any_order(kron, n):
    """Operand ordering at the edges of its tiles: random and reversed orders,
    one term by all (int64: exact), and a duplicate across the whole operand."""
    rng = np.random.default_rng(n)
    x = np.sort(rng.choice(40 * n + 100, n, replace=False)).astype(np.int32)
    e = np.stack([x, (x % 7).astype(np.int32) * 1000003])      # ascending in the second variable, then the first
    coef = np.arange(1, n + 1, dtype=np.int64)
    one = Poly(np.array([[5], [-3]], np.int32), np.array([-2], np.int64))
    by_code = np.lexsort((e[0], e[1]))
    for order in (rng.permutation(n), by_code[::-1]):
        ex, cf, _, _ = poly(kron, one, Poly(np.ascontiguousarray(e[:, order]), coef[order]))
        assert np.array_equal(to_np(ex), e[:, by_code] + np.array([[5], [-3]]))
        assert np.array_equal(to_np(cf), -2 * coef[by_code])
    e[:, 0] = e[:, -1]
    with pytest.raises(kron.KronError) as err:
        poly(kron, one, Poly(np.ascontiguousarray(e), coef))
    assert err.value.status == kron.KR_ERR_DUP


def test_runs_across_regions(kron):
    """Keys shared in one part of the range and distinct in the others, so that runs of both kinds meet."""
    rng = Rng(81)

    def both(which, seed):
        a, b = mp_sparse(which, 9, -1000, 1000, seed), random_poly(5, 2700, 0, 45, seed + 1)
        e = np.concatenate([a.exps, b.exps + np.array([[0], [0], [0], [0], [200]], np.int32)], axis=1)
        p = rng.perm(e.shape[1])
        return Poly(np.ascontiguousarray(e[:, p]), np.concatenate([a.coef, b.coef])[p])

    f, g = both("f", 82), both("g", 84)
    a = [to_np(x) for x in poly(kron, f, g)[:2]]
    b = [to_np(x) for x in poly(kron, f, g, table_slots=1 << 26)[:2]]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
