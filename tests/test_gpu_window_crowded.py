"""Windowed products whose keys crowd into a small part of a range that a few far terms made wide: cuts by sampled
quantiles, and the table where the keys are too close to be divided.  Results against the oracle; times against the
table in device memory (asked for by its size) on the same operands."""
import time

import numpy as np
import pytest

import oracle
from tests.gpu_compare import assert_poly_close, assert_poly_equal, assert_pseries_close, to_np
from tests.test_gpu_window import dev, poly, pseries
from workloads import Poly, PSeries, Rng, dense_total_degree, random_poly, random_pseries

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kron():
    import paper_1004_4548_gb300 as k
    k.load()
    return k


def far(p, *where):
    """The polynomial and one monomial of the last variable for each exponent given."""
    e = np.zeros((p.exps.shape[0], len(where)), np.int32)
    e[-1] = where
    return Poly(np.ascontiguousarray(np.concatenate([p.exps, e], axis=1)),
                np.concatenate([p.coef, np.arange(7, 7 + len(where), dtype=p.coef.dtype)]))


def line(n, seed):
    return Poly(np.arange(n, dtype=np.int32)[None, :], Rng(seed).nonzero_ints(-1000, 1000, n))


def stages(k, f, g):
    ctx = k.Context()
    ctx.set_profiling(True)
    poly(k, f, g, ctx=ctx)
    names = {n for n, _ in ctx.stages()}
    ctx.close()
    return names


def far_series(p, e):
    """The series and one term of exponent e in the first polynomial variable."""
    x = np.zeros((p.npoly, 1), np.int32)
    x[0] = e
    t = np.zeros((p.ntrig, 1), np.int32)
    t[-1] = 3
    return PSeries(np.ascontiguousarray(np.concatenate([p.exps, x], axis=1)),
                   np.ascontiguousarray(np.concatenate([p.trig, t], axis=1)),
                   np.concatenate([p.kind, np.ones(1, np.uint8)]), np.concatenate([p.coef, [0.75]]))


POLY = {
    "offsets_32": lambda: (far(dense_total_degree(4, 8, -100, 100, 1), 1 << 11), far(dense_total_degree(4, 7, -100, 100, 2), 1 << 10)),
    "offsets_64": lambda: (far(dense_total_degree(4, 8, -100, 100, 3), 10 ** 9), far(dense_total_degree(4, 7, -100, 100, 4), 10 ** 9)),
    "both_ends": lambda: (far(dense_total_degree(3, 12, -100, 100, 5), -10 ** 8, 10 ** 8), far(dense_total_degree(3, 11, -100, 100, 6), 10 ** 7)),
    # 32-bit offsets and a gap of more than 2^32 keys
    "wide_gap": lambda: (far(dense_total_degree(4, 10, -100, 100, 13), 500000), far(dense_total_degree(4, 10, -100, 100, 14), 480000)),
    "distinct": lambda: (far(random_poly(4, 600, -30, 30, 7), 10 ** 7), far(random_poly(4, 500, -30, 30, 8), -10 ** 7)),
    "a_line": lambda: (far(line(3000, 9), 10 ** 9), far(line(2990, 10), 10 ** 9)),              # 6000 keys: the table
    "wide_line": lambda: (far(line(400, 11), 10 ** 9), far(line(390, 12), 10 ** 9)),            # too few pairs for the table
}


@pytest.mark.parametrize("case", sorted(POLY))
def test_polynomials(kron, case):
    f, g = POLY[case]()
    r = oracle.poly_mul(f, g)
    for kw in ({}, {"host_out": True}, {"capacity": 1}):
        ex, cf, _, _ = poly(kron, f, g, **kw)
        assert_poly_equal(ex, cf, r, f"{case} {kw}")
    assert ("hll" in stages(kron, f, g)) == (case == "a_line")   # a table's size is estimated first
    ff, gf = Poly(f.exps, f.coef.astype(np.float64)), Poly(g.exps, g.coef.astype(np.float64))
    ex, cf, _, _ = poly(kron, ff, gf)
    assert_poly_close(ex, cf, oracle.poly_mul(ff, gf, keep_zero=True), 1e-12, case)


@pytest.mark.parametrize("e", [1 << 9, 10 ** 6])
def test_series(kron, e):
    f, g = far_series(random_pseries(2, 2, 700, 4, 6, 21), e), far_series(random_pseries(2, 2, 650, 4, 6, 22), e)
    assert_pseries_close(pseries(kron, f, g), oracle.poisson_mul(f, g, keep_zero=True), 1e-12)


def test_key_windows_and_truncation(kron):
    f, g = POLY["offsets_64"]()
    ex, cf, codes, _ = (to_np(x) if i < 3 else x for i, x in enumerate(poly(kron, f, g, want_codes=True)))
    cuts = [0, int(codes[cf.size // 5]), int(codes[cf.size // 2]), 0]
    parts = [poly(kron, f, g, code_lo=a, code_hi=b) for a, b in zip(cuts[:-1], cuts[1:])]
    assert np.array_equal(np.concatenate([to_np(p[0]) for p in parts], axis=1), ex)
    assert np.array_equal(np.concatenate([to_np(p[1]) for p in parts]), cf)
    keep = ex.sum(axis=0) <= 10 ** 9   # drops the far square
    t = [to_np(x) for x in poly(kron, f, g, trunc_degree=10 ** 9)[:2]]
    key = lambda e, c: sorted(zip(map(tuple, e.T.tolist()), c.tolist()))  # noqa: E731
    assert key(*t) == key(ex[:, keep], cf[keep])


def test_batches(kron):
    """A product that goes to the table beside others, in one call and replayed."""
    import torch
    jobs = [POLY[c]() for c in ("distinct", "a_line", "offsets_32", "offsets_64")] + \
        [(random_poly(2, 50, 0, 12, 31), random_poly(2, 60, 0, 12, 32))]
    want = [oracle.poly_mul(f, g) for f, g in jobs]
    up = [tuple(Poly(dev(p.exps), dev(p.coef)) for p in fg) for fg in jobs]
    pb = kron.PreparedBatch(up)
    pb.launch()
    torch.cuda.synchronize()
    for res in (kron.kron_mul_batch(up), pb.first_results(), pb.results()):
        for x, r in zip(res, want):
            assert x["status"] == 0
            assert_poly_equal(x["exps"], x["coef"], r)
    pb.close()


@pytest.mark.parametrize("case", ["simplex", "distinct"])
def test_not_slower_than_the_table(kron, case):
    """Cut by equal bins these took 27 and 390 times the table's time."""
    import torch
    f, g = {"simplex": lambda: (far(dense_total_degree(4, 12, -100, 100, 41), 10 ** 9),) * 2,
            "distinct": lambda: (far(random_poly(4, 3000, 0, 39, 42), 10 ** 9),) * 2}[case]()
    D = [dev(x) for x in (f.exps, f.coef, g.exps, g.coef)]

    def best(**kw):
        t = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            kron.poly_mul(*D, path=kron.KR_PATH_HASH, **kw)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t[1:])

    windows, table = best(), best(table_slots=1 << (23 if case == "distinct" else 16))
    assert windows < 3.0 * table, f"{case}: {windows * 1e6:.0f} us, the table {table * 1e6:.0f}"
