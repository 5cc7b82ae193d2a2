"""Windowed products run again: replays of batches that hold no other kind, and
phase repetitions after a limit was met (lowered limits, so that small products
meet them)."""
import numpy as np
import pytest

import oracle
from tests.gpu_compare import assert_poly_equal, assert_pseries_close, to_np
from tests.test_gpu_window import POLY, PSER, dev, poly, pseries
from tests.test_gpu_window_crowded import far
from workloads import dense_total_degree, random_poly

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kron():
    import paper_1004_4548_gb300 as k
    k.load()
    return k


@pytest.fixture
def limited(kron):
    """A context whose limits a test lowers."""
    ctx = kron.Context()
    yield lambda which, value: kron.kr_selftest_limit(ctx, which, value) or ctx
    ctx.close()


def up(p):
    return type(p)(*(dev(x.copy()) for x in vars(p).values()))


PREPARED = {
    "one_32": ([POLY["swapped"]], []),
    "one_64": ([POLY["offsets_64"]], []),
    "one_series": ([], [PSER["no_polynomial"]]),
    "several": ([POLY["swapped"], POLY["offsets_64"], POLY["clustered"]], [PSER["offsets_64"], PSER["cosines"]]),
}


@pytest.mark.parametrize("case", sorted(PREPARED))
def test_prepared_batch_of_windows_alone(kron, case):
    import torch
    polys, series = ([c() for c in cs] for cs in PREPARED[case])
    pb = kron.PreparedBatch([(up(f), up(g)) for f, g in polys + series], opts={"path": kron.KR_PATH_HASH})
    want = [r["nterms"] for r in pb.first_results()]
    for _ in range(3):
        pb.launch()
        torch.cuda.synchronize()
        res = pb.results()
        assert [r["status"] for r in res] == [0] * len(res) and [r["nterms"] for r in res] == want
        for r, (f, g) in zip(res, polys):
            assert_poly_equal(r["exps"], r["coef"], oracle.poly_mul(f, g), case)
        for r, (f, g) in zip(res[len(polys):], series):
            assert_pseries_close([r[k] for k in ("exps", "trig", "kind", "coef")], oracle.poisson_mul(f, g, keep_zero=True))
    pb.close()


@pytest.mark.parametrize("case", ["swapped", "offsets_64", "dense"])
def test_replay_keeps_the_statuses_it_finds(kron, case):
    """Exponents changed in place to a repeated term: the replay reports it, and the next one, mended, does not."""
    import torch
    f, g = POLY[case]() if case != "dense" else (random_poly(2, 50, 0, 12, 31), random_poly(2, 60, 0, 12, 32))
    F, G = up(f), up(g)
    pb = kron.PreparedBatch([(F, G)])
    whole = F.exps.clone()
    for exps, status in ((whole, 0), (torch.cat([whole[:, 1:2], whole[:, 1:]], 1), kron.KR_ERR_DUP), (whole, 0)):
        F.exps.copy_(exps)
        pb.launch()
        torch.cuda.synchronize()
        r = pb.results()[0]
        assert r["status"] == status
        if status == 0:
            assert_poly_equal(r["exps"], r["coef"], oracle.poly_mul(f, g), case)
    pb.close()


def test_short_estimate_is_repeated(kron, limited):
    """The room comes from an estimate that is always short: every product is repeated with full room."""
    limited(kron.KR_LIMIT_WINDOW_BYTES, 1.0)
    ctx = limited(kron.KR_LIMIT_WINDOW_ROOM, 0.5)
    for case in ("offsets_64", "swapped", "one_by_many"):
        f, g = POLY[case]()
        r = oracle.poly_mul(f, g)
        for host in (False, True):
            ex, cf, _, _ = poly(kron, f, g, ctx=ctx, host_out=host)
            assert_poly_equal(ex, cf, r, case)
    f, g = PSER["offsets_64"]()
    assert_pseries_close(pseries(kron, f, g, ctx=ctx), oracle.poisson_mul(f, g, keep_zero=True))
    jobs = [POLY["offsets_64"](), POLY["swapped"](), (random_poly(2, 50, 0, 12, 31), random_poly(2, 60, 0, 12, 32))]
    for n in (2, 3):   # windows alone, and beside a dense product
        res = kron.kron_mul_batch([(up(f), up(g)) for f, g in jobs[:n]], ctx=ctx)
        for x, (f, g) in zip(res, jobs):
            assert x["status"] == 0
            assert_poly_equal(x["exps"], x["coef"], oracle.poly_mul(f, g))


def test_estimated_room(kron, limited):
    """An estimate that suffices: no repetition, the same terms."""
    ctx = limited(kron.KR_LIMIT_WINDOW_BYTES, 1.0)
    f, g = POLY["shared_keys"]()
    ex, cf, _, _ = poly(kron, f, g, ctx=ctx)
    assert_poly_equal(ex, cf, oracle.poly_mul(f, g))
    assert np.array_equal(to_np(cf), to_np(poly(kron, f, g)[1]))


def test_pieces_run_out(kron, limited):
    """A product whose windows put down more pieces than there is room for goes through the table."""
    ctx = limited(kron.KR_LIMIT_WINDOW_PIECES, 3)

    def launches(call, c):
        before = c.launch_count()
        return call(), c.launch_count() - before

    for case in ("offsets_64", "swapped", "clustered", "clustered_64"):
        f, g = POLY[case]()
        r = oracle.poly_mul(f, g)
        for kw in ({}, {"host_out": True}, {"capacity": 1}, {"capacity": 1, "host_out": True}):
            (ex, cf, _, _), n = launches(lambda: poly(kron, f, g, ctx=ctx, **kw), ctx)
            assert_poly_equal(ex, cf, r, f"{case} {kw}")
            assert n > launches(lambda: poly(kron, f, g, **kw), kron.context())[1]   # the limit was met
    for case in ("offsets_64", "cosines"):
        f, g = PSER[case]()
        r = oracle.poisson_mul(f, g, keep_zero=True)
        for kw in ({}, {"host_out": True}, {"capacity": 1}):
            assert_pseries_close(pseries(kron, f, g, ctx=ctx, **kw), r, 1e-12, f"{case} {kw}")
    dup = random_poly(3, 40, -90, 90, 35)
    dup.exps[:, 1] = dup.exps[:, 0]
    jobs = [POLY["offsets_64"](), (random_poly(2, 50, 0, 12, 31), random_poly(2, 60, 0, 12, 32)), POLY["one_by_many"](),
            (dup, dup), POLY["swapped"]()]
    res = kron.kron_mul_batch([(up(f), up(g)) for f, g in jobs], ctx=ctx)
    for i, (x, (f, g)) in enumerate(zip(res, jobs)):
        assert x["status"] == (kron.KR_ERR_DUP if i == 3 else 0)
        if i != 3:
            assert_poly_equal(x["exps"], x["coef"], oracle.poly_mul(f, g), f"job {i}")


@pytest.mark.parametrize("failures", [1, 2, 3])
def test_out_of_memory(kron, failures):
    """A windowed product whose scratch does not fit runs again with estimated room, then through the table."""
    import torch
    f, g = POLY["shared_keys"]()
    p, q = PSER["offsets_64"]()
    r, rs = oracle.poly_mul(f, g), oracle.poisson_mul(p, q, keep_zero=True)
    calls = {"poly": (lambda c: poly(kron, f, g, ctx=c), lambda o: assert_poly_equal(o[0], o[1], r)),
             "host": (lambda c: poly(kron, f, g, ctx=c, host_out=True), lambda o: assert_poly_equal(o[0], o[1], r)),
             "series": (lambda c: pseries(kron, p, q, ctx=c), lambda o: assert_pseries_close(o, rs)),
             "batch": (lambda c: kron.kron_mul_batch([(up(f), up(g))], ctx=c, opts={"path": kron.KR_PATH_HASH}),
                       lambda o: assert_poly_equal(o[0]["exps"], o[0]["coef"], r))}
    for name, (call, check) in calls.items():
        ctx = kron.Context()
        kron.kr_selftest_limit(ctx, kron.KR_LIMIT_GROWTHS, failures)
        if failures < 3:
            check(call(ctx))
        else:
            with pytest.raises(kron.KronError) as err:
                call(ctx)
            assert err.value.status == kron.KR_ERR_OOM
        check(call(ctx))   # the next call is not affected
        ctx.close()
    # several products: a wave is split before its products give up their windows
    ctx = kron.Context()
    kron.kr_selftest_limit(ctx, kron.KR_LIMIT_GROWTHS, failures)
    for x in kron.kron_mul_batch([(up(f), up(g))] * 2, ctx=ctx):
        assert x["status"] == 0
        assert_poly_equal(x["exps"], x["coef"], r)
    ctx.close()
    torch.cuda.synchronize()


def test_host_outputs_take_room_for_their_terms(kron):
    """A product with far fewer terms than pairs, into host memory with room for every pair."""
    f = far(dense_total_degree(4, 12, -1000, 1000, 61), 10 ** 9)
    g = far(dense_total_degree(4, 11, -1000, 1000, 62), 10 ** 9)
    r = oracle.poly_mul(f, g)
    pairs = f.coef.size * g.coef.size
    assert 50 * r.coef.size < pairs
    ctx, base = kron.Context(), kron.Context()
    ex, cf, _, _ = poly(kron, f, g, ctx=ctx, host_out=True, capacity=pairs)
    assert_poly_equal(ex, cf, r)
    poly(kron, f, g, ctx=base)
    extra = ctx.scratch_bytes() - base.scratch_bytes()   # the decode's: 24 bytes a term, a quarter and 1 MB to spare
    assert extra <= 1.25 * 24 * r.coef.size + (2 << 20)
    ctx.close()
    base.close()
