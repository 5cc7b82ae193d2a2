"""Outputs are complete when a call returns, on whichever stream it ran."""
import pytest

import oracle
from tests.gpu_compare import assert_poly_equal, assert_pseries_close, to_np
from tests.test_gpu_window import dev
from workloads import PSeries, random_poly, random_pseries

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kron():
    import paper_1004_4548_gb300 as k
    k.load()
    return k


@pytest.mark.parametrize("given", [True, False])
def test_outputs_complete_on_return(kron, given):
    """torch's current stream is kept busy after the operands; the outputs are read on another stream at once.
    given: the call runs on that other stream; else on the current one, behind the busy work."""
    import torch
    f, g = random_poly(2, 9000, 0, 100, 1), random_poly(2, 9000, 0, 100, 2)   # room for 144,000 terms guessed, 40,401 used
    p, q = random_pseries(1, 2, 2000, 3, 10, 3), random_pseries(1, 2, 40, 3, 2, 4)
    D = [[dev(x) for x in (f.exps, f.coef, g.exps, g.coef)], [PSeries(*(dev(x) for x in vars(s).values())) for s in (p, q)]]
    r, rs = oracle.poly_mul(f, g), oracle.poisson_mul(p, q, keep_zero=True)
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    for _ in range(2):
        torch.cuda._sleep(200_000_000)   # about 0.1 s of the current stream
        a = kron.poly_mul(*D[0], stream=other if given else None)
        with torch.cuda.stream(other):
            ex, cf = (x.cpu() for x in a[:2])
        assert_poly_equal(ex, cf, r)
        torch.cuda._sleep(200_000_000)
        b = kron.poisson_mul(*D[1], stream=other if given else None)
        with torch.cuda.stream(other):
            b = [x.cpu() for x in b[:4]]
        assert_pseries_close(b, rs)
        del a
    assert to_np(cf).size == r.coef.size
