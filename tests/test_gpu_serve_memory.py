"""A worker's scratch after a request is within what admission predicted for it."""
import pytest

from tests.test_gpu_window import dev
from workloads import dense_total_degree, mp_sparse, poisson_random, random_poly

pytestmark = pytest.mark.gpu

REQUESTS = {
    "merging": lambda: (mp_sparse("f", 10, -1000, 1000, 1), mp_sparse("g", 10, -1000, 1000, 2)),
    "own_keys": lambda: (random_poly(5, 2000, -30, 30, 3), random_poly(5, 1500, -30, 30, 4)),
    "staged": lambda: (poisson_random(3800, 3, 4, 4, 8, 5, mag="unit"), poisson_random(2900, 3, 4, 4, 8, 6, mag="unit")),
    "dense": lambda: (dense_total_degree(4, 12, -9, 9, 7), dense_total_degree(4, 12, -9, 9, 8)),
    "small": lambda: (random_poly(3, 40, -90, 90, 9), random_poly(3, 50, -90, 90, 10)),
}


@pytest.mark.parametrize("case", sorted(REQUESTS))
def test_scratch_within_the_prediction(case):
    import torch
    from paper_1004_4548_gb300.serve import Request, Server
    f, g = (type(p)(*(dev(x) for x in vars(p).values())) for p in REQUESTS[case]())
    srv = Server(workers=1)
    r = Request(f, g, 0.0)
    predicted = srv.predict_bytes(r)   # before anything is learned
    w = srv.workers[0]
    with torch.cuda.stream(w.stream):
        srv._mul(w, [r])
        w.stream.synchronize()
    assert w.ctx.scratch_bytes() <= predicted, f"{w.ctx.scratch_bytes()} bytes, {predicted:.0f} predicted"
    srv.close()
