"""Admission: the memory predicted for a request covers the room that key windows take, whatever the observed
ratio of output terms says."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_1004_4548_gb300 import serve


def request(nf, ng, poisson):
    f, g = (SimpleNamespace(coef=np.empty(n, np.float64), **({"trig": None} if poisson else {})) for n in (nf, ng))
    return serve.Request(f, g, 0.0)


@pytest.mark.parametrize("poisson", [False, True])
@pytest.mark.parametrize("nf,ng", [(1, 1), (500, 700), (6188, 6188), (20000, 12000)])
@pytest.mark.parametrize("ratio", [1e-4, 0.3, 2.0])
def test_prediction_covers_the_windows(nf, ng, poisson, ratio):
    srv = serve.Server.__new__(serve.Server)
    srv.ratio = {False: ratio, True: ratio}
    updates = nf * ng * (2 if poisson else 1)
    need = 32 * updates if 32 * updates <= 16 << 30 else 32 * 1.1 * nf * ng * ratio
    assert srv.predict_bytes(request(nf, ng, poisson)) >= max(need, 64 * nf * ng * ratio)
