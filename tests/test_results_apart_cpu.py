"""The arrays of a batch's results are tensors of their own: a change of one in place does not reach autograd's version
of another, and each one's storage is its own array, not the batch's block."""
import copy

import numpy as np
import torch

from paper_1004_4548_gb300 import binding
from tests.test_views_cpu import host_view


def test_results_share_nothing(monkeypatch):
    monkeypatch.setattr(binding, "_view", host_view)
    block = np.zeros(4096, np.uint8)
    off = -block.ctypes.data % 256
    at = block.ctypes.data + off
    jobs, res = (binding.kr_job * 2)(), (binding.kr_result * 2)()
    for j in jobs:
        j.f.nvars, j.f.type = 3, binding.KR_F64
    for i, r in enumerate(res):
        r.path, r.nterms, r.coef, r.exps = 1, 7, at + 512 * i, at + 512 * i + 256
    a, b = binding._results(jobs, res, 2, 0)
    w = torch.ones(7, dtype=torch.float64, requires_grad=True)
    loss = (w * b["coef"]).sum()   # saves b's coefficients
    a["coef"].add_(1)
    loss.backward()
    for r in (a, b):
        for k in ("exps", "coef"):
            assert r[k].untyped_storage().nbytes() == r[k].numel() * r[k].element_size()
            assert copy.deepcopy(r[k]).untyped_storage().nbytes() == r[k].numel() * r[k].element_size()
