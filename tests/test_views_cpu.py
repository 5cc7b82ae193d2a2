"""Results of a batch as strided views: packed arrays share one tensor, arrays in several blocks get their
own, and both read the library's memory (host memory here, in the place of the device's)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1004_4548_gb300 import binding


def host_view(ptr, shape, typestr, device):
    if not ptr or 0 in shape:
        return torch.empty(shape)
    n = int(np.prod(shape)) * int(typestr[2])
    raw = np.ctypeslib.as_array(ctypes.cast(ptr, ctypes.POINTER(ctypes.c_uint8)), (n,))
    return torch.from_numpy(raw.view(np.dtype(typestr)).reshape(shape))


@pytest.mark.parametrize("blocks", [1, 2])
def test_batch_results(monkeypatch, blocks):
    monkeypatch.setattr(binding, "_view", host_view)
    block = np.zeros(4096, np.uint8)
    off = -block.ctypes.data % 256
    at = block.ctypes.data + off
    e, c = np.arange(21, dtype=np.int32).reshape(3, 7), np.arange(7, dtype=np.int64) - 3
    block[off:off + 56] = c.view(np.uint8)
    block[off + 256:off + 256 + 84] = e.reshape(-1).view(np.uint8)
    far = np.ascontiguousarray(e[:, ::-1])
    jobs, res = (binding.kr_job * 3)(), (binding.kr_result * 3)()
    for j in jobs:
        j.f.nvars, j.f.type = 3, binding.KR_I64
    res[0].path, res[0].nterms, res[0].exps, res[0].coef = 1, 7, at + 256, at
    res[1].status = binding.KR_ERR_DUP
    if blocks == 2:
        res[2].nterms, res[2].exps, res[2].coef = 7, far.ctypes.data, at
    out = binding._results(jobs, res, 3, 0)
    assert [r["status"] for r in out] == [0, binding.KR_ERR_DUP, 0] and out[0]["path"] == 1
    assert np.array_equal(out[0]["exps"].numpy(), e) and np.array_equal(out[0]["coef"].numpy(), c)
    assert out[0]["exps"].dtype == torch.int32 and out[0]["coef"].dtype == torch.int64
    assert out[1]["nterms"] == 0 and out[1]["coef"].shape[0] == 0
    if blocks == 2:
        assert np.array_equal(out[2]["exps"].numpy(), far)
    block[off] = 42   # the library's memory itself, not a copy
    assert int(out[0]["coef"][0]) & 0xff == 42
