"""decode_cands: values, layout (a contiguous score) and independence of the buffer, for whole,
single-record, empty, strided and unaligned buffers."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

REC = [("score", "<f8"), ("rot", "<i4"), ("idx", "<i4")]


def _rec(n):
    rec = np.zeros(n, dtype=REC)
    rec["score"] = np.random.default_rng(n).standard_normal(n)
    rec["score"][: n // 3] = np.nan
    rec["rot"], rec["idx"] = -np.arange(n), np.arange(n) + (1 << 20)
    return rec


def _buffer(rec, kind):
    raw = torch.from_numpy(rec.view(np.uint8).copy()).reshape(-1, sd.CAND_BYTES)
    if kind == "flat":
        return raw.reshape(-1)
    if kind == "strided":
        wide = torch.zeros((len(rec), sd.CAND_BYTES + 4), dtype=torch.uint8)
        wide[:, : sd.CAND_BYTES] = raw
        return wide[:, : sd.CAND_BYTES]
    if kind == "unaligned":
        wide = torch.zeros(raw.numel() + 5, dtype=torch.uint8)
        wide[5:] = raw.reshape(-1)
        return wide[5:]
    return raw


@pytest.mark.parametrize("kind", ["rows", "flat", "strided", "unaligned"])
@pytest.mark.parametrize("n", [0, 1, 2, 257])
def test_decode_cands(n, kind):
    rec = _rec(n)
    buf = _buffer(rec, kind)
    score, rot, idx = sd.decode_cands(buf)
    buf.fill_(7)
    assert score.is_contiguous() and score.dtype == torch.float64
    assert score.shape == rot.shape == idx.shape == (n,)
    assert np.array_equal(score.numpy().view(np.int64), rec["score"].view(np.int64))  # bits, NaN's too
    assert np.array_equal(rot.numpy(), rec["rot"]) and np.array_equal(idx.numpy(), rec["idx"])
    assert rot.stride() == idx.stride() == (2,)
    assert score.view(torch.int32).numel() == 2 * n
