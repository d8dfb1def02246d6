"""The radix-selecting top-k against a full sort: sizes around the CTA and the sort's powers of two,
heavy ties, signed zeros, infinities and NaN, keys equal up to the position."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu

REC = [("score", "<f8"), ("rot", "<i4"), ("idx", "<i4")]


def _records(kind, n, rng):
    rec = np.zeros(n, dtype=REC)
    rec["rot"] = rng.permutation(n)
    rec["idx"] = rng.integers(0, 1 << 24, n)
    if kind == "spread":
        rec["score"] = rng.standard_normal(n) * 10.0 ** rng.uniform(-300, 300, n)
    elif kind == "ties":
        rec["score"] = rng.integers(-2, 3, n) * 0.5
        rec["rot"] = rng.integers(-3, 4, n)
        rec["idx"] = rng.integers(0, 3, n)
    elif kind == "special":
        rec["score"] = rng.choice([0.0, -0.0, np.inf, -np.inf, np.nan, 1.0, -1.0, 5e-324], n)
    else:  # all records the same: the position decides
        rec["score"], rec["rot"], rec["idx"] = 1.25, 7, 9
    return rec


@pytest.mark.parametrize("kind", ["spread", "ties", "special", "same"])
@pytest.mark.parametrize("n,k", [(1, 1), (3, 5), (64, 64), (1023, 33), (1025, 1), (5000, 100), (70001, 1000), (70000, 4096)])
def test_top_k_matches_a_sort(n, k, kind):
    rec = _records(kind, n, np.random.default_rng(np.random.SeedSequence([n, k])))
    s = np.where(np.isnan(rec["score"]), -np.inf, rec["score"]) + 0.0
    order = np.lexsort((np.arange(n), rec["idx"], rec["rot"], -s))[:k]
    ctx = sd.Context(3, "f32", 0)
    cand = torch.from_numpy(rec.view(np.uint8).copy()).cuda()
    poses = ctx.top_k_poses(cand, k, grid=sd.Grid(256, 10.0), rescore_fp64=False)
    got = np.array([(p["score"], p["rot"], p["idx"]) for p in poses], dtype=REC)
    want = rec[order]
    m = min(n, k)
    assert np.array_equal(got["rot"][:m], want["rot"]) and np.array_equal(got["idx"][:m], want["idx"])
    assert np.array_equal(got["score"][:m], want["score"], equal_nan=True)
    assert (got["rot"][m:] == -1).all() and (got["idx"][m:] == -1).all() and (got["score"][m:] == -np.inf).all()
    ctx.close()
