"""The best one to four candidates (a pass each up to three, the radix selection from four) against a
full sort, over list sizes around the CTA, with ties, NaN and infinities, and past the list's end."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu

REC = [("score", "<f8"), ("rot", "<i4"), ("idx", "<i4")]


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 54001])
def test_few_match_a_sort(n, k):
    rng = np.random.default_rng(np.random.SeedSequence([n, k]))
    for kind in ("spread", "ties", "special", "same"):
        rec = np.zeros(n, dtype=REC)
        rec["rot"], rec["idx"] = rng.integers(-3, 4, n), rng.integers(0, 3, n)
        if kind == "spread":
            rec["score"] = rng.standard_normal(n)
        elif kind == "ties":
            rec["score"] = rng.integers(0, 2, n)
        elif kind == "special":
            rec["score"] = rng.choice([np.nan, -np.inf, np.inf, -0.0, 0.0], n, p=[0.4, 0.4, 0.0, 0.1, 0.1])
        else:
            rec["score"], rec["rot"], rec["idx"] = -np.inf, -1, -1
        rec["idx"][0] = 7  # one record differs where all else may be equal
        s = np.where(np.isnan(rec["score"]), -np.inf, rec["score"]) + 0.0
        order = np.lexsort((np.arange(n), rec["idx"], rec["rot"], -s))[:k]
        ctx = sd.Context(3, "f32", 0)
        cand = torch.from_numpy(rec.view(np.uint8).copy()).cuda()
        out = torch.zeros((k, sd.CAND_BYTES), dtype=torch.uint8, device="cuda")
        ctx._check(ctx.lib.sd_top_k_static(ctx.handle, cand.data_ptr(), n, k, out.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream))
        got = out.cpu().numpy().reshape(-1).view(REC)
        m = min(n, k)
        assert np.array_equal(got[:m].view(np.uint8), rec[order].view(np.uint8)), kind
        assert (got["rot"][m:] == -1).all() and (got["idx"][m:] == -1).all() and (got["score"][m:] == -np.inf).all()
        ctx.close()
