"""Selections of different sizes from two host threads at once: the kernel's shared-memory limit is one
value per device, so a small selection must not take it away from a large one about to launch."""

import threading

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


def test_two_threads_of_different_k():
    n, reps = 5000, 400
    rec = np.zeros(n, dtype=[("score", "<f8"), ("rot", "<i4"), ("idx", "<i4")])
    rec["score"] = np.random.default_rng(5).permutation(n)
    rec["rot"] = np.arange(n)
    cand = torch.from_numpy(rec.view(np.uint8).copy()).cuda()
    torch.cuda.synchronize()
    start, errors, outs = threading.Barrier(2), [], {}

    def work(k):
        try:
            ctx = sd.Context(3, "f32", 0)
            with torch.cuda.stream(torch.cuda.Stream()):
                out = torch.empty((k, sd.CAND_BYTES), dtype=torch.uint8, device="cuda")
                stream = torch.cuda.current_stream().cuda_stream
                start.wait()
                for _ in range(reps):
                    ctx._check(ctx.lib.sd_top_k_static(ctx.handle, cand.data_ptr(), n, k, out.data_ptr(), stream))
                torch.cuda.current_stream().synchronize()
            outs[k] = sd.decode_cands(out)[0].cpu().numpy()
            ctx.close()
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (2000, 4000)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for k in (2000, 4000):
        assert np.array_equal(outs[k], np.arange(n - 1, n - 1 - k, -1))
