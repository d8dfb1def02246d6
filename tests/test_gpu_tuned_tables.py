"""The product tables that an autotuner's trials made and its plan does not read are given back: the plan
not chosen makes its table anew at its first search, the chosen one does not."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


def test_trial_tables_are_given_back():
    N, L = 32, 8.0
    rng = np.random.default_rng(3)
    ctx = sd.Context(3, "f32", 0, sigma_g=0.3)
    fx, mv = (ctx.shape_from_samples(np.pad(rng.uniform(-0.7, 0.7, (200, 3)), ((0, 0), (0, 1))),
                                     rng.standard_normal((200, 2))) for _ in range(2))
    q = torch.tensor(rng.standard_normal((12, 4)), device="cuda")
    g = sd.Grid(N, L)

    def launches():
        n0 = sd.launch_count()
        out = sd.decode_cands(ctx.score_rotations(fx, mv, q, g))
        return sd.launch_count() - n0, out

    ctx.set_option("autotune", 1)
    _, tuned = launches()
    n1, _ = launches()
    n2, _ = launches()
    assert n1 == n2  # the chosen plan's table is there
    best = ctx.search_plan(mv, g, 12)["fft_plan"]
    ctx.set_option("fft_plan", 0 if best else 1)
    n3, other = launches()
    n4, _ = launches()
    assert n3 == n4 + 1  # the other plan's is made again
    assert (tuned[0] - other[0]).abs().max() <= 1e-5 * tuned[0].abs().max() and torch.equal(tuned[2], other[2])
    ctx.close()
