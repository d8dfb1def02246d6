"""Tuned and imported plans with fused spreading where the job cannot run it (a forced full forward plan, a
2D job, another kernel width): another spreading takes its place, with the same candidates."""

import json

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,w,fft", [(3, 6, 0), (2, 6, -1), (3, 5, -1), (3, 6, -1)])
def test_fused_plan_only_where_it_runs(dim, w, fft):
    N, L, P = 32, 8.0, 9
    rng = np.random.default_rng(np.random.SeedSequence([dim, w]))
    ctx = sd.Context(dim, "f32", 0, sigma_g=0.3, w=w)
    shapes = []
    for m in (80, 300):
        p = np.zeros((m, 4))
        p[:, :dim] = rng.uniform(-0.7, 0.7, (m, dim))
        shapes.append(ctx.shape_from_samples(p, rng.standard_normal((m, 2))))
    q = rng.standard_normal((P, 4))
    if dim == 2:
        q[:, 1:3] = 0
    q = torch.tensor(q, device="cuda")
    g = sd.Grid(N, L)
    want = sd.decode_cands(ctx.score_rotations(*shapes, q, g))
    ctx.set_option("autotune", 1)
    ctx.tune_import(json.dumps({"sdfdock_plans": 1, "plans": [
        {"key": f"{sd.SD_F32}|{dim}|{N}|{2 * N}|{s}|8", "batch": 4, "spread_bins": 1, "fft": 1} for s in range(8)]}))
    ctx.set_option("fft_plan", fft)
    plan = ctx.search_plan(shapes[1], g, P)
    runs = dim == 3 and w == 6 and fft != 0
    assert plan["batch"] == 4 and (plan["spread_bins"] == 1) == runs and (fft < 0 or plan["fft_plan"] == fft)
    got = sd.decode_cands(ctx.score_rotations(*shapes, q, g))
    assert (got[0] - want[0]).abs().max() <= 1e-5 * want[0].abs().max()
    assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    ctx.close()
