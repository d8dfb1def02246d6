"""Fused spreading's workspace limit (7 GiB a batch) where a tuned plan's batch is larger than the one the
job would have started from: the limit counts at the batch that runs.  Plans only; nothing is searched."""

import json

import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


# 108 bytes a sample and rotation and the bin tables, 64 rotations a batch: 1.09 million samples reach the limit
@pytest.mark.parametrize("m,fused", [(1_040_000, True), (1_120_000, False), (1_900_000, False)])
@pytest.mark.parametrize("default_fused", [0, 1])
def test_limit_holds_at_the_tuned_batch(m, fused, default_fused):
    N, L = 256, 8.0
    ctx = sd.Context(3, "f32", 0, sigma_g=0.1)
    pos = torch.rand((m, 4), device="cuda") - 0.5
    pos[:, 3] = 0
    mv = ctx.shape_from_samples(pos, torch.ones((m, 2), device="cuda"))
    g = sd.Grid(N, L)
    ctx.set_option("spread_fused", default_fused)
    assert ctx.search_plan(mv, g, 64)["batch"] < 64
    assert ctx.search_plan(mv, g, 64)["spread_bins"] == default_fused  # the default batch fits, or direct
    ctx.set_option("autotune", 1)
    lg = m.bit_length() - 1
    keys = [f"{sd.SD_F32}|3|{N}|{2 * N}|{s}|{lg}" for s in range(33)]
    ctx.tune_import(json.dumps({"sdfdock_plans": 1, "plans": [
        {"key": k, "batch": 64, "spread_bins": 1, "fft": 1} for k in keys]}))
    plan = ctx.search_plan(mv, g, 64)
    assert plan["batch"] == 64 and plan["spread_bins"] == (1 if fused else 0)
    ctx.close()
