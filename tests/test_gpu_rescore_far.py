"""The re-score where positions are so large against sigma that the FP32 screen cannot tell near pairs
from far ones: pairs of every distance reach the FP64 exponential, which is 0 for the far ones."""

import math

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far", [1e9, 3e12])
def test_far_pairs_add_nothing(far):
    sigma, N = 0.05, 32  # FP32 coordinates of `far` are 64 and 262144 apart
    m2 = 4000
    p1, p2 = np.zeros((1, 4)), np.zeros((m2, 4))
    p1[0, 0] = far
    p2[:, 0] = far + np.geomspace(2.0 ** -3, 24.0 if far < 1e10 else 1e5, m2)  # all round to p1 in FP32
    ctx = sd.Context(3, "f64", 0, sigma_g=sigma)
    fx = ctx.shape_from_samples(p1, np.array([[1.0, 0.0]]))
    mv = ctx.shape_from_samples(p2, np.stack([np.ones(m2), np.full(m2, -0.5)], 1))
    rec = np.zeros(1, dtype=[("score", "<f8"), ("rot", "<i4"), ("idx", "<i4")])
    rec["idx"] = (N // 2) * (1 + N + N * N)  # no translation
    q = torch.tensor([[1.0, 0, 0, 0]], dtype=torch.float64, device="cuda")
    pose = ctx.top_k_poses(torch.from_numpy(rec.view(np.uint8).copy()).cuda(), 1, fx, mv, q, sd.Grid(N, 5 * far))[0]
    s2 = 2 * sigma * sigma
    ref = (np.exp(-((p2[:, 0] - p1[0, 0]) ** 2) / (2 * s2)) * (2 * math.pi * s2) ** -1.5).sum()
    # rounding of the terms and the sum, and of the far terms' cutoff (e^-32 of the peak each)
    tol = 64 * 2.0 ** -52 * ref + m2 * math.exp(-32) * (2 * math.pi * s2) ** -1.5
    assert abs(pose["score_fp64"] - ref) <= tol
    assert abs(pose["score_fp64_im"] + 0.5 * ref) <= tol
    ctx.close()
