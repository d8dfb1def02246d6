"""Pruned 3D passes clear and read only the ball of the sub-box that the rotated taps reach: samples
on the sphere's surface, in every direction, against the full passes, which clear and read all of it."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0.0, 0.03, 0.71, 1.37])
@pytest.mark.parametrize("precision,N", [("f32", 16), ("f32", 48), ("f32", 96), ("f32", 192), ("f64", 32), ("f64", 64)])
def test_surface_samples_match_full_passes(precision, N, radius):
    L, m = 8.0, 700
    ctx = sd.Context(3, precision, 0, sigma_g=2.0 * L / (np.pi * N))
    rng = np.random.default_rng(np.random.SeedSequence([N, int(100 * radius), 41]))
    v = rng.standard_normal((m, 3))
    p = np.zeros((m, 4))
    p[:, :3] = radius * v / np.linalg.norm(v, axis=1, keepdims=True)
    p[:6, :3] = radius * np.concatenate([np.eye(3), -np.eye(3)])
    fx = ctx.shape_from_samples(np.pad(rng.uniform(-0.8, 0.8, (60, 3)), ((0, 0), (0, 1))),
                                rng.standard_normal((60, 2)))
    mv = ctx.shape_from_samples(p, rng.standard_normal((m, 2)))
    q = rng.standard_normal((7, 4))
    q[0] = (1, 0, 0, 0)
    q = torch.tensor(q, dtype=torch.float64, device="cuda")
    g = sd.Grid(N, L)
    ctx.set_option("batch", 2)  # the buffers of one batch hold the last one's passes
    ctx.set_option("fft_plan", 0)
    want = ctx.score_maps(fx, mv, q, g).cpu().numpy()
    ctx.set_option("fft_plan", 1)
    # as the other comparisons of the two plans allow, and for equal terms (radius 0) the sums'
    # rounding: m 2^-25 in FP32, 2.6 m / 2^29 in fixed-point tiles times four for the deconvolution
    tol = 1e-12 if precision == "f64" else 2e-6 + m * (4 * 2.6 / 2 ** 29 + 2.0 ** -25)
    off = {"spread_direct": 1, "spread_box": 0, "spread_fused": 0}
    for spread in ({}, {"spread_direct": 0, "spread_bin_side": 8}, {"spread_box": 1}, {"spread_fused": 1}):
        for k, val in {**off, **spread}.items():
            ctx.set_option(k, val)
        got = ctx.score_maps(fx, mv, q, g).cpu().numpy()
        for r in range(7):
            assert np.linalg.norm(got[r] - want[r]) <= tol * np.linalg.norm(want[r]), (spread, r)
    ctx.close()
