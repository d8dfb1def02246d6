"""The ball of the sub-box where it is used, 3D grids of 128 and more (256 points a line): pruned passes
that clear and read it alone against the full passes, in a workspace that a larger shape's search has
filled.  Samples on the sphere's surface, in every direction; every length, both precisions."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0.0, 0.03, 0.71, 1.37])
@pytest.mark.parametrize("precision,N", [("f32", 128), ("f32", 192), ("f32", 256), ("f64", 128), ("f64", 192), ("f64", 256)])
def test_ball_matches_full_passes(precision, N, radius):
    L, m, P = 8.0, 300, 3
    ctx = sd.Context(3, precision, 0, sigma_g=2.0 * L / (np.pi * N))
    rng = np.random.default_rng(np.random.SeedSequence([N, int(100 * radius), 43]))

    def surface(r, n):
        v = rng.standard_normal((n, 3))
        p = np.zeros((n, 4))
        p[:, :3] = r * v / np.linalg.norm(v, axis=1, keepdims=True)
        p[:6, :3] = r * np.concatenate([np.eye(3), -np.eye(3)])
        return ctx.shape_from_samples(p, rng.standard_normal((n, 2)))

    fx = ctx.shape_from_samples(np.pad(rng.uniform(-0.8, 0.8, (60, 3)), ((0, 0), (0, 1))), rng.standard_normal((60, 2)))
    mv, large = surface(radius, m), surface(1.8, 4000)
    q = rng.standard_normal((P, 4))
    q[0] = (1, 0, 0, 0)
    q = torch.tensor(q, device="cuda")
    g = sd.Grid(N, L)
    ctx.set_option("batch", 2)
    ctx.set_option("fft_plan", 0)
    ref = ctx.score_maps(fx, mv, q, g)
    ctx.set_option("fft_plan", 1)
    # as the other comparisons of the two plans allow, and for equal terms (radius 0) the sums'
    # rounding: m 2^-25 in FP32, 2.6 m / 2^29 in fixed-point tiles times four for the deconvolution
    tol = 1e-12 if precision == "f64" else 2e-6 + m * (4 * 2.6 / 2 ** 29 + 2.0 ** -25)
    off = {"spread_direct": 1, "spread_box": 0, "spread_fused": 0}
    for spread in ({}, {"spread_direct": 0, "spread_bin_side": 8}, {"spread_box": 1}):
        for k, val in {**off, **spread}.items():
            ctx.set_option(k, val)
        plan = ctx.search_plan(mv, g, P)
        assert plan["fft_plan"] == 1 and 2 * N >= 256 and plan["spread_bins"] != 1  # a sub-box, cleared by the ball
        ctx.set_option("fft_plan", 0)
        ctx.score_maps(fx, large, q, g)  # full passes of a larger sub-box fill the workspace
        ctx.set_option("fft_plan", 1)
        got = ctx.score_maps(fx, mv, q, g)
        for r in range(P):
            assert (got[r] - ref[r]).norm() <= tol * ref[r].norm(), (spread, r)
        s, _, idx = sd.decode_cands(ctx.score_rotations(fx, mv, q, g))
        peak = ref.real.amax(1).double()
        at = ref.real.gather(1, idx.long()[:, None])[:, 0].double()
        lim = 20 * tol * ref.abs().amax(1).double()  # a norm's error over the largest entry of a smooth map
        assert ((s - peak).abs() <= lim).all() and ((at - peak).abs() <= lim).all()
    ctx.close()
