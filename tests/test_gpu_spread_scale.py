"""The fixed-point scale of fused spreading: its bound on a tile's cells must hold where all the
samples fall in a few cells, on both sides of a bin and of a 32-cell stretch of x, and where bins
differ by orders of magnitude."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [48, 96, 256])
@pytest.mark.parametrize("jitter", [0.0, 1.0, 4.0])  # spread of a cluster, in cells
def test_clustered_samples_match_direct_spreading(N, jitter):
    L, m, n_clusters = 8.0, 600, 24
    ctx = sd.Context(3, "f32", 0, sigma_g=2.0 * L / (np.pi * N))
    rng = np.random.default_rng(np.random.SeedSequence([N, int(jitter), 31]))
    fx = ctx.shape_from_samples(np.pad(rng.uniform(-0.8, 0.8, (60, 3)), ((0, 0), (0, 1))),
                                rng.standard_normal((60, 2)))
    q = torch.tensor(rng.standard_normal((4, 4)), dtype=torch.float64, device="cuda")
    g = sd.Grid(N, L)
    # FP32 sums of m equal terms: m 2^-25 in one direction; a fixed-point cell of at most
    # m |c|, scaled to at least 2^29: 0.5 a tap over 216 taps against a kernel norm of 2.8,
    # 2.6 m / 2^29; four times that for the deconvolution, 2e-6 for the FP32 passes
    tol = 2e-6 + m * (4 * 2.6 / 2 ** 29 + 2.0 ** -25)
    for k in range(n_clusters // 8):
        centres = rng.uniform(-0.55, 0.55, (8, 3))
        p = np.zeros((8 * m // 8 + 1, 4))
        p[:-1, :3] = np.repeat(centres, m // 8, 0) if k else np.repeat(centres[:1], m, 0)
        p[:-1, :3] += jitter * (L / (2 * N)) * rng.uniform(-0.5, 0.5, (m, 3))
        p[-1, 0] = 1.0  # the sub-box's extent
        c = np.ones((m + 1, 2)) * (10.0 ** rng.uniform(-4, 0, (m + 1, 1)) if k == 2 else 1.0)
        mv = ctx.shape_from_samples(p, c)
        maps = []
        for fused in (1, 0):
            ctx.set_option("spread_fused", fused)
            assert (ctx.search_plan(mv, g, 4)["spread_bins"] == 1) == bool(fused)
            maps.append(ctx.score_maps(fx, mv, q, g).cpu().numpy())
        for r in range(4):
            assert np.linalg.norm(maps[0][r] - maps[1][r]) <= tol * np.linalg.norm(maps[1][r]), (k, r)
    ctx.close()
