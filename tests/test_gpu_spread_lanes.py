"""Direct spreading with eight lanes a sample against one thread a sample: the same rotations in batches
below and above the lines between the two (16,000, 20,000 and 60,000 samples a launch)."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("w", [4, 5, 6, 7, 8])
def test_lanes_match_threads(w, dim, precision):
    N, L, m, P = 32, 8.0, 5003, 13  # 5,003 samples a launch, 65,039 in one
    rng = np.random.default_rng(np.random.SeedSequence([w, dim]))
    ctx = sd.Context(dim, precision, 0, sigma_g=0.3, w=w)
    ctx.set_option("spread_direct", 1)
    shapes = []
    for n in (100, m):
        p = np.zeros((n, 4))
        p[:, :dim] = rng.uniform(-0.9, 0.9, (n, dim))
        shapes.append(ctx.shape_from_samples(p, rng.standard_normal((n, 2))))
    q = rng.standard_normal((P, 4))
    if dim == 2:
        q[:, 1:3] = 0
    q = torch.tensor(q, device="cuda")
    maps = {}
    for batch in (1, 3, 4, P):  # 5,003 to 65,039 samples a launch
        ctx.set_option("batch", batch)
        maps[batch] = ctx.score_maps(*shapes, q, sd.Grid(N, L))
    # two orders of the cells' sums (m terms of random sign) and of the transforms
    tol = 2e-6 if precision == "f32" else 1e-13
    for batch in (3, 4, P):
        for r in range(P):
            assert (maps[batch][r] - maps[1][r]).norm() <= tol * maps[1][r].norm(), (batch, r)
    ctx.close()
