"""2D searches on both sides of the lines between the half-spectrum passes' forms for few CTAs and for
many, against the real part of score_maps: every length, batches about the waves of 152 CTAs, pruned and
unpruned passes, one and several candidates."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu

# rotations a batch: CTAs of 16 (FP64 from N = 192: 8) columns a rotation are N / 32 rounded up (N / 16)
BATCHES = {"f32": {8: (1, 64), 16: (1, 64), 24: (1, 64), 32: (5, 64), 48: (48, 49), 64: (48, 49), 96: (32, 33), 128: (24, 25),
                   192: (16, 17), 256: (12, 13)},
           "f64": {8: (1, 64), 16: (1, 64), 24: (1, 64), 32: (5, 64), 48: (50, 64), 64: (50, 64), 96: (32, 40, 64),
                   128: (24, 32, 40, 64), 192: (5, 12, 18), 256: (5, 12, 24)}}


@pytest.mark.parametrize("reach", [0.6, 2.4])
@pytest.mark.parametrize("precision,N", [(p, N) for p in BATCHES for N in BATCHES[p]])
def test_forms_match_maps(precision, N, reach):
    L, m = 8.0, 60
    rng = np.random.default_rng(np.random.SeedSequence([N, int(10 * reach)]))
    ctx = sd.Context(2, precision, 0, sigma_g=2.0 * L / (np.pi * N))
    shapes = []
    for _ in range(2):
        p = np.zeros((m, 4))
        p[:, :2] = rng.uniform(-reach, reach, (m, 2))
        shapes.append(ctx.shape_from_samples(p, rng.standard_normal((m, 2))))
    P = max(BATCHES[precision][N])
    q = rng.standard_normal((P, 4))
    q[:, 1:3] = 0
    q = torch.tensor(q, device="cuda")
    g = sd.Grid(N, L)
    ref = ctx.score_maps(*shapes, q, g).real.double()
    scale = ref.abs().amax(1)
    # as the other comparison with the maps: rounding of two transforms of N^2 points, and of the atomic sums
    tol = 2 * (2.0 ** -23 if precision == "f32" else 2.0 ** -52) * max(4.0, 2 * np.log2(N)) * (4 if precision == "f64" else 1)
    for batch in BATCHES[precision][N]:
        ctx.set_option("batch", batch)
        for k_r in (1, 2, 4, 16):
            s, rot, idx = sd.decode_cands(ctx.score_rotations(*shapes, q, g, k_r=k_r))
            s, idx = s.reshape(P, k_r), idx.reshape(P, k_r).long()
            want = torch.topk(ref, k_r, dim=1).values
            assert ((s - want).abs().amax(1) <= tol * scale).all(), (batch, k_r)
            assert ((ref.gather(1, idx) - s).abs().amax(1) <= tol * scale).all(), (batch, k_r)
            assert (rot.reshape(P, k_r) == torch.arange(P, device="cuda")[:, None]).all()
            assert all(len(set(r)) == k_r for r in idx.tolist())
    ctx.close()
