"""The search's half-spectrum passes on long lines (3D grids of 128 and more) against the full inverse of
score_maps: each forward plan, both precisions, sub-boxes that fit half a line and that do not, kept
candidates of one and several.  One or two rotations."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


def _check(N, precision, reach, plan, rotations):
    L = 8.0
    rng = np.random.default_rng(np.random.SeedSequence([N, plan, int(10 * reach)]))
    ctx = sd.Context(3, precision, 0, sigma_g=2.0 * L / (np.pi * N))
    shapes = []
    for _ in range(2):
        p = np.zeros((60, 4))
        p[:, :3] = rng.uniform(-reach, reach, (60, 3))
        shapes.append(ctx.shape_from_samples(p, rng.standard_normal((60, 2))))
    q = torch.tensor(rng.standard_normal((rotations, 4)), device="cuda")
    g = sd.Grid(N, L)
    ctx.set_option("fft_plan", plan)
    assert ctx.search_plan(shapes[1], g, rotations)["fft_plan"] == plan
    ctx.set_option("fft_plan", 1 if reach < 1 else 0)  # the reference: the standard plan's maps
    ref = ctx.score_maps(*shapes, q, g).real.double()
    ctx.set_option("fft_plan", plan)
    scale = ref.abs().amax(1)
    # as the smaller grids' comparison: rounding of two transforms of N^3 points, and (FP64) of the atomic sums
    tol = 2 * (2.0 ** -23 if precision == "f32" else 2.0 ** -52) * max(4.0, 3 * np.log2(N)) * (4 if precision == "f64" else 1)
    for k_r in (1, 2, 4, 16):
        s, rot, idx = sd.decode_cands(ctx.score_rotations(*shapes, q, g, k_r=k_r))
        s, idx = s.reshape(rotations, k_r), idx.reshape(rotations, k_r).long()
        want = torch.topk(ref, k_r, dim=1).values
        assert ((s - want).abs().amax(1) <= tol * scale).all(), (k_r, ((s - want).abs().amax(1) / scale).tolist())
        assert ((ref.gather(1, idx) - s).abs().amax(1) <= tol * scale).all()
        assert (rot.reshape(rotations, k_r) == torch.arange(rotations, device="cuda")[:, None]).all()
        assert all(len(set(r.tolist())) == k_r for r in idx)
    ctx.close()


@pytest.mark.parametrize("plan", [0, 1, 2, 3])
def test_plans_of_384_points(plan):
    _check(192, "f32", 0.6, plan, 2)


# reach 0.6: the sub-box fits half a line; 2.4: it does not (full passes; their tables exceed 32 MB at 192 and 256)
@pytest.mark.parametrize("precision,N,reach,rotations", [("f32", 128, 0.6, 2), ("f32", 128, 2.4, 2), ("f32", 192, 2.4, 1),
                                                         ("f32", 256, 0.6, 2), ("f32", 256, 2.4, 1), ("f64", 128, 0.6, 2),
                                                         ("f64", 128, 2.4, 1), ("f64", 192, 0.6, 1), ("f64", 192, 2.4, 1),
                                                         ("f64", 256, 0.6, 1), ("f64", 256, 2.4, 1)])
def test_long_lines(precision, N, reach, rotations):
    _check(N, precision, reach, 1 if reach < 1 else 0, rotations)
    if reach < 1:
        _check(N, precision, reach, 0, rotations)
