"""The FP64 re-score against plain FP64 pair sums: its exponential over the whole cutoff range, block
remainders, 2D and 3D, both sample precisions."""

import math

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("m1,m2", [(1, 1), (33, 257), (300, 256), (1000, 777)])
@pytest.mark.parametrize("sigma", [0.05, 0.4, 3.0])
def test_rescore_matches_pair_sums(m1, m2, dim, precision, sigma):
    rng = np.random.default_rng(np.random.SeedSequence([m1, m2, dim]))
    real = np.float32 if precision == "f32" else np.float64
    pts, wts = [], []
    for m in (m1, m2):
        p = np.zeros((m, 4), real)
        p[:, :dim] = rng.uniform(-2, 2, (m, dim))
        pts.append(p)
        wts.append(rng.standard_normal((m, 2)).astype(real))
    ctx = sd.Context(dim, precision, 0, sigma_g=sigma)
    fx, mv = (ctx.shape_from_samples(p, w) for p, w in zip(pts, wts))
    N, L, k = 32, 12.0, 3
    q = rng.standard_normal((k, 4))
    if dim == 2:
        q[:, 1:3] = 0
    idx = rng.integers(0, N ** dim, k)
    rec = np.zeros(k, dtype=[("score", "<f8"), ("rot", "<i4"), ("idx", "<i4")])
    rec["score"], rec["rot"], rec["idx"] = [3.0, 2.0, 1.0], np.arange(k), idx
    poses = ctx.top_k_poses(torch.from_numpy(rec.view(np.uint8).copy()).cuda(), k, fx, mv,
                            torch.tensor(q, device="cuda"), sd.Grid(N, L))
    p1, p2 = (p[:, :dim].astype(np.float64) for p in pts)
    c1, c2 = (w[:, 0].astype(np.float64) + 1j * w[:, 1] for w in wts)
    s2 = 2 * sigma * sigma
    for r in range(k):
        w, x, y, z = q[r] / np.linalg.norm(q[r])
        R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                      [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                      [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])[:dim, :dim]
        i, t = int(idx[r]), []
        for _ in range(dim):
            t.append((i % N - N // 2) * L / N)
            i //= N
        d2 = (((p2 @ R.T + np.array(t))[:, None] - p1[None]) ** 2).sum(2)
        g = np.exp(-d2 / (2 * s2)) * (2 * math.pi * s2) ** (-dim / 2)
        terms = c2[:, None] * c1[None] * g
        ref, mag = terms.sum(), np.abs(terms).sum()
        # exponents to 32 in rounding, the sums, and pairs beyond the cutoff (e^-32 of the peak each)
        tol = 64 * 2.0 ** -52 * mag + m1 * m2 * math.exp(-32) * (2 * math.pi * s2) ** (-dim / 2) * 30
        assert abs(poses[r]["score_fp64"] - ref.real) <= tol
        assert abs(poses[r]["score_fp64_im"] - ref.imag) <= tol
    ctx.close()
