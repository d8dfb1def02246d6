"""The search's half-spectrum inverse against the full one: candidates of score_rotations against
the real part of score_maps (held to the oracle elsewhere), at every grid size, both precisions,
1D-tile remainders (N/2 below and above a CTA's columns), pruned and unpruned forward passes."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu

SIZES = [8, 16, 24, 32, 48, 64, 96, 128, 192, 256]


def _shapes(ctx, dim, m, seed, reach):
    rng = np.random.default_rng(np.random.SeedSequence([seed, 21]))
    out = []
    for _ in range(2):
        p = np.zeros((m, 4))
        p[:, :dim] = rng.uniform(-reach, reach, (m, dim))
        out.append(ctx.shape_from_samples(p, rng.standard_normal((m, 2))))
    return out


# reach 0.6: the sub-box fits half a line (pruned passes); 2.4: it does not
@pytest.mark.parametrize("reach", [0.6, 2.4])
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dim,N", [(2, N) for N in SIZES] + [(3, N) for N in SIZES if N <= 192])
def test_half_spectrum_matches_maps(dim, N, precision, reach):
    if dim == 3 and N > 96 and (precision == "f64" or reach > 1):
        pytest.skip("covered by the smaller grids; keeps the test small")
    L = 8.0
    ctx = sd.Context(dim, precision, 0, sigma_g=2.0 * L / (np.pi * N))
    fx, mv = _shapes(ctx, dim, 60, N + dim, reach)
    rng = np.random.default_rng(np.random.SeedSequence([N, 22]))
    q = torch.tensor(rng.standard_normal((3, 4)) if dim == 3 else
                     np.stack([np.cos([0.0, 0.7, 2.1]), np.zeros(3), np.zeros(3), np.sin([0.0, 0.7, 2.1])], 1),
                     dtype=torch.float64, device="cuda")
    g = sd.Grid(N, L)
    ref = ctx.score_maps(fx, mv, q, g).real.double()
    scale = ref.abs().amax(1)
    # rounding of two transforms of N^dim points: eps log2(N^dim) each, relative to the map's largest value
    tol = 2 * (2.0 ** -23 if precision == "f32" else 2.0 ** -52) * max(4.0, dim * np.log2(N))
    if precision == "f64":  # the sub-box's atomic sums differ between the two runs by rounding too
        tol *= 4
    for k_r in (1, 2, 3, 8, 16):
        if k_r > N ** dim:
            continue
        s, rot, idx = sd.decode_cands(ctx.score_rotations(fx, mv, q, g, k_r=k_r))
        s, idx = s.reshape(3, k_r), idx.reshape(3, k_r).long()
        want = torch.topk(ref, k_r, dim=1).values
        assert ((s - want).abs().amax(1) <= tol * scale).all(), (k_r, ((s - want).abs().amax(1) / scale).tolist())
        assert ((ref.gather(1, idx) - s).abs().amax(1) <= tol * scale).all()
        assert (rot.reshape(3, k_r) == torch.arange(3, device="cuda")[:, None]).all()
        assert all(len(set(r.tolist())) == k_r for r in idx)
    ctx.close()
