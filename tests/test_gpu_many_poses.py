"""Gradients and refinement of many poses at once against the same poses a few at a time: many are
finished by a launch of their own, few by the gather's last CTAs, and the samples are cut differently."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


def _setup(dim, precision, w, m):
    rng = np.random.default_rng(np.random.SeedSequence([dim, w, m]))
    ctx = sd.Context(dim, precision, 0, sigma_g=0.4, w=w)
    shapes = []
    for n in (200, m):
        p = np.zeros((n, 4))
        p[:, :dim] = rng.uniform(-1.5, 1.5, (n, dim))
        shapes.append(ctx.shape_from_samples(p, rng.standard_normal((n, 2))))
    return ctx, shapes, sd.Grid(32, 8.0), rng


def _poses(P, dim, rng, real):
    q, t = rng.standard_normal((P, 4)), rng.uniform(-1, 1, (P, 3))
    if dim == 2:
        q[:, 1:3] = 0
        t[:, 2] = 0
    return torch.tensor(q, device="cuda", dtype=real), torch.tensor(t, device="cuda", dtype=real)


# CTAs a pose times poses about the lines: 608 and 1,216 CTAs
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("w,m,P", [(6, 1, 1217), (6, 50, 608), (6, 50, 609), (6, 130, 1300), (4, 700, 500), (8, 65, 1217),
                                   (12, 257, 650)])
def test_gradients_of_many_poses(w, m, P, dim, precision):
    ctx, (fx, mv), g, rng = _setup(dim, precision, w, m)
    q, t = _poses(P, dim, rng, ctx.real)
    many = ctx.score_grad(fx, mv, g, q, t)
    few = [ctx.score_grad(fx, mv, g, q[i:i + 7].contiguous(), t[i:i + 7].contiguous()) for i in range(0, P, 7)]
    eps = torch.finfo(ctx.real).eps
    for a, b in zip(many, (torch.cat(x) for x in zip(*few))):
        # the same m products in another order: the running sums' rounding, m eps of the largest at worst
        assert (a - b).abs().max() <= (8 + m) * eps * b.abs().max()
    ctx.close()


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("method", [sd.REFINE_ASCENT, sd.REFINE_CG, sd.REFINE_DYNAMICS])
def test_refinement_of_many_poses(method, dim, precision):
    P, m, steps = 1300, 40, 4
    ctx, (fx, mv), g, rng = _setup(dim, precision, 6, m)
    q, t = _poses(P, dim, rng, ctx.real)
    if dim == 2:
        t = t[:, :2].contiguous()
    kw = dict(steps=steps, method=method, lr_t=0.01, lr_q=0.01, mass=50.0, inertia=50.0, dt=0.05)
    n0 = sd.launch_count()
    many = ctx.refine(fx, mv, g, q, t, **kw)
    n1 = sd.launch_count()
    few = [ctx.refine(fx, mv, g, q[i:i + 100], t[i:i + 100], **kw) for i in range(0, P, 100)]
    n2 = sd.launch_count()
    per_few = (n2 - n1) // 13
    assert per_few == steps + 1                 # a launch a step
    assert n1 - n0 >= 2 * (steps + 1)           # two, and the tables of the first call
    qf, tf, hf = torch.cat([x[0] for x in few]), torch.cat([x[1] for x in few]), torch.cat([x[2] for x in few], 1)
    eps = torch.finfo(ctx.real).eps
    # the sums' rounding (m eps) through four updates; the ascent divides by its largest gradient entry
    # and CG by its direction's length, so poses with a small gradient carry it enlarged
    tol = 4 * 100 * m * eps
    assert (many[2][0] - hf[0]).abs().max() <= (8 + m) * eps * hf[0].abs().max()
    worst = torch.maximum((many[0] - qf).abs().amax(1), (many[1] - tf).abs().amax(1))
    assert (worst <= tol).float().mean() > 0.98 and worst.median() <= tol / 20
    ctx.close()
