"""A search captured by the caller whose product table does not exist yet (the fixed shape has met the
grid through another call only): the table belongs to the shape, not to the graph."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


# N = 48: full passes only; 64: pruned ones
@pytest.mark.parametrize("dim,N", [(2, 48), (3, 48), (3, 64)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_captured_first_search(dim, N, precision):
    L = 8.0
    rng = np.random.default_rng(np.random.SeedSequence([dim, N]))
    ctx = sd.Context(dim, precision, 0, sigma_g=2.0 * L / (np.pi * N))

    def shape(seed, m=300):
        r = np.random.default_rng(seed)
        p = np.zeros((m, 4))
        p[:, :dim] = r.uniform(-0.6, 0.6, (m, dim))
        return ctx.shape_from_samples(p, r.standard_normal((m, 2)))

    other, fixed, twin, moving = shape(1), shape(2), shape(2), shape(3)
    q = rng.standard_normal((5, 4))
    if dim == 2:
        q[:, 1:3] = 0
    q = torch.tensor(q, device="cuda")
    g = sd.Grid(N, L)
    want = ctx.score_rotations(twin, moving, q, g).clone()
    ctx.score_rotations(other, moving, q, g)  # the kernels and the workspace are there
    ctx.score_maps(fixed, moving, q, g)       # and the fixed shape's spectrum
    out = torch.zeros_like(want)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        ctx.score_rotations(fixed, moving, q, g, out=out)
    assert not out.any()
    # the spreading's atomic sums come in any order: as the comparisons of two runs elsewhere allow
    tol = 2e-6 if precision == "f32" else 1e-12

    def check(got):
        (s, r, i), (ws, wr, wi) = sd.decode_cands(got), sd.decode_cands(want)
        assert (s - ws).abs().max() <= tol * ws.abs().max() and torch.equal(r, wr) and torch.equal(i, wi)

    for _ in range(2):
        out.zero_()
        graph.replay()
        check(out)
    del graph
    torch.cuda.synchronize()
    check(ctx.score_rotations(fixed, moving, q, g))  # the table outlives the graph
    ctx.close()
