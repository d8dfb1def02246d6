"""3D SDF builds on both sides of the line between all pairs and the boundary tree, against plain FP64
sums on a sample of the queries: partial sub-tiles and tiles, several tiles, closed solids and open
sample sets.  Each side launches its own kernels."""

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd
from test_gpu_sdf_tree import _boundary, _edge_terms, _reference

pytestmark = pytest.mark.gpu


def _queries(m, rng):
    q = np.zeros((0, 3))
    while len(q) < m:
        x = rng.uniform(-2.6, 2.6, (m + 1000, 3))
        q = np.concatenate([q, x[np.abs(np.linalg.norm(x, axis=1) - 1.5) > 0.05]])
    return q[:m]


@pytest.mark.parametrize("kind", ["closed", "open"])
@pytest.mark.parametrize("precision,n_b", [("f32", 40), ("f32", 257), ("f32", 2049), ("f32", 9000), ("f32", 60001),
                                           ("f64", 40), ("f64", 257), ("f64", 2049), ("f64", 25001)])
def test_both_routes_match_full_sums(precision, n_b, kind):
    rng = np.random.default_rng(np.random.SeedSequence([n_b, 31]))
    pos, nrm, area = _boundary(kind, n_b, rng)
    real = np.float32 if precision == "f32" else np.float64
    eps = np.finfo(real).eps
    last = 3300 + 60000000 // n_b if precision == "f32" else 500 + 25000000 // n_b  # all pairs up to here
    qry = _queries(last + 1, rng)
    pos, nrm, area, qry = (x.astype(real) for x in (pos, nrm, area, qry))
    pick = rng.choice(last, min(last, 2000, 40000000 // n_b), replace=False)
    dist, w, rho, mag = _reference(qry[pick], pos, nrm, area)
    # memberships of queries whose exact sum lies within rounding of 1/2 are not defined
    sure = (w - 0.5).abs() > (1e-4 if n_b < 50000 else 1e-3)
    assert sure.sum() > 0.9 * len(pick)
    ctx = sd.Context(3, precision, 0, sigma_g=0.1)
    launches = []
    for m in (last, last + 1):
        n0 = sd.launch_count()
        s, r = ctx.sdf_build(pos, nrm, area, qry[:m], np.ones(m), return_rho=True)
        launches.append(sd.launch_count() - n0)
        got = torch.view_as_complex(r)[torch.as_tensor(pick, device="cuda")]
        # as the tree's own test: ~100 eps of a term, and terms within rounding of the cut
        tol = 100 * eps * mag.amax() + 30 * eps * rho.abs().amax()
        assert ((got - rho).abs()[sure] <= tol + _edge_terms(qry[pick], pos, nrm, area, dist, eps)[sure]).all(), m
        s.free()
    assert launches[1] == launches[0] + 2  # nodes, tree, two of the list; pairs and their finish
    ctx.close()


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("m", [1, 31, 33, 257, 600])
def test_few_queries_take_all_pairs(m, precision):
    # distances and memberships alone (SD_PHI_SKIN), given memberships included
    rng = np.random.default_rng(m)
    pos, nrm, area = _boundary("closed", 20000, rng)
    qry = _queries(m, rng)
    real = np.float32 if precision == "f32" else np.float64
    pos, nrm, area, qry = (x.astype(real) for x in (pos, nrm, area, qry))
    ctx = sd.Context(3, precision, 0, phi=3, phi_radius=0.8)
    for pmc in (None, np.where(rng.random(m) < 0.5, -1, 1).astype(np.int8)):
        dist, w, _, _ = _reference(qry, pos, nrm, area)
        inside = w > 0.5 if pmc is None else torch.as_tensor(pmc, device="cuda") < 0
        xi = torch.where(inside, -dist, dist)
        _, r = ctx.sdf_build(pos, nrm, area, qry, np.ones(m), pmc=pmc, return_rho=True)
        g = lambda x: torch.exp(-2.0 * x * x) / (np.sqrt(2 * np.pi) * 0.5)  # noqa: E731
        tol = 1e-12 if precision == "f64" else 2e-5  # the distance's rounding times g's slope (< 1), a few eps
        assert (r[:, 0].double() - g(xi / 0.8 - 1)).abs().max() < tol
        assert (r[:, 1].double() - 3 * g(xi / 0.8 + 1)).abs().max() < tol
    ctx.close()


# splits of the truncated sum: 16 x 152 CTAs shared out among groups of 32 queries, four tiles a split
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("n_b,m", [(2047, 40), (2048, 40), (2304, 33), (20001, 1), (20001, 700), (70000, 300)])
def test_split_sums_match_full_sums(n_b, m, precision):
    rng = np.random.default_rng(np.random.SeedSequence([n_b, m, 33]))
    real = np.float32 if precision == "f32" else np.float64
    eps = np.finfo(real).eps
    for kind in ("closed", "open"):
        pos, nrm, area = _boundary(kind, n_b, rng)
        qry = _queries(m, rng)
        pos, nrm, area, qry = (x.astype(real) for x in (pos, nrm, area, qry))
        dist, w, rho, mag = _reference(qry, pos, nrm, area)
        sure = (w - 0.5).abs() > (1e-4 if n_b < 50000 else 1e-3)
        ctx = sd.Context(3, precision, 0, sigma_g=0.1)
        n0 = sd.launch_count()
        _, r = ctx.sdf_build(pos, nrm, area, qry, np.ones(m), return_rho=True)
        launches = sd.launch_count() - n0
        got = torch.view_as_complex(r)
        tol = 100 * eps * mag.amax() + 30 * eps * rho.abs().amax()
        assert ((got - rho).abs()[sure] <= tol + _edge_terms(qry, pos, nrm, area, dist, eps)[sure]).all()
        ctx.set_option("sdf_cull", 0)
        _, r0 = ctx.sdf_build(pos, nrm, area, qry, np.ones(m), return_rho=True)
        assert torch.equal(torch.view_as_complex(r0), got)  # what the boxes leave out adds nothing
        # the launches of a build whose boundary is too small to split, and one that adds the splits
        n0 = sd.launch_count()
        ctx.sdf_build(pos[:1000], nrm[:1000], area[:1000], qry, np.ones(m))
        assert launches == sd.launch_count() - n0 + 1
        ctx.close()
