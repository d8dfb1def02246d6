"""The 3D SDF passes over the boundary tree against plain FP64 sums: sample counts around the tile
(256) and sub-tile (32) sizes, query counts around a warp, closed solids and open, randomly oriented
sample sets (whose winding numbers fall anywhere, so the full-sum list is used), given memberships."""

import math

import numpy as np
import pytest
import torch

from paper_1712_00238_gb300 import sdfdock as sd

pytestmark = pytest.mark.gpu


def _boundary(kind, n, rng):
    z = 1 - (2 * np.arange(n) + 1) / n
    a = np.arange(n) * math.pi * (3 - math.sqrt(5))
    nrm = np.stack([np.sqrt(1 - z * z) * np.cos(a), np.sqrt(1 - z * z) * np.sin(a), z], 1)
    pos, area = 1.5 * nrm, np.full(n, 4 * math.pi * 2.25 / n)
    if kind == "open":
        pos = pos + 0.3 * rng.standard_normal((n, 3))
        nrm = rng.standard_normal((n, 3))
        nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
        area = area * rng.uniform(0.2, 6.0, n)
    return pos, nrm, area


def _reference(p, q, n, a, pmc=None):
    """|xi|, w / S, rho of Eq. 13 and the summed magnitudes, in FP64."""
    p, q, n, a = (torch.as_tensor(x, device="cuda").double() for x in (p, q, n, a))
    d = p[:, None] - q[None]
    eta = d.norm(dim=2)
    dot = (d * n[None]).sum(2)
    w = -(a * dot / eta ** 3).sum(1) / (4 * math.pi)
    inside = w > 0.5 if pmc is None else torch.as_tensor(pmc, device="cuda") < 0
    dist = eta.amin(1)
    xi = torch.where(inside, -dist, dist)[:, None]
    r = eta / dist[:, None]
    g = torch.exp(-2.0 * (r - 1) ** 2) / (math.sqrt(2 * math.pi) * 0.5) * (r - 1 <= 1.5)
    lam = torch.where(inside, -3.0, 1.0).double()[:, None]
    t = lam / math.sqrt(2 * math.pi) * g * dot / eta * a / torch.complex(xi * xi - eta * eta, 2 * xi * eta)
    return dist, w, t.sum(1), t.abs().sum(1)


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("kind", ["closed", "open", "given"])
@pytest.mark.parametrize("n_b,m", [(1, 1), (31, 33), (32, 31), (33, 300), (255, 64), (257, 65), (2049, 1000), (9000, 4001)])
def test_tree_matches_full_sums(n_b, m, kind, precision):
    rng = np.random.default_rng(np.random.SeedSequence([n_b, m, 7]))
    pos, nrm, area = _boundary("open" if kind == "open" else "closed", n_b, rng)
    real = np.float32 if precision == "f32" else np.float64
    eps = np.finfo(real).eps
    qry = rng.uniform(-2.6, 2.6, (4 * m, 3))
    keep = np.abs(np.linalg.norm(qry, axis=1) - 1.5) > 0.05
    qry = qry[keep][:m]
    pos, nrm, area, qry = (x.astype(real) for x in (pos, nrm, area, qry))
    pmc = np.where(rng.random(m) < 0.5, -1, 1).astype(np.int8) if kind == "given" else None
    dist, w, rho, mag = _reference(qry, pos, nrm, area, pmc)
    # memberships of queries whose exact sum lies within rounding of 1/2 are not defined
    sure = ((w - 0.5).abs() > 1e-4) if pmc is None else torch.ones(m, dtype=torch.bool, device="cuda")
    ctx = sd.Context(3, precision, 0, sigma_g=0.1)
    got = {}
    for level in (2, 0):
        ctx.set_option("sdf_cull", level)
        _, r = ctx.sdf_build(pos, nrm, area, qry, np.ones(m), pmc=pmc, return_rho=True)
        got[level] = torch.view_as_complex(r).clone()
    assert torch.equal(got[2], got[0])
    # a term: distances to a few eps of the coordinates, the exponent (<= 4.5) and its factors: ~100 eps
    tol = 100 * eps * mag.amax() + 30 * eps * rho.abs().amax()
    assert ((got[2] - rho).abs()[sure] <= tol + _edge_terms(qry, pos, nrm, area, dist, eps)[sure]).all()
    ctx.close()


def _edge_terms(p, q, n, a, dist, eps):
    """Magnitude of the terms whose eta / |xi| - 1 lies within rounding of the cut at 1.5."""
    p, q, n, a = (torch.as_tensor(x, device="cuda").double() for x in (p, q, n, a))
    d = p[:, None] - q[None]
    eta = d.norm(dim=2)
    r = eta / dist[:, None]
    near = (r - 2.5).abs() <= 40 * eps
    t = 3 / math.sqrt(2 * math.pi) * torch.exp(-2.0 * (r - 1) ** 2) / (math.sqrt(2 * math.pi) * 0.5) * a / (dist[:, None] ** 2 + eta ** 2)
    return (t * near).sum(1)


def test_tree_distances():
    # SD_PHI_SKIN depends on the signed distance alone
    rng = np.random.default_rng(5)
    pos, nrm, area = _boundary("closed", 3001, rng)
    qry = rng.uniform(-2.6, 2.6, (2000, 3))
    qry = qry[np.abs(np.linalg.norm(qry, axis=1) - 1.5) > 0.05]
    dist, w, _, _ = _reference(qry, pos, nrm, area)
    xi = torch.where(w > 0.5, -dist, dist)
    ctx = sd.Context(3, "f64", 0, phi=3, phi_radius=0.8)
    _, r = ctx.sdf_build(pos, nrm, area, qry, np.ones(len(qry)), return_rho=True)
    g = lambda x: torch.exp(-2.0 * x * x) / (math.sqrt(2 * math.pi) * 0.5)  # noqa: E731
    assert (r[:, 0] - g(xi / 0.8 - 1)).abs().max() < 1e-12
    assert (r[:, 1] - 3 * g(xi / 0.8 + 1)).abs().max() < 1e-12
    ctx.close()
