"""Performance cases: the calls a user of the library makes, over the range of sizes they are made at.

Kinds of case, each through the public Python binding:

* ``search``  - score_rotations: the best translation(s) of every rotation (one NUFFT each).
* ``pairs``   - score_pairs: several shape pairs on their own grids in one launch sequence.
* ``sdf``     - sdf_build: a shape's sampled density from oriented boundary samples.
* ``rescore`` - top_k_poses: global top-k of a candidate list with the FP64 re-score.
* ``grad``    - SdfScore forward and backward: score and pose gradient, as in a training loop.
* ``refine``  - Context.refine: on-device pose refinement.

Shapes (made from the seed on the GPU): ``spheres``, molecule-like packings of n spheres with radii
in [1.2, 2.0], 64 boundary samples and 40 density samples per sphere in a band of 2 (the docking and
uneven-batch workloads); ``peg``, a cylinder and a block with a blind bore, density samples in a
0.3 band (the mechanical workload); ``square``, a square peg and a plate with a square hole (2D).
"""

import math

import numpy as np
import torch

from paper_1712_00238_gb300 import sdfdock as sd

CUDA = "cuda:0"
PER_SPHERE, BND_PER_SPHERE = 40, 64
W = 6  # spreading width of every context (the library's default)


def listed():
    return [
        # the 2D peg-in-hole workload: FP64 throughout, 64 planar rotations, everything fits in L2
        dict(name="search_2d_f64", kind="search", shape="square", f64=True, m1=3700, m2=3500, N=128, L=6.6,
             sigma_g=0.02, n_r=64, k_r=1, tuned=False),
        # the smallest 3D call (a quick look at a coarse grid): latency and launches
        dict(name="search_tiny_3d", kind="search", shape="peg", f64=False, m1=1500, m2=1500, N=32, L=10.9,
             sigma_g=0.25, n_r=12, k_r=1, tuned=False),
        # small molecules, the four best translations of each rotation, library defaults
        dict(name="search_top4_96", kind="search", shape="spheres", f64=False, n1=203, n2=57, N=96, L=0.0,
             sigma_g=0.6, n_r=77, k_r=4, tuned=False),
        # the mechanical workload: 576 rotations x 128^3, autotuned and replayed as a graph
        dict(name="search_peg_128", kind="search", shape="peg", f64=False, m1=52636, m2=50342, N=128, L=10.9,
             sigma_g=0.03, n_r=576, k_r=1, tuned=True),
        # the docking workload (the largest single-pair search), a shard of its rotations
        dict(name="search_docking_192", kind="search", shape="spheres", f64=False, n1=2000, n2=500, N=192,
             L=153.6, sigma_g=0.6, n_r=600, k_r=1, tuned=True),
        # two large molecules on the largest grid, library defaults, an odd number of rotations
        dict(name="search_large_256", kind="search", shape="spheres", f64=False, n1=4500, n2=2900, N=256,
             L=0.0, sigma_g=0.6, n_r=45, k_r=1, tuned=False),
        # pairs of uneven sizes in one call (the uneven batch): grids 96, 128, 192 and 256, autotuned
        dict(name="pairs_uneven", kind="pairs", sigma_g=0.6, n_r=48, n1a=120, n2a=60, Na=96, n1b=900, n2b=210,
             Nb=128, n1c=310, n2c=1500, Nc=192, n1d=4100, n2d=1700, Nd=256),
        # density of the peg: 20,000 boundary samples, every query's nearest distance, membership and sum
        dict(name="sdf_peg", kind="sdf", shape="peg", f64=False, n_b=20000, m=50342),
        # density of a 5,000-sphere molecule (320,000 boundary samples)
        dict(name="sdf_spheres_5000", kind="sdf", shape="spheres", f64=False, n=5000, m=199433),
        # the docking search's last step: top 100 of 54,000 candidates, FP64 pair sums
        dict(name="rescore_docking_100", kind="rescore", n1=2000, n2=500, N=192, L=153.6, sigma_g=0.6,
             n_cand=54000, k=100),
        # gradient-driven refinement through autograd: 256 poses on the docking pair
        dict(name="grad_docking_256", kind="grad", n1=2000, n2=500, N=192, L=153.6, sigma_g=0.6, P=256),
        # refinement of a search's ten best poses on the device, small molecules
        dict(name="refine_10", kind="refine", n1=203, n2=57, N=96, L=0.0, sigma_g=0.6, P=10, steps=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(n1, n2):
    """Smallest grid with a spacing of at most 0.8 for two packings (the uneven batch's rule)."""
    L = _box(n1, n2)
    for N in (64, 96, 128, 192, 256):
        if L / N <= 0.8:
            return N
    return 256


def draw(rng):
    kind = rng.choice(["search", "search", "search", "search2d", "pairs", "sdf", "sdf", "rescore", "grad", "refine"])
    if kind == "search2d":
        m = _log(rng, 300, 6000)
        return dict(kind="search", shape="square", f64=True, m1=m + rng.randrange(90), m2=m,
                    N=rng.choice([32, 48, 64, 96, 128, 192, 256]), L=6.6, sigma_g=0.05, n_r=_log(rng, 5, 130),
                    k_r=rng.choice([1, 1, 3]), tuned=False)
    if kind == "search" and rng.random() < 0.3:
        m = _log(rng, 1200, 60000)
        N = rng.choice([48, 64, 96, 128])
        return dict(kind="search", shape="peg", f64=False, m1=m + rng.randrange(1000), m2=m, N=N, L=10.9,
                    sigma_g=8.0 / N, n_r=_log(rng, 8, 400), k_r=rng.choice([1, 1, 1, 2]), tuned=rng.random() < 0.5)
    if kind == "search":
        n1, n2 = _log(rng, 50, 5000), _log(rng, 50, 3000)
        N = _grid(n1, n2)
        n_r = _log(rng, 6, max(8, int(600 * min(1.0, (192 / N) ** 3 / 1.2))))
        return dict(kind="search", shape="spheres", f64=False, n1=n1, n2=n2, N=N, L=0.0, sigma_g=0.6, n_r=n_r,
                    k_r=rng.choice([1, 1, 1, 4]), tuned=rng.random() < 0.5)
    if kind == "pairs":
        c = dict(kind="pairs", sigma_g=0.6, n_r=_log(rng, 6, 48))
        for j in "abcd":
            n1, n2 = _log(rng, 50, 4000), _log(rng, 50, 1800)
            c.update({"n1" + j: n1, "n2" + j: n2, "N" + j: _grid(n1, n2)})
        return c
    if kind == "sdf":
        if rng.random() < 0.5:
            n_b = _log(rng, 500, 40000)
            return dict(kind="sdf", shape="peg", f64=rng.random() < 0.2 and n_b < 5000, n_b=n_b, m=_log(rng, 900, 60000))
        n = _log(rng, 50, 4900)
        return dict(kind="sdf", shape="spheres", f64=False, n=n, m=PER_SPHERE * n - rng.randrange(40))
    n1, n2 = _log(rng, 100, 2000), _log(rng, 50, 500)
    c = dict(kind=kind, n1=n1, n2=n2, N=_grid(n1, n2), L=0.0, sigma_g=0.6)
    if kind == "rescore":
        return dict(c, n_cand=_log(rng, 500, 54000), k=_log(rng, 4, 100))
    if kind == "grad":
        return dict(c, P=_log(rng, 3, 256))
    return dict(c, P=_log(rng, 2, 64), steps=rng.randrange(5, 26))


# ---------------------------------------------------------------------------
# shapes
# ---------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=CUDA)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=CUDA, dtype=torch.float64)


def _radius(n):
    """Bounding radius of a packing of n spheres with its band of density samples."""
    return 3.0 * n ** (1 / 3) + 4.6


def _box(n1, n2):
    return 2.0 * (_radius(n1) + _radius(n2)) + 2.0


def _directions(g, n):
    z = 2 * _rand(g, n) - 1
    a = 2 * math.pi * _rand(g, n)
    s = torch.sqrt(1 - z * z)
    return torch.stack([s * torch.cos(a), s * torch.sin(a), z], 1)


def _centres(g, n):
    """n sphere centres and radii: a jittered lattice of spacing 4.8, the n points nearest the origin."""
    k = int(math.ceil(0.75 * n ** (1 / 3))) + 2
    ax = torch.arange(-k, k + 1, device=CUDA, dtype=torch.float64) * 4.8
    p = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    p = p + 0.6 * (_rand(g, p.shape[0], 3) - 0.5)
    order = torch.argsort((p * p).sum(1))[:n]
    return p[order].contiguous(), 1.2 + 0.8 * _rand(g, n)


def _sphere_boundary(g, cen, rad):
    i = torch.arange(BND_PER_SPHERE, device=CUDA, dtype=torch.float64)
    z = 1 - (2 * i + 1) / BND_PER_SPHERE
    s = torch.sqrt(1 - z * z)
    a = i * math.pi * (3 - math.sqrt(5)) + 2 * math.pi * _rand(g, cen.shape[0], 1)
    nrm = torch.stack([s * torch.cos(a), s * torch.sin(a), z.expand_as(a)], -1)
    pos = cen[:, None] + rad[:, None, None] * nrm
    area = (4 * math.pi / BND_PER_SPHERE) * (rad * rad)[:, None].expand(-1, BND_PER_SPHERE)
    return pos.reshape(-1, 3), nrm.reshape(-1, 3), area.reshape(-1).contiguous()


def _sphere_queries(g, cen, rad, m):
    """m points in the band 0.7 <= |d| <= 2 of the union's surface: positions, signed distance, cell volume."""
    out = []
    left = m
    while left > 0:
        k = 2 * left + 64
        i = torch.randint(cen.shape[0], (k,), generator=g, device=CUDA)
        r = (_rand(g, k) * (rad[i] + 2.0) ** 3) ** (1 / 3)
        p = cen[i] + r[:, None] * _directions(g, k)
        d = torch.cat([(torch.cdist(q.float(), cen.float()) - rad.float()).amin(1) for q in p.split(16384)]).double()
        keep = (d.abs() >= 0.7) & (d.abs() <= 2.0)
        out.append(torch.cat([p[keep], d[keep, None]], 1)[:left])
        left -= out[-1].shape[0]
    q = torch.cat(out)
    vol = (4.8 ** 3 / PER_SPHERE) * (0.8 + 0.4 * _rand(g, m))
    return q[:, :3].contiguous(), q[:, 3].contiguous(), vol


def _cylinder(p):
    r = torch.hypot(p[:, 0], p[:, 1]) - 1.0
    z = p[:, 2].abs() - 1.5
    return torch.maximum(r, z).clamp_max(0) + torch.hypot(r.clamp_min(0), z.clamp_min(0))


def _block(p):
    e = p.abs() - torch.tensor([3.0, 3.0, 2.0], device=CUDA, dtype=torch.float64)
    box = e.amax(1).clamp_max(0) + e.clamp_min(0).norm(dim=1)
    bore = torch.maximum(torch.hypot(p[:, 0], p[:, 1]) - 1.02, -0.5 - p[:, 2])
    return torch.maximum(box, -bore)


def _square(p):
    e = p.abs() - 0.5
    return e.amax(1).clamp_max(0) + e.clamp_min(0).norm(dim=1)


def _plate(p):
    e, h = p.abs() - 2.0, p.abs() - 0.525
    return torch.maximum(e.amax(1).clamp_max(0) + e.clamp_min(0).norm(dim=1), -h.amax(1))


def _band_queries(g, dist, half, m, lo, band):
    """m points of a box with lo <= |distance| <= band: positions, signed distance, cell volume."""
    h = torch.tensor(half, device=CUDA, dtype=torch.float64)
    out, left = [], m
    seen = kept = 0
    while left > 0:
        p = (2 * _rand(g, 8 * left + 64, len(half)) - 1) * h
        d = dist(p)
        keep = (d.abs() >= lo) & (d.abs() <= band)
        seen, kept = seen + p.shape[0], kept + int(keep.sum())
        out.append(torch.cat([p[keep], d[keep, None]], 1)[:left])
        left -= out[-1].shape[0]
    q = torch.cat(out)
    cell = float(np.prod([2 * x for x in half])) * kept / seen / m
    return q[:, :-1].contiguous(), q[:, -1].contiguous(), cell * (0.9 + 0.2 * _rand(g, m))


def _cylinder_boundary(g, n):
    """Area-uniform samples of the cylinder (r = 1, length 3): side, then the two caps."""
    k = int(round(n * 0.75))
    off = _rand(g, 4)
    i = torch.arange(n, device=CUDA, dtype=torch.float64)
    u, v = (i * 0.7548776662466927 + off[0]) % 1.0, (i * 0.5698402909980532 + off[1]) % 1.0
    a = 2 * math.pi * u
    r = torch.sqrt(v)
    up = torch.where((torch.arange(n, device=CUDA) % 2) == 0, 1.0, -1.0).double()
    side = (torch.arange(n, device=CUDA) < k)[:, None]
    zero = torch.zeros_like(a)
    pos = torch.where(side, torch.stack([torch.cos(a), torch.sin(a), 3 * v - 1.5], 1),
                      torch.stack([r * torch.cos(a), r * torch.sin(a), 1.5 * up], 1))
    nrm = torch.where(side, torch.stack([torch.cos(a), torch.sin(a), zero], 1), torch.stack([zero, zero, up], 1))
    area = torch.where(side[:, 0], 6 * math.pi / k, 2 * math.pi / max(1, n - k)).to(torch.float64)
    return pos, nrm, area


def _density(d, vol, radius):
    """Weights rho v with the pattern of a skeletal density near a surface of the given curvature radius:
    mostly imaginary (on the medial axis zeta^2 is), +lambda2 / sigma inside, -lambda1 / sigma outside times
    the share of the directions in which the solid is seen."""
    seen = 1.0 - torch.sqrt(1.0 - (radius / (radius + d.clamp_min(0.0))) ** 2)
    mag = torch.where(d > 0, -2.0 * 0.5 * seen, 6.0 / (1.0 + 0.3 / radius)) * vol
    return torch.stack([0.2 * mag * torch.cos(2 * d), mag], 1)


def _samples(case, which, seed):
    """Positions, weights (both in the context's precision) of the fixed (1) or moving (2) shape."""
    g = _gen(seed, 10 + which)
    kind = case.get("shape", "spheres")
    if kind == "spheres":
        n = case["n%d" % which]
        cen, rad = _centres(g, n)
        p, d, vol = _sphere_queries(g, cen, rad, PER_SPHERE * n)
    elif kind == "peg":
        m = case["m%d" % which]
        if which == 1:
            p, d, vol = _band_queries(g, _block, (3.3, 3.3, 2.3), m, 0.05, 0.3)
        else:
            p, d, vol = _band_queries(g, _cylinder, (1.3, 1.3, 1.8), m, 0.04, 0.3)
    else:
        m = case["m%d" % which]
        half = 2.3 if which == 1 else 0.8
        p, d, vol = _band_queries(g, _plate if which == 1 else _square, (half, half), m, 0.01, 9.0)
    real = torch.float64 if case.get("f64") else torch.float32
    pos = torch.zeros((p.shape[0], 4), dtype=real, device=CUDA)
    pos[:, : p.shape[1]] = p
    return pos, _density(d, vol, {"spheres": 1.6, "peg": 1.0, "square": 4.0}[kind]).to(real)


def _quats(case, seed, n):
    g = _gen(seed, 3)
    if case.get("shape") == "square":  # planar rotations, evenly spaced
        a = math.pi * (torch.arange(n, device=CUDA, dtype=torch.float64) + _rand(g, 1)) / n
        q = torch.zeros((n, 4), dtype=torch.float64, device=CUDA)
        q[:, 0], q[:, 3] = torch.cos(a), torch.sin(a)
        return q
    u = _rand(g, 3, n)
    a, b, r, s = 2 * math.pi * u[1], 2 * math.pi * u[2], torch.sqrt(1 - u[0]), torch.sqrt(u[0])
    return torch.stack([r * torch.sin(a), r * torch.cos(a), s * torch.sin(b), s * torch.cos(b)], 1).contiguous()


def _start_poses(case, seed, P):
    """Rotations and translations within 10 of the receptor's centre (the refinement workload's starts)."""
    g = _gen(seed, 5)
    t = _directions(g, P) * (10.0 * _rand(g, P, 1) ** (1 / 3))
    return _quats(case, seed, P).float().contiguous(), t.float().contiguous()


def _side(case):
    return case["L"] if case["L"] > 0 else _box(case["n1"], case["n2"])


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

class State:
    """What a program keeps between calls; closing the context gives its device memory back."""

    def __init__(self, case):
        dim = 2 if case.get("shape") == "square" else 3
        sigma = {"sigma_g": case["sigma_g"]} if "sigma_g" in case else {}
        self.case = case
        self.ctx = sd.Context(dim, "f64" if case.get("f64") else "f32", 0, **sigma)
        self.stream = None
        if case.get("tuned") or case["kind"] == "pairs":  # as the benchmark runs: plans tuned, launches replayed
            self.ctx.set_option("autotune", 1)
            self.ctx.set_option("graph", 1)
            self.stream = torch.cuda.Stream()

    def __del__(self):
        self.ctx.close()


def _pair_cases(case):
    return [dict(shape="spheres", n1=case["n1" + j], n2=case["n2" + j], N=case["N" + j],
                 L=_box(case["n1" + j], case["n2" + j])) for j in "abcd"]


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "sdf":
        real = torch.float64 if case["f64"] else torch.float32
        g = _gen(seed, 1)
        if case["shape"] == "peg":
            b = _cylinder_boundary(g, case["n_b"])
            h_b = math.sqrt(8 * math.pi / case["n_b"])
            p, _, vol = _band_queries(g, _cylinder, (1.3, 1.3, 1.8), case["m"], min(h_b, 0.25), 0.3)
        else:
            cen, rad = _centres(g, case["n"])
            b = _sphere_boundary(g, cen, rad)
            p, _, vol = _sphere_queries(g, cen, rad, case["m"])
        pad = lambda x: torch.nn.functional.pad(x, (0, 4 - x.shape[1])).to(real).contiguous()  # noqa: E731
        s.args = (pad(b[0]), pad(b[1]), b[2].to(real).contiguous(), pad(p), vol.to(real).contiguous())
        torch.cuda.synchronize()
        return s
    if kind == "pairs":
        s.jobs = []
        for j, c in enumerate(_pair_cases(case)):
            fx, mv = (s.ctx.shape_from_samples(*_samples(c, k, seed * 7 + j)) for k in (1, 2))
            s.jobs.append((fx, mv, _quats(c, seed * 7 + j, case["n_r"]), sd.Grid(c["N"], c["L"])))
        s.outs = [torch.empty((case["n_r"], sd.CAND_BYTES), dtype=torch.uint8, device=CUDA) for _ in s.jobs]
        torch.cuda.synchronize()
        return s
    s.fixed, s.moving = (s.ctx.shape_from_samples(*_samples(case, k, seed)) for k in (1, 2))
    s.grid = sd.Grid(case["N"], _side(case))
    if kind == "search":
        s.quats = _quats(case, seed, case["n_r"])
        s.out = torch.empty((case["n_r"] * case["k_r"], sd.CAND_BYTES), dtype=torch.uint8, device=CUDA)
    elif kind == "rescore":
        # candidates of a finished search: one per rotation, the best of them in contact with the receptor
        g = _gen(seed, 4)
        n, N = case["n_cand"], case["N"]
        s.quats = _quats(case, seed, n)
        reach = (0.35 + 0.5 * _rand(g, n, 1)) * (_radius(case["n1"]) + _radius(case["n2"]))
        cell = torch.round(_directions(g, n) * reach * (N / s.grid.L)).long() % N
        cell = (cell + N // 2) % N
        rec = torch.zeros((n, 2), dtype=torch.float64, device=CUDA)
        rec[:, 0] = 100 * _rand(g, n)
        ri = rec.view(torch.int32).reshape(n, 4)
        ri[:, 2] = torch.arange(n, device=CUDA, dtype=torch.int32)
        ri[:, 3] = ((cell[:, 2] * N + cell[:, 1]) * N + cell[:, 0]).int()
        s.cand = rec.view(torch.uint8).reshape(n, 16)
    else:
        s.q, s.t = _start_poses(case, seed, case["P"])
    torch.cuda.synchronize()
    return s


def _cands(buf, f64):
    """Scores, rotations and translation indices of candidate records.  An FP32 context computes its
    scores in FP32 (the record only carries them in a 64-bit field): they are handed on as such."""
    score, rot, idx = sd.decode_cands(buf)
    return [score if f64 else score.float(), rot, idx]


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "search":
        if s.stream is None:
            return _cands(s.ctx.score_rotations(s.fixed, s.moving, s.quats, s.grid, k_r=case["k_r"]), case["f64"])
        with torch.cuda.stream(s.stream):
            s.ctx.score_rotations(s.fixed, s.moving, s.quats, s.grid, k_r=case["k_r"], out=s.out)
            return _cands(s.out, case["f64"])
    if kind == "pairs":
        with torch.cuda.stream(s.stream):
            outs, _ = s.ctx.score_pairs(s.jobs, outs=s.outs, stats=False)
            return [_cands(o, False) for o in outs]
    if kind == "sdf":
        shape, rho = s.ctx.sdf_build(*s.args, return_rho=True)
        shape.free()
        s.ctx.shapes.remove(shape)
        return rho
    if kind == "rescore":
        poses = s.ctx.top_k_poses(s.cand, case["k"], s.fixed, s.moving, s.quats, s.grid, rescore_fp64=True)
        return {key: np.array([p[key] for p in poses]) for key in ("score", "score_fp64", "score_fp64_im", "rot", "idx", "t")}
    if kind == "grad":
        q, t = s.q.detach().requires_grad_(True), s.t.detach().requires_grad_(True)
        score = sd.sdf_score(s.ctx, s.fixed, s.moving, s.grid, q, t)
        gq, gt = torch.autograd.grad(score.sum(), (q, t))
        return [score.detach(), gq, gt]
    q, t, hist = s.ctx.refine(s.fixed, s.moving, s.grid, s.q, s.t, case["steps"], method=sd.REFINE_ASCENT,
                              lr_t=0.05, lr_q=0.002)
    return [q, t, hist]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _search_work(dim, m1, m2, N, n_r, k_r, L, r2, real):
    """Samples, quaternions and the fixed spectrum in, candidates out; spreading, and the line transforms
    (5 n log2 n operations each) of the rotated shape's sub-box forward and of the kept modes back."""
    n = 2 * N
    s = min(2 * (int(r2 * n / L + W / 2) + 2), n)
    fwd, inv = 5 * n * math.log2(n), 5 * N * math.log2(N)
    if dim == 2:
        lines = s * fwd + N * (fwd + inv) + N * inv
    else:
        lines = (s * s + s * N + N * N) * fwd + 3 * N * N * inv
    flops = n_r * (lines + m2 * 4.0 * W ** dim + 6.0 * N ** dim)
    return (m1 + m2) * 6 * real + n_r * 32 + N ** dim * 2 * real + n_r * k_r * 16, flops


def work(case):
    kind = case["kind"]
    if kind == "search":
        real = 8 if case["f64"] else 4
        if case["shape"] == "spheres":
            m1, m2 = PER_SPHERE * case["n1"], PER_SPHERE * case["n2"]
            b, f = _search_work(3, m1, m2, case["N"], case["n_r"], case["k_r"], _side(case), _radius(case["n2"]), real)
        else:
            dim, r2 = (2, 1.1) if case["shape"] == "square" else (3, 2.1)
            b, f = _search_work(dim, case["m1"], case["m2"], case["N"], case["n_r"], case["k_r"], case["L"], r2, real)
        return {"bytes": b, "flops": f}
    if kind == "pairs":
        got = [_search_work(3, PER_SPHERE * c["n1"], PER_SPHERE * c["n2"], c["N"], case["n_r"], 1, c["L"],
                            _radius(c["n2"]), 4) for c in _pair_cases(case)]
        return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}
    if kind == "sdf":
        real = 8 if case["f64"] else 4
        n_b = case["n_b"] if case["shape"] == "peg" else BND_PER_SPHERE * case["n"]
        # the density's own sum reaches a small share of the pairs: 32 neighbours per query, 40 operations each
        return {"bytes": (9 * n_b + 7 * case["m"]) * real, "flops": case["m"] * 32.0 * 40}
    m1, m2 = PER_SPHERE * case["n1"], PER_SPHERE * case["n2"]
    if kind == "rescore":
        # samples and candidates in; each moving sample of a pose meets about 64 fixed ones within the cutoff
        return {"bytes": (m1 + m2) * 24 + case["n_cand"] * 16, "flops": case["k"] * m2 * 64.0 * 30}
    evals = case["P"] * (case.get("steps", 0) + 1)
    # samples, the fields on the oversampled grid once, poses in and gradients out
    return {"bytes": m2 * 24 + 32.0 * (2 * case["N"]) ** 3 + case["P"] * 60, "flops": evals * m2 * (16.0 * W ** 3 + 60)}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definitions
# ---------------------------------------------------------------------------

def _modes(N):
    return torch.fft.fftfreq(N, 1.0 / N, device=CUDA, dtype=torch.float64)


def _nudft(x, c, N, L, sign):
    """sum_j c_j exp(sign i k.x_j) on the modes, axes (z, y, x) or (y, x)."""
    k = 2 * math.pi * _modes(N) / L
    E = [torch.exp(1j * sign * x[:, a:a + 1] * k) for a in range(x.shape[1])]
    if x.shape[1] == 2:
        return (c[:, None] * E[1]).T @ E[0]
    return torch.stack([((c * E[2][:, z])[:, None] * E[1]).T @ E[0] for z in range(N)])


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([w * w + x * x - y * y - z * z, 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), w * w - x * x + y * y - z * z, 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), w * w - x * x - y * y + z * z], -1).reshape(3, 3)


def _exact_in(case, seed, dim):
    out = []
    for k in (1, 2):
        p, c = _samples(case, k, seed)
        out += [p[:, :dim].double(), torch.view_as_complex(c.double().contiguous())]
    return out


def _spectrum(p1, c1, N, L, sigma, dim):
    """exp(-s^2 |k|^2) F1 / L^d on the modes |kappa| < N/2."""
    kap = _modes(N)
    g = torch.exp(-(sigma * 2 * math.pi * kap / L) ** 2) * (kap > -N / 2)
    A = _nudft(p1, c1, N, L, -1) / L ** dim
    for a in range(dim):
        A = A * g.reshape([-1 if b == a else 1 for b in range(dim)])
    return A


def _exact_search(case, seed):
    dim = 2 if case["shape"] == "square" else 3
    N, L, k_r = case["N"], _side(case), case["k_r"]
    p1, c1, p2, c2 = _exact_in(case, seed, dim)
    if 8.0 * N ** dim * (p1.shape[0] + case["n_r"] * p2.shape[0]) > 5e12:
        return None
    A = _spectrum(p1, c1, N, L, case["sigma_g"], dim)
    sgn = 1.0 - 2.0 * (_modes(N).abs() % 2)
    for a in range(dim):
        A = A * sgn.reshape([-1 if b == a else 1 for b in range(dim)])
    best = []
    for q in _quats(case, seed, case["n_r"]):
        y = p2 @ _rotation(q)[:dim, :dim].T
        m = torch.fft.ifftn(A * _nudft(y, c2, N, L, 1)).real.reshape(-1) * N ** dim
        best.append(torch.topk(m, k_r).values)
    return [torch.cat(best), None, None]


def _exact_sdf(case, seed):
    s = prepare(case, seed)
    if s.args[0].shape[0] * case["m"] > 2e9:
        return None
    bnd, nrm, area, qry, _ = (x.double() for x in s.args)
    rho = []
    for p in qry[:, :3].split(max(1, 100_000_000 // bnd.shape[0])):
        diff = p[:, None] - bnd[None, :, :3]
        eta = diff.norm(dim=2)
        dot = (diff * nrm[None, :, :3]).sum(2)
        inside = -(area * dot / (4 * math.pi * eta ** 3)).sum(1) > 0.5
        xi = eta.amin(1)
        ratio = eta / xi[:, None]
        g = torch.exp(-0.5 * ((ratio - 1) / 0.5) ** 2) / (math.sqrt(2 * math.pi) * 0.5) * (ratio - 1 <= 1.5)
        xi = torch.where(inside, -xi, xi)[:, None]
        lam = torch.where(inside, -3.0, 1.0).double()[:, None]
        zeta2 = torch.complex(xi * xi - eta * eta, 2 * xi * eta)
        rho.append((lam / math.sqrt(2 * math.pi) * g * dot / eta * area / zeta2).sum(1))
    return torch.view_as_real(torch.cat(rho))


def _exact_grad(case, seed):
    N, L = case["N"], _side(case)
    p1, c1, p2, c2 = _exact_in(case, seed, 3)
    if 8.0 * N ** 3 * (p1.shape[0] + 4.0 * case["P"] * p2.shape[0]) > 5e12:
        return None
    A = _spectrum(p1, c1, N, L, case["sigma_g"], 3)
    k = 2 * math.pi * _modes(N) / L
    qs, ts = (x.double() for x in _start_poses(case, seed, case["P"]))
    out = []
    for q, t in zip(qs, ts):
        q, t = q.clone().requires_grad_(True), t.clone().requires_grad_(True)
        y = p2 @ _rotation(q).T + t
        yd = y.detach()
        E = [torch.exp(1j * yd[:, a:a + 1] * k) for a in range(3)]
        f, gy = 0.0, torch.zeros_like(yd)
        for z in range(N):  # per plane of modes: values and y, x derivatives at every sample
            u = E[1] @ A[z]
            du = (1j * k * E[1]) @ A[z]
            e = c2 * E[2][:, z]
            val = (u * E[0]).sum(1)
            f = f + (e * val).sum().real
            gy[:, 0] += (e * (u * (1j * k) * E[0]).sum(1)).real
            gy[:, 1] += (e * (du * E[0]).sum(1)).real
            gy[:, 2] += (e * 1j * k[z] * val).real
        gq, gt = torch.autograd.grad(y, (q, t), gy)
        out.append((f, gq, gt))
    return [torch.stack([x[i] for x in out]) for i in range(3)]


def exact(case, seed):
    if case["kind"] == "search":
        return _exact_search(case, seed)
    if case["kind"] == "sdf":
        return _exact_sdf(case, seed)
    if case["kind"] == "grad":
        return _exact_grad(case, seed)
    return None
