"""Performance cases of the tensorial template matching engine.

Each case is one call (or one step) that a program makes through the public
entry points: whole matching passes (``Matcher.run``, a captured batch), the
score map with rotations at its peaks only (``Matcher.match_peaks``), and the
single stages a program also calls by themselves (``ttm_local_stats``,
``build_template``, ``ttm_classical_ncc``, ``ttm_extract_peaks``).  Volumes
are Gaussian noise with randomly rotated copies of the template planted in
them, as a tomogram has; sizes are those of the benchmark's and the tests'
configurations (boxes of 9 to 64 voxels, volumes of 64^3 to 928 x 464 x 232,
orders 2 to 8, FP32 and mixed precision) and ragged ones between them.

``exact`` states in 64 bits what a call computes: w, score, the tensor
components, the best classical correlation and, where the maximum can be
searched by brute force, lambda.  A rotation has no such value (at a near-tie
of two maxima both are right), nor has the index of the best rotation.
"""

import math

import numpy as np
import torch

import paper_2311_07561_gb300 as ttm

SNR = 0.5
PSI = 1.533751168755204288118041      # psi^4 = psi + 4 (super-Fibonacci spiral)


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # the smallest whole call: a 64^3 subvolume against a 15^3 template,
        # where launches and latency count
        dict(name="match 64 s15", kind="match", x=64, y=64, z=64, s=15, n=4, rot=2000, mixed=False),
        # an ordinary subtomogram search, FP32: the 256^3 configuration
        dict(name="match 256 s32", kind="match", x=256, y=256, z=256, s=32, n=4, rot=10000,
             mixed=False),
        # half of a 512^3 tomogram with bf16 storage, order 4
        dict(name="match mixed 512x512x256 s40", kind="match", x=512, y=512, z=256, s=40, n=4,
             rot=10000, mixed=True),
        # the largest: a quarter of the 928 x 928 x 464 tomogram with its 64^3
        # template, order 6, bf16 storage
        dict(name="match mixed 928x464x232 s64 n6", kind="match", x=928, y=464, z=232, s=64, n=6,
             rot=20000, mixed=True),
        # a small particle: few mask voxels, where the planner takes the
        # direct correlation (mixed precision: on the tensor cores)
        dict(name="match mixed 130x121x97 s9", kind="match", x=130, y=121, z=97, s=9, n=4, rot=2000,
             mixed=True),
        # particle picking: the score map, rotations at the peaks only; a
        # ragged volume and an odd box
        dict(name="peaks 250x230x190 s33", kind="peaks", x=250, y=230, z=190, s=33, n=4, rot=5000,
             mixed=False),
        # the denominators alone (a program that normalises maps of its own)
        dict(name="stats 300x260x140 s25", kind="stats", x=300, y=260, z=140, s=25, n=2, rot=100),
        # a batch: several volumes, several templates, resident waves, one graph
        dict(name="batch 4 volumes 2 templates", kind="batch", x=160, y=144, z=128, volumes=4, s=24,
             s2=32, n=4, rot=3000, mib=2048),
        # folding a template, once per template: an ordinary and the largest one
        dict(name="build s32 n4", kind="build", s=32, n=4, rot=10000),
        dict(name="build s64 n6", kind="build", s=64, n=6, rot=20000),
        # the classical per-rotation comparator
        dict(name="classical 192x160x128 s24", kind="classical", x=192, y=160, z=128, s=24, rot=500),
        # peaks of maps that are there already (another threshold or radius)
        dict(name="extract 256", kind="extract", x=256, y=256, z=256, radius=12),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def box(lo, hi, least):
        """Extents of a ragged volume of lo..hi voxels, each at least `least`."""
        edge = log(lo, hi) ** (1.0 / 3.0)
        a, b = rng.uniform(0.75, 1.3), rng.uniform(0.75, 1.3)
        return {k: int(min(700, max(least, round(edge * f))))
                for k, f in (("x", a), ("y", b), ("z", 1.0 / (a * b)))}

    kind = rng.choice(["match", "match", "match", "peaks", "stats", "batch", "build", "classical",
                       "extract"])
    if kind in ("match", "peaks"):
        mixed = rng.random() < 0.5
        n = rng.choice([4, 4, 6] if kind == "peaks" else [2, 4, 4, 4, 6, 6, 8])
        s = int(round(log(9, 64 if n == 6 else 40)))
        most = {2: 1.6e7, 4: 1.6e7, 6: 8e6, 8: 4e5}[n]
        c = box(max(1.5e5, 3.5 * s ** 3), max(most, 5.0 * s ** 3), s + 3)
        return dict(kind=kind, **c, s=s, n=n, rot=int(log(500, 4000)), mixed=mixed)
    if kind == "stats":
        s = int(round(log(9, 56)))
        return dict(kind=kind, **box(max(1.5e5, 3.5 * s ** 3), 2.5e7, s + 3), s=s, n=2, rot=100)
    if kind == "batch":
        s = rng.randint(13, 32)
        return dict(kind=kind, **box(6e5, 4e6, s + 55), volumes=rng.randint(2, 6), s=s, s2=s + 7,
                    n=4, rot=1000, mib=rng.choice([256, 1024, 4096]))
    if kind == "build":
        n = rng.choice([2, 4, 4, 6])
        return dict(kind=kind, s=int(round(log(9, 64))), n=n, rot=int(log(300, 12000)))
    if kind == "classical":
        s = rng.randint(11, 40)
        return dict(kind=kind, **box(max(2e5, 3.5 * s ** 3), 5e6, s + 3), s=s, rot=int(log(40, 400)))
    return dict(kind=kind, **box(2e5, 3e7, 24), radius=rng.randint(1, 20))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _quadrature(n):
    """n near-uniform unit quaternions (super-Fibonacci spiral), float32."""
    s = np.arange(n) + 0.5
    r, big = np.sqrt(s / n), np.sqrt(1.0 - s / n)
    a, b = 2 * np.pi * s / math.sqrt(2.0), 2 * np.pi * s / PSI
    return np.stack([r * np.sin(a), r * np.cos(a), big * np.sin(b), big * np.cos(b)], 1).astype(np.float32)


def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(1000003 * what + seed)


def _rand(shape, g, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _axes(s):
    """Offsets from the box centre, (s, s, s) each, in (x, y, z) order."""
    o = torch.arange(s, device="cuda", dtype=torch.float64) - s // 2
    z, y, x = torch.meshgrid(o, o, o, indexing="ij")
    return x, y, z


def _radius(s):
    return (s - 1) // 2 if s % 2 else s // 2 - 1


def _mask(s):
    x, y, z = _axes(s)
    return (x * x + y * y + z * z <= _radius(s) ** 2).to(torch.float32)


def _rotations(q):
    """Rotation matrices of unit quaternions (real part first), (n, 3, 3)."""
    a, b, c, d = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([
        torch.stack([a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c)], 1),
        torch.stack([2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b)], 1),
        torch.stack([2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d], 1)], 1)


class _Blobs:
    """A particle: a sum of Gaussian blobs, sampled at any rotation."""

    def __init__(self, s, seed, what=1):
        g = _gen(seed, what)
        n = 5 if s < 20 else 30
        r = _radius(s)
        v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
        rad = 0.6 * r * _rand((n, 1), g) ** (1.0 / 3.0)
        self.s, self.centre = s, v / v.norm(dim=1, keepdim=True) * rad
        self.width = _rand((n,), g, 1.0, 2.0) * max(s / 24.0, 0.7)
        self.amp = _rand((n,), g, 0.5, 1.0)

    def sample(self, quats=None):
        """The box (float64) of each rotation, or of the particle itself."""
        R = torch.eye(3, device="cuda", dtype=torch.float64)[None] if quats is None else _rotations(quats)
        p = torch.einsum("rij,bj->rbi", R, self.centre)
        o = torch.arange(self.s, device="cuda", dtype=torch.float64) - self.s // 2
        e = torch.exp(-0.5 * ((o - p[..., None]) / self.width[None, :, None, None]) ** 2)   # (r, b, 3, s)
        return torch.einsum("b,rbz,rby,rbx->rzyx", self.amp, e[:, :, 2], e[:, :, 1], e[:, :, 0])


def _volume(case, seed, blobs, what=2):
    """Noise with planted copies, float32 (Z, Y, X); SNR over the planted boxes."""
    g = _gen(seed, what)
    X, Y, Z = case["x"], case["y"], case["z"]
    s = blobs.s
    n = int(min(60, max(2, X * Y * Z // (3 * s) ** 3)))
    q = torch.randn((n, 4), generator=g, device="cuda", dtype=torch.float64)
    copies = blobs.sample(q) * _mask(s)
    f = torch.zeros((Z, Y, X), device="cuda", dtype=torch.float32)
    at = torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    for k in range(n):
        x0, y0, z0 = (int(at[k, i] * (d - s + 1)) for i, d in enumerate((X, Y, Z)))
        f[z0:z0 + s, y0:y0 + s, x0:x0 + s] += copies[k].float()
    inside = copies[copies != 0]
    sigma = float(torch.sqrt(inside.var() / SNR))
    return f + sigma * torch.randn(f.shape, generator=g, device="cuda", dtype=torch.float32)


def _template(case, seed, s=None, what=1):
    s = s or case["s"]
    blobs = _Blobs(s, seed, what)
    return blobs, blobs.sample()[0].float(), _mask(s)


def _built(case, seed, s=None, what=1):
    blobs, t, m = _template(case, seed, s, what)
    comp, desc = ttm.build_template(t.cpu().numpy(), m.cpu().numpy(), case["n"], _quadrature(case["rot"]))
    return blobs, (comp, desc, m)


def _opts(case):
    o = ttm.PlanOpts()
    o.precision = ttm.TTM_PREC_MIXED if case.get("mixed") else ttm.TTM_PREC_FP32
    o.batch_mib = case.get("mib", 0)
    return o


def _dims(case):
    return case["x"], case["y"], case["z"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "build":
        # the raw template as a program has read it from a file, host arrays
        _, t, m = _template(case, seed)
        return dict(case=case, t=t.cpu().numpy(), m=m.cpu().numpy(), q=_quadrature(case["rot"]))
    if kind == "extract":
        g = _gen(seed, 7)
        shape = (case["z"], case["y"], case["x"])
        score = 0.1 * torch.rand(shape, generator=g, device="cuda")
        q = torch.randn(shape + (4,), generator=g, device="cuda")
        small = dict(case, s=5, n=2, rot=20)
        _, tmpl = _built(small, seed)
        m = ttm.Matcher([tmpl], [(_dims(case), 0)], opts=_opts(case))
        m.score[0].copy_(score)
        m.quat[0].copy_(q / q.norm(dim=-1, keepdim=True))
        m.lam[0].copy_(0.5 * score)
        return dict(case=case, m=m)
    if kind == "batch":
        first, t1 = _built(case, seed, case["s"], 1)
        _, t2 = _built(case, seed, case["s2"], 3)
        problems, vols = [], []
        for v in range(case["volumes"]):
            c = dict(case, x=case["x"] - 8 * v, z=case["z"] + 4 * v)
            f = _volume(c, seed, first, 11 + v)
            for k in (0, 1):
                problems.append((_dims(c), k))
                vols.append(f)
        m = ttm.Matcher([t1, t2], problems, opts=_opts(case))
        graph = m.capture(vols)
        return dict(case=case, m=m, vols=vols, graph=graph)
    if kind == "classical":
        blobs, tmpl = _built(dict(case, n=2, rot=50), seed)
        o = _opts(case)
        o.path = ttm.TTM_PATH_FFT
        m = ttm.Matcher([tmpl], [(_dims(case), 0)], opts=o)
        f = _volume(case, seed, blobs)
        ttm.ttm_local_stats(m.plan, [f], m.w, m.ws)
        ws = torch.empty(ttm.ttm_classical_workspace_size(m.plan, 0), dtype=torch.uint8, device="cuda")
        return dict(case=case, m=m, f=f, t=blobs.sample()[0].float().contiguous(), ws=ws,
                    q=torch.from_numpy(_quadrature(case["rot"])).cuda(),
                    best=torch.empty_like(f), index=torch.empty(f.shape, dtype=torch.int32, device="cuda"))
    blobs, tmpl = _built(case, seed)
    m = ttm.Matcher([tmpl], [(_dims(case), 0)], opts=_opts(case))
    return dict(case=case, m=m, vols=[_volume(case, seed, blobs)])


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def _most(cells, radius):
    """Peaks asked for: a number that the volume is sure to have."""
    return int(min(1000, max(1, cells // (8 * (2 * radius + 1) ** 3))))


def _records(p):
    return dict(at=np.stack([p["x"], p["y"], p["z"]], 1), score=p["score"].copy(),
                lam=p["lambda"].copy(), quat=p["q"].copy())


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "build":
        comp, desc = ttm.build_template(state["t"], state["m"], case["n"], state["q"])
        return dict(components=comp, mask_sum=float(desc.mask_sum))
    m = state["m"]
    if kind == "match":
        m.run(state["vols"])
        return dict(w=m.w, score=m.score, lam=m.lam, quat=m.quat)
    if kind == "batch":
        state["graph"].replay()
        return dict(w=m.w, score=m.score, lam=m.lam, quat=m.quat)
    if kind == "peaks":
        s, radius = case["s"], max(2, case["s"] // 3)
        inner = math.prod(d - s + 1 for d in _dims(case))
        p = m.match_peaks(state["vols"], 0, 0.0, radius, _most(inner, radius))
        return dict(w=m.w, score=m.score, peaks=_records(p))
    if kind == "stats":
        ttm.ttm_local_stats(m.plan, state["vols"], m.w, m.ws)
        return dict(w=m.w)
    if kind == "classical":
        ttm.ttm_classical_ncc(m.plan, 0, state["t"], state["q"], case["rot"], state["f"], m.w[0],
                              state["best"], state["index"], state["ws"])
        return dict(best=state["best"], index=state["index"])
    return dict(peaks=_records(m.peaks(0, 0.05, case["radius"],
                                       _most(math.prod(_dims(case)), case["radius"]))))


# --------------------------------------------------------------------------
# work one pass cannot do without
# --------------------------------------------------------------------------

def _k(n):
    return (n + 1) * (n + 2) * (n + 3) // 6


def _transform(vox):
    """Operations of one real 3D transform."""
    return 2.5 * vox * math.log2(max(vox, 2))


def _match_work(x, y, z, s, n, dense):
    vox, K = float(x * y * z), _k(n)
    inner = float((x - s + 1) * (y - s + 1) * (z - s + 1))
    fl = (K + 1) * _transform(vox) + 3.0 * K * vox + 5 * _transform(vox)     # maps, products, w
    # 32 evaluations of phi and ~30 power iterations per voxel: 400 K; the score alone: 3 K
    fl += inner * (400.0 * K if dense else 3.0 * K)
    return vox * (4 + (28 if dense else 8)) + 4.0 * K * s ** 3, fl


def work(case):
    kind = case["kind"]
    if kind in ("match", "peaks"):
        b, f = _match_work(*_dims(case), case["s"], case["n"], kind == "match")
    elif kind == "batch":
        b = f = 0.0
        for v in range(case["volumes"]):
            for s in (case["s"], case["s2"]):
                bb, ff = _match_work(case["x"] - 8 * v, case["y"], case["z"] + 4 * v, s, case["n"], True)
                b, f = b + bb, f + ff
    elif kind == "stats":
        vox = float(case["x"] * case["y"] * case["z"])
        b, f = 8.0 * vox, 5 * _transform(vox)
    elif kind == "build":
        inside = 4.19 * _radius(case["s"]) ** 3
        b = 4.0 * (_k(case["n"]) + 2) * case["s"] ** 3 + 16.0 * case["rot"]
        f = case["rot"] * inside * (30.0 + 2.0 * _k(case["n"]))
    elif kind == "classical":
        vox = float(case["x"] * case["y"] * case["z"])
        b, f = 16.0 * vox, case["rot"] * (2 * _transform(vox) + 5 * vox)
    else:
        vox = float(case["x"] * case["y"] * case["z"])
        b, f = 4.0 * vox, 6.0 * vox
    return {"bytes": b, "flops": f}


# --------------------------------------------------------------------------
# what a pass computes, in 64 bits
# --------------------------------------------------------------------------

def _rotated(t, m, q):
    """Rotated (trilinear, zero outside), masked, S-normalised copies at the
    mask's voxels: (rotations, voxels)."""
    s = t.shape[0]
    c = s // 2
    idx = m.reshape(-1).nonzero()[:, 0]
    mv = m.reshape(-1)[idx]
    off = torch.stack([a.reshape(-1)[idx] for a in _axes(s)], 0)              # (3, voxels)
    p = torch.einsum("rji,jv->riv", _rotations(q), off) + c                   # R^-1 (u - c)
    lo = p.floor()
    fr = p - lo
    lo = lo.long()
    pad = torch.zeros((s + 2,) * 3, device=t.device, dtype=t.dtype)
    pad[1:-1, 1:-1, 1:-1] = t
    flat = pad.reshape(-1)
    v = torch.zeros(p.shape[0], p.shape[2], device=t.device, dtype=t.dtype)
    for corner in range(8):
        w, at = 1.0, 0
        for axis, stride in ((0, 1), (1, s + 2), (2, (s + 2) ** 2)):
            bit = (corner >> axis) & 1
            w = w * (fr[:, axis] if bit else 1.0 - fr[:, axis])
            at = at + (lo[:, axis] + bit + 1).clamp(0, s + 1) * stride
        v += w * flat[at]
    one = mv.sum()
    mean = (v * mv).sum(1, keepdim=True) / one
    var = (v * v * mv).sum(1, keepdim=True) - mean * mean * one
    return idx, mv * (v - mean) / var.sqrt()


def _tuples(n):
    out = []

    def go(prefix, least):
        if len(prefix) == n:
            out.append(tuple(prefix))
            return
        for i in range(least, 4):
            go(prefix + [i], i)
    go([], 0)
    return out


def _mu(n):
    return torch.tensor([math.factorial(n) / math.prod(math.factorial(a.count(i)) for i in range(4))
                         for a in _tuples(n)], dtype=torch.float64, device="cuda")


def _powers(q, n):
    """q^alpha for every component, (points, K)."""
    return torch.stack([torch.stack([q[:, i] for i in a], 0).prod(0) for a in _tuples(n)], 1)


def _exact_template(t, m, n, rot):
    q = torch.from_numpy(_quadrature(rot)).cuda().double()
    s = t.shape[0]
    total = None
    step = max(1, int(6e7 / s ** 3))
    for j in range(0, rot, step):
        qq = q[j:j + step]
        idx, v = _rotated(t.double(), m.double(), qq)
        part = _powers(qq / qq.norm(dim=1, keepdim=True), n).T @ v / rot
        total = part if total is None else total + part
    out = torch.zeros((_k(n), s ** 3), device="cuda", dtype=torch.float64)
    out[:, idx] = total
    return out.reshape(_k(n), s, s, s)


def _spectrum(box, shape):
    """Half spectrum of a box whose centre voxel sits at the origin."""
    s = box.shape[-1]
    pad = torch.zeros(shape, device="cuda", dtype=torch.float64)
    pad[:s, :s, :s] = box
    return torch.fft.rfftn(pad.roll((-(s // 2),) * 3, (0, 1, 2)))


def _inside(shape, s):
    c = s // 2
    keep = torch.zeros(shape, device="cuda", dtype=torch.float64)
    keep[tuple(slice(c, d - (s - 1 - c)) for d in shape)] = 1.0
    return keep


def _exact_w(f, m):
    mean = f.mean()
    F = _spectrum(m.double(), f.shape).conj()
    a = f - mean
    s1 = torch.fft.irfftn(torch.fft.rfftn(a) * F, s=f.shape)
    s2 = torch.fft.irfftn(torch.fft.rfftn(a * a) * F, s=f.shape)
    var = s2 - s1 * s1 / m.double().sum()
    ok = var > 1e-6 * m.double().sum() * (a * a).mean()
    return torch.where(ok, var.clamp_min(1e-300).rsqrt(), torch.zeros_like(var)) * _inside(f.shape, m.shape[0])


def _exact_lambda(C, n):
    """max phi over unit quaternions, phi(Q) = C . Q^n, by grid search and
    shifted power steps from the best points; C is (K, voxels)."""
    mu = _mu(n)
    grid = torch.from_numpy(_quadrature(8192)).cuda().double()
    grid = grid / grid.norm(dim=1, keepdim=True)
    table = (_powers(grid, n) * mu).T
    where = {a: k for k, a in enumerate(_tuples(n))}
    full = torch.tensor([where[tuple(sorted((i, j, k, l)))] for i in range(4) for j in range(4)
                         for k in range(4) for l in range(4)], device="cuda")
    out = torch.zeros(C.shape[1], device="cuda", dtype=torch.float64)
    for v0 in range(0, C.shape[1], 16384):
        c = C[:, v0:v0 + 16384].T
        x = grid[(c @ table).topk(12, dim=1).indices]                          # (v, 12, 4)
        A = c[:, full].reshape(-1, 4, 64)
        shift = ((n - 1) * (c * c * mu).sum(1).sqrt())[:, None, None]
        best = None
        for _ in range(150):
            x3 = torch.einsum("vpi,vpj,vpk->vpijk", x, x, x).reshape(x.shape[0], 12, 64)
            g = torch.einsum("vpa,via->vpi", x3, A)
            best = (g * x).sum(-1)
            x = g + shift * x
            x = x / x.norm(dim=-1, keepdim=True).clamp_min(1e-300)
        out[v0:v0 + 16384] = best.max(1).values
    return out


def _exact_match(f, t, m, n, rot, lam):
    T = _exact_template(t, m, n, rot)
    f = f.double()
    w = _exact_w(f, m)
    F = torch.fft.rfftn(f - f.mean())
    mu = _mu(n)
    score = torch.zeros_like(f)
    maps = []
    for k in range(T.shape[0]):
        c = torch.fft.irfftn(F * _spectrum(T[k], f.shape).conj(), s=f.shape) * w
        score += mu[k] * c * c
        if lam:
            maps.append(c.reshape(-1))
    l = None
    if lam:
        l = _exact_lambda(torch.stack(maps, 0), n).reshape(f.shape) * _inside(f.shape, m.shape[0])
    return w, score.sqrt(), l


def exact(case, seed):
    kind = case["kind"]
    if kind == "build":
        _, t, m = _template(case, seed)
        return dict(components=_exact_template(t, m, case["n"], case["rot"]), mask_sum=float(m.double().sum()))
    if kind == "extract":
        return None          # selected and copied values, none computed
    if kind == "stats":
        blobs, _, m = _template(case, seed)
        return dict(w=[_exact_w(_volume(case, seed, blobs).double(), m)])
    if kind == "classical":
        blobs, t, m = _template(case, seed)
        f = _volume(case, seed, blobs).double()
        w, F, best = _exact_w(f, m), torch.fft.rfftn(f - f.mean()), None
        q = torch.from_numpy(_quadrature(case["rot"])).cuda().double()
        s = case["s"]
        for j in range(0, case["rot"], 32):
            idx, v = _rotated(t.double(), m.double(), q[j:j + 32])
            for r in range(v.shape[0]):
                one = torch.zeros(s ** 3, device="cuda", dtype=torch.float64)
                one[idx] = v[r]
                c = torch.fft.irfftn(F * _spectrum(one.reshape(s, s, s), f.shape).conj(), s=f.shape) * w
                best = c if best is None else torch.maximum(best, c)
        return dict(best=best, index=None)
    if kind == "batch":
        first, t1, m1 = _template(case, seed, case["s"], 1)
        _, t2, m2 = _template(case, seed, case["s2"], 3)
        out = dict(w=[], score=[], lam=None, quat=None)
        for v in range(case["volumes"]):
            f = _volume(dict(case, x=case["x"] - 8 * v, z=case["z"] + 4 * v), seed, first, 11 + v)
            for t, m in ((t1, m1), (t2, m2)):
                w, score, _ = _exact_match(f, t, m, case["n"], case["rot"], False)
                out["w"].append(w)
                out["score"].append(score)
        return out
    blobs, t, m = _template(case, seed)
    f = _volume(case, seed, blobs)
    lam = kind == "match" and case["n"] == 4 and f.numel() <= 300000
    w, score, l = _exact_match(f, t, m, case["n"], case["rot"], lam)
    if kind == "peaks":
        return dict(w=[w], score=[score], peaks=None)
    return dict(w=[w], score=[score], lam=[l], quat=None)
