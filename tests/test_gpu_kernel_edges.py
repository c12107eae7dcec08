"""The kernels at the sizes where their tiles, lists and variants end: FFT
passes of every long length, window statistics of small masks, template builds
over listed voxels, the candidates of the rotation search, peak lists.

Tolerances are those of the parity tests: 1e-4 on components, score and lambda
(FP32), 5e-3 with bf16 storage, 1e-5 relative on w, 2e-5 of the largest
component on templates; peaks exact.
"""

import numpy as np
import pytest

import synth
from oracle import ttm_oracle as o

pytestmark = pytest.mark.gpu

TOL = 1e-4
BF16_TOL = 5e-3


@pytest.fixture(scope="module")
def ttm():
    import os
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2311_07561_gb300 as ttm
    if not os.path.exists(ttm.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    ttm.load_library()
    return ttm


def _cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _maps(ttm, volume, comp, desc, mask, want_comp=False, **opts):
    import torch
    po = ttm.PlanOpts()
    for k, v in opts.items():
        setattr(po, k, v)
    Z, Y, X = volume.shape
    m = ttm.Matcher([(comp, desc, mask)], [((X, Y, Z), 0)], opts=po)
    comps = [torch.empty((desc.K, Z, Y, X), dtype=torch.float32, device="cuda")] if want_comp else None
    m.run([_cuda(volume)], components_out=comps)
    torch.cuda.synchronize()
    assert ttm.ttm_plan_device_status(m.plan, m.ws) == 0
    out = dict(w=m.w[0].cpu().numpy(), score=m.score[0].cpu().numpy(),
               quat=m.quat[0].cpu().numpy(), lam=m.lam[0].cpu().numpy(),
               comp=comps[0].cpu().numpy() if want_comp else None)
    box = ttm.ttm_plan_problem_fft_box(m.plan, 0) if opts.get("path") == ttm.TTM_PATH_FFT else None
    m.close()
    return out, box


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("length", [128, 144, 192, 240, 256, 320, 384, 512, 576, 640, 768, 1024])
def test_long_lines(ttm, length, axis):
    """One long line along x, y or z, the volume up to three voxels short of it
    (rows that start on 4, 8 or 16 bytes; columns that end in the padding)."""
    short = (length // 64 + axis) % 4
    shape = [18, 21, 23]
    shape[2 - axis] = length - short
    wl = synth.make_workload(shape, 7, 3, 2, 1.0, 2, 60, radius=3, seeds=(41, 42, 43))
    T = o.tensor_template(wl.template, wl.mask, wl.quadrature.astype(np.float64), wl.weights, 2)
    comp, desc = ttm.build_template(wl.template, wl.mask, 2, wl.quadrature)
    w_o, C_o = o.ttm_components(wl.volume, T, wl.mask)
    for precision, tol in ((ttm.TTM_PREC_FP32, TOL), (ttm.TTM_PREC_MIXED, BF16_TOL)):
        res, box = _maps(ttm, wl.volume, comp, desc, wl.mask, True, path=ttm.TTM_PATH_FFT,
                         precision=precision)
        assert box[axis] == length
        assert np.abs(res["comp"] - C_o).max() <= tol
        nz = w_o > 0
        assert np.array_equal(res["w"] > 0, nz)
        assert (np.abs(res["w"][nz] - w_o[nz]) / w_o[nz]).max() <= 1e-5


def _mask(kind, s):
    m = np.zeros((s, s, s), dtype=np.float32)
    rng = np.random.default_rng(s)
    if kind == "ball":
        m = synth.ball_mask(s)
    elif kind == "lopsided":             # runs that lie to one side, in few windows
        m[: s // 2 + 1, s // 2:, : s // 2 + 1] = 1
        m[0, s - 1, 0] = 0
    elif kind == "plane":
        m[s - 1] = 1
    elif kind == "scattered":            # as many windows as there are runs
        m = (rng.random((s, s, s)) < 0.4).astype(np.float32)
    return m


@pytest.mark.parametrize("kind", ["ball", "lopsided", "plane", "scattered"])
@pytest.mark.parametrize("s,shape", [(3, (5, 66, 35)), (6, (40, 9, 33)), (9, (23, 31, 64)),
                                     (15, (15, 47, 81)), (17, (30, 34, 38))])
def test_direct_statistics(ttm, s, shape, kind):
    rng = np.random.default_rng(5)
    mask = _mask(kind, s)
    volume = (rng.normal(size=shape) + 3.0).astype(np.float32)
    q = synth.super_fibonacci_quaternions(8).astype(np.float32)
    t = rng.normal(size=(s, s, s)).astype(np.float32)
    comp, desc = ttm.build_template(t, mask, 2, q)
    res, _ = _maps(ttm, volume, comp, desc, mask, path=ttm.TTM_PATH_DIRECT)
    w_o = o.local_stats_direct(volume, mask)[2]
    nz = w_o > 0
    assert np.array_equal(res["w"] > 0, nz)
    assert (np.abs(res["w"][nz] - w_o[nz]) / w_o[nz]).max() <= 1e-5


@pytest.mark.parametrize("s,n,n_rot,kind,scale", [
    (3, 2, 700, "ball", 1.0),            # fewer listed voxels than threads
    (5, 4, 1, "ball", 1.0),              # one node: no room for the tables
    (8, 4, 37, "ball", 1.0),             # nodes past a multiple of the step
    (10, 6, 150, "scattered", 1.0),
    (11, 4, 90, "full", 1.0),            # every voxel: the box build
    (13, 4, 200, "soft", 1.0),           # weights, not flags
    (12, 4, 120, "ball", 1e-25),         # squares below the FP32 range
    (12, 4, 120, "ball", 1e20),          # and above it
    (12, 8, 64, "lopsided", 1.0),
    (32, 4, 90, "ball", 1.0),            # two voxels per thread
    (40, 8, 320, "ball", 1.0),           # four, and few nodes of many voxels
    (70, 4, 310, "ball", 1.0),           # four at order 4, a ragged last chunk
])
def test_template_build(ttm, s, n, n_rot, kind, scale):
    t = (synth.blob_template(s, 4, seed=s).astype(np.float64) * scale).astype(np.float32)
    if kind == "soft":
        mask = synth.soft_ball_mask(s, s // 2, 2.0)
    else:
        mask = np.ones((s, s, s), np.float32) if kind == "full" else _mask(kind, s)
    q = synth.super_fibonacci_quaternions(n_rot).astype(np.float32)
    comp, desc = ttm.build_template(t, mask, n, q)
    T = o.tensor_template(t, mask, q.astype(np.float64), np.full(n_rot, 1.0 / n_rot), n)
    assert desc.mask_sum == pytest.approx(mask.sum(dtype=np.float64))
    assert np.abs(comp.cpu().numpy() - T).max() <= 2e-5 * np.abs(T).max()


@pytest.mark.parametrize("path", ["direct", "fft"])
@pytest.mark.parametrize("n,shape", [(2, (21, 20, 23)), (4, (23, 19, 37)), (6, (19, 22, 29))])
def test_candidates_one_by_one(ttm, n, shape, path):
    """With every candidate refined, one more can only raise lambda, and leaves
    what the others gave to the bit (whichever one it is refined beside, and
    however many the search keeps); lambda is phi at q."""
    wl = synth.make_workload(shape, 9, 3, 1, 1.0, n, 200, radius=4, seeds=(51, 52, 53))
    T = o.tensor_template(wl.template, wl.mask, wl.quadrature.astype(np.float64), wl.weights, n)
    comp, desc = ttm.build_template(wl.template, wl.mask, n, wl.quadrature)
    w_o, C_o = o.ttm_components(wl.volume, T, wl.mask)
    at = np.argwhere(w_o > 0)[::29]
    C_pts = C_o[:, at[:, 0], at[:, 1], at[:, 2]].T
    last = None
    for k in (1, 2, 3, 4):
        res, _ = _maps(ttm, wl.volume, comp, desc, wl.mask, n_grid=2048, n_cells=128,
                       n_candidates=k, n_refined=k,
                       path={"direct": ttm.TTM_PATH_DIRECT, "fft": ttm.TTM_PATH_FFT}[path])
        phi = o.phi_unique(C_pts, res["quat"][at[:, 0], at[:, 1], at[:, 2]].astype(np.float64), n)
        assert np.abs(phi - res["lam"][at[:, 0], at[:, 1], at[:, 2]]).max() <= TOL
        if last is not None:
            assert np.all(res["lam"] >= last["lam"])
            same = res["lam"] == last["lam"]
            assert np.array_equal(res["quat"][same], last["quat"][same])
            assert np.array_equal(res["score"], last["score"])
        last = res


@pytest.mark.parametrize("levels", [1, 3, 1000])
@pytest.mark.parametrize("shape", [(5, 5, 5), (7, 66, 9), (34, 11, 129), (65, 33, 17)])
def test_peak_lists(ttm, shape, levels):
    """Scores of one level (a single peak per cube of ties), of few and of
    many; cubes inside one block of voxels, over many and over the whole map."""
    Z, Y, X = shape
    rng = np.random.default_rng(Z)
    t = synth.blob_template(5, 3, seed=1)
    mask = synth.ball_mask(5, 2)
    comp, desc = ttm.build_template(t, mask, 2, synth.super_fibonacci_quaternions(10).astype(np.float32))
    m = ttm.Matcher([(comp, desc, mask)], [((X, Y, Z), 0)])
    score = (np.floor(rng.random(shape) * levels) / levels + 0.25).astype(np.float32)
    quat = np.zeros(shape + (4,), dtype=np.float32)
    quat[..., 0] = np.arange(score.size, dtype=np.float32).reshape(shape)
    for radius in (0, 1, 2, 5):
        for limit in (3, score.size):
            got = ttm.ttm_extract_peaks(m.plan, 0, _cuda(score), _cuda(quat), _cuda(score), 0.2,
                                        radius, limit, m.ws)
            expect = o.extract_peaks(score.astype(np.float64), 0.2, radius, limit)
            assert np.array_equal((got["z"].astype(np.int64) * Y + got["y"]) * X + got["x"], expect)
            assert np.array_equal(got["q"][:, 0], quat[..., 0].ravel()[expect])
            assert np.array_equal(got["lambda"], score.ravel()[expect])
    m.close()


@pytest.mark.parametrize("depth,s,n_rot", [(125, 9, 3), (141, 8, 34), (192, 15, 5), (239, 12, 2), (460, 9, 4)])
def test_classical_long_z(ttm, depth, s, n_rot):
    """Classical matching where a rotated template's own z transform runs
    inside the multiply (long z lines, three rotations and more in a batch; 34
    leaves a batch of two, which takes the passes one by one)."""
    import torch
    rng = np.random.default_rng(depth)
    shape = (depth, 23, 26)
    volume = rng.normal(size=shape).astype(np.float32)
    t, mask = synth.blob_template(s, 4, seed=s), synth.ball_mask(s)
    q = synth.shoemake_quaternions(n_rot, 4).astype(np.float32)
    comp, desc = ttm.build_template(t, mask, 2, synth.super_fibonacci_quaternions(20).astype(np.float32))
    po = ttm.PlanOpts()
    po.path = ttm.TTM_PATH_FFT
    m = ttm.Matcher([(comp, desc, mask)], [(shape[::-1], 0)], opts=po)
    vol = _cuda(volume)
    m.run([vol])
    best = torch.empty(shape, dtype=torch.float32, device="cuda")
    arg = torch.empty(shape, dtype=torch.int32, device="cuda")
    ws = torch.empty(ttm.ttm_classical_workspace_size(m.plan, 0), dtype=torch.uint8, device="cuda")
    ttm.ttm_classical_ncc(m.plan, 0, _cuda(t), _cuda(q), n_rot, vol, m.w[0], best, arg, ws)
    torch.cuda.synchronize()
    best, arg = best.cpu().numpy(), arg.cpu().numpy()
    m.close()
    c = o.classical_ncc(volume, t, mask, q.astype(np.float64))
    keep = o.interior_mask(shape, s)
    best_o = np.where(keep, c.max(axis=0), 0.0)
    assert np.abs(best - best_o).max() <= TOL
    zi, yi, xi = np.nonzero(keep)
    assert np.all(c[arg[zi, yi, xi], zi, yi, xi] >= best_o[zi, yi, xi] - TOL)


@pytest.mark.parametrize("shape", [(6, 5, 7), (33, 40, 70), (19, 9, 130)])
def test_peaks_of_small_cubes(ttm, shape):
    """Radii up to the last one that scans its cubes without cells, and the
    next: few levels, so that ties decide, and a map with many peaks."""
    Z, Y, X = shape
    rng = np.random.default_rng(X)
    t = synth.blob_template(5, 3, seed=1)
    comp, desc = ttm.build_template(t, synth.ball_mask(5, 2), 2,
                                    synth.super_fibonacci_quaternions(10).astype(np.float32))
    m = ttm.Matcher([(comp, desc, synth.ball_mask(5, 2))], [((X, Y, Z), 0)])
    quat = np.zeros(shape + (4,), dtype=np.float32)
    for levels in (2, 10 ** 6):
        score = (np.floor(rng.random(shape) * levels) / levels + 0.25).astype(np.float32)
        for radius in (1, 2, 3, 4, 5):
            got = ttm.ttm_extract_peaks(m.plan, 0, _cuda(score), _cuda(quat), _cuda(score), 0.2,
                                        radius, score.size, m.ws)
            expect = o.extract_peaks(score.astype(np.float64), 0.2, radius, score.size)
            assert np.array_equal((got["z"].astype(np.int64) * Y + got["y"]) * X + got["x"], expect)
    m.close()


@pytest.mark.parametrize("s,shape", [(5, (21, 20, 22)), (7, (33, 41, 66)), (9, (20, 21, 22)), (9, (37, 41, 40)),
                                     (11, (30, 43, 90)), (13, (52, 48, 47)), (15, (37, 41, 40)),
                                     (15, (64, 60, 62))])
def test_direct_statistics_of_both_forms(ttm, s, shape):
    """Volumes on both sides of the line between marching and one plane at a
    time, the marching ones with one to several planes per block."""
    rng = np.random.default_rng(s)
    mask = _mask("ball", s)
    volume = (rng.normal(size=shape) + 3.0).astype(np.float32)
    q = synth.super_fibonacci_quaternions(8).astype(np.float32)
    comp, desc = ttm.build_template(rng.normal(size=(s, s, s)).astype(np.float32), mask, 2, q)
    res, _ = _maps(ttm, volume, comp, desc, mask, path=ttm.TTM_PATH_DIRECT)
    w_o = o.local_stats_direct(volume, mask)[2]
    nz = w_o > 0
    assert np.array_equal(res["w"] > 0, nz)
    assert (np.abs(res["w"][nz] - w_o[nz]) / w_o[nz]).max() <= 1e-5


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_direct_statistics_beside_values_that_are_not_finite(ttm, value):
    """Columns of such values at a block's reference voxel: the windows that
    hold one have no w, every other window has its own."""
    s, shape = 5, (30, 44, 70)
    mask = _mask("ball", s)
    rng = np.random.default_rng(12)
    volume = (rng.normal(size=shape) + 3.0).astype(np.float32)
    q = synth.super_fibonacci_quaternions(8).astype(np.float32)
    comp, desc = ttm.build_template(rng.normal(size=(s, s, s)).astype(np.float32), mask, 2, q)
    touched = np.zeros(shape, bool)
    disc = mask.any(axis=0)
    w_o = o.local_stats_direct(volume, mask)[2]
    for x, y in ((18, 6), (18, 14), (50, 30)):
        volume[:, y, x] = value
        for dy, dx in np.argwhere(disc) - s // 2:
            touched[:, y - dy, x - dx] = True
    import torch
    po = ttm.PlanOpts()
    po.path = ttm.TTM_PATH_DIRECT
    m = ttm.Matcher([(comp, desc, mask)], [(shape[::-1], 0)], opts=po)
    ttm.ttm_local_stats(m.plan, [_cuda(volume)], m.w, m.ws)
    torch.cuda.synchronize()
    w = m.w[0].cpu().numpy()
    m.close()
    keep = (w_o > 0) & ~touched
    assert keep.sum() > 20000
    assert np.all(w[touched] == 0)
    assert (np.abs(w[keep] - w_o[keep]) / w_o[keep]).max() <= 1e-5


@pytest.mark.parametrize("shape", [(5, 600000, 5), (1100000, 5, 5)])
def test_peaks_of_long_axes(ttm, shape):
    """Maps longer in y or z than a launch grid's second and third extent of
    blocks; planted scores, some on both sides of that length."""
    import torch
    Z, Y, X = shape
    t = synth.blob_template(5, 3, seed=1)
    comp, desc = ttm.build_template(t, synth.ball_mask(5, 2), 2,
                                    synth.super_fibonacci_quaternions(10).astype(np.float32))
    m = ttm.Matcher([(comp, desc, synth.ball_mask(5, 2))], [((X, Y, Z), 0)])
    score = torch.zeros(shape, device="cuda")
    quat = torch.zeros(shape + (4,), device="cuda")
    at = [0, 7, 65535, 524279, 524280, 524288, 599999] + ([] if Z < Y else [1048559, 1048560, 1099999])
    flat = []
    for k, p in enumerate(at):
        v = (2 * Y + p) * X + 2 if Z < Y else (p * Y + 2) * X + 2
        score.view(-1)[v] = 1.0 + k
        flat.append((p, v, 1.0 + k))
    for radius in (0, 1, 3, 6):
        got = ttm.ttm_extract_peaks(m.plan, 0, score, quat, score, 0.5, radius, 100, m.ws)
        expect = [v for p, v, s in sorted(flat, key=lambda e: -e[2])
                  if not any(abs(p - p2) <= radius and s2 > s for p2, _, s2 in flat)]
        assert ((got["z"].astype(np.int64) * Y + got["y"]) * X + got["x"]).tolist() == expect
    m.close()


@pytest.mark.parametrize("s,n_rot", [(12, 40), (33, 90)])
@pytest.mark.parametrize("offset", [30.0, 1e4])
def test_template_build_far_from_zero(ttm, s, n_rot, offset):
    """A template on a large offset: its mean and variance under the mask come
    from sums that nearly cancel.  A sample is eight products and sums in FP32
    (weights of three factors), at most 12 roundings of the largest value, and
    the mean carries the same, on top of the bound for a template near zero."""
    t = (synth.blob_template(s, 4, seed=s).astype(np.float64) + offset).astype(np.float32)
    mask = synth.ball_mask(s, (s - 1) // 2 - 1)          # samples outside the box would be zero
    q = synth.super_fibonacci_quaternions(n_rot).astype(np.float32)
    comp, _ = ttm.build_template(t, mask, 4, q)
    T = o.tensor_template(t, mask, q.astype(np.float64), np.full(n_rot, 1.0 / n_rot), 4)
    scale = max(np.abs(o.rotated_normalised(t, mask, v)).max() for v in q[:8].astype(np.float64))
    spread = np.ptp(t[mask > 0]).astype(np.float64)
    bound = 2e-5 * np.abs(T).max() + 24 * 2.0 ** -24 * np.abs(t).max() * scale / spread * 2
    assert np.abs(comp.cpu().numpy() - T).max() <= bound


@pytest.mark.parametrize("n", [2, 4, 6])
def test_bits_of_the_scalar_forms(ttm, n):
    """w, score, lambda and q at 1500 voxels, to the bit what the scalar FFT
    passes and the scalar refinement gave before two lines or two candidates
    shared a register pair (recorded in tests/golden/scalar_passes.npz).  Lines
    of 144 and 160 points along z and x, of 48 along y."""
    import os
    gold = np.load(os.path.join(os.path.dirname(__file__), "golden", "scalar_passes.npz"))
    shape = (132, 36, 150)
    wl = synth.make_workload(shape, 9, 3, 2, 1.0, n, 200, radius=4, seeds=(71, 72, 73))
    comp, desc = ttm.build_template(wl.template, wl.mask, n, wl.quadrature)
    res, box = _maps(ttm, wl.volume, comp, desc, wl.mask, path=ttm.TTM_PATH_FFT)
    assert list(box) == [160, 48, 144]
    inner = tuple(d - 8 for d in shape)
    at = np.random.default_rng(9).choice(int(np.prod(inner)), 1500, replace=False)
    z, y, x = (i + 4 for i in np.unravel_index(at, inner))
    for k in ("w", "score", "lam", "quat"):
        assert np.array_equal(res[k][z, y, x], gold[f"{k}{n}"]), k


def _peaks_by_rank(score, threshold, radius):
    """The oracle's peaks (o.extract_peaks) for large cubes: ranks by score and,
    where equal, by falling index; a peak is the highest rank of its cube."""
    from scipy.ndimage import maximum_filter1d
    flat = score.ravel()
    rank = np.empty(flat.size, dtype=np.int64)
    rank[np.lexsort((-np.arange(flat.size), flat))] = np.arange(flat.size)
    best = rank = rank.reshape(score.shape)
    for axis in range(3):
        best = maximum_filter1d(best, 2 * radius + 1, axis=axis, mode="constant", cval=-1)
    idx = np.nonzero(((best == rank) & (score > threshold)).ravel())[0]
    return idx[np.lexsort((idx, -flat[idx]))]


@pytest.mark.parametrize("shape", [(5, 5, 5), (29, 40, 70), (70, 21, 33), (66, 67, 69)])
@pytest.mark.parametrize("levels", [1, 2, 4, 10 ** 6])
def test_peaks_of_large_cubes(ttm, shape, levels):
    """Cubes that hold many cells, up to the largest radius, in maps with a few
    levels (equal scores in whole cells) and with none alike."""
    Z, Y, X = shape
    rng = np.random.default_rng(Y)
    mask = synth.ball_mask(5, 2)
    comp, desc = ttm.build_template(synth.blob_template(5, 3, seed=1), mask, 2,
                                    synth.super_fibonacci_quaternions(10).astype(np.float32))
    m = ttm.Matcher([(comp, desc, mask)], [((X, Y, Z), 0)])
    quat = np.zeros(shape + (4,), dtype=np.float32)
    score = (np.floor(rng.random(shape) * levels) / levels + 0.25).astype(np.float32)
    if shape == (5, 5, 5):
        assert np.array_equal(_peaks_by_rank(score, 0.2, 3), o.extract_peaks(score.astype(np.float64), 0.2, 3, 125))
    for radius in (5, 6, 9, 13, 20, 32):
        got = ttm.ttm_extract_peaks(m.plan, 0, _cuda(score), _cuda(quat), _cuda(score), 0.2,
                                    radius, score.size, m.ws)
        expect = _peaks_by_rank(score, 0.2, radius)
        assert np.array_equal((got["z"].astype(np.int64) * Y + got["y"]) * X + got["x"], expect)
    m.close()


@pytest.mark.parametrize("s,n,n_rot,kind,scale", [
    (6, 4, 180, "ball", 1.0), (6, 4, 179, "ball", 1.0),      # either side of the node count
    (10, 2, 400, "scattered", 1.0), (10, 2, 399, "scattered", 1.0),
    (9, 6, 40, "lopsided", 1.0), (9, 8, 20, "ball", 1.0),
    (3, 2, 700, "full", 1.0), (4, 6, 300, "ball", 1.0),      # no room for the tables
    (13, 4, 200, "soft", 1.0), (32, 2, 20, "soft", 1.0), (33, 2, 20, "soft", 1.0),
    (23, 4, 20, "ball", 1.0), (24, 4, 20, "ball", 1.0),      # either side of the edge
    (12, 4, 200, "ball", 1e-25), (12, 4, 200, "ball", 1e20),
])
def test_template_build_of_both_forms(ttm, s, n, n_rot, kind, scale):
    """Boxes and node counts on both sides of the line between the build over
    every voxel and the one over the mask's, and soft masks summed by either."""
    t = (synth.blob_template(s, 4, seed=s).astype(np.float64) * scale).astype(np.float32)
    if kind == "soft":
        mask = synth.soft_ball_mask(s, s // 2, 2.0)
    else:
        mask = np.ones((s, s, s), np.float32) if kind == "full" else _mask(kind, s)
    q = synth.super_fibonacci_quaternions(n_rot).astype(np.float32)
    w = np.random.default_rng(s).random(n_rot).astype(np.float32)
    w /= w.sum()
    comp, desc = ttm.build_template(t, mask, n, q, weights=w)
    T = o.tensor_template(t, mask, q.astype(np.float64), w.astype(np.float64), n)
    assert desc.mask_sum == pytest.approx(mask.sum(dtype=np.float64))
    assert np.abs(comp.cpu().numpy() - T).max() <= 2e-5 * np.abs(T).max()
