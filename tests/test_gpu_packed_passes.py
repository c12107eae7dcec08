"""The packed FFT passes at every length they are compiled for, on the sides
that short boxes do not reach.

The packed column passes take spectra whose rows are whole tiles of columns,
which rows of fewer than 128 points never are, so long y lines need a box of 128
points or more along x.  The packed multiply gives a CTA a second column tile
only where there are more tiles than SMs.  Tolerances are those of the parity
tests: 1e-4 on the components (FP32), 5e-3 with bf16 storage, 1e-5 relative on w.
"""

import numpy as np
import pytest

import synth
from oracle import ttm_oracle as o

pytestmark = pytest.mark.gpu

TOL = 1e-4
BF16_TOL = 5e-3
LONG = [128, 144, 160, 192, 240, 256, 288, 320, 384, 480, 512, 576, 640, 768, 960, 1024]


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


def _check(ttm, shape, box, seeds):
    """Components and w of a (Z, Y, X) volume on the FFT path against the oracle."""
    import torch
    wl = synth.make_workload(list(shape), 7, 3, 2, 1.0, 2, 60, radius=3, seeds=seeds)
    T = o.tensor_template(wl.template, wl.mask, wl.quadrature.astype(np.float64), wl.weights, 2)
    comp, desc = ttm.build_template(wl.template, wl.mask, 2, wl.quadrature)
    w_o, C_o = o.ttm_components(wl.volume, T, wl.mask)
    nz = w_o > 0
    for precision, tol in ((ttm.TTM_PREC_FP32, TOL), (ttm.TTM_PREC_MIXED, BF16_TOL)):
        po = ttm.PlanOpts()
        po.path, po.precision = ttm.TTM_PATH_FFT, precision
        m = ttm.Matcher([(comp, desc, wl.mask)], [(shape[::-1], 0)], opts=po)
        assert list(ttm.ttm_plan_problem_fft_box(m.plan, 0)) == box
        out = torch.empty((desc.K,) + tuple(shape), dtype=torch.float32, device="cuda")
        m.run([_cuda(wl.volume)], components_out=[out])
        torch.cuda.synchronize()
        assert ttm.ttm_plan_device_status(m.plan, m.ws) == 0
        w = m.w[0].cpu().numpy()
        assert np.abs(out.cpu().numpy() - C_o).max() <= tol
        assert np.array_equal(w > 0, nz)
        assert (np.abs(w[nz] - w_o[nz]) / w_o[nz]).max() <= 1e-5
        m.close()


@pytest.mark.parametrize("length", LONG)
def test_long_y_lines(ttm, length):
    """Rows of 113 to 126 voxels (a pitch of 72: nine tiles of eight columns,
    seven of them padding), lines up to three voxels short."""
    short = length // 64 % 4
    _check(ttm, (14, length - short, 113 + length // 16 % 14), [128, length, 16], (61, 62, 63))


@pytest.mark.parametrize("length", [160, 288, 480, 960])
def test_long_x_rows(ttm, length):
    short = length // 32 % 4
    _check(ttm, (17, 22, length - short), [length, 32, 32], (64, 65, 66))


@pytest.mark.parametrize("length", [n for n in LONG if n <= 512])
def test_long_z_lines_over_many_tiles(ttm, length):
    """48 x 72 columns: 216 tiles of 16 columns or 432 of 8, more than SMs, so
    a CTA goes on to a second tile with its image and components copied ahead."""
    short = length // 64 % 4
    _check(ttm, (length - short, 35, 113), [128, 48, length], (67, 68, 69))


@pytest.mark.parametrize("depth,s,n_rot", [(126, 9, 3), (142, 8, 35), (190, 11, 5), (237, 12, 7), (253, 9, 4),
                                           (381, 9, 3), (477, 7, 3)])
def test_classical_over_many_tiles(ttm, depth, s, n_rot):
    """The same columns in classical matching, where the templates' z transform
    runs inside the multiply; 35 rotations leave a last batch of three."""
    import torch
    rng = np.random.default_rng(depth)
    shape = (depth, 35, 113)
    volume = rng.normal(size=shape).astype(np.float32)
    t, mask = synth.blob_template(s, 4, seed=s), synth.ball_mask(s)
    q = synth.shoemake_quaternions(n_rot, 4).astype(np.float32)
    comp, desc = ttm.build_template(t, mask, 2, synth.super_fibonacci_quaternions(20).astype(np.float32))
    po = ttm.PlanOpts()
    po.path = ttm.TTM_PATH_FFT
    m = ttm.Matcher([(comp, desc, mask)], [(shape[::-1], 0)], opts=po)
    vol = _cuda(volume)
    ttm.ttm_local_stats(m.plan, [vol], m.w, m.ws)
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
