// Peaks of the TTM position score (Sec. 3.4 of the paper: the Frobenius norm
// of C_n(x) locates candidate matches).  A voxel is a peak when its score
// exceeds the threshold and beats every other voxel of the (2r+1)^3 cube
// around it; equal scores go to the lower linear index.
//
// Three passes: the voxels above the threshold that are the largest of their
// 3^3 cube (a few in a hundred) with the maxima of 4^3 cells, then those that
// no cell inside their cube beats, then the voxels of the cubes that are left
// (up to radius 4 the cubes at once).
// Few loads per voxel are needed either way, so the passes are bound by L1/L2
// and latency, not by the (2r+1) loads per axis of a separable maximum (256^3,
// r = 12: 1559 us).
#include <algorithm>

#include "ttm_internal.h"

namespace ttm {

namespace {

struct PeakRec {
    int idx;
    float score;
    float lambda;
    float q[4];
    int pad;
};

// Voxels above the threshold that no voxel of their 3^3 cube beats (radius 0:
// every voxel above the threshold), and the maxima of the cells of kCell^3
// voxels.  A CTA owns 32 x 8 x W voxels; a thread walks the planes of one
// (x, y) and keeps what its neighbours' planes held, so a voxel costs nine
// loads that hit L1.  The CTA's survivors are gathered in shared memory and
// take their list slots with one atomic (one per warp and plane made the
// counter the limit: 249 us at 256^3, now 66).  No two survivors are within
// one voxel of each other on every axis, so prod ceil(d / 2) bounds them.
// W planes per CTA: 16, or 4 in maps too small to give every SM two CTAs of 16
// (the planes are a chain of loads: 50 x 41 x 37, nothing above the threshold, the
// whole call 53 -> 44 us; 51 with a separable maximum).
constexpr int kCell = 4;

template <int W>
__global__ void __launch_bounds__(256) peak_candidates_kernel(
    const float* __restrict__ score, int X, int Y, int Z, int radius, float thr,
    int* __restrict__ cand, int* __restrict__ n_cand, float* __restrict__ cells) {
    __shared__ int found[256 * W];
    __shared__ int n_found, base_s;
    __shared__ float part[8][32 / kCell][W / kCell];      // [y][cell x][cell z]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // block (bx, by, bz) of a one-dimensional grid: y and z may be longer than
    // a grid's second and third extent
    const unsigned nbx = (unsigned)(X + 31) / 32, nby = (unsigned)(Y + 7) / 8;
    const int bx = (int)(blockIdx.x % nbx), by = (int)(blockIdx.x / nbx % nby),
              bz = (int)(blockIdx.x / nbx / nby);
    const int x = bx * 32 + lane;
    const int y = by * 8 + warp;
    const int z0 = bz * W, z1 = min(z0 + W, Z);
    const size_t plane = (size_t)X * Y;
    const bool in = x < X && y < Y;
    const int xc = min(x, X - 1), yc = min(y, Y - 1);
    const int xl = max(xc - 1, 0), xr = min(xc + 1, X - 1);
    const int yl = max(yc - 1, 0), yr = min(yc + 1, Y - 1);
    if (t == 0) n_found = 0;
    __syncthreads();
    // the 3 x 3 square of plane z about (x, y), neighbours outside the volume
    // clamped onto its voxels: the centre, the maximum of the square, and the
    // maxima of its voxels before (a lower linear index) and after the centre
    struct Square {
        float centre, all, before, after;
    };
    auto square = [&](int z) {
        const float* p = score + (size_t)z * plane;
        const float* a = p + (size_t)yl * X;
        const float* b = p + (size_t)yc * X;
        const float* c = p + (size_t)yr * X;
        Square q;
        q.centre = __ldg(b + xc);
        const float ra = fmaxf(fmaxf(__ldg(a + xl), __ldg(a + xc)), __ldg(a + xr));
        const float rc = fmaxf(fmaxf(__ldg(c + xl), __ldg(c + xc)), __ldg(c + xr));
        const float l = __ldg(b + xl);
        q.after = fmaxf(__ldg(b + xr), rc);
        q.before = fmaxf(y > 0 ? ra : -INFINITY, x > 0 ? l : -INFINITY);
        q.all = fmaxf(fmaxf(ra, fmaxf(l, q.centre)), q.after);
        return q;
    };
    float below = z0 > 0 ? square(z0 - 1).all : -INFINITY;
    Square here = square(z0);
    float cell = -INFINITY;
#pragma unroll 4
    for (int z = z0; z < z0 + W; ++z) {
        if (z < z1) {
            const Square above = square(min(z + 1, Z - 1));
            const float mid = here.centre;
            const bool lost = radius > 0 && (below >= mid || here.before >= mid || here.after > mid ||
                                             above.all > mid);
            if (in && mid > thr && !lost)
                found[atomicAdd(&n_found, 1)] = (int)((size_t)z * plane + (size_t)y * X + x);
            cell = fmaxf(cell, in ? mid : -INFINITY);
            below = here.all;
            here = above;
        }
        if ((z & (kCell - 1)) == kCell - 1) {                 // z0 is a multiple of kCell
            for (int o = 1; o < kCell; o <<= 1)
                cell = fmaxf(cell, __shfl_xor_sync(0xffffffffu, cell, o));
            if ((lane & (kCell - 1)) == 0) part[warp][lane / kCell][(z - z0) / kCell] = cell;
            cell = -INFINITY;
        }
    }
    __syncthreads();
    if (t == 0 && n_found) base_s = atomicAdd(n_cand, n_found);
    const int CX = (X + kCell - 1) / kCell, CY = (Y + kCell - 1) / kCell, CZ = (Z + kCell - 1) / kCell;
    if (t < 2 * (32 / kCell) * (W / kCell)) {
        const int cx = t % (32 / kCell), cy = (t / (32 / kCell)) % 2, cz = t / (2 * (32 / kCell));
        float m = part[cy * kCell][cx][cz];
#pragma unroll
        for (int k = 1; k < kCell; ++k) m = fmaxf(m, part[cy * kCell + k][cx][cz]);
        const int gx = bx * (32 / kCell) + cx, gy = by * 2 + cy, gz = bz * (W / kCell) + cz;
        if (gx < CX && gy < CY && gz < CZ) cells[((size_t)gz * CY + gy) * CX + gx] = m;
    }
    __syncthreads();
    for (int k = t; k < n_found; k += 256) cand[base_s + k] = found[k];
}

__device__ __forceinline__ void emit_peak(int v, const float* __restrict__ score,
                                          const float* __restrict__ quat, const float* __restrict__ lam,
                                          PeakRec* __restrict__ list, int cap, int* __restrict__ count) {
    const int slot = atomicAdd(count, 1);
    if (slot >= cap) return;
    PeakRec rec;
    rec.idx = v;
    rec.score = score[v];
    rec.lambda = lam ? lam[v] : 0.f;
    const float4 q = quat ? reinterpret_cast<const float4*>(quat)[v] : make_float4(1.f, 0.f, 0.f, 0.f);
    rec.q[0] = q.x; rec.q[1] = q.y; rec.q[2] = q.z; rec.q[3] = q.w;
    rec.pad = 0;
    list[slot] = rec;
}

// radius 0 and 1: every candidate is a peak
__global__ void __launch_bounds__(256) peak_all_kernel(
    const float* __restrict__ score, const float* __restrict__ quat, const float* __restrict__ lam,
    const int* __restrict__ cand, const int* __restrict__ n_cand, PeakRec* __restrict__ list, int cap,
    int* __restrict__ count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < *n_cand; i += gridDim.x * blockDim.x)
        emit_peak(cand[i], score, quat, lam, list, cap, count);
}

// cells of an axis (C of them, N voxels) whose every voxel is within r of p (the
// last cell ends at the volume)
__device__ __forceinline__ void cell_span(int p, int r, int N, int C, int& first, int& last) {
    const int lo = max(p - r, 0), hi = min(p + r, N - 1);
    first = (lo + kCell - 1) / kCell;
    last = hi == N - 1 ? C - 1 : (hi + 1) / kCell - 1;
}

// Order of visits from the middle outwards: 0, -1, +1, -2, +2, ...
__device__ __forceinline__ int outward(int k) { return (k & 1) ? -((k + 1) >> 1) : k >> 1; }

// One thread per candidate: it reads the maxima of the cells that lie wholly
// inside its (2r+1)^3 cube, the planes and rows of cells nearest it first, and
// leaves at the first that is higher.  A cell stands for 64 voxels, so most leave
// after a read or two.  The rest are listed for peak_scan_kernel.  FAR (radius 16
// and more): one thread looks at five planes and rows of cells, the scan at the
// others, and an equal cell below the candidate's own layer beats it too (it holds
// that score at a lower linear index).
constexpr int kNearCells = 5;
constexpr int kFarRadius = 16;

template <bool FAR>
__global__ void __launch_bounds__(256) peak_cells_kernel(
    const float* __restrict__ score, int X, int Y, int Z, int r, const int* __restrict__ cand,
    const int* __restrict__ n_cand, const float* __restrict__ cells, int* __restrict__ left,
    int* __restrict__ n_left) {
    const int n = *n_cand;
    const int CX = (X + kCell - 1) / kCell, CY = (Y + kCell - 1) / kCell, CZ = (Z + kCell - 1) / kCell;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int v = __ldg(cand + i);
        const float s = __ldg(score + v);
        const int row = v / X, x = v - row * X, z = row / Y, y = row - z * Y;
        int fx, ex, fy, ey, fz, ez;
        cell_span(x, r, X, CX, fx, ex);
        cell_span(y, r, Y, CY, fy, ey);
        cell_span(z, r, Z, CZ, fz, ez);
        const int cy = y / kCell, cz = z / kCell;
        const int nz = FAR ? kNearCells : 2 * max(ez - cz, cz - fz) + 1;
        const int ny = FAR ? kNearCells : 2 * max(ey - cy, cy - fy) + 1;
        bool beaten = false;
        for (int kz = 0; kz < nz && !beaten; ++kz) {
            const int gz = cz + outward(kz);
            if (gz < fz || gz > ez) continue;
            for (int ky = 0; ky < ny && !beaten; ++ky) {
                const int gy = cy + outward(ky);
                if (gy < fy || gy > ey) continue;
                const float* c = cells + ((size_t)gz * CY + gy) * CX;
                for (int gx = fx; gx <= ex; ++gx) {
                    if constexpr (FAR) {
                        const float m = __ldg(c + gx);
                        beaten = beaten || m > s || (m == s && gz < cz);
                    } else {
                        beaten = beaten || __ldg(c + gx) > s;
                    }
                }
            }
        }
        if (!beaten) left[atomicAdd(n_left, 1)] = v;
    }
}

// Radius 2 to 4: one warp per candidate.  The cube has 125 to 729 voxels and
// hardly a whole cell, and a few voxels in a hundred are candidates: cells that
// turn almost none of them away, then a CTA with its block-wide votes for each,
// took longer than the separable maximum these passes replace (256 x 251 x 259
// of noise, peak kernels: r = 1 465 us before them, 1552 with a CTA each, 123
// now; r = 2 515, 1255, 316; r = 3 553, 644, 361; r = 4 621, 433, 393; at r = 5
// the cells pay: 260 against 438).
constexpr int kWarpRadius = 4;

__global__ void __launch_bounds__(256) peak_warp_kernel(
    const float* __restrict__ score, const float* __restrict__ quat, const float* __restrict__ lam,
    int X, int Y, int Z, int r, const int* __restrict__ cand, const int* __restrict__ n_cand,
    PeakRec* __restrict__ list, int cap, int* __restrict__ count) {
    const int n = *n_cand, lane = threadIdx.x & 31;
    for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += gridDim.x * 8) {
        const int v = __ldg(cand + i);
        const float s = __ldg(score + v);
        const int row = v / X, x = v - row * X, z = row / Y, y = row - z * Y;
        const int xa = max(x - r, 0), w = min(x + r, X - 1) - xa + 1;
        const int ya = max(y - r, 0), h = min(y + r, Y - 1) - ya + 1;
        const int za = max(z - r, 0), d = min(z + r, Z - 1) - za + 1;
        bool beaten = false;
        for (int e0 = 0; e0 < w * h * d && !beaten; e0 += 128) {    // four loads in flight
            bool hit = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int e = e0 + 32 * j + lane;
                if (e >= w * h * d) break;
                const int rr = e / w, rz = rr / h;
                const int o_at = ((za + rz) * Y + ya + (rr - rz * h)) * X + xa + (e - rr * w);
                const float o = __ldg(score + o_at);
                hit = hit || o > s || (o == s && o_at < v);
            }
            beaten = __any_sync(0xffffffffu, hit);
        }
        if (!beaten && lane == 0) emit_peak(v, score, quat, lam, list, cap, count);
    }
}

// One CTA per candidate that no cell beat: its threads read the cube plane by
// plane, the nearest first, up to the first voxel that beats it (a higher score,
// or an equal one at a lower linear index).  A candidate that survives is a peak.
// FAR: the rest of the cells inside the cube first, and then of the planes outside
// the candidate's own layer of cells only what lies beside the cells (the whole
// call in us, separable maximum / without FAR / now: 256^3 of noise, r = 32, 14651 /
// 624 / 431, r = 20 4605 / 324 / 276; 50 x 41 x 37, r = 32, 3438 / 190 / 114, with
// three levels of score 76 / 238 / 114.  At r = 12 what is left is too little to
// pay for finding it: 266, with FAR 293).
template <bool FAR>
__global__ void __launch_bounds__(256) peak_scan_kernel(
    const float* __restrict__ score, const float* __restrict__ quat, const float* __restrict__ lam,
    int X, int Y, int Z, int r, const int* __restrict__ left, const int* __restrict__ n_left,
    const float* __restrict__ cells, PeakRec* __restrict__ list, int cap, int* __restrict__ count) {
    const int n = *n_left;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const int v = left[i];
        const float s = score[v];
        const int row = v / X, x = v - row * X, z = row / Y, y = row - z * Y;
        const int xa = max(x - r, 0), w = min(x + r, X - 1) - xa + 1;
        const int ya = max(y - r, 0), h = min(y + r, Y - 1) - ya + 1;
        bool beaten = false;
        // rows and columns of a plane that the cells cover, and the planes
        int x0 = 0, x1 = 0, y0 = 0, y1 = 0, z0 = 0, z1 = 0;
        if constexpr (FAR) {
            const int CX = (X + kCell - 1) / kCell, CY = (Y + kCell - 1) / kCell, CZ = (Z + kCell - 1) / kCell;
            int fx, ex, fy, ey, fz, ez;
            cell_span(x, r, X, CX, fx, ex);
            cell_span(y, r, Y, CY, fy, ey);
            cell_span(z, r, Z, CZ, fz, ez);
            const int nx = ex - fx + 1, ny = ey - fy + 1, nz = ez - fz + 1;
            if (nx > 0 && ny > 0 && nz > 0) {
                bool hit = false;
#pragma unroll 4
                for (int e = threadIdx.x; e < nx * ny * nz; e += 256) {
                    const int gy = e / nx, gz = gy / ny;
                    const float m = __ldg(cells + ((size_t)(fz + gz) * CY + fy + gy - gz * ny) * CX + fx + e - gy * nx);
                    hit = hit || m > s || (m == s && fz + gz < z / kCell);
                }
                beaten = __syncthreads_or(hit);
                x0 = fx * kCell - xa, x1 = (ex + 1) * kCell - xa;
                y0 = fy * kCell - ya, y1 = (ey + 1) * kCell - ya;
                z0 = fz * kCell, z1 = (ez + 1) * kCell;
            }
        }
        for (int k = 0; k <= 2 * r && !beaten; k += 2) {      // two planes a step
            bool hit = false;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int zz = z + outward(k + j);
                if (k + j > 2 * r || zz < 0 || zz >= Z) continue;
                const bool beside = FAR && zz / kCell != z / kCell && zz >= z0 && zz < z1;
                for (int e = threadIdx.x; e < w * h; e += 256) {
                    const int ry = e / w, rx = e - ry * w;
                    if (FAR && beside && rx >= x0 && rx < x1 && ry >= y0 && ry < y1) continue;
                    const int o_at = (zz * Y + ya + ry) * X + xa + rx;
                    const float o = __ldg(score + o_at);
                    hit = hit || o > s || (o == s && o_at < v);
                }
            }
            beaten = __syncthreads_or(hit);
        }
        if (beaten || threadIdx.x != 0) continue;
        emit_peak(v, score, quat, lam, list, cap, count);
    }
}

// Running maximum of c_j(x) = w(x) corr_j(x) over a batch of rotations j0..j0+nb-1
// (Algorithm 1 reduced over the rotation set); first index wins ties.  Outside
// the interior (where no correlation is computed) both outputs are 0.  Bound by
// HBM: the nb maps are read once, eight loads in flight per thread.
__global__ void __launch_bounds__(128) best_rotation_kernel(const float* __restrict__ corr, int nb, int j0,
                                                            const float* __restrict__ w, int X, int Y,
                                                            int Z, int s, float* __restrict__ best,
                                                            int* __restrict__ best_j, int first) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    if (x >= X) return;
    const size_t nvox = (size_t)X * Y * Z, v = ((size_t)z * Y + y) * X + x;
    if (!(interior(x, X, s) && interior(y, Y, s) && interior(z, Z, s))) {
        if (first) {
            best[v] = 0.f;
            best_j[v] = 0;
        }
        return;
    }
    const float wv = w[v];
    float b = first ? -INFINITY : best[v];
    int bj = first ? 0 : best_j[v];
#pragma unroll 8
    for (int j = 0; j < nb; ++j) {
        const float c = wv * __ldg(corr + (size_t)j * nvox + v);
        if (c > b) { b = c; bj = j0 + j; }
    }
    best[v] = b;
    best_j[v] = bj;
}

}  // namespace

ttm_status launch_best_rotation(const float* corr, int nb, int j0, const float* w, int X, int Y, int Z,
                                int s, float* best, int* best_j, bool first, cudaStream_t st,
                                long long* cnt) {
    if (Y > 65535 || Z > 65535) return TTM_ERR_UNSUPPORTED;
    const dim3 grid((unsigned)((X + 127) / 128), (unsigned)Y, (unsigned)Z);
    best_rotation_kernel<<<grid, 128, 0, st>>>(corr, nb, j0, w, X, Y, Z, s, best, best_j, first ? 1 : 0);
    return after_launch(cnt);
}

size_t peak_record_bytes() { return sizeof(PeakRec); }

ttm_status launch_peak_candidates_full(const float* score, const float* quat, const float* lam,
                                       int X, int Y, int Z, float thr, int radius, float* tmp_a,
                                       float* tmp_b, void* list, int cap, int* d_count,
                                       cudaStream_t st, long long* cnt) {
    // tmp_a: the candidates (one per voxel at most).  tmp_b: the cell maxima,
    // then the candidates left after them; prod ceil(d / 4) cells and, from
    // radius 1 up, prod ceil(d / 2) candidates fit its nvox entries (a multiple
    // of 64, which covers the smallest volumes).  The lists' lengths sit beside
    // the peak count; the caller has set all three to zero.
    const int CX = (X + kCell - 1) / kCell, CY = (Y + kCell - 1) / kCell, CZ = (Z + kCell - 1) / kCell;
    int* cand = reinterpret_cast<int*>(tmp_a);
    float* cells = tmp_b;
    int* left = reinterpret_cast<int*>(tmp_b) + (size_t)CX * CY * CZ;
    int* n_cand = d_count + 1;
    int* n_left = d_count + 2;
    PeakRec* recs = reinterpret_cast<PeakRec*>(list);
    // fewer than 2^31 voxels in boxes of 3^3 and more: the blocks fit one extent
    const unsigned columns = (unsigned)((X + 31) / 32) * (unsigned)((Y + 7) / 8);
    if (columns * (unsigned)((Z + 15) / 16) >= 304u)
        peak_candidates_kernel<16><<<columns * (unsigned)((Z + 15) / 16), 256, 0, st>>>(
            score, X, Y, Z, radius, thr, cand, n_cand, cells);
    else
        peak_candidates_kernel<4><<<columns * (unsigned)((Z + 3) / 4), 256, 0, st>>>(
            score, X, Y, Z, radius, thr, cand, n_cand, cells);
    TTM_TRY(after_launch(cnt));
    // no more candidates than voxels, or from radius 1 up than every second one
    // along each axis
    const size_t most = radius == 0 ? (size_t)X * Y * Z
                                    : (size_t)((X + 1) / 2) * ((Y + 1) / 2) * (size_t)((Z + 1) / 2);
    auto blocks = [&](size_t per) { return (unsigned)std::min<size_t>(152 * 8, (most + per - 1) / per); };
    if (radius <= 1) {                                   // the first pass took the whole cube
        peak_all_kernel<<<blocks(256), 256, 0, st>>>(score, quat, lam, cand, n_cand, recs, cap, d_count);
        return after_launch(cnt);
    }
    if (radius <= kWarpRadius) {
        peak_warp_kernel<<<blocks(8), 256, 0, st>>>(score, quat, lam, X, Y, Z, radius, cand, n_cand, recs,
                                                    cap, d_count);
        return after_launch(cnt);
    }
    const bool far = radius >= kFarRadius;
    auto cells_pass = far ? peak_cells_kernel<true> : peak_cells_kernel<false>;
    auto scan_pass = far ? peak_scan_kernel<true> : peak_scan_kernel<false>;
    cells_pass<<<blocks(256), 256, 0, st>>>(score, X, Y, Z, radius, cand, n_cand, cells, left, n_left);
    TTM_TRY(after_launch(cnt));
    scan_pass<<<blocks(1), 256, 0, st>>>(score, quat, lam, X, Y, Z, radius, left, n_left, cells, recs, cap,
                                         d_count);
    return after_launch(cnt);
}

}  // namespace ttm
