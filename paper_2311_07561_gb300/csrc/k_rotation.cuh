// Per-voxel TTM score and rotation (kernel template; instantiated per order n
// in k_rotation_n*.cu) (Sec. 3.2-3.4 of the paper).
//
//   C_alpha(x) = w(x) Corr_alpha(x)
//   score(x)   = ||C_n(x)||_F = sqrt(sum_alpha mu_alpha C_alpha^2)          (Sec. 3.4)
//   lambda(x)  = max_{|Q|=1} phi(Q),  phi(Q) = C_n(x) . Q^(n)                (Sec. 3.3)
//   q(x)       = argmax, the dominant Z-eigenvector of C_n(x)                (Sec. 3.1)
//
// One thread per interior voxel.  The maximum is searched on a fixed grid of unit
// quaternions (half sphere, sorted into regions of equal size): phi at every grid point is a
// dot product with a precomputed row mu_alpha q_g^alpha staged in shared memory
// and read as a broadcast.  The best point of each region competes for a short
// list of n_cand candidates.  Every candidate takes two shifted power steps
// (x <- normalise(C x^{n-1} + sigma x), sigma = (n-1) score, the SS-HOPM step
// of Kolda & Mayo 2011, monotone for this shift); the n_refine (<= kRefine)
// best of the points reached are then refined by Riemannian Newton steps on the sphere,
// each accepted only if phi does not decrease (otherwise the power step is
// taken).  The largest refined value wins.
#pragma once
#include <cuda_bf16.h>

#include "ttm_f2.cuh"
#include "ttm_internal.h"

namespace ttm {

namespace rot {

constexpr int kRotThreads = 128;
constexpr int kChunk = 128;       // grid points staged per step
constexpr int kMaxCand = 8;
constexpr int kRefine = 4;        // candidates refined by Newton after the power steps

// correlation maps are float or bf16 (mixed precision)
__device__ __forceinline__ float ldcorr(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ldcorr(const __nv_bfloat16* p) { return __bfloat162float(__ldg(p)); }

// The problems and units of one launch (RotBatch, in the kernel parameters,
// read in place: the kernels take their arguments as __grid_constant__).
struct SearchArgs {
    RotBatch b;
    UnitList list;          // optional unit list (peaks; one problem per launch)
    const float* gm;        // n_grid x K4 (SIMT search)
    const int* cell_end;    // n_grid
    int n_grid;
    int n_cand;             // candidates the refinement reads
};

struct PolishArgs {
    RotBatch b;
    UnitList list;          // optional unit list (peaks) and strided outputs
    const float* gq;        // n_grid x 4
    int n_cand, newton, n_refine;
    int n_grid;             // a candidate from n_grid up is none: 0xFFFF, or what a
                            // search that gave up has left unwritten
};

static_assert(kRotThreads == kRotTile, "one block of the SIMT kernels is one tile");

// segment of tile t: segments are in tile order, so s only moves forward
static __device__ __forceinline__ int seg_of(const RotBatch& b, uint32_t t, int s = 0) {
    while (s + 1 < b.n && t >= b.seg[s + 1].tile0) ++s;
    return s;
}

// The score sum_alpha mu_alpha C_alpha^2 is accumulated in two halves, the
// components below score_split<N>() and the rest, added at the end (two shorter
// chains): every kernel that writes a score map sums in this same order, so the
// maps agree bit for bit.
template <int N>
__host__ __device__ constexpr int score_split() { return ((n_comp(N) + 1 + 15) / 16) * 8; }

// end of the units [.., u1) and the voxel of unit i, with an optional list
static __device__ __forceinline__ uint32_t list_end(const UnitList& l, uint32_t u1) {
    if (!l.count) return u1;
    const int c = *l.count;
    return c <= 0 ? 0u : ((uint32_t)c < u1 ? (uint32_t)c : u1);
}
static __device__ __forceinline__ size_t unit_voxel(const VoxBox& b, const UnitList& l, uint32_t i) {
    return l.idx ? (size_t)l.idx[(size_t)i * l.stride] : b.voxel(i);
}

// score = ||C||_F with C = w Corr at the interior voxels, 0 elsewhere; the
// same arithmetic as the search kernels.  Block (x segment, y, z).
template <int N, typename CT>
__global__ void __launch_bounds__(128) score_only_kernel(const CT* __restrict__ corr,
                                                         const float* __restrict__ w, int X, int Y,
                                                         size_t nvox, VoxBox box,
                                                         float* __restrict__ score) {
    constexpr int K = n_comp(N);
    constexpr Sym<N> S{};
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    if (x >= X) return;
    const size_t v = ((size_t)z * Y + y) * X + x;
    const bool in = (uint32_t)(x - box.x0) < box.nx && (uint32_t)(y - box.y0) < box.ny &&
                    (uint32_t)(z - box.z0) < box.nz;
    float ss0 = 0.f, ss1 = 0.f;
    if (in) {
        const float wv = __ldg(w + v);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float c = wv * ldcorr(corr + (size_t)k * nvox + v);
            if (k < score_split<N>()) ss0 = fmaf((float)S.mu[k], c * c, ss0);
            else ss1 = fmaf((float)S.mu[k], c * c, ss1);
        }
    }
    score[v] = sqrtf(ss0 + ss1);
}

// keep the kMaxCand largest (value, index) pairs, sorted descending
static __device__ __forceinline__ void insert_candidate(float (&tv)[kMaxCand], int (&ti)[kMaxCand],
                                                 float val, int idx) {
#pragma unroll
    for (int k = 0; k < kMaxCand; ++k) {
        if (val > tv[k]) {
            float t = tv[k]; tv[k] = val; val = t;
            int u = ti[k]; ti[k] = idx; idx = u;
        }
    }
}

static __device__ __forceinline__ void store_candidates(uint16_t* cand, size_t v, const int (&ti)[kMaxCand],
                                                 bool active) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t lo = active ? (uint32_t)(ti[2 * k] & 0xFFFF) : 0xFFFFu;
        uint32_t hi = active ? (uint32_t)(ti[2 * k + 1] & 0xFFFF) : 0xFFFFu;
        w[k] = lo | (hi << 16);
    }
    reinterpret_cast<uint4*>(cand)[v] = make_uint4(w[0], w[1], w[2], w[3]);
}

template <int N>
struct Geo {
    static constexpr int K = n_comp(N);
    static constexpr int K4 = (K + 3) & ~3;
};

// H = C x^{N-2} (symmetric 4x4, 10 entries in the order of HessTab pairs)
template <int N>
__device__ __forceinline__ void hess(const float (&C)[Geo<N>::K4], const float x[4], float h[10]) {
    constexpr HessTab<N> T{};
    Monomials<N - 2> mb;
    monomials<N - 2>(x, mb);
    float mw[HessTab<N>::KB];
#pragma unroll
    for (int b = 0; b < HessTab<N>::KB; ++b) mw[b] = (float)T.mult[b] * mb.v[b];
#pragma unroll
    for (int p = 0; p < 10; ++p) {
        float acc = 0.f;
#pragma unroll
        for (int b = 0; b < HessTab<N>::KB; ++b) acc = fmaf(mw[b], C[T.comp[p][b]], acc);
        h[p] = acc;
    }
}

// full 4x4 from the 10 stored entries (pairs i <= j in row order)
static __device__ __forceinline__ void unpack(const float h[10], float H[4][4]) {
    int p = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j) {
            H[i][j] = h[p];
            H[j][i] = h[p];
            ++p;
        }
}

static __device__ __forceinline__ void normalise4(float x[4]) {
    float n2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2] + x[3] * x[3];
    float inv = rsqrtf(n2);
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] *= inv;
}

// value and gradient pieces at x: H = C x^{N-2}, g = H x = C x^{N-1}, lam = x.g
template <int N>
__device__ __forceinline__ void eval_at(const float (&C)[Geo<N>::K4], const float x[4],
                                        float H[4][4], float g[4], float& lam) {
    float h[10];
    hess<N>(C, x, h);
    unpack(h, H);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        g[i] = H[i][0] * x[0] + H[i][1] * x[1] + H[i][2] * x[2] + H[i][3] * x[3];
    lam = g[0] * x[0] + g[1] * x[1] + g[2] * x[2] + g[3] * x[3];
}

// Riemannian Newton direction on the unit sphere for maximising phi:
//   P ((N-1) H - lam I) P eta = -(g - lam x),  eta orthogonal to x,
// solved as A eta = (g - lam x) with A = -P B P + sig x x^T, which is SPD
// exactly when the tangent Hessian is negative definite.  Returns false if
// the Cholesky factorisation breaks down (not near a maximum).  Pivots are
// inverted with rsqrt, so the solve has no division.
template <int N>
__device__ __forceinline__ bool newton_dir(const float H[4][4], const float g[4], const float x[4],
                                           float lam, float sig, float eta[4]) {
    float B[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) B[i][j] = (float)(N - 1) * H[i][j] - (i == j ? lam : 0.f);
    float Bx[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) Bx[i] = B[i][0] * x[0] + B[i][1] * x[1] + B[i][2] * x[2] + B[i][3] * x[3];
    const float xBx = x[0] * Bx[0] + x[1] * Bx[1] + x[2] * Bx[2] + x[3] * Bx[3];
    // A = -B + x (Bx)^T + (Bx) x^T + (sig - x^T B x) x x^T, lower triangle only
    const float cxx = sig - xBx;
    float A[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j)
            A[i][j] = fmaf(cxx * x[i], x[j], fmaf(x[i], Bx[j], fmaf(Bx[i], x[j], -B[i][j])));
    float r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = g[i] - lam * x[i];
    const float tiny = 1e-9f * sig;
    float L[4][4] = {};
    float inv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float d = A[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
        if (!(d > tiny)) return false;
        inv[j] = rsqrtf(d);
#pragma unroll
        for (int i = j + 1; i < 4; ++i) {
            float v = A[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) v -= L[i][k] * L[j][k];
            L[i][j] = v * inv[j];
        }
    }
    float y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float v = r[i];
#pragma unroll
        for (int k = 0; k < i; ++k) v -= L[i][k] * y[k];
        y[i] = v * inv[i];
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        float v = y[i];
#pragma unroll
        for (int k = i + 1; k < 4; ++k) v -= L[k][i] * eta[k];
        eta[i] = v * inv[i];
    }
    return true;
}

// g = C x^{N-1} (the gradient of phi divided by N) and lam = x . g
template <int N>
__device__ __forceinline__ void grad_at(const float (&C)[Geo<N>::K4], const float x[4], float g[4],
                                        float& lam) {
    constexpr GradTab<N> T{};
    Monomials<N - 1> mg;
    monomials<N - 1>(x, mg);
    float mw[GradTab<N>::KG];
#pragma unroll
    for (int b = 0; b < GradTab<N>::KG; ++b) mw[b] = (float)T.mult[b] * mg.v[b];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int b = 0; b < GradTab<N>::KG; ++b) acc = fmaf(mw[b], C[T.comp[i][b]], acc);
        g[i] = acc;
    }
    lam = g[0] * x[0] + g[1] * x[1] + g[2] * x[2] + g[3] * x[3];
}

// Two shifted power (SS-HOPM) steps x <- normalise(C x^{N-1} + sigma x) from
// x (the SS-HOPM step of Kolda & Mayo 2011, monotone for this shift); with
// want_lam, lam = phi at the point reached (one more evaluation).
template <int N>
__device__ __forceinline__ void power_steps(const float (&C)[Geo<N>::K4], float sigma, float x[4],
                                            float& lam, bool want_lam) {
    float g[4];
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        grad_at<N>(C, x, g, lam);
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = g[i] + sigma * x[i];
        normalise4(x);
    }
    if (want_lam) grad_at<N>(C, x, g, lam);
}

// Riemannian Newton steps on the sphere from x; a trial that lowers phi is
// rejected and replaced by a power step from the last accepted point (power
// steps with this shift never lower phi).  newton trials are evaluated; no
// direction is formed after the last one.  One evaluation site per iteration
// keeps the code small.
template <int N>
__device__ void refine(const float (&C)[Geo<N>::K4], float sigma, int newton, float x[4],
                       float& lam_out) {
    float xa[4] = {x[0], x[1], x[2], x[3]};
    float ga[4], la = -INFINITY;
    float xt[4] = {x[0], x[1], x[2], x[3]};
    bool trial_newton = false;
    const float eps = 1e-6f * sigma;
    const int iters = 1 + newton;
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        float H[4][4], g[4], lam;
        const bool last = it + 1 == iters;
        // the last trial needs only phi: from order 6 on C x^(n-1) (4 sums)
        // is cheaper than C x^(n-2) (10 sums)
        if (N >= 6 && last && it > 0) grad_at<N>(C, xt, g, lam);
        else eval_at<N>(C, xt, H, g, lam);
        if (trial_newton && lam < la - eps) {
            if (last) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) xt[i] = ga[i] + sigma * xa[i];
            normalise4(xt);
            trial_newton = false;
            continue;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            xa[i] = xt[i];
            ga[i] = g[i];
        }
        la = lam;
        if (last) break;
        float eta[4];
        if (newton_dir<N>(H, ga, xa, la, sigma, eta)) {
            const float en2 = eta[0] * eta[0] + eta[1] * eta[1] + eta[2] * eta[2] + eta[3] * eta[3];
            const float clip = en2 > 0.0625f ? 0.25f * rsqrtf(en2) : 1.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) xt[i] = xa[i] + clip * eta[i];
            trial_newton = true;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) xt[i] = ga[i] + sigma * xa[i];
            trial_newton = false;
        }
        normalise4(xt);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = xa[i];
    lam_out = la;
}

// ---- two candidates at a time (orders 2, 4 and 6) --------------------------
// The refinement is bound by the FMA pipe's register reads: scalar FMAs with
// three different registers each ran at 78-86 lanes a clock and SM, packed
// ones (fma.rn.f32x2, two FMAs per instruction) at 108.  So two candidates of
// a voxel go through the evaluations and the Newton solves together, one in
// each half of a register pair; the components, which both share, are kept as
// pairs of equal halves (2 K registers: 168 at order 6, which leaves two CTAs
// per SM and still gains; the 330 of order 8 do not fit).  Every half carries
// the operations of the scalar code in its order, so the results are the same
// bits.  Whole runs, evaluations packed -> solves too: order 4 at 512 x 512 x
// 256, 29.8 -> 28.4 ms; order 6 at 928 x 464 x 232, all scalar before, 49.7 ->
// 47.6 ms.
template <int M>
struct Monomials2 {
    F2 v[n_comp(M) > 0 ? n_comp(M) : 1];
};

template <int M>
__device__ __forceinline__ void monomials2(const F2 (&x)[4], Monomials2<M>& out) {
    if constexpr (M == 0) {
        out.v[0] = f2(1.0f, 1.0f);
    } else if constexpr (M == 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) out.v[k] = x[k];
    } else {
        Monomials2<M - 1> prev;
        monomials2<M - 1>(x, prev);
        constexpr MonoTab<M> T{};
#pragma unroll
        for (int k = 0; k < n_comp(M); ++k) out.v[k] = f2_mul(prev.v[T.parent[k]], x[T.var[k]]);
    }
}

// a . b in the scalar code's order: a0 b0 + (a1 b1), then a2 b2, a3 b3
__device__ __forceinline__ F2 f2_dot(const F2 (&a)[4], const F2 (&b)[4]) {
    return f2_fma(a[3], b[3], f2_fma(a[2], b[2], f2_fma(a[0], b[0], f2_mul(a[1], b[1]))));
}

// Row i of a symmetric matrix times x.  At order 2 the matrix is C itself and the
// Newton matrix differs from it in the diagonal alone, so the scalar code forms
// the off-diagonal products of the two once, rounded, and only what one of them
// has to itself is fused.  (A packed multiplication and the packed addition after
// it are fused all the same, so a rounded product that is added is scalar.)
__device__ __forceinline__ F2 f2_round_mul(F2 a, F2 b) {
    return f2(__fmul_rn(f2_get(a, 0), f2_get(b, 0)), __fmul_rn(f2_get(a, 1), f2_get(b, 1)));
}
template <int N>
__device__ __forceinline__ F2 f2_row(int i, const F2 (&a)[4], const F2 (&b)[4]) {
    if (N != 2 || i == 3) return f2_dot(a, b);
    const F2 last = f2_round_mul(a[3], b[3]);
    if (i == 2) return f2_add(f2_fma(a[2], b[2], f2_fma(a[0], b[0], f2_mul(a[1], b[1]))), last);
    const F2 s = i == 0 ? f2_fma(a[0], b[0], f2_mul(a[1], b[1])) : f2_fma(a[1], b[1], f2_mul(a[0], b[0]));
    return f2_add(f2_add(s, f2_round_mul(a[2], b[2])), last);
}

// the gradient of grad_at for two points (its lam is f2_dot(x, g))
template <int N>
__device__ __forceinline__ void grad2_at(const F2 (&C)[Geo<N>::K], const F2 (&x)[4], F2 (&g)[4]) {
    constexpr GradTab<N> T{};
    Monomials2<N - 1> mg;
    monomials2<N - 1>(x, mg);
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] = f2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < GradTab<N>::KG; ++b) {
        const F2 mw = T.mult[b] == 1 ? mg.v[b]
                                     : f2_mul(f2((float)T.mult[b], (float)T.mult[b]), mg.v[b]);
#pragma unroll
        for (int i = 0; i < 4; ++i) g[i] = f2_fma(mw, C[T.comp[i][b]], g[i]);
    }
}

// eval_at for two points; h = the 10 entries of H
template <int N>
__device__ __forceinline__ void eval2_at(const F2 (&C)[Geo<N>::K], const F2 (&x)[4], F2 (&h)[10],
                                         F2 (&g)[4], F2& lam) {
    constexpr HessTab<N> T{};
    Monomials2<N - 2> mb;
    monomials2<N - 2>(x, mb);
#pragma unroll
    for (int p = 0; p < 10; ++p) h[p] = f2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < HessTab<N>::KB; ++b) {
        const F2 mw = T.mult[b] == 1 ? mb.v[b]
                                     : f2_mul(f2((float)T.mult[b], (float)T.mult[b]), mb.v[b]);
#pragma unroll
        for (int p = 0; p < 10; ++p) h[p] = f2_fma(mw, C[T.comp[p][b]], h[p]);
    }
    // rows of the symmetric matrix stored as pairs i <= j
    const F2 H[4][4] = {{h[0], h[1], h[2], h[3]}, {h[1], h[4], h[5], h[6]},
                        {h[2], h[5], h[7], h[8]}, {h[3], h[6], h[8], h[9]}};
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] = f2_row<N>(i, H[i], x);
    lam = f2_dot(g, x);
}

// normalise4 for two points
static __device__ __forceinline__ void normalise2(F2 (&x)[4]) {
    const F2 n2 = f2_dot(x, x);
    const F2 inv = f2(rsqrtf(f2_get(n2, 0)), rsqrtf(f2_get(n2, 1)));
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = f2_mul(x[i], inv);
}

// power_steps for two candidates
template <int N>
__device__ __forceinline__ void power_steps2(const F2 (&C)[Geo<N>::K], float sigma, F2 (&x)[4],
                                             F2& lam, bool want_lam) {
    const F2 sig = f2(sigma, sigma);
    F2 g[4];
    lam = f2(0.f, 0.f);
#pragma unroll 1
    for (int s = 0; s < 3; ++s) {
        if (s == 2 && !want_lam) break;
        grad2_at<N>(C, x, g);
        if (s == 2) {
            lam = f2_dot(x, g);
            break;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = f2_fma(sig, x[i], g[i]);
        normalise2(x);
    }
}

// newton_dir for two points: h = the entries of H, ok = each half's success.
// A half whose factorisation breaks down leaves values that nobody reads.
template <int N>
__device__ __forceinline__ void newton_dir2(const F2 (&h)[10], const F2 (&g)[4], const F2 (&x)[4],
                                            F2 lam, float sig, F2 (&eta)[4], bool (&ok)[2]) {
    const F2 minus = f2(-1.f, -1.f), nl = f2_mul(lam, minus);
    const F2 order = f2((float)(N - 1), (float)(N - 1));
    F2 B[4][4];
    int p = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j, ++p) {
            B[i][j] = i == j ? f2_fma(order, h[p], nl) : f2_mul(order, h[p]);
            B[j][i] = B[i][j];
        }
    F2 Bx[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) Bx[i] = f2_row<N>(i, B[i], x);
    const F2 cxx = f2_sub(f2_dot(x, Bx), f2(sig, sig));
#pragma unroll
    for (int i = 0; i < 4; ++i) Bx[i] = f2_mul(Bx[i], minus);
    // nA = -A and nL = -L: the same factorisation with every sign turned, as
    // packed operations take no negated operand
    F2 nA[4][4], nL[4][4], inv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const F2 cx = f2_mul(cxx, x[i]);
#pragma unroll
        for (int j = 0; j <= i; ++j)
            nA[i][j] = f2_fma(cx, x[j], f2_fma(x[i], Bx[j], f2_fma(Bx[i], x[j], B[i][j])));
    }
    const float tiny = 1e-9f * sig;
    ok[0] = ok[1] = true;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        F2 d = nA[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) d = f2_fma(nL[j][k], nL[j][k], d);
        const float da = -f2_get(d, 0), db = -f2_get(d, 1);
        ok[0] = ok[0] && da > tiny;
        ok[1] = ok[1] && db > tiny;
        inv[j] = f2(rsqrtf(da), rsqrtf(db));
#pragma unroll
        for (int i = j + 1; i < 4; ++i) {
            F2 v = nA[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) v = f2_fma(nL[i][k], nL[j][k], v);
            nL[i][j] = f2_mul(v, inv[j]);
        }
    }
    F2 y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        F2 v = f2_fma(nl, x[i], g[i]);
#pragma unroll
        for (int k = 0; k < i; ++k) v = f2_fma(nL[i][k], y[k], v);
        y[i] = f2_mul(v, inv[i]);
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        F2 v = y[i];
#pragma unroll
        for (int k = i + 1; k < 4; ++k) v = f2_fma(nL[k][i], eta[k], v);
        eta[i] = f2_mul(v, inv[i]);
    }
}

static __device__ __forceinline__ F2 f2_pick(bool a, bool b, F2 yes, F2 no) {
    return f2(a ? f2_get(yes, 0) : f2_get(no, 0), b ? f2_get(yes, 1) : f2_get(no, 1));
}

// refine for two points: from xt to the last accepted points xa and their
// values.  Both halves form the Newton point; a half that goes by a power step
// (a rejected trial, or no direction) takes g + sigma x of its accepted point
// in its place before the common normalisation.
template <int N>
__device__ __forceinline__ void refine2(const F2 (&C)[Geo<N>::K], float sigma, int newton,
                                        F2 (&xt)[4], F2 (&xa)[4], float& la, float& lb) {
    const float eps = 1e-6f * sigma;
    const F2 sig = f2(sigma, sigma);
    const int iters = 1 + newton;
    F2 ga[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        xa[i] = xt[i];
        ga[i] = f2(0.f, 0.f);
    }
    la = lb = -INFINITY;
    bool ta = false, tb = false;   // the trial is a Newton point
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        const bool last = it + 1 == iters;
        F2 h[10], g[4], lam;
        // the last trial needs only phi (see refine)
        if (N >= 6 && last && it > 0) {
            grad2_at<N>(C, xt, g);
            lam = f2_dot(xt, g);
        } else eval2_at<N>(C, xt, h, g, lam);
        const float va = f2_get(lam, 0), vb = f2_get(lam, 1);
        const bool keep_a = !(ta && va < la - eps), keep_b = !(tb && vb < lb - eps);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            xa[i] = f2_pick(keep_a, keep_b, xt[i], xa[i]);
            ga[i] = f2_pick(keep_a, keep_b, g[i], ga[i]);
        }
        la = keep_a ? va : la;
        lb = keep_b ? vb : lb;
        if (last) break;
        F2 eta[4];
        bool ok[2];
        newton_dir2<N>(h, g, xt, lam, sigma, eta, ok);
        const F2 en2 = f2_dot(eta, eta);
        const float ea = f2_get(en2, 0), eb = f2_get(en2, 1);
        const F2 clip = f2(ea > 0.0625f ? 0.25f * rsqrtf(ea) : 1.f,
                           eb > 0.0625f ? 0.25f * rsqrtf(eb) : 1.f);
        ta = ok[0] && keep_a;
        tb = ok[1] && keep_b;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            xt[i] = f2_pick(ta, tb, f2_fma(clip, eta[i], xa[i]), f2_fma(sig, xa[i], ga[i]));
        normalise2(xt);
    }
}

// keep the kRefine largest values with their points, sorted descending
static __device__ __forceinline__ void keep_point(float (&kl)[kRefine], float (&kx)[kRefine][4], float l,
                                                  float (&x)[4]) {
#pragma unroll
    for (int s = 0; s < kRefine; ++s) {
        const bool up = l > kl[s];
        const float tl = kl[s];
        kl[s] = up ? l : kl[s];
        l = up ? tl : l;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float tx = kx[s][i];
            kx[s][i] = up ? x[i] : kx[s][i];
            x[i] = up ? tx : x[i];
        }
    }
}

template <int N> constexpr bool kPairs = N <= 6;

// Refinement of a voxel's candidates, two at a time (orders 2, 4 and 6); the
// scalar loops of polish_kernel state the steps.
template <int N>
__device__ __forceinline__ void polish_pairs(const float (&Cs)[Geo<N>::K4], float score,
                                             const uint32_t (&cw)[4], const PolishArgs& a,
                                             float& best_l, float (&best_q)[4]) {
    constexpr int K = Geo<N>::K;
    F2 C[K];
#pragma unroll
    for (int k = 0; k < K; ++k) C[k] = f2(Cs[k], Cs[k]);
    const float sigma = (float)(N - 1) * score;
    best_l = -INFINITY;
    const bool rank = a.n_cand > a.n_refine;
    float kl[kRefine], kx[kRefine][4];
#pragma unroll
    for (int s = 0; s < kRefine; ++s) {
        kl[s] = -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) kx[s][i] = 0.f;
    }
    const int nc = a.n_cand < kMaxCand ? a.n_cand : kMaxCand;
#pragma unroll 1
    for (int k = 0; k < nc; k += 2) {
        const uint32_t pair = k < 4 ? (k < 2 ? cw[0] : cw[1]) : (k < 6 ? cw[2] : cw[3]);
        const int ia = (int)(pair & 0xFFFFu);
        if (ia >= a.n_grid) break;
        int ib = (int)(pair >> 16);
        const bool two = k + 1 < nc && ib < a.n_grid;
        if (!two) ib = ia;
        F2 x[4], lam;
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = f2(__ldg(a.gq + 4 * ia + i), __ldg(a.gq + 4 * ib + i));
        power_steps2<N>(C, sigma, x, lam, rank);
        const float la = rank ? f2_get(lam, 0) : -(float)k;
        const float lb = rank ? f2_get(lam, 1) : -(float)(k + 1);
        float xa[4], xb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            xa[i] = f2_get(x[i], 0);
            xb[i] = f2_get(x[i], 1);
        }
        keep_point(kl, kx, la, xa);
        if (!two) break;
        keep_point(kl, kx, lb, xb);
    }
#pragma unroll 1
    for (int s = 0; s < kRefine; s += 2) {
        if (s >= a.n_refine || !((s == 0 ? kl[0] : kl[2]) > -INFINITY)) break;
        const bool two = s + 1 < a.n_refine && (s == 0 ? kl[1] : kl[3]) > -INFINITY;
        F2 xt[4], xa[4];
        float la, lb;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // the kept points s and s + 1, picked with compile-time indices
            const float p = s == 0 ? kx[0][i] : kx[2][i];
            xt[i] = f2(p, !two ? p : (s == 0 ? kx[1][i] : kx[3][i]));
        }
        refine2<N>(C, sigma, a.newton, xt, xa, la, lb);
        if (la > best_l) {
            best_l = la;
#pragma unroll
            for (int i = 0; i < 4; ++i) best_q[i] = f2_get(xa[i], 0);
        }
        if (two && lb > best_l) {
            best_l = lb;
#pragma unroll
            for (int i = 0; i < 4; ++i) best_q[i] = f2_get(xa[i], 1);
        }
    }
    static_assert(kRefine == 4 && kMaxCand % 2 == 0, "points in pairs");
}

// Score and search: C_alpha = w Corr_alpha, score = ||C||_F, phi at every grid
// point, best point of each region, the n_cand best regions -> candidate grid
// indices (0xFFFF = none).  One thread per voxel; the grid table is staged in
// shared memory and read as broadcasts.
template <int N, typename CT>
__global__ void __launch_bounds__(kRotThreads) search_simt_kernel(const __grid_constant__ SearchArgs a) {
    constexpr int K = Geo<N>::K;
    constexpr int K4 = Geo<N>::K4;
    constexpr Sym<N> S{};
    extern __shared__ __align__(16) float sm[];
    float* Mt = sm;                                   // kChunk x K4
    int* ends = reinterpret_cast<int*>(sm + kChunk * K4);

    const RotSeg& sg = a.b.seg[seg_of(a.b, blockIdx.x)];
    const CT* corr = reinterpret_cast<const CT*>(sg.corr);
    const size_t i = sg.u0 + (size_t)(blockIdx.x - sg.tile0) * kRotTile + threadIdx.x;
    const bool in_range = i < list_end(a.list, sg.u1);
    const size_t v = in_range ? unit_voxel(sg.box, a.list, (uint32_t)i) : 0;
    const float wv = in_range ? __ldg(sg.w + v) : 0.f;
    float C[K4];
#pragma unroll
    for (int k = 0; k < K4; ++k) C[k] = 0.f;
    float ss0 = 0.f, ss1 = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float c = in_range ? wv * ldcorr(corr + (size_t)k * sg.nvox + v) : 0.f;
        C[k] = c;
        if (k < score_split<N>()) ss0 = fmaf((float)S.mu[k], c * c, ss0);
        else ss1 = fmaf((float)S.mu[k], c * c, ss1);
    }
    const float score = sqrtf(ss0 + ss1);
    const bool active = in_range && score > 0.f;

    float tv[kMaxCand];
    int ti[kMaxCand];
#pragma unroll
    for (int k = 0; k < kMaxCand; ++k) { tv[k] = -INFINITY; ti[k] = 0xFFFF; }
    float cur = -INFINITY;
    int curi = 0;
    const bool any_active = __syncthreads_or(active);
    for (int g0 = 0; g0 < a.n_grid && any_active; g0 += kChunk) {
        const int gn = min(kChunk, a.n_grid - g0);
        __syncthreads();
        const float4* src = reinterpret_cast<const float4*>(a.gm + (size_t)g0 * K4);
        float4* dst = reinterpret_cast<float4*>(Mt);
        for (int e = threadIdx.x; e < gn * (K4 / 4); e += blockDim.x) dst[e] = __ldg(src + e);
        for (int e = threadIdx.x; e < gn; e += blockDim.x) ends[e] = __ldg(a.cell_end + g0 + e);
        __syncthreads();
        for (int gg = 0; gg < gn; ++gg) {
            const float4* row = reinterpret_cast<const float4*>(Mt + gg * K4);
            float phi = 0.f;
#pragma unroll
            for (int c4 = 0; c4 < K4 / 4; ++c4) {
                const float4 m = row[c4];
                phi = fmaf(m.x, C[4 * c4 + 0], phi);
                phi = fmaf(m.y, C[4 * c4 + 1], phi);
                phi = fmaf(m.z, C[4 * c4 + 2], phi);
                phi = fmaf(m.w, C[4 * c4 + 3], phi);
            }
            if (phi > cur) { cur = phi; curi = g0 + gg; }
            if (ends[gg]) {
                insert_candidate(tv, ti, cur, curi);
                cur = -INFINITY;
            }
        }
    }
    if (!in_range) return;
    sg.score[v] = score;
    store_candidates(sg.cand, i, ti, active);
}

// CTAs per SM the refinement's registers are sized for: four (128 registers)
// at orders 2 and 4; two from order 6 on, whose K = 84 components as pairs fill
// 168 (three CTAs spill 250 bytes a thread) and whose K = 165 at order 8 take
// all there are
template <int N> constexpr int polish_ctas() { return N <= 4 ? 4 : 2; }

// Refinement of the candidates and the outputs: lambda = the largest refined
// phi, q its maximiser (canonical sign), C_alpha optionally.
template <int N, typename CT>
__global__ void __launch_bounds__(kRotThreads, polish_ctas<N>()) polish_kernel(const __grid_constant__ PolishArgs a) {
    constexpr int K = Geo<N>::K;
    constexpr int K4 = Geo<N>::K4;
    const RotSeg& sg = a.b.seg[seg_of(a.b, blockIdx.x)];
    const CT* corr = reinterpret_cast<const CT*>(sg.corr);
    const size_t i = sg.u0 + (size_t)(blockIdx.x - sg.tile0) * kRotTile + threadIdx.x;
    if (i >= list_end(a.list, sg.u1)) return;
    const size_t v = unit_voxel(sg.box, a.list, (uint32_t)i);
    const float wv = __ldg(sg.w + v);
    float C[K4];
#pragma unroll
    for (int k = 0; k < K4; ++k) C[k] = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float c = wv * ldcorr(corr + (size_t)k * sg.nvox + v);
        C[k] = c;
        if (sg.comp_out) sg.comp_out[(size_t)k * sg.nvox + v] = c;
    }
    const float score = __ldg(sg.score + v);
    const uint4 cr = __ldg(reinterpret_cast<const uint4*>(sg.cand) + i);
    const uint32_t cw[4] = {cr.x, cr.y, cr.z, cr.w};
    float best_l = 0.f;
    float best_q[4] = {1.f, 0.f, 0.f, 0.f};
    if (score > 0.f && (int)(cw[0] & 0xFFFFu) < a.n_grid) {
        if constexpr (kPairs<N>) {
            polish_pairs<N>(C, score, cw, a, best_l, best_q);
        } else {
        const float sigma = (float)(N - 1) * score;
        best_l = -INFINITY;
        // phase 1: two power steps from every candidate; the kRefine best
        // (by phi at the point reached) are kept, sorted descending.  When
        // every candidate is refined the ranking only orders the refinement:
        // the candidates keep the search's order and phi is not evaluated
        const bool rank = a.n_cand > a.n_refine;
        float kl[kRefine], kx[kRefine][4];
#pragma unroll
        for (int s = 0; s < kRefine; ++s) {
            kl[s] = -INFINITY;
#pragma unroll
            for (int i = 0; i < 4; ++i) kx[s][i] = 0.f;
        }
#pragma unroll 1
        for (int k = 0; k < a.n_cand && k < kMaxCand; ++k) {
            const int gi = (int)((cw[k >> 1] >> (16 * (k & 1))) & 0xFFFFu);
            if (gi >= a.n_grid) break;
            float x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = __ldg(a.gq + 4 * gi + i);
            float l;
            power_steps<N>(C, sigma, x, l, rank);
            if (!rank) l = -(float)k;
#pragma unroll
            for (int s = 0; s < kRefine; ++s) {
                const bool up = l > kl[s];
                const float tl = kl[s];
                kl[s] = up ? l : kl[s];
                l = up ? tl : l;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float tx = kx[s][i];
                    kx[s][i] = up ? x[i] : kx[s][i];
                    x[i] = up ? tx : x[i];
                }
            }
        }
        // phase 2: Newton refinement of the n_refine best kept points
#pragma unroll 1
        for (int s = 0; s < kRefine; ++s) {
            if (s >= a.n_refine) break;
            // the kept point s, picked with compile-time indices (registers,
            // no local memory)
            float ls = -INFINITY, x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < kRefine; ++j) {
                const bool pick = j == s;
                ls = pick ? kl[j] : ls;
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = pick ? kx[j][i] : x[i];
            }
            if (!(ls > -INFINITY)) break;
            float l;
            refine<N>(C, sigma, a.newton, x, l);
            if (l > best_l) {
                best_l = l;
#pragma unroll
                for (int i = 0; i < 4; ++i) best_q[i] = x[i];
            }
        }
        }
        // canonical representative of {q, -q}: first non-zero component positive
        float sgn = 1.f;
        if (best_q[0] != 0.f) sgn = best_q[0] < 0.f ? -1.f : 1.f;
        else if (best_q[1] != 0.f) sgn = best_q[1] < 0.f ? -1.f : 1.f;
        else if (best_q[2] != 0.f) sgn = best_q[2] < 0.f ? -1.f : 1.f;
        else sgn = best_q[3] < 0.f ? -1.f : 1.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) best_q[i] *= sgn;
    }
    if (a.list.out_stride > 0) {
        float* qo = sg.quat + i * (size_t)a.list.out_stride;
#pragma unroll
        for (int k = 0; k < 4; ++k) qo[k] = best_q[k];
        if (sg.lambda) sg.lambda[i * (size_t)a.list.out_stride] = best_l;
        return;
    }
    reinterpret_cast<float4*>(sg.quat)[v] = make_float4(best_q[0], best_q[1], best_q[2], best_q[3]);
    if (sg.lambda) sg.lambda[v] = best_l;
}

// search_done: run only the refinement; search_only: run only the SIMT search
template <int N, typename CT>
ttm_status launch_n_t(const SearchArgs& s, const PolishArgs& p, bool search_done, bool search_only,
                      cudaStream_t st, long long* cnt) {
    if (s.b.ntiles == 0) return TTM_OK;
    const unsigned blocks = s.b.ntiles;
    if (!search_done) {
        const size_t smem = (size_t)kChunk * Geo<N>::K4 * sizeof(float) + kChunk * sizeof(int);
        TTM_CUDA_TRY(cudaFuncSetAttribute(search_simt_kernel<N, CT>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        search_simt_kernel<N, CT><<<blocks, kRotThreads, smem, st>>>(s);
        TTM_TRY(after_launch(cnt));
    }
    if (search_only) return TTM_OK;
    polish_kernel<N, CT><<<blocks, kRotThreads, 0, st>>>(p);
    return after_launch(cnt);
}

template <int N>
ttm_status launch_n(const SearchArgs& s, const PolishArgs& p, bool search_done, bool search_only,
                    bool bf16, cudaStream_t st, long long* cnt) {
    return bf16 ? launch_n_t<N, __nv_bfloat16>(s, p, search_done, search_only, st, cnt)
                : launch_n_t<N, float>(s, p, search_done, search_only, st, cnt);
}

}  // namespace rot

template <int N>
ttm_status launch_rotation_n(const rot::SearchArgs& s, const rot::PolishArgs& p, bool search_done,
                             bool search_only, bool bf16, cudaStream_t st, long long* cnt);

// tensor-core grid search for orders 4 and 6 with the default 2048-point grid
// in 128 regions (k_search_tc.cu); returns TTM_ERR_UNSUPPORTED otherwise
bool search_tc_supported(int n_order, int n_grid, int n_cells);
ttm_status launch_search_tc(int n_order, const rot::SearchArgs& s, const uint16_t* grid_fp16,
                            int* status, bool bf16, cudaStream_t st, long long* cnt);

}  // namespace ttm
