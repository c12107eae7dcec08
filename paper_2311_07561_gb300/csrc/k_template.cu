// Tensor template build (Sec. 3.2 of the paper; template normalisation as in
// Algorithm 1 and the formulas for ||P_S t||_S and <t, 1>_S in Sec. 2).
//
//   t~_j = m (t_{R_j} - <t_{R_j}, m>/<1, m>) / sqrt(<t_{R_j}^2, m> - <t_{R_j}, m>^2/<1, m>)
//   T_alpha(u) = sum_j w_j q_j^alpha t~_j(u)
//
// Kernel 1 rotates and normalises a chunk of quadrature nodes, one CTA per
// node (the per-node reductions stay inside the CTA, in FP64).  Kernel 2 folds
// the chunk into the K components: a [K x J] x [J x s^3] product on CUDA cores
// with the coefficients w_j q_j^alpha staged in shared memory.
#include "ttm_f2.cuh"
#include "ttm_internal.h"

namespace ttm {

namespace {

constexpr int kRotThreads = 512;

__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
        if (threadIdx.x == 0) red[0] = r;
    }
    __syncthreads();
    return red[0];
}

// <1, m> by one CTA of kRotThreads threads or more (the order of the sum is part
// of the result; further threads add nothing).  16 loads in flight, then 4, then
// one: an FP64 addition costs its 16 clocks a warp also where a predicate skips it
template <int G>
__device__ __forceinline__ void mask_add(const float* __restrict__ m, int n, int& i, double& acc) {
    for (; i + (G - 1) * kRotThreads < n; i += G * kRotThreads) {
        float v[G];
#pragma unroll
        for (int k = 0; k < G; ++k) v[k] = __ldg(m + i + k * kRotThreads);
#pragma unroll
        for (int k = 0; k < G; ++k)
            if (v[k] != 0.f) acc += (double)v[k];
    }
}

__device__ __forceinline__ double mask_sum(const float* __restrict__ m, int n, double* red) {
    double acc = 0.0;
    int i = threadIdx.x < kRotThreads ? threadIdx.x : n;
    mask_add<16>(m, n, i, acc);
    mask_add<4>(m, n, i, acc);
    mask_add<1>(m, n, i, acc);
    return block_sum(acc, red);
}

__global__ void __launch_bounds__(kRotThreads) mask_sum_kernel(const float* __restrict__ m,
                                                               int n, double* out) {
    __shared__ double red[32];
    const double s = mask_sum(m, n, red);
    if (threadIdx.x == 0) *out = s;
}

// t_R(u) = t(c + R^-1 (u - c)), trilinear, zero outside the s^3 box.  The
// eight taps are read unconditionally from clamped indices, a tap outside
// the box carrying weight zero (the same sum, term by term, as skipping it),
// so that every load of a voxel can be in flight at once.
__device__ __forceinline__ float sample_rotated(const float* __restrict__ t, int s, float c,
                                                const float Rt[9], int ux, int uy, int uz) {
    float vx = ux - c, vy = uy - c, vz = uz - c;
    // R^-1 = R^T: p_i = sum_k R[k][i] v_k
    float px = Rt[0] * vx + Rt[1] * vy + Rt[2] * vz + c;
    float py = Rt[3] * vx + Rt[4] * vy + Rt[5] * vz + c;
    float pz = Rt[6] * vx + Rt[7] * vy + Rt[8] * vz + c;
    float fx0 = floorf(px), fy0 = floorf(py), fz0 = floorf(pz);
    int x0 = (int)fx0, y0 = (int)fy0, z0 = (int)fz0;
    float ax = px - fx0, ay = py - fy0, az = pz - fz0;
    float tap[8], wt[8];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz) {
        const int zz = z0 + dz;
        const bool iz = zz >= 0 && zz < s;
        const int zc = min(max(zz, 0), s - 1);
        const float wz = dz ? az : 1.0f - az;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int yy = y0 + dy;
            const bool iy = yy >= 0 && yy < s;
            const int yc = min(max(yy, 0), s - 1);
            const float wy = dy ? ay : 1.0f - ay;
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                const int xx = x0 + dx;
                const bool ix = xx >= 0 && xx < s;
                const int xc = min(max(xx, 0), s - 1);
                const float wx = dx ? ax : 1.0f - ax;
                const int k = (dz * 2 + dy) * 2 + dx;
                tap[k] = __ldg(t + ((size_t)zc * s + yc) * s + xc);
                wt[k] = (iz && iy && ix) ? wz * wy * wx : 0.0f;
            }
        }
    }
    float acc = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) acc += wt[k] * tap[k];
    return acc;
}

// rotation matrix of the quaternion at q (normalised on use), rows of R stored
// transposed: Rt[3*i + k] = R[k][i]
__device__ __forceinline__ void node_rotation(const float* __restrict__ q, float* Rt) {
    float a = q[0], b = q[1], cc = q[2], d = q[3];
    float inv = rsqrtf(a * a + b * b + cc * cc + d * d);
    a *= inv; b *= inv; cc *= inv; d *= inv;
    float R00 = 1.f - 2.f * (cc * cc + d * d), R01 = 2.f * (b * cc - a * d), R02 = 2.f * (b * d + a * cc);
    float R10 = 2.f * (b * cc + a * d), R11 = 1.f - 2.f * (b * b + d * d), R12 = 2.f * (cc * d - a * b);
    float R20 = 2.f * (b * d - a * cc), R21 = 2.f * (cc * d + a * b), R22 = 1.f - 2.f * (b * b + cc * cc);
    Rt[0] = R00; Rt[1] = R10; Rt[2] = R20;
    Rt[3] = R01; Rt[4] = R11; Rt[5] = R21;
    Rt[6] = R02; Rt[7] = R12; Rt[8] = R22;
}

__global__ void __launch_bounds__(kRotThreads) rotate_normalise_kernel(
    const float* __restrict__ t, const float* __restrict__ m, int s,
    const float* __restrict__ quats, int j0, float* __restrict__ out, double mask_sum,
    int* bad) {
    __shared__ double red[32];
    __shared__ float Rt[9];
    const int j = j0 + blockIdx.x;
    if (threadIdx.x == 0) node_rotation(quats + 4 * j, Rt);
    __syncthreads();
    float R[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) R[i] = Rt[i];
    const int s3 = s * s * s;
    const float c = (float)(s / 2);
    float* o = out + (size_t)blockIdx.x * s3;
    double t1 = 0.0, t2 = 0.0;
#pragma unroll 4
    for (int u = threadIdx.x; u < s3; u += blockDim.x) {
        int ux = u % s, uy = (u / s) % s, uz = u / (s * s);
        float v = sample_rotated(t, s, c, R, ux, uy, uz);
        o[u] = v;
        float mm = m[u];
        t1 += (double)(mm * v);
        t2 += (double)(mm * v) * v;
    }
    double T1 = block_sum(t1, red);
    double T2 = block_sum(t2, red);
    double var = T2 - T1 * T1 / mask_sum;
    if (!(var > 0.0)) {
        if (threadIdx.x == 0) atomicOr(bad, 1);
        var = 1.0;
    }
    const float off = (float)(T1 / mask_sum);
    const float scl = (float)(1.0 / sqrt(var));
    for (int u = threadIdx.x; u < s3; u += blockDim.x) o[u] = m[u] * (o[u] - off) * scl;
}

constexpr int kFoldThreads = 256;
constexpr int kFoldJ = 32;        // quadrature nodes staged per step
constexpr int kFoldA = 40;        // components per pass (registers per thread)

// Components A0 .. A0 + kFoldA - 1 (a compile-time range, so the exponent
// table is indexed by constants and stays out of local memory).
template <int N, int A0>
__global__ void __launch_bounds__(kFoldThreads, 2) fold_kernel(
    const float* __restrict__ quats, const float* __restrict__ weights, float inv_nrot, int j0,
    int nj, const float* __restrict__ rot, int s3, float* __restrict__ comp, int first) {
    constexpr Sym<N> S{};
    constexpr int K = n_comp(N);
    constexpr int na = K - A0 < kFoldA ? K - A0 : kFoldA;
    const int a0 = A0;
    __shared__ __align__(16) float coef[kFoldJ][kFoldA];
    static_assert(kFoldA % 4 == 0, "coefficients are read as float4");
    static_assert(kFoldJ <= kFoldThreads, "one thread per staged node");
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    float acc[kFoldA];
#pragma unroll
    for (int a = 0; a < kFoldA; ++a) acc[a] = 0.0f;
    for (int jb = 0; jb < nj; jb += kFoldJ) {
        __syncthreads();
        if (threadIdx.x < kFoldJ) {
            // thread jj: w_j q_j^alpha of its node for the pass's components
            const int jj = threadIdx.x;
            const bool live = jb + jj < nj;
            const int j = j0 + jb + (live ? jj : 0);
            float q[4] = {quats[4 * j], quats[4 * j + 1], quats[4 * j + 2], quats[4 * j + 3]};
            const float inv = rsqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) q[i] *= inv;
            const float w = weights ? weights[j] : inv_nrot;
#pragma unroll
            for (int a = 0; a < kFoldA; ++a) {
                float p = 0.0f;
                if (live && a < na) {
                    p = w;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int r = 0; r < S.e[(A0 + a) % K][i]; ++r) p *= q[i];
                }
                coef[jj][a] = p;
            }
        }
        __syncthreads();
        if (u < s3) {
            const int jn = min(kFoldJ, nj - jb);
            // the block's kFoldJ samples of this voxel, all loads in flight at
            // once (nodes past jn carry zero coefficients)
            float rr[kFoldJ];
#pragma unroll
            for (int jj = 0; jj < kFoldJ; ++jj)
                rr[jj] = jj < jn ? __ldg(rot + (size_t)(jb + jj) * s3 + u) : 0.f;
#pragma unroll
            for (int jj = 0; jj < kFoldJ; ++jj) {
                const float r = rr[jj];
                // one 16-byte broadcast read per four FMAs
                const float4* c4 = reinterpret_cast<const float4*>(&coef[jj][0]);
#pragma unroll
                for (int a4 = 0; a4 < kFoldA / 4; ++a4) {
                    const float4 c = c4[a4];
                    acc[4 * a4 + 0] = fmaf(c.x, r, acc[4 * a4 + 0]);
                    acc[4 * a4 + 1] = fmaf(c.y, r, acc[4 * a4 + 1]);
                    acc[4 * a4 + 2] = fmaf(c.z, r, acc[4 * a4 + 2]);
                    acc[4 * a4 + 3] = fmaf(c.w, r, acc[4 * a4 + 3]);
                }
            }
        }
    }
    if (u < s3) {
        for (int a = 0; a < na; ++a) {
            float* dst = comp + (size_t)(a0 + a) * s3 + u;
            *dst = first ? acc[a] : *dst + acc[a];
        }
    }
}

// ---- the same over the mask's voxels only ----------------------------------
// A ball fills half of its box, every voxel outside it is multiplied by zero,
// and the eight clamped, bounds-tested taps of a sample cost more than their
// sum.  So the build lists the mask's voxels once, in bricks of 4 x 4 x 2 (a
// warp's samples stay close together in the rotated template), keeps the
// template as cells {t(x, y), t(x+1, y), t(x, y+1), t(x+1, y+1)} with a border of
// zeros (two 16-byte loads a sample), rotates into rows of the listed voxels
// and leaves the normalisation to the fold, which has to load them anyway.
// 64^3, order 6, 20000 rotations: rotation 75.6 ms and fold 46.5 ms over all
// voxels with scalar FMAs; listed 28.9 ms together, the fold 15.5 of them.
struct VoxelList {            // what the prepass leaves in the workspace header
    double mask_sum;
    int bad;                  // a rotated copy has no variance under the mask
    int n;                    // mask voxels
    int odd;                  // template or mask values that are not finite
    int soft;                 // mask values other than 0 and 1
    int summed;               // mask_sum holds the sum of a soft mask
};

__device__ __forceinline__ int brick_voxel(int e, int s) {     // packed x | y << 8 | z << 16, or -1
    const int bx = (s + 3) / 4;
    const int in = e & 31, b = e >> 5;
    const int x = (b % bx) * 4 + (in & 3), y = (b / bx % bx) * 4 + ((in >> 2) & 3),
              z = (b / (bx * bx)) * 2 + (in >> 4);
    return x < s && y < s && z < s ? x | y << 8 | z << 16 : -1;
}
__device__ __forceinline__ int unpack_voxel(int p, int s) {
    return (((p >> 16) & 255) * s + ((p >> 8) & 255)) * s + (p & 255);
}

constexpr int kListThreads = 1024;
// boxes up to this edge: a CTA more sums the mask where it is soft, beside the
// ones that count, so that the host need not wait twice (order 4, 50 nodes: 24^3
// 111 -> 94 us, all voxels 95; 32^3 136 -> 117); a larger mask would take that CTA
// longer than the wait
constexpr int kListSumEdge = 32;

// mask voxels per CTA of brick-ordered positions; the flags of VoxelList
__global__ void __launch_bounds__(kListThreads) list_count_kernel(const float* __restrict__ t,
                                                                  const float* __restrict__ m, int s,
                                                                  int* __restrict__ counts, int blocks,
                                                                  VoxelList* __restrict__ out) {
    if ((int)blockIdx.x == blocks) {
        __shared__ double red[32];
        const int n = s * s * s;
        bool any = false;
#pragma unroll 4
        for (int i = threadIdx.x; i < n; i += kListThreads) {
            const float v = __ldg(m + i);
            any = any || (v != 0.f && v != 1.f);
        }
        if (!__syncthreads_or(any)) return;
        const double sum = mask_sum(m, n, red);
        if (threadIdx.x == 0) {
            out->mask_sum = sum;
            out->summed = 1;
        }
        return;
    }
    const int p = brick_voxel(blockIdx.x * kListThreads + threadIdx.x, s);
    const float mv = p >= 0 ? m[unpack_voxel(p, s)] : 0.f;
    const float tv = p >= 0 ? t[unpack_voxel(p, s)] : 0.f;
    const int c = __syncthreads_count(mv != 0.f);
    const bool odd = __syncthreads_or(!isfinite(mv) || !isfinite(tv));
    const bool soft = __syncthreads_or(mv != 0.f && mv != 1.f);
    if (threadIdx.x == 0) {
        counts[blockIdx.x] = c;
        if (odd) atomicOr(&out->odd, 1);
        if (soft) atomicOr(&out->soft, 1);
    }
}

__global__ void __launch_bounds__(kListThreads) list_write_kernel(const float* __restrict__ m, int s,
                                                                  const int* __restrict__ counts,
                                                                  int* __restrict__ list,
                                                                  VoxelList* __restrict__ out) {
    __shared__ int warp_n[32], base_s;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) base_s = 0;
    __syncthreads();
    int before = 0;
    for (int b = t; b < (int)blockIdx.x; b += kListThreads) before += counts[b];
    for (int o = 16; o > 0; o >>= 1) before += __shfl_down_sync(0xffffffffu, before, o);
    if (lane == 0 && before) atomicAdd(&base_s, before);
    const int p = brick_voxel(blockIdx.x * kListThreads + t, s);
    const bool in = p >= 0 && m[unpack_voxel(p, s)] != 0.f;
    const uint32_t bits = __ballot_sync(0xffffffffu, in);
    if (lane == 0) warp_n[warp] = __popc(bits);
    __syncthreads();
    int at = base_s;
    for (int w = 0; w < warp; ++w) at += warp_n[w];
    if (in) list[at + __popc(bits & ((1u << lane) - 1u))] = p;
    if (blockIdx.x == gridDim.x - 1 && t == kListThreads - 1) out->n = at + __popc(bits);
}

// cell (x, y, z) of the bordered template, x, y = -2 .. s, z = -2 .. s + 1
__global__ void __launch_bounds__(256) cells_kernel(const float* __restrict__ t, int s,
                                                    float4* __restrict__ cells) {
    const int side = s + 3;
    const int e = blockIdx.x * 256 + threadIdx.x;
    if (e >= side * side * (side + 1)) return;
    const int x = e % side - 2, y = e / side % side - 2, z = e / (side * side) - 2;
    auto at = [&](int xx, int yy) {
        return (unsigned)xx < (unsigned)s && (unsigned)yy < (unsigned)s && (unsigned)z < (unsigned)s
            ? t[((size_t)z * s + yy) * s + xx] : 0.f;
    };
    cells[e] = make_float4(at(x, y), at(x + 1, y), at(x, y + 1), at(x + 1, y + 1));
}

// s + e = a + b exactly.  Additions by name, here and for the squares: one that
// the compiler fuses with the product before it sums something else.
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// row length of the rotated samples: rows start on 16 bytes
__host__ __device__ constexpr size_t rot_pitch(int n) { return ((size_t)n + 3) & ~(size_t)3; }

// One CTA per node: raw samples of the listed voxels, and the node's offset
// and scale.  FP64 runs at 1/64 of the FP32 rate here, so four samples (and
// their squares) are summed in FP32, every addition's and product's remainder
// kept; one FP64 addition takes the sum, and the remainders, 2^-24 of the sums,
// add up in FP32 (a rounding of 2^-48).
__global__ void __launch_bounds__(640, 2) rotate_list_kernel(
    const float4* __restrict__ cells, const float* __restrict__ m, int s,
    const float* __restrict__ quats, int j0, const int* __restrict__ list, int n, int soft,
    float* __restrict__ out, float2* __restrict__ norm, double mask_sum, int* bad) {
    __shared__ double red[32];
    __shared__ float Rt[9];
    const int j = j0 + blockIdx.x;
    if (threadIdx.x == 0) node_rotation(quats + 4 * j, Rt);
    __syncthreads();
    float R[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) R[i] = Rt[i];
    const float c = (float)(s / 2);
    const int side = s + 3, plane = side * side;
    const float top = (float)s;
    float* o = out + (size_t)blockIdx.x * rot_pitch(n);
    double t1 = 0.0, t2 = 0.0;
    float e1 = 0.f, e2 = 0.f;
    for (int i0 = threadIdx.x; i0 < n; i0 += 4 * blockDim.x) {
        float a[4], v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * blockDim.x;
            a[k] = v[k] = 0.f;
            if (i < n) {
                const int p = __ldg(list + i);
                const float vx = (p & 255) - c, vy = ((p >> 8) & 255) - c, vz = (p >> 16) - c;
                // R^-1 = R^T: p_i = sum_k R[k][i] v_k
                const float px = R[0] * vx + R[1] * vy + R[2] * vz + c;
                const float py = R[3] * vx + R[4] * vy + R[5] * vz + c;
                const float pz = R[6] * vx + R[7] * vy + R[8] * vz + c;
                const float fx = floorf(px), fy = floorf(py), fz = floorf(pz);
                const float ax = px - fx, ay = py - fy, az = pz - fz;
                // cells beyond the border are zero like the border's
                const int x = (int)fminf(fmaxf(fx, -2.f), top) + 2;
                const int y = (int)fminf(fmaxf(fy, -2.f), top) + 2;
                const int z = (int)fminf(fmaxf(fz, -2.f), top) + 2;
                const float4* q = cells + (z * side + y) * side + x;
                const float4 lo = __ldg(q), hi = __ldg(q + plane);
                const float bx = 1.0f - ax, by = 1.0f - ay, bz = 1.0f - az;
                float acc = 0.0f;
                acc += (bz * by * bx) * lo.x;
                acc += (bz * by * ax) * lo.y;
                acc += (bz * ay * bx) * lo.z;
                acc += (bz * ay * ax) * lo.w;
                acc += (az * by * bx) * hi.x;
                acc += (az * by * ax) * hi.y;
                acc += (az * ay * bx) * hi.z;
                acc += (az * ay * ax) * hi.w;
                o[i] = acc;
                v[k] = acc;
                a[k] = soft ? __fmul_rn(__ldg(m + unpack_voxel(p, s)), acc) : acc;
            }
        }
        float ea, eb, ec, q[4], r = 0.f;
        const float s1 = two_sum(two_sum(a[0], a[1], ea), two_sum(a[2], a[3], eb), ec);
        t1 += (double)s1;
        e1 += (ea + eb) + ec;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[k] = __fmul_rn(a[k], v[k]);
            r += fmaf(a[k], v[k], -q[k]);
        }
        const float s2 = two_sum(two_sum(q[0], q[1], ea), two_sum(q[2], q[3], eb), ec);
        t2 += (double)s2;
        e2 += ((ea + eb) + ec) + r;
    }
    t1 += (double)e1;
    t2 += (double)e2;
    double T1 = block_sum(t1, red);
    double T2 = block_sum(t2, red);
    if (!(T2 > 1e-20 && T2 < 1e30)) {
        // squares near the ends of the FP32 range: every term in FP64
        t1 = t2 = 0.0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const float v = o[i];
            const float a = soft ? __ldg(m + unpack_voxel(__ldg(list + i), s)) * v : v;
            t1 += (double)a;
            t2 += (double)a * v;
        }
        T1 = block_sum(t1, red);
        T2 = block_sum(t2, red);
    }
    if (threadIdx.x == 0) {
        double var = T2 - T1 * T1 / mask_sum;
        if (!(var > 0.0)) {
            atomicOr(bad, 1);
            var = 1.0;
        }
        norm[blockIdx.x] = make_float2((float)(T1 / mask_sum), (float)(1.0 / sqrt(var)));
    }
}

// w_j q_j^alpha of node j, one row of kp values per node (zero from K on)
template <int N>
__global__ void __launch_bounds__(128) coef_kernel(const float* __restrict__ quats,
                                                   const float* __restrict__ weights, float inv_nrot,
                                                   int j0, int nj, int kp, float* __restrict__ coef) {
    constexpr Sym<N> S{};
    constexpr int K = n_comp(N);
    const int jj = blockIdx.x * 128 + threadIdx.x;
    if (jj >= nj) return;
    const int j = j0 + jj;
    float q[4] = {quats[4 * j], quats[4 * j + 1], quats[4 * j + 2], quats[4 * j + 3]};
    const float inv = rsqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] *= inv;
    const float w = weights ? weights[j] : inv_nrot;
    float* row = coef + (size_t)jj * kp;
#pragma unroll
    for (int a = 0; a < K; ++a) {
        float p = w;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int r = 0; r < S.e[a][i]; ++r) p *= q[i];
        row[a] = p;
    }
    for (int a = K; a < kp; ++a) row[a] = 0.f;
}

// T_alpha(u) over the listed voxels, A components (blockIdx.y) and V voxels per
// thread: a coefficient pair read from shared memory (a broadcast) feeds V
// packed FMAs of two components each.  The samples, coefficients and norms of
// the next nodes are copied into shared memory while this step's are folded
// (loading them into registers at the step's start left the FMA pipe idle two
// thirds of the time: 30.5 ms at 64^3, order 6, 20000 rotations).  Bound by the
// shared-memory reads: 16 bytes for every lane take four clocks of the SM even
// when they are one broadcast, so a coefficient quad has to feed four voxels (8
// packed FMAs, four clocks of the FMA pipes).  A component's sum runs over the
// nodes in order, as in fold_kernel.
constexpr int kFold2Threads = 128;

// V = 4: a thread's voxels are neighbours, copied and read as one float4
template <int A, int V> constexpr int fold_ctas() { return V == 4 ? (A > 28 ? 2 : 3) : 6; }

__device__ __forceinline__ void copy_async(void* dst, const void* src, int bytes) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (bytes == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
    else if (bytes == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

template <int A, int V>
__global__ void __launch_bounds__(kFold2Threads, (fold_ctas<A, V>())) fold_list_kernel(
    const float* __restrict__ coef, int kp, int K, int nj, const float* __restrict__ rot,
    const float2* __restrict__ norm, const float* __restrict__ m, int s,
    const int* __restrict__ list, int n, float* __restrict__ comp, int first) {
    static_assert(A % 4 == 0, "coefficients are copied and read four at a time");
    constexpr int J = V == 4 ? 8 : 16;                // nodes per step
    __shared__ __align__(16) float cs[2][J][A];
    __shared__ __align__(16) float raw[2][J][V * kFold2Threads];
    __shared__ __align__(8) float2 ns[2][J];
    const int a0 = blockIdx.y * A;
    const int t = threadIdx.x;
    const int s3 = s * s * s;
    int at[V], vox[V];
    float mv[V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
        const int i = (blockIdx.x * kFold2Threads + t) * V + k;
        at[k] = i < n ? i : -1;
        vox[k] = at[k] >= 0 ? unpack_voxel(__ldg(list + i), s) : 0;
        mv[k] = at[k] >= 0 ? __ldg(m + vox[k]) : 0.f;
    }
    F2 acc[V][A / 2];
#pragma unroll
    for (int k = 0; k < V; ++k)
#pragma unroll
        for (int a = 0; a < A / 2; ++a) acc[k][a] = f2(0.f, 0.f);
    const size_t pitch = rot_pitch(n);
    // nodes jb .. jb + J - 1 (zeros past the last, and for threads past the
    // list; a row's padding is copied, never used)
    auto stage = [&](int jb, int buf) {
#pragma unroll
        for (int jj = 0; jj < J; ++jj) {
            float* d = &raw[buf][jj][V * t];
            if (jb + jj < nj && at[0] >= 0) copy_async(d, rot + (jb + jj) * pitch + at[0], 4 * V);
            else
#pragma unroll
                for (int k = 0; k < V; ++k) d[k] = 0.f;
        }
        for (int e = t; e < J * (A / 4); e += kFold2Threads) {
            const int jj = e / (A / 4), q = e - jj * (A / 4);
            float4* d = reinterpret_cast<float4*>(&cs[buf][jj][0]) + q;
            if (jb + jj < nj) copy_async(d, coef + (size_t)(jb + jj) * kp + a0 + 4 * q, 16);
            else *d = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (t < J) {
            if (jb + t < nj) copy_async(&ns[buf][t], norm + jb + t, 8);
            else ns[buf][t] = make_float2(0.f, 0.f);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    stage(0, 0);
    int buf = 0;
    for (int jb = 0; jb < nj; jb += J, buf ^= 1) {
        if (jb + J < nj) {
            stage(jb + J, buf ^ 1);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
#pragma unroll
        for (int jj = 0; jj < J; ++jj) {
            const float2 nm = ns[buf][jj];
            float rw[V];
            if constexpr (V == 4) {
                const float4 q = *reinterpret_cast<const float4*>(&raw[buf][jj][V * t]);
                rw[0] = q.x; rw[1] = q.y; rw[2] = q.z; rw[3] = q.w;
            } else {
#pragma unroll
                for (int k = 0; k < V; ++k) rw[k] = raw[buf][jj][V * t + k];
            }
            F2 r[V];
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const float x = mv[k] * (rw[k] - nm.x) * nm.y;
                r[k] = f2(x, x);
            }
            const float4* c4 = reinterpret_cast<const float4*>(&cs[buf][jj][0]);
#pragma unroll
            for (int q = 0; q < A / 4; ++q) {
                const float4 c = c4[q];
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    acc[k][2 * q] = f2_fma(f2(c.x, c.y), r[k], acc[k][2 * q]);
                    acc[k][2 * q + 1] = f2_fma(f2(c.z, c.w), r[k], acc[k][2 * q + 1]);
                }
            }
        }
        __syncthreads();                              // the buffer takes the next copies
    }
#pragma unroll
    for (int k = 0; k < V; ++k) {
        if (at[k] < 0) continue;
#pragma unroll
        for (int a = 0; a < A; ++a) {
            if (a0 + a >= K) break;
            float* dst = comp + (size_t)(a0 + a) * s3 + vox[k];
            const float x = f2_get(acc[k][a / 2], a & 1);
            *dst = first ? x : *dst + x;
        }
    }
}

}  // namespace

ttm_status launch_mask_sum(const float* m, int s, double* d_out, cudaStream_t st, long long* cnt) {
    mask_sum_kernel<<<1, kRotThreads, 0, st>>>(m, s * s * s, d_out);
    return after_launch(cnt);
}

ttm_status launch_rotate_normalise(const float* t, const float* m, int s, const float* quats,
                                   int j0, int nj, float* out, double mask_sum, int* d_bad,
                                   cudaStream_t st, long long* cnt) {
    if (nj <= 0) return TTM_OK;
    rotate_normalise_kernel<<<nj, kRotThreads, 0, st>>>(t, m, s, quats, j0, out, mask_sum, d_bad);
    return after_launch(cnt);
}

// one launch per kFoldA components: A0 = 0, kFoldA, ... below K
template <int N, int A0 = 0>
static ttm_status fold_passes(const float* quats, const float* weights, float inv, int j0, int nj,
                              const float* rot, int s3, float* comp, bool first, dim3 grid,
                              cudaStream_t st, long long* cnt) {
    if constexpr (A0 < n_comp(N)) {
        fold_kernel<N, A0><<<grid, kFoldThreads, 0, st>>>(quats, weights, inv, j0, nj, rot, s3, comp,
                                                         first);
        TTM_TRY(after_launch(cnt));
        return fold_passes<N, A0 + kFoldA>(quats, weights, inv, j0, nj, rot, s3, comp, first, grid,
                                          st, cnt);
    } else {
        return TTM_OK;
    }
}

ttm_status launch_fold_components(int n_order, const float* quats, const float* weights,
                                  int n_rot_total, int j0, int nj, const float* rot, int s3,
                                  float* comp, bool first, cudaStream_t st, long long* cnt) {
    const float inv = 1.0f / (float)n_rot_total;
    const dim3 grid((s3 + kFoldThreads - 1) / kFoldThreads);
    switch (n_order) {
        case 2: return fold_passes<2>(quats, weights, inv, j0, nj, rot, s3, comp, first, grid, st, cnt);
        case 4: return fold_passes<4>(quats, weights, inv, j0, nj, rot, s3, comp, first, grid, st, cnt);
        case 6: return fold_passes<6>(quats, weights, inv, j0, nj, rot, s3, comp, first, grid, st, cnt);
        case 8: return fold_passes<8>(quats, weights, inv, j0, nj, rot, s3, comp, first, grid, st, cnt);
        default: return TTM_ERR_UNSUPPORTED;
    }
}

// ---- build over the listed mask voxels --------------------------------------

namespace {
int list_blocks(int s) {
    const int b = (s + 3) / 4, z = (s + 1) / 2;
    return (b * b * z * 32 + kListThreads - 1) / kListThreads;
}
// components per pass of fold_list_kernel, and the coefficient rows' length:
// one pass of 36 at order 4, three of 28 at order 6 (six at order 8) with four
// voxels per thread where that gives every SM two CTAs, else 12 with two, else
// 12 with one
constexpr int kFoldNarrow = 12;
constexpr int fold_wide(int K) { return K <= 36 ? 36 : 28; }
constexpr int fold_row(int K) {
    const int wide = (K + fold_wide(K) - 1) / fold_wide(K) * fold_wide(K);
    const int narrow = (K + kFoldNarrow - 1) / kFoldNarrow * kFoldNarrow;
    return wide > narrow ? wide : narrow;
}

template <int N>
ttm_status fold_list_n(const TemplateBuild& b, const float* quats, const float* weights, int n_rot,
                       int j0, int nj, float* comp, bool first, cudaStream_t st, long long* cnt) {
    constexpr int K = n_comp(N);
    constexpr int A = fold_wide(K);
    const int kp = fold_row(K);
    coef_kernel<N><<<(nj + 127) / 128, 128, 0, st>>>(quats, weights, 1.0f / (float)n_rot, j0, nj, kp,
                                                     b.coef);
    TTM_TRY(after_launch(cnt));
    const int wide = (K + A - 1) / A;
    const int narrow = (K + kFoldNarrow - 1) / kFoldNarrow;
    auto blocks = [&](int v) { return (b.n + v * kFold2Threads - 1) / (v * kFold2Threads); };
    if (K > kFoldNarrow && blocks(4) * wide >= 304) {
        fold_list_kernel<A, 4><<<dim3(blocks(4), wide), kFold2Threads, 0, st>>>(
            b.coef, kp, K, nj, b.rot, b.norm, b.mask, b.s, b.list, b.n, comp, first);
    } else if (blocks(2) * narrow >= 152) {
        fold_list_kernel<kFoldNarrow, 2><<<dim3(blocks(2), narrow), kFold2Threads, 0, st>>>(
            b.coef, kp, K, nj, b.rot, b.norm, b.mask, b.s, b.list, b.n, comp, first);
    } else {
        fold_list_kernel<kFoldNarrow, 1><<<dim3(blocks(1), narrow), kFold2Threads, 0, st>>>(
            b.coef, kp, K, nj, b.rot, b.norm, b.mask, b.s, b.list, b.n, comp, first);
    }
    return after_launch(cnt);
}
}  // namespace

static_assert(sizeof(VoxelList) <= 64, "the prepass results sit in the workspace header");

// The prepass: voxel list and flags into the header at `head` (a binary mask's
// sum is its number of voxels: no mask sum is formed, whose FP64 additions in one
// CTA took 150 us at 64^3); the
// list at the start of `area`, its CTA counts at the end of the area_floats.
ttm_status launch_build_prepass(const float* t, const float* m, int s, void* head, float* area,
                                size_t area_floats, cudaStream_t st, long long* cnt) {
    VoxelList* vl = reinterpret_cast<VoxelList*>(head);
    const int nb = list_blocks(s);
    int* counts = reinterpret_cast<int*>(area + area_floats - nb);
    list_count_kernel<<<nb + (s <= kListSumEdge ? 1 : 0), kListThreads, 0, st>>>(t, m, s, counts, nb, vl);
    TTM_TRY(after_launch(cnt));
    list_write_kernel<<<nb, kListThreads, 0, st>>>(m, s, counts, reinterpret_cast<int*>(area), vl);
    return after_launch(cnt);
}

// Whether the build goes over listed voxels, as far as that can be said before
// they are counted.  The prepass needs the list and its counts side by side in
// the area, the layout its tables.  A small box with few nodes is folded before
// the list is made: its prepass and further launches take 8 to 15 us, and the box
// build's time grows by 0.09, 0.1, 0.22 and 0.4 us a node at orders 2, 4, 6 and 8
// (us of the call, all voxels / listed: order 2, 10^3, 300 nodes 84 / 89, 600 117 /
// 106; order 4, 10^3, 150 80 / 88, 200 94 / 85; order 6, 8^3, 30 77 / 70; order 8,
// 8^3, 10 93 / 103, 30 94 / 76).  From 24^3 on the list costs no more than the mask
// sum that it saves (order 4, 24^3, 10 nodes 92 / 94, 50 95 / 88; 32^3, 10 155 / 142).
bool build_takes_list(int s, int n_order, int n_rot, int nj, size_t area_floats) {
    if (area_floats < (size_t)s * s * s + (size_t)list_blocks(s)) return false;
    const size_t side = (size_t)s + 3;
    if (4 * side * side * (side + 1) + (size_t)nj * (fold_row(n_comp(n_order)) + 2 + 4) > area_floats) return false;
    const int least = n_order == 2 ? 400 : n_order == 4 ? 180 : n_order == 6 ? 40 : 20;
    return s >= 24 || n_rot >= least;
}

// The sum of a finite mask from the prepass, where it has one.
bool build_mask_count(const void* head_host, double* mask_sum) {
    const VoxelList& vl = *reinterpret_cast<const VoxelList*>(head_host);
    if (vl.odd || (vl.soft && !vl.summed)) return false;
    *mask_sum = vl.soft ? vl.mask_sum : (double)vl.n;
    return true;
}

// Splits the area behind the list: cells, norms, coefficients, rotated rows of
// up to nj nodes.  False where they do not fit (a mask that fills its box, a
// handful of nodes) or values are not finite: the build then takes every voxel.
bool build_layout(const void* head_host, const float* m, double mask_sum, int s, int n_order, int nj,
                  float* area, size_t area_floats, TemplateBuild* out) {
    const VoxelList& vl = *reinterpret_cast<const VoxelList*>(head_host);
    if (vl.odd || vl.n < 1) return false;
    const size_t side = (size_t)s + 3;
    auto up = [](size_t v) { return (v + 63) & ~(size_t)63; };
    const size_t list = up((size_t)vl.n), cells = up(4 * side * side * (side + 1)), norm = up(2 * (size_t)nj),
                 coef = up((size_t)nj * fold_row(n_comp(n_order))), rot = (size_t)nj * rot_pitch(vl.n);
    if (list + cells + norm + coef + rot > area_floats) return false;
    out->s = s; out->n = vl.n; out->soft = vl.soft; out->mask = m;
    out->mask_sum = mask_sum;
    out->list = reinterpret_cast<int*>(area);
    out->cells = area + list;
    out->norm = reinterpret_cast<float2*>(area + list + cells);
    out->coef = area + list + cells + norm;
    out->rot = area + list + cells + norm + coef;
    return true;
}

ttm_status launch_build_cells(const TemplateBuild& b, const float* t, cudaStream_t st, long long* cnt) {
    const int side = b.s + 3;
    cells_kernel<<<(side * side * (side + 1) + 255) / 256, 256, 0, st>>>(t, b.s, reinterpret_cast<float4*>(b.cells));
    return after_launch(cnt);
}

// nodes j0 .. j0 + nj - 1 rotated and folded into the components
ttm_status launch_build_nodes(const TemplateBuild& b, int n_order, const float* quats,
                              const float* weights, int n_rot, int j0, int nj, float* comp,
                              int* d_bad, cudaStream_t st, long long* cnt) {
    // small masks: fewer warps to reduce per node; few nodes (the 304 to 608 that
    // a box from 39^3 on leaves room for): two CTAs hold all the threads an SM
    // takes at 48 registers; many nodes: 256.  Builds of order 2, 2400 nodes, ms
    // with 128 / 256 / 640 threads: 20^3 (3071 voxels) 0.332 / 0.348 / 0.380, 24^3
    // (5575) 0.356 / 0.365 / 0.400, 28^3 0.455 / 0.448 / 0.462, 36^3 0.821 / 0.673
    // / 0.723, 40^3 1.15 / 0.845 / 0.812, 48^3 2.56 / 1.60 / 1.16, 64^3 6.34 / 3.73
    // / 2.28, 127^3 (1000 nodes) 50 / 26.6 / 12.6; 300 nodes: 24^3 0.220 / 0.216 /
    // 0.203, 32^3 0.260 / 0.230 / 0.207.  384 threads beat 640 at 42^3 and 44^3
    // (0.873 against 0.987, 1.07 against 1.20), elsewhere from 39^3 on they lose.
    const int threads = b.n < 4096 ? 128 : nj <= 4 * 152 ? 640 : 256;
    rotate_list_kernel<<<nj, threads, 0, st>>>(reinterpret_cast<const float4*>(b.cells), b.mask, b.s,
                                               quats, j0, b.list, b.n, b.soft, b.rot, b.norm,
                                               b.mask_sum, d_bad);
    TTM_TRY(after_launch(cnt));
    switch (n_order) {
        case 2: return fold_list_n<2>(b, quats, weights, n_rot, j0, nj, comp, j0 == 0, st, cnt);
        case 4: return fold_list_n<4>(b, quats, weights, n_rot, j0, nj, comp, j0 == 0, st, cnt);
        case 6: return fold_list_n<6>(b, quats, weights, n_rot, j0, nj, comp, j0 == 0, st, cnt);
        case 8: return fold_list_n<8>(b, quats, weights, n_rot, j0, nj, comp, j0 == 0, st, cnt);
        default: return TTM_ERR_UNSUPPORTED;
    }
}

}  // namespace ttm
