// Two-level line FFTs, two lines at a time in packed arithmetic.
//
// The two-level passes (k_fft2.cuh) issue 65-78 instructions per point, about
// 36 of them FP32 operations, on lines whose FP32 work and HBM traffic would
// each take 40% of their time.  Here a thread transforms two neighbouring
// lines together, one in each half of a register pair (fma/add/sub.rn.f32x2:
// half the FP32 instructions), the samples reach shared memory in 16-byte
// cp.async copies (spectrum rows are padded to whole 32-byte sectors, so no
// copy is split or predicated) and leave in stores of both lines, and the
// twiddles come from shared memory as ready pairs: about 25 instructions per
// point.  The factors, the order of the operations and their roundings are
// those of the scalar passes, so the results are the same bits.
#pragma once

#include "ttm_f2.cuh"

namespace ttm {
namespace fftk {

// a complex sample of two lines: real and imaginary pairs
struct C2 {
    F2 re, im;
};

__device__ __forceinline__ F2 dup2(float x) { return f2(x, x); }
__device__ __forceinline__ C2 c2_add(C2 a, C2 b) { return C2{f2_add(a.re, b.re), f2_add(a.im, b.im)}; }
__device__ __forceinline__ C2 c2_sub(C2 a, C2 b) { return C2{f2_sub(a.re, b.re), f2_sub(a.im, b.im)}; }
// a + SIGN i b and a - SIGN i b
template <int SIGN>
__device__ __forceinline__ C2 c2_addi(C2 a, C2 b) {
    return SIGN < 0 ? C2{f2_add(a.re, b.im), f2_sub(a.im, b.re)} : C2{f2_sub(a.re, b.im), f2_add(a.im, b.re)};
}
template <int SIGN>
__device__ __forceinline__ C2 c2_subi(C2 a, C2 b) { return c2_addi<-SIGN>(a, b); }
// a * (c + i s).  Of the two products of each part one is rounded and the other
// fused into the sum; which one decides the last bit, and the scalar cmul leaves
// it to the compiler.  Inside the transforms that fuses a.x c in the real part
// and a.y c in the imaginary one (read off the scalar passes' responses to
// single samples); where |c| = |s| the two parts share their products and the
// choice is another.
template <bool AYR, bool AYI>
__device__ __forceinline__ C2 c2_mul(C2 a, F2 c, F2 s, F2 ns) {
    return C2{AYR ? f2_fma(a.im, ns, f2_mul(a.re, c)) : f2_fma(a.re, c, f2_mul(a.im, ns)),
              AYI ? f2_fma(a.im, c, f2_mul(a.re, s)) : f2_fma(a.re, s, f2_mul(a.im, c))};
}
__device__ __forceinline__ C2 c2_mulc(C2 a, float c, float s) {      // constants
    const F2 cc = dup2(c), ss = dup2(s), ns = dup2(-s);
    if ((c == s || c == -s) && c > 0.f) return c2_mul<false, false>(a, cc, ss, ns);
    if (c == s && c < 0.f) return c2_mul<true, true>(a, cc, ss, ns);
    return c2_mul<false, true>(a, cc, ss, ns);
}
template <int SIGN>
__device__ __forceinline__ C2 c2_mi(C2 a) {                          // SIGN i a
    const F2 neg = dup2(-1.f);
    return SIGN < 0 ? C2{a.im, f2_mul(a.re, neg)} : C2{f2_mul(a.im, neg), a.re};
}
template <int N, int SIGN>
__device__ __forceinline__ C2 c2_tw(C2 a, int m) {                   // mul_tw
    const int r = ((m % N) + N) % N;
    if (r == 0) return a;
    if (2 * r == N) return C2{f2_mul(a.re, dup2(-1.f)), f2_mul(a.im, dup2(-1.f))};
    if (4 * r == N) return c2_mi<SIGN>(a);
    if (4 * r == 3 * N) return c2_mi<-SIGN>(a);
    const float2 w = tw_const<N, SIGN>(r);
    return c2_mulc(a, w.x, w.y);
}

// dft4 of a, b, c, d; with CI the third input is SIGN i c
template <int SIGN, bool CI>
__device__ __forceinline__ void c2_dft4(C2& a, C2& b, C2& c, C2& d) {
    const C2 s02 = CI ? c2_addi<SIGN>(a, c) : c2_add(a, c), d02 = CI ? c2_subi<SIGN>(a, c) : c2_sub(a, c);
    const C2 s13 = c2_add(b, d), d13 = c2_sub(b, d);
    a = c2_add(s02, s13);
    b = c2_addi<SIGN>(d02, d13);
    c = c2_sub(s02, s13);
    d = c2_subi<SIGN>(d02, d13);
}

template <int N, int SIGN>
__device__ __forceinline__ void c2_dft(C2 (&v)[N]);

template <int R, int SIGN>
__device__ __forceinline__ void c2_dft_small(C2 (&v)[R]) {
    if constexpr (R == 2) {
        const C2 a = v[0], b = v[1];
        v[0] = c2_add(a, b);
        v[1] = c2_sub(a, b);
    } else if constexpr (R == 4) {
        c2_dft4<SIGN, false>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        C2 u[8];
#pragma unroll
        for (int n2 = 0; n2 < 2; ++n2) {
            C2 a = v[n2], b = v[n2 + 2], c = v[n2 + 4], d = v[n2 + 6];
            c2_dft4<SIGN, false>(a, b, c, d);
            u[n2 + 0] = a; u[n2 + 2] = b; u[n2 + 4] = c; u[n2 + 6] = d;
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            const C2 a = u[2 * k1], b = u[2 * k1 + 1];
            if (k1 == 2) {
                v[k1] = c2_addi<SIGN>(a, b);
                v[k1 + 4] = c2_subi<SIGN>(a, b);
            } else {
                const float2 w = w16<SIGN>(2 * k1);
                const C2 t = k1 == 0 ? b : c2_mulc(b, w.x, w.y);
                v[k1] = c2_add(a, t);
                v[k1 + 4] = c2_sub(a, t);
            }
        }
    } else if constexpr (R == 3) {
        const C2 s = c2_add(v[1], v[2]), e = c2_sub(v[1], v[2]);
        const F2 h = dup2(-0.5f), p = dup2(kS3), n = dup2(-kS3);
        const C2 m{f2_fma(h, s.re, v[0].re), f2_fma(h, s.im, v[0].im)};
        v[0] = c2_add(v[0], s);
        const C2 plus{f2_fma(p, e.im, m.re), f2_fma(n, e.re, m.im)};      // m - i kS3 e
        const C2 minus{f2_fma(n, e.im, m.re), f2_fma(p, e.re, m.im)};     // m + i kS3 e
        v[1] = SIGN < 0 ? plus : minus;
        v[2] = SIGN < 0 ? minus : plus;
    } else if constexpr (R == 5) {
        const C2 t1 = c2_add(v[1], v[4]), t2 = c2_add(v[2], v[3]);
        const C2 t3 = c2_sub(v[1], v[4]), t4 = c2_sub(v[2], v[3]);
        const F2 c1 = dup2(kC51), c2 = dup2(kC52), s1 = dup2(kS51), s2 = dup2(kS52), n1 = dup2(-kS51);
        const C2 a1{f2_fma(c2, t2.re, f2_fma(c1, t1.re, v[0].re)), f2_fma(c2, t2.im, f2_fma(c1, t1.im, v[0].im))};
        const C2 a2{f2_fma(c1, t2.re, f2_fma(c2, t1.re, v[0].re)), f2_fma(c1, t2.im, f2_fma(c2, t1.im, v[0].im))};
        const C2 b1{f2_fma(s1, t3.re, f2_mul(s2, t4.re)), f2_fma(s1, t3.im, f2_mul(s2, t4.im))};
        const C2 b2{f2_fma(s2, t3.re, f2_mul(n1, t4.re)), f2_fma(s2, t3.im, f2_mul(n1, t4.im))};
        v[0] = c2_add(v[0], c2_add(t1, t2));
        v[1] = c2_addi<SIGN>(a1, b1);
        v[4] = c2_subi<SIGN>(a1, b1);
        v[2] = c2_addi<SIGN>(a2, b2);
        v[3] = c2_subi<SIGN>(a2, b2);
    } else {
        static_assert(R == 16, "radix 2, 3, 4, 5, 8 or 16");
        C2 u[16];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            C2 a = v[n2], b = v[n2 + 4], c = v[n2 + 8], d = v[n2 + 12];
            c2_dft4<SIGN, false>(a, b, c, d);
            u[4 * 0 + n2] = a; u[4 * 1 + n2] = b; u[4 * 2 + n2] = c; u[4 * 3 + n2] = d;
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            C2 a = u[4 * k1], b = u[4 * k1 + 1], c = u[4 * k1 + 2], d = u[4 * k1 + 3];
            if (k1 > 0) {
                const float2 wb = w16<SIGN>(k1), wc = w16<SIGN>(2 * k1), wd = w16<SIGN>(3 * k1);
                b = c2_mulc(b, wb.x, wb.y);
                if (k1 != 2) c = c2_mulc(c, wc.x, wc.y);
                d = c2_mulc(d, wd.x, wd.y);
            }
            if (k1 == 2) c2_dft4<SIGN, true>(a, b, c, d);          // W16^4 = -i
            else c2_dft4<SIGN, false>(a, b, c, d);
            v[k1] = a; v[k1 + 4] = b; v[k1 + 8] = c; v[k1 + 12] = d;
        }
    }
}

template <int N, int P, int SIGN>
__device__ __forceinline__ void c2_dft_split(C2 (&v)[N]) {
    constexpr int Q = N / P;
    C2 t[N];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        C2 a[P];
#pragma unroll
        for (int p = 0; p < P; ++p) a[p] = v[Q * p + q];
        c2_dft<P, SIGN>(a);
#pragma unroll
        for (int k1 = 0; k1 < P; ++k1) t[k1 * Q + q] = c2_tw<N, SIGN>(a[k1], q * k1);
    }
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) {
        C2 b[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) b[q] = t[k1 * Q + q];
        c2_dft<Q, SIGN>(b);
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) v[k1 + P * k2] = b[k2];
    }
}

template <int N, int SIGN>
__device__ __forceinline__ void c2_dft(C2 (&v)[N]) {
    if constexpr (N == 1) {
        return;
    } else if constexpr (base_radix(N)) {
        c2_dft_small<N, SIGN>(v);
    } else {
        c2_dft_split<N, split_p(N), SIGN>(v);
    }
}

// ---- samples in shared and global memory ------------------------------------
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
// two neighbouring complex samples (8-byte aligned bf16 pairs, 16-byte float2)
__device__ __forceinline__ C2 c2_load(const float2* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    return C2{f2(q.x, q.z), f2(q.y, q.w)};
}
__device__ __forceinline__ C2 c2_load(const __nv_bfloat162* p) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    return C2{f2(bf_lo(q.x), bf_lo(q.y)), f2(bf_hi(q.x), bf_hi(q.y))};
}
__device__ __forceinline__ void c2_store(float2* p, C2 v) {
    *reinterpret_cast<float4*>(p) =
        make_float4(f2_get(v.re, 0), f2_get(v.im, 0), f2_get(v.re, 1), f2_get(v.im, 1));
}
__device__ __forceinline__ void c2_store(__nv_bfloat162* p, C2 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(f2_get(v.re, 0), f2_get(v.im, 0));
    const __nv_bfloat162 b = __floats2bfloat162_rn(f2_get(v.re, 1), f2_get(v.im, 1));
    uint2 q;
    memcpy(&q.x, &a, 4);
    memcpy(&q.y, &b, 4);
    *reinterpret_cast<uint2*>(p) = q;
}

// every copy of this thread, committed or not
__device__ __forceinline__ void cp_async_wait_every() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

// W_L^m as pairs: cos, SIGN-adjusted sin of table entry m
template <int SIGN>
__device__ __forceinline__ void fill_tw(float4* dst, const float2* __restrict__ tw, int n, int t, int nt) {
    for (int m = t; m < n; m += nt) {
        float2 w = __ldg(tw + m);
        if (SIGN > 0) w.y = -w.y;
        dst[m] = make_float4(w.x, w.x, w.y, w.y);
    }
}
template <int SIGN>
__device__ __forceinline__ C2 c2_mul_tab(C2 a, const float4* w) {
    const float4 q = *w;
    const F2 c = f2(q.x, q.y), s = f2(q.z, q.w);
    // -(a.y s) = (a.y s) (-1); the table's values fuse a.x s forward, and a.y c
    // inverse, where the sine is negated first
    return C2{f2_fma(a.re, c, f2_mul(f2_mul(a.im, s), dup2(-1.f))),
              SIGN > 0 ? f2_fma(a.im, c, f2_mul(a.re, s)) : f2_fma(a.re, s, f2_mul(a.im, c))};
}

// Split of the packed passes: the two-level one, except at 128, whose scalar pass
// takes the factor 16 first
template <int L> struct PackSplit { static constexpr int L1 = TwoLevel<L>::L1, L2 = TwoLevel<L>::L2; };
template <> struct PackSplit<128> { static constexpr int L1 = 8, L2 = 16; };

// ---- column pass -------------------------------------------------------------
// Tiles of 2 NP neighbouring columns (NP pairs) of one plane; a thread is one
// (sample, pair) of a step.  A tile's copies start when every thread has the
// samples of the staging buffer in registers, one or two tiles ahead.
template <int L1, int L2, int NP> constexpr size_t c2_exchange() { return (size_t)L2 * (L1 + 1) * NP * 16; }
template <int L1, int L2, int NP, typename PS> constexpr size_t colsp_smem(int stages) {
    return (size_t)L1 * L2 * (stages * 2 * NP * sizeof(PS) + 16) + c2_exchange<L1, L2, NP>();
}
// registers a thread needs: the larger of the two transforms' pairs
template <int L1, int L2> constexpr int c2_regs() {
    constexpr int big = L1 > L2 ? L1 : L2;
    return big <= 16 ? 160 : big <= 20 ? 208 : 255;
}
// CTAs per SM that registers and shared memory leave
template <int L1, int L2, int NP, typename PS> constexpr int colsp_fit(int stages) {
    constexpr int by_regs = 65536 / (L1 * NP * ((c2_regs<L1, L2>() + 7) / 8 * 8));
    const int by_smem = (int)((size_t)227 * 1024 / (colsp_smem<L1, L2, NP, PS>(stages) + 1024));
    return by_regs < by_smem ? by_regs : by_smem;
}
// staging buffers: two where one or two CTAs fit and the second costs none
// (512 FP32: 238 -> 216 us; with three CTAs and more it measured slower)
template <int L1, int L2, int NP, typename PS> constexpr int colsp_stages() {
    return colsp_fit<L1, L2, NP, PS>(1) <= 2 && colsp_fit<L1, L2, NP, PS>(2) >= colsp_fit<L1, L2, NP, PS>(1)
        ? 2 : 1;
}
template <int L1, int L2, int NP, typename PS> constexpr int colsp_ctas() {
    return colsp_fit<L1, L2, NP, PS>(colsp_stages<L1, L2, NP, PS>());
}

// first step: samples x[n1 + L1 n2] of one pair of lines -> exchange
template <int L1, int L2, int SIGN, int NP>
__device__ __forceinline__ void c2_step_a(C2 (&v)[L2], float4* zx, const float4* tws, int n1, int pair) {
    c2_dft<L2, SIGN>(v);
#pragma unroll
    for (int k2 = 0; k2 < L2; ++k2) {
        if (k2 > 0) v[k2] = c2_mul_tab<SIGN>(v[k2], tws + n1 * k2);
        zx[(k2 * (L1 + 1) + n1) * NP + pair] =
            make_float4(f2_get(v[k2].re, 0), f2_get(v[k2].re, 1), f2_get(v[k2].im, 0), f2_get(v[k2].im, 1));
    }
}
template <int L1, int SIGN, int NP>
__device__ __forceinline__ void c2_step_b(C2 (&u)[L1], const float4* zx, int k2, int pair) {
#pragma unroll
    for (int m = 0; m < L1; ++m) {
        const float4 q = zx[(k2 * (L1 + 1) + m) * NP + pair];
        u[m] = C2{f2(q.x, q.y), f2(q.z, q.w)};
    }
    c2_dft<L1, SIGN>(u);
}

template <int L1, int L2, int SIGN, int NP, typename PS>
__global__ void __launch_bounds__(L1 * NP, (colsp_ctas<L1, L2, NP, PS>())) colsp_t(
    PS* __restrict__ data, int B, const float2* __restrict__ tw, ColsMap mp, int ntb, uint32_t ntiles,
    ColsIn ci) {
    constexpr int L = L1 * L2;
    constexpr int T = L1 * NP, TB = 2 * NP;
    constexpr int kSeg = TB * (int)sizeof(PS) / 16;          // 16-byte copies per line sample
    constexpr int kSt = colsp_stages<L1, L2, NP, PS>();
    extern __shared__ __align__(16) unsigned char smp[];
    float4* tws = reinterpret_cast<float4*>(smp);
    float4* zx = tws + L;
    PS* st = reinterpret_cast<PS*>(smp + (size_t)L * 16 + c2_exchange<L1, L2, NP>());
    const int t = threadIdx.x;
    const int n1 = t / NP, pair = t % NP;
    auto plane_of = [&](uint32_t tile, int& b0) {
        const uint32_t plane = tile / (uint32_t)ntb;
        b0 = (int)(tile - plane * (uint32_t)ntb) * TB;
        return cols_plane_base(mp, (size_t)mp.p0 + plane, L, B);
    };
    auto copy = [&](uint32_t tile, int buf) {
        int b0;
        const PS* src = data + plane_of(tile, b0) + b0;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(st + (size_t)buf * L * TB);
        for (int e = t; e < ci.len * kSeg; e += T) {
            const int q = e / kSeg, seg = e % kSeg;
            int l = q - ci.c;
            if (l < 0) l += L;
            cp_async16(dst + (uint32_t)(l * TB * (int)sizeof(PS) + seg * 16),
                       reinterpret_cast<const char*>(src + (size_t)l * B) + seg * 16);
        }
    };
    uint32_t tile = blockIdx.x;
    if (tile >= ntiles) return;
    if (ci.len < L) {
        uint4* z = reinterpret_cast<uint4*>(st);
        for (int e = t; e < kSt * L * kSeg; e += T) z[e] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    // kSt tiles ahead, one copy group each (an empty one past the end)
#pragma unroll
    for (int q = 0; q < kSt; ++q) {
        if (tile + q * gridDim.x < ntiles) copy(tile + q * gridDim.x, q);
        cp_async_commit();
    }
    fill_tw<SIGN>(tws, tw, L, t, T);
    const F2 sc = dup2(ci.scale);
    for (int buf = 0; tile < ntiles; tile += gridDim.x, buf = kSt == 2 ? buf ^ 1 : 0) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kSt - 1) : "memory");
        __syncthreads();                  // samples (and twiddles) in place, exchange free
        {
            const PS* in = st + (size_t)buf * L * TB;
            C2 v[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) v[n2] = c2_load(in + (n1 + L1 * n2) * TB + 2 * pair);
            c2_step_a<L1, L2, SIGN, NP>(v, zx, tws, n1, pair);
        }
        __syncthreads();
        int b0;
        PS* base = data + plane_of(tile, b0) + b0;
        if (tile + kSt * gridDim.x < ntiles) copy(tile + kSt * gridDim.x, buf);
        cp_async_commit();
#pragma unroll 1
        for (int it = t; it < L2 * NP; it += T) {
            const int k2 = it / NP, pb = it % NP;
            C2 u[L1];
            c2_step_b<L1, SIGN, NP>(u, zx, k2, pb);
            PS* o = base + (size_t)k2 * B + 2 * pb;
            const size_t step = (size_t)L2 * B;
#pragma unroll
            for (int k1 = 0; k1 < L1; ++k1) {
                const int l = k2 + L2 * k1;
                if (l >= mp.lo && l <= mp.hi) {
                    if (ci.scale != 1.f) u[k1] = C2{f2_mul(u[k1].re, sc), f2_mul(u[k1].im, sc)};
                    c2_store(o, u[k1]);
                }
                o += step;
            }
        }
    }
}

// ---- z lines of F(f) conj(T_k), inverse ---------------------------------------
// Pairs per tile and component buffers per team, by length and sample type
// (measured, 35 components unless said; us scalar pass -> packed).  64-byte row
// segments count for more than teams: bf16 samples take 8 pairs (240: 4 pairs
// 6670, 8 pairs 3566, scalar 4571) except where that leaves one team of the
// four (384: 2605, 2114, 2417) or none (512).  A second component buffer pays
// where it costs few teams.
template <int L, typename TS> struct MulPlan {
    static constexpr bool bf = sizeof(TS) == 4;
    static constexpr int NP = bf ? (L == 384 || L == 512 ? 4 : 8) : (L == 128 ? 8 : 4);
    static constexpr int MS = bf ? (L <= 192 || L == 512 ? 2 : 1)
                                 : (L == 128 || L == 288 || L == 320 || L == 480 ? 1 : 2);
    static constexpr bool on = bf ? L <= 512 : L <= 480;
};
// BOX: the template lines come as they are before their own z transform (a
// rotated template's box: len planes, the rest zero).  The team transforms a
// line forward, multiplies, and goes on, the products where the samples were:
// the template spectra are neither written nor read (128 points, boxes of 24,
// 500 templates: 2152 us of z pass and 2622 of multiply -> 3276).
// Persistent CTAs over column tiles; the teams of a CTA (L1 NP threads with
// a named barrier each) share the tile's image samples in shared memory (the
// next tile's arrive meanwhile) and take the components in turn.
template <int L1, int L2, int NP, int MS, typename TS> constexpr size_t mulp_team() {
    return (size_t)L1 * L2 * 2 * NP * sizeof(TS) * MS + c2_exchange<L1, L2, NP>();
}
template <int L1, int L2, int NP, bool BOX> constexpr size_t mulp_shared() {
    // two image tiles, twiddles
    return (size_t)L1 * L2 * (2 * 2 * NP * sizeof(float2) + (BOX ? 32 : 16));
}
template <int L1, int L2, int NP, int MS, typename TS, bool BOX = false> constexpr int mulp_teams() {
    constexpr size_t room = (size_t)226 * 1024;
    constexpr int by_smem = mulp_shared<L1, L2, NP, BOX>() < room
        ? (int)((room - mulp_shared<L1, L2, NP, BOX>()) / mulp_team<L1, L2, NP, MS, TS>()) : 0;
    constexpr int by_regs = 65536 / (L1 * NP * ((c2_regs<L1, L2>() + 7) / 8 * 8));
    constexpr int n = by_smem < by_regs ? by_smem : by_regs;
    return n > 8 ? 8 : n;
}
template <int L1, int L2, int NP, int MS, typename TS, bool BOX = false> constexpr size_t mulp_smem() {
    return mulp_shared<L1, L2, NP, BOX>() +
           mulp_teams<L1, L2, NP, MS, TS, BOX>() * mulp_team<L1, L2, NP, MS, TS>();
}

template <int L1, int L2, int NP, int MS, typename TS, typename PS, bool BOX>
__global__ void __launch_bounds__(L1 * NP * mulp_teams<L1, L2, NP, MS, TS, BOX>(), 1) mulp_t(
    const float2* __restrict__ spec, const TS* __restrict__ tspec, PS* __restrict__ out, int B, int K,
    const float2* __restrict__ tw, int lo, int hi, uint32_t ntiles, ColsIn ci) {
    constexpr int L = L1 * L2;
    constexpr int T = L1 * NP, TB = 2 * NP;
    constexpr int kTeams = mulp_teams<L1, L2, NP, MS, TS, BOX>();
    constexpr int kSegF = TB * (int)sizeof(float2) / 16, kSegT = TB * (int)sizeof(TS) / 16;
    extern __shared__ __align__(16) unsigned char smp[];
    float4* tws = reinterpret_cast<float4*>(smp);
    const float4* twf = tws + L;                                            // BOX: forward
    float2* img = reinterpret_cast<float2*>(smp + (size_t)L * (BOX ? 32 : 16));   // two tiles
    const int team = threadIdx.x / T, t = threadIdx.x % T;
    unsigned char* mine = smp + mulp_shared<L1, L2, NP, BOX>() + team * mulp_team<L1, L2, NP, MS, TS>();
    float4* zx = reinterpret_cast<float4*>(mine);
    TS* st = reinterpret_cast<TS*>(mine + c2_exchange<L1, L2, NP>());
    const int n1 = t / NP, pair = t % NP;
    const size_t plane = (size_t)L * B;
    auto sync_team = [&] { asm volatile("bar.sync %0, %1;\n" ::"r"(1 + team), "n"(T) : "memory"); };
    auto copy_image = [&](uint32_t tile, int buf) {
        const float2* src = spec + (size_t)tile * TB;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(img + (size_t)buf * L * TB);
        for (int e = threadIdx.x; e < L * kSegF; e += T * kTeams) {
            const int l = e / kSegF, seg = e % kSegF;
            cp_async16(dst + (uint32_t)(e * 16), reinterpret_cast<const char*>(src + (size_t)l * B) + seg * 16);
        }
    };
    // item i of the team: component team + i kTeams of the tile, tile after tile
    const int per = team < K ? (K - team + kTeams - 1) / kTeams : 0;
    auto copy_comp = [&](uint32_t tile, int k, int buf) {
        const TS* src = tspec + (size_t)k * plane + (size_t)tile * TB;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(st + (size_t)buf * L * TB);
        for (int e = t; e < (BOX ? ci.len : L) * kSegT; e += T) {
            const int seg = e % kSegT;
            int l = e / kSegT - (BOX ? ci.c : 0);
            if (l < 0) l += L;
            cp_async16(dst + (uint32_t)((l * kSegT + seg) * 16), reinterpret_cast<const char*>(src + (size_t)l * B) + seg * 16);
        }
    };
    uint32_t tile = blockIdx.x;
    if (tile >= ntiles) return;
    // the next item to copy, MS ahead of the one at work; one copy
    // group per item (an empty one past the end).  The image of the tile after
    // next joins the group that follows its call.
    uint32_t ct = tile;
    int ck = team, cbuf = 0;
    auto copy_next = [&] {
        if (per > 0 && ct < ntiles) {
            copy_comp(ct, ck, cbuf);
            ck += kTeams;
            if (ck >= K) { ck = team; ct += gridDim.x; }
        }
        cp_async_commit();
        cbuf = cbuf + 1 == MS ? 0 : cbuf + 1;
    };
    copy_image(tile, 0);
#pragma unroll
    for (int q = 0; q < MS; ++q) copy_next();
    fill_tw<+1>(tws, tw, L, threadIdx.x, T * kTeams);
    if constexpr (BOX) fill_tw<-1>(tws + L, tw, L, threadIdx.x, T * kTeams);
    int buf = 0, cur = 0;
    for (; tile < ntiles; tile += gridDim.x, buf ^= 1) {
        const bool more = tile + gridDim.x < ntiles;
        if (tile == blockIdx.x) asm volatile("cp.async.wait_group %0;\n" ::"n"(MS - 1) : "memory");
        else cp_async_wait_every();
        __syncthreads();                 // the tile's image in place, the other buffer free
        if (more) copy_image(tile + gridDim.x, buf ^ 1);
        const float2* im = img + (size_t)buf * L * TB;
        for (int k = team; k < K; k += kTeams) {
            asm volatile("cp.async.wait_group %0;\n" ::"n"(MS - 1) : "memory");
            sync_team();                 // the component in place, the exchange free
            TS* in = st + (size_t)cur * L * TB;
            auto product = [&](int at, C2 q) {            // F(f) conj(q) of two columns
                const float4 f = *reinterpret_cast<const float4*>(im + at);
                const float2 a = cmulc(make_float2(f.x, f.y), make_float2(f2_get(q.re, 0), f2_get(q.im, 0)));
                const float2 b = cmulc(make_float2(f.z, f.w), make_float2(f2_get(q.re, 1), f2_get(q.im, 1)));
                return C2{f2(a.x, b.x), f2(a.y, b.y)};
            };
            if constexpr (BOX) {
                {
                    C2 v[L2];
#pragma unroll
                    for (int n2 = 0; n2 < L2; ++n2) {
                        const int l = n1 + L1 * n2, d = l + ci.c >= L ? l + ci.c - L : l + ci.c;
                        v[n2] = d < ci.len ? c2_load(in + l * TB + 2 * pair) : C2{dup2(0.f), dup2(0.f)};
                    }
                    c2_step_a<L1, L2, -1, NP>(v, zx, twf, n1, pair);
                }
                sync_team();
                const F2 sc = dup2(ci.scale);
#pragma unroll 1
                for (int it = t; it < L2 * NP; it += T) {
                    const int k2 = it / NP, pb = it % NP;
                    C2 u[L1];
                    c2_step_b<L1, -1, NP>(u, zx, k2, pb);
#pragma unroll
                    for (int k1 = 0; k1 < L1; ++k1) {
                        const int at = (k2 + L2 * k1) * TB + 2 * pb;
                        if (ci.scale != 1.f) u[k1] = C2{f2_mul(u[k1].re, sc), f2_mul(u[k1].im, sc)};
                        c2_store(in + at, product(at, u[k1]));
                    }
                }
                sync_team();             // the products in place, the exchange free
            }
            {
                C2 v[L2];
#pragma unroll
                for (int n2 = 0; n2 < L2; ++n2) {
                    const int at = (n1 + L1 * n2) * TB + 2 * pair;
                    if constexpr (BOX) v[n2] = c2_load(in + at);
                    else v[n2] = product(at, c2_load(in + at));
                }
                c2_step_a<L1, L2, +1, NP>(v, zx, tws, n1, pair);
            }
            sync_team();
            copy_next();
            cur = cur + 1 == MS ? 0 : cur + 1;
            PS* base = out + (size_t)k * plane + (size_t)tile * TB;
#pragma unroll 1
            for (int it = t; it < L2 * NP; it += T) {
                const int k2 = it / NP, pb = it % NP;
                C2 u[L1];
                c2_step_b<L1, +1, NP>(u, zx, k2, pb);
                PS* o = base + (size_t)k2 * B + 2 * pb;
                const size_t step = (size_t)L2 * B;
#pragma unroll
                for (int k1 = 0; k1 < L1; ++k1) {
                    const int l = k2 + L2 * k1;
                    if (l >= lo && l <= hi) c2_store(o, u[k1]);
                    o += step;
                }
            }
        }
    }
    cp_async_wait_every();
}

// ---- half-spectrum rows -> real x lines -----------------------------------------
// Pairs of kept rows (neighbours in the order z, y).  The rows of a tile are
// copied whole into shared memory, the next tile's while this one's second
// step runs; a thread of the first step reads the samples of its two rows, and
// their mirrored ones, from there.  HALF: through a complex transform of half
// the length (rows_c2r_half_t), else of the whole length with the Hermitian
// extension.
constexpr int kRowThreads = 128;
// row pairs per tile: the first step's items fill the CTA once or twice, the
// second step's once
template <int L1, int L2> constexpr int rowp_pairs() {
    return L2 <= 8 ? 2 * kRowThreads / L1 : L1 >= 32 ? 2 * kRowThreads / L1 : kRowThreads / L1;
}
template <int L1, int L2, bool HALF> constexpr int rowp_len() { return L1 * L2 * (HALF ? 2 : 1); }
template <int L1, int L2, bool HALF, typename PS> constexpr size_t rowp_smem() {
    constexpr int L = rowp_len<L1, L2, HALF>(), NR = 2 * rowp_pairs<L1, L2>();
    return (size_t)L1 * L2 * 16 * (HALF ? 2 : 1) + (size_t)rowp_pairs<L1, L2>() * L2 * (L1 + 1) * 16 +
           (size_t)NR * spec_pitch(L) * sizeof(PS) + (size_t)2 * NR * 16;
}
template <int L1, int L2, bool HALF, typename PS> constexpr int rowp_ctas() {
    constexpr int by_regs = 65536 / (kRowThreads * ((c2_regs<L1, L2>() + 7) / 8 * 8));
    constexpr int by_smem = (int)((size_t)227 * 1024 / (rowp_smem<L1, L2, HALF, PS>() + 1024));
    return by_regs < by_smem ? by_regs : by_smem;
}

template <int L1, int L2, bool HALF, typename PS, typename RT>
__global__ void __launch_bounds__(kRowThreads, (rowp_ctas<L1, L2, HALF, PS>())) rowsp_t(
    const PS* __restrict__ in, int X, int Y, int Z, FftGeom g, RT* __restrict__ out, int n_batch,
    const float2* __restrict__ tw, FftKeep keep) {
    constexpr int M = L1 * L2;                          // length of the complex transform
    constexpr int L = rowp_len<L1, L2, HALF>();
    constexpr int XP = spec_pitch(L);
    constexpr int NPR = rowp_pairs<L1, L2>(), NR = 2 * NPR;
    constexpr int kSeg = ((L / 2 + 1) * (int)sizeof(PS) + 15) / 16;
    static_assert(XP * sizeof(PS) % 16 == 0, "rows of whole copies");
    struct Row {
        long long src, dst;                             // -1: no row / not written
    };
    extern __shared__ __align__(16) unsigned char smp[];
    float4* twm = reinterpret_cast<float4*>(smp);       // W_M^j (inverse)
    float4* twl = twm + M;                              // HALF: W_L^-k, k < M
    float4* zx = twm + (HALF ? 2 : 1) * M;
    PS* st = reinterpret_cast<PS*>(zx + NPR * L2 * (L1 + 1));
    Row* rows = reinterpret_cast<Row*>(st + NR * XP);   // two tiles in turn
    const int t = threadIdx.x;
    const int ny = keep.y1 - keep.y0 + 1, nz = keep.z1 - keep.z0 + 1;
    const size_t per_item = (size_t)nz * ny;
    const size_t nrows = (size_t)n_batch * per_item;
    const size_t ntiles = (nrows + NR - 1) / NR;
    auto list_rows = [&](size_t tile, Row* r) {
        if (t >= NR) return;
        const size_t q = tile * NR + t;
        Row w{-1, -1};
        if (q < nrows) {
            const size_t item = q / per_item;
            const uint32_t rr = (uint32_t)(q - item * per_item);
            const int z = keep.z0 + (int)(rr / (uint32_t)ny), y = keep.y0 + (int)(rr % (uint32_t)ny);
            w.src = (long long)(((item * g.Zp + z) * (size_t)g.Yp + y) * XP);
            if (y < Y && z < Z) w.dst = (long long)(item * ((size_t)X * Y * Z) + ((size_t)z * Y + y) * X);
        }
        r[t] = w;
    };
    auto copy = [&](const Row* r) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(st);
        for (int e = t; e < NR * kSeg; e += kRowThreads) {
            const int row = e / kSeg, seg = e - row * kSeg;
            const long long src = r[row].src;
            if (src >= 0)
                cp_async16(dst + (uint32_t)(row * XP * (int)sizeof(PS) + seg * 16),
                           reinterpret_cast<const char*>(in + src) + seg * 16);
        }
        cp_async_commit();
    };
    size_t tile = blockIdx.x;
    if (tile >= ntiles) return;
    list_rows(tile, rows);
    __syncthreads();
    copy(rows);
    for (int m = t; m < M; m += kRowThreads) {
        float2 w = __ldg(tw + (HALF ? 2 * m : m));
        twm[m] = make_float4(w.x, w.x, -w.y, -w.y);
        if constexpr (HALF) {
            w = __ldg(tw + m);
            twl[m] = make_float4(w.x, w.x, -w.y, -w.y);
        }
    }
    const int xk0 = keep.x0, xk1 = min(keep.x1, X - 1);
    for (int cur = 0; tile < ntiles; tile += gridDim.x, cur ^= 1) {
        const bool more = tile + gridDim.x < ntiles;
        cp_async_wait_all();
        __syncthreads();                 // the rows in place, the exchange and the other list free
        if (more) list_rows(tile + gridDim.x, rows + (cur ^ 1) * NR);
#pragma unroll 1
        for (int it = t; it < NPR * L1; it += kRowThreads) {
            const int rp = it / L1, n1 = it % L1;
            const PS* pa = st + (2 * rp) * XP;
            const PS* pb = pa + XP;
            auto sample = [&](int k) {
                const float2 a = ldc(pa + k), b = ldc(pb + k);
                return C2{f2(a.x, b.x), f2(a.y, b.y)};
            };
            C2 v[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) {
                const int k = n1 + L1 * n2;
                if constexpr (HALF) {
                    // Z[k] = (a + b) + i (a - b) W_L^-k, b = conj X[M - k]
                    const C2 a = sample(k), c = sample(M - k);
                    const float4 w = twl[k];
                    const C2 e{f2_sub(a.re, c.re), f2_add(a.im, c.im)};
                    const C2 d = c2_mul<false, true>(e, f2(w.x, w.y), f2(w.z, w.w),
                                                     f2_mul(f2(w.z, w.w), dup2(-1.f)));
                    v[n2] = C2{f2_sub(f2_add(a.re, c.re), d.im), f2_add(f2_sub(a.im, c.im), d.re)};
                } else {
                    v[n2] = sample(k <= L / 2 ? k : L - k);
                    if (k > L / 2) v[n2].im = f2_mul(v[n2].im, dup2(-1.f));      // conj X[L - k]
                }
            }
            c2_dft<L2, +1>(v);
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) {
                if (k2 > 0) v[k2] = c2_mul_tab<+1>(v[k2], twm + n1 * k2);
                zx[(rp * L2 + k2) * (L1 + 1) + n1] = make_float4(f2_get(v[k2].re, 0), f2_get(v[k2].re, 1),
                                                                f2_get(v[k2].im, 0), f2_get(v[k2].im, 1));
            }
        }
        __syncthreads();
        if (more) copy(rows + (cur ^ 1) * NR);
#pragma unroll 1
        for (int it = t; it < NPR * L2; it += kRowThreads) {
            const int rp = it / L2, k2 = it % L2;
            C2 u[L1];
#pragma unroll
            for (int m = 0; m < L1; ++m) {
                const float4 q = zx[(rp * L2 + k2) * (L1 + 1) + m];
                u[m] = C2{f2(q.x, q.y), f2(q.z, q.w)};
            }
            c2_dft<L1, +1>(u);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const long long dst = rows[cur * NR + 2 * rp + half].dst;
                if (dst < 0) continue;
                RT* o = out + dst;
                if constexpr (HALF) {
                    const bool pair_ok = (reinterpret_cast<uintptr_t>(o) & (2 * sizeof(RT) - 1)) == 0;
#pragma unroll
                    for (int k1 = 0; k1 < L1; ++k1) {
                        const int x = 2 * (k2 + L2 * k1);   // z[m] = (y[2m], y[2m+1])
                        const float a = f2_get(u[k1].re, half), b = f2_get(u[k1].im, half);
                        if (pair_ok && x >= xk0 && x + 1 <= xk1) {
                            str2(o + x, a, b);
                        } else {
                            if (x >= xk0 && x <= xk1) str(o + x, a);
                            if (x + 1 >= xk0 && x + 1 <= xk1) str(o + x + 1, b);
                        }
                    }
                } else {
#pragma unroll
                    for (int k1 = 0; k1 < L1; ++k1) {
                        const int x = k2 + L2 * k1;
                        if (x >= xk0 && x <= xk1) str(o + x, f2_get(u[k1].re, half));
                    }
                }
            }
        }
    }
}

// ---- real x lines -> half-spectrum rows (rows_r2c_half_t, two rows a thread) ----
// The rows of a tile are copied into shared memory (16, 8 or 4 bytes a copy, as
// their alignment allows), the next tile's while this one goes through its
// second step and the pairing; after the second step the transforms Z go back
// to shared memory, where X[k] finds Z[k] and Z[M - k].
template <int L1, int L2> constexpr bool rowsf_ok() { return rowp_pairs<L1, L2>() * L2 <= kRowThreads; }
template <int L1, int L2> constexpr size_t rowsf_smem() {
    constexpr int M = L1 * L2, NR = 2 * rowp_pairs<L1, L2>();
    return (size_t)M * 16 + (size_t)rowp_pairs<L1, L2>() * L2 * (L1 + 1) * 16 + (size_t)NR * 2 * M * 4 +
           (size_t)2 * NR * 8;
}
template <int L1, int L2> constexpr int rowsf_ctas() {
    constexpr int by_regs = 65536 / (kRowThreads * ((c2_regs<L1, L2>() + 7) / 8 * 8));
    constexpr int by_smem = (int)((size_t)227 * 1024 / (rowsf_smem<L1, L2>() + 1024));
    return by_regs < by_smem ? by_regs : by_smem;
}

template <int L1, int L2>
__global__ void __launch_bounds__(kRowThreads, (rowsf_ctas<L1, L2>())) rowsf_t(
    const float* __restrict__ f, int X, int Y, int Z, FftGeom g, float2* __restrict__ out,
    const float2* __restrict__ tw, int mode, double* __restrict__ moments, int vec) {
    constexpr int M = L1 * L2, L = 2 * M;
    constexpr int XP = spec_pitch(L);
    constexpr int NPR = rowp_pairs<L1, L2>(), NR = 2 * NPR;
    extern __shared__ __align__(16) unsigned char smp[];
    float4* twm = reinterpret_cast<float4*>(smp);                 // W_M^j
    float4* zx = twm + M;
    float* st = reinterpret_cast<float*>(zx + NPR * L2 * (L1 + 1));
    long long* rows = reinterpret_cast<long long*>(st + NR * L);  // inputs of two tiles in turn, -1: zero row
    __shared__ double part[kRowThreads / 32];
    __shared__ float mean_s;
    const int t = threadIdx.x;
    const size_t nrows = (size_t)g.Yp * g.Zp;
    const size_t ntiles = (nrows + NR - 1) / NR;
    auto list_rows = [&](size_t tile, long long* r) {
        if (t >= NR) return;
        const size_t q = tile * NR + t;
        long long src = -1;
        if (q < nrows) {
            const uint32_t y = (uint32_t)(q % (size_t)g.Yp), z = (uint32_t)(q / (size_t)g.Yp);
            if (y < (uint32_t)Y && z < (uint32_t)Z) src = (long long)(((size_t)z * Y + y) * X);
        }
        r[t] = src;
    };
    auto copy = [&](const long long* r) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(st);
        const int per = X / vec;                                  // copies per row
        for (int e = t; e < NR * per; e += kRowThreads) {
            const int row = e / per, c = (e - row * per) * vec;
            const long long src = r[row];
            if (src < 0) continue;
            const uint32_t d = dst + (uint32_t)(row * L + c) * 4;
            if (vec == 4) cp_async16(d, f + src + c);
            else if (vec == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(f + src + c) : "memory");
            else cp_async4(d, f + src + c);
        }
        cp_async_commit();
    };
    size_t tile = blockIdx.x;
    if (tile >= ntiles) return;
    if (t == 0) mean_s = mode ? (float)(moments[0] / ((double)X * Y * Z)) : 0.f;
    list_rows(tile, rows);
    for (int e = t; e < NR * L; e += kRowThreads) st[e] = 0.f;    // samples from X on stay zero
    __syncthreads();
    copy(rows);
    for (int m = t; m < M; m += kRowThreads) {
        const float2 w = __ldg(tw + 2 * m);
        twm[m] = make_float4(w.x, w.x, w.y, w.y);
    }
    const float mean = mean_s;
    float q4 = 0.f;                                               // mode 2: sum of (f - mean)^4
    for (int cur = 0; tile < ntiles; tile += gridDim.x, cur ^= 1) {
        const bool more = tile + gridDim.x < ntiles;
        const long long* mine = rows + cur * NR;
        cp_async_wait_all();
        __syncthreads();                 // the rows in place, the exchange and the other list free
        if (more) list_rows(tile + gridDim.x, rows + (cur ^ 1) * NR);
#pragma unroll 1
        for (int it = t; it < NPR * L1; it += kRowThreads) {
            const int rp = it / L1, n1 = it % L1;
            const bool ina = mine[2 * rp] >= 0, inb = mine[2 * rp + 1] >= 0;
            const float* pa = st + (2 * rp) * L;
            C2 v[L2];
#pragma unroll
            for (int n2 = 0; n2 < L2; ++n2) {
                const int x = 2 * (n1 + L1 * n2);
                float2 a = *reinterpret_cast<const float2*>(pa + x);
                float2 b = *reinterpret_cast<const float2*>(pa + L + x);
                a.x = ina && x < X ? a.x - mean : 0.f;
                a.y = ina && x + 1 < X ? a.y - mean : 0.f;
                b.x = inb && x < X ? b.x - mean : 0.f;
                b.y = inb && x + 1 < X ? b.y - mean : 0.f;
                if (mode == 2) {
                    a.x *= a.x; a.y *= a.y; b.x *= b.x; b.y *= b.y;
                    q4 = fmaf(a.x, a.x, fmaf(a.y, a.y, q4));
                    q4 = fmaf(b.x, b.x, fmaf(b.y, b.y, q4));
                }
                v[n2] = C2{f2(a.x, b.x), f2(a.y, b.y)};
            }
            c2_dft<L2, -1>(v);
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) {
                if (k2 > 0) v[k2] = c2_mul_tab<-1>(v[k2], twm + n1 * k2);
                zx[(rp * L2 + k2) * (L1 + 1) + n1] = make_float4(f2_get(v[k2].re, 0), f2_get(v[k2].re, 1),
                                                                f2_get(v[k2].im, 0), f2_get(v[k2].im, 1));
            }
        }
        __syncthreads();
        if (more) copy(rows + (cur ^ 1) * NR);
        const int rp = t / L2, k2 = t % L2;
        C2 u[L1];
        if (rp < NPR) {
#pragma unroll
            for (int m = 0; m < L1; ++m) {
                const float4 q = zx[(rp * L2 + k2) * (L1 + 1) + m];
                u[m] = C2{f2(q.x, q.y), f2(q.z, q.w)};
            }
            c2_dft<L1, -1>(u);
        }
        __syncthreads();                 // the exchange takes Z
        if (rp < NPR) {
#pragma unroll
            for (int k1 = 0; k1 < L1; ++k1)
                zx[rp * M + k2 + L2 * k1] = make_float4(f2_get(u[k1].re, 0), f2_get(u[k1].re, 1),
                                                        f2_get(u[k1].im, 0), f2_get(u[k1].im, 1));
        }
        __syncthreads();
        for (int e = t; e < NPR * (M + 1); e += kRowThreads) {
            const int p = e / (M + 1), k = e - p * (M + 1);
            const size_t q = tile * NR + 2 * p;
            if (q >= nrows) continue;
            const float4 za = zx[p * M + (k == M ? 0 : k)], zb = zx[p * M + (k == 0 ? 0 : M - k)];
            const C2 a{f2(za.x, za.y), f2(za.z, za.w)}, b{f2(zb.x, zb.y), f2(zb.z, zb.w)};
            const float2 w = __ldg(tw + k);
            const F2 h = dup2(0.5f);
            // b stands for conj Z[M - k]
            const C2 s{f2_mul(h, f2_add(a.re, b.re)), f2_mul(h, f2_sub(a.im, b.im))};
            const C2 d = c2_mul<false, false>(C2{f2_mul(h, f2_sub(a.re, b.re)), f2_mul(h, f2_add(a.im, b.im))},
                                              dup2(w.x), dup2(w.y), dup2(-w.y));
            const F2 re = f2_add(s.re, d.im), im = f2_sub(s.im, d.re);     // s - i d
            out[q * XP + k] = make_float2(f2_get(re, 0), f2_get(im, 0));
            if (q + 1 < nrows) out[(q + 1) * XP + k] = make_float2(f2_get(re, 1), f2_get(im, 1));
        }
    }
    if (mode == 2) {
        double d = q4;
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if ((t & 31) == 0) part[t >> 5] = d;
        __syncthreads();
        if (t == 0) {
            double s4 = 0.0;
            for (int k = 0; k < kRowThreads / 32; ++k) s4 += part[k];
            if (s4 != 0.0) atomicAdd(moments + 2, s4);
        }
    }
}

}  // namespace fftk
}  // namespace ttm
