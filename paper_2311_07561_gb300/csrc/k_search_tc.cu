// Tensor-core grid search of the per-voxel rotation for tensor orders 4 and 6
// (Sec. 3.3-3.4 of the paper: the rotation is the maximiser of
// phi(Q) = C_n(x) . Q^(n) on the unit sphere).
//
// phi at the 2048 grid points of every voxel is one dense contraction,
//   Phi[v, g] = sum_alpha Cn[v, alpha] M[g, alpha],  M[g, alpha] = mu_alpha q_g^alpha,
// with Cn = C / ||C||_F (a positive per-voxel scale changes no ranking).  It runs
// on the 5th-generation tensor cores: tcgen05.mma kind::f16 (FP16 operands,
// FP32 accumulation) with M = 128 voxels, N = 256 grid points and K = KP (the
// K components, a constant column that adds +1 to phi, zero padding to a
// multiple of 16: 48 for order 4, 96 for order 6), D in tensor memory.
//
// One persistent CTA per SM, thirteen warps in three roles; a tile is 128
// consecutive voxels of the interior box (voxel l of the tile = TMEM lane l):
//   warps 0-7   reduce: per 256-point chunk each warp reads its 32 lanes of half
//               of the columns (warps 0-3 the first, 4-7 the second) with
//               tcgen05.ld and keeps, per grid region of 16 consecutive points,
//               the best point, and the best KC regions;
//   warps 8-11  produce: one thread per voxel loads the K correlations, writes
//               the score and the normalised components as one FP16 row of A;
//   warp 12     one thread issues the MMAs of a 256-point chunk into one half
//               of the 512-column accumulator while the other half is reduced.
// The roles meet on mbarriers only, so the next tile's components are loaded,
// normalised and stored, and its first chunk multiplied, while the last chunks
// of the current tile are reduced: A is free as soon as the MMAs of the last
// chunk are done, two chunks of reduction before its next row is needed, so
// one A buffer is enough.  The FP16 grid table (G x KP, K-major core-matrix
// layout without swizzle, stored chunk by chunk of 256 points) is bulk-copied
// into shared memory once per CTA (192 KB; the first tile's MMAs start with
// the first chunk) or, where it does not fit (order 6 with 2048 points),
// streamed through four 48 KB buffers from L2.
//
// What bounds it: the integer ALU of the reduction, 1.5 operations per value
// (one LOP3 to pack the key, half a three-input maximum), 64 lanes a clock:
// 3.5 clocks per 128-lane column measured alone, 4.1 with two regions kept
// and 5.0 with eight (sixteen reducing warps of 80 registers, which is all that
// six warps on a scheduler leave each, were no faster: 512 x 512 x 256 in 28.6
// ms against 28.4); the MMAs take 1.5 (KP = 48) or 3 (KP = 96).  With every
// role in the same warps, one after the other, a tile of 1024 columns at KP =
// 96 took 12000 clocks and one of 2048 columns at KP = 48 took 17300.
//
// The roles meet on mbarriers alone (a named barrier waits without a limit),
// and every wait on one is bounded.  On expiry the whole warp leaves its role's
// loop (the lanes vote: the tensor-memory loads behind a wait take all 32), the
// other roles' waits expire after it, the kernel records TTM_ERR_TIMEOUT, waits
// once more for its MMAs and copies in flight, frees its TMEM and exits.
#include <climits>

#include <cuda_fp16.h>

#include "k_rotation.cuh"

namespace ttm {

namespace {

constexpr int kReduceWarps = 8;      // warps w and w + 4 read the same TMEM lanes
constexpr int kProduceWarps = 4;     // one thread per voxel of a tile
constexpr int kThreads = 32 * (kReduceWarps + kProduceWarps + 1);
constexpr int kChunkN = 256;         // grid points per MMA
constexpr int kGroupN = kChunkN / 2; // columns a reducing warp reads of a chunk

// Shapes for K tensor components, G grid points (1024 or 2048) and KC kept
// regions: padded K, shared-memory sizes, and whether the grid table is
// resident or streamed through a ring of kRing chunk buffers.
template <int K, int G, int KC>
struct TcShape {
    static constexpr int kChunks = G / kChunkN;
    static constexpr int KP = ((K + 1 + 15) / 16) * 16;          // + constant column
    static constexpr int kCore = KP / 8;                         // core-matrix columns along K
    static constexpr uint32_t ABytes = (uint32_t)kCore * 16 * 128;
    static constexpr uint32_t ChunkBytes = (uint32_t)kCore * (kChunkN / 8) * 128;
    static constexpr bool Stream = (uint64_t)ChunkBytes * kChunks > 200u * 1024u;
    static constexpr int kRing = Stream ? 4 : kChunks;
    static constexpr uint32_t BBytes = ChunkBytes * kRing;
    // the second column group's best keys, for two tiles in turn
    static constexpr uint32_t MergeBytes = 2u * KC * 128 * 4;
    static constexpr uint32_t Smem = BBytes + ABytes + MergeBytes;
    static_assert(kChunks % 2 == 0, "a tile starts in TMEM half 0");
    static_assert(Smem <= 226u * 1024u, "shared memory");
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: K-major, no swizzle; lbo = byte distance of
// core matrices adjacent along K, sbo = along M/N
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// kind::f16 instruction descriptor: D FP32, A and B FP16, both K-major, M = 128, N = 256
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kChunkN >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t phase) {
    return mbar_wait_bounded(bar, phase, kMbarWaitPolls);
}
// The same by all lanes of a warp, with one answer for all of them.  The vote on
// a first poll keeps the loop, whose lanes may part, off the usual path (search of
// the 256^3 case: 3.51 ms, 3.57 with a vote after the loop alone, 3.51 without
// votes).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t phase) {
    if (__all_sync(0xffffffffu, mbar_wait_bounded(bar, phase, 1))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, phase));
}

// MMAs of one 256-point chunk whose B block (KP/8 x 32 core matrices, K-block
// major) starts at b_chunk; A is 128 x KP (KP/8 x 16 core matrices)
template <int KP>
__device__ __forceinline__ void issue_chunk(uint32_t tmem_d, uint32_t a_base, uint32_t b_chunk,
                                           uint32_t bar) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
    for (int s = 0; s < KP / 16; ++s) {
        const uint64_t ad = smem_desc(a_base + (uint32_t)(2 * s) * 16 * 128, 16 * 128, 128);
        const uint64_t bd = smem_desc(b_chunk + (uint32_t)(2 * s) * (kChunkN / 8) * 128,
                                      (kChunkN / 8) * 128, 128);
        asm volatile(
            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
            "l"(ad), "l"(bd), "r"(kIdesc), "r"(s) : "memory");
    }
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
        : "memory");
}

// (c ? a : b) bit by bit: one LOP3 whose b operand is an immediate
template <int B>
__device__ __forceinline__ int select_bits(int a, int c) {
    int d;
    asm("lop3.b32 %0, %1, %2, %3, 0xE4;" : "=r"(d) : "r"(a), "n"(B), "r"(c));
    return d;
}

// key[j] = (r[j] & ~2047) | (15 - j % 16) for j = J..M-1 (compile-time j)
template <int J, int M>
__device__ __forceinline__ void pack_keys(int (&key)[M], const uint32_t (&r)[M], int mask) {
    if constexpr (J < M) {
        key[J] = select_bits<15 - (J & 15)>((int)r[J], mask);
        pack_keys<J + 1, M>(key, r, mask);
    }
}

// compare-exchange for a descending order
__device__ __forceinline__ void cx(int& hi, int& lo) {
    const int a = max(hi, lo);
    lo = min(hi, lo);
    hi = a;
}

// top (8, descending) := the 8 largest of top and n (4, descending): the
// element-wise max of top and reversed n is bitonic, then three half-cleaner
// stages sort it
__device__ __forceinline__ void merge4(int (&top)[8], int (&n)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) top[4 + i] = max(top[4 + i], n[3 - i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) cx(top[i], top[i + 4]);
#pragma unroll
    for (int i = 0; i < 8; i += 4) { cx(top[i], top[i + 2]); cx(top[i + 1], top[i + 3]); }
#pragma unroll
    for (int i = 0; i < 8; i += 2) cx(top[i], top[i + 1]);
}

// the same for two lists of 8
__device__ __forceinline__ void merge8(int (&top)[8], const int (&n)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) top[i] = max(top[i], n[7 - i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) cx(top[i], top[i + 4]);
#pragma unroll
    for (int i = 0; i < 8; i += 4) { cx(top[i], top[i + 2]); cx(top[i + 1], top[i + 3]); }
#pragma unroll
    for (int i = 0; i < 8; i += 2) cx(top[i], top[i + 1]);
}

// one thread: arm the barrier for `bytes` and start a bulk copy global -> shared
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// 32 TMEM columns of this warp's 32 lanes into r; the copy completes at
// tmem_wait32, which names r as modified so nothing reads r before it
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
          "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
          "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
          "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
          "=r"(r[30]), "=r"(r[31])
        : "r"(addr)
        : "memory");
}

__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]),
                   "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// 32 columns = 2 regions of 16 -> their best keys n0, n1.  phi + 1 >= 0
// (|phi| <= 1 for unit-norm C), so its float bits order like the values; the
// low 11 bits become the code 2047 - g of the grid index g: first only the
// position in the region (15 - j, one LOP3 per value), the region part (low0 =
// 2047 - grid index of column 0) is added to each region's maximum
__device__ __forceinline__ void region_max32(const uint32_t (&r)[32], int low0, int& n0, int& n1) {
    int key[32];
    pack_keys<0, 32>(key, r, ~2047);
    int nk[2];
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2) {
        // three-input integer maxima, 16 -> 6 -> 2 -> 1
        const int* k16 = key + 16 * q2;
        const int m0 = __vimax3_s32(k16[0], k16[1], k16[2]);
        const int m1 = __vimax3_s32(k16[3], k16[4], k16[5]);
        const int m2 = __vimax3_s32(k16[6], k16[7], k16[8]);
        const int m3 = __vimax3_s32(k16[9], k16[10], k16[11]);
        const int m4 = __vimax3_s32(k16[12], k16[13], k16[14]);
        const int a0 = __vimax3_s32(m0, m1, m2);
        const int a1 = __vimax3_s32(m3, m4, k16[15]);
        nk[q2] = max(a0, a1) + (low0 - 16 * q2 - 15);
    }
    n0 = nk[0];
    n1 = nk[1];
}

// top (KC, descending) := the KC largest of top and the four keys n
__device__ __forceinline__ void keep_best(int (&top)[8], int (&n)[4]) {
    cx(n[0], n[1]); cx(n[2], n[3]); cx(n[0], n[2]); cx(n[1], n[3]); cx(n[1], n[2]);
    merge4(top, n);
}
__device__ __forceinline__ void keep_best(int (&top)[2], int (&n)[4]) {
    cx(n[0], n[1]); cx(n[2], n[3]);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
        // second of two descending pairs: the larger of the lower first and
        // the seconds (the lower pair's own second cannot exceed its first)
        const int lo = min(top[0], n[i]);
        top[0] = max(top[0], n[i]);
        top[1] = __vimax3_s32(lo, top[1], n[i + 1]);
    }
}
__device__ __forceinline__ void merge_best(int (&top)[8], const int (&n)[8]) { merge8(top, n); }
__device__ __forceinline__ void merge_best(int (&top)[2], const int (&n)[2]) {
    const int lo = min(top[0], n[0]);
    top[0] = max(top[0], n[0]);
    top[1] = __vimax3_s32(lo, top[1], n[1]);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

// 104 registers: what the produced row of K = 84 components needs
template <typename CT, int N, int G, int KC>
__global__ void __maxnreg__(104) search_tc_kernel(const __grid_constant__ rot::SearchArgs a,
                                                  const unsigned char* __restrict__ gtab,
                                                  int* status) {
    using Sh = TcShape<n_comp(N), G, KC>;
    constexpr int kChunks = Sh::kChunks;
    constexpr int K = n_comp(N);
    constexpr int KP = Sh::KP;
    constexpr int kRing = Sh::kRing;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t full_s[2];      // MMAs of a chunk done, per TMEM half
    __shared__ __align__(8) uint64_t read_s[2];      // TMEM half read by every reducing warp
    __shared__ __align__(8) uint64_t afull_s, afree_s;   // A written / read by all its MMAs
    __shared__ __align__(8) uint64_t load_s[kRing];  // grid-chunk copies
    __shared__ __align__(8) uint64_t merge_s[kReduceWarps / 2];   // a tile's keys of warp w + 4 stored
    __shared__ uint32_t tmem_base_s;
    const int t = threadIdx.x;
    const int warp = t >> 5, lane = t & 31;
    unsigned char* As = sm + Sh::BBytes;
    int* merge = reinterpret_cast<int*>(sm + Sh::BBytes + Sh::ABytes);   // [2][KC][128]
    const uint32_t full0 = smem_u32(&full_s[0]), read0 = smem_u32(&read_s[0]);
    const uint32_t afull = smem_u32(&afull_s), afree = smem_u32(&afree_s);
    const uint32_t load0 = smem_u32(&load_s[0]), merge0 = smem_u32(&merge_s[0]);
    const uint32_t a_base = smem_u32(As), b_base = smem_u32(sm);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(
                         smem_u32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (t == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(full0 + 8 * b, 1);
            mbar_init(read0 + 8 * b, kReduceWarps);
        }
        mbar_init(afull, kProduceWarps);
        mbar_init(afree, 1);
        for (int b = 0; b < kRing; ++b) mbar_init(load0 + 8 * b, 1);
        for (int b = 0; b < kReduceWarps / 2; ++b) mbar_init(merge0 + 8 * b, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_base_s;
    bool ok = true;

    // tiles of the launch (with a unit list, one problem: the listed units)
    size_t ntiles = a.b.ntiles;
    if (a.list.count) {
        const uint32_t uend = rot::list_end(a.list, a.b.seg[0].u1);
        ntiles = ((uend > a.b.seg[0].u0 ? uend - a.b.seg[0].u0 : 0) + 127) / 128;
    }
    // tiles of this CTA, and its chunks in order: chunk q of the CTA is chunk
    // q % kChunks of tile q / kChunks and goes through TMEM half q & 1
    const uint32_t mine = blockIdx.x < ntiles
        ? (uint32_t)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0u;

    if (warp < kReduceWarps) {
        // ---- reduce ------------------------------------------------------
        const int grp = warp >> 2;
        const int lane_t = (warp & 3) * 32 + lane;
        const uint32_t cols0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)grp * kGroupN;
        int sidx = 0;
        uint32_t ra[32], rb[32];
        for (uint32_t n = 0; n < mine && ok; ++n) {
            // packed keys: the float bits of phi + 1 with the low 11 bits replaced
            // by (2047 - grid index): one integer max gives the best point of a
            // region (ties: lower index) at 2.4e-4 resolution of the normalised
            // phi; top holds the KC best region keys, descending
            int top[KC];
#pragma unroll
            for (int k = 0; k < KC; ++k) top[k] = INT_MIN;
#pragma unroll 1
            for (int c = 0; c < kChunks; ++c) {
                const uint32_t h = c & 1, use = (n * kChunks + c) >> 1;   // use-th chunk of half h
                if (!mbar_wait_warp(full0 + 8 * h, use & 1u)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t cols = cols0 + h * kChunkN;
                const int low0 = 2047 - (c * kChunkN + grp * kGroupN);
                // four loads of 32 columns, the next one in flight while the
                // previous one is reduced
                int nk[4];
                tmem_ld32(cols, ra);
                tmem_wait32(ra);
                tmem_ld32(cols + 32, rb);
                region_max32(ra, low0, nk[0], nk[1]);
                tmem_wait32(rb);
                tmem_ld32(cols + 64, ra);
                region_max32(rb, low0 - 32, nk[2], nk[3]);
                keep_best(top, nk);
                tmem_wait32(ra);
                tmem_ld32(cols + 96, rb);
                region_max32(ra, low0 - 64, nk[0], nk[1]);
                tmem_wait32(rb);
                // this warp has read half h: the chunk after next may take it
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(read0 + 8 * h);
                region_max32(rb, low0 - 96, nk[2], nk[3]);
                keep_best(top, nk);
            }
            if (!ok) break;
            // the second group hands its keys to the first (warps w and w + 4
            // share lanes and an mbarrier).  Two buffers in turn: the second
            // group is at most two chunks ahead of the first, so it comes back
            // to a buffer, and to a phase, only after the first has taken it.
            int* mg = merge + (n & 1) * KC * 128 + lane_t;
            if (grp == 1) {
#pragma unroll
                for (int k = 0; k < KC; ++k) mg[k * 128] = top[k];
                __syncwarp();
                if (lane == 0) mbar_arrive(merge0 + 8 * (warp & 3));
            } else {
                if (!mbar_wait_warp(merge0 + 8 * warp, n & 1u)) { ok = false; break; }
                int other[KC];
#pragma unroll
                for (int k = 0; k < KC; ++k) other[k] = mg[k * 128];
                merge_best(top, other);
                const uint32_t tile = blockIdx.x + n * gridDim.x;
                sidx = rot::seg_of(a.b, tile, sidx);
                const RotSeg& sg = a.b.seg[sidx];
                const size_t i = sg.u0 + (size_t)(tile - sg.tile0) * 128 + lane_t;
                if (i < rot::list_end(a.list, sg.u1)) {
                    int ti[rot::kMaxCand];
#pragma unroll
                    for (int k = 0; k < rot::kMaxCand; ++k)
                        ti[k] = k < KC && top[k < KC ? k : 0] != INT_MIN
                            ? 2047 - (top[k < KC ? k : 0] & 2047) : 0xFFFF;
                    // (a voxel of score 0 has candidates too: the refinement
                    // looks at the score first)
                    rot::store_candidates(sg.cand, i, ti, true);
                }
            }
        }
    } else if (warp < kReduceWarps + kProduceWarps) {
        // ---- produce -----------------------------------------------------
        constexpr Sym<N> S{};
        const int lane_t = t - 32 * kReduceWarps;
        int sidx = 0;
        for (uint32_t n = 0; n < mine; ++n) {
            const uint32_t tile = blockIdx.x + n * gridDim.x;
            sidx = rot::seg_of(a.b, tile, sidx);
            const RotSeg& sg = a.b.seg[sidx];
            const size_t i = sg.u0 + (size_t)(tile - sg.tile0) * 128 + lane_t;
            const bool in = i < rot::list_end(a.list, sg.u1);
            const size_t v = in ? rot::unit_voxel(sg.box, a.list, (uint32_t)i) : 0;
            const float wv = in ? __ldg(sg.w + v) : 0.f;
            const size_t step = sg.nvox;
            const CT* src = reinterpret_cast<const CT*>(sg.corr) + v;
            CT raw[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                raw[k] = in ? __ldg(src) : CT(0.f);
                src += step;
            }
            // C = w Corr and the score, summed in the two halves of
            // rot::score_split as every kernel that writes a score
            float C[K], ss0 = 0.f, ss1 = 0.f;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                C[k] = (float)raw[k] * wv;
                if (k < rot::score_split<N>()) ss0 = fmaf((float)S.mu[k], C[k] * C[k], ss0);
                else ss1 = fmaf((float)S.mu[k], C[k] * C[k], ss1);
            }
            const float score = sqrtf(ss0 + ss1);
            if (in) sg.score[v] = score;
            const float inv = score > 0.f ? 1.f / score : 0.f;
            // the row of A: components, the constant 1 that adds +1 to every
            // phi, zeros
            uint32_t row[KP / 2];
#pragma unroll
            for (int j = 0; j < KP / 2; ++j) {
                const float lo = 2 * j < K ? C[2 * j < K ? 2 * j : 0] * inv : (2 * j == K ? 1.f : 0.f);
                const float hi = 2 * j + 1 < K ? C[2 * j + 1 < K ? 2 * j + 1 : 0] * inv
                                               : (2 * j + 1 == K ? 1.f : 0.f);
                const __half2 hh = __halves2half2(__float2half_rn(lo), __float2half_rn(hi));
                row[j] = *reinterpret_cast<const uint32_t*>(&hh);
            }
            if (n > 0 && !mbar_wait_warp(afree, (n - 1) & 1u)) { ok = false; break; }
#pragma unroll
            for (int kc = 0; kc < Sh::kCore; ++kc)
                *reinterpret_cast<uint4*>(As + ((kc * 16 + (lane_t >> 3)) * 8 + (lane_t & 7)) * 16) =
                    make_uint4(row[4 * kc], row[4 * kc + 1], row[4 * kc + 2], row[4 * kc + 3]);
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(afull);
        }
    } else {
      if (lane == 0 && mine > 0) {
        // ---- issue -------------------------------------------------------
        uint32_t loading = 0u;                    // copies issued and not yet waited for
        uint32_t nload = 0u;                      // chunks copied so far, in order
        const uint32_t nq = mine * kChunks;
        auto load = [&](uint32_t q) {             // chunk q of the CTA into its buffer
            const uint32_t b = q % kRing;
            bulk_load(b_base + b * Sh::ChunkBytes, gtab + (size_t)(q % kChunks) * Sh::ChunkBytes,
                      Sh::ChunkBytes, load0 + 8 * b);
            loading |= 1u << b;
            nload = q + 1;
        };
        for (uint32_t q = 0; q < (uint32_t)kRing && q < nq; ++q) load(q);
        uint32_t pending = 0u;                    // MMAs committed to full_s[h], not seen done
        uint32_t q = 0;
        for (uint32_t n = 0; n < mine && ok; ++n) {
            if (!mbar_wait(afull, n & 1u)) { ok = false; break; }
            for (int c = 0; c < kChunks; ++c, ++q) {
                const uint32_t h = q & 1u, use = q >> 1;
                if (use > 0 && !mbar_wait(read0 + 8 * h, (use - 1) & 1u)) { ok = false; break; }
                pending &= ~(1u << h);            // read, so its MMAs were done
                const uint32_t b = q % kRing;
                if (Sh::Stream || n == 0) {
                    if (!mbar_wait(load0 + 8 * b, (q / kRing) & 1u)) { ok = false; break; }
                    loading &= ~(1u << b);
                }
                issue_chunk<KP>(tmem + h * kChunkN, a_base, b_base + b * Sh::ChunkBytes, full0 + 8 * h);
                if (c == kChunks - 1)
                    asm volatile(
                        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                        ::"r"(afree) : "memory");
                pending |= 1u << h;
                // the buffer of the previous chunk takes the next copy once its
                // MMAs are done (this chunk's are queued behind them)
                if (Sh::Stream && q > 0 && q - 1 + kRing < nq) {
                    if (!mbar_wait(full0 + 8 * (h ^ 1u), ((q - 1) >> 1) & 1u)) { ok = false; ++q; break; }
                    load(q - 1 + kRing);
                }
            }
        }
        // MMAs and copies in flight finish before the memory is released: also
        // when every chunk was issued, as a reducing warp that gave up on the
        // last of them does not wait for it
        for (uint32_t hh = 0; hh < 2; ++hh)
            if ((pending >> hh) & 1u) {
                const uint32_t last = q > 0 && ((q - 1) & 1u) == hh ? q - 1 : q - 2;
                mbar_wait(full0 + 8 * hh, (last >> 1) & 1u);
            }
        for (uint32_t b = 0; b < (uint32_t)kRing; ++b)
            if ((loading >> b) & 1u) {
                uint32_t lq = b;                  // the buffer's latest copy
                while (lq + kRing < nload) lq += kRing;
                mbar_wait(load0 + 8 * b, (lq / kRing) & 1u);
            }
      }
      __syncwarp();
    }
    if (!__syncthreads_and(ok) && t == 0) atomicExch(status, TTM_ERR_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem) : "memory");
}

}  // namespace

template <typename CT, int N, int G, int KC>
static ttm_status launch_tc_t(const rot::SearchArgs& s, const uint16_t* grid_fp16, int* status,
                              cudaStream_t st, long long* cnt) {
    constexpr uint32_t smem = TcShape<n_comp(N), G, KC>::Smem;
    TTM_CUDA_TRY(cudaFuncSetAttribute(search_tc_kernel<CT, N, G, KC>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int dev = 0, sms = 0;
    TTM_CUDA_TRY(cudaGetDevice(&dev));
    TTM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t ntiles = s.b.ntiles;
    if (ntiles == 0) return TTM_OK;
    const unsigned grid = (unsigned)(ntiles < (size_t)sms ? ntiles : (size_t)sms);
    search_tc_kernel<CT, N, G, KC><<<grid, kThreads, smem, st>>>(
        s, reinterpret_cast<const unsigned char*>(grid_fp16), status);
    return after_launch(cnt);
}

// the refinement reads the first n_cand candidates: with one or two (the
// default of order 6) the search keeps two regions instead of eight, which
// takes 0.8 of the 5.0 clocks per column off its reduction
template <typename CT, int N, int G>
static ttm_status launch_tc_k(const rot::SearchArgs& s, const uint16_t* grid_fp16, int* status,
                              cudaStream_t st, long long* cnt) {
    return s.n_cand <= 2 ? launch_tc_t<CT, N, G, 2>(s, grid_fp16, status, st, cnt)
                         : launch_tc_t<CT, N, G, 8>(s, grid_fp16, status, st, cnt);
}

// grids of 2048 points in 128 regions, or 1024 points in 64 regions, of 16
bool search_tc_supported(int n_order, int n_grid, int n_cells) {
    return (n_order == 4 || n_order == 6) && (n_grid == 2048 || n_grid == 1024) &&
           n_cells == n_grid / 16;
}

ttm_status launch_search_tc(int n_order, const rot::SearchArgs& s, const uint16_t* grid_fp16,
                            int* status, bool bf16, cudaStream_t st, long long* cnt) {
    if ((s.n_grid != 2048 && s.n_grid != 1024) || !grid_fp16) return TTM_ERR_UNSUPPORTED;
    const bool g1 = s.n_grid == 1024;
    if (n_order == 4) {
        if (g1) return bf16 ? launch_tc_k<__nv_bfloat16, 4, 1024>(s, grid_fp16, status, st, cnt)
                            : launch_tc_k<float, 4, 1024>(s, grid_fp16, status, st, cnt);
        return bf16 ? launch_tc_k<__nv_bfloat16, 4, 2048>(s, grid_fp16, status, st, cnt)
                    : launch_tc_k<float, 4, 2048>(s, grid_fp16, status, st, cnt);
    }
    if (n_order == 6) {
        if (g1) return bf16 ? launch_tc_k<__nv_bfloat16, 6, 1024>(s, grid_fp16, status, st, cnt)
                            : launch_tc_k<float, 6, 1024>(s, grid_fp16, status, st, cnt);
        return bf16 ? launch_tc_k<__nv_bfloat16, 6, 2048>(s, grid_fp16, status, st, cnt)
                    : launch_tc_k<float, 6, 2048>(s, grid_fp16, status, st, cnt);
    }
    return TTM_ERR_UNSUPPORTED;
}

// FP16 grid table in the kernel's shared-memory layout, chunk by chunk of 256
// points: element (g, k) of the 2048 x KP matrix [mu_k q_g^k | 1 | 0...] at
// chunk g / 256, core matrix (k / 8, (g % 256) / 8), row g % 8, column k % 8,
// core matrices ordered k-block-major within the chunk.
void build_grid_fp16(const float* m_rows, int K, int K4, int n_grid, std::vector<uint16_t>& out) {
    const int KP = ((K + 1 + 15) / 16) * 16;
    out.assign((size_t)n_grid * KP, 0);
    for (int g = 0; g < n_grid; ++g)
        for (int k = 0; k < KP; ++k) {
            // column K holds the constant 1 paired with A's constant column,
            // adding +1 to every phi
            float v = k < K ? m_rows[(size_t)g * K4 + k] : (k == K ? 1.f : 0.f);
            __half h = __float2half_rn(v);
            const int c = g / kChunkN, gl = g % kChunkN;
            const size_t idx = (size_t)c * kChunkN * KP +
                               ((((size_t)(k / 8) * (kChunkN / 8) + gl / 8) * 8 + gl % 8) * 8 + k % 8);
            out[idx] = __half_as_ushort(h);
        }
}

}  // namespace ttm
