// Streaming kernel on the 5th-generation tensor cores (up to 64 tokens): the packed weights stream through
// shared memory once, are unpacked into tensor memory as the A operand of tcgen05.mma kind::i8 (UMMA M = 128
// channels), and meet the tokens as a narrow B operand (UMMA N = 16, 32, 48 or 64).
//
//  * Work.  A cluster of C CTAs (1, 2, 4 or 8) takes tiles of 128 channels, of up to four matrices that share their
//    activations; rank r of it the r-th share of K (K-splitting of Sec. II-D), in blocks of 256 k = 8 KB of packed weights.
//    The ranks exchange their sums of a tile through distributed shared memory, each adding up a part of the token
//    columns in rank order: the order is fixed by the launch, so results repeat bit for bit.
//  * Roles.  One thread brings weights (64-byte rows, 64-byte swizzle) and activations (128-byte swizzle) by TMA;
//    four or eight warps unpack a channel per lane, 64 registers of int8 lanes for 256 k, into tensor memory
//    (tcgen05.st), which the shared memory's 128 B/clk would not bear beside the copies; one warp issues the MMAs; four or
//    eight warps drain the accumulators (lane = channel, column = token): a conversion and half a packed FMA per value.
//  * Up to 32 tokens a CTA has 12 warps, 112 KB and 256 columns of tensor memory, so that two are resident per SM and one
//    computes while the other waits or, under programmatic dependent launch, while the previous kernel ends; with 64
//    tokens one CTA of 20 warps has them all.  Registers are dealt by setmaxnreg so that hardly anything spills (16 bytes
//    at most, in two instances for 64 tokens; a few words per block, local memory beside the copies, made
//    8192 x (28672 + 28672) at 32 tokens 94 us instead of 54).
//  * Sums.  Chains of eight or six groups by FMA; a chain joins the running sum with what that addition rounds away going into
//    the next chain, and the ranks' shares are added in the same way: the error does not depend on the length of a row.
//    Distance from sums in 64 bits, one running total / this: 4096 x (14336 + 14336) at 64 tokens, groups of 64, one share
//    9.5e-8 / 4.6e-8; 28672 x 8192, groups of 64, four shares 7.5e-8 / 4.0e-8; 8192 x 8192, groups of 128, four shares
//    5.5e-8 / 4.6e-8.  The other kernels are at 5.1e-8 and more at these sizes.
//  * Bound (8192 x (28672 + 28672), groups of 128, 32 tokens, 44 us, 3.0 TB/s): issue slots, 59 % busy: 2000 warp instructions
//    per block of 8 KB, of which unpack and drain (a conversion and half a packed FMA per value and group) are a good half
//    and waits and bookkeeping the rest.  On the kernel with stationary activations (mma.sync) the same launch takes 58 us.
//    Not kept: conversion through the bits of 1.5 * 2^23, by integer adds (50 us); eight drain warps at 32 tokens (45);
//    unpack warps with 64 registers (4 to 19 % more per launch); blocks dealt evenly over CTAs with cut tiles summed through
//    global memory (3 us more per small launch); one running total, or pairs of groups added first, which are 4 to 6 % faster
//    at 64 tokens and groups of 64 or 128, and too far off (above).
//  * A wait is one barrier per warp: lanes of a warp that polled different barriers saw phases that had not completed.
//  * Every wait on an mbarrier is bounded, as in the other tensor-core kernels.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "w2a8_tc.cuh"

namespace w2a8 {

constexpr int kTsMaxMats = 4;
constexpr int kTsBM = 128;                  // channels of a tile (UMMA M, TMEM lanes)
constexpr int kTsWBytes = kTsBM * 64;       // packed weights of a block
constexpr int kTsMaxCluster = 8;

struct TsMat {
    const void *w_scale;
    void *y;
    int tile_end;         // tiles of this matrix and of all before it
    int N;
    int ldy;
};

struct TsParams {
    TsMat mat[kTsMaxMats];
    const float *a_scale;
    int *status;
    int nmats, M, G, KB;  // KB: blocks of a row
    int C;                // CTAs per cluster = shares of K
    int blk_per, blk_extra;       // rank r owns blk_per (+ 1 if r < blk_extra) blocks of every row
    int tiles, nclusters; // cluster c takes tiles c, c + nclusters, ...
    int bpg;              // blocks per scale group (groups of whole blocks)
    int y16;
    unsigned polls;       // bound of every wait
};

struct TsMaps {
    CUtensorMap w[kTsMaxMats];
    CUtensorMap act;
};

// NT: tokens that are drained (16, 24, 32, 48, 64); SPP: 64-k slices per scale group, 0 = groups of whole blocks, kTsRow = one
// group per row.
constexpr int kTsRow = -1;
template <int NT, int SPP>
struct TsCfg {
    static constexpr int BN = (NT + 15) / 16 * 16;                // UMMA N
    static constexpr int kCtasPerSm = NT <= 32 ? 2 : 1;
    static constexpr int kDrainWarps = NT > 32 ? 8 : 4;
    static constexpr int kUnpackSets = NT <= 32 ? 1 : 2;          // sets of four warps, on alternate blocks
    static constexpr int DC = NT * 4 / kDrainWarps;               // token columns of a drain warp
    static constexpr int kFirstUnpack = 4, kFirstDrain = 4 + 4 * kUnpackSets;
    static constexpr int kThreads = 32 * (kFirstDrain + kDrainWarps);
    static constexpr int kTmemCols = NT <= 32 ? 256 : 512;
    static constexpr int AS = NT <= 32 ? 2 : 4;     // unpacked blocks in tensor memory
    static constexpr int kAccCols = kTmemCols - 64 * AS;
    static constexpr int GPB = SPP <= 0 ? 1 : 4 / SPP;            // groups of a block
    static constexpr int UG = SPP <= 0 ? 1 : GPB * BN <= 64 ? GPB : 2;   // groups of a unit = hand-off between MMA and drain
    static constexpr int UPB = GPB / UG;                          // units of a block
    static constexpr int kUnitCols = UG * BN;
    // A chain of additions is kChain blocks (groups of whole blocks: groups) long, eight groups and with groups of 128 six
    // (four cost 2 to 5 % of a launch, eight save nothing and are further off on short rows).  The running sums of the
    // second half of a thread's columns are in shared memory where the registers do not hold them.
    static constexpr int kChain = SPP <= 0 ? 8 : SPP == 2 ? 3 : 8 / GPB;
    static constexpr int kHiShared = SPP != kTsRow && DC > 16 ? DC / 2 : 0;
    static constexpr int kHiBytes = kHiShared * 4 * 32 * kDrainWarps;
    static constexpr int kUnits = kAccCols / kUnitCols;
    // One barrier says that a block is unpacked and its accumulators are free, where both come round alike.
    static constexpr bool kFold = SPP > 0 && UPB == 1 && kUnits >= AS;
    static constexpr int NU = kFold ? AS : kUnits > 4 ? 4 : kUnits;      // units in flight
    static constexpr int kStageBytes = kTsWBytes + BN * 256;
    static constexpr int kSumBytes = kTsBM * (DC == 24 ? 32 : DC) * kDrainWarps;     // a tile's sums, in pieces of 16 bytes
    static constexpr int kRing = ((kCtasPerSm == 2 ? 112 : 224) * 1024 - 2048 - 2 * kSumBytes) / kStageBytes;
    static constexpr size_t kSmem = (size_t)kRing * kStageBytes + 2 * kSumBytes + kHiBytes + 1024;
    static constexpr bool kUnitBarrier = SPP <= 0 || UPB > 1;     // else a block's barrier says it all
    // Registers per thread: the launch has 80 or 96 (what the launch bounds leave, rounded down to a multiple of eight, and
    // what the compiler reports for every instance); setmaxnreg moves some of the first warps' to the drain warps.
    static constexpr int kRegs = NT <= 32 ? 80 : 96, kRegsFirst = NT <= 32 ? 24 : 32, kRegsDrain = NT <= 32 ? 136 : 128;
    static_assert(kFirstUnpack * (kRegs - kRegsFirst) >= kDrainWarps * (kRegsDrain - kRegs), "");
    static_assert(kSmem + 1024 <= (kCtasPerSm == 2 ? 113 : 227) * 1024, "");
    static_assert(NU >= 2 && AS < kRing, "");
};

__device__ __forceinline__ void ts_mma_i8_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void ts_tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void ts_tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void ts_tmem_ld(uint32_t taddr, int (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void ts_tmem_ld(uint32_t taddr, int (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void ts_tmem_ld(uint32_t taddr, int (&v)[24]) {
    ts_tmem_ld(taddr, reinterpret_cast<int (&)[16]>(v[0]));
    ts_tmem_ld(taddr + 16, reinterpret_cast<int (&)[8]>(v[16]));
}
__device__ __forceinline__ void ts_tmem_ld(uint32_t taddr, int (&v)[32]) { pf_tmem_ld32(taddr, v); }
// Joins two chains (a0, a1) with the running sums (h0, h1), packed fp32.  What the addition rounds away stays behind in
// the chains and goes into the next join.
__device__ __forceinline__ void ts_join2(float &h0, float &h1, float &a0, float &a1) {
    asm("{\n\t.reg .b64 h, a, s, z, m;\n\t"
        "mov.b64 h, {%0, %1};\n\tmov.b64 a, {%2, %3};\n\tmov.b64 m, {%4, %4};\n\t"
        "add.rn.f32x2 s, h, a;\n\t"
        "fma.rn.f32x2 z, h, m, s;\n\t"        // s - h: the part of the chain that the sum took
        "fma.rn.f32x2 a, z, m, a;\n\t"        // the rest
        "mov.b64 {%0, %1}, s;\n\tmov.b64 {%2, %3}, a;\n\t}"
        : "+f"(h0), "+f"(h1), "+f"(a0), "+f"(a1) : "f"(-1.f));
}
__device__ __forceinline__ void ts_st_shared2(uint32_t addr, float x, float y) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}
template <int N>
__device__ __forceinline__ void ts_maxreg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void ts_maxreg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// N floats into another CTA's shared memory, counted by its barrier, in the widest pieces that N divides into
template <int N>
__device__ __forceinline__ void ts_send(uint32_t addr, uint32_t bar, int rank, const float *v) {
    uint32_t ra, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(bar), "r"(rank));
    constexpr int P = N % 4 == 0 ? 4 : N % 2 == 0 ? 2 : 1;
#pragma unroll
    for (int j = 0; j < N; j += P) {
        if constexpr (P == 4)
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                         ::"r"(ra + j * 4), "r"(__float_as_uint(v[j])), "r"(__float_as_uint(v[j + 1])), "r"(__float_as_uint(v[j + 2])),
                           "r"(__float_as_uint(v[j + 3])), "r"(rb) : "memory");
        else if constexpr (P == 2)
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                         ::"r"(ra + j * 4), "r"(__float_as_uint(v[j])), "r"(__float_as_uint(v[j + 1])), "r"(rb) : "memory");
        else
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                         ::"r"(ra + j * 4), "r"(__float_as_uint(v[j])), "r"(rb) : "memory");
    }
}
template <int N>
__device__ __forceinline__ void ts_ld_shared(float (&v)[N], uint32_t addr) {
    constexpr int P = N % 4 == 0 ? 4 : 2;
    static_assert(N % P == 0, "");
#pragma unroll
    for (int j = 0; j < N; j += P) {
        if constexpr (P == 4)
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[j]), "=f"(v[j + 1]), "=f"(v[j + 2]), "=f"(v[j + 3])
                         : "r"(addr + j * 4) : "memory");
        else
            asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[j]), "=f"(v[j + 1]) : "r"(addr + j * 4) : "memory");
    }
}
// pf_wait for data that other CTAs of the cluster wrote
__device__ __forceinline__ bool ts_wait_cluster(uint32_t bar, unsigned parity, volatile int *abort_flag, unsigned polls) {
    for (unsigned i = 0; i < polls; ++i) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if ((i & 63u) == 63u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

// Bounded wait of a converged warp (pf_wait_all) whose first look costs a poll, a vote and a branch: most waits find their
// barrier complete, and what the warps spend on looking was a third of all instructions.
__device__ __forceinline__ bool ts_wait(uint32_t bar, unsigned parity, volatile int *abort_flag, unsigned polls) {
    if (__all_sync(0xFFFFFFFFu, pf_mbar_try_wait(bar, parity))) return true;
    return pf_wait_all(bar, parity, abort_flag, polls);
}

template <int NT, int SPP, bool H16>
__global__ void __launch_bounds__(TsCfg<NT, SPP>::kThreads, TsCfg<NT, SPP>::kCtasPerSm)
w2a8_tstream_kernel(const __grid_constant__ TsMaps maps, const __grid_constant__ TsParams p) {
    using C = TsCfg<NT, SPP>;
    constexpr int BN = C::BN, R = C::kRing, AS = C::AS, NU = C::NU, UG = C::UG, DC = C::DC;
    extern __shared__ unsigned char ts_smem[];
    __shared__ __align__(8) unsigned long long bar_w[R], bar_b[R], bar_done[R], bar_a[AS], bar_full[NU], bar_free[NU];
    __shared__ __align__(8) unsigned long long bar_sum[2][C::kDrainWarps];
    __shared__ float tok_scale[NT];
    __shared__ __align__(8) unsigned long long bar_mma;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_s, copies_w_s, copies_b_s;
    volatile int *abort_flag = &abort_s;

    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t stage0 = (pf_smem_u32(ts_smem) + 1023u) & ~1023u;
    // this CTA's share of K, and its tiles
    const int nc = p.C, rank = nc > 1 ? (int)cluster_ctarank() : 0;
    int cl;
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(cl));
    const int kb_lo = rank * p.blk_per + min(rank, p.blk_extra), nb = p.blk_per + (rank < p.blk_extra ? 1 : 0);
    const int ntiles = (p.tiles - cl + p.nclusters - 1) / p.nclusters, n = ntiles * nb;      // blocks of this CTA
    // matrix of a tile, and the tile's first channel there
    auto mat_of = [&](int tile, int &n0) -> int {
        int i = 0, first = 0;
#pragma unroll
        for (int j = 1; j < kTsMaxMats; ++j)
            if (j < p.nmats && tile >= p.mat[j - 1].tile_end) { i = j; first = p.mat[j - 1].tile_end; }
        n0 = (tile - first) * kTsBM;
        return i;
    };

    if (threadIdx.x == 0) {
        abort_s = copies_w_s = copies_b_s = 0;
        pf_mbar_init(pf_smem_u32(&bar_mma), 1);
        for (int i = 0; i < R; ++i) {
            pf_mbar_init(pf_smem_u32(&bar_w[i]), 1);
            pf_mbar_init(pf_smem_u32(&bar_b[i]), 1);
            pf_mbar_init(pf_smem_u32(&bar_done[i]), 1);
        }
        for (int i = 0; i < AS; ++i) pf_mbar_init(pf_smem_u32(&bar_a[i]), 4 + (C::kFold ? C::kDrainWarps : 0));
        for (int i = 0; i < NU; ++i) {
            pf_mbar_init(pf_smem_u32(&bar_full[i]), 1);
            pf_mbar_init(pf_smem_u32(&bar_free[i]), C::kDrainWarps);
        }
        for (int i = 0; i < 2 * C::kDrainWarps; ++i) pf_mbar_init(pf_smem_u32(&bar_sum[0][0] + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        pf_fence_proxy_async();
    }
    if (warp == 1) pf_tmem_alloc(pf_smem_u32(&tmem_slot), C::kTmemCols);
    pf_tc_fence_before();
    __syncthreads();
    pf_tc_fence_after();
    // every CTA of the cluster has its barriers: arrive here, wait before the first access to another CTA
    int nsum = 0;                                       // (drain warps) tiles summed so far
    if (nc > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const uint32_t sums0 = stage0 + R * C::kStageBytes;
    const uint32_t tmem_a = tmem_slot, tmem_acc = tmem_slot + 64 * AS;
    // Programmatic dependent launch: weights and scales are frozen, everything up to the first unpacked blocks
    // overlaps the tail of the previous kernel of the stream.  Roles that touch anything else, or that could wait for
    // one that does, wait for that kernel first (a wait's limit covers this kernel's own work only).
    pdl_launch_dependents();

    if (warp < C::kFirstUnpack) {
        ts_maxreg_dec<C::kRegsFirst>();
        if (warp == 0 && lane == 0) {
            // ===== TMA producer =============================================================
            int tile = cl, kb = 0, n0;
            int mi = mat_of(tile, n0);
            auto advance = [&]() {
                if (++kb == nb) {
                    kb = 0;
                    tile += p.nclusters;
                    if (tile < p.tiles) mi = mat_of(tile, n0);
                }
            };
            auto load_w = [&](int s) {
                pf_tma_load_2d(stage0 + s * C::kStageBytes, &maps.w[mi], (kb_lo + kb) * 16, n0, pf_smem_u32(&bar_w[s]));
            };
            auto load_b = [&](int s, int k, uint32_t bar) {
                const uint32_t dst = stage0 + s * C::kStageBytes + kTsWBytes;
                pf_tma_load_2d(dst, &maps.act, (kb_lo + k) * 256, 0, bar);
                pf_tma_load_2d(dst + BN * 128, &maps.act, (kb_lo + k) * 256 + 128, 0, bar);
            };
            const int head = min(R, n);
            for (int i = 0; i < head; ++i) {
                pf_mbar_arrive_expect_tx(pf_smem_u32(&bar_w[i]), kTsWBytes);
                load_w(i);
                advance();
            }
            asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.act) : "memory");
            pdl_wait();
            for (int i = 0, k = 0; i < head; ++i) {
                pf_mbar_arrive_expect_tx(pf_smem_u32(&bar_b[i]), BN * 256);
                load_b(i, k, pf_smem_u32(&bar_b[i]));
                if (++k == nb) k = 0;
            }
            copies_b_s = head;
            copies_w_s = head;
            int s = 0;
            uint32_t ph = 0;
            for (int i = R; i < n; ++i) {
                if (!pf_wait(pf_smem_u32(&bar_done[s]), ph, abort_flag, p.polls)) break;
                // (the MMA warp learns of these activations from the unpack warps, which wait for both)
                pf_mbar_arrive_expect_tx(pf_smem_u32(&bar_w[s]), C::kStageBytes);
                load_w(s);
                load_b(s, kb, pf_smem_u32(&bar_w[s]));
                copies_w_s = i + 1;
                advance();
                if (++s == R) { s = 0; ph ^= 1u; }
            }
        } else if (warp == 1) {
            // ===== MMA issuer: the warp walks, one elected lane issues ========================
            const bool lead = pf_elect();
            if (lead) pdl_wait();
            __syncwarp();
            const uint64_t b_desc0 = pf_smem_desc(stage0 + kTsWBytes);
            const uint32_t b_lo = (uint32_t)b_desc0, b_hi = (uint32_t)(b_desc0 >> 32);
            constexpr uint32_t idesc = pf_instr_desc(kTsBM, BN);
            int s = 0, as = 0, un = 0;
            uint32_t aph = 0, uph = 0, so = 0;
            bool ok = true;
            [[maybe_unused]] int kb = 0;
            [[maybe_unused]] bool fresh = true;         // (groups of whole blocks) the next block opens a unit
            const int first_left = SPP == 0 ? p.bpg - kb_lo % p.bpg : nb;
            [[maybe_unused]] int left = first_left;
            for (int i = 0; i < n; ++i) {
                if (i < R) ok = ts_wait(pf_smem_u32(&bar_b[s]), 0, abort_flag, p.polls);
                if (SPP <= 0 && fresh) ok = ok && ts_wait(pf_smem_u32(&bar_free[un]), uph, abort_flag, p.polls);
                ok = ok && ts_wait(pf_smem_u32(&bar_a[as]), aph, abort_flag, p.polls);
                if (!ok) break;
                auto step = [&](int j, uint32_t d, uint32_t acc) {
                    const uint32_t koff = ((j >> 2) * BN * 128 + (j & 3) * 32) >> 4;
                    ts_mma_i8_tmem(d, tmem_a + as * 64 + 8 * j, ((uint64_t)b_hi << 32) | (b_lo + so + koff), idesc, acc);
                };
                if constexpr (SPP > 0) {
#pragma unroll
                    for (int u = 0; u < C::UPB; ++u) {
                        if constexpr (!C::kFold) ok = ts_wait(pf_smem_u32(&bar_free[un]), uph, abort_flag, p.polls);
                        if (!ok) break;
                        pf_tc_fence_after();
                        if (lead) {
                            const uint32_t d = tmem_acc + un * C::kUnitCols;
#pragma unroll
                            for (int j = 0; j < 8 / C::UPB; ++j) step(u * (8 / C::UPB) + j, d + (j / (2 * SPP)) * BN, j % (2 * SPP) != 0 ? 1u : 0u);
                            if constexpr (C::kUnitBarrier) pf_mma_commit(pf_smem_u32(&bar_full[un]));
                        }
                        if (++un == NU) { un = 0; uph ^= 1u; }
                    }
                    if (!ok) break;
                } else {
                    pf_tc_fence_after();
                    const bool last = --left == 0 || kb + 1 == nb;
                    if (lead) {
                        const uint32_t d = tmem_acc + un * C::kUnitCols;
                        step(0, d, fresh ? 0u : 1u);
#pragma unroll
                        for (int j = 1; j < 8; ++j) step(j, d, 1u);
                        if (last) pf_mma_commit(pf_smem_u32(&bar_full[un]));
                    }
                    fresh = last;
                    if (last) {
                        left = SPP == 0 ? p.bpg : nb;
                        if (++un == NU) { un = 0; uph ^= 1u; }
                    }
                    if (++kb == nb) { kb = 0; left = first_left; }
                }
                if (lead) pf_mma_commit(pf_smem_u32(&bar_done[s]));
                so += C::kStageBytes >> 4;
                if (++s == R) { s = 0; so = 0; }
                if (++as == AS) { as = 0; aph ^= 1u; }
            }
            // every MMA has ended, also where the drain warps need not have waited for it, and where a wait gave up
            if (lead) pf_mma_commit(pf_smem_u32(&bar_mma));
            pf_wait_own(pf_smem_u32(&bar_mma), 0);
            __syncwarp();
        }
    } else if (warp < C::kFirstDrain) {
        // ===== unpack warps: a lane's channel of a block, 16 words -> 64 columns of int8 lanes ========
        const int set = (warp - C::kFirstUnpack) >> 2, q = warp & 3;
        const int row = q * 32 + lane;
        const uint32_t tlane = tmem_a + ((uint32_t)(q * 32) << 16);
        const uint32_t row_off = row * 64, sw = (row >> 1) & 3;
        int s = set, as = set % AS;                     // ring slot, place in tensor memory
        uint32_t ph = 0;
        bool got = true;
        uint32_t w[4][4];                               // [t][slice]
        auto load = [&](int slot) {
            const uint32_t base = stage0 + slot * C::kStageBytes + row_off;
#pragma unroll
            for (int t = 0; t < 4; ++t)
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[t][0]), "=r"(w[t][1]), "=r"(w[t][2]), "=r"(w[t][3])
                             : "r"(base + ((t ^ sw) << 4)));
        };
        if (set < n) {
            got = ts_wait(pf_smem_u32(&bar_w[s]), 0, abort_flag, p.polls);
            load(s);
        }
        int ds = (set + 2 * R - AS) % R;                // slot of block i - AS
        uint32_t dph = 1u;                              // its parity (flips whenever ds comes round to 0)
        for (int i = set; i < n && got; i += C::kUnpackSets) {
            if (i >= AS) {                              // the MMAs of block i - AS have read this place
                if (i < AS + C::kUnpackSets) pdl_wait();
                got = ts_wait(pf_smem_u32(&bar_done[ds]), dph, abort_flag, p.polls);
                pf_tc_fence_after();
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t v[32];
#pragma unroll
                for (int sl = 0; sl < 2; ++sl)
#pragma unroll
                    for (int t = 0; t < 4; ++t)
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[16 * sl + 4 * t + j] = lane_codes(w[t][2 * h + sl], j);
                ts_tmem_st32(tlane + as * 64 + 32 * h, v);
            }
            // the next block's words on their way while the stores finish
            s += C::kUnpackSets;
            if (s >= R) { s -= R; ph ^= 1u; }
            if (i + C::kUnpackSets < n) {
                got = got && ts_wait(pf_smem_u32(&bar_w[s]), ph, abort_flag, p.polls);
                load(s);
            }
            ts_tmem_st_wait();
            pf_tc_fence_before();
            __syncwarp();
            if (lane == 0) pf_mbar_arrive(pf_smem_u32(&bar_a[as]));
            as = (as + C::kUnpackSets) % AS;
            ds += C::kUnpackSets;
            if (ds >= R) { ds -= R; dph ^= 1u; }
        }
    } else {
        ts_maxreg_inc<C::kRegsDrain>();
        // ===== drain warps ==============================================================
        const int q = warp & 3, d = warp - C::kFirstDrain, col0 = (d >> 2) * DC;
        const uint32_t tlane = tmem_acc + ((uint32_t)(q * 32) << 16) + col0;
#pragma unroll
        for (int un = 0; un < NU; ++un) {
            if (lane == 0) pf_mbar_arrive(pf_smem_u32(C::kFold ? &bar_a[un] : &bar_free[un]));
        }
        // scales of a block (groups of 64, 128) or group, two ahead of the block that is drained
        struct Scales { uint32_t r[4]; };
        int tile = cl, kb = 0;                          // block that is drained
        int ptile = cl, pkb = 0, left = n;              // block whose scales are requested next
        const char *srow = nullptr;
        auto locate = [&](int t) {
            int n0;
            const int i = mat_of(t, n0);
            const int ch = min(n0 + q * 32 + lane, p.mat[i].N - 1);
            srow = reinterpret_cast<const char *>(p.mat[i].w_scale) + (size_t)ch * p.G * (H16 ? 2 : 4) +
                   (SPP <= 0 ? 0 : kb_lo * C::GPB * (H16 ? 2 : 4));
        };
        locate(ptile);
        // (groups of whole blocks) group of the block that is requested next, blocks left of it
        const int gi0 = SPP == 0 ? kb_lo / p.bpg : 0, first_left = SPP == 0 ? (gi0 + 1) * p.bpg - kb_lo : nb;
        int pgi = gi0, pleft = first_left;
        constexpr int kStep = SPP <= 0 ? 0 : C::GPB * (H16 ? 2 : 4);      // scale bytes of a block
        auto request = [&]() -> Scales {
            Scales sc = {};
            if (left == 0) return sc;
            --left;
            if constexpr (kStep == 16) {
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(srow)); sc.r[0] = v.x; sc.r[1] = v.y; sc.r[2] = v.z; sc.r[3] = v.w;
            } else if constexpr (kStep == 8) {
                const uint2 v = __ldg(reinterpret_cast<const uint2 *>(srow)); sc.r[0] = v.x; sc.r[1] = v.y;
            } else if constexpr (kStep == 4) {
                sc.r[0] = __ldg(reinterpret_cast<const uint32_t *>(srow));
            } else {
                if constexpr (H16) sc.r[0] = __ldg(reinterpret_cast<const unsigned short *>(srow) + pgi);
                else sc.r[0] = __ldg(reinterpret_cast<const uint32_t *>(srow) + pgi);
                if (SPP == 0 && --pleft == 0) { ++pgi; pleft = p.bpg; }
            }
            srow += kStep;
            if (++pkb == nb) {
                pkb = 0; ptile += p.nclusters; pgi = gi0; pleft = first_left;
                if (left > 0) locate(ptile);
            }
            return sc;
        };
        auto scale = [&](const Scales &sc, int g) -> float {       // g is a constant after unrolling
            if constexpr (!H16) return __uint_as_float(sc.r[g]);
            else {
                const __half2 h = *reinterpret_cast<const __half2 *>(&sc.r[g >> 1]);
                return (g & 1) ? __high2float(h) : __low2float(h);
            }
        };
        Scales sc_cur, sc_n1 = request(), sc_n2 = request();
        pdl_wait();
        if (warp == C::kFirstDrain)
            for (int j = lane; j < NT; j += 32) tok_scale[j] = p.a_scale[min(j, p.M - 1)] * (1.0f / kCodeGain);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * C::kDrainWarps) : "memory");
        constexpr int HS = C::kHiShared, HR = DC - HS;
        float acc[DC], hi[HR];                          // chains, running sums (the last HS columns': hi_s, in pairs)
        const uint32_t hi_s = sums0 + 2 * C::kSumBytes + (d * 32 + lane) * 8;
        constexpr uint32_t kHiStep = C::kDrainWarps * 32 * 8;
        int s = 0, un = 0, chain;
        float largest;                                  // scale of this tile's row so far
        auto clear = [&]() {
#pragma unroll
            for (int j = 0; j < DC; ++j) acc[j] = 0.f;
#pragma unroll
            for (int j = 0; j < HR; ++j) hi[j] = 0.f;
#pragma unroll
            for (int j = 0; j < HS; j += 2) ts_st_shared2(hi_s + j / 2 * kHiStep, 0.f, 0.f);
            chain = 0;
            largest = 0.f;
        };
        clear();
        uint32_t ph = 0, uph = 0;
        bool got = true;
        // One group per row: shares are summed as the integers they are and scaled once, so that the split of K adds no
        // rounding (8192 x 8192 at 64 tokens 4.3e-8 from sums in 64 bits with scaled shares, 3.6e-8 with integers).
        constexpr bool whole = SPP == kTsRow;
        [[maybe_unused]] int gleft = first_left;
        auto drain_unit = [&](int g0) {
            // All groups of the unit for CH columns at a time (more staged values spill, and local memory is slow beside
            // the copies).
            constexpr int CH = UG == 4 ? 8 : DC == 32 ? 16 : DC;
            const uint32_t at = tlane + un * C::kUnitCols;
#pragma unroll
            for (int c = 0; c < DC; c += CH) {
                int v[UG][CH];
#pragma unroll
                for (int g = 0; g < UG; ++g) ts_tmem_ld(at + g * BN + c, v[g]);
                pf_tmem_ld_wait();
                if (c + CH == DC) {
                    pf_tc_fence_before();
                    __syncwarp();
                    if (lane == 0) pf_mbar_arrive(pf_smem_u32(C::kFold ? &bar_a[un] : &bar_free[un]));
                    if (++un == NU) { un = 0; uph ^= 1u; }
                }
                float f[UG];
#pragma unroll
                for (int g = 0; g < UG; ++g) {
                    f[g] = scale(sc_cur, g0 + g);
                    if (c == 0) largest = fmaxf(largest, fabsf(f[g]));
                }
                if constexpr (whole) {
#pragma unroll
                    for (int j = 0; j < CH; ++j) acc[c + j] = __int_as_float(v[0][j]);
                } else {
#pragma unroll
                    for (int g = 0; g < UG; ++g)
#pragma unroll
                        for (int j = 0; j < CH; j += 2) pf_fma2(acc[c + j], acc[c + j + 1], (float)v[g][j], (float)v[g][j + 1], f[g]);
                }
            }
        };
        auto join = [&]() {
            chain = 0;
#pragma unroll
            for (int j = 0; j < HR; j += 2) ts_join2(hi[j], hi[j + 1], acc[j], acc[j + 1]);
#pragma unroll
            for (int j = 0; j < HS; j += 2) {
                float h[2];
                ts_ld_shared<2>(h, hi_s + j / 2 * kHiStep);
                ts_join2(h[0], h[1], acc[HR + j], acc[HR + j + 1]);
                ts_st_shared2(hi_s + j / 2 * kHiStep, h[0], h[1]);
            }
            // A row's integers add up to less than 2^31.  Sums that may be infinite are plain ones: an infinity minus itself is
            // not what an addition left over.  (A vote in front of the branch cost 4 % of a launch at 16 tokens.)
            if (largest >= 0x1p96f) {
#pragma unroll
                for (int j = 0; j < DC; ++j) acc[j] = 0.f;
            }
        };
        for (int i = 0; i < n; ++i) {
            sc_cur = sc_n1; sc_n1 = sc_n2; sc_n2 = request();
            const bool row_end = kb + 1 == nb;
            if constexpr (SPP > 0) {
#pragma unroll
                for (int u = 0; u < C::UPB; ++u) {
                    if constexpr (C::kUnitBarrier) got = got && ts_wait(pf_smem_u32(&bar_full[un]), uph, abort_flag, p.polls);
                    else                           got = got && ts_wait(pf_smem_u32(&bar_done[s]), ph, abort_flag, p.polls);
                    pf_tc_fence_after();
                    drain_unit(u * UG);
                }
                if (++chain == C::kChain) join();
            } else if (--gleft == 0 || row_end) {
                gleft = row_end ? first_left : SPP == 0 ? p.bpg : nb;
                got = got && ts_wait(pf_smem_u32(&bar_full[un]), uph, abort_flag, p.polls);
                pf_tc_fence_after();
                drain_unit(0);
                if (!whole && ++chain == C::kChain) join();
            }
            if (++s == R) { s = 0; ph ^= 1u; }
            if (!got) break;
            if (row_end) {
                // ---- this CTA's share of the tile's sums is complete ---------------------------
                if constexpr (!whole) {
#pragma unroll
                    for (int j = 0; j < HR; ++j) acc[j] += hi[j];
#pragma unroll
                    for (int j = 0; j < HS; j += 2) {
                        float h[2];
                        ts_ld_shared<2>(h, hi_s + j / 2 * kHiStep);
                        acc[HR + j] += h[0];
                        acc[HR + j + 1] += h[1];
                    }
                }
                const float row_scale = whole ? scale(sc_cur, 0) : 0.f;
                auto scaled = [&](float bits) -> float { return (float)__float_as_int(bits) * row_scale; };
                int n0;
                const int mi = mat_of(tile, n0);
                const int ch = n0 + q * 32 + lane;
                const bool valid = ch < p.mat[mi].N;
                const int ldy = p.mat[mi].ldy;
                char *y = reinterpret_cast<char *>(p.mat[mi].y);
                auto store = [&](int m, float sum) {
                    const float v = sum * tok_scale[m];
                    if (m < p.M && valid) {
                        const size_t at = (size_t)m * ldy + ch;
                        if (H16 && p.y16) reinterpret_cast<__nv_bfloat16 *>(y)[at] = __float2bfloat16_rn(v);
                        else              reinterpret_cast<float *>(y)[at] = v;
                    }
                };
                // Shares are exchanged through distributed shared memory: rank r adds up the r-th part of every
                // thread's columns, in rank order (of 24 columns eight ranks have parts of 4, not 3, and the last two none: with
                // 4-byte stores 14336 x 4096 took 14 instead of 10 us at 24 tokens; a rank without columns gets a word, to keep step).  The buffers alternate: a CTA that is two tiles ahead has received what
                // its peers sent after reading theirs.
                auto exchange = [&](auto cc) {
                    constexpr int CC = decltype(cc)::value, PC = DC == 24 ? (24 / CC + 3) / 4 * 4 : DC / CC, kParts = DC / PC;
                    constexpr uint32_t kFrom = C::kDrainWarps * 32 * PC * 4;       // bytes from one rank
                    const uint32_t buf = sums0 + (nsum & 1) * C::kSumBytes + (d * 32 + lane) * (PC * 4);
                    const uint32_t bar = pf_smem_u32(&bar_sum[nsum & 1][d]);
                    if (nsum == 0) cluster_wait_acquire();
                    __syncwarp();
                    if (lane == 0) pf_mbar_arrive_expect_tx(bar, (CC - 1) * (rank < kParts ? 32 * PC * 4 : 4));
#pragma unroll
                    for (int r = 0; r < CC; ++r) {
                        if (r == rank) continue;
                        if (r < kParts)     ts_send<PC>(buf + rank * kFrom, bar, r, acc + (r < kParts ? r : 0) * PC);
                        else if (lane == 0) ts_send<1>(buf + rank * kFrom, bar, r, acc);
                    }
                    got = __all_sync(0xFFFFFFFFu, ts_wait_cluster(bar, (nsum >> 1) & 1, abort_flag, p.polls));
                    ++nsum;
                    if (rank >= kParts) return;
                    float sum[PC], rest[PC];
#pragma unroll
                    for (int r = 0; r < CC; ++r) {
                        float v[PC];
                        ts_ld_shared<PC>(v, buf + r * kFrom);
#pragma unroll
                        for (int j = 0; j < PC; ++j) {
                            const float x = r < kParts && r == rank ? acc[(r < kParts ? r : 0) * PC + j] : v[j];
                            if (r == 0) { sum[j] = x; rest[j] = 0.f; continue; }
                            if (whole) { sum[j] = __int_as_float(__float_as_int(sum[j]) + __float_as_int(x)); continue; }
                            const float s2 = sum[j] + x, took = s2 - sum[j];      // exact sum = s2 + what is left of both terms
                            rest[j] += (sum[j] - (s2 - took)) + (x - took);
                            sum[j] = s2;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < PC; ++j)          // (an infinite sum has no rest)
                        store(col0 + rank * PC + j, whole ? scaled(sum[j]) : rest[j] == rest[j] ? sum[j] + rest[j] : sum[j]);
                };
                if (nc == 1) {
#pragma unroll
                    for (int j = 0; j < DC; ++j) store(col0 + j, whole ? scaled(acc[j]) : acc[j]);
                } else if (nc == 2) exchange(std::integral_constant<int, 2>{});
                else if (nc == 4)   exchange(std::integral_constant<int, 4>{});
                else                exchange(std::integral_constant<int, 8>{});
                clear();
            }
            if (++kb == nb) { kb = 0; tile += p.nclusters; }
        }
    }

    // ---- wind down ---------------------------------------------------------------------
    __syncwarp();
    if (nc > 1 && nsum == 0) cluster_wait_acquire();
    pf_tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (abort_s) {
        // A wait gave up.  Nothing may be on its way into this CTA's shared memory when it leaves: neither its own copies
        // nor sums of its peers, which have left or wait here as well once the cluster barrier opens (it counts the threads
        // that have not exited).  The pause covers stores that were under way, many times over.
        if (threadIdx.x == 0) {
            atomicExch(p.status, W2A8_ERR_TIMEOUT);
            for (int i = max(0, copies_w_s - R); i < copies_w_s; ++i) pf_wait_own(pf_smem_u32(&bar_w[i % R]), (uint32_t)(i / R) & 1u);
            for (int i = 0; i < copies_b_s; ++i) pf_wait_own(pf_smem_u32(&bar_b[i]), 0);
        }
        __syncthreads();
        if (nc > 1) {
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            cluster_wait_acquire();
            __nanosleep(20000);
        }
    }
    if (warp == 1) {
        pf_tc_fence_after();
        pf_tmem_dealloc(tmem_slot, C::kTmemCols);
    }
}

// ---- host side -----------------------------------------------------------------------
bool gemv_preferred(int M, int K, int group, int tiles, int count);
double stat_estimate(int M, int K, int group, int pairs);

bool tstream_supported(int M, int K, int group) {
    if (M < 1 || M > 64 || K % kBlockK != 0) return false;
    if ((long long)64 * 254 * group >= (1ll << 31)) return false;           // int32 accumulator range
    return group == 64 || group == 128 || group % 256 == 0;
}
static int ts_tokens(int M) { return M <= 16 ? 16 : M <= 24 ? 24 : M <= 32 ? 32 : M <= 48 ? 48 : 64; }

// Time of a launch in us, by token width and group (64, 128, more): a start, one per block of cost, round with an exchange
// of sums, and level of C.
struct TsTimes { double start, block, round, level; };
static const TsTimes kTsTimes[5][3] = {
    {{1.891, 0.340, 0.482, -0.054}, {1.889, 0.289, 0.457, -0.038}, {2.738, 0.234, 0.411, -0.236}},
    {{2.652, 0.420, 0.573, -0.040}, {2.444, 0.320, 0.609, -0.095}, {3.033, 0.258, 0.457, -0.159}},
    {{3.459, 0.471, 0.919, -0.456}, {3.396, 0.338, 0.835, -0.446}, {3.451, 0.263, 0.606, -0.302}},
    {{3.317, 0.429, 0.729, -0.005}, {3.190, 0.294, 0.589, 0.071}, {3.874, 0.221, 0.332, 0.002}},
    {{4.577, 0.488, 1.237, -0.560}, {4.311, 0.331, 1.059, -0.474}, {4.526, 0.226, 0.605, -0.197}}
};
static const TsTimes &ts_times(int M, int group) {
    const int nt = ts_tokens(M);
    return kTsTimes[nt == 16 ? 0 : nt == 24 ? 1 : nt == 32 ? 2 : nt == 48 ? 3 : 4][group == 64 ? 0 : group == 128 ? 1 : 2];
}

// Shares of K and clusters for a launch over `tiles` tiles of `KB` blocks: those of the least estimated time, which is
// returned.  The cost counts blocks that one CTA works off after the other, in full rounds of the resident clusters and a
// last one; a block takes twice as long where every SM has a CTA as where few have, and 30 % more with two CTAs on each.
// Fitted to 2280 launches of the layers' and of random matrices at 9 to 64 tokens with every C (7 % rms); the choice loses
// 1.0 % on average against the best C.
static double ts_plan(int tiles, int KB, const int *resident, const TsTimes &t, int *C, int *nclusters) {
    const int forced = env_int("W2A8_TSTREAM_C", 0);
    const double sms = sm_count();
    auto load = [&](double ctas) { return 1.0 + std::min(1.0, ctas / sms) + 0.3 * std::max(0.0, ctas / sms - 1.0); };
    double best = 1e30;
    for (int c = 1, level = 0; c <= kTsMaxCluster; c *= 2, ++level) {
        if (c > KB || resident[c] < 1 || (forced > 0 && c != forced)) continue;
        const int ncl = std::min(tiles, resident[c]), full = tiles / ncl, left = tiles % ncl, share = (KB + c - 1) / c;
        const double cost = share * (full * load((double)ncl * c) + (left > 0 ? load((double)left * c) : 0.0));
        const double us = t.start + t.block * cost + (c > 1 ? t.round * (full + (left > 0)) : 0.0) + t.level * level;
        if (us < best) { best = us; *C = c; *nclusters = ncl; }
    }
    return best;
}

// Whether the kernel takes a launch over `count` matrices of `tiles16` 16-channel tiles in all (9 to 64 tokens).
// Compared are the estimates of its own launch and of the kernel with stationary activations, whose plan is the alternative
// or (above 32 tokens, where the alternative is a launch per matrix, 2.5 us each; at 64 the tensor-core kernel) close to it.
// Measured on B200 (us per call, before / this kernel, groups of 64 | 128 | one scale per channel):
//   16 tokens: 8192 x 8192 10.1 / 9.3 | 9.9 / 8.6 | 8.7 / 8.2; 28672 x 8192 21.9 stays | 21.3 stays | 19.9 / 17.3;
//   4096 x (14336 + 14336) 13.1 stays | 12.4 stays | 11.7 / 10.7; 2560 x 3840 7.5 / 3.7 | 7.3 / 3.5 | 7.1 / 3.6
//   24 tokens: 8192 x 8192 11.7 / 11.5 | 11.1 / 9.8 | 10.8 / 8.7; 8192 x (28672 + 28672) 49.4 stays | 44.5 stays |
//   44.2 / 34.8
//   32 tokens: 8192 x (8192 + 1024 + 1024) 16.1 stays | 15.2 / 15.1 | 14.3 / 12.7; 8192 x 8192 14.1 / 12.4 | 13.3 /
//   10.3 | 12.6 / 9.0; 8192 x (28672 + 28672) 62.9 stays | 58.1 / 44.3 | 55.4 / 35.6; 28672 x 8192 41.0 / 31.9 |
//   37.9 / 24.3 | 36.4 / 18.9
//   48 tokens: 8192 x 8192 17.1 / 16.2 | 16.0 / 12.3 | 15.1 / 10.9; 28672 x 8192 80.6 / 45.7 | 71.2 / 32.4 | 68.0 /
//   25.5
//   64 tokens: 4096 x 4096 10.0 stays | 10.8 / 7.8 | 9.8 / 7.3; 4096 x (14336 + 14336) 40.3 / 32.4 | 31.3 / 23.7 |
//   25.7 / 17.0; 8192 x (28672 + 28672) 135.4 / 115.7 | 103.2 / 82.4 | 76.5 / 54.8; 14336 x 4096 22.2 / 17.5 | 18.3
//   / 13.2 | 20.7 / 11.6
// Small launches stay where they were, by their number of 8 KB blocks: their alternatives are not what the estimate describes
// (us, before / this kernel: at 32 tokens 4096 x 4096, 512 blocks, 5.7 / 6.9 | 5.8 / 5.8 | 5.1 / 5.7; at 48 8.3 / 8.3 | 6.3 / 6.7;
// 2048 x 2048, 128 blocks, 3.2 / 5.2), and so does everything of up to 8 tokens (4096 x (14336 + 14336) 9.4 / 11.2).
// Rows of 1536 to 3840 values that the persistent kernel does not hold in registers leave it at 9 to 16 tokens, up to where
// the kernel with stationary activations has them (3840 x 47392, groups of 128, 11 tokens 15.7 / 18.9).
// Short rows stay too, below 1536 values with groups of 64 and below 2048 with groups of 128: a short row is summed no better here, and by
// the other kernels in more parts (1024 x 20928, groups of 128, 64 tokens: 5.1e-8 from sums in 64 bits, 5.6e-8 here).  At 64 tokens so do
// fewer than eight groups of 256 values and more, whose integers the tensor-core kernel never cuts, and groups of 128 with
// binary16 scales, whose products it adds without rounding for longer (8192 x 8192 3.8e-8, 4.0e-8 here).
// Of 4244 launches of random sets of matrices (9 to 64 tokens, groups of 64, 128, 1024 and one scale, some single
// matrices with binary16 scales) the rule moved 2337 here: their time fell by 1.49 on average (geometric), 23 took more
// than 1.5 % longer, 8 more than 5 %, 16 % at most; the distance from sums in 64 bits grew for 11 (binary16 scales in
// groups of 1024, or rows below 2048), by 2.7 % at most.
// W2A8_TSTREAM = 0 never, 2 whenever it supports the shape; any switch that forces a plan of another kernel keeps it out.
bool tstream_takes(int M, int K, int group, int tiles16, int count, bool h16) {
    if (!tstream_supported(M, K, group)) return false;
    const int mode = env_int("W2A8_TSTREAM", 1);
    if (mode == 0) return false;
    if (mode == 2) return true;
    if (M <= 8 || (group == 64 && K < 1536) || (group == 128 && K < 2048)) return false;
    if (M == 64 && ((group > 128 && group < K && K / group < 8) || (h16 && group == 128))) return false;
    const int KB = K / kBlockK, tiles = (tiles16 + 7) / 8, pairs = (tiles16 + 1) / 2;
    const long long blocks = (long long)tiles * KB;
    const long long least = M <= 32 ? (count > 1 && M > 24 ? 700 : 1536) : M <= 48 && count == 1 ? 1024 : 300;
    const bool odd_row = M <= 16 && !h16 && KB >= 6 && KB < 16 && KB != 8 && blocks >= 100 && (long long)pairs * KB < 12288;
    if (blocks < least && !odd_row) return false;
    if (env_int("W2A8_STAT", 1) == 2 || env_int("W2A8_GEMV", 1) == 2) return false;
    for (const char *name : {"W2A8_STAT_C", "W2A8_CHUNKS", "W2A8_TG", "W2A8_RING", "W2A8_MT", "W2A8_CLUSTER",
                             "W2A8_MIN_WARPS", "W2A8_RELAX"})
        if (env_set(name)) return false;
    if (M == 64)
        for (const char *name : {"W2A8_PREFILL", "W2A8_TC_KIND", "W2A8_PF_SPLIT", "W2A8_PF_KSPLIT", "W2A8_PF_WIDE"})
            if (env_set(name)) return false;
    if (odd_row && gemv_preferred(M, K, group, tiles16, count)) return true;
    if (blocks < least) return false;
    const int sms = sm_count(), per_sm = ts_tokens(M) <= 32 ? 2 : 1;
    int resident[kTsMaxCluster + 1] = {}, C, ncl;       // (what the device reports for a whole B200: 148, 74, 33, 15)
    for (int c = 1; c <= kTsMaxCluster; c *= 2) resident[c] = (int)(sms / c * (c == 4 ? 0.9 : c == 8 ? 0.84 : 1.0)) * per_sm;
    if (per_sm == 2) resident[8] = resident[8] * 3 / 4;
    const double mine = ts_plan(tiles, KB, resident, ts_times(M, group), &C, &ncl);
    double other = stat_estimate(M, K, group, pairs);
    if (other < 0) other = 4.6 + 1.0e-3 * (double)blocks * ((M + 7) / 8);
    if (M > 32) other += 2.5 * (count - 1);
    return mine < 0.95 * other;
}

template <int NT, int SPP, bool H16>
static cudaError_t launch_ts_inst(const TsMaps &maps, TsParams &p, cudaStream_t st) {
    using C = TsCfg<NT, SPP>;
    auto kernel = w2a8_tstream_kernel<NT, SPP, H16>;
    static PerDeviceFlags configured, carved;   // per kernel instantiation
    if (cudaError_t e = allow_dynamic_smem(kernel, configured, (int)C::kSmem)) return e;
    if (!carved.done[current_device()].load(std::memory_order_acquire)) {
        if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100)) return e;
        carved.done[current_device()].store(true, std::memory_order_release);
    }
    // Clusters of C CTAs that are resident at once.  The query answers for one CTA per SM; with 256 columns of tensor
    // memory, 112 KB and half of the registers two are resident (clusters of eight: about three quarters of that).
    static PerDeviceTable<kTsMaxCluster + 1> clusters;
    const int *resident = clusters.get(current_device(), [&](int *n) {
        for (int c = 1; c <= kTsMaxCluster; c *= 2) {
            const int found = C::kCtasPerSm * resident_clusters(kernel, c, C::kThreads, C::kSmem);
            n[c] = C::kCtasPerSm == 2 && c == 8 && found > 1 ? found * 3 / 4 : found;
        }
    });
    if (ts_plan(p.tiles, p.KB, resident, ts_times(p.M, SPP == 1 ? 64 : SPP == 2 ? 128 : 256), &p.C, &p.nclusters) > 1e29)
        return cudaErrorNotSupported;
    p.blk_per = p.KB / p.C; p.blk_extra = p.KB % p.C;
    return launch_kernel_clusters(kernel, dim3((unsigned)(p.nclusters * p.C)), dim3(C::kThreads), C::kSmem, st, pdl_enabled(),
                                  make_uint2((unsigned)p.C, 1u), maps, p);
}
template <int NT, bool H16>
static cudaError_t launch_ts_spp(const TsMaps &maps, TsParams &p, int spp, cudaStream_t st) {
    return spp == 1 ? launch_ts_inst<NT, 1, H16>(maps, p, st)
         : spp == 2 ? launch_ts_inst<NT, 2, H16>(maps, p, st)
         : p.G == 1 ? launch_ts_inst<NT, kTsRow, H16>(maps, p, st) : launch_ts_inst<NT, 0, H16>(maps, p, st);
}
template <bool H16>
static cudaError_t launch_ts_nt(const TsMaps &maps, TsParams &p, int spp, cudaStream_t st) {
    switch (ts_tokens(p.M)) {
        case 16: return launch_ts_spp<16, H16>(maps, p, spp, st);
        case 24: return launch_ts_spp<24, H16>(maps, p, spp, st);
        case 32: return launch_ts_spp<32, H16>(maps, p, spp, st);
        case 48: return launch_ts_spp<48, H16>(maps, p, spp, st);
        default: return launch_ts_spp<64, H16>(maps, p, spp, st);
    }
}

// Enqueue one launch over `count` matrices (1 .. 4) that share their activations.  kStatNoPlan: nothing was launched,
// because no cluster is resident (a small partition of a GPU).
int launch_tstream(const int8_t *a, const float *a_scale, int count, const uint32_t *const *packed,
                   const void *const *w_scale, void *const *y, const int *N, const int *ldy, int M, int K, int group,
                   void *workspace, cudaStream_t st, bool h16, bool y16) {
    if (count < 1 || count > kTsMaxMats || !tstream_supported(M, K, group)) return W2A8_ERR_SHAPE;
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return W2A8_ERR_CUDA;
    TsMaps maps = {};
    TsParams p = {};
    const cuuint32_t estr[2] = {1u, 1u};
    int tiles = 0;
    for (int i = 0; i < count; ++i) {
        tiles += (N[i] + kTsBM - 1) / kTsBM;
        p.mat[i].w_scale = w_scale[i]; p.mat[i].y = y[i]; p.mat[i].N = N[i]; p.mat[i].ldy = ldy[i]; p.mat[i].tile_end = tiles;
        const cuuint64_t dims[2] = {(cuuint64_t)(K / 16), (cuuint64_t)N[i]};
        const cuuint64_t strides[1] = {(cuuint64_t)(K / 4)};
        const cuuint32_t box[2] = {16u, (cuuint32_t)kTsBM};                    // 64 bytes x 128 channels
        if (encode(&maps.w[i], CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t *>(packed[i]), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return W2A8_ERR_CUDA;
    }
    {
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)M};
        const cuuint64_t strides[1] = {(cuuint64_t)K};
        const cuuint32_t box[2] = {128u, (cuuint32_t)((ts_tokens(M) + 15) / 16 * 16)};
        if (encode(&maps.act, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(a), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return W2A8_ERR_CUDA;
    }
    p.a_scale = a_scale; p.nmats = count; p.M = M; p.G = K / group; p.KB = K / kBlockK;
    p.bpg = group >= kBlockK ? group / kBlockK : 1;
    p.y16 = h16 && y16 ? 1 : 0;
    p.tiles = tiles;
    p.status = reinterpret_cast<int *>(workspace);
    p.polls = (unsigned)env_int("W2A8_TSTREAM_POLLS", (int)kPfWaitPolls);
    const int spp = group == 64 ? 1 : group == 128 ? 2 : 0;
    const cudaError_t e = h16 ? launch_ts_nt<true>(maps, p, spp, st) : launch_ts_nt<false>(maps, p, spp, st);
    return e == cudaSuccess ? W2A8_OK : e == cudaErrorNotSupported ? kStatNoPlan : W2A8_ERR_CUDA;
}

}  // namespace w2a8
