// Streaming kernel with stationary activations (up to a few hundred tokens): the weights stream past
// activations that stay in shared memory, and every weight is unpacked once per group of up to 64 tokens.
//
//  * Work.  A cluster of C CTAs owns a contiguous range of channel pairs (32 channels); rank r of it
//    owns the r-th share of the 256-k blocks (K-splitting of Sec. II-D) and keeps the activations of
//    that share in shared memory.  A "cell" is one pair x one block: 2 KB of packed weights plus its
//    scales.  A CTA's cells (pairs of a round x its blocks) are dealt to its warps as equal contiguous
//    runs, so no warp waits for a larger tile than its neighbour's; a pair cut between warps is summed
//    from its last part to its first, in place in one shared-memory slot (each warp adds what the next
//    one left there), and the ranks' slots are added in rank order through distributed shared memory.
//    All orders are fixed by the launch: results repeat bit for bit.
//  * Inner step: mma.sync m16n8k32 int8, the weight tile as the 16-row operand (w2a8_cell.cuh).  Two
//    tiles share each activation fragment, so a fragment is read from shared memory once per 32
//    channels.
//  * One CTA of 8 warps per SM with up to 255 registers: two warps per scheduler, but enough registers for
//    the compiler to keep many MMAs in flight.  Against two CTAs (128 registers) or 16 and 12 warps:
//    14336 x 4096 at 32 tokens 12.9 / 13.7 us, at 64 tokens 22.1 / 26.9; 8192 x (28672 + 28672) at 16 tokens
//    35.3 / 44.
//  * Bound.  32 tokens: the chain unpack - MMA - promotion inside a warp (583 warp instructions per cell, of which
//    64 MMAs, 128 packed promotions and 112 of unpack; with two warps per scheduler one issues every 3.2 clk: issue
//    slots 32 %, tensor pipe 28 % busy, ncu at 14336 x 4096); 64 tokens: the MMA pipe at half its rate (425 of 1190 TOPS with 2 warps
//    per scheduler); small problems: the 4 to 5 us that a launch costs beside the stream (a cold prologue, the
//    activations after the dependency wait, two cluster barriers).
#include "w2a8_cell.cuh"

namespace w2a8 {

bool gemv_preferred(int M, int K, int group, int tiles, int count);
bool gemv_half_sm(int M, int K);
bool one_shot_keeps(int M, int N, int K, int group, bool h16);
bool prefill_supported(int M, int N, int K, int group);
bool prefill_preferred(int M, int N, int K, int group, bool can_split);
size_t prefill_workspace_bytes(int M, int N, int K, int group);
double many_token_seconds(int M, int N, int K, int group);

constexpr int kStMaxMats = 4;
constexpr int kStWSlot = 4 * 32 * 16;         // weights of a cell: four channel rows per lane x 16 B
constexpr int kStSSlot = 32 * 16;             // its scales: 32 channels x 16 B
constexpr int kStSlot = kStWSlot + kStSSlot;
constexpr int kStMaxCluster = 8;

struct StMat {
    const uint32_t *packed;
    const void *w_scale;
    void *y;
    int pair_end;         // pairs of this matrix and of all before it
    int N;
    int ldy;
};

struct StParams {
    StMat mat[kStMaxMats];
    const int8_t *a;
    const float *a_scale;
    int nmats, M, K, G, blocks, words_per_row;
    int blocks_per_group;
    int C;                        // CTAs per cluster = shares of K
    int blk_per, blk_extra;       // rank r owns blk_per (+ 1 if r < blk_extra) blocks
    uint32_t nb_inv[2];           // ceil(65536 / n) for n = blk_per, blk_per + 1
    int pair_per, pair_extra;     // cluster c owns pair_per (+ 1 if c < pair_extra) pairs
    int round_pairs;              // pairs per round = sum slots
    int tgroups;                  // token groups of 8 * MT tokens; neighbouring clusters take the same pairs of different groups
    int y16;
    int s_wide;                   // scales are copied 16 bytes at a time (every row starts on a 16-byte boundary)
    int pairs;                    // (host)
};

__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t local, uint32_t rank) {
    uint32_t remote;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(remote) : "memory");
    return v;
}

constexpr int kStWarps = 8;

// MT: 8-token slabs of a token group; SPP: 64-k slices per scale group (capped at 4); H16: binary16
// scales; RING: landing slots (cells) per warp.
template <int MT, int SPP, bool H16, int RING>
__global__ void __launch_bounds__(kStWarps * 32, 1)
w2a8_stat_kernel(const __grid_constant__ StParams p) {
    constexpr int W = kStWarps, kThreads = W * 32;
    constexpr int SPB = 4 / SPP;                    // scales per block and channel
    constexpr int kActBlock = 8 * MT * 256;         // activations of one block in shared memory
    constexpr int kSlotFloats = MT * 2 * 32 * 4;    // sums of one pair
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float tok_scale[8 * MT];
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);
    const int gq = lane >> 2, t = lane & 3;
    const int C = p.C, rank = C > 1 ? (int)cluster_ctarank() : 0;
    int cl;
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(cl));
    int m_base = 0;                        // first token of this cluster's group
    if (p.tgroups > 1) { const int all = cl; cl = all / p.tgroups; m_base = (all - cl * p.tgroups) * (8 * MT); }
    const int mrows = min(8 * MT, p.M - m_base);
    // (shares computed on the host: a launch runs its prologue once, and divisions are long cold code)
    const int kb_lo = rank * p.blk_per + min(rank, p.blk_extra), nb = p.blk_per + (rank < p.blk_extra ? 1 : 0);
    const uint32_t nb_inv = rank < p.blk_extra ? p.nb_inv[1] : p.nb_inv[0];
    const int nb_max = p.blk_per + (p.blk_extra > 0 ? 1 : 0);
    // this cluster's pairs, in rounds of round_pairs
    const int pr_lo = cl * p.pair_per + min(cl, p.pair_extra), npairs = p.pair_per + (cl < p.pair_extra ? 1 : 0);

    unsigned char *ring = smem + warp * (RING * kStSlot);
    const uint32_t ring_u32 = smem_u32(ring);
    const uint32_t act_u32 = smem_u32(smem) + W * RING * kStSlot;
    float *sums = reinterpret_cast<float *>(smem + W * RING * kStSlot + nb_max * kActBlock);

    // matrix of a pair, and the pair's first channel there
    auto mat_of = [&](int pair, int &n0) -> int {
        int i = 0, first = 0;
#pragma unroll
        for (int j = 1; j < kStMaxMats; ++j)
            if (j < p.nmats && pair >= p.mat[j - 1].pair_end) { i = j; first = p.mat[j - 1].pair_end; }
        n0 = (pair - first) * 32;
        return i;
    };
    // this warp's run of cells in the round that starts at pair r0: [lo, hi) of pairs x blocks
    auto run_of = [&](int r0, int &lo, int &hi) {
        const int cells = min(p.round_pairs, npairs - r0) * nb;
        lo = cells * warp / W;
        hi = cells * (warp + 1) / W;
    };

    // ---- request side ------------------------------------------------------------------
    // A cursor over this warp's cells, ring slots ahead of the compute.  Everything that is not an
    // addition happens once per matrix or round.
    constexpr int kScaleStep = SPP == 4 ? 0 : SPB * (H16 ? 2 : 4);        // scale bytes from a block to the next
    const int row_bytes = p.words_per_row * 4;
    const char *q_w = nullptr, *q_s = nullptr;    // this lane's unit of the cell's first row; scales of channel `lane`
    int q_r0 = -p.round_pairs, q_pair = 0, q_kb = 0, q_left = 0, q_relocate = 0, q_second = 0;
    auto q_locate = [&]() {
        int n0;
        const int i = mat_of(q_pair, n0);
        const int N = p.mat[i].N;
        const bool two = n0 + 16 < N;                     // a matrix may end with half a pair: its tile again
        q_w = reinterpret_cast<const char *>(p.mat[i].packed) + (size_t)(n0 + gq) * row_bytes + 64 * (kb_lo + q_kb) + 16 * t;
        q_second = two ? 16 * row_bytes : 0;
        const int ch = n0 + (two ? lane : (lane & 15));
        q_s = reinterpret_cast<const char *>(p.mat[i].w_scale) + (size_t)ch * (p.G * (H16 ? 2 : 4)) + (kb_lo + q_kb) * kScaleStep;
        q_relocate = p.mat[i].pair_end - (two && (N & 16) ? 1 : 0);
    };
    auto q_next_round = [&]() {
        int c, hi;
        do {
            q_r0 += p.round_pairs;
            if (q_r0 >= npairs) return;
            run_of(q_r0, c, hi);
        } while (c == hi);
        q_left = hi - c;
        const int pi = (c * nb_inv) >> 16;
        q_kb = c - pi * nb;
        q_pair = pr_lo + q_r0 + pi;
        q_locate();
    };
    auto request = [&](int slot) {
        if (q_left == 0) return;
        const uint32_t dst = ring_u32 + slot * kStSlot + lane * 16;
        cp_async16(dst, q_w);
        cp_async16(dst + 512, q_w + 8 * row_bytes);
        cp_async16(dst + 1024, q_w + q_second);
        cp_async16(dst + 1536, q_w + q_second + 8 * row_bytes);
        const uint32_t sdst = dst + kStWSlot;
        if constexpr (SPP == 4) {
            const int gi = p.blocks_per_group >= p.blocks ? 0 : (kb_lo + q_kb) / p.blocks_per_group;
            if constexpr (H16) cp_async4(sdst, reinterpret_cast<const void *>(reinterpret_cast<uintptr_t>(q_s + 2 * gi) & ~(uintptr_t)3));
            else               cp_async4(sdst, q_s + 4 * gi);
        } else if constexpr (kScaleStep == 16) {          // whole blocks: a block's scales of a channel are one aligned unit
            cp_async16(sdst, q_s);
        } else if (p.s_wide) {
            // The 16 bytes around the block's scales, past L1: the rings leave it 28 KB, less than the lines that
            // the 8 x 32 rows in flight would hold, so pieces of 8 or 4 bytes (which can only go through L1) missed
            // it block after block (28672 x 8192, groups of 128: 24.8 / 17.5 us at 8 tokens, 38.9 / 37.8 at 32;
            // 8192 x 28672 at 32 33.1 / 32.4).  Small launches are ahead with the pieces (4096 x 14336 at 32 tokens
            // 10.97 / 11.12, 4096 x 4096 at 64 10.1 / 10.7): the host decides by the number of cells.
            cp_async16(sdst, reinterpret_cast<const void *>(reinterpret_cast<uintptr_t>(q_s) & ~(uintptr_t)15));
        } else if constexpr (kScaleStep == 8) {
            cp_async8(sdst, q_s);
        } else {
            cp_async4(sdst, q_s);
        }
        q_w += 64;
        q_s += kScaleStep;
        ++q_kb;
        if (--q_left == 0) {
            q_next_round();
        } else if (q_kb == nb) {
            q_kb = 0;
            ++q_pair;
            if (q_pair == q_relocate) {
                q_locate();
            } else {
                q_w += (size_t)32 * row_bytes - 64 * nb;
                q_s += (size_t)32 * (p.G * (H16 ? 2 : 4)) - nb * kScaleStep;
            }
        }
    };
    q_next_round();
    // weights and scales are frozen data: requested before the wait for the previous kernel
#pragma unroll 1
    for (int r = 0; r < RING - 1; ++r) {
        request(r);
        cp_async_commit();
    }
    pdl_launch_dependents();
    pdl_wait();

    // ---- activations of this CTA's blocks ------------------------------------------------
    // [block][token][256 B], the 64-byte slices of odd rows swapped in pairs so that the eight lanes of
    // a fragment load's phase hit different banks.  Rows past the last token are left as they are: token
    // columns of an MMA are independent, and those columns are never stored.
    {
        const int ch = (threadIdx.x & 15) * 16;
        int m = threadIdx.x >> 4, kb = 0;
        for (;;) {
            while (m >= mrows) { m -= mrows; ++kb; }
            if (kb >= nb) break;
            cp_async16(act_u32 + kb * kActBlock + m * 256 + (ch ^ ((m & 1) << 6)),
                       p.a + (size_t)(m_base + m) * p.K + (kb_lo + kb) * kBlockK + ch);
            m += kThreads / 16;
        }
    }
    cp_async_commit();
    if (threadIdx.x < 8 * MT) tok_scale[threadIdx.x] = p.a_scale[m_base + min((int)threadIdx.x, mrows - 1)] * (1.0f / kCodeGain);
    cp_async_wait_all();
    __syncthreads();
    const uint32_t b_even = act_u32 + gq * 256 + t * 16 + ((gq & 1) << 6), b_odd = b_even - ((gq & 1) << 7);

    // Constants of the inner step as opaque registers: as literals they are written anew for many of
    // the instructions that read them.
    int magic[4];
    unsigned long long minus_magic;
    uint32_t mask, flip;
    asm volatile("mov.b32 %0, %4;\n\tmov.b32 %1, %4;\n\tmov.b32 %2, %4;\n\tmov.b32 %3, %4;"
                 : "=r"(magic[0]), "=r"(magic[1]), "=r"(magic[2]), "=r"(magic[3]) : "n"(kMagicInt));
    asm volatile("mov.b64 %0, {%1, %1};" : "=l"(minus_magic) : "f"(-kMagicFloat));
    asm volatile("mov.b32 %0, 0xC0C0C0C0;\n\tmov.b32 %1, 0x80808080;" : "=r"(mask), "=r"(flip));
    // lane_codes; j is a constant after unrolling
    auto codes = [&](uint32_t word, int j) -> uint32_t {
        const uint32_t x = j == 3 ? word : word << (6 - 2 * j);
        uint32_t r;
        asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(r) : "r"(x), "r"(mask), "r"(flip));
        return r;
    };
    // (acc0, acc1) += sc * (float(d0), float(d1)), as promote2
    auto promote = [&](float &acc0, float &acc1, int d0, int d1, float sc) {
        asm("{\n\t.reg .b64 a, b, c;\n\t"
            "mov.b64 a, {%2, %3};\n\t"
            "add.rn.f32x2 a, a, %5;\n\t"
            "mov.b64 b, {%4, %4};\n\t"
            "mov.b64 c, {%0, %1};\n\t"
            "fma.rn.f32x2 c, a, b, c;\n\t"
            "mov.b64 {%0, %1}, c;\n\t}"
            : "+f"(acc0), "+f"(acc1) : "r"(d0), "r"(d1), "f"(sc), "l"(minus_magic));
    };

    // ---- compute side --------------------------------------------------------------------
    int slot = 0, pslot = RING - 1;
    bool reading = false;                  // a cluster barrier phase (everybody has read the sums) is open
    for (int r0 = 0; r0 < npairs; r0 += p.round_pairs) {
        const int round_n = min(p.round_pairs, npairs - r0);
        int c, hi;
        run_of(r0, c, hi);
        int pi = (c * nb_inv) >> 16, kb0 = c - pi * nb;
        while (c < hi) {
            const int kb1 = min(nb, kb0 + hi - c);
            float acc[2][MT][4];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][mt][j] = 0.f;
#pragma unroll 1
            for (int kb = kb0; kb < kb1; ++kb) {
                // the slot consumed in the previous step is free: refill it, then wait for this one
                __syncwarp();
                request(pslot);
                cp_async_commit();
                cp_async_wait_group<RING - 1>();
                __syncwarp();                                   // the scales were copied by other lanes
                const unsigned char *sl = ring + slot * kStSlot;
                pslot = slot;
                slot = slot + 1 == RING ? 0 : slot + 1;
                uint32_t w[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(sl + i * 512 + lane * 16);
                    w[i][0] = v.x; w[i][1] = v.y; w[i][2] = v.z; w[i][3] = v.w;
                }
                uint32_t odd_scale = 0;
                if constexpr (H16 && SPP == 4) {
                    // the copied word starts at an even scale; the wanted one may be its second half
                    int n0;
                    const int mi = mat_of(pr_lo + r0 + pi, n0);
                    const int gi = p.blocks_per_group >= p.blocks ? 0 : (kb_lo + kb) / p.blocks_per_group;
                    const int tile = n0 + 16 < p.mat[mi].N ? 16 : 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        odd_scale |= (((n0 + (i >> 1) * tile + (i & 1) * 8 + gq) * p.G + gi) & 1) << i;
                }
                // the block's scales inside their slot (whole 16 bytes: groups of 64, fp32)
                const int s_off = SPP == 4 || kScaleStep == 16 || !p.s_wide ? 0 : ((kb_lo + kb) * kScaleStep) & 15;
                // scale of slice s for rows gq, gq + 8 of both tiles (i = 0 .. 3)
                auto scale = [&](int i, int s) -> float {
                    const unsigned char *ss = sl + kStWSlot + (i * 8 + gq) * 16 + s_off;
                    if constexpr (!H16)          return reinterpret_cast<const float *>(ss)[s / SPP];
                    else if constexpr (SPP != 4) return __half2float(reinterpret_cast<const __half *>(ss)[s / SPP]);
                    else                         return __half2float(reinterpret_cast<const __half *>(ss)[(odd_scale >> i) & 1]);
                };
                const uint32_t be = b_even + kb * kActBlock, bo = b_odd + kb * kActBlock;
                // Slices are taken S at a time (a group, or half of a larger group: a promotion costs less than
                // accumulators that outlive the unpacked weights).
                constexpr int S = SPP == 1 ? 1 : 2;
#pragma unroll
                for (int s0 = 0; s0 < 4; s0 += S) {
                    uint32_t A[S][2][8];
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                A[s][i][2 * j] = codes(w[2 * i][s0 + s], j);
                                A[s][i][2 * j + 1] = codes(w[2 * i + 1][s0 + s], j);
                            }
                    float sc[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) sc[i] = scale(i, s0);
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        int D[2][4];
#pragma unroll
                        for (int s = 0; s < S; ++s) {
                            uint4 B;
                            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(B.x), "=r"(B.y), "=r"(B.z), "=r"(B.w)
                                         : "r"((((s0 + s) & 1) ? bo : be) + mt * 2048 + (s0 + s) * 64));
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const uint32_t (&a)[8] = A[s][i];
                                if (s == 0) mma_s8_16x8x32_pure(D[i], a[0], a[1], a[2], a[3], B.x, B.y, magic);
                                else        mma_s8_16x8x32_pure(D[i], a[0], a[1], a[2], a[3], B.x, B.y, D[i]);
                                mma_s8_16x8x32_pure(D[i], a[4], a[5], a[6], a[7], B.z, B.w, D[i]);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            promote(acc[i][mt][0], acc[i][mt][1], D[i][0], D[i][1], sc[2 * i]);
                            promote(acc[i][mt][2], acc[i][mt][3], D[i][2], D[i][3], sc[2 * i + 1]);
                        }
                    }
                }
            }
            // ---- this part of the pair: add what the following parts left, leave the sum -------
            if (reading) { cluster_wait(); reading = false; }   // the slots of the previous round have been read
            float4 *dst = reinterpret_cast<float4 *>(sums + pi * kSlotFloats) + lane;
            c += kb1 - kb0;
            if (kb1 < nb) {
                int next = warp + 1;                                      // the warp that has the next cell
                while (round_n * nb * (next + 1) / W <= c) ++next;
                asm volatile("bar.sync %0, 64;" ::"r"(next) : "memory");
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        const float4 v = dst[(mt * 2 + i) * 32];
                        acc[i][mt][0] += v.x; acc[i][mt][1] += v.y; acc[i][mt][2] += v.z; acc[i][mt][3] += v.w;
                    }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    dst[(mt * 2 + i) * 32] = make_float4(acc[i][mt][0], acc[i][mt][1], acc[i][mt][2], acc[i][mt][3]);
            if (kb0 > 0) {
                __syncwarp();
                asm volatile("bar.arrive %0, 64;" ::"r"(warp) : "memory");
            }
            ++pi;
            kb0 = 0;
        }
        __syncwarp();
        if (reading) { cluster_wait(); reading = false; }
        // ---- the round's outputs: ranks in order, token scale, store ----------------------
        if (C > 1) cluster_sync(); else __syncthreads();
        const uint32_t sums_u32 = smem_u32(sums) + lane * 16;
        // one (pair, slab, tile) per warp and step: everything but the loads and stores is warp-uniform
        for (int q = rank * W + warp; q < round_n * (MT * 2); q += C * W) {
            float4 part[kStMaxCluster];
#pragma unroll
            for (int k = 0; k < kStMaxCluster; ++k)
                part[k] = k < C ? ld_cluster_f32x4(sums_u32 + q * 512, k) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 v = part[0];
#pragma unroll
            for (int k = 1; k < kStMaxCluster; ++k) { v.x += part[k].x; v.y += part[k].y; v.z += part[k].z; v.w += part[k].w; }
            const int i = q & 1, mt = (q >> 1) % MT, pj = (q >> 1) / MT;
            int n0;
            const int mi = mat_of(pr_lo + r0 + pj, n0);
            if (n0 + i * 16 < p.mat[mi].N) {
                const size_t ldy = p.mat[mi].ldy;
                const int m = mt * 8 + 2 * t;
                const size_t at = (size_t)(m_base + m) * ldy + n0 + i * 16 + gq;
                const float s0 = tok_scale[m], s1 = tok_scale[m + 1];
                if (H16 && p.y16) {
                    __nv_bfloat16 *y = reinterpret_cast<__nv_bfloat16 *>(p.mat[mi].y) + at;
                    if (m < mrows) { y[0] = __float2bfloat16_rn(v.x * s0); y[8] = __float2bfloat16_rn(v.z * s0); }
                    if (m + 1 < mrows) { y[ldy] = __float2bfloat16_rn(v.y * s1); y[ldy + 8] = __float2bfloat16_rn(v.w * s1); }
                } else {
                    float *y = reinterpret_cast<float *>(p.mat[mi].y) + at;
                    if (m < mrows) { y[0] = v.x * s0; y[8] = v.z * s0; }
                    if (m + 1 < mrows) { y[ldy] = v.y * s1; y[ldy + 8] = v.w * s1; }
                }
            }
        }
        __syncwarp();
        if (C > 1) { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); reading = true; }
        else __syncthreads();
    }
    if (reading) cluster_wait();           // nobody leaves while its sums may be read
}

// ---- host side -----------------------------------------------------------------------
constexpr size_t kStBudget = 225 * 1024;      // dynamic shared memory per CTA
constexpr int st_ring(int mt) { return mt <= 2 ? 4 : mt <= 4 ? 3 : 2; }
// Token groups and slabs per group: groups of at most 64 tokens, all of the same width.
static int st_tgroups(int M) { return (M + 63) / 64; }
static int st_slabs(int M) { return ((M + 7) / 8 + st_tgroups(M) - 1) / st_tgroups(M); }

static bool stat_supported(int M, int K, int group) {
    if (K % kBlockK != 0 || M < 1 || st_tgroups(M) > 16) return false;
    // the activations of an eighth of K have to fit beside the rings and one slot of sums
    const int mt = st_slabs(M), nb = (K / kBlockK + kStMaxCluster - 1) / kStMaxCluster;
    const size_t budget = kStBudget;
    if ((size_t)kStWarps * st_ring(mt) * kStSlot + (size_t)nb * mt * 2048 + mt * 1024 > budget) return false;
    return group == 64 || group == 128 || group % 256 == 0;
}

// Whether the kernel takes a launch over `count` matrices of `tiles` 16-channel tiles in all.  Measured on
// B200 (us per GEMM call, group 64, back to back over rotating weight copies; before / this kernel):
//   1 .. 4 tokens: only matrices of the size of the 70B layer's, where the shorter prologue of the other
//     kernels no longer counts: 28672 x 8192 17.7 / 16.8 at 1 token, 22.2 / 17.4 at 4; 8192 x (28672 + 28672)
//     31.5 / 30.2 at 3 (groups of 128 32.2 / 27.6, one scale 28.5 / 24.7), but 28.7 / 29.4 at 1; 8192 x 8192 7.1 / 7.2,
//     q|k|v 8192 x 10240 8.8 / 9.0.  Binary16 scales: 8192 x 28672 21.5 / 16.2 at 1, 23.5 / 16.3 at 4; 8192 x 8192
//     6.6 / 6.9, 4096 x 14336 5.2 / 6.1.
//   5 .. 8 tokens: 8192 x (28672 + 28672) 36.0 / 30.9, 28672 x 8192 23.0 / 18.3, 8192 x (10240 + 1024 + 1024) 10.3 / 9.8;
//     but 14336 x 4096 7.8 / 8.6, gate|up 4096 x (14336 + 14336) 9.0 / 11.0, 8192 x (8192 + 1024 + 1024) 8.9 / 9.45 (groups of
//     128 9.0 / 9.0, one scale 8.5 / 8.0).  Against the persistent kernel in its two-CTAs-per-SM form, 5120 x (8192 +
//     8192) at 6 tokens: 8.3 / 9.3, of 128 8.0 / 9.1, one scale 7.8 / 7.7; 5120 x (14336 + 14336) 13.1 / 13.0;
//   9 .. 16 tokens: gate|up 13.9 / 13.0, 8192 x 8192 10.6 / 9.7, 8192 x (28672 + 28672) 65.2 / 35.3,
//     28672 x 8192 29.9 / 21.8; but 4096 x 14336 8.3 / 8.8, 14336 x 4096 9.5 / 9.7.  Where only the one-shot
//     kernel is left (binary16 scales): 4096 x 14336 9.9 / 8.2, 14336 x 4096 11.1 / 9.6, 4096 x 4096 4.1 / 4.9.
//   17 .. 32 tokens: 4096 x 14336 12.7 / 9.8, 14.7 / 11.9; gate|up 25.5 / 15.7, 29.3 / 18.9; 14336 x 4096
//     16.5 / 10.7, 17.3 / 12.9; 8192 x (28672 + 28672) 127 / 49, 133 / 63; but 4096 x 4096 4.9 / 5.5, 5.6 / 6.9:
//     a launch costs 4 to 5 us beside the stream, so small problems stay where they were, unless the
//     alternative is a launch per matrix (q|k|v 4096 x 6144 12.0 / 8.7).
//   33 .. 64 tokens: 4096 x 4096 8.8 / 7.2, 11.8 / 9.9; 4096 x 14336 20.6 / 13.5, 27.9 / 20.3; 14336 x 4096
//     29.1 / 14.6, 34.4 / 22.1; 8192 x 8192 29.1 / 16.1, 37.2 / 23.5.  But where the one-shot kernel has all its CTAs resident
//     at once it stays: 4096 x 4096 at 48 tokens 6.1 / 7.7 (groups of 128) and 5.9 / 7.5 (one scale), 2560 x 4096 4.4 / 7.4,
//     8192 x 2048 at 40 6.9 / 8.6; and on short rows, 2048 x 5120 at 48 5.6 / 6.8 (not 2560 x 3840, whose K it splits over
//     two waves of CTAs: 9.9 / 6.7).  At 64 tokens the tensor-core
//     kernel takes what the estimate below gives it: 14336 x 4096 18.9 / 22.7 (128), 4096 x 14336 13.4 / 18.9 (one scale),
//     8192 x 28672 40.1 / 63.8 (one scale), 52.3 / 66.2 (128); but not on a K split that needs more than the fixed scratch of
//     w2a8_gemm_static, 14336 x 5120 (128) 32.0 / 31.5.
//   64 .. 256 tokens: about 5 us + 0.27 ns per cell and slab (a little more for K > 8192, where clusters of six
//     and eight leave SMs idle), against the model of the tensor-core kernels: 4096 x 4096 at 100 tokens
//     13.1 / 12.5, 4096 x 14336 at 140 40.6 / 38.1, but at 100 22.0 / 31.1 and at 200 40.6 / 56.4, 14336 x 4096 at 140
//     39.6 / 46.1.
// W2A8_STAT = 0 never, 2 whenever it supports the shape; any switch that forces a plan of another kernel
// keeps it out.
bool stat_takes(int M, int K, int group, int tiles, int count, bool h16) {
    if (!stat_supported(M, K, group)) return false;
    const int mode = env_int("W2A8_STAT", 1);
    if (mode == 0) return false;
    if (mode == 2) return true;
    if (M > 256) return false;
    for (const char *name : {"W2A8_CHUNKS", "W2A8_TG", "W2A8_RING", "W2A8_MT", "W2A8_CLUSTER", "W2A8_MIN_WARPS",
                             "W2A8_RELAX"})
        if (env_set(name)) return false;
    if (env_int("W2A8_GEMV", 1) == 2) return false;
    const long long blocks = K / kBlockK, cells = (long long)((tiles + 1) / 2) * blocks;
    if (M <= 4) return cells >= 24576 && (h16 || blocks > (M == 1 ? 64 : 16));
    if (M <= 8) {
        const long long least = group <= 128 && gemv_half_sm(M, K) ? 16384 : group <= 64 ? 12288 : 8192;
        return gemv_preferred(M, K, group, tiles, count) && blocks > 16 && cells >= least;
    }
    if (M <= 16 && !h16 && gemv_preferred(M, K, group, tiles, count)) return cells >= (blocks > 16 ? 8192 : 12288);
    if (M <= 32) return cells >= (count > 1 ? 1536 : 4096);
    if (count > 1) return false;                  // (more than 32 tokens: a launch per matrix)
    if (M >= 64)
        for (const char *name : {"W2A8_PREFILL", "W2A8_TC_KIND", "W2A8_PF_SPLIT", "W2A8_PF_KSPLIT", "W2A8_PF_WIDE"})
            if (env_set(name)) return false;
    const bool tensor_cores = M >= 64 && prefill_supported(M, tiles * 16, K, group) &&
                              prefill_preferred(M, tiles * 16, K, group, true) &&
                              (M > 64 || prefill_workspace_bytes(M, tiles * 16, K, group) <= W2A8_STATIC_SCRATCH_BYTES);
    if (M < 64 || (M == 64 && !tensor_cores))
        return cells >= 1024 && !one_shot_keeps(M, tiles * 16, K, group, h16);
    const double mine = 5.0e-6 + 0.27e-9 * (blocks > 32 ? 1.15 : 1.0) * (double)cells * st_tgroups(M) * st_slabs(M);
    return mine < 0.95 * many_token_seconds(M, tiles * 16, K, group);
}

struct StPlan { int C, round_pairs, nclusters; size_t smem; };

// The plan: C, pairs per round.  One cell of one warp is the unit of cost.  (C = 2 is ahead of 4 at equal
// cells per warp: gate|up of the 8B layer 19.3 / 21.9 us at 32 tokens, 13.4 / 14.2 at 16.)
static bool stat_plan(int M, int K, int pairs, const int *resident, StPlan *out) {
    StPlan pl = {};
    const int mt = st_slabs(M), w = kStWarps, blocks = K / kBlockK, tg = st_tgroups(M);
    const size_t budget = kStBudget;
    const size_t slot_bytes = (size_t)mt * 1024, act_block = (size_t)mt * 2048;
    const int forced = env_int("W2A8_STAT_C", 0);
    double best = 1e30;
    for (int C = 1; C <= kStMaxCluster && C <= blocks; ++C) {
        if (forced > 0 && C != forced) continue;
        const int nb = (blocks + C - 1) / C;
        const size_t fixed = (size_t)w * st_ring(mt) * kStSlot + nb * act_block;
        if (fixed + slot_bytes > budget) continue;
        int ncl = resident[C] / tg;                       // clusters per token group
        if (ncl < 1) continue;
        if (ncl > pairs) ncl = pairs;
        const int per = (pairs + ncl - 1) / ncl;
        int cap = (int)((budget - fixed) / slot_bytes);
        while (cap > 1 && (long long)cap * nb * nb >= 65536) --cap;      // (the kernel divides by nb with a 16-bit reciprocal)
        const int rounds = (per + cap - 1) / cap, rp = (per + rounds - 1) / rounds;
        double cost = 0;
        for (int r = 0; r < rounds; ++r) cost += ((r + 1 < rounds ? rp : per - rp * (rounds - 1)) * nb + w - 1) / w;
        cost += 0.7 * rounds + 0.05 * nb * mt / 4.0 + 0.4 * C;
        if (cost < best) {
            best = cost;
            pl.C = C; pl.round_pairs = rp; pl.nclusters = ncl;
            pl.smem = fixed + rp * slot_bytes;
        }
    }
    *out = pl;
    return best < 1e29;
}

// Estimated time of a launch on a whole B200 in us, from its plan: a start, rounds, ranks, and cells of one warp (up to 64
// tokens; 1260 launches of random matrices at 9 to 63 tokens, groups of 64, 128 and one scale: 7 % rms).  Negative: no plan.
double stat_estimate(int M, int K, int group, int pairs) {
    static const int resident[kStMaxCluster + 1] = {0, 148, 74, 45, 33, 26, 22, 20, 15};
    StPlan pl;
    if (!stat_supported(M, K, group) || !stat_plan(M, K, pairs, resident, &pl)) return -1.0;
    const int nb = (K / kBlockK + pl.C - 1) / pl.C, per = (pairs + pl.nclusters - 1) / pl.nclusters;
    const int rounds = (per + pl.round_pairs - 1) / pl.round_pairs;
    int cells = 0;
    for (int r = 0; r < rounds; ++r)
        cells += ((r + 1 < rounds ? pl.round_pairs : per - pl.round_pairs * (rounds - 1)) * nb + kStWarps - 1) / kStWarps;
    const double a = group == 64 ? 0.089 : group == 128 ? 0.072 : 0.113, b = group == 64 ? 0.273 : group == 128 ? 0.249 : 0.2335;
    return 2.15 + 1.18 * rounds + 0.364 * pl.C + cells * (a + b * st_slabs(M));
}

template <int MT, int SPP, bool H16>
static cudaError_t launch_stat_inst(StParams &p, cudaStream_t st) {
    auto kernel = w2a8_stat_kernel<MT, SPP, H16, st_ring(MT)>;
    constexpr size_t budget = kStBudget;
    static PerDeviceFlags configured;   // per kernel instantiation
    if (cudaError_t e = allow_dynamic_smem(kernel, configured, (int)budget)) return e;
    // Clusters of C CTAs that are resident at once (clusters are placed inside one GPC, so the count is not
    // slots / C: 74, 45, 33, 26, 22, 15 for C = 2, 3, 4, 5, 6, 8).  A larger grid would run a second wave of a few clusters.
    static PerDeviceTable<kStMaxCluster + 1> clusters;
    const int *resident = clusters.get(current_device(), [&](int *n) {
        for (int C = 1; C <= kStMaxCluster; ++C) {
            const int found = resident_clusters(kernel, C, kStWarps * 32, budget);
            n[C] = found > 0 ? found : sm_count() / C;
        }
    });
    StPlan pl;
    if (!stat_plan(p.M, p.K, p.pairs, resident, &pl)) return cudaErrorNotSupported;
    p.C = pl.C; p.round_pairs = pl.round_pairs;
    p.blk_per = p.blocks / pl.C; p.blk_extra = p.blocks % pl.C;
    for (int i = 0; i < 2; ++i) p.nb_inv[i] = (65536 + p.blk_per + i - 1) / (p.blk_per + i);
    p.tgroups = st_tgroups(p.M);
    p.pair_per = p.pairs / pl.nclusters; p.pair_extra = p.pairs % pl.nclusters;
    return launch_kernel_clusters(kernel, dim3(pl.nclusters * p.tgroups * pl.C), dim3(kStWarps * 32), pl.smem, st, pdl_enabled(),
                                  make_uint2((unsigned)pl.C, 1u), p);
}
template <int MT, bool H16>
static cudaError_t launch_stat_spp(StParams &p, int spp, cudaStream_t st) {
    return spp == 1 ? launch_stat_inst<MT, 1, H16>(p, st)
         : spp == 2 ? launch_stat_inst<MT, 2, H16>(p, st) : launch_stat_inst<MT, 4, H16>(p, st);
}
template <bool H16>
static cudaError_t launch_stat_mt(StParams &p, int spp, cudaStream_t st) {
    switch (st_slabs(p.M)) {
        case 1: return launch_stat_spp<1, H16>(p, spp, st);
        case 2: return launch_stat_spp<2, H16>(p, spp, st);
        case 3: return launch_stat_spp<3, H16>(p, spp, st);
        case 4: return launch_stat_spp<4, H16>(p, spp, st);
        case 5: return launch_stat_spp<5, H16>(p, spp, st);
        case 6: return launch_stat_spp<6, H16>(p, spp, st);
        case 7: return launch_stat_spp<7, H16>(p, spp, st);
        default: return launch_stat_spp<8, H16>(p, spp, st);
    }
}

// Enqueue one launch over `count` matrices (1 .. 4) that share their activations.  kStatNoPlan: nothing was launched,
// because no cluster size holds the activations and is resident for every token group (a small partition of a GPU,
// or a forced W2A8_STAT_C); how many clusters are resident is only known here, with a context.
int launch_stat(const int8_t *a, const float *a_scale, int count, const uint32_t *const *packed,
                const void *const *w_scale, void *const *y, const int *N, const int *ldy, int M, int K, int group,
                cudaStream_t st, bool h16, bool y16) {
    if (count < 1 || count > kStMaxMats) return W2A8_ERR_SHAPE;
    ShapeInfo si;
    if (!shape_ok(M, N[0], K, group, &si)) return W2A8_ERR_SHAPE;
    StParams p = {};
    int pairs = 0;
    for (int i = 0; i < count; ++i) {
        pairs += (N[i] + 31) / 32;
        p.mat[i].packed = packed[i]; p.mat[i].w_scale = w_scale[i]; p.mat[i].y = y[i];
        p.mat[i].pair_end = pairs; p.mat[i].N = N[i]; p.mat[i].ldy = ldy[i];
    }
    p.a = a; p.a_scale = a_scale; p.nmats = count; p.M = M; p.K = K; p.G = si.G; p.blocks = si.blocks;
    p.words_per_row = si.words_per_row; p.blocks_per_group = (group + kBlockK - 1) / kBlockK;
    p.pairs = pairs;
    p.s_wide = (si.G * (h16 ? 2 : 4)) % 16 == 0 && (long long)pairs * si.blocks >= 12288;
    for (int i = 0; i < count; ++i)
        if (reinterpret_cast<uintptr_t>(w_scale[i]) % 16 != 0) p.s_wide = 0;
    p.y16 = y16 ? 1 : 0;
    const cudaError_t e = h16 ? launch_stat_mt<true>(p, si.spp, st) : launch_stat_mt<false>(p, si.spp, st);
    return e == cudaSuccess ? W2A8_OK : e == cudaErrorNotSupported ? kStatNoPlan : W2A8_ERR_CUDA;
}

}  // namespace w2a8
