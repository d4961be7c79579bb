// Batched decode of up to 32 sequences with per-sequence masks in ONE pass over the layer (16-bit layers):
//   h[b, j] = keep(b, j) * z(w_gate_j . x_b, w_up_j . x_b),   y_b = sum_j h[b, j] * w_down_j,   keep(b, j) = (A_bj >= tau_b)
// (Algorithm 2's masked FFN for every sequence of the batch).  With eight or more sequences that cut 40-50 % each,
// the union of the kept sets is the whole layer, so the layer is streamed densely, every row once, and the masks
// only zero entries of h.  Both contractions run on the 5th-generation tensor cores with the weights as the A
// operand (128 TMEM lanes) and the sequences as the N = 16 or 32 (SEQS) columns:
//
//   phase 1   D1[neuron, b] = W_gate/up[neuron, :] . x_b          A = weight rows (K-major), B = x (K-major),
//             K = d_model in blocks of 64 columns, four interleaved K splits in separate TMEM columns (short
//             accumulation chains), summed by the epilogue in fp32.
//   h         one epilogue thread per neuron: gate / up of its sequences from TMEM, neuron value, keep bits from
//             the score vectors, and h split into three 16-bit parts (h = h1 + h2 + h3), because the second
//             contraction takes 16-bit operands and y is held to 1e-5.  bf16 parts hold all of fp32's bits; fp16 parts
//             end at 65504 (beyond: NaN) and at 3e-8, so a small h of an fp16 layer loses bits (1e-4: 3e-4 of it).
//   phase 2   D2[column, (part, b)] = sum_j W_down_t[j, column] * h_part[b, j]   A = down rows as they lie in memory
//             (MN-major: columns contiguous), B = the three parts of h as 3 SEQS rows (K-major): ONE instruction of
//             N = 48 / 96 per 16 neurons and 128 columns, the three column groups added by the epilogue.  A member's
//             column tiles go through the tensor memory in equal sets of at most 512 / (3 SEQS) tiles; a tile of the
//             next set waits until the epilogue has read the tile whose columns it takes.
//
// Bound by HBM: every weight byte once per launch (13B layer: 425 MB = 65 us at the copy rate).  17-32 sequences as
// one launch of 32 columns instead of two of 16: the weights are read once instead of twice, at the price of twice
// the x tile and h image in shared memory (five ring stages instead of seven at 13824 neurons).
// Between the phases HBM has only the ring to fill, so h (two warps per quarter of the lanes), its exchange (all loads
// of a thread in flight together, rows of absent sequences left out) and the final sums (equal runs for every CTA,
// nineteen loads in flight) are kept short.  A call measured, as two launches or one of 16 columns at first / now: 32
// sequences of a 13B layer 153.7 / 80.3 us, 16 of it 77.2 / 74.9, 6 of 4096 x 14336 67.9 / 64.8, 6 of 5120 x 4100 62.6 /
// 61.0, 24 of 1024 x 4100 46.2 / 24.0 (whole steps, with cognitive load: 8 of 4096 x 14336 69.5, 32 of the 13B layer 95.4).
// Asking phase 2's boxes into L2 meanwhile (cp.async.bulk.prefetch.tensor, 8 to 48 stages) cost
// 2.5 to 8 us: the requests are paid for twice.
//
// Work split: 4 CTAs that begin one after another form a group.  Member m of group g streams the gate / up rows of its own
// rows_blk neurons (phase 1), the four members exchange their parts of h through global memory (each writes its
// slice of the operand image, a byte counter per group in the control block, bounded wait; the producer keeps
// prefetching meanwhile), and in phase 2 member m streams column slice m (a quarter of d_model) of the down rows
// of all four members' neurons, column tile by column tile, so that a finished tile's partial output is stored
// while the next tile streams.  Every weight byte is read once, and a group writes ONE partial output
// [B, d_model] instead of one per CTA.  After the CTAs have met (grid_meet) all threads sum the groups' partials in group order
// and write y.
//
// One persistent CTA per SM, 320 threads: warp 0 TMA producer (64-column boxes of rows_blk rows, 128-byte swizzle,
// mbarrier ring), warp 1 TMEM allocation + MMA issue from one thread, warps 2-9 epilogues.  Every wait is bounded;
// on expiry the CTA raises CLADA_STATUS_TIMEOUT, drains its copies and frees its tensor memory.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "ffn_batch.cuh"
#include "ffn_common.cuh"
#include "tc_common.cuh"

namespace clada {

constexpr int kBdEpi = 256;          // epilogue threads: two warps per quarter of the TMEM lanes, half the sequences each
constexpr int kBdThreads = 64 + kBdEpi;
constexpr int kBdMembers = 4;        // CTAs per group = column slices of phase 2
constexpr int kBdKSplit = 4;         // interleaved K splits of phase 1
constexpr int kBdMaxStages = 8;
constexpr int kBdMaxRows = 128;      // neurons per CTA (TMEM lanes)
constexpr int kBdMaxTiles = 16;      // 128-column tiles per member (kMaxDModel columns)
constexpr int kBdParts = 3;          // 16-bit parts of h
constexpr uint32_t kBdTmemCols = 512;
// bytes of a 64-neuron block of the h image: (parts x sequences) rows of 128 bytes
__host__ __device__ constexpr uint32_t bd_img_block(int seqs) { return (uint32_t)(kBdParts * seqs) * 128u; }
// column tiles whose partial outputs (parts x sequences columns each) fit the tensor memory together
constexpr int bd_tiles_in_tmem(int seqs) { return (int)kBdTmemCols / (kBdParts * seqs); }
constexpr int kBdGroupWord0 = 8;     // group byte counters: control-block words 8..63
constexpr int kBdMaxGroups = 4 * (64 - kBdGroupWord0);
constexpr size_t kBdSmemMin = 120 * 1024;

// Opt-in timeline (-DCLADA_BD_TRACE): %globaltimer stamps per CTA, 64 slots, written by the thread that passes the point.
#ifdef CLADA_BD_TRACE
__device__ unsigned long long *g_bd_trace = nullptr;  // [n_ctas][64]
#define BD_TRACE(slot)                                                \
    do {                                                              \
        if (g_bd_trace) {                                             \
            unsigned long long t_;                                    \
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_));     \
            g_bd_trace[(size_t)blockIdx.x * 64 + (slot)] = t_;        \
        }                                                             \
    } while (0)
#define BD_CLOCK(slot)                                                           \
    do {                                                                         \
        if (g_bd_trace) g_bd_trace[(size_t)blockIdx.x * 64 + (slot)] = clock64(); \
    } while (0)
#else
#define BD_TRACE(slot) \
    do {               \
    } while (0)
#define BD_CLOCK(slot) \
    do {               \
    } while (0)
#endif

struct BdParams {
    int d_model, d_ff, B;
    int rows_blk;        // neurons per CTA
    int rpad;            // rows_blk rounded up to 16 (K steps of phase 2)
    int n_groups;
    int n_stages;
    int n_tiles, tps;    // 128-column tiles of d_model; tiles per member
    int tile_set;        // tiles per TMEM set of phase 2: tps in equal sets of at most bd_tiles_in_tmem
    int act, dtype;
    uint32_t idesc_p1, idesc_p2;
    const float *scores;  // [B, d_ff]
    const float *tau;
    long long tau_stride;
    void *y;
    size_t y_stride;
    int y_dtype;
    float *partials;      // [n_groups, B, d_model]
    unsigned char *himg;  // [n_groups] images of the phase-2 B operand: K blocks x (3 parts x sequences x 128 bytes)
    WsCtrl *ctrl;
    int32_t *status;
};

// 2-D tiled TMA load with an L2 eviction hint.
__device__ __forceinline__ void bd_tma_load(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar,
                                            uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], "
        "[%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void bd_ld(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void bd_ld(uint32_t taddr, uint32_t (&r)[16]) { tc_ld16(taddr, r); }
// Shared-memory descriptor of an MN-major operand tile with 128-byte swizzle: 64 contiguous elements along M per
// 128-byte row, 8 K rows per 1024-byte atom; the next 8 K rows follow 1024 bytes on (stride byte offset), the next
// 64 elements along M lie lbo_bytes on (leading byte offset).
__device__ __forceinline__ uint64_t bd_smem_desc_mn(uint32_t addr, uint32_t lbo_bytes) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3fffu);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3fffu) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// Byte offset of element (row n = SEQS part + sequence, k) in the K-major, 128-byte-swizzled image of the
// [3 SEQS, K] operand: blocks of 64 k, 8-row atoms of 1024 bytes, 16-byte chunks XORed with the row inside the atom.
template <int SEQS>
__device__ __forceinline__ uint32_t bd_himg_off(int k, int n) {
    const int kb = k >> 6, kk = k & 63;
    return (uint32_t)kb * bd_img_block(SEQS) + (uint32_t)(n >> 3) * 1024u + (uint32_t)(n & 7) * 128u +
           (uint32_t)(((kk >> 3) ^ (n & 7)) << 4) + (uint32_t)(kk & 7) * 2u;
}
__device__ __forceinline__ uint16_t bd_to16(int dtype, float v, float &back) {
    if (dtype == CLADA_F16) {
        const __half h = __float2half_rn(v);
        back = __half2float(h);
        return __half_as_ushort(h);
    }
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    back = __bfloat162float(h);
    return __bfloat16_as_ushort(h);
}
// The MMAs of one phase-2 stage (up to 8 K steps of 16 neurons), issued back to back from descriptors computed
// beforehand: the issuing thread's own instructions between two MMAs are what limits their rate.
//   da: MN-major descriptor of the stage's first 16 rows (the next K step lies 2048 bytes on);
//   dhv: the K-major descriptors of the member's K steps in the h image, computed once per launch and member.
__device__ __forceinline__ void bd_issue_stage(uint32_t d_y, uint64_t da, const uint64_t (&dhv)[kBdMaxRows / 16], int ksteps,
                                               uint32_t acc, uint32_t idesc) {
#pragma unroll
    for (int k = 0; k < kBdMaxRows / 16; ++k)
        if (k < ksteps) tc_mma(d_y, da + 128 * k, dhv[k], k > 0 ? 1u : acc, idesc);
}
// The K-major descriptors of a member's K steps in the h image: the next step lies 32 bytes on, after the fourth
// step of a 64-neuron block the next block follows.
template <int SEQS>
__device__ __forceinline__ void bd_member_descs(uint64_t dh0, int mm, int ksteps, uint64_t (&dhv)[kBdMaxRows / 16]) {
#pragma unroll
    for (int k = 0; k < kBdMaxRows / 16; ++k) {
        const int kk16 = mm * ksteps + k;
        dhv[k] = dh0 + (uint64_t)(kk16 >> 2) * (bd_img_block(SEQS) >> 4) + (uint64_t)(kk16 & 3) * 2;
    }
}
__device__ __forceinline__ void bd_epi_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kBdEpi) : "memory"); }

template <int SEQS>
__global__ void __launch_bounds__(kBdThreads, 1)
sparse_ffn_batch_dense_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_wg,
                              const __grid_constant__ CUtensorMap map_wu, const __grid_constant__ CUtensorMap map_wd,
                              const BdParams p) {
    extern __shared__ unsigned char bd_smem_raw[];
    const uint32_t smem0 = (tc_smem_u32(bd_smem_raw) + 1023u) & ~1023u;
    __shared__ __align__(8) uint64_t s_full[kBdMaxStages], s_empty[kBdMaxStages], s_p1_full, s_h_own, s_h_all,
        s_tile_full[kBdMaxTiles], s_tile_read[kBdMaxTiles];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort, s_group_ok, s_cta;

    constexpr int kPer = SEQS / 2;  // sequences of an epilogue warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool gated = act_is_gated(p.act);
    const int n_kblocks = (p.d_model + kTcTileK - 1) / kTcTileK;
    const int n_stages = p.n_stages;
    const uint32_t box_bytes = (uint32_t)p.rows_blk * 128u;     // what one weight box delivers
    const uint32_t slot_bytes = (uint32_t)p.rpad * 128u;        // where the next box of a stage starts
    const uint32_t stage_bytes = 2u * slot_bytes + SEQS * 128u; // gate | up | x   or   down columns 0-63 | 64-127
    const int kimg_blocks = (kBdMembers * p.rpad + 63) / 64;
    const uint32_t img_bytes = (uint32_t)kimg_blocks * bd_img_block(SEQS);
    const uint32_t himg_s = smem0 + (uint32_t)n_stages * stage_bytes;  // the group's h image in shared memory

    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) {
            tc_mbar_init(tc_smem_u32(&s_full[s]), 1);
            tc_mbar_init(tc_smem_u32(&s_empty[s]), 1);
        }
        tc_mbar_init(tc_smem_u32(&s_p1_full), 1);
        tc_mbar_init(tc_smem_u32(&s_h_own), kBdEpi);
        tc_mbar_init(tc_smem_u32(&s_h_all), kBdEpi);
        for (int t = 0; t < kBdMaxTiles; ++t) {
            tc_mbar_init(tc_smem_u32(&s_tile_full[t]), 1);
            tc_mbar_init(tc_smem_u32(&s_tile_read[t]), kBdEpi);
        }
        s_abort = 0;
        s_group_ok = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // Rows rows_blk .. rpad-1 of every box slot are never written by a copy but are read by the last K step of
    // phase 2 (against h = 0): they must hold finite values.
    if (p.rpad > p.rows_blk) {
        const int pad_vecs = (p.rpad - p.rows_blk) * 8;  // 16-byte vectors per slot
        for (int i = threadIdx.x; i < n_stages * 2 * pad_vecs; i += kBdThreads) {
            const int slot = i / pad_vecs, v = i - slot * pad_vecs;
            const uint32_t a = smem0 + (uint32_t)(slot >> 1) * stage_bytes + (uint32_t)(slot & 1) * slot_bytes + box_bytes +
                               (uint32_t)v * 16u;
            asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&s_tmem_base)),
                     "r"(kBdTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    volatile int *abort_flag = &s_abort;
    pdl_launch_dependents();
    pdl_wait();  // x, the scores and the thresholds may come from the launch before
    // CTAs are numbered in the order in which they begin.  The launch is a plain one, so nothing promises that all CTAs
    // are resident at a time; but with these numbers every group but the last one begun is complete whenever a CTA
    // waits, goes through to the end by itself and makes room for the others.  The last one's three CTAs at most wait, in
    // group_wait, for a member that other work keeps off the SMs; the waits behind it (of the MMA thread for the others' h,
    // of the producer for the stages that hold their rows) are as long.
    if (threadIdx.x == 0) s_cta = (int)grid_enter(p.ctrl);
    __syncthreads();
    const int cta = s_cta;
    const int grp = cta / kBdMembers, mem = cta - grp * kBdMembers;
    const bool active = grp < p.n_groups;  // the CTAs behind the last whole group only join the meeting and the sums
    const int t0 = mem * p.tps;
    const int nt = max(0, min(p.tps, p.n_tiles - t0));          // this member's column tiles in phase 2
    const int j0 = cta * p.rows_blk;                            // this CTA's first neuron
    if (threadIdx.x == 0) BD_TRACE(0);

    if (active && warp == 0) {
        // ---- TMA producer ----------------------------------------------------------------------
        if (lane == 0) {
            const uint64_t stream_policy = policy_evict_first(), keep_policy = policy_evict_last();
            int kc = 0, s = 0;
            uint32_t par = 0;
            bool ok = true;
            for (int kb = 0; kb < n_kblocks && ok; ++kb, ++kc) {  // phase 1: gate | up | x, one K block per stage
                if (!tc_mbar_wait(tc_smem_u32(&s_empty[s]), par ^ 1, abort_flag)) {
                    ok = false;
                    break;
                }
                const uint32_t bar = tc_smem_u32(&s_full[s]);
                const uint32_t dst = smem0 + (uint32_t)s * stage_bytes;
                tc_mbar_expect_tx(bar, SEQS * 128u + (gated ? 2u : 1u) * box_bytes);
                bd_tma_load(dst + 2u * slot_bytes, &map_x, kb * kTcTileK, 0, bar, keep_policy);
                bd_tma_load(dst, &map_wg, kb * kTcTileK, j0, bar, stream_policy);
                if (gated) bd_tma_load(dst + slot_bytes, &map_wu, kb * kTcTileK, j0, bar, stream_policy);
                if (++s == n_stages) {
                    s = 0;
                    par ^= 1;
                }
            }
            BD_TRACE(14);
            // Phase 2, one column tile of one member's rows per stage: first this CTA's own rows for every tile of the
            // first set (their h is here before the group's exchange is over), then tile by tile the other three
            // members' rows; a tile of a later set takes its four members' rows in the same order.
            auto issue_p2 = [&](int mm, int t) -> bool {
                if (!tc_mbar_wait(tc_smem_u32(&s_empty[s]), par ^ 1, abort_flag, kPlaceLimit)) return false;
                const int rows0 = (grp * kBdMembers + mm) * p.rows_blk;
                const uint32_t bar = tc_smem_u32(&s_full[s]);
                const uint32_t dst = smem0 + (uint32_t)s * stage_bytes;
                tc_mbar_expect_tx(bar, 2u * box_bytes);
                bd_tma_load(dst, &map_wd, (t0 + t) * kTcTileM, rows0, bar, stream_policy);
                bd_tma_load(dst + slot_bytes, &map_wd, (t0 + t) * kTcTileM + 64, rows0, bar, stream_policy);
                ++kc;
                if (++s == n_stages) {
                    s = 0;
                    par ^= 1;
                }
                return true;
            };
            for (int t = 0; t < min(nt, p.tile_set) && ok; ++t) ok = issue_p2(mem, t);
            for (int t = 0; t < nt && ok; ++t) {
                if (t >= p.tile_set) ok = issue_p2(mem, t);
                for (int mo = 0; mo < kBdMembers - 1 && ok; ++mo) ok = issue_p2(mo + (mo >= mem ? 1 : 0), t);
            }
            BD_TRACE(15);
            if (!ok) *abort_flag = 1;
            for (int i = max(0, kc - n_stages); i < kc; ++i) {  // never leave with copies in flight
                int never = 0;
                if (!tc_mbar_wait(tc_smem_u32(&s_full[i % n_stages]), (i / n_stages) & 1, &never)) *abort_flag = 1;
            }
        }
    } else if (active && warp == 1) {
        // ---- MMA issuer ------------------------------------------------------------------------
        if (lane == 0) {
            int s = 0;
            uint32_t par = 0;
            bool ok = true;
            // One thread issues every MMA, so its instruction count per MMA bounds the rate (an MMA of N <= 48 takes
            // the tensor pipe ~44 cycles): descriptors are advanced by additions, never rebuilt.
            const uint64_t desc0 = tc_smem_desc(smem0);  // K-major descriptor of the ring's first byte
            const uint64_t stage16 = stage_bytes >> 4, slot16 = slot_bytes >> 4;
            uint64_t dstage = desc0;                     // descriptor of the current stage's first byte
            for (int kb = 0; kb < n_kblocks && ok; ++kb) {
                if (!tc_mbar_wait(tc_smem_u32(&s_full[s]), par, abort_flag)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (kb == 0) BD_TRACE(1);
                const uint64_t dg = dstage, du = dstage + slot16, dx = dstage + 2 * slot16;
                const uint32_t d_g = tmem_base + (uint32_t)(kb % kBdKSplit) * (2 * SEQS);  // this K split's columns
                const uint32_t acc0 = kb >= kBdKSplit ? 1u : 0u;
#pragma unroll
                for (int k = 0; k < kTcTileK / 16; ++k) {
                    tc_mma(d_g, dg + 2 * k, dx + 2 * k, k > 0 ? 1u : acc0, p.idesc_p1);
                    if (gated) tc_mma(d_g + SEQS, du + 2 * k, dx + 2 * k, k > 0 ? 1u : acc0, p.idesc_p1);
                }
                tc_commit(tc_smem_u32(&s_empty[s]));
                dstage += stage16;
                if (++s == n_stages) {
                    s = 0;
                    par ^= 1;
                    dstage = desc0;
                }
            }
            if (ok) tc_commit(tc_smem_u32(&s_p1_full));
            BD_TRACE(2);
            // Phase 2 writes over the phase-1 columns: the epilogue has read them before it lets s_h_own complete.
            // A: the stage's two boxes as one MN-major tile, 16 rows (2048 bytes) further per K step.  B: the h image,
            // 32 bytes further per K step and from the fourth step of a 64-neuron block on to the next block.
            const int ksteps = p.rpad / 16;
            const uint64_t dmn0 = bd_smem_desc_mn(smem0, slot_bytes);
            const uint64_t dh0 = tc_smem_desc(himg_s);
            uint64_t dstage2 = dmn0 + (uint64_t)s * stage16;
            auto run_p2 = [&](const uint64_t (&dhv)[kBdMaxRows / 16], int slot, uint32_t acc) -> bool {  // one stage's MMAs
                if (!tc_mbar_wait(tc_smem_u32(&s_full[s]), par, abort_flag)) return false;
                tc_fence_after();
                bd_issue_stage(tmem_base + (uint32_t)(slot * kBdParts * SEQS), dstage2, dhv, ksteps, acc, p.idesc_p2);
                tc_commit(tc_smem_u32(&s_empty[s]));
                dstage2 += stage16;
                if (++s == n_stages) {
                    s = 0;
                    par ^= 1;
                    dstage2 = dmn0;
                }
                return true;
            };
            // the B descriptors of the four members' K steps stay in registers for the whole phase
            uint64_t dh_own[kBdMaxRows / 16], dh_oth[kBdMembers - 1][kBdMaxRows / 16];
            bd_member_descs<SEQS>(dh0, mem, ksteps, dh_own);
#pragma unroll
            for (int mo = 0; mo < kBdMembers - 1; ++mo) bd_member_descs<SEQS>(dh0, mo + (mo >= mem ? 1 : 0), ksteps, dh_oth[mo]);
            // (left to itself the compiler forms them anew between the MMAs: a step of 6 sequences 61.0 us on 5120 x 4100 and
            // 52.6 on 4096 x 9000 as it stands, 66.6 and 56.3 without these lines)
#pragma unroll
            for (int k = 0; k < kBdMaxRows / 16; ++k) {
                asm volatile("" : "+l"(dh_own[k]));
#pragma unroll
                for (int mo = 0; mo < kBdMembers - 1; ++mo) asm volatile("" : "+l"(dh_oth[mo][k]));
            }
            // this CTA's own part of h is in shared memory first; the other members' parts follow the exchange
            if (ok && !tc_mbar_wait(tc_smem_u32(&s_h_own), 0, abort_flag)) ok = false;
            tc_fence_after();
            BD_TRACE(3);
            for (int t = 0; t < min(nt, p.tile_set) && ok; ++t) ok = run_p2(dh_own, t, 0u);
            if (ok && !tc_mbar_wait(tc_smem_u32(&s_h_all), 0, abort_flag, kPlaceLimit)) ok = false;
            tc_fence_after();
            for (int t = 0, slot = 0; t < nt && ok; ++t) {
                if (t >= p.tile_set) {  // the slot's tile of the set before has to be out of the tensor memory
                    ok = tc_mbar_wait(tc_smem_u32(&s_tile_read[t - p.tile_set]), 0, abort_flag);
                    tc_fence_after();
                    if (ok) ok = run_p2(dh_own, slot, 0u);
                }
#pragma unroll
                for (int mo = 0; mo < kBdMembers - 1; ++mo)
                    if (ok) ok = run_p2(dh_oth[mo], slot, 1u);
                if (++slot == p.tile_set) slot = 0;
                if (ok) tc_commit(tc_smem_u32(&s_tile_full[t]));  // this tile's partial output is complete
            }
            BD_TRACE(4);
            if (!ok) *abort_flag = 1;
        }
    } else if (active) {
        // ---- epilogue warps (2..): warp w reads TMEM lanes 32 (w % 4) .. +31; twins take half the sequences each ----
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const int b0 = half * kPer;                  // this warp's first sequence
        const int r = quarter * 32 + lane;           // this thread's neuron of the CTA (phase 1), column of a tile (phase 2)
        const int etid = threadIdx.x - 64;
        const int j = j0 + r;
        const bool row_ok = r < p.rows_blk && j < p.d_ff;
        unsigned keep = 0;                           // bit i: sequence b0 + i keeps neuron j
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int b = b0 + i;
            if (b < p.B && row_ok && __ldg(p.scores + (size_t)b * p.d_ff + j) >= __ldg(p.tau + (size_t)b * p.tau_stride))
                keep |= 1u << i;
        }
        bool ok = tc_mbar_wait(tc_smem_u32(&s_p1_full), 0, abort_flag);
        tc_fence_after();
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        if (etid == 0) BD_TRACE(5);
        if (ok) {
            const int n_splits = min(kBdKSplit, n_kblocks);
            const int k = mem * p.rpad + r;  // this CTA's slice of the image, written where phase 2 reads it
            const uint32_t row0 = himg_s + bd_himg_off<SEQS>(k & ~63, 0) + (uint32_t)(k & 7) * 2u;  // row n: see bd_himg_off
            const uint32_t chunk = (uint32_t)(k & 63) >> 3;
            if (b0 < p.B) {
                float g[kPer], u[kPer];
#pragma unroll
                for (int i = 0; i < kPer; ++i) g[i] = u[i] = 0.f;
                for (int sp = 0; sp < n_splits; ++sp) {
                    uint32_t rg[kPer], ru[kPer];
                    const uint32_t col = t_lane + (uint32_t)(sp * 2 * SEQS + b0);
                    bd_ld(col, rg);
                    if (gated) bd_ld(col + SEQS, ru);
                    tc_wait_ld();
#pragma unroll
                    for (int i = 0; i < kPer; ++i) {
                        g[i] += __uint_as_float(rg[i]);
                        if (gated) u[i] += __uint_as_float(ru[i]);
                    }
                }
                if (r < p.rpad) {  // rows rows_blk .. rpad-1 are the zero padding of the K steps
                    const uint32_t at0 = row0 + (uint32_t)(b0 >> 3) * 1024u;  // b0 is a multiple of 8
#pragma unroll
                    for (int i = 0; i < kPer; ++i) {
                        if (b0 + i >= p.B) break;
                        float h = ((keep >> i) & 1u) ? neuron_value_f(p.act, g[i], u[i]) : 0.f;
                        const uint32_t at = at0 + (uint32_t)(i >> 3) * 1024u + (uint32_t)(i & 7) * 128u + ((chunk ^ (uint32_t)(i & 7)) << 4);
#pragma unroll
                        for (int part = 0; part < kBdParts; ++part) {
                            float back;
                            const uint16_t bits = bd_to16(p.dtype, h, back);
                            h -= back;
                            asm volatile("st.shared.u16 [%0], %1;" ::"r"(at + part * (SEQS / 8) * 1024u), "h"(bits) : "memory");
                        }
                    }
                }
            }
        }
        if (ok) {  // the MMA thread may start on this CTA's own down rows
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();  // phase 2 writes over the TMEM columns this thread has read
            tc_mbar_arrive(tc_smem_u32(&s_h_own));
        }
        bd_epi_sync();
        unsigned char *img = p.himg + (size_t)grp * img_bytes;
        // The exchange in 16-byte chunks: thread -> chunk etid % 16 of a member's slice (rpad <= 128) in row etid / 16 of
        // every run of kRowsPass rows; rows of absent sequences are left out.
        constexpr int kRowsPass = kBdEpi / 16, kPasses = kBdParts * SEQS / kRowsPass;
        const int c8 = 8 * (etid & 15);
        auto present = [&](int pass) { return c8 < p.rpad && (pass * kRowsPass + (etid >> 4)) % SEQS < p.B; };
        auto chunk_off = [&](int pass, int m) { return bd_himg_off<SEQS>(m * p.rpad + c8, pass * kRowsPass + (etid >> 4)); };
        if (ok) {  // the slice goes to global memory for the other three members
#pragma unroll
            for (int pass = 0; pass < kPasses; ++pass) {
                if (!present(pass)) continue;
                const uint32_t off = chunk_off(pass, mem);
                __stcg(reinterpret_cast<uint4 *>(img + off), lds128(himg_s + off));
            }
            __threadfence();
        }
        if (etid == 0) BD_TRACE(6);
        bd_epi_sync();
        // group exchange: one byte counter per group; every member adds 1 when its part of h is in global memory
        if (etid == 0) {
            unsigned *word = reinterpret_cast<unsigned *>(p.ctrl) + kBdGroupWord0 + (grp >> 2);
            const unsigned shift = 8u * (unsigned)(grp & 3);
            int gok = 0;
            if (ok && !*abort_flag) {
                asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(word), "r"(1u << shift) : "memory");
                gok = group_wait(p.ctrl, word, shift, kBdMembers, (unsigned)(grp + 1) * kBdMembers) ? 1 : 0;
            }
            s_group_ok = gok;
            BD_TRACE(7);
        }
        bd_epi_sync();
        ok = ok && s_group_ok != 0;
        if (ok) {
            uint4 v[kBdMembers - 1][kPasses];  // the other members' slices: all loads go out together
#pragma unroll
            for (int mo = 0; mo < kBdMembers - 1; ++mo)
#pragma unroll
                for (int pass = 0; pass < kPasses; ++pass)
                    if (present(pass))
                        v[mo][pass] = __ldcg(reinterpret_cast<const uint4 *>(img + chunk_off(pass, mo + (mo >= mem ? 1 : 0))));
#pragma unroll
            for (int mo = 0; mo < kBdMembers - 1; ++mo)
#pragma unroll
                for (int pass = 0; pass < kPasses; ++pass)
                    if (present(pass))
                        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(himg_s + chunk_off(pass, mo + (mo >= mem ? 1 : 0))),
                                     "r"(v[mo][pass].x), "r"(v[mo][pass].y), "r"(v[mo][pass].z), "r"(v[mo][pass].w)
                                     : "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_mbar_arrive(tc_smem_u32(&s_h_all));
            if (etid == 0) BD_TRACE(8);
            // ---- phase 2 epilogue: each column tile of the group's partial output as soon as it is complete ----------
            for (int t = 0; t < nt && ok; ++t) {
                ok = tc_mbar_wait(tc_smem_u32(&s_tile_full[t]), 0, abort_flag);
                tc_fence_after();
                if (t == 0 && etid == 0) BD_TRACE(9);
                if (!ok) break;
                const int i = (t0 + t) * kTcTileM + r;
                const uint32_t t_col = t_lane + (uint32_t)((t % p.tile_set) * kBdParts * SEQS);
                uint32_t rp[kBdParts][kPer];
                if (b0 < p.B) {
#pragma unroll
                    for (int part = 0; part < kBdParts; ++part) bd_ld(t_col + (uint32_t)(part * SEQS + b0), rp[part]);
                    tc_wait_ld();
                }
                tc_fence_before();  // read: the next set's tile may take the columns
                tc_mbar_arrive(tc_smem_u32(&s_tile_read[t]));
                if (i < p.d_model) {
#pragma unroll
                    for (int e = 0; e < kPer; ++e)
                        if (b0 + e < p.B)  // the three parts' column groups, added in part order
                            p.partials[((size_t)grp * p.B + b0 + e) * p.d_model + i] =
                                (__uint_as_float(rp[0][e]) + __uint_as_float(rp[1][e])) + __uint_as_float(rp[2][e]);
                }
            }
        }
        if (etid == 0) BD_TRACE(10);
        if (!ok) *abort_flag = 1;
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) BD_TRACE(11);
    if (threadIdx.x == 0 && s_abort && p.status) atomicOr(p.status, CLADA_STATUS_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kBdTmemCols) : "memory");
    }
    // ---- all groups' partial outputs are in global memory after the meeting: sum them in group order ----------
    const GridPart mine = grid_meet(p.ctrl, gridDim.x, cta, 32);
    if (mine.parts < 0 && threadIdx.x == 0 && p.status) atomicOr(p.status, CLADA_STATUS_TIMEOUT);
    if (mine.parts <= 0) return;
    if (threadIdx.x == 0) BD_TRACE(12);
    if (mine.part == 0 && threadIdx.x < 64 - kBdGroupWord0)  // every member has passed its group's counter: clear them
        reinterpret_cast<unsigned *>(p.ctrl)[kBdGroupWord0 + threadIdx.x] = 0u;
    const int d4 = p.d_model / 4;
    // a part is an equal run of (sequence, four columns)
    const int share = (p.B * d4 + mine.parts - 1) / mine.parts;
    const int it0 = mine.part * share, it1 = min(p.B * d4, it0 + share);
    for (int it = it0 + threadIdx.x; it < it1; it += kBdThreads) {
        const int b = it / d4, q = it - b * d4;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 *src = reinterpret_cast<const float4 *>(p.partials) + (size_t)b * d4 + q;
        for (int g0 = 0; g0 < p.n_groups; g0 += 19) {
            float4 v[19];
#pragma unroll
            for (int e = 0; e < 19; ++e)
                v[e] = g0 + e < p.n_groups ? __ldcg(src + (size_t)(g0 + e) * p.B * d4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 19; ++e) {
                s.x += v[e].x; s.y += v[e].y; s.z += v[e].z; s.w += v[e].w;
            }
        }
        char *yb = static_cast<char *>(p.y) + b * p.y_stride;
        if (p.y_dtype == CLADA_F32) {
            reinterpret_cast<float4 *>(yb)[q] = s;
        } else {
            reinterpret_cast<uint2 *>(yb)[q] = pack4_16bit(p.y_dtype, s);
        }
    }
    if (threadIdx.x == 0) BD_TRACE(13);
}

// ---- host side ------------------------------------------------------------------------------

struct BdPlan {
    int seqs;  // the kernel's instance: 16 or 32 sequences
    int rows_blk, rpad, n_groups, n_tiles, tps, tile_set, n_stages;
    size_t smem, partial_bytes, himg_bytes;
};

// The split of a layer over the device's CTAs, or false when this kernel does not take the layer.
static bool bd_plan(const clada_layer *layer, int B, const DeviceInfo &di, BdPlan *pl) {
    if (layer->dtype != CLADA_BF16 && layer->dtype != CLADA_F16) return false;
    if (B < 1 || B > kDenseMaxSeqs) return false;
    pl->seqs = B <= 16 ? 16 : 32;
    if (layer->d_model % 8 != 0 || layer->d_model > kMaxDModel) return false;
    pl->n_groups = di.num_sms / kBdMembers;
    if (pl->n_groups < 1 || pl->n_groups > kBdMaxGroups) return false;
    const int n_ctas = pl->n_groups * kBdMembers;
    pl->rows_blk = (layer->d_ff + n_ctas - 1) / n_ctas;
    if (pl->rows_blk > kBdMaxRows) return false;
    pl->rpad = (pl->rows_blk + 15) / 16 * 16;
    pl->n_tiles = (layer->d_model + kTcTileM - 1) / kTcTileM;
    pl->tps = (pl->n_tiles + kBdMembers - 1) / kBdMembers;
    if (pl->tps > kBdMaxTiles) return false;
    const int sets = (pl->tps + bd_tiles_in_tmem(pl->seqs) - 1) / bd_tiles_in_tmem(pl->seqs);
    pl->tile_set = (pl->tps + sets - 1) / sets;
    const size_t stage_bytes = 2 * (size_t)pl->rpad * 128 + (size_t)pl->seqs * 128;
    const size_t kimg_blocks = ((size_t)kBdMembers * pl->rpad + 63) / 64;
    pl->himg_bytes = kimg_blocks * bd_img_block(pl->seqs);
    const size_t budget = (size_t)di.max_smem_optin - 1024;  // static arrays: barriers and flags
    // behind the ring: the h image; at least 16 KB, because a phase-1 A tile is always 128 rows high and with few
    // neurons per CTA the tile of the last stage reaches past its own slot
    const size_t tail = std::max<size_t>(pl->himg_bytes, 16384);
    if (budget < 1024 + tail + 3 * stage_bytes) return false;
    pl->n_stages = (int)std::min<size_t>(kBdMaxStages, (budget - 1024 - tail) / stage_bytes);
    // never two CTAs on an SM (more than half of its shared memory): the second would wait for tensor memory that the
    // first gives back only at its end
    pl->smem = std::max<size_t>(1024 + (size_t)pl->n_stages * stage_bytes + tail, kBdSmemMin);
    pl->partial_bytes = (size_t)pl->n_groups * B * layer->d_model * sizeof(float);
    return true;
}

bool ffn_batch_dense_supported(const clada_layer *layer, int B) {
    DeviceInfo di;
    BdPlan pl;
    return device_info(&di) == CLADA_OK && bd_plan(layer, B, di, &pl);
}

// Scratch behind the control block: the groups' partial outputs, then their h images.
size_t ffn_batch_dense_scratch_bytes(const clada_layer *layer, int B) {
    DeviceInfo di;
    BdPlan pl;
    if (device_info(&di) != CLADA_OK || !bd_plan(layer, B, di, &pl)) return 0;
    return ((pl.partial_bytes + 255) & ~(size_t)255) + (size_t)pl.n_groups * pl.himg_bytes;
}

int launch_ffn_batch_dense(const clada_layer *layer, int B, const void *x, const float *scores, const float *tau,
                           long long tau_stride, void *y, int y_dtype, void *ws, int32_t *status, cudaStream_t st) {
    static bool configured[2][64] = {};
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != CLADA_OK) return rc;
    BdPlan pl;
    if (!bd_plan(layer, B, di, &pl)) return CLADA_ERR_UNSUPPORTED;
    EncodeTiledFn enc;
    rc = encode_fn(&enc);
    if (rc != CLADA_OK) return rc;
    const bool gated = act_is_gated(layer->activation);
    CUtensorMap map_x, map_wg, map_wu, map_wd;
    if ((rc = make_map(enc, &map_x, x, B, layer->d_model, layer->dtype, pl.seqs)) != CLADA_OK) return rc;
    if ((rc = make_map(enc, &map_wg, layer->w_gate, layer->d_ff, layer->d_model, layer->dtype, pl.rows_blk)) != CLADA_OK)
        return rc;
    if ((rc = make_map(enc, &map_wu, gated ? layer->w_up : layer->w_gate, layer->d_ff, layer->d_model, layer->dtype,
                       pl.rows_blk)) != CLADA_OK)
        return rc;
    if ((rc = make_map(enc, &map_wd, layer->w_down_t, layer->d_ff, layer->d_model, layer->dtype, pl.rows_blk)) != CLADA_OK)
        return rc;
    BdParams p;
    p.d_model = layer->d_model;
    p.d_ff = layer->d_ff;
    p.B = B;
    p.rows_blk = pl.rows_blk;
    p.rpad = pl.rpad;
    p.n_groups = pl.n_groups;
    p.n_stages = pl.n_stages;
    p.n_tiles = pl.n_tiles;
    p.tps = pl.tps;
    p.act = layer->activation;
    p.dtype = layer->dtype;
    p.tile_set = pl.tile_set;
    p.idesc_p1 = tc_instr_desc(layer->dtype, pl.seqs);
    p.idesc_p2 = tc_instr_desc(layer->dtype, kBdParts * pl.seqs) | (1u << 15);  // A (the down rows) is MN-major
    p.scores = scores;
    p.tau = tau;
    p.tau_stride = tau_stride;
    p.y = y;
    p.y_stride = (size_t)layer->d_model * elem_size(y_dtype);
    p.y_dtype = y_dtype;
    p.partials = reinterpret_cast<float *>(static_cast<char *>(ws) + kWsCtrlBytes);
    p.himg = reinterpret_cast<unsigned char *>(static_cast<char *>(ws) + kWsCtrlBytes + ((pl.partial_bytes + 255) & ~(size_t)255));
    p.ctrl = static_cast<WsCtrl *>(ws);
    p.status = status;
    const void *kernel = pl.seqs == 16 ? reinterpret_cast<const void *>(sparse_ffn_batch_dense_kernel<16>)
                                       : reinterpret_cast<const void *>(sparse_ffn_batch_dense_kernel<32>);
    if (!configured[pl.seqs == 16][di.device & 63]) {
        CLADA_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)((size_t)di.max_smem_optin - 1024)));
        configured[pl.seqs == 16][di.device & 63] = true;
    }
    void *args[] = {&map_x, &map_wg, &map_wu, &map_wd, &p};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(di.num_sms);
    cfg.blockDim = dim3(kBdThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CLADA_CUDA_TRY(cudaLaunchKernelExC(&cfg, kernel, args));
    return CLADA_OK;
}

}  // namespace clada

#ifdef CLADA_BD_TRACE
extern "C" int clada_bd_trace_buffer(unsigned long long *buf) {
    CLADA_CUDA_TRY(cudaMemcpyToSymbol(clada::g_bd_trace, &buf, sizeof buf));
    return CLADA_OK;
}
#endif
