// Decode of several sequences from nested index lists in shared passes over the layer:
//   h[b, j] = z(w_gate_j . x_b, w_up_j . x_b)   for j in list_b,      y_b = sum_{j in list_b} h[b, j] w_down_t[j, :]
//
// Every sequence gets the bits that a launch of its own gives it (sparse_ffn_kernel): the same tree for every dot
// product, the same order of neurons and partial rows in every sum.  What the sequences share are the reads: a gate or
// up row is fetched from HBM once for all sequences that list it; a down row is fetched once per sequence, from L2 where it
// is still there.  No row that nobody lists is read, and h stays in fp32.  Four launches, chained programmatically, none of
// which waits for CTAs of its own grid:
//
//   nested_keep_kernel    the lists' heads as keep bits, 32 neurons a word; counts, levels and indices checked here
//   nested_hidden_kernel  the union of the heads shared out evenly; a producer warp streams gate | up rows through a ring
//                         of stages with bulk copies, a lane per row; a free consumer warp takes the next neuron (no
//                         CTA-wide step at all), up to four of its sequences at a time, x from shared memory.  Bound by the
//                         consumers' instructions (0.5 a cycle and scheduler, half of the HBM rate).
//   nested_down_kernel    CTA c adds up, list after list, the down rows of the share that CTA c of a single launch takes;
//                         its rows are on their way before the hidden values are waited for.  Bound by HBM and L2 (5 to
//                         6 TB/s with a third of the rows from L2).
//   nested_sums_kernel    column sums of the partial rows
//
// Measured (us a step with its cognitive load, a launch per sequence / this way): four of 2048 x 16384, a vocabulary of
// 256000, 96.3 / 68.6; three, four and eight of 2048 x 16384 78.3 / 64.7, 103 / 73.5, 201 / 121; of 4096 x 11008 92.7 / 84.5,
// 121 / 99, 236 / 183; of 5120 x 13824 133 / 123, 176 / 143, 346 / 287; of 1024 x 4100 41.2 / 31.4, 53.8 / 33.3, 103 / 45.9.
// Which batches do: at nb_plan.
#include <algorithm>

#include "common.cuh"
#include "ffn_common.cuh"
#include "nested_batch.cuh"

namespace clada {

struct NbParams {
    const void *w_gate, *w_up, *w_down_t;
    const void *x;           // [nb, d_model]
    const int32_t *order;    // [nb, d_ff]
    const int32_t *counts;   // [nb, 4]
    const int32_t *level;    // [nb]
    void *y;                 // [nb, d_model]
    int y_dtype;
    int32_t *count_out;      // [nb] or null
    float *hidden;           // [nb, d_ff]
    unsigned *words;         // [nb, chunks]
    float *partials;         // [nb, n_shares * groups, d_model]
    int32_t *status;
    int d_model, d_ff, act, nb;
    int n_shares;            // shares of a list: CTAs of a single launch
};

constexpr int kNbConsWarps = 15;                      // consumer warps of the hidden pass, at most
constexpr int kNbThreads = (kNbConsWarps + 1) * kWarp;
constexpr int kNbMaxStages = 48;
constexpr int kNbKeepThreads = 1024;
constexpr int kNbStatic = 9 * 1024;  // room for static shared memory

// The leading entries of list b that count: clamped into the layer as the single launch clamps them.
__device__ __forceinline__ int nb_count(const NbParams &p, int b, bool &bad) {
    const int lv = __ldcg(p.level + b);
    const int n = __ldcg(p.counts + (size_t)b * 4 + (lv & 3));
    bad |= lv < 0 || lv > 3 || n < 0 || n > p.d_ff;
    return min(max(n, 0), p.d_ff);
}
__device__ __forceinline__ int nb_share(int n, int c, int n_shares) {  // as split_at of the single launch
    return (int)(((unsigned)n * (unsigned)c) / (unsigned)n_shares);
}

// One CTA per sequence: bits set in shared memory, words written out.
__global__ void __launch_bounds__(kNbKeepThreads)
nested_keep_kernel(const NbParams p) {
    extern __shared__ unsigned s_words[];
    const int b = blockIdx.x, chunks = (p.d_ff + kWarp - 1) / kWarp;
    for (int q = threadIdx.x; q < chunks; q += kNbKeepThreads) s_words[q] = 0u;
    __syncthreads();
    pdl_wait();
    // Only now: a kernel behind this one that has not waited yet may read what was there before this one (x, the lists).
    pdl_launch_dependents();
    bool bad = false;
    const int n = nb_count(p, b, bad);
    const int32_t *list = p.order + (size_t)b * p.d_ff;
    for (int i0 = 0; i0 < n; i0 += 8 * kNbKeepThreads) {
        int j[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * kNbKeepThreads + threadIdx.x;
            j[u] = i < n ? __ldcg(list + i) : -1;
            bad |= i < n && (j[u] < 0 || j[u] >= p.d_ff);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (i0 + u * kNbKeepThreads + (int)threadIdx.x >= n) continue;
            const int k = min(max(j[u], 0), p.d_ff - 1);
            atomicOr(&s_words[k >> 5], 1u << (k & 31));
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < chunks; q += kNbKeepThreads) p.words[(size_t)b * chunks + q] = s_words[q];
    if (bad && p.status) atomicOr(p.status, CLADA_STATUS_BAD_INDEX);
    if (threadIdx.x == 0 && p.count_out) p.count_out[b] = n;
}

// Hidden values of one neuron for the next S of its sequences (bits; the last one again when there are fewer) by one warp.
// The single launch has 32 VW threads on a row: lane l here plays the threads l, l + 32, ..., one after another, so step w
// forms what warp w has there.  Its warp totals come from a halving butterfly (the tree of one value is that of any
// butterfly: partners 16, 8, 4, 2, 1 lanes away), and the VW totals of a value are added as there, neighbours first.  The
// steps stay a loop: unrolled altogether, with four sequences, the warps of a CTA were spread over more code than the
// instruction cache holds (72 us for the pass where the loop takes 28).  x widened to fp32 in shared memory was slower, too.
template <typename T, int VW, int NV, bool GATED, int S>
__device__ __forceinline__ unsigned nb_hidden(unsigned bits, const uint32_t rows, const uint32_t row_bytes, const int vpr,
                                              const uint32_t xs0, const int act, const int lane, float *s_tot, const int F,
                                              float *out) {
    constexpr int P = Pairs<T>::kPairs;
    constexpr int N = GATED ? 2 * S : S;  // values: sequence by sequence its gate and (gated) up sum
    int b[S];
    uint32_t xs[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        b[s] = s == 0 || bits ? __ffs(bits) - 1 : b[s > 0 ? s - 1 : 0];
        if (bits) bits &= bits - 1;
        xs[s] = xs0 + (uint32_t)b[s] * row_bytes;
    }
    __syncwarp();  // the totals of the call before are read
#pragma unroll 2
    for (int w = 0; w < VW; ++w) {
        float2 sg[S], su[S];
#pragma unroll
        for (int s = 0; s < S; ++s) sg[s] = su[s] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int vec = w * kWarp + lane + k * VW * kWarp;
            if (vec < vpr) {
                const uint32_t at = (uint32_t)vec * 16u;
                float2 fg[P], fu[P];
                Pairs<T>::unpack(lds128(rows + at), fg);
                if (GATED) Pairs<T>::unpack(lds128(rows + row_bytes + at), fu);
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    float2 fx[P];
                    Pairs<T>::unpack(lds128(xs[s] + at), fx);
#pragma unroll
                    for (int e = 0; e < P; ++e) {
                        sg[s] = __ffma2_rn(fg[e], fx[e], sg[s]);
                        if (GATED) su[s] = __ffma2_rn(fu[e], fx[e], su[s]);
                    }
                }
            }
        }
        float v[N];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            v[GATED ? 2 * s : s] = sg[s].x + sg[s].y;
            if (GATED) v[2 * s + 1] = su[s].x + su[s].y;
        }
        int o = 16;
#pragma unroll
        for (int n = N / 2; n >= 1; n >>= 1, o >>= 1) {
            const bool hi = lane & o;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const float send = hi ? v[i] : v[i + n];
                v[i] = (hi ? v[i + n] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
#pragma unroll
        for (int q = 16 / N; q >= 1; q >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], q);
        // lane l holds value l N / 32
        if (lane % (32 / N) == 0) s_tot[lane / (32 / N) * VW + w] = v[0];
    }
    __syncwarp();
    const float4 *t = reinterpret_cast<const float4 *>(s_tot + lane % N * VW);
    float q[VW / 4];
#pragma unroll
    for (int i = 0; i < VW / 4; ++i) {
        const float4 f = t[i];
        q[i] = (f.x + f.y) + (f.z + f.w);
    }
    const float tot = VW == 8 ? q[0] + q[1] : (q[0] + q[1]) + (q[VW / 4 - 2] + q[VW / 4 - 1]);
    const float up = __shfl_xor_sync(0xffffffffu, tot, 1);
    const float h = neuron_value_f(act, tot, up);
#pragma unroll
    for (int s = 0; s < S; ++s)
        if (lane == (GATED ? 2 * s : s)) out[(size_t)b[s] * F] = h;
    return bits;
}

template <typename T, int VW, int NV, bool GATED>
__global__ void __launch_bounds__(kNbThreads, 1)
nested_hidden_kernel(const NbParams p, const int n_stages, const int n_cons) {
    constexpr int E = Elem<T>::kPerVec;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = blockIdx.x, n_ctas = gridDim.x;
    const int F = p.d_ff, vpr = p.d_model / E;
    const uint32_t row_bytes = (uint32_t)vpr * 16u;
    const uint32_t stage_bytes = (GATED ? 2u : 1u) * row_bytes;
    const int chunks = (F + kWarp - 1) / kWarp;

    // dynamic shared memory: ring | x of all sequences | full, empty | list | keep bits of the list's neurons
    const uint32_t ring = smem_u32(smem_raw), xs0 = ring + (uint32_t)n_stages * stage_bytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw + (size_t)n_stages * stage_bytes + (size_t)p.nb * row_bytes);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kNbMaxStages);
    int *s_list = reinterpret_cast<int *>(bars + 2 * kNbMaxStages);
    int *s_keep = s_list + (F / n_ctas + 2);
    __shared__ int s_wtot[kNbThreads / kWarp], s_next;
    __shared__ __align__(16) float s_tot[kNbConsWarps][8 * VW];  // warp totals of up to eight values

    if (tid == 0) {
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(full0 + 8 * s, 1);   // the producer's expect_tx arrival
            mbar_init(empty0 + 8 * s, 1);  // the warp that took the neuron
        }
        s_next = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // x was there before nested_keep_kernel, which lets this kernel start only after its own wait
    for (int i = tid; i < p.nb * vpr; i += kNbThreads) {
        const uint4 q = __ldcg(static_cast<const uint4 *>(p.x) + i);
        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(xs0 + (uint32_t)i * 16u), "r"(q.x), "r"(q.y), "r"(q.z), "r"(q.w)
                     : "memory");
    }
    pdl_wait();
    pdl_launch_dependents();  // nested_down_kernel reads the lists and the down rows before its wait

    // ---- this CTA's equal share of the union, in ascending order ---------------------------------------------
    // A thread takes one 32-neuron chunk per batch; the batches are walked twice, first to count them all.
    auto union_word = [&](int q) {
        unsigned w = 0;
        if (q < chunks)
            for (int b = 0; b < p.nb; ++b) w |= p.words[(size_t)b * chunks + q];
        return w;
    };
    const int n_batches = (chunks + kNbThreads - 1) / kNbThreads;
    int n_act = 0, total = 0;
    unsigned first_word = 0;
    for (int walk = 0; walk < 2; ++walk) {
        const int r0 = nb_share(total, cta, n_ctas), r1 = nb_share(total, cta + 1, n_ctas);
        n_act = 0;
        for (int bt = 0; bt < n_batches; ++bt) {
            const int q = bt * kNbThreads + tid;
            const unsigned wu = walk == 1 && bt == 0 ? first_word : union_word(q);
            if (bt == 0) first_word = wu;
            const int cnt = __popc(wu);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            __syncthreads();
            if (lane == kWarp - 1) s_wtot[warp] = incl;
            __syncthreads();
            int wbase = 0, btot = 0;
#pragma unroll
            for (int w = 0; w < kNbThreads / kWarp; ++w) {
                const int v = s_wtot[w];
                wbase += w < warp ? v : 0;
                btot += v;
            }
            const int fr = n_act + wbase + incl - cnt;
            n_act += btot;
            if (walk == 0) continue;
            unsigned todo = __ballot_sync(0xffffffffu, fr < r1 && fr + cnt > r0);
            while (todo) {  // the warp that owns a chunk of the share writes it out, one lane per neuron
                const int t = __ffs(todo) - 1;
                todo &= todo - 1;
                const unsigned wb = __shfl_sync(0xffffffffu, wu, t);
                const int rank = __shfl_sync(0xffffffffu, fr, t) + __popc(wb & ((1u << lane) - 1u));
                const int qq = bt * kNbThreads + warp * kWarp + t;
                if (((wb >> lane) & 1u) && rank >= r0 && rank < r1 && guard_slot(rank - r0, F / n_ctas + 2, p.status)) {
                    int bits = 0;
                    for (int b = 0; b < p.nb; ++b) bits |= (int)((p.words[(size_t)b * chunks + qq] >> lane) & 1u) << b;
                    s_list[rank - r0] = qq * kWarp + lane;
                    s_keep[rank - r0] = bits;
                }
            }
        }
        total = n_act;
    }
    const int my_n = nb_share(total, cta + 1, n_ctas) - nb_share(total, cta, n_ctas);
    __syncthreads();  // list, keep bits, x and the mbarriers are ready

    bool timed_out = false;
    if (warp == kNbConsWarps) {
        // ---- producer ------------------------------------------------------------------------------------
        // A lane per row, several neurons at a time: what one thread needs for a copy is more than a short row's time.
        constexpr int kPerNeuron = GATED ? 2 : 1;
        const int run = min(16, max(1, n_stages / 3));  // well below n_stages: all of a run's stages are waited for at once
        const int q = lane / kPerNeuron, r = lane % kPerNeuron;
        const char *W = static_cast<const char *>(GATED && r == 1 ? p.w_up : p.w_gate);
        const uint64_t stream_policy = policy_evict_first();
        int i0 = 0;
        for (; i0 < my_n; i0 += run) {
            const int i = i0 + q, s = i % n_stages;
            const bool mine = q < run && i < my_n;
            if (mine && !mbar_wait(empty0 + 8 * s, ((i / n_stages) & 1) ^ 1)) timed_out = true;  // fresh: parity 1 passes
            if (__any_sync(0xffffffffu, timed_out)) break;
            if (mine && r == 0) mbar_expect_tx(full0 + 8 * s, stage_bytes);
            __syncwarp();
            if (mine)
                bulk_load_row_hint(ring + (uint32_t)s * stage_bytes + (uint32_t)r * row_bytes,
                                   W + (size_t)guard_row(s_list[i], F, p.status) * row_bytes, row_bytes, full0 + 8 * s, stream_policy);
        }
        // Never leave with copies in flight: the last use of every stage must have landed.
        const int issued = min(i0, my_n);
        for (int i = max(0, issued - n_stages) + lane; i < issued; i += kWarp)
            if (!mbar_wait(full0 + 8 * (i % n_stages), (i / n_stages) & 1)) timed_out = true;
    } else if (warp < n_cons) {
        // ---- consumers: whoever is free takes the next neuron ------------------------------------------------
        for (;;) {
            int i = 0;
            if (lane == 0) i = atomicAdd(&s_next, 1);
            i = __shfl_sync(0xffffffffu, i, 0);
            if (i >= my_n) break;
            const int use = i / n_stages, s = i - use * n_stages;
            // The stage's use before this one may still be on its way (its warp waits for it): a wait by parity for this use
            // would pass at once, so that one's hand-back is waited for first.
            if (use > 0 && !timed_out && !mbar_wait(empty0 + 8 * s, (use - 1) & 1)) timed_out = true;
            if (!timed_out && !mbar_wait(full0 + 8 * s, use & 1)) timed_out = true;
            const uint32_t rows = ring + (uint32_t)s * stage_bytes;
            float *out = p.hidden + s_list[i];
            for (unsigned bits = (unsigned)s_keep[i]; bits;) {
                const int left = __popc(bits);
                bits = left > 2    ? nb_hidden<T, VW, NV, GATED, 4>(bits, rows, row_bytes, vpr, xs0, p.act, lane, s_tot[warp], F, out)
                       : left == 2 ? nb_hidden<T, VW, NV, GATED, 2>(bits, rows, row_bytes, vpr, xs0, p.act, lane, s_tot[warp], F, out)
                                   : nb_hidden<T, VW, NV, GATED, 1>(bits, rows, row_bytes, vpr, xs0, p.act, lane, s_tot[warp], F, out);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + 8 * s);
        }
    }
    if (timed_out && p.status) atomicOr(p.status, CLADA_STATUS_TIMEOUT);
}

// CTA c takes share c of every list, one list after the other; down rows come through a ring of single rows per consumer
// group (a ring's uses are all one group's, in order).  NPC: neurons per chunk of the single launch; its group g takes
// chunks g, g + GROUPS, ...
template <typename T, int NV, int GROUPS, int NPC>
__global__ void __launch_bounds__(kFfnThreads, 1)
nested_down_kernel(const NbParams p, const int n_stages) {  // stages of a group's ring
    constexpr int E = Elem<T>::kPerVec, P = Pairs<T>::kPairs;
    constexpr int GT = kConsumers / GROUPS;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = blockIdx.x, F = p.d_ff, vpr = p.d_model / E;
    const uint32_t row_bytes = (uint32_t)vpr * 16u;
    // dynamic shared memory: rings | full, empty of all rings | list | hidden values
    const uint32_t ring0 = smem_u32(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw + (size_t)GROUPS * n_stages * row_bytes);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kNbMaxStages);
    int *s_list = reinterpret_cast<int *>(bars + 2 * kNbMaxStages);
    float *s_h = reinterpret_cast<float *>(s_list + p.nb * (F / p.n_shares + 2));
    __shared__ int s_r0[kNestedBatchMax], s_first[kNestedBatchMax + 1];
    if (tid == 0) {
        for (int s = 0; s < GROUPS * n_stages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, kConsWarps / GROUPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // The lists and the layer were there before nested_keep_kernel and nested_hidden_kernel began.
    if (warp == 1) {
        bool bad = false;
        const int n = lane < p.nb ? nb_count(p, lane, bad) : 0;
        const int r0 = nb_share(n, c, p.n_shares), mine = nb_share(n, c + 1, p.n_shares) - r0;
        int end = mine;
#pragma unroll
        for (int o = 1; o < kNestedBatchMax; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += t;
        }
        if (lane < p.nb) {
            s_r0[lane] = r0;
            s_first[lane] = end - mine;
            if (lane == p.nb - 1) s_first[p.nb] = end;
        }
    }
    __syncthreads();
    for (int b = 0; b < p.nb; ++b) {
        const int first = s_first[b], n = s_first[b + 1] - first;
        const int32_t *list = p.order + (size_t)b * F + s_r0[b];
        for (int i = tid; i < n; i += kFfnThreads) s_list[first + i] = min(max(__ldcg(list + i), 0), F - 1);
    }
    __syncthreads();

    bool timed_out = false;
    if (warp == kConsWarps) {
        // ---- producer ------------------------------------------------------------------------------------
        // A lane per row, a chunk of every group at a time.
        const char *Wd = static_cast<const char *>(p.w_down_t);
        const uint64_t policy = policy_evict_last();  // the other sequences of the pass read the row again
        const int g = lane / NPC, u = lane % NPC;
        int done = 0;  // rows of this lane's group so far
        bool stop = false;
        for (int b = 0; b < p.nb && !stop; ++b) {
            const int first = s_first[b], n = s_first[b + 1] - first;
            for (int i0 = 0; i0 < n; i0 += GROUPS * NPC) {
                const int i = i0 + lane, m = done + u, s = g * n_stages + m % n_stages;
                const bool mine = g < GROUPS && i < n;
                if (mine && !mbar_wait(empty0 + 8 * s, ((m / n_stages) & 1) ^ 1)) timed_out = true;
                stop = __any_sync(0xffffffffu, timed_out);
                if (stop) break;
                if (mine) {
                    mbar_expect_tx(full0 + 8 * s, row_bytes);
                    bulk_load_row_hint(ring0 + (uint32_t)s * row_bytes,
                                       Wd + (size_t)guard_row(s_list[first + i], F, p.status) * row_bytes, row_bytes, full0 + 8 * s,
                                       policy);
                }
                done += min(NPC, max(0, n - i0 - g * NPC));
            }
        }
        // Never leave with copies in flight: the last use of every stage must have landed.
        if (u == 0 && g < GROUPS)
            for (int m = max(0, done - n_stages); m < done; ++m)
                if (!mbar_wait(full0 + 8 * (g * n_stages + m % n_stages), (m / n_stages) & 1)) timed_out = true;
    } else {
        // ---- consumers -----------------------------------------------------------------------------------
        const int grp = tid / GT, gt = tid - grp * GT;
        bool vok[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) vok[k] = gt + k * GT < vpr;
        const uint32_t ring = ring0 + (uint32_t)(grp * n_stages) * row_bytes + (uint32_t)gt * 16u;
        const uint32_t full = full0 + 8 * grp * n_stages, empty = empty0 + 8 * grp * n_stages;
        pdl_wait();  // the hidden values
        pdl_launch_dependents();
        for (int b = 0; b < p.nb; ++b) {
            const int first = s_first[b], n = s_first[b + 1] - first;
            for (int i = tid; i < n; i += kConsumers) s_h[first + i] = __ldcg(p.hidden + (size_t)b * F + s_list[first + i]);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kConsumers) : "memory");
        int s = 0;
        uint32_t par = 0;
        for (int b = 0; b < p.nb; ++b) {
            const int first = s_first[b], n = s_first[b + 1] - first;
            float2 acc[NV][P];
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int e = 0; e < P; ++e) acc[k][e] = make_float2(0.f, 0.f);
            for (int i0 = grp * NPC; i0 < n; i0 += GROUPS * NPC) {
                const int s0 = s;
                uint4 q[NPC][NV];
#pragma unroll
                for (int u = 0; u < NPC; ++u) {
                    if (i0 + u >= n) continue;
                    if (!timed_out && !mbar_wait(full + 8 * s, par)) timed_out = true;
#pragma unroll
                    for (int k = 0; k < NV; ++k)
                        if (vok[k]) q[u][k] = lds128(ring + (uint32_t)s * row_bytes + (uint32_t)(k * GT) * 16u);
                    if (++s == n_stages) {
                        s = 0;
                        par ^= 1;
                    }
                }
                __syncwarp();
                if (lane < NPC && i0 + lane < n) mbar_arrive(empty + 8 * (s0 + lane < n_stages ? s0 + lane : s0 + lane - n_stages));
#pragma unroll
                for (int u = 0; u < NPC; ++u) {
                    if (i0 + u >= n) continue;
                    const float hv = s_h[first + i0 + u];
                    const float2 h2 = make_float2(hv, hv);
#pragma unroll
                    for (int k = 0; k < NV; ++k) {
                        if (!vok[k]) continue;
                        float2 fd[P];
                        Pairs<T>::unpack(q[u][k], fd);
#pragma unroll
                        for (int e = 0; e < P; ++e) acc[k][e] = __ffma2_rn(h2, fd[e], acc[k][e]);
                    }
                }
            }
            float *mine = p.partials + (((size_t)b * p.n_shares + c) * GROUPS + grp) * p.d_model;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                if (!vok[k]) continue;
                float4 *dst = reinterpret_cast<float4 *>(mine + (size_t)(gt + k * GT) * E);
#pragma unroll
                for (int e = 0; e < P; e += 2) dst[e / 2] = make_float4(acc[k][e].x, acc[k][e].y, acc[k][e + 1].x, acc[k][e + 1].y);
            }
        }
    }
    if (timed_out && p.status) atomicOr(p.status, CLADA_STATUS_TIMEOUT);
}

// Column sums of the partial rows in the single launch's order: "lane" l adds rows l, l + 32, ... in order, the 32 sums
// combine as by a butterfly (partners 16, 8, 4, 2, 1 away).  Eight neighbouring threads read a whole line of one row.
constexpr int kNbSumThreads = 256, kNbSumVecs = kNbSumThreads / kWarp;
__global__ void __launch_bounds__(kNbSumThreads)
nested_sums_kernel(const NbParams p, const int n_rows) {
    __shared__ float4 s_sum[kWarp][kNbSumVecs];
    const int v = threadIdx.x % kNbSumVecs, l = threadIdx.x / kNbSumVecs, d4 = p.d_model / 4;
    const int b = blockIdx.y, g = blockIdx.x * kNbSumVecs + v;
    pdl_wait();
    pdl_launch_dependents();
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g < d4) {
        const float4 *part = reinterpret_cast<const float4 *>(p.partials) + (size_t)b * n_rows * d4 + g;
        for (int rb = 0; rb < n_rows; rb += 10 * kWarp) {
            float4 q[10];
#pragma unroll
            for (int u = 0; u < 10; ++u) {
                const int r = rb + u * kWarp + l;
                q[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (r < n_rows) q[u] = __ldcg(part + (size_t)r * d4);
            }
#pragma unroll
            for (int u = 0; u < 10; ++u) {
                s.x += q[u].x; s.y += q[u].y; s.z += q[u].z; s.w += q[u].w;
            }
        }
    }
    s_sum[l][v] = s;
#pragma unroll
    for (int o = kWarp / 2; o > 0; o >>= 1) {
        __syncthreads();
        if (l < o) {
            const float4 t = s_sum[l + o][v];
            s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
            s_sum[l][v] = s;
        }
    }
    if (l == 0 && g < d4) {
        char *yb = static_cast<char *>(p.y) + (size_t)b * p.d_model * (p.y_dtype == CLADA_F32 ? 4 : 2);
        if (p.y_dtype == CLADA_F32)
            reinterpret_cast<float4 *>(yb)[g] = s;
        else
            reinterpret_cast<uint2 *>(yb)[g] = pack4_16bit(p.y_dtype, s);
    }
}

// ---- host side ------------------------------------------------------------------------------

static size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }
static int nb_vpr(const clada_layer *L) { return L->d_model / (L->dtype == CLADA_F32 ? 4 : 8); }

struct NbPlan {
    int n_stages, n_cons, n_rows;  // stages and consumer warps of the hidden pass; rows of a group's ring of the down pass
    size_t smem_hidden, smem_down, smem_keep;
};

// Which batches take a pass; measured against a launch per sequence, both in graphs, layers of 4096 to 24576 neurons, lists of
// independent random neurons, of ones half shared, of the same ones and of none in common (times a pass / its launches):
//   four and more  0.55 to 0.98 up to 6144 columns (lists without a neuron in common up to 1.10), while the ring has five stages
//                  beside x; with four 1.1 to 1.2 (7168 gated columns from six sequences on, 8192 from four)
//   three          0.80 to 1.0 on rows of up to 256 vectors and of 512 and more, with six stages (with five, 8192 gated columns,
//                  1.04 to 1.06); on rows of 257 to 511 a single launch is at its best: layers without a gate 1.03 to 1.14, gated ones
//                  0.94 to 1.0 up to 80 MB a matrix (2304 x 16384, 3072 x 12288), 1.01 to 1.06 beyond
//   two            steps of 1024 x 4100 26.7 / 26.6 us, 2048 x 16384 51.5 / 52.6, 4096 x 11008 59.8 / 68.7, 5120 x 13824 88.5 / 96.9
static bool nb_plan(const clada_layer *L, int nb, const DeviceInfo &di, NbPlan *pl) {
    const int vpr = nb_vpr(L);
    const bool gated = act_is_gated(L->activation);
    if (nb < kNestedBatchMin || nb > kNestedBatchMax || vpr > 2 * kConsumers || L->d_ff > kSingleMaxDff) return false;
    const size_t row = (size_t)vpr * 16, stage = (gated ? 2 : 1) * row;
    if (nb == 3 && vpr > kConsumers / 2 && vpr < kConsumers && (!gated || row * L->d_ff > ((size_t)80 << 20))) return false;
    const size_t cap = (size_t)(L->d_ff / di.num_sms + 2);
    const size_t tail = (size_t)nb * row + 2 * kNbMaxStages * sizeof(uint64_t) + 2 * cap * sizeof(int);
    const size_t budget = (size_t)di.max_smem_optin - kNbStatic;
    if (budget < tail + (nb == 3 ? 6 : 5) * stage) return false;
    const int fit = (int)std::min<size_t>(kNbMaxStages, (budget - tail) / stage);
    pl->n_cons = std::min(fit - std::max(2, fit / 3), kNbConsWarps);  // the other stages are on their way
    pl->n_stages = fit;
    pl->smem_hidden = (size_t)pl->n_stages * stage + tail;
    const int groups = ffn_groups(vpr);
    const size_t down_tail = 2 * kNbMaxStages * sizeof(uint64_t) + 2 * (size_t)nb * cap * sizeof(int);
    if (budget < down_tail + 8 * groups * row) return false;  // a chunk is up to eight rows
    pl->n_rows = (int)std::min<size_t>(kNbMaxStages, (budget - down_tail) / row) / groups;
    pl->smem_down = (size_t)groups * pl->n_rows * row + down_tail;
    pl->smem_keep = (size_t)((L->d_ff + 31) / 32) * sizeof(unsigned);
    return true;
}

bool nested_batch_supported(const clada_layer *layer, int nb) {
    DeviceInfo di;
    NbPlan pl;
    return device_info(&di) == CLADA_OK && nb_plan(layer, nb, di, &pl);
}

size_t nested_batch_scratch_bytes(const clada_layer *L, int nb, int num_sms) {
    return align256((size_t)nb * L->d_ff * sizeof(float)) + align256((size_t)nb * ((L->d_ff + 31) / 32) * sizeof(unsigned)) +
           align256((size_t)nb * num_sms * ffn_groups(nb_vpr(L)) * L->d_model * sizeof(float));
}

static int nb_launch(const void *kernel, dim3 grid, int threads, size_t smem, cudaStream_t st, void **args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CLADA_CUDA_TRY(cudaLaunchKernelExC(&cfg, kernel, args));
    return CLADA_OK;
}

template <typename T, int NV, bool GATED, int GROUPS>
static int nb_launch_variant(NbParams p, const NbPlan &pl, const DeviceInfo &di, cudaStream_t st) {
    constexpr int kVw = kConsumers / GROUPS / kWarp;
    constexpr int kNpc = (!GATED && NV == 1) ? 2 * GS : GS;
    static bool configured[64] = {};
    auto hidden = nested_hidden_kernel<T, kVw, NV, GATED>;
    auto down = nested_down_kernel<T, NV, GROUPS, kNpc>;
    if (!configured[di.device & 63]) {
        CLADA_CUDA_TRY(cudaFuncSetAttribute(hidden, cudaFuncAttributeMaxDynamicSharedMemorySize, di.max_smem_optin - kNbStatic));
        CLADA_CUDA_TRY(cudaFuncSetAttribute(down, cudaFuncAttributeMaxDynamicSharedMemorySize, di.max_smem_optin - kNbStatic));
        configured[di.device & 63] = true;
    }
    int n_stages = pl.n_stages, n_cons = pl.n_cons, n_ring = pl.n_rows, n_rows = p.n_shares * GROUPS;
    void *args1[] = {&p};
    void *args2[] = {&p, &n_stages, &n_cons};
    void *args3[] = {&p, &n_ring};
    void *args4[] = {&p, &n_rows};
    int rc = nb_launch(reinterpret_cast<const void *>(nested_keep_kernel), dim3(p.nb), kNbKeepThreads, pl.smem_keep, st, args1);
    if (rc == CLADA_OK)
        rc = nb_launch(reinterpret_cast<const void *>(hidden), dim3(di.num_sms), kNbThreads, pl.smem_hidden, st, args2);
    if (rc == CLADA_OK)
        rc = nb_launch(reinterpret_cast<const void *>(down), dim3(p.n_shares), kFfnThreads, pl.smem_down, st, args3);
    if (rc == CLADA_OK)
        rc = nb_launch(reinterpret_cast<const void *>(nested_sums_kernel), dim3((p.d_model / 4 + kNbSumVecs - 1) / kNbSumVecs, p.nb),
                       kNbSumThreads, 0, st, args4);
    return rc;
}

template <typename T>
static int nb_launch_typed(const NbParams &p, int vpr, const NbPlan &pl, const DeviceInfo &di, cudaStream_t st) {
    const bool gated = act_is_gated(p.act);  // the instances of launch_ffn_single
    if (vpr <= kConsumers / 2)
        return gated ? nb_launch_variant<T, 1, true, 2>(p, pl, di, st) : nb_launch_variant<T, 1, false, 2>(p, pl, di, st);
    if (vpr <= kConsumers)
        return gated ? nb_launch_variant<T, 1, true, 1>(p, pl, di, st) : nb_launch_variant<T, 1, false, 1>(p, pl, di, st);
    return gated ? nb_launch_variant<T, 2, true, 1>(p, pl, di, st) : nb_launch_variant<T, 2, false, 1>(p, pl, di, st);
}

int launch_nested_batch(const clada_layer *layer, int nb, const void *x, const int32_t *order, const int32_t *counts,
                        const int32_t *level, void *y, int y_dtype, int32_t *count_out, void *ws, int32_t *status,
                        cudaStream_t st) {
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != CLADA_OK) return rc;
    NbPlan pl;
    if (!nb_plan(layer, nb, di, &pl)) return CLADA_ERR_UNSUPPORTED;
    char *base = static_cast<char *>(ws) + kWsCtrlBytes;
    NbParams p;
    p.w_gate = layer->w_gate;
    p.w_up = layer->w_up;
    p.w_down_t = layer->w_down_t;
    p.x = x;
    p.order = order;
    p.counts = counts;
    p.level = level;
    p.y = y;
    p.y_dtype = y_dtype;
    p.count_out = count_out;
    p.hidden = reinterpret_cast<float *>(base);
    base += align256((size_t)nb * layer->d_ff * sizeof(float));
    p.words = reinterpret_cast<unsigned *>(base);
    base += align256((size_t)nb * ((layer->d_ff + 31) / 32) * sizeof(unsigned));
    p.partials = reinterpret_cast<float *>(base);
    p.status = status;
    p.d_model = layer->d_model;
    p.d_ff = layer->d_ff;
    p.act = layer->activation;
    p.nb = nb;
    p.n_shares = di.num_sms;
    const int vpr = nb_vpr(layer);
    return layer->dtype == CLADA_F32    ? nb_launch_typed<float>(p, vpr, pl, di, st)
           : layer->dtype == CLADA_BF16 ? nb_launch_typed<__nv_bfloat16>(p, vpr, pl, di, st)
                                        : nb_launch_typed<__half>(p, vpr, pl, di, st);
}

}  // namespace clada
