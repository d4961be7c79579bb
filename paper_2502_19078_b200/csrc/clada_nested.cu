// Nested index lists: the four masks of a sequence in one list.
//
// Eq. final_threshold yields tau_base * m with m in {1, 1+lambda, 1+gamma, (1+lambda)+gamma}, and a kept set
// is { j : A_j >= tau }, so every kept set is a leading part of the neurons listed in descending order of
// score.  Once after prefill, per sequence:
//   order  = neurons by descending score, equal scores by ascending index        [d_ff] int32
//   counts = |{ j : A_j >= tau_base * m_k }| for the four multipliers            [4]    int32
// A decode step then needs the load level k = I(s > tau_s) + 2 I(H > tau_H) (clada_cogload_level) and reads
// order[0 .. counts[k]): no per-step threshold test, ranking or compaction, and the per-sequence state
// is one int32 list instead of the fp32 scores plus masks.
//
// Up to kSortMaxN neurons are sorted in shared memory (block_sort.cuh).  Wider layers, and small calls (nested_by_rank),
// take a rank sort: a neuron's place in the list is the number of neurons that come before it -- those with a larger score, or an equal score and
// a smaller index -- so every place can be computed independently and exactly.  A sequence is shared by several CTAs;
// each holds the whole score vector in shared memory (as bit patterns: scores are norms, so the patterns of the
// positive ones order them; see score_key for the rest) and ranks its slice, one warp per neuron, lanes striding over
// the vector.  The four counts come from the first CTA of the sequence by a block-wide sum.  The multipliers are
// formed on the host exactly as the adjustment kernel forms them (fp32, one addition at a time), the thresholds with
// one fp32 multiplication.
#include <math.h>

#include <algorithm>

#include "block_sort.cuh"
#include "common.cuh"
#include "nvtx_ranges.cuh"

namespace clada {

constexpr int kNestThreads = 1024;
constexpr int kNestMaxN = 32768;  // the score vector must fit shared memory (4 bytes per neuron)

struct NestMults {
    float m[4];
};

// Sort key of a score: scores are norms, so the bit patterns of the positive ones order them.  What is not a
// positive number is put where the selection A_j >= tau puts it: NaN compares false with every threshold and
// sorts after everything (key 0); zero of either sign and anything negative sort just before it (key 1).
__device__ __forceinline__ unsigned score_key(float a) {
    if (a > 0.f) return __float_as_uint(a) + 1u;
    return a != a ? 0u : 1u;
}

__global__ void __launch_bounds__(kNestThreads)
nested_build_kernel(const float *__restrict__ scores, int d_ff, const float *__restrict__ tau_base,
                    long long tau_stride, const NestMults mults, int32_t *__restrict__ order,
                    int32_t *__restrict__ counts) {
    extern __shared__ unsigned s_key[];
    __shared__ int s_part[kNestThreads / kWarp][4];
    const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *A = scores + (size_t)b * d_ff;
    for (int i = tid; i < d_ff; i += kNestThreads) s_key[i] = score_key(A[i]);
    __syncthreads();
    const int e0 = (int)(((long long)d_ff * blockIdx.x) / gridDim.x);
    const int e1 = (int)(((long long)d_ff * (blockIdx.x + 1)) / gridDim.x);
    // before(e) = #{k < e : key_k >= key_e} + #{k > e : key_k > key_e}: one comparison per pair, four pairs per
    // 16-byte shared-memory load; the vector that holds e and the ragged end of the row go element by element.
    const uint4 *s_vec = reinterpret_cast<const uint4 *>(s_key);
    const int nvec = d_ff / 4;
    for (int e = e0 + warp; e < e1; e += kNestThreads / kWarp) {
        const unsigned a = s_key[e];
        const int ev = e >> 2;
        int before = 0;
        for (int v = lane; v < min(ev, nvec); v += kWarp) {
            const uint4 q = s_vec[v];
            before += (q.x >= a) + (q.y >= a) + (q.z >= a) + (q.w >= a);
        }
        for (int v = ev + 1 + lane; v < nvec; v += kWarp) {
            const uint4 q = s_vec[v];
            before += (q.x > a) + (q.y > a) + (q.z > a) + (q.w > a);
        }
        {
            int k = -1;  // lanes 0..3: the vector around e; lanes 4..: the elements after the last whole vector
            if (lane < 4) {
                if (ev < nvec) k = ev * 4 + lane;
            } else if (nvec * 4 + lane - 4 < d_ff) {
                k = nvec * 4 + lane - 4;
            }
            if (k >= 0 && k != e) {
                const unsigned v = s_key[k];
                before += k < e ? (v >= a) : (v > a);
            }
        }
        before = warp_sum(before);
        if (lane == 0) order[(size_t)b * d_ff + before] = e;
    }
    if (blockIdx.x == 0) {
        float tau[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) tau[k] = __fmul_rn(tau_base[(size_t)b * tau_stride], mults.m[k]);
        int c[4] = {0, 0, 0, 0};
        for (int i = tid; i < d_ff; i += kNestThreads) {
            const float a = A[i];
#pragma unroll
            for (int k = 0; k < 4; ++k) c[k] += (a >= tau[k]) ? 1 : 0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int w = warp_sum(c[k]);
            if (lane == 0) s_part[warp][k] = w;
        }
        __syncthreads();
        if (tid < 4) {
            int tot = 0;
            for (int w = 0; w < kNestThreads / kWarp; ++w) tot += s_part[w][tid];
            counts[(size_t)b * 4 + tid] = tot;
        }
    }
}

// Layers of at most kSortMaxN neurons: one or a few CTAs per sequence sort in shared memory
// (block_sort); each CTA of a sequence prepares the same table and writes its slice of the list, CTA 0 also counts.
// Measured (lists of 8 sequences of 14336 neurons, back-to-back calls): 194.5 us a call with the bitonic network alone,
// 16.4 us with four CTAs that each scatter everything, 12.5 with eight (13.2 with six CTAs, 14.0 with four), 11.5 now.
__global__ void __launch_bounds__(kSortThreads, 1)
nested_sort_kernel(const float *__restrict__ scores, int d_ff, const float *__restrict__ tau_base,
                   long long tau_stride, const NestMults mults, int32_t *__restrict__ order,
                   int32_t *__restrict__ counts) {
    extern __shared__ __align__(16) unsigned char s_sort[];
    __shared__ int s_part[kSortThreads / kWarp][4];
    const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *A = scores + (size_t)b * d_ff;
    pdl_launch_dependents();
    pdl_wait();
    float tau[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) tau[k] = __fmul_rn(tau_base[(size_t)b * tau_stride], mults.m[k]);
    int c[4] = {0, 0, 0, 0};
    // complementing the score's key turns ascending keys into descending scores; what is not a positive number has
    // key 0 or 1, an infinity the largest
    const int r0 = (int)(((long long)d_ff * blockIdx.x) / gridDim.x);
    const int r1 = (int)(((long long)d_ff * (blockIdx.x + 1)) / gridDim.x);
    block_sort(
        d_ff, ~0x7f800000u, ~2u, r0, r1, s_sort, [&](int i) { return A[i]; },
        [&](float a) {
#pragma unroll
            for (int k = 0; k < 4; ++k) c[k] += (a >= tau[k]) ? 1 : 0;
            return ~score_key(a);
        },
        [&](int rank, int i, unsigned) { order[(size_t)b * d_ff + rank] = i; });
    if (blockIdx.x != 0) return;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int w = warp_sum(c[k]);
        if (lane == 0) s_part[warp][k] = w;
    }
    __syncthreads();
    if (tid < 4) {
        int tot = 0;
        for (int w = 0; w < kSortThreads / kWarp; ++w) tot += s_part[w][tid];
        counts[(size_t)b * 4 + tid] = tot;
    }
}

// CTAs per sequence of the rank sort: enough to occupy the device, at least 32 neurons each.
static int nested_rank_split(const DeviceInfo &di, int B, int d_ff) {
    return std::max(1, std::min((di.num_sms + B - 1) / B, (d_ff + 31) / 32));
}
// CTAs per sequence of the sort.  A CTA of a sequence repeats the counting for the sake of shorter last passes: eight at
// most (twelve and sixteen measured for 1 to 16 sequences: 5 % at 11008 and 16384 neurons, nothing below).
static int nested_sort_parts(const DeviceInfo &di, int B, int d_ff) {
    return std::max(1, std::min({8, di.num_sms / B, (d_ff + 1023) / 1024}));
}
// Whether the rank sort is the faster one.  Its warps go through the whole vector once per neuron of their CTA's share, one
// launch-bound round trip otherwise (3 us), where the sort's passes over its counters and pieces take 6.5 to 8 us whatever the
// size; so it takes the calls of few rounds, fewer when its CTAs do not all fit the device at once.  Measured at 148 SMs
// (us, rank / sort): one sequence of 1376 4.4/7.2, 4096 6.3/8.1, 5000 8.4/8.3; two of 3000 7.4/7.8, 4096 8.7/8.1; four of
// 2048 6.9/7.6, 2560 8.6/7.6; 16 of 512 6.3/6.7, 24 of 512 7.9/6.7; 74 of 256 5.8/6.7, 100 of 256 9.3/6.7; 300 of 64
// 7.8/18.3.  Over 390 shapes of 64 to 4700 neurons and 1 to 300 sequences the rule is within 5 % of the faster one.
static bool nested_by_rank(const DeviceInfo &di, int B, int d_ff) {
    const long long split = nested_rank_split(di, B, d_ff), ctas = split * B;
    const long long rounds = ((d_ff + split - 1) / split + kNestThreads / kWarp - 1) / (kNestThreads / kWarp);
    const long long sort_waves = ((long long)nested_sort_parts(di, B, d_ff) * B + di.num_sms - 1) / di.num_sms;
    return rounds * (d_ff + 1500) <= (ctas <= di.num_sms ? 9000 : 2400 + 2500 * sort_waves);
}

}  // namespace clada

using namespace clada;

extern "C" int clada_nested_build(const float *scores, int32_t B, int32_t d_ff, const float *tau_base,
                                  int64_t tau_stride, float lambda, float gamma, int32_t *order, int32_t *counts,
                                  void *stream) {
    CLADA_RANGE("clada_nested_build");
    if (!scores || !tau_base || !order || !counts) return CLADA_ERR_NULL;
    if (B <= 0 || d_ff <= 0 || tau_stride < 0) return CLADA_ERR_SHAPE;
    if (d_ff > kNestMaxN || B > 65535) return CLADA_ERR_UNSUPPORTED;
    NestMults mults;
    {
        // level k = I(s > tau_s) + 2 I(H > tau_H); the sums are taken as the adjustment takes them:
        // start from 1, add lambda if the first indicator holds, then gamma if the second does
        volatile float one = 1.0f;
        volatile float m1 = one + lambda;
        volatile float m2 = one + gamma;
        volatile float m3 = m1 + gamma;
        mults.m[0] = one;
        mults.m[1] = m1;
        mults.m[2] = m2;
        mults.m[3] = m3;
    }
    static bool configured[64] = {};
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != CLADA_OK) return rc;
    if (!configured[di.device & 63]) {
        CLADA_CUDA_TRY(cudaFuncSetAttribute(nested_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            kNestMaxN * (int)sizeof(unsigned)));
        CLADA_CUDA_TRY(cudaFuncSetAttribute(nested_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)kSortSmem));
        configured[di.device & 63] = true;
    }
    if (d_ff <= kSortMaxN && !nested_by_rank(di, B, d_ff)) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(nested_sort_parts(di, B, d_ff), B);
        cfg.blockDim = dim3(kSortThreads);
        cfg.dynamicSmemBytes = kSortSmem;
        cfg.stream = static_cast<cudaStream_t>(stream);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        CLADA_CUDA_TRY(cudaLaunchKernelEx(&cfg, nested_sort_kernel, scores, (int)d_ff, tau_base, (long long)tau_stride, mults,
                                          order, counts));
        return CLADA_OK;
    }
    nested_build_kernel<<<dim3(nested_rank_split(di, B, d_ff), B), kNestThreads, (size_t)d_ff * sizeof(unsigned),
                          static_cast<cudaStream_t>(stream)>>>(scores, d_ff, tau_base, tau_stride, mults, order,
                                                               counts);
    CLADA_CUDA_TRY(cudaGetLastError());
    return CLADA_OK;
}
