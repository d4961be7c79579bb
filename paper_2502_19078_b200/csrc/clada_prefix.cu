// Prefill statistics (Eq. neuron_activation) on CUDA cores, fp32 accumulation, any dtype:
//   z[t,j] = silu(x_t . w_gate_j) * (x_t . w_up_j),   A[b,j] = sqrt(sum_{t in b} z[t,j]^2) * ||W_out,j||
// plus the fp64 guard-band refinement and the one-call prefill entry point.
//
// The GEMM never writes z: each CTA owns a (token tile, neuron tile) pair that lies inside one
// prompt, keeps both accumulators (gate and up) in registers, and its epilogue squares and sums
// over the tile's tokens into one fp32 partial per neuron.  A second kernel adds a prompt's
// partials in tile order, so scores are bit-identical run to run.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "nvtx_ranges.cuh"
#include "prefix_common.cuh"

namespace clada {

constexpr int BM = 64, BK = 16;

// Shared memory of a K block, transposed and in the layer's own element type: x, gate, up.  Two K blocks; the token
// sums take the same bytes afterwards.
template <typename T, int BN>
constexpr size_t pf_smem() {
    const size_t ring = 2 * (size_t)BK * (BM + 2 * BN) * sizeof(T), sums = 16 * (size_t)BN * sizeof(float);
    return ring > sums ? ring : sums;
}
// N = 4 or 8 consecutive elements from shared memory as fp32.
template <typename T, int N> __device__ __forceinline__ void pf_load(const T *p, float (&f)[N]) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(p + i);
            f[i] = v.x; f[i + 1] = v.y; f[i + 2] = v.z; f[i + 3] = v.w;
        }
    } else if constexpr (N == 8) {
        Elem<T>::unpack(*reinterpret_cast<const uint4 *>(p), f);
    } else {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        float h[8];
        Elem<T>::unpack(make_uint4(v.x, v.y, 0u, 0u), h);
#pragma unroll
        for (int i = 0; i < 4; ++i) f[i] = h[i];
    }
}

// A CTA owns 64 tokens x BN neurons (gate and up), a thread 8 tokens x NT neurons.  Bound by the FMA pipes, so
// everything else stays out of the way: packed two-wide FMAs, operands in shared memory in their 16 bits (a 16-byte
// load returns 512 bytes to a warp's registers, four cycles whatever is broadcast: fp32 operands kept that path busy
// for most of the FMAs' time), the next K block fetched into registers while this one is multiplied.  Every
// accumulator is one chain over k in ascending order.
// NT = 8 (BN = 128) halves the shared-memory loads per FMA; NT = 4 (BN = 64) has the smaller steps (launch_prefix_partials
// chooses).
// Measured with z written (2048 tokens, 4096 x 11008, bf16; 369 GFLOP): 9.53 ms with 4 x 4 per thread and fp32 operands
// in shared memory, 7.5 ms as one CTA of 256 neurons per SM, 6.3 ms (59 TFLOP/s) as two CTAs of 128.  fp32 layers, the
// whole call: 9.66 ms with 4 x 4 per thread, 8.19 now; one prompt of 64 tokens on 512 x 1376: 62.6 us, 51.7 now.
// z of 16-bit layers on the tensor cores was tried twice.  Rows as three 8-bit digits with integer sums (0.9 ms) lose what
// is small beside a row's largest element: scores off by 2e-5 (an outlier channel 3000 times the others) to 5e-4 (10000
// times, over weights 1000 times smaller), 1e-6 here.  16-bit products, each MMA's 16 added up in fp32 (1.4 ms), are
// truncated once: z low by 3e-8 (bf16) to 8e-8 (fp16), and the search's curve off by 6e-8 to 1.7e-7, 4e-9 to 3e-8 here.
template <typename T, int NT, int BN>
__global__ void __launch_bounds__(8 * BN / NT, NT == 8 ? 2 : 3)
prefix_partials_kernel(const T *__restrict__ X, const T *__restrict__ Wg, const T *__restrict__ Wu,
                       int d_model, int d_ff, const SeqTable tab, float *__restrict__ partials,
                       float *__restrict__ zt, long long zt_stride, int act) {
    constexpr int kThreads = 8 * BN / NT;
    constexpr int E = Elem<T>::kPerVec;
    constexpr int kVecsX = BM * BK / E, kVecsW = BN * BK / E;             // 16-byte vectors of a K block
    constexpr int kVecX = (kVecsX + kThreads - 1) / kThreads, kVecW = (kVecsW + kThreads - 1) / kThreads;  // per thread
    // neurons of a thread: NT consecutive ones, or (fp32, NT = 8) two runs of four that keep a warp's loads contiguous
    constexpr int kRun = NT * sizeof(T) > 16 ? 4 : NT;
    extern __shared__ __align__(16) unsigned char s_pf_raw[];
    T *s_pf = reinterpret_cast<T *>(s_pf_raw);
    constexpr int kXs = BK * BM, kWs = BK * BN;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ty = (warp & 1) * 4 + (lane >> 3);   // tokens 8 ty .. 8 ty + 7
    const int tx = (warp >> 1) * 8 + (lane & 7);
    auto neuron = [&](int j) { return (j / kRun) * (BN / (NT / kRun)) + tx * kRun + j % kRun; };
    const int n0 = blockIdx.x * BN;
    int b;
    long long t0, t1;
    locate_tile(tab, blockIdx.y, BM, b, t0, t1);

    // Vector v of an operand's K block: row v % rows, column v / rows of 16 bytes, so that consecutive threads store
    // consecutive rows (no bank conflicts in the transposed layout).
    uint4 qx[kVecX], qg[kVecW], qu[kVecW];
    auto fetch = [&](int k0) {  // d_model % 8 == 0: a vector is all in or all out
#pragma unroll
        for (int i = 0; i < kVecX; ++i) {
            const int v = tid + i * kThreads, r = v % BM, c = k0 + v / BM * E;
            qx[i] = make_uint4(0, 0, 0, 0);
            if (v < kVecsX && c < d_model && t0 + r < t1)
                qx[i] = *reinterpret_cast<const uint4 *>(X + (size_t)(t0 + r) * d_model + c);
        }
#pragma unroll
        for (int i = 0; i < kVecW; ++i) {
            const int v = tid + i * kThreads, r = v % BN, c = k0 + v / BN * E;
            qg[i] = qu[i] = make_uint4(0, 0, 0, 0);
            if (v < kVecsW && c < d_model && n0 + r < d_ff) {
                qg[i] = *reinterpret_cast<const uint4 *>(Wg + (size_t)(n0 + r) * d_model + c);
                if (Wu) qu[i] = *reinterpret_cast<const uint4 *>(Wu + (size_t)(n0 + r) * d_model + c);  // null: no gate projection
            }
        }
    };
    auto store = [&](T *buf) {
        T *gs = buf + kXs, *us = gs + kWs;
#pragma unroll
        for (int i = 0; i < kVecX; ++i) {
            const int v = tid + i * kThreads, r = v % BM, c = v / BM * E;
            if (v >= kVecsX) break;
            const T *f = reinterpret_cast<const T *>(&qx[i]);
#pragma unroll
            for (int e = 0; e < E; ++e) buf[(c + e) * BM + r] = f[e];
        }
#pragma unroll
        for (int i = 0; i < kVecW; ++i) {
            const int v = tid + i * kThreads, r = v % BN, c = v / BN * E;
            if (v >= kVecsW) break;
            const T *f = reinterpret_cast<const T *>(&qg[i]), *h = reinterpret_cast<const T *>(&qu[i]);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                gs[(c + e) * BN + r] = f[e];
                us[(c + e) * BN + r] = h[e];
            }
        }
    };

    float2 ag[8][NT / 2], au[8][NT / 2];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NT / 2; ++j) ag[i][j] = au[i][j] = make_float2(0.f, 0.f);

    T *cur = s_pf, *nxt = s_pf + kXs + 2 * kWs;
    fetch(0);
    store(cur);
    __syncthreads();
    for (int k0 = 0; k0 < d_model; k0 += BK) {
        const bool more = k0 + BK < d_model;
        if (more) fetch(k0 + BK);
        const T *xs = cur + ty * 8, *gs = cur + kXs, *us = gs + kWs;
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            float x[8], g[NT], u[NT];
            pf_load(xs + k * BM, x);
#pragma unroll
            for (int r = 0; r < NT; r += kRun) {
                float t[kRun];
                pf_load(gs + k * BN + neuron(r), t);
#pragma unroll
                for (int e = 0; e < kRun; ++e) g[r + e] = t[e];
                pf_load(us + k * BN + neuron(r), t);
#pragma unroll
                for (int e = 0; e < kRun; ++e) u[r + e] = t[e];
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float2 xx = make_float2(x[i], x[i]);
#pragma unroll
                for (int j = 0; j < NT / 2; ++j) {
                    ag[i][j] = __ffma2_rn(xx, make_float2(g[2 * j], g[2 * j + 1]), ag[i][j]);
                    au[i][j] = __ffma2_rn(xx, make_float2(u[2 * j], u[2 * j + 1]), au[i][j]);
                }
            }
        }
        if (more) store(nxt);
        __syncthreads();
        T *t = cur;
        cur = nxt;
        nxt = t;
    }
    // epilogue: z^2 summed over groups of 4 tokens, then over the tile's 16 groups in order
    // (the offline threshold search also wants z itself, neuron-major: zt[j, t])
    float *s_red = reinterpret_cast<float *>(s_pf_raw);  // [16][BN]; every thread is past its last read of the ring
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int n = neuron(j);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float s = 0.f;
#pragma unroll
            for (int i = 4 * q; i < 4 * q + 4; ++i) {
                const float g = j & 1 ? ag[i][j >> 1].y : ag[i][j >> 1].x, u = j & 1 ? au[i][j >> 1].y : au[i][j >> 1].x;
                const float z = neuron_value_f(act, g, u);  // padded token rows give exactly 0
                s = fmaf(z, z, s);
                const long long t = t0 + ty * 8 + i;
                if (zt && t < t1 && n0 + n < d_ff) zt[(size_t)(n0 + n) * zt_stride + t] = z;
            }
            s_red[(2 * ty + q) * BN + n] = s;
        }
    }
    __syncthreads();
    for (int n = tid; n < BN && n0 + n < d_ff; n += kThreads) {
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r) s += s_red[r * BN + n];
        partials[(size_t)blockIdx.y * d_ff + n0 + n] = s;
    }
}

template <typename T, int NT, int BN>
static int launch_prefix_variant(const clada_layer *L, const void *X, const SeqTable &tab, int n_mtiles, float *partials,
                                 float *zt, long long zt_stride, const DeviceInfo &di, cudaStream_t st) {
    static bool configured[64] = {};
    if (!configured[di.device & 63]) {  // the K blocks may need the opt-in
        CLADA_CUDA_TRY(cudaFuncSetAttribute(prefix_partials_kernel<T, NT, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)pf_smem<T, BN>()));
        configured[di.device & 63] = true;
    }
    const dim3 grid((L->d_ff + BN - 1) / BN, n_mtiles);
    prefix_partials_kernel<T, NT, BN><<<grid, 8 * BN / NT, pf_smem<T, BN>(), st>>>(
        static_cast<const T *>(X), static_cast<const T *>(L->w_gate), static_cast<const T *>(L->w_up), L->d_model, L->d_ff,
        tab, partials, zt, zt_stride, L->activation);
    CLADA_CUDA_TRY(cudaGetLastError());
    return CLADA_OK;
}

template <typename T>
static int launch_prefix_partials(const clada_layer *L, const void *X, const SeqTable &tab, int n_mtiles, float *partials,
                                  float *zt, long long zt_stride, cudaStream_t st) {
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != CLADA_OK) return rc;
    // An SM's time goes with the tiles it gets, and a tile of NT = 8 takes 1.85 times one of NT = 4: the variant whose whole
    // number of tiles per SM comes out cheaper.  With one tile an SM NT = 8 has half the warps it needs.  Measured (fp32, us,
    // NT = 8 / 4): 512 x 1376 with 1000 tokens (2 against 3 tiles) 127 / 102, 1500 (2, 4) 127 / 133, 2000 (3, 5) 187 / 162,
    // 4096 (5, 10) 296 / 311; 1024 x 4096 with 400 (2, 4) 233 / 245, 640 (3, 5) 345 / 307; 4096 x 11008 with 200 (3, 5) 1330 /
    // 1180, 512 (5, 10) 2186 / 2356.
    const long long per_sm8 = ((long long)n_mtiles * ((L->d_ff + 127) / 128) + di.num_sms - 1) / di.num_sms;
    const long long per_sm4 = ((long long)n_mtiles * ((L->d_ff + 63) / 64) + di.num_sms - 1) / di.num_sms;
    if (per_sm8 > 1 && 20 * per_sm4 > 37 * per_sm8)
        return launch_prefix_variant<T, 8, 128>(L, X, tab, n_mtiles, partials, zt, zt_stride, di, st);
    return launch_prefix_variant<T, 4, 64>(L, X, tab, n_mtiles, partials, zt, zt_stride, di, st);
}

// ---- scores from the tile sums, and which of them lie in the guard band -----------------------

constexpr int kFinThreads = 256;
struct GuardMults {
    int n;  // 0: no guard band
    float m[8];
    float rel_band;
};
// The guard band's part of the workspace.  Every CTA of the kernel below owns a run of 256 neurons of a sequence and
// leaves that run's candidates, compacted, at cand[b * d_ff + 256 run ..] and their number in count[b * runs + run]:
// no counter has to be cleared before, and the candidates come in one order whatever the timing.
struct GuardBuf {
    int *cand, *count;
    double2 *part;  // [n_slots] shares of the sums over tokens (guard_refine_kernel)
    int n_slots;
    int *done;      // CTAs of guard_refine_kernel that have finished; cleared here
};

// partials == nullptr: the scores are there already, only the candidates are wanted.
__global__ void __launch_bounds__(kFinThreads)
prefix_finalize_kernel(const float *__restrict__ partials, const SeqTable tab, int tile, int d_ff,
                       const float *__restrict__ w_down_norm, float *__restrict__ scores,
                       const float *__restrict__ tau_base, const GuardMults gm, const GuardBuf gb) {
    const int j = blockIdx.x * kFinThreads + threadIdx.x;
    const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_launch_dependents();
    int first = 0, n = 0;  // this prompt's tiles; at most 65535 tiles of tokens, so 32 bits do
    if (partials) {
        auto tiles = [&](int q) { return ((int)(tab.off[q + 1] - tab.off[q]) + tile - 1) / tile; };
        for (int q = lane; q < b; q += kWarp) first += tiles(q);
        first = __reduce_add_sync(0xffffffffu, first);
        n = tiles(b);
    }
    pdl_wait();
    float a = 0.f;
    if (j < d_ff) {
        if (partials) {
            const float *src = partials + (size_t)first * d_ff + j;
            float s = 0.f;
            for (int t0 = 0; t0 < n; t0 += 8) {  // eight loads in flight, added in tile order
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = t0 + u < n ? src[(size_t)(t0 + u) * d_ff] : 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (t0 + u < n) s += v[u];
            }
            a = __fmul_rn(sqrtf(s), w_down_norm[j]);
            scores[(size_t)b * d_ff + j] = a;
        } else {
            a = scores[(size_t)b * d_ff + j];
        }
    }
    if (gm.n == 0) return;
    __shared__ int s_n[kFinThreads / kWarp];
    bool near = false;
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        if (g < gm.n) {
            const float thr = tau_base[b] * gm.m[g];
            near |= fabsf(a - thr) <= gm.rel_band * fabsf(thr);
        }
    }
    near = near && j < d_ff;
    const unsigned bal = __ballot_sync(0xffffffffu, near);
    if (lane == 0) s_n[warp] = __popc(bal);
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kFinThreads / kWarp; ++w) {
        base += w < warp ? s_n[w] : 0;
        total += s_n[w];
    }
    if (near) gb.cand[(size_t)b * d_ff + blockIdx.x * kFinThreads + base + __popc(bal & ((1u << lane) - 1u))] = j;
    if (threadIdx.x == 0) gb.count[b * gridDim.x + blockIdx.x] = total;
    if (threadIdx.x == 0 && blockIdx.x == 0 && b == 0) *gb.done = 0;
}

// Chunked prefill: the same tile sums added into a running sum of squares per (prompt, neuron) ...
// Latency-bound: with one load after the other 7.1 us for the 16 tiles of 2000 tokens (14336 neurons); its launch, the
// finishing one and the down projection's are chained to what runs before them.  A chunk of 256 tokens (4096 x 11008), three
// calls, 109 us before and 102.6 now; of 2000 tokens (4096 x 14336) 627 and 624, which is within what runs differ by.
__global__ void prefix_accumulate_kernel(const float *__restrict__ partials, const SeqTable tab, int tile, int d_ff,
                                         float *__restrict__ sumsq) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = blockIdx.y;
    int first = 0;
    for (int q = 0; q < b; ++q) first += tiles_of(tab.off[q + 1] - tab.off[q], tile);
    const int n = tiles_of(tab.off[b + 1] - tab.off[b], tile);
    pdl_launch_dependents();
    pdl_wait();
    if (j >= d_ff) return;
    float s = sumsq[(size_t)b * d_ff + j];
    for (int t0 = 0; t0 < n; t0 += 16) {  // sixteen loads in flight, added in tile order
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = t0 + u < n ? partials[(size_t)(first + t0 + u) * d_ff + j] : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u)
            if (t0 + u < n) s += v[u];
    }
    sumsq[(size_t)b * d_ff + j] = s;
}

// ... and, after the last chunk, the scores from it.
__global__ void prefix_finish_kernel(const float *__restrict__ sumsq, int B, int d_ff,
                                     const float *__restrict__ w_down_norm, float *__restrict__ scores) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    if (i >= (size_t)B * d_ff) return;
    scores[i] = __fmul_rn(sqrtf(sumsq[i]), w_down_norm[i % d_ff]);
}

// ---- guard band -----------------------------------------------------------------------------

// A 16-byte vector widened to fp64 (exact).  For bf16 the double is assembled from the bit fields with
// integer operations: converting through the float-to-double instruction runs at a sixteenth of the ALU
// rate and was the guard band's bottleneck.  Zeros, denormals, inf and NaN take the conversion.
template <typename T> struct Widen;
template <> struct Widen<float> {
    __device__ static __forceinline__ void run(const uint4 &v, double (&o)[4]) {
        o[0] = (double)__uint_as_float(v.x); o[1] = (double)__uint_as_float(v.y);
        o[2] = (double)__uint_as_float(v.z); o[3] = (double)__uint_as_float(v.w);
    }
};
__device__ __forceinline__ double bf16_bits_to_double(uint32_t b) {  // b: 16 significant bits
    const uint32_t ex = (b >> 7) & 0xffu;
    if (ex == 0u || ex == 255u) return (double)__uint_as_float(b << 16);
    const uint32_t hi = ((b & 0x8000u) << 16) | ((ex + 896u) << 20) | ((b & 0x7fu) << 13);
    return __hiloint2double((int)hi, 0);
}
// IEEE half: 1 sign, 5 exponent (bias 15), 10 fraction bits -> double (bias 1023, fraction at bit 42 of 52).
__device__ __forceinline__ double f16_bits_to_double(uint32_t b) {  // b: 16 significant bits
    const uint32_t ex = (b >> 10) & 0x1fu;
    if (ex == 0u || ex == 31u) return (double)__half2float(__ushort_as_half((unsigned short)b));
    const uint32_t hi = ((b & 0x8000u) << 16) | ((ex + 1008u) << 20) | ((b & 0x3ffu) << 10);
    return __hiloint2double((int)hi, 0);
}
template <> struct Widen<__half> {
    __device__ static __forceinline__ void run(const uint4 &v, double (&o)[8]) {
        o[0] = f16_bits_to_double(v.x & 0xffffu); o[1] = f16_bits_to_double(v.x >> 16);
        o[2] = f16_bits_to_double(v.y & 0xffffu); o[3] = f16_bits_to_double(v.y >> 16);
        o[4] = f16_bits_to_double(v.z & 0xffffu); o[5] = f16_bits_to_double(v.z >> 16);
        o[6] = f16_bits_to_double(v.w & 0xffffu); o[7] = f16_bits_to_double(v.w >> 16);
    }
};
template <> struct Widen<__nv_bfloat16> {
    __device__ static __forceinline__ void run(const uint4 &v, double (&o)[8]) {
        o[0] = bf16_bits_to_double(v.x & 0xffffu); o[1] = bf16_bits_to_double(v.x >> 16);
        o[2] = bf16_bits_to_double(v.y & 0xffffu); o[3] = bf16_bits_to_double(v.y >> 16);
        o[4] = bf16_bits_to_double(v.z & 0xffffu); o[5] = bf16_bits_to_double(v.z >> 16);
        o[6] = bf16_bits_to_double(v.w & 0xffffu); o[7] = bf16_bits_to_double(v.w >> 16);
    }
};

// The same widening in three integer operations per element, off by a power of two: the exponent field of the 16-bit
// value is taken over as it is, so the double is x * 2^-896 (bf16) or 2^-1008 (fp16), exactly, zeros and denormals
// included (they become the double's zeros and denormals).  Weights are multiplied by kUp, which leaves room below
// their products with x; a finished sum times kBack is in true scale.  Infinities and NaN become numbers: the caller
// looks for them (nonfinite()).
template <typename T> struct Scaled;
template <> struct Scaled<float> {
    static constexpr double kUp = 1.0, kBack = 1.0;
    struct Peak {};
    __device__ static __forceinline__ void peak(Peak &, const uint4 &) {}
    __device__ static __forceinline__ bool nonfinite(const Peak &) { return false; }
    __device__ static __forceinline__ double get(const uint4 &v, int e) {
        return (double)__uint_as_float(e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w);
    }
};
__device__ __forceinline__ uint32_t word_of(const uint4 &v, int w) { return w == 0 ? v.x : w == 1 ? v.y : w == 2 ? v.z : v.w; }
template <> struct Scaled<__nv_bfloat16> {
    static constexpr double kUp = 0x1p1023, kBack = 0x1p769;  // scale 2^-896: x w 2^(1023 - 2 * 896)
    struct Peak { __nv_bfloat162 m = __nv_bfloat162(__ushort_as_bfloat16(0), __ushort_as_bfloat16(0)); };
    __device__ static __forceinline__ void peak(Peak &p, const uint4 &v) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t u = word_of(v, w);
            p.m = __hmax2_nan(p.m, __habs2(*reinterpret_cast<const __nv_bfloat162 *>(&u)));
        }
    }
    __device__ static __forceinline__ bool nonfinite(const Peak &p) {
        const uint32_t u = *reinterpret_cast<const uint32_t *>(&p.m) & 0x7fff7fffu;
        return (u & 0xffffu) >= 0x7f80u || (u >> 16) >= 0x7f80u;
    }
    __device__ static __forceinline__ double get(const uint4 &v, int e) {
        const uint32_t u = word_of(v, e >> 1);
        return __hiloint2double(((int)(e & 1 ? u : u << 16) >> 3) & (int)0x8fffe000u, 0);
    }
};
template <> struct Scaled<__half> {
    static constexpr double kUp = 0x1p1023, kBack = 0x1p993;  // scale 2^-1008
    struct Peak { __half2 m = __half2(__ushort_as_half(0), __ushort_as_half(0)); };
    __device__ static __forceinline__ void peak(Peak &p, const uint4 &v) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t u = word_of(v, w);
            p.m = __hmax2_nan(p.m, __habs2(*reinterpret_cast<const __half2 *>(&u)));
        }
    }
    __device__ static __forceinline__ bool nonfinite(const Peak &p) {
        const uint32_t u = *reinterpret_cast<const uint32_t *>(&p.m) & 0x7fff7fffu;
        return (u & 0xffffu) >= 0x7c00u || (u >> 16) >= 0x7c00u;
    }
    __device__ static __forceinline__ double get(const uint4 &v, int e) {
        const uint32_t u = word_of(v, e >> 1);
        return __hiloint2double(((int)(e & 1 ? u : u << 16) >> 6) & (int)0x81fffc00u, 0);
    }
};

constexpr int kRefThreads = 256;
constexpr int kRefTok = 8;        // tokens of a warp's pass
constexpr int kRefCand = 2;       // candidates of a unit
static_assert(kRefTok * kRefCand * 2 == kWarp, "one value per lane after the butterfly");

// g or u of one (token, neuron) row pair by one warp with the general widening: rows that hold infinities or NaN.
template <typename T>
__device__ __noinline__ double guard_dot_general(const uint4 *x, const uint4 *w, int vpr) {
    constexpr int E = Elem<T>::kPerVec;
    double s = 0.0;
    for (int v = threadIdx.x & 31; v < vpr; v += kWarp) {
        double fx[E], fw[E];
        Widen<T>::run(x[v], fx);
        Widen<T>::run(w[v], fw);
#pragma unroll
        for (int e = 0; e < E; ++e) s = fma(fw[e], fx[e], s);
    }
    return warp_sum(s);
}

// The candidates' scores again with fp64 products and sums.  A unit is two candidates of one prompt and a run of its
// tokens; SPLIT warps share a pass over eight tokens, each with its part of the row's 16-byte vectors, and every widened
// element of x meets four widened weights (gate and up of two candidates), every weight eight tokens.  So the double-precision FMA
// pipe sets the pace (it was the shared-memory path before: one 8-byte weight per FMA) and x is read once per two
// candidates.  Runs are cut so that every CTA gets about four units; a candidate's shares of the sum over tokens meet
// in the last CTA to finish, in one order.  With many short prompts the plan, the search for a unit's prompt and the last
// sums are what takes time: a warp each, binary search, eight lanes a candidate.
// Measured (bf16, refinement with its search for candidates, first version with a CTA per candidate / now): 8 prompts of
// 256-4096 tokens of a 5120 x 13824 layer 2650 / 880 us, one of 512 (4096 x 11008) 43 / 29, 30 of 100 (256 x 1000) 14.2 /
// 15.4, 64 of 16 (1024 x 4096) 15.0 / 14.8 (37 and 50 with one thread for the plan and the last sums prompt by prompt); the
// whole call for the prompt of 512 tokens 126-135 / 112-127.
template <typename T, int SPLIT>
__global__ void __launch_bounds__(kRefThreads, 1)
guard_refine_kernel(const T *__restrict__ X, const T *__restrict__ Wg, const T *__restrict__ Wu,
                    const T *__restrict__ Wd_t, int d_model, int d_ff, const SeqTable tab, const GuardBuf gb, int runs,
                    float *__restrict__ scores, int act) {
    constexpr int E = Elem<T>::kPerVec;
    constexpr int kWarps = kRefThreads / kWarp;
    using S = Scaled<T>;
    __shared__ int s_n[kMaxSeqs];             // candidates per prompt
    __shared__ int s_slot[kMaxSeqs + 1];      // their first slots
    __shared__ int s_unit[kMaxSeqs + 1];      // their first units
    __shared__ int s_cut[kMaxSeqs + 1];       // candidates of the prompts before that are cut into runs
    __shared__ int s_run_tokens, s_last;
    __shared__ int s_j[kRefCand];
    __shared__ double s_val[2][kWarps][kWarp];  // a pass's values per warp; the next pass may start while they are read
    __shared__ double s_zz[kWarps][kRefCand], s_nn[kWarps][kRefCand];
    __shared__ int s_odd[kWarps / SPLIT];
    constexpr int kPass = kWarps / SPLIT * kRefTok;  // tokens of a CTA's pass
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int vpr = d_model / E;
    pdl_launch_dependents();
    pdl_wait();
    for (int b0 = warp; b0 < tab.B; b0 += 4 * kWarps) {  // four prompts at a time, their loads in flight together
        int n[4] = {0, 0, 0, 0};
        for (int r = lane; r < runs; r += kWarp) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (b0 + i * kWarps < tab.B) n[i] += gb.count[(b0 + i * kWarps) * runs + r];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            n[i] = __reduce_add_sync(0xffffffffu, n[i]);
            if (lane == 0 && b0 + i * kWarps < tab.B) s_n[b0 + i * kWarps] = n[i];
        }
    }
    __syncthreads();
    if (warp == 0) {  // four prompts a lane (with one thread for all of them, 64 prompts cost 11 us)
        static_assert(kMaxSeqs <= 4 * kWarp, "four prompts a lane");
        int t[4], groups[4];  // at most 65535 tiles of tokens: 32 bits do
        float work = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int b = 4 * lane + i;
            t[i] = b < tab.B ? (int)(tab.off[b + 1] - tab.off[b]) : 0;
            groups[i] = b < tab.B ? (s_n[b] + kRefCand - 1) / kRefCand : 0;
            work += (float)groups[i] * (float)t[i];
        }
        work = warp_sum(work);
        int tokens = ((int)(work / (float)(4 * gridDim.x) / (float)kPass) + 1) * kPass;
        for (;; tokens *= 2) {  // until the shares have room (a prompt that is one run needs none)
            constexpr float kMany = 1 << 25;  // more shares than there ever is room for: the sums stay within 32 bits
            int slots[4], units[4], cuts[4], slot_sum = 0, unit_sum = 0, cut_sum = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = t[i] > tokens ? (t[i] + tokens - 1) / tokens : 1;
                slots[i] = slot_sum;
                units[i] = unit_sum;
                cuts[i] = cut_sum;
                if (r > 1) {
                    slot_sum = (int)fminf((float)slot_sum + (float)s_n[4 * lane + i] * (float)r, kMany);
                    cut_sum += s_n[4 * lane + i];
                }
                unit_sum += groups[i] * r;
            }
            int slot_end = slot_sum, unit_end = unit_sum, cut_end = cut_sum;
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, slot_end, o), c = __shfl_up_sync(0xffffffffu, unit_end, o),
                          e = __shfl_up_sync(0xffffffffu, cut_end, o);
                if (lane >= o) {
                    slot_end += a;
                    unit_end += c;
                    cut_end += e;
                }
            }
            if (__shfl_sync(0xffffffffu, slot_end, kWarp - 1) <= gb.n_slots) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int b = 4 * lane + i;
                    if (b < tab.B) {
                        s_slot[b] = slot_end - slot_sum + slots[i];
                        s_unit[b] = unit_end - unit_sum + units[i];
                        s_cut[b] = cut_end - cut_sum + cuts[i];
                    }
                }
                if (lane == kWarp - 1) {
                    s_unit[tab.B] = unit_end;
                    s_cut[tab.B] = cut_end;
                }
                break;
            }
        }
        if (lane == 0) s_run_tokens = tokens;
    }
    __syncthreads();
    const int run_tokens = s_run_tokens, n_units = s_unit[tab.B];
    if (n_units == 0) return;
    // The prompt that number i falls into: the last one whose first number is not beyond it (the one before it is empty).
    auto prompt_of = [&](const int *first, int i) {
        int lo = 0, hi = tab.B;  // first[lo] <= i < first[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (first[mid] <= i) lo = mid; else hi = mid;
        }
        return lo;
    };
    int buf = 0;
    for (int unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
        const int b = prompt_of(s_unit, unit);
        const int groups = (s_n[b] + kRefCand - 1) / kRefCand;
        const int group = (unit - s_unit[b]) % groups, run = (unit - s_unit[b]) / groups;
        const long long T_b = tab.off[b + 1] - tab.off[b];
        const int n_runs = (int)(T_b > run_tokens ? (T_b + run_tokens - 1) / run_tokens : 1);
        const int n_cand = min(kRefCand, s_n[b] - group * kRefCand);
        if (warp < kRefCand) {  // the group's neurons: the warp-th one is candidate group * 2 + warp of its prompt
            int left = group * kRefCand + min(warp, n_cand - 1);
            for (int r0 = 0; r0 < runs; r0 += kWarp) {
                const int c = r0 + lane < runs ? gb.count[b * runs + r0 + lane] : 0;
                int incl = c;
#pragma unroll
                for (int o = 1; o < kWarp; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const int all = __shfl_sync(0xffffffffu, incl, kWarp - 1);
                if (left < all) {
                    if (left >= incl - c && left < incl)
                        s_j[warp] = gb.cand[(size_t)b * d_ff + (size_t)(r0 + lane) * kFinThreads + left - (incl - c)];
                    break;
                }
                left -= all;
            }
        }
        __syncthreads();
        const uint4 *rows[2 * kRefCand];  // gate, up of the first candidate, then of the second
#pragma unroll
        for (int c = 0; c < kRefCand; ++c) {
            rows[2 * c] = reinterpret_cast<const uint4 *>(Wg + (size_t)s_j[c] * d_model);
            rows[2 * c + 1] = reinterpret_cast<const uint4 *>((Wu ? Wu : Wg) + (size_t)s_j[c] * d_model);  // null: not used
        }
        const long long t_end = min(tab.off[b + 1], tab.off[b] + (long long)(run + 1) * run_tokens);
        const int part = warp % SPLIT, team = warp / SPLIT;
        double zz = 0.0;  // lane: of one token and candidate per pass (even lanes of the team's first warp)
        for (long long t0 = tab.off[b] + (long long)run * run_tokens; t0 < t_end; t0 += kPass) {
            const long long tw = t0 + team * kRefTok;
            const uint4 *x = reinterpret_cast<const uint4 *>(X + (size_t)tw * d_model);
            const int n_tok = (int)max(0LL, min((long long)kRefTok, t_end - tw));
            double acc[kWarp];  // value 4 token + 2 candidate + (1: up)
#pragma unroll
            for (int i = 0; i < kWarp; ++i) acc[i] = 0.0;
            typename S::Peak peak;
            uint4 xv[kRefTok], wv[2 * kRefCand];
            auto fetch = [&](int v) {
#pragma unroll
                for (int t = 0; t < kRefTok; ++t) {
                    xv[t] = make_uint4(0, 0, 0, 0);
                    if (t < n_tok && v < vpr) xv[t] = ldg_stream(x + (size_t)t * vpr + v);
                }
#pragma unroll
                for (int r = 0; r < 2 * kRefCand; ++r) {
                    wv[r] = make_uint4(0, 0, 0, 0);
                    if (v < vpr) wv[r] = __ldg(rows[r] + v);
                }
            };
            fetch(part * kWarp + lane);
            for (int v = part * kWarp + lane; v - lane < vpr; v += SPLIT * kWarp) {
                uint4 xc[kRefTok], wc[2 * kRefCand];
#pragma unroll
                for (int t = 0; t < kRefTok; ++t) xc[t] = xv[t];
#pragma unroll
                for (int r = 0; r < 2 * kRefCand; ++r) wc[r] = wv[r];
                fetch(v + SPLIT * kWarp);
#pragma unroll
                for (int t = 0; t < kRefTok; ++t) S::peak(peak, xc[t]);
#pragma unroll
                for (int r = 0; r < 2 * kRefCand; ++r) S::peak(peak, wc[r]);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    double w[2 * kRefCand];
#pragma unroll
                    for (int r = 0; r < 2 * kRefCand; ++r) w[r] = S::get(wc[r], e) * S::kUp;
#pragma unroll
                    for (int t = 0; t < kRefTok; ++t) {
                        const double xe = S::get(xc[t], e);
#pragma unroll
                        for (int r = 0; r < 2 * kRefCand; ++r) acc[4 * t + r] = fma(w[r], xe, acc[4 * t + r]);
                    }
                }
            }
            // warp sums by a halving butterfly: lane i ends up with value i
#pragma unroll
            for (int o = kWarp / 2; o > 0; o >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int i = 0; i < o; ++i) {
                    const double send = up ? acc[i] : acc[i + o];
                    acc[i] = (up ? acc[i + o] : acc[i]) + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            const bool odd = __any_sync(0xffffffffu, S::nonfinite(peak));
            s_val[buf][warp][lane] = acc[0];
            if (part == 0 && lane == 0) s_odd[team] = 0;
            __syncthreads();
            if (odd && lane == 0) s_odd[team] = 1;
            __syncthreads();
            if (part == 0) {  // the team's first warp adds the parts in order and forms the neuron values
                double val = 0.0;
#pragma unroll
                for (int q = 0; q < SPLIT; ++q) val += s_val[buf][warp + q][lane];
                val *= S::kBack;
                if (s_odd[team]) {
                    for (int i = 0; i < 4 * n_tok; ++i) {
                        const double dot = guard_dot_general<T>(x + (size_t)(i >> 2) * vpr, rows[i & 3], vpr);
                        if (lane == i) val = dot;
                    }
                }
                const double other = __shfl_xor_sync(0xffffffffu, val, 1);
                if (!(lane & 1) && (lane >> 2) < n_tok) {
                    const double z = neuron_value_d(act, val, other);
                    zz += z * z;
                }
            }
            buf ^= 1;
        }
        // ||w_down||^2 of both candidates, and the sums over the CTA
        double nn[kRefCand];
#pragma unroll
        for (int c = 0; c < kRefCand; ++c) {
            nn[c] = 0.0;
            if (run == 0) {
                const uint4 *wd = reinterpret_cast<const uint4 *>(Wd_t + (size_t)s_j[c] * d_model);
                for (int v = tid; v < vpr; v += kRefThreads) {
                    double fd[E];
                    Widen<T>::run(wd[v], fd);
#pragma unroll
                    for (int e = 0; e < E; ++e) nn[c] = fma(fd[e], fd[e], nn[c]);
                }
                nn[c] = warp_sum(nn[c]);
            }
            const double zc = warp_sum((lane >> 1 & 1) == c ? zz : 0.0);  // odd lanes hold zero
            if (lane == 0) {
                s_zz[warp][c] = zc;
                s_nn[warp][c] = nn[c];
            }
        }
        __syncthreads();
        if (tid < n_cand) {
            double a = 0.0, n2 = 0.0;
            for (int w = 0; w < kWarps; ++w) {
                a += s_zz[w][tid];
                n2 += s_nn[w][tid];
            }
            const int j = s_j[tid];
            if (n_runs == 1)
                scores[(size_t)b * d_ff + j] = (float)(sqrt(a) * sqrt(n2));
            else  // this run's share; the first run's slot carries the norm, the second's the neuron
                gb.part[s_slot[b] + (size_t)(group * kRefCand + tid) * n_runs + run] =
                    make_double2(a, run == 0 ? n2 : (double)j);
        }
        __syncthreads();
    }
    // the last CTA adds the shares of every candidate that was cut into runs, eight lanes each (with a warp each and prompt
    // after prompt, 30 prompts cost 12 us)
    const int n_cut = s_cut[tab.B];
    if (n_cut == 0) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(gb.done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int sub = lane & 7;
    for (int p0 = warp * 4; p0 < n_cut; p0 += 4 * kWarps) {
        const int p = p0 + (lane >> 3), b = prompt_of(s_cut, min(p, n_cut - 1));
        double a = 0.0, y = 0.0;
        if (p < n_cut) {
            const int n_runs = (int)((tab.off[b + 1] - tab.off[b] + run_tokens - 1) / run_tokens);
            const double2 *share = gb.part + s_slot[b] + (size_t)(p - s_cut[b]) * n_runs;
            for (int r0 = sub; r0 < n_runs; r0 += 64) {  // eight loads in flight
                double2 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = r0 + 8 * i < n_runs ? __ldcg(share + r0 + 8 * i) : make_double2(0.0, 0.0);
                if (r0 < 2) y = v[0].y;
#pragma unroll
                for (int i = 0; i < 8; ++i) a += v[i].x;
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        const double n2 = __shfl_sync(0xffffffffu, y, lane & ~7), j = __shfl_sync(0xffffffffu, y, (lane & ~7) + 1);
        if (sub == 0 && p < n_cut) scores[(size_t)b * d_ff + (int)j] = (float)(sqrt(a) * sqrt(n2));
    }
}

// ---- host side ------------------------------------------------------------------------------

static int build_table(const int64_t *seq_offsets, int32_t B, SeqTable *tab, int *n_mtiles) {
    if (!seq_offsets) return CLADA_ERR_NULL;
    if (B <= 0) return CLADA_ERR_SHAPE;
    if (B > kMaxSeqs) return CLADA_ERR_UNSUPPORTED;
    tab->B = B;
    long long tiles = 0;
    for (int b = 0; b <= B; ++b) {
        tab->off[b] = seq_offsets[b];
        if (seq_offsets[b] < 0 || (b > 0 && seq_offsets[b] < seq_offsets[b - 1])) return CLADA_ERR_SHAPE;
        if (b > 0) tiles += tiles_of(seq_offsets[b] - seq_offsets[b - 1], BM);
    }
    if (tiles > 65535) return CLADA_ERR_UNSUPPORTED;
    *n_mtiles = (int)tiles;
    return CLADA_OK;
}

static size_t partials_bytes(int n_mtiles, int d_ff) {
    return (((size_t)n_mtiles * d_ff * sizeof(float)) + 255) & ~(size_t)255;
}

template <typename T>
static int run_scores(const clada_layer *L, const void *X, const SeqTable &tab, int n_mtiles, float *scores,
                      float *partials, cudaStream_t st, float *zt = nullptr, long long zt_stride = 0) {
    if (n_mtiles > 0) {
        const int rc = launch_prefix_partials<T>(L, X, tab, n_mtiles, partials, zt, zt_stride, st);
        if (rc != CLADA_OK) return rc;
    }
    return launch_prefix_finalize(partials, tab, BM, L->d_ff, L->w_down_norm, scores, st);
}

int run_prefix_scores_with_z(const clada_layer *layer, const void *X, const int64_t *seq_offsets, int32_t B,
                             float *scores, float *partials, float *zt, cudaStream_t st) {
    SeqTable tab;
    int n_mtiles = 0;
    int rc = build_table(seq_offsets, B, &tab, &n_mtiles);
    if (rc != CLADA_OK) return rc;
    if (layer->dtype == CLADA_F32)
        return run_scores<float>(layer, X, tab, n_mtiles, scores, partials, st, zt, seq_offsets[B]);
    if (layer->dtype == CLADA_BF16)
        return run_scores<__nv_bfloat16>(layer, X, tab, n_mtiles, scores, partials, st, zt, seq_offsets[B]);
    return run_scores<__half>(layer, X, tab, n_mtiles, scores, partials, st, zt, seq_offsets[B]);
}

size_t prefix_partials_bytes_cuda_core(const int64_t *seq_offsets, int32_t B, int d_ff) {
    long long tiles = 0;
    for (int b = 0; b < B; ++b) tiles += tiles_of(seq_offsets[b + 1] - seq_offsets[b], BM);
    return partials_bytes((int)tiles, d_ff);
}

// One launch of the chain statistics -> scores and candidates -> refinement -> selection: its latency hides under the
// launch before it.
template <typename... P, typename... A>
static int launch_chained(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CLADA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    return CLADA_OK;
}

// Scores from tile sums (partials), or the scores as they are (null), and with gm.n > 0 their candidates.
static int launch_finalize(const float *partials, const SeqTable &tab, int tile, int d_ff, const float *w_down_norm,
                           float *scores, const float *tau_base, const GuardMults &gm, const GuardBuf &gb,
                           cudaStream_t st) {
    return launch_chained(prefix_finalize_kernel, dim3((d_ff + kFinThreads - 1) / kFinThreads, tab.B), kFinThreads, st,
                          partials, tab, tile, d_ff, w_down_norm, scores, tau_base, gm, gb);
}

int launch_prefix_finalize(const float *partials, const SeqTable &tab, int tile, int d_ff,
                           const float *w_down_norm, float *scores, cudaStream_t st) {
    return launch_finalize(partials, tab, tile, d_ff, w_down_norm, scores, nullptr, GuardMults{}, GuardBuf{}, st);
}

// The guard band's buffers behind the tile sums of clada_prefix_scores, in the bytes that clada_workspace_bytes holds
// for them.
static int guard_buffers(const clada_layer *layer, int32_t B, int n_mtiles, void *ws, size_t ws_bytes, GuardBuf *gb) {
    const size_t off = kWsCtrlBytes + partials_bytes(n_mtiles, layer->d_ff);
    const size_t all = (size_t)B * layer->d_ff, runs = (size_t)B * ((layer->d_ff + kFinThreads - 1) / kFinThreads);
    const size_t need = off + 256 + 512 * sizeof(double2) + all * 2 * sizeof(int);
    if (ws_bytes < need) return CLADA_ERR_WORKSPACE;
    char *base = static_cast<char *>(ws);
    gb->done = reinterpret_cast<int *>(base + off);
    gb->cand = reinterpret_cast<int *>(base + off + 256);
    gb->count = gb->cand + all;
    const size_t part = (off + 256 + (all + runs) * sizeof(int) + 15) & ~(size_t)15;
    gb->part = reinterpret_cast<double2 *>(base + part);
    gb->n_slots = (int)std::min<size_t>((need - part) / sizeof(double2), 1u << 30);
    return CLADA_OK;
}

static int guard_mults_of(const float *guard_mults, int32_t n_guard, float rel_band, GuardMults *gm) {
    if (n_guard <= 0 || n_guard > 8 || !(rel_band >= 0.f)) return CLADA_ERR_SHAPE;
    gm->n = n_guard;
    gm->rel_band = rel_band;
    for (int g = 0; g < 8; ++g) gm->m[g] = g < n_guard ? guard_mults[g] : 0.f;
    return CLADA_OK;
}

// Four warps share a row when each of them then has 32 vectors of it; of a narrower row two or one, whose passes take more
// tokens (16, 32 or 64 a CTA).
template <typename T>
static int launch_refine(const clada_layer *L, const void *X, const SeqTable &tab, const GuardBuf &gb, float *scores,
                         int n_ctas, cudaStream_t st) {
    const int vpr = L->d_model / Elem<T>::kPerVec;
    auto kernel = vpr >= 4 * kWarp ? guard_refine_kernel<T, 4> : (vpr >= 2 * kWarp ? guard_refine_kernel<T, 2> : guard_refine_kernel<T, 1>);
    return launch_chained(kernel, dim3(n_ctas), kRefThreads, st, static_cast<const T *>(X),
                          static_cast<const T *>(L->w_gate), static_cast<const T *>(L->w_up),
                          static_cast<const T *>(L->w_down_t), L->d_model, L->d_ff, tab, gb,
                          (L->d_ff + kFinThreads - 1) / kFinThreads, scores, L->activation);
}
static int run_refine(const clada_layer *L, const void *X, const SeqTable &tab, const GuardBuf &gb, float *scores,
                      cudaStream_t st) {
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != CLADA_OK) return rc;
    if (L->dtype == CLADA_F32) return launch_refine<float>(L, X, tab, gb, scores, di.num_sms, st);
    if (L->dtype == CLADA_BF16) return launch_refine<__nv_bfloat16>(L, X, tab, gb, scores, di.num_sms, st);
    return launch_refine<__half>(L, X, tab, gb, scores, di.num_sms, st);
}

}  // namespace clada

using namespace clada;

// Statistics and scores of the prompts; with gm.n > 0 also the candidates of the guard band around tau_base (their
// buffers in *gb, the prompt table in *tab), for run_refine.
static int prefix_scores_guarded(const clada_layer *layer, const void *X, const int64_t *seq_offsets, int32_t B,
                                 float *scores, void *ws, size_t ws_bytes, int32_t *status, const float *tau_base,
                                 const GuardMults &gm, SeqTable *tab, GuardBuf *gb, void *stream) {
    int rc = validate_layer(layer, true);
    if (rc != CLADA_OK) return rc;
    if (!X || !scores) return CLADA_ERR_NULL;
    if (!aligned16(X)) return CLADA_ERR_ALIGN;
    int n_mtiles = 0;
    rc = build_table(seq_offsets, B, tab, &n_mtiles);
    if (rc != CLADA_OK) return rc;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CLADA_ERR_WORKSPACE;
    if (ws_bytes < kWsCtrlBytes + partials_bytes(n_mtiles, layer->d_ff)) return CLADA_ERR_WORKSPACE;
    GuardBuf none = {};
    if (gm.n > 0 && (rc = guard_buffers(layer, B, n_mtiles, ws, ws_bytes, gb)) != CLADA_OK) return rc;
    float *partials = reinterpret_cast<float *>(static_cast<char *>(ws) + kWsCtrlBytes);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int tile = BM;
    if (layer->dtype == CLADA_F32) {
        if (n_mtiles > 0) rc = launch_prefix_partials<float>(layer, X, *tab, n_mtiles, partials, nullptr, 0, st);
    } else {  // bf16 / fp16: tensor cores (128-token tiles: never more partial rows than the 64-token tiling above)
        rc = run_prefix_partials_tc(layer, X, *tab, seq_offsets[B], partials, status, st);
        tile = kTcTokenTile;
    }
    if (rc != CLADA_OK) return rc;
    return launch_finalize(partials, *tab, tile, layer->d_ff, layer->w_down_norm, scores, tau_base, gm,
                           gm.n > 0 ? *gb : none, st);
}

extern "C" {

int clada_prefix_scores(const clada_layer *layer, const void *X, const int64_t *seq_offsets, int32_t B,
                        float *scores, void *ws, size_t ws_bytes, int32_t *status, void *stream) {
    CLADA_RANGE("clada_prefix_scores");
    SeqTable tab;
    return prefix_scores_guarded(layer, X, seq_offsets, B, scores, ws, ws_bytes, status, nullptr, GuardMults{}, &tab,
                                 nullptr, stream);
}

int clada_prefix_accumulate(const clada_layer *layer, const void *X, const int64_t *seq_offsets, int32_t B,
                            float *sumsq, void *Z, void *ws, size_t ws_bytes, int32_t *status, void *stream) {
    CLADA_RANGE("clada_prefix_accumulate");
    int rc = validate_layer(layer, false);
    if (rc != CLADA_OK) return rc;
    if (!X || !sumsq) return CLADA_ERR_NULL;
    if (!aligned16(X) || (Z && !aligned16(Z))) return CLADA_ERR_ALIGN;
    if (Z && layer->dtype == CLADA_F32) return CLADA_ERR_UNSUPPORTED;  // hidden activations: tensor-core route only
    if (Z && layer->d_ff % 8 != 0) return CLADA_ERR_SHAPE;  // rows of Z are written as 16-byte vectors
    SeqTable tab;
    int n_mtiles = 0;
    rc = build_table(seq_offsets, B, &tab, &n_mtiles);
    if (rc != CLADA_OK) return rc;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CLADA_ERR_WORKSPACE;
    if (ws_bytes < kWsCtrlBytes + partials_bytes(n_mtiles, layer->d_ff)) return CLADA_ERR_WORKSPACE;
    float *partials = reinterpret_cast<float *>(static_cast<char *>(ws) + kWsCtrlBytes);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int tile = BM;
    if (layer->dtype == CLADA_F32) {
        if (n_mtiles > 0) {
            rc = launch_prefix_partials<float>(layer, X, tab, n_mtiles, partials, nullptr, 0, st);
            if (rc != CLADA_OK) return rc;
        }
    } else {
        rc = run_prefix_partials_tc(layer, X, tab, seq_offsets[B], partials, status, st, Z);
        if (rc != CLADA_OK) return rc;
        tile = kTcTokenTile;
    }
    return launch_chained(prefix_accumulate_kernel, dim3((layer->d_ff + 127) / 128, tab.B), 128, st, partials, tab, tile, layer->d_ff,
                          sumsq);
}

int clada_prefix_finish(const clada_layer *layer, const float *sumsq, int32_t B, float *scores, void *stream) {
    CLADA_RANGE("clada_prefix_finish");
    int rc = validate_layer(layer, true);
    if (rc != CLADA_OK) return rc;
    if (!sumsq || !scores) return CLADA_ERR_NULL;
    if (B <= 0) return CLADA_ERR_SHAPE;
    const size_t n = (size_t)B * layer->d_ff;
    return launch_chained(prefix_finish_kernel, dim3((unsigned)((n + 255) / 256)), 256, static_cast<cudaStream_t>(stream), sumsq, B,
                          layer->d_ff, layer->w_down_norm, scores);
}

int clada_prefill_down(const clada_layer *layer, const void *w_down, const void *Z, int64_t T, void *Y,
                       int32_t y_dtype, void *ws, size_t ws_bytes, int32_t *status, void *stream) {
    CLADA_RANGE("clada_prefill_down");
    int rc = validate_layer(layer, false);
    if (rc != CLADA_OK) return rc;
    if (!w_down || !Z || !Y) return CLADA_ERR_NULL;
    if (T < 0) return CLADA_ERR_SHAPE;
    if (layer->dtype == CLADA_F32) return CLADA_ERR_UNSUPPORTED;  // tensor-core route: bf16 / fp16 layers
    if (!dtype_ok(y_dtype)) return CLADA_ERR_DTYPE;
    if (layer->d_ff % 8 != 0) return CLADA_ERR_SHAPE;  // rows of Z and of w_down must be 16-byte multiples
    if (!aligned16(w_down) || !aligned16(Z) || !aligned16(Y)) return CLADA_ERR_ALIGN;
    if (ws && ((reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < kWsCtrlBytes)) return CLADA_ERR_WORKSPACE;
    // the scratch behind the workspace's control block (which this call leaves alone) holds split partial outputs
    void *scratch = ws ? static_cast<char *>(ws) + kWsCtrlBytes : nullptr;
    return run_down_tc(layer, w_down, Z, T, Y, y_dtype, scratch, ws ? ws_bytes - kWsCtrlBytes : 0, status,
                       static_cast<cudaStream_t>(stream));
}

int clada_refine_scores(const clada_layer *layer, const void *X, const int64_t *seq_offsets, int32_t B,
                        const float *tau_base, const float *guard_mults, int32_t n_guard, float rel_band,
                        float *scores, void *ws, size_t ws_bytes, int32_t *status, void *stream) {
    CLADA_RANGE("clada_refine_scores");
    (void)status;
    int rc = validate_layer(layer, false);
    if (rc != CLADA_OK) return rc;
    if (!X || !scores || !tau_base || !guard_mults) return CLADA_ERR_NULL;
    GuardMults gm;
    if ((rc = guard_mults_of(guard_mults, n_guard, rel_band, &gm)) != CLADA_OK) return rc;
    if (!aligned16(X)) return CLADA_ERR_ALIGN;
    SeqTable tab;
    int n_mtiles = 0;
    rc = build_table(seq_offsets, B, &tab, &n_mtiles);
    if (rc != CLADA_OK) return rc;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CLADA_ERR_WORKSPACE;
    GuardBuf gb;
    if ((rc = guard_buffers(layer, B, n_mtiles, ws, ws_bytes, &gb)) != CLADA_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    rc = launch_finalize(nullptr, tab, 1, layer->d_ff, nullptr, scores, tau_base, gm, gb, st);
    return rc != CLADA_OK ? rc : run_refine(layer, X, tab, gb, scores, st);
}

int clada_prefix_select(const clada_layer *layer, const void *X, const int64_t *seq_offsets, int32_t B,
                        const float *tau_base, const float *guard_mults, int32_t n_guard, float *scores,
                        uint8_t *mask, int32_t *idx, int32_t *count, void *ws, size_t ws_bytes,
                        int32_t *status, void *stream) {
    CLADA_RANGE("clada_prefix_select");
    if (!tau_base || n_guard <= 0 || !guard_mults) {
        const int rc = clada_prefix_scores(layer, X, seq_offsets, B, scores, ws, ws_bytes, status, stream);
        if (rc != CLADA_OK || !tau_base) return rc;
        return clada_select(scores, B, layer->d_ff, tau_base, 1, mask, idx, count, stream);
    }
    GuardMults gm;
    SeqTable tab;
    GuardBuf gb;
    int rc = validate_layer(layer, true);
    if (rc != CLADA_OK) return rc;
    if ((rc = guard_mults_of(guard_mults, n_guard, 1e-4f, &gm)) != CLADA_OK) return rc;
    rc = prefix_scores_guarded(layer, X, seq_offsets, B, scores, ws, ws_bytes, status, tau_base, gm, &tab, &gb, stream);
    if (rc == CLADA_OK) rc = run_refine(layer, X, tab, gb, scores, static_cast<cudaStream_t>(stream));
    if (rc != CLADA_OK) return rc;
    return clada_select(scores, B, layer->d_ff, tau_base, 1, mask, idx, count, stream);
}

}  // extern "C"
