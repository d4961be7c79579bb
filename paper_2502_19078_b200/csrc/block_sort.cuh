// Sorting one sequence's neurons by score inside a CTA (nested lists, threshold search).
#pragma once

#include "common.cuh"

namespace clada {

constexpr int kSortThreads = 1024;
constexpr int kSortMaxN = 16384;                       // 8-byte keys of the next power of two in shared memory
constexpr int kSortPer = kSortMaxN / kSortThreads;     // elements per thread
constexpr int kSortBuckets = 8192;
constexpr int kSortMaxBucket = 256;                    // fuller buckets: bitonic network
constexpr size_t kSortSmem = (size_t)kSortMaxN * 8 + (size_t)(kSortBuckets + 1) * 4;

// Ranks n <= kSortMaxN elements by ascending (key, index), all kSortThreads threads of the CTA taking part.
//   load(i)              element i from memory
//   key_of(value)        its 32-bit key; called once per element
//   reg_lo, reg_hi       keys in between are regular; the few outside (zeros, infinities, NaNs) go before / after them
//   emit(rank, i, key)   called once per element whose rank is in [r0, r1)
//
// Scores of one sequence lie within a few octaves, so the regular keys' range cut into 8190 equal pieces leaves a few
// elements per piece: count, scan, scatter, and every element's rank is its piece's start plus the number of smaller
// (key, index) pairs in the piece.  Five passes over the elements instead of the 105 of the bitonic network, which
// remains for keys that crowd into a piece (many equal scores).  Only the pieces that hold ranks of [r0, r1) are
// scattered and ranked (a comparison of piece numbers in registers tells which), so CTAs that share a sequence repeat the
// counting alone.  Bound by latency, memory's first and shared memory's afterwards.  The order inside a piece's slots is
// arrival order; the ranks do not depend on it.  Measured: lists of 8 sequences of 14336 neurons take 194.5 us a call with
// the network, 12.5 with every element's piece looked up and the counters scanned one by one (a warp's in four banks), 11.5
// now; 32 of them 14.0 / 12.5, 16 of 16384 13.7 / 12.2 (back-to-back calls; on scores not seen before half of the gain).
template <typename Load, typename KeyOf, typename Emit>
__device__ void block_sort(int n, unsigned reg_lo, unsigned reg_hi, int r0, int r1, unsigned char *smem, Load load,
                           KeyOf key_of, Emit emit) {
    unsigned long long *s_key = reinterpret_cast<unsigned long long *>(smem);
    int *s_cnt = reinterpret_cast<int *>(smem + (size_t)kSortMaxN * 8);
    __shared__ unsigned s_min[kSortThreads / kWarp], s_max[kSortThreads / kWarp];
    __shared__ int s_wtot[kSortThreads / kWarp], s_wmax[kSortThreads / kWarp], s_edge[2], s_piece[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    unsigned key[kSortPer], slot[kSortPer];
    unsigned kmin = 0xffffffffu, kmax = 0u;
    {
        decltype(load(0)) value[kSortPer];  // all loads in flight together
#pragma unroll
        for (int e = 0; e < kSortPer; ++e) {
            value[e] = {};
            if (tid + e * kSortThreads < n) value[e] = load(tid + e * kSortThreads);
        }
#pragma unroll
        for (int e = 0; e < kSortPer; ++e) key[e] = tid + e * kSortThreads < n ? key_of(value[e]) : 0u;
    }
#pragma unroll
    for (int e = 0; e < kSortPer; ++e) {
        const int i = tid + e * kSortThreads;
        if (i < n && key[e] >= reg_lo && key[e] <= reg_hi) {
            kmin = min(kmin, key[e]);
            kmax = max(kmax, key[e]);
        }
    }
    for (int i = tid; i <= kSortBuckets; i += kSortThreads) s_cnt[i] = 0;
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
        s_min[warp] = kmin;
        s_max[warp] = kmax;
    }
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, s_min[lane]);
    kmax = __reduce_max_sync(0xffffffffu, s_max[lane]);
    const unsigned span = kmax >= kmin ? kmax - kmin : 0u;
    constexpr unsigned kPieces = kSortBuckets - 2;
    const unsigned scale = span < kPieces ? 0u : (unsigned)(((unsigned long long)kPieces << 32) / ((unsigned long long)span + 1ull));
    auto bucket_of = [&](unsigned k) -> int {
        if (k < kmin) return 0;
        if (k > kmax) return kSortBuckets - 1;
        return 1 + (int)(scale ? __umulhi(k - kmin, scale) : k - kmin);
    };
#pragma unroll
    for (int e = 0; e < kSortPer; ++e) {
        if (tid + e * kSortThreads < n) slot[e] = (unsigned)atomicAdd(&s_cnt[bucket_of(key[e])], 1);
    }
    __syncthreads();
    // exclusive scan of the counters (eight consecutive ones per thread) and the fullest piece
    constexpr int kPer = kSortBuckets / kSortThreads;
    static_assert(kPer % 4 == 0, "counters as 16-byte vectors (one by one a warp's would share four banks)");
    int4 *own = reinterpret_cast<int4 *>(s_cnt + tid * kPer);
    int c[kPer], sum = 0, fullest = 0;
#pragma unroll
    for (int q = 0; q < kPer; q += 4) {
        const int4 v = own[q / 4];
        c[q] = v.x; c[q + 1] = v.y; c[q + 2] = v.z; c[q + 3] = v.w;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        sum += c[q];
        fullest = max(fullest, c[q]);
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    fullest = __reduce_max_sync(0xffffffffu, fullest);
    if (lane == kWarp - 1) s_wtot[warp] = incl;
    if (lane == 0) s_wmax[warp] = fullest;
    __syncthreads();
    fullest = __reduce_max_sync(0xffffffffu, s_wmax[lane]);
    if (fullest <= kSortMaxBucket) {
        int base = __reduce_add_sync(0xffffffffu, lane < warp ? s_wtot[lane] : 0) + incl - sum;
        int start[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            start[q] = base;
            base += c[q];
            // the pieces that hold the first and the last rank asked for
            if (start[q] <= r0 && r0 < base) {
                s_piece[0] = tid * kPer + q;
                s_edge[0] = start[q];
            }
            if (start[q] < r1 && r1 <= base) {
                s_piece[1] = tid * kPer + q;
                s_edge[1] = base;
            }
        }
#pragma unroll
        for (int q = 0; q < kPer; q += 4) own[q / 4] = make_int4(start[q], start[q + 1], start[q + 2], start[q + 3]);
        if (tid == kSortThreads - 1) s_cnt[kSortBuckets] = n;
        __syncthreads();
        if (r0 >= r1) return;
        // scatter the elements of the pieces from one to the other
        const int piece0 = s_piece[0], piece1 = s_piece[1];
#pragma unroll
        for (int e = 0; e < kSortPer; ++e) {
            const int i = tid + e * kSortThreads;
            if (i < n) {
                const int b = bucket_of(key[e]);
                if (b >= piece0 && b <= piece1)
                    s_key[s_cnt[b] + (int)slot[e]] = ((unsigned long long)key[e] << 32) | (unsigned)i;
            }
        }
        __syncthreads();
        // by position: the lanes of a warp share their pieces, so their reads are broadcasts
        for (int p = s_edge[0] + tid; p < s_edge[1]; p += kSortThreads) {
            const unsigned long long mine = s_key[p];
            const int b = bucket_of((unsigned)(mine >> 32));
            const int first = s_cnt[b], last = s_cnt[b + 1];
            int rank = first;
            for (int q = first; q < last; ++q) rank += s_key[q] < mine ? 1 : 0;
            if (rank >= r0 && rank < r1) emit(rank, (int)(mine & 0xffffffffull), (unsigned)(mine >> 32));
        }
        return;
    }
    int n_pow2 = 2;
    while (n_pow2 < n) n_pow2 <<= 1;
#pragma unroll
    for (int e = 0; e < kSortPer; ++e) {
        const int i = tid + e * kSortThreads;
        if (i < n_pow2) s_key[i] = i < n ? ((unsigned long long)key[e] << 32) | (unsigned)i : ~0ull;  // padding sorts last
    }
    __syncthreads();
    for (int k = 2; k <= n_pow2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < n_pow2; i += kSortThreads) {
                const int l = i ^ j;
                if (l > i) {
                    const unsigned long long x = s_key[i], y = s_key[l];
                    const bool ascending = (i & k) == 0;
                    if ((x > y) == ascending) {
                        s_key[i] = y;
                        s_key[l] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int p = r0 + tid; p < r1; p += kSortThreads) emit(p, (int)(s_key[p] & 0xffffffffull), (unsigned)(s_key[p] >> 32));
}

}  // namespace clada
