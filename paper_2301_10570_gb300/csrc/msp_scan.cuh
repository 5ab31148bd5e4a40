// msp_scan.cuh -- single-pass device scan with a decoupled look-back, and the
// look-back itself for kernels that scan sizes they compute on the way
// (octree levels, traversal depths).
//
// Blocks take tiles in order from a counter, so every tile's predecessors have
// started; a tile publishes its sum (flag 1) before it looks back, then its
// inclusive prefix (flag 2), as one 64-bit word (flag in the top two bits).
// The look-back reads 32 predecessors per step with a warp, waiting on each
// for at most spin_limit polls; a wait that gives up sets timeout_bit in
// *overflow and counts the tile as 0 (the result is then wrong and the host
// reports it).
#pragma once

#include <algorithm>

#include "msp_internal.cuh"

namespace msp {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr unsigned long long kValMask = (1ull << 62) - 1;
constexpr int kSpinLimit = 1 << 22;
constexpr int kSelftestSpins = 1 << 12;      // of the waits that are made to run out

__device__ __forceinline__ long long warp_incl_scan(long long v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// exclusive scan over a block of kScanThreads of one value per thread; returns
// the block total
__device__ __forceinline__ long long block_excl_scan(long long v, long long* total) {
    __shared__ long long warp_sums[kScanThreads / 32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        long long s = lane < kScanThreads / 32 ? warp_sums[lane] : 0;
        long long si = warp_incl_scan(s);
        if (lane < kScanThreads / 32) warp_sums[lane] = si - s;
        if (lane == kScanThreads / 32 - 1) *total = si;
    }
    __syncthreads();
    long long r = inc - v + warp_sums[w];
    __syncthreads();
    return r;
}

// Publishes tile t's W values (each below 2^62) and returns, in every lane of
// the one warp that calls, the sums of the tiles before it.  st: W words per
// tile, each with a flag of its own.
template <int W>
__device__ __forceinline__ void look_back(volatile unsigned long long* st, int64_t t,
                                          const long long (&own)[W], long long (&excl)[W],
                                          int64_t* overflow, int64_t timeout_bit, int spin_limit) {
    const int lane = threadIdx.x & 31;
    bool done[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
        excl[k] = 0;
        done[k] = false;
        if (lane == 0)
            st[W * t + k] = (t == 0 ? 2ull : 1ull) << 62 | ((unsigned long long)own[k] & kValMask);
    }
    for (int64_t j = t - 1; j >= 0; j -= 32) {
        const int64_t jj = j - lane;
        unsigned long long w[W];
#pragma unroll
        for (int k = 0; k < W; ++k) w[k] = jj >= 0 ? st[W * jj + k] : 2ull << 62;
        bool all = true;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            // lanes past tile 0 count as a prefix of 0
            int spin = 0;
            while ((w[k] >> 62) == 0 && spin < spin_limit) {
                ++spin;
                w[k] = st[W * jj + k];
            }
            if ((w[k] >> 62) == 0) {
                atomicOr(reinterpret_cast<unsigned long long*>(overflow),
                         (unsigned long long)timeout_bit);
                w[k] = 2ull << 62;
            }
            const unsigned pmask = __ballot_sync(0xffffffffu, (w[k] >> 62) == 2);
            const int stop = pmask ? __ffs(pmask) - 1 : 31;   // first prefix, else all 32
            long long val = !done[k] && lane <= stop ? (long long)(w[k] & kValMask) : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
            excl[k] += val;
            done[k] = done[k] || pmask != 0;
            all = all && done[k];
        }
        if (all) break;
    }
#pragma unroll
    for (int k = 0; k < W; ++k)
        if (lane == 0 && t > 0)
            st[W * t + k] = 2ull << 62 | ((unsigned long long)(excl[k] + own[k]) & kValMask);
}

// Exclusive scan of in(i), i < *n_dev: out(i, sum before i, out.read(i)) for every
// i (nothing that read reads is written by the scan), then
// fin(total) once (also for no element).  status[0]: the tile counter,
// status[1 + tile]: the tiles' words, zero on entry.
template <class In, class Out, class Fin>
__global__ void __launch_bounds__(kScanThreads)
k_scan_1p(In in, Out out, Fin fin, const int64_t* __restrict__ n_dev, unsigned long long* status,
          int64_t* __restrict__ overflow, int64_t timeout_bit, int spin_limit) {
    __shared__ int32_t s_v[kScanTile + kScanTile / 32];
    __shared__ long long s_tot, s_excl;
    __shared__ int64_t s_tile;
    if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);    // while n is read
    const int64_t n = *n_dev;
    const int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    if (ntiles == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) fin((int64_t)0);
        return;
    }
    for (;;) {
        __syncthreads();
        const int64_t t = s_tile;
        __syncthreads();
        if (t >= ntiles) break;
        const int64_t t0 = t * kScanTile;
        // coalesced load into shared memory (one padding word per 32), and what
        // the output will read: all loads of a thread in flight at once
        typename Out::Read rd[kScanItems];
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const int j = threadIdx.x + k * kScanThreads;
            const int64_t i = t0 + j;
            s_v[j + (j >> 5)] = i < n ? in(i) : 0;
            if (i < n) rd[k] = out.read(i);
        }
        __syncthreads();
        // each thread: kScanItems consecutive values
        long long v[kScanItems];
        long long sum = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const int j = threadIdx.x * kScanItems + k;
            v[k] = s_v[j + (j >> 5)];
            sum += v[k];
        }
        const long long pre = block_excl_scan(sum, &s_tot);
        const long long agg = s_tot;
        if (threadIdx.x < 32) {
            const long long own[1] = {agg};
            long long excl[1];
            look_back<1>(status + 1, t, own, excl, overflow, timeout_bit, spin_limit);
            if (threadIdx.x == 0) s_excl = excl[0];
        }
        __syncthreads();
        const long long excl = s_excl;
        // offsets through shared memory, handed out in order
        long long run = excl + pre;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const int j = threadIdx.x * kScanItems + k;
            s_v[j + (j >> 5)] = (int32_t)run;
            run += v[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const int j = threadIdx.x + k * kScanThreads;
            const int64_t i = t0 + j;
            if (i < n) out(i, s_v[j + (j >> 5)], rd[k]);
        }
        if (t == ntiles - 1 && threadIdx.x == 0) fin((int64_t)(excl + agg));
        if (ntiles <= gridDim.x) break;        // every block has had its one tile
        if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);
    }
}

// inputs, outputs and endings of the scans
struct ScanI32 {
    const int32_t* p;
    __device__ int32_t operator()(int64_t i) const { return p[i]; }
};
struct ScanU8 {
    const uint8_t* p;
    __device__ int32_t operator()(int64_t i) const { return p[i]; }
};
// 1 where the sorted key changes: the first entry of a segment
struct ScanHeads {
    const uint64_t* key;
    __device__ int32_t operator()(int64_t i) const { return i == 0 || key[i] != key[i - 1]; }
};
struct ScanStore {
    int32_t* out;
    struct Read {};
    __device__ Read read(int64_t) const { return Read{}; }
    __device__ void operator()(int64_t i, int32_t v, const Read&) const { out[i] = v; }
};
// first[k] = the first entry of segment k
struct ScanFirsts {
    ScanHeads head;
    int32_t* first;
    using Read = int32_t;
    __device__ Read read(int64_t i) const { return head(i); }
    __device__ void operator()(int64_t i, int32_t v, Read h) const {
        if (h) first[v] = (int32_t)i;
    }
};
struct ScanTotal {
    int64_t* dst;        // may be null
    __device__ void operator()(int64_t total) const {
        if (dst) *dst = total;
    }
};
// the total also as the entry after the offsets
struct ScanTotalAfter {
    int64_t* dst;
    int32_t* off;
    const int64_t* n;
    __device__ void operator()(int64_t total) const {
        *dst = total;
        off[*n] = (int32_t)total;
    }
};
// the number of segments, and the end of the last one
struct ScanSegments {
    int64_t* dst;
    int32_t* first;
    const int64_t* n;
    __device__ void operator()(int64_t total) const {
        *dst = total;
        first[total] = (int32_t)*n;
    }
};

// a tile counter and one status word per tile
inline int64_t scan_status_words(int64_t n_cap) {
    return std::max<int64_t>((n_cap + kScanTile - 1) / kScanTile, 1) + 1;
}
inline unsigned long long* scan_status(msp_ctx& c, int64_t n_cap) {
    return c.sd_tmp.ensure<unsigned long long>((size_t)scan_status_words(n_cap));
}

// cleared: the scan's status words, if an earlier kernel has cleared them (no
// other scan in between); otherwise they are cleared here
template <class In, class Out, class Fin>
inline void scan_launch(msp_ctx& c, In in, Out out, Fin fin, const int64_t* n_dev, int64_t n_cap,
                        cudaStream_t s, unsigned long long* cleared = nullptr) {
    const int64_t tiles_cap = scan_status_words(n_cap) - 1;
    unsigned long long* status = cleared ? cleared : scan_status(c, n_cap);
    if (!cleared)
        MSP_CUDA(cudaMemsetAsync(status, 0, ((size_t)tiles_cap + 1) * sizeof(unsigned long long), s));
    const int G = (int)std::min<int64_t>(tiles_cap, (int64_t)c.sm_count * 4);
    k_scan_1p<<<G, kScanThreads, 0, s>>>(in, out, fin, n_dev, status, &dcounts(c)->overflow,
                                         kScanTimeoutBit, kSpinLimit);
    MSP_LAUNCH("scan");
}

}  // namespace msp
