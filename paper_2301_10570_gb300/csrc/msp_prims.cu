// msp_prims.cu -- device-wide exclusive scan and stable LSD radix sort used by
// the tree build, the pair lists, the descent and the request resolution.
#include "msp_scan.cuh"

namespace msp {

namespace {

// ---------------------------------------------------------------------------
// Stable LSD radix sort, one kernel per digit, the published single-pass scheme
// (Adinets and Merrill, "Onesweep: A Faster Least Significant Digit Radix Sort for
// GPUs", 2022; the look-back of Merrill and Garland, "Single-pass Parallel Prefix
// Scan with Decoupled Look-back", 2016).  A first kernel counts the digits of every
// pass in one reading of the keys; then each pass reads, ranks and writes its tiles
// once: a tile publishes its digit counts, looks back over its predecessors' (as the
// scan of msp_scan.cuh, eight tiles per step), and so knows where each of its digits
// goes without a histogram per tile, its scan and a second reading of the keys.
// The tile is put in digit order in shared memory first, so that the writes of a
// digit are contiguous.  Bound by latency below some 100,000 keys (a pass is one
// chain of tile number, loads, ranks, look-back and stores, about 9 us cold) and by
// the look-back and the scattered writes above.  The sorts of a rebuilt step at
// 262,144 neurons (63, 13 and 16 bits): 275 us in 60 launches with a histogram,
// three scan kernels and a scatter per 8-bit digit, 157 us in 14 launches now
// (serialised, cold); the step 822 -> 732 us.  Nine bits a digit: 7 passes for a Morton key.
// ---------------------------------------------------------------------------
constexpr int kRsThreads = 256;
constexpr int kRsItems = 8;
constexpr int kRsTile = kRsThreads * kRsItems;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsMaxBits = 9;                  // two digits per thread
constexpr int kRsBins = 1 << kRsMaxBits;
constexpr int kRsMaxPasses = 8;                // of 64 bits
constexpr int kRsLook = 8;                     // predecessors read per step
// a status word: flag (none, counts, prefix) and the 31-bit counts of digits
// 2 t and 2 t + 1 (n < 2^31)
constexpr unsigned long long kRsVal = (1ull << 31) - 1;

// Digit counts of all passes (hist: zero on entry), and the passes' status
// words cleared for the tiles that *n_dev (or n) elements fill.
__global__ void __launch_bounds__(kRsThreads)
k_rs_hist(const uint64_t* __restrict__ keys, int64_t n_host, const int64_t* __restrict__ n_dev,
          int passes, int bits, int32_t* __restrict__ hist,
          unsigned long long* __restrict__ status, int64_t status_stride) {
    __shared__ int32_t h[kRsMaxPasses * kRsBins];
    const int64_t n = n_dev ? *n_dev : n_host;
    const int bins = 1 << bits;
    for (int k = threadIdx.x; k < passes * bins; k += kRsThreads) h[k] = 0;
    const int64_t tid = blockIdx.x * (int64_t)kRsThreads + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * kRsThreads;
    const int64_t words = (n + kRsTile - 1) / kRsTile * (bins / 2);
    for (int ps = 0; ps < passes; ++ps)
        for (int64_t k = tid; k < words; k += stride) status[ps * status_stride + k] = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = tid - lane; i0 < n; i0 += stride) {
        const bool in = i0 + lane < n;
        const uint64_t key = in ? keys[i0 + lane] : 0ull;
        const unsigned act = __ballot_sync(0xffffffffu, in);
        for (int ps = 0; ps < passes; ++ps) {
            const int d = (int)((key >> (ps * bits)) & (uint64_t)(bins - 1));
            // the high digits of neighbouring keys are often all the same
            int same = 0;
            if (act == 0xffffffffu) __match_all_sync(0xffffffffu, d, &same);
            if (same) {
                if (lane == 0) atomicAdd(&h[ps * bins + d], 32);
            } else if (in) {
                atomicAdd(&h[ps * bins + d], 1);
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < passes * bins; k += kRsThreads)
        if (h[k]) atomicAdd(&hist[k], h[k]);
}

// One pass.  tile_ctr hands out the tiles in order (zero on entry), so every
// tile's predecessors have started; a wait of more than SPINS polls gives
// up, counts the tile as 0 and sets timeout_bit in *overflow.
template <int SPINS>
__global__ void __launch_bounds__(kRsThreads, 3)
k_rs_pass(const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin,
          uint64_t* __restrict__ kout, int32_t* __restrict__ vout, int64_t n_host,
          const int64_t* __restrict__ n_dev, int shift, int bits,
          const int32_t* __restrict__ hist, int32_t* __restrict__ tile_ctr,
          unsigned long long* status_, int64_t* __restrict__ overflow, int64_t timeout_bit) {
    __shared__ uint64_t s_key[kRsTile];
    __shared__ int32_t s_val[kRsTile];
    __shared__ uint16_t s_cnt[kRsWarps][kRsBins];   // per warp: count, then offset, of a digit
    __shared__ int32_t s_off[kRsBins];              // where it starts in the tile
    __shared__ int32_t s_dst[kRsBins];              // output minus tile position
    __shared__ int32_t s_warp[kRsWarps];
    __shared__ int32_t s_tile;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int bins = 1 << bits;
    // the reads that start a pass run together: the first tile's number, the
    // element count, the digits' totals (scanned while the keys are on their way)
    if (t == 0) s_tile = atomicAdd(tile_ctr, 1);
    const int32_t h0 = 2 * t < bins ? hist[2 * t] : 0, h1 = 2 * t < bins ? hist[2 * t + 1] : 0;
    const int64_t n = n_dev ? *n_dev : n_host;
    const int ntiles = (int)((n + kRsTile - 1) / kRsTile);
    volatile unsigned long long* status = status_;
    // exclusive sums over the digits, two per thread
    auto digit_scan = [&](int32_t a, int32_t b) {
        int32_t inc = a + b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) s_warp[w] = inc;
        __syncthreads();
        int32_t before = 0;
        for (int k = 0; k < w; ++k) before += s_warp[k];
        __syncthreads();
        return before + inc - (a + b);
    };
    int32_t base0 = -1;         // where digit 2 t starts in the output
    const unsigned lt = (1u << lane) - 1u;
    for (;;) {
        for (int k = t; k < kRsWarps * kRsBins / 2; k += kRsThreads)
            reinterpret_cast<uint32_t*>(&s_cnt[0][0])[k] = 0u;
        __syncthreads();
        const int tile = s_tile;
        if (tile >= ntiles) break;
        // warp w takes 256 consecutive elements, lane-consecutive per round;
        // an element's rank is its digit's count in the warp so far
        const int64_t base = (int64_t)tile * kRsTile + w * (32 * kRsItems) + lane;
        uint64_t key[kRsItems];
        int32_t val[kRsItems];
        int rank[kRsItems];
#pragma unroll
        for (int r = 0; r < kRsItems; ++r) {
            const bool in = base + 32 * r < n;
            key[r] = in ? kin[base + 32 * r] : 0ull;
            val[r] = in ? vin[base + 32 * r] : 0;
        }
        if (base0 < 0) base0 = digit_scan(h0, h1);
#pragma unroll
        for (int r = 0; r < kRsItems; ++r) {
            const bool in = base + 32 * r < n;
            const int d = in ? (int)((key[r] >> shift) & (uint64_t)(bins - 1)) : bins;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const int before = in ? s_cnt[w][d] : 0;
            rank[r] = before + __popc(peers & lt);
            __syncwarp();
            if (in && (peers & lt) == 0) s_cnt[w][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // the tile's digit counts; the warps' counts become offsets
        int32_t c0 = 0, c1 = 0;
        if (2 * t < bins)
#pragma unroll
            for (int k = 0; k < kRsWarps; ++k) {
                uint32_t* p = reinterpret_cast<uint32_t*>(&s_cnt[k][2 * t]);
                const uint32_t v = *p;
                *p = (uint32_t)c0 | ((uint32_t)c1 << 16);
                c0 += (int32_t)(v & 0xffffu);
                c1 += (int32_t)(v >> 16);
            }
        unsigned long long* mine = status_ + (int64_t)tile * (bins / 2) + t;
        auto word = [](unsigned long long flag, int64_t a, int64_t b) {
            return flag << 62 | (unsigned long long)b << 31 | (unsigned long long)a;
        };
        if (2 * t < bins)
            *(volatile unsigned long long*)mine = word(tile == 0 ? 2 : 1, c0, c1);
        const int32_t e = digit_scan(c0, c1);
        if (2 * t < bins) {
            s_off[2 * t] = e;
            s_off[2 * t + 1] = e + c0;
            int64_t p0 = 0, p1 = 0;      // the digits' counts in the tiles before
            bool done = tile == 0;
            for (int j = tile - 1; j >= 0 && !done; j -= kRsLook) {
                unsigned long long v[kRsLook];
#pragma unroll
                for (int k = 0; k < kRsLook; ++k)
                    v[k] = j - k >= 0 ? status[(int64_t)(j - k) * (bins / 2) + t] : 2ull << 62;
#pragma unroll
                for (int k = 0; k < kRsLook; ++k) {
                    if (done) continue;
                    int spin = 0;
                    while ((v[k] >> 62) == 0 && spin < SPINS) {
                        ++spin;
                        v[k] = status[(int64_t)(j - k) * (bins / 2) + t];
                    }
                    if ((v[k] >> 62) == 0)
                        atomicOr(reinterpret_cast<unsigned long long*>(overflow),
                                 (unsigned long long)timeout_bit);
                    p0 += (int64_t)(v[k] & kRsVal);
                    p1 += (int64_t)((v[k] >> 31) & kRsVal);
                    done = (v[k] >> 62) != 1;
                }
            }
            if (tile > 0) *(volatile unsigned long long*)mine = word(2, p0 + c0, p1 + c1);
            s_dst[2 * t] = (int32_t)(base0 + p0 - e);
            s_dst[2 * t + 1] = (int32_t)(base0 + h0 + p1 - (e + c0));
        }
        __syncthreads();
        // into digit order, then out
#pragma unroll
        for (int r = 0; r < kRsItems; ++r)
            if (base + 32 * r < n) {
                const int d = (int)((key[r] >> shift) & (uint64_t)(bins - 1));
                const int pos = s_off[d] + s_cnt[w][d] + rank[r];
                s_key[pos] = key[r];
                s_val[pos] = val[r];
            }
        __syncthreads();
        const int m = (int)min((int64_t)kRsTile, n - (int64_t)tile * kRsTile);
        for (int i = t; i < m; i += kRsThreads) {
            const uint64_t k = s_key[i];
            const int64_t o = (int64_t)s_dst[(int)((k >> shift) & (uint64_t)(bins - 1))] + i;
            // a wait that gave up may leave a wrong offset
            if (o >= 0 && o < n) {
                kout[o] = k;
                vout[o] = s_val[i];
            }
        }
        if (ntiles <= (int)gridDim.x) break;        // every block has had its one tile
        __syncthreads();
        if (t == 0) s_tile = atomicAdd(tile_ctr, 1);
    }
}

}  // namespace

namespace {
__global__ void k_dev_set(int64_t* dst, int64_t v) { *dst = v; }
}  // namespace

void dev_set(int64_t* dst, int64_t v, cudaStream_t s) {
    k_dev_set<<<1, 1, 0, s>>>(dst, v);
    MSP_LAUNCH("dev_set");
}
void pull_counts(msp_ctx& c, cudaStream_t s) {
    MSP_CUDA(cudaMemcpyAsync(c.hcount, c.dcount.p, sizeof(DevCounts), cudaMemcpyDeviceToHost, s));
    MSP_CUDA(cudaStreamSynchronize(s));
    if (c.hcount->overflow & kScanTimeoutBit) {
        c.hcount->overflow &= ~kScanTimeoutBit;
        dev_set(&dcounts(c)->overflow, c.hcount->overflow, s);
        throw Error(MSP_ERR_TIMEOUT, "a bounded wait of the device scan gave up");
    }
}

void scan_dev(msp_ctx& c, const int32_t* in, int32_t* out, const int64_t* n_dev, int64_t n_cap,
              int64_t* total_dst, cudaStream_t s) {
    scan_launch(c, ScanI32{in}, ScanStore{out}, ScanTotal{total_dst}, n_dev, n_cap, s);
}

// The bounded waits of the scan and of the sort, exercised: the tile counter
// starts at 1, so tile 0 is never taken and its status never published; the tiles
// after it wait on it at most kSelftestSpins polls, give up, record the timeout
// bit and finish.  The next pull_counts then reports MSP_ERR_TIMEOUT.  (The look-back
// of the octree levels, the traversal depths and the compaction is the scan's.)
void scan_wait_selftest(msp_ctx& c, cudaStream_t s) {
    const int64_t n = 3 * (int64_t)kScanTile;
    int32_t* in = c.cnt.ensure<int32_t>((size_t)n);
    int32_t* out = c.off.ensure<int32_t>((size_t)n);
    int64_t* nd = c.gm_cnt.ensure<int64_t>(4);
    unsigned long long* status = c.sd_tmp.ensure<unsigned long long>(4 + 1);
    MSP_CUDA(cudaMemsetAsync(in, 0, (size_t)n * sizeof(int32_t), s));
    MSP_CUDA(cudaMemsetAsync(status, 0, 5 * sizeof(unsigned long long), s));
    dev_set(reinterpret_cast<int64_t*>(status), 1, s);       // tile 0 is skipped
    dev_set(nd, n, s);
    k_scan_1p<<<3, kScanThreads, 0, s>>>(ScanI32{in}, ScanStore{out}, ScanTotal{nd + 1}, nd, status,
                                         &dcounts(c)->overflow, kScanTimeoutBit, kSelftestSpins);
    MSP_LAUNCH("scan_wait_selftest");
}

void sort_wait_selftest(msp_ctx& c, cudaStream_t s) {
    const int64_t n = 3 * (int64_t)kRsTile;
    const int bits = 8, bins = 1 << bits;
    uint64_t* key[2] = {c.rq_key0.ensure<uint64_t>((size_t)n), c.keys1.ensure<uint64_t>((size_t)n)};
    int32_t* val[2] = {c.rq_val0.ensure<int32_t>((size_t)n), c.vals1.ensure<int32_t>((size_t)n)};
    int32_t* hist = c.rs_hist.ensure<int32_t>((size_t)kRsMaxPasses * (kRsBins + 1));
    unsigned long long* status = c.rs_status.ensure<unsigned long long>((size_t)(3 * bins / 2));
    MSP_CUDA(cudaMemsetAsync(key[0], 0, (size_t)n * sizeof(uint64_t), s));
    MSP_CUDA(cudaMemsetAsync(val[0], 0, (size_t)n * sizeof(int32_t), s));
    MSP_CUDA(cudaMemsetAsync(hist, 0, (size_t)(bins + 2) * sizeof(int32_t), s));
    k_rs_hist<<<3, kRsThreads, 0, s>>>(key[0], n, nullptr, 1, bits, hist, status, 3 * bins / 2);
    MSP_LAUNCH("rs_hist");
    // the tile counter (hist[bins], with the zero above it) starts at 1
    dev_set(reinterpret_cast<int64_t*>(hist + bins), 1, s);
    k_rs_pass<kSelftestSpins><<<3, kRsThreads, 0, s>>>(key[0], val[0], key[1], val[1], n, nullptr, 0, bits, hist,
                                       hist + bins, status, &dcounts(c)->overflow, kScanTimeoutBit);
    MSP_LAUNCH("sort_wait_selftest");
}

static int rs_passes(int64_t n_cap, int bits) {
    return n_cap <= 1 || bits <= 0 ? 0 : (bits + kRsMaxBits - 1) / kRsMaxBits;
}

// bits of a digit, status words of a pass
static int rs_digit(int passes, int bits) { return (bits + passes - 1) / passes; }
static int64_t rs_stride(int64_t n_cap, int per) {
    return (n_cap + kRsTile - 1) / kRsTile * ((1 << per) / 2);
}

void radix_reserve(msp_ctx& c, int64_t n_cap, int bits) {
    const int passes = rs_passes(n_cap, bits);
    if (passes == 0) return;
    c.rs_hist.ensure<int32_t>((size_t)kRsMaxPasses * (kRsBins + 1));
    c.rs_status.ensure<unsigned long long>(
        (size_t)(passes * rs_stride(n_cap, rs_digit(passes, bits))));
}

bool radix_from_tmp(int64_t n_cap, int bits) { return (rs_passes(n_cap, bits) & 1) != 0; }

void radix_sort_dev(msp_ctx& c, uint64_t* keys, int32_t* vals, uint64_t* keys_tmp,
                    int32_t* vals_tmp, const int64_t* n_dev, int64_t n_cap, int bits,
                    cudaStream_t s) {
    const int passes = rs_passes(n_cap, bits);
    if (passes == 0) return;
    radix_reserve(c, n_cap, bits);
    const int per = rs_digit(passes, bits), bins = 1 << per;
    const int64_t tiles_cap = (n_cap + kRsTile - 1) / kRsTile, stride = rs_stride(n_cap, per);
    // digit counts and tile counters (cleared here), status words (cleared
    // by the counting kernel, as many as the elements need)
    int32_t* hist = c.rs_hist.get<int32_t>();
    int32_t* ctr = hist + passes * bins;
    unsigned long long* status = c.rs_status.get<unsigned long long>();
    MSP_CUDA(cudaMemsetAsync(hist, 0, (size_t)passes * (bins + 1) * sizeof(int32_t), s));
    uint64_t *ka = keys, *kb = keys_tmp;
    int32_t *va = vals, *vb = vals_tmp;
    if (passes & 1) {
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    const int gh = (int)std::min<int64_t>((n_cap + 4 * kRsThreads - 1) / (4 * kRsThreads),
                                          (int64_t)c.sm_count * 4);
    k_rs_hist<<<gh, kRsThreads, 0, s>>>(ka, n_cap, n_dev, passes, per, hist, status, stride);
    MSP_LAUNCH("rs_hist");
    const int g = (int)std::min<int64_t>(tiles_cap, (int64_t)c.sm_count * 3);
    for (int ps = 0; ps < passes; ++ps) {
        k_rs_pass<kSpinLimit><<<g, kRsThreads, 0, s>>>(ka, va, kb, vb, n_cap, n_dev, ps * per, per,
                                           hist + ps * bins, ctr + ps, status + ps * stride,
                                           &dcounts(c)->overflow, kScanTimeoutBit);
        MSP_LAUNCH("rs_pass");
        std::swap(ka, kb);
        std::swap(va, vb);
    }
}

}  // namespace msp

// ---------------------------------------------------------------------------
// The counter-based generator of every draw, on caller-given counters and
// keys (msp_philox of include/msp.h)
// ---------------------------------------------------------------------------
namespace {
__global__ void k_philox_blocks(int64_t n, const uint32_t* __restrict__ ctr,
                                const uint32_t* __restrict__ key, uint32_t* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c[4] = {ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]};
        msp::philox4x32_10(c, key[2 * i], key[2 * i + 1]);
        out[4 * i] = c[0];
        out[4 * i + 1] = c[1];
        out[4 * i + 2] = c[2];
        out[4 * i + 3] = c[3];
    }
}
}  // namespace

extern "C" msp_status msp_philox(int64_t n, const uint32_t* ctr, const uint32_t* key,
                                 uint32_t* out, void* stream) {
    if (n < 0) {
        msp::set_last_error("msp_philox: n must not be negative");
        return MSP_ERR_INVALID_ARG;
    }
    if (n == 0) return MSP_OK;
    if (!ctr || !key || !out) {
        msp::set_last_error("msp_philox: null pointer");
        return MSP_ERR_INVALID_ARG;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_philox_blocks<<<msp::grid_for(n, 256), 256, 0, s>>>(n, ctr, key, out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        msp::set_last_error(cudaGetErrorString(e));
        return MSP_ERR_CUDA;
    }
    msp::g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
    msp::set_last_error("");
    return MSP_OK;
}
