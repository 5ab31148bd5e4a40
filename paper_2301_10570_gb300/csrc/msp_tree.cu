// msp_tree.cu -- steps a1-a4: Morton keys, stable sort + gather into a
// Morton-ordered float4 array, the adaptive octree (Section 3.2) built level
// by level, and the per-box sums of vacant elements and centroids.
#include "msp_scan.cuh"

namespace msp {

namespace {

// q = floor((v - o) * scale) in single precision with round-to-nearest, then
// clamped to the 2^21 grid; NaN maps to 0.
__device__ inline uint32_t quantise(float v, float o, float scale) {
    float f = floorf(__fmul_rn(__fsub_rn(v, o), scale));
    if (!(f >= 0.0f)) return 0u;
    if (f >= 2097152.0f) return 2097151u;
    return (uint32_t)f;
}

// start of a build; also copies the caller's counts (cp.n > 0) and clears the
// status words of the element scan and (n_arrive > 0) the arrival counters of the
// aggregation
__global__ void k_build_init(DevCounts* dc, int64_t n, unsigned long long* __restrict__ status,
                             int64_t n_status, int32_t* __restrict__ arrive, int64_t n_arrive,
                             CountCopy cp) {
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    if (i0 == 0) {
        dc->n = n;
        dc->bad_pos = 0;
        dc->pos_sum = 0;
    }
    for (int64_t i = i0; i < n_status; i += step) status[i] = 0;
    for (int64_t i = i0; i < n_arrive; i += step) arrive[i] = 0;
    for (int k = 0; k < 4; ++k) {
        // 16 bytes at a time where the caller's array allows it
        const int64_t nv = reinterpret_cast<uintptr_t>(cp.src[k]) % 16 == 0 ? cp.n / 16 : 0;
        for (int64_t i = i0; i < nv; i += step)
            reinterpret_cast<uint4*>(cp.dst[k])[i] = reinterpret_cast<const uint4*>(cp.src[k])[i];
        for (int64_t i = 16 * nv + i0; i < cp.n; i += step) cp.dst[k][i] = cp.src[k][i];
    }
}

// order-independent checksum of the positions: the sum over i (modulo 2^64)
// of a mix of i and every bit of the three coordinates (the finaliser of
// SplitMix64, Steele, Lea, Flood, "Fast splittable pseudorandom number
// generators", OOPSLA 2014, applied twice)
__device__ inline unsigned long long pos_mix(unsigned long long h) {
    h ^= h >> 30;
    h *= 0xBF58476D1CE4E5B9ull;
    h ^= h >> 27;
    h *= 0x94D049BB133111EBull;
    h ^= h >> 31;
    return h;
}

__device__ inline unsigned long long pos_hash(int64_t i, float x, float y, float z) {
    const unsigned long long xy = ((unsigned long long)__float_as_uint(x) << 32) |
                                  __float_as_uint(y);
    const unsigned long long h = pos_mix(xy ^ ((unsigned long long)i * 0x9E3779B97F4A7C15ull));
    return pos_mix(h ^ ((unsigned long long)__float_as_uint(z) * 0xD6E8FEB86659FD93ull));
}

// adds the block's sum to *out (one atomic per block: one per warp, at
// 1,000,000 neurons, took longer than reading the positions)
__device__ inline void add_pos_sum(unsigned long long acc, unsigned long long* out) {
    __shared__ unsigned long long s_sum;
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, acc);
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(out, s_sum);
}

__global__ void k_pos_sum(const float* __restrict__ x, const float* __restrict__ y,
                          const float* __restrict__ z, int64_t n,
                          unsigned long long* __restrict__ out) {
    unsigned long long acc = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        acc += pos_hash(i, x[i], y[i], z[i]);
    add_pos_sum(acc, out);
}

// End of a graph step's build, in its last kernel (k_aggregate_tree).
struct BuildEnd {
    DevCounts* dc;
    bool graph;              // otherwise nothing to do (the host looks)
    // octree kept: the positions must be those of the build that made it
    // (checksum ref) and the arrays that build's (stamp gen), or the step halts
    bool keep;
    uint64_t ref, gen;
    // more elements than the selection's buffers hold leave the step with no
    // element (every element kernel is bounded by the count)
    int64_t elem_cap;
    __device__ void operator()() const {
        if (!graph) return;
        if (keep && (dc->pos_sum != ref || dc->tree_gen != gen)) dc->bad_pos = 1;
        if (dc->n_elem > elem_cap) {
            dc->halt |= kHaltElements;
            dc->n_elem = 0;
        }
    }
};

// The first kernel of a build that makes the octree anew, and the last moment at
// which the arrays of the one before are whole: the build's own stamp, which no
// capture holds yet and which a build that fails later on leaves too.
__device__ __forceinline__ void put_stamp(DevCounts* dc, uint64_t stamp) {
    if (blockIdx.x == 0 && threadIdx.x == 0) dc->tree_gen = stamp;
}

// keys; a position outside [origin, origin + side) or not finite is counted
// (the build then fails: the tree's boxes must contain their points)
__global__ void k_morton(const float* __restrict__ x, const float* __restrict__ y,
                         const float* __restrict__ z, int64_t n, float ox, float oy, float oz,
                         float side, float scale, uint64_t* __restrict__ keys,
                         int32_t* __restrict__ vals, DevCounts* dc, uint64_t stamp) {
    put_stamp(dc, stamp);
    bool any_bad = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        any_bad |= !(x[i] >= ox && x[i] < ox + side && y[i] >= oy && y[i] < oy + side &&
                     z[i] >= oz && z[i] < oz + side);
        uint32_t qx = quantise(x[i], ox, scale);
        uint32_t qy = quantise(y[i], oy, scale);
        uint32_t qz = quantise(z[i], oz, scale);
        keys[i] = (spread_by3(qx) << 2) | (spread_by3(qy) << 1) | spread_by3(qz);
        vals[i] = (int32_t)i;
    }
    if (__any_sync(0xffffffffu, any_bad) && (threadIdx.x & 31) == 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&dc->bad_pos), 1ull);
}

// Keys of independent networks in local frames.  Neuron i belongs to the
// network k with off[k] <= i < off[k+1]; that network's cell at level L0 has
// the grid coordinates 2 (k mod G, (k / G) mod G, k / G^2), G = 2^(L0-1), and
// the neuron's position is relative to the cell's low corner, inside
// [0, cs).  Each axis of the key holds the cell's coordinate in its top L0
// bits and the local position, quantised on the same grid, below them: the
// key the point would have in one common frame, without ever forming its
// position in that frame in single precision.
__global__ void k_morton_frames(const float* __restrict__ x, const float* __restrict__ y,
                                const float* __restrict__ z, int64_t n,
                                const int64_t* __restrict__ off, int64_t nf, int L0, float cs,
                                float scale, uint64_t* __restrict__ keys,
                                int32_t* __restrict__ vals, DevCounts* dc, uint64_t stamp) {
    put_stamp(dc, stamp);
    const int sh = kMortonBits - L0;
    const uint32_t qmax = (1u << sh) - 1u;
    const int64_t G = 1ll << (L0 - 1);
    bool any_bad = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = nf;   // off[lo] <= i < off[hi]
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (off[mid] <= i) lo = mid; else hi = mid;
        }
        const uint32_t cx = (uint32_t)(2 * (lo % G)), cy = (uint32_t)(2 * ((lo / G) % G)),
                       cz = (uint32_t)(2 * (lo / (G * G)));
        any_bad |= !(x[i] >= 0.f && x[i] < cs && y[i] >= 0.f && y[i] < cs && z[i] >= 0.f &&
                     z[i] < cs);
        const uint32_t qx = (cx << sh) | min(quantise(x[i], 0.f, scale), qmax);
        const uint32_t qy = (cy << sh) | min(quantise(y[i], 0.f, scale), qmax);
        const uint32_t qz = (cz << sh) | min(quantise(z[i], 0.f, scale), qmax);
        keys[i] = (spread_by3(qx) << 2) | (spread_by3(qy) << 1) | spread_by3(qz);
        vals[i] = (int32_t)i;
    }
    if (__any_sync(0xffffffffu, any_bad) && (threadIdx.x & 31) == 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&dc->bad_pos), 1ull);
}

__device__ __forceinline__ uint32_t pack_counts(uint8_t type, uint8_t va, uint8_t vde, uint8_t vdi) {
    return (uint32_t)(type ? 1u : 0u) | ((uint32_t)va << 8) | ((uint32_t)vde << 16) |
           ((uint32_t)vdi << 24);
}
// the dendrite weights, and their log2 (-inf for none), added in the exponent
__device__ __forceinline__ void put_weights(int64_t j, uint8_t vde, uint8_t vdi, float2* wts,
                                            float2* lw) {
    wts[j] = make_float2((float)vde, (float)vdi);
    lw[j] = make_float2(vde ? log2f((float)vde) : -INFINITY, vdi ? log2f((float)vdi) : -INFINITY);
}

// the octree's first levels in one block (k_tree_top), and the cells of the last
constexpr int kTopLevels = 4;
constexpr int kTopCells = 1 << (3 * kTopLevels);

// points and weights into sorted order; and where the cells of level kTopLevels
// start: cells[i] = the first point of a cell >= i, i in [0, kTopCells]
__global__ void k_gather(const int32_t* __restrict__ order, int64_t n, const float* __restrict__ x,
                         const float* __restrict__ y, const float* __restrict__ z,
                         const uint8_t* __restrict__ type, const uint8_t* __restrict__ va,
                         const uint8_t* __restrict__ vde, const uint8_t* __restrict__ vdi,
                         int32_t* __restrict__ perm, float4* __restrict__ pts,
                         float2* __restrict__ wts, float2* __restrict__ lw,
                         const uint64_t* __restrict__ keys, int32_t* __restrict__ cells) {
    constexpr int kShift = 3 * (kMortonBits - kTopLevels);
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = order[j];
        const int cell = (int)(keys[j] >> kShift) & (kTopCells - 1);
        const int prev = j > 0 ? (int)(keys[j - 1] >> kShift) & (kTopCells - 1) : -1;
        for (int k = prev + 1; k <= cell; ++k) cells[k] = (int32_t)j;
        if (j == n - 1)
            for (int k = cell + 1; k <= kTopCells; ++k) cells[k] = (int32_t)n;
        perm[j] = i;
        pts[j] = make_float4(x[i], y[i], z[i],
                             __uint_as_float(pack_counts(type[i], va[i], vde[i], vdi[i])));
        put_weights(j, vde[i], vdi[i], wts, lw);
    }
}

// A build that keeps the sorted order: the positions' checksum (read in the
// caller's order, coalesced) and the counts gathered again; the sorted
// positions are those of the build that made the order, or the checksum tells
// and the octree is built anew.  Bound by the gather's 32-byte sectors.
// 1,000,000 neurons: 33 us for a full gather and 18 for the checksum before, 21 now.
__global__ void k_gather_counts(int64_t n, const float* __restrict__ x,
                                const float* __restrict__ y, const float* __restrict__ z,
                                const uint8_t* __restrict__ type, const uint8_t* __restrict__ va,
                                const uint8_t* __restrict__ vde, const uint8_t* __restrict__ vdi,
                                const int32_t* __restrict__ perm, float4* __restrict__ pts,
                                float2* __restrict__ wts, float2* __restrict__ lw,
                                unsigned long long* __restrict__ sum) {
    unsigned long long acc = 0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        acc += pos_hash(j, x[j], y[j], z[j]);
        const int32_t i = perm[j];
        pts[j].w = __uint_as_float(pack_counts(type[i], va[i], vde[i], vdi[i]));
        put_weights(j, vde[i], vdi[i], wts, lw);
    }
    add_pos_sum(acc, sum);
}

// The octree arrays and the split rule of a build.  Per-network leaf
// capacities (cap non-null, points in frames): a box at or below the frame
// level splits above its network's capacity, a box above it (several
// networks' cells) always splits.
struct LevelArgs {
    int64_t n;
    const uint64_t* keys;
    uint8_t* level;
    uint64_t* prefix;
    int32_t *first, *count, *parent, *child_first;
    uint8_t* nchild;
    int leaf_capacity, max_depth;
    const int32_t* cap;
    int frame_level;
    int64_t nf;
    int64_t node_cap;
};

__device__ __forceinline__ bool splits(const LevelArgs& a, int64_t i, int level, int32_t c) {
    int cap = a.leaf_capacity;
    if (a.cap)
        cap = level >= a.frame_level ? a.cap[box_frame(a.prefix[i], level, a.frame_level, a.nf)] : -1;
    return c > cap && level < a.max_depth;
}

// First index in [lo, hi) whose octant (at shift) is at least o; octants are
// non-decreasing inside a box because the higher bits are the box prefix.
// Seven probes at once leave an eighth of the range: a chain of 6 reads
// instead of 18 in a box of 262,144 points.
__device__ __forceinline__ int32_t octant_lower_bound(const uint64_t* __restrict__ keys, int32_t lo,
                                                      int32_t hi, int shift, uint32_t o) {
    while (lo < hi) {
        const int64_t len = hi - lo;
        uint64_t k[7];
#pragma unroll
        for (int p = 0; p < 7; ++p) k[p] = keys[lo + (int32_t)(len * (p + 1) >> 3)];
        int below = 0;
#pragma unroll
        for (int p = 0; p < 7; ++p) below += ((k[p] >> shift) & 7u) < o;
        const int32_t l0 = lo;
        if (below > 0) lo = l0 + (int32_t)(len * below >> 3) + 1;
        if (below < 7) hi = l0 + (int32_t)(len * (below + 1) >> 3);
    }
    return lo;
}

// Octant boundaries of box i (level `level`), 8 lanes per box: lane o returns
// the start and end of octant o (empty unless the box splits).  Whole warps
// take part (4 boxes per warp).
__device__ __forceinline__ void octant_split(const LevelArgs& a, bool valid, int64_t i, int level,
                                             int32_t& start, int32_t& end) {
    const int o = threadIdx.x & 7;
    int32_t lo = 0, e = 0;
    if (valid) {
        const int32_t c = a.count[i];
        lo = e = a.first[i];
        if (splits(a, i, level, c))
            e = octant_lower_bound(a.keys, lo, lo + c, 3 * (kMortonBits - (level + 1)),
                                   (uint32_t)o + 1);
    }
    const int32_t prev = __shfl_up_sync(0xffffffffu, e, 1);
    end = e;
    start = o == 0 ? lo : prev;
}

// The children of box i, one per lane with a non-empty octant: first child at
// cf, this lane's child at ci; grp: the box's non-empty octants.
__device__ __forceinline__ void emit_children(const LevelArgs& a, int64_t i, int level,
                                              unsigned grp, int64_t cf, int64_t ci, int32_t start,
                                              int32_t end) {
    const int o = threadIdx.x & 7;
    if (o == 0) {
        a.child_first[i] = (int32_t)cf;
        a.nchild[i] = (uint8_t)__popc(grp);
    }
    if (end > start) {
        a.level[ci] = (uint8_t)(level + 1);
        a.prefix[ci] = (a.prefix[i] << 3) | (uint64_t)o;
        a.first[ci] = start;
        a.count[ci] = end - start;
        a.parent[ci] = (int32_t)i;
        a.child_first[ci] = -1;
        a.nchild[ci] = 0;
    }
}

// The root and the levels below it down to level `levels` (at most kTopLevels) by
// one block, a block barrier between levels instead of a launch each.  A box's
// octants are looked up in cells, where the cells of level kTopLevels start in the
// keys (k_gather finds them on its way).  Bound by the chain of barriers and of
// reads of what the level above wrote.  262,144 / 21,013 neurons (serialised,
// cold), down to level 4: 33 + 14 / 25 + 11 us with a search per box and level,
// three levels here and the fourth a launch; 12 / 10 us now.
constexpr int kTopRounds = (1 << (3 * (kTopLevels - 1))) / 128;   // of 128 boxes

__global__ void __launch_bounds__(1024) k_tree_top(LevelArgs a, int levels,
                                                   const int32_t* __restrict__ cells,
                                                   DevCounts* dc) {
    __shared__ int32_t s_b[kTopCells + 1];
    __shared__ int s_off[32 * kTopRounds];
    __shared__ int s_tot;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        dc->level_start[0] = 0;
        dc->level_start[1] = 1;
        dc->overflow &= ~16ll;
        dc->more_levels = 0;
        a.level[0] = 0;
        a.prefix[0] = 0;
        a.first[0] = 0;
        a.count[0] = (int32_t)a.n;
        a.parent[0] = -1;
        a.child_first[0] = -1;
        a.nchild[0] = 0;
    }
    // (inside [0, n] also after a sort whose wait gave up, which the host reports)
    if (a.n > 0)
        for (int i = threadIdx.x; i <= kTopCells; i += 1024)
            s_b[i] = (int32_t)min((uint32_t)cells[i], (uint32_t)a.n);
    int64_t l0 = 0, nl = 1;
    for (int l = 0; l < levels; ++l) {
        __syncthreads();
        const int64_t next0 = l0 + nl;
        int32_t start[kTopRounds], end[kTopRounds];
        unsigned m[kTopRounds];
#pragma unroll
        for (int r = 0; r < kTopRounds; ++r) {
            const int64_t k = 128 * r + 4 * w + (lane >> 3), i = l0 + k;
            start[r] = end[r] = 0;              // of octant lane & 7
            if (k < nl && splits(a, i, l, a.count[i])) {
                const int sh = 3 * (kTopLevels - l - 1);
                const int cell = (int)(a.prefix[i] << 3) + (lane & 7);
                start[r] = s_b[cell << sh];
                end[r] = s_b[(cell + 1) << sh];
            }
            m[r] = __ballot_sync(0xffffffffu, end[r] > start[r]);
            if (lane == 0) s_off[32 * r + w] = __popc(m[r]);
        }
        __syncthreads();
        if (w == 0) {
            int v[kTopRounds], sum = 0;
#pragma unroll
            for (int r = 0; r < kTopRounds; ++r) {
                v[r] = s_off[kTopRounds * lane + r];
                sum += v[r];
            }
            int inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            int run = inc - sum;
#pragma unroll
            for (int r = 0; r < kTopRounds; ++r) {
                s_off[kTopRounds * lane + r] = run;
                run += v[r];
            }
            if (lane == 31) s_tot = inc;
        }
        __syncthreads();
        // the node arrays could not hold the level (a bound that cannot be
        // exceeded; guarded all the same)
        const bool fits = next0 + s_tot <= a.node_cap;
        if (!fits && threadIdx.x == 0) {
            dc->overflow |= 16;
            dc->need_nodes = next0 + s_tot;
        }
#pragma unroll
        for (int r = 0; r < kTopRounds; ++r) {
            const int64_t k = 128 * r + 4 * w + (lane >> 3);
            const int64_t at = next0 + s_off[32 * r + w];
            const unsigned grp = (m[r] >> (lane & ~7)) & 0xffu;
            if (k < nl && grp && fits)
                emit_children(a, l0 + k, l, grp, at + __popc(m[r] & ((1u << (lane & ~7)) - 1u)),
                              at + __popc(m[r] & ((1u << lane) - 1u)), start[r], end[r]);
        }
        const int64_t made = fits ? s_tot : 0;
        if (threadIdx.x == 0) dc->level_start[l + 2] = next0 + made;
        l0 = next0;
        nl = made;
    }
}

// One level: the children of the boxes [level_start[l], level_start[l+1]),
// appended in box order.  A tile of 128 boxes finds its octant boundaries,
// publishes its number of children, looks back and writes them: one launch
// (the count, its scan and the writing with a second search took 24 us a
// level; serialised, cold).  COUNT_ONLY: whether a box of the level would
// split (more_levels).
constexpr int kLevelRounds = 4;
constexpr int kLevelTile = 32 * kLevelRounds;

template <bool COUNT_ONLY>
__global__ void __launch_bounds__(256)
k_tree_level(LevelArgs a, int level, DevCounts* dc, unsigned long long* status,
             int64_t timeout_bit) {
    __shared__ int s_off[8 * kLevelRounds];
    __shared__ int s_tot;
    __shared__ long long s_excl;
    __shared__ int64_t s_tile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (!COUNT_ONLY && threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);
    const int64_t l0 = dc->level_start[level], nl = dc->level_start[level + 1] - l0;
    const int64_t next0 = l0 + nl;
    if (COUNT_ONLY) {
        bool any = false;
        for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nl;
             k += (int64_t)gridDim.x * blockDim.x)
            any |= splits(a, l0 + k, level, a.count[l0 + k]);
        if (__any_sync(0xffffffffu, any) && lane == 0)
            atomicOr(reinterpret_cast<unsigned long long*>(&dc->more_levels), 1ull);
        return;
    }
    const int64_t ntiles = (nl + kLevelTile - 1) / kLevelTile;
    if (ntiles == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) dc->level_start[level + 2] = next0;
        return;
    }
    for (;;) {
        __syncthreads();
        const int64_t t = s_tile;
        if (t >= ntiles) break;
        int32_t start[kLevelRounds], end[kLevelRounds];
        unsigned m[kLevelRounds];
#pragma unroll
        for (int r = 0; r < kLevelRounds; ++r) {
            const int64_t k = t * kLevelTile + 32 * r + 4 * w + (lane >> 3);
            octant_split(a, k < nl, l0 + k, level, start[r], end[r]);
            m[r] = __ballot_sync(0xffffffffu, end[r] > start[r]);
            if (lane == 0) s_off[8 * r + w] = __popc(m[r]);
        }
        __syncthreads();
        if (w == 0) {
            const int v = s_off[lane];
            int inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            s_off[lane] = inc - v;
            const long long own[1] = {(long long)__shfl_sync(0xffffffffu, inc, 31)};
            long long excl[1];
            look_back<1>(status + 1, t, own, excl, &dc->overflow, timeout_bit, kSpinLimit);
            if (lane == 0) {
                s_excl = excl[0];
                s_tot = (int)own[0];
            }
        }
        __syncthreads();
        const int64_t at0 = next0 + s_excl;
        const bool fits = at0 + s_tot <= a.node_cap;
#pragma unroll
        for (int r = 0; r < kLevelRounds; ++r) {
            const int64_t k = t * kLevelTile + 32 * r + 4 * w + (lane >> 3);
            const int64_t at = at0 + s_off[8 * r + w];
            const unsigned grp = (m[r] >> (lane & ~7)) & 0xffu;
            if (k < nl && grp && fits)
                emit_children(a, l0 + k, level, grp,
                              at + __popc(m[r] & ((1u << (lane & ~7)) - 1u)),
                              at + __popc(m[r] & ((1u << lane) - 1u)), start[r], end[r]);
        }
        if (t == ntiles - 1 && threadIdx.x == 0) {
            int64_t e = at0 + s_tot;
            if (e > a.node_cap) {
                atomicOr(reinterpret_cast<unsigned long long*>(&dc->overflow), 16ull);
                dc->need_nodes = e;
                e = next0;
            }
            dc->level_start[level + 2] = e;
        }
        if (ntiles <= gridDim.x) break;        // every block has had its one tile
        __syncthreads();
        if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);
    }
}

// Box aggregates, one launch for the whole octree.  A leaf sums its points;
// an inner box combines its children, and it is computed by the warp of its
// last child to finish: every box, once written, adds one to its parent's
// arrival counter (an acquire-release atomic: the box's results are visible
// before the arrival, the siblings' after it), and the warp that brings the
// counter to the parent's child count resets it and goes on with the parent,
// up to the root.
// Centroids are accumulated as weighted offsets from the box's geometric
// centre so that single precision keeps them accurate (with frames, the
// centre in the box's network's own frame: box_axis).  A leaf's lanes take its
// points, an inner box's lanes its children (at most 8).  A fixed butterfly
// (lane distances 16, 8, 4, 2, 1) sums the lanes: the vacant elements by the
// warp's integer reduction, the six offset sums by halving what a lane keeps
// while it halves the lanes (8 shuffles instead of 30), which leaves each sum in
// a lane of its own, where it is divided by its weight.  The order of every sum
// is fixed whichever warp computes a box, so the results are those of a
// level-by-level pass.  The counters are zero on entry (cleared by the build
// before an eager build and whenever their buffer is new; every complete launch
// leaves them zero).
//
// Bound by the chain of arrivals (a release each) and instruction issue.
// Serialised, cold: 1,000,000 neurons 47 -> 41 us with the halving butterfly and
// leaf_of kept, 65,536 in leaves of at most 8: 61 -> 50 us.
struct AggArgs {
    int frame_level;
    float ox, oy, oz, side;
    const float4* pts;
    const uint8_t* level;
    const uint64_t* prefix;
    const int32_t *first, *count, *parent, *child_first;
    const uint8_t* nchild;
    int4* sums;
    float4 *ca, *cd;
    int32_t* leaf_of;            // null: as they are (octree kept)
    int32_t* arrive;
};

// cf: the box's first child (-1: a leaf), nc: its children
__device__ __forceinline__ void aggregate_box(const AggArgs& a, int64_t i, int32_t cf, int nc,
                                              int lane) {
    const uint64_t pre = a.prefix[i];
    const int lv = (int)a.level[i];
    const float bs = ldexpf(a.side, -lv);
    const float g[3] = {a.ox + ((float)box_axis(pre, 0, lv, a.frame_level) + 0.5f) * bs,
                        a.oy + ((float)box_axis(pre, 1, lv, a.frame_level) + 0.5f) * bs,
                        a.oz + ((float)box_axis(pre, 2, lv, a.frame_level) + 0.5f) * bs};
    int aE = 0, aI = 0, wE = 0, wI = 0;
    float sa[3] = {0.f, 0.f, 0.f}, sd[3] = {0.f, 0.f, 0.f};
    if (cf < 0) {
        const int32_t f = a.first[i], c = a.count[i];
        for (int32_t j = f + lane; j < f + c; j += 32) {
            const float4 p = a.pts[j];
            const uint32_t w = __float_as_uint(p.w);
            const int ax = (int)pk_axon(w), de = (int)pk_de(w), di = (int)pk_di(w);
            if (pk_type(w)) aI += ax; else aE += ax;
            wE += de;
            wI += di;
            const float fa = (float)ax, fd = (float)(de + di);
            const float dx = p.x - g[0], dy = p.y - g[1], dz = p.z - g[2];
            sa[0] = fmaf(fa, dx, sa[0]); sa[1] = fmaf(fa, dy, sa[1]); sa[2] = fmaf(fa, dz, sa[2]);
            sd[0] = fmaf(fd, dx, sd[0]); sd[1] = fmaf(fd, dy, sd[1]); sd[2] = fmaf(fd, dz, sd[2]);
            if (a.leaf_of) a.leaf_of[j] = (int32_t)i;
        }
    } else if (lane < nc) {
        // the children were written by other warps: read them from L2
        const int4 sm = __ldcg(&a.sums[cf + lane]);
        const float4 a4 = __ldcg(&a.ca[cf + lane]), d4 = __ldcg(&a.cd[cf + lane]);
        aE = sm.x; aI = sm.y; wE = sm.z; wI = sm.w;
        const float fa = (float)(sm.x + sm.y), fd = (float)(sm.z + sm.w);
        sa[0] = fa * (a4.x - g[0]); sa[1] = fa * (a4.y - g[1]); sa[2] = fa * (a4.z - g[2]);
        sd[0] = fd * (d4.x - g[0]); sd[1] = fd * (d4.y - g[1]); sd[2] = fd * (d4.z - g[2]);
    }
    aE = __reduce_add_sync(0xffffffffu, aE);
    aI = __reduce_add_sync(0xffffffffu, aI);
    wE = __reduce_add_sync(0xffffffffu, wE);
    wI = __reduce_add_sync(0xffffffffu, wI);
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
    float v[3];                       // lanes 0-15: axons, 16-31: dendrites
#pragma unroll
    for (int d = 0; d < 3; ++d)
        v[d] = (h16 ? sd[d] : sa[d]) + __shfl_xor_sync(0xffffffffu, h16 ? sa[d] : sd[d], 16);
    const float u0 = (h8 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h8 ? v[0] : v[2], 8);
    const float u1 = v[1] + __shfl_xor_sync(0xffffffffu, v[1], 8);
    const bool one = !h8 && h4;       // axis 0: neither half, 1: h4, 2: h8
    float x = (one ? u1 : u0) + __shfl_xor_sync(0xffffffffu, h8 || h4 ? u0 : u1, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    // lanes 0, 4, 8 (16, 20, 24): the axes; lanes 12, 28: the weights; lane 1: sums
    if ((lane & 3) == 0) {
        const int q = (lane >> 2) & 3;
        const float t = (float)(h16 ? wE + wI : aE + aI);
        const float gq = q == 0 ? g[0] : (q == 1 ? g[1] : g[2]);
        float* out = reinterpret_cast<float*>(h16 ? a.cd + i : a.ca + i);
        out[q] = q == 3 ? (t > 0.f ? t : 0.f) : (t > 0.f ? gq + x / t : gq);
    } else if (lane == 1) {
        a.sums[i] = make_int4(aE, aI, wE, wI);
    }
}

// arrival at a parent: release for the box's own results, acquire for its
// siblings' (the last arrival reads them)
__device__ __forceinline__ int arrive_acq_rel(int32_t* p) {
    int old;
    asm volatile("atom.add.acq_rel.gpu.s32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
    return old;
}

// nodes_end: the node count (device memory); one warp per leaf
__global__ void k_aggregate_tree(const BuildEnd end, const int64_t* __restrict__ nodes_end,
                                 const AggArgs a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) end();
    const int64_t nn = *nodes_end;
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < nn; k += nw) {
        if (a.child_first[k] >= 0) continue;      // inner boxes: done by their last child's warp
        int64_t i = k;
        int32_t cf = -1, p = a.parent[k];
        int nc = 0;
        for (;;) {
            // the parent's place in the octree, read while the box is summed
            int32_t pcf = 0, pp = -1;
            int pnc = 0;
            if (p >= 0) {
                pcf = a.child_first[p];
                pnc = (int)a.nchild[p];
                pp = a.parent[p];
            }
            aggregate_box(a, i, cf, nc, lane);
            if (p < 0) break;
            __syncwarp();                         // the lanes' writes before the arrival
            int last = 0;
            if (lane == 0) {
                last = arrive_acq_rel(&a.arrive[p]) == pnc - 1;
                if (last) a.arrive[p] = 0;
            }
            last = __shfl_sync(0xffffffffu, last, 0);
            if (!last) break;
            __syncwarp();                         // the lanes' reads after lane 0's acquire
            i = p;
            cf = pcf;
            nc = pnc;
            p = pp;
        }
    }
}

// A warp per node, handed out by the hardware as warps finish, at most per_sm
// blocks per SM: 64 where the number of nodes is known (two replayed steps of
// 1,000,000 neurons 4633 us with 16, 4565 with 64), 16 where `nodes` is a bound far
// above it and most blocks would only leave.
int agg_grid(int64_t nodes, int64_t sm_count, int per_sm) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((nodes + 3) / 4, sm_count * per_sm));
}

}  // namespace

void build_tree(msp_ctx& c, int64_t n, const float* x, const float* y, const float* z,
                const uint8_t* type, const uint8_t* va, const uint8_t* vde, const uint8_t* vdi,
                cudaStream_t s, const CountCopy* copy) {
    NvtxRange nv_("msp build_tree");
    const bool was_built = c.tree_built, prev_kept = c.tree_reused;
    const int64_t prev_n = c.n;
    if (!c.graph_mode) {
        c.tree_built = false;
        c.attraction_done = false;
        c.tree_reused = false;
    }
    c.n = n;
    const msp_config& cfg = c.cfg;
    DevCounts* dc = dcounts(c);
    size_t nn = (size_t)(n > 0 ? n : 1);
    uint64_t* k0 = c.keys0.ensure<uint64_t>(nn);
    uint64_t* k1 = c.keys1.ensure<uint64_t>(nn);
    int32_t* v0 = c.vals0.ensure<int32_t>(nn);
    int32_t* v1 = c.vals1.ensure<int32_t>(nn);
    int32_t* perm = c.perm.ensure<int32_t>(nn);
    float4* pts = c.pts.ensure<float4>(nn);
    float2* wts = c.wts.ensure<float2>(nn);
    float2* lw = c.lw.ensure<float2>(nn);
    int32_t* eoff = c.elem_off.ensure<int32_t>(nn + 1);
    int32_t* leaf_of = c.leaf_of.ensure<int32_t>(nn);
    int32_t* cells = c.top_cells.ensure<int32_t>(kTopCells + 1);
    const int B = 256;
    const int G = grid_for(n, B, (int64_t)c.sm_count * 16);
    // box centres: in the domain's frame, or (frames) in each network's own
    const bool framed = c.frame_level > 0;
    const float o3[3] = {framed ? 0.f : cfg.origin[0], framed ? 0.f : cfg.origin[1],
                         framed ? 0.f : cfg.origin[2]};
    if (framed && n != c.frame_off_host.back())
        throw Error(MSP_ERR_INVALID_ARG, "the frames (msp_set_frames) hold a different number "
                                         "of neurons");
    auto agg_args = [&](int32_t* lo) {
        return AggArgs{c.frame_level, o3[0], o3[1], o3[2], cfg.side, pts,
                       c.nd_level.get<uint8_t>(), c.nd_prefix.get<uint64_t>(),
                       c.nd_first.get<int32_t>(), c.nd_count.get<int32_t>(),
                       c.nd_parent.get<int32_t>(), c.nd_child_first.get<int32_t>(),
                       c.nd_nchild.get<uint8_t>(), c.nd_sums.get<int4>(), c.nd_ca.get<float4>(),
                       c.nd_cd.get<float4>(), lo, c.nd_arrive.get<int32_t>()};
    };
    unsigned long long* scan_st = scan_status(c, n);
    const int64_t n_scan_st = scan_status_words(n);

    // An eager build on the positions of the last build keeps its sorted order
    // and octree, which depend on the positions only: their checksum tells.
    // After a build that kept them the next one is expected to as well and goes
    // ahead, its checksum read with its counts (a step of 4,096 neurons spends
    // 20 us on a second synchronisation); otherwise the checksum is read first.
    // Positions that move right after a kept build cost that expectation once: the
    // counts and aggregates of the old octree and a synchronisation (4,096 neurons
    // 159 -> 175 us a build, 1,048,576 457 -> 522; a kept build is 45 and 104).
    // Inside the whole-step graph the positions are those of the last eager
    // build, or the graph halts.  A full-build replay may have built another
    // octree since: the arrays' generation stamp tells.
    auto kept = [&] {
        return c.hcount->pos_sum == c.pos_sum_ref && c.hcount->tree_gen == c.tree_gen;
    };
    const bool may_keep = !c.graph_mode && was_built && n == prev_n && n > 0;
    const bool graph_keep = c.graph_mode && c.tree_built && !c.graph_full_build;
    const bool expect = may_keep && prev_kept;
    const int64_t n_arrive = may_keep ? (int64_t)(c.nd_arrive.bytes / sizeof(int32_t)) : 0;
    k_build_init<<<grid_for(std::max({n_scan_st, n_arrive, copy ? n / 8 : 0}), B,
                            (int64_t)c.sm_count * 2), B, 0, s>>>(
        dc, n, scan_st, n_scan_st, c.nd_arrive.get<int32_t>(), n_arrive, copy ? *copy : CountCopy{});
    MSP_LAUNCH("build_init");
    bool keep = graph_keep || expect;
    const BuildEnd end{dc, c.graph_mode, graph_keep, c.pos_sum_ref, c.tree_gen, c.graph_elem_cap};
    if (!keep && n > 0 && !c.graph_mode) {
        k_pos_sum<<<G, B, 0, s>>>(x, y, z, n, reinterpret_cast<unsigned long long*>(&dc->pos_sum));
        MSP_LAUNCH("pos_sum");
        if (may_keep) {
            MSP_CUDA(cudaMemcpyAsync(&c.hcount->pos_sum, &dc->pos_sum, 2 * sizeof(uint64_t),
                                     cudaMemcpyDeviceToHost, s));   // and tree_gen
            MSP_CUDA(cudaStreamSynchronize(s));
            keep = kept();
            if (keep) MSP_CUDA(cudaMemsetAsync(&dc->pos_sum, 0, sizeof(uint64_t), s));
        }
    }

    // the octree kept: the counts are gathered again and the aggregates recomputed
    if (keep) {
        if (n > 0) {
            k_gather_counts<<<G, B, 0, s>>>(n, x, y, z, type, va, vde, vdi, perm, pts, wts, lw,
                                            reinterpret_cast<unsigned long long*>(&dc->pos_sum));
            MSP_LAUNCH("gather_counts");
            scan_launch(c, ScanU8{va}, ScanStore{eoff}, ScanTotalAfter{&dc->n_elem, eoff, &dc->n},
                        &dc->n, n, s, scan_st);
        } else {
            dev_set(&dc->n_elem, 0, s);
        }
        k_aggregate_tree<<<agg_grid(c.n_nodes, c.sm_count, 64), 128, 0, s>>>(
            end, &dc->level_start[c.tree_levels + 1], agg_args(nullptr));
        MSP_LAUNCH("aggregate");
        if (c.graph_mode) return;
        pull_counts(c, s);              // the one synchronisation of the build
        if (kept()) {
            c.n_elem = c.hcount->n_elem;
            c.tree_built = true;
            c.tree_reused = true;
            return;
        }
        // the positions changed after all (dc->pos_sum is their checksum)
    }
    // every eager build that gets here has a stamp of its own, a replay one that
    // no capture and no eager build holds
    const uint64_t stamp = c.graph_mode ? ~0ull : ++c.tree_gen;
    if (!c.graph_mode) c.lists_valid = false;

    // a1 + a2: keys, stable sort, gather into Morton order
    if (n > 0) {
        const bool odd = radix_from_tmp(n, 3 * kMortonBits);
        uint64_t* mk = odd ? k1 : k0;
        int32_t* mv = odd ? v1 : v0;
        if (framed) {
            k_morton_frames<<<G, B, 0, s>>>(x, y, z, n, c.frame_off.get<int64_t>(),
                                            (int64_t)c.frame_off_host.size() - 1, c.frame_level,
                                            ldexpf(cfg.side, -c.frame_level), c.morton_scale, mk,
                                            mv, dc, stamp);
            MSP_LAUNCH("morton_frames");
        } else {
            k_morton<<<G, B, 0, s>>>(x, y, z, n, cfg.origin[0], cfg.origin[1], cfg.origin[2],
                                     cfg.side, c.morton_scale, mk, mv, dc, stamp);
            MSP_LAUNCH("morton");
        }
        radix_sort_dev(c, k0, v0, k1, v1, nullptr, n, 3 * kMortonBits, s);
        k_gather<<<G, B, 0, s>>>(v0, n, x, y, z, type, va, vde, vdi, perm, pts, wts, lw, k0, cells);
        MSP_LAUNCH("gather");
        // element offsets: exclusive prefix of the vacant axonal counts
        scan_launch(c, ScanU8{va}, ScanStore{eoff}, ScanTotalAfter{&dc->n_elem, eoff, &dc->n},
                    &dc->n, n, s, keep ? nullptr : scan_st);
    } else {
        dev_set(&dc->n_elem, 0, s);
        dev_set(reinterpret_cast<int64_t*>(&dc->tree_gen), (int64_t)stamp, s);
    }

    // a3: level-synchronous octree; the level sizes stay in device memory.
    // Levels are built down to the previous tree's depth + 1 (a first guess
    // from n and the leaf capacity otherwise); if a box of the last built level
    // would still split, the tree is rebuilt with all levels.
    int L = c.depth_hint;
    if (L < 0) {
        L = 3;
        for (int64_t m = std::max<int64_t>(n / std::max(cfg.leaf_capacity, 1), 1); m > 1; m >>= 3) ++L;
    } else {
        L += 1;
    }
    L = std::min(std::max(L, 0), cfg.max_depth);
    const int Gt = (int)std::max<int64_t>(1, (int64_t)c.sm_count * 8);
    int min_cap = cfg.leaf_capacity;
    if (framed && c.frame_plans)
        for (int32_t v : c.frame_cap_host) min_cap = std::min(min_cap, (int)v);
    // scratch of later steps (msp_direct's lists among them), sized here
    c.cnt.ensure<int32_t>(nn + 8);
    c.off.ensure<int32_t>(nn + 8);
    // boxes at level l: at most min(8^l, n), and (l >= 1) at most 8 children
    // of each box of level l-1 that splits, i.e. holds more than C neurons
    const int64_t splitters = (int64_t)nn / ((int64_t)min_cap + 1);
    auto level_cap = [&](int l) -> int64_t {
        int64_t c = l < 8 ? std::min<int64_t>((int64_t)1 << (3 * l), (int64_t)nn) : (int64_t)nn;
        if (l >= 1) c = std::min<int64_t>(c, 8 * splitters);
        return std::max<int64_t>(c, 1);
    };
    for (;;) {
        int64_t cap = 0;
        for (int l = 0; l <= L; ++l) cap += level_cap(l);
        cap += 8;
        c.nd_level.ensure<uint8_t>((size_t)cap);
        c.nd_prefix.ensure<uint64_t>((size_t)cap);
        c.nd_first.ensure<int32_t>((size_t)cap);
        c.nd_count.ensure<int32_t>((size_t)cap);
        c.nd_parent.ensure<int32_t>((size_t)cap);
        c.nd_child_first.ensure<int32_t>((size_t)cap);
        c.nd_nchild.ensure<uint8_t>((size_t)cap);
        c.nd_sums.ensure<int4>((size_t)cap);
        c.nd_ca.ensure<float4>((size_t)cap);
        c.nd_cd.ensure<float4>((size_t)cap);
        // the arrival counters: cleared before an eager build and whenever
        // the buffer is new (a graph's dry run may build one level deeper than
        // the eager build and grow it); a replay finds them as the last
        // complete launch left them, zero
        const size_t arrive_bytes = c.nd_arrive.bytes;
        int32_t* arrive = c.nd_arrive.ensure<int32_t>((size_t)cap);
        if (!c.graph_mode || c.nd_arrive.bytes != arrive_bytes)
            MSP_CUDA(cudaMemsetAsync(arrive, 0, c.nd_arrive.bytes, s));
        LevelArgs la;
        la.n = n;
        la.keys = k0;
        la.level = c.nd_level.get<uint8_t>();
        la.prefix = c.nd_prefix.get<uint64_t>();
        la.first = c.nd_first.get<int32_t>();
        la.count = c.nd_count.get<int32_t>();
        la.parent = c.nd_parent.get<int32_t>();
        la.child_first = c.nd_child_first.get<int32_t>();
        la.nchild = c.nd_nchild.get<uint8_t>();
        la.leaf_capacity = cfg.leaf_capacity;
        la.max_depth = cfg.max_depth;
        la.cap = framed && c.frame_plans ? c.frame_cap.get<int32_t>() : nullptr;
        la.frame_level = c.frame_level;
        la.nf = (int64_t)c.frame_off_host.size() - 1;
        la.node_cap = cap;
        // the top levels in one block, then a launch per level; per level a
        // tile counter and one status word per tile, cleared together
        const int top = std::min(L, kTopLevels);
        auto words = [&](int l) { return 1 + (level_cap(l) + kLevelTile - 1) / kLevelTile; };
        int64_t nw = 0;
        for (int l = top; l < L; ++l) nw += words(l);
        unsigned long long* st = c.lv_status.ensure<unsigned long long>((size_t)std::max<int64_t>(nw, 1));
        if (nw > 0) MSP_CUDA(cudaMemsetAsync(st, 0, (size_t)nw * sizeof(unsigned long long), s));
        k_tree_top<<<1, 1024, 0, s>>>(la, top, cells, dc);
        MSP_LAUNCH("tree_top");
        for (int l = top; l < L; ++l) {
            const int64_t tiles = words(l) - 1;
            k_tree_level<false><<<(unsigned)std::min<int64_t>(tiles, (int64_t)c.sm_count * 4), 256, 0,
                                  s>>>(la, l, dc, st, kScanTimeoutBit);
            MSP_LAUNCH("tree_level");
            st += words(l);
        }
        // would a box of the last built level still split?
        if (L < cfg.max_depth) {
            k_tree_level<true><<<grid_for(level_cap(L), 256, Gt), 256, 0, s>>>(la, L, dc, nullptr, 0);
            MSP_LAUNCH("tree_more");
        }
        // a4: aggregates, leaves up to the root in one launch
        k_aggregate_tree<<<agg_grid(cap, c.sm_count, 16), 128, 0, s>>>(
            end, &dc->level_start[L + 1], agg_args(leaf_of));
        MSP_LAUNCH("aggregate");
        // inside the whole-step graph the tree of the same positions has the
        // same levels; a deeper one sets more_levels, which halts the graph
        if (c.graph_mode) return;
        pull_counts(c, s);          // the one synchronisation of the build
        if (c.hcount->bad_pos)
            throw Error(MSP_ERR_INVALID_ARG,
                        framed ? "a position is outside its frame's cell [0, side / 2^level) "
                                 "or not finite"
                               : "a position is outside [origin, origin + side) or not finite");
        if (c.hcount->overflow & 16) throw Error(MSP_ERR_CHECK, "octree node capacity exceeded");
        if (c.hcount->more_levels > 0 && L < cfg.max_depth) {
            L = cfg.max_depth;
            continue;
        }
        break;
    }
    const DevCounts& hc = *c.hcount;
    int depth = 0;
    for (int l = 1; l <= L; ++l)
        if (hc.level_start[l + 1] > hc.level_start[l]) depth = l;
    c.level_start.assign(hc.level_start, hc.level_start + depth + 2);
    c.n_nodes = hc.level_start[depth + 1];
    c.tree_depth = depth;
    c.depth_hint = depth;
    c.n_elem = hc.n_elem;
    c.tree_levels = L;
    c.pos_sum_ref = hc.pos_sum;
    c.tree_built = true;
}

}  // namespace msp
