// msp_select.cu -- steps a11-a12: the level-synchronous descent of
// Algorithm 1 with Algorithm 2's choice (candidate attractions, total, uniform
// draw, upper_bound over the inclusive prefix sums), the per-element draw of a
// dendrite neuron inside the chosen leaf, and the resolution of the requests
// at the dendrite side (Section 4).  Also the vacancy random walk and the
// consumption of formed synapses.
#include <algorithm>

#include "msp_scan.cuh"

namespace msp {

__device__ inline float ex2_approx_sel(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__constant__ float c_inv_fact_sel[kMaxP] = {1.f, 1.f, 0.5f, 1.f / 6.f, 1.f / 24.f, 1.f / 120.f,
                                            1.f / 720.f, 1.f / 5040.f};

namespace {

struct Tree {
    const uint8_t* level;
    const int32_t* first;
    const int32_t* count;
    const int32_t* child_first;
    const uint8_t* nchild;
    const int4* sums;
    const float4* ca;
    const float4* cd;
};

struct Exps {
    const float* A;
    const float* M;
    int64_t first;
    int p;
    float inv_sigma;
};

// W(X, Y) of one channel from the expansions (pairs below a translated
// pair): M2L of A(Y) about c_A(X), dotted with the axon moments M(X).  Whole
// warp; the result is returned to every lane.
__device__ float warp_far_w(const Tree& tr, const Exps& ex, int32_t X, int32_t Y, int ch,
                            float* H, float* b0, float* b1) {
    const int lane = threadIdx.x & 31;
    const int p = ex.p, p2 = p * p, p3 = p2 * p;
    if (X < ex.first || Y < ex.first) return 0.f;
    float4 a = tr.ca[X], d = tr.cd[Y];
    if (lane < 3) {
        float x = (lane == 0 ? a.x - d.x : (lane == 1 ? a.y - d.y : a.z - d.z)) * ex.inv_sigma;
        float* h = H + 16 * lane;
        float h0 = __expf(-x * x);
        h[0] = h0;
        if (2 * p - 2 >= 1) h[1] = 2.f * x * h0;
        for (int k = 1; k < 2 * p - 2; ++k) h[k + 1] = 2.f * x * h[k] - 2.f * (float)k * h[k - 1];
    }
    const float* Ag = ex.A + (int64_t)(Y - ex.first) * p3 * 2 + ch;
    const float* Mg = ex.M + ((int64_t)(X - ex.first) * 2 + ch) * p3;
    for (int i = lane; i < p3; i += 32) b0[i] = Ag[2 * i];
    __syncwarp();
    for (int o = lane; o < p3; o += 32) {
        int c0 = o / p2, r = o - c0 * p2;
        float s = 0.f;
        for (int k = 0; k < p; ++k) s = fmaf(H[k + c0], b0[k * p2 + r], s);
        b1[o] = s;
    }
    __syncwarp();
    for (int o = lane; o < p3; o += 32) {
        int c0 = o / p2, c1 = (o / p) % p, k2 = o % p;
        float s = 0.f;
        for (int k = 0; k < p; ++k) s = fmaf(H[16 + k + c1], b1[c0 * p2 + k * p + k2], s);
        b0[o] = s;
    }
    __syncwarp();
    float w = 0.f;
    for (int o = lane; o < p3; o += 32) {
        int c0 = o / p2, c1 = (o / p) % p, c2 = o % p;
        float s = 0.f;
        for (int k = 0; k < p; ++k) s = fmaf(H[32 + k + c2], b0[c0 * p2 + c1 * p + k], s);
        float sc = c_inv_fact_sel[c0] * c_inv_fact_sel[c1] * c_inv_fact_sel[c2];
        if ((c0 + c1 + c2) & 1) sc = -sc;
        w = fmaf(s * sc, Mg[o], w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    __syncwarp();
    return w;
}

// Algorithm 2's last steps: negative candidates (truncation) count as zero;
// -1 when the total is at most kMinAttraction; upper_bound over the inclusive
// prefix sums, and the last positive candidate when rounding puts r at the
// total.  The candidates, their prefix sums and r = U * total are double-FP32
// values (hi + lo; the sign of a value is that of hi).
// (All loops have the constant bound of 8 candidates, so nothing is indexed at run
// time and the candidates stay in registers.)
__device__ __forceinline__ int draw_index(const float2 (&w)[8], int k, uint64_t bits53) {
    float2 pre[8];
    float2 tot = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (i < k) tot = ff_add(tot, w[i].x > 0.f ? w[i] : make_float2(0.f, 0.f));
        pre[i] = tot;
    }
    if (!(tot.x > kMinAttractionF)) return -1;
    const float2 r = ff_mul(ff_uniform(bits53), tot);
    int at = -1, last = -1;
#pragma unroll
    for (int i = 7; i >= 0; --i) {
        if (i < k && ff_gt(pre[i], r)) at = i;
        if (i < k && last < 0 && w[i].x > 0.f) last = i;
    }
    return at >= 0 ? at : last;
}

constexpr int kDescWarps = 4;

// The item counts of the steps rotate through DevCounts::items: step k reads its
// input count from slot k % 3, appends to the next (zeroed by the step before) and
// zeroes the third for the step after.

// Start of a selection: by one thread the counters and the items of both channels
// at (root, root), where the root has vacancies and attraction in that channel; no
// partner and nothing accepted yet, empty request groups (ng > 0: unless the last
// selection left them empty), the status words of its scans.  One launch instead
// of two and four clears (a clear of 2 us each and a gap: a selection of 4,096
// neurons is bound by its launches).
__global__ void k_select_init(const int4* __restrict__ sums, const float4* __restrict__ pw,
                              Item* __restrict__ items, DevCounts* dc, int64_t n,
                              int32_t* __restrict__ partner, uint8_t* __restrict__ acc,
                              int32_t* __restrict__ gcnt, int64_t ng,
                              unsigned long long* __restrict__ status, int64_t n_status) {
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (i0 == 0) {
        const int4 rs = sums[0];
        const float4 rw = pw[0];
        int64_t k = 0;
        if (rs.x > 0 && rw.x > kMinAttractionF) items[k++] = Item{0, 0, 0, 0};
        if (rs.y > 0 && rw.z > kMinAttractionF) items[k++] = Item{0, 0, 0, 1};
        dc->items[0] = k;
        dc->items[1] = 0;
        dc->n_leaf = 0;
        dc->leaf_next = 0;
        dc->draws = 0;
        dc->n_groups = 2 * n;
        dc->overflow &= ~38ll;      // the selection's bits; bit 0 (pair table) stays
    }
    const int64_t ne = dc->n_elem;
    for (int64_t i = i0; i < ne; i += stride) {
        partner[i] = -1;
        acc[i] = 0;
    }
    for (int64_t i = i0; i < ng; i += stride) gcnt[i] = 0;
    for (int64_t i = i0; i < n_status; i += stride) status[i] = 0;
}

// appends v of the lanes with `has` to list (one atomic per warp)
__device__ __forceinline__ void append_items(bool has, const Item& v, unsigned long long* n,
                                             Item* list, int64_t cap, unsigned long long* overflow,
                                             unsigned long long bit) {
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(n, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (!has) return;
    const int64_t slot = (int64_t)base + __popc(m & ((1u << lane) - 1u));
    if (slot < cap) list[slot] = v;
    else atomicOr(overflow, bit);
}

struct DescArgs {
    Tree tr;
    Exps ex;
    const uint8_t* kind;
    const int32_t* pcf;
    const float2* pw;            // pair q: E at 2 q, I at 2 q + 1 (hi, lo)
    uint64_t seed;
    StepRef stp;
    Item* items[2];              // step k reads items[k & 1]
    int64_t cap_out;
    Item* leaf_out;
    int64_t cap_leaf;
    DevCounts* dc;
};
// floats of shared memory per warp: Hermite functions and two sets of coefficients
__host__ __device__ constexpr int desc_warp_floats(int p) { return 48 + 2 * p * p * p; }

// One level step of the descent by `nwarp` warps, this one `warp`.  A warp takes
// four items, 8 lanes each (lane i of a group for the item's axon child i): a
// leaf pair goes to the per-element draw; a dendrite leaf is kept by every axon
// child with vacancies; otherwise each axon child draws among the children of Y
// from the pair table.  Items below a translated pair (candidates' attractions
// evaluated as translations by the whole warp) follow, one at a time.  Bound by
// the chain of dependent reads (item, boxes, candidates) of the few items of a
// step; everything that does not depend on the one before is read together.
__device__ __forceinline__ void descend_step(const DescArgs& a, int step_k, int64_t warp,
                                             int64_t nwarp, float* sm) {
    const Tree& tr = a.tr;
    const uint64_t step = a.stp.get();
    const int lane = threadIdx.x & 31;
    const int sub = lane & 7;
    DevCounts* dc = a.dc;
    auto ull = [](int64_t* p) { return reinterpret_cast<unsigned long long*>(p); };
    unsigned long long *n_out = ull(&dc->items[(step_k + 1) % 3]), *n_leaf = ull(&dc->n_leaf),
                       *overflow = ull(&dc->overflow);
    const Item* in = a.items[step_k & 1];
    Item* out = a.items[(step_k + 1) & 1];
    // the count may exceed the buffer (items past it were not stored and the
    // overflow bit is set)
    const int64_t n_in = min(__ldcg(&dc->items[step_k % 3]), a.cap_out);
    if (warp == 0 && lane == 0) dc->items[(step_k + 2) % 3] = 0;
    for (int64_t k0 = 4 * warp; k0 < n_in; k0 += 4 * nwarp) {
        const int64_t k = k0 + (lane >> 3);
        Item it = {0, 0, -1, 0}, nx = {0, 0, -1, 0};
        bool far_item = false, drew = false, leaf_pair = false, keep = false;
        if (k < n_in) {
            const int4 raw = __ldcg(reinterpret_cast<const int4*>(in) + k);
            it = Item{raw.x, raw.y, raw.z, raw.w};
            const int32_t X = it.X, Y = it.Y;
            const int ch = it.ch;
            const int32_t cx = tr.child_first[X], cy = tr.child_first[Y];
            const int nx_ch = tr.nchild[X], ny = tr.nchild[Y];
            const uint32_t ly1 = (uint32_t)tr.level[Y] + 1u;
            const int kd = it.q >= 0 ? a.kind[it.q] : (int)kPruned;
            const int32_t cfq = it.q >= 0 ? a.pcf[it.q] : -1;
            const bool lx = cx < 0, ly = cy < 0;
            const bool split = kd == kSplit;
            const int32_t cf = split ? cfq : -1;
            // a split pair whose children did not fit in the pair table (the
            // step is halted and redone with a larger table): nothing to read
            if (split && cf < 0) {
            } else if (lx && ly) {
                // form_synapse: the leaf pair goes to the per-element draw
                leaf_pair = sub == 0;
            } else if (!lx && ly) {
                // the dendrite side is a leaf: every axon child with vacancies
                // of this channel keeps it, without a draw
                if (sub < nx_ch) {
                    const int4 sc = tr.sums[cx + sub];
                    keep = (ch ? sc.y : sc.x) > 0;
                    if (split) keep = a.pw[2 * (int64_t)(cf + sub) + ch].x > kMinAttractionF && keep;
                    nx = Item{cx + sub, Y, split ? cf + sub : -1, ch};
                }
            } else if (split) {
                // a draw among the children of Y, for X itself (X a leaf) or
                // for each axon child of X (both inner); the candidates'
                // attractions are in the pair table
                if (sub < (lx ? 1 : nx_ch)) {
                    const int32_t xc = lx ? X : cx + sub;
                    const int4 sc = tr.sums[xc];
                    const int64_t c0 = cf + (int64_t)sub * ny;
                    float2 wk[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        wk[j] = j < ny ? a.pw[2 * (c0 + j) + ch] : make_float2(0.f, 0.f);
                    if (lx || (ch ? sc.y : sc.x) != 0) {
                        const uint32_t c1 = ly1 | ((uint32_t)ch << 8) | (kTagDescend << 16);
                        const int kk =
                            draw_index(wk, ny, philox_bits53(a.seed, (uint32_t)xc, c1, step));
                        drew = true;
                        keep = kk >= 0;
                        nx = Item{xc, cy + kk, (int32_t)(c0 + kk), ch};
                    }
                }
            } else {
                far_item = true;
            }
        }
        append_items(leaf_pair, it, n_leaf, a.leaf_out, a.cap_leaf, overflow, 4ull);
        append_items(keep, nx, n_out, out, a.cap_out, overflow, 2ull);
        const unsigned dm = __ballot_sync(0xffffffffu, drew);
        if (lane == 0 && dm) atomicAdd(ull(&dc->draws), (unsigned long long)__popc(dm));
        // below a translated pair: each candidate's attraction is a
        // translation the whole warp evaluates
        unsigned fm = __ballot_sync(0xffffffffu, far_item && sub == 0);
        while (fm) {
            const int src = __ffs(fm) - 1;
            fm &= fm - 1;
            const int32_t X = __shfl_sync(0xffffffffu, it.X, src);
            const int32_t Y = __shfl_sync(0xffffffffu, it.Y, src);
            const int ch = __shfl_sync(0xffffffffu, it.ch, src);
            const bool lx = tr.child_first[X] < 0;
            const int ny = tr.nchild[Y];
            const int32_t cy = tr.child_first[Y];
            const int nsrc = lx ? 1 : tr.nchild[X];
            for (int i = 0; i < nsrc; ++i) {
                const int32_t xc = lx ? X : tr.child_first[X] + i;
                if (!lx) {
                    const int4 sc = tr.sums[xc];
                    if ((ch ? sc.y : sc.x) == 0) continue;
                }
                float mine = 0.f;            // lane j: candidate j
                for (int j = 0; j < ny; ++j) {
                    const float v = warp_far_w(tr, a.ex, xc, cy + j, ch, sm, sm + 48,
                                               sm + 48 + a.ex.p * a.ex.p * a.ex.p);
                    if (lane == j) mine = v;
                }
                float2 wk[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    wk[j] = make_float2(__shfl_sync(0xffffffffu, mine, j), 0.f);
                if (lane == 0) {
                    const uint32_t c1 = (uint32_t)(tr.level[Y] + 1) | ((uint32_t)ch << 8) |
                                        (kTagDescend << 16);
                    const int kk = draw_index(wk, ny, philox_bits53(a.seed, (uint32_t)xc, c1, step));
                    atomicAdd(ull(&dc->draws), 1ull);
                    if (kk >= 0) {
                        const unsigned long long slot = atomicAdd(n_out, 1ull);
                        const Item far_nx = {xc, cy + kk, -1, ch};
                        if ((int64_t)slot < a.cap_out) out[slot] = far_nx;
                        else atomicOr(overflow, 2ull);
                    }
                }
                __syncwarp();
            }
        }
    }
}

// The first steps in one block: the items of a step are distinct (X, channel)
// with disjoint boxes X no deeper than the step, so at most 2 * 8^k, one round of
// 32 warps up to step 2.
constexpr int kDescTop = 3, kDescTopWarps = 32;
__global__ void __launch_bounds__(kDescTopWarps * 32) k_descend_top(const DescArgs a, int steps) {
    extern __shared__ float s_desc[];
    const int w = threadIdx.x >> 5;
    for (int k = 0; k < steps; ++k) {
        descend_step(a, k, w, kDescTopWarps, s_desc + w * desc_warp_floats(a.ex.p));
        __syncthreads();
    }
}

// Then a launch per step, with as many blocks as the step may have items for.
// 1,000,000 neurons (serialised, cold): 82 us in eight launches whose candidates
// lay in local memory, 64 in six; 4,096 neurons 30 in four, 22 in two.
__global__ void __launch_bounds__(kDescWarps * 32, 8) k_descend(const DescArgs a, int step_k) {
    extern __shared__ float s_desc[];
    const int w = threadIdx.x >> 5;
    descend_step(a, step_k, (int64_t)blockIdx.x * kDescWarps + w, (int64_t)gridDim.x * kDescWarps,
                 s_desc + w * desc_warp_floats(a.ex.p));
}

// Per-element draw inside the chosen dendrite leaf, one warp per leaf pair
// (X, Y, channel), or per part of X's neurons where there are few leaf pairs,
// taken from a device work counter: the warp stages Y's points with their
// weights of the channel in shared memory and takes X's neurons of that
// channel with vacant axons up to 32 at a time.  Their weights w_s K(t,s) of
// the sources s != t of Y, truncated at the cutoff, are summed in exact 64-bit
// fixed point (scale 2^shift; a weight is at most 255: integer adds are exact
// and full rate, where double precision adds are scarce on this GPU; weights
// below 2^-shift, far below exp(-cutoff^2) for the cutoffs the library
// accepts, count as zero).  A lane sums a neuron's sources, or with at most 16
// neurons a slice of them, and keeps the prefix sums of kLdBlocks blocks.  The
// element draws r_e = floor(U_e tot) (U_e with 53 bits) are then handed out to
// the lanes evenly, whatever each neuron's number of elements: the slice and
// the block by the prefix sums, the source (the first one whose inclusive
// prefix exceeds r_e) by evaluating that one block again.
//
// Bound by instruction issue: about 17 instructions per weight.  Against a
// walk over blocks of 32 sources by each lane for its own neuron's elements
// (the warp waited for its slowest lane) and one warp for a leaf pair whatever
// their number (serialised, cold): 1,048,576 neurons 322 -> 155 us, 262,144 in
// clusters 305 -> 95, 21,013 (some 700 leaf pairs) 223 -> 30 us.
constexpr int kLdWarps = 4;
constexpr int kLdStage = 256;
constexpr int kLdBlocks = 16;              // prefix sums per lane

// weight of source j: the staged point {x, y, z, w} or, for leaves of more
// than kLdStage points, global memory
struct LdSrc {
    const float4* sp;
    const float4* pts;
    const float2* wts;
    int32_t sf;
    int ch;
    __device__ float4 get(int j) const {
        if (sp) return sp[j];
        const float4 S = pts[sf + j];
        return make_float4(S.x, S.y, S.z, ch ? wts[sf + j].y : wts[sf + j].x);
    }
};

// floor(v * 2^shift) for a finite 0 <= v < 2^8 (shift <= 40), exact, from the
// bits of v on the integer pipe (a float to 64-bit integer conversion runs on
// the FP64 unit, which is scarce on this GPU): the mantissa at the place of
// the largest exponent, 2^47, shifted down by what the exponent lacks; v = 0
// (and anything below 2^-shift) shifts out
__device__ __forceinline__ uint64_t fixed_point(float v, int shift) {
    const uint32_t b = __float_as_uint(v);
    const uint32_t m = (b & 0x7fffffu) | 0x800000u;
    const int s = min(174 - shift - (int)(b >> 23), 63);
    return ((uint64_t)m << 24) >> s;
}

// the weights of two sources at once (paired FP32: each element rounded as in
// the scalar form); a source at position self (relative to the leaf) is t
// itself
__device__ __forceinline__ void ld_weight2(const float4& T, const float4& S0, const float4& S1,
                                           float k2, float rc2, int shift, uint64_t& v0,
                                           uint64_t& v1) {
    const float2 dx = __fadd2_rn(make_float2(T.x, T.x), make_float2(-S0.x, -S1.x));
    const float2 dy = __fadd2_rn(make_float2(T.y, T.y), make_float2(-S0.y, -S1.y));
    const float2 dz = __fadd2_rn(make_float2(T.z, T.z), make_float2(-S0.z, -S1.z));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    const float2 e = __fmul2_rn(make_float2(-r2.x, -r2.y), make_float2(k2, k2));
    const float2 ws =
        __fmul2_rn(make_float2(S0.w, S1.w), make_float2(ex2_approx_sel(e.x), ex2_approx_sel(e.y)));
    v0 = fixed_point(r2.x < rc2 ? ws.x : 0.f, shift);
    v1 = fixed_point(r2.y < rc2 ? ws.y : 0.f, shift);
}

// per-network truncation radii (points in frames with per-network plans):
// the squared radius of the axon leaf's network
struct FrameRc2 {
    const float* rc2;          // per network, or null: the kernel's rc2 everywhere
    const uint64_t* prefix;
    const uint8_t* level;
    int frame_level;
    int64_t nf;
};

__global__ void __launch_bounds__(kLdWarps * 32)
k_leaf_draw_w(const Item* __restrict__ items, const int64_t* __restrict__ n_leaf, int64_t cap_leaf,
              unsigned long long* __restrict__ next, const int32_t* __restrict__ nfirst,
              const int32_t* __restrict__ ncount, const float4* __restrict__ pts,
              const float2* __restrict__ wts, const int32_t* __restrict__ perm,
              const int32_t* __restrict__ eoff, float k2, float rc2_all, FrameRc2 fr,
              uint64_t seed, StepRef stp,
              int32_t* __restrict__ partner, int32_t* __restrict__ gcnt, int64_t n,
              unsigned long long* __restrict__ draw_ctr, const int64_t* __restrict__ n_elem) {
    __shared__ float4 s_pts[kLdWarps][kLdStage];
    __shared__ uint64_t s_pre[kLdWarps][kLdBlocks][32];   // inclusive prefix per block and lane
    __shared__ float4 s_T[kLdWarps][32];                  // a round's neurons
    __shared__ int32_t s_tl[kLdWarps][32], s_a[kLdWarps][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t step = stp.get();
    const int64_t ne = *n_elem;
    const int64_t n_items = min(*n_leaf, cap_leaf);
    // parts per leaf pair: a few thousand units keep the chip's warps busy
    // (a leaf pair alone is one long chain)
    const int lgK = n_items >= 8192 ? 0 : (n_items >= 4096 ? 1 : (n_items >= 2048 ? 2 : 3));
    unsigned long long draws = 0;
    for (;;) {
        unsigned long long k = 0;
        if (lane == 0) k = atomicAdd(next, 1ull);
        k = __shfl_sync(0xffffffffu, k, 0);
        if ((int64_t)(k >> lgK) >= n_items) break;
        const Item it = items[k >> lgK];
        const int part = (int)(k & ((1u << lgK) - 1u));
        const int32_t tf = nfirst[it.X], tc = ncount[it.X];
        const int parts = min(1 << lgK, (tc + 47) / 48);
        if (part >= parts) continue;
        const int32_t tend = (int32_t)((int64_t)tc * (part + 1) / parts);
        int32_t pos = (int32_t)((int64_t)tc * part / parts);
        const int ch = it.ch;
        const float rc2 =
            fr.rc2 ? fr.rc2[box_frame(fr.prefix[it.X], fr.level[it.X], fr.frame_level, fr.nf)]
                   : rc2_all;
        const int32_t sf = nfirst[it.Y], sc = ncount[it.Y];
        const bool own = it.X == it.Y;         // a neuron may meet itself
        // fixed-point scale: sc weights of at most 2^8 must stay below 2^63
        int lg = 0;
        while ((1 << lg) < sc + 1 && lg < 30) ++lg;
        const int shift = min(40, 55 - lg);
        LdSrc src{nullptr, pts, wts, sf, ch};
        if (sc <= kLdStage) {
            __syncwarp();
            for (int j = lane; j < sc; j += 32) {
                const float4 S = pts[sf + j];
                s_pts[w][j] = make_float4(S.x, S.y, S.z, ch ? wts[sf + j].y : wts[sf + j].x);
            }
            __syncwarp();
            src.sp = s_pts[w];
        }
        while (pos < tend) {
            // up to 32 of X's neurons of the channel with vacant axons, from pos on
            int nt = 0;
            while (pos < tend && nt < 32) {
                const int32_t tt = tf + pos + lane;
                float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
                if (pos + lane < tend) P = pts[tt];
                const uint32_t tw = __float_as_uint(P.w);
                const bool mine =
                    pos + lane < tend && pk_axon(tw) > 0 && (pk_type(tw) ? 1 : 0) == ch;
                const unsigned mask = __ballot_sync(0xffffffffu, mine);
                const int room = 32 - nt, cnt = __popc(mask);
                const int take = min(cnt, room);
                const int rank = __popc(mask & ((1u << lane) - 1u));
                if (mine && rank < take) {
                    s_tl[w][nt + rank] = tt;
                    s_T[w][nt + rank] = P;
                }
                nt += take;
                if (take < cnt) {
                    // continue after the lane of the last target taken
                    pos += (int32_t)__fns(mask, 0, take) + 1;
                    break;
                }
                pos += 32;
            }
            __syncwarp();
            if (nt == 0) continue;
            // S lanes per target when the round has few targets (S = 32 / nt,
            // at most 8; TS = nt lanes per slice, the last 32 - S TS lanes idle):
            // lane = q * TS + ti takes target ti and slice q of the sources
            const int TS = nt <= 16 ? nt : 32;
            const int S = nt <= 16 ? min(8, 32 / TS) : 1;
            const int ti = lane % TS, q = lane / TS;
            const bool act = ti < nt && q < S;
            const int L = (sc + S - 1) / S;
            // blocks of bs sources (an even number), kLdBlocks per slice
            const int bs = max(2, ((L + kLdBlocks - 1) / kLdBlocks + 1) & ~1);
            const float4 T = s_T[w][act ? ti : 0];
            const int32_t t = s_tl[w][act ? ti : 0];
            const int j0 = min(q * L, sc), j1 = min(j0 + L, sc);
            // the slice's block sums (integer sums: exact, the same as one
            // walk over all sources)
            uint64_t part_sum = 0;
            if (act) {
                const int self = own ? t - sf : -1;
                for (int b = 0; b < kLdBlocks; ++b) {
                    const int ja = j0 + b * bs, jb = min(ja + bs, j1);
                    int j = ja;
                    for (; j + 1 < jb; j += 2) {
                        uint64_t v0, v1;
                        ld_weight2(T, src.get(j), src.get(j + 1), k2, rc2, shift, v0, v1);
                        if (own) {
                            v0 = j == self ? 0ull : v0;
                            v1 = j + 1 == self ? 0ull : v1;
                        }
                        part_sum += v0 + v1;
                    }
                    if (j < jb) {
                        uint64_t v0, v1;
                        const float4 Sj = src.get(j);
                        ld_weight2(T, Sj, Sj, k2, rc2, shift, v0, v1);
                        part_sum += own && j == self ? 0ull : v0;
                    }
                    s_pre[w][b][lane] = part_sum;
                }
            }
            // the slices' offsets (an inclusive scan over q; a lane reads only
            // from lanes of the same target below it), added to the prefix sums
            uint64_t incl = part_sum;
            for (int o = TS; o < S * TS; o <<= 1) {
                const uint64_t up = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += up;
            }
            if (S > 1 && act && q > 0) {
                const uint64_t off = incl - part_sum;
                for (int b = 0; b < kLdBlocks; ++b) s_pre[w][b][lane] += off;
            }
            // the neurons' numbers of draws, and their running sum
            const uint64_t tot = __shfl_sync(0xffffffffu, incl, (S - 1) * TS + ti);
            int a = 0;
            if (lane < nt) {
                const int32_t to = perm[t];
                a = (int)pk_axon(__float_as_uint(T.w));
                if (tot == 0 || (int64_t)eoff[to] + a > ne) a = 0;
            }
            int run = a;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, run, o);
                if (lane >= o) run += up;
            }
            s_a[w][lane] = run - a;
            const int total = __shfl_sync(0xffffffffu, run, 31);
            __syncwarp();
            for (int d0 = 0; d0 < total; d0 += 32) {
                const int d = d0 + lane;
                if (d >= total) continue;
                // the drawing neuron: the last one whose draws start at or
                // before d (neurons without draws share the next one's start)
                int u = 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (s_a[w][u + o] <= d) u += o;
                const int e = d - s_a[w][u];
                const int32_t tu = s_tl[w][u], to = perm[tu];
                const float4 Tu = s_T[w][u];
                uint32_t o4[4];
                philox_draw(seed, (uint32_t)to, (uint32_t)e | ((uint32_t)ch << 8) | (kTagLeaf << 16),
                            step, o4);
                const uint64_t u53 = (((uint64_t)o4[0] << 32) | o4[1]) >> 11;
                const uint64_t r =
                    __umul64hi(u53 << 11, s_pre[w][kLdBlocks - 1][(S - 1) * TS + u]);   // floor(U tot)
                int sq = 0;
                while (sq + 1 < S && s_pre[w][kLdBlocks - 1][sq * TS + u] <= r) ++sq;
                const int ln = sq * TS + u;
                int b = 0;                     // the first block whose prefix exceeds r
#pragma unroll
                for (int o = kLdBlocks / 2; o > 0; o >>= 1)
                    if (s_pre[w][b + o - 1][ln] <= r) b += o;
                uint64_t pre = b > 0 ? s_pre[w][b - 1][ln]
                                     : (sq > 0 ? s_pre[w][kLdBlocks - 1][ln - TS] : 0ull);
                const int self = own ? tu - sf : -1;
                int j = sq * L + b * bs;
                const int je = min(min(sq * L + (b + 1) * bs, (sq + 1) * L), sc);
                int hit = -1;
                for (; j + 1 < je; j += 2) {
                    uint64_t v0, v1;
                    ld_weight2(Tu, src.get(j), src.get(j + 1), k2, rc2, shift, v0, v1);
                    pre += j == self ? 0ull : v0;
                    if (pre > r) {
                        hit = j;
                        break;
                    }
                    pre += j + 1 == self ? 0ull : v1;
                    if (pre > r) {
                        hit = j + 1;
                        break;
                    }
                }
                if (hit < 0) hit = je - 1;     // the block's sum exceeds r
                const int32_t dend = perm[sf + hit];
                partner[eoff[to] + e] = dend;
                atomicAdd(&gcnt[(ch ? n : 0) + dend], 1);    // the request's group
                ++draws;
            }
            __syncwarp();
        }
    }
    for (int o = 16; o > 0; o >>= 1) draws += __shfl_xor_sync(0xffffffffu, draws, o);
    if (lane == 0 && draws) atomicAdd(draw_ctr, draws);
}

// a12: the requests grouped by (channel, dendrite), group g = channel * n +
// dendrite, by a counting sort: counts per group (added by the leaf draw), their
// exclusive scan, and a scatter that takes each request's slot from its group's
// count (counting it back down to zero).  The order inside a group is left to the
// atomics; the ranking below does not depend on it.
// key = priority << 32 | group, val = element; cap bounds the slots (the
// buffers' length): a slot outside it (counts that do not match) is not
// written and sets bit 5 of *overflow
__global__ void k_req_scatter(int64_t n, const uint8_t* __restrict__ type,
                              const uint8_t* __restrict__ va, const int32_t* __restrict__ eoff,
                              const int32_t* __restrict__ partner, const int32_t* __restrict__ goff,
                              int32_t* __restrict__ gcnt, uint64_t seed, StepRef stp,
                              uint64_t* __restrict__ key, int32_t* __restrict__ val,
                              int32_t* __restrict__ owner,
                              const int64_t* __restrict__ n_elem, int64_t cap,
                              int64_t* __restrict__ overflow) {
    const uint64_t step = stp.get();
    const int64_t ne = *n_elem;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int a = va[t];
        const int32_t e0 = eoff[t];
        if ((int64_t)e0 + a > ne) continue;
        const int64_t base = type[t] ? n : 0;
        for (int k = 0; k < a; ++k) {
            const int32_t s = partner[e0 + k];
            if (s < 0) continue;
            uint32_t o[4];
            philox_draw(seed, (uint32_t)t, (uint32_t)k | (kTagAccept << 16), step, o);
            const int64_t g = base + s;
            const int64_t r = (int64_t)goff[g] + atomicSub(&gcnt[g], 1) - 1;
            if (r < 0 || r >= cap) {
                atomicOr(reinterpret_cast<unsigned long long*>(overflow), 32ull);
                continue;
            }
            key[r] = ((uint64_t)o[0] << 32) | (uint32_t)g;
            val[r] = e0 + k;
            owner[e0 + k] = (int32_t)t;
        }
    }
}

// A dendrite neuron accepts, per channel, its first `capacity` requests in
// (priority, element) order: the rank of request i is the number of requests
// of its group before it in that order.  Groups are small (the requests one
// neuron receives), so each request counts over its group directly, unless the
// group fits.  accepted: 0, or 1 + the channel.  A group whose count the scatter
// did not bring back to zero sets bit 5 of *overflow.
__global__ void k_accept(const uint64_t* __restrict__ key, const int32_t* __restrict__ val,
                         const int32_t* __restrict__ goff, const int32_t* __restrict__ gcnt,
                         const int64_t* __restrict__ nr_dev, int64_t n,
                         const uint8_t* __restrict__ vde, const uint8_t* __restrict__ vdi,
                         uint8_t* __restrict__ accepted, int64_t* __restrict__ overflow) {
    const int64_t nr = *nr_dev;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t ki = key[i];
        const int64_t g = (int64_t)(uint32_t)ki;
        const uint32_t pr = (uint32_t)(ki >> 32);
        const int32_t ei = val[i];
        const bool inh = g >= n;
        const int64_t s = inh ? g - n : g;
        const int cap = inh ? vdi[s] : vde[s];
        if (gcnt[g] != 0) atomicOr(reinterpret_cast<unsigned long long*>(overflow), 32ull);
        const int64_t j0 = goff[g], j1 = g + 1 < 2 * n ? (int64_t)goff[g + 1] : nr;
        int rank = 0;
        if (j1 - j0 > cap)
            for (int64_t j = j0; j < j1 && rank < cap; ++j) {
                const uint32_t pj = (uint32_t)(key[j] >> 32);
                rank += pj < pr || (pj == pr && val[j] < ei);
            }
        accepted[ei] = rank < cap ? (inh ? 2 : 1) : 0;
    }
}

// The scan over the elements that writes the synapses, in element order: an
// accepted element's prefix is its synapse's index.  (A scan and a pass over the
// neurons took 22 us of 1,000,000 neurons, this takes 13; bound by the latency of
// its reads, so k_scan_1p has all of a thread's in flight at once.)
struct ScanAccepted {
    const uint8_t* acc;
    __device__ int32_t operator()(int64_t i) const { return acc[i] != 0; }
};
struct ScanEmit {
    const uint8_t* acc;
    const int32_t *owner, *partner;
    int32_t *pre, *post;
    uint8_t* type;
    struct Read {
        int32_t owner, partner;
        uint8_t acc;
    };
    __device__ Read read(int64_t i) const { return Read{owner[i], partner[i], acc[i]}; }
    __device__ void operator()(int64_t, int32_t v, const Read& e) const {
        if (!e.acc) return;
        pre[v] = e.owner;
        post[v] = e.partner;
        type[v] = e.acc - 1;
    }
};
// the number of synapses, and in a graph step the step's end
struct ScanSynapses {
    DevCounts* dc;
    int64_t* n_syn;
    GraphEnd end;
    __device__ void operator()(int64_t total) const {
        dc->n_syn = total;
        if (n_syn) *n_syn = total;
        end(dc);
    }
};

__global__ void k_walk(int64_t n, uint64_t seed, StepRef stp, uint8_t* __restrict__ va,
                       uint8_t* __restrict__ vde, uint8_t* __restrict__ vdi,
                       const int64_t* __restrict__ halt) {
    if (halt && *halt) return;
    const uint64_t step = stp.get();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint8_t* v[3] = {va, vde, vdi};
        for (int ch = 0; ch < 3; ++ch) {
            uint32_t o[4];
            philox_draw(seed, (uint32_t)i, (uint32_t)ch | (kTagWalk << 16), step, o);
            int nv = (int)v[ch][i] + ((o[0] & 1u) ? 1 : -1);
            nv = nv < 0 ? 0 : (nv > kMaxVacancy ? kMaxVacancy : nv);
            v[ch][i] = (uint8_t)nv;
        }
    }
}

__device__ inline void sat_dec(uint8_t* p) {
    // byte-wise saturating decrement through the containing 32-bit word
    uintptr_t addr = reinterpret_cast<uintptr_t>(p);
    unsigned int* word = reinterpret_cast<unsigned int*>(addr & ~uintptr_t(3));
    unsigned int sh = (unsigned int)(addr & 3u) * 8u;
    unsigned int old = *word, assumed;
    do {
        assumed = old;
        unsigned int b = (assumed >> sh) & 0xffu;
        if (b == 0) return;
        old = atomicCAS(word, assumed, assumed - (1u << sh));
    } while (old != assumed);
}

__global__ void k_commit(const int64_t* __restrict__ n_syn, int64_t capacity,
                         const int32_t* __restrict__ pre, const int32_t* __restrict__ post,
                         const uint8_t* __restrict__ styp, uint8_t* va, uint8_t* vde, uint8_t* vdi,
                         const int64_t* __restrict__ halt) {
    if (halt && *halt) return;
    int64_t m = *n_syn;
    if (m > capacity) m = capacity;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m;
         k += (int64_t)gridDim.x * blockDim.x) {
        sat_dec(va + pre[k]);
        sat_dec((styp[k] ? vdi : vde) + post[k]);
    }
}

}  // namespace

void select_partners(msp_ctx& c, uint64_t step, const uint8_t* type_dev, const uint8_t* va_dev,
                     const uint8_t* vde_dev, const uint8_t* vdi_dev, int32_t* partner,
                     int32_t* syn_pre, int32_t* syn_post, uint8_t* syn_type, int64_t* n_syn,
                     cudaStream_t s) {
    NvtxRange nv_("msp select_partners");
    if (!c.attraction_done) throw Error(MSP_ERR_NOT_BUILT, "msp_attraction must run first");
    const msp_config& cfg = c.cfg;
    // the element count: exact from the build, or (whole-step graph) the
    // capacity of its buffers (the vacancy walk's bound, or the host-buffer
    // call's); kernels read the exact count from device memory and never
    // index past it
    const int64_t n = c.n, ne = c.graph_mode ? c.graph_elem_cap : c.n_elem;
    const int B = 256;
    const float k2 = (float)(1.4426950408889634 / (cfg.sigma * cfg.sigma));
    // inside a leaf the kernel is truncated at the radius that prunes box pairs
    const float rc2 = (float)((cfg.cutoff * cfg.sigma) * (cfg.cutoff * cfg.sigma));
    c.n_draws = c.n_requests = c.n_synapses = 0;
    if (ne == 0) {
        MSP_CUDA(cudaMemsetAsync(n_syn, 0, sizeof(int64_t), s));
        if (!c.graph_mode) MSP_CUDA(cudaStreamSynchronize(s));
        return;
    }
    DevCounts* dc = dcounts(c);
    const StepRef stp{step, c.graph_mode ? &dc->step : nullptr};
    const int ge = grid_for(ne, B, (int64_t)c.sm_count * 16);
    Tree tr;
    tr.level = c.nd_level.get<uint8_t>();
    tr.first = c.nd_first.get<int32_t>();
    tr.count = c.nd_count.get<int32_t>();
    tr.child_first = c.nd_child_first.get<int32_t>();
    tr.nchild = c.nd_nchild.get<uint8_t>();
    tr.sums = c.nd_sums.get<int4>();
    // expansion centres (the geometric ones with centre_mode 1)
    tr.ca = c.cfg.centre_mode == 1 ? c.nd_gc.get<float4>() : c.nd_ca.get<float4>();
    tr.cd = c.cfg.centre_mode == 1 ? c.nd_gc.get<float4>() : c.nd_cd.get<float4>();
    Exps ex;
    ex.A = c.expA.get<float>();
    ex.M = c.expM.get<float>();
    ex.first = c.exp_first;
    ex.p = cfg.p;
    ex.inv_sigma = (float)(1.0 / cfg.sigma);

    // a11: the level steps of the descent.  At step k every inner box of an
    // item is at level k (inner boxes always go one level down; a leaf stays),
    // and an item of two leaves goes to the per-element draw, so depth + 1
    // steps empty the item list.
    const int64_t cap_items = 2 * c.n_nodes + 64, cap_leaf = 2 * c.n_nodes + 64;
    Item* ib[2] = {c.items0.ensure<Item>((size_t)cap_items), c.items1.ensure<Item>((size_t)cap_items)};
    Item* lit = c.leaf_items.ensure<Item>((size_t)cap_leaf);
    // the group counts: cleared before an eager selection and whenever the
    // buffer is new; every complete scatter counts them back down to zero
    const size_t ng = (size_t)std::max<int64_t>(2 * n, 1);
    const size_t gcnt_bytes = c.rq_gcnt.bytes;
    int32_t* gcnt = c.rq_gcnt.ensure<int32_t>(ng);
    const bool clear_gcnt = !c.graph_mode || c.rq_gcnt.bytes != gcnt_bytes;
    int32_t* goff = c.rq_goff.ensure<int32_t>(ng);
    uint8_t* acc = c.accepted.ensure<uint8_t>((size_t)ne);
    uint64_t* k0 = c.rq_key0.ensure<uint64_t>((size_t)ne);
    int32_t* v0 = c.rq_val0.ensure<int32_t>((size_t)ne);
    int32_t* owner = c.rq_owner.ensure<int32_t>((size_t)ne);
    // status words of the two scans, one after the other
    const int64_t n_st0 = scan_status_words((int64_t)ng), n_st1 = scan_status_words(ne);
    unsigned long long* st0 = c.sd_tmp.ensure<unsigned long long>((size_t)(n_st0 + n_st1));
    k_select_init<<<grid_for(std::max<int64_t>(ne, clear_gcnt ? (int64_t)ng : 0), B,
                             (int64_t)c.sm_count * 8), B, 0, s>>>(
        c.nd_sums.get<int4>(), c.pr_w.get<float4>(), ib[0], dc, n, partner, acc, gcnt,
        clear_gcnt ? (int64_t)(c.rq_gcnt.bytes / sizeof(int32_t)) : 0, st0, n_st0 + n_st1);
    MSP_LAUNCH("select_init");
    auto ull = [](int64_t* p) { return reinterpret_cast<unsigned long long*>(p); };
    const int n_steps = c.tree_depth + 1;
    const DescArgs da{tr, ex, c.pr_kind.get<uint8_t>(), c.pr_cf.get<int32_t>(),
                      c.pr_w.get<float2>(), cfg.seed, stp, {ib[0], ib[1]}, cap_items, lit, cap_leaf,
                      dc};
    const int top = std::min(n_steps, kDescTop);
    const size_t warp_bytes = desc_warp_floats(cfg.p) * sizeof(float);
    allow_shared(k_descend_top, kDescTopWarps * warp_bytes,
                 kDescTopWarps * desc_warp_floats(kMaxP) * sizeof(float));
    k_descend_top<<<1, kDescTopWarps * 32, kDescTopWarps * warp_bytes, s>>>(da, top);
    MSP_LAUNCH("descend_top");
    for (int k = top; k < n_steps; ++k) {
        // at most two items (channels) for each of 8^k boxes, 16 a block
        const int64_t most = std::min<int64_t>(cap_items, (int64_t)2 << std::min(3 * k, 40));
        k_descend<<<grid_for(most, 4 * kDescWarps, (int64_t)c.sm_count * 16), kDescWarps * 32,
                    kDescWarps * warp_bytes, s>>>(da, k);
        MSP_LAUNCH("descend");
    }
    // one warp per leaf pair, from a device work counter
    FrameRc2 frc{nullptr, c.nd_prefix.get<uint64_t>(), c.nd_level.get<uint8_t>(), c.frame_level,
                 (int64_t)c.frame_off_host.size() - 1};
    if (c.frame_level > 0 && c.frame_plans) frc.rc2 = c.frame_rc2.get<float>();
    k_leaf_draw_w<<<(int)std::max<int64_t>(1, (int64_t)c.sm_count * 8), kLdWarps * 32, 0, s>>>(
        lit, &dc->n_leaf, cap_leaf, ull(&dc->leaf_next), c.nd_first.get<int32_t>(),
        c.nd_count.get<int32_t>(), c.pts.get<float4>(), c.wts.get<float2>(),
        c.perm.get<int32_t>(), c.elem_off.get<int32_t>(), k2, rc2, frc, cfg.seed, stp, partner,
        gcnt, n, ull(&dc->draws), &dc->n_elem);
    MSP_LAUNCH("leaf_draw");

    // a12: requests grouped by (channel, dendrite), ranked by (priority, element)
    const int gn = grid_for(n, B, (int64_t)c.sm_count * 16);
    scan_launch(c, ScanI32{gcnt}, ScanStore{goff}, ScanTotal{&dc->n_req}, &dc->n_groups, (int64_t)ng,
                s, st0);
    k_req_scatter<<<gn, B, 0, s>>>(n, type_dev, va_dev, c.elem_off.get<int32_t>(), partner, goff,
                                   gcnt, cfg.seed, stp, k0, v0, owner, &dc->n_elem, (int64_t)ne,
                                   &dc->overflow);
    MSP_LAUNCH("req_scatter");
    k_accept<<<ge, B, 0, s>>>(k0, v0, goff, gcnt, &dc->n_req, n, vde_dev, vdi_dev, acc,
                              &dc->overflow);
    MSP_LAUNCH("accept");
    const bool aligned = reinterpret_cast<uintptr_t>(n_syn) % sizeof(int64_t) == 0;
    GraphEnd end = c.graph_end;
    end.on = c.graph_mode;
    end.left_slot = n_steps % 3;
    scan_launch(c, ScanAccepted{acc}, ScanEmit{acc, owner, partner, syn_pre, syn_post, syn_type},
                ScanSynapses{dc, aligned ? n_syn : nullptr, end}, &dc->n_elem, ne, s, st0 + n_st0);
    if (!aligned)
        MSP_CUDA(cudaMemcpyAsync(n_syn, &dc->n_syn, sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
    if (c.graph_mode) return;       // checked on the device (GraphEnd)
    pull_counts(c, s);              // the one synchronisation of the selection
    const DevCounts& hc = *c.hcount;
    if (hc.overflow & 6) throw Error(MSP_ERR_CHECK, "descent item capacity exceeded");
    if (hc.overflow & 32) throw Error(MSP_ERR_CHECK, "request groups inconsistent");
    if (hc.items[n_steps % 3] != 0) throw Error(MSP_ERR_CHECK, "descent did not terminate");
    c.n_draws = hc.draws;
    c.n_requests = hc.n_req;
    c.n_synapses = hc.n_syn;
}

void vacancy_walk(msp_ctx& c, int64_t n, uint64_t step, uint8_t* va, uint8_t* vde, uint8_t* vdi,
                  cudaStream_t s) {
    if (n <= 0) return;
    DevCounts* dc = dcounts(c);
    const StepRef stp{step, c.graph_mode ? &dc->step : nullptr};
    k_walk<<<grid_for(n, 256, (int64_t)c.sm_count * 16), 256, 0, s>>>(
        n, c.cfg.seed, stp, va, vde, vdi, c.graph_mode ? &dc->halt : nullptr);
    MSP_LAUNCH("walk");
}

void commit_synapses(msp_ctx& c, const int64_t* n_syn, int64_t capacity, const int32_t* pre,
                     const int32_t* post, const uint8_t* styp, uint8_t* va, uint8_t* vde,
                     uint8_t* vdi, cudaStream_t s) {
    if (capacity <= 0) return;
    k_commit<<<grid_for(capacity, 256, (int64_t)c.sm_count * 16), 256, 0, s>>>(
        n_syn, capacity, pre, post, styp, va, vde, vdi,
        c.graph_mode ? &dcounts(c)->halt : nullptr);
    MSP_LAUNCH("commit");
}

}  // namespace msp
