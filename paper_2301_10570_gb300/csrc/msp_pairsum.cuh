// msp_pairsum.cuh -- sums over the near-field leaf pairs that need no result
// per pair: the walk shared by the derivatives (msp_grad.cu) and the synapse
// length (msp_length.cu), forward (per target, over its partner leaves'
// sources) and transposed (per source, over its partner leaves' targets).
//
// The set of near-field pairs is symmetric: the traversal starts at (root,
// root), splits both sides alike, and the cutoff test does not change when the
// boxes change places; only translated pairs break it, and these sums refuse
// them.  So the segment of leaf L in the list sorted by target leaf names the
// partners of L in both directions, and the transposed sums need no list of
// their own.
//
// One block of 4 warps takes a segment (longest first), its warps the partner
// leaves round-robin.  A warp reads 32 partner ranges at a time and walks
// their points as one sequence, 64 per staged unit: every lane loads two
// points and stores them as one staged pair (paired FP32, 16-byte stores), so
// a leaf's size does not matter to the staging.  A lane holds R evaluation
// points; when the points' groups fit in npr = 2^k < 32 lanes, 32 / npr lanes
// share a group, each over an interleaved slice of the staged pairs.
#pragma once

#include "msp_internal.cuh"

namespace msp {

constexpr int kPsWarps = 4;
constexpr int kPsUnit = 64;                  // points per staged unit
constexpr int kPsPairs = 2 * kPsUnit / 2;    // staged pairs of a chunk (two units)
constexpr int kPsList = 128;                 // evaluation slots per pass
// per sorted point: bit 0 type, bit 1 a > 0, a in the high byte
constexpr uint32_t kPsInh = 1u, kPsAct = 2u;

__device__ __forceinline__ float ps_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The points of a segment's partner ranges, chunk by chunk.  range(m) maps a
// partner leaf's (first point, count) to the range to stage (count 0: none);
// stage(a, b, two, slot) stores points a and b (b only if two) as staged pair
// `slot`; eval(mp) evaluates the staged pairs [0, mp) (the first unit's come
// first).  meta: the warp's own 32 entries of shared memory.
template <class Range, class Stage, class Eval>
__device__ __forceinline__ void ps_walk(const int2* __restrict__ src, int32_t i0, int32_t i1,
                                        int2* meta, Range range, Stage stage, Eval eval) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned le = 0xffffffffu >> (31 - lane);
    for (int32_t cb = i0 + w; cb < i1; cb += 32 * kPsWarps) {
        const int32_t mi = cb + kPsWarps * lane;
        int2 m = make_int2(0, 0);
        if (mi < i1) m = range(src[mi]);
        // the non-empty ranges, one per lane
        const unsigned nz = __ballot_sync(0xffffffffu, m.y > 0);
        __syncwarp();
        if (m.y > 0) meta[__popc(nz & le) - 1] = m;
        __syncwarp();
        m = lane < __popc(nz) ? meta[lane] : make_int2(0, 0);
        int inc = m.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        const int tot = __shfl_sync(0xffffffffu, inc, 31);
        const int start = inc - m.y, shift = m.x - start;
        // the point at position p + lane: the last range that starts at or
        // before it, from the ranges' starts as a bit mask over 32 positions
        auto point = [&](int p) {
            const int rel = start - p;
            const unsigned bit = m.y > 0 && rel >= 0 && rel < 32 ? 1u << rel : 0u;
            const unsigned starts = __reduce_or_sync(0xffffffffu, bit);
            const int before = __popc(__ballot_sync(0xffffffffu, m.y > 0 && rel < 0));
            const int k = before + __popc(starts & le) - 1;
            return __shfl_sync(0xffffffffu, shift, k) + p + lane;
        };
        for (int q = 0; q < tot; q += 2 * kPsUnit) {
            int mp = 0;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int left = min(tot - q - r * kPsUnit, kPsUnit);
                if (left > 0) {
                    const int half = (left + 1) >> 1, p = q + r * kPsUnit;
                    const int32_t a = point(p), b = point(p + half);
                    if (lane < half) stage(a, b, lane < left - half, mp + lane);
                    mp += half;
                }
            }
            __syncwarp();
            eval(mp);
        }
    }
}

// Slots per lane: R = 1..RMAX with the smallest time per staged pair, npr
// lanes (a power of two) times the larger of the arithmetic (per4 quarter
// cycles an SM and slot) and the shared-memory delivery (lds cycles an SM).
// slots(R) is the number of slots with padding.
template <int RMAX, class Slots>
__device__ __forceinline__ int ps_choose_r(Slots slots, int per4, int lds) {
    int R = RMAX, best = 1 << 30;
    for (int r = RMAX; r >= 1; --r) {
        const int g = (slots(r) + r - 1) / r;
        if (g > 32) continue;
        int npr = 1;
        while (npr < g) npr <<= 1;
        const int cost = npr * max(per4 * r, 4 * lds);
        if (cost < best) {
            best = cost;
            R = r;
        }
    }
    return R;
}

// The pass list of a target leaf's next targets (a > 0), by one warp: the
// excitatory ones, padding (-1) up to a multiple of R when inhibitory ones
// follow, the inhibitory ones, so that a lane's R slots share a channel.  At
// most `most` targets from position pos on.  Returns through the pointers the
// slots, R and the position to resume at.
template <int RMAX>
__device__ __forceinline__ void ps_list_targets(const uint16_t* __restrict__ fl, int32_t lf,
                                                int32_t lc, int32_t pos, int most, int per4,
                                                int lds, int32_t* list, int* s_np, int* s_pos,
                                                int* s_R) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int nt = 0, nE = 0;
    int32_t p = pos, end = lc;
    for (; p < lc; p += 32) {
        const uint32_t f = p + lane < lc ? fl[lf + p + lane] : 0u;
        const unsigned mk = __ballot_sync(0xffffffffu, (f & kPsAct) != 0);
        const unsigned mE = __ballot_sync(0xffffffffu, (f & kPsAct) && !(f & kPsInh));
        const int room = most - nt;
        if (__popc(mk) > room) {
            // the room-th target ends the pass: resume at the one after it
            unsigned keep = mk;
            for (int k = 0; k < room; ++k) keep &= keep - 1u;
            const int stop = __ffs(keep) - 1;
            nE += __popc(mE & ((1u << stop) - 1u));
            nt = most;
            end = p + stop;
            break;
        }
        nt += __popc(mk);
        nE += __popc(mE);
    }
    const int nI = nt - nE;
    auto padded = [&](int R) { return nt + (nI > 0 ? (R - nE % R) % R : 0); };
    const int R = ps_choose_r<RMAX>(padded, per4, lds);
    const int pad = padded(R) - nt;
    int we = 0, wi = nE + pad;
    for (int32_t q = pos; q < end; q += 32) {
        const uint32_t f = q + lane < end ? fl[lf + q + lane] : 0u;
        const bool isE = (f & kPsAct) && !(f & kPsInh), isI = (f & kPsAct) && (f & kPsInh);
        const unsigned mE = __ballot_sync(0xffffffffu, isE), mI = __ballot_sync(0xffffffffu, isI);
        if (isE) list[we + __popc(mE & lt)] = lf + q + lane;
        if (isI) list[wi + __popc(mI & lt)] = lf + q + lane;
        we += __popc(mE);
        wi += __popc(mI);
    }
    if (lane < pad) list[nE + lane] = -1;
    if (lane == 0) {
        *s_np = nt + pad;
        *s_pos = end;
        *s_R = R;
    }
}

// lanes of a pass: group j (of npr) and slice ksl (of slices)
struct PsLanes {
    int npr, slices, j, ksl;
    __device__ PsLanes(int np, int R) {
        int lg = 0;
        while ((1 << lg) < (np + R - 1) / R) ++lg;
        const int lane = threadIdx.x & 31;
        npr = 1 << lg;
        slices = 32 >> lg;
        j = lane & (npr - 1);
        ksl = lane >> lg;
    }
    // the slices' sums of a value, in a fixed order
    __device__ float sum(float v) const {
        for (int o = npr; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
};

// Forward staging: sources a and b of the sorted points with their weights of
// both channels (w: sorted order), scaled and relative to O: A = (-x0, -x1,
// -y0, -y1), E = (-z0, -z1, wE0, wE1), I = (-z0, -z1, wI0, wI1); E and I are
// one 16-byte entry apart from a multiple of 128 bytes, so that lanes of
// both channels read different banks.
struct PsFwdStage {
    float4 A[kPsPairs], E[kPsPairs + 1], I[kPsPairs];
};

__device__ __forceinline__ void ps_stage_fwd(PsFwdStage& st, const float4* __restrict__ pts,
                                             const float2* __restrict__ w, int32_t a, int32_t b,
                                             bool two, int slot, const float4& O, float sqk) {
    const float4 S0 = pts[a], S1 = pts[two ? b : a];
    const float2 w0 = w[a], w1 = two ? w[b] : make_float2(0.f, 0.f);
    const float2 k = make_float2(sqk, sqk);
    const float2 x = __fmul2_rn(__fadd2_rn(make_float2(O.x, O.x), make_float2(-S0.x, -S1.x)), k);
    const float2 y = __fmul2_rn(__fadd2_rn(make_float2(O.y, O.y), make_float2(-S0.y, -S1.y)), k);
    const float2 z = __fmul2_rn(__fadd2_rn(make_float2(O.z, O.z), make_float2(-S0.z, -S1.z)), k);
    st.A[slot] = make_float4(x.x, x.y, y.x, y.y);
    st.E[slot] = make_float4(z.x, z.y, w0.x, w1.x);
    st.I[slot] = make_float4(z.x, z.y, w0.y, w1.y);
}

// Transposed staging: the targets of one channel, packed (PsPacked, filled by
// k_grad_pack and k_len_pack) as {x, y, z, sorted index}; difference form: A = (-x0,
// -x1, -y0, -y1), B = (-z0, -z1, ..); D: the sorted indices (own leaf only).
struct PsAdjStage {
    float4 A[kPsPairs], B[kPsPairs];
    float2 C[kPsPairs];
    int2 D[kPsPairs];
};

// The packed targets: those of the excitatory channel in sorted order, then
// the inhibitory ones; off[ch * n + j] is the position of the first one at or
// after sorted point j (off has 2 n + 1 entries), so leaf (f, c) holds the
// packed range [off[ch n + f], off[ch n + f + c]).
struct PsPacked {
    const float4* pt;
    const int32_t* off;
};
// flags and offsets of fl's targets (scan), leaving the scatter to the caller
const int32_t* ps_offsets(msp_ctx& c, const uint16_t* fl, cudaStream_t s);

}  // namespace msp
