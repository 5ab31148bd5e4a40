// msp_grad.cu -- derivatives of the attraction (Eq. 8), the adjoint of the
// near field: with K(t,s) = exp(-r^2/sigma^2) = 2^-q, q = r^2 log2(e)/sigma^2,
//   u(t)      = sum_{s != t} w_s^{T(t)} K                        (a_t > 0)
//   du/dsigma = sum_{s != t} w_s^{T(t)} K 2 r^2 / sigma^3
//             = (2 / (sigma log2 e)) sum_{s != t} w_s^{T(t)} q 2^-q
//   dL/dw^T_s = sum_{t != s, a_t > 0, T(t) = T} g_t K(t,s)   for L = sum_t g_t u(t)
// summed over the near-field leaf pairs of the last attraction (a plan
// without translated pairs), at counts the caller passes (the tree's own
// counts only chose the pairs).  Both directions run one block per leaf over its
// segment of the pair list sorted by target leaf: the near-field pairs are
// symmetric (msp_pairsum.cuh), so the segment names the leaf's partners as
// sources and as targets; the partners' points are staged in shared memory.
// Every sum has a fixed order: the results are reproducible.  The distance
// is formed as a difference (no expanded form), in single precision.
#include <algorithm>
#include <cmath>

#include "msp_hostdev.cuh"
#include "msp_pairsum.cuh"

namespace msp {

namespace {

// sorted-order inputs: the weights (w^E, w^I) and the targets' flags; grads of
// points without terms stay zero (out of the pair sums)
__global__ void k_grad_gather(int64_t n, const int32_t* __restrict__ perm,
                              const uint8_t* __restrict__ type, const uint8_t* __restrict__ va,
                              const uint8_t* __restrict__ vde, const uint8_t* __restrict__ vdi,
                              float2* __restrict__ w, uint16_t* __restrict__ fl) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = perm[s];
        w[s] = make_float2((float)vde[c], (float)vdi[c]);
        fl[s] = (uint16_t)((type[c] ? kPsInh : 0u) | (va[c] ? kPsAct : 0u) | ((uint32_t)va[c] << 8));
    }
}

// entries of the packed targets' scan: [0, n) excitatory, [n, 2n) inhibitory,
// one zero after them
__global__ void k_ps_flags(int64_t n, const uint16_t* __restrict__ fl, int32_t* __restrict__ flag,
                           int64_t* __restrict__ scan_n) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *scan_n = 2 * n + 1;
        flag[2 * n] = 0;
    }
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t f = fl[s];
        flag[s] = (f & kPsAct) && !(f & kPsInh);
        flag[n + s] = (f & kPsAct) && (f & kPsInh);
    }
}

// the packed targets with their g
__global__ void k_grad_pack(int64_t n, const uint16_t* __restrict__ fl,
                            const int32_t* __restrict__ off, const int32_t* __restrict__ perm,
                            const float4* __restrict__ pts, const float* __restrict__ g,
                            float4* __restrict__ pt, float* __restrict__ pg) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t f = fl[s];
        if (!(f & kPsAct)) continue;
        const int32_t k = off[((f & kPsInh) ? n : 0) + s];
        const float4 P = pts[s];
        pt[k] = make_float4(P.x, P.y, P.z, __int_as_float((int32_t)s));
        pg[k] = g[perm[s]];
    }
}

// FORWARD: u(t) = sum w K and sum w q K (times dscale: du/dsigma) for the
// targets of the block's leaf.  The distance is formed as a difference: the
// second sum needs q itself, which the expanded exponent gives only with an
// absolute error that is large against q for the closest pairs.  Two terms:
// dx = t - s (s staged negated), q = fma(dx, dx, fma(dy, dy, dz dz)), K =
// 2^-q.  SELF: a source may be the target itself (sorted index); its term is
// zero.
constexpr int kGrFwdR = 4;

template <int R, bool SELF>
__device__ __forceinline__ void gr_fwd_eval(const float4* sA, const float4* sW, int mp, int ksl,
                                            int slices, const float2 (&tx)[R],
                                            const float2 (&ty)[R], const float2 (&tz)[R],
                                            const int32_t (&e)[R], int32_t first, int32_t second,
                                            float2 (&a0)[R], float2 (&a1)[R]) {
#pragma unroll 2
    for (int j = ksl; j < mp; j += slices) {
        const float4 A = sA[j], B = sW[j];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 dx = __fadd2_rn(tx[r], make_float2(A.x, A.y));
            const float2 dy = __fadd2_rn(ty[r], make_float2(A.z, A.w));
            const float2 dz = __fadd2_rn(tz[r], make_float2(B.x, B.y));
            const float2 q = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            float2 K = make_float2(ps_ex2(-q.x), ps_ex2(-q.y));
            if (SELF) {
                K.x = first + j == e[r] ? 0.f : K.x;
                K.y = second + j == e[r] ? 0.f : K.y;
            }
            const float2 wk = __fmul2_rn(make_float2(B.z, B.w), K);
            a0[r] = __fadd2_rn(a0[r], wk);
            a1[r] = __ffma2_rn(wk, q, a1[r]);
        }
    }
}

template <int R>
__device__ __forceinline__ void gr_fwd_pass(const int32_t* list, int np, int32_t i0, int32_t i1,
                                            int32_t lf, int32_t lc, const float4& O,
                                            const int2* __restrict__ src,
                                            const float4* __restrict__ pts,
                                            const float2* __restrict__ wt,
                                            const uint16_t* __restrict__ fl, float sqk,
                                            PsFwdStage& st, int2* meta, float2* red) {
    const int lane = threadIdx.x & 31;
    const PsLanes ln(np, R);
    float2 tx[R], ty[R], tz[R], a0[R], a1[R];
    int32_t e[R];
    bool inh = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int slot = R * ln.j + r;
        e[r] = slot < np ? list[slot] : -1;
        const int32_t t = e[r] >= 0 ? e[r] : lf;
        if (r == 0) inh = e[0] >= 0 && (fl[t] & kPsInh);
        const float4 T = pts[t];
        const float x = (T.x - O.x) * sqk, y = (T.y - O.y) * sqk, z = (T.z - O.z) * sqk;
        tx[r] = make_float2(x, x);
        ty[r] = make_float2(y, y);
        tz[r] = make_float2(z, z);
        a0[r] = a1[r] = make_float2(0.f, 0.f);
    }
    const float4* sW = inh ? st.I : st.E;
    bool self = false;
    ps_walk(
        src, i0, i1, meta,
        [&](int2 m) {
            if (m.x == lf) {
                self = true;
                m.y = 0;
            }
            return m;
        },
        [&](int32_t a, int32_t b, bool two, int slot) {
            ps_stage_fwd(st, pts, wt, a, b, two, slot, O, sqk);
        },
        [&](int mp) {
            gr_fwd_eval<R, false>(st.A, sW, mp, ln.ksl, ln.slices, tx, ty, tz, e, 0, 0, a0, a1);
        });
    // L's own points, where a target skips itself
    if (__any_sync(0xffffffffu, self))
        for (int32_t p = 0; p < lc; p += kPsUnit) {
            const int left = min(lc - p, kPsUnit), half = (left + 1) >> 1;
            __syncwarp();
            if (lane < half)
                ps_stage_fwd(st, pts, wt, lf + p + lane, lf + p + half + lane, lane < left - half,
                             lane, O, sqk);
            __syncwarp();
            gr_fwd_eval<R, true>(st.A, sW, half, ln.ksl, ln.slices, tx, ty, tz, e, lf + p,
                                 lf + p + half, a0, a1);
        }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float s0 = ln.sum(a0[r].x + a0[r].y), s1 = ln.sum(a1[r].x + a1[r].y);
        if (ln.ksl == 0 && R * ln.j + r < np) red[R * ln.j + r] = make_float2(s0, s1);
    }
}

__global__ void __launch_bounds__(kPsWarps * 32, 6)
k_grad_forward(const int32_t* __restrict__ seg_first, const int64_t* __restrict__ nseg_dev,
               const int32_t* __restrict__ order, const int32_t* __restrict__ pairs,
               const int32_t* __restrict__ pX, const int2* __restrict__ src,
               const int32_t* __restrict__ nfirst, const int32_t* __restrict__ ncount,
               const float4* __restrict__ pts, const float2* __restrict__ wt,
               const uint16_t* __restrict__ fl, const int32_t* __restrict__ perm, float sqk,
               float dscale, float* __restrict__ u, float* __restrict__ du) {
    __shared__ PsFwdStage st[kPsWarps];
    __shared__ int2 meta[kPsWarps][32];
    __shared__ float2 red[kPsWarps][kPsList];
    __shared__ int32_t list[kPsList];
    __shared__ int s_np, s_pos, s_R;
    const int w = threadIdx.x >> 5;
    const int64_t nseg = *nseg_dev;
    for (int64_t b = blockIdx.x; b < nseg; b += gridDim.x) {
        const int32_t sg = order[b], i0 = seg_first[sg], i1 = seg_first[sg + 1];
        const int32_t L = pX[pairs[i0]], lf = nfirst[L], lc = ncount[L];
        // positions relative to a point of L before scaling: small operands,
        // so the differences keep their precision
        const float4 O = pts[lf];
        for (int32_t pos = 0; pos < lc;) {
            // up to 4 R slots a pass; nine paired FP32 instructions a slot
            // (18 quarter cycles an SM), two 16-byte loads a staged pair
            if (w == 0)
                ps_list_targets<kGrFwdR>(fl, lf, lc, pos, kPsList - kGrFwdR + 1, 18, 8, list,
                                         &s_np, &s_pos, &s_R);
            __syncthreads();
            const int np = s_np, R = s_R;
            pos = s_pos;
            if (np > 0) {
#define MSP_GR_FWD(RR)                                                                        \
    gr_fwd_pass<RR>(list, np, i0, i1, lf, lc, O, src, pts, wt, fl, sqk, st[w], meta[w], red[w])
                if (R == 1) MSP_GR_FWD(1);
                else if (R == 2) MSP_GR_FWD(2);
                else if (R == 3) MSP_GR_FWD(3);
                else MSP_GR_FWD(4);
#undef MSP_GR_FWD
            }
            __syncthreads();
            for (int k = threadIdx.x; k < np; k += kPsWarps * 32) {
                if (list[k] < 0) continue;
                float2 v = red[0][k];
#pragma unroll
                for (int q = 1; q < kPsWarps; ++q) {
                    v.x += red[q][k].x;
                    v.y += red[q][k].y;
                }
                const int32_t c = perm[list[k]];
                if (u) u[c] = v.x;
                if (du) du[c] = v.y * dscale;
            }
            __syncthreads();
        }
    }
}

// TRANSPOSED: for every point s of the block's leaf, sum_t g_t K(t,s) over the
// partner leaves' targets of one channel after the other.  FAST, the expanded
// form while every point of the pass has |s^|^2 <= kGrFastT2: with the point
// held as 2 s^ and a staged target as (t^, -|t^|^2), E = 2 s^.t^ - |t^|^2 and
// K = 2^E 2^-|s^|^2 (the last factor applied once per point; E <= |s^|^2).
constexpr float kGrFastT2 = 20.f;
constexpr int kGrAdjR = 5;

template <int R, bool SELF, bool FAST>
__device__ __forceinline__ void gr_adj_eval(const PsAdjStage& st, int mp, int ksl, int slices,
                                            const float2 (&tx)[R], const float2 (&ty)[R],
                                            const float2 (&tz)[R], const int32_t (&e)[R],
                                            float2 (&acc)[R]) {
#pragma unroll 2
    for (int j = ksl; j < mp; j += slices) {
        const float4 A = st.A[j], B = st.B[j];
        const float2 C = FAST ? st.C[j] : make_float2(B.z, B.w);
        const int2 D = SELF ? st.D[j] : make_int2(0, 0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float2 K;
            if (FAST) {
                const float2 E = __ffma2_rn(
                    tx[r], make_float2(A.x, A.y),
                    __ffma2_rn(ty[r], make_float2(A.z, A.w),
                               __ffma2_rn(tz[r], make_float2(B.x, B.y), make_float2(B.z, B.w))));
                K = make_float2(ps_ex2(E.x), ps_ex2(E.y));
            } else {
                const float2 dx = __fadd2_rn(tx[r], make_float2(A.x, A.y));
                const float2 dy = __fadd2_rn(ty[r], make_float2(A.z, A.w));
                const float2 dz = __fadd2_rn(tz[r], make_float2(B.x, B.y));
                const float2 q = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                K = make_float2(ps_ex2(-q.x), ps_ex2(-q.y));
            }
            if (SELF) {
                K.x = D.x == e[r] ? 0.f : K.x;
                K.y = D.y == e[r] ? 0.f : K.y;
            }
            acc[r] = __ffma2_rn(C, K, acc[r]);
        }
    }
}

template <int R, bool FAST>
__device__ __forceinline__ void gr_adj_pass(int32_t first, int np, int32_t i0, int32_t i1,
                                            int32_t lf, int32_t lc, int64_t n, const float4& O,
                                            const int2* __restrict__ src,
                                            const float4* __restrict__ pts, const PsPacked pk,
                                            const float* __restrict__ pg, float sqk,
                                            PsAdjStage& st, int2* meta, float2* red) {
    const int lane = threadIdx.x & 31;
    const PsLanes ln(np, R);
    float2 tx[R], ty[R], tz[R], acc[R];
    float sc[R], sE[R];
    int32_t e[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int slot = R * ln.j + r;
        e[r] = first + (slot < np ? slot : 0);
        const float4 T = pts[e[r]];
        const float x = (T.x - O.x) * sqk, y = (T.y - O.y) * sqk, z = (T.z - O.z) * sqk;
        const float f = FAST ? 2.f : 1.f;
        tx[r] = make_float2(f * x, f * x);
        ty[r] = make_float2(f * y, f * y);
        tz[r] = make_float2(f * z, f * z);
        sc[r] = FAST ? ps_ex2(-fmaf(x, x, fmaf(y, y, z * z))) : 1.f;
        sE[r] = 0.f;
    }
    auto stage = [&](int32_t a, int32_t b, bool two, int slot) {
        const float4 S0 = pk.pt[a], S1 = pk.pt[two ? b : a];
        const float2 g = make_float2(pg[a], two ? pg[b] : 0.f);
        const float2 k = make_float2(sqk, sqk);
        float2 x = __fmul2_rn(__fadd2_rn(make_float2(S0.x, S1.x), make_float2(-O.x, -O.x)), k);
        float2 y = __fmul2_rn(__fadd2_rn(make_float2(S0.y, S1.y), make_float2(-O.y, -O.y)), k);
        float2 z = __fmul2_rn(__fadd2_rn(make_float2(S0.z, S1.z), make_float2(-O.z, -O.z)), k);
        if (FAST) {
            const float2 q = __ffma2_rn(x, x, __ffma2_rn(y, y, __fmul2_rn(z, z)));
            st.A[slot] = make_float4(x.x, x.y, y.x, y.y);
            st.B[slot] = make_float4(z.x, z.y, -q.x, -q.y);
            st.C[slot] = g;
        } else {
            st.A[slot] = make_float4(-x.x, -x.y, -y.x, -y.y);
            st.B[slot] = make_float4(-z.x, -z.y, g.x, g.y);
        }
        st.D[slot] = make_int2(__float_as_int(S0.w), two ? __float_as_int(S1.w) : -1);
    };
#pragma unroll 1
    for (int ch = 0; ch < 2; ++ch) {
        const int32_t* off = pk.off + ch * n;
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = make_float2(0.f, 0.f);
        bool self = false;
        ps_walk(
            src, i0, i1, meta,
            [&](int2 m) {
                if (m.x == lf) {
                    self = true;
                    return make_int2(0, 0);
                }
                const int32_t a = off[m.x];
                return make_int2(a, off[m.x + m.y] - a);
            },
            stage,
            [&](int mp) {
                gr_adj_eval<R, false, FAST>(st, mp, ln.ksl, ln.slices, tx, ty, tz, e, acc);
            });
        // L's own targets, where a point skips itself
        if (__any_sync(0xffffffffu, self)) {
            const int32_t a0 = off[lf], a1 = off[lf + lc];
            for (int32_t p = a0; p < a1; p += kPsUnit) {
                const int left = min(a1 - p, kPsUnit), half = (left + 1) >> 1;
                __syncwarp();
                if (lane < half) stage(p + lane, p + half + lane, lane < left - half, lane);
                __syncwarp();
                gr_adj_eval<R, true, FAST>(st, half, ln.ksl, ln.slices, tx, ty, tz, e, acc);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float v = ln.sum(acc[r].x + acc[r].y) * sc[r];
            if (ch == 0) {
                sE[r] = v;
            } else if (ln.ksl == 0 && R * ln.j + r < np) {
                red[R * ln.j + r] = make_float2(sE[r], v);
            }
        }
    }
}

__global__ void __launch_bounds__(kPsWarps * 32, 6)
k_grad_adjoint(const int32_t* __restrict__ seg_first, const int64_t* __restrict__ nseg_dev,
               const int32_t* __restrict__ order, const int32_t* __restrict__ pairs,
               const int32_t* __restrict__ pX, const int2* __restrict__ src,
               const int32_t* __restrict__ nfirst, const int32_t* __restrict__ ncount, int64_t n,
               const float4* __restrict__ pts, const PsPacked pk, const float* __restrict__ pg,
               const int32_t* __restrict__ perm, float sqk, float* __restrict__ gE,
               float* __restrict__ gI) {
    __shared__ PsAdjStage st[kPsWarps];
    __shared__ int2 meta[kPsWarps][32];
    __shared__ float2 red[kPsWarps][kPsList];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nseg = *nseg_dev;
    for (int64_t b = blockIdx.x; b < nseg; b += gridDim.x) {
        const int32_t sg = order[b], i0 = seg_first[sg], i1 = seg_first[sg + 1];
        const int32_t L = pX[pairs[i0]], lf = nfirst[L], lc = ncount[L];
        const float4 O = pts[lf];
        for (int32_t pos = 0; pos < lc; pos += kPsList) {
            const int np = min(lc - pos, kPsList);
            // expanded form: four paired FP32 instructions a slot, 40 bytes a
            // staged pair; the same choice in every warp
            const int R = ps_choose_r<kGrAdjR>([&](int) { return np; }, 8, 10);
            float m2 = 0.f;
            for (int k = lane; k < np; k += 32) {
                const float4 T = pts[lf + pos + k];
                const float x = (T.x - O.x) * sqk, y = (T.y - O.y) * sqk, z = (T.z - O.z) * sqk;
                m2 = fmaxf(m2, fmaf(x, x, fmaf(y, y, z * z)));
            }
            for (int o = 16; o > 0; o >>= 1) m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
            const bool fast = m2 <= kGrFastT2;
#define MSP_GR_ADJ(RR, FF)                                                                      \
    gr_adj_pass<RR, FF>(lf + pos, np, i0, i1, lf, lc, n, O, src, pts, pk, pg, sqk, st[w],       \
                        meta[w], red[w])
            if (!fast) {
                // wide leaves: few, two points a lane up to 64, else four
                if (np <= 64) MSP_GR_ADJ(2, false);
                else MSP_GR_ADJ(4, false);
            } else if (R == 1) MSP_GR_ADJ(1, true);
            else if (R == 2) MSP_GR_ADJ(2, true);
            else if (R == 3) MSP_GR_ADJ(3, true);
            else if (R == 4) MSP_GR_ADJ(4, true);
            else MSP_GR_ADJ(5, true);
#undef MSP_GR_ADJ
            __syncthreads();
            for (int k = threadIdx.x; k < np; k += kPsWarps * 32) {
                float2 v = red[0][k];
#pragma unroll
                for (int q = 1; q < kPsWarps; ++q) {
                    v.x += red[q][k].x;
                    v.y += red[q][k].y;
                }
                const int32_t c = perm[lf + pos + k];
                if (gE) gE[c] = v.x;
                if (gI) gI[c] = v.y;
            }
            __syncthreads();
        }
    }
}

}  // namespace

const int32_t* ps_offsets(msp_ctx& c, const uint16_t* fl, cudaStream_t s) {
    const int64_t n = c.n;
    DevCounts* dc = dcounts(c);
    int32_t* flag = c.gr_flag.ensure<int32_t>((size_t)2 * n + 1);
    int32_t* off = c.gr_off.ensure<int32_t>((size_t)2 * n + 1);
    k_ps_flags<<<grid_for(n, 256, (int64_t)c.sm_count * 16), 256, 0, s>>>(n, fl, flag, &dc->scan_n);
    MSP_LAUNCH("ps_flags");
    scan_dev(c, flag, off, &dc->scan_n, 2 * n + 1, nullptr, s);
    return off;
}

void attraction_grad(msp_ctx& c, const uint8_t* type, const uint8_t* va, const uint8_t* vde,
                     const uint8_t* vdi, const float* g, float* u, float* dud, float* gE,
                     float* gI, cudaStream_t s) {
    NvtxRange nv_("msp attraction_grad");
    if (!c.attraction_done) throw Error(MSP_ERR_NOT_BUILT, "msp_attraction must run first");
    if (c.n_far > 0)
        throw Error(MSP_ERR_INVALID_ARG,
                    "derivatives need a plan without translated pairs (rho_max = 0)");
    if ((gE || gI) && !g) throw Error(MSP_ERR_INVALID_ARG, "weight gradients need g");
    const int64_t n = c.n;
    if (n == 0) return;
    const msp_config& cfg = c.cfg;
    const int B = 256;
    const int G = grid_for(n, B, (int64_t)c.sm_count * 16);
    DevCounts* dc = dcounts(c);
    float2* wt = c.gr_w.ensure<float2>((size_t)n);
    uint16_t* fl = c.gr_fl.ensure<uint16_t>((size_t)n);
    const int32_t* perm = c.perm.get<int32_t>();
    k_grad_gather<<<G, B, 0, s>>>(n, perm, type, va, vde, vdi, wt, fl);
    MSP_LAUNCH("grad_gather");
    const float sqk = (float)std::sqrt(1.4426950408889634 / (cfg.sigma * cfg.sigma));
    const float dscale = (float)(2.0 / (cfg.sigma * 1.4426950408889634));
    // the segments in the near field's order (longest first) and its source
    // ranges, kept with the lists
    const int32_t *segf = c.seg_first.get<int32_t>(), *order = c.nf_oval0.get<int32_t>(),
                  *list = c.p2p_val0.get<int32_t>(), *pX = c.pr_X.get<int32_t>(),
                  *nfirst = c.nd_first.get<int32_t>(), *ncount = c.nd_count.get<int32_t>();
    const int2* src = c.nf_src.get<int2>();
    const float4* pts = c.pts.get<float4>();
    const int nb = (int)std::min<int64_t>(std::max<int64_t>(c.n_nodes, 1), 1 << 30);
    const bool adjoint = gE || gI;
    const int32_t* off = nullptr;
    float4* pt = nullptr;
    float* pg = nullptr;
    auto pack = [&] {
        off = ps_offsets(c, fl, s);
        pt = c.gr_pt.ensure<float4>((size_t)n);
        pg = c.gr_tmp.ensure<float>((size_t)n);
        k_grad_pack<<<G, B, 0, s>>>(n, fl, off, perm, pts, g, pt, pg);
        MSP_LAUNCH("grad_pack");
    };
    // an output may lie over g: g is gathered before any is written then (else
    // while the forward sums run, so that a first call's allocations overlap them)
    bool over = false;
    for (const float* o : {u, dud, gE, gI}) over |= o && adjoint && meets(o, 4 * n, g, 4 * n);
    if (over) pack();
    if (u || dud) {
        if (u) MSP_CUDA(cudaMemsetAsync(u, 0, (size_t)n * sizeof(float), s));
        if (dud) MSP_CUDA(cudaMemsetAsync(dud, 0, (size_t)n * sizeof(float), s));
        k_grad_forward<<<nb, kPsWarps * 32, 0, s>>>(segf, &dc->nseg, order, list, pX, src, nfirst,
                                                    ncount, pts, wt, fl, perm, sqk, dscale, u, dud);
        MSP_LAUNCH("grad_forward");
    }
    if (adjoint) {
        if (!over) pack();
        if (gE) MSP_CUDA(cudaMemsetAsync(gE, 0, (size_t)n * sizeof(float), s));
        if (gI) MSP_CUDA(cudaMemsetAsync(gI, 0, (size_t)n * sizeof(float), s));
        k_grad_adjoint<<<nb, kPsWarps * 32, 0, s>>>(segf, &dc->nseg, order, list, pX, src, nfirst,
                                                    ncount, n, pts, PsPacked{pt, off}, pg, perm,
                                                    sqk, gE, gI);
        MSP_LAUNCH("grad_adjoint");
    }
}

}  // namespace msp
