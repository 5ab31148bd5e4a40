// msp_length.cu -- the expected mean synapse length and its gradient, the
// loss of the differentiation workload.
//
// An axonal element of t draws dendrite s with probability w_s K(t,s) / u(t)
// (Eq. 1 with the kernel of Eq. 8, K = exp(-r^2/sigma^2); w = the continuous
// dendritic weights of t's channel), so its synapse is l(t) = v(t)/u(t) long
// on average, with
//   u(t) = sum_s w_s K,   v(t) = sum_s w_s K r.
// Over the vacant axonal elements (a_t > 0, u(t) > 0; A = sum of their a_t):
//   m = sum_t a_t l(t) / A,   loss = (m - target)^2,
//   dm/dsigma = sum_t a_t (v' u - v u') / (A u^2),  with ' = d/dsigma:
//               u' = sum w K 2 r^2 / sigma^3,  v' = sum w K r 2 r^2 / sigma^3,
//   dm/dw^T_s = sum_{t: T(t) = T} K(t,s) (alpha_t r - beta_t),
//               alpha_t = a_t / (A u), beta_t = a_t v / (A u^2),
// and every loss derivative is 2 (m - target) times m's.  The sums run over
// the near-field leaf pairs of the last attraction (a plan without
// translations: K r has no Hermite expansion), u, v and their sigma
// derivatives per target leaf, then the transposed sums per source leaf over
// its partner leaves' targets of one channel after the other (both walks in
// msp_pairsum.cuh).  Coordinates are scaled by sqk = sqrt(log2 e)/sigma
// relative to the leaf's first point, so that q = |t^ - s^|^2 gives K = 2^-q
// and r = rs sqrt(q), rs = sigma/sqrt(log2 e); rs is applied to the sums.
// A lane's sums join its running totals by Kahan's compensated summation
// after every 64 staged points (the transposed terms are signed: their partial
// sums exceed their total; a fold per 32 partner leaves raised the error of
// the weight gradients from 3.4e-7 to 4.7e-7).  The lanes' and the warps' totals are
// joined with their compensations and rounded once: joined plainly, the weight
// gradients of 3,000 to 131,072 neurons were 10 to 30 % further from 64 bits
// (20,000 in two clusters: 4.5e-7 joined plainly, 3.4e-7 so), at the same time.
// Every sum has a fixed order, so the results are reproducible; the scalar
// reductions run in double.
//
// Bound by the FP32 pipe, the special function unit (EX2 and SQRT per term)
// and instruction issue.  131,072 clustered neurons (cutoff 5 sigma, leaf
// capacity 128), against chunks of 32 with mixed channels per lane, in no order
// of length, and a list sorted anew by source leaf: forward 1.51 -> 0.82 ms
// (1.06 -> 0.60 G warp instructions), transposed 1.67 + 0.1 -> 0.64 + 0.02 ms;
// the blocks' partials by one thread cost another 0.08 ms.
#include <algorithm>
#include <cmath>

#include "msp_pairsum.cuh"

namespace msp {

namespace {

constexpr double kLog2e = 1.4426950408889634;

__device__ inline float len_sqrt(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ inline void kahan_add(float& acc, float& cmp, float v) {
    const float y = __fsub_rn(v, cmp);
    const float t = __fadd_rn(acc, y);
    cmp = __fsub_rn(__fsub_rn(t, acc), y);
    acc = t;
}

// sorted-order inputs: the weights, and the flags with a in the high byte
__global__ void k_len_gather(int64_t n, const int32_t* __restrict__ perm,
                             const uint8_t* __restrict__ type, const uint8_t* __restrict__ va,
                             const float* __restrict__ we, const float* __restrict__ wi,
                             float2* __restrict__ w, uint16_t* __restrict__ fl) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = perm[s];
        w[s] = make_float2(we[c], wi[c]);
        fl[s] = (uint16_t)((type[c] ? kPsInh : 0u) | (va[c] ? kPsAct : 0u) | ((uint32_t)va[c] << 8));
    }
}

__device__ __forceinline__ float len_count(uint16_t f) { return (float)(f >> 8); }

// A lane's running totals with their compensations, N per slot, in shared
// memory (touched once per unit; the registers are the loop's)
template <int R, int N>
struct LenTotals {
    float* p;      // this thread's entry; entries lie kPsWarps * 32 floats apart
    __device__ explicit LenTotals(float* base) : p(base + threadIdx.x) {
        for (int k = 0; k < 2 * R * N; ++k) p[k * kPsWarps * 32] = 0.f;
    }
    __device__ void add(int k, float v) const {
        float acc = p[2 * k * kPsWarps * 32], cmp = p[(2 * k + 1) * kPsWarps * 32];
        kahan_add(acc, cmp, v);
        p[2 * k * kPsWarps * 32] = acc;
        p[(2 * k + 1) * kPsWarps * 32] = cmp;
    }
    // the total over the slices of a group, in a fixed order, with what it lost
    // (Kahan's compensation is what the total gained)
    __device__ float2 get(int k, const PsLanes& ln) const {
        float h = p[2 * k * kPsWarps * 32], c = -p[(2 * k + 1) * kPsWarps * 32];
        for (int o = ln.npr; o < 32; o <<= 1)
            ff_acc(h, c, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, c, o));
        return make_float2(h, c);
    }
};

// the sum of the warps' totals get(q), rounded once
template <class Get>
__device__ __forceinline__ float len_warps(Get get) {
    float2 v = get(0);
#pragma unroll
    for (int q = 1; q < kPsWarps; ++q) {
        const float2 x = get(q);
        ff_acc(v.x, v.y, x.x, x.y);
    }
    return __fadd_rn(v.x, v.y);
}

// FORWARD: per target t with a_t > 0, over the staged sources (w: the source's
// weight of t's channel)
//   U = sum w K, V = sum w K sqrt(q), QU = sum w K q, QV = sum w K q sqrt(q)
// (V and QV in units of rs).  SELF: a source may be t itself; its
// kernel is zero.
constexpr int kLenFwdR = 3;

template <int R, bool SELF>
__device__ __forceinline__ void len_fwd_eval(const float4* sA, const float4* sW, int j0, int mp,
                                             int slices, const float2 (&tx)[R],
                                             const float2 (&ty)[R], const float2 (&tz)[R],
                                             const int32_t (&e)[R], int32_t first, int32_t second,
                                             float2 (&p)[R][4]) {
    for (int j = j0; j < mp; j += slices) {
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
            const float2 wr = __fmul2_rn(wk, make_float2(len_sqrt(q.x), len_sqrt(q.y)));
            p[r][0] = __fadd2_rn(p[r][0], wk);
            p[r][1] = __fadd2_rn(p[r][1], wr);
            p[r][2] = __ffma2_rn(wk, q, p[r][2]);
            p[r][3] = __ffma2_rn(wr, q, p[r][3]);
        }
    }
}

template <int R>
__device__ __forceinline__ void len_fwd_pass(const int32_t* list, int np, int32_t i0, int32_t i1,
                                             int32_t lf, int32_t lc, const float4& O,
                                             const int2* __restrict__ src,
                                             const float4* __restrict__ pts,
                                             const float2* __restrict__ wt,
                                             const uint16_t* __restrict__ fl, float sqk,
                                             PsFwdStage& st, int2* meta, float* totals,
                                             float2 (*red)[4]) {
    const int lane = threadIdx.x & 31;
    const PsLanes ln(np, R);
    const LenTotals<R, 4> tot(totals);
    float2 tx[R], ty[R], tz[R], p[R][4];
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
#pragma unroll
        for (int k = 0; k < 4; ++k) p[r][k] = make_float2(0.f, 0.f);
    }
    auto fold = [&] {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tot.add(4 * r + k, __fadd_rn(p[r][k].x, p[r][k].y));
                p[r][k] = make_float2(0.f, 0.f);
            }
    };
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
            // a fold per unit of 64 sources
            len_fwd_eval<R, false>(st.A, sW, ln.ksl, min(mp, kPsUnit / 2), ln.slices, tx, ty, tz, e,
                                   0, 0, p);
            fold();
            if (mp > kPsUnit / 2) {
                len_fwd_eval<R, false>(st.A, sW, kPsUnit / 2 + ln.ksl, mp, ln.slices, tx, ty, tz, e,
                                       0, 0, p);
                fold();
            }
        });
    // L's own points, where a target skips itself
    if (__any_sync(0xffffffffu, self)) {
        for (int32_t q = 0; q < lc; q += kPsUnit) {
            const int left = min(lc - q, kPsUnit), half = (left + 1) >> 1;
            __syncwarp();
            if (lane < half)
                ps_stage_fwd(st, pts, wt, lf + q + lane, lf + q + half + lane, lane < left - half,
                             lane, O, sqk);
            __syncwarp();
            len_fwd_eval<R, true>(st.A, sW, ln.ksl, half, ln.slices, tx, ty, tz, e, lf + q,
                                  lf + q + half, p);
            fold();
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 v = tot.get(4 * r + k, ln);
            if (ln.ksl == 0 && R * ln.j + r < np) red[R * ln.j + r][k] = v;
        }
    }
}

__global__ void __launch_bounds__(kPsWarps * 32, 5)
k_len_forward(const int32_t* __restrict__ seg_first, const int64_t* __restrict__ nseg_dev,
              const int32_t* __restrict__ order, const int32_t* __restrict__ pairs,
              const int32_t* __restrict__ pX, const int2* __restrict__ src,
              const int32_t* __restrict__ nfirst, const int32_t* __restrict__ ncount,
              const float4* __restrict__ pts, const float2* __restrict__ wt,
              const uint16_t* __restrict__ fl, float sqk, float4* __restrict__ sums) {
    __shared__ PsFwdStage st[kPsWarps];
    __shared__ int2 meta[kPsWarps][32];
    __shared__ float totals[2 * kLenFwdR * 4 * kPsWarps * 32];
    __shared__ float2 red[kPsWarps][32 * kLenFwdR][4];     // totals and what they lost
    __shared__ int32_t list[kPsList];
    __shared__ int s_np, s_pos, s_R;
    const int w = threadIdx.x >> 5;
    const int64_t nseg = *nseg_dev;
    for (int64_t b = blockIdx.x; b < nseg; b += gridDim.x) {
        const int32_t sg = order[b], i0 = seg_first[sg], i1 = seg_first[sg + 1];
        const int32_t L = pX[pairs[i0]], lf = nfirst[L], lc = ncount[L];
        const float4 O = pts[lf];
        for (int32_t pos = 0; pos < lc;) {
            // twelve paired FP32 instructions a slot, two 16-byte loads a pair
            if (w == 0)
                ps_list_targets<kLenFwdR>(fl, lf, lc, pos, 32 * kLenFwdR - kLenFwdR + 1, 24, 8,
                                          list, &s_np, &s_pos, &s_R);
            __syncthreads();
            const int np = s_np, R = s_R;
            pos = s_pos;
            if (np > 0) {
#define MSP_LEN_FWD(RR)                                                                        \
    len_fwd_pass<RR>(list, np, i0, i1, lf, lc, O, src, pts, wt, fl, sqk, st[w], meta[w], totals, \
                     red[w])
                if (R == 1) MSP_LEN_FWD(1);
                else if (R == 2) MSP_LEN_FWD(2);
                else MSP_LEN_FWD(3);
#undef MSP_LEN_FWD
            }
            __syncthreads();
            for (int k = threadIdx.x; k < 4 * np; k += kPsWarps * 32)
                if (list[k >> 2] >= 0)
                    reinterpret_cast<float*>(sums + list[k >> 2])[k & 3] =
                        len_warps([&](int q) { return red[q][k >> 2][k & 3]; });
            __syncthreads();
        }
    }
}

// TRANSPOSED: for every point s of the block's leaf and each channel T,
//   G_T = sum_{t: T(t) = T} K (alpha_t r - beta_t)
// over the partner leaves' targets of the channel, staged as A = (-x0, -x1,
// -y0, -y1), B = (-z0, -z1, alpha0, alpha1), C = (-beta0, -beta1) (alpha times
// rs), D = the sorted indices.
constexpr int kLenAdjR = 4;

template <int R, bool SELF>
__device__ __forceinline__ void len_adj_eval(const PsAdjStage& st, int j0, int mp, int slices,
                                             const float2 (&tx)[R], const float2 (&ty)[R],
                                             const float2 (&tz)[R], const int32_t (&e)[R],
                                             float2 (&p)[R]) {
    for (int j = j0; j < mp; j += slices) {
        const float4 A = st.A[j], B = st.B[j];
        const float2 C = st.C[j];
        const int2 D = SELF ? st.D[j] : make_int2(0, 0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 dx = __fadd2_rn(tx[r], make_float2(A.x, A.y));
            const float2 dy = __fadd2_rn(ty[r], make_float2(A.z, A.w));
            const float2 dz = __fadd2_rn(tz[r], make_float2(B.x, B.y));
            const float2 q = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            float2 K = make_float2(ps_ex2(-q.x), ps_ex2(-q.y));
            if (SELF) {
                K.x = D.x == e[r] ? 0.f : K.x;
                K.y = D.y == e[r] ? 0.f : K.y;
            }
            const float2 f =
                __ffma2_rn(make_float2(B.z, B.w), make_float2(len_sqrt(q.x), len_sqrt(q.y)), C);
            p[r] = __ffma2_rn(K, f, p[r]);
        }
    }
}

template <int R>
__device__ __forceinline__ void len_adj_pass(int32_t first, int np, int32_t i0, int32_t i1,
                                             int32_t lf, int32_t lc, int64_t n, const float4& O,
                                             const int2* __restrict__ src,
                                             const float4* __restrict__ pts, const PsPacked pk,
                                             const float2* __restrict__ cf, float sqk,
                                             PsAdjStage& st, int2* meta, float* totals,
                                             float2 (*red)[2]) {
    const int lane = threadIdx.x & 31;
    const PsLanes ln(np, R);
    const LenTotals<R, 2> tot(totals);
    float2 tx[R], ty[R], tz[R], p[R];
    int32_t e[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int slot = R * ln.j + r;
        e[r] = first + (slot < np ? slot : 0);
        const float4 T = pts[e[r]];
        const float x = (T.x - O.x) * sqk, y = (T.y - O.y) * sqk, z = (T.z - O.z) * sqk;
        tx[r] = make_float2(x, x);
        ty[r] = make_float2(y, y);
        tz[r] = make_float2(z, z);
        p[r] = make_float2(0.f, 0.f);
    }
    auto stage = [&](int32_t a, int32_t b, bool two, int slot) {
        const float4 S0 = pk.pt[a], S1 = pk.pt[two ? b : a];
        const float2 c0 = cf[a], c1 = two ? cf[b] : make_float2(0.f, 0.f);
        const float2 k = make_float2(sqk, sqk);
        const float2 x = __fmul2_rn(__fadd2_rn(make_float2(O.x, O.x), make_float2(-S0.x, -S1.x)), k);
        const float2 y = __fmul2_rn(__fadd2_rn(make_float2(O.y, O.y), make_float2(-S0.y, -S1.y)), k);
        const float2 z = __fmul2_rn(__fadd2_rn(make_float2(O.z, O.z), make_float2(-S0.z, -S1.z)), k);
        st.A[slot] = make_float4(x.x, x.y, y.x, y.y);
        st.B[slot] = make_float4(z.x, z.y, c0.x, c1.x);
        st.C[slot] = make_float2(c0.y, c1.y);
        st.D[slot] = make_int2(__float_as_int(S0.w), two ? __float_as_int(S1.w) : -1);
    };
#pragma unroll 1
    for (int ch = 0; ch < 2; ++ch) {
        const int32_t* off = pk.off + ch * n;
        auto fold = [&] {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                tot.add(2 * r + ch, __fadd_rn(p[r].x, p[r].y));
                p[r] = make_float2(0.f, 0.f);
            }
        };
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
                // a fold per unit of 64 targets
                len_adj_eval<R, false>(st, ln.ksl, min(mp, kPsUnit / 2), ln.slices, tx, ty, tz, e, p);
                fold();
                if (mp > kPsUnit / 2) {
                    len_adj_eval<R, false>(st, kPsUnit / 2 + ln.ksl, mp, ln.slices, tx, ty, tz, e,
                                           p);
                    fold();
                }
            });
        // L's own targets, where a point skips itself
        if (__any_sync(0xffffffffu, self)) {
            const int32_t a0 = off[lf], a1 = off[lf + lc];
            for (int32_t q = a0; q < a1; q += kPsUnit) {
                const int left = min(a1 - q, kPsUnit), half = (left + 1) >> 1;
                __syncwarp();
                if (lane < half) stage(q + lane, q + half + lane, lane < left - half, lane);
                __syncwarp();
                len_adj_eval<R, true>(st, ln.ksl, half, ln.slices, tx, ty, tz, e, p);
                fold();
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
            const float2 v = tot.get(2 * r + ch, ln);
            if (ln.ksl == 0 && R * ln.j + r < np) red[R * ln.j + r][ch] = v;
        }
    }
}

__global__ void __launch_bounds__(kPsWarps * 32, 6)
k_len_adjoint(const int32_t* __restrict__ seg_first, const int64_t* __restrict__ nseg_dev,
              const int32_t* __restrict__ order, const int32_t* __restrict__ pairs,
              const int32_t* __restrict__ pX, const int2* __restrict__ src,
              const int32_t* __restrict__ nfirst, const int32_t* __restrict__ ncount, int64_t n,
              const float4* __restrict__ pts, const PsPacked pk, const float2* __restrict__ cf,
              const int32_t* __restrict__ perm, float sqk, float* __restrict__ gE,
              float* __restrict__ gI) {
    __shared__ PsAdjStage st[kPsWarps];
    __shared__ int2 meta[kPsWarps][32];
    __shared__ float totals[2 * kLenAdjR * 2 * kPsWarps * 32];
    __shared__ float2 red[kPsWarps][kPsList][2];           // totals and what they lost
    const int w = threadIdx.x >> 5;
    const int64_t nseg = *nseg_dev;
    for (int64_t b = blockIdx.x; b < nseg; b += gridDim.x) {
        const int32_t sg = order[b], i0 = seg_first[sg], i1 = seg_first[sg + 1];
        const int32_t L = pX[pairs[i0]], lf = nfirst[L], lc = ncount[L];
        const float4 O = pts[lf];
        for (int32_t pos = 0; pos < lc; pos += kPsList) {
            const int np = min(lc - pos, kPsList);
            // EX2 and SQRT for two sources a slot (the special function unit's
            // 17 quarter cycles), 40 bytes a staged pair
            const int R = ps_choose_r<kLenAdjR>([&](int) { return np; }, 17, 10);
#define MSP_LEN_ADJ(RR)                                                                        \
    len_adj_pass<RR>(lf + pos, np, i0, i1, lf, lc, n, O, src, pts, pk, cf, sqk, st[w], meta[w], \
                     totals, red[w])
            if (R == 1) MSP_LEN_ADJ(1);
            else if (R == 2) MSP_LEN_ADJ(2);
            else if (R == 3) MSP_LEN_ADJ(3);
            else MSP_LEN_ADJ(4);
#undef MSP_LEN_ADJ
            __syncthreads();
            for (int k = threadIdx.x; k < np; k += kPsWarps * 32) {
                const int32_t c = perm[lf + pos + k];
                if (gE) gE[c] = len_warps([&](int q) { return red[q][k][0]; });
                if (gI) gI[c] = len_warps([&](int q) { return red[q][k][1]; });
            }
            __syncthreads();
        }
    }
}

constexpr int kLenRedThreads = 256;

// per block: the partial sums A = sum a, S = sum a V/U, D = sum a (V'U - VU')/U^2
// over the targets it takes (a > 0, U > 0), in double, reduced in a fixed
// order; V' / U' are QV / QU times dscale = 2 / (sigma log2 e)
__global__ void __launch_bounds__(kLenRedThreads)
k_len_reduce(int64_t n, const uint16_t* __restrict__ fl, const float4* __restrict__ sums,
             double rs, double dscale, double* __restrict__ part) {
    __shared__ double red[3][kLenRedThreads];
    double A = 0.0, S = 0.0, D = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const float a = len_count(fl[t]);
        if (!(a > 0.f)) continue;
        const float4 s4 = sums[t];
        const double U = s4.x, V = rs * s4.y;
        if (!(U > 0.0)) continue;
        const double dU = dscale * s4.z, dV = dscale * rs * s4.w;
        A += a;
        S += a * V / U;
        D += a * (dV * U - V * dU) / (U * U);
    }
    red[0][threadIdx.x] = A;
    red[1][threadIdx.x] = S;
    red[2][threadIdx.x] = D;
    __syncthreads();
    for (int o = kLenRedThreads / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 3; ++k) part[3 * blockIdx.x + k] = red[k][0];
}

// the blocks' partials, added in a fixed order by one block; res = {loss, m,
// dloss/dsigma, dm/dsigma, A, f}
__global__ void __launch_bounds__(kLenRedThreads)
k_len_final(const double* __restrict__ part, int nblocks, double target, double* __restrict__ res) {
    __shared__ double red[3][kLenRedThreads];
    double v[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += kLenRedThreads)
        for (int k = 0; k < 3; ++k) v[k] += part[3 * b + k];
    for (int k = 0; k < 3; ++k) red[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int o = kLenRedThreads / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x) return;
    const double A = red[0][0], S = red[1][0], D = red[2][0];
    const double m = A > 0.0 ? S / A : 0.0;
    const double dm = A > 0.0 ? D / A : 0.0;
    const double f = 2.0 * (m - target);
    res[0] = (m - target) * (m - target);
    res[1] = m;
    res[2] = f * dm;
    res[3] = dm;
    res[4] = A;
    res[5] = f;
}

// the packed targets: point, and (f alpha_t rs, -f beta_t), f = 2 (m - target)
__global__ void k_len_pack(int64_t n, const uint16_t* __restrict__ fl,
                           const int32_t* __restrict__ off, const float4* __restrict__ pts,
                           const float4* __restrict__ sums, const double* __restrict__ res,
                           double rs, float4* __restrict__ pt, float2* __restrict__ cf) {
    const double A = res[4], f = res[5];
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t fw = fl[t];
        if (!(fw & kPsAct)) continue;
        const float a = len_count((uint16_t)fw);
        const float4 s4 = sums[t];
        const double U = s4.x, V = rs * s4.y;
        float2 c = make_float2(0.f, 0.f);
        if (U > 0.0 && A > 0.0)
            c = make_float2((float)(rs * (f * a / (A * U))), (float)(-(f * a * V / (A * U * U))));
        const int32_t k = off[((fw & kPsInh) ? n : 0) + t];
        const float4 P = pts[t];
        pt[k] = make_float4(P.x, P.y, P.z, __int_as_float((int32_t)t));
        cf[k] = c;
    }
}

}  // namespace

void length_loss(msp_ctx& c, const uint8_t* type, const uint8_t* va, const float* we,
                 const float* wi, double target, double* out4, float* gE, float* gI,
                 cudaStream_t s) {
    NvtxRange nv_("msp length_loss");
    if (!c.attraction_done) throw Error(MSP_ERR_NOT_BUILT, "msp_attraction must run first");
    if (c.n_far > 0)
        throw Error(MSP_ERR_INVALID_ARG,
                    "the synapse length needs a plan without translated pairs (rho_max = 0)");
    const int64_t n = c.n;
    for (int k = 0; k < 4; ++k) out4[k] = 0.0;
    if (n == 0) return;
    const msp_config& cfg = c.cfg;
    const int B = 256;
    const int G = grid_for(n, B, (int64_t)c.sm_count * 16);
    DevCounts* dc = dcounts(c);
    float2* wt = c.gr_w.ensure<float2>((size_t)n);
    uint16_t* fl = c.gr_fl.ensure<uint16_t>((size_t)n);
    const int32_t* perm = c.perm.get<int32_t>();
    k_len_gather<<<G, B, 0, s>>>(n, perm, type, va, we, wi, wt, fl);
    MSP_LAUNCH("len_gather");
    const float sqk = (float)std::sqrt(kLog2e / (cfg.sigma * cfg.sigma));
    const double rs = cfg.sigma / std::sqrt(kLog2e);
    const double dscale = 2.0 / (cfg.sigma * kLog2e);
    // the segments in the near field's order (longest first) and its source
    // ranges, kept with the lists
    const int32_t *segf = c.seg_first.get<int32_t>(), *order = c.nf_oval0.get<int32_t>(),
                  *list = c.p2p_val0.get<int32_t>(), *pX = c.pr_X.get<int32_t>(),
                  *nfirst = c.nd_first.get<int32_t>(), *ncount = c.nd_count.get<int32_t>();
    const int2* src = c.nf_src.get<int2>();
    const float4* pts = c.pts.get<float4>();
    const int nb = (int)std::min<int64_t>(std::max<int64_t>(c.n_nodes, 1), 1 << 30);
    float4* sums = c.ln_sums.ensure<float4>((size_t)n);
    MSP_CUDA(cudaMemsetAsync(sums, 0, (size_t)n * sizeof(float4), s));
    k_len_forward<<<nb, kPsWarps * 32, 0, s>>>(segf, &dc->nseg, order, list, pX, src, nfirst, ncount,
                                               pts, wt, fl, sqk, sums);
    MSP_LAUNCH("len_forward");
    const int Gr = (int)std::min<int64_t>(grid_for(n, kLenRedThreads), (int64_t)c.sm_count * 4);
    double* part = c.ln_part.ensure<double>((size_t)3 * Gr + 8);
    k_len_reduce<<<Gr, kLenRedThreads, 0, s>>>(n, fl, sums, rs, dscale, part);
    MSP_LAUNCH("len_reduce");
    double* res = part + 3 * Gr;
    k_len_final<<<1, kLenRedThreads, 0, s>>>(part, Gr, target, res);
    MSP_LAUNCH("len_final");
    if (gE || gI) {
        if (gE) MSP_CUDA(cudaMemsetAsync(gE, 0, (size_t)n * sizeof(float), s));
        if (gI) MSP_CUDA(cudaMemsetAsync(gI, 0, (size_t)n * sizeof(float), s));
        const int32_t* off = ps_offsets(c, fl, s);
        float4* pt = c.gr_pt.ensure<float4>((size_t)n);
        float2* cf = c.ln_coef.ensure<float2>((size_t)n);
        k_len_pack<<<G, B, 0, s>>>(n, fl, off, pts, sums, res, rs, pt, cf);
        MSP_LAUNCH("len_pack");
        k_len_adjoint<<<nb, kPsWarps * 32, 0, s>>>(segf, &dc->nseg, order, list, pX, src, nfirst,
                                                   ncount, n, pts, PsPacked{pt, off}, cf, perm, sqk,
                                                   gE, gI);
        MSP_LAUNCH("len_adjoint");
    }
    MSP_CUDA(cudaMemcpyAsync(out4, res, 4 * sizeof(double), cudaMemcpyDeviceToHost, s));
    MSP_CUDA(cudaStreamSynchronize(s));
}

}  // namespace msp
