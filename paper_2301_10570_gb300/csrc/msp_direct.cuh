// msp_direct.cuh -- the all-pairs attraction (Eq. 8 over every neuron): the
// device code shared by msp_direct (a context's sorted copy) and
// msp_direct_noalloc (the caller's arrays, fixed scratch).
//
// Every term is w exp2(-k2 |t - s|^2), the distance formed from the unscaled
// single precision positions (a difference of near positions is exact, scaled
// coordinates would not be).  What bounds it is the FP32 pipe: eight paired
// FP32 instructions and two EX2 per two terms, 16 terms per SM and clock at
// 128 FP32 lanes.  Two sources sit in one staged pair, so that each term runs
// as one half of a paired instruction, and a lane holds R targets, so that the
// two 16-byte shared loads of a staged pair serve 2 R terms.
//
// Terms that single precision evaluates to exactly zero are left out: EX2 of
// an argument below -126 flushes to zero, so a tile of sources whose bounding
// box is farther from the targets' box than k2 d^2 = kDirZero (with a margin
// for the rounding of d^2) adds nothing, bit for bit.  Of the tile pairs of
// 131,072 neurons in 8 clusters 17 % remain.  Measured there: 9.08 ms with one
// target per lane, scalar FP32 and every pair evaluated, 1.00 ms now.
#pragma once

#include "msp_hostdev.cuh"
#include "msp_internal.cuh"

namespace msp {

constexpr float kDirZero = 127.f;
constexpr int kDirTile = 128;          // sources per staged tile
constexpr int kDirListPts = 1024;      // neurons per block of the target lists

__device__ __forceinline__ float dir_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// neuron i as {x, y, z, packed bytes}: the sorted copy, or the caller's arrays
struct DirPacked {
    const float4* __restrict__ pts;
    __device__ float4 get(int64_t i) const { return pts[i]; }
};
struct DirRaw {
    const float *__restrict__ x, *__restrict__ y, *__restrict__ z;
    const uint8_t *__restrict__ type, *__restrict__ va, *__restrict__ vde, *__restrict__ vdi;
    __device__ float4 get(int64_t i) const {
        const uint32_t w = (uint32_t)(type[i] ? 1u : 0u) | ((uint32_t)va[i] << 8) |
                           ((uint32_t)vde[i] << 16) | ((uint32_t)vdi[i] << 24);
        return make_float4(x[i], y[i], z[i], __uint_as_float(w));
    }
};

// one staged pair of sources, A = (-x0, -x1, -y0, -y1), B = (-z0, -z1, w0, w1),
// against one target: the weighted kernels of both are added to acc
template <bool MASK>
__device__ __forceinline__ void dir_term(const float4& A, const float4& B, float2 tx, float2 ty,
                                         float2 tz, float2 mk2, bool keep0, bool keep1,
                                         float2& acc) {
    const float2 dx = __fadd2_rn(tx, make_float2(A.x, A.y));
    const float2 dy = __fadd2_rn(ty, make_float2(A.z, A.w));
    const float2 dz = __fadd2_rn(tz, make_float2(B.x, B.y));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    const float2 E = __fmul2_rn(r2, mk2);
    float2 w = make_float2(B.z, B.w);
    if (MASK) {
        w.x = keep0 ? w.x : 0.f;
        w.y = keep1 ? w.y : 0.f;
    }
    acc = __ffma2_rn(w, make_float2(dir_ex2(E.x), dir_ex2(E.y)), acc);
}

// Kahan's compensated addition of a tile's sum
__device__ __forceinline__ void dir_kahan(float& acc, float& comp, float v) {
    const float y = __fsub_rn(v, comp);
    const float t = __fadd_rn(acc, y);
    comp = __fsub_rn(__fsub_rn(t, acc), y);
    acc = t;
}

// Up to kDirSmallN neurons: a block takes 32 consecutive targets, one per
// lane, and its 32 warps take tiles of 32 sources round-robin, so that a few
// hundred targets still give thousands of warps; one launch, no lists.  FR: a
// target takes only the sources of its own network (the cell in the keys' top
// bits).
constexpr int kDirSmallN = 8192;
constexpr int kDirSmallWarps = 32;

template <bool FR, class Src>
__global__ void __launch_bounds__(kDirSmallWarps * 32, 1)
k_dir_small(int64_t n, Src src, float k2, const uint64_t* __restrict__ keys, int fsh,
            const int32_t* __restrict__ perm, float* __restrict__ u) {
    __shared__ float4 sA[kDirSmallWarps][16], sB[kDirSmallWarps][2][17];
    __shared__ float red[kDirSmallWarps][33];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * 32 + lane;
    const float4 T = src.get(t < n ? t : n - 1);
    const uint32_t tw = __float_as_uint(T.w);
    const int ch = pk_type(tw) ? 1 : 0;
    const uint32_t tcell = FR ? (uint32_t)(keys[t < n ? t : n - 1] >> fsh) : 0u;
    const float2 tx = make_float2(T.x, T.x), ty = make_float2(T.y, T.y), tz = make_float2(T.z, T.z);
    const float2 mk2 = make_float2(-k2, -k2);
    float* fA = reinterpret_cast<float*>(sA[w]);
    float* fE = reinterpret_cast<float*>(sB[w][0]);
    float* fI = reinterpret_cast<float*>(sB[w][1]);
    const int jj = lane >> 1, h = lane & 1;
    float acc = 0.f, comp = 0.f;
    for (int64_t s0 = 32 * w; s0 < n; s0 += 32 * kDirSmallWarps) {
        const int64_t s = s0 + lane;
        const bool in = s < n;
        float4 S = make_float4(3e30f, 3e30f, 3e30f, 0.f);
        if (in) S = src.get(s);
        const uint32_t sw = __float_as_uint(S.w);
        const uint32_t scell = FR && in ? (uint32_t)(keys[s] >> fsh) : 0xffffffffu;
        __syncwarp();
        fA[4 * jj + h] = -S.x;
        fA[4 * jj + 2 + h] = -S.y;
        fE[4 * jj + h] = -S.z;
        fI[4 * jj + h] = -S.z;
        fE[4 * jj + 2 + h] = (float)pk_de(sw);
        fI[4 * jj + 2 + h] = (float)pk_di(sw);
        __syncwarp();
        const float4* B = sB[w][ch];
        float2 p = make_float2(0.f, 0.f);
        const bool own = s0 < (int64_t)blockIdx.x * 32 + 32 && s0 + 32 > (int64_t)blockIdx.x * 32;
        if (!FR && !own) {
#pragma unroll
            for (int j = 0; j < 16; ++j) dir_term<false>(sA[w][j], B[j], tx, ty, tz, mk2, true, true, p);
        } else {
#pragma unroll 4
            for (int j = 0; j < 16; ++j) {
                bool k0 = s0 + 2 * j != t, k1 = s0 + 2 * j + 1 != t;
                if (FR) {
                    k0 = k0 && __shfl_sync(0xffffffffu, scell, 2 * j) == tcell;
                    k1 = k1 && __shfl_sync(0xffffffffu, scell, 2 * j + 1) == tcell;
                }
                dir_term<true>(sA[w][j], B[j], tx, ty, tz, mk2, k0, k1, p);
            }
        }
        dir_kahan(acc, comp, __fadd_rn(p.x, p.y));
    }
    red[w][lane] = __fsub_rn(acc, comp);
    __syncthreads();
    // warp w sums target w over the warps: lane l holds warp l's part
    const int64_t tt = (int64_t)blockIdx.x * 32 + w;
    float v = red[lane][w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && tt < n) {
        const float4 P = src.get(tt);
        u[perm ? perm[tt] : tt] = pk_axon(__float_as_uint(P.w)) > 0 ? v : 0.f;
    }
}

// The target lists: excitatory targets in order from list[0] up, inhibitory
// ones from list[n - 1] down (in order, so that the targets of a block lie
// close together and few tiles are in reach of their box).  First the numbers
// of each block's targets per channel (bcnt), u = 0 for the neurons without
// vacant axons, the bounding box of every kDirTile neurons (six floats; the
// whole space if a coordinate is not finite, so that such a tile is always
// evaluated) and, with copy, the packed copy.
__device__ __forceinline__ void dir_classes(int64_t i, int64_t n, float4 P, bool& e, bool& h) {
    const uint32_t pw = __float_as_uint(P.w);
    const bool act = i < n && pk_axon(pw) > 0, inh = pk_type(pw) != 0;
    e = act && !inh;
    h = act && inh;
}

template <class Src>
__global__ void __launch_bounds__(256)
k_dir_count(int64_t n, Src src, float4* __restrict__ copy, const int32_t* __restrict__ perm,
            int32_t* __restrict__ bcnt, float* __restrict__ bounds, float* __restrict__ u) {
    __shared__ int s_cnt[2][8];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // warp w takes the 128 neurons (one tile) from base on, 32 at a time
    const int64_t base = (int64_t)blockIdx.x * kDirListPts + w * kDirTile;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    int nE = 0, nI = 0;
    bool odd = false;
#pragma unroll
    for (int r = 0; r < kDirTile / 32; ++r) {
        const int64_t i = base + 32 * r + lane;
        bool e = false, h = false;
        if (i < n) {
            const float4 P = src.get(i);
            dir_classes(i, n, P, e, h);
            if (copy) copy[i] = P;
            if (!e && !h) u[perm ? perm[i] : i] = 0.f;
            const float v[3] = {P.x, P.y, P.z};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                odd |= !(fabsf(v[d]) < INFINITY);
                lo[d] = fminf(lo[d], v[d]);
                hi[d] = fmaxf(hi[d], v[d]);
            }
        }
        nE += __popc(__ballot_sync(0xffffffffu, e));
        nI += __popc(__ballot_sync(0xffffffffu, h));
    }
    odd = __any_sync(0xffffffffu, odd);
#pragma unroll
    for (int d = 0; d < 3; ++d)
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    if (lane < 6 && base < n) {
        const float b = lane < 3 ? (lane == 0 ? lo[0] : (lane == 1 ? lo[1] : lo[2]))
                                 : (lane == 3 ? hi[0] : (lane == 4 ? hi[1] : hi[2]));
        bounds[6 * (base / kDirTile) + lane] = odd ? (lane < 3 ? -INFINITY : INFINITY) : b;
    }
    if (lane == 0) {
        s_cnt[0][w] = nE;
        s_cnt[1][w] = nI;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        int t = 0;
        for (int k = 0; k < 8; ++k) t += s_cnt[threadIdx.x][k];
        bcnt[2 * blockIdx.x + threadIdx.x] = t;
    }
}

// then the entries: a block adds up the counts of the blocks before it; the
// last one writes the totals
template <class Src>
__global__ void __launch_bounds__(256)
k_dir_lists(int64_t n, Src src, const int32_t* __restrict__ bcnt, int32_t* __restrict__ list,
            int32_t* __restrict__ cnt) {
    __shared__ int s_cnt[2][32], s_part[2][8];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = (int64_t)blockIdx.x * kDirListPts + w * kDirTile;
    int pE = 0, pI = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += 256) {
        pE += bcnt[2 * k];
        pI += bcnt[2 * k + 1];
    }
    pE = __reduce_add_sync(0xffffffffu, pE);
    pI = __reduce_add_sync(0xffffffffu, pI);
    if (lane == 0) {
        s_part[0][w] = pE;
        s_part[1][w] = pI;
    }
    unsigned mE[kDirTile / 32], mI[kDirTile / 32];
#pragma unroll
    for (int r = 0; r < kDirTile / 32; ++r) {
        const int64_t i = base + 32 * r + lane;
        bool e = false, h = false;
        if (i < n) dir_classes(i, n, src.get(i), e, h);
        mE[r] = __ballot_sync(0xffffffffu, e);
        mI[r] = __ballot_sync(0xffffffffu, h);
        if (lane == 0) {
            s_cnt[0][4 * w + r] = __popc(mE[r]);
            s_cnt[1][4 * w + r] = __popc(mI[r]);
        }
    }
    __syncthreads();
    // exclusive offsets of the block's 32 groups of 32, one warp per channel
    if (w < 2) {
        int before = lane < 8 ? s_part[w][lane] : 0;
        before = __reduce_add_sync(0xffffffffu, before);
        const int c = s_cnt[w][lane];
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        s_cnt[w][lane] = before + inc - c;
        if (lane == 31 && blockIdx.x == gridDim.x - 1) cnt[w] = before + inc;
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kDirTile / 32; ++r) {
        const int32_t i = (int32_t)(base + 32 * r + lane);
        if ((mE[r] >> lane) & 1u) list[s_cnt[0][4 * w + r] + __popc(mE[r] & lt)] = i;
        if ((mI[r] >> lane) & 1u) list[n - 1 - (s_cnt[1][4 * w + r] + __popc(mI[r] & lt))] = i;
    }
}

// The squared gap of two bounding boxes {lo, hi}
__device__ __forceinline__ float dir_gap2(const float (&lo)[3], const float (&hi)[3],
                                          const float* __restrict__ b) {
    float g2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float g = fmaxf(fmaxf(b[d] - hi[d], lo[d] - b[3 + d]), 0.f);
        g2 = fmaf(g, g, g2);
    }
    return g2;
}

// A block takes 32 R targets of one channel from the lists, R per lane; its NW
// warps hold the same targets and take the source tiles round-robin (tile k:
// warp k mod NW), each staging its tile in its own shared memory; a tile's sum
// joins the lane's total by Kahan's summation and the warps' totals are added
// in order, so u does not depend on which targets share a block.  MASK
// evaluation: tiles that hold one of the targets, and with FR tiles of several
// networks or of another network than some target's.
template <int R, int NW, bool FR>
__global__ void __launch_bounds__(NW * 32, R == 4 && !FR ? 3 : 2)
k_dir_tiles(int64_t n, const float4* __restrict__ pts, const int32_t* __restrict__ list,
            const int32_t* __restrict__ cnt, const float* __restrict__ bounds, float k2,
            const uint64_t* __restrict__ keys, int fsh, const int32_t* __restrict__ perm,
            float* __restrict__ u) {
    constexpr int kT = 32 * R;
    __shared__ float4 sA[NW][kDirTile / 2], sB[NW][kDirTile / 2];
    __shared__ uint32_t sc[FR ? NW : 1][FR ? kDirTile : 1];
    __shared__ float red[NW][kT];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nE = cnt[0], nI = cnt[1];
    // the inhibitory targets first: fewer, so their boxes are wider and their
    // blocks longer
    const int bI = (nI + kT - 1) / kT;
    const int ch = (int)blockIdx.x < bI ? 1 : 0;
    const int first = ((int)blockIdx.x - (ch ? 0 : bI)) * kT;
    const int m = min((ch ? nI : nE) - first, kT);      // targets of the block
    if (m <= 0) return;
    int32_t tq[R];
    float2 tx[R], ty[R], tz[R];
    uint32_t tcell[R];
    float acc[R], comp[R];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    int32_t tmin = 0x7fffffff, tmax = -1;
    uint32_t cmin = 0xffffffffu, cmax = 0u;
    bool odd = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // slots past the end repeat the block's first target (not written)
        const int slot = 32 * r + lane;
        const int k = first + (slot < m ? slot : 0);
        tq[r] = ch ? list[n - 1 - k] : list[k];
        const float4 T = pts[tq[r]];
        tx[r] = make_float2(T.x, T.x);
        ty[r] = make_float2(T.y, T.y);
        tz[r] = make_float2(T.z, T.z);
        acc[r] = comp[r] = 0.f;
        tcell[r] = FR ? (uint32_t)(keys[tq[r]] >> fsh) : 0u;
        cmin = min(cmin, tcell[r]);
        cmax = max(cmax, tcell[r]);
        tmin = min(tmin, tq[r]);
        tmax = max(tmax, tq[r]);
        const float v[3] = {T.x, T.y, T.z};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            odd |= !(fabsf(v[d]) < INFINITY);
            lo[d] = fminf(lo[d], v[d]);
            hi[d] = fmaxf(hi[d], v[d]);
        }
    }
    odd = __any_sync(0xffffffffu, odd);
    tmin = __reduce_min_sync(0xffffffffu, tmin);
    tmax = __reduce_max_sync(0xffffffffu, tmax);
    cmin = __reduce_min_sync(0xffffffffu, cmin);
    cmax = __reduce_max_sync(0xffffffffu, cmax);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
        if (odd) {
            lo[d] = -INFINITY;
            hi[d] = INFINITY;
        }
    }
    const float2 mk2 = make_float2(-k2, -k2);
    float* fA = reinterpret_cast<float*>(sA[w]);
    float* fB = reinterpret_cast<float*>(sB[w]);
    const int ntile = (int)((n + kDirTile - 1) / kDirTile);
    for (int c0 = w; c0 < ntile; c0 += 32 * NW) {
        // the warp's next 32 tiles, one per lane: which of them to evaluate
        const int ck = c0 + NW * lane;
        bool need = ck < ntile;
        bool mask = false;
        if (need) {
            need = !(dir_gap2(lo, hi, bounds + 6 * (int64_t)ck) * k2 > kDirZero);
            const int32_t i0 = ck * kDirTile, i1 = (int32_t)min((int64_t)i0 + kDirTile, n) - 1;
            mask = i0 <= tmax && i1 >= tmin;
            if (FR && need) {
                const uint32_t a = (uint32_t)(keys[i0] >> fsh), b = (uint32_t)(keys[i1] >> fsh);
                need = a <= cmax && b >= cmin;
                mask |= !(a == b && cmin == cmax && a == cmin);
            }
        }
        const unsigned mm = __ballot_sync(0xffffffffu, mask);
        unsigned todo = __ballot_sync(0xffffffffu, need);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const int32_t i0 = (c0 + NW * l) * kDirTile;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kDirTile / 32; ++r) {
                const int k = 32 * r + lane;
                const int64_t i = (int64_t)i0 + k;
                float4 S = make_float4(3e30f, 3e30f, 3e30f, 0.f);
                if (i < n) S = pts[i];
                const uint32_t sw = __float_as_uint(S.w);
                const int jj = k >> 1, h = k & 1;
                fA[4 * jj + h] = -S.x;
                fA[4 * jj + 2 + h] = -S.y;
                fB[4 * jj + h] = -S.z;
                fB[4 * jj + 2 + h] = (float)(ch ? pk_di(sw) : pk_de(sw));
                if (FR) sc[w][k] = i < n ? (uint32_t)(keys[i] >> fsh) : 0xffffffffu;
            }
            __syncwarp();
            float2 p[R];
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = make_float2(0.f, 0.f);
            if (!((mm >> l) & 1u)) {
#pragma unroll 2
                for (int j = 0; j < kDirTile / 2; ++j) {
                    const float4 A = sA[w][j], B = sB[w][j];
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        dir_term<false>(A, B, tx[r], ty[r], tz[r], mk2, true, true, p[r]);
                }
            } else {
                for (int j = 0; j < kDirTile / 2; ++j) {
                    const float4 A = sA[w][j], B = sB[w][j];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        bool k0 = i0 + 2 * j != tq[r], k1 = i0 + 2 * j + 1 != tq[r];
                        if (FR) {
                            k0 = k0 && sc[w][2 * j] == tcell[r];
                            k1 = k1 && sc[w][2 * j + 1] == tcell[r];
                        }
                        dir_term<true>(A, B, tx[r], ty[r], tz[r], mk2, k0, k1, p[r]);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) dir_kahan(acc[r], comp[r], __fadd_rn(p[r].x, p[r].y));
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) red[w][32 * r + lane] = __fsub_rn(acc[r], comp[r]);
    __syncthreads();
    for (int slot = threadIdx.x; slot < m; slot += NW * 32) {
        const float v = sum_totals<NW>([&](int k) { return red[k][slot]; });
        const int32_t t = ch ? list[n - 1 - (first + slot)] : list[first + slot];
        u[perm ? perm[t] : t] = v;
    }
}

// scratch after the list (n int32): the lists' counts, each list block's
// counts and the tiles' boxes, at most n + 8 words for n > kDirSmallN
struct DirScratch {
    int32_t *cnt, *bcnt;
    float* bounds;
    DirScratch(int32_t* p, int64_t n)
        : cnt(p), bcnt(p + 2), bounds(reinterpret_cast<float*>(p + 2 + 2 * blocks(n))) {}
    static __host__ __device__ constexpr int64_t blocks(int64_t n) {
        return (n + kDirListPts - 1) / kDirListPts;
    }
    static __host__ __device__ constexpr int64_t words(int64_t n) {
        return 2 + 2 * blocks(n) + 6 * ((n + kDirTile - 1) / kDirTile);
    }
};
static_assert(DirScratch::words(kDirSmallN + 1) <= kDirSmallN + 9, "the scratch words suffice");

// The evaluation over listed targets: three launches.  R and NW by the number
// of neurons: 4 targets per lane serve a staged pair best, but 128 targets a
// block leave the chip idle below about 300 blocks.
template <bool FR, class Src>
inline void dir_launch_tiles(int64_t n, Src src, float4* copy, const float4* pts, int32_t* list,
                             const DirScratch& t, float k2, const uint64_t* keys, int fsh,
                             const int32_t* perm, float* u, cudaStream_t s) {
    const unsigned gl = (unsigned)DirScratch::blocks(n);
    k_dir_count<<<gl, 256, 0, s>>>(n, src, copy, perm, t.bcnt, t.bounds, u);
    k_dir_lists<<<gl, 256, 0, s>>>(n, src, t.bcnt, list, t.cnt);
    if (n >= 40'000) {
        const unsigned g = (unsigned)((n + 127) / 128 + 1);
        k_dir_tiles<4, 8, FR><<<g, 256, 0, s>>>(n, pts, list, t.cnt, t.bounds, k2, keys, fsh, perm, u);
    } else {
        const unsigned g = (unsigned)((n + 63) / 64 + 1);
        k_dir_tiles<2, 16, FR><<<g, 512, 0, s>>>(n, pts, list, t.cnt, t.bounds, k2, keys, fsh, perm, u);
    }
}

}  // namespace msp
