// msp_fmm.cu -- steps a5-a10: dual traversal with the separation / cutoff
// rule, Hermite coefficients (Eq. 7), Hermite-to-Taylor translation (Eq. 7
// composed with the Taylor expansion of Eq. 6), Taylor evaluation (Eq. 6), the
// exact near field (Eq. 8) and the box-pair attraction table.
#include <algorithm>
#include <cmath>

#include "msp_hostdev.cuh"
#include "msp_scan.cuh"

namespace msp {

struct Geo {
    long long g2[kMortonBits + 1];   // prune when sum of squared box gaps >= g2[level]
    int l_far;                       // boxes at level >= l_far may carry expansions
    long long m2l_min_pairs;
    int mac_mode;                    // 1: Algorithm 2's count rule
    int c1;                          // its dendrite threshold
    // per-network cutoffs (points in frames): the thresholds of the finer
    // box's network, [network][level], for levels at or below frame_level
    const long long* fg2;
    int frame_level;
    int64_t nf;
};

__device__ inline float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__constant__ float c_inv_fact[kMaxP] = {1.f, 1.f, 0.5f, 1.f / 6.f, 1.f / 24.f, 1.f / 120.f,
                                        1.f / 720.f, 1.f / 5040.f};

namespace {

struct NodeView {
    const uint8_t* level;
    const uint64_t* prefix;
    const int32_t* first;
    const int32_t* count;
    const int32_t* child_first;
    const uint8_t* nchild;
    const int4* sums;
};

// A pair is pruned by the cutoff only: a box pair without vacant axonal or
// dendritic elements contributes exactly zero (log2 0 = -inf in every term,
// or no target), so the lists depend on the positions alone and the step
// graph can keep them across steps.
__device__ inline uint8_t classify(const NodeView& nv, const Geo& geo, int32_t X, int32_t Y) {
    const int4 sy = nv.sums[Y];
    int lx = nv.level[X], ly = nv.level[Y];
    int lf = lx > ly ? lx : ly;
    uint64_t px = nv.prefix[X], py = nv.prefix[Y];
    long long gsum = 0, gmax = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        long long lox = (long long)compact_by3(px >> (2 - d)) << (lf - lx);
        long long hix = lox + (1ll << (lf - lx));
        long long loy = (long long)compact_by3(py >> (2 - d)) << (lf - ly);
        long long hiy = loy + (1ll << (lf - ly));
        long long g = 0;
        if (loy - hix > g) g = loy - hix;
        if (lox - hiy > g) g = lox - hiy;
        gsum += g * g;
        if (g > gmax) gmax = g;
    }
    long long thr = geo.g2[lf];
    if (geo.fg2 && lf >= geo.frame_level) {
        // both boxes in one network: its cutoff; in two networks: at least a
        // cell apart, beyond every network's cutoff
        const int64_t k = box_frame(lx == lf ? px : py, lf, geo.frame_level, geo.nf);
        thr = geo.fg2[k * (kMortonBits + 1) + lf];
    }
    if (gsum >= thr) return kPruned;
    const bool leafx = nv.child_first[X] < 0, leafy = nv.child_first[Y] < 0;
    const int lmin = lx < ly ? lx : ly;
    if (geo.mac_mode == 1) {
        // Algorithm 2: a leaf side is evaluated directly; an inner dendrite
        // box with more than c1 vacant dendrites is expanded; else direct
        // (boxes above l_far, which is 0 unless the points sit in frames,
        // are split)
        if (leafx && leafy) return kP2P;
        if (!leafx && !leafy && X != Y && lmin >= geo.l_far && sy.z + sy.w > geo.c1)
            return kFar;
        return kSplit;
    }
    if (lmin >= geo.l_far && gmax >= 1 &&
        (long long)nv.count[X] * (long long)nv.count[Y] >= geo.m2l_min_pairs)
        return kFar;
    if (leafx && leafy) return kP2P;
    return kSplit;
}

// The traversal's tables and lists: the pair table, and as the pairs are
// classified, in pair order, the split pairs (pair, first child, child count,
// 0), the near-field pairs with their target leaf as the key of the sort that
// groups them, and the far pairs.
struct TravArgs {
    NodeView nv;
    Geo geo;
    int32_t *pX, *pY, *pcf;
    uint8_t *kind, *pnb;
    float4* pw;
    int64_t cap;
    int4* split;
    uint64_t* p2p_key;
    int32_t *p2p_q, *far_q;
    DevCounts* dc;
};

// Tile t of depth d (pairs q0 + 256 t ..., one per thread): classifies them
// and counts their children and the kinds; with the sums of the tiles before
// (excl(own, ex) gives them to every thread) writes the children, one
// contiguous block per pair, axon-child major, from next0 on, and the list
// entries.  A pair's children are written by its warp, 32 at a time.  Bound by
// latency at the sizes of one network; the step of a rebuilding replay at
// 262,144 neurons (five depths) went from 732 to 608 us with this and the
// octree's one-launch levels (classification, scan, writing and the three
// lists' flags, scans and compactions were 24 launches).
//
// Children that do not fit in the table (overflow bit 0) are not written and
// their pair has none; the fitting ones are a prefix of the depth's children,
// and the next depth ends there.  The caller grows the table and redoes the
// traversal.
constexpr int kTravTile = 256;

template <class Excl>
__device__ __forceinline__ void trav_tile(const TravArgs& a, int d, int64_t t, int64_t q0,
                                          int64_t nq, int64_t next0, bool last, Excl exclusive) {
    __shared__ int s_w[4][kTravTile / 32];
    __shared__ int s_tot[4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t k = t * kTravTile + threadIdx.x, q = q0 + k;
    const bool in = k < nq;
    int32_t X = 0, Y = 0;
    uint8_t kd = kPruned;
    int nb = 0;
    int2 child = make_int2(0, 0);      // the first child of X (X if a leaf), of Y (Y if a leaf)
    int ny = 1;
    if (in) {
        X = a.pX[q];
        Y = a.pY[q];
        kd = classify(a.nv, a.geo, X, Y);
        a.kind[q] = kd;
        a.pw[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kd == kSplit) {
            const int32_t cx = a.nv.child_first[X], cy = a.nv.child_first[Y];
            const int nx = cx < 0 ? 1 : a.nv.nchild[X];
            ny = cy < 0 ? 1 : a.nv.nchild[Y];
            nb = nx * ny;
            child = make_int2(cx < 0 ? X : cx, cy < 0 ? Y : cy);
        }
    }
    // offsets inside the tile
    int inc = nb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    const unsigned mS = __ballot_sync(0xffffffffu, in && kd == kSplit);
    const unsigned mP = __ballot_sync(0xffffffffu, in && kd == kP2P);
    const unsigned mF = __ballot_sync(0xffffffffu, in && kd == kFar);
    if (lane == 31) s_w[0][w] = inc;
    if (lane == 0) {
        s_w[1][w] = __popc(mS);
        s_w[2][w] = __popc(mP);
        s_w[3][w] = __popc(mF);
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        int run = 0;
#pragma unroll
        for (int j = 0; j < kTravTile / 32; ++j) {
            const int v = s_w[threadIdx.x][j];
            s_w[threadIdx.x][j] = run;
            run += v;
        }
        s_tot[threadIdx.x] = run;
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    const int pre = s_w[0][w] + inc - nb;
    long long ex[4];
    exclusive(s_tot, ex);             // a block barrier
    const int64_t c0 = next0 + ex[0];
    if (in) {
        const int64_t cf = c0 + pre;
        const bool stored = kd == kSplit && cf + nb <= a.cap;
        a.pcf[q] = stored ? (int32_t)cf : -1;
        if (stored) a.pnb[q] = (uint8_t)nb;
        if (kd == kSplit) {
            a.split[a.dc->split_start[d] + ex[1] + s_w[1][w] + __popc(mS & lt)] =
                make_int4((int32_t)q, stored ? (int32_t)cf : -1, nb, 0);
            // the first pair whose children do not fit
            if (!stored && cf <= a.cap) a.dc->depth_start[d + 2] = cf;
        } else if (kd == kP2P) {
            const int64_t r = a.dc->p2p_start[d] + ex[2] + s_w[2][w] + __popc(mP & lt);
            a.p2p_key[r] = (uint64_t)X;
            a.p2p_q[r] = (int32_t)q;
        } else if (kd == kFar) {
            a.far_q[a.dc->far_start[d] + ex[3] + s_w[3][w] + __popc(mF & lt)] = (int32_t)q;
        }
    }
    // a split pair's children by the whole warp, 32 at a time
    const int rcp = (2048 + ny - 1) / ny;         // floor(c / ny) = c rcp >> 11 for c < 64, ny <= 8
    for (unsigned todo = mS; todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        const int lnb = __shfl_sync(0xffffffffu, nb, l), lpre = __shfl_sync(0xffffffffu, pre, l);
        const int lny = __shfl_sync(0xffffffffu, ny, l), lrcp = __shfl_sync(0xffffffffu, rcp, l);
        const int2 lc = make_int2(__shfl_sync(0xffffffffu, child.x, l),
                                  __shfl_sync(0xffffffffu, child.y, l));
        const int64_t f = c0 + lpre;
        if (f + lnb > a.cap) break;                // nor do the ones after it fit
        for (int k2 = lane; k2 < lnb; k2 += 32) {
            const int i = k2 * lrcp >> 11;
            a.pX[f + k2] = lc.x + i;
            a.pY[f + k2] = lc.y + k2 - i * lny;
        }
    }
    if (last && threadIdx.x == 0) {
        DevCounts* dc = a.dc;
        const int64_t end = c0 + s_tot[0];
        if (end <= a.cap) {
            dc->depth_start[d + 2] = end;
        } else {
            atomicOr(reinterpret_cast<unsigned long long*>(&dc->overflow), 1ull);
            atomicMax(reinterpret_cast<unsigned long long*>(&dc->need_pairs),
                      (unsigned long long)end);
        }
        dc->n_split = dc->split_start[d + 1] = dc->split_start[d] + ex[1] + s_tot[1];
        dc->n_p2p = dc->p2p_start[d + 1] = dc->p2p_start[d] + ex[2] + s_tot[2];
        dc->n_far = dc->far_start[d + 1] = dc->far_start[d] + ex[3] + s_tot[3];
    }
}

// a depth without pairs: its lists and the next depth are empty
__device__ __forceinline__ void trav_empty(DevCounts* dc, int d) {
    dc->depth_start[d + 2] = dc->depth_start[d + 1];
    dc->n_split = dc->split_start[d + 1] = dc->split_start[d];
    dc->n_p2p = dc->p2p_start[d + 1] = dc->p2p_start[d];
    dc->n_far = dc->far_start[d + 1] = dc->far_start[d];
}

// the root pair (root, root) and the depths before kTopDepths (1 and at most
// 64 pairs: one tile each) by one block
constexpr int kTopDepths = 2;

__global__ void __launch_bounds__(kTravTile) k_trav_top(TravArgs a, int64_t n, int depths) {
    DevCounts* dc = a.dc;
    if (threadIdx.x == 0) {
        dc->depth_start[0] = 0;
        dc->depth_start[1] = n > 0 ? 1 : 0;
        dc->split_start[0] = dc->p2p_start[0] = dc->far_start[0] = 0;
        dc->overflow &= ~1ll;       // the traversal's bit; the build's (16) stays for the step check
        dc->need_pairs = 0;
        dc->interactions = 0;
        if (n > 0) {
            a.pX[0] = 0;
            a.pY[0] = 0;
        }
    }
    for (int d = 0; d < depths; ++d) {
        __syncthreads();
        const int64_t q0 = dc->depth_start[d], next0 = dc->depth_start[d + 1], nq = next0 - q0;
        __syncthreads();
        if (nq == 0) {
            if (threadIdx.x == 0) trav_empty(dc, d);
        } else {
            trav_tile(a, d, 0, q0, nq, next0, true, [](const int (&)[4], long long (&ex)[4]) {
                ex[0] = ex[1] = ex[2] = ex[3] = 0;
                __syncthreads();
            });
        }
    }
}

// one depth; status: a tile counter and W words per tile (trav_pack), zero on
// entry; W = 2: no pair is far.  (A third word costs 1 us a depth: two rebuilt
// steps of 262,144 neurons 9 us.)
template <int W>
__global__ void __launch_bounds__(kTravTile)
k_trav_depth(TravArgs a, int d, unsigned long long* status, int64_t timeout_bit) {
    __shared__ int64_t s_tile;
    __shared__ long long s_ex[W];
    DevCounts* dc = a.dc;
    if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);
    const int64_t q0 = dc->depth_start[d], next0 = dc->depth_start[d + 1], nq = next0 - q0;
    const int64_t ntiles = (nq + kTravTile - 1) / kTravTile;
    if (ntiles == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) trav_empty(dc, d);
        return;
    }
    for (;;) {
        __syncthreads();
        const int64_t t = s_tile;
        if (t >= ntiles) break;
        trav_tile(a, d, t, q0, nq, next0, t == ntiles - 1,
                  [&](const int (&tot)[4], long long (&ex)[4]) {
            long long e[W];
            if (threadIdx.x < 32) {
                long long own[W];
                trav_pack(tot, own);
                look_back<W>(status + 1, t, own, e, &dc->overflow, timeout_bit, kSpinLimit);
                if (threadIdx.x == 0)
#pragma unroll
                    for (int k = 0; k < W; ++k) s_ex[k] = e[k];
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < W; ++k) e[k] = s_ex[k];
            trav_unpack(e, ex);
        });
        if (ntiles <= gridDim.x) break;        // every block has had its one tile
        __syncthreads();
        if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);
    }
}

// ---------------------------------------------------------------------------
// a6: Hermite coefficients of the dendritic weights (Eq. 7) and axon moments
// M_beta = sum_t a_t ((t - c_A)/sigma)^beta, per channel, one block per box.
// A holds a coefficient's two channels side by side (the translations read them as
// one 8-byte pair), M and B channel after channel.
// ---------------------------------------------------------------------------
constexpr int kP2MThreads = 128;
constexpr int kP2MChunk = 32;

// The order is a template parameter: with it in a register the divisions of
// every index by p and the loops over powers were most of the instructions.
// 20 k boxes of at most 20 points, order 4: 76 us before, 20 us.  Bound by the
// chain of a block's few steps (load, powers, sums), not by its 1 KB a box.
template <int P>
__global__ void __launch_bounds__(kP2MThreads)
k_p2m(int64_t first_node, float inv_sigma, const float4* __restrict__ pts,
      const int32_t* __restrict__ nfirst, const int32_t* __restrict__ ncount,
      const float4* __restrict__ ca, const float4* __restrict__ cd, float* __restrict__ A,
      float* __restrict__ M) {
    constexpr int P2 = P * P, P3 = P2 * P;
    // powers of a point's offset from the dendritic [0] and axonal [1] centre
    __shared__ float pow_[2][kP2MChunk][3][P];
    __shared__ float wgt[kP2MChunk][4];
    const int64_t node = first_node + blockIdx.x;
    const float4 cD = cd[node], cA = ca[node];
    const int32_t f = nfirst[node], c = ncount[node];
    constexpr int NACC = (4 * P3 + kP2MThreads - 1) / kP2MThreads;
    float acc[NACC];
#pragma unroll
    for (int r = 0; r < NACC; ++r) acc[r] = 0.f;
    for (int base = 0; base < c; base += kP2MChunk) {
        const int m = min(kP2MChunk, c - base);
        if (base) __syncthreads();
        // thread (point, centre, dimension)
        for (int t = threadIdx.x; t < m * 6; t += kP2MThreads) {
            const int j = t / 6, g = (t % 6) / 3, d = t % 3;
            const float4 pt = pts[f + base + j];
            const float4 c4 = g ? cA : cD;
            const float v = ((d == 0 ? pt.x : (d == 1 ? pt.y : pt.z)) -
                             (d == 0 ? c4.x : (d == 1 ? c4.y : c4.z))) * inv_sigma;
            float pv = 1.f;
#pragma unroll
            for (int k = 0; k < P; ++k) {
                pow_[g][j][d][k] = pv;
                pv *= v;
            }
            if (t % 6 == 0) {
                const uint32_t w = __float_as_uint(pt.w);
                const float a = (float)pk_axon(w);
                const bool inh = pk_type(w) != 0;
                wgt[j][0] = (float)pk_de(w);
                wgt[j][1] = (float)pk_di(w);
                wgt[j][2] = inh ? 0.f : a;
                wgt[j][3] = inh ? a : 0.f;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < NACC; ++r) {
            const int idx = threadIdx.x + r * kP2MThreads;
            if (idx >= 4 * P3) continue;
            const int which = idx / P3, a = idx % P3;
            const int a0 = a / P2, a1 = (a / P) % P, a2 = a % P;
            const float(*pw)[3][P] = pow_[which >> 1];
            float s = acc[r];
            for (int j = 0; j < m; ++j)
                s = fmaf(wgt[j][which] * pw[j][0][a0], pw[j][1][a1] * pw[j][2][a2], s);
            acc[r] = s;
        }
    }
    const int64_t e = (int64_t)blockIdx.x;
#pragma unroll
    for (int r = 0; r < NACC; ++r) {
        const int idx = threadIdx.x + r * kP2MThreads;
        if (idx >= 4 * P3) continue;
        const int which = idx / P3, a = idx % P3;
        if (which < 2)
            A[(e * P3 + a) * 2 + which] = acc[r] * c_inv_fact[a / P2] *
                                          c_inv_fact[(a / P) % P] * c_inv_fact[a % P];
        else
            M[(e * 2 + which - 2) * P3 + a] = acc[r];
    }
}

// ---------------------------------------------------------------------------
// a7: translations.  With Delta = (c_A - c_D)/sigma and H_d[n] = h_n(Delta_d),
//   B_beta(X <- Y) = (-1)^|beta| / beta!  sum_alpha A_alpha(Y) H0[a0+b0] H1[a1+b1] H2[a2+b2]
// done as three passes over one dimension each (p^4 multiply-adds per pass
// and channel), and W(X,Y) = sum_beta B_beta(X <- Y) M_beta(X).  The far pairs
// are grouped by target box X (stable sort of the list by X); one warp takes
// all pairs of one X in list order, so B(X) = sum_Y B(X <- Y) is summed in
// registers in a fixed order (reproducible, no atomics) and added to B once.
// A pass is one column per lane (channel and the two indices it does not
// sum over), staged through the warp's shared memory between passes; the
// last pass's columns are the lane's own for every pair of X.
// ---------------------------------------------------------------------------
__device__ inline void hermite_row(float x, float* h, int nmax) {
    const float h0 = __expf(-x * x);
    h[0] = h0;
    if (nmax >= 1) h[1] = 2.f * x * h0;
    for (int k = 1; k < nmax; ++k) h[k + 1] = 2.f * x * h[k] - 2.f * (float)k * h[k - 1];
}

constexpr int kM2LWarps = 4;

template <int P>
__global__ void __launch_bounds__(kM2LWarps * 32)
k_m2l_seg(const int32_t* __restrict__ seg_first, const int64_t* __restrict__ nseg_dev,
          const int32_t* __restrict__ list, int64_t exp_first, float inv_sigma,
          const int32_t* __restrict__ pX, const int32_t* __restrict__ pY,
          const float4* __restrict__ ca, const float4* __restrict__ cd,
          const float* __restrict__ A, const float* __restrict__ M, float* __restrict__ B,
          float4* __restrict__ pw) {
    constexpr int P2 = P * P, P3 = P2 * P;
    constexpr int NC = 2 * P2;                 // columns of a pass (two channels)
    constexpr int NL = (NC + 31) / 32;         // columns per lane
    constexpr int NH = 2 * P - 1;              // Hermite functions h_0 .. h_{2p-2}
    __shared__ float sbuf[kM2LWarps][2][2 * P3];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* s0 = sbuf[w][0];
    float* s1 = sbuf[w][1];
    // (-1)^|beta| / beta! of the lane's last-pass columns (c, b0, b1)
    float scale[NL][P];
#pragma unroll
    for (int j = 0; j < NL; ++j) {
        const int col = lane + 32 * j;
        const int b0 = (col / P) % P, b1 = col % P;
#pragma unroll
        for (int b2 = 0; b2 < P; ++b2) {
            const float f = c_inv_fact[b0] * c_inv_fact[b1] * c_inv_fact[b2];
            scale[j][b2] = ((b0 + b1 + b2) & 1) ? -f : f;
        }
    }
    const int64_t nseg = *nseg_dev;
    for (int64_t sg = (int64_t)blockIdx.x * kM2LWarps + w; sg < nseg;
         sg += (int64_t)gridDim.x * kM2LWarps) {
        const int32_t i0 = seg_first[sg], i1 = seg_first[sg + 1];
        const int32_t X = pX[list[i0]];
        const int64_t ex = X - exp_first;
        const float4 a = ca[X];
        float acc[NL][P], mm[NL][P];
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int col = lane + 32 * j;
            const int c = col / P2, b0 = (col / P) % P, b1 = col % P;
#pragma unroll
            for (int b2 = 0; b2 < P; ++b2) {
                acc[j][b2] = 0.f;
                mm[j][b2] = col < NC ? M[(ex * 2 + c) * P3 + b0 * P2 + b1 * P + b2] : 0.f;
            }
        }
        // the next pair's list entry, centre and coefficients are loaded
        // while the current pair is translated (a chain of dependent loads)
        constexpr int NA = (2 * P3 + 31) / 32;     // coefficients per lane
        int32_t qn = list[i0];
        int32_t yn = pY[qn];
        float4 dn = cd[yn];
        float an[NA];
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const int e = lane + 32 * k;
            an[k] = e < 2 * P3 ? A[(yn - exp_first) * 2 * P3 + e] : 0.f;
        }
        for (int32_t i = i0; i < i1; ++i) {
            const int32_t q = qn;
            const float4 d = dn;
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const int e = lane + 32 * k;
                if (e < 2 * P3) s0[(e & 1) * P3 + (e >> 1)] = an[k];
            }
            if (i + 1 < i1) {
                qn = list[i + 1];
                yn = pY[qn];
                dn = cd[yn];
#pragma unroll
                for (int k = 0; k < NA; ++k) {
                    const int e = lane + 32 * k;
                    an[k] = e < 2 * P3 ? A[(yn - exp_first) * 2 * P3 + e] : 0.f;
                }
            }
            float H[NH];
            hermite_row((a.x - d.x) * inv_sigma, H, NH - 1);
            __syncwarp();
            // pass 0 (over a0): column (c, a1, a2) -> s1[c][b0][a1][a2]
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                const int col = lane + 32 * j;
                if (col >= NC) break;
                const int c = col / P2, r = col % P2;
                float v[P];
#pragma unroll
                for (int k = 0; k < P; ++k) v[k] = s0[c * P3 + k * P2 + r];
#pragma unroll
                for (int o = 0; o < P; ++o) {
                    float t = 0.f;
#pragma unroll
                    for (int k = 0; k < P; ++k) t = fmaf(H[k + o], v[k], t);
                    s1[c * P3 + o * P2 + r] = t;
                }
            }
            hermite_row((a.y - d.y) * inv_sigma, H, NH - 1);
            __syncwarp();
            // pass 1 (over a1): column (c, b0, a2) -> s0[c][b0][b1][a2]
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                const int col = lane + 32 * j;
                if (col >= NC) break;
                const int c = col / P2, b0 = (col / P) % P, a2 = col % P;
                const int base = c * P3 + b0 * P2 + a2;
                float v[P];
#pragma unroll
                for (int k = 0; k < P; ++k) v[k] = s1[base + k * P];
#pragma unroll
                for (int o = 0; o < P; ++o) {
                    float t = 0.f;
#pragma unroll
                    for (int k = 0; k < P; ++k) t = fmaf(H[k + o], v[k], t);
                    s0[base + o * P] = t;
                }
            }
            hermite_row((a.z - d.z) * inv_sigma, H, NH - 1);
            __syncwarp();
            // pass 2 (over a2): the lane's own columns (c, b0, b1)
            float w0 = 0.f, w1 = 0.f;
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                const int col = lane + 32 * j;
                if (col >= NC) break;
                const int base = (col / P2) * P3 + (col % P2) * P;
                float v[P];
#pragma unroll
                for (int k = 0; k < P; ++k) v[k] = s0[base + k];
                float wc = 0.f;
#pragma unroll
                for (int o = 0; o < P; ++o) {
                    float t = 0.f;
#pragma unroll
                    for (int k = 0; k < P; ++k) t = fmaf(H[k + o], v[k], t);
                    t *= scale[j][o];
                    acc[j][o] += t;
                    wc = fmaf(t, mm[j][o], wc);
                }
                if (col < P2) w0 += wc; else w1 += wc;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                w0 += __shfl_xor_sync(0xffffffffu, w0, o);
                w1 += __shfl_xor_sync(0xffffffffu, w1, o);
            }
            if (lane == 0) pw[q] = make_float4(w0, 0.f, w1, 0.f);
            __syncwarp();      // s0 is the next pair's staging
        }
        // B(X) += the sum over X's far pairs (no other warp adds to B(X) here)
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int col = lane + 32 * j;
            if (col >= NC) break;
            const int c = col / P2, b0 = (col / P) % P, b1 = col % P;
            float* Bx = B + (ex * 2 + c) * P3 + b0 * P2 + b1 * P;
#pragma unroll
            for (int b2 = 0; b2 < P; ++b2) Bx[b2] += acc[j][b2];
        }
    }
}

// Order 4 (the paper's): a pass has 16 columns per channel, so a quarter of a warp
// takes a pair, two columns a lane, and the quarters alternate over X's pairs; both
// channels share the Hermite functions and run as the two halves of paired FMAs;
// the next pair's coefficients are loaded while the current pair is translated.
// Per pair the products and sums of W(X,Y) are those of the general kernel in the
// same order; B(X) adds the pairs of each quarter and then the quarters.  Blocks
// take four targets and leave (the numbers of pairs per target differ widely: a
// grid of resident blocks striding over the targets took 0.93 ms).
// 4.9 M pairs of 65,536 neurons: 1.47 ms in the general kernel, 0.58 ms here (0.67
// with list entry, source box and coefficients read one pair ahead, 0.72 with the
// channels' coefficients read one by one too, 0.74 with half a warp a pair, 1.47
// with unpadded rows: bank conflicts).  Bound by instruction issue: 48 paired
// FMAs of a pair's 90 instructions, the rest Hermite functions and staging.
__global__ void __launch_bounds__(kM2LWarps * 32, 4)
k_m2l_seg4(const int32_t* __restrict__ seg_first, const int64_t* __restrict__ nseg_dev,
           const int32_t* __restrict__ list, int64_t exp_first, float inv_sigma,
           const int32_t* __restrict__ pX, const int32_t* __restrict__ pY,
           const float4* __restrict__ ca, const float4* __restrict__ cd,
           const float* __restrict__ A, const float* __restrict__ M, float* __restrict__ B,
           float4* __restrict__ pw) {
    constexpr int P = 4, P3 = 64, QW = 88;
    // a quarter's coefficients between passes: [b0][a1][a2] with rows of 20 and 4,
    // [b0][b1][a2] with rows of 20 and 5, quarters 88 apart (16 lanes write or
    // read 16 different pairs of banks in every pass)
    __shared__ float2 s_t0[kM2LWarps][4 * QW], s_t1[kM2LWarps][4 * QW];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, quarter = lane >> 3, r = lane & 7;
    float2* t0 = s_t0[w] + QW * quarter;
    float2* t1 = s_t1[w] + QW * quarter;
    const int hi = r >> 2, lo = r & 3;       // the lane's columns: (hi, lo) and (hi + 2, lo)
    float scale[2][P];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int b2 = 0; b2 < P; ++b2) {
            const float f = c_inv_fact[hi + 2 * j] * c_inv_fact[lo] * c_inv_fact[b2];
            scale[j][b2] = ((hi + lo + b2) & 1) ? -f : f;
        }
    const int64_t nseg = *nseg_dev;
    for (int64_t sg = (int64_t)blockIdx.x * kM2LWarps + w; sg < nseg;
         sg += (int64_t)gridDim.x * kM2LWarps) {
        const int32_t i0 = seg_first[sg], i1 = seg_first[sg + 1];
        const int32_t X = pX[list[i0]];
        const int64_t ex = X - exp_first;
        const float4 a4 = ca[X];
        float2 mm[2][P], acc[2][P];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float4 m0 = reinterpret_cast<const float4*>(M + (ex * 2) * P3)[r + 8 * j];
            const float4 m1 = reinterpret_cast<const float4*>(M + (ex * 2 + 1) * P3)[r + 8 * j];
            mm[j][0] = make_float2(m0.x, m1.x);
            mm[j][1] = make_float2(m0.y, m1.y);
            mm[j][2] = make_float2(m0.z, m1.z);
            mm[j][3] = make_float2(m0.w, m1.w);
#pragma unroll
            for (int k = 0; k < P; ++k) acc[j][k] = make_float2(0.f, 0.f);
        }
        // the next pair's centre and coefficients are loaded while the current
        // pair is translated, its source box a pair earlier and the list entry
        // two (a chain of dependent reads longer than a pair's work)
        auto entry = [&](int32_t i) { return (uint32_t)i < (uint32_t)i1 ? list[i] : -1; };
        auto source = [&](int32_t q) { return q >= 0 ? pY[q] : -1; };
        int32_t q = entry(i0 + quarter), q1 = entry(i0 + 4 + quarter), q2 = entry(i0 + 8 + quarter);
        float4 d = a4;
        float2 v[2][P];
        auto load = [&](int32_t Y) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int k = 0; k < P; ++k) v[j][k] = make_float2(0.f, 0.f);
            if (Y < 0) return;
            d = cd[Y];
            const float2* Ay = reinterpret_cast<const float2*>(A) + (Y - exp_first) * P3 + r;
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int k = 0; k < P; ++k)
                    v[j][k] = Ay[16 * k + 8 * j];
        };
        load(source(q));
        int32_t y1 = source(q1);
        for (int32_t ib = i0; (uint32_t)ib < (uint32_t)i1; ib += 4) {
            const bool in = q >= 0;
            const int32_t qc = q;
            float H[8];
            const float4 dc = d;
            auto apply = [&](const float2 (&c)[P], int o) {
                float2 t = make_float2(0.f, 0.f);
#pragma unroll
                for (int k = 0; k < P; ++k)
                    t = __ffma2_rn(make_float2(H[k + o], H[k + o]), c[k], t);
                return t;
            };
            // over a0: column (a1, a2) -> [b0][a1][a2]
            hermite_row((a4.x - dc.x) * inv_sigma, H, 2 * P - 2);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int o = 0; o < P; ++o) t0[20 * o + r + 8 * j] = apply(v[j], o);
            load(y1);
            q = q1;
            y1 = source(q2);
            q1 = q2;
            q2 = entry(ib + 12 + quarter);
            __syncwarp();
            // over a1: column (b0, a2) -> [b0][b1][a2]
            hermite_row((a4.y - dc.y) * inv_sigma, H, 2 * P - 2);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float2 c[P];
#pragma unroll
                for (int k = 0; k < P; ++k) c[k] = t0[20 * (hi + 2 * j) + 4 * k + lo];
#pragma unroll
                for (int o = 0; o < P; ++o) t1[20 * (hi + 2 * j) + 5 * o + lo] = apply(c, o);
            }
            __syncwarp();
            // over a2: column (b0, b1)
            hermite_row((a4.z - dc.z) * inv_sigma, H, 2 * P - 2);
            float2 wc[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float2 c[P];
#pragma unroll
                for (int k = 0; k < P; ++k) c[k] = t1[20 * (hi + 2 * j) + 5 * lo + k];
                wc[j] = make_float2(0.f, 0.f);
#pragma unroll
                for (int o = 0; o < P; ++o) {
                    const float2 t = __fmul2_rn(apply(c, o), make_float2(scale[j][o], scale[j][o]));
                    acc[j][o] = __fadd2_rn(acc[j][o], t);
                    wc[j] = __ffma2_rn(t, mm[j][o], wc[j]);
                }
            }
            float2 ws = __fadd2_rn(wc[0], wc[1]);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                ws.x += __shfl_xor_sync(0xffffffffu, ws.x, o);
                ws.y += __shfl_xor_sync(0xffffffffu, ws.y, o);
            }
            if (r == 0 && in) pw[qc] = make_float4(ws.x, 0.f, ws.y, 0.f);
        }
        // B(X) += the sum over X's far pairs (no other warp adds to B(X) here):
        // quarters 0, 1 write the excitatory columns, 2, 3 the inhibitory ones
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < P; ++k)
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) {
                    acc[j][k].x += __shfl_xor_sync(0xffffffffu, acc[j][k].x, o);
                    acc[j][k].y += __shfl_xor_sync(0xffffffffu, acc[j][k].y, o);
                }
        const int j = quarter & 1, ch = quarter >> 1;
        float4* Bx = reinterpret_cast<float4*>(B + (ex * 2 + ch) * P3) + r + 8 * j;
        float4 b = *Bx;
        float add[P];
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const float2 t = j ? acc[1][k] : acc[0][k];
            add[k] = ch ? t.y : t.x;
        }
        b.x += add[0];
        b.y += add[1];
        b.z += add[2];
        b.w += add[3];
        *Bx = b;
    }
}

// keys of the far pairs [first, nfar) of `list` for the grouping by target box
__global__ void k_m2l_keys(const int32_t* __restrict__ list, const int64_t* __restrict__ nfar,
                           const int64_t* __restrict__ first, const int32_t* __restrict__ pX,
                           uint64_t* __restrict__ key, int32_t* __restrict__ val,
                           int64_t* __restrict__ count) {
    const int64_t k0 = first ? *first : 0, n = *nfar - k0;
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = n > 0 ? n : 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t q = list[k0 + i];
        key[i] = (uint64_t)pX[q];
        val[i] = q;
    }
}

// ---------------------------------------------------------------------------
// a8: Taylor evaluation (Eq. 6) at every target from each of its boxes that
// carries an expansion; initialises u_sorted and (uo not null) the caller's u.
// reuse not null: first launch of an attraction that keeps its lists; clears
// the counters that the traversal would have cleared.
// ---------------------------------------------------------------------------
__global__ void k_l2p(int64_t n, int64_t exp_first, int p, float inv_sigma,
                      const float4* __restrict__ pts, const int32_t* __restrict__ leaf_of,
                      const int32_t* __restrict__ parent, const float4* __restrict__ ca,
                      const float* __restrict__ B, const int32_t* __restrict__ perm,
                      float* __restrict__ u, float* __restrict__ uo, DevCounts* reuse) {
    if (reuse && blockIdx.x == 0 && threadIdx.x == 0) {
        reuse->overflow &= ~1ll;
        reuse->interactions = 0;
    }
    const int p3 = p * p * p;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        float4 P = pts[j];
        uint32_t pw = __float_as_uint(P.w);
        float acc = 0.f;
        if (pk_axon(pw) > 0) {
            int ch = pk_type(pw) ? 1 : 0;
            int32_t node = leaf_of[j];
            while (node >= exp_first) {
                float4 c = ca[node];
                float x[3] = {(P.x - c.x) * inv_sigma, (P.y - c.y) * inv_sigma,
                              (P.z - c.z) * inv_sigma};
                float px[3][kMaxP];
                for (int d = 0; d < 3; ++d) {
                    float v = 1.f;
                    for (int k = 0; k < p; ++k) {
                        px[d][k] = v;
                        v *= x[d];
                    }
                }
                const float* Bn = B + ((int64_t)(node - exp_first) * 2 + ch) * p3;
                int i = 0;
                for (int b0 = 0; b0 < p; ++b0)
                    for (int b1 = 0; b1 < p; ++b1) {
                        float s = 0.f;
                        float f01 = px[0][b0] * px[1][b1];
                        for (int b2 = 0; b2 < p; ++b2) s = fmaf(Bn[i++], px[2][b2], s);
                        acc = fmaf(f01, s, acc);
                    }
                node = parent[node];
            }
        }
        u[j] = acc;
        if (uo) uo[perm[j]] = acc;
    }
}

// a10: attraction of a split pair = sum over its child block, in double-FP32
// (compensated FP32 sums: no double precision instruction, which this GPU
// runs at 1/64 of the single precision rate).  The split pairs of each depth
// are listed once per traversal (the list keeps pair order, each entry with
// its child block); 8 lanes take one split pair, lane c summing children c,
// c + 8, ... (coalesced: 8 consecutive 16-byte entries per step, all loaded
// before the sum), then a fixed butterfly over the 8 lanes.  Both orders are
// fixed, so the table is reproducible.  sb = [first, end) of the depth's
// entries in split; an entry is (pair, first child, child count, 0).
__device__ __forceinline__ void reduce_depth(const int64_t* __restrict__ sb,
                                             const int4* __restrict__ split, float4* pw,
                                             int64_t warp, int64_t nwarp) {
    const int64_t s0 = sb[0], ns = sb[1] - sb[0];
    const int lane = threadIdx.x & 31, sub = lane & 7;
    // the loop bound is uniform across the warp (its 4 groups shuffle together)
    for (int64_t k0 = 4 * warp; k0 < ns; k0 += 4 * nwarp) {
        const int64_t k = k0 + (lane >> 3);
        int4 ent = make_int4(-1, -1, 0, 0);
        if (k < ns) ent = split[s0 + k];
        const int32_t q = ent.x, cf = ent.y;
        const int nb = cf >= 0 ? ent.z : 0;     // cf < 0: children not stored (overflow)
        // a lane's children (at most 8 of a block of 64) loaded before they
        // are summed, in compensated running sums of both channels
        float4 v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (sub + 8 * t < nb) v[t] = pw[cf + sub + 8 * t];
        float eh = 0.f, ec = 0.f, ih = 0.f, ic = 0.f;
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (sub + 8 * t < nb) {
                ff_acc(eh, ec, v[t].x, v[t].y);
                ff_acc(ih, ic, v[t].z, v[t].w);
            }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const float oeh = __shfl_xor_sync(0xffffffffu, eh, o);
            const float oec = __shfl_xor_sync(0xffffffffu, ec, o);
            const float oih = __shfl_xor_sync(0xffffffffu, ih, o);
            const float oic = __shfl_xor_sync(0xffffffffu, ic, o);
            ff_acc(eh, ec, oeh, oec);
            ff_acc(ih, ic, oih, oic);
        }
        if (sub == 0 && cf >= 0) {
            const float2 e = ff_two_sum(eh, ec), i = ff_two_sum(ih, ic);
            pw[q] = make_float4(e.x, e.y, i.x, i.y);
        }
    }
}
__global__ void k_reduce_split(const int64_t* __restrict__ sb, const int4* __restrict__ split,
                               float4* pw) {
    reduce_depth(sb, split, pw, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                 ((int64_t)gridDim.x * blockDim.x) >> 5);
}
// The last depths (at most 64 split pairs and the root's) in one block, the others
// with as many blocks as the depth may have pairs for: a step of two networks of
// 21 k 1209 -> 1193 us (4 and 5 launches of 1216 blocks each before).
constexpr int kReduceTop = 2;
__global__ void __launch_bounds__(512) k_reduce_top(const int64_t* __restrict__ sb,
                                                    const int4* __restrict__ split, float4* pw,
                                                    int depths) {
    for (int d = depths - 1; d >= 0; --d) {
        reduce_depth(sb + d, split, pw, threadIdx.x >> 5, blockDim.x >> 5);
        __syncthreads();
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
static NodeView node_view(msp_ctx& c) {
    NodeView nv;
    nv.level = c.nd_level.get<uint8_t>();
    nv.prefix = c.nd_prefix.get<uint64_t>();
    nv.first = c.nd_first.get<int32_t>();
    nv.count = c.nd_count.get<int32_t>();
    nv.child_first = c.nd_child_first.get<int32_t>();
    nv.nchild = c.nd_nchild.get<uint8_t>();
    nv.sums = c.nd_sums.get<int4>();
    return nv;
}

static int bits_for(int64_t v) {
    int b = 1;
    while (b < 63 && (1ll << b) <= v) ++b;
    return b;
}

void attraction(msp_ctx& c, float* u_dev, cudaStream_t s) {
    NvtxRange nv_("msp attraction");
    if (!c.tree_built) throw Error(MSP_ERR_NOT_BUILT, "msp_build_tree must run first");
    if (!c.graph_mode) {
        c.attraction_done = false;
        c.last_was_graph = false;
    }
    const msp_config& cfg = c.cfg;
    const int64_t n = c.n;
    const int B = 256;
    // inside a stream capture the near-field events become graph nodes
    cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
    MSP_CUDA(cudaStreamIsCapturing(s, &cst));
    const unsigned ev_flags = cst == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : 0u;
    NodeView nv = node_view(c);
    Geo geo;
    for (int l = 0; l <= kMortonBits; ++l) geo.g2[l] = c.g2[l];
    geo.fg2 = c.frame_level > 0 && c.frame_plans ? c.frame_g2.get<long long>() : nullptr;
    geo.frame_level = c.frame_level;
    geo.nf = (int64_t)c.frame_off_host.size() - 1;
    geo.l_far = c.l_far;
    geo.m2l_min_pairs = cfg.m2l_min_pairs;
    geo.mac_mode = cfg.mac_mode;
    geo.c1 = cfg.c1;
    const int p = cfg.p, p3 = p * p * p;
    const float inv_sigma = (float)(1.0 / cfg.sigma);

    DevCounts* dc = dcounts(c);
    // traversal depth d holds the pairs whose finer box is at level d, so the
    // tree depth bounds the number of depths
    const int D = c.tree_depth + 1;
    // replays of the step graph that reuse the octree keep the traversal and
    // its lists too: the cutoff rule depends on the positions only (the count
    // rule of Algorithm 2 depends on the vacant counts and is redone)
    if (c.pair_cap <= 0) c.pair_cap = std::max<int64_t>(64 * c.n_nodes, 1 << 16);
    // an eager attraction on a reused octree keeps the lists of the last one,
    // provided no buffer that holds them is about to grow (which would lose
    // them)
    auto holds = [&](const DBuf& b, size_t elem) {
        return b.bytes >= (size_t)c.pair_cap * elem;
    };
    const bool lists_fit = holds(c.pr_X, 4) && holds(c.pr_Y, 4) && holds(c.pr_kind, 1) &&
                           holds(c.pr_cf, 4) && holds(c.pr_nb, 1) && holds(c.pr_w, 16) &&
                           holds(c.p2p_val0, 4) && holds(c.far_q, 4) && holds(c.split_q, 16) &&
                           holds(c.nf_src, 8) &&
                           holds(c.nf_w32, 8) &&
                           (c.exp_nodes == 0 || (holds(c.m2_key0, 8) && holds(c.m2_val0, 4)));
    const bool reuse_lists =
        cfg.mac_mode == 0 && ((c.graph_mode && !c.graph_full_build) ||
                              (!c.graph_mode && c.tree_reused && c.lists_valid && lists_fit));
    const int Gt = (int)std::max<int64_t>(1, (int64_t)c.sm_count * 8);
    for (int attempt = 0;; ++attempt) {
    const int64_t cap = c.pair_cap;
    if (cap > 0x7fffffffll) throw Error(MSP_ERR_CAPACITY, "pair count exceeds int32");
    c.pr_X.ensure<int32_t>((size_t)cap);
    c.pr_Y.ensure<int32_t>((size_t)cap);
    c.pr_kind.ensure<uint8_t>((size_t)cap);
    c.pr_cf.ensure<int32_t>((size_t)cap);
    c.pr_nb.ensure<uint8_t>((size_t)cap);
    c.pr_w.ensure<float4>((size_t)cap);
    uint8_t* kind = c.pr_kind.get<uint8_t>();

    int32_t* far_q = c.far_q.ensure<int32_t>((size_t)cap);
    int4* split = c.split_q.ensure<int4>((size_t)cap);
    int32_t* pv0 = c.p2p_val0.ensure<int32_t>((size_t)cap);
    int32_t* seg_first = c.seg_first.ensure<int32_t>((size_t)c.n_nodes + 2);
    // the step graph's replays keep the traversal and the lists of the eager
    // attraction of the same positions (guarded by the build's checksum and
    // generation stamp); k_l2p restarts the near field's work counter
    if (!reuse_lists) {
    // a5: breadth-first dual traversal from (root, root): the first depths in
    // one launch, then one per depth (status words cleared together; depth d
    // holds at most 64^d pairs), each writing its part of the lists
    const int xbits = bits_for(c.n_nodes);
    const bool odd = radix_from_tmp(cap, xbits);
    uint64_t* pk0 = c.p2p_key0.ensure<uint64_t>((size_t)cap);
    uint64_t* pk1 = c.p2p_key1.ensure<uint64_t>((size_t)cap);
    int32_t* pv1 = c.p2p_val1.ensure<int32_t>((size_t)cap);
    TravArgs ta;
    ta.nv = nv;
    ta.geo = geo;
    ta.pX = c.pr_X.get<int32_t>();
    ta.pY = c.pr_Y.get<int32_t>();
    ta.pcf = c.pr_cf.get<int32_t>();
    ta.kind = kind;
    ta.pnb = c.pr_nb.get<uint8_t>();
    ta.pw = c.pr_w.get<float4>();
    ta.cap = cap;
    ta.split = split;
    ta.p2p_key = odd ? pk1 : pk0;
    ta.p2p_q = odd ? pv1 : pv0;
    ta.far_q = far_q;
    ta.dc = dc;
    auto tiles_at = [&](int d) {
        const int64_t pairs = d < 5 ? std::min<int64_t>((int64_t)1 << (6 * d), cap) : cap;
        return (pairs + kTravTile - 1) / kTravTile;
    };
    const int dtop = std::min(D, kTopDepths);
    const int words = c.l_far <= c.tree_depth ? 3 : 2;      // a far pair's boxes: levels from l_far on
    int64_t nw = 0;
    for (int d = dtop; d < D; ++d) nw += 1 + words * tiles_at(d);
    unsigned long long* st = c.tv_status.ensure<unsigned long long>((size_t)std::max<int64_t>(nw, 1));
    if (nw > 0) MSP_CUDA(cudaMemsetAsync(st, 0, (size_t)nw * sizeof(unsigned long long), s));
    k_trav_top<<<1, kTravTile, 0, s>>>(ta, n, dtop);
    MSP_LAUNCH("trav_top");
    for (int d = dtop; d < D; ++d) {
        const int64_t tiles = tiles_at(d);
        (words == 3 ? k_trav_depth<3> : k_trav_depth<2>)<<<
            (unsigned)std::min<int64_t>(tiles, (int64_t)c.sm_count * 6), kTravTile, 0, s>>>(
            ta, d, st, kScanTimeoutBit);
        MSP_LAUNCH("trav_depth");
        st += 1 + words * tiles;
    }
    // the near-field list grouped by target leaf (at most one segment per box)
    radix_sort_dev(c, pk0, pv0, pk1, pv1, &dc->n_p2p, cap, xbits, s);
    const ScanHeads head{pk0};
    scan_launch(c, head, ScanFirsts{head, seg_first}, ScanSegments{&dc->nseg, seg_first, &dc->n_p2p},
                &dc->n_p2p, cap, s);
    }

    // a6: expansions of every box at level >= l_far
    c.exp_first = c.l_far <= c.tree_depth ? c.level_start[c.l_far] : c.n_nodes;
    c.exp_nodes = c.n_nodes - c.exp_first;
    size_t ecount = (size_t)std::max<int64_t>(c.exp_nodes, 1) * 2 * p3;
    float* eA = c.expA.ensure<float>(ecount);
    float* eM = c.expM.ensure<float>(ecount);
    float* eB = c.expB.ensure<float>(ecount);
    // expansion centres: the centroids, or the geometric centres (centre_mode 1)
    const bool geo = c.cfg.centre_mode == 1;
    const float4* eca = c.nd_ca.get<float4>();
    const float4* ecd = c.nd_cd.get<float4>();
    if (geo && c.exp_nodes > 0) {
        geo_centres(c, s);
        eca = ecd = c.nd_gc.get<float4>();
    }
    if (c.exp_nodes > 0) {
        MSP_CUDA(cudaMemsetAsync(eB, 0, ecount * sizeof(float), s));
#define MSP_P2M_CASE(PP)                                                                    \
    case PP:                                                                                \
        k_p2m<PP><<<(unsigned)c.exp_nodes, kP2MThreads, 0, s>>>(                            \
            c.exp_first, inv_sigma, c.pts.get<float4>(), c.nd_first.get<int32_t>(),         \
            c.nd_count.get<int32_t>(), eca, ecd, eA, eM);                                   \
        break;
        switch (p) {
            MSP_P2M_CASE(1) MSP_P2M_CASE(2) MSP_P2M_CASE(3) MSP_P2M_CASE(4)
            MSP_P2M_CASE(5) MSP_P2M_CASE(6) MSP_P2M_CASE(7) MSP_P2M_CASE(8)
            default: throw Error(MSP_ERR_INVALID_ARG, "expansion order out of range");
        }
#undef MSP_P2M_CASE
        MSP_LAUNCH("p2m");
    }
    // a7: translations, accumulating B(X) and W(X,Y); with geometric centres
    // the pairs that share an offset share one operator (matrix products),
    // the rest one pair at a time
    if (c.exp_nodes > 0) {
        const int32_t* mq = far_q;
        const int64_t* first = nullptr;
        if (geo && m2l_gemm_fits(p)) {
            int64_t* fb = nullptr;
            mq = m2l_gemm(c, far_q, &dc->n_far, cap, eA, eM, eB, c.pr_w.get<float4>(), &fb, s);
            first = fb;
        }
        // the pairs [first, n_far) of mq grouped by target box
        uint64_t* mk0 = c.m2_key0.ensure<uint64_t>((size_t)cap);
        uint64_t* mk1 = c.m2_key1.ensure<uint64_t>((size_t)cap);
        int32_t* mv0 = c.m2_val0.ensure<int32_t>((size_t)cap);
        int32_t* mv1 = c.m2_val1.ensure<int32_t>((size_t)cap);
        int32_t* mseg = c.m2_seg.ensure<int32_t>((size_t)c.n_nodes + 2);
        if (!reuse_lists || geo) {
            const int xbits = bits_for(c.n_nodes);
            const bool odd = radix_from_tmp(cap, xbits);
            k_m2l_keys<<<Gt, B, 0, s>>>(mq, &dc->n_far, first, c.pr_X.get<int32_t>(),
                                        odd ? mk1 : mk0, odd ? mv1 : mv0, &dc->m2l_n);
            MSP_LAUNCH("m2l_keys");
            radix_sort_dev(c, mk0, mv0, mk1, mv1, &dc->m2l_n, cap, xbits, s);
            const ScanHeads head{mk0};
            scan_launch(c, head, ScanFirsts{head, mseg}, ScanSegments{&dc->m2l_nseg, mseg, &dc->m2l_n},
                        &dc->m2l_n, cap, s);
        }
        const int gm = (int)c.sm_count * 8;
#define MSP_M2L_CASE(PP)                                                                       \
    case PP:                                                                                   \
        k_m2l_seg<PP><<<gm, kM2LWarps * 32, 0, s>>>(mseg, &dc->m2l_nseg, mv0, c.exp_first,    \
                                                    inv_sigma, c.pr_X.get<int32_t>(),         \
                                                    c.pr_Y.get<int32_t>(), eca, ecd, eA, eM,  \
                                                    eB, c.pr_w.get<float4>());                \
        break;
        switch (p) {
            MSP_M2L_CASE(1) MSP_M2L_CASE(2) MSP_M2L_CASE(3)
            case 4:
                k_m2l_seg4<<<(unsigned)((c.exp_nodes + kM2LWarps - 1) / kM2LWarps), kM2LWarps * 32,
                             0, s>>>(mseg, &dc->m2l_nseg, mv0, c.exp_first, inv_sigma,
                                     c.pr_X.get<int32_t>(), c.pr_Y.get<int32_t>(), eca, ecd, eA, eM,
                                     eB, c.pr_w.get<float4>());
                break;
            MSP_M2L_CASE(5) MSP_M2L_CASE(6) MSP_M2L_CASE(7) MSP_M2L_CASE(8)
            default: throw Error(MSP_ERR_INVALID_ARG, "expansion order out of range");
        }
#undef MSP_M2L_CASE
        MSP_LAUNCH("m2l");
    }
    // a8: Taylor evaluation initialises u in sorted order; a9 adds the near field
    float* us = c.u_sorted.ensure<float>((size_t)std::max<int64_t>(n, 1));
    unsigned long long* work = reinterpret_cast<unsigned long long*>(&dc->interactions);
    if (n > 0) {
        k_l2p<<<grid_for(n, B, (int64_t)c.sm_count * 16), B, 0, s>>>(
            n, c.exp_first, p, inv_sigma, c.pts.get<float4>(), c.leaf_of.get<int32_t>(),
            c.nd_parent.get<int32_t>(), eca, eB, c.perm.get<int32_t>(), us, u_dev,
            reuse_lists ? dc : nullptr);
        MSP_LAUNCH("l2p");
        MSP_CUDA(cudaEventRecordWithFlags(c.ev_nf0, s, ev_flags));
        launch_near_field(c, seg_first, &dc->nseg, c.n_nodes, pv0, cap, us, u_dev, work,
                          reuse_lists, s);
        MSP_CUDA(cudaEventRecordWithFlags(c.ev_nf1, s, ev_flags));
    }
    c.nf_timed = n > 0;
    // a10: pair table, deepest pairs first
    for (int dd = D - 1; dd >= kReduceTop; --dd) {
        // at most 64^dd pairs of this depth, four a warp
        const int64_t pairs = std::min<int64_t>((int64_t)1 << std::min(6 * dd, 40), cap);
        k_reduce_split<<<grid_for(8 * pairs, B, Gt), B, 0, s>>>(&dc->split_start[dd], split,
                                                               c.pr_w.get<float4>());
        MSP_LAUNCH("reduce_split");
    }
    k_reduce_top<<<1, 512, 0, s>>>(dc->split_start, split, c.pr_w.get<float4>(),
                                   std::min(D, kReduceTop));
    MSP_LAUNCH("reduce_top");
    // inside the whole-step graph the table does not grow: an overflow halts
    // the graph (checked on the device after the selection)
    if (c.graph_mode) return;
    pull_counts(c, s);              // the one synchronisation of the attraction
    const DevCounts& hc = *c.hcount;
    if (hc.overflow & 1) {
        // the pair table was too small: the traversal stopped at the first depth
        // that did not fit, so its count is a lower bound; grow and redo
        if (attempt >= 8) throw Error(MSP_ERR_CAPACITY, "pair table overflow after growth");
        c.pair_cap = std::max(2 * cap, hc.need_pairs + hc.need_pairs / 2 + 1024);
        continue;
    }
    int nd = 0;
    for (int d = 0; d < D; ++d)
        if (hc.depth_start[d + 1] > hc.depth_start[d]) nd = d + 1;
    c.depth_start.assign(hc.depth_start, hc.depth_start + nd + 1);
    c.n_pairs = hc.depth_start[D];
    c.n_far = hc.n_far;
    c.n_p2p = hc.n_p2p;
    c.n_p2p_targets = hc.nseg;
    c.p2p_interactions = hc.interactions;
    // keep a quarter of headroom for the next call
    c.pair_cap = std::max(c.pair_cap, c.n_pairs + c.n_pairs / 4 + 1024);
    break;
    }
    c.attraction_done = true;
    c.lists_valid = cfg.mac_mode == 0;
}

}  // namespace msp
