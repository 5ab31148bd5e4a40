// msp_neuron.cu -- the neuron side of the Model of Structural Plasticity
// (Section 3.1, Table 1), which produces the vacant elements the synapse
// search consumes: electrical activity with Poisson spiking, calcium,
// synaptic-element growth on the Gaussian growth curve, and the deletion of
// synapses a neuron no longer has elements for.
//
// Readings (the paper states the model in words):
//   activity   x <- x + (x0 - x)/tau_x + I + c_in * (edges s -> t whose s
//              spiked in the previous step); the neuron spikes when a uniform
//              draw U in [0,1) (24 bits of Philox) is below x, unless it
//              spiked in one of the last `refractory` steps;
//   calcium    Ca <- Ca - decay * Ca, plus beta on a spike;
//   elements   z <- max(z + g(Ca), 0), g(Ca) = mu (2 exp(-((Ca-xi)/zeta)^2) - 1),
//              xi = (eta + eps)/2, zeta = (eps - eta)/(2 sqrt(ln 2)): zero at
//              eta and eps, mu halfway (the growth curve of the cited model);
//   deletion   a side with more bound synapses than floor(z) deletes the
//              excess, uniformly at random (the excess edges with the
//              smallest Philox priorities, ties by edge position); an edge
//              chosen by either side goes; vacant = floor(z) - bound.
// The state decides integers (a spike, a floor), so every floating-point
// operation is single precision with explicit rounding intrinsics in the
// order written (no contraction into FMAs), and exp is computed here from its
// definition; the result is then reproducible bit for bit.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "msp_scan.cuh"

namespace msp {

namespace {

constexpr uint32_t kTagSpike = 5u, kTagDelAxon = 6u, kTagDelDend = 7u;

__device__ __forceinline__ uint32_t nr_draw(uint64_t seed, uint32_t c0, uint32_t c1,
                                            uint64_t step) {
    uint32_t o[4];
    philox_draw(seed, c0, c1, step, o);
    return o[0];
}

// exp(x), single precision: Cody and Waite's reduction x = n ln 2 + r with
// ln 2 = 0.693359375 - 2.12194440e-4 (n times the first part is exact), the
// degree-7 Taylor polynomial of e^r (|r| <= 0.35) and the scale 2^n; 0 below
// -87.  Rounded operation by operation.
__device__ float nr_expf(float x) {
    if (x < -87.0f) return 0.0f;
    const float n = floorf(__fadd_rn(__fmul_rn(x, 1.44269504f), 0.5f));
    float r = __fadd_rn(x, -__fmul_rn(n, 0.693359375f));
    r = __fadd_rn(r, __fmul_rn(n, 2.12194440e-4f));
    float p = 1.98412698e-4f;
    p = __fadd_rn(__fmul_rn(p, r), 1.38888889e-3f);
    p = __fadd_rn(__fmul_rn(p, r), 8.33333333e-3f);
    p = __fadd_rn(__fmul_rn(p, r), 4.16666667e-2f);
    p = __fadd_rn(__fmul_rn(p, r), 1.66666667e-1f);
    p = __fadd_rn(__fmul_rn(p, r), 0.5f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f);
    const float s = __uint_as_float((uint32_t)((int)n + 127) << 23);
    return __fmul_rn(p, s);
}

// a growth curve's middle and width
struct NrCurve {
    float xi, zeta;
};

__device__ __forceinline__ NrCurve nr_curve(float eta, float eps) {
    NrCurve c;
    c.xi = __fmul_rn(__fadd_rn(eta, eps), 0.5f);
    c.zeta = __fdiv_rn(__fadd_rn(eps, -eta), __fmul_rn(2.0f, 0.832554611f));
    return c;
}

__device__ __forceinline__ float nr_growth(float ca, const NrCurve& c, float mu) {
    const float q = __fdiv_rn(__fadd_rn(ca, -c.xi), c.zeta);
    const float e = nr_expf(-__fmul_rn(q, q));
    return __fmul_rn(mu, __fadd_rn(__fadd_rn(e, e), -1.0f));
}

// The input of a step is event driven: the outgoing edges of each neuron, as
// a compressed list by presynaptic neuron rebuilt at the start of every
// call, and two input-count buffers; a neuron that spikes in step k adds one
// to the next buffer for each of its outgoing edges, which step k + 1 reads
// (and clears).  Edges naming a neuron outside [0, n) are skipped.
__global__ void k_out_degree(const int64_t* __restrict__ n_edges, int64_t cap, int64_t n,
                             const int32_t* __restrict__ pre, const int32_t* __restrict__ post,
                             int32_t* __restrict__ deg) {
    const int64_t m = min(*n_edges, cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = pre[e], b = post[e];
        if (a < 0 || a >= n || b < 0 || b >= n) continue;
        atomicAdd(&deg[a], 1);
    }
}

// targets of each neuron's outgoing edges at [off[s], off[s] + deg[s]) (the
// order inside a neuron's range does not matter: only counts are formed)
__global__ void k_out_fill(const int64_t* __restrict__ n_edges, int64_t cap, int64_t n,
                           const int32_t* __restrict__ pre, const int32_t* __restrict__ post,
                           const int32_t* __restrict__ off, int32_t* __restrict__ cursor,
                           int32_t* __restrict__ targets) {
    const int64_t m = min(*n_edges, cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = pre[e], b = post[e];
        if (a < 0 || a >= n || b < 0 || b >= n) continue;
        targets[off[a] + atomicAdd(&cursor[a], 1)] = b;
    }
}

// the input of the first step of a call: last step's spikes
__global__ void k_seed_input(int64_t n, const uint8_t* __restrict__ spiked,
                             const int32_t* __restrict__ off, const int32_t* __restrict__ deg,
                             const int32_t* __restrict__ targets, int32_t* __restrict__ inp) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x)
        if (spiked[t])
            for (int32_t j = off[t], j1 = off[t] + deg[t]; j < j1; ++j) atomicAdd(&inp[targets[j]], 1);
}

// The state of one neuron through one step (Section 3.1): activity with
// input `in`, the spike draw (o: its random word), calcium, the three element
// counts.  Returns the spike.
struct NrState {
    float x, ca, za, ze, zi;
    uint32_t rf;
};

__device__ __forceinline__ uint32_t nr_spike_word(uint64_t seed, uint32_t t, uint64_t step) {
    return nr_draw(seed, t, kTagSpike << 16, step);
}

__device__ __forceinline__ int nr_update(NrState& v, int32_t in, uint32_t o,
                                         const msp_neuron_params& mp, const NrCurve& axon,
                                         const NrCurve& dend) {
    float d = __fadd_rn(mp.x0, -v.x);
    d = __fdiv_rn(d, mp.tau_x);
    float xt = __fadd_rn(v.x, d);
    xt = __fadd_rn(xt, mp.background);
    xt = __fadd_rn(xt, __fmul_rn(mp.input_per_spike, (float)in));
    v.x = xt;
    int s = 0;
    if (v.rf > 0) {
        v.rf -= 1;
    } else {
        const float u = __fmul_rn((float)(o >> 8), 1.0f / 16777216.0f);
        s = u < xt;
        if (s) v.rf = (uint32_t)mp.refractory;
    }
    float ca = __fadd_rn(v.ca, -__fmul_rn(v.ca, mp.decay_ca));
    if (s) ca = __fadd_rn(ca, mp.beta_ca);
    v.ca = ca;
    const float a = __fadd_rn(v.za, nr_growth(ca, axon, mp.mu));
    const float gd = nr_growth(ca, dend, mp.mu);
    const float e = __fadd_rn(v.ze, gd);
    const float i = __fadd_rn(v.zi, gd);
    v.za = a > 0.0f ? a : 0.0f;
    v.ze = e > 0.0f ? e : 0.0f;
    v.zi = i > 0.0f ? i : 0.0f;
    return s;
}

// The same for two neurons at a time in paired FP32 (each element rounded as
// in the scalar form: the results are the same bit for bit).  The divisors are
// the model's constants, so a division is four paired instructions: with zh =
// RN(1/y) and zl = RN(1/y - zh) from the host, q0 = x zh + x zl is within an ulp
// of x/y, and q0 + (x - q0 y) zh is then the correctly rounded quotient
// (Markstein, IBM J. Res. Dev. 34 (1990); the two-word reciprocal as in
// Brisebarre, Muller and Raina, IEEE Trans. Computers 53 (2004)), for y whose
// significand is not all ones and away from overflow and underflow, which
// nr_fast on the host and nr_safe below make sure of.
struct NrDiv {
    float y, zh, zl;
};
struct NrFast {
    float xi_a, xi_d;
    NrDiv tau, zeta_a, zeta_d;
};

__device__ __forceinline__ float2 nr_both(float v) { return make_float2(v, v); }

// A paired product that stays rounded: a paired product and sum, also with
// explicit rounding, are contracted into one paired FMA (measured: the results
// are the fused ones).  The FMA with an addend of minus zero, which the
// compiler cannot see, is the rounded product.
__constant__ float c_minus_zero = -0.0f;

__device__ __forceinline__ float2 nr_mul2(float2 a, float2 b) {
    return __ffma2_rn(a, b, nr_both(c_minus_zero));
}
__device__ __forceinline__ float2 nr_add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

__device__ __forceinline__ float2 nr_div2(float2 x, const NrDiv& d) {
    const float2 q = __ffma2_rn(x, nr_both(d.zh), nr_mul2(x, nr_both(d.zl)));
    const float2 r = __ffma2_rn(q, nr_both(-d.y), x);
    return __ffma2_rn(r, nr_both(d.zh), q);
}

// nr_expf of both
__device__ __forceinline__ float2 nr_expf2(float2 x) {
    const float2 y = nr_add2(nr_mul2(x, nr_both(1.44269504f)), nr_both(0.5f));
    const float2 n = make_float2(floorf(y.x), floorf(y.y));
    float2 r = nr_add2(x, nr_mul2(n, nr_both(-0.693359375f)));
    r = nr_add2(r, nr_mul2(n, nr_both(2.12194440e-4f)));
    float2 p = nr_both(1.98412698e-4f);
    p = nr_add2(nr_mul2(p, r), nr_both(1.38888889e-3f));
    p = nr_add2(nr_mul2(p, r), nr_both(8.33333333e-3f));
    p = nr_add2(nr_mul2(p, r), nr_both(4.16666667e-2f));
    p = nr_add2(nr_mul2(p, r), nr_both(1.66666667e-1f));
    p = nr_add2(nr_mul2(p, r), nr_both(0.5f));
    p = nr_add2(nr_mul2(p, r), nr_both(1.0f));
    p = nr_add2(nr_mul2(p, r), nr_both(1.0f));
    const float2 s = make_float2(__uint_as_float((uint32_t)((int)n.x + 127) << 23),
                                 __uint_as_float((uint32_t)((int)n.y + 127) << 23));
    const float2 e = nr_mul2(p, s);
    return make_float2(x.x < -87.0f ? 0.0f : e.x, x.y < -87.0f ? 0.0f : e.y);
}

__device__ __forceinline__ float2 nr_growth2(float2 ca, float xi, const NrDiv& zeta, float mu) {
    const float2 q = nr_div2(nr_add2(ca, nr_both(-xi)), zeta);
    const float2 qq = nr_mul2(q, q);
    const float2 e = nr_expf2(make_float2(-qq.x, -qq.y));
    return nr_mul2(nr_both(mu), nr_add2(nr_add2(e, e), nr_both(-1.0f)));
}

// the differences the divisions take are zero or normal numbers of moderate
// size while the state is (the constants are: nr_fast)
__device__ __forceinline__ bool nr_safe(float2 x, float2 ca) {
    return fmaxf(fabsf(x.x), fabsf(x.y)) < 1e18f && fmaxf(fabsf(ca.x), fabsf(ca.y)) < 1e18f &&
           x.x == x.x && x.y == x.y && ca.x == ca.x && ca.y == ca.y;
}

__device__ __forceinline__ uint32_t nr_update2(float2& x, float2& ca, float2& za, float2& ze,
                                               float2& zi, uint32_t (&rf)[2], int32_t in0,
                                               int32_t in1, uint32_t o0, uint32_t o1,
                                               const msp_neuron_params& mp, const NrFast& f) {
    float2 xt = nr_add2(x, nr_div2(nr_add2(nr_both(mp.x0), make_float2(-x.x, -x.y)), f.tau));
    xt = nr_add2(xt, nr_both(mp.background));
    xt = nr_add2(xt, nr_mul2(nr_both(mp.input_per_spike), make_float2((float)in0, (float)in1)));
    x = xt;
    const float2 u = nr_mul2(make_float2((float)(o0 >> 8), (float)(o1 >> 8)),
                                nr_both(1.0f / 16777216.0f));
    const bool s0 = rf[0] == 0 && u.x < xt.x, s1 = rf[1] == 0 && u.y < xt.y;
    rf[0] = s0 ? (uint32_t)mp.refractory : rf[0] - (rf[0] > 0);
    rf[1] = s1 ? (uint32_t)mp.refractory : rf[1] - (rf[1] > 0);
    // ca - decay ca: the product negated by its factor (the same rounding)
    float2 c = nr_add2(ca, nr_mul2(ca, nr_both(-mp.decay_ca)));
    const float2 cb = nr_add2(c, nr_both(mp.beta_ca));
    c = make_float2(s0 ? cb.x : c.x, s1 ? cb.y : c.y);
    ca = c;
    const float2 ga = nr_growth2(c, f.xi_a, f.zeta_a, mp.mu);
    const float2 gd = nr_growth2(c, f.xi_d, f.zeta_d, mp.mu);
    const float2 a = nr_add2(za, ga), e = nr_add2(ze, gd), i = nr_add2(zi, gd);
    za = make_float2(a.x > 0.0f ? a.x : 0.0f, a.y > 0.0f ? a.y : 0.0f);
    ze = make_float2(e.x > 0.0f ? e.x : 0.0f, e.y > 0.0f ? e.y : 0.0f);
    zi = make_float2(i.x > 0.0f ? i.x : 0.0f, i.y > 0.0f ? i.y : 0.0f);
    return (uint32_t)s0 | (uint32_t)s1 << 8;
}

// One step of every neuron: consumes (and clears) its input count in `cur`;
// a spike adds one to `next` for each outgoing edge.  With vec4 set (every
// array 16-byte aligned, the byte arrays 4-byte aligned) a thread takes four
// consecutive neurons with 16-byte loads and stores, so that more of the
// state is in flight per thread; the last n mod 4 neurons (or all, without
// vec4) go one per thread.  The step is bound by the latency of its loads:
// at most 48 registers (no spills) keep five blocks resident per SM.
__global__ void __launch_bounds__(256, 5)
k_neuron_step(int64_t n, int vec4, uint64_t seed, uint64_t step,
                              msp_neuron_params mp, int32_t* __restrict__ cur,
                              int32_t* __restrict__ next, const int32_t* __restrict__ off,
                              const int32_t* __restrict__ deg, const int32_t* __restrict__ targets,
                              float* __restrict__ x, uint8_t* __restrict__ refr,
                              float* __restrict__ calcium, float* __restrict__ za,
                              float* __restrict__ ze, float* __restrict__ zi,
                              uint8_t* __restrict__ spiked) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n4 = vec4 ? n / 4 : 0;
    const NrCurve axon = nr_curve(mp.eta_axon, mp.eps), dend = nr_curve(mp.eta_dend, mp.eps);
    for (int64_t q = tid; q < n4; q += stride) {
        const int4 in4 = reinterpret_cast<const int4*>(cur)[q];
        const float4 x4 = reinterpret_cast<const float4*>(x)[q];
        const float4 c4 = reinterpret_cast<const float4*>(calcium)[q];
        const float4 a4 = reinterpret_cast<const float4*>(za)[q];
        const float4 e4 = reinterpret_cast<const float4*>(ze)[q];
        const float4 i4 = reinterpret_cast<const float4*>(zi)[q];
        const uint32_t r4 = reinterpret_cast<const uint32_t*>(refr)[q];
        reinterpret_cast<int4*>(cur)[q] = make_int4(0, 0, 0, 0);
        const int32_t ins[4] = {in4.x, in4.y, in4.z, in4.w};
        NrState v[4] = {{x4.x, c4.x, a4.x, e4.x, i4.x, r4 & 0xffu},
                        {x4.y, c4.y, a4.y, e4.y, i4.y, (r4 >> 8) & 0xffu},
                        {x4.z, c4.z, a4.z, e4.z, i4.z, (r4 >> 16) & 0xffu},
                        {x4.w, c4.w, a4.w, e4.w, i4.w, r4 >> 24}};
        uint32_t sp = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int s = nr_update(v[k], ins[k], nr_spike_word(seed, (uint32_t)(4 * q + k), step), mp,
                                    axon, dend);
            sp |= (uint32_t)s << (8 * k);
            if (s) {
                // the outgoing edges are read only for the neurons that spiked
                const int32_t j0 = off[4 * q + k], j1 = j0 + deg[4 * q + k];
                for (int32_t j = j0; j < j1; ++j) atomicAdd(&next[targets[j]], 1);
            }
        }
        reinterpret_cast<float4*>(x)[q] = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
        reinterpret_cast<float4*>(calcium)[q] = make_float4(v[0].ca, v[1].ca, v[2].ca, v[3].ca);
        reinterpret_cast<float4*>(za)[q] = make_float4(v[0].za, v[1].za, v[2].za, v[3].za);
        reinterpret_cast<float4*>(ze)[q] = make_float4(v[0].ze, v[1].ze, v[2].ze, v[3].ze);
        reinterpret_cast<float4*>(zi)[q] = make_float4(v[0].zi, v[1].zi, v[2].zi, v[3].zi);
        reinterpret_cast<uint32_t*>(refr)[q] = v[0].rf | (v[1].rf << 8) | (v[2].rf << 16) |
                                               (v[3].rf << 24);
        reinterpret_cast<uint32_t*>(spiked)[q] = sp;
    }
    for (int64_t t = 4 * n4 + tid; t < n; t += stride) {
        const int32_t in = cur[t];
        cur[t] = 0;
        NrState v = {x[t], calcium[t], za[t], ze[t], zi[t], refr[t]};
        const int s = nr_update(v, in, nr_spike_word(seed, (uint32_t)t, step), mp, axon, dend);
        x[t] = v.x;
        calcium[t] = v.ca;
        za[t] = v.za;
        ze[t] = v.ze;
        zi[t] = v.zi;
        refr[t] = (uint8_t)v.rf;
        spiked[t] = (uint8_t)s;
        if (s)
            for (int32_t j = off[t], j1 = off[t] + deg[t]; j < j1; ++j)
                atomicAdd(&next[targets[j]], 1);
    }
}

// Many steps of every neuron in one launch: a block keeps the state of its
// share of the neurons, in groups of four, in shared memory from the first step
// to the last, and only the input counts travel through memory.  One
// cooperative block per SM; a step ends with a grid-wide barrier (the spikes of
// step k are step k + 1's input), whose waiting time holds the next step's
// random draws.  A barrier wait of more than SPINS polls (and four for each edge of
// the network, whose numbers per neuron have no bound) sets timeout_bit
// in *overflow and every later wait is skipped: the kernel always ends (the
// counts are then wrong, and the next synchronising call reports it).
//
// Bound by the step's chain (input counts, update, spikes' edge lists, barrier;
// issue 39 % busy).  100 steps of 1,048,576 neurons: 1.9 ms with a launch per
// step (the state read and written every step, 1.35 waves of five blocks per
// SM, 290 instructions per neuron), 1.41 ms on the chip with 254, 1.17 ms with
// paired FP32 and divisions by reciprocals (174).
struct NrRun {
    int64_t n4, n;              // groups of four; neurons (the last n mod 4 one per thread)
    int per;                    // groups per block
    int n_steps;
    uint64_t seed, first_step;
    msp_neuron_params mp;
    int32_t *inp0, *inp1;       // input counts of even and odd steps
    const int32_t *off, *deg, *targets;
    const int64_t* n_edges;     // of the caller's list, at most cap (null: none)
    int64_t cap;
    float *x, *ca, *za, *ze, *zi;
    uint8_t *refr, *spiked;
    unsigned int* barrier;      // arrivals, zero on entry
    int64_t* overflow;
    int64_t timeout_bit;
    NrFast fast;                // of FAST: the constants allow nr_update2
};
// bytes of shared memory per group: five floats and a random word for each
// neuron, the refractory counts and the spikes as bytes, an entry of the list
// of spiking neurons for each
constexpr int kNrGroupBytes = 6 * 16 + 8 + 8;
constexpr int kNrMaxGroups = 220 * 1024 / kNrGroupBytes;

// A spiking neuron's edges are one thread's work (60 ns an edge; a poll takes
// longer): four polls more for each edge of the network.  Whether the arrivals
// reached the goal.  (Out of line: inside the kernel it made a step 1 % slower.)
__device__ __noinline__ bool nr_wait_longer(volatile unsigned int* arrivals, unsigned int goal,
                                            const int64_t* n_edges, int64_t cap) {
    int64_t more = n_edges ? 4 * min(max(*n_edges, (int64_t)0), cap) : 0;
    while (*arrivals < goal && more > 0) --more;
    return *arrivals >= goal;
}

template <bool FAST, int SPINS>
__global__ void __launch_bounds__(1024, 1) k_neuron_run(NrRun a) {
    extern __shared__ float4 nr_sm[];
    __shared__ int s_dead, s_nsp[2];
    const int T = blockDim.x, per = a.per;
    const int64_t q0 = (int64_t)blockIdx.x * per;
    const int cnt = (int)max((int64_t)0, min((int64_t)per, a.n4 - q0));
    float4 *sx = nr_sm, *sc = sx + per, *sa = sc + per, *se = sa + per, *si = se + per;
    uint4* so = reinterpret_cast<uint4*>(si + per);
    uint32_t *sr = reinterpret_cast<uint32_t*>(so + per), *ss = sr + per;
    uint16_t* sl = reinterpret_cast<uint16_t*>(ss + per);
    const NrCurve axon = nr_curve(a.mp.eta_axon, a.mp.eps),
                  dend = nr_curve(a.mp.eta_dend, a.mp.eps);
    if (threadIdx.x == 0) s_dead = s_nsp[0] = s_nsp[1] = 0;
    auto draw = [&](uint64_t step) {
        for (int i = threadIdx.x; i < cnt; i += T) {
            const uint32_t t = (uint32_t)(4 * (q0 + i));
            so[i] = make_uint4(nr_spike_word(a.seed, t, step), nr_spike_word(a.seed, t + 1, step),
                               nr_spike_word(a.seed, t + 2, step), nr_spike_word(a.seed, t + 3, step));
        }
    };
    for (int i = threadIdx.x; i < cnt; i += T) {
        const int64_t q = q0 + i;
        sx[i] = reinterpret_cast<const float4*>(a.x)[q];
        sc[i] = reinterpret_cast<const float4*>(a.ca)[q];
        sa[i] = reinterpret_cast<const float4*>(a.za)[q];
        se[i] = reinterpret_cast<const float4*>(a.ze)[q];
        si[i] = reinterpret_cast<const float4*>(a.zi)[q];
        sr[i] = reinterpret_cast<const uint32_t*>(a.refr)[q];
    }
    auto spike = [&](int64_t t, int32_t* next) {
        const int32_t j0 = a.off[t], j1 = j0 + a.deg[t];
        for (int32_t e = j0; e < j1; ++e) atomicAdd(&next[a.targets[e]], 1);
    };
    // a thread only touches its own groups: no barrier between these phases
    draw(a.first_step);
    __syncthreads();
    for (int st = 0; st < a.n_steps; ++st) {
        const uint64_t step = a.first_step + (uint64_t)st;
        int32_t* cur = (st & 1) ? a.inp1 : a.inp0;
        int32_t* next = (st & 1) ? a.inp0 : a.inp1;
        for (int i = threadIdx.x; i < cnt; i += T) {
            const int64_t q = q0 + i;
            // counts other SMs added: past the L1
            const int4 in4 = __ldcg(reinterpret_cast<const int4*>(cur) + q);
            const float4 x = sx[i], ca = sc[i], za = sa[i], ze = se[i], zi = si[i];
            const uint4 o = so[i];
            const uint32_t rf = sr[i];
            if (in4.x | in4.y | in4.z | in4.w)
                __stcg(reinterpret_cast<int4*>(cur) + q, make_int4(0, 0, 0, 0));
            uint32_t sp = 0;
            const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
            const float2 c0 = make_float2(ca.x, ca.y), c1 = make_float2(ca.z, ca.w);
            if (FAST && nr_safe(x0, c0) && nr_safe(x1, c1)) {
                float2 v[2][5] = {{x0, c0, make_float2(za.x, za.y), make_float2(ze.x, ze.y),
                                   make_float2(zi.x, zi.y)},
                                  {x1, c1, make_float2(za.z, za.w), make_float2(ze.z, ze.w),
                                   make_float2(zi.z, zi.w)}};
                uint32_t r[2][2] = {{rf & 0xffu, (rf >> 8) & 0xffu}, {(rf >> 16) & 0xffu, rf >> 24}};
                sp = nr_update2(v[0][0], v[0][1], v[0][2], v[0][3], v[0][4], r[0], in4.x, in4.y, o.x,
                                o.y, a.mp, a.fast);
                sp |= nr_update2(v[1][0], v[1][1], v[1][2], v[1][3], v[1][4], r[1], in4.z, in4.w, o.z,
                                 o.w, a.mp, a.fast) << 16;
                sx[i] = make_float4(v[0][0].x, v[0][0].y, v[1][0].x, v[1][0].y);
                sc[i] = make_float4(v[0][1].x, v[0][1].y, v[1][1].x, v[1][1].y);
                sa[i] = make_float4(v[0][2].x, v[0][2].y, v[1][2].x, v[1][2].y);
                se[i] = make_float4(v[0][3].x, v[0][3].y, v[1][3].x, v[1][3].y);
                si[i] = make_float4(v[0][4].x, v[0][4].y, v[1][4].x, v[1][4].y);
                sr[i] = r[0][0] | r[0][1] << 8 | r[1][0] << 16 | r[1][1] << 24;
            } else {
                const int32_t ins[4] = {in4.x, in4.y, in4.z, in4.w};
                const uint32_t ow[4] = {o.x, o.y, o.z, o.w};
                NrState v[4] = {{x.x, ca.x, za.x, ze.x, zi.x, rf & 0xffu},
                                {x.y, ca.y, za.y, ze.y, zi.y, (rf >> 8) & 0xffu},
                                {x.z, ca.z, za.z, ze.z, zi.z, (rf >> 16) & 0xffu},
                                {x.w, ca.w, za.w, ze.w, zi.w, rf >> 24}};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    sp |= (uint32_t)nr_update(v[k], ins[k], ow[k], a.mp, axon, dend) << (8 * k);
                sx[i] = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
                sc[i] = make_float4(v[0].ca, v[1].ca, v[2].ca, v[3].ca);
                sa[i] = make_float4(v[0].za, v[1].za, v[2].za, v[3].za);
                se[i] = make_float4(v[0].ze, v[1].ze, v[2].ze, v[3].ze);
                si[i] = make_float4(v[0].zi, v[1].zi, v[2].zi, v[3].zi);
                sr[i] = v[0].rf | (v[1].rf << 8) | (v[2].rf << 16) | (v[3].rf << 24);
            }
            ss[i] = sp;
            if (sp) {
                int at = atomicAdd(&s_nsp[st & 1], __popc(sp));
                for (uint32_t m = sp; m; m &= m - 1)
                    sl[at++] = (uint16_t)(4 * i + ((__ffs(m) - 1) >> 3));
            }
        }
        __syncthreads();
        // the outgoing edges of the neurons that spiked, one neuron per thread
        for (int k = threadIdx.x; k < s_nsp[st & 1]; k += T) spike(4 * q0 + sl[k], next);
        if (threadIdx.x == 0) s_nsp[(st + 1) & 1] = 0;
        // the last n mod 4 neurons, their state in memory
        const int64_t tid = (int64_t)blockIdx.x * T + threadIdx.x;
        for (int64_t t = 4 * a.n4 + tid; t < a.n; t += (int64_t)gridDim.x * T) {
            const int32_t in = __ldcg(cur + t);
            __stcg(cur + t, 0);
            NrState v = {a.x[t], a.ca[t], a.za[t], a.ze[t], a.zi[t], a.refr[t]};
            const int s = nr_update(v, in, nr_spike_word(a.seed, (uint32_t)t, step), a.mp, axon, dend);
            a.x[t] = v.x;
            a.ca[t] = v.ca;
            a.za[t] = v.za;
            a.ze[t] = v.ze;
            a.zi[t] = v.zi;
            a.refr[t] = (uint8_t)v.rf;
            a.spiked[t] = (uint8_t)s;
            if (s) spike(t, next);
        }
        if (st + 1 == a.n_steps) break;
        // arrive, draw for the next step, wait
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(a.barrier, 1u);
        draw(step + 1);
        if (threadIdx.x == 0 && !s_dead) {
            const unsigned int goal = (unsigned int)(st + 1) * gridDim.x;
            volatile unsigned int* b = a.barrier;
            int spin = 0;
            while (*b < goal && spin < SPINS) ++spin;
            if (*b < goal && !nr_wait_longer(b, goal, a.n_edges, a.cap)) {
                s_dead = 1;
                atomicOr(reinterpret_cast<unsigned long long*>(a.overflow),
                         (unsigned long long)a.timeout_bit);
            }
            __threadfence();
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < cnt; i += T) {
        const int64_t q = q0 + i;
        reinterpret_cast<float4*>(a.x)[q] = sx[i];
        reinterpret_cast<float4*>(a.ca)[q] = sc[i];
        reinterpret_cast<float4*>(a.za)[q] = sa[i];
        reinterpret_cast<float4*>(a.ze)[q] = se[i];
        reinterpret_cast<float4*>(a.zi)[q] = si[i];
        reinterpret_cast<uint32_t*>(a.refr)[q] = sr[i];
        reinterpret_cast<uint32_t*>(a.spiked)[q] = ss[i];
    }
}

// ---------------------------------------------------------------------------
// Update of synapses.  The 3 n sides are groups: neuron t's outgoing synapses
// are group t, its incoming ones of type T group n + 2 t + T.  At 1,048,576
// neurons with 1.5 synapses each: 0.71 ms with both sides' edges sorted whole
// and the list compacted through a copy, 0.29 ms now (the synchronisation of
// the check included).
// ---------------------------------------------------------------------------
constexpr unsigned long long kBadWait = 1ull << 40;

// bound synapses per group; counts the edges naming a neuron outside [0, n),
// and an edge count above the capacity; kBadWait more where a wait before gave up
__global__ void k_bound(const int64_t* __restrict__ n_edges, int64_t cap, int64_t n,
                        const int32_t* __restrict__ pre, const int32_t* __restrict__ post,
                        const uint8_t* __restrict__ typ, int32_t* __restrict__ bound,
                        unsigned long long* __restrict__ bad, const int64_t* __restrict__ overflow,
                        int64_t timeout_bit) {
    const int64_t m0 = *n_edges;
    if (blockIdx.x == 0 && threadIdx.x == 0 && (*overflow & timeout_bit)) atomicAdd(bad, kBadWait);
    if (blockIdx.x == 0 && threadIdx.x == 0 && (m0 < 0 || m0 > cap)) atomicAdd(bad, 1ull);
    const int64_t m = min(max(m0, (int64_t)0), cap);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = pre[e], b = post[e];
        if (a < 0 || a >= n || b < 0 || b >= n) {
            atomicAdd(bad, 1ull);
            continue;
        }
        atomicAdd(&bound[a], 1);
        atomicAdd(&bound[n + 2 * (int64_t)b + (typ[e] ? 1 : 0)], 1);
    }
}

__device__ __forceinline__ int32_t floor_count(float z) { return (int32_t)floorf(z); }

// excess per group: bound - floor(z) when positive; also the edge count (the
// list's own changes under the compaction) and the number of (side, edge) entries
__global__ void k_excess(int64_t n, const float* __restrict__ za, const float* __restrict__ ze,
                         const float* __restrict__ zi, const int32_t* __restrict__ bound,
                         int32_t* __restrict__ excess, const int64_t* __restrict__ n_edges,
                         int64_t* __restrict__ m_out, int64_t* __restrict__ groups_out, int sides,
                         int64_t* __restrict__ entries_out) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *m_out = *n_edges;
        *groups_out = 3 * n;
        *entries_out = sides * *n_edges;
    }
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        excess[t] = max(bound[t] - floor_count(za[t]), 0);
        excess[n + 2 * t] = max(bound[n + 2 * t] - floor_count(ze[t]), 0);
        excess[n + 2 * t + 1] = max(bound[n + 2 * t + 1] - floor_count(zi[t]), 0);
    }
}

// Only the groups with an excess choose among their edges: the others' edges
// stay out of the sort.  Where such a group's edges start in (group, priority)
// order:
struct ScanOverfull {
    const int32_t *bound, *excess;
    __device__ int32_t operator()(int64_t g) const { return excess[g] > 0 ? bound[g] : 0; }
};
// and the entries (side, edge) of the sides side0, side0 + 1, ... in edge
// order, kept where their group has an excess: key (group << 32 | priority),
// value the edge's position
struct DelEntries {
    const int64_t* m;
    int64_t n;
    int side0;
    const int32_t *pre, *post;
    const uint8_t* typ;
    const int32_t* excess;
    __device__ int64_t edge(int64_t i, int& side) const {
        const int64_t me = *m;
        side = side0 + (i >= me);
        return i >= me ? i - me : i;
    }
    __device__ int64_t group(int64_t e, int side) const {
        return side ? n + 2 * (int64_t)post[e] + (typ[e] ? 1 : 0) : (int64_t)pre[e];
    }
    __device__ int32_t operator()(int64_t i) const {
        int side;
        const int64_t e = edge(i, side);
        return excess[group(e, side)] > 0;
    }
};
struct DelKeys {
    DelEntries in;
    uint64_t seed, step;
    uint64_t* key;
    int32_t* val;
    using Read = int64_t;                       // the group, or -1: not kept
    __device__ Read read(int64_t i) const {
        int side;
        const int64_t e = in.edge(i, side), g = in.group(e, side);
        return in.excess[g] > 0 ? g : -1;
    }
    __device__ void operator()(int64_t i, int32_t at, Read g) const {
        if (g < 0) return;
        int side;
        const int64_t e = in.edge(i, side);
        const uint32_t tag = (side ? kTagDelDend : kTagDelAxon) << 16;
        key[at] = ((uint64_t)g << 32) | nr_draw(seed, (uint32_t)e, tag, step);
        val[at] = (int32_t)e;
    }
};

// in sorted order, the first excess[group] edges of each group are deleted;
// g0: the first group of the sorted sides
__global__ void k_del_mark(const int64_t* __restrict__ n_entries, const uint64_t* __restrict__ key,
                           const int32_t* __restrict__ val, const int32_t* __restrict__ start,
                           int64_t g0, const int32_t* __restrict__ excess,
                           uint8_t* __restrict__ del) {
    const int64_t m = *n_entries;
    const int32_t s0 = start[g0];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = (int64_t)(key[i] >> 32);
        if (i - (start[g] - s0) < excess[g]) del[val[i]] = 1;
    }
}

// The list compacted in place, order kept: a tile of edges is in registers
// before it publishes its count, so when a later tile knows where its edges go,
// every edge in that place has been read.  Tiles before the first deleted edge
// write nothing.  A deleted edge leaves its groups' bound counts.
constexpr int kCompactTile = 2048;

__global__ void __launch_bounds__(256)
k_compact_edges(const int64_t* __restrict__ m_dev, int64_t n, const uint8_t* __restrict__ del,
                int32_t* pre, int32_t* post, uint8_t* typ, int32_t* __restrict__ bound,
                int64_t* __restrict__ n_edges, unsigned long long* status,
                int64_t* __restrict__ overflow, int64_t timeout_bit) {
    __shared__ int s_off[64];
    __shared__ int s_tot;
    __shared__ long long s_excl;
    __shared__ int64_t s_tile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t m = *m_dev, ntiles = (m + kCompactTile - 1) / kCompactTile;
    for (;;) {
        if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(&status[0], 1ull);
        __syncthreads();
        const int64_t t = s_tile;
        if (t >= ntiles) break;
        int32_t a[8], b[8];
        uint8_t c[8];
        unsigned keep[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int64_t e = t * kCompactTile + 256 * r + threadIdx.x;
            const bool in = e < m, k = in && !del[e];
            a[r] = in ? pre[e] : 0;
            b[r] = in ? post[e] : 0;
            c[r] = in ? typ[e] : 0;
            keep[r] = __ballot_sync(0xffffffffu, k);
            if (lane == 0) s_off[8 * r + w] = __popc(keep[r]);
            if (in && !k) {
                atomicSub(&bound[a[r]], 1);
                atomicSub(&bound[n + 2 * (int64_t)b[r] + (c[r] ? 1 : 0)], 1);
            }
        }
        __syncthreads();
        if (w == 0) {
            // 64 counts, two per lane
            const int v0 = s_off[2 * lane], v1 = s_off[2 * lane + 1];
            int inc = v0 + v1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            s_off[2 * lane] = inc - v0 - v1;
            s_off[2 * lane + 1] = inc - v1;
            const long long own[1] = {(long long)__shfl_sync(0xffffffffu, inc, 31)};
            long long excl[1];
            __threadfence();          // the tile's reads before its count
            look_back<1>(status + 1, t, own, excl, overflow, timeout_bit, kSpinLimit);
            __threadfence();          // the others' counts before this tile's writes
            if (lane == 0) {
                s_excl = excl[0];
                s_tot = (int)own[0];
            }
        }
        __syncthreads();
        const int64_t excl = s_excl;
        const int cnt = (int)min((int64_t)kCompactTile, m - t * kCompactTile);
        if (excl < t * kCompactTile || s_tot < cnt) {
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if ((keep[r] >> lane) & 1u) {
                    const int64_t q =
                        excl + s_off[8 * r + w] + __popc(keep[r] & ((1u << lane) - 1u));
                    pre[q] = a[r];
                    post[q] = b[r];
                    typ[q] = c[r];
                }
        }
        if (t == ntiles - 1 && threadIdx.x == 0) *n_edges = excl + s_tot;
        __syncthreads();
    }
}

__global__ void k_vacancies(int64_t n, const float* __restrict__ za, const float* __restrict__ ze,
                            const float* __restrict__ zi, const int32_t* __restrict__ bound,
                            uint8_t* __restrict__ va, uint8_t* __restrict__ ve,
                            uint8_t* __restrict__ vi) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        va[t] = (uint8_t)min(max(floor_count(za[t]) - bound[t], 0), 255);
        ve[t] = (uint8_t)min(max(floor_count(ze[t]) - bound[n + 2 * t], 0), 255);
        vi[t] = (uint8_t)min(max(floor_count(zi[t]) - bound[n + 2 * t + 1], 0), 255);
    }
}

// append formed synapses at the end of the edge list (up to the capacity)
__global__ void k_append(const int64_t* __restrict__ n_syn, int64_t syn_cap,
                         const int32_t* __restrict__ sp, const int32_t* __restrict__ sq,
                         const uint8_t* __restrict__ st, const int64_t* __restrict__ n_edges,
                         int64_t cap, int32_t* __restrict__ pre, int32_t* __restrict__ post,
                         uint8_t* __restrict__ typ) {
    const int64_t m0 = *n_edges, k = min(*n_syn, syn_cap);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < k;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = m0 + i;
        if (e >= cap) break;
        pre[e] = sp[i];
        post[e] = sq[i];
        typ[e] = st[i];
    }
}

__global__ void k_append_count(const int64_t* __restrict__ n_syn, int64_t syn_cap, int64_t cap,
                               int64_t* __restrict__ n_edges, int64_t* __restrict__ overflow) {
    const int64_t m = *n_edges + min(*n_syn, syn_cap);
    if (m > cap) {
        *overflow |= 32;
        *n_edges = cap;
    } else {
        *n_edges = m;
    }
}

// The constants of nr_update2, and whether it may be used: divisors of moderate
// size whose significand is not all ones, and subtrahends (x0, the curves'
// middles) not so small that a difference could underflow in the division.
bool nr_fast(const msp_neuron_params& mp, NrFast& f) {
    auto div = [](float y, NrDiv& d) {
        d.y = y;
        d.zh = (float)(1.0 / (double)y);
        d.zl = (float)(1.0 / (double)y - (double)d.zh);
        uint32_t bits;
        std::memcpy(&bits, &y, 4);
        return std::fabs(y) >= 0x1p-30f && std::fabs(y) <= 0x1p30f && (bits & 0x7fffffu) != 0x7fffffu;
    };
    auto moderate = [](float v) { return std::fabs(v) >= 0x1p-60f && std::fabs(v) <= 0x1p60f; };
    const float w = 2.0f * 0.832554611f;
    f.xi_a = (mp.eta_axon + mp.eps) * 0.5f;
    f.xi_d = (mp.eta_dend + mp.eps) * 0.5f;
    const bool ok = div(mp.tau_x, f.tau) & div((mp.eps - mp.eta_axon) / w, f.zeta_a) &
                    div((mp.eps - mp.eta_dend) / w, f.zeta_d);
    return ok && moderate(mp.x0) && moderate(f.xi_a) && moderate(f.xi_d);
}

int bits_for_neuron(int64_t v) {
    int b = 1;
    while (b < 62 && ((int64_t)1 << b) <= v) ++b;
    return b;
}

}  // namespace

void neuron_steps(msp_ctx& c, int64_t n, uint64_t first_step, int n_steps,
                  const msp_neuron_params& mp, const int64_t* n_edges, int64_t cap,
                  const int32_t* pre, const int32_t* post, float* x, uint8_t* refr,
                  float* calcium, float* za, float* ze, float* zi, uint8_t* spiked,
                  cudaStream_t s) {
    NvtxRange nv_("msp neuron_steps");
    if (n <= 0 || n_steps <= 0) return;
    // two input-count buffers, the second at a 16-byte boundary
    const int64_t n_pad = (n + 3) & ~(int64_t)3;
    int32_t* inp = c.nr_inp.ensure<int32_t>((size_t)2 * n_pad);
    int32_t* deg = c.nr_bout.ensure<int32_t>((size_t)n);
    int32_t* off = c.nr_sout.ensure<int32_t>((size_t)n);
    int32_t* cursor = c.nr_xout.ensure<int32_t>((size_t)n);
    int32_t* targets = c.nr_pos.ensure<int32_t>((size_t)std::max<int64_t>(cap, 1));
    int64_t* cnt = c.nr_cnt.ensure<int64_t>(4);
    const int ge = (int)c.sm_count * 8;
    const int gn = grid_for(n, 256, (int64_t)c.sm_count * 16);
    // outgoing edges by presynaptic neuron
    MSP_CUDA(cudaMemsetAsync(deg, 0, (size_t)n * sizeof(int32_t), s));
    MSP_CUDA(cudaMemsetAsync(cursor, 0, (size_t)n * sizeof(int32_t), s));
    MSP_CUDA(cudaMemsetAsync(inp, 0, (size_t)2 * n_pad * sizeof(int32_t), s));
    k_out_degree<<<ge, 256, 0, s>>>(n_edges, cap, n, pre, post, deg);
    MSP_LAUNCH("out_degree");
    dev_set(cnt, n, s);
    scan_dev(c, deg, off, cnt, n, cnt + 2, s);
    k_out_fill<<<ge, 256, 0, s>>>(n_edges, cap, n, pre, post, off, cursor, targets);
    MSP_LAUNCH("out_fill");
    k_seed_input<<<gn, 256, 0, s>>>(n, spiked, off, deg, targets, inp);
    MSP_LAUNCH("seed_input");
    // four neurons per thread where every array allows 16-byte (bytes: 4-byte) access
    auto al = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; };
    const int32_t* inp1 = inp + n_pad;
    const int vec4 = al(inp, 16) && al(inp1, 16) && al(off, 16) && al(deg, 16) && al(x, 16) &&
                     al(calcium, 16) && al(za, 16) && al(ze, 16) && al(zi, 16) && al(refr, 4) &&
                     al(spiked, 4);
    // several steps in one launch while the state fits the chip's shared
    // memory (four neurons to a group, kNrMaxGroups groups an SM: 1.22 M neurons on
    // 152 SMs): one block per SM (fewer for small networks), the
    // groups spread evenly over the blocks
    const int64_t n4 = n / 4;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(c.sm_count, n4 / 64));
    const int64_t per = (n4 + blocks - 1) / blocks;      // groups per block
    if (vec4 && n_steps >= 2 && n4 > 0 && per <= kNrMaxGroups &&
        (uint64_t)n_steps * (uint64_t)blocks < 0xffffffffull) {
        const int64_t rounds = (per + 1023) / 1024;
        const int T = (int)(((per + rounds - 1) / rounds + 31) / 32 * 32);
        NrRun r;
        r.n4 = n4;
        r.n = n;
        r.per = (int)per;
        r.n_steps = n_steps;
        r.seed = c.cfg.seed;
        r.first_step = first_step;
        r.mp = mp;
        r.inp0 = inp;
        r.inp1 = inp + n_pad;
        r.off = off;
        r.deg = deg;
        r.targets = targets;
        r.n_edges = n_edges;
        r.cap = cap;
        r.x = x;
        r.ca = calcium;
        r.za = za;
        r.ze = ze;
        r.zi = zi;
        r.refr = refr;
        r.spiked = spiked;
        r.barrier = reinterpret_cast<unsigned int*>(cnt + 3);
        r.overflow = &dcounts(c)->overflow;
        r.timeout_bit = kScanTimeoutBit;
        const bool fast = nr_fast(mp, r.fast);
        MSP_CUDA(cudaMemsetAsync(r.barrier, 0, sizeof(int64_t), s));
        const size_t smem = (size_t)per * kNrGroupBytes;
        const void* kernel = fast ? (const void*)k_neuron_run<true, kSpinLimit>
                                  : (const void*)k_neuron_run<false, kSpinLimit>;
        allow_shared(kernel, smem, (size_t)kNrMaxGroups * kNrGroupBytes);
        void* args[] = {&r};
        // refused where the process may not have a block on every SM that the
        // device reports: the steps then go one by one
        const cudaError_t e =
            c.refuse_cooperative
                ? cudaErrorCooperativeLaunchTooLarge
                : cudaLaunchCooperativeKernel(kernel, dim3((unsigned)blocks), dim3((unsigned)T), args,
                                              smem, s);
        if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) {
            cuda_check(e, "cudaLaunchCooperativeKernel");
            MSP_LAUNCH("neuron_run");
            return;
        }
        (void)cudaGetLastError();
    }
    const int gv = grid_for(vec4 ? (n + 3) / 4 : n, 256, (int64_t)c.sm_count * 16);
    for (int k = 0; k < n_steps; ++k) {
        int32_t* cur = inp + (size_t)(k & 1) * n_pad;
        int32_t* next = inp + (size_t)((k + 1) & 1) * n_pad;
        k_neuron_step<<<gv, 256, 0, s>>>(n, vec4, c.cfg.seed, first_step + (uint64_t)k, mp, cur,
                                          next, off, deg, targets, x, refr, calcium, za, ze, zi,
                                          spiked);
        MSP_LAUNCH("neuron_step");
    }
}

// The barrier's bounded wait, exercised: the arrivals start one below zero, so the
// one block's own arrival does not complete the first step; it waits at most
// kSelftestSpins polls, records the timeout bit and goes on to the end.
void barrier_wait_selftest(msp_ctx& c, cudaStream_t s) {
    const int64_t n = 256;
    const int groups = (int)n / 4;
    NrRun r = {};
    r.n4 = groups;
    r.n = n;
    r.per = groups;
    r.n_steps = 3;
    r.mp.x0 = r.mp.eps = 0.5f;
    r.mp.tau_x = 5.0f;
    r.mp.eta_axon = r.mp.eta_dend = 0.25f;
    const size_t ints = (size_t)4 * n;               // input counts, edge starts and numbers
    int32_t* zero = c.nr_inp.ensure<int32_t>(ints);
    MSP_CUDA(cudaMemsetAsync(zero, 0, ints * sizeof(int32_t), s));
    r.inp0 = zero;
    r.inp1 = zero + n;
    r.off = zero + 2 * n;
    r.deg = zero + 3 * n;
    r.targets = r.off;                               // no edges: not read
    float* state = c.nr_key0.ensure<float>((size_t)6 * n);
    MSP_CUDA(cudaMemsetAsync(state, 0, (size_t)6 * n * sizeof(float), s));
    r.x = state;
    r.ca = state + n;
    r.za = state + 2 * n;
    r.ze = state + 3 * n;
    r.zi = state + 4 * n;
    r.refr = reinterpret_cast<uint8_t*>(state + 5 * n);
    r.spiked = r.refr + n;
    int64_t* cnt = c.nr_cnt.ensure<int64_t>(4);
    r.barrier = reinterpret_cast<unsigned int*>(cnt + 3);
    MSP_CUDA(cudaMemsetAsync(r.barrier, 0xff, sizeof(int64_t), s));
    r.overflow = &dcounts(c)->overflow;
    r.timeout_bit = kScanTimeoutBit;
    void* args[] = {&r};
    MSP_CUDA(cudaLaunchCooperativeKernel((const void*)k_neuron_run<false, kSelftestSpins>, dim3(1),
                                         dim3(groups), args, (size_t)groups * kNrGroupBytes, s));
    MSP_LAUNCH("barrier_wait_selftest");
}

void update_synapses(msp_ctx& c, int64_t n, uint64_t step, const float* za, const float* ze,
                     const float* zi, int64_t* n_edges, int32_t* pre, int32_t* post, uint8_t* typ,
                     int64_t cap, uint8_t* va, uint8_t* ve, uint8_t* vi, cudaStream_t s) {
    NvtxRange nv_("msp update_synapses");
    if (n <= 0) return;
    const size_t ecap = (size_t)std::max<int64_t>(cap, 1);
    int32_t* bound = c.nr_bin.ensure<int32_t>((size_t)3 * n);
    int32_t* excess = c.nr_xin.ensure<int32_t>((size_t)3 * n);
    int32_t* start = c.nr_sin.ensure<int32_t>((size_t)3 * n);
    uint8_t* del = c.nr_del.ensure<uint8_t>(ecap);
    // bad edges, edges, groups, entries, kept entries
    int64_t* cnt = c.nr_upd.ensure<int64_t>(8);
    // both sides' entries in one sort; one side at a time where they could exceed
    // the sort's 2^31, or where the memory or its limit does not hold both (60
    // bytes an edge, 31 for one side; 42 were enough for a sort per side and a
    // copy of the list)
    const int bits = 32 + bits_for_neuron(3 * n);
    int sides = cap < (1ll << 30) ? 2 : 1;
    auto reserve = [&] {
        const size_t ncap = sides * ecap;
        c.nr_key0.ensure<uint64_t>(ncap);
        c.nr_key1.ensure<uint64_t>(ncap);
        c.nr_val0.ensure<int32_t>(ncap);
        c.nr_val1.ensure<int32_t>(ncap);
        radix_reserve(c, (int64_t)ncap, bits);
        scan_status(c, std::max<int64_t>((int64_t)ncap, 3 * n));
    };
    try {
        reserve();
    } catch (const Error& e) {
        if (sides == 1 || e.code != MSP_ERR_OOM) throw;
        (void)cudaGetLastError();
        for (DBuf* b : {&c.nr_key0, &c.nr_key1, &c.nr_val0, &c.nr_val1, &c.rs_status}) b->release();
        sides = 1;
        reserve();
    }
    const int64_t ncap = sides * (int64_t)ecap;
    uint64_t *k0 = c.nr_key0.get<uint64_t>(), *k1 = c.nr_key1.get<uint64_t>();
    int32_t *v0 = c.nr_val0.get<int32_t>(), *v1 = c.nr_val1.get<int32_t>();
    const int ge = (int)c.sm_count * 8;
    const int gn = grid_for(n, 256, (int64_t)c.sm_count * 16);
    // the edges must name neurons in [0, n) and fit the capacity; a wait of the
    // steps before that gave up is reported here, before the edges change
    MSP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int64_t), s));
    MSP_CUDA(cudaMemsetAsync(bound, 0, (size_t)3 * n * sizeof(int32_t), s));
    k_bound<<<ge, 256, 0, s>>>(n_edges, cap, n, pre, post, typ, bound,
                               reinterpret_cast<unsigned long long*>(cnt), &dcounts(c)->overflow,
                               kScanTimeoutBit);
    MSP_LAUNCH("bound");
    int64_t bad = 0;
    MSP_CUDA(cudaMemcpyAsync(&bad, cnt, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MSP_CUDA(cudaStreamSynchronize(s));
    if ((unsigned long long)bad >= kBadWait) pull_counts(c, s);      // throws
    if (bad) throw Error(MSP_ERR_INVALID_ARG, "an edge names a neuron outside [0, n), or the "
                                              "edge count exceeds the capacity");
    MSP_CUDA(cudaMemsetAsync(del, 0, ecap, s));
    k_excess<<<gn, 256, 0, s>>>(n, za, ze, zi, bound, excess, n_edges, cnt + 1, cnt + 2, sides,
                                cnt + 3);
    MSP_LAUNCH("excess");
    scan_launch(c, ScanOverfull{bound, excess}, ScanStore{start}, ScanTotal{nullptr}, cnt + 2, 3 * n,
                s);
    const bool odd = radix_from_tmp(ncap, bits);
    for (int side0 = 0; side0 < 2; side0 += sides) {
        const DelEntries in{cnt + 1, n, side0, pre, post, typ, excess};
        scan_launch(c, in, DelKeys{in, c.cfg.seed, step, odd ? k1 : k0, odd ? v1 : v0},
                    ScanTotal{cnt + 4}, cnt + 3, ncap, s);
        radix_sort_dev(c, k0, v0, k1, v1, cnt + 4, ncap, bits, s);
        k_del_mark<<<ge, 256, 0, s>>>(cnt + 4, k0, v0, start, side0 ? n : 0, excess, del);
        MSP_LAUNCH("del_mark");
    }
    // compaction, order kept; the bound counts follow
    const int64_t tiles = std::max<int64_t>((cap + kCompactTile - 1) / kCompactTile, 1);
    unsigned long long* st = c.sd_tmp.ensure<unsigned long long>((size_t)tiles + 1);
    MSP_CUDA(cudaMemsetAsync(st, 0, ((size_t)tiles + 1) * sizeof(unsigned long long), s));
    k_compact_edges<<<(unsigned)std::min<int64_t>(tiles, (int64_t)c.sm_count * 4), 256, 0, s>>>(
        cnt + 1, n, del, pre, post, typ, bound, n_edges, st, &dcounts(c)->overflow, kScanTimeoutBit);
    MSP_LAUNCH("compact_edges");
    k_vacancies<<<gn, 256, 0, s>>>(n, za, ze, zi, bound, va, ve, vi);
    MSP_LAUNCH("vacancies");
}

void append_synapses(msp_ctx& c, const int64_t* n_syn, int64_t syn_cap, const int32_t* sp,
                     const int32_t* sq, const uint8_t* st, int64_t* n_edges, int32_t* pre,
                     int32_t* post, uint8_t* typ, int64_t cap, cudaStream_t s) {
    NvtxRange nv_("msp append_synapses");
    DevCounts* dc = dcounts(c);
    k_append<<<(int)c.sm_count * 8, 256, 0, s>>>(n_syn, syn_cap, sp, sq, st, n_edges, cap, pre,
                                                  post, typ);
    MSP_LAUNCH("append");
    k_append_count<<<1, 1, 0, s>>>(n_syn, syn_cap, cap, n_edges, &dc->overflow);
    MSP_LAUNCH("append_count");
    pull_counts(c, s);
    if (c.hcount->overflow & 32) {
        dev_set(&dc->overflow, c.hcount->overflow & ~32ll, s);
        throw Error(MSP_ERR_CAPACITY, "edge list capacity exceeded: the excess synapses were dropped");
    }
}

}  // namespace msp
