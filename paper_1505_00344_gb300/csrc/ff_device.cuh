// ff_device.cuh -- device code of the integrator: kernel arguments, the
// per-system right-hand sides f(x, p) in FP32, the RK4 / Euler steppers and the
// persistent integration kernel template.
//
// Layout: state is structure-of-arrays, plane k (state variable k) at
// x + k * pitch, pitch a multiple of 256 floats, so a thread owning PPT
// consecutive particles reads and writes each plane with one PPT*4-byte vector
// access (16 bytes at PPT = 4).  Each thread keeps its particles' state in
// registers for all steps of a launch: the only global traffic of an
// n-step launch is one read and one write of the state (plus the Kahan
// compensation and the per-particle parameter when enabled).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ff.h"
#include "ff_draw.cuh"
#include "ff_project.cuh"

namespace ff {

constexpr float kLog2e = 1.4426950408889634f;

// Base-2 exponential and reciprocal as PTX's approximate instructions with
// subnormal inputs and results flushed to zero (.ftz).  Supporting subnormals
// costs extra instructions per call (ncu counted 195 fewer per HH3 particle-step
// with these); no argument here is subnormal, and a subnormal exponential only
// ever meets 1 + e, which rounds to 1 either way.  Accuracy is checked through
// the parity tests against the FP64 oracle.
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Work handed out to warps as they come free.  A persistent grid's scheduler favours its older
// warps, so equal shares leave some warps done early and the rest alone at the end (11.4 of 16
// warps of the Lorenz adjoint sweep were active on average).  Each warp takes its own task first
// and then the next one from the queue; the last warp to find none clears the queue for the
// next launch, so launches on one stream, also replayed from a graph, share one.
struct WorkQueue {
    unsigned next;  // tasks handed out beyond the first of every warp
    unsigned done;  // warps that found none
};

// f(task) for the calling warp's tasks of 0 .. n_tasks - 1 (n_tasks < 2^31), all its lanes
// together; the queue serves `blocks` blocks, of which this is number `block`.
template <class F>
__device__ __forceinline__ void warp_tasks(WorkQueue* queue, int64_t n_tasks, unsigned block, unsigned blocks, F&& f) {
    const unsigned warps = blocks * (blockDim.x >> 5), lane = threadIdx.x & 31;
    // warp-major as warp_major_first: a partial first round spreads over all blocks
    for (int64_t w = (int64_t)(threadIdx.x >> 5) * blocks + block; w < n_tasks;) {
        f(w);
        __syncwarp();
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(&queue->next, 1u);
        w = (int64_t)warps + __shfl_sync(0xffffffffu, t, 0);
    }
    if (lane == 0 && atomicInc(&queue->done, warps - 1) == warps - 1) atomicExch(&queue->next, 0u);
}
template <class F>
__device__ __forceinline__ void warp_tasks(WorkQueue* queue, int64_t n_tasks, F&& f) {
    warp_tasks(queue, n_tasks, blockIdx.x, gridDim.x, f);
}

struct IntegrateArgs {
    float* x;              // state planes
    float* comp;           // Kahan compensation planes (KAHAN only)
    const float* pparam;   // per-particle parameter values (PP only)
    int64_t n_vec;         // work items = particles processed / PPT
    int64_t pitch;         // floats between planes
    int64_t n_steps;       // steps in this launch
    int dim;               // planes actually stored (LINEAR may use fewer than its DIM)
    int n_groups;
    int pidx;              // parameter replaced by pparam (PP only)
    int pad_;
    int64_t gstart[FF_MAX_GROUPS];  // first particle of each group
    float gh[FF_MAX_GROUPS];        // signed step of each group
    float p[FF_MAX_PARAMS];         // system parameters (FP32)
    int64_t gend[FF_MAX_GROUPS];    // one past the last processed particle of each group
    int gblk[FF_MAX_GROUPS + 1];    // group-uniform kernels: first block of each group (prefix)
    // particle reset (RESET variants only)
    const struct ResetTable* reset;  // group boxes, sizes, seeds and state bounds (device)
    uint32_t* age;                   // steps since each particle's last reset
    uint32_t* resets;                // resets of each particle
    int64_t step0;                   // global step number before this launch
    int check_every;
    uint32_t max_age;                // 0 = no age limit
    // fused projection + splat after the last step (group-uniform packed Lorenz kernel only)
    int64_t n_real;                  // seeded particles (the rest are padding)
    ViewArgs view;
    // taped runs: before step ck_first + k * ck_every of this launch (k = 0, 1, ... while below
    // n_steps) the state is written to checkpoint slot ck_slot0 + k; ckpt null: no checkpoints
    float* ckpt;                     // slot q at ckpt + q * ck_stride (dim planes of pitch floats)
    int64_t ck_stride;
    int ck_first, ck_every, ck_slot0, ck_pad_;
    // kernels that hand out their work: the system's queues, one per group (ungrouped kernels use the first)
    WorkQueue* queue;
};

// Checkpoint slot for the state as the launch loads it (a chunk that starts with
// the launch), or null.  The kernels write it before any step or change of form.
__device__ __forceinline__ float* start_checkpoint(const IntegrateArgs& a) {
    return (a.ckpt && a.ck_first == 0) ? a.ckpt + (int64_t)a.ck_slot0 * a.ck_stride : nullptr;
}

// The step loop of one launch.  step() advances the state one step; before each
// later checkpoint step of a taped run, save(slot) writes the state to its slot
// in the form, and with the roundings, of a launch that ends there followed by
// one that starts there, so a taped run passes through the states of a run split
// into launches at its checkpoints.
// TAPE false compiles the checkpoints out (kernels that never run taped).
template <int UNROLL, bool TAPE = true, class Step, class Save>
__device__ __forceinline__ void run_steps(const IntegrateArgs& a, int n_steps, Step&& step, Save&& save) {
    if constexpr (!TAPE) {
#pragma unroll UNROLL
        for (int s = 0; s < n_steps; ++s) step();
    } else {
        const bool at0 = a.ckpt && a.ck_first == 0;  // written at load (start_checkpoint)
        int next = a.ckpt ? (at0 ? a.ck_every : a.ck_first) : n_steps;
        int slot = a.ck_slot0 + (at0 ? 1 : 0);
        int s = 0;
        for (;;) {
            const int end = next < n_steps ? next : n_steps;
#pragma unroll UNROLL
            for (; s < end; ++s) step();
            if (s >= n_steps) break;
            save(slot);
            ++slot;
            next += a.ck_every;
        }
    }
}

// Reset data of a system, in device memory (read only when a particle resets).
struct ResetTable {
    DrawBox box[FF_MAX_GROUPS][FF_MAX_DIM];
    int64_t count[FF_MAX_GROUPS];             // particles of the whole group (a slice's is its group's)
    int64_t first[FF_MAX_GROUPS];             // index within the whole group of the group's first particle
    uint64_t seed[FF_MAX_GROUPS];
    float blo[FF_MAX_DIM], bhi[FF_MAX_DIM];
    int has_bounds;
};

// ---------------------------------------------------------------------------
// Right-hand sides.  Each has DIM (registers per particle state), NP (params)
// and f(x, p, dx).  All arithmetic in FP32; exp via ex2_ftz with the log2(e)
// factor folded into the argument, reciprocals via rcp_ftz.
// ---------------------------------------------------------------------------

// Linear test system dx/dt = A x, A padded to 8x8 (row-major) by the host;
// unused rows/columns are zero so padded components stay zero.
struct Linear {
    static constexpr int DIM = 8;
    static constexpr int NP = 64;
    static constexpr int MAX_BLOCK = 256;  // room for 64 parameters in registers
    __device__ __forceinline__ static void f(const float (&x)[DIM], const float* p, float (&dx)[DIM]) {
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < DIM; ++j) s = fmaf(p[i * DIM + j], x[j], s);
            dx[i] = s;
        }
    }
};

// Harmonic oscillator: dx = v, dv = -w^2 x.
struct Harmonic {
    static constexpr int DIM = 2;
    static constexpr int NP = 1;
    static constexpr int MAX_BLOCK = 512;
    __device__ __forceinline__ static void f(const float (&x)[DIM], const float* p, float (&dx)[DIM]) {
        dx[0] = x[1];
        dx[1] = -(p[0] * p[0]) * x[0];
    }
};

// Wilson-Cowan E-I pair (paper Eq. 1-2):
//   tauE dE = -E + S(wEE E - wEI I + P),  tauI dI = -I + S(wIE E - wII I + Q),
//   S(a) = 1 / (1 + exp(-gain (a - threshold))).
struct WilsonCowan {
    static constexpr int DIM = 2;
    static constexpr int NP = 10;
    static constexpr int MAX_BLOCK = 512;
    __device__ __forceinline__ static void f(const float (&x)[DIM], const float* p, float (&dx)[DIM]) {
        const float E = x[0], I = x[1];
        // the logistic's exponent -gain (a - th), a = wE E - wI I + drive, as one affine form
        // of E and I in base 2 (the constants depend on the parameters only, so a step loop
        // forms them once), and (S - x) / tau as S / tau - x / tau: from a stage point to its
        // derivative the dependent chain is two FMAs, ex2, an add, rcp and one FMA
        const float g2 = p[8] * kLog2e;
        const float argE = fmaf(-g2 * p[0], E, fmaf(g2 * p[1], I, g2 * (p[9] - p[4])));
        const float argI = fmaf(-g2 * p[2], E, fmaf(g2 * p[3], I, g2 * (p[9] - p[5])));
        const float SE = rcp_ftz(1.0f + ex2_ftz(argE)), SI = rcp_ftz(1.0f + ex2_ftz(argI));
        const float iE = __fdividef(1.0f, p[6]), iI = __fdividef(1.0f, p[7]);
        dx[0] = fmaf(SE, iE, -E * iE);
        dx[1] = fmaf(SI, iI, -I * iI);
    }
};

// Lorenz (paper Eq. 3-5): dx = sigma (y - x), dy = x (r - z) - y, dz = x y - beta z.
struct Lorenz {
    static constexpr int DIM = 3;
    static constexpr int NP = 3;
    static constexpr int MAX_BLOCK = 512;
    __device__ __forceinline__ static void f(const float (&x)[DIM], const float* p, float (&dx)[DIM]) {
        dx[0] = p[0] * (x[1] - x[0]);
        dx[1] = fmaf(x[0], p[1] - x[2], -x[1]);
        dx[2] = fmaf(x[0], x[1], -(p[2] * x[2]));
    }
};

// Three Hodgkin-Huxley neurons (paper Eq. 6-11), state (V, m, h, n, s) per
// neuron, all-to-all synapses; rates of Hodgkin & Huxley 1952, rest near -65 mV.
// The rate exponentials share one exp2: with u = V + 65 and q = exp(-u/80),
// exp(-u/20) = q^4, exp(-u/10) = q^8, and exp(-(V+40)/10), exp(-(V+55)/10),
// exp(-(V+35)/10) are e^2.5, e^1 and e^3 times q^8; beta_m and the synaptic
// sigmoid take one exp2 each, their constant factors folded into the exponent.
// The four reciprocals are formed two at a time (1/a = b / (a b)).  alpha_m,
// alpha_n = v / (1 - exp(-v/10)) switch to the Bernoulli series for |v/10| <
// 0.5, where the FP32 difference would cancel.  5 MUFU operations per neuron.
//
// One neuron's right-hand side is written once over a lane type: O = HHScalar
// (one neuron) or, further below, the packed pair type (two lanes of one f32x2
// register).  Every operation is explicit, so both forms give the same bits lane
// by lane -- with one care: the toolchain fuses an f32x2 product whose only use
// is an f32x2 addition or subtraction into one fused operation, which the float
// form keeps as two roundings, so such places are written as explicit fused
// operations (checked on 65,536 random neuron states: no lane differs).
struct HHScalar {
    using T = float;
    using M = bool;
    __device__ __forceinline__ static T k(float c) { return c; }
    __device__ __forceinline__ static T add(T a, T b) { return __fadd_rn(a, b); }
    __device__ __forceinline__ static T sub(T a, T b) { return __fsub_rn(a, b); }
    __device__ __forceinline__ static T mul(T a, T b) { return __fmul_rn(a, b); }
    __device__ __forceinline__ static T fma(T a, T b, T c) { return fmaf(a, b, c); }
    __device__ __forceinline__ static T ex2(T a) { return ex2_ftz(a); }
    __device__ __forceinline__ static T rcp(T a) { return rcp_ftz(a); }
    __device__ __forceinline__ static M small(T y) { return fabsf(y) < 0.5f; }
    __device__ __forceinline__ static T sel(M c, T a, T b) { return c ? a : b; }
    // a - t y with one rounding
    __device__ __forceinline__ static T fms(T t, T y, T a) { return fmaf(-t, y, a); }
};

// Parameter-derived constants of the neuron right-hand side.
// The conductances come divided by the capacitance C (and the caller passes the drive as
// I_i / C), so that dV/dt is the current sum itself.
template <class O> struct HHConst {
    typename O::T gNaC, gKC, gLC, ENa, EK, EL, gsynC, Esyn, inv_tr, neg_inv_td, neg_sig2, sig2_theta;
};

template <class O>
__device__ __forceinline__ HHConst<O> hh_const(const float* p) {
    HHConst<O> c;
    const float invC = __fdividef(1.0f, p[0]);
    c.gNaC = O::k(__fmul_rn(p[1], invC));
    c.gKC = O::k(__fmul_rn(p[2], invC));
    c.gLC = O::k(__fmul_rn(p[3], invC));
    c.ENa = O::k(p[4]);
    c.EK = O::k(p[5]);
    c.EL = O::k(p[6]);
    c.gsynC = O::k(__fmul_rn(p[7], invC));
    c.Esyn = O::k(p[8]);
    c.inv_tr = O::k(__fdividef(1.0f, p[12]));
    c.neg_inv_td = O::k(-__fdividef(1.0f, p[13]));
    const float sig2 = p[14] * kLog2e;
    c.neg_sig2 = O::k(-sig2);
    c.sig2_theta = O::k(sig2 * p[15]);
    return c;
}

// Bernoulli series of y / (1 - exp(-y)) = 1 + y/2 + y^2/12 - y^4/720 + y^6/30240
// (the next term, -y^8/1209600, is below 3.3e-9 for |y| < 0.5).
template <class O>
__device__ __forceinline__ typename O::T bernoulli_series_t(typename O::T y) {
    const auto y2 = O::mul(y, y);
    const auto even = O::fma(y2, O::fma(y2, O::fma(y2, O::k(1.0f / 30240.0f), O::k(-1.0f / 720.0f)),
                                        O::k(1.0f / 12.0f)), O::k(1.0f));
    return O::fma(O::k(0.5f), y, even);
}

// Derivatives of one neuron: V, m, h, n, s its state, `others` the sum of the
// other neurons' s, `driveC` its injected current divided by C (hh_drive_c).
template <class O>
__device__ __forceinline__ void hh_neuron(typename O::T V, typename O::T m, typename O::T h, typename O::T n,
                                          typename O::T s, typename O::T others, typename O::T driveC,
                                          const HHConst<O>& c, typename O::T (&d)[5]) {
    using T = typename O::T;
    constexpr float kE25 = 12.182493960703473f;  // e^2.5
    constexpr float kE1 = 2.718281828459045f;    // e^1
    constexpr float kE3 = 20.085536923187668f;   // e^3
    // q = e^(-(V+65)/80) = 2^(kQ V + kQ0); beta_m = 4 e^(-(V+65)/18) = 2^(kB V + kB0)
    constexpr float kQ = -kLog2e / 80.0f, kQ0 = 65.0f * (-kLog2e / 80.0f);
    constexpr float kB = -kLog2e / 18.0f, kB0 = 65.0f * (-kLog2e / 18.0f) + 2.0f;
    const T one = O::k(1.0f);
    const T q = O::ex2(O::fma(V, O::k(kQ), O::k(kQ0)));
    const T q2 = O::mul(q, q), q4 = O::mul(q2, q2), q8 = O::mul(q4, q4);
    const T bm = O::ex2(O::fma(V, O::k(kB), O::k(kB0)));
    const T ah = O::mul(O::k(0.07f), q4);
    const T es = O::ex2(O::fma(c.neg_sig2, V, c.sig2_theta));  // e^(sig (theta - V))
    // alpha_m = g(ym), alpha_n = g(yn) / 10 with g(y) = y / (1 - e^-y),
    // ym = (V + 40) / 10, yn = (V + 55) / 10, e^-ym = e^2.5 q^8, e^-yn = e q^8
    const T ym = O::fma(V, O::k(0.1f), O::k(4.0f)), yn = O::fma(V, O::k(0.1f), O::k(5.5f));
    const auto sm = O::small(ym), sn = O::small(yn);  // series there
    const T dm = O::sel(sm, one, O::fma(O::k(-kE25), q8, one));
    const T dn = O::sel(sn, one, O::fma(O::k(-kE1), q8, one));
    const T rmn = O::rcp(O::mul(dm, dn));
    // yn - ym = 1.5, so at most one of the two lies in the series band: one series serves both
    const T ser = bernoulli_series_t<O>(O::sel(sm, ym, yn));
    const T am = O::sel(sm, ser, O::mul(O::mul(ym, dn), rmn));
    const T an = O::mul(O::k(0.1f), O::sel(sn, ser, O::mul(O::mul(yn, dm), rmn)));
    // beta_h = 1 / (1 + e^3 q^8), act = 1 / (1 + es)
    const T ph = O::fma(O::k(kE3), q8, one), ps = O::add(one, es);
    const T r = O::rcp(O::mul(ph, ps));
    const T act = O::mul(ph, r);  // beta_h = ps r enters only the h gate, fused there
    const T m3h = O::mul(O::mul(O::mul(m, m), m), h);
    const T n2 = O::mul(n, n), n4 = O::mul(n2, n2);
    // dV/dt = (I_i + sum of g (E - V)) / C with every term already divided by C
    T u = O::fma(c.gLC, O::sub(c.EL, V), driveC);
    u = O::fma(O::mul(c.gNaC, m3h), O::sub(c.ENa, V), u);
    u = O::fma(O::mul(c.gKC, n4), O::sub(c.EK, V), u);
    u = O::fma(O::mul(c.gsynC, others), O::sub(c.Esyn, V), u);
    d[0] = u;
    // gates: a (1 - y) - b y = a - (a + b) y, with one rounding on both lane types (the
    // toolchain would fuse the f32x2 form of an unfused product and difference anyway)
    d[1] = O::fms(O::add(am, bm), m, am);
    d[2] = O::fms(O::fma(ps, r, ah), h, ah);  // ah + bh with bh = ps r, fused likewise
    d[3] = O::fms(O::fma(O::k(0.125f), q, an), n, an);  // beta_n = q / 8, an exact product
    d[4] = O::fma(O::mul(act, c.inv_tr), O::sub(one, s), O::mul(s, c.neg_inv_td));
}

// Neuron i's drive I_i / C, formed the same way on every path (one rounding).
__device__ __forceinline__ float hh_drive_c(const float* p, int i) {
    return __fmul_rn(p[9 + i], __fdividef(1.0f, p[0]));
}

struct HH3 {
    static constexpr int DIM = 15;
    static constexpr int NP = 16;
    static constexpr int MAX_BLOCK = 256;  // 15-dimensional state, stages and rates in registers
    static constexpr int MIN_BLOCKS = 3;   // resident blocks of MAX_BLOCK threads the register budget aims at
    __device__ __forceinline__ static void f(const float (&x)[DIM], const float* p, float (&dx)[DIM]) {
        const HHConst<HHScalar> c = hh_const<HHScalar>(p);
        const float s_sum = __fadd_rn(__fadd_rn(x[4], x[9]), x[14]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float d[5];
            hh_neuron<HHScalar>(x[5 * i], x[5 * i + 1], x[5 * i + 2], x[5 * i + 3], x[5 * i + 4],
                                __fsub_rn(s_sum, x[5 * i + 4]), hh_drive_c(p, i), c, d);
#pragma unroll
            for (int k = 0; k < 5; ++k) dx[5 * i + k] = d[k];
        }
    }
};

// ---------------------------------------------------------------------------
// Steppers.  acc() returns the stage-weighted sum a and its scale sc so that
// the step is x += sc * a; the update (plain or compensated) is applied by the
// kernel.  RK4: k1 = f(x), k2 = f(x + h/2 k1), k3 = f(x + h/2 k2),
// k4 = f(x + h k3), a = k1 + 2 k2 + 2 k3 + k4, sc = h/6.  Euler: a = f(x), sc = h.
// ---------------------------------------------------------------------------

template <class R>
struct GenericRK4 {
    static constexpr int D = R::DIM;
    float h1, h2, h6;
    const float* p;
    __device__ __forceinline__ void init(float h, const float* prm) {
        h1 = h;
        h2 = 0.5f * h;
        h6 = h * (1.0f / 6.0f);
        p = prm;
    }
    __device__ __forceinline__ void to_internal(float (&)[D]) const {}
    __device__ __forceinline__ void from_internal(float (&)[D]) const {}
    __device__ __forceinline__ void acc(const float (&x)[D], float (&a)[D], float (&sc)[D]) const {
        float k[D], xs[D];
        if constexpr (D > 8) {
            // large systems: one copy of f in a loop over the four stages, so the step's
            // code fits the instruction caches (the weights 1 make fmaf(1, k, a) = a + k,
            // so the result is the same as the unrolled form's)
#pragma unroll
            for (int i = 0; i < D; ++i) { xs[i] = x[i]; a[i] = 0.0f; }
#pragma unroll 1
            for (int st = 0; st < 4; ++st) {
                R::f(xs, p, k);
                const float w = (st == 1 || st == 2) ? 2.0f : 1.0f;  // fmaf(1, k, 0) = k
#pragma unroll
                for (int i = 0; i < D; ++i) a[i] = fmaf(w, k[i], a[i]);
                if (st == 3) break;
                const float c = (st == 2) ? h1 : h2;
#pragma unroll
                for (int i = 0; i < D; ++i) xs[i] = fmaf(c, k[i], x[i]);
            }
#pragma unroll
            for (int i = 0; i < D; ++i) sc[i] = h6;
        } else {
            R::f(x, p, k);
#pragma unroll
            for (int i = 0; i < D; ++i) { a[i] = k[i]; xs[i] = fmaf(h2, k[i], x[i]); }
            R::f(xs, p, k);
#pragma unroll
            for (int i = 0; i < D; ++i) { a[i] = fmaf(2.0f, k[i], a[i]); xs[i] = fmaf(h2, k[i], x[i]); }
            R::f(xs, p, k);
#pragma unroll
            for (int i = 0; i < D; ++i) { a[i] = fmaf(2.0f, k[i], a[i]); xs[i] = fmaf(h1, k[i], x[i]); }
            R::f(xs, p, k);
#pragma unroll
            for (int i = 0; i < D; ++i) { a[i] = a[i] + k[i]; sc[i] = h6; }
        }
    }
};

template <class R>
struct GenericEuler {
    static constexpr int D = R::DIM;
    float h1;
    const float* p;
    __device__ __forceinline__ void init(float h, const float* prm) { h1 = h; p = prm; }
    __device__ __forceinline__ void to_internal(float (&)[D]) const {}
    __device__ __forceinline__ void from_internal(float (&)[D]) const {}
    __device__ __forceinline__ void acc(const float (&x)[D], float (&a)[D], float (&sc)[D]) const {
        R::f(x, p, a);
#pragma unroll
        for (int i = 0; i < D; ++i) sc[i] = h1;
    }
};

// RK4 on Lorenz with sigma folded into the x-component's stage and final
// scales: with d = y - x, k_x = sigma d, so x + c h k_x = x + (c h sigma) d and
// the x-part of the weighted sum is carried in units of d.  Same arithmetic
// as the generic stepper up to rounding, 41 instead of 45 FP32 instructions.
struct LorenzRK4 {
    static constexpr int D = 3;
    float h1, h2, h6, sh1, sh2, sh6, r, b;
    __device__ __forceinline__ void init(float h, const float* prm) {
        const float s = prm[0];
        r = prm[1];
        b = prm[2];
        h1 = h;
        h2 = 0.5f * h;
        h6 = h * (1.0f / 6.0f);
        sh1 = s * h1;
        sh2 = s * h2;
        sh6 = s * h6;
    }
    __device__ __forceinline__ void to_internal(float (&)[D]) const {}
    __device__ __forceinline__ void from_internal(float (&)[D]) const {}
    __device__ __forceinline__ void acc(const float (&x)[D], float (&a)[D], float (&sc)[D]) const {
        float d, ky, kz, X, Y, Z;
        // stage 1
        d = x[1] - x[0];
        ky = fmaf(x[0], r - x[2], -x[1]);
        kz = fmaf(x[0], x[1], -(b * x[2]));
        a[0] = d; a[1] = ky; a[2] = kz;
        X = fmaf(sh2, d, x[0]); Y = fmaf(h2, ky, x[1]); Z = fmaf(h2, kz, x[2]);
        // stage 2
        d = Y - X;
        ky = fmaf(X, r - Z, -Y);
        kz = fmaf(X, Y, -(b * Z));
        a[0] = fmaf(2.0f, d, a[0]); a[1] = fmaf(2.0f, ky, a[1]); a[2] = fmaf(2.0f, kz, a[2]);
        X = fmaf(sh2, d, x[0]); Y = fmaf(h2, ky, x[1]); Z = fmaf(h2, kz, x[2]);
        // stage 3
        d = Y - X;
        ky = fmaf(X, r - Z, -Y);
        kz = fmaf(X, Y, -(b * Z));
        a[0] = fmaf(2.0f, d, a[0]); a[1] = fmaf(2.0f, ky, a[1]); a[2] = fmaf(2.0f, kz, a[2]);
        X = fmaf(sh1, d, x[0]); Y = fmaf(h1, ky, x[1]); Z = fmaf(h1, kz, x[2]);
        // stage 4
        d = Y - X;
        ky = fmaf(X, r - Z, -Y);
        kz = fmaf(X, Y, -(b * Z));
        a[0] = a[0] + d; a[1] = a[1] + ky; a[2] = a[2] + kz;
        sc[0] = sh6; sc[1] = h6; sc[2] = h6;
    }
};

// RK4 on Lorenz in the shifted variable zt = z - r.  RK4 commutes with affine
// changes of variables, so this is the same map as the unshifted step up to
// rounding; in zt the RHS reads  dx = sigma d,  dy = -(x zt + y),
// dzt = x y - beta zt - beta r, which saves the (r - z) subtraction: 37 FP32
// instructions per step (negations are free operand modifiers).  The shift is
// applied once per launch on load and undone on store.
struct LorenzRK4Shift {
    static constexpr int D = 3;
    float h1, h2, h6, sh1, sh2, sh6, r, nb, nbr;
    __device__ __forceinline__ void init(float h, const float* prm) {
        const float s = prm[0];
        r = prm[1];
        nb = -prm[2];
        nbr = nb * r;
        h1 = h;
        h2 = 0.5f * h;
        h6 = h * (1.0f / 6.0f);
        sh1 = s * h1;
        sh2 = s * h2;
        sh6 = s * h6;
    }
    __device__ __forceinline__ void to_internal(float (&x)[D]) const { x[2] = x[2] - r; }
    __device__ __forceinline__ void from_internal(float (&x)[D]) const { x[2] = x[2] + r; }
    __device__ __forceinline__ void acc(const float (&x)[D], float (&a)[D], float (&sc)[D]) const {
        float d, A, kz, X, Y, Z;
        // stage 1 (A = -k_y)
        d = x[1] - x[0];
        A = fmaf(x[0], x[2], x[1]);
        kz = fmaf(x[0], x[1], fmaf(nb, x[2], nbr));
        a[0] = d; a[1] = A; a[2] = kz;
        X = fmaf(sh2, d, x[0]); Y = fmaf(-h2, A, x[1]); Z = fmaf(h2, kz, x[2]);
        // stage 2
        d = Y - X;
        A = fmaf(X, Z, Y);
        kz = fmaf(X, Y, fmaf(nb, Z, nbr));
        a[0] = fmaf(2.0f, d, a[0]); a[1] = fmaf(2.0f, A, a[1]); a[2] = fmaf(2.0f, kz, a[2]);
        X = fmaf(sh2, d, x[0]); Y = fmaf(-h2, A, x[1]); Z = fmaf(h2, kz, x[2]);
        // stage 3
        d = Y - X;
        A = fmaf(X, Z, Y);
        kz = fmaf(X, Y, fmaf(nb, Z, nbr));
        a[0] = fmaf(2.0f, d, a[0]); a[1] = fmaf(2.0f, A, a[1]); a[2] = fmaf(2.0f, kz, a[2]);
        X = fmaf(sh1, d, x[0]); Y = fmaf(-h1, A, x[1]); Z = fmaf(h1, kz, x[2]);
        // stage 4
        d = Y - X;
        A = fmaf(X, Z, Y);
        kz = fmaf(X, Y, fmaf(nb, Z, nbr));
        a[0] = a[0] + d; a[1] = a[1] + A; a[2] = a[2] + kz;
        sc[0] = sh6; sc[1] = -h6; sc[2] = h6;
    }
};

// RK4 on Wilson-Cowan with a shorter dependent chain between stages.  The
// logistic's base-2 exponents are affine in the state, arg = A x + c, so at a
// stage point P = x + c_s k they are arg(x) + c_s A k, and with k = (S - Q) / tau
// (Q the point k was taken at, S its logistic values)
//   arg(P) = [arg(x) - c_s A (Q / tau)] + c_s A (S / tau).
// The bracket needs only Q and runs beside the exponentials, so from the
// reciprocals to the next exponentials the chain is two FMAs instead of four
// (k, the stage point, and the two FMAs of the exponent).  The stage points and
// k themselves are formed as in the generic stepper for the weighted sum; the
// exponents differ from the ones taken at those points by rounding only.
struct WilsonCowanRK4 {
    static constexpr int D = 2;
    float h1, h2, h6;
    float aE, bE, cE, aI, bI, cI;  // exponent of the E (I) logistic: aE E + bE I + cE (aI E + bI I + cI)
    float iE, iI;                  // 1 / tau
    float uE, vE, uI, vI;          // exponent change per unit of S: aE / tauE, bE / tauI, aI / tauE, bI / tauI
    __device__ __forceinline__ void init(float h, const float* p) {
        const float g2 = p[8] * kLog2e;
        aE = -g2 * p[0];
        bE = g2 * p[1];
        cE = g2 * (p[9] - p[4]);
        aI = -g2 * p[2];
        bI = g2 * p[3];
        cI = g2 * (p[9] - p[5]);
        iE = __fdividef(1.0f, p[6]);
        iI = __fdividef(1.0f, p[7]);
        uE = aE * iE;
        vE = bE * iI;
        uI = aI * iE;
        vI = bI * iI;
        h1 = h;
        h2 = 0.5f * h;
        h6 = h * (1.0f / 6.0f);
    }
    __device__ __forceinline__ void to_internal(float (&)[D]) const {}
    __device__ __forceinline__ void from_internal(float (&)[D]) const {}
    __device__ __forceinline__ void acc(const float (&x)[D], float (&a)[D], float (&sc)[D]) const {
        const float E = x[0], I = x[1];
        // stage 1: the right-hand side at x
        const float argE = fmaf(aE, E, fmaf(bE, I, cE)), argI = fmaf(aI, E, fmaf(bI, I, cI));
        float SE = rcp_ftz(1.0f + ex2_ftz(argE)), SI = rcp_ftz(1.0f + ex2_ftz(argI));
        float QE = E, QI = I;  // the point the current k is taken at
        float kE = fmaf(SE, iE, -QE * iE), kI = fmaf(SI, iI, -QI * iI);
        a[0] = kE;
        a[1] = kI;
#pragma unroll
        for (int st = 2; st <= 4; ++st) {
            const float c = (st == 4) ? h1 : h2;
            // beside the chain: the stage point and the part of its exponents known from Q
            const float PE = fmaf(c, kE, E), PI = fmaf(c, kI, I);
            const float cuE = c * uE, cvE = c * vE, cuI = c * uI, cvI = c * vI;
            const float qE = fmaf(-cuE, QE, fmaf(-cvE, QI, argE)), qI = fmaf(-cuI, QE, fmaf(-cvI, QI, argI));
            // on the chain: two FMAs from the reciprocals to the exponents
            const float eE = fmaf(cvE, SI, fmaf(cuE, SE, qE)), eI = fmaf(cvI, SI, fmaf(cuI, SE, qI));
            SE = rcp_ftz(1.0f + ex2_ftz(eE));
            SI = rcp_ftz(1.0f + ex2_ftz(eI));
            QE = PE;
            QI = PI;
            kE = fmaf(SE, iE, -QE * iE);
            kI = fmaf(SI, iI, -QI * iI);
            if (st < 4) {
                a[0] = fmaf(2.0f, kE, a[0]);
                a[1] = fmaf(2.0f, kI, a[1]);
            } else {
                a[0] = a[0] + kE;
                a[1] = a[1] + kI;
            }
        }
        sc[0] = h6;
        sc[1] = h6;
    }
};

template <class R, int METHOD, bool KAHAN> struct StepperFor { using type = GenericRK4<R>; };
template <bool KAHAN> struct StepperFor<WilsonCowan, FF_RK4, KAHAN> { using type = WilsonCowanRK4; };
template <class R, bool KAHAN> struct StepperFor<R, FF_EULER, KAHAN> { using type = GenericEuler<R>; };
// the compensated variant keeps z unshifted so that no rounding escapes the compensation
template <> struct StepperFor<Lorenz, FF_RK4, true> { using type = LorenzRK4; };
template <> struct StepperFor<Lorenz, FF_RK4, false> { using type = LorenzRK4Shift; };

// ---------------------------------------------------------------------------
// Vector access of PPT consecutive floats.
// ---------------------------------------------------------------------------
template <int PPT> struct Vec;
template <> struct Vec<1> {
    __device__ __forceinline__ static void load(const float* p, float (&v)[1]) { v[0] = __ldcs(p); }
    __device__ __forceinline__ static void store(float* p, const float (&v)[1]) { __stcs(p, v[0]); }
};
template <> struct Vec<2> {
    __device__ __forceinline__ static void load(const float* p, float (&v)[2]) {
        float2 t = __ldcs(reinterpret_cast<const float2*>(p));
        v[0] = t.x; v[1] = t.y;
    }
    __device__ __forceinline__ static void store(float* p, const float (&v)[2]) {
        __stcs(reinterpret_cast<float2*>(p), make_float2(v[0], v[1]));
    }
};
template <> struct Vec<4> {
    __device__ __forceinline__ static void load(const float* p, float (&v)[4]) {
        float4 t = __ldcs(reinterpret_cast<const float4*>(p));
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
    __device__ __forceinline__ static void store(float* p, const float (&v)[4]) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
    }
};

// Reset test and re-draw of one particle (paper Sec. 2.1, Appendix A).  The
// state is tested in external coordinates; a reset particle gets the draws of
// its next reset block, loses its compensation and restarts its age.
template <int D, class Stepper>
__device__ __forceinline__ void reset_check(const IntegrateArgs& a, const Stepper& st, float (&x)[D], float (&c)[D],
                                         uint32_t& age, uint32_t& nres, int g, int64_t i) {
    const ResetTable* t = a.reset;
    float e[D];
#pragma unroll
    for (int k = 0; k < D; ++k) e[k] = x[k];
    st.from_internal(e);
    bool out = a.max_age > 0u && age >= a.max_age;
    if (t->has_bounds)
        for (int k = 0; k < a.dim; ++k) out |= !(e[k] >= t->blo[k] && e[k] <= t->bhi[k]);
    if (!out) return;
    const uint32_t r = nres + 1u;
    const uint64_t j = (uint64_t)(t->first[g] + (i - a.gstart[g]));  // index within the whole group
    const uint64_t base = ((uint64_t)r * (uint64_t)t->count[g] + j) * (uint64_t)a.dim;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        if (k < a.dim) {
            e[k] = draw_value(splitmix64_mix(t->seed[g] + (base + (uint64_t)k + 1u) * kSplitMixGamma), t->box[g][k]);
        } else {
            e[k] = 0.0f;
        }
        c[k] = 0.0f;
        x[k] = e[k];
    }
    st.to_internal(x);
    age = 0u;
    nres = r;
}

// ---------------------------------------------------------------------------
// The persistent integrator.  Grid-stride over work items of PPT consecutive
// particles; each work item loads its state once, runs n_steps steps with the
// state in registers and stores it once.
// ---------------------------------------------------------------------------
// One work item (PPT consecutive particles starting at t * PPT) of the integrator:
// load, n_steps steps with the state in registers, store.  `a` may live in the
// kernel's argument block or, for batched launches, in a device table.
// TAPE: the launch may carry checkpoints (a.ckpt); false compiles them out.
template <class R, int METHOD, bool KAHAN, bool PP, int PPT, bool RESET, bool TAPE = true>
__device__ __forceinline__ void integrate_item(const IntegrateArgs& a, int64_t t, int n_steps_run) {
    constexpr int D = R::DIM;
    using Stepper = typename StepperFor<R, METHOD, KAHAN>::type;
    const int64_t i0 = t * PPT;
    float x[PPT][D];
    float c[PPT][D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        float v[PPT], w[PPT];
        if (k < a.dim) {
            Vec<PPT>::load(a.x + k * a.pitch + i0, v);
            if (KAHAN) Vec<PPT>::load(a.comp + k * a.pitch + i0, w);
        } else {
#pragma unroll
            for (int j = 0; j < PPT; ++j) { v[j] = 0.f; w[j] = 0.f; }
        }
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
            x[j][k] = v[j];
            c[j][k] = KAHAN ? w[j] : 0.f;
        }
        if (float* ck0 = TAPE ? start_checkpoint(a) : nullptr; ck0 && k < a.dim)
            Vec<PPT>::store(ck0 + k * a.pitch + i0, v);
    }
    float prm[PPT][R::NP];
    Stepper st[PPT];
    int grp[PPT];
    uint32_t age[PPT], nres[PPT];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
        const int64_t i = i0 + j;
        float h = a.gh[0];
        grp[j] = 0;
#pragma unroll
        for (int g = 1; g < FF_MAX_GROUPS; ++g)
            if (g < a.n_groups && i >= a.gstart[g]) { h = a.gh[g]; grp[j] = g; }
        if (RESET) {
            age[j] = a.age[i];
            nres[j] = a.resets[i];
        }
        float pv = 0.f;
        if (PP) pv = a.pparam[i];
#pragma unroll
        for (int q = 0; q < R::NP; ++q) prm[j][q] = (PP && q == a.pidx) ? pv : a.p[q];
        st[j].init(h, prm[j]);
        st[j].to_internal(x[j]);
    }
    const int n_steps = n_steps_run;  // the host splits launches at 2^30 steps
    // steps until the next reset check (global step numbers that are multiples of check_every)
    int countdown = RESET ? a.check_every - (int)(a.step0 % a.check_every) : 0;
    auto step = [&]() {
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
            float acc[D], sc[D];
            st[j].acc(x[j], acc, sc);
#pragma unroll
            for (int k = 0; k < D; ++k) {
                if (KAHAN) {
                    const float y = fmaf(sc[k], acc[k], -c[j][k]);
                    const float tt = __fadd_rn(x[j][k], y);
                    c[j][k] = __fsub_rn(__fsub_rn(tt, x[j][k]), y);
                    x[j][k] = tt;
                } else {
                    x[j][k] = fmaf(sc[k], acc[k], x[j][k]);
                }
            }
            if (RESET) age[j] += 1u;
        }
        if (RESET && --countdown == 0) {
            countdown = a.check_every;
#pragma unroll
            for (int j = 0; j < PPT; ++j) reset_check<D>(a, st[j], x[j], c[j], age[j], nres[j], grp[j], i0 + j);
        }
    };
    auto save = [&](int slot) {
        // the end of a launch (back from the stepper's internal form) and the start of the next
#pragma unroll
        for (int j = 0; j < PPT; ++j) st[j].from_internal(x[j]);
        float* ck = a.ckpt + (int64_t)slot * a.ck_stride;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            if (k < a.dim) {
                float v[PPT];
#pragma unroll
                for (int j = 0; j < PPT; ++j) v[j] = x[j][k];
                Vec<PPT>::store(ck + k * a.pitch + i0, v);
            }
        }
#pragma unroll
        for (int j = 0; j < PPT; ++j) st[j].to_internal(x[j]);
    };
    // a step of a large system is long enough on its own; unrolling only grows the code
    run_steps<(D > 8) ? 1 : 4, TAPE>(a, n_steps, step, save);
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
        st[j].from_internal(x[j]);
        if (RESET) {
            a.age[i0 + j] = age[j];
            a.resets[i0 + j] = nres[j];
        }
    }
#pragma unroll
    for (int k = 0; k < D; ++k) {
        if (k < a.dim) {
            float v[PPT], w[PPT];
#pragma unroll
            for (int j = 0; j < PPT; ++j) { v[j] = x[j][k]; w[j] = c[j][k]; }
            Vec<PPT>::store(a.x + k * a.pitch + i0, v);
            if (KAHAN) Vec<PPT>::store(a.comp + k * a.pitch + i0, w);
        }
    }
}

// First item of this thread in a grid-stride loop of nb blocks (stride nb *
// blockDim, items in runs of 32 per warp).  Runs go out warp-major -- warp k of
// every block before warp k + 1 of any -- so the last, partial round of a
// persistent grid spreads over all blocks and SMs instead of falling on the
// first blocks whole.  Needs blockDim a multiple of 32.
__device__ __forceinline__ int64_t warp_major_first(int64_t block_in_range, int64_t nb) {
    return ((int64_t)(threadIdx.x >> 5) * nb + block_in_range) * 32 + (threadIdx.x & 31);
}

// Minimum resident blocks for a system's launch bound: R::MIN_BLOCKS where given, else 1.
template <class R, class = void> struct MinBlocks { static constexpr int value = 1; };
template <class R> struct MinBlocks<R, decltype((void)R::MIN_BLOCKS)> { static constexpr int value = R::MIN_BLOCKS; };

// Particle reset is never taped, so its variants carry no checkpoints.
template <class R, int METHOD, bool KAHAN, bool PP, int PPT, bool RESET = false, bool TAPE = !RESET>
__global__ void __launch_bounds__(R::MAX_BLOCK, MinBlocks<R>::value) integrate_kernel(const __grid_constant__ IntegrateArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = warp_major_first(blockIdx.x, gridDim.x); t < a.n_vec; t += stride)
        integrate_item<R, METHOD, KAHAN, PP, PPT, RESET, TAPE>(a, t, (int)a.n_steps);
}

// ---------------------------------------------------------------------------
// Packed-pair RK4 for Lorenz.  Blackwell executes two FP32 lanes per thread
// with one add/sub/mul/fma.rn.f32x2 instruction, which halves the issue slots
// the 37 FP32 operations of a step need, so the step is bound by the FP32
// pipes rather than by instruction issue.  Each f32x2 register holds the same
// quantity of two consecutive particles.  The arithmetic is the shifted step
// above (zt = z - r); the f32x2 forms have no operand negation, so the
// negated step sizes of the y-component are kept as constants.
// ---------------------------------------------------------------------------
struct f2 {
    unsigned long long v;
};
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 p, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

struct LorenzPairConsts {
    f2 h1, h2, h6, nh1, nh2, nh6, sh1, sh2, sh6, nb, nbr;
};

__device__ __forceinline__ void lorenz_rk4_pair(f2& x, f2& y, f2& z, const LorenzPairConsts& c, f2 two) {
    f2 d, A, kz, X, Y, Z, ad, aA, az;
    // stage 1 (A = -k_y, z is the shifted zt)
    d = sub2(y, x);
    A = fma2(x, z, y);
    kz = fma2(x, y, fma2(c.nb, z, c.nbr));
    ad = d; aA = A; az = kz;
    X = fma2(c.sh2, d, x); Y = fma2(c.nh2, A, y); Z = fma2(c.h2, kz, z);
    // stage 2
    d = sub2(Y, X);
    A = fma2(X, Z, Y);
    kz = fma2(X, Y, fma2(c.nb, Z, c.nbr));
    ad = fma2(two, d, ad); aA = fma2(two, A, aA); az = fma2(two, kz, az);
    X = fma2(c.sh2, d, x); Y = fma2(c.nh2, A, y); Z = fma2(c.h2, kz, z);
    // stage 3
    d = sub2(Y, X);
    A = fma2(X, Z, Y);
    kz = fma2(X, Y, fma2(c.nb, Z, c.nbr));
    ad = fma2(two, d, ad); aA = fma2(two, A, aA); az = fma2(two, kz, az);
    X = fma2(c.sh1, d, x); Y = fma2(c.nh1, A, y); Z = fma2(c.h1, kz, z);
    // stage 4
    d = sub2(Y, X);
    A = fma2(X, Z, Y);
    kz = fma2(X, Y, fma2(c.nb, Z, c.nbr));
    ad = add2(ad, d); aA = add2(aA, A); az = add2(az, kz);
    x = fma2(c.sh6, ad, x); y = fma2(c.nh6, aA, y); z = fma2(c.h6, az, z);
}

template <bool PP, int NPAIR>
__global__ void __launch_bounds__(512) lorenz_rk4_x2_kernel(const __grid_constant__ IntegrateArgs a) {
    constexpr int PPT = 2 * NPAIR;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const f2 two = pack2(2.0f, 2.0f);
    for (int64_t t = warp_major_first(blockIdx.x, gridDim.x); t < a.n_vec; t += stride) {
        const int64_t i0 = t * PPT;
        float xs[PPT], ys[PPT], zs[PPT];
        Vec<PPT>::load(a.x + i0, xs);
        Vec<PPT>::load(a.x + a.pitch + i0, ys);
        Vec<PPT>::load(a.x + 2 * a.pitch + i0, zs);
        if (float* ck0 = start_checkpoint(a)) {
            Vec<PPT>::store(ck0 + i0, xs);
            Vec<PPT>::store(ck0 + a.pitch + i0, ys);
            Vec<PPT>::store(ck0 + 2 * a.pitch + i0, zs);
        }
        float h[PPT], sg[PPT], r[PPT], b[PPT];
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
            const int64_t i = i0 + j;
            h[j] = a.gh[0];
#pragma unroll
            for (int g = 1; g < FF_MAX_GROUPS; ++g)
                if (g < a.n_groups && i >= a.gstart[g]) h[j] = a.gh[g];
            const float pv = PP ? a.pparam[i] : 0.0f;
            sg[j] = (PP && a.pidx == 0) ? pv : a.p[0];
            r[j] = (PP && a.pidx == 1) ? pv : a.p[1];
            b[j] = (PP && a.pidx == 2) ? pv : a.p[2];
        }
        f2 X[NPAIR], Y[NPAIR], Z[NPAIR];
        LorenzPairConsts c[NPAIR];
#pragma unroll
        for (int q = 0; q < NPAIR; ++q) {
            const int u = 2 * q, v = 2 * q + 1;
            X[q] = pack2(xs[u], xs[v]);
            Y[q] = pack2(ys[u], ys[v]);
            Z[q] = pack2(zs[u] - r[u], zs[v] - r[v]);
            const float h2u = 0.5f * h[u], h2v = 0.5f * h[v];
            const float h6u = h[u] * (1.0f / 6.0f), h6v = h[v] * (1.0f / 6.0f);
            c[q].h1 = pack2(h[u], h[v]);
            c[q].h2 = pack2(h2u, h2v);
            c[q].h6 = pack2(h6u, h6v);
            c[q].nh1 = pack2(-h[u], -h[v]);
            c[q].nh2 = pack2(-h2u, -h2v);
            c[q].nh6 = pack2(-h6u, -h6v);
            c[q].sh1 = pack2(sg[u] * h[u], sg[v] * h[v]);
            c[q].sh2 = pack2(sg[u] * h2u, sg[v] * h2v);
            c[q].sh6 = pack2(sg[u] * h6u, sg[v] * h6v);
            c[q].nb = pack2(-b[u], -b[v]);
            c[q].nbr = pack2(-b[u] * r[u], -b[v] * r[v]);
        }
        auto save = [&](int slot) {
            float* ck = a.ckpt + (int64_t)slot * a.ck_stride;
            float cx[PPT], cy[PPT], cz[PPT];
#pragma unroll
            for (int q = 0; q < NPAIR; ++q) {
                const int u = 2 * q, v = 2 * q + 1;
                unpack2(X[q], cx[u], cx[v]);
                unpack2(Y[q], cy[u], cy[v]);
                unpack2(Z[q], cz[u], cz[v]);
                cz[u] = cz[u] + r[u];
                cz[v] = cz[v] + r[v];
                Z[q] = pack2(cz[u] - r[u], cz[v] - r[v]);
            }
            Vec<PPT>::store(ck + i0, cx);
            Vec<PPT>::store(ck + a.pitch + i0, cy);
            Vec<PPT>::store(ck + 2 * a.pitch + i0, cz);
        };
        run_steps<2>(a, (int)a.n_steps, [&]() {
#pragma unroll
            for (int q = 0; q < NPAIR; ++q) lorenz_rk4_pair(X[q], Y[q], Z[q], c[q], two);
        }, save);
#pragma unroll
        for (int q = 0; q < NPAIR; ++q) {
            const int u = 2 * q, v = 2 * q + 1;
            unpack2(X[q], xs[u], xs[v]);
            unpack2(Y[q], ys[u], ys[v]);
            unpack2(Z[q], zs[u], zs[v]);
            zs[u] = zs[u] + r[u];
            zs[v] = zs[v] + r[v];
        }
        Vec<PPT>::store(a.x + i0, xs);
        Vec<PPT>::store(a.x + a.pitch + i0, ys);
        Vec<PPT>::store(a.x + 2 * a.pitch + i0, zs);
    }
}

// Group-uniform variant of the packed kernel.  Blocks are dealt out to the
// groups in proportion to their sizes (gblk), so a block's group -- and with
// it the step sizes and the sigma/beta constants -- is the same for every
// thread of the block; those constants are computed once per block from the
// argument block instead of living in per-thread registers, which leaves room
// for more resident warps.  Used when every group starts on a multiple of the
// particles per thread and a per-particle parameter, if any, is r.
template <bool PP_R, int NPAIR, bool SPLAT = false>
__global__ void __launch_bounds__(512) lorenz_rk4_x2u_kernel(const __grid_constant__ IntegrateArgs a) {
    constexpr int PPT = 2 * NPAIR;
    int g = 0;
#pragma unroll
    for (int q = 1; q < FF_MAX_GROUPS; ++q)
        if (q < a.n_groups && (int)blockIdx.x >= a.gblk[q]) g = q;
    const int64_t nb = a.gblk[g + 1] - a.gblk[g];
    const int64_t first = a.gstart[g] / PPT, last = a.gend[g] / PPT;
    const float h = a.gh[g], sg = a.p[0], b = a.p[2];
    const float h2 = 0.5f * h, h6 = h * (1.0f / 6.0f);
    LorenzPairConsts c;
    c.h1 = pack2(h, h);
    c.h2 = pack2(h2, h2);
    c.h6 = pack2(h6, h6);
    c.nh1 = pack2(-h, -h);
    c.nh2 = pack2(-h2, -h2);
    c.nh6 = pack2(-h6, -h6);
    c.sh1 = pack2(sg * h, sg * h);
    c.sh2 = pack2(sg * h2, sg * h2);
    c.sh6 = pack2(sg * h6, sg * h6);
    c.nb = pack2(-b, -b);
    const float nbr_sys = -b * a.p[1];
    const f2 two = pack2(2.0f, 2.0f);
    const int64_t stride = nb * blockDim.x;
    for (int64_t t = first + warp_major_first(blockIdx.x - a.gblk[g], nb); t < last; t += stride) {
        const int64_t i0 = t * PPT;
        float xs[PPT], ys[PPT], zs[PPT], r[PPT];
        Vec<PPT>::load(a.x + i0, xs);
        Vec<PPT>::load(a.x + a.pitch + i0, ys);
        Vec<PPT>::load(a.x + 2 * a.pitch + i0, zs);
        if (PP_R) Vec<PPT>::load(a.pparam + i0, r);
        if (float* ck0 = SPLAT ? nullptr : start_checkpoint(a)) {  // the fused frame is never taped
            Vec<PPT>::store(ck0 + i0, xs);
            Vec<PPT>::store(ck0 + a.pitch + i0, ys);
            Vec<PPT>::store(ck0 + 2 * a.pitch + i0, zs);
        }
        f2 X[NPAIR], Y[NPAIR], Z[NPAIR], NBR[NPAIR];
#pragma unroll
        for (int q = 0; q < NPAIR; ++q) {
            const int u = 2 * q, v = 2 * q + 1;
            const float ru = PP_R ? r[u] : a.p[1], rv = PP_R ? r[v] : a.p[1];
            X[q] = pack2(xs[u], xs[v]);
            Y[q] = pack2(ys[u], ys[v]);
            Z[q] = pack2(zs[u] - ru, zs[v] - rv);
            NBR[q] = PP_R ? pack2(-b * ru, -b * rv) : pack2(nbr_sys, nbr_sys);
        }
        auto save = [&](int slot) {
            float* ck = a.ckpt + (int64_t)slot * a.ck_stride;
            float cx[PPT], cy[PPT], cz[PPT];
#pragma unroll
            for (int q = 0; q < NPAIR; ++q) {
                const int u = 2 * q, v = 2 * q + 1;
                const float ru = PP_R ? r[u] : a.p[1], rv = PP_R ? r[v] : a.p[1];
                unpack2(X[q], cx[u], cx[v]);
                unpack2(Y[q], cy[u], cy[v]);
                unpack2(Z[q], cz[u], cz[v]);
                cz[u] = cz[u] + ru;
                cz[v] = cz[v] + rv;
                Z[q] = pack2(cz[u] - ru, cz[v] - rv);
            }
            Vec<PPT>::store(ck + i0, cx);
            Vec<PPT>::store(ck + a.pitch + i0, cy);
            Vec<PPT>::store(ck + 2 * a.pitch + i0, cz);
        };
        run_steps<2, !SPLAT>(a, (int)a.n_steps, [&]() {
#pragma unroll
            for (int q = 0; q < NPAIR; ++q) {
                LorenzPairConsts cq = c;
                cq.nbr = NBR[q];
                lorenz_rk4_pair(X[q], Y[q], Z[q], cq, two);
            }
        }, save);
#pragma unroll
        for (int q = 0; q < NPAIR; ++q) {
            const int u = 2 * q, v = 2 * q + 1;
            unpack2(X[q], xs[u], xs[v]);
            unpack2(Y[q], ys[u], ys[v]);
            unpack2(Z[q], zs[u], zs[v]);
            zs[u] = zs[u] + (PP_R ? r[u] : a.p[1]);
            zs[v] = zs[v] + (PP_R ? r[v] : a.p[1]);
        }
        Vec<PPT>::store(a.x + i0, xs);
        Vec<PPT>::store(a.x + a.pitch + i0, ys);
        Vec<PPT>::store(a.x + 2 * a.pitch + i0, zs);
        if (SPLAT && ((a.view.mask >> g) & 1u)) {
            // the render step on the final states held in registers: one count per drawn particle
#pragma unroll
            for (int j = 0; j < PPT; ++j) {
                if (i0 + j >= a.n_real) continue;
                const float rj = PP_R ? r[j] : a.p[1];
                auto coord = [&](int ax) { return ax == 0 ? xs[j] : ax == 1 ? ys[j] : ax == 2 ? zs[j] : rj; };
                const float u = coord(a.view.axes[0]), v = coord(a.view.axes[1]), w = coord(a.view.axes[2]);
                int col, row;
                const bool drawn = a.view.ndim == 2 ? pixel_of<2>(a.view, u, v, w, col, row)
                                                    : pixel_of<3>(a.view, u, v, w, col, row);
                if (drawn) atomicAdd(&a.view.image[(int64_t)row * a.view.W + col], 1u);
            }
        }
    }
}

// Host-side launch of one integrator variant (defined per system in its own
// translation unit so the variants compile in parallel).
struct LaunchShape {
    int ppt;
    int block;
    int blocks_per_sm;  // 0 = occupancy limit
    int num_sms;
};

// The shape with blocks of at most `most` threads.  A limit of blocks per SM keeps its threads: it counts
// blocks of the block size it came with, at most that of the system's one-particle kernel.
inline LaunchShape with_block_of(LaunchShape s, int most, int one_particle = 512) {
    const int block = s.block < one_particle ? s.block : one_particle;
    if (s.blocks_per_sm > 0 && block > most) s.blocks_per_sm = s.blocks_per_sm * block / most;
    if (s.block > most) s.block = most;
    return s;
}

cudaError_t launch_integrate(int rhs_id, int method, bool kahan, bool pp, const IntegrateArgs& a,
                             const LaunchShape& shape, cudaStream_t stream);
cudaError_t launch_integrate_lorenz(int method, bool kahan, bool pp, const IntegrateArgs& a,
                                    const LaunchShape& shape, cudaStream_t stream);
bool lorenz_uniform_packed(int method, bool kahan, bool pp, const IntegrateArgs& a, const LaunchShape& shape);
cudaError_t launch_integrate_lorenz_splat(bool pp, const IntegrateArgs& a, const LaunchShape& shape,
                                          cudaStream_t stream);
// Compensated RK4 for Lorenz as packed pairs (ff_integrate_lorenz_kahan.cu), where the
// shape allows it (2 or 4 particles per thread, aligned groups, no reset, parameter r at most).
bool lorenz_kahan_packed(int method, bool pp, const IntegrateArgs& a, const LaunchShape& shape);
cudaError_t launch_integrate_lorenz_kahan(bool pp, const IntegrateArgs& a, const LaunchShape& shape,
                                          cudaStream_t stream);
cudaError_t launch_integrate_wc(int method, bool kahan, bool pp, const IntegrateArgs& a,
                                const LaunchShape& shape, cudaStream_t stream);
// Wilson-Cowan and Lorenz with particle reset as packed pairs (ff_integrate_reset.cu).
bool reset_pairs(int rhs_id, int method, bool kahan, bool pp, const IntegrateArgs& a);
cudaError_t launch_reset_pairs(int rhs_id, const IntegrateArgs& a, const LaunchShape& shape, cudaStream_t stream);
cudaError_t launch_integrate_hh3(int method, bool kahan, bool pp, const IntegrateArgs& a,
                                 const LaunchShape& shape, cudaStream_t stream);
cudaError_t launch_integrate_linear(int rhs_id, int method, bool kahan, bool pp,
                                    const IntegrateArgs& a, const LaunchShape& shape,
                                    cudaStream_t stream);

// Block size for work too small to give every SM a block: narrowed, in whole
// warps down to one, until the blocks cover the SMs.  A small ensemble then runs
// one or a few warps per SM instead of crowding a few SMs, whose sub-partitions
// would share their MUFU and FP32 pipes between the warps of one step chain.
inline int spread_block(int block, int64_t items, int num_sms) {
    if (num_sms < 1 || items >= (int64_t)block * num_sms) return block;
    const int64_t per_sm = (items + num_sms - 1) / num_sms;
    const int64_t b = (per_sm + 31) / 32 * 32;
    return b < 32 ? 32 : (b < block ? (int)b : block);
}

// The integrator kernel a launch helper last started on this host thread, with
// its grid and block (ff_last_launch reports it; defined in ff_api.cu).
struct LaunchRecord {
    const void* kernel = nullptr;
    int grid = 0, block = 0;
};
LaunchRecord& last_launch_record();

// Grid for a persistent launch: enough blocks to cover the work, at most
// blocks_per_sm (or the occupancy limit) per SM.  The block size is clamped to
// the kernel's compiled maximum (its launch bound).
template <class Kernel, class... First>
inline cudaError_t persistent_launch(Kernel kernel, const IntegrateArgs& a, const LaunchShape& s0,
                                     cudaStream_t stream, First... first) {
    LaunchShape s = s0;
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
    if (e != cudaSuccess) return e;
    if (s.block > attr.maxThreadsPerBlock) s.block = attr.maxThreadsPerBlock / 32 * 32;
    s.block = spread_block(s.block, a.n_vec, s.num_sms);
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, s.block, 0);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const int per_sm = (s.blocks_per_sm > 0 && s.blocks_per_sm < occ) ? s.blocks_per_sm : occ;
    const int64_t need = (a.n_vec + s.block - 1) / s.block;
    const int64_t cap = (int64_t)per_sm * s.num_sms;
    const int grid = (int)(need < cap ? need : cap);
    if (grid < 1) return cudaSuccess;
    kernel<<<grid, s.block, 0, stream>>>(first..., a);
    last_launch_record() = LaunchRecord{(const void*)kernel, grid, s.block};
    return cudaGetLastError();
}

// Dispatch over (method, Kahan, per-particle parameter, particles per thread).
template <class R, int METHOD, bool KAHAN, bool PP>
inline cudaError_t launch_ppt(const IntegrateArgs& a, const LaunchShape& s, cudaStream_t st) {
    if constexpr (R::DIM <= 4) {
        switch (s.ppt) {
        case 1: return persistent_launch(integrate_kernel<R, METHOD, KAHAN, PP, 1>, a, s, st);
        case 2: return persistent_launch(integrate_kernel<R, METHOD, KAHAN, PP, 2>, a, s, st);
        case 4: return persistent_launch(integrate_kernel<R, METHOD, KAHAN, PP, 4>, a, s, st);
        default: return cudaErrorInvalidValue;
        }
    }
    else {
        // large systems run at their register limit: untaped launches take a variant without
        // the checkpoint code
        if (s.ppt != 1) return cudaErrorInvalidValue;
        if (a.ckpt) return persistent_launch(integrate_kernel<R, METHOD, KAHAN, PP, 1, false, true>, a, s, st);
        return persistent_launch(integrate_kernel<R, METHOD, KAHAN, PP, 1, false, false>, a, s, st);
    }
}

// Resetting particles: the scalar kernel, one particle per thread.
template <class R>
inline cudaError_t launch_reset_variants(int method, bool kahan, bool pp, const IntegrateArgs& a0,
                                         const LaunchShape& s0, cudaStream_t st) {
    IntegrateArgs a = a0;
    LaunchShape s = s0;
    a.n_vec = a0.n_vec * s0.ppt;
    s.ppt = 1;
    if (method == FF_RK4) {
        if (kahan) return pp ? persistent_launch(integrate_kernel<R, FF_RK4, true, true, 1, true>, a, s, st)
                             : persistent_launch(integrate_kernel<R, FF_RK4, true, false, 1, true>, a, s, st);
        return pp ? persistent_launch(integrate_kernel<R, FF_RK4, false, true, 1, true>, a, s, st)
                  : persistent_launch(integrate_kernel<R, FF_RK4, false, false, 1, true>, a, s, st);
    }
    if (kahan) return pp ? persistent_launch(integrate_kernel<R, FF_EULER, true, true, 1, true>, a, s, st)
                         : persistent_launch(integrate_kernel<R, FF_EULER, true, false, 1, true>, a, s, st);
    return pp ? persistent_launch(integrate_kernel<R, FF_EULER, false, true, 1, true>, a, s, st)
              : persistent_launch(integrate_kernel<R, FF_EULER, false, false, 1, true>, a, s, st);
}

// Deal the persistent grid's blocks out to the groups in proportion to their
// sizes (at least one block per group) and launch the group-uniform kernel.
template <class Kernel>
inline cudaError_t uniform_launch(Kernel kernel, const IntegrateArgs& a0, const LaunchShape& s0,
                                  cudaStream_t stream) {
    LaunchShape s = s0;
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
    if (e != cudaSuccess) return e;
    if (s.block > attr.maxThreadsPerBlock) s.block = attr.maxThreadsPerBlock / 32 * 32;
    IntegrateArgs a = a0;
    const int ppt = s.ppt;
    int64_t items_all = 0;
    for (int g = 0; g < a.n_groups; ++g) items_all += (a.gend[g] - a.gstart[g] + ppt - 1) / ppt;
    s.block = spread_block(s.block, items_all, s.num_sms);
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, s.block, 0);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const int per_sm = (s.blocks_per_sm > 0 && s.blocks_per_sm < occ) ? s.blocks_per_sm : occ;
    const int64_t total = (int64_t)per_sm * s.num_sms;
    int next = 0;
    for (int g = 0; g < a.n_groups; ++g) {
        const int64_t items = (a.gend[g] - a.gstart[g] + ppt - 1) / ppt;
        int64_t nb = items_all > 0 ? (total * items + items_all / 2) / items_all : 1;
        const int64_t need = (items + s.block - 1) / s.block;
        if (nb > need) nb = need;
        if (nb < 1) nb = 1;
        a.gblk[g] = next;
        next += (int)nb;
    }
    a.gblk[a.n_groups] = next;
    kernel<<<next, s.block, 0, stream>>>(a);
    last_launch_record() = LaunchRecord{(const void*)kernel, next, s.block};
    return cudaGetLastError();
}

template <class R>
inline cudaError_t launch_variants(int method, bool kahan, bool pp, const IntegrateArgs& a,
                                   const LaunchShape& s, cudaStream_t st) {
    if (a.reset) return launch_reset_variants<R>(method, kahan, pp, a, s, st);
    if (method == FF_RK4) {
        if (kahan) return pp ? launch_ppt<R, FF_RK4, true, true>(a, s, st) : launch_ppt<R, FF_RK4, true, false>(a, s, st);
        return pp ? launch_ppt<R, FF_RK4, false, true>(a, s, st) : launch_ppt<R, FF_RK4, false, false>(a, s, st);
    }
    if (kahan) return pp ? launch_ppt<R, FF_EULER, true, true>(a, s, st) : launch_ppt<R, FF_EULER, true, false>(a, s, st);
    return pp ? launch_ppt<R, FF_EULER, false, true>(a, s, st) : launch_ppt<R, FF_EULER, false, false>(a, s, st);
}

// ---------------------------------------------------------------------------
// Packed-pair RK4 for HH3: neurons 0 and 1 of a particle share f32x2 registers
// (lane 0 neuron 0, lane 1 neuron 1) and run the neuron right-hand side above
// with packed add/sub/mul/fma, which halves the issue slots of their FP32
// arithmetic; neuron 2 runs the scalar form.  The transcendental and compare
// steps work lane by lane.  Lane by lane the arithmetic is that of HH3::f, so
// the step equals the generic stepper's bit for bit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

struct HHPair {
    using T = f2;
    struct M {
        bool a, b;
    };
    __device__ __forceinline__ static T k(float c) { return pack2(c, c); }
    __device__ __forceinline__ static T add(T a, T b) { return add2(a, b); }
    __device__ __forceinline__ static T sub(T a, T b) { return sub2(a, b); }
    __device__ __forceinline__ static T mul(T a, T b) { return mul2(a, b); }
    __device__ __forceinline__ static T fma(T a, T b, T c) { return fma2(a, b, c); }
    __device__ __forceinline__ static T ex2(T v) {
        float a, b;
        unpack2(v, a, b);
        return pack2(ex2_ftz(a), ex2_ftz(b));
    }
    __device__ __forceinline__ static T rcp(T v) {
        float a, b;
        unpack2(v, a, b);
        return pack2(rcp_ftz(a), rcp_ftz(b));
    }
    __device__ __forceinline__ static M small(T y) {
        float a, b;
        unpack2(y, a, b);
        return M{fabsf(a) < 0.5f, fabsf(b) < 0.5f};
    }
    __device__ __forceinline__ static T sel(M c, T x, T y) {
        float xa, xb, ya, yb;
        unpack2(x, xa, xb);
        unpack2(y, ya, yb);
        return pack2(c.a ? xa : ya, c.b ? xb : yb);
    }
    // a - t y with one rounding: f32x2 has no negated-operand form in PTX, and the toolchain
    // fuses a product whose only use is this subtraction into one fused operation (the
    // bit-identity tests of the one- and two-particle HH3 kernels depend on it and check it)
    __device__ __forceinline__ static T fms(T t, T y, T a) { return sub2(a, mul2(t, y)); }
};

// The weighted sum k1 + 2 k2 + 2 k3 + k4 after stage st (0..3; unrolled loops), a the sum before it.
template <class O>
__device__ __forceinline__ typename O::T rk4_weigh(int st, typename O::T k, typename O::T a) {
    return st == 0 ? k : (st == 3 ? O::add(a, k) : O::fma(O::k(2.0f), k, a));
}

struct HH3RK4Packed {
    static constexpr int D = 15;
    float h1, h2, h6;
    const float* p;
    __device__ __forceinline__ void init(float h, const float* prm) {
        h1 = h;
        h2 = 0.5f * h;
        h6 = h * (1.0f / 6.0f);
        p = prm;
    }
    __device__ __forceinline__ void to_internal(float (&)[D]) const {}
    __device__ __forceinline__ void from_internal(float (&)[D]) const {}
    __device__ __forceinline__ void acc(const float (&x)[D], float (&a)[D], float (&sc)[D]) const {
        const HHConst<HHPair> c2 = hh_const<HHPair>(p);
        const HHConst<HHScalar> c1 = hh_const<HHScalar>(p);
        const f2 drive01 = pack2(hh_drive_c(p, 0), hh_drive_c(p, 1));
        const float drive2 = hh_drive_c(p, 2);
        f2 X[5], XS[5], A[5], K[5];
        float x2[5], xs2[5], a2[5], k2[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            X[k] = pack2(x[k], x[5 + k]);
            XS[k] = X[k];
            x2[k] = x[10 + k];
            xs2[k] = x2[k];
        }
        // the stages unrolled: 4% faster than a stage loop (65,536 particles of hh3_1M)
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            float s0, s1;
            unpack2(XS[4], s0, s1);
            const float s_sum = __fadd_rn(__fadd_rn(s0, s1), xs2[4]);
            hh_neuron<HHPair>(XS[0], XS[1], XS[2], XS[3], XS[4], sub2(pack2(s_sum, s_sum), XS[4]), drive01, c2, K);
            hh_neuron<HHScalar>(xs2[0], xs2[1], xs2[2], xs2[3], xs2[4], __fsub_rn(s_sum, xs2[4]), drive2, c1, k2);
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                A[k] = rk4_weigh<HHPair>(st, K[k], A[k]);
                a2[k] = rk4_weigh<HHScalar>(st, k2[k], a2[k]);
            }
            if (st == 3) break;
            const float cst = (st == 2) ? h1 : h2;
            const f2 C = pack2(cst, cst);
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                XS[k] = fma2(C, K[k], X[k]);
                xs2[k] = fmaf(cst, k2[k], x2[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            unpack2(A[k], a[k], a[5 + k]);
            a[10 + k] = a2[k];
        }
#pragma unroll
        for (int i = 0; i < D; ++i) sc[i] = h6;
    }
};
template <bool KAHAN> struct StepperFor<HH3, FF_RK4, KAHAN> { using type = HH3RK4Packed; };

// ---------------------------------------------------------------------------
// RK4 for HH3 with two particles per work item, packed across particles: every
// f32x2 register holds one state variable of particles 2t (lane 0) and 2t + 1
// (lane 1), and all three neurons run the neuron right-hand side over f32x2.  The
// one-particle stepper (HH3RK4Packed) packs neurons 0 and 1 and runs neuron 2 on
// floats; here no neuron runs on floats, so a particle-step issues about three
// quarters of the instructions.  Lane by lane the operations are those of HH3::f
// and of the RK4 stepper, in the same order, so every state is the one-particle
// kernel's to the bit (the adjoint's recomputation still reproduces the taped
// states).  `a` may live in the argument block or, batched, in a device table.
// ---------------------------------------------------------------------------
// The neuron constants of two particles' parameter vectors, per lane (the
// fields of hh_const<HHScalar>, each formed as it forms them).
__device__ __forceinline__ HHConst<HHPair> hh_const_pair(const float* pa, const float* pb) {
    const HHConst<HHScalar> a = hh_const<HHScalar>(pa), b = hh_const<HHScalar>(pb);
    HHConst<HHPair> c;
    c.gNaC = pack2(a.gNaC, b.gNaC);
    c.gKC = pack2(a.gKC, b.gKC);
    c.gLC = pack2(a.gLC, b.gLC);
    c.ENa = pack2(a.ENa, b.ENa);
    c.EK = pack2(a.EK, b.EK);
    c.EL = pack2(a.EL, b.EL);
    c.gsynC = pack2(a.gsynC, b.gsynC);
    c.Esyn = pack2(a.Esyn, b.Esyn);
    c.inv_tr = pack2(a.inv_tr, b.inv_tr);
    c.neg_inv_td = pack2(a.neg_inv_td, b.neg_inv_td);
    c.neg_sig2 = pack2(a.neg_sig2, b.neg_sig2);
    c.sig2_theta = pack2(a.sig2_theta, b.sig2_theta);
    return c;
}

// Steps and parameter vectors of particles i0 and, with PER 2, i0 + 1 (PER 1: i0 twice).
template <bool PP, int PER = 2>
__device__ __forceinline__ void hh_pair_params(const IntegrateArgs& a, int64_t i0, float (&hs)[2],
                                               float (&pa)[HH3::NP], float (&pb)[HH3::NP]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int64_t i = i0 + j * (PER - 1);
        hs[j] = a.gh[0];
#pragma unroll
        for (int g = 1; g < FF_MAX_GROUPS; ++g)
            if (g < a.n_groups && i >= a.gstart[g]) hs[j] = a.gh[g];
    }
    const float pva = PP ? a.pparam[i0] : 0.0f, pvb = PP ? a.pparam[i0 + PER - 1] : 0.0f;
#pragma unroll
    for (int q = 0; q < HH3::NP; ++q) {
        pa[q] = (PP && q == a.pidx) ? pva : a.p[q];
        pb[q] = (PP && q == a.pidx) ? pvb : a.p[q];
    }
}

template <bool PP, bool TAPE>
__device__ __forceinline__ void hh3_rk4_x2_item(const IntegrateArgs& a, int64_t t, int n_steps) {
    constexpr int D = HH3::DIM;
    const int64_t i0 = 2 * t;
    f2 X[D];
    float* ck0 = TAPE ? start_checkpoint(a) : nullptr;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        float v[2];
        Vec<2>::load(a.x + k * a.pitch + i0, v);
        if (ck0) Vec<2>::store(ck0 + k * a.pitch + i0, v);
        X[k] = pack2(v[0], v[1]);
    }
    float hs[2], pa[HH3::NP], pb[HH3::NP];
    hh_pair_params<PP>(a, i0, hs, pa, pb);
    const HHConst<HHPair> c = hh_const_pair(pa, pb);
    f2 drive[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) drive[n] = pack2(hh_drive_c(pa, n), hh_drive_c(pb, n));
    // the stepper's constants, per lane: h, h/2, h/6
    const f2 H1 = pack2(hs[0], hs[1]);
    const f2 H2 = pack2(0.5f * hs[0], 0.5f * hs[1]);
    const f2 H6 = pack2(hs[0] * (1.0f / 6.0f), hs[1] * (1.0f / 6.0f));
    auto step = [&]() {
        f2 XS[D], A[D];
#pragma unroll
        for (int k = 0; k < D; ++k) XS[k] = X[k];
        // the stages unrolled: 4% faster than a stage loop on hh3_1M (168 registers)
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            const f2 s_sum = add2(add2(XS[4], XS[9]), XS[14]);
            f2 K[D];
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                f2 d[5];
                hh_neuron<HHPair>(XS[5 * n], XS[5 * n + 1], XS[5 * n + 2], XS[5 * n + 3], XS[5 * n + 4],
                                  sub2(s_sum, XS[5 * n + 4]), drive[n], c, d);
#pragma unroll
                for (int k = 0; k < 5; ++k) K[5 * n + k] = d[k];
            }
#pragma unroll
            for (int k = 0; k < D; ++k) A[k] = rk4_weigh<HHPair>(st, K[k], A[k]);
            if (st == 3) break;
            const f2 C = (st == 2) ? H1 : H2;
#pragma unroll
            for (int k = 0; k < D; ++k) XS[k] = fma2(C, K[k], X[k]);
        }
#pragma unroll
        for (int k = 0; k < D; ++k) X[k] = fma2(H6, A[k], X[k]);
    };
    auto save = [&](int slot) {
        float* ck = a.ckpt + (int64_t)slot * a.ck_stride;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            float v[2];
            unpack2(X[k], v[0], v[1]);
            Vec<2>::store(ck + k * a.pitch + i0, v);
        }
    };
    run_steps<1, TAPE>(a, n_steps, step, save);
#pragma unroll
    for (int k = 0; k < D; ++k) {
        float v[2];
        unpack2(X[k], v[0], v[1]);
        Vec<2>::store(a.x + k * a.pitch + i0, v);
    }
}

}  // namespace ff
