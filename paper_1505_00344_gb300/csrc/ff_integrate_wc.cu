// Integrator variants for the Wilson-Cowan E-I model (paper Eq. 1-2).
#include "ff_device.cuh"

namespace ff {

namespace {

// RK4 as packed f32x2 pairs with group-uniform constants, for ensembles that fill the GPU.
// There the exponential-and-reciprocal unit bounds the step (an exponential takes 1/32, a
// reciprocal 1/16 of a clock and SM per lane), and beside it instruction issue: the
// one-particle stepper issues 66 FP32 operations and 16 of that unit's per step, 0.95 clocks
// per SM and particle-step where the unit alone needs 0.75.  Here the two logistics of a stage
// share one reciprocal, 1/a = b / (a b), which takes the unit to 0.5 clocks; the FP32
// operations go out two lanes an instruction; and 1/tau is folded into the step constants
// (K = tau k = S - x), which leaves 50 of them.  The exponents are clamped at 60 so that the
// product of two denominators stays finite: a logistic below 2^-60 then reads 2^-60, far
// below an ulp of the S - x it enters.  The dependent chain of a stage is longer than the
// one-particle stepper's, so ensembles too small to hide it keep that one.  2,097,152
// particles x 200 steps: 1,267 us one particle per thread, 1,144 us in pairs with two
// reciprocals a stage, 904 us with one, 860 us with the step loop unrolled twice; four logistics on
// one reciprocal (920 us) and four particles per thread (925 us) gave nothing.  With the pairs
// handed out to warps instead of in equal shares it is 816 us.  The exponential
// unit is then about three quarters busy, the FP32 pipe 58%.
struct WCWideConsts {
    f2 aE, bE, cE, aI, bI, cI;      // base-2 exponents of the logistics: aE E + bE I + cE, aI E + bI I + cI
    f2 h2E, h2I, h1E, h1I, h6E, h6I;  // h/2, h and h/6 over tau
};

__device__ __forceinline__ f2 ex2_clamped(f2 arg) {
    float u, v;
    unpack2(arg, u, v);
    asm("min.NaN.f32 %0, %0, 0f42700000;" : "+f"(u));  // 60; a NaN stays one
    asm("min.NaN.f32 %0, %0, 0f42700000;" : "+f"(v));
    return pack2(ex2_ftz(u), ex2_ftz(v));
}

// K = S - (E, I) at the stage point (E, I).
__device__ __forceinline__ void wc_wide_k(f2 E, f2 I, const WCWideConsts& c, f2& KE, f2& KI) {
    const f2 one = HHPair::k(1.0f);
    const f2 pE = add2(one, ex2_clamped(fma2(c.aE, E, fma2(c.bE, I, c.cE))));
    const f2 pI = add2(one, ex2_clamped(fma2(c.aI, E, fma2(c.bI, I, c.cI))));
    const f2 r = HHPair::rcp(mul2(pE, pI));
    KE = sub2(mul2(pI, r), E);
    KI = sub2(mul2(pE, r), I);
}

// Blocks are dealt out to the groups (uniform_launch, pairs of particles).  WIDE groups run the
// packed pairs; a small group beside them runs the one-particle stepper, a pair one
// particle after the other.  Groups may start and end inside an aligned pair.
__global__ void __launch_bounds__(256) wc_rk4_x2u_kernel(const __grid_constant__ IntegrateArgs a, uint32_t wide) {
    int g = 0;
#pragma unroll
    for (int q = 1; q < FF_MAX_GROUPS; ++q)
        if (q < a.n_groups && (int)blockIdx.x >= a.gblk[q]) g = q;
    const int64_t nb = a.gblk[g + 1] - a.gblk[g];
    const int64_t start = a.gstart[g], end = a.gend[g], pairs = (end - start + 1) / 2;
    WilsonCowanRK4 s;
    s.init(a.gh[g], a.p);
    if (!((wide >> g) & 1u)) {
        const int64_t stride = nb * blockDim.x;
        for (int64_t t = warp_major_first(blockIdx.x - a.gblk[g], nb); t < pairs; t += stride)
            for (int64_t i = start + 2 * t; i < start + 2 * t + 2 && i < end; ++i) {
                float x[2] = {a.x[i], a.x[a.pitch + i]};
                run_steps<2, false>(a, (int)a.n_steps, [&]() {
                    float acc[2], sc[2];
                    s.acc(x, acc, sc);
                    x[0] = fmaf(sc[0], acc[0], x[0]);
                    x[1] = fmaf(sc[1], acc[1], x[1]);
                }, [](int) {});
                a.x[i] = x[0];
                a.x[a.pitch + i] = x[1];
            }
        return;
    }
    WCWideConsts c;
    c.aE = HHPair::k(s.aE); c.bE = HHPair::k(s.bE); c.cE = HHPair::k(s.cE);
    c.aI = HHPair::k(s.aI); c.bI = HHPair::k(s.bI); c.cI = HHPair::k(s.cI);
    c.h1E = HHPair::k(s.h1 * s.iE); c.h1I = HHPair::k(s.h1 * s.iI);
    c.h2E = HHPair::k(s.h2 * s.iE); c.h2I = HHPair::k(s.h2 * s.iI);
    c.h6E = HHPair::k(s.h6 * s.iE); c.h6I = HHPair::k(s.h6 * s.iI);
    const f2 two = HHPair::k(2.0f);
    warp_tasks(a.queue + g, (pairs + 31) / 32, blockIdx.x - a.gblk[g], (unsigned)nb, [&](int64_t task) {
        const int64_t t = task * 32 + (threadIdx.x & 31);
        if (t >= pairs) return;
        const int64_t i0 = start + 2 * t;
        const bool vec = (start & 1) == 0 && i0 + 1 < end, has1 = i0 + 1 < end;
        float xs[2], ys[2];
        if (vec) {
            Vec<2>::load(a.x + i0, xs);
            Vec<2>::load(a.x + a.pitch + i0, ys);
        } else {
            xs[0] = a.x[i0];
            ys[0] = a.x[a.pitch + i0];
            xs[1] = has1 ? a.x[i0 + 1] : 0.0f;
            ys[1] = has1 ? a.x[a.pitch + i0 + 1] : 0.0f;
        }
        f2 E = pack2(xs[0], xs[1]), I = pack2(ys[0], ys[1]);
        run_steps<2, false>(a, (int)a.n_steps, [&]() {
            f2 KE, KI, AE, AI;
            wc_wide_k(E, I, c, KE, KI);
            AE = KE; AI = KI;
            wc_wide_k(fma2(c.h2E, KE, E), fma2(c.h2I, KI, I), c, KE, KI);
            AE = fma2(two, KE, AE); AI = fma2(two, KI, AI);
            wc_wide_k(fma2(c.h2E, KE, E), fma2(c.h2I, KI, I), c, KE, KI);
            AE = fma2(two, KE, AE); AI = fma2(two, KI, AI);
            wc_wide_k(fma2(c.h1E, KE, E), fma2(c.h1I, KI, I), c, KE, KI);
            AE = add2(AE, KE); AI = add2(AI, KI);
            E = fma2(c.h6E, AE, E);
            I = fma2(c.h6I, AI, I);
        }, [](int) {});
        unpack2(E, xs[0], xs[1]);
        unpack2(I, ys[0], ys[1]);
        if (vec) {
            Vec<2>::store(a.x + i0, xs);
            Vec<2>::store(a.x + a.pitch + i0, ys);
        } else {
            a.x[i0] = xs[0];
            a.x[a.pitch + i0] = ys[0];
            if (has1) {
                a.x[i0 + 1] = xs[1];
                a.x[a.pitch + i0 + 1] = ys[1];
            }
        }
    });
}

}  // namespace

cudaError_t launch_integrate_wc(int method, bool kahan, bool pp, const IntegrateArgs& a,
                                const LaunchShape& shape, cudaStream_t stream) {
    if (method == FF_RK4 && !kahan && shape.ppt == 2) {
        // The pairs round differently (within the parity bar), so a particle's kernel must not hang on
        // what happens to be launched with it: it goes by the size of its whole group, of which
        // this system may hold a slice, and taped steps, whose adjoint recomputes them, stay
        // with the one-particle stepper.  100 steps on 152 SMs, one particle per thread / in
        // pairs: 65,536 particles 32 / 32 us, 98,304 43.5 / 43, 131,072 54 / 43, 262,144 93 / 73;
        // below, the pairs' longer chain loses (20 / 25).
        if (!pp && !a.reset && !shape.taped && shape.wide)
            return uniform_launch(wc_rk4_x2u_kernel, a, shape, stream, shape.wide);
        IntegrateArgs a1 = a;
        LaunchShape s1 = shape;
        a1.n_vec = a.n_vec * 2;
        s1.ppt = 1;
        return launch_variants<WilsonCowan>(method, kahan, pp, a1, s1, stream);
    }
    return launch_variants<WilsonCowan>(method, kahan, pp, a, shape, stream);
}
}  // namespace ff
