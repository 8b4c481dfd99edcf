// ff_wc_pair.cuh -- Wilson-Cowan RK4 on a packed pair of particles with the constants of one group.
#pragma once

#include "ff_device.cuh"

namespace ff {

// Lane by lane the operations of WilsonCowanRK4::acc and the plain update, so the one-particle
// stepper's bits.  The constants that enter negated are kept negated too (f32x2 operands have no sign).
struct WilsonCowanPair {
    static constexpr int D = 2, SHIFTED = -1;
    f2 aE, bE, cE, aI, bI, cI, iE, iI, niE, niI;
    f2 c[2], u[2][4], n[2][4];  // per stage constant (h/2, h): itself; +- (uE, vE, uI, vI) times it
    f2 h6;
    __device__ __forceinline__ void init(float h, const float* p) {
        WilsonCowanRK4 s;
        s.init(h, p);
        aE = pack2(s.aE, s.aE); bE = pack2(s.bE, s.bE); cE = pack2(s.cE, s.cE);
        aI = pack2(s.aI, s.aI); bI = pack2(s.bI, s.bI); cI = pack2(s.cI, s.cI);
        iE = pack2(s.iE, s.iE); iI = pack2(s.iI, s.iI);
        niE = pack2(-s.iE, -s.iE); niI = pack2(-s.iI, -s.iI);
        h6 = pack2(s.h6, s.h6);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float cs = q ? s.h1 : s.h2;
            c[q] = pack2(cs, cs);
            const float w[4] = {__fmul_rn(cs, s.uE), __fmul_rn(cs, s.vE), __fmul_rn(cs, s.uI), __fmul_rn(cs, s.vI)};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                u[q][k] = pack2(w[k], w[k]);
                n[q][k] = pack2(-w[k], -w[k]);
            }
        }
    }
    __device__ __forceinline__ float shift() const { return 0.0f; }
    __device__ __forceinline__ static f2 logistic(f2 arg) {  // 1 / (1 + 2^arg)
        const f2 p = add2(HHPair::k(1.0f), HHPair::ex2(arg));
        return HHPair::rcp(p);
    }
    // WilsonCowanRK4::acc and the plain update, lane by lane
    __device__ __forceinline__ void step(f2 (&x)[D]) const {
        const f2 E = x[0], I = x[1], two = HHPair::k(2.0f);
        const f2 argE = fma2(aE, E, fma2(bE, I, cE)), argI = fma2(aI, E, fma2(bI, I, cI));
        f2 SE = logistic(argE), SI = logistic(argI), QE = E, QI = I;
        f2 kE = fma2(SE, iE, mul2(QE, niE)), kI = fma2(SI, iI, mul2(QI, niI));
        f2 AE = kE, AI = kI;
#pragma unroll
        for (int st = 2; st <= 4; ++st) {
            const int q = st == 4 ? 1 : 0;
            const f2 PE = fma2(c[q], kE, E), PI = fma2(c[q], kI, I);
            const f2 qE = fma2(n[q][0], QE, fma2(n[q][1], QI, argE)), qI = fma2(n[q][2], QE, fma2(n[q][3], QI, argI));
            const f2 eE = fma2(u[q][1], SI, fma2(u[q][0], SE, qE)), eI = fma2(u[q][3], SI, fma2(u[q][2], SE, qI));
            SE = logistic(eE);
            SI = logistic(eI);
            QE = PE;
            QI = PI;
            kE = fma2(SE, iE, mul2(QE, niE));
            kI = fma2(SI, iI, mul2(QI, niI));
            AE = st < 4 ? fma2(two, kE, AE) : add2(AE, kE);
            AI = st < 4 ? fma2(two, kI, AI) : add2(AI, kI);
        }
        x[0] = fma2(h6, AE, E);
        x[1] = fma2(h6, AI, I);
    }
};

}  // namespace ff
