// Integrator variants for the Wilson-Cowan E-I model (paper Eq. 1-2).
#include "ff_wc_pair.cuh"

namespace ff {

namespace {

// RK4 as packed f32x2 pairs with group-uniform constants, for ensembles that fill the GPU: the
// one-particle stepper's bits (WilsonCowanPair).  There the exponential-and-reciprocal unit bounds the
// step (an exponential takes 1/32, a reciprocal 1/16 of a clock and SM per lane: 0.75 clocks for the 8
// of either), and beside it instruction issue, which the pairs halve: 2,097,152 particles x 100 steps
// 636 us one particle per thread, 552 us in pairs, 91% of that unit's 503 us.  (One reciprocal for the two
// logistics of a stage takes 410 us, but rounds each of them twice more; brought back to the separate
// reciprocals' precision by a Newton step each, over the whole range, 606 us.)  Blocks are dealt out to the groups
// (uniform_launch) and their warps take tasks of 32 pairs from the group's queue.  Groups may start
// and end inside an aligned pair.
__global__ void __launch_bounds__(256) wc_rk4_x2u_kernel(const __grid_constant__ IntegrateArgs a) {
    int g = 0;
#pragma unroll
    for (int q = 1; q < FF_MAX_GROUPS; ++q)
        if (q < a.n_groups && (int)blockIdx.x >= a.gblk[q]) g = q;
    const int64_t nb = a.gblk[g + 1] - a.gblk[g];
    const int64_t start = a.gstart[g], end = a.gend[g], pairs = (end - start + 1) / 2;
    WilsonCowanPair s;
    s.init(a.gh[g], a.p);
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
        f2 X[2] = {pack2(xs[0], xs[1]), pack2(ys[0], ys[1])};
        run_steps<2, false>(a, (int)a.n_steps, [&]() { s.step(X); }, [](int) {});
        unpack2(X[0], xs[0], xs[1]);
        unpack2(X[1], ys[0], ys[1]);
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
        // Pairs where some group has 650 particles per SM or more; the bits are the same either way.
        // Resets, a parameter per particle and launches that write checkpoints have kernels of their
        // own.  Small blocks spread a few rounds of warps evenly over the SMs, large ones suit many
        // rounds.  100 steps on 152 SMs, one particle per thread / pairs in blocks of 128 / of 256:
        // 98,800 particles 40.9 / 38.7 / 47.3 us, 131,072 51.3 / 49.2 / 47.6, 200,000 68.9 / 68.9 / 67.4,
        // 262,144 91.9 / 78.6 / 87.4, 524,288 168 / 147 / 147, 1,048,576 325 / 285 / 276, 2,097,152 636 / 552 / 552.
        bool wide = false;
        for (int g = 0; g < a.n_groups; ++g) {
            const int64_t end = a.gend[g] < a.n_real ? a.gend[g] : a.n_real;
            wide = wide || end - a.gstart[g] >= 650 * (int64_t)shape.num_sms;
        }
        if (wide && !pp && !a.reset && !a.ckpt)
            return uniform_launch(wc_rk4_x2u_kernel, a,
                                  with_block_of(shape, a.n_real < 2500 * (int64_t)shape.num_sms ? 128 : 256), stream);
        IntegrateArgs a1 = a;
        LaunchShape s1 = shape;
        a1.n_vec = a.n_vec * 2;
        s1.ppt = 1;
        return launch_variants<WilsonCowan>(method, kahan, pp, a1, s1, stream);
    }
    return launch_variants<WilsonCowan>(method, kahan, pp, a, shape, stream);
}
}  // namespace ff
