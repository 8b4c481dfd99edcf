// ff_integrate_reset.cu -- RK4 with particle reset (paper Sec. 2.1, Appendix A) as packed
// f32x2 pairs with group-uniform constants, for Wilson-Cowan and Lorenz.
//
// The step's operations are those of the one-particle steppers (WilsonCowanRK4,
// LorenzRK4Shift) lane by lane, and so are the reset test and the draws: states, ages and
// reset counts are the one-particle kernel's to the bit.  What bounded that kernel, beside
// issuing every FP32 operation for one particle, were the bounds, read again from the
// device table at each check, and the re-draws: in an ensemble that runs backward out of its
// bounds some lane of a warp resets at most steps, and the warp takes the whole re-draw each
// time.  Here the bounds stay in registers, the counter of a particle's next re-draw is
// carried (one 64-bit addition instead of three multiplications per reset), and a lane
// whose two particles both reset takes them in turn, so that a warp pays for one re-draw
// where 64 particles rarely need a second.  1,000,000 Wilson-Cowan particles, half of them
// backward, 200 steps with the unit-square reset at each: 1,064 us -> 735 us.
#include "ff_wc_pair.cuh"

namespace ff {

namespace {

// Packed steppers: D state variables, constants of one group, one step of a pair.  Variable
// SHIFTED loses shift() on the way into the stepper's form (Lorenz keeps z - r).
struct LorenzPair {
    static constexpr int D = 3, SHIFTED = 2;
    LorenzPairConsts c;
    float r;
    __device__ __forceinline__ void init(float h, const float* p) {
        LorenzRK4Shift s;
        s.init(h, p);
        r = s.r;
        c.h1 = pack2(s.h1, s.h1); c.h2 = pack2(s.h2, s.h2); c.h6 = pack2(s.h6, s.h6);
        c.nh1 = pack2(-s.h1, -s.h1); c.nh2 = pack2(-s.h2, -s.h2); c.nh6 = pack2(-s.h6, -s.h6);
        c.sh1 = pack2(s.sh1, s.sh1); c.sh2 = pack2(s.sh2, s.sh2); c.sh6 = pack2(s.sh6, s.sh6);
        c.nb = pack2(s.nb, s.nb);
        c.nbr = pack2(s.nbr, s.nbr);
    }
    __device__ __forceinline__ float shift() const { return r; }
    __device__ __forceinline__ void step(f2 (&x)[D]) const { lorenz_rk4_pair(x[0], x[1], x[2], c, HHPair::k(2.0f)); }
};

template <class S>
__global__ void __launch_bounds__(256) reset_pair_kernel(const __grid_constant__ IntegrateArgs a) {
    constexpr int D = S::D;
    int g = 0;
#pragma unroll
    for (int q = 1; q < FF_MAX_GROUPS; ++q)
        if (q < a.n_groups && (int)blockIdx.x >= a.gblk[q]) g = q;
    const int64_t nb = a.gblk[g + 1] - a.gblk[g];
    const int64_t first = a.gstart[g] / 2, last = a.gend[g] / 2;
    S st;
    st.init(a.gh[g], a.p);
    const ResetTable* t = a.reset;
    const bool has_bounds = t->has_bounds != 0;
    float blo[D], bhi[D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        blo[k] = t->blo[k];
        bhi[k] = t->bhi[k];
    }
    // draw n of the group's stream is the finaliser of seed + n gamma; particle j's r-th reset
    // takes n = (r count + j) dim + 1, ..., so its next one starts count dim gamma further on
    const uint64_t block_of_draws = (uint64_t)t->count[g] * (uint64_t)D * kSplitMixGamma;
    auto item = [&](int64_t it) {
        const int64_t i0 = 2 * it;
        f2 X[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            float v[2];
            Vec<2>::load(a.x + k * a.pitch + i0, v);
            X[k] = pack2(v[0], v[1]);
            if (k == S::SHIFTED) X[k] = pack2(v[0] - st.shift(), v[1] - st.shift());
        }
        uint2 age2 = *reinterpret_cast<const uint2*>(a.age + i0), res2 = *reinterpret_cast<const uint2*>(a.resets + i0);
        uint32_t age[2] = {age2.x, age2.y}, nres[2] = {res2.x, res2.y};
        uint64_t next[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint64_t jg = (uint64_t)(t->first[g] + (i0 + j - a.gstart[g]));
            next[j] = t->seed[g] + (((uint64_t)nres[j] + 1u) * (uint64_t)t->count[g] + jg) * (uint64_t)D * kSplitMixGamma +
                      kSplitMixGamma;
        }
        int countdown = a.check_every - (int)(a.step0 % a.check_every);  // steps until the next check
        for (int s = 0; s < (int)a.n_steps; ++s) {
            st.step(X);
            age[0] += 1u;
            age[1] += 1u;
            if (--countdown != 0) continue;
            countdown = a.check_every;
            float e[2][D];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                unpack2(X[k], e[0][k], e[1][k]);
                if (k == S::SHIFTED) { e[0][k] = e[0][k] + st.shift(); e[1][k] = e[1][k] + st.shift(); }
            }
            bool out[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                out[j] = a.max_age > 0u && age[j] >= a.max_age;
                if (has_bounds) {
#pragma unroll
                    for (int k = 0; k < D; ++k) out[j] |= !(e[j][k] >= blo[k] && e[j][k] <= bhi[k]);
                }
            }
            while (out[0] || out[1]) {
                const int j = out[0] ? 0 : 1;
                uint64_t z = j == 0 ? next[0] : next[1];
#pragma unroll
                for (int k = 0; k < D; ++k, z += kSplitMixGamma) {
                    float v = draw_value(splitmix64_mix(z), t->box[g][k]);
                    if (k == S::SHIFTED) v = v - st.shift();
                    float u0, u1;
                    unpack2(X[k], u0, u1);
                    X[k] = pack2(j == 0 ? v : u0, j == 0 ? u1 : v);
                }
                if (j == 0) {
                    next[0] += block_of_draws;
                    age[0] = 0u;
                    nres[0] += 1u;
                    out[0] = false;
                } else {
                    next[1] += block_of_draws;
                    age[1] = 0u;
                    nres[1] += 1u;
                    out[1] = false;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < D; ++k) {
            float v[2];
            unpack2(X[k], v[0], v[1]);
            if (k == S::SHIFTED) { v[0] = v[0] + st.shift(); v[1] = v[1] + st.shift(); }
            Vec<2>::store(a.x + k * a.pitch + i0, v);
        }
        *reinterpret_cast<uint2*>(a.age + i0) = make_uint2(age[0], age[1]);
        *reinterpret_cast<uint2*>(a.resets + i0) = make_uint2(nres[0], nres[1]);
    };
    // Wilson-Cowan's items, whose re-draws make them uneven, are handed out (780 -> 760 us); Lorenz's
    // step constants leave the uniform registers in that loop (330 -> 362 us), so it keeps equal shares
    const unsigned block = blockIdx.x - a.gblk[g];
    if constexpr (S::SHIFTED < 0) {
        warp_tasks(a.queue + g, (last - first + 31) / 32, block, (unsigned)nb, [&](int64_t task) {
            const int64_t it = first + task * 32 + (threadIdx.x & 31);
            if (it < last) item(it);
        });
    } else {
        const int64_t stride = nb * blockDim.x;
        for (int64_t it = first + warp_major_first(block, nb); it < last; it += stride) item(it);
    }
}

}  // namespace

// Whether the packed reset kernel runs: plain RK4 on a system it has, no per-particle
// parameter, every group starting on an even particle (a pair has one group).
bool reset_pairs(int rhs_id, int method, bool kahan, bool pp, const IntegrateArgs& a) {
    if (!a.reset || method != FF_RK4 || kahan || pp) return false;
    if (rhs_id != FF_RHS_WILSON_COWAN && rhs_id != FF_RHS_LORENZ) return false;
    for (int g = 0; g < a.n_groups; ++g)
        if (a.gstart[g] % 2 != 0) return false;
    return true;
}

cudaError_t launch_reset_pairs(int rhs_id, const IntegrateArgs& a, const LaunchShape& shape, cudaStream_t stream) {
    LaunchShape s = with_block_of(shape, 256);
    s.ppt = 2;
    if (rhs_id == FF_RHS_WILSON_COWAN) return uniform_launch(reset_pair_kernel<WilsonCowanPair>, a, s, stream);
    return uniform_launch(reset_pair_kernel<LorenzPair>, a, s, stream);
}

}  // namespace ff
