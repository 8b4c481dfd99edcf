// Integrator variants for three coupled Hodgkin-Huxley neurons (paper Eq. 6-11).
#include "ff_device.cuh"

namespace ff {

namespace {

// Two particles per thread, all three neurons packed across the pair (hh3_rk4_x2_item).
// The queue comes as a parameter of its own, before the arguments: read from the end of
// IntegrateArgs the same code took 5,041 us (5,172 in another process) for 1,048,576 particles x
// 200 steps with the state copies, this way 4,960.
template <bool PP, bool TAPE>
__global__ void __launch_bounds__(HH3::MAX_BLOCK / 2, 3) hh3_rk4_x2_kernel(
        WorkQueue* queue, const __grid_constant__ IntegrateArgs a) {
    // handed out (equal shares: 1,048,576 particles x 200 steps 5,021 us, handed out 4,894 us)
    warp_tasks(queue, (a.n_vec + 31) / 32, [&](int64_t w) {
        const int64_t t = w * 32 + (threadIdx.x & 31);
        if (t < a.n_vec) hh3_rk4_x2_item<PP, TAPE>(a, t, (int)a.n_steps);
    });
}

// One neuron per lane: lanes 3j, 3j + 1 and 3j + 2 of a warp (j < 10) hold neurons 0, 1 and 2
// of one particle (PER 1, floats) or of the particle pair 2j, 2j + 1 of the warp's 20 (PER 2, one
// f32x2 register per quantity); lanes 30 and 31 compute on a copy of a particle and write nothing.
// The neurons meet only in the sum of the three s, which goes round the triple by shuffles in
// the order of HH3::f, so the states are the other kernels' to the bit.  For ensembles too small
// to fill the GPU a step takes the latency and issue of one warp's instructions: here a warp holds
// 10 or 20 particles where the other kernels hold 32 or 64.  Measured, 100 steps with w warps on
// every SM sub-partition: 9 + 18 w us on floats, 41, 72, 104, 136, 168 us in pairs, against
// 10 + 91 w us of the particle-pair kernel and 104 us up to 19,456 particles, then 131, 227 of
// one particle per thread: 12,345 particles take 63 us instead of 104.  R is HH3.
// (A bound of 20 warps per SM instead of 16 measured 8% slower on pairs.)
template <class R, int PER> struct LaneType { using type = HHPair; };
template <class R> struct LaneType<R, 1> { using type = HHScalar; };

template <int PER> struct LaneOps;  // the lane type's loads, stores and constants
template <> struct LaneOps<1> {
    using T = float;
    __device__ __forceinline__ static T load(const float* p) { return *p; }
    __device__ __forceinline__ static void store(float* p, T v) { *p = v; }
    __device__ __forceinline__ static T shfl(T v, int src) { return __shfl_sync(0xffffffffu, v, src); }
    __device__ __forceinline__ static T join(float a, float) { return a; }
    __device__ __forceinline__ static HHConst<HHScalar> consts(const float* pa, const float*) {
        return hh_const<HHScalar>(pa);
    }
};
template <> struct LaneOps<2> {
    using T = f2;
    __device__ __forceinline__ static T load(const float* p) {
        float v[2];
        Vec<2>::load(p, v);
        return pack2(v[0], v[1]);
    }
    __device__ __forceinline__ static void store(float* p, T x) {
        float v[2];
        unpack2(x, v[0], v[1]);
        Vec<2>::store(p, v);
    }
    __device__ __forceinline__ static T shfl(T v, int src) {
        T r;
        r.v = __shfl_sync(0xffffffffu, v.v, src);
        return r;
    }
    __device__ __forceinline__ static T join(float a, float b) { return pack2(a, b); }
    __device__ __forceinline__ static HHConst<HHPair> consts(const float* pa, const float* pb) {
        return hh_const_pair(pa, pb);
    }
};

template <class R, int PER, bool PP, bool TAPE>
__global__ void __launch_bounds__(32, 16) lane_integrate_kernel(const __grid_constant__ IntegrateArgs a) {
    using O = typename LaneType<R, PER>::type;
    using T = typename O::T;
    using L = LaneOps<PER>;
    constexpr int kWarp = 10 * PER;  // particles per warp
    const int lane = threadIdx.x;
    const int j = lane / 3, n = lane - 3 * j, src0 = 3 * j;  // lanes 30 and 31: their sums are discarded
    const int64_t tasks = (a.n_vec + kWarp - 1) / kWarp;  // n_vec: particles, a multiple of 4
    for (int64_t w = blockIdx.x; w < tasks; w += gridDim.x) {
        const int64_t first = w * kWarp, own = first + PER * j;
        const bool valid = lane < 30 && own < a.n_vec;
        const int64_t i0 = valid ? own : first;  // a multiple of PER, so the loads are aligned
        float* ck0 = TAPE ? start_checkpoint(a) : nullptr;
        T X[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) X[k] = L::load(a.x + (int64_t)(5 * n + k) * a.pitch + i0);
        auto put = [&](float* planes) {
#pragma unroll
            for (int k = 0; k < 5; ++k)
                if (valid) L::store(planes + (int64_t)(5 * n + k) * a.pitch + i0, X[k]);
        };
        if (ck0) put(ck0);
        float hs[2], pa[R::NP], pb[R::NP];
        hh_pair_params<PP, PER>(a, i0, hs, pa, pb);
        const HHConst<O> c = L::consts(pa, pb);
        const T drive = L::join(hh_drive_c(pa, n), hh_drive_c(pb, n));
        const T H1 = L::join(hs[0], hs[1]), H2 = L::join(0.5f * hs[0], 0.5f * hs[1]);
        const T H6 = L::join(hs[0] * (1.0f / 6.0f), hs[1] * (1.0f / 6.0f));
        auto step = [&]() {
            T XS[5], A[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) XS[k] = X[k];
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                const T s_sum = O::add(O::add(L::shfl(XS[4], src0), L::shfl(XS[4], src0 + 1)), L::shfl(XS[4], src0 + 2));
                T K[5];
                hh_neuron<O>(XS[0], XS[1], XS[2], XS[3], XS[4], O::sub(s_sum, XS[4]), drive, c, K);
#pragma unroll
                for (int k = 0; k < 5; ++k) A[k] = rk4_weigh<O>(st, K[k], A[k]);
                if (st == 3) break;
                const T C = (st == 2) ? H1 : H2;
#pragma unroll
                for (int k = 0; k < 5; ++k) XS[k] = O::fma(C, K[k], X[k]);
            }
#pragma unroll
            for (int k = 0; k < 5; ++k) X[k] = O::fma(H6, A[k], X[k]);
        };
        run_steps<1, TAPE>(a, (int)a.n_steps, step, [&](int slot) { put(a.ckpt + (int64_t)slot * a.ck_stride); });
        put(a.x);
    }
}

// Launch of a lane kernel: blocks of one warp, which spread evenly over the SMs.
template <int PER, bool PP, bool TAPE>
cudaError_t lane_launch_one(const IntegrateArgs& a, const LaunchShape& s, cudaStream_t stream) {
    auto kernel = lane_integrate_kernel<HH3, PER, PP, TAPE>;
    int occ = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 32, 0);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const int limit = with_block_of(s, 32, HH3::MAX_BLOCK).blocks_per_sm;  // the caller's, in warps
    const int per_sm = (limit > 0 && limit < occ) ? limit : occ;
    const int64_t need = (a.n_vec + 10 * PER - 1) / (10 * PER), cap = (int64_t)per_sm * s.num_sms;
    const int grid = (int)(need < cap ? need : cap);
    if (grid < 1) return cudaSuccess;
    kernel<<<grid, 32, 0, stream>>>(a);
    last_launch_record() = LaunchRecord{(const void*)kernel, grid, 32};
    return cudaGetLastError();
}

template <int PER>
cudaError_t lane_launch(bool pp, const IntegrateArgs& a, const LaunchShape& s, cudaStream_t stream) {
    if (a.ckpt) return pp ? lane_launch_one<PER, true, true>(a, s, stream) : lane_launch_one<PER, false, true>(a, s, stream);
    return pp ? lane_launch_one<PER, true, false>(a, s, stream) : lane_launch_one<PER, false, false>(a, s, stream);
}

}  // namespace

cudaError_t launch_integrate_hh3(int method, bool kahan, bool pp, const IntegrateArgs& a,
                                 const LaunchShape& shape, cudaStream_t stream) {
    if (shape.ppt == 2) {
        const int64_t n = a.n_vec * 2;  // particles
        const int64_t subs = 4 * (int64_t)shape.num_sms;  // SM sub-partitions
        IntegrateArgs a1 = a;
        LaunchShape s1 = shape;
        a1.n_vec = n;
        s1.ppt = 1;
        // Euler, the compensated update and particle reset: one particle per thread
        if (method != FF_RK4 || kahan || a.reset) return launch_variants<HH3>(method, kahan, pp, a1, s1, stream);
        // The plain RK4 kernels give the same bits, so the ensemble's size decides.  Three warps of
        // 10 particles on a sub-partition take 63 us per 100 steps and two of 20 take 72, four of 10
        // take 82; five warps of 20 take 168 us and one and two pair warps (64 particles) 102
        // and 193, so the pairs are ahead where one warp of them is nearly full and beyond 100
        // particles a sub-partition.
        if (n <= 30 * subs) return lane_launch<1>(pp, a1, s1, stream);
        if (n <= 100 * subs && !(n > 60 * subs && n <= 64 * subs)) return lane_launch<2>(pp, a1, s1, stream);
        if (a.ckpt)
            return pp ? persistent_launch(hh3_rk4_x2_kernel<true, true>, a, shape, stream, a.queue)
                      : persistent_launch(hh3_rk4_x2_kernel<false, true>, a, shape, stream, a.queue);
        return pp ? persistent_launch(hh3_rk4_x2_kernel<true, false>, a, shape, stream, a.queue)
                  : persistent_launch(hh3_rk4_x2_kernel<false, false>, a, shape, stream, a.queue);
    }
    return launch_variants<HH3>(method, kahan, pp, a, shape, stream);
}

}  // namespace ff
