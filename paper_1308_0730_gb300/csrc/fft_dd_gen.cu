// Kernels and launchers of the mixed-radix double-float passes (tile functions in
// fft_dd.cuh).
#include "fft_dd.cuh"

namespace mvd {

namespace {

// Mixed-radix double-float passes: four blocks of 256 threads per SM. At 64 registers they
// spill (bytes stored and loaded: z with the product 188 and 332, update 112 and 328, ratio
// 124 and 244, the others at most 76 and 112), but they wait on loads more than they issue:
// 300x180x150, a view update with 3, 4 and 5 blocks (the tiles sized to fit, all passes
// together) 739, 661 and 698 us.
constexpr int kDdGenBlocks = 4;

__global__ void __launch_bounds__(kGenThreads, kDdGenBlocks) k_dd_x_forward(const __grid_constant__ DdX a) {
    extern __shared__ cdd smd[];
    pass_wait();
    dd_x_forward_tile<false>(a, blockIdx.x, smd);
}

__global__ void __launch_bounds__(kGenThreads, kDdGenBlocks) k_dd_x_ratio(const __grid_constant__ DdX a) {
    extern __shared__ cdd smd[];
    pass_wait();
    dd_x_ratio_tile<false>(a, blockIdx.x, smd);
}

template <int MODE>
__global__ void __launch_bounds__(kGenThreads, kDdGenBlocks) k_dd_x_update(const __grid_constant__ DdXU u) {
    extern __shared__ cdd smd[];
    pass_wait();
    dd_x_update_tile<false, MODE>(u, blockIdx.x, smd);
}

template <int S, bool F32 = false>
__global__ void __launch_bounds__(kGenThreads, kDdGenBlocks) k_dd_y(const __grid_constant__ DdY a) {
    extern __shared__ cdd smd[];
    pass_wait();
    dd_y_tile<false, S, F32>(a, blockIdx.x, smd);
}

template <bool MUL>
__global__ void __launch_bounds__(kGenThreads, kDdGenBlocks) k_dd_z(const __grid_constant__ DdZ a) {
    extern __shared__ cdd smd[];
    pass_wait();
    dd_z_tile<false, MUL>(a, blockIdx.x, smd);
}

template <typename K, typename A>
mvd_status launch(K kern, const A& a, const LineGeo& g, long grid, cudaStream_t st, const char* name, int cls) {
    const size_t smem = dd_smem(g);
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return cuda_status(e, name);
    prof_begin(cls, st);
    e = launch_pass(kern, dim3((unsigned)grid), g.T, smem, st, a);
    prof_end(cls, st);
    if (e != cudaSuccess) return cuda_status(e, name);
    count_launch();
    return check_launch(name);
}

}  // namespace

mvd_status dd_forward_real_generic(const FftGeom& g, const float* src, cdd* S2, cudaStream_t st) {
    DdX a = dd_x_args(g.X, g.YZ, g.px, g.tw2x);
    a.src = src;
    a.S2 = S2;
    return launch(k_dd_x_forward, a, a.g, dd_x_tiles(g.px, g.YZ), st, "dd x forward", KC_DD_X_FORWARD);
}

mvd_status dd_x_ratio_generic(const FftGeom& g, cdd* S2, const float* phi, float eps, cudaStream_t st, float2* S) {
    DdX a = dd_x_args(g.X, g.YZ, g.px, g.tw2x);
    a.S2 = S2;
    a.S = S;
    a.phi = phi;
    a.eps = eps;
    return launch(k_dd_x_ratio, a, a.g, dd_x_tiles(g.px, g.YZ), st, "dd x ratio", KC_DD_X_RATIO);
}

mvd_status dd_y_generic(const FftGeom& g, cdd* S2, int inverse, const float2* S1, cudaStream_t st) {
    DdY a = dd_y_args(g.Xh, g.Z, g.py, g.tw2y, S2);
    a.S1 = S1;
    return launch(S1 ? k_dd_y<-1, true> : inverse ? k_dd_y<+1> : k_dd_y<-1>, a, a.g, dd_y_tiles(g.py, g.Xh, g.Z), st,
                  "dd y", KC_DD_Y);
}

mvd_status dd_x_update_generic(const FftGeom& g, const cdd* S2, float* psi, float eps, cudaStream_t st,
                               const float* wt, float lam, const float* inv_s, int accumulate) {
    DdXU u{};
    u.x = dd_x_args(g.X, g.YZ, g.px, g.tw2x);
    u.x.S2 = const_cast<cdd*>(S2);
    u.x.eps = eps;
    u.psi = psi;
    u.wt = wt;
    u.lam = lam;
    u.inv_s = inv_s;
    return launch(accumulate ? k_dd_x_update<4> : k_dd_x_update<1>, u, u.x.g, dd_x_tiles(g.px, g.YZ), st, "dd x update",
                  KC_X_UPDATE);
}

mvd_status dd_x_inverse_real_generic(const FftGeom& g, const cdd* S2, float* dst, cudaStream_t st) {
    DdXU u{};
    u.x = dd_x_args(g.X, g.YZ, g.px, g.tw2x);
    u.x.S2 = const_cast<cdd*>(S2);
    u.psi = dst;
    return launch(k_dd_x_update<0>, u, u.x.g, dd_x_tiles(g.px, g.YZ), st, "dd x inverse", KC_X_UPDATE);
}

mvd_status dd_z_generic(const FftGeom& g, cdd* S2, const cdd* K2, double scale, cudaStream_t st) {
    const float hi = (float)scale;
    DdZ a = dd_z_args(g.Y, g.YZ, g.pz, g.tw2z, S2, K2, dd{hi, (float)(scale - (double)hi)});
    return launch(K2 ? k_dd_z<true> : k_dd_z<false>, a, a.g, dd_z_tiles(g.pz, g.Y, g.Xh), st, K2 ? "dd z" : "dd z forward",
                  K2 ? KC_DD_Z_MUL : KC_SETUP);
}

}  // namespace mvd
