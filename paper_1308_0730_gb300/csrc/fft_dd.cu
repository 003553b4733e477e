// Kernels and launchers of the register-resident double-float passes (tile
// functions in fft_dd_fast.cuh); other lengths go to fft_dd_gen.cu.
#include <type_traits>

#include "fft_dd_fast.cuh"

namespace mvd {

namespace {

// register-resident double-float passes (power-of-two lengths)
template <int L, int S, int IO = 0>
__global__ void __launch_bounds__(kDdThreads, dd_blocks(dd_e(L))) k_ddf_y(cdd* S2, long nlines, const cdd* tw2, float2* S1) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_y_tile<L, S, false, IO>(S2, nlines, tw2, blockIdx.x, smd, S1);
}

template <int L, bool MUL>
__global__ void __launch_bounds__(512) k_ddf_z(cdd* S2, const cdd* K2, int Y, long YZ, int ntiles_y, dd scale,
                                               const cdd* tw2) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_z_tile<L, MUL, false>(S2, K2, Y, YZ, ntiles_y, scale, tw2, blockIdx.x, smd);
}

template <int L>
__global__ void __launch_bounds__(z2_threads(L), 3) k_ddf_z2_pipe(cdd* S2, const cdd* K2, int Y, long YZ, int ntiles_y,
                                                              const cdd* tw2, long ntiles) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_z2_pipe<L>(S2, K2, Y, YZ, ntiles_y, tw2, ntiles, smd);
}

template <int L>
__global__ void __launch_bounds__(kDdThreads, dd_blocks(dd_e(L))) k_ddf_x_forward(const __grid_constant__ DdXFast a) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_x_forward_tile<L, false>(a, blockIdx.x, smd);
}

template <int L>
__global__ void __launch_bounds__(kDdThreads) k_ddf_x_inverse(const __grid_constant__ DdXFast a) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_x_inverse_tile<L, false>(a, blockIdx.x, smd);
}

template <int L>
__global__ void __launch_bounds__(kDdThreads, dd_blocks(kXInvE)) k_ddf_x_ratio(const __grid_constant__ DdXFast a) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_x_ratio_tile<L, false>(a, blockIdx.x, smd);
}

template <int L, int MODE>
__global__ void __launch_bounds__(kDdThreads, dd_blocks(kXInvE)) k_ddf_x_update(const __grid_constant__ DdXUpd a) {
    extern __shared__ cdd smd[];
    pass_wait();
    ddf_x_update_tile<L, MODE>(a, blockIdx.x, smd);
}




template <typename F>
bool with_dd_len(int L, F&& f) {
    switch (L) {
        case 32: f(std::integral_constant<int, 32>{}); return true;
        case 64: f(std::integral_constant<int, 64>{}); return true;
        case 128: f(std::integral_constant<int, 128>{}); return true;
        case 256: f(std::integral_constant<int, 256>{}); return true;
        case 512: f(std::integral_constant<int, 512>{}); return true;
        case 1024: f(std::integral_constant<int, 1024>{}); return true;
        default: return false;
    }
}

template <typename K, typename... Args>
mvd_status launch_raw(K kern, long grid, int threads, size_t smem, cudaStream_t st, const char* name, int cls,
                      Args... args) {
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return cuda_status(e, name);
    prof_begin(cls, st);
    e = launch_pass(kern, dim3((unsigned)grid), threads, smem, st, args...);
    prof_end(cls, st);
    if (e != cudaSuccess) return cuda_status(e, name);
    count_launch();
    return check_launch(name);
}

// blocks of a persistent launch: as many as fit on every SM at once, at most one per tile
template <typename K>
long persistent_grid(K kern, int threads, size_t smem, long ntiles) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    allow_smem(kern);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const long g = (long)per_sm * (sms > 0 ? sms : 1);
    return g < ntiles ? g : ntiles;
}

DdXFast ddf_args(const FftGeom& g) {
    DdXFast a{};
    a.YZ = g.YZ;
    a.tw2 = g.tw2x;
    a.plan = g.px;
    return a;
}

}  // namespace

mvd_status dd_forward_real(const FftGeom& g, const float* src, cdd* S2, cudaStream_t st) {
    if (g.fast && dd_fast_length(g.X)) {
        mvd_status rc = MVD_ERR_UNSUPPORTED;
        DdXFast a = ddf_args(g);
        a.src = src;
        a.S2 = S2;
        with_dd_len(g.X, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            rc = launch_raw(k_ddf_x_forward<L>, gen_div_up(g.YZ, 2 * ddf_pairs(L, dd_e(L))), kDdThreads, ddf_xf_smem(L), st,
                            "dd x forward (fast)", KC_DD_X_FORWARD, a);
        });
        return rc;
    }
    return dd_forward_real_generic(g, src, S2, st);
}

bool dd_fast_x(const FftGeom& g) { return g.fast && dd_fast_length(g.X); }

mvd_status dd_x_inverse_real(const FftGeom& g, const cdd* S2, float* dst, cudaStream_t st) {
    if (!(g.fast && dd_fast_length(g.X))) {
        set_error("dd x inverse: length %d has no register-resident double-float transform", g.X);
        return MVD_ERR_UNSUPPORTED;
    }
    mvd_status rc = MVD_ERR_UNSUPPORTED;
    DdXFast a = ddf_args(g);
    a.S2 = const_cast<cdd*>(S2);
    a.dst = dst;
    with_dd_len(g.X, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        rc = launch_raw(k_ddf_x_inverse<L>, gen_div_up(g.YZ, 2 * ddf_pairs(L, kXInvE)), kDdThreads, ddf_x_smem(L), st,
                        "dd x inverse (fast)", KC_DD_X_RATIO, a);
    });
    return rc;
}

mvd_status dd_x_ratio(const FftGeom& g, cdd* S2, const float* phi, float eps, cudaStream_t st, float2* S) {
    if (g.fast && dd_fast_length(g.X)) {
        mvd_status rc = MVD_ERR_UNSUPPORTED;
        DdXFast a = ddf_args(g);
        a.S2 = S2;
        a.S = S;
        a.phi = phi;
        a.eps = eps;
        with_dd_len(g.X, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            rc = launch_raw(k_ddf_x_ratio<L>, gen_div_up(g.YZ, 2 * ddf_pairs(L, kXInvE)), kDdThreads, ddf_ratio_smem(L), st,
                            "dd x ratio (fast)", KC_DD_X_RATIO, a);
        });
        return rc;
    }
    return dd_x_ratio_generic(g, S2, phi, eps, st, S);
}

mvd_status dd_y(const FftGeom& g, cdd* S2, int inverse, cudaStream_t st) {
    if (g.fast && dd_fast_length(g.Y)) {
        mvd_status rc = MVD_ERR_UNSUPPORTED;
        const long nl = (long)g.Xh * g.Z;
        with_dd_len(g.Y, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            rc = launch_raw(inverse ? k_ddf_y<L, +1> : k_ddf_y<L, -1>, gen_div_up(nl, ddf_y_lines(L)), kDdThreads,
                            ddf_y_smem(L), st, "dd y (fast)", KC_DD_Y, S2, nl, g.tw2y, (float2*)nullptr);
        });
        return rc;
    }
    return dd_y_generic(g, S2, inverse, nullptr, st);
}

mvd_status dd_y_from_f32(const FftGeom& g, const float2* S1, cdd* S2, cudaStream_t st) {
    if (!(g.fast && dd_fast_length(g.Y))) return dd_y_generic(g, S2, 0, S1, st);
    mvd_status rc = MVD_ERR_UNSUPPORTED;
    const long nl = (long)g.Xh * g.Z;
    with_dd_len(g.Y, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        rc = launch_raw(k_ddf_y<L, -1, 1>, gen_div_up(nl, ddf_y_lines(L)), kDdThreads, ddf_y_smem(L), st,
                        "dd y (FP32 in)", KC_DD_Y, S2, nl, g.tw2y, const_cast<float2*>(S1));
    });
    return rc;
}

mvd_status dd_x_update(const FftGeom& g, const cdd* S2, float* psi, float eps, cudaStream_t st, const float* wt,
                       float lam, const float* inv_s, int accumulate) {
    if (!dd_fast_x(g)) return dd_x_update_generic(g, S2, psi, eps, st, wt, lam, inv_s, accumulate);
    mvd_status rc = MVD_ERR_UNSUPPORTED;
    DdXUpd a{S2, psi, g.YZ, eps, g.tw2x, wt, lam, inv_s};
    with_dd_len(g.X, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        rc = launch_raw(accumulate ? k_ddf_x_update<L, 4> : k_ddf_x_update<L, 1>, gen_div_up(g.YZ, 2 * ddf_pairs(L, kXInvE)),
                        kDdThreads, ddf_ratio_smem(L), st, "dd x update", KC_X_UPDATE, a);
    });
    return rc;
}

static mvd_status ddf_z(const FftGeom& g, cdd* S2, const cdd* K2, dd scale, bool mul, cudaStream_t st) {
    mvd_status rc = MVD_ERR_UNSUPPORTED;
    with_dd_len(g.Z, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        constexpr int Q = ddf_z_cols(L);
        const int threads = Q * (L / dd_e(L));
        const int nty = (int)gen_div_up(g.Y, Q);
        rc = launch_raw(mul ? k_ddf_z<L, true> : k_ddf_z<L, false>, (long)g.Xh * nty, threads, ddf_z_smem(L), st,
                        "dd z (fast)", mul ? KC_DD_Z_MUL : KC_SETUP, S2, K2, g.Y, g.YZ, nty, scale, g.tw2z);
    });
    return rc;
}

mvd_status dd_z_mul(const FftGeom& g, cdd* S2, const cdd* K2, cudaStream_t st) {
    if (g.fast && ddf_z2_length(g.Z)) {
        mvd_status rc = MVD_ERR_UNSUPPORTED;
        with_dd_len(g.Z, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            if constexpr (ddf_z2_length(L)) {
                constexpr int Q = z2_cols(L);
                const int nty = (int)gen_div_up(g.Y, Q);
                const long nt = (long)g.Xh * nty;
                const size_t smem = ddf_z2_pipe_smem(L);
                rc = launch_raw(k_ddf_z2_pipe<L>, persistent_grid(k_ddf_z2_pipe<L>, z2_threads(L), smem, nt),
                                z2_threads(L), smem, st, "dd z", KC_DD_Z_MUL, S2, K2, g.Y, g.YZ, nty, g.tw2z, nt);
            }
        });
        return rc;
    }
    if (g.fast && dd_fast_length(g.Z)) return ddf_z(g, S2, K2, dd{1.f, 0.f}, true, st);
    return dd_z_generic(g, S2, K2, 1.0, st);
}

mvd_status dd_z_forward_scaled(const FftGeom& g, cdd* S2, double scale, cudaStream_t st) {
    const float hi = (float)scale;
    if (g.fast && dd_fast_length(g.Z)) return ddf_z(g, S2, nullptr, dd{hi, (float)(scale - (double)hi)}, false, st);
    return dd_z_generic(g, S2, nullptr, scale, st);
}

}  // namespace mvd
