// Direct periodic 3D convolution for small kernels, with the update's
// elementwise steps fused into the epilogue:
//   ratio : r   = phi / max(psi * P, eps)        (Eq. 15 / Eq. 51, first half)
//   update: psi = max(psi . (r * K), eps)         (Eq. 15 / Eq. 220, second half)
// (f * k)(x) = sum_d k(d) f((x - d) mod dims), d = tap index - (K-1)/2.
//
// The tiling and its cost are in box_conv.cuh; the elementwise steps run in its
// epilogue. Measured (GB300): see k_direct.
#include "box_conv.cuh"
#include "common.cuh"
#include "fft.cuh"

namespace mvd {

namespace {

// The boxes this engine takes: those whose input tile (32 x 1 x 4 outputs plus
// the box's halo) and taps fit in 200 KB of shared memory.
constexpr size_t kMaxSmem = 200 * 1024;

inline bool box_fits(const int kd[3], int ty) {
    const size_t T = (size_t)kd[0] * kd[1] * kd[2];
    const size_t tile = (size_t)(32 + kd[0] - 1) * (ty + kd[1] - 1) * (4 + kd[2] - 1);
    return (T + tile) * sizeof(float) <= kMaxSmem;
}

struct DArgs {
    BoxConv c;
    const float* phi;
    float* out;  // r (ratio), psi (update) or plain output
    float eps;
    const float* wt;     // update: when set, apply the fraction wt of the change (partial overlap)
    float lam;           // update: Tikhonov regularisation (0 = none)
    const float* inv_s;  // update / accumulate: zero boundary, 1 / sensitivity
    int splits, mode;
};

enum { M_RATIO, M_UPDATE, M_CONV, M_ADD, M_ACCUMULATE };

// M_RATIO: out = phi / max(conv, eps); M_UPDATE: out = max(out . conv, eps); M_CONV: out = conv;
// M_ADD: out += conv; M_ACCUMULATE: out *= conv (the combined update's product).
__device__ __forceinline__ void finish(const DArgs& a, long g, float acc) {
    if (a.mode == M_RATIO) {
        a.out[g] = __ldg(a.phi + g) / fmaxf(acc, a.eps);
    } else if (a.mode == M_UPDATE) {
        const float p = a.out[g];
        a.out[g] = fmaxf(p * (a.wt || a.lam != 0.f || a.inv_s ? update_factor(acc - 1.f, p, a.wt, g, a.lam, a.inv_s)
                                                              : acc),
                         a.eps);
    } else if (a.mode == M_CONV) {
        a.out[g] = acc;
    } else if (a.mode == M_ADD) {
        a.out[g] += acc;
    } else {
        a.out[g] *= a.inv_s ? acc * __ldg(a.inv_s + g) : acc;
    }
}

// KX: the box's length in x, 0 for those without a kernel of their own, -1 for planes staged in
// rows. Blocks of 256 threads have 80 registers, for three of them per SM: with one kernel for
// both sizes of block the 8-row tiles took 82 to 103, which left two (97x83x61, 9x9x15: 48.4
// against 44.7 us a launch); held to 80, blocks of 512 gain nothing (three updates of 32^3: 69
// and 73 us).
template <int NY, int KX, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 3 : 1) k_direct(const __grid_constant__ DArgs a) {
    extern __shared__ float4 smem4[];
    pass_wait();
    bc_tile<NY, KX, true, false>(a.c, blockIdx.x, blockIdx.y, blockIdx.z, a.splits, reinterpret_cast<float*>(smem4),
                                 [&](int x, int y, int z, float acc) {
        finish(a, (long)x + (long)a.c.ox * (y + (long)a.c.oy * z), acc);
    });
}

// One tap: nothing to stage, memory bound (two views of 128^3: 82 us an iteration through the
// tiles, 72 with one output row per thread; 27 here; 32^3 23, 19 and 8.7).
__global__ void __launch_bounds__(256) k_point(const __grid_constant__ DArgs a, long n) {
    pass_wait();
    const float t = __ldg(a.c.taps);
    for (long g = blockIdx.x * 256L + threadIdx.x; g < n; g += 256L * gridDim.x) finish(a, g, t * a.c.in[g]);
}

template <int NY, int THREADS>
auto kernel_for(int kx) {
    switch (kx) {  // the short rows, whose loop and remainder would cost as much as their taps
        case 3: return k_direct<NY, 3, THREADS>;
        case 5: return k_direct<NY, 5, THREADS>;
        case 7: return k_direct<NY, 7, THREADS>;
        case 9: return k_direct<NY, 9, THREADS>;
        case 11: return k_direct<NY, 11, THREADS>;
        case 13: return k_direct<NY, 13, THREADS>;
        case 15: return k_direct<NY, 15, THREADS>;
        case 17: return k_direct<NY, 17, THREADS>;
        case -1: return k_direct<NY, -1, THREADS>;
        default: return k_direct<NY, 0, THREADS>;
    }
}

// ty 0 or 8: the cheaper of the 16- and 8-row tiles (bc_plan); 4, 2, 1: the 8-row tile
mvd_status launch(DArgs& a, int mode, cudaStream_t st, const char* name, int ty = 0) {
    BoxConv& c = a.c;
    const int kd[3] = {c.kx, c.ky, c.kz};
    BcPlan p{};
    if (!direct_supported(kd) || !bc_plan(c.ox, c.oy, c.oz, c.kx, c.ky, c.kz, ty == 0 || ty == 8 ? 2 : 1, &p)) {
        set_error("%s: kernel box %dx%dx%d too large for the direct engine", name, kd[0], kd[1], kd[2]);
        return MVD_ERR_UNSUPPORTED;
    }
    c.ck = p.ck;
    c.cy = p.cy;
    c.cx = p.cx;
    a.splits = p.s;
    a.mode = mode;
    const int kx = p.cy < c.ky || p.cx < c.kx ? -1 : c.kx;
    auto kern = p.ny == 2 ? kernel_for<2, 256>(kx) : p.warps == 8 ? kernel_for<1, 256>(kx) : kernel_for<1, 512>(kx);
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return cuda_status(e, name);
    const int nz = p.planes();
    const dim3 grid((c.ox + kBcTX - 1) / kBcTX, (c.oy + 8 * p.ny - 1) / (8 * p.ny), (c.oz + nz - 1) / nz);
    const long n = (long)c.ox * c.oy * c.oz, points = (n + 255) / 256;
    const int cls = mode == M_RATIO ? KC_DIRECT_RATIO
                                    : (mode == M_UPDATE || mode == M_ACCUMULATE) ? KC_DIRECT_UPDATE : KC_DIRECT_CONV;
    prof_begin(cls, st);
    if (c.kx * c.ky * c.kz == 1)
        e = launch_pass(k_point, dim3((unsigned)(points < 152 * 16 ? points : 152 * 16)), 256, 0, st, a, n);
    else
        e = launch_pass(kern, grid, 32 * p.warps, p.smem, st, a);
    prof_end(cls, st);
    if (e != cudaSuccess) return cuda_status(e, name);
    count_launch();
    return check_launch(name);
}

// (f * k)(x) = sum_t k(K - 1 - t) f(x + t - h): the taps reversed, the input starting h before the output
DArgs make(const int dims[3], const float* in, const float* k, const int kd[3]) {
    DArgs a{};
    BoxConv& c = a.c;
    c.in = in;
    c.taps = k;
    c.ix = c.ox = dims[0];
    c.iy = c.oy = dims[1];
    c.iz = c.oz = dims[2];
    c.kx = kd[0];
    c.ky = kd[1];
    c.kz = kd[2];
    c.offx = -((kd[0] - 1) / 2);
    c.offy = -((kd[1] - 1) / 2);
    c.offz = -((kd[2] - 1) / 2);
    c.mir = 1;
    return a;
}

}  // namespace

bool direct_supported(const int kd[3]) { return box_fits(kd, 1); }

mvd_status direct_ratio(const int dims[3], const float* psi, const float* k, const int kd[3],
                        const float* phi, float eps, float* r, cudaStream_t st, int ty) {
    DArgs a = make(dims, psi, k, kd);
    a.phi = phi;
    a.out = r;
    a.eps = eps;
    return launch(a, M_RATIO, st, "direct ratio", ty);
}

mvd_status direct_update(const int dims[3], const float* r, const float* k, const int kd[3],
                         float* psi, float eps, cudaStream_t st, int ty, const float* wt, float lam,
                         const float* inv_s) {
    DArgs a = make(dims, r, k, kd);
    a.out = psi;
    a.eps = eps;
    a.wt = wt;
    a.lam = lam;
    a.inv_s = inv_s;
    return launch(a, M_UPDATE, st, "direct update", ty);
}

mvd_status direct_accumulate(const int dims[3], const float* r, const float* k, const int kd[3], float* prod,
                             cudaStream_t st, int ty, const float* inv_s) {
    DArgs a = make(dims, r, k, kd);
    a.out = prod;
    a.inv_s = inv_s;
    return launch(a, M_ACCUMULATE, st, "direct accumulate", ty);
}

mvd_status direct_conv(const int dims[3], const float* in, const float* k, const int kd[3], float* out,
                       cudaStream_t st) {
    DArgs a = make(dims, in, k, kd);
    a.out = out;
    return launch(a, M_CONV, st, "direct conv");
}

mvd_status direct_conv_add(const int dims[3], const float* in, const float* k, const int kd[3], float* out,
                           cudaStream_t st) {
    DArgs a = make(dims, in, k, kd);
    a.out = out;
    return launch(a, M_ADD, st, "direct conv add");
}

}  // namespace mvd
