// FP32 passes of any {2,3,5}-smooth length as tile-level device functions: the
// per-volume kernels (fft_passes.cu) run one tile per block, the persistent batch
// kernel (batch.cu) runs whichever tile its work queue hands out. CO = true makes
// every load of data written inside the same launch (spectrum, estimate) an L2 load,
// as the batch kernel requires. Transforms and tile geometry: lines.cuh.
//
// Layout and contract as in fft_passes.cu: spectrum S[kx][z][y], two real
// x-lines per complex line, 1/M folded into the kernel spectra.
#pragma once

#include "dd.cuh"
#include "fft.cuh"
#include "lines.cuh"

namespace mvd {

constexpr int kGenThreads = 256;

__host__ __device__ inline long gen_div_up(long a, long b) { return (a + b - 1) / b; }

// rows of half spectra staged by an x inverse: odd stride
__host__ __device__ inline int x_half_stride(int X) { return (X / 2 + 1) | 1; }

// geometry of the x (lines = row pairs), y and z passes
__host__ __device__ inline LineGeo gen_x_geo(const FftPlan& p) {
    LineGeo g{};
    g.L = p.L;
    g.ln = tile_lines_log2(p, f32_tile_rule(), 32);
    const int hs = 2 * x_half_stride(p.L);  // 2n staged rows share one exchange buffer
    g.ls = line_stride_for(p.L > hs ? p.L : hs, g.n(), 16);
    g.T = tile_threads(p, g.ln);
    return g;
}
__host__ __device__ inline LineGeo gen_line_geo(const FftPlan& p, int most) {
    LineGeo g{};
    g.L = p.L;
    g.ln = tile_lines_log2(p, f32_tile_rule(), most);
    g.ls = line_stride_for(p.L, g.n(), 16);
    g.T = tile_threads(p, g.ln);
    return g;
}
__host__ __device__ inline size_t gen_smem(const LineGeo& g) { return (size_t)2 * g.n() * g.ls * sizeof(float2); }

struct GenX {
    LineGeo g;
    int X, Xh;
    long YZ;
    FftPlan plan;
    const float* src;  // real rows (forward from a real volume)
    float2* S;
    const float* phi;  // ratio epilogue
    float* psi;        // update epilogue / real output
    float eps;
    const float* wt;   // when set, the update applies the fraction wt of the change (partial overlap)
    float lam;         // Tikhonov regularisation of the update (0 = none)
    const float* inv_s;  // zero boundary: 1 / sensitivity of the update's view, or none
};

__host__ __device__ inline GenX gen_x_args(int X, long YZ, const FftPlan& plan) {
    GenX a{};
    a.g = gen_x_geo(plan);
    a.X = X;
    a.Xh = X / 2 + 1;
    a.YZ = YZ;
    a.plan = plan;
    return a;
}
__host__ __device__ inline long gen_x_tiles(const FftPlan& p, long YZ) { return gen_div_up(YZ, 2 * gen_x_geo(p).n()); }

// the half spectra of rows rho0 .. rho0 + 2n - 1 into H (row r at r * x_half_stride)
template <bool CO>
__device__ __forceinline__ void gen_gather(const GenX& a, float2* H, long rho0, int nrows) {
    const int hs = x_half_stride(a.X), lr = a.g.ln + 1;
    const float2* S = a.S + rho0;
    for (int t = threadIdx.x; t < (a.Xh << lr); t += blockDim.x) {
        const int row = t & ((1 << lr) - 1), k = t >> lr;
        const bool ok = row < nrows;
        if constexpr (CO)  // an 8-byte asynchronous copy would go through L1
            H[row * hs + k] = ok ? ld2<CO>(S + (long)k * a.YZ + row) : make_float2(0.f, 0.f);
        else
            cp_async8(H + row * hs + k, ok ? S + (long)k * a.YZ + row : a.S, ok);
    }
    cp_async_wait_all();
}

// real volume -> spectrum, one tile of 2n rows; pair p = rows p and n + p
template <bool CO>
__device__ void gen_x_forward_tile(const GenX& a, long tile, float2* sm) {
    const int n = a.g.n(), ls = a.g.ls;
    const long rho0 = tile * 2 * n;
    const int nrows = (int)min((long)2 * n, a.YZ - rho0);
    const float* src = a.src + rho0 * a.X;
    const float2* F = line_transform<-1, float2, true, false, CO>(
        a.g, a.plan, a.plan.tw + 3 * a.X, sm, sm + n * ls, nullptr,
        [&](int p, int i) {
            return make_float2(p < nrows ? ld1<CO>(src + p * a.X + i) : 0.f,
                               n + p < nrows ? ld1<CO>(src + (n + p) * a.X + i) : 0.f);
        },
        [&](float2* buf, int p, int i, float2 v) { buf[p * ls + i] = v; });
    __syncthreads();
    float2* S = a.S + rho0;
    unpack_tile<float2>(F, ls, a.X, a.g.ln, nrows, [&](int k, int row, float2 v) { S[(long)k * a.YZ + row] = v; });
}

// inverse x of the tile's rows: last(buf, p, element, value)
template <bool CO, typename Last>
__device__ __forceinline__ float2* gen_x_inverse_lines(const GenX& a, long rho0, int nrows, float2* sm, Last&& last) {
    const int n = a.g.n(), hs = x_half_stride(a.X);
    float2* H = sm + n * a.g.ls;
    gen_gather<CO>(a, H, rho0, nrows);
    __syncthreads();
    return line_transform<+1, float2, false, true, CO>(
        a.g, a.plan, a.plan.tw + 3 * a.X, sm, H, nullptr,
        [&](int p, int k) {
            const bool up = k <= a.X / 2;
            const int kk = up ? k : a.X - k;
            return pack_pair(H[p * hs + kk], H[(n + p) * hs + kk], up);
        },
        last);
}

// spectrum -> inverse x -> r = phi / max(b, eps) -> forward x of r - 1 -> spectrum
// (transforming r - 1 instead of r keeps the large mean of r out of the FP32
// back-projection's rounding; the update adds the 1 back, since K sums to 1)
template <bool CO>
__device__ void gen_x_ratio_tile(const GenX& a, long tile, float2* sm) {
    const int n = a.g.n(), ls = a.g.ls;
    const long rho0 = tile * 2 * n;
    const int nrows = (int)min((long)2 * n, a.YZ - rho0);
    const float* phi = a.phi + rho0 * a.X;
    prefetch_rows(phi, nrows * a.X * 4);
    float2* R = gen_x_inverse_lines<CO>(a, rho0, nrows, sm, [&](float2* buf, int p, int i, float2 v) {
        const float ra = p < nrows ? __ldg(phi + p * a.X + i) / fmaxf(v.x, a.eps) - 1.f : 0.f;
        const float rb = n + p < nrows ? __ldg(phi + (n + p) * a.X + i) / fmaxf(v.y, a.eps) - 1.f : 0.f;
        buf[p * ls + i] = make_float2(ra, rb);
    });
    __syncthreads();
    const float2* F = line_transform<-1, float2, false, false, CO>(
        a.g, a.plan, a.plan.tw + 3 * a.X, R == sm ? sm + n * ls : sm, R, nullptr,
        [&](int p, int i) { return R[p * ls + i]; },
        [&](float2* buf, int p, int i, float2 v) { buf[p * ls + i] = v; });
    __syncthreads();
    float2* S = a.S + rho0;
    unpack_tile<float2>(F, ls, a.X, a.g.ln, nrows, [&](int k, int row, float2 v) { S[(long)k * a.YZ + row] = v; });
}

// MODE 0: plain real output ; 1: psi = max(psi . update_factor(c - 1), eps) ; 4: acc *= c (the
// combined update's product of view factors; acc in a.psi). The lines hold (r - 1) * K = c - 1.
template <bool CO, int MODE>
__device__ void gen_x_inverse_tile(const GenX& a, long tile, float2* sm) {
    const int n = a.g.n();
    const long rho0 = tile * 2 * n;
    const int nrows = (int)min((long)2 * n, a.YZ - rho0);
    if (MODE != 0) prefetch_rows(a.psi + rho0 * a.X, nrows * a.X * 4);
    gen_x_inverse_lines<CO>(a, rho0, nrows, sm, [&](float2*, int p, int i, float2 v) {
        const float cv[2] = {v.x, v.y};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = p + h * n;
            if (row >= nrows) continue;
            const long at = (rho0 + row) * a.X + i;
            if (MODE == 0) {
                a.psi[at] = cv[h];
                continue;
            }
            const float old = ld1<CO>(a.psi + at);
            if (MODE == 1)
                a.psi[at] = fmaxf(old * update_factor(cv[h], old, a.wt, at, a.lam, a.inv_s), a.eps);
            else
                a.psi[at] = old * (cv[h] + 1.f) * (a.inv_s ? __ldg(a.inv_s + at) : 1.f);
        }
    });
}

struct GenY {
    LineGeo g;
    long nlines;
    FftPlan plan;
    float2* S;
};

__host__ __device__ inline GenY gen_y_args(int Xh, int Z, const FftPlan& plan, float2* S) {
    GenY a{};
    a.g = gen_line_geo(plan, 32);
    a.nlines = (long)Xh * Z;
    a.plan = plan;
    a.S = S;
    return a;
}
__host__ __device__ inline long gen_y_tiles(const FftPlan& p, int Xh, int Z) {
    return gen_div_up((long)Xh * Z, gen_line_geo(p, 32).n());
}

// complex FFT along y: the spectrum is nlines = Xh*Z contiguous lines of Y
template <bool CO, int S>
__device__ void gen_y_tile(const GenY& a, long tile, float2* sm) {
    const int n = a.g.n(), L = a.g.L;
    const long l0 = tile * n;
    const int nl = (int)min((long)n, a.nlines - l0);
    float2* s = a.S + l0 * L;
    line_transform<S, float2, true, true, CO>(
        a.g, a.plan, a.plan.tw + 3 * L, sm, sm + n * a.g.ls, nullptr,
        [&](int l, int i) { return l < nl ? ld2<CO>(s + l * L + i) : make_float2(0.f, 0.f); },
        [&](float2*, int l, int i, float2 v) {
            if (l < nl) s[l * L + i] = v;
        });
}

struct GenZ {
    LineGeo g;
    int Y, ntiles_y;
    long YZ;
    FftPlan plan;
    float2* S;
    const float2* K;
    float scale;
};

__host__ __device__ inline GenZ gen_z_args(int Y, long YZ, const FftPlan& plan, float2* S, const float2* K,
                                           float scale) {
    GenZ a{};
    a.g = gen_line_geo(plan, Y);
    a.Y = Y;
    a.ntiles_y = (int)gen_div_up(Y, a.g.n());
    a.YZ = YZ;
    a.plan = plan;
    a.S = S;
    a.K = K;
    a.scale = scale;
    return a;
}
__host__ __device__ inline long gen_z_tiles(const FftPlan& p, int Y, int Xh) {
    return (long)Xh * gen_div_up(Y, gen_line_geo(p, Y).n());
}

// along z at fixed (kx, y0..y0+n-1): MUL -> forward, times K, inverse;
// otherwise forward, times scale
template <bool CO, bool MUL>
__device__ void gen_z_tile(const GenZ& a, long tile, float2* sm) {
    const int n = a.g.n(), ls = a.g.ls;
    const int kx = (int)(tile / a.ntiles_y);
    const int y0 = (int)(tile - (long)kx * a.ntiles_y) * n;
    const int nq = min(n, a.Y - y0);
    const long base = (long)kx * a.YZ + y0;
    float2* s = a.S + base;
    const float2* tw = a.plan.tw + 3 * a.g.L;
    auto src = [&](int q, int z) { return q < nq ? ld2<CO>(s + (long)z * a.Y + q) : make_float2(0.f, 0.f); };
    if (!MUL) {
        line_transform<-1, float2, false, false, CO>(a.g, a.plan, tw, sm, sm + n * ls, nullptr, src,
                                          [&](float2*, int q, int z, float2 v) {
                                              if (q < nq) s[(long)z * a.Y + q] = cscale(v, a.scale);
                                          });
        return;
    }
    const float2* K = a.K + base;
    for (int z = threadIdx.x; z < a.g.L; z += blockDim.x) prefetch_l2(K + (long)z * a.Y);
    float2* F = line_transform<-1, float2, false, false, CO>(a.g, a.plan, tw, sm, sm + n * ls, nullptr, src,
                                                  [&](float2* buf, int q, int z, float2 v) {
                                                      buf[q * ls + z] =
                                                          q < nq ? cmul(v, __ldg(K + (long)z * a.Y + q)) : v;
                                                  });
    __syncthreads();
    line_transform<+1, float2, false, false, CO>(
        a.g, a.plan, tw, F == sm ? sm + n * ls : sm, F, nullptr, [&](int q, int z) { return F[q * ls + z]; },
        [&](float2*, int q, int z, float2 v) {
            if (q < nq) s[(long)z * a.Y + q] = v;
        });
}

}  // namespace mvd
