// Double-float passes of any {2,3,5}-smooth length (tile-level device functions;
// transforms and tile geometry: lines.cuh). Same layout as the FP32 passes:
// spectrum S2[kx][z][y] of complex double-float (16 bytes, adp.cuh), two real
// x-lines per complex line. The forward blur b = psi * P_v runs entirely in
// double-float; the ratio pass rounds b to FP32, forms r - 1 = phi / max(b, eps) - 1,
// transforms it along x in FP32 and hands that spectrum over in FP32 (or widened
// exactly into S2); the back-projection's other passes, the update's x inverse
// included, run in double-float.
//
// CO = true makes loads of data written inside the same launch L2 loads (the
// persistent batch kernel).
#pragma once

#include "adp.cuh"
#include "dd.cuh"
#include "fft_generic.cuh"
#include "lines.cuh"

namespace mvd {

// spectra are read once per pass: past L1, which keeps the twiddles
template <bool CO>
__device__ __forceinline__ cdp ld_cdp(const cdd* p) {
    return cdp_load_cg(p);
}

// geometry: as gen_x_geo, gen_line_geo with 16-byte elements; the ratio's FP32 lines
// (stride line_stride_for(X, n, 16)) go two to one double-float line
__host__ __device__ inline LineGeo dd_x_geo(const FftPlan& p, TileRule rule = dd_tile_rule()) {
    LineGeo g{};
    g.L = p.L;
    g.ln = tile_lines_log2(p, rule, 32);
    int least = 2 * x_half_stride(p.L);
    const int f = line_stride_for(p.L, g.n(), 16);
    least = least > f ? least : f;
    g.ls = line_stride_for(least > p.L ? least : p.L, g.n(), 8);
    g.T = tile_threads(p, g.ln);
    return g;
}
__host__ __device__ inline LineGeo dd_line_geo(const FftPlan& p, int most, TileRule rule = dd_tile_rule()) {
    LineGeo g{};
    g.L = p.L;
    g.ln = tile_lines_log2(p, rule, most);
    g.ls = line_stride_for(p.L, g.n(), 8);
    g.T = tile_threads(p, g.ln);
    return g;
}
__host__ __device__ inline size_t dd_smem(const LineGeo& g) { return (size_t)2 * g.n() * g.ls * sizeof(cdd); }

struct DdX {
    LineGeo g;
    int X, Xh;
    long YZ;
    FftPlan plan;           // radices of X
    const cdd* tw2;         // double-float twiddles of X
    const float* src;       // real rows
    cdd* S2;                // double-float spectrum
    const float* phi;       // observed view
    float eps;
    float2* S;              // ratio: the FP32 spectrum of r - 1 goes here when set, else into S2
};

__host__ __device__ inline DdX dd_x_args(int X, long YZ, const FftPlan& plan, const cdd* tw2,
                                         TileRule rule = dd_tile_rule()) {
    DdX a{};
    a.g = dd_x_geo(plan, rule);
    a.X = X;
    a.Xh = X / 2 + 1;
    a.YZ = YZ;
    a.plan = plan;
    a.tw2 = tw2;
    return a;
}
__host__ __device__ inline long dd_x_tiles(const FftPlan& p, long YZ, TileRule rule = dd_tile_rule()) {
    return gen_div_up(YZ, 2 * dd_x_geo(p, rule).n());
}

// pair p = rows (p, n + p): complex line a + i b, exact in double-float
template <bool CO>
__device__ void dd_x_forward_tile(const DdX& a, long tile, cdd* sm) {
    __shared__ unsigned w[8];
    const int n = a.g.n(), ls = a.g.ls;
    const long rho0 = tile * 2 * n;
    const int nrows = (int)min((long)2 * n, a.YZ - rho0);
    const float* src = a.src + rho0 * a.X;
    const cdd* F = line_transform<-1, cdp, true, false, CO>(
        a.g, a.plan, a.tw2 + 2 * a.X, sm, sm + n * ls, w,
        [&](int p, int i) {
            return cdp_from(p < nrows ? ld1<CO>(src + p * a.X + i) : 0.f,
                            n + p < nrows ? ld1<CO>(src + (n + p) * a.X + i) : 0.f);
        },
        [&](cdd* buf, int p, int i, cdp v) { cdp_store(buf + p * ls + i, v); });
    __syncthreads();
    cdd* S2 = a.S2 + rho0;
    unpack_tile<cdp>(F, ls, a.X, a.g.ln, nrows, [&](int k, int row, cdp v) { cdp_store(S2 + (long)k * a.YZ + row, v); });
}

// inverse x of the tile's rows: the half spectra staged by asynchronous copies (all in
// flight at once), then last(buf, p, element, value)
template <bool CO, typename Last>
__device__ __forceinline__ cdd* dd_x_inverse_lines(const DdX& a, long rho0, int nrows, cdd* sm, unsigned* w,
                                                   Last&& last) {
    const int n = a.g.n(), hs = x_half_stride(a.X), lr = a.g.ln + 1;
    cdd* H = sm + n * a.g.ls;
    const cdd* S2 = a.S2 + rho0;
    for (int t = threadIdx.x; t < (a.Xh << lr); t += blockDim.x) {
        const int row = t & ((1 << lr) - 1), k = t >> lr;
        const bool ok = row < nrows;
        cp_async16(H + row * hs + k, ok ? S2 + (long)k * a.YZ + row : a.S2, ok);
    }
    cp_async_wait_all();
    __syncthreads();
    return line_transform<+1, cdp, false, true, CO>(
        a.g, a.plan, a.tw2 + 2 * a.X, sm, H, w,
        [&](int p, int k) {
            const bool up = k <= a.X / 2;
            const int kk = up ? k : a.X - k;
            return pack_pair(cdp_load(H + p * hs + kk), cdp_load(H + (n + p) * hs + kk), up);
        },
        last);
}

// The back-projection's last pass in double-float: inverse x of S2, the
// result (c - 1) rounded to FP32 once, then MODE 1: psi = max(psi .
// update_factor, eps); MODE 4: acc = acc . c . inv_s (the combined update's
// product); MODE 0: psi = the rounded result (plain real output).
struct DdXU {
    DdX x;
    float* psi;
    const float* wt;
    float lam;
    const float* inv_s;
};

template <bool CO, int MODE>
__device__ void dd_x_update_tile(const DdXU& u, long tile, cdd* sm) {
    __shared__ unsigned w[8];
    const DdX& a = u.x;
    const int n = a.g.n();
    const long rho0 = tile * 2 * n;
    const int nrows = (int)min((long)2 * n, a.YZ - rho0);
    const long base = rho0 * a.X;
    if (MODE != 0) prefetch_rows(u.psi + base, nrows * a.X * 4);
    dd_x_inverse_lines<CO>(a, rho0, nrows, sm, w, [&](cdd*, int p, int i, cdp v) {
        const float2 z = cdp_round(v);
        const float cv[2] = {z.x, z.y};  // c - 1 of rows p and n + p
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = p + h * n;
            if (row >= nrows) continue;
            const long at = base + (row * a.X + i);
            if (MODE == 0) {
                u.psi[at] = cv[h];
                continue;
            }
            const float ps = ld1<CO>(u.psi + at);
            if (MODE == 1)
                u.psi[at] = fmaxf(ps * update_factor(cv[h], ps, u.wt, at, u.lam, u.inv_s), a.eps);
            else
                u.psi[at] = ps * (cv[h] + 1.f) * (u.inv_s ? __ldg(u.inv_s + at) : 1.f);
        }
    });
}

// double-float spectrum -> inverse x -> b (rounded to FP32) -> r - 1 with
// r = phi / max(b, eps) -> FP32 forward x -> the FP32 spectrum S (or S2)
template <bool CO>
__device__ void dd_x_ratio_tile(const DdX& a, long tile, cdd* sm) {
    __shared__ unsigned w[8];
    const int n = a.g.n();
    const long rho0 = tile * 2 * n;
    const int nrows = (int)min((long)2 * n, a.YZ - rho0);
    const float* phi = a.phi + rho0 * a.X;
    prefetch_rows(phi, nrows * a.X * 4);
    LineGeo gf = a.g;
    gf.ls = line_stride_for(a.X, n, 16);
    // the last stage leaves r - 1 in FP32 lines in the buffer it does not read
    cdd* Rd = dd_x_inverse_lines<CO>(a, rho0, nrows, sm, w, [&](cdd* buf, int p, int i, cdp v) {
        const float2 z = cdp_round(v);
        const float ba = fmaxf(z.x, a.eps), bb = fmaxf(z.y, a.eps);
        const float ra = p < nrows ? __ldg(phi + p * a.X + i) / ba - 1.f : 0.f;
        const float rb = n + p < nrows ? __ldg(phi + (n + p) * a.X + i) / bb - 1.f : 0.f;
        reinterpret_cast<float2*>(buf)[p * gf.ls + i] = make_float2(ra, rb);
    });
    __syncthreads();
    const float2* R = reinterpret_cast<const float2*>(Rd);
    float2* A = reinterpret_cast<float2*>(Rd == sm ? sm + n * a.g.ls : sm);  // two FP32 buffers in the other one
    const float2* F = line_transform<-1, float2, false, false, CO>(
        gf, a.plan, a.plan.tw + 3 * a.X, A, A + n * gf.ls, nullptr, [&](int p, int i) { return R[p * gf.ls + i]; },
        [&](float2* buf, int p, int i, float2 v) { buf[p * gf.ls + i] = v; });
    __syncthreads();
    if (a.S) {
        float2* S = a.S + rho0;
        unpack_tile<float2>(F, gf.ls, a.X, a.g.ln, nrows, [&](int k, int row, float2 v) { S[(long)k * a.YZ + row] = v; });
    } else {
        cdd* S2 = a.S2 + rho0;
        unpack_tile<float2>(F, gf.ls, a.X, a.g.ln, nrows,
                            [&](int k, int row, float2 v) { cdp_store(S2 + (long)k * a.YZ + row, cdp_from(v.x, v.y)); });
    }
}

struct DdY {
    LineGeo g;
    long nlines;
    FftPlan plan;
    const cdd* tw2;
    cdd* S2;
    const float2* S1;  // when set, the lines come from this FP32 spectrum (widened exactly)
};

__host__ __device__ inline DdY dd_y_args(int Xh, int Z, const FftPlan& plan, const cdd* tw2, cdd* S2,
                                         TileRule rule = dd_tile_rule()) {
    DdY a{};
    a.g = dd_line_geo(plan, 32, rule);
    a.nlines = (long)Xh * Z;
    a.plan = plan;
    a.tw2 = tw2;
    a.S2 = S2;
    return a;
}
__host__ __device__ inline long dd_y_tiles(const FftPlan& p, int Xh, int Z, TileRule rule = dd_tile_rule()) {
    return gen_div_up((long)Xh * Z, dd_line_geo(p, 32, rule).n());
}

template <bool CO, int S, bool F32 = false>
__device__ void dd_y_tile(const DdY& a, long tile, cdd* sm) {
    __shared__ unsigned w[8];
    const int n = a.g.n(), L = a.g.L;
    const long l0 = tile * n;
    const int nl = (int)min((long)n, a.nlines - l0);
    cdd* s = a.S2 + l0 * L;
    const float2* s1 = a.S1 + l0 * L;
    line_transform<S, cdp, true, true, CO>(
        a.g, a.plan, a.tw2 + 2 * L, sm, sm + n * a.g.ls, w,
        [&](int l, int i) {
            if (l >= nl) return cdp_zero();
            if constexpr (F32) {
                const float2 f = ld2<CO>(s1 + l * L + i);
                return cdp_from(f.x, f.y);
            } else {
                return ld_cdp<CO>(s + l * L + i);
            }
        },
        [&](cdd*, int l, int i, cdp v) {
            if (l < nl) cdp_store(s + l * L + i, v);
        });
}

struct DdZ {
    LineGeo g;
    int Y, ntiles_y;
    long YZ;
    FftPlan plan;
    const cdd* tw2;
    cdd* S2;
    const cdd* K2;  // double-float kernel spectrum (MUL)
    dd scale;       // forward-only scale
};

__host__ __device__ inline DdZ dd_z_args(int Y, long YZ, const FftPlan& plan, const cdd* tw2, cdd* S2, const cdd* K2,
                                         dd scale, TileRule rule = dd_tile_rule()) {
    DdZ a{};
    a.g = dd_line_geo(plan, Y, rule);
    a.Y = Y;
    a.ntiles_y = (int)gen_div_up(Y, a.g.n());
    a.YZ = YZ;
    a.plan = plan;
    a.tw2 = tw2;
    a.S2 = S2;
    a.K2 = K2;
    a.scale = scale;
    return a;
}
__host__ __device__ inline long dd_z_tiles(const FftPlan& p, int Y, int Xh, TileRule rule = dd_tile_rule()) {
    return (long)Xh * gen_div_up(Y, dd_line_geo(p, Y, rule).n());
}

// columns: element z of column q at base + z*Y + q, n consecutive q per tile
template <bool CO, bool MUL>
__device__ void dd_z_tile(const DdZ& a, long tile, cdd* sm) {
    __shared__ unsigned w[8];
    const int n = a.g.n(), ls = a.g.ls;
    const int kx = (int)(tile / a.ntiles_y);
    const int y0 = (int)(tile - (long)kx * a.ntiles_y) * n;
    const int nq = min(n, a.Y - y0);
    const long base = (long)kx * a.YZ + y0;
    cdd* s = a.S2 + base;
    const cdd* tw = a.tw2 + 2 * a.g.L;
    auto src = [&](int q, int z) { return q < nq ? ld_cdp<CO>(s + (long)z * a.Y + q) : cdp_zero(); };
    if (!MUL) {
        line_transform<-1, cdp, false, false, CO>(a.g, a.plan, tw, sm, sm + n * ls, w, src, [&](cdd*, int q, int z, cdp v) {
            if (q < nq) cdp_store(s + (long)z * a.Y + q, cdp_scale(v, a.scale));
        });
        return;
    }
    // the last forward stage multiplies by the kernel spectrum
    const cdd* K = a.K2 + base;
    for (int z = threadIdx.x; z < a.g.L; z += blockDim.x) prefetch_l2(K + (long)z * a.Y);
    cdd* F = line_transform<-1, cdp, false, false, CO>(a.g, a.plan, tw, sm, sm + n * ls, w, src,
                                           [&](cdd* buf, int q, int z, cdp v) {
                                               if (q < nq) v = cdp_mul_pair(v, cdp_load_cg(K + (long)z * a.Y + q));
                                               cdp_store(buf + q * ls + z, v);
                                           });
    __syncthreads();
    line_transform<+1, cdp, false, false, CO>(
        a.g, a.plan, tw, F == sm ? sm + n * ls : sm, F, w,
        [&](int q, int z) { return cdp_load(F + q * ls + z); },
        [&](cdd*, int q, int z, cdp v) {
            if (q < nq) cdp_store(s + (long)z * a.Y + q, v);
        });
}

}  // namespace mvd
