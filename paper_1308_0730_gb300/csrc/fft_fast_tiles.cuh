// Tile-level device functions of the register-resident FFT passes
// (power-of-two line lengths), shared by the per-volume kernels
// (fft_fast.cu) and the persistent batch kernel (batch.cu). A tile is what
// one 256-thread block handles. CO = true turns loads of data written inside
// the same launch (spectrum, estimate) into L2 loads, as the batch kernel
// requires.
#pragma once

#include "dd.cuh"
#include "fft_fast.cuh"
#include "lines.cuh"

namespace mvd {

constexpr int kFastThreads = 256;

// tile sizes: x rows per tile, y lines per tile, z columns per tile
__host__ __device__ constexpr int fast_x_rows(int L) { return 2 * (kFastThreads / (L / kE)); }
__host__ __device__ constexpr int fast_y_lines(int L) { return kFastThreads / (L / kE); }
__host__ __device__ constexpr int fast_z_cols(int L) {
    return (kFastThreads / (L / kE)) >= 8 ? kFastThreads / (L / kE) : 8;
}
__host__ __device__ constexpr size_t fast_x_smem(int L) { return (size_t)fast_x_rows(L) * line_stride(L) * sizeof(float2); }
__host__ __device__ constexpr size_t fast_y_smem(int L) { return (size_t)fast_y_lines(L) * line_stride(L) * sizeof(float2); }
__host__ __device__ constexpr size_t fast_z_smem(int L) { return (size_t)fast_z_cols(L) * line_stride(L) * sizeof(float2); }

// y pass: Xh*Z contiguous lines of length Y; lines of one warp are adjacent
template <int L, int S, bool CO>
__device__ __forceinline__ void fast_y_tile(float2* __restrict__ spec, long nlines, const float2* __restrict__ tw,
                                            long tile, float2* sm) {
    using F = LineFFT<L, S, true>;
    constexpr int TPL = F::TPL;
    constexpr int LPC = kFastThreads / TPL;
    const int li = threadIdx.x / TPL, t = threadIdx.x - li * TPL;
    const long line = tile * LPC + li;
    const bool ok = line < nlines;
    float2* g = spec + line * L;
    float2 v[kE];
#pragma unroll
    for (int q = 0; q < kE; ++q) v[q] = ok ? ld2<CO>(g + t + TPL * q) : make_float2(0.f, 0.f);
    F::run(v, sm + li * line_stride(L), t, tw);
    if (ok) {
#pragma unroll
        for (int q = 0; q < kE; ++q) g[t + TPL * q] = v[q];
    }
}

// z pass: Q lines (consecutive y) of one kx plane; thread = q + Q * t so each
// warp reads rows of consecutive y. Needs Q * L/16 threads per block.
template <int L, bool MUL, bool CO>
__device__ __forceinline__ void fast_z_tile(float2* __restrict__ spec, const float2* __restrict__ K, int Y, long YZ,
                                            int ntiles_y, float scale, const float2* __restrict__ tw, long tile,
                                            float2* sm) {
    constexpr int TPL = L / kE;
    constexpr int Q = fast_z_cols(L);
    const int q = threadIdx.x % Q, t = threadIdx.x / Q;
    const int kx = (int)(tile / ntiles_y);
    const int y0 = (int)(tile - (long)kx * ntiles_y) * Q;
    const bool ok = y0 + q < Y;
    const long base = (long)kx * YZ + y0 + q;
    float2* line_sm = sm + q * line_stride(L);
    float2 v[kE];
#pragma unroll
    for (int i = 0; i < kE; ++i) v[i] = ok ? ld2<CO>(spec + base + (long)(t + TPL * i) * Y) : make_float2(0.f, 0.f);
    LineFFT<L, -1, false>::run(v, line_sm, t, tw);
    if (MUL) {
#pragma unroll
        for (int i = 0; i < kE; ++i) {
            const float2 k = ok ? __ldg(K + base + (long)(t + TPL * i) * Y) : make_float2(0.f, 0.f);
            v[i] = cmul(v[i], k);
        }
        __syncthreads();  // the exchange buffer is reused by the inverse transform
        LineFFT<L, +1, false>::run(v, line_sm, t, tw);
    } else {
#pragma unroll
        for (int i = 0; i < kE; ++i) v[i] = cscale(v[i], scale);
    }
    if (ok) {
#pragma unroll
        for (int i = 0; i < kE; ++i) spec[base + (long)(t + TPL * i) * Y] = v[i];
    }
}

// x passes: P pairs of rows per tile (rows rho0+p and rho0+P+p form pair p)
struct XFast {
    const float* src;
    float2* spec;
    const float* phi;
    float* psi;
    long YZ;
    float eps;
    const float2* tw;
    const float* wt;   // when set, the update applies the fraction wt of the change (partial overlap)
    float lam;         // Tikhonov regularisation of the update (0 = none)
    const float* inv_s;  // zero boundary: 1 / sensitivity of the update's view, or none
};

// write the packed forward spectra (natural order in registers) as the two
// half spectra of each pair, coalesced over rows
template <int L>
__device__ __forceinline__ void x_store_halves(const XFast& a, float2 (&v)[kE], float2* sm, int p, int t, long rho0,
                                               int nrows) {
    constexpr int TPL = L / kE, P = kFastThreads / TPL, LS = line_stride(L), XH = L / 2 + 1;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kE; ++q) sm[p * LS + pad16(t + TPL * q)] = v[q];
    __syncthreads();
    constexpr int NTOT = XH * 2 * P, NIT = (NTOT + kFastThreads - 1) / kFastThreads;
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
        const int idx = threadIdx.x + i * kFastThreads;
        const int k = idx / (2 * P), row = idx - k * 2 * P;
        if (idx >= NTOT || row >= nrows) continue;
        const int pp = row < P ? row : row - P;
        const float2 zk = sm[pp * LS + pad16(k)];
        const float2 zm = cconj(sm[pp * LS + pad16(k == 0 ? 0 : L - k)]);
        float2 val;
        if (row < P) {
            val = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y + zm.y));
        } else {
            const float2 d = csub(zk, zm);
            val = make_float2(0.5f * d.y, -0.5f * d.x);
        }
        a.spec[(long)k * a.YZ + rho0 + row] = val;
    }
}

// Read both half spectra of each pair and build Z = A + i B (natural order). They are
// gathered by asynchronous copies, all in flight at once and in no registers; row r
// (r < P: A of pair r, else B of pair r - P) sits at the odd stride XH, so that a warp's
// rows of one k and a line's ascending and descending runs both fall on distinct banks.
template <int L, bool CO>
__device__ __forceinline__ void x_load_packed(const XFast& a, float2 (&v)[kE], float2* sm, int p, int t, long rho0,
                                              int nrows) {
    constexpr int TPL = L / kE, P = kFastThreads / TPL, XH = L / 2 + 1;
    static_assert(2 * P * XH <= P * line_stride(L), "the gathered rows exceed the lines' buffer");
    const float2* spec = a.spec + rho0;
    if constexpr (CO) {  // an 8-byte asynchronous copy would go through L1: all loads before the first store
        constexpr int KS = kFastThreads / (2 * P), N = (XH + KS - 1) / KS;  // k of a thread's elements: KS apart
        static_assert(KS >= 1, "a tile has more rows than threads");
        const int row = threadIdx.x % (2 * P), k0 = threadIdx.x / (2 * P);
        float2 t[N];
#pragma unroll
        for (int j = 0; j < N; ++j)
            t[j] = row < nrows && k0 + j * KS < XH ? ld2<CO>(spec + (long)(k0 + j * KS) * a.YZ + row) : make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (k0 + j * KS < XH) sm[row * XH + k0 + j * KS] = t[j];
    } else {
        for (int idx = threadIdx.x; idx < XH * 2 * P; idx += kFastThreads) {
            const int k = idx / (2 * P), row = idx - k * 2 * P;
            const bool ok = row < nrows;
            cp_async8(sm + row * XH + k, ok ? spec + (long)k * a.YZ + row : a.spec, ok);
        }
        cp_async_wait_all();
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kE; ++q) {
        const int k = t + TPL * q;
        const int kk = k <= L / 2 ? k : L - k;
        const float2 A = sm[p * XH + kk], B = sm[(P + p) * XH + kk];
        v[q] = k <= L / 2 ? make_float2(A.x - B.y, A.y + B.x)
                          : make_float2(A.x + B.y, B.x - A.y);  // conj(A) + i conj(B)
    }
    __syncthreads();
}

template <int L, bool CO>
__device__ __forceinline__ void fast_x_forward_tile(const XFast& a, long tile, float2* sm) {
    constexpr int TPL = L / kE, P = kFastThreads / TPL, LS = line_stride(L);
    const int p = threadIdx.x / TPL, t = threadIdx.x - p * TPL;
    const long rho0 = tile * 2 * P;
    const int nrows = (int)min((long)2 * P, a.YZ - rho0);
    const bool oka = p < nrows, okb = P + p < nrows;
    const float* ra = a.src + (rho0 + p) * L;
    const float* rb = a.src + (rho0 + P + p) * L;
    float2 v[kE];
#pragma unroll
    for (int q = 0; q < kE; ++q) {
        const int n = t + TPL * q;
        v[q] = make_float2(oka ? ld1<CO>(ra + n) : 0.f, okb ? ld1<CO>(rb + n) : 0.f);
    }
    LineFFT<L, -1, true>::run(v, sm + p * LS, t, a.tw);
    x_store_halves<L>(a, v, sm, p, t, rho0, nrows);
}

// MODE 0: ratio -> forward ; 1: psi update ; 2: plain real output ;
// 4: acc *= c (the combined update's product of view factors; acc in a.psi)
template <int L, int MODE, bool CO>
__device__ __forceinline__ void fast_x_inverse_tile(const XFast& a, long tile, float2* sm) {
    constexpr int TPL = L / kE, P = kFastThreads / TPL, LS = line_stride(L);
    const int p = threadIdx.x / TPL, t = threadIdx.x - p * TPL;
    const long rho0 = tile * 2 * P;
    const int nrows = (int)min((long)2 * P, a.YZ - rho0);
    const bool oka = p < nrows, okb = P + p < nrows;
    // the epilogue's operand rows (phi for the ratio, psi for the update) come into L2
    // meanwhile: loaded here they would hold 32 registers through the transform. The persistent
    // batch kernel (CO: two blocks, 128 registers) has those, and hides less: four volumes of
    // 128^3 in FP32 1.48 ms with prefetches and one gathered value at a time, 1.27 so.
    if (!CO && MODE == 0) prefetch_rows(a.phi + rho0 * L, nrows * L * 4);
    if (!CO && (MODE == 1 || MODE == 4)) prefetch_rows(a.psi + rho0 * L, nrows * L * 4);
    float2 v[kE];
    x_load_packed<L, CO>(a, v, sm, p, t, rho0, nrows);
    const long ra = (rho0 + p) * L, rb = (rho0 + P + p) * L;
    float2 w[kE];
    auto operands = [&] {
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            const int n = t + TPL * q;
            if (MODE == 0)
                w[q] = make_float2(oka ? __ldg(a.phi + ra + n) : 0.f, okb ? __ldg(a.phi + rb + n) : 0.f);
            else
                w[q] = make_float2(oka ? ld1<CO>(a.psi + ra + n) : 0.f, okb ? ld1<CO>(a.psi + rb + n) : 0.f);
        }
    };
    if (CO && MODE != 2) operands();
    LineFFT<L, +1, true>::run(v, sm + p * LS, t, a.tw);
    if (MODE == 0) {
        if (!CO) operands();  // all loads before the first division (whose slow path is a branch)
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            // r - 1 (see the generic ratio pass): the update adds the 1 back
            const float xa = oka ? w[q].x / fmaxf(v[q].x, a.eps) - 1.f : 0.f;
            const float xb = okb ? w[q].y / fmaxf(v[q].y, a.eps) - 1.f : 0.f;
            v[q] = make_float2(xa, xb);
        }
        LineFFT<L, -1, true>::run(v, sm + p * LS, t, a.tw);
        x_store_halves<L>(a, v, sm, p, t, rho0, nrows);
    } else {
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            const int n = t + TPL * q;
            if (MODE == 1) {
                // v = c - 1 (weights and regularisation: update_factor)
                const float pa = CO ? w[q].x : oka ? ld1<CO>(a.psi + ra + n) : 0.f;
                const float pb = CO ? w[q].y : okb ? ld1<CO>(a.psi + rb + n) : 0.f;
                if (oka) a.psi[ra + n] = fmaxf(pa * update_factor(v[q].x, pa, a.wt, ra + n, a.lam, a.inv_s), a.eps);
                if (okb) a.psi[rb + n] = fmaxf(pb * update_factor(v[q].y, pb, a.wt, rb + n, a.lam, a.inv_s), a.eps);
            } else if (MODE == 4) {  // combined update: multiply this view's factor into the product
                if (oka)
                    a.psi[ra + n] = ld1<CO>(a.psi + ra + n) * (v[q].x + 1.f) * (a.inv_s ? __ldg(a.inv_s + ra + n) : 1.f);
                if (okb)
                    a.psi[rb + n] = ld1<CO>(a.psi + rb + n) * (v[q].y + 1.f) * (a.inv_s ? __ldg(a.inv_s + rb + n) : 1.f);
            } else {
                if (oka) a.psi[ra + n] = v[q].x;
                if (okb) a.psi[rb + n] = v[q].y;
            }
        }
    }
}

}  // namespace mvd
