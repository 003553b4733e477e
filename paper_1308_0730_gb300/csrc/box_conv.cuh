// Tiled 3D convolution sums on the FP32 pipe, shared by the direct engine
// (periodic volumes) and the compound-kernel algebra (small kernels, zero
// outside their boxes):
//   out(o) = sum_t tap(t) in(o + t + off),   o on the output box, t on the tap box.
//
// What bounds it: the FMAs (taps x outputs, 128 per SM and clock) and the
// shared-memory returns (128 bytes per clock: a float4 per lane takes four clocks,
// also where all lanes read the same one). Hence the register tile:
//   - a thread holds 8 consecutive x by NY consecutive y outputs; per input row and
//     4 taps it loads one new float4 of the row and one of taps per output row, for
//     32 NY FMAs: 4 (1 + NY) clocks of returns against 8 NY of FMAs. (4 x outputs
//     would need 4 (1 + NY) against 4 NY; 32 rows per warp were slower than 16 or 8
//     at every size tried: too few warps.)
//   - four lanes of a warp lie along x, eight along y; the row stride is an odd
//     number of float4, so the eight lanes of a quarter-warp (two rows, every second
//     float4) fall on distinct banks. A block's warps (8, or 16) cover nz planes
//     times S splits of the tap planes (tap plane kz belongs to split kz mod S):
//     small volumes get S = 8, so that 32^3 outputs still fill the SMs, large ones 1;
//   - input planes and taps are staged CK tap planes at a time by 4-byte
//     asynchronous copies (all in flight at once), two or more blocks per SM
//     overlapping one's copies with another's sums.
// Measured against one output row per thread with scalar loads (GB300, one launch,
// us): 32^3 outputs, 13x7x7 box 52.9 -> 8.3; 97x83x61, 9x9x15 222 -> 44;
// 120x110x100, 15x15x41 about 0.46 of the FMA peak (660 us).
// The order of each output's sum in the direct engine depends on S only (and, where not one
// row of taps fits, on the pieces): not on NY, CK, the warps or the rows staged at a time,
// whose chains run on from one staging to the next. The compensated sums of the kernel
// algebra add what each staging gives.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "fft.cuh"

namespace mvd {

constexpr int kBcTX = 32;
constexpr int kBcPiece = 512;  // taps of a row staged at a time where not one whole row fits
constexpr size_t kBcMaxSmem = 226 * 1024;  // kMaxDynSmem

// one convolution: input box, tap box, output box; `off` is the input index of
// (output 0, tap 0) per axis; mir reads the taps reversed on every axis
struct BoxConv {
    const float* in;
    const float* taps;
    int ix, iy, iz;
    int kx, ky, kz;
    int ox, oy, oz;
    int offx, offy, offz;
    int mir;
    int ck, cy, cx;  // tap planes, tap rows of each and taps of a row staged at a time
};

__host__ __device__ inline int bc_wx(int kx) { return ((kBcTX + kx - 1 + 3) & ~3) | 4; }  // an odd number of float4
__host__ __device__ inline int bc_kxp(int kx) { return (kx + 3) & ~3; }
inline size_t bc_smem(int kx, int ky, int ck, int ny, int nz, int warps) {
    const size_t tile = (size_t)bc_wx(kx) * (8 * ny + ky - 1) * (nz + ck - 1);
    const size_t taps = (size_t)bc_kxp(kx) * ky * ck;
    const size_t red = (size_t)warps * 256 * ny;  // the partial sums of the splits reuse the staging
    return sizeof(float) * (tile + taps > red ? tile + taps : red);
}

struct BcPlan {
    int ny, s, ck, cy, cx, warps;
    size_t smem;
    double cost;  // SM clocks of the whole grid, for comparing plans
    int planes() const { return warps / s; }
};

// Splits of the tap planes: enough warps for 8 per SM at eight rows per warp.
inline int bc_splits(long warps, int kz) {
    int s = 1;
    while (s < 8 && warps * s < 152L * 8 && s < kz) s *= 2;
    return s;
}

// Staged tap planes and estimated cost of blocks of `warps` warps over tiles of 8 ny
// rows; false where not even one tap row of one plane fits. Three blocks of eight
// warps per SM where the staging allows it, else two; boxes of which no whole plane
// fits are staged a few rows at a time, and (pieces) a piece of a row at a time.
inline bool bc_plan_ny(int ox, int oy, int oz, int kx_all, int ky, int kz, int ny, int s, int warps, BcPlan* p,
                       bool pieces = false) {
    const int nz = warps / s;
    if (nz < 1) return false;
    const int kx = pieces && kx_all > kBcPiece ? kBcPiece : kx_all, np = (kx_all + kx - 1) / kx;
    const size_t want[3] = {74 * 1024, 110 * 1024, kBcMaxSmem};
    int ck = 0;
    for (int i = 0; i < 3 && ck == 0; ++i) {
        int c = 0;
        while (c < kz && bc_smem(kx, ky, c + 1, ny, nz, warps) <= want[i]) ++c;
        const int least = i < 2 ? (kz < 8 ? kz : 8) : 1;  // few planes per stage would mean mostly halo loads
        if (c < kz && c >= s) c = c / s * s;
        if (c >= least) ck = c;
    }
    int cy = ky;
    if (ck == 0)
        for (ck = 1; cy > 0 && bc_smem(kx, cy, 1, ny, nz, warps) > kBcMaxSmem;) cy -= cy > 64 ? 16 : 1;
    if (cy <= 0 || (oy + 8 * ny - 1) / (8 * ny) > 65535) return false;
    *p = BcPlan{ny, s, ck, cy, kx, warps, bc_smem(kx, cy, ck, ny, nz, warps), 0.0};
    const long blocks = (long)((ox + 31) / 32) * ((oy + 8 * ny - 1) / (8 * ny)) * ((oz + nz - 1) / nz);
    const int most = 24 / warps;
    int res = (int)((227 * 1024) / (p->smem + 1024));
    res = res > most ? most : res;
    const double nf = kx / 4 + 1, planes = (double)np * ((kz + s - 1) / s);
    const double chunks = (double)np * ((kz + ck - 1) / ck) * ((ky + cy - 1) / cy);
    // issue slots of a warp: the FMAs and loads of its (row, output) pairs, about 20 more
    // per row; the copies of its share of the tile's rows and of the taps
    const double sums = planes * (ny * ky * (8.0 * kx + nf) + (ky + ny - 1) * (20.0 + nf));
    const double copies = chunks * ((8.0 * ny + cy - 1) * (nz + ck - 1) / warps * (25.0 + 4.0 * (bc_wx(kx) / 32 + 1)) +
                                    bc_kxp(kx) * (double)cy * ck / (32.0 * warps) * 30.0);
    const double lds = 4.0 * warps * planes * nf * ((ky + ny - 1) + ny * ky);  // shared-memory clocks of a block
    const double busy = (ny == 2 ? 1.3 : 1.15) * (warps * (sums + copies) / 4 > lds ? warps * (sums + copies) / 4 : lds);
    auto round = [&](double n) {  // n blocks on one SM: its issue slots, or the latency of one warp's chain
        const double lat = 2.5 * (sums + copies);
        return (n * busy > lat ? n * busy : lat) + 2500.0 * chunks;
    };
    const long slots = 152L * res, full = blocks / slots, rem = blocks - full * slots;
    p->cost = full * round(res) + (rem ? round((double)((rem + 151) / 152)) : 0.0);
    return true;
}

// The cheapest of 16- and 8-row tiles (ny_max limits it) for blocks of eight warps,
// and of 8-row tiles for sixteen, which read the halo of a small volume's few planes
// half as often; a box so tall that no tile of nz planes fits takes more splits, and one so
// wide that no row of taps fits (from about 6400) is staged in pieces of rows.
inline bool bc_plan(int ox, int oy, int oz, int kx, int ky, int kz, int ny_max, BcPlan* best) {
    bool any = false;
    for (int s = bc_splits((long)((ox + 31) / 32) * ((oy + 7) / 8) * oz, kz); s <= 8 && !any; s *= 2)
        for (int ny = ny_max; ny >= 1; ny /= 2)
            for (int warps = 8; warps <= (ny == 1 ? 16 : 8); warps *= 2) {
                BcPlan p{};
                if (bc_plan_ny(ox, oy, oz, kx, ky, kz, ny, s, warps, &p) && (!any || p.cost < best->cost))
                    *best = p, any = true;
            }
    if (any) return true;
    const int s = bc_splits((long)((ox + 31) / 32) * ((oy + 7) / 8) * oz, kz);
    if (!bc_plan_ny(ox, oy, oz, kx, ky, kz, 1, s, 8, best, true)) return false;
    best->ck = 1;  // a chain runs on over the stagings of one plane
    return true;
}

// A batch of convolutions of small kernels (zero outside their boxes), one
// launch for up to kBcMaxJobs of them: every output box gets its own tiles.
constexpr int kBcMaxJobs = 16;
struct BoxJob {
    BoxConv c;
    float* out;
    int add;     // out += sum, else out = sum
    int mirror;  // outputs written reversed on every axis
};

__device__ __forceinline__ void cp_async4(float* dst_smem, const float* src, bool valid) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst_smem));
    const int n = valid ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// taps t[0..N-1] against the input window w[0..10] of the outputs x..x+7
template <int N>
__device__ __forceinline__ void bc_taps(float (&acc)[8], const float4& t, const float4& a0, const float4& a1,
                                        const float4& b) {
    const float w[12] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w, b.x, b.y, b.z, b.w};
    const float tt[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = fmaf(tt[j], w[i + j], acc[i]);
}

// One input row against the tap rows of outputs 0..NY-1 (tp: output 0's tap row;
// output o's is o rows earlier). KX > 0: the taps of a row are known at compile
// time, everything unrolls; KX == 0: nf groups of four and rem more (box sizes are
// odd: one or three); KX < 0: nf and rem of a piece of a row, rem may be zero.
template <int NY, int KX>
__device__ __forceinline__ void bc_row(const float* in, const float* tp, int kxp, int nf, int rem, float (&acc)[NY][8]) {
    auto ld = [](const float* p) { return *reinterpret_cast<const float4*>(p); };
    float4 a0 = ld(in), a1 = ld(in + 4), b = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (KX > 0) {
        constexpr int KP = (KX + 3) & ~3;
#pragma unroll
        for (int c = 0; c < KX / 4; ++c) {
            b = ld(in + 4 * c + 8);
#pragma unroll
            for (int o = 0; o < NY; ++o) bc_taps<4>(acc[o], ld(tp - o * KP + 4 * c), a0, a1, b);
            a0 = a1;
            a1 = b;
        }
        if (KX % 4 == 3) b = ld(in + (KX & ~3) + 8);
#pragma unroll
        for (int o = 0; o < NY; ++o) bc_taps<KX % 4>(acc[o], ld(tp - o * KP + (KX & ~3)), a0, a1, b);
    } else {
#pragma unroll 3  // the window turns over three float4: no register moves
        for (int c = 0; c < nf; ++c) {
            b = ld(in + 4 * c + 8);
#pragma unroll
            for (int o = 0; o < NY; ++o) bc_taps<4>(acc[o], ld(tp - o * kxp + 4 * c), a0, a1, b);
            a0 = a1;
            a1 = b;
        }
        if (rem == 3) {
            b = ld(in + 4 * nf + 8);
#pragma unroll
            for (int o = 0; o < NY; ++o) bc_taps<3>(acc[o], ld(tp - o * kxp + 4 * nf), a0, a1, b);
        } else if (KX == 0 || rem == 1) {
#pragma unroll
            for (int o = 0; o < NY; ++o) bc_taps<1>(acc[o], ld(tp - o * kxp + 4 * nf), a0, a1, b);
        }
    }
}

// the outputs lo..hi of the window that input row iy reaches
template <int NY, int KX>
__device__ __forceinline__ void bc_rows(int lo, int hi, const float* in, const float* tp, int kxp, int nf, int rem,
                                        float (&acc)[NY][8]) {
    if constexpr (NY == 1) {
        bc_row<1, KX>(in, tp, kxp, nf, rem, acc);
    } else {
        if (lo == 0 && hi == NY - 1) return bc_row<NY, KX>(in, tp, kxp, nf, rem, acc);
        // an edge row: one output at a time
#pragma unroll
        for (int o = 0; o < NY; ++o)
            if (o >= lo && o <= hi) {
                float one[1][8];
#pragma unroll
                for (int i = 0; i < 8; ++i) one[0][i] = acc[o][i];
                bc_row<1, KX>(in, tp - o * kxp, kxp, nf, rem, one);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[o][i] = one[0][i];
            }
    }
}

// The tile (bx, by, bz) of convolution j; epi(x, y, z, sum) receives every output
// of the tile that lies inside the output box, once. WRAP: the input box is
// periodic; else zero outside. COMP: every row's sum is formed on its own, the
// rows of a plane are added, and the planes' sums are added with compensation
// (Kahan), so the error does not grow with the box; otherwise a plane's taps are
// one chain and the planes' sums are added plainly (boxes of the direct engine), also
// where its rows are staged cy at a time. KX < 0: planes are staged in rows, and rows in pieces
// of j.cx (a multiple of four, or the whole row); kernels without COMP and of other KX take
// whole planes only (the chains would hold registers through the staging).
template <int NY, int KX, bool WRAP, bool COMP, typename Epi>
__device__ __forceinline__ void bc_tile(const BoxConv& j, int bx, int by, int bz, int S, float* smem, Epi&& epi) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lx = lane & 3, ly = lane >> 2;
    const int nw = blockDim.x >> 5, nz = nw / S, s = warp & (S - 1), zl = warp / S;
    const int x0 = bx * kBcTX, y0 = by * 8 * NY, z0 = bz * nz;
    constexpr bool PIECES = KX < 0, CHAIN = PIECES && !COMP;
    const int px = PIECES ? j.cx : j.kx;
    const int wx = bc_wx(px), kxp = bc_kxp(px);
    int nf = px >> 2, rem = px & 3;
    float* tile = smem;
    float* taps = smem + (size_t)wx * (8 * NY + j.cy - 1) * (nz + j.ck - 1);
    const float inv_kxp = 1.0f / (float)kxp;
    // tap planes whose input planes touch the box for some output of the block
    int klo = 0, khi = j.kz;
    if (!WRAP) {
        klo = max(0, -(z0 + j.offz) - (nz - 1));
        khi = min(j.kz, j.iz - (z0 + j.offz));
    }
    int p0 = 0;                            // first tap of the piece
    auto column = [&](int i, bool& okx) {  // input column of tile column i
        int gx = x0 + j.offx + (PIECES ? p0 : 0) + i;
        okx = gx >= 0 && gx < j.ix;
        if (WRAP) return gx < 0 ? gx + j.ix : (gx >= j.ix ? min(gx - j.ix, j.ix - 1) : gx);
        return okx ? gx : 0;
    };
    bool oka, okb;
    int gxa = column(lane, oka), gxb = column(lane + 32, okb);
    float acc[NY][8], tot[NY][8], cmp[NY][8];
#pragma unroll
    for (int o = 0; o < NY; ++o)
#pragma unroll
        for (int i = 0; i < 8; ++i) tot[o][i] = 0.f, cmp[o][i] = 0.f;
    for (int k0 = klo; k0 < khi; k0 += j.ck)
        for (int q0 = 0; q0 < j.ky; q0 += j.cy)
            for (p0 = 0; p0 < (PIECES ? j.kx : 1); p0 += PIECES ? j.cx : 1) {
                const int ck = min(j.ck, khi - k0), cy = min(j.cy, j.ky - q0);
                const int nx = PIECES ? min(j.cx, j.kx - p0) : j.kx;  // taps of the piece's rows
                if constexpr (PIECES) {
                    gxa = column(lane, oka), gxb = column(lane + 32, okb);
                    nf = nx >> 2, rem = nx & 3;
                }
                const int wy = 8 * NY + cy - 1, rows = (nz + ck - 1) * wy;
                const int iy0 = y0 + j.offy + q0;  // input row of the tile's first
                const float inv_cy = 1.0f / (float)cy;
                // each warp copies every nw-th row; a lane's columns (and their wrap) are the same in every row
                int p = warp / wy, iy = warp - p * wy;
                for (int r = warp; r < rows; r += nw) {
                    int gz = z0 + j.offz + k0 + p, gy = iy0 + iy;
                    bool ok = true;
                    if (WRAP) {  // one turn covers every input of a valid output; the rest only needs a valid address
                        gz = gz < 0 ? gz + j.iz : (gz >= j.iz ? min(gz - j.iz, j.iz - 1) : gz);
                        gy = gy < 0 ? gy + j.iy : (gy >= j.iy ? min(gy - j.iy, j.iy - 1) : gy);
                    } else {
                        ok = gz >= 0 && gz < j.iz && gy >= 0 && gy < j.iy;
                    }
                    const float* row = j.in + (ok ? (long)j.ix * (gy + (long)j.iy * gz) : 0L);
                    float* dst = tile + (size_t)r * wx + lane;
                    cp_async4(dst, row + gxa, WRAP || (ok && oka));
                    if (lane + 32 < wx) cp_async4(dst + 32, row + gxb, WRAP || (ok && okb));
                    for (int i = lane + 64; i < wx; i += 32) {
                        bool okx;
                        const int gx = column(i, okx);
                        cp_async4(dst + i - lane, row + gx, WRAP || (ok && okx));
                    }
                    for (iy += nw; iy >= wy; iy -= wy) ++p;
                }
                const int nt = ck * cy * kxp;
                for (int i = threadIdx.x; i < nt; i += blockDim.x) {
                    const int r = small_div(i, inv_kxp), kx = i - r * kxp;
                    const int kz = small_div(r, inv_cy), ky = r - kz * cy;
                    const bool ok = kx < nx;
                    long t = (PIECES ? p0 : 0) + kx + (long)j.kx * (q0 + ky + (long)j.ky * (k0 + kz));
                    if (j.mir) t = (long)j.kx * j.ky * j.kz - 1 - t;
                    cp_async4(taps + i, ok ? j.taps + t : j.taps, ok);
                }
                asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
                __syncthreads();
                int ilo = 0, ihi = cy + NY - 1;  // rows of a thread's window that hold input for some lane
                if (!WRAP) {
                    ilo = max(0, -iy0 - 7 * NY);
                    ihi = min(ihi, j.iy - iy0);
                }
                for (int kk = (s - k0) & (S - 1); kk < ck; kk += S) {
                    const float* in = tile + ((size_t)(zl + kk) * wy + ly * NY + ilo) * wx + 8 * lx;
                    const float* tp = taps + ((size_t)kk * cy + ilo) * kxp;
                    float pl[NY][8];
#pragma unroll
                    for (int o = 0; o < NY; ++o)
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if (!CHAIN || (q0 == 0 && p0 == 0)) acc[o][i] = 0.f;  // CHAIN: ck is 1, one plane at a time
                            pl[o][i] = 0.f;
                        }
                    for (int iy = ilo; iy < ihi; ++iy, in += wx, tp += kxp) {
                        const int lo = max(0, iy - cy + 1), hi = min(NY - 1, iy);
                        bc_rows<NY, KX>(lo, hi, in, tp, kxp, nf, rem, acc);
                        if (COMP) {
#pragma unroll
                            for (int o = 0; o < NY; ++o)
#pragma unroll
                                for (int i = 0; i < 8; ++i) pl[o][i] += acc[o][i], acc[o][i] = 0.f;
                        }
                    }
#pragma unroll
                    for (int o = 0; o < NY; ++o)
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if (COMP) {
                                const float y = __fsub_rn(pl[o][i], cmp[o][i]);
                                const float t = __fadd_rn(tot[o][i], y);
                                cmp[o][i] = __fsub_rn(__fsub_rn(t, tot[o][i]), y);
                                tot[o][i] = t;
                            } else if (!CHAIN || (q0 + cy == j.ky && p0 + nx == j.kx)) {
                                tot[o][i] += acc[o][i];
                            }
                        }
                }
                __syncthreads();
            }
    if (S == 1) {
        const int z = z0 + zl;
        if (z >= j.oz) return;
#pragma unroll
        for (int o = 0; o < NY; ++o) {
            const int y = y0 + ly * NY + o;
            if (y >= j.oy) break;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (x0 + 8 * lx + i < j.ox) epi(x0 + 8 * lx + i, y, z, tot[o][i]);
        }
        return;
    }
    // the splits' partial sums: slot (split, plane, row, x)
    const int plane = 8 * NY * kBcTX;
    float* red = smem + (size_t)(s * nz + zl) * plane;
#pragma unroll
    for (int o = 0; o < NY; ++o) {
        float4* r = reinterpret_cast<float4*>(red + (ly * NY + o) * kBcTX + 8 * lx);
        r[0] = make_float4(tot[o][0], tot[o][1], tot[o][2], tot[o][3]);
        r[1] = make_float4(tot[o][4], tot[o][5], tot[o][6], tot[o][7]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nz * plane; i += blockDim.x) {
        float v = smem[i];
        for (int q = 1; q < S; ++q) v += smem[i + q * nz * plane];
        const int x = x0 + (i & 31), y = y0 + (i >> 5) % (8 * NY), z = z0 + i / (8 * NY * kBcTX);
        if (x < j.ox && y < j.oy && z < j.oz) epi(x, y, z, v);
    }
}

// out(d) (+)= sum_t tap(t) in(d + t) for d on the centred box od, t on the centred
// box td, `in` zero outside its centred box id; with mir the taps are reversed
inline BoxJob box_job(const float* in, const int id[3], const float* taps, const int td[3], bool mir, float* out,
                      const int od[3], bool add = false, bool mirror = false) {
    BoxJob j{};
    BoxConv& c = j.c;
    c.in = in;
    c.taps = taps;
    c.ix = id[0], c.iy = id[1], c.iz = id[2];
    c.kx = td[0], c.ky = td[1], c.kz = td[2];
    c.ox = od[0], c.oy = od[1], c.oz = od[2];
    c.offx = (id[0] - td[0] - od[0] + 1) / 2;  // the boxes are odd: half widths add up exactly
    c.offy = (id[1] - td[1] - od[1] + 1) / 2;
    c.offz = (id[2] - td[2] - od[2] + 1) / 2;
    c.mir = mir ? 1 : 0;
    j.out = out;
    j.add = add ? 1 : 0;
    j.mirror = mirror ? 1 : 0;
    return j;
}

mvd_status box_convs(std::vector<BoxJob> jobs, cudaStream_t st);

}  // namespace mvd
