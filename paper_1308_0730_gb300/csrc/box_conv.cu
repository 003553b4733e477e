// Convolutions of small kernels with small kernels (the compound-kernel algebra
// and its vector-Jacobian product), batched; tiling in box_conv.cuh.
#include "box_conv.cuh"
#include "common.cuh"

namespace mvd {

namespace {

struct BoxJobs {
    BoxJob j[kBcMaxJobs];
};

// two blocks per SM: the compensated sums take four registers per output
template <int NY, int KX>
__global__ void __launch_bounds__(256, 2) k_box_conv(const __grid_constant__ BoxJobs jobs, int splits) {
    extern __shared__ float4 smem4[];
    pass_wait();
    const BoxJob& b = jobs.j[blockIdx.y];
    const int nz = 8 / splits;
    const int tx = (b.c.ox + kBcTX - 1) / kBcTX, ty = (b.c.oy + 8 * NY - 1) / (8 * NY), tz = (b.c.oz + nz - 1) / nz;
    const int t = blockIdx.x;
    if (t >= tx * ty * tz) return;
    bc_tile<NY, KX, false, true>(b.c, t % tx, (t / tx) % ty, t / (tx * ty), splits, reinterpret_cast<float*>(smem4),
                             [&](int x, int y, int z, float acc) {
        long g = (long)x + (long)b.c.ox * (y + (long)b.c.oy * z);
        if (b.mirror) g = (long)b.c.ox * b.c.oy * b.c.oz - 1 - g;
        b.out[g] = b.add ? b.out[g] + acc : acc;
    });
}

}  // namespace

mvd_status box_convs(std::vector<BoxJob> jobs, cudaStream_t st) {
    for (size_t first = 0; first < jobs.size(); first += kBcMaxJobs) {
        BoxJobs a{};
        const int n = (int)(jobs.size() - first < (size_t)kBcMaxJobs ? jobs.size() - first : kBcMaxJobs);
        long warps = 0;
        int kz = 1;
        for (int i = 0; i < n; ++i) {
            const BoxConv& c = jobs[first + i].c;
            a.j[i] = jobs[first + i];
            warps += (long)((c.ox + 31) / 32) * ((c.oy + 7) / 8) * c.oz;
            kz = c.kz > kz ? c.kz : kz;
        }
        // one tile height and split for the batch: the cheapest over all its boxes
        const int s0 = bc_splits(warps, kz);
        int ny = 0, s = s0;
        BcPlan plan[kBcMaxJobs];
        size_t smem = 0;
        double best = 0.0;
        auto take = [&](int t, bool pieces) {  // the batch in tiles of 8 t rows, if every box fits and it is cheaper
            double cost = 0.0;
            size_t sm = 0;
            BcPlan ps[kBcMaxJobs];
            for (int i = 0; i < n; ++i) {
                const BoxConv& c = a.j[i].c;
                if (!bc_plan_ny(c.ox, c.oy, c.oz, c.kx, c.ky, c.kz, t, s, 8, ps + i, pieces)) return;
                cost += ps[i].cost;
                sm = ps[i].smem > sm ? ps[i].smem : sm;
            }
            if (ny != 0 && cost >= best) return;
            best = cost, ny = t, smem = sm;
            for (int i = 0; i < n; ++i) plan[i] = ps[i];
        };
        for (; s <= 8; s *= 2) {
            take(2, false);
            take(1, false);
            if (ny) break;
        }
        const bool pieces = ny == 0;  // a box of which not one row of taps fits
        if (pieces) {
            s = s0;
            take(1, true);
        }
        if (ny == 0) {
            set_error("compound kernels: a PSF box is too large for the tiled convolution");
            return MVD_ERR_UNSUPPORTED;
        }
        long tiles = 1;
        const int nz = 8 / s;
        for (int i = 0; i < n; ++i) {
            BoxConv& c = a.j[i].c;
            c.ck = plan[i].ck;
            c.cy = plan[i].cy;
            c.cx = plan[i].cx;
            const long t = (long)((c.ox + 31) / 32) * ((c.oy + 8 * ny - 1) / (8 * ny)) * ((c.oz + nz - 1) / nz);
            tiles = t > tiles ? t : tiles;
        }
        auto kern = pieces ? k_box_conv<1, -1> : ny == 2 ? k_box_conv<2, 0> : k_box_conv<1, 0>;
        cudaError_t e = allow_smem(kern);
        if (e != cudaSuccess) return cuda_status(e, "box convolutions");
        e = launch_pass(kern, dim3((unsigned)tiles, (unsigned)n), 256, smem, st, a, s);
        if (e != cudaSuccess) return cuda_status(e, "box convolutions");
        count_launch();
        MVD_TRY(check_launch("box convolutions"));
    }
    return MVD_OK;
}

}  // namespace mvd
