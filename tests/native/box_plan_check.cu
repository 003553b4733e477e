// Prints the direct engine's tiling (csrc/box_conv.cuh, compiled here for the CPU) for the
// volumes and boxes on standard input, one "X Y Z Kx Ky Kz ty" per line:
// "ny s ck cy cx warps smem", or "none".
#include <cstdio>

#include "box_conv.cuh"

int main() {
    int X, Y, Z, kx, ky, kz, ty;
    while (std::scanf("%d %d %d %d %d %d %d", &X, &Y, &Z, &kx, &ky, &kz, &ty) == 7) {
        mvd::BcPlan p{};
        if (mvd::bc_plan(X, Y, Z, kx, ky, kz, ty == 8 ? 2 : 1, &p))
            std::printf("%d %d %d %d %d %d %zu\n", p.ny, p.s, p.ck, p.cy, p.cx, p.warps, p.smem);
        else
            std::printf("none\n");
    }
    return 0;
}
