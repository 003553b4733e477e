// Host check of the double-float FFT lines: the butterflies of csrc/adp.cuh (the code the
// passes run, compiled here for the CPU) in the passes' stage schedules, against a direct
// 80-bit DFT of the same input.
//
//   regs:  the register-resident lengths with their own plans and constants (dd_e points
//          per thread, and 8 in the x inverse: LineFFTDD's HEAD and SHIFT);
//   mixed: {2,3,5}-smooth plans as lines.cuh runs them: the first stage in plain
//          double-float, then aligned stages from adf_second_exp of its outputs' bound,
//          adf_gen_shift coarser per stage. The same line with an exact first stage (80
//          bits) gives the error that the schedule cannot do without.
//
// Prints per (plan, input pattern), means over 8 inputs: the largest error over L * (input
// bound), the same with an exact first stage, and over all inputs the largest |hi| / q at
// an aligned stage's input and output as log2, and whether every aligned output's hi lies
// on its grid.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "fft_dd_fast.cuh"
using namespace mvd;
typedef long double ld;

static cdp make(ld re, ld im) {
    const float rh = (float)re, ih = (float)im;
    return cdp{f2_of(rh, ih), f2_of((float)(re - rh), (float)(im - ih))};
}
static void value(cdp v, ld& re, ld& im) {
    float a, b, c, d;
    f2_get(v.h, a, b);
    f2_get(v.l, c, d);
    re = (ld)a + c;
    im = (ld)b + d;
}

template <typename C>
static void bfly(int R, cdp* v, C c) {
    switch (R) {
        case 9: DftP<9, -1>::run(v, c); break;
        case 8: DftP<8, -1>::run(v, c); break;
        case 6: DftP<6, -1>::run(v, c); break;
        case 5: DftP<5, -1>::run(v, c); break;
        case 4: DftP<4, -1>::run(v, c); break;
        case 3: DftP<3, -1>::run(v, c); break;
        default: DftP<2, -1>::run(v, c); break;
    }
}
static void bfly_aligned(int R, cdp* v, f2 c) {
    if (R == 16)
        DftP<16, -1>::run(v, c);
    else
        bfly(R, v, c);
}

struct Plan {
    std::vector<int> radix;
    int head = 0, shift = 0;  // regs; 0: mixed
    int length() const {
        int L = 1;
        for (int r : radix) L *= r;
        return L;
    }
};
template <int L, int E>
static Plan regs_plan() {
    Plan p;
    for (int s = 0; s < plan_e_nst(L, E); ++s) p.radix.push_back(plan_e_radix(L, E, s));
    p.head = LineFFTDD<L, E, -1, true>::HEAD;
    p.shift = LineFFTDD<L, E, -1, true>::SHIFT;
    return p;
}

struct Seen {
    double in = -1e9, out = -1e9;
    bool on_grid = true;
};
static double bits(cdp v, int e) {
    const float m = cdp_absmax(v, 0.f);
    return m > 0.f ? std::log2((double)m) - e : -1e9;
}

static std::vector<cdp> transform(std::vector<cdp> x, const Plan& p, bool exact_first, Seen* seen) {
    const int L = (int)x.size();
    std::vector<cdp> tw(L), y(L);
    for (int m = 0; m < L; ++m) tw[m] = make(cosl(-2 * M_PIl * m / L), sinl(-2 * M_PIl * m / L));
    int e = 0, Ns = 1;
    float M = 0.f;
    if (p.head) {
        for (cdp v : x) M = cdp_absmax(v, M);
        e = p.head == 18 ? adf_exp_for<18>(M) : adf_exp_for<19>(M);
    }
    for (size_t s = 0; s < p.radix.size(); ++s) {
        const int R = p.radix[s];
        if (p.head)
            e += s ? p.shift : 0;
        else if (s > 0)
            e = s == 1 ? adf_second_exp(M) : e + adf_gen_shift(p.radix[s - 1]);
        const bool aligned = p.head || s > 0;
        const f2 c = f2_dup(adf_const_exp2(e));
        for (int j = 0; j < L / R; ++j) {
            const int k = j % Ns;
            cdp v[16];
            for (int r = 0; r < R; ++r) v[r] = x[j + r * (L / R)];
            if (!aligned && exact_first) {
                ld re[16], im[16];
                for (int m = 0; m < R; ++m) {
                    re[m] = im[m] = 0;
                    for (int r = 0; r < R; ++r) {
                        const ld a = -2 * M_PIl * ((r * m) % R) / R;
                        ld xr, xi;
                        value(v[r], xr, xi);
                        re[m] += xr * cosl(a) - xi * sinl(a);
                        im[m] += xr * sinl(a) + xi * cosl(a);
                    }
                }
                for (int m = 0; m < R; ++m) v[m] = make(re[m], im[m]);
            } else if (!aligned) {
                bfly(R, v, Unaligned{});
            } else {
                v[0] = cdp_align(v[0], c);
                for (int r = 1; r < R; ++r)
                    v[r] = s ? cdp_cmul<-1>(v[r], tw[r * k * (L / (Ns * R))], c) : cdp_align(v[r], c);
                for (int r = 0; r < R; ++r) seen->in = std::fmax(seen->in, bits(v[r], e));
                bfly_aligned(R, v, c);
                const float q = std::ldexp(1.f, e);
                for (int r = 0; r < R; ++r) {
                    float h[2];
                    f2_get(v[r].h, h[0], h[1]);
                    seen->out = std::fmax(seen->out, bits(v[r], e));
                    seen->on_grid = seen->on_grid && std::fmod(h[0], q) == 0.f && std::fmod(h[1], q) == 0.f;
                }
            }
            if (s == 0)
                for (int r = 0; r < R; ++r) M = cdp_absmax(v[r], M);
            for (int r = 0; r < R; ++r) y[(j / Ns) * Ns * R + k + r * Ns] = v[r];
        }
        x.swap(y);
        Ns *= R;
    }
    return x;
}

int main(int argc, char** argv) {
    const bool regs = argc > 1 && argv[1][0] == 'r';
    std::vector<Plan> plans;
    if (regs) {
        plans = {regs_plan<32, dd_e(32)>(),     regs_plan<64, dd_e(64)>(),     regs_plan<128, dd_e(128)>(),
                 regs_plan<256, dd_e(256)>(),   regs_plan<512, dd_e(512)>(),   regs_plan<1024, dd_e(1024)>(),
                 regs_plan<128, kXInvE>(),      regs_plan<256, kXInvE>(),      regs_plan<1024, kXInvE>()};
    } else {
        for (std::vector<int> r : std::vector<std::vector<int>>{{9, 6, 5}, {6, 5, 5}, {9, 5, 4}, {5, 5, 4}, {9, 8},
                                                                {6, 6}, {9, 9, 9}, {5, 5, 3}, {8, 6, 5}, {4, 4, 4},
                                                                {3, 3, 3, 3}, {2, 2, 3}, {9, 6, 5, 2}, {8, 8, 4, 4}})
            plans.push_back(Plan{r});
    }
    std::mt19937_64 g(11);
    std::uniform_real_distribution<double> U(0, 1);
    for (const Plan& p : plans) {
        const int L = p.length(), T = 8;
        std::vector<ld> cs(L), sn(L);
        for (int m = 0; m < L; ++m) cs[m] = cosl(-2 * M_PIl * m / L), sn[m] = sinl(-2 * M_PIl * m / L);
        for (int pat = 0; pat < 8; ++pat) {
            ld err = 0, ref = 0;
            Seen seen;
            for (int t = 0; t < T; ++t) {
                std::vector<cdp> x(L);
                std::vector<ld> xr(L), xi(L), wr(L), wi(L);
                ld bound = 0;
                const int f = 1 + (int)(U(g) * (L - 1));
                const double ph = U(g), lvl = 1 + U(g);
                for (int n = 0; n < L; ++n) {
                    const ld a = 2 * M_PIl * ((ld)((long)f * n % L) / L + ph);
                    ld re = 0, im = 0;
                    switch (pat) {
                        case 0: re = U(g); im = U(g); break;                         // uniform
                        case 1: re = 3.7 * lvl; im = -1.1; break;                    // constant
                        case 2: re = U(g) < 0.01 ? 1e6 * U(g) : 1e-3 * U(g); break;  // spikes
                        case 3:                                                      // 8 decades
                            re = powl(10.0L, -8 * U(g)) * (U(g) - .5);
                            im = powl(10.0L, -8 * U(g)) * (U(g) - .5);
                            break;
                        case 4: re = (n & 1) ? -lvl : 1; im = -re; break;            // alternating
                        case 5: re = cosl(a); im = sinl(a); break;                   // one tone
                        case 6: re = U(g) * 1e3 + U(g) * 1e-5; im = U(g) * 1e-4; break;  // low parts
                        default:  // the largest sums: both parts at the bound, signs along a tone
                            re = cosl(a) + sinl(a) >= 0 ? 1.9999 : -1.9999;
                            im = cosl(a) - sinl(a) >= 0 ? 1.9999 : -1.9999;
                    }
                    x[n] = make(re, im);
                    value(x[n], xr[n], xi[n]);
                    bound = fmaxl(bound, fmaxl(fabsl(xr[n]), fabsl(xi[n])));
                }
                for (int k = 0; k < L; ++k) {
                    wr[k] = wi[k] = 0;
                    for (int n = 0; n < L; ++n) {
                        const int m = (int)((long)n * k % L);
                        wr[k] += xr[n] * cs[m] - xi[n] * sn[m];
                        wi[k] += xr[n] * sn[m] + xi[n] * cs[m];
                    }
                }
                auto worst = [&](const std::vector<cdp>& y) {
                    ld m = 0;
                    for (int k = 0; k < L; ++k) {
                        ld a, b;
                        value(y[k], a, b);
                        m = fmaxl(m, fmaxl(fabsl(a - wr[k]), fabsl(b - wi[k])));
                    }
                    return m / (bound * L);
                };
                Seen dummy;
                err += worst(transform(x, p, false, &seen)) / T;
                ref += regs ? 0 : worst(transform(x, p, true, &dummy)) / T;
            }
            printf("%d:%d %d %.6Le %.6Le %.3f %.3f %d\n", L, p.radix[0], pat, err, ref, seen.in, seen.out, (int)seen.on_grid);
        }
    }
    return 0;
}
