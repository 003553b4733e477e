// Aligned double-float (adf.cuh) on packed pairs: a complex value is two 64-bit
// register pairs, the high parts (re, im) and the low parts (re, im), and every
// operation is one two-lane FP32 instruction (add/mul/fma.rn.f32x2, each lane
// rounded as its scalar form). The steps are those of adf.cuh, operation for
// operation, so the results are bit-identical to it. The same
// butterflies also run without a grid (Unaligned: TwoSum sums, renormalised products), as
// the first stage of a mixed-radix line does.
//
// Why: the FFT passes are bound by issue slots and shared memory, not by the FP32
// lanes. One radix-8 stage with its twiddles takes 23 instructions per point
// against 42 in scalar form; alone it runs at 117 lanes per clock and SM (the
// FP32 peak) and 2.93 points per clock against 2.42. The exchange of re and im that a
// product by i needs and the broadcast of a twiddle's part to both lanes cost almost
// nothing (operand selection). Packing two lines instead of re and im gave the same
// rate for twice the registers.
//
// In memory (global and shared) a complex double-float is 16 bytes in the order
// re.hi, im.hi, re.lo, im.lo, so that a 16-byte load gives the two pairs.
#pragma once

#include "dd.cuh"

namespace mvd {

typedef unsigned long long f2;  // two FP32 lanes: low word = first

#if defined(__CUDA_ARCH__)
#define MVD_F2_OP(NAME, PTX)                                              \
    __host__ __device__ __forceinline__ f2 NAME(f2 a, f2 b) {             \
        f2 d;                                                             \
        asm(PTX " %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));               \
        return d;                                                         \
    }
__host__ __device__ __forceinline__ f2 f2_of(float a, float b) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__host__ __device__ __forceinline__ void f2_get(f2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
MVD_F2_OP(f2_add, "add.rn.f32x2")
MVD_F2_OP(f2_sub, "sub.rn.f32x2")
MVD_F2_OP(f2_mul, "mul.rn.f32x2")
__host__ __device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
#else  // the same roundings lane by lane, for host checks
#define MVD_F2_OP(NAME, OP)                                               \
    __host__ __device__ __forceinline__ f2 NAME(f2 a, f2 b) {             \
        float ax, ay, bx, by;                                             \
        f2_get(a, ax, ay);                                                \
        f2_get(b, bx, by);                                                \
        return f2_of(ax OP bx, ay OP by);                                 \
    }
union f2_lanes {
    f2 v;
    float f[2];
};
__host__ __device__ __forceinline__ f2 f2_of(float a, float b) {
    f2_lanes u;
    u.f[0] = a, u.f[1] = b;
    return u.v;
}
__host__ __device__ __forceinline__ void f2_get(f2 v, float& a, float& b) {
    f2_lanes u;
    u.v = v;
    a = u.f[0], b = u.f[1];
}
MVD_F2_OP(f2_add, +)
MVD_F2_OP(f2_sub, -)
MVD_F2_OP(f2_mul, *)
__host__ __device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    float ax, ay, bx, by, cx, cy;
    f2_get(a, ax, ay);
    f2_get(b, bx, by);
    f2_get(c, cx, cy);
    return f2_of(fmaf(ax, bx, cx), fmaf(ay, by, cy));
}
#endif
#undef MVD_F2_OP
__host__ __device__ __forceinline__ f2 f2_neg(f2 a) { return a ^ 0x8000000080000000ull; }
__host__ __device__ __forceinline__ f2 f2_swap(f2 a) {
    float x, y;
    f2_get(a, x, y);
    return f2_of(y, x);
}
__host__ __device__ __forceinline__ f2 f2_dup(float a) { return f2_of(a, a); }

// complex double-float: h = (re.hi, im.hi), l = (re.lo, im.lo)
struct cdp {
    f2 h, l;
};

__host__ __device__ __forceinline__ cdp cdp_from4(float4 v) { return {f2_of(v.x, v.y), f2_of(v.z, v.w)}; }
__host__ __device__ __forceinline__ cdp cdp_load(const cdd* p) { return cdp_from4(*reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ cdp cdp_load_cg(const cdd* p) { return cdp_from4(__ldcg(reinterpret_cast<const float4*>(p))); }
__device__ __forceinline__ cdp cdp_load_nc(const cdd* p) { return cdp_from4(__ldg(reinterpret_cast<const float4*>(p))); }
__host__ __device__ __forceinline__ void cdp_store(cdd* p, cdp a) {
    float4 v;
    f2_get(a.h, v.x, v.y);
    f2_get(a.l, v.z, v.w);
    *reinterpret_cast<float4*>(p) = v;
}
__host__ __device__ __forceinline__ cdp cdp_zero() { return {0ull, 0ull}; }
__host__ __device__ __forceinline__ cdp cdp_from(float re, float im) { return {f2_of(re, im), 0ull}; }
// the value rounded to FP32 (re, im)
__host__ __device__ __forceinline__ float2 cdp_round(cdp a) {
    float x, y;
    f2_get(f2_add(a.h, a.l), x, y);
    return make_float2(x, y);
}
__host__ __device__ __forceinline__ float cdp_absmax(cdp a, float m) {
    float x, y;
    f2_get(a.h, x, y);
    return fmaxf(m, fmaxf(fabsf(x), fabsf(y)));
}

__host__ __device__ __forceinline__ cdp cdp_add(cdp a, cdp b) { return {f2_add(a.h, b.h), f2_add(a.l, b.l)}; }
__host__ __device__ __forceinline__ cdp cdp_sub(cdp a, cdp b) { return {f2_sub(a.h, b.h), f2_sub(a.l, b.l)}; }
__host__ __device__ __forceinline__ cdp cdp_half(cdp a) {  // exact
    const f2 k = f2_dup(0.5f);
    return {f2_mul(a.h, k), f2_mul(a.l, k)};
}
// the sign pair of a product by s i: s i (x + i y) = (-s y) + i (s x)
template <int S>
__host__ __device__ __forceinline__ f2 f2_si() {
    return f2_of(S > 0 ? -1.f : 1.f, S > 0 ? 1.f : -1.f);
}
// a + S i b (exact product by +-1, then the same rounding as an add)
template <int S>
__host__ __device__ __forceinline__ cdp cdp_addi(cdp a, cdp b) {
    const f2 s = f2_si<S>();
    return {f2_fma(f2_swap(b.h), s, a.h), f2_fma(f2_swap(b.l), s, a.l)};
}
template <int S>
__host__ __device__ __forceinline__ cdp cdp_muli(cdp a) {  // S i a, exact
    const f2 s = f2_si<S>();
    return {f2_mul(f2_swap(a.h), s), f2_mul(f2_swap(a.l), s)};
}
__host__ __device__ __forceinline__ cdp cdp_neg(cdp a) { return {f2_neg(a.h), f2_neg(a.l)}; }
__host__ __device__ __forceinline__ cdp cdp_conj(cdp a) {
    return {a.h ^ 0x8000000000000000ull, a.l ^ 0x8000000000000000ull};
}

// onto the grid of the constant pair c (adf_align)
__host__ __device__ __forceinline__ cdp cdp_align(cdp x, f2 c) {
    const f2 h = f2_sub(f2_add(x.h, c), c);
    return {h, f2_add(f2_sub(x.h, h), x.l)};
}
// lane-wise products by the double-float constants (kh + kl), aligned (adf_mulk)
__host__ __device__ __forceinline__ cdp cdp_mulk(cdp a, f2 kh, f2 kl, f2 c) {
    const f2 h = f2_sub(f2_add(f2_mul(a.h, kh), c), c);
    f2 r = f2_fma(a.h, kh, f2_neg(h));
    r = f2_fma(a.h, kl, r);
    return {h, f2_fma(a.l, kh, r)};
}
__host__ __device__ __forceinline__ cdp cdp_mulk(cdp a, dd k, f2 c) { return cdp_mulk(a, f2_dup(k.hi), f2_dup(k.lo), c); }
// by an FP32-exact constant (adf_mulf)
__host__ __device__ __forceinline__ cdp cdp_mulf(cdp a, float k, f2 c) {
    const f2 kk = f2_dup(k), h = f2_sub(f2_add(f2_mul(a.h, kk), c), c);
    return {h, f2_fma(a.l, kk, f2_fma(a.h, kk, f2_neg(h)))};
}
// x w (S < 0) or x conj(w) (S > 0), w a forward twiddle, aligned (adf_cmul): 14 instructions
template <int S>
__host__ __device__ __forceinline__ cdp cdp_cmul(cdp x, cdp w, f2 c) {
    float rh, ih, rl, il;
    f2_get(w.h, rh, ih);
    f2_get(w.l, rl, il);
    const cdp xs{f2_swap(x.h), f2_swap(x.l)};
    const cdp q = S < 0 ? cdp_mulk(xs, f2_of(-ih, ih), f2_of(-il, il), c) : cdp_mulk(xs, f2_of(ih, -ih), f2_of(il, -il), c);
    return cdp_add(cdp_mulk(x, f2_dup(rh), f2_dup(rl), c), q);
}

// double-float sums without a grid (Knuth's TwoSum of the high parts): x + y, x - y and
// x + S i y, 8 instructions each
__host__ __device__ __forceinline__ cdp cdp_two_add(cdp x, cdp y) {
    const f2 s = f2_add(x.h, y.h), nb = f2_sub(x.h, s);  // minus what s took of y
    const f2 e = f2_add(f2_sub(x.h, f2_add(s, nb)), f2_add(y.h, nb));
    return {s, f2_add(e, f2_add(x.l, y.l))};
}
__host__ __device__ __forceinline__ cdp cdp_two_sub(cdp x, cdp y) {
    const f2 s = f2_sub(x.h, y.h), nb = f2_sub(x.h, s);
    const f2 e = f2_add(f2_sub(x.h, f2_add(s, nb)), f2_sub(nb, y.h));
    return {s, f2_add(e, f2_sub(x.l, y.l))};
}
// x plus y with its parts exchanged and multiplied by the signs s (exact)
__host__ __device__ __forceinline__ cdp cdp_two_addx(cdp x, cdp y, f2 s) {
    const f2 yh = f2_swap(y.h);
    const f2 t = f2_fma(yh, s, x.h), nb = f2_sub(x.h, t);
    const f2 e = f2_add(f2_sub(x.h, f2_add(t, nb)), f2_fma(yh, s, nb));
    return {t, f2_add(e, f2_fma(f2_swap(y.l), s, x.l))};
}
template <int S>
__host__ __device__ __forceinline__ cdp cdp_two_addi(cdp x, cdp y) {
    return cdp_two_addx(x, y, f2_si<S>());
}
// x y as an unevaluated pair (dd_dot2_pair): 16 instructions
__host__ __device__ __forceinline__ cdp cdp_mul_pair(cdp x, cdp y) {
    float rh, ih, rl, il;
    f2_get(y.h, rh, ih);
    f2_get(y.l, rl, il);
    const f2 xs = f2_swap(x.h), rr = f2_dup(rh), ii = f2_of(-ih, ih);
    const f2 p = f2_mul(x.h, rr), q = f2_mul(xs, ii);
    f2 e = f2_fma(x.h, rr, f2_neg(p)), f = f2_fma(xs, ii, f2_neg(q));
    e = f2_fma(x.h, f2_dup(rl), e);
    e = f2_fma(x.l, rr, e);
    f = f2_fma(xs, f2_of(-il, il), f);
    f = f2_fma(f2_swap(x.l), ii, f);
    const f2 s = f2_add(p, q), bb = f2_sub(s, p);
    const f2 t = f2_add(f2_sub(p, f2_sub(s, bb)), f2_sub(q, bb));
    return {s, f2_add(t, f2_add(e, f))};
}

// x s for a real double-float s, renormalised (dd_mul)
__host__ __device__ __forceinline__ cdp cdp_scale(cdp x, dd s) {
    const f2 sh = f2_dup(s.hi), p = f2_mul(x.h, sh);
    f2 e = f2_fma(x.h, sh, f2_neg(p));
    e = f2_fma(x.h, f2_dup(s.lo), e);
    e = f2_fma(x.l, sh, e);
    const f2 h = f2_add(p, e);
    return {h, f2_sub(e, f2_sub(h, p))};
}

// The operations of a small DFT, on the grid of a constant pair c or, for Unaligned, in
// plain double-float (values on no common grid: the first stage of a mixed-radix line)
struct Unaligned {};
__host__ __device__ __forceinline__ cdp cdp_add(cdp a, cdp b, f2) { return cdp_add(a, b); }
__host__ __device__ __forceinline__ cdp cdp_add(cdp a, cdp b, Unaligned) { return cdp_two_add(a, b); }
__host__ __device__ __forceinline__ cdp cdp_sub(cdp a, cdp b, f2) { return cdp_sub(a, b); }
__host__ __device__ __forceinline__ cdp cdp_sub(cdp a, cdp b, Unaligned) { return cdp_two_sub(a, b); }
template <int S>
__host__ __device__ __forceinline__ cdp cdp_addi(cdp a, cdp b, f2) { return cdp_addi<S>(a, b); }
template <int S>
__host__ __device__ __forceinline__ cdp cdp_addi(cdp a, cdp b, Unaligned) { return cdp_two_addi<S>(a, b); }
__host__ __device__ __forceinline__ cdp cdp_mulk(cdp a, dd k, Unaligned) { return cdp_scale(a, k); }
__host__ __device__ __forceinline__ cdp cdp_mulf(cdp a, float k, Unaligned) {  // k a power of two: exact
    return {f2_mul(a.h, f2_dup(k)), f2_mul(a.l, f2_dup(k))};
}
// x (r + i S s) for double-float constants r, s
template <int S>
__host__ __device__ __forceinline__ cdp cdp_mulc(cdp x, dd r, dd s, f2 c) {
    const cdp xs{f2_swap(x.h), f2_swap(x.l)};
    return cdp_add(cdp_mulk(x, r, c), cdp_mulk(xs, f2_of(-S * s.hi, S * s.hi), f2_of(-S * s.lo, S * s.lo), c));
}
template <int S>
__host__ __device__ __forceinline__ cdp cdp_mulc(cdp x, dd r, dd s, Unaligned) {
    const cdp p = cdp_mul_pair(x, cdp{f2_of(r.hi, S * s.hi), f2_of(r.lo, S * s.lo)});
    const f2 h = f2_add(p.h, p.l);
    return {h, f2_sub(p.l, f2_sub(h, p.h))};
}

// small DFTs y[m] = sum_r v[r] exp(S 2 pi i r m / R); C: f2 (aligned) or Unaligned
template <int R, int S>
struct DftP;

template <int S>
struct DftP<2, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        const cdp a = v[0], b = v[1];
        v[0] = cdp_add(a, b, c);
        v[1] = cdp_sub(a, b, c);
    }
};

template <int S>
struct DftP<4, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        const cdp t0 = cdp_add(v[0], v[2], c), t1 = cdp_sub(v[0], v[2], c);
        const cdp t2 = cdp_add(v[1], v[3], c), t3 = cdp_sub(v[1], v[3], c);
        v[0] = cdp_add(t0, t2, c);
        v[2] = cdp_sub(t0, t2, c);
        v[1] = cdp_addi<S>(t1, t3, c);
        v[3] = cdp_addi<-S>(t1, t3, c);
    }
};

template <int S>
struct DftP<8, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        cdp e[4] = {v[0], v[2], v[4], v[6]};
        cdp o[4] = {v[1], v[3], v[5], v[7]};
        DftP<4, S>::run(e, c);
        DftP<4, S>::run(o, c);
        // o1 (1 + S i) h and o3 (-1 + S i) h, h = sqrt(2)/2
        const dd hd = MVD_DD(0.70710678118654752440);
        const cdp w1 = cdp_mulk(cdp_addi<S>(o[1], o[1], c), hd, c);
        const cdp w3 = cdp_mulk(cdp_addi<-S>(o[3], o[3], c), hd, c);  // its negative
        v[0] = cdp_add(e[0], o[0], c);
        v[4] = cdp_sub(e[0], o[0], c);
        v[1] = cdp_add(e[1], w1, c);
        v[5] = cdp_sub(e[1], w1, c);
        v[2] = cdp_addi<S>(e[2], o[2], c);
        v[6] = cdp_addi<-S>(e[2], o[2], c);
        v[3] = cdp_sub(e[3], w3, c);
        v[7] = cdp_add(e[3], w3, c);
    }
};

template <int S>
struct DftP<3, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        const cdp t = cdp_add(v[1], v[2], c), u = cdp_sub(v[1], v[2], c);
        const dd hd = MVD_DD(0.86602540378443864676);  // sin(2 pi / 3)
        const cdp m = cdp_add(v[0], cdp_mulf(t, -0.5f, c), c), j = cdp_mulk(u, hd, c);
        v[0] = cdp_add(v[0], t, c);
        v[1] = cdp_addi<S>(m, j, c);
        v[2] = cdp_addi<-S>(m, j, c);
    }
};

template <int S>
struct DftP<5, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        const dd c1 = MVD_DD(0.30901699437494742410), c2 = MVD_DD(-0.80901699437494742410);
        const dd s1 = MVD_DD(0.95105651629515357212), s2 = MVD_DD(0.58778525229247312917);
        const cdp t1 = cdp_add(v[1], v[4], c), u1 = cdp_sub(v[1], v[4], c);
        const cdp t2 = cdp_add(v[2], v[3], c), u2 = cdp_sub(v[2], v[3], c);
        const cdp a0 = v[0];
        const cdp m1 = cdp_add(a0, cdp_add(cdp_mulk(t1, c1, c), cdp_mulk(t2, c2, c), c), c);
        const cdp m2 = cdp_add(a0, cdp_add(cdp_mulk(t1, c2, c), cdp_mulk(t2, c1, c), c), c);
        const cdp j1 = cdp_add(cdp_mulk(u1, s1, c), cdp_mulk(u2, s2, c), c);
        const cdp j2 = cdp_sub(cdp_mulk(u1, s2, c), cdp_mulk(u2, s1, c), c);
        v[0] = cdp_add(a0, cdp_add(t1, t2, c), c);
        v[1] = cdp_addi<S>(m1, j1, c);
        v[4] = cdp_addi<-S>(m1, j1, c);
        v[2] = cdp_addi<S>(m2, j2, c);
        v[3] = cdp_addi<-S>(m2, j2, c);
    }
};

// length 6 as 2 x 3 with coprime factors (Good-Thomas): no twiddles between
template <int S>
struct DftP<6, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        cdp a[3] = {cdp_add(v[0], v[3], c), cdp_add(v[2], v[5], c), cdp_add(v[4], v[1], c)};
        cdp b[3] = {cdp_sub(v[0], v[3], c), cdp_sub(v[2], v[5], c), cdp_sub(v[4], v[1], c)};
        DftP<3, S>::run(a, c);
        DftP<3, S>::run(b, c);
        v[0] = a[0], v[4] = a[1], v[2] = a[2];
        v[3] = b[0], v[1] = b[1], v[5] = b[2];
    }
};

// length 9 as 3 x 3 with the internal twiddles exp(s 2 pi i m / 9), m = 1, 2, 4
template <int S>
struct DftP<9, S> {
    template <typename C>
    __host__ __device__ __forceinline__ static cdp mul_root(cdp x, int m, C c) {
        const double cr = m == 1 ? 0.76604444311897803520 : m == 2 ? 0.17364817766693034885 : -0.93969262078590838405;
        const double si = m == 1 ? 0.64278760968653932632 : m == 2 ? 0.98480775301220805936 : 0.34202014332566873304;
        return cdp_mulc<S>(x, MVD_DD(cr), MVD_DD(si), c);
    }
    template <typename C>
    __host__ __device__ __forceinline__ static void run(cdp* v, C c) {
        cdp c0[3] = {v[0], v[3], v[6]};
        cdp c1[3] = {v[1], v[4], v[7]};
        cdp c2[3] = {v[2], v[5], v[8]};
        DftP<3, S>::run(c0, c);
        DftP<3, S>::run(c1, c);
        DftP<3, S>::run(c2, c);
        cdp r0[3] = {c0[0], c1[0], c2[0]};
        cdp r1[3] = {c0[1], mul_root(c1[1], 1, c), mul_root(c2[1], 2, c)};
        cdp r2[3] = {c0[2], mul_root(c1[2], 2, c), mul_root(c2[2], 4, c)};
        DftP<3, S>::run(r0, c);
        DftP<3, S>::run(r1, c);
        DftP<3, S>::run(r2, c);
        v[0] = r0[0], v[3] = r0[1], v[6] = r0[2];
        v[1] = r1[0], v[4] = r1[1], v[7] = r1[2];
        v[2] = r2[0], v[5] = r2[1], v[8] = r2[2];
    }
};

// length 16 as 4 x 4: radix 4 over n1 for each n2 (n = 4 n1 + n2), twiddles
// exp(S 2 pi i n2 k1 / 16), radix 4 over n2 (k = k1 + 4 k2). Inputs bounded by 2^18 q:
// the first sums reach 2^20.5 q (the products' range is 2^22 q), the outputs 2^22.5 q.
template <int S>
struct DftP<16, S> {
    __host__ __device__ __forceinline__ static void run(cdp* v, f2 c) {
        const dd c1 = MVD_DD(0.92387953251128675613), s1 = MVD_DD(0.38268343236508977173);
        const dd nc1 = MVD_DD(-0.92387953251128675613), ns1 = MVD_DD(-0.38268343236508977173);
        const dd h = MVD_DD(0.70710678118654752440), nh = MVD_DD(-0.70710678118654752440);
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            cdp x[4] = {v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]};
            DftP<4, S>::run(x, c);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) v[n2 + 4 * k1] = x[k1];
        }
        // v[n2 + 4 k1] times w^(n2 k1)
        v[5] = cdp_mulc<S>(v[5], c1, s1, c);
        v[9] = cdp_mulk(cdp_addi<S>(v[9], v[9]), h, c);
        v[13] = cdp_mulc<S>(v[13], s1, c1, c);
        v[6] = cdp_mulk(cdp_addi<S>(v[6], v[6]), h, c);
        v[10] = cdp_muli<S>(v[10]);
        v[14] = cdp_mulk(cdp_addi<-S>(v[14], v[14]), nh, c);
        v[7] = cdp_mulc<S>(v[7], s1, c1, c);
        v[11] = cdp_mulk(cdp_addi<-S>(v[11], v[11]), nh, c);
        v[15] = cdp_mulc<S>(v[15], nc1, ns1, c);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) DftP<4, S>::run(v + 4 * k1, c);
        // v[4 k1 + k2] -> k1 + 4 k2
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = a + 1; b < 4; ++b) {
                const cdp t = v[4 * a + b];
                v[4 * a + b] = v[4 * b + a];
                v[4 * b + a] = t;
            }
    }
};

}  // namespace mvd
