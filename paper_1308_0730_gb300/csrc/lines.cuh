// Mixed-radix Stockham transforms of the n lines of a tile in shared memory, for any
// {2,3,5}-smooth length, on double-float (cdp, adp.cuh) or FP32 (float2) values.
//
// What bounds these passes is instructions (index arithmetic beside the butterflies)
// and the blocks in flight, not memory. Hence:
//   - n is a power of two and consecutive threads take consecutive lines (thread t:
//     line t mod n, butterfly t / n), so the only division left is j / Ns, a float
//     reciprocal; every access of a quarter-warp goes to n lines whose stride puts
//     them on different banks, whatever the radix;
//   - the first stage takes its inputs from a functor (global memory, or the staged
//     half spectra of an x inverse) and the last stage gives its outputs to one
//     (global memory, the ratio, the update, the kernel product): no pass over the
//     tile only loads, multiplies or stores;
//   - double-float runs on packed pairs: the first stage in plain double-float (its
//     inputs share no grid), the later ones aligned on the tile's grid (adf.cuh), which
//     the bound of the first stage's outputs gives. Aligning the inputs instead, with the
//     worst growth of every stage assumed, costs 1.5 bits in the mean and 3 on lines with
//     spikes (errors against 80-bit transforms, tests/native/line_host_check.cu), and was
//     no faster: a view update of 300x180x150 584 us, now 582, 288x288x144 754 and 729,
//     90x60x48 100 and 98, but 200x96x100 200 and 212;
//   - tiles of up to 1700 points (54 KB with both exchange buffers) and blocks of as
//     many threads as the second stage has butterflies: four or more per SM; operands
//     that only the last stage reads are prefetched into L2 when the block starts.
//
// Measured on 300x180x150 (us a launch, against passes that load, transform and store one
// after another): x forward 100 -> 51, y 65 -> 39, z 135 -> 90, ratio 207 -> 116, update
// 158 -> 81. Loads in flight bound them still (a third of the warps resident).
#pragma once

#include "adf.cuh"
#include "adp.cuh"
#include "fft.cuh"

namespace mvd {

// line stride in elements: `per` elements make 128 bytes (8 double-float, 16 FP32);
// n >= per lines take an odd stride, fewer are spread per / n apart
__host__ __device__ inline int line_stride_for(int least, int n, int per) {
    if (n >= per) return least | 1;
    const int m = 2 * per / n, r = per / n;
    return least + ((r - least % m) + m) % m;
}

// tile geometry of lines of length L: n = 2^ln lines, strides ls (elements of the
// pass's type), T threads
struct LineGeo {
    int L, ln, ls, T;
    __host__ __device__ int n() const { return 1 << ln; }
};

// What a pass's tiles may hold: points, and whether a tile's first-stage butterflies are at
// most 256, one for each thread of a block (a second, mostly empty round of them took
// 100x108x72 from 120 to 127 us a view update)
struct TileRule {
    int points;
    bool one_round;
};
__host__ __device__ constexpr TileRule dd_tile_rule() { return {1700, true}; }
__host__ __device__ constexpr TileRule f32_tile_rule() { return {2560, false}; }

// lines per tile: the largest power of two (at most `most` lines) that the rule allows
__host__ __device__ inline int tile_lines_log2(const FftPlan& p, TileRule r, int most) {
    int ln = 0;
    const int nb = p.nst ? p.L / p.radix[0] : 1;
    while ((2 << ln) <= 32 && (1 << ln) < most && (p.L << (ln + 1)) <= r.points &&
           (!r.one_round || (nb << (ln + 1)) <= 256))
        ++ln;
    return ln;
}
__host__ __device__ inline int tile_threads(const FftPlan& p, int ln) {
    const int r = p.nst > 1 ? p.radix[1] : p.nst ? p.radix[0] : 1;
    const int t = ((((p.L / r) << ln) + 31) / 32) * 32;
    return t < 64 ? 64 : (t > 256 ? 256 : t);
}

// values of a transform: memory type, twiddles in the plan's stage order, arithmetic
template <typename V>
struct LineV;

template <>
struct LineV<cdp> {
    using Mem = cdd;
    static constexpr bool kAligned = true;
    __device__ __forceinline__ static cdp load(const cdd* p) { return cdp_load(p); }
    __device__ __forceinline__ static void store(cdd* p, cdp v) { cdp_store(p, v); }
    template <int S>
    __device__ __forceinline__ static cdp tmul(cdp x, const cdd* tw, f2 c) {
        return cdp_cmul<S>(x, cdp_load_nc(tw), c);
    }
    __device__ __forceinline__ static cdp align(cdp x, f2 c) { return cdp_align(x, c); }
    __device__ __forceinline__ static float absmax(cdp x, float m) { return cdp_absmax(x, m); }
    template <int R, int S, typename C>
    __device__ __forceinline__ static void dft(cdp* v, C c) {
        DftP<R, S>::run(v, c);
    }
};

template <>
struct LineV<float2> {
    using Mem = float2;
    static constexpr bool kAligned = false;
    __device__ __forceinline__ static float2 load(const float2* p) { return *p; }
    __device__ __forceinline__ static void store(float2* p, float2 v) { *p = v; }
    template <int S>
    __device__ __forceinline__ static float2 tmul(float2 x, const float2* tw, f2) {
        return cmul(x, twiddle<S>(tw, 0));
    }
    __device__ __forceinline__ static float2 align(float2 x, f2) { return x; }
    __device__ __forceinline__ static float absmax(float2, float m) { return m; }
    template <int R, int S, typename C>
    __device__ __forceinline__ static void dft(float2* v, C) {
        Dft<R, S>::run(v);
    }
};

// The block's largest value of mx (>= 0), through 8 words of shared memory: written
// before a block barrier, read after it
__device__ __forceinline__ void put_bound(float mx, unsigned* w) {
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = m;
}
__device__ __forceinline__ float get_bound(const unsigned* w) {
    const unsigned lane = threadIdx.x & 31;  // one word a lane: the loop over the words held more registers
    return __uint_as_float(__reduce_max_sync(0xffffffffu, lane < blockDim.x >> 5 ? w[lane] : 0u));
}

// Which butterfly of a stage thread t takes: consecutive threads along the n lines, or
// (ROWS) along a line, for stages that read or write global memory whose lines are
// contiguous. Shared memory then sees consecutive elements, or every R-th one where a
// first stage writes.
template <bool ROWS>
struct Butterfly {
    int ln, nb;
    float inv_nb;
    __device__ __forceinline__ Butterfly(const LineGeo& g, int nb_) : ln(g.ln), nb(nb_), inv_nb(1.0f / (float)nb_) {}
    __device__ __forceinline__ void at(int t, int& line, int& j) const {
        if constexpr (ROWS) {
            line = small_div(t, inv_nb);
            j = t - line * nb;
        } else {
            line = t & ((1 << ln) - 1);
            j = t >> ln;
        }
    }
};

// First stage: elements j + r L/R of a line from src(line, element), outputs to
// out(line, element, value); mx: the largest component of the thread's outputs.
// ROWS radices whose stride in shared memory would put a quarter-warp on one or two
// banks (8, 4, 2) keep the other mapping.
template <int R, int S, typename V, bool ROWS, typename Src, typename Out>
__device__ __forceinline__ void line_first(const LineGeo& g, Src&& src, Out&& out, float& mx) {
    using T = LineV<V>;
    const int nb = g.L / R, total = nb << g.ln;
    const Butterfly<ROWS && (R == 6 || R % 2 == 1)> bf(g, nb);
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int line, j;
        bf.at(t, line, j);
        V v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src(line, j + r * nb);
        T::template dft<R, S>(v, Unaligned{});
#pragma unroll
        for (int r = 0; r < R; ++r) {
            mx = T::absmax(v[r], mx);
            out(line, j * R + r, v[r]);
        }
    }
}

// A later stage (Ns points combined before it) from the shared buffer A
template <int R, int S, typename V, bool ROWS, typename Out>
__device__ __forceinline__ void line_stage(const LineGeo& g, const typename LineV<V>::Mem* A, int Ns,
                                           const typename LineV<V>::Mem* tw, f2 c, Out&& out) {
    using T = LineV<V>;
    const int nb = g.L / R, total = nb << g.ln;
    const float inv_ns = 1.0f / (float)Ns;
    const Butterfly<ROWS> bf(g, nb);
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int line, j;
        bf.at(t, line, j);
        const int jq = small_div(j, inv_ns), k = j - jq * Ns;
        const typename T::Mem* a = A + line * g.ls + j;
        V v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = T::load(a + r * nb);
        v[0] = T::align(v[0], c);
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = T::template tmul<S>(v[r], tw + (r - 1) * Ns + k, c);
        T::template dft<R, S>(v, c);
        const int d = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) out(line, d + r * Ns, v[r]);
    }
}

// A middle stage, shared buffer to shared buffer: one function per radix, sign and type
// for every pass (inlined into each they would triple the code)
template <int R, int S, typename V>
__device__ __noinline__ void line_middle(const LineGeo& g, const typename LineV<V>::Mem* from,
                                         typename LineV<V>::Mem* to, int Ns, const typename LineV<V>::Mem* tw, f2 c) {
    line_stage<R, S, V, false>(g, from, Ns, tw, c, [&](int line, int i, V v) { LineV<V>::store(to + line * g.ls + i, v); });
}

// Any stage, shared buffer to shared buffer (Ns = 1: the first, without twiddles or a
// grid); returns the largest component of the first stage's outputs
template <int R, int S, typename V>
__device__ __noinline__ float line_any(const LineGeo& g, const typename LineV<V>::Mem* from,
                                       typename LineV<V>::Mem* to, int Ns, const typename LineV<V>::Mem* tw, f2 c) {
    using T = LineV<V>;
    float mx = 0.f;
    if (Ns == 1) {
        line_first<R, S, V, false>(
            g, [&](int line, int i) { return T::load(from + line * g.ls + i); },
            [&](int line, int i, V v) { T::store(to + line * g.ls + i, v); }, mx);
    } else {
        line_stage<R, S, V, false>(g, from, Ns, tw, c, [&](int line, int i, V v) { T::store(to + line * g.ls + i, v); });
    }
    return mx;
}

// CALL(R) for the plan's radices (10 in FP32 plans only)
#define MVD_RADIX_SWITCH(R, CALL)            \
    switch (R) {                             \
        case 8: CALL(8); break;              \
        case 9: CALL(9); break;              \
        case 6: CALL(6); break;              \
        case 5: CALL(5); break;              \
        case 4: CALL(4); break;              \
        case 3: CALL(3); break;              \
        case 10:                             \
            if constexpr (!T::kAligned) {    \
                CALL(10);                    \
            }                                \
            break;                           \
        default: CALL(2); break;             \
    }

// Transforms the tile's lines (sign S): src(line, element) -> last(buf, line, element,
// value), where buf is the shared buffer the last stage does not read (the caller's to
// fill or ignore). A and B: exchange buffers, n lines of stride g.ls; src may read B
// (not A) and global memory the pass itself overwrites through `last`. tw: the stage-
// ordered twiddles of the plan. The caller synchronises before (what src reads) and
// after. Returns buf. RIN, ROUT: the first / last stage runs along the lines (Butterfly).
// STAGED: every stage goes through shared memory by the functions above, src and last in
// loops of their own (the persistent batch kernel: with the stages inlined into all of its
// passes it took eight minutes to compile).
template <int S, typename V, bool RIN, bool ROUT, bool STAGED, typename Src, typename Last>
__device__ __forceinline__ typename LineV<V>::Mem* line_transform(const LineGeo& g, const FftPlan& p,
                                                                  const typename LineV<V>::Mem* tw,
                                                                  typename LineV<V>::Mem* A, typename LineV<V>::Mem* B,
                                                                  unsigned* w, Src&& src, Last&& last) {
    using T = LineV<V>;
    typename T::Mem *from = A, *to = B;
    float mx = 0.f;
    int e = 0;
    if constexpr (STAGED) {
        const int total = g.L << g.ln;
        const Butterfly<RIN> in(g, g.L);
        const Butterfly<ROUT> res(g, g.L);
        for (int t = threadIdx.x; t < total; t += blockDim.x) {
            int line, i;
            in.at(t, line, i);
            T::store(A + line * g.ls + i, src(line, i));
        }
        __syncthreads();
        int Ns = 1;
        for (int s = 0; s < p.nst; ++s) {
            const int R = p.radix[s];
            f2 c = 0;
            if constexpr (T::kAligned) {
                if (s > 0) e = s == 1 ? adf_second_exp(get_bound(w)) : e + adf_gen_shift(p.radix[s - 1]);
                c = f2_dup(adf_const_exp2(e));
            }
#define MVD_CALL(RR) mx = line_any<RR, S, V>(g, from, to, Ns, tw, c)
            MVD_RADIX_SWITCH(R, MVD_CALL)
#undef MVD_CALL
            if constexpr (T::kAligned) {
                if (s == 0) put_bound(mx, w);
            }
            __syncthreads();
            if (s > 0) tw += (R - 1) * Ns;
            Ns *= R;
            typename T::Mem* x = from;
            from = to;
            to = x;
        }
        for (int t = threadIdx.x; t < total; t += blockDim.x) {
            int line, i;
            res.at(t, line, i);
            last(to, line, i, T::load(from + line * g.ls + i));
        }
        return to;
    }
    if (p.nst > 0) {
        auto out = [&](int line, int i, V v) { T::store(A + line * g.ls + i, v); };
#define MVD_CALL(RR) line_first<RR, S, V, RIN>(g, src, out, mx)
        MVD_RADIX_SWITCH(p.radix[0], MVD_CALL)
#undef MVD_CALL
    } else if ((int)threadIdx.x < g.n()) {  // an axis of length 1
        T::store(A + threadIdx.x * g.ls, src((int)threadIdx.x, 0));
    }
    if constexpr (T::kAligned) put_bound(mx, w);
    __syncthreads();
    if (p.nst <= 1) {  // a line of at most 10 points
        for (int t = threadIdx.x; t < (g.L << g.ln); t += blockDim.x) {
            const int line = t & (g.n() - 1), i = t >> g.ln;
            last(to, line, i, T::load(from + line * g.ls + i));
        }
        return to;
    }
    if constexpr (T::kAligned) e = adf_second_exp(get_bound(w));
    int Ns = p.radix[0];
    for (int s = 1; s < p.nst; ++s) {
        const int R = p.radix[s];
        f2 c = 0;
        if constexpr (T::kAligned) {
            if (s > 1) e += adf_gen_shift(p.radix[s - 1]);
            c = f2_dup(adf_const_exp2(e));
        }
        if (s + 1 == p.nst) {
            auto out = [&](int line, int i, V v) { last(to, line, i, v); };
#define MVD_CALL(RR) line_stage<RR, S, V, ROUT>(g, from, Ns, tw, c, out)
            MVD_RADIX_SWITCH(R, MVD_CALL)
#undef MVD_CALL
            break;
        }
#define MVD_CALL(RR) line_middle<RR, S, V>(g, from, to, Ns, tw, c)
        MVD_RADIX_SWITCH(R, MVD_CALL)
#undef MVD_CALL
        __syncthreads();
        tw += (R - 1) * Ns;
        Ns *= R;
        typename T::Mem* x = from;
        from = to;
        to = x;
    }
    return to;
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// `bytes` contiguous bytes at p, by the whole block
__device__ __forceinline__ void prefetch_rows(const void* p, int bytes) {
    for (int i = threadIdx.x * 128; i < bytes; i += blockDim.x * 128) prefetch_l2(static_cast<const char*>(p) + i);
}

// The two half spectra A, B of the real rows p and n + p from the transformed complex
// line z = a + i b of pair p: A = (z_k + conj z_-k) / 2, B = (z_k - conj z_-k) / (2 i)
__device__ __forceinline__ void unpack_pair(cdp zk, cdp zm, cdp& a, cdp& b) {
    zm = cdp_conj(zm);  // a line of one stage is on no grid
    a = cdp_half(cdp_two_add(zk, zm));
    b = cdp_half(cdp_muli<-1>(cdp_two_sub(zk, zm)));
}
__device__ __forceinline__ void unpack_pair(float2 zk, float2 zm, float2& a, float2& b) {
    a = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
    b = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
}
// and back: the full spectrum of a + i b at k (up: k <= L/2) or at L - k
__device__ __forceinline__ cdp pack_pair(cdp a, cdp b, bool up) {
    // up: a + i b; else conj(a - i b) = conj(a) + i conj(b)
    const f2 c = up ? 0ull : 0x8000000000000000ull;
    a.h ^= c, a.l ^= c;
    return cdp_two_addx(a, b, up ? f2_of(-1.f, 1.f) : f2_of(1.f, 1.f));
}
__device__ __forceinline__ float2 pack_pair(float2 a, float2 b, bool up) {
    return up ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, b.x - a.y);
}

// F: transformed lines (natural order, stride ls); store(k, row, value) receives the
// half spectra of the tile's rows
template <typename V, typename Store>
__device__ __forceinline__ void unpack_tile(const typename LineV<V>::Mem* F, int ls, int L, int ln, int nrows,
                                            Store&& store) {
    const int n = 1 << ln, m = (L / 2 + 1) << ln;
    for (int t = threadIdx.x; t < m; t += blockDim.x) {
        const int p = t & (n - 1), k = t >> ln;
        if (p >= nrows) continue;
        V a, b;
        unpack_pair(LineV<V>::load(F + p * ls + k), LineV<V>::load(F + p * ls + (k == 0 ? 0 : L - k)), a, b);
        store(k, p, a);
        if (n + p < nrows) store(k, n + p, b);
    }
}

}  // namespace mvd
