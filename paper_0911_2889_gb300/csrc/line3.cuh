// line3.cuh -- transforms of lines of L = 3 * 2^A points, the lengths of the
// step's alias-free grid (see flame_step.cuh).
//
// A line is transformed by mixed-radix Stockham passes: one pass of radix
// 3 F and power-of-two passes of radix at most 4 F, with F = 1, 2 or 4.
//   * The 3 F pass sits at the spectral end of the transform: first in the
//     inverse (spectrum -> points), last in the forward transform.  A third
//     of a retained line's spectrum is padding, so a thread that holds the 3 F
//     entries t + r TS (r < 3 F, TS = L / (3 F)) holds F of them known to be
//     zero (pass A) or not wanted (pass C): the compiler drops them.
//   * At the physical end a thread holds the 4 F points t + r TP,
//     TP = L / (4 F) = 3/4 TS: a quarter of a line's threads sit the
//     power-of-two passes out, which costs no issue slots (they wait at the
//     barriers), and the inverse transform's output is the forward one's
//     input without an exchange.
// F = 4 (radix 12 and 16, three passes for 3072 points) does the fewest
// shared-memory exchanges; F = 1 and 2 give a line more threads with shorter
// chains, for grids too small to fill the SMs.
//
// Radix 3 F is done by the prime-factor map (3 x F, no twiddles between).
#pragma once

#include "fft_engine.cuh"

namespace flame {

// ----------------------------------------------------------------------------
// In-register DFTs of 3, 6 and 12 points, natural order in and out
// ----------------------------------------------------------------------------
template <int DIR, class V> __device__ __forceinline__ void dft3(CV<V> &x0, CV<V> &x1, CV<V> &x2) {
    using Real = decltype(x0.re.x);
    constexpr double kS = 0.866025403784438646763723170752936183;  // sin(pi/3)
    const V half = vbc_as((Real)0.5, V{}), sd = vbc_as((Real)kS, V{});
    const CV<V> t = cadd(x1, x2), d = csub(x1, x2);
    const CV<V> m{vfma(vneg(t.re), half, x0.re), vfma(vneg(t.im), half, x0.im)};
    x0 = cadd(x0, t);
    // x1 = m + DIR i kS d, x2 = m - DIR i kS d
    const CV<V> p{vfma(vneg(d.im), sd, m.re), vfma(d.re, sd, m.im)}, n{vfma(d.im, sd, m.re), vfma(vneg(d.re), sd, m.im)};
    x1 = DIR > 0 ? p : n;
    x2 = DIR > 0 ? n : p;
}

// N = 3 F points (F = 1, 2, 4): n = (F n1 + 3 n2) mod N, k = (ka k1 + kb k2)
// mod N with ka = 1 (mod 3), 0 (mod F) and kb = 0 (mod 3), 1 (mod F)
template <int F, int DIR, class V> __device__ __forceinline__ void dft_3f(CV<V> (&x)[3 * F]) {
    constexpr int N = 3 * F;
    constexpr int ka = F == 1 ? 1 : 4, kb = F == 1 ? 0 : F == 2 ? 3 : 9;
    CV<V> y[N];
    static_for<0, F>([&](auto n2c) {
        constexpr int n2 = decltype(n2c)::value;
        CV<V> a = x[(3 * n2) % N], b = x[(F + 3 * n2) % N], c = x[(2 * F + 3 * n2) % N];
        dft3<DIR>(a, b, c);
        y[n2] = a;
        y[F + n2] = b;
        y[2 * F + n2] = c;
    });
    static_for<0, 3>([&](auto k1c) {
        constexpr int k1 = decltype(k1c)::value;
        CV<V> s[F];
#pragma unroll
        for (int i = 0; i < F; ++i) s[i] = y[F * k1 + i];
        dft<F, DIR>(s);
        static_for<0, F>([&](auto k2c) {
            constexpr int k2 = decltype(k2c)::value;
            x[(ka * k1 + kb * k2) % N] = s[k2];
        });
    });
}

// ----------------------------------------------------------------------------
// The pass plan of a line
// ----------------------------------------------------------------------------
constexpr int gcd_c(int a, int b) { return b == 0 ? a : gcd_c(b, a % b); }

// PRODUCTS: the last pass forms its twiddles (butterflies)
template <int A_, int F_, bool PRODUCTS_ = false> struct Plan3 {
    static constexpr bool PRODUCTS = PRODUCTS_;
    static constexpr int A = A_, F = F_, LF = F == 4 ? 2 : F == 2 ? 1 : 0;
    static_assert(F == 1 || F == 2 || F == 4, "F");
    static_assert(A >= LF + 2, "a line needs 12 F points");
    static constexpr int L = 3 << A, ES = 3 * F, EP = 4 * F, TS = L / ES, TP = L / EP;
    // the 2^(A - LF) points left by the radix-3F pass, as NQ radices
    static constexpr int NB = A - LF, MB = LF + 2, NQ = (NB + MB - 1) / MB;
    __host__ __device__ static constexpr int q_radix(int i) { return 1 << (NB / NQ + (i < NB % NQ ? 1 : 0)); }
    // pass s = 0 .. NQ of the inverse (INV) or forward transform
    template <bool INV> __host__ __device__ static constexpr bool spectral(int s) { return INV ? s == 0 : s == NQ; }
    template <bool INV> __host__ __device__ static constexpr int radix(int s) {
        return spectral<INV>(s) ? ES : q_radix(INV ? s - 1 : s);
    }
    template <bool INV> __host__ __device__ static constexpr int stride(int s) {  // product of the radices before s
        int n = 1;
        for (int i = 0; i < s; ++i) n *= radix<INV>(i);
        return n;
    }
    // twiddles of pass s >= 1: [(q-1) Ns + m] = exp(2 pi i q m / (r Ns)), q = 1 .. r-1, m < Ns; the
    // inverse's passes, then the forward's (stored with the + sign, conjugated by the forward)
    template <bool INV> __host__ __device__ static constexpr int tw_offset(int s) {
        int off = 0;
        if (!INV) off = tw_offset<true>(NQ + 1);
        for (int i = 1; i < s; ++i) off += (radix<INV>(i) - 1) * stride<INV>(i);
        return off;
    }
    __host__ __device__ static constexpr int kTwLen() { return tw_offset<false>(NQ + 1); }
    // Padding of the exchange after pass s, for W slots per shared-memory
    // wavefront: P slots every D.  Pass 0 stores runs of r slots per thread,
    // shifted by one slot whenever the runs come back to the same bank;
    // later passes store runs of Ns slots, and P makes a run go on in the
    // banks where the one before it ended.  Checked for all lengths by
    // enumeration: at most 1.5 wavefronts where 1 is the least.
    template <bool INV> __host__ __device__ static constexpr int pad_d(int s, int W) {
        const int r = radix<INV>(s);
        return s == 0 ? r / gcd_c(r, W) * W : stride<INV>(s) * r;
    }
    template <bool INV> __host__ __device__ static constexpr int pad_p(int s, int W) {
        if (s == 0) return 1;
        const int ns = stride<INV>(s), v = (ns - ns * radix<INV>(s)) % W;
        return v < 0 ? v + W : v;
    }
    template <bool INV> __host__ __device__ static constexpr int slots_dir(int W) {
        int m = L;
        for (int s = 0; s < NQ; ++s) {
            const int v = L + pad_p<INV>(s, W) * ((L - 1) / pad_d<INV>(s, W));
            m = v > m ? v : m;
        }
        return m;
    }
    // slots of a line's exchange buffer (a multiple of 8: two-line buffers stay 128-byte aligned)
    __host__ __device__ static constexpr int slots(int W) {
        const int a = slots_dir<true>(W), b = slots_dir<false>(W);
        return ((a > b ? a : b) + 7) & ~7;
    }
};
// slots per 128-byte wavefront of an exchange buffer: two lines take 16 bytes a
// slot (FP64: in each of two planes), one line keeps separate planes of 4
// (FP32) or 8 (FP64) bytes
template <class V> constexpr int kSlotsPerWave =
    std::is_same<V, float2>::value || std::is_same<V, double2>::value ? 8 : std::is_same<V, F1>::value ? 32 : 16;

// ----------------------------------------------------------------------------
// Twiddle allocation of a line: the tables of F = 1, 2, 4 (where the line is
// long enough), then exp(2 pi i k / 2L), k < L, for rows of 2 L points
// ----------------------------------------------------------------------------
template <int A, int F> __host__ __device__ constexpr int tw3_len() {
    if constexpr (A >= (F == 4 ? 4 : F == 2 ? 3 : 2)) return Plan3<A, F>::kTwLen();
    else return 0;
}
template <int A, int F> __host__ __device__ constexpr int tw3_offset() {
    return (F > 1 ? tw3_len<A, 1>() : 0) + (F > 2 ? tw3_len<A, 2>() : 0);
}
template <int A> __host__ __device__ constexpr int tw3_real_offset() { return tw3_offset<A, 4>() + tw3_len<A, 4>(); }
template <int A> __host__ __device__ constexpr int tw3_alloc_len() { return tw3_real_offset<A>() + (3 << A); }

constexpr int kMinA = 2, kMaxA = 10;  // lines of 12 .. 3072 points
// calls f(integral_constant<A>) for a line exponent lo <= a <= kMaxA known at
// run time (host)
template <int lo = kMinA, class Fn> static void with_a(int a, Fn &&f) {
    if constexpr (lo <= kMaxA) {
        if (a == lo) f(std::integral_constant<int, lo>{});
        else with_a<lo + 1>(a, f);
    }
}

inline size_t tw3_len_of(int a) {
    size_t n = 0;
    with_a(a, [&](auto ac) { n = tw3_alloc_len<decltype(ac)::value>(); });
    return n;
}
// The least a with 3 * 2^a >= 3 K + 1 points (at least 12): 2^a >= K + 1
inline int step_exponent(int K) {
    int a = kMinA;
    while ((1 << a) < K + 1) ++a;
    return a;
}

// ----------------------------------------------------------------------------
// Passes
// ----------------------------------------------------------------------------
// A plan with PRODUCTS, FP32: in the last pass w^q for q = 4a + b is the product
// w^(4a) w^b of two table entries, 6 loads for radix 16 instead of 15 (a 3072-point
// line's last pass reads 9 KB of its table instead of 23).  Such a twiddle is off
// by up to about 2 * 2^-24 (the entries' errors and the product's), a table entry
// by 0.7 * 2^-24, so only the rows of 3072 points take it, whose 4096-point
// predecessors on the public grid had products of two entries too: 4096x8192
// 136.1 -> 134.5 us a step, 2048x8192 74.0 -> 73.0.  Relative L2 error of the
// step's increment (nonlinear only, flat spectrum, mean of 4): 4096x8192 3.85e-7
// against 3.80e-7 with entries and 4.21e-7 on the public grid.  (In all passes
// from 768 points on: 3.91e-7 for 133.7 us, and 1024x2048 3.54e-7 against
// 3.38e-7 for 16.9 us instead of 17.0.)
template <class C, class PL> constexpr bool kTwiddleProducts = sizeof(C) == 8 && PL::PRODUCTS;

// Pass S on a thread's E points x[i] = element t + i T (T = L / E): B = E / r
// butterflies j = t + b T, twiddles, DFTs.
template <class PL, int DIR, bool INV, int S, int E, class V, class C>
__device__ __forceinline__ void butterflies(CV<V> (&x)[E], int t, const C *__restrict__ tw) {
    constexpr int r = PL::template radix<INV>(S), Ns = PL::template stride<INV>(S), T = PL::L / E, B = E / r;
#pragma unroll
    for (int b = 0; b < B; ++b) {
        CV<V> y[r];
#pragma unroll
        for (int q = 0; q < r; ++q) y[q] = x[b + B * q];
        if constexpr (Ns > 1) {
            const int j = t + b * T, m = Ns >= PL::L / r ? j : j % Ns;
            const C *w0 = tw + PL::template tw_offset<INV>(S) + m;
            if constexpr (kTwiddleProducts<C, PL> && S == PL::NQ && r >= 8) {
                C lo[4], hi = C{1, 0};  // w^1 .. w^3, w^(4a)
#pragma unroll
                for (int q = 1; q < 4; ++q) lo[q] = __ldg(w0 + (q - 1) * Ns);
#pragma unroll
                for (int q = 1; q < r; ++q) {
                    if (q % 4 == 0) hi = __ldg(w0 + (q - 1) * Ns);
                    const C l = lo[q % 4];
                    const C w = q < 4 ? l : q % 4 == 0 ? hi : C{hi.x * l.x - hi.y * l.y, hi.x * l.y + hi.y * l.x};
                    y[q] = cmul_s(y[q], w.x, DIR > 0 ? w.y : -w.y);
                }
            } else {
#pragma unroll
                for (int q = 1; q < r; ++q) {
                    const C w = __ldg(w0 + (q - 1) * Ns);
                    y[q] = cmul_s(y[q], w.x, DIR > 0 ? w.y : -w.y);
                }
            }
        }
        if constexpr (r % 3 == 0) dft_3f<r / 3, DIR>(y);
        else dft<r, DIR>(y);
#pragma unroll
        for (int q = 0; q < r; ++q) x[b + B * q] = y[q];
    }
}
// Stores pass S's results to the exchange buffer.
template <class PL, bool INV, int S, int E, class V>
__device__ __forceinline__ void put(const CV<V> (&x)[E], int t, const Planes<V> &sm) {
    constexpr int W = kSlotsPerWave<V>;
    constexpr int r = PL::template radix<INV>(S), Ns = PL::template stride<INV>(S), T = PL::L / E, B = E / r;
    constexpr int D = PL::template pad_d<INV>(S, W), P = PL::template pad_p<INV>(S, W);
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int j = t + b * T;
        // pass 0: r j + q, padded per D = a multiple of r; later: blocks of Ns r = D
        const int base = S == 0 ? r * j + P * (j / (D / r)) : (j / Ns) * (Ns * r + P) + j % Ns;
#pragma unroll
        for (int q = 0; q < r; ++q) sm.st_raw(base + q * Ns, x[b + B * q]);
    }
}
// Reads a thread's E points from the exchange after pass S.
template <class PL, bool INV, int S, int E, class V>
__device__ __forceinline__ void get(CV<V> (&x)[E], int t, const Planes<V> &sm) {
    constexpr int W = kSlotsPerWave<V>, T = PL::L / E;
    constexpr int D = PL::template pad_d<INV>(S, W), P = PL::template pad_p<INV>(S, W);
    if constexpr (T % D == 0) {
        const int base = t + P * (t / D);
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = sm.ld_raw(base + i * (T + P * (T / D)));
    } else if constexpr (D % T == 0) {
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = sm.ld_raw(t + i * T + P * (i * T / D));
    } else {
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = sm.ld_raw(t + i * T + P * ((t + i * T) / D));
    }
}

// A thread's place in a CTA of `lines` lines: its line and its index t within
// it, in the spectral layout (TS threads a line) or the physical one (TP).
struct Place {
    int line, t;
    bool on;  // the thread takes part
};
template <int T> __device__ __forceinline__ Place place(int lines) {
    const int line = (int)threadIdx.x / T;
    return {line, (int)threadIdx.x % T, line < lines};
}

// ... where the CTA is `lines` lines of TS threads exactly
template <int T> __device__ __forceinline__ Place place_all() { return {(int)threadIdx.x / T, (int)threadIdx.x % T, true}; }

// Inverse transform (sign +): spectral layout xs in, physical layout xp out.
// buf(line) is the line's exchange buffer; all threads of the CTA take part in
// the barriers.  First the pass at the spectral end, stored to the buffers;
// after a barrier, the rest.  Nothing may read the buffers any more when the
// first begins.
template <class PL, class V, class C, class Buf>
__device__ __forceinline__ void inverse3_first(CV<V> (&xs)[PL::ES], Place s, Buf buf, const C *__restrict__ tw) {
    if (s.on) {
        butterflies<PL, 1, true, 0>(xs, s.t, tw);
        put<PL, true, 0>(xs, s.t, buf(s.line));
    }
}
template <class PL, class V, class C, class Buf>
__device__ __forceinline__ void inverse3_rest(CV<V> (&xp)[PL::EP], Place p, Buf buf, const C *__restrict__ tw) {
    if (p.on) {
        get<PL, true, 0>(xp, p.t, buf(p.line));
        butterflies<PL, 1, true, 1>(xp, p.t, tw);
    }
    static_for<1, PL::NQ>([&](auto sc) {
        constexpr int S = decltype(sc)::value;
        __syncthreads();
        if (p.on) put<PL, true, S>(xp, p.t, buf(p.line));
        __syncthreads();
        if (p.on) {
            get<PL, true, S>(xp, p.t, buf(p.line));
            butterflies<PL, 1, true, S + 1>(xp, p.t, tw);
        }
    });
}
template <class PL, class V, class C, class Buf>
__device__ __forceinline__ void inverse3(CV<V> (&xs)[PL::ES], CV<V> (&xp)[PL::EP], Place s, Place p, Buf buf,
                                         const C *__restrict__ tw) {
    inverse3_first<PL>(xs, s, buf, tw);
    __syncthreads();
    inverse3_rest<PL>(xp, p, buf, tw);
}

// Forward transform (sign -): physical layout xp in, spectral layout xs out.
// FRESH: nothing reads the buffers any more when the call begins.
template <class PL, bool FRESH, class V, class C, class Buf>
__device__ __forceinline__ void forward3(CV<V> (&xp)[PL::EP], CV<V> (&xs)[PL::ES], Place p, Place s, Buf buf,
                                         const C *__restrict__ tw) {
    if (p.on) butterflies<PL, -1, false, 0>(xp, p.t, tw);
    static_for<0, PL::NQ - 1>([&](auto sc) {
        constexpr int S = decltype(sc)::value;
        if constexpr (S > 0 || !FRESH) __syncthreads();
        if (p.on) put<PL, false, S>(xp, p.t, buf(p.line));
        __syncthreads();
        if (p.on) {
            get<PL, false, S>(xp, p.t, buf(p.line));
            butterflies<PL, -1, false, S + 1>(xp, p.t, tw);
        }
    });
    if constexpr (PL::NQ > 1 || !FRESH) __syncthreads();
    if (p.on) put<PL, false, PL::NQ - 1>(xp, p.t, buf(p.line));
    __syncthreads();
    if (s.on) {
        get<PL, false, PL::NQ - 1>(xs, s.t, buf(s.line));
        butterflies<PL, -1, false, PL::NQ>(xs, s.t, tw);
    }
}

}  // namespace flame
