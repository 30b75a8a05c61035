// flame_step.cuh -- the step's passes on its alias-free grid.
//
// The quadratic term of eq. (SivCurv1c) is wanted on the retained harmonics
// |k_i| <= K_i only.  The product of two fields with K harmonics has 2 K; on a
// grid of L points harmonic m folds onto m - L, so the retained ones stay
// clean as long as L - 2 K > K: L >= 3 K + 1 points give the same coefficients
// as the N >= 4 K + 1 points of the augmented array of Sec. 3 (the 3/2 rule of
// pseudospectral methods, Orszag 1971), and the same mean of |grad Phi|^2.
// The step therefore transforms on L1 x L2 points, L = 3 * 2^a the least such
// length >= 3 K + 1: 3/4 of the public grid a side by default, less for a
// truncated box.  At 4096 x 8192 the row pass does 9/16 of the transforms and
// the workspaces hold 3/4 of the bytes (uv 101 MB, gk 50 MB).
//
// Three passes over HBM, as on the public grid:
//   A (columns): Phi(., k2) -> the row spectra of w = d1 Phi + i d2 Phi at
//                k2 and -k2, for all j1:  W(j1, k2) and W(j1, -k2).  Both are
//                inverse transforms of the same column:
//                  W(., k2)        = synthesis of (i s1 k1 - s2 k2) Phi,
//                  conj W(., -k2)  = synthesis of (i s1 k1 + s2 k2) Phi
//   B (rows):    w = inverse transform of W along k2, g = |w|^2 =
//                |grad Phi|^2, its forward real transform, k2 <= K2 kept
//   C (columns): forward transform along j1, |k1| <= K1 kept, update.
// Layouts:
//   uv  per (row pair, k2): W of both rows at k2, then at -k2.  FP32: (re, re,
//       im, im) of rows 2p, 2p+1, 16 bytes a sign, the two-line form pass B
//       works in; FP64: (re, im) of row 2p, then of row 2p+1.  Pass A writes
//       whole 32-byte sectors and a row pair is one contiguous block.  (With
//       +k2 and -k2 in planes of their own pass A's tensor stores wrote half
//       sectors: 4096x8192 40 -> 81 us.)
//   gk  g_index
// One extra CTA of pass B derives the step's coefficients and one of pass C
// the mean mode and the time (coef_cta, finish_cta).
#pragma once

#include "flame_kernels.cuh"
#include "line3.cuh"

namespace flame {

template <class V> constexpr int kLanes = sizeof(V) / sizeof(V{}.x);  // lines per thread
template <class R, int A, int F, class C> __device__ __forceinline__ const C *tab3(const void *tw) {
    return static_cast<const C *>(tw) + tw3_offset<A, F>();
}
// exchange buffer of line (or line pair) `line`, `slots` slots each
template <class V, class R> __device__ __forceinline__ Planes<V> planes3(unsigned char *smem, int line, int slots) {
    if constexpr (std::is_same<V, float2>::value) return Planes<V>(reinterpret_cast<V *>(smem) + (size_t)line * 2 * slots);
    else if constexpr (kLanes<V> == 2) return Planes<V>(reinterpret_cast<V *>(smem) + (size_t)line * 2 * slots, 0, slots);
    else return Planes<V>(reinterpret_cast<R *>(smem) + (size_t)line * 2 * slots, slots);
}
// bytes of a CTA's exchange buffers
template <class R, class V, class PL> __host__ __device__ constexpr size_t exchange_bytes(int lines) {
    return (size_t)lines * PL::slots(kSlotsPerWave<V>) * 2 * sizeof(V);
}
// Complex index of the (row pair, k2) entry that holds row j1: 4 complex
// numbers, two per sign.  FP32: -k2 comes first where k2 / 4 is odd, so that the
// 16-byte reads of one sign at 8 consecutive k2 in pass B's shared memory meet
// no bank twice.
template <class R> __host__ __device__ __forceinline__ int w_half(int k2, bool minus) {
    return sizeof(R) == 4 ? (int)minus ^ ((k2 >> 2) & 1) : (int)minus;
}
__host__ __device__ __forceinline__ size_t w_index(int j1, int k2, int ldk) { return 4 * ((size_t)(j1 >> 1) * ldk + k2); }
// Complex index of G(j1, k2) in gk: per (column pair, row pair) rows 2p, 2p+1
// of column 2q, then of 2q+1.  A column pair is contiguous (pass C), a row
// pair's sector too (pass B, which parks both rows of a column at once).
__host__ __device__ __forceinline__ size_t g_index(int j1, int k2, int n1) {
    return 2 * (size_t)(k2 >> 1) * n1 + 4 * (j1 >> 1) + 2 * (k2 & 1) + (j1 & 1);
}
// W(j1, +-k2) of one row.  What the previous kernel wrote is read by plain loads,
// never __ldg or through __restrict__: those may move ahead of griddep_wait.
template <class R> __device__ __forceinline__ CplxT<R> ld_w(const CplxT<R> *uv, int j1, int k2, int ldk, bool minus) {
    const CplxT<R> *e = uv + w_index(j1, k2, ldk) + 2 * w_half<R>(k2, minus);
    if constexpr (std::is_same<R, float>::value) {
        const float4 q = *reinterpret_cast<const float4 *>(e);
        return j1 & 1 ? CplxT<R>{q.y, q.w} : CplxT<R>{q.x, q.z};
    } else return e[j1 & 1];
}
// ... written by two adjacent threads, rows 2i and 2i+1 (all threads call it):
// FP32, one shuffle, and each thread writes 8 of the 16 bytes
template <class R> __device__ __forceinline__ void st_w(CplxT<R> *uv, int j1, int k2, int ldk, bool minus, CplxT<R> v, bool on) {
    CplxT<R> *e = uv + w_index(j1, k2, ldk) + 2 * w_half<R>(k2, minus);
    if constexpr (std::is_same<R, float>::value) {
        const bool odd = j1 & 1;
        const R got = __shfl_xor_sync(0xffffffffu, odd ? v.x : v.y, 1);
        if (on) e[odd] = odd ? CplxT<R>{got, v.y} : CplxT<R>{v.x, got};
    } else if (on) e[j1 & 1] = v;
}
// Two lines per thread: lane 0 of x is W(n, k2), lane 1 conj W(n, -k2), rows
// 2i and 2i+1 in adjacent threads (TP is even).  One shuffle gives the even
// thread both rows at k2 and the odd one both at -k2, as uv holds them.
__device__ __forceinline__ float4 w_pair(CV<float2> x, bool odd) {
    const float2 plus = make_float2(x.re.x, x.im.x), minus = make_float2(x.re.y, -x.im.y);
    const float2 give = odd ? plus : minus;
    const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, 1), __shfl_xor_sync(0xffffffffu, give.y, 1));
    const float2 r0 = odd ? got : plus, r1 = odd ? minus : got;
    return make_float4(r0.x, r1.x, r0.y, r1.y);
}

// The tile that starts when this one ends, `by` tiles further (the CTAs
// resident at once; 0: no prefetch), in this flame or, in an ensemble's
// launch, a later one: its input is prefetched into L2, behind this tile's own
// loads.
struct Ahead {
    int by, ntiles;
    const FlameDesc *ds;  // ensemble: its descriptors (flame = blockIdx.y), else null
    template <class Fn> __device__ __forceinline__ void run(const FlameDesc &d, int tile, Fn prefetch) const {
        if (threadIdx.x != 0 || by <= 0) return;
        const int t = tile + by;
        if (!ds) {
            if (t < ntiles) prefetch(d, t);
        } else {
            const int f = (int)blockIdx.y + t / ntiles;
            if (f < (int)gridDim.y) prefetch(ds[f], t % ntiles);
        }
    }
};

// Pass A: column k2 of the box.  Two lines per thread (V = float2): lane 0 is
// W(., k2), lane 1 conj W(., -k2); one line per thread: lines 2u and 2u+1 of
// the CTA are the two of its column u.
template <class R, class V, int A, int F, bool TMA>
__device__ __forceinline__ void stepA_body(const FlameDesc &d, int tile, const Ahead &ahead, const CUtensorMap *tm) {
    griddep_wait();
    using C = CplxT<R>;
    using PL = Plan3<A, F>;
    constexpr int NL = kLanes<V>, LPC = 2 / NL, SL = PL::slots(kSlotsPerWave<V>);
    extern __shared__ __align__(128) unsigned char smstep[];
    const StepArgs &a = d.a;
    const int G = blockDim.x / (PL::TS * LPC);
    // (two lines per thread: CTAs are whole lines)
    const Place s = NL == 2 ? place_all<PL::TS>() : place<PL::TS>(G * LPC), p = place<PL::TP>(G * LPC);
    const int ld1 = 2 * a.K1 + 1;
    const C *state = static_cast<const C *>(d.state);
    C *__restrict__ uv = static_cast<C *>(d.uv);
    CV<V> xs[PL::ES];
    {
        const int k2 = tile * G + s.line / LPC;
        const C *col = state + (size_t)k2 * ld1 + a.K1;
        const R s1 = scale1<R>(a), s2k2 = scale2<R>(a) * (R)k2;
#pragma unroll
        for (int r = 0; r < PL::ES; ++r) {
            xs[r] = CV<V>{vzero(V{}), vzero(V{})};
            if (r >= F && r < 2 * F) continue;  // padding: K1 < 2^A = F TS
            const int n = s.t + r * PL::TS, k1 = r < F ? n : n - PL::L;
            const bool in_box = s.on && k2 <= a.K2 && (r < F ? n <= a.K1 : k1 >= -a.K1);
            if (in_box && FLAME_IN(d.status, (long long)k2 * ld1 + a.K1 + k1, box_len(a), kSiteAState)) {
                C phi = col[k1];
                if (k1 == 0 && k2 == 0) phi = C{0, 0};
                const R f = s1 * (R)k1;
                const C da{-f * phi.y, f * phi.x}, db{s2k2 * phi.x, s2k2 * phi.y};
                if constexpr (NL == 2) {
                    xs[r] = pack2<R>(C{da.x - db.x, da.y - db.y}, C{da.x + db.x, da.y + db.y});
                } else {
                    const R sg = s.line & 1 ? (R)1 : (R)-1;
                    xs[r] = CV<V>{{fma_rn(sg, db.x, da.x)}, {fma_rn(sg, db.y, da.y)}};
                }
            }
        }
    }
    ahead.run(d, tile, [&](const FlameDesc &q, int t) {  // that tile's columns
        const int c = t * G, nc = min(G, q.a.K2 + 1 - c);
        if (nc > 0) l2_prefetch(static_cast<const C *>(q.state) + (size_t)c * ld1, (size_t)nc * ld1 * sizeof(C));
    });
    auto buf = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    CV<V> xp[PL::EP];
    inverse3<PL>(xs, xp, s, p, buf, tab3<R, A, F, C>(d.tw1));
    griddep_launch();
    const int k2 = tile * G + p.line / LPC;
    const bool valid = p.on && k2 <= a.K2;
    if constexpr (NL == 1) {
        const int f = p.line & 1;
        if constexpr (PL::TP % 2 == 0) {
#pragma unroll
            for (int i = 0; i < PL::EP; ++i) {
                const int n = p.t + i * PL::TP;
                const bool on = valid && FLAME_IN(d.status, w_index(n, k2, a.ldk) + 3, uv_len(a), kSiteAUv);
                st_w<R>(uv, n, k2, a.ldk, f, C{xp[i].re.x, f ? -xp[i].im.x : xp[i].im.x}, on);
            }
        } else if (valid) {  // lines of 12 F points: rows one by one
#pragma unroll
            for (int i = 0; i < PL::EP; ++i) {
                const int n = p.t + i * PL::TP;
                if (!FLAME_IN(d.status, w_index(n, k2, a.ldk) + 3, uv_len(a), kSiteAUv)) continue;
                C *e = uv + w_index(n, k2, a.ldk) + 2 * w_half<R>(k2, f);
                const C v{xp[i].re.x, f ? -xp[i].im.x : xp[i].im.x};
                if constexpr (sizeof(R) == 4) {
                    R *w = reinterpret_cast<R *>(e) + (n & 1);
                    w[0] = v.x;
                    w[2] = v.y;
                } else e[n & 1] = v;
            }
        }
    } else if constexpr (TMA) {
        // The column is parked in shared memory in uv's order (32 bytes a row
        // pair) and the copy engine writes the scattered sectors.
        __syncthreads();  // the transform's last exchange has been read
        static_assert(PL::TP % 2 == 0, "row pairs in adjacent threads");
        auto park = [&](int line) { return reinterpret_cast<float4 *>(smstep) + (size_t)line * SL; };
        const bool odd = threadIdx.x & 1;
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) {
            const float4 w = w_pair(xp[i], odd);
            if (p.on) park(p.line)[((p.t + i * PL::TP) & ~1) + w_half<R>(k2, odd)] = w;
        }
        fence_async_smem();
        __syncthreads();
        const bool aligned = (__cvta_generic_to_shared(smstep) & 127) == 0;
        if (aligned) {
            const int c = tile * G + s.line;
            if (s.on && s.t == 0 && c <= a.K2) {
                constexpr int BP = uv3_box_pairs(PL::L);
#pragma unroll 1
                for (int p0 = 0; p0 < PL::L / 2; p0 += BP)
                    if (FLAME_IN(d.status, c, a.ldk, kSiteATma) && FLAME_IN(d.status, p0, a.n1 >> 1, kSiteATma))
                        tma_store_3d(tm, park(s.line) + 2 * p0, 0, c, p0);
                bulk_commit_and_wait_read();
            }
        } else if (valid) {
            const float4 *q = park(p.line);
#pragma unroll
            for (int i = 0; i < PL::EP; ++i) {
                const int n = p.t + i * PL::TP;
                const size_t w = w_index(n, k2, a.ldk) + 2 * (n & 1);  // the halves as parked
                if (FLAME_IN(d.status, w + 1, uv_len(a), kSiteAUv)) *reinterpret_cast<float4 *>(uv + w) = q[n];
            }
        }
    } else {
        static_assert(PL::TP % 2 == 0, "row pairs in adjacent threads");
        const bool odd = threadIdx.x & 1;
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) {
            const float4 v = w_pair(xp[i], odd);
            const size_t w = w_index(p.t + i * PL::TP, k2, a.ldk) + 2 * w_half<R>(k2, odd);
            if (valid && FLAME_IN(d.status, w + 1, uv_len(a), kSiteAUv)) *reinterpret_cast<float4 *>(uv + w) = v;
        }
    }
}

// The inputs of the two half-length inverse transforms of a row of 2 L points
// at index n: the even grid points take W[n] + W[n - L], the odd ones
// (W[n] - W[n - L]) exp(2 pi i n / 2L) (harmonics L apart fold; for an index
// only one of them reaches the other is zero).  n = t + r TS, so
// exp(2 pi i n / 2L) = wt exp(i pi r / 3F): one table entry per thread and
// compile-time roots.
struct Roots24 {  // cos and sin of k pi / 12, k = 0 .. 11
    static constexpr double C1 = 0.965925826289068286749743199728897368, S1 = 0.258819045102520762348898837624048328;
    static constexpr double C2 = 0.866025403784438646763723170752936183, S2 = 0.5;
    static constexpr double C3 = 0.707106781186547524400844362104849039;
    static constexpr double c[12] = {1.0, C1, C2, C3, S2, S1, 0.0, -S1, -S2, -C3, -C2, -C1};
    static constexpr double s[12] = {0.0, S1, S2, C3, C2, C1, 1.0, C1, C2, C3, S2, S1};
};
// b exp(i pi r / ES), ES = 3, 6 or 12
template <int r, int ES, class C> __device__ __forceinline__ C mul_root24(C b) {
    using Real = decltype(C::x);
    constexpr int k = r * (12 / ES);
    constexpr Real cr = (Real)Roots24::c[k], ci = (Real)Roots24::s[k];
    if constexpr (k == 0) return b;
    else if constexpr (k == 6) return C{-b.y, b.x};
    else return C{fma_rn(b.x, cr, -(b.y * ci)), fma_rn(b.x, ci, b.y * cr)};
}

// G[k] and G[L - k] of a row from H[k] and H[L - k] of h[m] = g[2m] + i g[2m+1]
// (E = (H[k] + conj H[L-k]) / 2, O = (H[k] - conj H[L-k]) / 2i, w = exp(2 pi i
// k / 2L)): E + O conj w and conj(E - O conj w).
template <class V, class C> __device__ __forceinline__ void real_post(CV<V> h, CV<V> hc, C w, CV<V> &lo, CV<V> &hi) {
    using Real = decltype(C::x);
    const V hf = vbc_as((Real)0.5, V{});
    const CV<V> E{vmul(vadd(h.re, hc.re), hf), vmul(vsub(h.im, hc.im), hf)};
    const CV<V> O{vmul(vadd(h.im, hc.im), hf), vmul(vsub(hc.re, h.re), hf)};
    const CV<V> Ow = cmul_s(O, w.x, -w.y);
    lo = cadd(E, Ow);
    hi = CV<V>{vsub(E.re, Ow.re), vsub(Ow.im, E.im)};
}

// Bulk copy of a block (16-byte aligned, a multiple of 16 bytes) from global
// to shared memory by one thread, and the wait of all threads for it on the
// mbarrier `bar`, which the copying thread initialises: a CTA barrier has to
// come between.  The wait ends after a second; false: the block has not come.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, unsigned long long *bar, bool issue = true) {
    const unsigned sb = (unsigned)__cvta_generic_to_shared(bar), sd = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sb), "r"(bytes) : "memory");
    if (bytes && issue)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sd),
                     "l"(reinterpret_cast<unsigned long long>(src)), "r"(bytes), "r"(sb)
                     : "memory");
}
__device__ __forceinline__ bool bulk_wait(unsigned long long *bar) {
    const unsigned sb = (unsigned)__cvta_generic_to_shared(bar);
    const long long start = clock64();
    unsigned done = 0;
    do {
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(sb) : "memory");
    } while (!done && clock64() - start < 1LL << 31);
    return done;
}
// All threads, at the barrier behind the reads of the block: false, and the
// status says so, where some thread's wait ran out.  What the CTA read may not
// be the block then: it makes its part of the output NaN, so that a caller
// who does not ask for the status sees it too, and returns, behind one more
// bounded wait for the copy that may still be on its way into its shared memory.
__device__ __forceinline__ bool bulk_read(bool came, unsigned long long *bar, int *status) {
    if (__syncthreads_and(came)) return true;
    if (threadIdx.x == 0) atomicOr(status, 1 << kStatusTimeout);
    bulk_wait(bar);
    return false;
}

// Twiddles exp(2 pi i k / 2L) of the real post-processing, k = t + r TS: rows of
// 3072 points form them from one entry per thread and compile-time roots, as
// the inverse transforms' odd points do; shorter rows read the table, which is
// what keeps the step's rounding error at that of the public grid's rows.  1024x2048,
// increment (nonlinear only, flat spectrum): 3.379e-7 with roots, 3.354e-7 so,
// 3.376e-7 on the public grid; an ensemble of 96 443.4 -> 446.1 us a step,
// 1024x2048 level.  (Both from the table: 3.306e-7, but 460 us.)
template <int A> constexpr bool kPostRoots = A == kMaxA;

// Pass B, two lines per thread (FP32): one row pair per group of TS threads,
// the lanes its two rows.  The even and the odd points are two inverse
// transforms with an exchange buffer each, whose first passes run together as
// the row pair's W come out of shared memory; the even buffer then takes g at
// the even points, the odd one the forward transform of g, and the even one G
// on its way out (32 bytes of gk per column and row pair: 2/3 of a buffer).
// Bound by the latency between its barriers at two CTAs of 256 threads per SM
// (the shared-memory pipe is 42 % busy, the six exchanges most of it; issue 37 %;
// stalls per issue: barrier 2.5, loads 1.3, shared memory 1.0).  4096x8192 (1536 pairs of 3072-point
// rows): 123 -> 75 us, 1.99 TB/s of its 151 MB (three 4096-point transforms a
// row pair before; on this grid, 155 -> 136 us a step by this form).
template <class R, int A, bool TMA>
__device__ __forceinline__ void stepB2_body(const FlameDesc &d, int tile, const Ahead &ahead, const CUtensorMap *tm) {
    using V = float2;
    using C = CplxT<R>;
    using PL = Plan3<A, 4, A == kMaxA>;
    constexpr int L = PL::L, TS = PL::TS, TP = PL::TP, ES = PL::ES, SL = PL::slots(kSlotsPerWave<V>);
    extern __shared__ __align__(128) unsigned char smstep[];
    const StepArgs &a = d.a;
    const C *uv = static_cast<const C *>(d.uv);
    C *__restrict__ gk = static_cast<C *>(d.gk);
    const int G = blockDim.x / TS;
    const Place s = place_all<TS>(), p = place<TP>(G);
    const int pair = tile * G + s.line;
    const bool valid = s.on && pair < (a.n1 >> 1);
    // The CTA's row pairs (one contiguous block) come in by one bulk copy, into
    // the exchange buffers, which nothing uses yet.
    __shared__ __align__(8) unsigned long long loaded;
    if (threadIdx.x == 0) {
        const int np = min(G, (a.n1 >> 1) - tile * G);
        const size_t first = w_index(2 * tile * G, 0, a.ldk), len = (size_t)np * 4 * a.ldk;
        if (FLAME_IN(d.status, first + len - 1, uv_len(a), kSiteBUv))
            bulk_load(smstep, uv + first, (unsigned)(len * sizeof(C)), &loaded, !FLAME_STALL(a.flags));
        else bulk_load(smstep, uv, 0, &loaded);
    }
    ahead.run(d, tile, [&](const FlameDesc &q, int t) {  // that tile's row pairs
        const int p0 = t * G, np = min(G, (q.a.n1 >> 1) - p0);
        if (np > 0) l2_prefetch(static_cast<const C *>(q.uv) + w_index(2 * p0, 0, q.a.ldk), (size_t)np * 4 * q.a.ldk * sizeof(C));
    });
    auto even = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    auto odd = [&](int line) { return planes3<V, R>(smstep, G + line, SL); };
    const C *tw = tab3<R, A, 4, C>(d.twm);
    const C *P = static_cast<const C *>(d.twm) + tw3_real_offset<A>() + s.t;
    const C wt = __ldg(P);  // exp(2 pi i t / 2L)
    __syncthreads();  // the barrier's initialisation
    const bool came = bulk_wait(&loaded);

    CV<V> xs[ES];
    {
        // W at n = t + i TS (i < 8: K2 < 2^(A+1) = 8 TS) and at n - L (n = t + (i + 4) TS), both rows
        const float4 *src = reinterpret_cast<const float4 *>(smstep) + (size_t)s.line * 2 * a.ldk;  // two per k
        CV<V> up[8], um[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int n = s.t + i * TS, km = L - (s.t + (i + 4) * TS);
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f), m = q;
            if (valid && n <= a.K2) q = src[2 * n + w_half<R>(n, false)];
            if (valid && km <= a.K2) m = src[2 * km + w_half<R>(km, true)];
            up[i] = CV<V>{make_float2(q.x, q.y), make_float2(q.z, q.w)};
            um[i] = CV<V>{make_float2(m.x, m.y), make_float2(m.z, m.w)};
        }
        if (!bulk_read(came, &loaded, d.status)) {  // (a barrier: the block has been read)
            const R nan = (R)__int_as_float(0x7fc00000);
            for (int k = s.t; valid && k <= a.K2; k += TS)
                if (FLAME_IN(d.status, g_index(2 * pair, k, a.n1) + 1, gk_len(a), kSiteBGk))
                    *reinterpret_cast<float4 *>(gk + g_index(2 * pair, k, a.n1)) = make_float4(nan, nan, nan, nan);
            return;
        }
        CV<V> xo[ES];
        static_for<0, ES>([&](auto rc) {
            constexpr int r = decltype(rc)::value;
            constexpr int ip = r < 8 ? r : 0, im = r >= 4 ? r - 4 : 0;
            if constexpr (r < 4) xs[r] = xo[r] = up[ip];
            else if constexpr (r >= 8) xs[r] = um[im], xo[r] = CV<V>{vneg(um[im].re), vneg(um[im].im)};
            else xs[r] = cadd(up[ip], um[im]), xo[r] = csub(up[ip], um[im]);
        });
        inverse3_first<PL>(xs, s, even, tw);
        static_for<0, ES>([&](auto rc) {
            constexpr int r = decltype(rc)::value;
            const C w = mul_root24<r, ES>(wt);
            xo[r] = cmul_s(xo[r], w.x, w.y);
        });
        inverse3_first<PL>(xo, s, odd, tw);
    }
    __syncthreads();
    V g[PL::EP];  // |w|^2 at the even, then at the odd points of both rows
    V *hp = reinterpret_cast<V *>(even(p.line).p) + p.t;
#pragma unroll 1
    for (int parity = 0;; ++parity) {
        // (the loop's addresses are to be formed in it: formed before it they spill)
        Place q = p;
        asm volatile("" : "+r"(q.line), "+r"(q.t), "+l"(tw));
        CV<V> xp[PL::EP];
        inverse3_rest<PL>(xp, q, [&](int line) { return planes3<V, R>(smstep, parity * G + line, SL); }, tw);
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) g[i] = vfma(xp[i].re, xp[i].re, vmul(xp[i].im, xp[i].im));
        if (parity == 1) break;
        __syncthreads();  // the even buffers have been read
        if (p.on) {
#pragma unroll
            for (int i = 0; i < PL::EP; ++i) hp[i * TP] = g[i];
        }
    }
    // h[m] = g[2m] + i g[2m+1] of both rows
    CV<V> xp[PL::EP], hk[ES];
    if (p.on) {
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) xp[i] = CV<V>{hp[i * TP], g[i]};  // the thread's own slots
    }
    forward3<PL, false>(xp, hk, p, s, odd, tw);
    griddep_launch();
    // real-input post-processing: the pairs (k, L - k), k <= L/2
    C post[ES / 2];  // exp(2 pi i k / 2L)
    static_for<0, ES / 2>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        post[r] = kPostRoots<A> ? mul_root24<r, ES>(wt) : r == 0 ? wt : __ldg(P + r * TS);
    });
    __syncthreads();
    const Planes<V> sm = odd(s.line);
    if (s.on) {
#pragma unroll
        for (int r = ES / 2; r < ES; ++r) sm.st_raw(s.t + r * TS, hk[r]);
        if (s.t == 0) sm.st_raw(0, hk[0]);
    }
    __syncthreads();
    const bool staged = TMA && (__cvta_generic_to_shared(smstep) & 127) == 0;
    float4 *hs = even(s.line).p;  // g has been read
    auto emit = [&](int k, CV<V> Y) {
        const float4 v = make_float4(Y.re.x, Y.im.x, Y.re.y, Y.im.y);  // rows 2p, 2p+1
        if (staged) hs[k] = v;
        else if (FLAME_IN(d.status, g_index(2 * pair, k, a.n1) + 1, gk_len(a), kSiteBGk))
            *reinterpret_cast<float4 *>(gk + g_index(2 * pair, k, a.n1)) = v;
    };
    if (valid) {
        static_for<0, ES / 2>([&](auto rc) {
            constexpr int r = decltype(rc)::value;
            const int k = s.t + r * TS, kc = L - k;
            if (k <= a.K2 || kc <= a.K2) {
                CV<V> lo, hi;
                real_post(hk[r], sm.ld_raw(k == 0 ? 0 : kc), post[r], lo, hi);
                if (k <= a.K2) emit(k, lo);
                if (kc <= a.K2) emit(kc, hi);
            }
        });
        // k = L/2 is its own partner: G = conj H
        if (s.t == 0 && L / 2 <= a.K2) emit(L / 2, CV<V>{hk[ES / 2].re, vneg(hk[ES / 2].im)});
    }
    if constexpr (TMA) {
        if (staged) {
            fence_async_smem();
            __syncthreads();
            if (s.t == 0 && valid) {
                const int nq = (a.ldk + 1) >> 1, BQ = gk_box_pairs(a.ldk);
#pragma unroll 1
                for (int q0 = 0; q0 < nq; q0 += BQ)
                    if (FLAME_IN(d.status, pair, a.n1 >> 1, kSiteBTma) && FLAME_IN(d.status, q0, (gk_len(a) / a.n1) >> 1, kSiteBTma))
                        tma_store_3d(tm, hs + 2 * q0, 0, pair, q0);
                bulk_commit_and_wait_read();
            }
        }
    }
}

// Pass B, one line per thread: RW rows per unit (2, or 1 for FP64 rows whose
// pair does not fit in shared memory), lines 2 q + s = the points 2m + s of
// row q in the inverse transforms, line q = row q in the forward one.
template <class R, int A, int F, int RW>
__device__ __forceinline__ void stepB1_body(const FlameDesc &d, int unit0) {
    using V = typename OneOf<R>::type;
    using C = CplxT<R>;
    using PL = Plan3<A, F>;
    constexpr int L = PL::L, TS = PL::TS, TP = PL::TP, ES = PL::ES, SL = PL::slots(kSlotsPerWave<V>);
    extern __shared__ __align__(128) unsigned char smstep[];
    const StepArgs &a = d.a;
    const C *uv = static_cast<const C *>(d.uv);
    C *__restrict__ gk = static_cast<C *>(d.gk);
    const int U = blockDim.x / (2 * RW * TS), lines = 2 * RW * U;  // units of the CTA
    const Place s = place<TS>(lines), p = place<TP>(lines);
    auto buf = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    const C *tw = tab3<R, A, F, C>(d.twm);
    const C *P = static_cast<const C *>(d.twm) + tw3_real_offset<A>();
    const int first = unit0 * U * RW;  // the CTA's first row
    CV<V> xs[ES];
    {
        const int row = first + (s.line >> 1);
        const bool odd = s.line & 1, valid = s.on && row < a.n1;
#pragma unroll
        for (int r = 0; r < ES; ++r) {
            const int n = s.t + r * TS, km = L - n;
            C up{0, 0}, um{0, 0};
            // loads without branches (element 0 where there is none): a forced
            // 512x1024 run 596 -> 579 us
            if (r < 2 * F) {
                const bool in = valid && n <= a.K2 && FLAME_IN(d.status, w_index(row, n, a.ldk) + 3, uv_len(a), kSiteBUv);
                const C v = ld_w<R>(uv, in ? row : 0, in ? n : 0, a.ldk, false);
                if (in) up = v;
            }
            if (r >= F) {
                const bool in = valid && km <= a.K2 && FLAME_IN(d.status, w_index(row, km, a.ldk) + 3, uv_len(a), kSiteBUv);
                const C v = ld_w<R>(uv, in ? row : 0, in ? km : 0, a.ldk, true);
                if (in) um = v;
            }
            C z{up.x + um.x, up.y + um.y};
            if (odd) {
                const C o{up.x - um.x, up.y - um.y}, w = __ldg(P + n);  // exp(2 pi i n / 2L)
                z = C{fma_rn(o.x, w.x, -(o.y * w.y)), fma_rn(o.x, w.y, o.y * w.x)};
            }
            xs[r] = CV<V>{{z.x}, {z.y}};
        }
    }
    CV<V> xp[PL::EP];
    inverse3<PL>(xs, xp, s, p, buf, tw);
    R *h = reinterpret_cast<R *>(smstep + (size_t)lines * SL * 2 * sizeof(R));  // g of row q at h[2 L q + j]
    if (p.on) {
#pragma unroll
        for (int i = 0; i < PL::EP; ++i)
            h[2 * L * (p.line >> 1) + 2 * (p.t + i * TP) + (p.line & 1)] =
                fma_rn(xp[i].re.x, xp[i].re.x, xp[i].im.x * xp[i].im.x);
    }
    __syncthreads();
    const int rows = RW * U;
    const Place fp{p.line, p.t, p.line < rows}, fs{s.line, s.t, s.line < rows};
    if (fp.on) {
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) {
            const C g = reinterpret_cast<const C *>(h)[L * fp.line + fp.t + i * TP];
            xp[i] = CV<V>{{g.x}, {g.y}};
        }
    }
    forward3<PL, true>(xp, xs, fp, fs, buf, tw);
    griddep_launch();
    __syncthreads();
    const int row = first + fs.line;
    const Planes<V> sm = buf(fs.line);
    if (fs.on) {
#pragma unroll
        for (int r = 0; r < ES; ++r) {
            if (TS * (r + 1) > L / 2) sm.st_raw(fs.t + r * TS, xs[r]);
        }
        if (fs.t == 0) sm.st_raw(0, xs[0]);
    }
    __syncthreads();
    if (!fs.on || row >= a.n1) return;
    auto emit = [&](int k, CV<V> Y) {
        const size_t i = g_index(row, k, a.n1);
        if (FLAME_IN(d.status, i, gk_len(a), kSiteBGk)) gk[i] = C{Y.re.x, Y.im.x};
    };
#pragma unroll
    for (int r = 0; r < ES; ++r) {
        if (TS * r > L / 2) continue;
        const int k = fs.t + r * TS, kc = L - k;
        if (k <= L / 2 && (k <= a.K2 || kc <= a.K2)) {
            CV<V> lo, hi;
            real_post(xs[r], sm.ld_raw(k == 0 ? 0 : kc), __ldg(P + k), lo, hi);
            if (k <= a.K2) emit(k, lo);
            if (kc <= a.K2 && kc != k) emit(kc, hi);
        }
    }
}

// Pass C: columns 2 u, 2 u + 1 of gk; two lines per thread (lanes) or lines
// 2u, 2u+1 of the CTA.  FUSE_A: pass A of the next step on the updated
// columns (two lines per thread, tensor stores).
template <class R, class V, int A, int F, bool GEN, bool FUSE_A = false>
__device__ __forceinline__ void stepC_body(const FlameDesc &d, int tile, const Ahead &ahead, const CUtensorMap *tm) {
    griddep_wait();
    using C = CplxT<R>;
    using PL = Plan3<A, F>;
    constexpr int NL = kLanes<V>, LPC = 2 / NL, L = PL::L, TS = PL::TS, TP = PL::TP, SL = PL::slots(kSlotsPerWave<V>);
    static_assert(!FUSE_A || NL == 2, "the fused pass is a two-line kernel");
    extern __shared__ __align__(128) unsigned char smstep[];
    const StepArgs &a = d.a;
    const C *gk = static_cast<const C *>(d.gk);
    const C *state = static_cast<const C *>(d.state);
    const C *tw = tab3<R, A, F, C>(d.tw1);
    const int G = blockDim.x / (TS * LPC);
    const Place s = NL == 2 ? place_all<TS>() : place<TS>(G * LPC), p = place<TP>(G * LPC);
    const int ld1 = 2 * a.K1 + 1;
    const CoefR<R> cfs = load_coef<R>(d.coef);  // derived by pass B
    CV<V> xp[PL::EP];
    {
        // the line's (first) column
        const int c = 2 * (tile * G + p.line / LPC) + (NL == 1 ? p.line & 1 : 0);
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) {
            const int n = p.t + i * TP;
            const bool in = p.on && c <= a.K2 && FLAME_IN(d.status, g_index(n, c, L) + (NL == 2 ? 2 : 0), gk_len(a), kSiteCGk);
            const C *q = gk + g_index(n, c, L);
            const C q0 = in ? *q : C{0, 0};
            if constexpr (NL == 2) xp[i] = pack2<R>(q0, in && c < a.K2 ? q[2] : C{0, 0});
            else xp[i] = CV<V>{{q0.x}, {q0.y}};
        }
    }
    ahead.run(d, tile, [&](const FlameDesc &q, int t) {  // that tile's column pairs
        const int c = 2 * t * G, nc = min(2 * G, q.a.K2 + 1 - c);
        if (nc > 0) {
            l2_prefetch(static_cast<const C *>(q.gk) + (size_t)c * L, (size_t)nc * L * sizeof(C));
            l2_prefetch(static_cast<const C *>(q.state) + (size_t)c * ld1, (size_t)nc * ld1 * sizeof(C));
        }
    });
    auto buf = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    CV<V> xs[PL::ES];
    forward3<PL, true>(xp, xs, p, s, buf, tw);

    const int c0 = 2 * (tile * G + s.line / LPC) + (NL == 1 ? s.line & 1 : 0);
    const C *col = state + (size_t)c0 * ld1 + a.K1;
    C *ocol = static_cast<C *>(d.state_out) + (size_t)c0 * ld1 + a.K1;
    // the band entries of this thread: r < F (k1 = n) and r >= 2F (k1 = n - L);
    // read after the transform, from the L2 window over the state
    auto k1_of = [&](int i) { return i < F ? s.t + i * TS : s.t + (i + F) * TS - L; };
    auto in_box = [&](int i, int side) {
        const int k1 = k1_of(i);
        return s.on && c0 + side <= a.K2 && (i < F ? k1 <= a.K1 : k1 >= -a.K1);
    };
    griddep_launch();  // (behind the loads, which it would hold back)
    const bool lin = !(a.flags & kNonlinearOnly), nl = !(a.flags & kLinearOnly);
    const EpiArgs<R> ea{cfs, scale1<R>(a), scale2<R>(a), GEN ? d.stage : kStageEuler, lin, nl};
    const C *fcol = GEN && d.forcing ? static_cast<const C *>(d.forcing) + (size_t)c0 * ld1 + a.K1 : nullptr;
    C *scol = GEN && d.save ? static_cast<C *>(d.save) + (size_t)c0 * ld1 + a.K1 : nullptr;
    int bad = 0;
    C nphi[2 * F][NL];  // the updated entries (kept for the fused pass A)
#pragma unroll
    for (int side = 0; side < NL; ++side) {
        C phi[2 * F];
#pragma unroll
        for (int i = 0; i < 2 * F; ++i) {
            const bool in = in_box(i, side) && FLAME_IN(d.status, (long long)(c0 + side) * ld1 + a.K1 + k1_of(i), box_len(a), kSiteCState);
            phi[i] = in ? col[(long)side * ld1 + k1_of(i)] : C{0, 0};
        }
#pragma unroll
        for (int i = 0; i < 2 * F; ++i) {
            nphi[i][side] = C{0, 0};
            const int k1 = k1_of(i), k2 = c0 + side;
            if (!in_box(i, side) || (k2 == 0 && k1 < 0)) continue;  // k2 = 0, k1 < 0: the mirror of +k1
            const CV<V> x = xs[i < F ? i : i + F];
            C gh;
            if constexpr (NL == 2) gh = side == 0 ? lane0<R>(x) : lane1<R>(x);
            else gh = C{x.re.x, x.im.x};
            const int off = side * ld1;
            update_entry<R, GEN>(d, ea, k1, k2, gh, phi[i], ocol + off, fcol ? fcol + off : nullptr,
                                 scol ? scol + off : nullptr, nphi[i][side], bad);
        }
    }
    if (bad) atomicOr(d.status, 1 << kStatusNonfinite);
    if constexpr (FUSE_A) {
        // The k2 = 0 column's k1 < 0 half was written by other threads (the
        // conjugate mirror) and is read back after the barrier.
        __syncthreads();
        if (c0 == 0 && s.on) {
#pragma unroll
            for (int i = F; i < 2 * F; ++i)
                if (k1_of(i) >= -a.K1 && FLAME_IN(d.status, a.K1 + k1_of(i), box_len(a), kSiteCState)) nphi[i][0] = ocol[k1_of(i)];
        }
        auto park = [&](int line) { return reinterpret_cast<float4 *>(smstep) + (size_t)line * SL; };
        const bool odd = threadIdx.x & 1;
        C *uv = static_cast<C *>(d.uv);
        const bool aligned = (__cvta_generic_to_shared(smstep) & 127) == 0;
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            const int k2 = c0 + side;
            const R s2k2 = ea.s2 * (R)k2;
#pragma unroll
            for (int r = 0; r < PL::ES; ++r) {
                xs[r] = CV<V>{vzero(V{}), vzero(V{})};
                if (r >= F && r < 2 * F) continue;
                const int i = r < F ? r : r - F;
                if (!in_box(i, side)) continue;
                C ph = side == 0 ? nphi[i][0] : nphi[i][1];
                if (k1_of(i) == 0 && k2 == 0) ph = C{0, 0};
                const R f = ea.s1 * (R)k1_of(i);
                const C da{-f * ph.y, f * ph.x}, db{s2k2 * ph.x, s2k2 * ph.y};
                xs[r] = pack2<R>(C{da.x - db.x, da.y - db.y}, C{da.x + db.x, da.y + db.y});
            }
            __syncthreads();
            inverse3<PL>(xs, xp, s, p, buf, tw);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < PL::EP; ++i) {
                const float4 w = w_pair(xp[i], odd);
                if (p.on) park(p.line)[((p.t + i * TP) & ~1) + w_half<R>(k2, odd)] = w;
            }
            fence_async_smem();
            __syncthreads();
            if (aligned) {
                if (s.on && s.t == 0 && k2 <= a.K2) {
                    constexpr int BP = uv3_box_pairs(L);
#pragma unroll 1
                    for (int p0 = 0; p0 < L / 2; p0 += BP)
                        if (FLAME_IN(d.status, k2, a.ldk, kSiteCAUv) && FLAME_IN(d.status, p0, a.n1 >> 1, kSiteCAUv))
                            tma_store_3d(tm, park(s.line) + 2 * p0, 0, k2, p0);
                    bulk_commit_and_wait_read();
                }
            } else if (p.on) {
                const int kp = 2 * (tile * G + p.line) + side;
                const float4 *q = park(p.line);
                for (int i = 0; i < PL::EP; ++i) {
                    const int n = p.t + i * TP;
                    const size_t w = w_index(n, kp, a.ldk) + 2 * (n & 1);
                    if (kp <= a.K2 && FLAME_IN(d.status, w + 1, uv_len(a), kSiteCAUv)) *reinterpret_cast<float4 *>(uv + w) = q[n];
                }
            }
        }
    }
}

// ----------------------------------------------------------------------------
// Twiddle tables of a line of 3 * 2^A points (FP64, rounded once).  The angle
// is reduced to an eighth of a turn in integers first: 3 * 2^a is no power of
// two, and 2 pi times a rounded fraction would cost the last bit or two.
// ----------------------------------------------------------------------------
__device__ inline void cos_sin_of(long num, long den, double &c, double &s) {  // 2 pi num / den
    num %= den;  // den is even
    const bool flip = 2 * num > den;  // (half, 1): the conjugate of den - num
    if (flip) num = den - num;
    const bool left = 4 * num > den;  // (quarter, half]: mirrored at the imaginary axis;
    if (left) num = den - 2 * num;    // in units of 1 / (2 den) from here on
    else num = 2 * num;
    const bool swap = 4 * num > den;  // (eighth, quarter]
    if (swap) num = den / 2 - num;
    double sv, cv;
    sincospi((double)num / (double)den, &sv, &cv);  // angle 2 pi num / (2 den)
    c = swap ? sv : cv;
    s = swap ? cv : sv;
    if (left) c = -c;
    if (flip) s = -s;
}
// One entry per thread: an FP64 sine and cosine take microseconds.
template <class R, int A> __global__ void k_twiddles3(CplxT<R> *tab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    long num = -1, den = 1;
    auto table = [&](auto fc, auto ic) {
        constexpr int F = decltype(fc)::value;
        constexpr bool INV = decltype(ic)::value;
        if constexpr (A >= (F == 4 ? 4 : F == 2 ? 3 : 2)) {
            using PL = Plan3<A, F>;
            static_for<1, PL::NQ + 1>([&](auto sc) {
                constexpr int S = decltype(sc)::value, r = PL::template radix<INV>(S), Ns = PL::template stride<INV>(S);
                const int j = i - (tw3_offset<A, F>() + PL::template tw_offset<INV>(S));
                if (j >= 0 && j < (r - 1) * Ns) {
                    num = (long)(j / Ns + 1) * (j % Ns);
                    den = r * Ns;
                }
            });
        }
    };
    static_for<0, 3>([&](auto lf) {
        constexpr int F = 1 << decltype(lf)::value;
        table(std::integral_constant<int, F>{}, std::true_type{});
        table(std::integral_constant<int, F>{}, std::false_type{});
    });
    if (i >= tw3_real_offset<A>() && i < tw3_alloc_len<A>()) {
        num = i - tw3_real_offset<A>();
        den = 6L << A;
    }
    if (num < 0) return;
    double c, s;
    cos_sin_of(num, den, c, s);
    tab[i] = CplxT<R>{(R)c, (R)s};
}

// ----------------------------------------------------------------------------
// Kernels: one flame (descriptor by value) or the flames of one ensemble class
// (descriptor array, flame = blockIdx.y)
// ----------------------------------------------------------------------------
// Passes A and C of one flame may be launched over part of their tiles
// (flame_step_host); the launch that holds tile 0 of pass C has the extra CTA.
// Threads of a CTA, and CTAs per SM to allot registers for: 128 registers for
// two lines of 16 points a thread; one line of EP points takes about 4 EP
// (FP32) or 8 EP (FP64) less than 64 besides.
template <class R, class V, int A, int F, int LINES> constexpr int kStepThreads =
    kLanes<V> == 2 ? 256 : (LINES * Plan3<A, F>::TS > 32 ? LINES * Plan3<A, F>::TS : 32);
template <class R, class V, int A, int F, int LINES> constexpr int kStepBlocks =
    kLanes<V> == 2 ? 2 : (sizeof(R) == 8 ? (F == 4 ? 512 : F == 2 ? 640 : 1024) : 1024) / kStepThreads<R, V, A, F, LINES>;

template <class R, class V, int A, int F>
__global__ void __launch_bounds__(kStepThreads<R, V, A, F, 2>, kStepBlocks<R, V, A, F, 2>) k_stepA(FlameDesc d, int pf) {
    stepA_body<R, V, A, F, false>(d, blockIdx.x + d.tile0, Ahead{pf, (int)gridDim.x + d.tile0, nullptr}, nullptr);
}
template <class R, int A>
__global__ void __launch_bounds__(256, 2) k_stepAt(FlameDesc d, int pf, const __grid_constant__ CUtensorMap tm) {
    stepA_body<R, float2, A, 4, true>(d, blockIdx.x + d.tile0, Ahead{pf, (int)gridDim.x + d.tile0, nullptr}, &tm);
}
template <class R, class V, int A, int F>
__global__ void __launch_bounds__(kStepThreads<R, V, A, F, 2>, kStepBlocks<R, V, A, F, 2>) k_stepA_n(const FlameDesc *__restrict__ ds, int pf) {
    stepA_body<R, V, A, F, false>(ds[blockIdx.y], blockIdx.x, Ahead{pf, (int)gridDim.x, ds}, nullptr);
}

template <class R, int A>
__global__ void __launch_bounds__(256, 2) k_stepB(FlameDesc d, int pf) {
    if (blockIdx.x == 0) return coef_cta<R>(d);
    griddep_wait();
    stepB2_body<R, A, false>(d, blockIdx.x - 1, Ahead{pf, (int)gridDim.x - 1, nullptr}, nullptr);
}
template <class R, int A>
__global__ void __launch_bounds__(256, 2) k_stepBt(FlameDesc d, int pf, const __grid_constant__ CUtensorMap tm) {
    if (blockIdx.x == 0) return coef_cta<R>(d);
    griddep_wait();
    stepB2_body<R, A, true>(d, blockIdx.x - 1, Ahead{pf, (int)gridDim.x - 1, nullptr}, &tm);
}
template <class R, int A> __global__ void __launch_bounds__(256, 2) k_stepB_n(const FlameDesc *__restrict__ ds, int pf) {
    if (blockIdx.x == 0) return coef_cta<R>(ds[blockIdx.y]);
    griddep_wait();
    stepB2_body<R, A, false>(ds[blockIdx.y], blockIdx.x - 1, Ahead{pf, (int)gridDim.x - 1, ds}, nullptr);
}
template <class R, int A, int F, int RW>
__global__ void __launch_bounds__(kStepThreads<R, typename OneOf<R>::type, A, F, 2 * RW>, kStepBlocks<R, typename OneOf<R>::type, A, F, 2 * RW>)
 k_stepB1(FlameDesc d) {
    if (blockIdx.x == 0) return coef_cta<R>(d);
    griddep_wait();
    stepB1_body<R, A, F, RW>(d, blockIdx.x - 1);
}
template <class R, int A, int F, int RW>
__global__ void __launch_bounds__(kStepThreads<R, typename OneOf<R>::type, A, F, 2 * RW>, kStepBlocks<R, typename OneOf<R>::type, A, F, 2 * RW>)
 k_stepB1_n(const FlameDesc *__restrict__ ds) {
    if (blockIdx.x == 0) return coef_cta<R>(ds[blockIdx.y]);
    griddep_wait();
    stepB1_body<R, A, F, RW>(ds[blockIdx.y], blockIdx.x - 1);
}

// Plain pass C with THREE: 80 registers a thread, three CTAs per SM, for launches
// of several waves (three_ctas in flame_step_ops.cuh).
template <class R, class V, int A, int F, bool GEN, bool THREE> constexpr int kStepBlocksC =
    THREE ? 3 : kStepBlocks<R, V, A, F, 2>;
template <class R, class V, int A, int F, bool GEN, bool THREE = false>
__global__ void __launch_bounds__(kStepThreads<R, V, A, F, 2>, kStepBlocksC<R, V, A, F, GEN, THREE>) k_stepC(FlameDesc d, int pf) {
    const int extra = d.tile0 == 0 ? 1 : 0;
    if (extra && blockIdx.x == 0) return finish_cta<R, GEN, true>(d);
    stepC_body<R, V, A, F, GEN>(d, blockIdx.x - extra + d.tile0, Ahead{pf, (int)gridDim.x - extra + d.tile0, nullptr}, nullptr);
}
template <class R, class V, int A, int F, bool GEN, bool THREE = false>
__global__ void __launch_bounds__(kStepThreads<R, V, A, F, 2>, kStepBlocksC<R, V, A, F, GEN, THREE>) k_stepC_n(const FlameDesc *__restrict__ ds, int pf) {
    if (blockIdx.x == 0) return finish_cta<R, GEN, true>(ds[blockIdx.y]);
    stepC_body<R, V, A, F, GEN>(ds[blockIdx.y], blockIdx.x - 1, Ahead{pf, (int)gridDim.x - 1, ds}, nullptr);
}
template <class R, int A, bool GEN>
__global__ void __launch_bounds__(256, 2) k_stepCA(FlameDesc d, int pf, const __grid_constant__ CUtensorMap tm) {
    if (blockIdx.x == 0) return finish_cta<R, GEN, true>(d);
    stepC_body<R, float2, A, 4, GEN, true>(d, blockIdx.x - 1, Ahead{pf, (int)gridDim.x - 1, nullptr}, &tm);
}

}  // namespace flame
