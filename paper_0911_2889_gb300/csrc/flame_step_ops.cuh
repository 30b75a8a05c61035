// flame_step_ops.cuh -- launch geometry and launchers of the step's passes on
// the alias-free grid (flame_step.cuh).  FP64 is instantiated by
// flame_step_f64.cu; the FP32 launchers are split over flame_step_f32_*.cu so
// that their kernels compile in parallel.
#pragma once

#include <algorithm>

#include "flame_launch.cuh"
#include "flame_step.cuh"

namespace flame {

// Two lines per thread: FP32 lines of 192 points and more.  Shorter lines
// have too few pairs to fill warps, and FP64 has no paired instructions.
template <class R> constexpr bool two_line(int a) { return sizeof(R) == 4 && a >= 6; }
// One line per thread: all of FP64, and FP32 up to 1536 points (a pair of
// 3072-point rows would not leave shared memory for a second CTA).
template <class R> constexpr bool one_line(int a) { return sizeof(R) == 8 || a <= 9; }
// Points per thread of the one-line kernels (4 F, spectral end 3 F).  FP64: a warp
// instruction holds its SM quarter for some 68 cycles, so short lines spread
// over more warps (256x512: 28.6 us a step with F = 1 for 192 points, 38.9 with
// 2; 128x256 21.6 against 33.7), and long ones take the plan with the fewest
// twiddles (1024x2048: 254 us with F = 4, 258 with 2).
template <class R> constexpr int one_line_f(int a) {
    if (sizeof(R) == 8) return a <= 6 ? 1 : a <= 7 ? 2 : 4;
    return a <= 5 ? 1 : a <= 8 ? 2 : 4;
}
// FLAME_FP64_POINTS=8: the FP64 lines of up to 96 points with 8 points per
// thread instead of 4 (read at every launch, so tests can run both)
static bool fp64_points8() {
    const char *v = getenv("FLAME_FP64_POINTS");
    return v && strcmp(v, "8") == 0;
}
// rows per unit of the one-line pass B: FP32 a pair where its lines fit 512
// threads and its buffers shared memory, else one.  FP64 one: it is bound by
// the FP64 units of the fullest SM, and single rows spread better (512x1024:
// 192 pairs leave 41 of 152 SMs with two).
template <class R, int A, int F> constexpr int rows_of() {
    if (sizeof(R) == 8) return 1;
    using V = typename OneOf<R>::type;
    const size_t pair = exchange_bytes<R, V, Plan3<A, F>>(4) + (size_t)4 * (3 << A) * sizeof(R);
    return 4 * Plan3<A, F>::TS <= 512 && pair <= kSmemBudget ? 2 : 1;
}

// calls f(A, F) for a one-line kernel of lines of 3 * 2^a points
template <class R, class Fn> static void with_one_line(int a, Fn &&f) {
    with_a(a, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        if constexpr (one_line<R>(A)) {
            if constexpr (sizeof(R) == 8 && A >= 3 && A <= 5) {
                if (fp64_points8()) {
                    f(ac, std::integral_constant<int, 2>{});
                    return;
                }
            }
            f(ac, std::integral_constant<int, one_line_f<R>(A)>{});
        }
    });
}
template <class Fn> static void with_two_line(int a, Fn &&f) { with_a<6>(a, f); }

// CTA of a two-line kernel: line pairs of 2^a / 4 threads each, up to 256
// threads, fewer pairs where a grid would not span two CTAs per SM.
static Geom geom_two_line(int a, int nlines, size_t per_line) {
    const int T = 1 << (a - 2);
    int G = T >= 256 ? 1 : 256 / T;
    while (G > 1 && G * per_line > kSmemBudget) G >>= 1;
    while (G > 1 && (nlines + G - 1) / G < 2 * sm_count()) G >>= 1;
    return Geom{G * T, (nlines + G - 1) / G, ((G * per_line + 127) & ~(size_t)127)};
}
template <int A> static size_t pair_bytes() { return exchange_bytes<float, float2, Plan3<A, 4>>(1); }
// pass B's two-line CTA: two exchange buffers per row pair
template <int A> static Geom geom_b2(int npairs) { return geom_two_line(A, npairs, 2 * pair_bytes<A>()); }
// CTA of a one-line kernel: units of `lines` lines, as many as fill a warp
template <class R, int A, int F> static Geom geom_one_line(int units, int lines, size_t extra) {
    using PL = Plan3<A, F>;
    using V = typename OneOf<R>::type;
    const int T = lines * PL::TS, U = T >= 32 ? 1 : 32 / T;
    return Geom{U * T, (units + U - 1) / U, exchange_bytes<R, V, PL>(U * lines) + U * extra};
}
template <class R, int A, int F> static Geom geom_b1(int n1) {
    constexpr int RW = rows_of<R, A, F>();
    return geom_one_line<R, A, F>(n1 / RW, 2 * RW, (size_t)RW * 2 * (3 << A) * sizeof(R));
}

template <class R>
cudaError_t Ops<R>::init_twiddles3(C *tab, int a, cudaStream_t s) {
    cudaError_t e = cudaErrorInvalidValue;
    with_a(a, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        e = launch_k(k_twiddles3<R, A>, dim3((tw3_alloc_len<A>() + 127) / 128), 128, 0, s, tab);
    });
    return e;
}

template <class R> cudaError_t Ops<R>::init_kappa(R *kap, const StepArgs &a, cudaStream_t s) {
    const long n = (long)(2 * a.K1 + 1) * a.ldk;
    return launch_k(k_kappa<R>, dim3((unsigned)std::min<long>((n + 255) / 256, 8L * sm_count())), 256, 0, s, kap, a);
}

// variant: kVariantTma = the tensor-store write-out through uv_map (two-line
// kernels), kVariantOneLine = one line per thread, others: direct stores
template <class R>
cudaError_t Ops<R>::passA(const FlameDesc &d, cudaStream_t s, int variant, const CUtensorMap *uv_map) {
    cudaError_t err = cudaErrorInvalidValue;
    const int ncol = d.a.K2 + 1;
    if (!two_line<R>(d.a.la) || (variant == kVariantOneLine && one_line<R>(d.a.la))) {
        with_one_line<R>(d.a.la, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value;
            using V = typename OneOf<R>::type;
            const Geom g = geom_one_line<R, A, F>(ncol, 2, 0);
            err = launch_s(d.l2_state, pdl_on(sizeof(R) == 8, d.a), k_stepA<R, V, A, F>, dim3(d.tiles ? d.tiles : g.blocks), g.threads, g.smem, s, d, 0);
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) with_two_line(d.a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_two_line(A, ncol, pair_bytes<A>());
        const dim3 grid(d.tiles ? d.tiles : g.blocks);
        if (variant == kVariantTma && uv_map) {
            const int pf = resident_ctas((const void *)k_stepAt<R, A>, g);
            err = launch_s(d.l2_state, pdl_on(sizeof(R) == 8, d.a), k_stepAt<R, A>, grid, g.threads, g.smem, s, d, pf, *uv_map);
        } else {
            const int pf = resident_ctas((const void *)k_stepA<R, float2, A, 4>, g);
            err = launch_s(d.l2_state, pdl_on(sizeof(R) == 8, d.a), k_stepA<R, float2, A, 4>, grid, g.threads, g.smem, s, d, pf);
        }
    });
    return err;
}
template <class R>
cudaError_t Ops<R>::passA_batch(const FlameDesc *ds, int n, const StepArgs &a, cudaStream_t s, int variant) {
    cudaError_t err = cudaErrorInvalidValue;
    if (!two_line<R>(a.la) || (variant == kVariantOneLine && one_line<R>(a.la))) {
        with_one_line<R>(a.la, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value;
            const Geom g = geom_one_line<R, A, F>(a.K2 + 1, 2, 0);
            err = launch_k(k_stepA_n<R, typename OneOf<R>::type, A, F>, dim3(g.blocks, n), g.threads, g.smem, s, ds, 0);
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) with_two_line(a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_two_line(A, n * (a.K2 + 1), pair_bytes<A>());
        const int G = g.threads >> (A - 2);
        const int pf = resident_ctas((const void *)k_stepA_n<R, float2, A, 4>, g);
        err = launch_k(k_stepA_n<R, float2, A, 4>, dim3((a.K2 + G) / G, n), g.threads, g.smem, s, ds, pf);
    });
    return err;
}

// variant: kVariantTmaB = the tensor-store write-out through gk_map (two-line
// kernels), kVariantOneLineB = one line per thread, others: direct stores
template <class R>
cudaError_t Ops<R>::passB(const FlameDesc &d, cudaStream_t s, int variant, const CUtensorMap *gk_map) {
    cudaError_t err = cudaErrorInvalidValue;
    const L2Window none{nullptr, 0, 0.f};
    if (!two_line<R>(d.a.lb) || (variant == kVariantOneLineB && one_line<R>(d.a.lb))) {
        with_one_line<R>(d.a.lb, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value, RW = rows_of<R, A, F>();
            const Geom g = geom_b1<R, A, F>(d.a.n1);
            err = launch_s(none, pdl_on(sizeof(R) == 8, d.a), k_stepB1<R, A, F, RW>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) with_two_line(d.a.lb, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_b2<A>(d.a.n1 / 2);
        if ((variant == kVariantTmaB || variant == kVariantTmaB4) && gk_map) {
            const int pf = resident_ctas((const void *)k_stepBt<R, A>, g);
            err = launch_s(none, pdl_on(sizeof(R) == 8, d.a), k_stepBt<R, A>, dim3(g.blocks + 1), g.threads, g.smem, s, d, pf, *gk_map);
        } else {
            const int pf = resident_ctas((const void *)k_stepB<R, A>, g);
            err = launch_s(none, pdl_on(sizeof(R) == 8, d.a), k_stepB<R, A>, dim3(g.blocks + 1), g.threads, g.smem, s, d, pf);
        }
    });
    return err;
}
template <class R>
cudaError_t Ops<R>::passB_batch(const FlameDesc *ds, int n, const StepArgs &a, cudaStream_t s, int variant) {
    cudaError_t err = cudaErrorInvalidValue;
    if (!two_line<R>(a.lb) || (variant == kVariantOneLineB && one_line<R>(a.lb))) {
        with_one_line<R>(a.lb, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value, RW = rows_of<R, A, F>();
            const Geom g = geom_b1<R, A, F>(a.n1);
            err = launch_k(k_stepB1_n<R, A, F, RW>, dim3(g.blocks + 1, n), g.threads, g.smem, s, ds);
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) with_two_line(a.lb, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_b2<A>(n * (a.n1 / 2));
        const int G = g.threads >> (A - 2);
        const int pf = resident_ctas((const void *)k_stepB_n<R, A>, g);
        err = launch_k(k_stepB_n<R, A>, dim3((a.n1 / 2 + G - 1) / G + 1, n), g.threads, g.smem, s, ds, pf);
    });
    return err;
}

// Plain pass C, two lines per thread, three CTAs per SM (k_stepC's THREE): columns
// of 3072 points in more than two waves of two CTAs, which are then a wave
// less.  us a step with two, with three: 4096x8192 137.3, 134.5; 4096x4096 72.5,
// 72.5; 4096x2048 (under a wave) 40.9, 42.7; 4096x512 19.3, 20.7 (direct stores).
// Shorter columns have 1.7 waves at most (2048x4096 40.5, 41.5).  Ensembles take
// three always: of 96 uneven flames 448.8 us, by this rule 451.0 (of 8 flames of
// 512x1024 25.7, 24.5; of 96 of 256x512 55.5, with two 64.6).
static bool three_ctas(int tiles) { return tiles > 4 * sm_count(); }

template <class R> cudaError_t Ops<R>::passC(const FlameDesc &d, cudaStream_t s) {
    cudaError_t err = cudaErrorInvalidValue;
    const int npair = (d.a.K2 + 2) / 2, extra = d.tile0 == 0 ? 1 : 0;
    const bool gen = general_epilogue(d);
    auto launch = [&](auto plain, auto general, const Geom &g, bool prefetch) {
        const int pf = prefetch ? resident_ctas((const void *)(gen ? general : plain), g) : 0;
        return launch_s(d.l2_state, pdl_on(sizeof(R) == 8, d.a), gen ? general : plain, dim3((d.tiles ? d.tiles : g.blocks) + extra), g.threads, g.smem,
                        s, d, pf);
    };
    if (!two_line<R>(d.a.la) || (d.onec && one_line<R>(d.a.la))) {
        with_one_line<R>(d.a.la, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value;
            using V = typename OneOf<R>::type;
            err = launch(k_stepC<R, V, A, F, false>, k_stepC<R, V, A, F, true>, geom_one_line<R, A, F>(npair, 2, 0), false);
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) with_two_line(d.a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_two_line(A, npair, pair_bytes<A>());
        const auto general = k_stepC<R, float2, A, 4, true>;
        if constexpr (A == kMaxA)
            if (three_ctas(d.tiles ? d.tiles : g.blocks)) {
                err = launch(k_stepC<R, float2, A, 4, false, true>, general, g, true);
                return;
            }
        err = launch(k_stepC<R, float2, A, 4, false>, general, g, true);
    });
    return err;
}
template <class R>
cudaError_t Ops<R>::passC_batch(const FlameDesc *ds, int n, const StepArgs &a, cudaStream_t s, bool onec, bool gen) {
    cudaError_t err = cudaErrorInvalidValue;
    const int npair = (a.K2 + 2) / 2;
    if (!two_line<R>(a.la) || (onec && one_line<R>(a.la))) {
        with_one_line<R>(a.la, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value;
            using V = typename OneOf<R>::type;
            const Geom g = geom_one_line<R, A, F>(npair, 2, 0);
            err = launch_k(gen ? k_stepC_n<R, V, A, F, true> : k_stepC_n<R, V, A, F, false>, dim3(g.blocks + 1, n),
                            g.threads, g.smem, s, ds, 0);
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) with_two_line(a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_two_line(A, n * npair, pair_bytes<A>());
        const int G = g.threads >> (A - 2);
        const auto kernel = gen ? k_stepC_n<R, float2, A, 4, true> : k_stepC_n<R, float2, A, 4, false, true>;
        err = launch_k(kernel, dim3((npair + G - 1) / G + 1, n), g.threads, g.smem, s, ds, resident_ctas((const void *)kernel, g));
    });
    return err;
}

template <class R>
cudaError_t Ops<R>::passCA(const FlameDesc &d, cudaStream_t s, const CUtensorMap *uv_map) {
    cudaError_t err = cudaErrorNotSupported;
    if constexpr (sizeof(R) == 4) {
        if (!uv_map || !two_line<R>(d.a.la)) return err;
        with_two_line(d.a.la, [&](auto ac) {
            constexpr int A = decltype(ac)::value;
            const Geom g = geom_two_line(A, (d.a.K2 + 2) / 2, pair_bytes<A>());
            const auto kernel = general_epilogue(d) ? k_stepCA<R, A, true> : k_stepCA<R, A, false>;
            const int pf = resident_ctas((const void *)kernel, g);
            err = launch_s(d.l2_state, pdl_on(sizeof(R) == 8, d.a), kernel, dim3(g.blocks + 1), g.threads, g.smem, s, d, pf, *uv_map);
        });
    }
    return err;
}

// Columns per tile of pass A and column pairs per tile of pass C (tiles =
// CTAs), for partial launches (flame_step_host).
template <class R> void Ops<R>::tiles(const StepArgs &a, int variant, int *colsA, int *pairsC) {
    const int npair = (a.K2 + 2) / 2;
    if (!two_line<R>(a.la) || (variant == kVariantOneLine && one_line<R>(a.la))) {
        with_one_line<R>(a.la, [&](auto ac, auto fc) {
            constexpr int A = decltype(ac)::value, F = decltype(fc)::value, T = 2 * Plan3<A, F>::TS;
            *colsA = geom_one_line<R, A, F>(a.K2 + 1, 2, 0).threads / T;
            *pairsC = geom_one_line<R, A, F>(npair, 2, 0).threads / T;
        });
        return;
    }
    with_two_line(a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        *colsA = geom_two_line(A, a.K2 + 1, pair_bytes<A>()).threads >> (A - 2);
        *pairsC = geom_two_line(A, npair, pair_bytes<A>()).threads >> (A - 2);
    });
}

}  // namespace flame
