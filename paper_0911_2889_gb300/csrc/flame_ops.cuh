// flame_ops.cuh -- launch geometry and launchers of the kernels.  FP64 is
// instantiated whole by flame_f64.cu; the FP32 launchers are split over
// flame_f32_*.cu so that their kernels compile in parallel.
#pragma once

#include "flame_adjoint.cuh"
#include "flame_launch.cuh"

namespace flame {

template <class R> static size_t group_smem(int logn) {
    return 2 * (size_t)plane_len(1 << logn) * sizeof(typename VecOf<R>::type);
}

// G line groups of T = 2^logn / 16 threads per CTA: up to 256 threads and
// the shared-memory budget, but no more groups than keep at least two CTAs
// per SM busy (small grids spread over the whole GPU).
template <class R> static Geom make_geom(int logn, int nlines, size_t extra = 0) {
    const int T = (1 << logn) >> 4;
    int G = T >= kThreadsTarget ? 1 : kThreadsTarget / T;
    const size_t per = group_smem<R>(logn) + extra;
    while (G > 1 && (G * per > kSmemBudget || G * T > kMaxThreads)) G >>= 1;
    while (G > 1 && (nlines + G - 1) / G < 2 * sm_count()) G >>= 1;

    Geom g;
    g.threads = G * T;
    g.blocks = (nlines + G - 1) / G;
    g.smem = G * per;
    return g;
}

// Line lengths with compile-time kernels: FP32 2^LO .. 2^12; everything else (and
// FP64) runs the runtime-length kernels (LOG = 0).
template <class R, int LO = 8, class F> static void with_log(int logn, F &&f) {
    bool done = false;
    if constexpr (sizeof(R) == 4) {
        static_for<LO, 13>([&](auto lc) {
            if (!done && logn == decltype(lc)::value) {
                f(lc);
                done = true;
            }
        });
    }
    if (!done) f(std::integral_constant<int, 0>{});
}

template <class R> cudaError_t Ops<R>::init_twiddles(C *tab, int logN, cudaStream_t s) {
    return launch_k(k_twiddles<R>, dim3((tw_table_len(logN, 4) + 255) / 256, 3), 256, 0, s, tab, logN);
}

template <class R>
cudaError_t Ops<R>::box_from_spec(const C *spec, C *state, double *mean, int n1, int n2, int K1, int K2,
                                  cudaStream_t s, int *status) {
    const long total = (long)(2 * K1 + 1) * (K2 + 1);
    const int blocks = (int)std::min<long>((total + 255) / 256, 8L * sm_count());
    return launch_k(k_box_from_spec<R>, dim3(blocks), 256, 0, s, spec, state, mean, n1, n2, K1, K2, status);
}

// Lines of 2^5 .. 2^10 points where 16 points a thread would leave an SM fewer
// than 256 threads: 4 points a thread.  Those transforms are bound by the
// latency of one thread's chain and by launches, not by bytes.  Per transform
// (graph), 16 -> 4 points: FP32 256x256 7.2 -> 4.7 us (with the second pass a
// programmatic dependent launch, below), 512x512 7.2 -> 5.7, 512x2048 11.0 -> 10.0,
// FP64 128x256 58 -> 18.5, 512x512 70 -> 23.6, 512x2048 92.5 -> 88.  Grids
// with more lines than that stay with 16 points: fewer exchanges.
// Programmatic dependent launch of the second pass: FP32 0.4 to 1 us a
// transform; FP64 off (512x1024 43.6 -> 45.4 c2r, 44.6 -> 52.3 r2c with it).
template <class R, class F> static bool with_short_lines(int logn, int npairs, bool split, F &&f) {
    bool done = false;
    if (((long)npairs << logn) / 16 < 256L * sm_count() && !(sizeof(R) == 4 && split))
        static_for<5, 11>([&](auto lc) {
            if (logn == decltype(lc)::value) {
                f(lc);
                done = true;
            }
        });
    return done;
}

// row pairs per CTA of short lines: up to 64 threads, and a CTA for every SM
static int short_groups(int npairs, int T) {
    int G = 1;
    while (2 * G * T <= 64 && npairs / (2 * G) >= sm_count()) G *= 2;
    return G;
}

template <class R>
cudaError_t Ops<R>::rows_r2c(const R *in, C *out, int n1, int logm, const C *tw, const C *tw1, cudaStream_t s, int *status) {
    Geom g = make_geom<R>(logm, n1 / 2);
    cudaError_t err = cudaSuccess;
    if (with_short_lines<R>(logm, n1 / 2, fft_split(sizeof(R) == 8, n1, logm) > 1, [&](auto lc) {
            constexpr int L = decltype(lc)::value;
            const int G = short_groups(n1 / 2, (1 << L) / 4);
            err = launch_k(k_rows_r2c<R, L, 4>, dim3(n1 / 2 / G), G * (1 << L) / 4, G * cols_group_bytes<R, 4>(1 << L, 1), s, in,
                           out, n1, logm, tw, status);
        }))
        return err;
    with_log<R>(logm, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        if constexpr (sizeof(R) == 4 && L >= 9)
            if (fft_split(false, n1, logm) == 4) {
                err = launch_k(k_rows4_r2c<L>, dim3(n1 / 4), (1 << L) / 8, 2 * group_smem<R>(L), s, in, out, n1, tw,
                               tw1 + tw_real_offset(__builtin_ctz(n1)), sm_count() * (4096 >> L), status);
                return;
            }
        err = launch_k(k_rows_r2c<R, L>, dim3(g.blocks), g.threads, g.smem, s, in, out, n1, logm, tw, status);
    });
    return err;
}

template <class R>
cudaError_t Ops<R>::rows_c2r(const C *in, R *out, int n1, int logm, const C *tw, const C *tw1, cudaStream_t s, int *status) {
    Geom g = make_geom<R>(logm, n1 / 2);
    cudaError_t err = cudaSuccess;
    if (with_short_lines<R>(logm, n1 / 2, fft_split(sizeof(R) == 8, n1, logm) > 1, [&](auto lc) {
            constexpr int L = decltype(lc)::value;
            const int G = short_groups(n1 / 2, (1 << L) / 4);
            err = launch_s(L2Window{nullptr, 0, 0.f}, sizeof(R) == 4, k_rows_c2r<R, L, 4>, dim3(n1 / 2 / G), G * (1 << L) / 4,
                           G * cols_group_bytes<R, 4>(1 << L, 1), s, in, out, n1, logm, tw, status);
        }))
        return err;
    with_log<R>(logm, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        if constexpr (sizeof(R) == 4 && L >= 9)
            if (fft_split(false, n1, logm) == 4) {
                err = launch_s(L2Window{nullptr, 0, 0.f}, true, k_rows4_c2r<L>, dim3(n1 / 4), (1 << L) / 8,
                               2 * group_smem<R>(L), s, in, out, n1, tw, tw1 + tw_real_offset(__builtin_ctz(n1)),
                               sm_count() * (4096 >> L), status);
                return;
            }
        err = launch_s(L2Window{nullptr, 0, 0.f}, sizeof(R) == 4, k_rows_c2r<R, L>, dim3(g.blocks), g.threads, g.smem, s, in, out, n1,
                       logm, tw, status);
    });
    return err;
}

template <class R>
cudaError_t Ops<R>::cols(const C *in, C *out, int logn, int split, int ncols, int ld, int dir, const C *tw, cudaStream_t s,
                         int *status) {
    const int npairs = (ncols + 1) / 2;
    // the next wave's tile into L2 where the array is too large to stay there
    // (4096x8192 -2 and -6 us; 4096x2048, which stays, +0.5)
    const int ahead = split > 1 && ((size_t)split << logn) * ld * sizeof(C) > ((size_t)64 << 20) ? 2 * sm_count() : 0;
    cudaError_t err = cudaSuccess;
    // r2c: behind the row pass; not behind the 64-thread CTAs of split rows of
    // 1024 points, among which the early column CTAs crowd in (1024x1024 16.5 us
    // against 9.7, 2048x1024 17.1 against 14.1; 2048x2048 18.0 against 18.9 without)
    const bool pdl = dir < 0 && sizeof(R) == 4 && !(split > 1 && ncols < 1024);
    auto go = [&](auto kernel, int threads, int G, size_t smem) {
        err = launch_s(L2Window{nullptr, 0, 0.f}, pdl, kernel, dim3((npairs + G - 1) / G, split), threads, smem, s, in,
                       out, logn, ncols, ld, tw, ahead, status);
    };
    if (with_short_lines<R>(logn, npairs, split > 1, [&](auto lc) {
            constexpr int L = decltype(lc)::value, T = (1 << L) / 4;
            // adjacent columns in one CTA, up to 32 bytes of a row a warp
            int G = sizeof(R) == 4 ? 4 : 2;
            while (G > 1 && (npairs < G * sm_count() || G * T > 256)) G >>= 1;
            const size_t smem = G * cols_group_bytes<R, 4>(1 << L, G);
            if (dir < 0) go(k_cols<R, -1, L, 4>, G * T, G, smem);
            else go(k_cols<R, 1, L, 4>, G * T, G, smem);
        }))
        return err;
    const int n = 1 << logn, T = n >> 4;
    const Geom g = make_geom<R>(logn, npairs * split);
    with_log<R>(logn, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        const int G = g.threads / T;
        if (dir < 0) go(k_cols<R, -1, L>, g.threads, G, G * cols_group_bytes<R>(n, G));
        else go(k_cols<R, 1, L>, g.threads, G, G * cols_group_bytes<R>(n, G));
    });
    return err;
}

// FP64 lines of 2^4 .. 2^7 points: 8 points per thread, one line pair per
// CTA (the runtime kernels give such lines 2^LOG/16 threads, a quarter warp
// at 128 points, and are bound by the latency of their FP64 chains)
template <class R> static bool small_fp64(int logn) { return sizeof(R) == 8 && logn >= 4 && logn <= 7; }
// Points per thread of those kernels, which a step with its area runs: 4 (a warp
// per 128-point line pair), or 8 with FLAME_FP64_POINTS=8 (read at every launch,
// so tests can run both).  The lines' FP64 chains are latency-bound, and a full
// warp per line pair halves each thread's: when the plain step ran them too,
// 128x256 took 46.1 us a step with 4 and 78.4 with 8.
static int fp64_points() {
    const char *v = getenv("FLAME_FP64_POINTS");
    return (v && strcmp(v, "8") == 0) ? 8 : 4;
}
template <class R, int E> static Geom geom_small_fp64(int logn, int nlines, size_t extra) {
    Geom g;
    g.threads = (1 << logn) / E;
    g.blocks = nlines;
    g.smem = 2 * (size_t)plane_len_e<E>(1 << logn) * sizeof(typename VecOf<R>::type) + extra;
    return g;
}
// CTA of the one-line kernels (k_passA1, k_passC1): `groups` line groups of
// 2^logn / E threads, each with its own exchange planes, and `extra` bytes more;
// one CTA per unit
template <class R, int E> static Geom geom_short1(int logn, int units, int groups, size_t extra) {
    Geom g;
    g.threads = groups * ((1 << logn) / E);
    g.blocks = units;
    g.smem = (size_t)groups * 2 * plane_len_e<E>(1 << logn) * sizeof(R) + extra;
    return g;
}
// FP32 columns with one-line kernels (E = 16): 2^8 .. 2^10 points (1024x2048,
// pass A + C: 8.3 + 12.0 us against 9.9 + 12.4 us with two lines per thread;
// longer columns fill the SMs with pairs: 2048x2048 55 against 30 us a step)
template <class R> static bool one_line_fp32(int logn) { return sizeof(R) == 4 && logn >= 8 && logn <= 10; }
// calls f(integral_constant<E>) with the chosen points per thread
template <class F> static void with_fp64_points(F &&f) {
    if (fp64_points() == 4) f(std::integral_constant<int, 4>{});
    else f(std::integral_constant<int, 8>{});
}

// Passes A and B of a step with the area are programmatic dependent launches in
// FP32 (FLAME_PDL=0: not): 512x1024 25.8 -> 24.8 us a step, 1024x2048 31.9 -> 31.4,
// 4096x8192 365 -> 364.5.  Pass C is not (1024x2048 34.5): early column CTAs take
// SMs that the row pass, one CTA per SM, still needs.
template <class R> static bool pdl_area() {
    const char *v = getenv("FLAME_PDL");
    return sizeof(R) == 4 && !(v && strcmp(v, "0") == 0);
}

// Passes A and C on the public grid: the steps that record the surface area
// (whose sum is over that grid's points).
template <class R>
cudaError_t Ops<R>::passA_full(const FlameDesc &d, cudaStream_t s, const CUtensorMap *uv_map) {
    cudaError_t err = cudaErrorInvalidValue;
    if constexpr (sizeof(R) == 8) if (small_fp64<R>(d.a.logn1)) {
        with_fp64_points([&](auto ec) {
            constexpr int E = decltype(ec)::value;
            const Geom g = geom_short1<R, E>(d.a.logn1, d.a.K2 + 1, 2, 0);
            static_for<4, 8>([&](auto lc) {
                constexpr int L = decltype(lc)::value;
                if (d.a.logn1 == L)
                    err = launch_s(d.l2_state, pdl_area<R>(), k_passA1<R, L, E>, dim3(g.blocks), g.threads, g.smem, s, d);
            });
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) if (one_line_fp32<R>(d.a.logn1)) {
        const Geom g = geom_short1<R, 16>(d.a.logn1, d.a.K2 + 1, 2, 0);
        static_for<8, 11>([&](auto lc) {
            constexpr int L = decltype(lc)::value;
            if (d.a.logn1 == L)
                err = launch_s(d.l2_state, pdl_area<R>(), k_passA1<R, L, 16>, dim3(g.blocks), g.threads, g.smem, s, d);
        });
        return err;
    }
    const Geom g = make_geom<R>(d.a.logn1, d.a.K2 + 1);
    with_log<R, 11>(d.a.logn1, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        if constexpr (sizeof(R) == 4 && L > 0) if (uv_map) {  // tensor-store write-out
            const int pf = resident_ctas((const void *)k_passAt<R, L>, g);
            err = launch_s(d.l2_state, pdl_area<R>(), k_passAt<R, L>, dim3(g.blocks), g.threads, g.smem, s, d, pf, *uv_map);
            return;
        }
        const int pf = resident_ctas((const void *)k_passA<R, L>, g);
        err = launch_s(d.l2_state, pdl_area<R>(), k_passA<R, L>, dim3(g.blocks), g.threads, g.smem, s, d, pf);
    });
    return err;
}

// pass B with 8 points per thread: 512-thread CTAs, padding every 8 slots
template <class R> static Geom geom_passB8(int logm, int nlines) {
    const int T = (1 << logm) >> 3;
    const int G = T >= 512 ? 1 : 512 / T;
    Geom g;
    g.threads = G * T;
    g.blocks = (nlines + G - 1) / G;
    g.smem = (size_t)G * (2 * (size_t)plane_len_e<8>(1 << logm) * sizeof(typename VecOf<R>::type) +
                          (size_t)(1 << logm) * sizeof(typename VecOf<R>::c));
    return g;
}

template <class R> cudaError_t Ops<R>::passB_area(const FlameDesc &d, cudaStream_t s) {
    using Vt = typename VecOf<R>::type;
    const int M = 1 << d.a.logm;
    cudaError_t err = cudaErrorNotSupported;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return cudaErrorNotSupported;
    }
    const size_t area_extra = 3 * (size_t)M * sizeof(Vt);
    if constexpr (sizeof(R) == 8) if (small_fp64<R>(d.a.logm)) {
        with_fp64_points([&](auto ec) {
            constexpr int E = decltype(ec)::value;
            Geom g = geom_small_fp64<R, E>(d.a.logm, d.a.n1 / 2, (size_t)M * sizeof(typename VecOf<R>::c) + area_extra);
            if (g.smem + 4096 > (size_t)optin) return;
            static_for<4, 8>([&](auto lc) {
                constexpr int L = decltype(lc)::value;
                if (d.a.logm == L)
                    err = launch_s(L2Window{nullptr, 0, 0.f}, pdl_area<R>(), k_passB_area<R, L, E, 128>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
            });
        });
        return err;
    }
    // FP32 compile-time rows: 8 points per thread, 512-thread CTAs (one per
    // SM: the area buffers take most of the shared memory, and 16 warps hide
    // more latency than the 8 of 16 points per thread)
    if constexpr (sizeof(R) == 4) if (d.a.logm >= 8 && d.a.logm <= 12) {
        Geom g = geom_passB8<R>(d.a.logm, d.a.n1 / 2);
        const int G = g.threads / (M / 8);
        g.smem += (size_t)G * area_extra;
        if (g.smem + 4096 > (size_t)optin) return cudaErrorNotSupported;
        with_log<R>(d.a.logm, [&](auto lc) {
            constexpr int L = decltype(lc)::value;
            if constexpr (L > 0) err = launch_s(L2Window{nullptr, 0, 0.f}, pdl_area<R>(), k_passB_area<R, L, 8, 512>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
        });
        if (err != cudaSuccess) return err;
        return cudaGetLastError();
    }
    // other rows: the runtime-length kernel
    const Geom g = make_geom<R>(d.a.logm, d.a.n1 / 2, (size_t)M * sizeof(typename VecOf<R>::c) + area_extra);
    if (g.smem + 4096 > (size_t)optin) return cudaErrorNotSupported;
    return launch_s(L2Window{nullptr, 0, 0.f}, pdl_area<R>(), k_passB_area<R, 0, 16, 256>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
}

template <class R> cudaError_t Ops<R>::passC_full(const FlameDesc &d, cudaStream_t s) {
    cudaError_t err = cudaErrorInvalidValue;
    if constexpr (sizeof(R) == 8) if (small_fp64<R>(d.a.logn1)) {
        with_fp64_points([&](auto ec) {
            constexpr int E = decltype(ec)::value;
            const Geom g = geom_short1<R, E>(d.a.logn1, (d.a.K2 + 2) / 2, 2, 0);
            static_for<4, 8>([&](auto lc) {
                constexpr int L = decltype(lc)::value;
                if (d.a.logn1 == L)
                    err = launch_w(d.l2_state, k_passC1<R, L, E>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
            });
        });
        return err;
    }
    if constexpr (sizeof(R) == 4) if (one_line_fp32<R>(d.a.logn1)) {
        const Geom g = geom_short1<R, 16>(d.a.logn1, (d.a.K2 + 2) / 2, 2, 0);
        static_for<8, 11>([&](auto lc) {
            constexpr int L = decltype(lc)::value;
            if (d.a.logn1 == L)
                err = launch_w(d.l2_state, k_passC1<R, L, 16>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
        });
        return err;
    }
    const Geom g = make_geom<R>(d.a.logn1, (d.a.K2 + 2) / 2);
    with_log<R, 11>(d.a.logn1, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        const int pf = resident_ctas((const void *)k_passC<R, L>, g);
        err = launch_w(d.l2_state, k_passC<R, L>, dim3(g.blocks + 1), g.threads, g.smem, s, d, pf);
    });
    return err;
}

// one row per CTA (N2/32 threads): exchange buffer + one parked row
template <class R> static Geom geom_row1(int logm, int nrows) {
    Geom g;
    g.threads = (1 << logm) >> 4;
    g.blocks = nrows;
    g.smem = group_smem<R>(logm) + (size_t)(1 << logm) * sizeof(typename VecOf<R>::c);
    return g;
}

// The area and adjoint kernels take the column length (log2 N1) or the
// half row length (log2 N2/2) as their compile-time LOG (0: any length).
template <class R> cudaError_t Ops<R>::area(const AdjDesc &d, cudaStream_t s) {
    const StepArgs &a = d.a;
    Geom ga = make_geom<R>(a.logn1, a.K2 + 1);
    Geom gb = geom_row1<R>(a.logm, a.n1);
    cudaError_t e = cudaSuccess;
    with_log<R>(a.logn1, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        e = launch_k(k_areaA<R, L>, dim3(ga.blocks), ga.threads, ga.smem, s, d);
    });
    with_log<R>(a.logm, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        if (e == cudaSuccess) e = launch_k(k_areaB<R, L>, dim3(gb.blocks), gb.threads, gb.smem, s, d);
    });
    with_log<R>(a.logn1, [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        if (e == cudaSuccess) e = launch_k(k_areaC<R, L>, dim3(ga.blocks), ga.threads, ga.smem, s, d);
    });
    return e;
}

// CTA of an adjoint kernel: lines of T threads, up to 128 threads, fewer lines
// where they would not span two CTAs per SM
template <class R, int A> static Geom geom_adj(int nlines) {
    using V = typename VecOf<R>::type;
    using PL = Plan3<A, adj_f<R>(A)>;
    int G = PL::TS >= 128 ? 1 : 128 / PL::TS;
    while (G > 1 && (G * PL::TS > 32) && (nlines + G - 1) / G < 2 * sm_count()) G >>= 1;
    return Geom{G * PL::TS, (nlines + G - 1) / G, exchange_bytes<R, V, PL>(G)};
}
template <class R> cudaError_t Ops<R>::adj_step(const AdjDesc &d, cudaStream_t s) {
    const StepArgs &a = d.a;
    FlameDesc f;
    memset(&f, 0, sizeof f);
    f.a = a;
    f.state = const_cast<void *>(d.state);
    f.uv = d.uv;
    f.tw1 = d.tw1;
    f.status = d.status;
    cudaError_t e = passA(f, s, a.la <= 8 ? kVariantOneLine : kVariantDirect);
    if (e != cudaSuccess) return e;
    with_a(a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_adj<R, A>((a.K2 + 2) / 2);
        e = launch_s(L2Window{nullptr, 0, 0.f}, pdl_on(sizeof(R) == 8, a), k_adjL<R, A>, dim3(g.blocks + 1), g.threads, g.smem, s, d);
    });
    with_a(a.lb, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_adj<R, A>(a.n1);
        if (e == cudaSuccess) e = launch_s(L2Window{nullptr, 0, 0.f}, pdl_on(sizeof(R) == 8, a), k_adjB<R, A>, dim3(g.blocks), g.threads, g.smem, s, d);
    });
    with_a(a.la, [&](auto ac) {
        constexpr int A = decltype(ac)::value;
        const Geom g = geom_adj<R, A>(a.K2 + 1);
        if (e == cudaSuccess) e = launch_s(L2Window{nullptr, 0, 0.f}, pdl_on(sizeof(R) == 8, a), k_adjC<R, A>, dim3(g.blocks), g.threads, g.smem, s, d);
    });
    return e;
}

}  // namespace flame
