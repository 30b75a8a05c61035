// flame_adjoint.cuh -- kernels of the area objective and of the discrete
// adjoint of the explicit step (project-added; the paper has neither).
//
// Conventions (inner product on spectra: <X, Y> = Re sum over the full
// spectrum of conj(X_k) Y_k; synthesis  phi(x) = sum_k Phi_k e^{ik.x};
// analysis  hat(a)_k = sum_x a(x) e^{-ik.x}):
//
//   area   A = sum_x w R sqrt(R^2 + |grad phi|^2),  R = r0 + phi,
//          w = (2 pi)^2 / (N1 N2 s1 s2);
//          dA/dPhi_k = hat(a)_k - i kappa_1 hat(b1)_k - i kappa_2 hat(b2)_k with
//          a = w (S + R^2/S), b_i = w R d_i phi / S, S = sqrt(R^2 + |grad phi|^2).
//   adjoint of one Euler step at (Phi_n, t_n), lambda = lambda_{n+1}:
//          lambda_n = lambda + dt (omega_k lambda + c P_k)   (k != 0),
//          P = (1/(N1 N2)) [ -i kappa_1 hat(q1) - i kappa_2 hat(q2) ],
//          q_i = 2 ell d_i phi_n,  ell = synthesis of lambda (with lambda_0),
//          lambda_0 unchanged; dL/dgamma += <lambda, dt |kappa|/(2 r0) Phi_n>.
#pragma once

#include "flame_step.cuh"

namespace flame {

template <class R> __device__ __forceinline__ CplxT<R> cmulc(CplxT<R> a, CplxT<R> b) {
    return CplxT<R>{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}

// --- area, pass A: columns of (i s1 k1 Phi, Phi with the mean mode) ---------
// writes uv[j1][k2] = (U, P) with U = synthesis of i s1 k1 Phi and P the
// column synthesis of Phi (the mean mode at k = 0).
template <class R, int LOG> __global__ void __launch_bounds__(256, kMinBlocks<R>) k_areaA(AdjDesc d) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    extern __shared__ __align__(16) unsigned char smraw[];
    const StepArgs &a = d.a;
    const C *state = static_cast<const C *>(d.state);
    C *uv = static_cast<C *>(d.uv);
    const int N1 = 1 << a.logn1, T = N1 >> 4;
    const int G = blockDim.x / T, g = threadIdx.x / T, t = threadIdx.x % T;
    const int ld1 = 2 * a.K1 + 1;
    const int k2 = blockIdx.x * G + g;
    const bool valid = k2 <= a.K2;
    V *base = reinterpret_cast<V *>(smraw) + (size_t)g * 2 * plane_len(N1);
    auto sm = make_planes(base, N1);
    const C *col = state + (size_t)k2 * ld1 + a.K1;
    const double mean0 = *d.mean;
    CV<V> x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        x[r] = CV<V>{vzero(V{}), vzero(V{})};
        if (r < 4 || r >= 12) {
            const int n = t + r * T;
            const int k1 = (r < 4) ? n : n - N1;
            const bool in_box = valid && ((r < 4) ? (n <= a.K1) : (k1 >= -a.K1));
            if (in_box) {
                C phi = col[k1];
                if (k1 == 0 && k2 == 0) phi = C{(R)mean0, 0};
                const R f = scale1<R>(a) * (R)k1;
                x[r] = pack2<R>(C{-f * phi.y, f * phi.x}, phi);
            }
        }
    }
    fft_line<1, LOG>(x, a.logn1, t, sm, static_cast<const C *>(d.tw1));
    if (valid) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int n = t + r * T;
            st_uv<R>(uv + uv_index(n, k2, a.ldk), lane0<R>(x[r]), lane1<R>(x[r]));
        }
    }
}

// Half-band inverse of one row: from the row spectrum S[k] (k = -K2..K2,
// S[-k] = conj S[k] unless `full`) builds the lanes Y_q[k mod M] =
// S[k] e^{2 pi i k q / N2} (q = 0, 1) and transforms them; lane q of x[r]
// is then the synthesis at grid point 2m + q, m = t + r T.
template <class R, int LOG, class Get>
__device__ __forceinline__ void halfband_ifft(CV<typename VecOf<R>::type> (&x)[16], const StepArgs &a, int t,
                                              const CplxT<R> *P, const CplxT<R> *twm, Get get, bool valid,
                                              void *smbase) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    const int M = 1 << a.logm, T = M >> 4;
    auto sm = make_planes(static_cast<V *>(smbase), M);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int n = t + r * T;
        const int kk = (r < 8) ? n : M - n;
        C z{0, 0};
        if (valid && kk <= a.K2) z = get(kk, r < 8);
        C w = __ldg(P + kk);
        C z1 = (r < 8) ? C{z.x * w.x - z.y * w.y, z.x * w.y + z.y * w.x}
                       : C{z.x * w.x + z.y * w.y, z.y * w.x - z.x * w.y};
        x[r] = pack2<R>(z, z1);
    }
    fft_line<1, LOG>(x, a.logm, t, sm, twm);
}

// Forward real transform of two real rows given as h_q[m] = f_q[2m] + i
// f_q[2m+1] in the lanes of x (q = 0, 1); on return out(k, Y) is called for
// k = 0..K2 (r < 8) with Y the pair of analyses (lane 0: f_0, lane 1: f_1).
template <class R, int LOG, class Out>
__device__ __forceinline__ void real_fwd(CV<typename VecOf<R>::type> (&x)[16], const StepArgs &a, int t,
                                         const CplxT<R> *P, const CplxT<R> *twm, void *smbase, bool valid,
                                         Out out) {
    using V = typename VecOf<R>::type;
    const int M = 1 << a.logm, T = M >> 4;
    auto sm = make_planes(static_cast<V *>(smbase), M);
    fft_line<-1, LOG>(x, a.logm, t, sm, twm);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; ++r) sm.st(t + r * T, x[r]);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int k = t + r * T;
        if (valid && k <= a.K2) {
            CV<V> h = x[r], hc = sm.ld((M - k) & (M - 1));
            const R hf = (R)0.5;
            CV<V> E{vmul(vadd(h.re, hc.re), vbc(hf)), vmul(vsub(h.im, hc.im), vbc(hf))};
            CV<V> O{vmul(vadd(h.im, hc.im), vbc(hf)), vmul(vsub(hc.re, h.re), vbc(hf))};
            auto w = __ldg(P + k);
            out(k, cadd(E, cmul_s(O, w.x, -w.y)));
        }
    }
    __syncthreads();
}

// --- area, pass B: one row per group ----------------------------------------
// u + iv from U, V = i s2 k2 P; phi from P; pointwise area terms; forward
// real transforms of a, b1, b2.  Writes aw[k2][j1] = (hat a, hat b1) and
// gk[k2][j1] = hat b2 (column-major), rowsum[j1] = sum_x of w R S over the row.
template <class R, int LOG> __global__ void __launch_bounds__(256, kMinBlocks<R>) k_areaB(AdjDesc d) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ double red[256];  // one per thread (blockDim = N2/32 <= 256)
    const StepArgs &a = d.a;
    const C *uv = static_cast<const C *>(d.uv);
    const C *twm = static_cast<const C *>(d.twm);
    const int M = 1 << a.logm, T = M >> 4;
    const int t = threadIdx.x;  // one group per CTA
    const int row = blockIdx.x;
    const bool valid = row < a.n1;
    V *base = reinterpret_cast<V *>(smraw);
    C *park = reinterpret_cast<C *>(base + 2 * plane_len(M));  // M entries
    const C *P = twm + tw_real_offset(a.logm);
    const C *src = uv + uv_index(valid ? row : 0, 0, a.ldk);  // element kk at src + 4 kk
    const R s2 = scale2<R>(a);
    // phi at 2m, 2m+1 (real parts of the two lanes), parked
    CV<V> x[16];
    halfband_ifft<R, LOG>(x, a, t, P, twm,
                     [&](int kk, bool pos) {
                         UV<R> e = ld_uv<R>(src + 4 * (size_t)kk);
                         return pos ? e.v : C{e.v.x, -e.v.y};
                     },
                     valid, base);
#pragma unroll
    for (int r = 0; r < 16; ++r) park[t + r * T] = C{x[r].re.x, x[r].re.y};
    // u + iv at 2m, 2m+1
    halfband_ifft<R, LOG>(x, a, t, P, twm,
                     [&](int kk, bool pos) {
                         UV<R> e = ld_uv<R>(src + 4 * (size_t)kk);
                         const R f = s2 * (R)kk;
                         C Vv{-f * e.v.y, f * e.v.x};  // i s2 k2 P
                         if (pos) return C{e.u.x - Vv.y, e.u.y + Vv.x};
                         return C{e.u.x + Vv.y, Vv.x - e.u.y};
                     },
                     valid, base);
    const double r0 = *d.t;
    const R w = (R)((2.0 * 3.14159265358979323846) * (2.0 * 3.14159265358979323846) /
                    ((double)a.n1 * (double)a.n2 * a.s1 * a.s2));
    double part = 0.0;
    C hb2[16];
    CV<V> y[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        C ph = park[t + r * T];
        R av[2], b1[2], b2[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const R u = q == 0 ? x[r].re.x : x[r].re.y;
            const R v = q == 0 ? x[r].im.x : x[r].im.y;
            const R Rr = (R)r0 + (q == 0 ? ph.x : ph.y);
            const R S = sqrt(Rr * Rr + u * u + v * v);
            part += (double)(w * Rr * S);
            av[q] = w * (S + Rr * Rr / S);
            b1[q] = w * Rr * u / S;
            b2[q] = w * Rr * v / S;
        }
        y[r] = pack2<R>(C{av[0], av[1]}, C{b1[0], b1[1]});
        hb2[r] = C{b2[0], b2[1]};
    }
    if (!valid) part = 0.0;
    C *aw = static_cast<C *>(d.aw);
    C *gk = static_cast<C *>(d.gk);
    real_fwd<R, LOG>(y, a, t, P, twm, base, valid, [&](int k, CV<V> Y) {
        C *dst = aw + 2 * ((size_t)k * a.n1 + row);
        st_uv<R>(dst, lane0<R>(Y), lane1<R>(Y));
    });
#pragma unroll
    for (int r = 0; r < 16; ++r) y[r] = pack2<R>(hb2[r], C{0, 0});
    real_fwd<R, LOG>(y, a, t, P, twm, base, valid, [&](int k, CV<V> Y) { gk[(size_t)k * a.n1 + row] = lane0<R>(Y); });
    const double sum = cta_sum(part, red);
    if (t == 0 && valid) d.rowsum[row] = sum;
}

// --- area, pass C: one column per group -------------------------------------
// forward column transforms of (hat a, hat b1) and hat b2, combination
// grad = A - i s1 k1 B1 - i s2 k2 B2 on the box; block 0 also reduces the
// row sums into the area and writes dA/dPhi_0.
template <class R, int LOG> __global__ void __launch_bounds__(256, kMinBlocks<R>) k_areaC(AdjDesc d) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    extern __shared__ __align__(16) unsigned char smraw[];
    const StepArgs &a = d.a;
    const int N1 = 1 << a.logn1, T = N1 >> 4;
    const int G = blockDim.x / T, g = threadIdx.x / T, t = threadIdx.x % T;
    const int ld1 = 2 * a.K1 + 1;
    const int k2 = blockIdx.x * G + g;
    const bool valid = k2 <= a.K2;
    V *base = reinterpret_cast<V *>(smraw) + (size_t)g * 2 * plane_len(N1);
    auto sm = make_planes(base, N1);
    const C *tw1 = static_cast<const C *>(d.tw1);
    const C *aw = static_cast<const C *>(d.aw) + 2 * (size_t)(valid ? k2 : 0) * N1;
    const C *gk = static_cast<const C *>(d.gk) + (size_t)(valid ? k2 : 0) * N1;
    // hat b2 first (only the box rows are kept), then (hat a, hat b1)
    CV<V> x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int n = t + r * T;
        x[r] = pack2<R>(valid ? gk[n] : C{0, 0}, C{0, 0});
    }
    fft_line<-1, LOG>(x, a.logn1, t, sm, tw1);
    C B2[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) B2[i] = lane0<R>(x[i < 4 ? i : i + 8]);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int n = t + r * T;
        UV<R> e = valid ? ld_uv<R>(aw + 2 * n) : UV<R>{C{0, 0}, C{0, 0}};
        x[r] = pack2<R>(e.u, e.v);
    }
    fft_line<-1, LOG>(x, a.logn1, t, sm, tw1);
    C *grad = static_cast<C *>(d.grad);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = i < 4 ? i : i + 8;
        const int n = t + r * T;
        const int k1 = (r < 4) ? n : n - N1;
        const bool in_box = valid && ((r < 4) ? (n <= a.K1) : (k1 >= -a.K1));
        if (in_box) {
            C A = lane0<R>(x[r]), B1 = lane1<R>(x[r]);
            const R f1 = scale1<R>(a) * (R)k1, f2 = scale2<R>(a) * (R)k2;
            // A - i f1 B1 - i f2 B2
            C gr{A.x + f1 * B1.y + f2 * B2[i].y, A.y - f1 * B1.x - f2 * B2[i].x};
            if (k1 == 0 && k2 == 0) {
                *d.dmean = (double)A.x;
                gr = C{0, 0};
            }
            if (grad) grad[(size_t)k2 * ld1 + k1 + a.K1] = gr;
        }
    }
    if (blockIdx.x == 0) {  // (one thread's sum of 512 rows took 17 of the kernel's 36 us)
        __shared__ double red[256];
        double v = 0.0;
        for (int i = threadIdx.x; i < a.n1; i += blockDim.x) v += d.rowsum[i];
        const double sum = cta_sum(v, red);
        if (threadIdx.x == 0) *d.area = sum;
    }
}

// ----------------------------------------------------------------------------
// The adjoint step, on the step's alias-free grid: its products 2 ell d_i phi
// are quadratic too, and only their retained harmonics are wanted.  Pass A of
// the step gives W = the row spectra of d1 phi + i d2 phi; then
//   L (columns): lambda -> its row spectra, for all j1
//   B (rows):    ell and d_i phi on the row, q_i = 2 ell d_i phi, forward real
//                transforms of q_1 and q_2
//   C (columns): forward transforms, P, the update of lambda, dL/dgamma
// Two lines per thread throughout (two columns, even and odd points, q_1 and
// q_2); 3 F and 4 F points a thread, F by adj_f.
// ----------------------------------------------------------------------------
// (512x1024: with the public grid, 16 points a thread and every CTA deriving
// the coefficients, an adjoint step's four kernels took 38 us.)
template <class R> __host__ __device__ constexpr int adj_f(int a) {
    return a == 2 ? 1 : sizeof(R) == 8 ? (a <= 6 ? 1 : a <= 9 ? 2 : 4) : (a <= 8 ? 2 : 4);
}
// complex index of lambda's row spectrum (j1, k2): row pairs interleaved
__host__ __device__ __forceinline__ size_t l_index(int j1, int k2, int ldk) {
    return 2 * ((size_t)(j1 >> 1) * ldk + k2) + (j1 & 1);
}
// ... and its extent (lambda's row spectra lie in gk)
__host__ __device__ __forceinline__ long long l_len(const StepArgs &a) { return (long long)a.n1 * a.ldk; }

// Columns c0, c0 + 1 of lambda (lambda_0 at k = 0); the extra CTA derives the
// step's coefficients for pass C (and dt / (2 t_n), dL/dgamma's factor).
template <class R, int A> __global__ void __launch_bounds__(256, kMinBlocks<R>) k_adjL(AdjDesc d) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    using PL = Plan3<A, adj_f<R>(A)>;
    constexpr int F = PL::F, SL = PL::slots(kSlotsPerWave<V>);
    extern __shared__ __align__(128) unsigned char smstep[];
    const StepArgs &a = d.a;
    griddep_wait();
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            store_coef<R>(d.coef, a, *d.t, false);
            d.coef[10] = a.dt / (2.0 * d.coef[0]);
        }
        griddep_launch();
        return;
    }
    const int G = blockDim.x / PL::TS, ld1 = 2 * a.K1 + 1;
    const Place s = place_all<PL::TS>(), p = place<PL::TP>(G);
    const double l0 = *d.lam0;
    CV<V> xs[PL::ES];
    {
        const int c0 = 2 * ((blockIdx.x - 1) * G + s.line);
        const C *la = static_cast<const C *>(d.lam) + (size_t)c0 * ld1 + a.K1, *lb = la + ld1;
#pragma unroll
        for (int r = 0; r < PL::ES; ++r) {
            xs[r] = CV<V>{vzero(V{}), vzero(V{})};
            if (r >= F && r < 2 * F) continue;
            const int n = s.t + r * PL::TS, k1 = r < F ? n : n - PL::L;
            const bool in_box = r < F ? n <= a.K1 : k1 >= -a.K1;
            [[maybe_unused]] const long long i = (long long)c0 * ld1 + a.K1 + k1;
            C p0 = in_box && c0 <= a.K2 && FLAME_IN(d.status, i, box_len(a), kSiteAdjLam) ? la[k1] : C{0, 0};
            const C p1 = in_box && c0 + 1 <= a.K2 && FLAME_IN(d.status, i + ld1, box_len(a), kSiteAdjLam) ? lb[k1] : C{0, 0};
            if (c0 == 0 && k1 == 0) p0 = C{(R)l0, 0};
            xs[r] = pack2<R>(p0, p1);
        }
    }
    auto buf = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    CV<V> xp[PL::EP];
    inverse3<PL>(xs, xp, s, p, buf, tab3<R, A, F, C>(d.tw1));
    griddep_launch();
    if (!p.on) return;
    C *out = static_cast<C *>(d.gk);
    const int c0 = 2 * ((blockIdx.x - 1) * G + p.line);
#pragma unroll
    for (int i = 0; i < PL::EP; ++i) {
        const size_t n = l_index(p.t + i * PL::TP, c0, a.ldk);
        if (c0 <= a.K2 && FLAME_IN(d.status, n, l_len(a), kSiteAdjRow)) out[n] = lane0<R>(xp[i]);
        if (c0 + 1 <= a.K2 && FLAME_IN(d.status, n + 2, l_len(a), kSiteAdjRow)) out[n + 2] = lane1<R>(xp[i]);
    }
}

// The inputs of a row's two half-length inverse transforms (as in the step's
// pass B), get(k, minus) the row spectrum at +-k, 0 <= k <= K2.
template <class PL, class R, class V, class Get>
__device__ __forceinline__ void half_inputs(CV<V> (&x)[PL::ES], int t, bool valid, int K2, const CplxT<R> *P, Get get) {
    using C = CplxT<R>;
#pragma unroll
    for (int r = 0; r < PL::ES; ++r) {
        const int n = t + r * PL::TS, km = PL::L - n;
        const C up = r < 2 * PL::F && valid && n <= K2 ? get(n, false) : C{0, 0};
        const C um = r >= PL::F && valid && km <= K2 ? get(km, true) : C{0, 0};
        const C o{up.x - um.x, up.y - um.y}, w = __ldg(P + n);
        x[r] = pack2<R>(C{up.x + um.x, up.y + um.y}, C{fma_rn(o.x, w.x, -(o.y * w.y)), fma_rn(o.x, w.y, o.y * w.x)});
    }
}

// One row per group: ell and w = d1 phi + i d2 phi at the even and odd points
// (lanes), q_i = 2 ell d_i phi, forward transforms of h_i[m] = q_i[2m] + i
// q_i[2m+1] (lanes i = 1, 2); aw[k2][j1] = (hat q1, -i s2 k2 hat q2).
template <class R, int A> __global__ void __launch_bounds__(256, kMinBlocks<R>) k_adjB(AdjDesc d) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    using PL = Plan3<A, adj_f<R>(A)>;
    constexpr int F = PL::F, L = PL::L, TS = PL::TS, ES = PL::ES, SL = PL::slots(kSlotsPerWave<V>);
    extern __shared__ __align__(128) unsigned char smstep[];
    const StepArgs &a = d.a;
    griddep_wait();
    const int G = blockDim.x / TS;
    const Place s = place_all<TS>(), p = place<PL::TP>(G);
    const int row = blockIdx.x * G + s.line;
    const bool valid = row < a.n1;
    auto buf = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    const C *tw = tab3<R, A, F, C>(d.twm);
    const C *P = static_cast<const C *>(d.twm) + tw3_real_offset<A>();
    const C *lrow = static_cast<const C *>(d.gk), *uv = static_cast<const C *>(d.uv);
    V ell[PL::EP];
    {
        CV<V> xs[ES], xp[PL::EP];
        half_inputs<PL, R>(xs, s.t, valid, a.K2, P, [&](int k, bool minus) {
            const size_t n = l_index(row, k, a.ldk);
            const C e = FLAME_IN(d.status, n, l_len(a), kSiteAdjRow) ? lrow[n] : C{0, 0};
            return minus ? C{e.x, -e.y} : e;
        });
        inverse3<PL>(xs, xp, s, p, buf, tw);
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) ell[i] = vadd(xp[i].re, xp[i].re);  // 2 ell
    }
    CV<V> xp[PL::EP];
    {
        CV<V> xs[ES];
        half_inputs<PL, R>(xs, s.t, valid, a.K2, P, [&](int k, bool minus) {
            return FLAME_IN(d.status, w_index(row, k, a.ldk) + 3, uv_len(a), kSiteAdjUv) ? ld_w<R>(uv, row, k, a.ldk, minus)
                                                                                          : C{0, 0};
        });
        __syncthreads();  // the exchange buffers are free
        inverse3<PL>(xs, xp, s, p, buf, tw);
    }
#pragma unroll
    for (int i = 0; i < PL::EP; ++i) {
        const V q1 = vmul(ell[i], xp[i].re), q2 = vmul(ell[i], xp[i].im);
        xp[i] = CV<V>{V{q1.x, q2.x}, V{q1.y, q2.y}};
    }
    CV<V> hk[ES];
    forward3<PL, false>(xp, hk, p, s, buf, tw);
    griddep_launch();
    __syncthreads();
    const Planes<V> sm = buf(s.line);
#pragma unroll
    for (int r = 0; r < ES; ++r)
        if (TS * (r + 1) > L / 2) sm.st_raw(s.t + r * TS, hk[r]);
    if (s.t == 0) sm.st_raw(0, hk[0]);
    __syncthreads();
    if (!valid) return;
    C *aw = static_cast<C *>(d.aw);
    const R s2 = scale2<R>(a);
    auto emit = [&](int k, CV<V> Y) {
        const C q2 = lane1<R>(Y);
        const R f = s2 * (R)k;
        if (FLAME_IN(d.status, 2 * ((long long)k * a.n1 + row) + 1, uv_len(a), kSiteAdjAw))
            st_uv<R>(aw + 2 * ((size_t)k * a.n1 + row), lane0<R>(Y), C{f * q2.y, -f * q2.x});  // -i f q2
    };
#pragma unroll
    for (int r = 0; r < ES; ++r) {
        if (TS * r > L / 2) continue;
        const int k = s.t + r * TS, kc = L - k;
        if (k <= L / 2 && (k <= a.K2 || kc <= a.K2)) {
            CV<V> lo, hi;
            real_post(hk[r], sm.ld_raw(k == 0 ? 0 : kc), __ldg(P + k), lo, hi);
            if (k <= a.K2) emit(k, lo);
            if (kc <= a.K2 && kc != k) emit(kc, hi);
        }
    }
}

// One column per group: forward column transforms of (hat q1, -i k2 hat q2),
// P = (-i s1 k1 Q1 + Q2) / (N1 N2), lambda update on the box, k2 = 0 column
// from its k1 > 0 half, dL/dgamma contribution (FP64, one atomic per block).
template <class R, int A> __global__ void __launch_bounds__(256, kMinBlocks<R>) k_adjC(AdjDesc d) {
    using V = typename VecOf<R>::type;
    using C = CplxT<R>;
    using PL = Plan3<A, adj_f<R>(A)>;
    constexpr int F = PL::F, L = PL::L, TS = PL::TS, SL = PL::slots(kSlotsPerWave<V>);
    extern __shared__ __align__(128) unsigned char smstep[];
    __shared__ double red[256];
    const StepArgs &a = d.a;
    griddep_wait();
    const int G = blockDim.x / TS, ld1 = 2 * a.K1 + 1;
    const Place s = place_all<TS>(), p = place<PL::TP>(G);
    const CoefR<R> cfs = load_coef<R>(d.coef);  // derived by k_adjL
    CV<V> xp[PL::EP];
    {
        const int k2 = blockIdx.x * G + p.line;
        const C *aw = static_cast<const C *>(d.aw) + 2 * (size_t)k2 * L;
#pragma unroll
        for (int i = 0; i < PL::EP; ++i) {
            const int n = p.t + i * PL::TP;
            const bool in = p.on && k2 <= a.K2 && FLAME_IN(d.status, 2 * ((long long)k2 * L + n) + 1, uv_len(a), kSiteAdjAw);
            const UV<R> e = in ? ld_uv<R>(aw + 2 * n) : UV<R>{C{0, 0}, C{0, 0}};
            xp[i] = pack2<R>(e.u, e.v);
        }
    }
    auto buf = [&](int line) { return planes3<V, R>(smstep, line, SL); };
    CV<V> xs[PL::ES];
    forward3<PL, true>(xp, xs, p, s, buf, tab3<R, A, F, C>(d.tw1));
    griddep_launch();
    const int k2 = blockIdx.x * G + s.line;
    const bool lin = !(a.flags & kNonlinearOnly), nl = !(a.flags & kLinearOnly);
    const R ra = cfs.a, rb = cfs.b, rcs = cfs.cs, rdt = cfs.dt;
    const R s1 = scale1<R>(a), s2 = scale2<R>(a);
    const C *lam = static_cast<const C *>(d.lam) + (size_t)k2 * ld1 + a.K1;
    C *lout = static_cast<C *>(d.lam_out) + (size_t)k2 * ld1 + a.K1;
    const C *phi = static_cast<const C *>(d.state) + (size_t)k2 * ld1 + a.K1;
    double dg = 0.0;  // sum of 2 kappa (lambda . Phi); times dt / (2 r0) at the end
#pragma unroll
    for (int r = 0; r < PL::ES; ++r) {
        if (r >= F && r < 2 * F) continue;
        const int n = s.t + r * TS, k1 = r < F ? n : n - L;
        const bool in_box = k2 <= a.K2 && (r < F ? n <= a.K1 : k1 >= -a.K1);
        // k2 = 0, k1 < 0: conjugate mirror of +k1, written (and counted in
        // the gamma gradient, with the same value) by the owner of +k1
        if (!in_box || (k1 == 0 && k2 == 0) || (k2 == 0 && k1 < 0)) continue;
        const long long bi = (long long)k2 * ld1 + a.K1 + k1;
        if (!FLAME_IN(d.status, bi, box_len(a), kSiteAdjLam) || !FLAME_IN(d.status, bi, box_len(a), kSiteAdjState)) continue;
        const R f1 = s1 * (R)k1;
        const C Q1 = lane0<R>(xs[r]), Q2 = lane1<R>(xs[r]);
        const C Pk{f1 * Q1.y + Q2.x, -f1 * Q1.x + Q2.y};  // -i f1 Q1 + Q2
        const C l = lam[k1];
        R kap;
        if (sizeof(R) == 8 && d.kap) kap = static_cast<const R *>(d.kap)[bi];
        else kap = kappa_norm<R>(f1, s2 * (R)k2);
        if (lin) {
            const C ph = phi[k1];
            // weight 2: k2 > 0 stands for +-k; k2 = 0 here counts +k1 and -k1
            dg += 2.0 * (double)kap * ((double)l.x * ph.x + (double)l.y * ph.y);
        }
        const R om = lin ? kap * (rb - kap * ra) : (R)0;
        const R cn = nl ? rcs : (R)0;
        const C nw{l.x + rdt * (om * l.x + cn * Pk.x), l.y + rdt * (om * l.y + cn * Pk.y)};
        lout[k1] = nw;
        if (k2 == 0 && FLAME_IN(d.status, a.K1 - k1, box_len(a), kSiteAdjLam)) lout[-k1] = C{nw.x, -nw.y};
    }
    const double sum = cta_sum(dg, red);
    if (threadIdx.x == 0 && sum != 0.0) atomicAdd(d.dgamma, sum * d.coef[10]);
}

}  // namespace flame
