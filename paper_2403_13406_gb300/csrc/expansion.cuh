// expansion.cuh -- the entropic relaxation parameter from the expansion of the entropy about the
// equilibrium.
//
// With B(t) = sum_k B_k(t delta_k) (systems.cuh) the root t* > 0 of B(t) = B(-1) is all that the
// relaxation needs.  B(t) = c_2 t^2 + c_3 t^3 + ..., and the coefficients have closed forms, so a
// smooth cell needs no evaluation of B: dividing B(t) - B(-1) by t + 1 leaves
//   H(e) = sum_n c_n P_n(1 + e) = 0,  P_n(t) = (t^n - (-1)^n) / (t + 1) = t P_{n-1}(t) - (-1)^n,  P_1 = 1,
// whose root e = t* - 1 = -c_3 / c_2 + ... has full relative precision however close the cell is to
// equilibrium: B(1) - B(-1), in which all digits cancel there, is never formed.
//
// Coefficients, with q = delta / f in the smooth limit:
//  - scalar systems: d B_k / d h = 2 h / (D (1 + sqrt(1 + x))) with D = D2_k, x = b12_k h / D^2, and
//    2 / (1 + sqrt(1 + x)) = sum_n C_n (-x / 4)^n with the Catalan numbers C_n, hence
//    c_{n+2} = C_n / (n + 2) sum_k (delta_k^2 / D_k) y_k^n,  y_k = -b12_k delta_k / (4 D_k^2).
//  - shallow water: a population is a function of eta = h_1 / f_1, R = sign (h_d - v_d h_1) / (f_1 c) and
//    kappa = g h / (2 c^2) alone (c = nu + sign v_d; f_1 its equilibrium depth).  With beta = sign b / c
//    (b the dual velocity's deviation), along the axis B_k / (f_1 c^2) is the stationary value over beta of
//      Psi(beta) = kappa (eta + beta)^2 / (1 - beta) - R beta - (1 + eta) beta^2 / 2,
//    and across it the kinetic energy adds (h_t - v_t h_1)^2 / (2 f_1 (1 + eta)).  Psi is stationary, so beta to
//    order t^2 (beta_1, beta_2) gives B_k through t^5.
//
// The terms left out are bounded by the `size` of the cell, the ratio of successive terms: up to `most` (of
// SmoothRoot and Expansion) the root of the truncated H is the root to the rounding of omega.  Rougher cells
// take rough_root: Newton on B(t) - B(-1) from the truncated root, with B in the forms above (for
// shallow water z = (eta + beta) / (1 - beta), (1 + z)(1 - beta) = 1 + eta, turns the stationarity of Psi into a
// cubic in z), and what that does not certify, the general safeguarded search (entropic_omega).
// Worst error of omega over 60 000 random cells per system (1D and 2D shallow water and Burgers, deviations of 1e-7 ...
// 0.5 of f, states up to the edge of the domain), against a bisection in 113 bits, by the cell's place in the domain
// ((|v| + sqrt(g h)) / nu, or |c u| / V q / 2, below 0.9 / 0.99 / 0.999 / 0.99999):
//   FP32  smooth  6e-8 / 2e-7 / 2e-6 / 1e-5    rough  6e-6 / 4e-6 / 6e-5 / 6e-4    general search  3e-3 / 2e-3 / 3e-2 / 1
//   FP64  smooth  4e-17 / 9e-17 / 3e-16 / 2e-15   rough  1.2e-14 / 5e-15 / 7e-14 / 1e-12   general  2e-14 / 3e-14 / 3e-13 / 3e-2
// Both round to nearest: next to the edge the diagnostics' bar of 64 roundings (7.6e-6 in FP32) is exceeded in 0.1 % of
// such cells, on the general search alone in 1.3 %.
//
// The root-find bounds every entropic kernel (instruction issue in FP32, the FP64 pipe, 2 lanes a clock
// and SM, in FP64).  Two evaluations of B by inner Newton solves, a quartic model through them and its
// certificate took 652 thread instructions per 1D shallow-water cell-stage in all; with the expansion 299.
// Before -> after: 1D shallow water N = 2^20, FP32, 409 -> 186 us per step; 2D Burgers 4096^2, FP32, 296 -> 141 us
// per stage; 1D shallow water N = 100003, FP64, 3.26 -> 0.82 ms per step.  With the populations in packed pairs and
// two coefficients for very smooth cells (SmoothRoot) 215 instructions, 137 us per step and 110 us per stage (FP32).
#pragma once

#include "systems.cuh"

namespace eslbm {

// Reciprocal and square root of normal positive numbers to about one unit in the last place: the
// hardware's approximation, in FP64 with one third-order step of Newton's iteration for 1/x (relative
// error e -> e^3) and of the binomial series for 1/sqrt(x) (e -> 5/16 e^3).
__host__ __device__ __forceinline__ float rcp_fast(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}
__host__ __device__ __forceinline__ double rcp_fast(double x)
{
#ifdef __CUDA_ARCH__
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
#else
    return 1.0 / x;
#endif
}
__host__ __device__ __forceinline__ float sqrt_fast(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return sqrtf(x);
#endif
}
__host__ __device__ __forceinline__ double sqrt_fast(double x)
{
#ifdef __CUDA_ARCH__
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double s = x * r;
    const double e = fma(-s, r, 1.0);
    return fma(s, e * fma(e, 0.375, 0.5), s);
#else
    return sqrt(x);
#endif
}
template <class R> struct Eps;
template <> struct Eps<float> { static constexpr float value = 1.1920929e-7f; };
template <> struct Eps<double> { static constexpr double value = 2.220446049250313e-16; };

// Positive and far enough from the ends of the range that rcp_fast neither takes it for zero nor flushes its
// reciprocal (its argument is subnormal or above 2^126 in FP32, 2^1022 in FP64).
// FP64: from the upper word, off the FP64 pipe.
__host__ __device__ __forceinline__ bool ordinary(float x) { return x >= 0x1p-124f && x <= 0x1p124f; }
__host__ __device__ __forceinline__ bool ordinary(double x)
{
#ifdef __CUDA_ARCH__
    return (unsigned)__double2hiint(x) - (3u << 20) < (2040u << 20);
#else
    return x >= 0x1p-1020 && x < 0x1p1020;
#endif
}
// the upper bound alone, for x >= 0
__host__ __device__ __forceinline__ bool below_top(float x) { return x <= 0x1p124f; }
__host__ __device__ __forceinline__ bool below_top(double x)
{
#ifdef __CUDA_ARCH__
    return (unsigned)__double2hiint(x) < (2043u << 20);
#else
    return x < 0x1p1020;
#endif
}

// Root e of H(e) with c[n] the coefficient of t^(n + 2), N of them: the quadratic model of H about 0 (exact to
// e^5 relative to c_2), then in FP64 `steps` Newton steps on all of H.
template <class R, int N> __host__ __device__ __forceinline__ R expansion_root(const R *c, int steps)
{
    const R rc = rcp_fast(c[0]);
    R r[N];
#pragma unroll
    for (int n = 1; n < N; ++n) r[n] = c[n] * rc;
    // H and its first two derivatives at e = 0: P_n(1), P_n'(1), P_n''(1) / 2 up to n = 7
    R h0 = r[1], h1 = R(1) + r[1] + R(2) * r[2], h2 = r[1] + R(2) * r[2];
    if constexpr (N > 3) {
        h0 += r[3];
        h1 += R(2) * r[3];
        h2 += R(4) * r[3];
    }
    if constexpr (N > 4) h1 += R(3) * r[4];
    if constexpr (N > 5) h0 += r[5];
    const R g = rcp_fast(h1);
    R e = -h0 * g;
    e = -(h0 + h2 * e * e) * g;
    for (int i = 0; i < steps; ++i) {
        const R t = R(1) + e;
        R p = R(1) + e * t, H = e + r[1] * p;
        R sgn = R(-1);
#pragma unroll
        for (int n = 2; n < N; ++n) {
            p = t * p + sgn;
            H += r[n] * p;
            sgn = -sgn;
        }
        e -= H * rcp_fast(h1 + R(2) * h2 * e);
    }
    return e;
}

// Expansion<Sys, R>: build(P, u, delta) computes the coefficients c[0 .. N) of t^2 ... and `size`, the
// scale of successive terms; false outside the domain or for non-finite data.
template <class Sys, class R> struct Expansion;

template <int DIM, class R> struct Expansion<Scalar<DIM, true>, R> {
    static constexpr int Q = Lattice<DIM>::Q;
    static constexpr int N = sizeof(R) == 4 ? 6 : 8;
    // largest size at which the terms left out (286 y^8 of c_2) and the root's own error after one Newton step (y^7)
    // are below the FP64 rounding of omega (the mixed mode's evaluation; SmoothRoot holds FP32's); beyond most_rough
    // (4 y -> 1: the edge of the domain) the closed form does not help
    static constexpr R most = R(0.004);
    static constexpr R most_rough = R(0.2);
    R c[N], size;
    R a[Q], y[Q];

    __host__ __device__ __forceinline__ bool build(const ParamsR<R> &P, const R *u, const R *delta)
    {
        bool ok = true;
        R S[N];
#pragma unroll
        for (int n = 0; n < N; ++n) S[n] = R(0);
        size = R(0);
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const R cj = R(Lattice<DIM>::sign(k)) * P.c[Lattice<DIM>::axis(k)] * P.inv2V;
            const R D = R(1) / R(Q) + cj * u[0];
            ok &= D > R(0);
            const R dr = delta[k] * rcp_fast(D);
            a[k] = delta[k] * dr;
            y[k] = R(-0.5) * cj * (dr * rcp_fast(D));
            ok &= fabs(y[k]) <= most_rough;
            size = fmax(size, fabs(y[k]));
            R p = a[k];
            S[0] += p;
#pragma unroll
            for (int n = 1; n < N; ++n) {
                p *= y[k];
                S[n] += p;
            }
        }
        constexpr double cat[8] = {1.0 / 2, 1.0 / 3, 2.0 / 4, 5.0 / 5, 14.0 / 6, 42.0 / 7, 132.0 / 8, 429.0 / 9};
#pragma unroll
        for (int n = 0; n < N; ++n) c[n] = R(cat[n]) * S[n];
        return ok;
    }

    // B(t) and dB/dt
    __host__ __device__ __forceinline__ bool eval(R t, R &B, R &dB) const
    {
        R b = R(0), db = R(0);
        bool ok = true;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const R X = R(1) - R(4) * y[k] * t;
            ok &= X > R(0);
            const R s = sqrt_fast(X);
            const R q = rcp_fast(R(1) + s);
            const R aq = a[k] * q;
            db += aq;
            b += aq * (q * (R(1) + R(2) * s));
        }
        B = b * (t * t) * R(2.0 / 3.0);
        dB = db * (R(2) * t);
        return ok;
    }
};

template <int DIM, class R> struct Expansion<ShallowWater<DIM>, R> {
    static constexpr int Q = Lattice<DIM>::Q, M = DIM + 1;
    static constexpr int N = 4;
    // sizes measured as above: at most, the error is 1e-16 in FP64; three times that size multiplies it by 3^5
    static constexpr R most = R(3e-4);
    static constexpr R most_rough = R(2);
    R c[N], size;
    R kap[Q], cv[Q], eta[Q], rr[Q], w[Q], zt[Q], z1[Q], z2[Q];

    __host__ __device__ __forceinline__ bool build(const ParamsR<R> &P, const R *u, const R *delta)
    {
        bool ok = u[0] > R(0);
        const R rh = rcp_fast(u[0]);
        const R rf = R(2) * P.V * rh;          // 1 / f_1 = rf / c
        const R gh2 = R(0.5) * P.g * u[0];
        const R hV = u[0] * P.inv2V;
        const R nu = R(2) * P.V / R(Q);
        R v[DIM];
#pragma unroll
        for (int j = 0; j < DIM; ++j) v[j] = u[1 + j] * rh;
#pragma unroll
        for (int n = 0; n < N; ++n) c[n] = R(0);
        size = R(0);
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const int d = Lattice<DIM>::axis(k);
            const R sg = R(Lattice<DIM>::sign(k));
            const R ck = nu + sg * v[d];
            const R rc = rcp_fast(ck);
            const R rc2 = rc * rc;
            const R kp = gh2 * rc2;
            const R curv = R(1) - R(2) * kp;
            ok &= (ck > R(0)) & (curv > R(0));
            const R L = rcp_fast(curv);
            const R e1 = delta[k * M] * (rf * rc);
            const R R1 = (sg * rf * rc2) * (delta[k * M + 1 + d] - v[d] * delta[k * M]);
            const R A = (e1 - R1) * L;
            const R b1 = A - e1;
            const R wk = hV * ck * (ck * ck);
            const R A2 = A * A, Ab = A * b1, b11 = b1 * b1;
            const R n2 = kp * (R(2) * Ab + A2) - e1 * b1;  // (1 - 2 kappa) beta_2
            const R b2 = n2 * L;
            const R kA2 = kp * A2;
            const R sz = L * (fabs(e1 + R1) + R(6) * kp * fabs(A)) + fabs(A) + fabs(e1);
            ok &= sz <= most_rough;
            size = fmax(size, sz);
            c[0] += wk * (kp * (e1 * e1) + R(0.5) * curv * b11);
            c[1] += wk * (kA2 * b1 - R(0.5) * e1 * b11);
            c[2] += wk * (R(0.5) * b2 * n2 + kA2 * b11);
            c[3] += wk * (kp * (b2 * (b2 * (b1 + R(2) * A) + R(2) * Ab * (b1 + A)) + A2 * b11 * b1) -
                          R(0.5) * e1 * (b2 * b2));
            if constexpr (DIM == 2) {
                const R tau = delta[k * M + 2 - d] - v[1 - d] * delta[k * M];
                R z = R(0.5) * tau * tau * (rf * rc);
                zt[k] = z;
                c[0] += z;
                z *= -e1;
                c[1] += z;
                z *= -e1;
                c[2] += z;
                c[3] -= z * e1;
            }
            kap[k] = kp;
            cv[k] = curv;
            eta[k] = e1;
            rr[k] = R1;
            w[k] = wk;
            z1[k] = A;
            z2[k] = b2 + b1 * A;
        }
        return ok;
    }

    // B(t) and dB/dt.  z = (eta + beta) / (1 - beta) solves kappa z^3 + 3 kappa z^2 - k1 z + k0 = 0 (Newton from
    // the expansion, the populations in step); with R eliminated by the stationarity of Psi,
    //   Psi = kappa [(eta + z beta)^2 - 2 z^2 beta] + ((1 + eta) / 2 - kappa) beta^2
    // has no cancellation at leading order.
    __host__ __device__ __forceinline__ bool eval(R t, R &B, R &dB) const
    {
        constexpr R tol = R(sizeof(R) == 4 ? 1e-4 : 1e-9);
        R z[Q], k0[Q], k1[Q];
        bool ok = true, more = true;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const R et = t * eta[k];
            k1[k] = cv[k] + t * (eta[k] + rr[k]);
            k0[k] = t * (eta[k] - rr[k]) + et * et;
            z[k] = t * (z1[k] + t * z2[k]);
        }
        for (int it = 0; it < 6 && more; ++it) {
            more = false;
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const R g = k0[k] + z[k] * (kap[k] * z[k] * (R(3) + z[k]) - k1[k]);
                const R gp = R(3) * kap[k] * z[k] * (R(2) + z[k]) - k1[k];
                ok &= gp < R(0);
                const R dz = g * rcp_fast(gp);
                z[k] -= dz;
                more |= !(fabs(dz) <= tol * fabs(z[k]));
            }
        }
        ok &= !more;
        R b = R(0), db = R(0);
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const R et = t * eta[k], m = R(1) + et;
            const R q = R(1) + z[k];
            ok &= (m > R(0)) & (q > R(0));
            const R be = (z[k] - et) * rcp_fast(q);
            const R b2 = be * be, x = et + z[k] * be;
            b += w[k] * (kap[k] * (x * x - R(2) * z[k] * z[k] * be) + R(0.5) * (cv[k] + et) * b2);
            db += w[k] * ((R(2) * kap[k] * z[k] - R(0.5) * b2) * eta[k] - be * rr[k]);
            if constexpr (DIM == 2) {
                const R rm = rcp_fast(m), q2 = zt[k] * t * rm;
                b += q2 * t;
                db += q2 * (R(1) + rm);
            }
        }
        B = b;
        dB = db;
        return ok;
    }
};

// Two values, one for each of a pair of opposite populations (k and k + Q/2): on the device pairs of FP32
// are the packed operands of one instruction, so the common path issues half as many.
template <class R> struct Two {
    R x, y;
};
template <class R> __host__ __device__ __forceinline__ Two<R> two(R x, R y) { return {x, y}; }
template <class R> __host__ __device__ __forceinline__ Two<R> two(R x) { return {x, x}; }
template <class R> __host__ __device__ __forceinline__ Two<R> fma2(const Two<R> &a, const Two<R> &b, const Two<R> &c)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(R) == 4) {
        const float2 r = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), make_float2(c.x, c.y));
        return {r.x, r.y};
    }
#endif
    return {fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}
template <class R> __host__ __device__ __forceinline__ Two<R> operator*(const Two<R> &a, const Two<R> &b)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(R) == 4) {
        const float2 r = __fmul2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
        return {r.x, r.y};
    }
#endif
    return {a.x * b.x, a.y * b.y};
}
template <class R> __host__ __device__ __forceinline__ Two<R> operator+(const Two<R> &a, const Two<R> &b)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(R) == 4) {
        const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
        return {r.x, r.y};
    }
#endif
    return {a.x + b.x, a.y + b.y};
}
template <class R> __host__ __device__ __forceinline__ Two<R> rcp2(const Two<R> &a) { return {rcp_fast(a.x), rcp_fast(a.y)}; }

// SmoothRoot<Sys, R>::find: the root e of a smooth cell from the expansion (the terms of Expansion, in pairs of
// populations); false where the cell is too rough for it or outside the domain.  Its measure of roughness is
// the sum of squares sq of the terms' ratios.  Very smooth cells (FP32, up to `few`: the terms of order
// size^3 in omega are below its rounding) need c_2 and c_3 only: e = -c_3 / (c_2 + c_3).  c_2 scales with the square of
// the fields (h V^2 size^2 for shallow water): in thin films, h of 1e-21 and below in FP32, it is subnormal while the
// deviation is ordinary, rcp_fast takes it for zero and e is infinite or NaN, which omega_of refuses.
template <class Sys, class R> struct SmoothRoot;

template <int DIM, class R> struct SmoothRoot<Scalar<DIM, true>, R> {
    static constexpr int Q = Lattice<DIM>::Q;
    static constexpr int N = Expansion<Scalar<DIM, true>, R>::N;
    static constexpr R few = sizeof(R) == 4 ? R(2.5e-3) : R(0);
    static constexpr R most = sizeof(R) == 4 ? R(0.04) : R(0.004);

    __host__ __device__ static __forceinline__ bool find(const ParamsR<R> &P, const R *u, const R *delta, R &e)
    {
        Two<R> S0 = two(R(0)), S1 = two(R(0)), sq = two(R(0)), y[Q / 2], p[Q / 2];
        bool ok = true;
#pragma unroll
        for (int k = 0; k < Q / 2; ++k) {
            const R cj = P.c[Lattice<DIM>::axis(k)] * P.inv2V;
            const R s = cj * u[0];
            ok &= fabs(s) < R(1) / R(Q);
            const Two<R> rD = rcp2(two(R(1) / R(Q) + s, R(1) / R(Q) - s));
            const Two<R> d = two(delta[k], delta[k + Q / 2]);
            const Two<R> dr = d * rD, a = d * dr;
            y[k] = dr * (rD * two(R(-0.5) * cj, R(0.5) * cj));
            sq = fma2(y[k], y[k], sq);
            p[k] = a * y[k];
            S0 = S0 + a;
            S1 = S1 + p[k];
        }
        const R q = sq.x + sq.y;
        const R s0 = S0.x + S0.y, s1 = S1.x + S1.y;
        // (2 c_2 from the top of the range: rcp_fast would flush its reciprocal)
        if (!(ok && q <= most * most && below_top(s0))) return false;
        constexpr R tiny = Eps<R>::value / R(16);
        if (sizeof(R) == 4 && q <= few * few) {
            const R c3 = s1 * R(2.0 / 3.0);  // over c_2 = s0 / 2
            e = q <= tiny * tiny ? R(0) : -c3 * rcp_fast(s0 + c3);
            return true;
        }
        if (q <= tiny * tiny) {
            e = R(0);
            return true;
        }
        constexpr double cat[8] = {1.0 / 2, 1.0 / 3, 2.0 / 4, 5.0 / 5, 14.0 / 6, 42.0 / 7, 132.0 / 8, 429.0 / 9};
        R c[N];
        c[0] = R(cat[0]) * s0;
        c[1] = R(cat[1]) * s1;
#pragma unroll
        for (int n = 2; n < N; ++n) {
            Two<R> S = two(R(0));
#pragma unroll
            for (int k = 0; k < Q / 2; ++k) {
                p[k] = p[k] * y[k];
                S = S + p[k];
            }
            c[n] = R(cat[n]) * (S.x + S.y);
        }
        e = expansion_root<R, N>(c, sizeof(R) == 4 ? 0 : 1);
        return true;
    }
};

template <int DIM, class R> struct SmoothRoot<ShallowWater<DIM>, R> {
    static constexpr int Q = Lattice<DIM>::Q, M = DIM + 1;
    static constexpr R few = sizeof(R) == 4 ? R(2e-3) : R(0);
    static constexpr R most = sizeof(R) == 4 ? R(0.02) : R(3e-4);

    __host__ __device__ static __forceinline__ bool find(const ParamsR<R> &P, const R *u, const R *delta, R &e)
    {
        const R rh = rcp_fast(u[0]);
        const R rf = R(2) * P.V * rh;  // 1 / f_1 = rf / c
        const R gh = P.g * u[0], gh2 = R(0.5) * gh;
        const R hV = u[0] * P.inv2V;
        const R nu = R(2) * P.V / R(Q);
        bool ok = u[0] > R(0);
        Two<R> C2 = two(R(0)), C3 = two(R(0)), sq = two(R(0));
        Two<R> kp[Q / 2], e1[Q / 2], A[Q / 2], b1[Q / 2], w[Q / 2], L[Q / 2], zt[Q / 2];
#pragma unroll
        for (int k = 0; k < Q / 2; ++k) {
            constexpr int H = Q / 2;
            const int d = Lattice<DIM>::axis(k);
            const R v = u[1 + d] * rh;
            const R t = nu - fabs(v);  // min c
            ok &= (t > R(0)) & (t * t > gh);
            const Two<R> c = two(nu + v, nu - v);
            const Two<R> rc = rcp2(c), rc2 = rc * rc;
            kp[k] = two(gh2) * rc2;
            const Two<R> cv = fma2(two(R(-2)), kp[k], two(R(1)));
            L[k] = rcp2(cv);
            const Two<R> d0 = two(delta[k * M], delta[(k + H) * M]);
            const Two<R> d1 = two(delta[k * M + 1 + d], delta[(k + H) * M + 1 + d]);
            const Two<R> frc = two(rf) * rc;
            e1[k] = d0 * frc;
            const Two<R> r1 = (rc2 * two(rf, -rf)) * fma2(two(-v), d0, d1);
            A[k] = fma2(two(R(-1)), r1, e1[k]) * L[k];
            b1[k] = fma2(two(R(-1)), e1[k], A[k]);
            w[k] = (two(hV) * c) * (c * c);
            const Two<R> e11 = e1[k] * e1[k], A2 = A[k] * A[k], b11 = b1[k] * b1[k];
            sq = fma2(L[k] * L[k], e11 + A2, sq);
            C2 = fma2(w[k], fma2(kp[k], e11, (two(R(0.5)) * cv) * b11), C2);
            C3 = fma2(w[k], fma2(kp[k] * A2, b1[k], (two(R(-0.5)) * e1[k]) * b11), C3);
            if constexpr (DIM == 2) {
                const R vt = u[2 - d] * rh;
                const Two<R> d2 = two(delta[k * M + 2 - d], delta[(k + H) * M + 2 - d]);
                const Two<R> tau = fma2(two(-vt), d0, d2);
                const Two<R> z = (two(R(0.5)) * frc) * (tau * tau);
                zt[k] = z * e1[k];
                C2 = C2 + z;
                C3 = fma2(two(R(-1)), zt[k], C3);
            }
        }
        const R q = sq.x + sq.y;
        if (!(ok && q <= most * most)) return false;
        constexpr R tiny = Eps<R>::value / R(64);
        R c[4];
        c[0] = C2.x + C2.y;
        c[1] = C3.x + C3.y;
        if (q <= tiny * tiny) {  // |e| <= 4 size; c_2 may have underflowed
            e = R(0);
            return true;
        }
        if (sizeof(R) == 4 && q <= few * few) {
            e = -c[1] * rcp_fast(c[0] + c[1]);
            return true;
        }
        Two<R> C4 = two(R(0)), C5 = two(R(0));
#pragma unroll
        for (int k = 0; k < Q / 2; ++k) {
            const Two<R> Ab = A[k] * b1[k], A2 = A[k] * A[k], b11 = b1[k] * b1[k], kA2 = kp[k] * A2;
            const Two<R> n2 = fma2(kp[k], fma2(two(R(2)), Ab, A2), (two(R(-1)) * e1[k]) * b1[k]);
            const Two<R> b2 = n2 * L[k];
            C4 = fma2(w[k], fma2(two(R(0.5)) * b2, n2, kA2 * b11), C4);
            const Two<R> in = fma2(b2, fma2(two(R(2)), A[k], b1[k]), two(R(2)) * Ab * (b1[k] + A[k]));
            const Two<R> s5 = fma2(kp[k] * b2, in, kA2 * (b11 * b1[k]));
            C5 = fma2(w[k], fma2(two(R(-0.5)) * e1[k], b2 * b2, s5), C5);
            if constexpr (DIM == 2) {
                const Two<R> z = zt[k] * e1[k];
                C4 = C4 + z;
                C5 = fma2(two(R(-1)) * z, e1[k], C5);
            }
        }
        c[2] = C4.x + C4.y;
        c[3] = C5.x + C5.y;
        e = expansion_root<R, 4>(c, sizeof(R) == 4 ? 0 : 1);
        return true;
    }
};

// Cells too rough for the truncated expansion: Newton on B(t) - B(-1) from its root; then the general search.
template <class Sys, class R>
__host__ __device__ __forceinline__ bool rough_root(const ParamsR<R> &P, const R *u, const R *delta, R &omega)
{
    Expansion<Sys, R> X;
    if (!X.build(P, u, delta)) return false;
    R E0, dE0;
    if (!X.eval(R(-1), E0, dE0) || !(E0 > R(0))) return false;
    R t = R(1) + expansion_root<R, Expansion<Sys, R>::N>(X.c, 0);
    if (!(t > R(0.25) && t < R(2))) t = R(1);
    constexpr R tol = R(sizeof(R) == 4 ? 1e-4 : 1e-9);
    R dt = R(1), dB = R(1);
    for (int it = 0; it < 8; ++it) {
        R B;
        if (!X.eval(t, B, dB) || !ordinary(dB)) return false;
        dt = (B - E0) * rcp_fast(dB);
        t -= dt;
        if (!(t > R(0.1) && t < R(2.5))) return false;
        if (fabs(dt) <= tol) break;
    }
    if (!(fabs(dt) <= tol && t < P.t_max)) return false;
    // (the Newton point of a convex F lies above its root by less than dt^2, below the rounding of omega)
    omega = R(1) + t;
    return true;
}

// omega of a cell that the truncated expansion does not certify; out of line, so that its registers do
// not add to those of the kernels' common path
template <class Sys, class R>
__device__ __noinline__ R rough_omega(const ParamsR<R> &P, const R *u, const R *delta, bool &fallback)
{
    R w;
    if (rough_root<Sys, R>(P, u, delta, w)) {
        fallback = false;
        return w;
    }
    typename Sys::template Ctx<R> cx;
    Sys::template prepare<R>(P, u, delta, cx);
    return entropic_omega<Sys, R>(P, cx, fallback);
}

// omega = 1 + t* (no root: 1, and fallback is set)
template <class Sys, class R>
__device__ __forceinline__ R omega_of(const ParamsR<R> &P, const R *u, const R *delta, bool &fallback)
{
    R e;
    // (a smooth cell's |e| is a few times its size, at most 0.2; the lower bound refuses -infinity)
    if (SmoothRoot<Sys, R>::find(P, u, delta, e) && e > R(-0.5) && e < P.e_max) {
        fallback = false;
        return R(2) + e;
    }
    R uu[Sys::M], dd[Sys::Q * Sys::M];
#pragma unroll
    for (int m = 0; m < Sys::M; ++m) uu[m] = u[m];
#pragma unroll
    for (int i = 0; i < Sys::Q * Sys::M; ++i) dd[i] = delta[i];
    bool fb = false;
    const R w = rough_omega<Sys, R>(P, uu, dd, fb);
    fallback = fb;
    return w;
}

}  // namespace eslbm
