// Device math for the PixVOD sweep kernels: SE(3) exponential / logarithm,
// packed symmetric storage, Cholesky factorisation and triangular solves.
// Templated on the arithmetic type (float for the production path, double for
// the verification path).
//
// se(3) convention (App. C.2): xi = [theta; rho], Exp(xi) = (Exp_SO3(theta),
// V(theta) rho), V = I + B [theta]x + C [theta]x^2, A = sin t / t,
// B = (1 - cos t)/t^2, C = (t - sin t)/t^3 with t = |theta|.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

// Every function here is also compiled for the host (PV_HD), so that the same
// arithmetic can be exercised by host-side checks; on the device the scalar
// wrappers below select CUDA's device functions.
#define PV_HD __host__ __device__ __forceinline__

namespace pv {

// ---------------------------------------------------------------------------
// scalar wrappers (precise CUDA math functions, selected by type)
// ---------------------------------------------------------------------------
PV_HD float v_fma(float a, float b, float c) { return fmaf(a, b, c); }
PV_HD double v_fma(double a, double b, double c) { return fma(a, b, c); }
PV_HD float v_sqrt(float x) { return sqrtf(x); }
PV_HD double v_sqrt(double x) { return sqrt(x); }
PV_HD float v_exp(float x) { return expf(x); }
PV_HD double v_exp(double x) { return exp(x); }
PV_HD float v_atan2(float y, float x) { return atan2f(y, x); }
PV_HD double v_atan2(double y, double x) { return atan2(y, x); }
PV_HD float v_floor(float x) { return floorf(x); }
PV_HD double v_floor(double x) { return floor(x); }
PV_HD float v_abs(float x) { return fabsf(x); }
PV_HD double v_abs(double x) { return fabs(x); }
PV_HD bool v_finite(float x) { return isfinite(x); }
PV_HD bool v_finite(double x) { return isfinite(x); }
// reciprocal square root and quotient: the float path uses the approximate
// hardware forms (a few ulp), the double (verification) path the exact ones
#ifdef __CUDA_ARCH__
PV_HD void v_sincos(float x, float* s, float* c) { sincosf(x, s, c); }
PV_HD void v_sincos(double x, double* s, double* c) { sincos(x, s, c); }
PV_HD float v_rsqrt(float x) { return rsqrtf(x); }
PV_HD double v_rsqrt(double x) { return rsqrt(x); }
PV_HD float v_div(float a, float b) { return __fdividef(a, b); }
#else
PV_HD void v_sincos(float x, float* s, float* c) { *s = sinf(x); *c = cosf(x); }
PV_HD void v_sincos(double x, double* s, double* c) { *s = sin(x); *c = cos(x); }
PV_HD float v_rsqrt(float x) { return 1.0f / sqrtf(x); }
PV_HD double v_rsqrt(double x) { return 1.0 / sqrt(x); }
PV_HD float v_div(float a, float b) { return a / b; }
#endif
PV_HD double v_div(double a, double b) { return a / b; }

// Precision-dependent series limits: below ab_series_max the A/B quotients use
// their power series to t^6; below 1 rad (C) and d_series_max (D) the other
// coefficients use their power series with enough terms for the type's epsilon.
template <typename T> struct Prec;
// Float: below ab_series_max = 0.3 rad the A/B series truncate below 2e-10, and
// the logarithm recovers the angle from s = sin(t) with the arcsine series to
// s^9 when s < 0.2 and cos(t) > 0 (truncation below 5e-10), so small rotations
// need no trigonometric calls.
template <> struct Prec<float> {
    static constexpr int c_terms = 7;
    static constexpr float d_series_max = 1.0f;
    static constexpr float ab_series_max = 0.3f;
    static constexpr float asin_series_max = 0.2f;
};
template <> struct Prec<double> {
    static constexpr int c_terms = 12;
    static constexpr double d_series_max = 0.5;
    static constexpr double ab_series_max = 1e-8;
    static constexpr double asin_series_max = 0.0;
};

// (t - sin t)/t^3 = sum_k (-1)^k t^(2k) / (2k+3)!, k < c_terms, evaluated in
// Horner form with the coefficients computed at compile time
__host__ __device__ constexpr double series_C_coef(int k) {
    double f = 1.0;
    for (int i = 2; i <= 2 * k + 3; ++i) f *= double(i);
    return (k % 2 ? -1.0 : 1.0) / f;
}

template <typename T, int K, int N>
PV_HD T series_C_from(T t2) {
    constexpr double c = series_C_coef(K);
    if constexpr (K + 1 < N)
        return T(c) + t2 * series_C_from<T, K + 1, N>(t2);
    else
        return T(c);
}

template <typename T>
PV_HD T series_C(T t2) {
    return series_C_from<T, 0, Prec<T>::c_terms>(t2);
}

// D(t) = (1 - A/(2B))/t^2 = 1/t^2 - cot(t/2)/(2t), the [theta]x^2 coefficient of
// V^-1; from the Laurent series of cot: 1/12 + t^2/720 + t^4/30240 + t^6/1209600
// + t^8/47900160 + t^10/1892437580.3 + ... (used below d_series_max).
template <typename T>
PV_HD T series_D(T t2) {
    return T(1) / T(12) + t2 * (T(1) / T(720) + t2 * (T(1) / T(30240) + t2 * (T(1) / T(1209600) +
           t2 * (T(1) / T(47900160) + t2 * (T(1) / T(1892437580.3183))))));
}

// sin t / t = 1 - t^2/3! + t^4/5! - t^6/7!; (1 - cos t)/t^2 = 1/2! - t^2/4! + t^4/6! - t^6/8!
template <typename T>
PV_HD void series_AB(T t2, T* A, T* B) {
    *A = T(1) - t2 * (T(1) / T(6) - t2 * (T(1) / T(120) - t2 * (T(1) / T(5040))));
    *B = T(0.5) - t2 * (T(1) / T(24) - t2 * (T(1) / T(720) - t2 * (T(1) / T(40320))));
}

template <typename T>
PV_HD void coef_AB(T t, T* A, T* B) {
    if (t < Prec<T>::ab_series_max) {
        series_AB(t * t, A, B);
    } else {
        T s, c, sh, ch;
        v_sincos(t, &s, &c);
        v_sincos(T(0.5) * t, &sh, &ch);
        *A = s / t;
        T q = sh / (T(0.5) * t);
        *B = T(0.5) * q * q;
    }
}

template <typename T>
PV_HD T coef_C(T t, T A) {
    if (t < T(1)) return series_C(t * t);
    return (T(1) - A) / (t * t);
}

template <typename T>
PV_HD T coef_D(T t, T A, T B) {
    if (t < Prec<T>::d_series_max) return series_D(t * t);
    return (T(1) - A / (T(2) * B)) / (t * t);
}

// ---------------------------------------------------------------------------
// 3x3 helpers (row-major)
// ---------------------------------------------------------------------------
template <typename T>
PV_HD void mat3_mul(const T* a, const T* b, T* c) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            c[3 * i + j] = a[3 * i] * b[j] + a[3 * i + 1] * b[3 + j] + a[3 * i + 2] * b[6 + j];
}

template <typename T>
PV_HD void mat3_vec(const T* a, const T* x, T* y) {
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = a[3 * i] * x[0] + a[3 * i + 1] * x[1] + a[3 * i + 2] * x[2];
}

template <typename T>
PV_HD void mat3T_vec(const T* a, const T* x, T* y) {
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = a[i] * x[0] + a[3 + i] * x[1] + a[6 + i] * x[2];
}

// M = I + a W + b W^2 for W = [w]x, using W^2 = w w^T - |w|^2 I
template <typename T>
PV_HD void so3_poly(const T* w, T a, T b, T* M) {
    T t2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    M[0] = T(1) + b * (w[0] * w[0] - t2);
    M[4] = T(1) + b * (w[1] * w[1] - t2);
    M[8] = T(1) + b * (w[2] * w[2] - t2);
    M[1] = -a * w[2] + b * w[0] * w[1];
    M[3] = a * w[2] + b * w[0] * w[1];
    M[2] = a * w[1] + b * w[0] * w[2];
    M[6] = -a * w[1] + b * w[0] * w[2];
    M[5] = -a * w[0] + b * w[1] * w[2];
    M[7] = a * w[0] + b * w[1] * w[2];
}

// Exp: xi (6) -> R (9), t (3). Below ab_series_max the coefficients come from
// their power series in t^2, so small rotations take no square root, division
// or trigonometric call.
// Exp with V(theta) (t = V rho) returned as well (the adjoint uses it)
template <typename T>
PV_HD void se3_exp_V(const T* xi, T* R, T* t, T* V) {
    T t2 = xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2];
    T A, B, C;
    if (t2 < Prec<T>::ab_series_max * Prec<T>::ab_series_max) {
        series_AB(t2, &A, &B);
        C = series_C(t2);
    } else {
        T th = v_sqrt(t2);
        coef_AB(th, &A, &B);
        C = coef_C(th, A);
    }
    so3_poly(xi, A, B, R);
    so3_poly(xi, B, C, V);
    mat3_vec(V, xi + 3, t);
}

// Log: R (9), t (3) -> xi (6); rotation angles below pi. With w = vee(R - R^T)/2,
// s = |w| = sin(t) and c = cos(t): theta = w t / s = w / A. For s below
// asin_series_max (and c > 0) t / s = asin(s) / s comes from the arcsine series
// 1 + s^2/6 + 3 s^4/40 + 5 s^6/112 + 35 s^8/1152 and t^2 = s^2 (t / s)^2, so small
// rotations take no square root, division or trigonometric call.
// The logarithm from w = vee(R - R^T)/2, c = (tr R - 1)/2 and t (se3_log below
// computes w and c; the adjoint differentiates this part in w, c and t).
template <typename T>
PV_HD void se3_log_wct(T w0, T w1, T w2, T c, const T* t, T* xi, T* Vi) {
    static_assert(Prec<T>::asin_series_max <= Prec<T>::d_series_max / 2, "series D range");
    T s2 = w0 * w0 + w1 * w1 + w2 * w2;
    T ratio, D;
    if (s2 < Prec<T>::asin_series_max * Prec<T>::asin_series_max && c > T(0)) {
        ratio = T(1) + s2 * (T(1) / T(6) + s2 * (T(3) / T(40) + s2 * (T(5) / T(112) + s2 * (T(35) / T(1152)))));
        D = series_D(s2 * ratio * ratio);
    } else {
        T th = v_atan2(v_sqrt(s2), c);
        T A, B;
        coef_AB(th, &A, &B);
        ratio = T(1) / A;
        D = coef_D(th, A, B);
    }
    xi[0] = w0 * ratio;
    xi[1] = w1 * ratio;
    xi[2] = w2 * ratio;
    so3_poly(xi, T(-0.5), D, Vi);
    mat3_vec(Vi, t, xi + 3);
}

template <typename T>
PV_HD void se3_log(const T* R, const T* t, T* xi) {
    T Vi[9];
    se3_log_wct(T(0.5) * (R[7] - R[5]), T(0.5) * (R[2] - R[6]), T(0.5) * (R[3] - R[1]),
                T(0.5) * (R[0] + R[4] + R[8] - T(1)), t, xi, Vi);
}

// (R1, t1) * (R2, t2)
template <typename T>
PV_HD void se3_mul(const T* R1, const T* t1, const T* R2, const T* t2, T* R, T* t) {
    mat3_mul(R1, R2, R);
    mat3_vec(R1, t2, t);
    t[0] += t1[0];
    t[1] += t1[1];
    t[2] += t1[2];
}

// (R1, t1)^-1 * (R2, t2) = (R1^T R2, R1^T (t2 - t1))
template <typename T>
PV_HD void se3_invmul(const T* R1, const T* t1, const T* R2, const T* t2, T* R, T* t) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            R[3 * i + j] = R1[i] * R2[j] + R1[3 + i] * R2[3 + j] + R1[6 + i] * R2[6 + j];
    T d[3] = {t2[0] - t1[0], t2[1] - t1[1], t2[2] - t1[2]};
    mat3T_vec(R1, d, t);
}

// ---------------------------------------------------------------------------
// poses as unit quaternions (the sweep's Exp, Log and relative poses)
// ---------------------------------------------------------------------------
// q = (w, v) with rotation angle t: w = cos(t/2), v = sin(t/2) theta/t. Against
// rotation matrices, Exp, relative pose and Log take 110 instead of 172 FP
// operations per neighbour, in shorter dependent chains, and a pose held through
// the neighbour loop takes 7 registers instead of 12. Every fused operation here
// is written out, so a value does not depend on the kernel that computes it (the
// adjoint's recomputation of a sweep takes the same roundings).

template <typename T> constexpr bool is_scalar_v = false;
template <> constexpr bool is_scalar_v<float> = true;
template <> constexpr bool is_scalar_v<double> = true;

// number of terms of the small-angle series (angles below 0.3 rad)
template <typename T> struct QuatPrec;
template <> struct QuatPrec<float> {
    static constexpr int terms = 4;       // of cos(t/2), sin(t/2)/t and C: truncated below 1e-11
    static constexpr int asin_terms = 5;  // of asin(s)/s for s^2 < 0.0225: truncated below 2e-10
    static constexpr int d_terms = 4;     // of D: truncated below 2e-12
};
template <> struct QuatPrec<double> {
    static constexpr int terms = 9;
    static constexpr int asin_terms = 11;
    static constexpr int d_terms = 8;
};
constexpr double QUAT_T2_MAX = 0.09;    // Exp: squared angle below which the series are used
constexpr double QUAT_S2_MAX = 0.0223;  // Log: squared sine of the half angle below which they are

// sum_k (-x)^k / (2k + FIRST)! times 4^-k when HALF, k < N
template <typename T, int FIRST, bool HALF, int N>
PV_HD T quat_series(T x) {
    constexpr auto coef = [](int k) constexpr {
        double f = 1.0;
        for (int i = 2; i <= 2 * k + FIRST; ++i) f *= double(i);
        for (int i = 0; i < k && HALF; ++i) f *= 4.0;
        return (k % 2 ? -1.0 : 1.0) / f;
    };
    T r = T(coef(N - 1));
#pragma unroll
    for (int k = N - 2; k >= 0; --k) r = v_fma(r, x, T(coef(k)));
    return r;
}

// asin(s)/s = sum_k (2k)! / (4^k k!^2 (2k + 1)) s^(2k)
template <typename T, int N>
PV_HD T asin_series(T s2) {
    constexpr auto coef = [](int k) constexpr {
        double c = 1.0;
        for (int i = 0; i < k; ++i) c *= (2.0 * i + 1.0) / (2.0 * i + 2.0);
        return c / (2.0 * k + 1.0);
    };
    T r = T(coef(N - 1));
#pragma unroll
    for (int k = N - 2; k >= 0; --k) r = v_fma(r, s2, T(coef(k)));
    return r;
}

// D(t) = sum_k |B_2k+2| t^(2k) / (2k + 2)!, k < N (Bernoulli numbers)
template <typename T, int N>
PV_HD T d_series(T t2) {
    constexpr double c[8] = {1.0 / 12, 1.0 / 720, 1.0 / 30240, 1.0 / 1209600, 1.0 / 47900160,
                             691.0 / 1307674368000.0, 1.0 / 74724249600.0, 3617.0 / 510 / 20922789888000.0};
    T r = T(c[N - 1]);
#pragma unroll
    for (int k = N - 2; k >= 0; --k) r = v_fma(r, t2, T(c[k]));
    return r;
}

// c = a x b
template <typename T>
PV_HD void cross3(const T* a, const T* b, T* c) {
    c[0] = v_fma(a[1], b[2], -(a[2] * b[1]));
    c[1] = v_fma(a[2], b[0], -(a[0] * b[2]));
    c[2] = v_fma(a[0], b[1], -(a[1] * b[0]));
}
template <typename T>
PV_HD T dot3(const T* a, const T* b) {
    return v_fma(a[2], b[2], v_fma(a[1], b[1], a[0] * b[0]));
}

// Exp: xi (6) -> q (4: w, v), t (3) = V rho = rho + B theta x rho + C theta x (theta x rho)
template <typename T>
PV_HD void se3_exp_q(const T* xi, T* q, T* t) {
    const T t2 = dot3(xi, xi);
    T sh, C;  // sin(t/2)/t; C as in se3_exp_V
    if (t2 < T(QUAT_T2_MAX)) {
        constexpr int N = QuatPrec<T>::terms;
        q[0] = quat_series<T, 0, true, N>(t2);
        sh = T(0.5) * quat_series<T, 1, true, N>(t2);
        C = quat_series<T, 3, false, N>(t2);
    } else {
        const T th = v_sqrt(t2);
        T s;
        v_sincos(T(0.5) * th, &s, &q[0]);
        sh = s / th;
        C = coef_C(th, T(2) * sh * q[0]);
    }
    const T B = T(2) * (sh * sh);
    q[1] = sh * xi[0];
    q[2] = sh * xi[1];
    q[3] = sh * xi[2];
    T c[3], e[3];
    cross3(xi, xi + 3, c);
    cross3(xi, c, e);
#pragma unroll
    for (int i = 0; i < 3; ++i) t[i] = v_fma(C, e[i], v_fma(B, c[i], xi[3 + i]));
}

// Log: q, t (3) -> xi (6); rotation angles below pi
template <typename T>
PV_HD void se3_log_q(const T* q, const T* t, T* xi) {
    const T s2 = dot3(q + 1, q + 1);
    T ratio, D;  // theta = ratio v
    if (s2 < T(QUAT_S2_MAX)) {  // of either sign: -q is the same rotation, and v may vanish
        ratio = (q[0] < T(0) ? T(-2) : T(2)) * asin_series<T, QuatPrec<T>::asin_terms>(s2);
        D = d_series<T, QuatPrec<T>::d_terms>(s2 * (ratio * ratio));
    } else {
        const T s = v_sqrt(s2), w = v_abs(q[0]);
        const T th = T(2) * v_atan2(s, w);
        ratio = (q[0] < T(0) ? -th : th) / s;
        // (1 - (t/2) cot(t/2)) / t^2
        D = th < Prec<T>::d_series_max ? series_D(th * th) : (T(1) - T(0.5) * th * w / s) / (th * th);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) xi[i] = ratio * q[1 + i];
    T c[3], e[3];
    cross3(xi, t, c);
    cross3(xi, c, e);
#pragma unroll
    for (int i = 0; i < 3; ++i) xi[3 + i] = v_fma(D, e[i], v_fma(T(-0.5), c[i], t[i]));
}

// rotation matrix of q
template <typename T>
PV_HD void quat_matrix(const T* q, T* R) {
    const T x2 = q[1] + q[1], y2 = q[2] + q[2], z2 = q[3] + q[3];
    const T wx = q[0] * x2, wy = q[0] * y2, wz = q[0] * z2;
    R[0] = v_fma(-q[3], z2, v_fma(-q[2], y2, T(1)));
    R[4] = v_fma(-q[3], z2, v_fma(-q[1], x2, T(1)));
    R[8] = v_fma(-q[2], y2, v_fma(-q[1], x2, T(1)));
    R[1] = v_fma(q[1], y2, -wz);
    R[3] = v_fma(q[1], y2, wz);
    R[2] = v_fma(q[1], z2, wy);
    R[6] = v_fma(q[1], z2, -wy);
    R[5] = v_fma(q[2], z2, -wx);
    R[7] = v_fma(q[2], z2, wx);
}

// q = a b (S = 1) or conj(a) b (S = -1)
template <int S, typename T>
PV_HD void quat_mul(const T* a, const T* b, T* q) {
    const T av[3] = {S * a[1], S * a[2], S * a[3]};
    q[0] = v_fma(-av[2], b[3], v_fma(-av[1], b[2], v_fma(-av[0], b[1], a[0] * b[0])));
    q[1] = v_fma(-av[2], b[2], v_fma(av[1], b[3], v_fma(av[0], b[0], a[0] * b[1])));
    q[2] = v_fma(-av[0], b[3], v_fma(av[2], b[1], v_fma(av[1], b[0], a[0] * b[2])));
    q[3] = v_fma(-av[1], b[1], v_fma(av[0], b[2], v_fma(av[2], b[0], a[0] * b[3])));
}

// y = R(q) x (S = 1) or R(q)^T x (S = -1): x + 2 (v x (v x x) + S w v x x)
template <int S, typename T>
PV_HD void quat_rotate(const T* q, const T* x, T* y) {
    T c[3], e[3];
    cross3(q + 1, x, c);
    cross3(q + 1, c, e);
    const T w = S * q[0];
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = v_fma(T(2), v_fma(w, c[i], e[i]), x[i]);
}

// residual of an identity factor (Eq. 5) at the receiver (qi, ti) from a sender at
// Exp(xj): Log(Exp(xj)^-1 (qi, ti))
template <typename T>
PV_HD void se3_between(const T* xj, const T* qi, const T* ti, T* r) {
    T qj[4], tj[3], qr[4], tr[3];
    se3_exp_q(xj, qj, tj);
    quat_mul<-1>(qj, qi, qr);
    const T d[3] = {ti[0] - tj[0], ti[1] - tj[1], ti[2] - tj[2]};
    quat_rotate<-1>(qj, d, tr);
    se3_log_q(qr, tr, r);
}

// mean update: Log((q, t) Exp(tau))
template <typename T>
PV_HD void se3_update(const T* q, const T* t, const T* tau, T* xn) {
    T qt[4], tt[3], qn[4], tn[3];
    se3_exp_q(tau, qt, tt);
    quat_mul<1>(q, qt, qn);
    quat_rotate<1>(q, tt, tn);
#pragma unroll
    for (int i = 0; i < 3; ++i) tn[i] += t[i];
    se3_log_q(qn, tn, xn);
}

// Exp as (R, t): through the quaternion for plain scalars, so that every kernel
// has the same pose of a pixel; through se3_exp_V for other types (the tape)
template <typename T>
PV_HD void se3_exp(const T* xi, T* R, T* t) {
    if constexpr (is_scalar_v<T>) {
        T q[4];
        se3_exp_q(xi, q, t);
        quat_matrix(q, R);
    } else {
        T V[9];
        se3_exp_V(xi, R, t, V);
    }
}

// ---------------------------------------------------------------------------
// packed lower-triangular symmetric storage: (r, c), r >= c -> r(r+1)/2 + c
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int pidx(int r, int c) { return r >= c ? r * (r + 1) / 2 + c : c * (c + 1) / 2 + r; }

// In-place Cholesky of a packed N x N SPD matrix: A = L L^T, L packed lower.
// inv_diag receives 1 / L(j, j). Returns false on a non-positive (or NaN) pivot.
template <int N, typename T>
PV_HD bool chol_packed(T* A, T* inv_diag) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        T d = A[pidx(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) d -= A[pidx(j, k)] * A[pidx(j, k)];
        ok = ok && (d > T(0));
        T inv = v_rsqrt(d > T(0) ? d : T(1));
        T ljj = (d > T(0) ? d : T(1)) * inv;
        A[pidx(j, j)] = ljj;
        inv_diag[j] = inv;
#pragma unroll
        for (int i = j + 1; i < N; ++i) {
            T v = A[pidx(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) v -= A[pidx(i, k)] * A[pidx(j, k)];
            A[pidx(i, j)] = v * inv;
        }
    }
    return ok;
}

// Solve L y = b in place (L packed lower from chol_packed).
template <int N, typename T>
PV_HD void fwd_solve(const T* L, const T* inv_diag, T* b) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        T v = b[i];
#pragma unroll
        for (int k = 0; k < i; ++k) v -= L[pidx(i, k)] * b[k];
        b[i] = v * inv_diag[i];
    }
}

// Solve L^T x = y in place.
template <int N, typename T>
PV_HD void bwd_solve(const T* L, const T* inv_diag, T* b) {
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
        T v = b[i];
#pragma unroll
        for (int k = i + 1; k < N; ++k) v -= L[pidx(k, i)] * b[k];
        b[i] = v * inv_diag[i];
    }
}

// The same two solves with 1/L_ii stored on the diagonal of L in place of L_ii
// (a factor whose diagonal is only used through its inverse).
template <int N, typename T>
PV_HD void fwd_solve_id(const T* L, T* b) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        T v = b[i];
#pragma unroll
        for (int k = 0; k < i; ++k) v -= L[pidx(i, k)] * b[k];
        b[i] = v * L[pidx(i, i)];
    }
}
template <int N, typename T>
PV_HD void bwd_solve_id(const T* L, T* b) {
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
        T v = b[i];
#pragma unroll
        for (int k = i + 1; k < N; ++k) v -= L[pidx(k, i)] * b[k];
        b[i] = v * L[pidx(i, i)];
    }
}

// ---------------------------------------------------------------------------
// identity messages
// ---------------------------------------------------------------------------
// Inverse of a symmetric positive definite 6x6 matrix (packed; A is destroyed)
// by A = L D L^T, L^-1 in place and A^-1 = L^-T D^-1 L^-1. False on a
// non-positive (or NaN) pivot, which then stands as 1.
template <typename T>
PV_HD bool inverse6(T* A, T* Ai) {
    bool ok = true;
    T id[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const T d = A[pidx(j, j)];
        ok = ok && (d > T(0));
        id[j] = v_div(T(1), d > T(0) ? d : T(1));
        T v[6];
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            v[i] = A[pidx(i, j)];
            A[pidx(i, j)] = -(v[i] * id[j]);  // -L
        }
#pragma unroll
        for (int i = j + 1; i < 6; ++i)
#pragma unroll
            for (int l = j + 1; l <= i; ++l) A[pidx(i, l)] = v_fma(A[pidx(i, j)], v[l], A[pidx(i, l)]);
    }
    // M = L^-1 below its unit diagonal, column by column
#pragma unroll
    for (int c = 0; c < 5; ++c)
#pragma unroll
        for (int r = c + 2; r < 6; ++r)
#pragma unroll
            for (int k = c + 1; k < r; ++k) A[pidx(r, c)] = v_fma(A[pidx(r, k)], A[pidx(k, c)], A[pidx(r, c)]);
    // row r of A^-1: D^-1_r M_rc + sum over k > r of (D^-1_k M_kr) M_kc
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        T n[6];
#pragma unroll
        for (int k = r + 1; k < 6; ++k) n[k] = id[k] * A[pidx(k, r)];
#pragma unroll
        for (int c = 0; c <= r; ++c) {
            T s = c == r ? id[r] : id[r] * A[pidx(r, c)];
#pragma unroll
            for (int k = r + 1; k < 6; ++k) s = v_fma(n[k], A[pidx(k, c)], s);
            Ai[pidx(r, c)] = s;
        }
    }
    return ok;
}

// y = S x for packed symmetric S, in one fixed order of operations
template <typename T>
PV_HD void sym6_mv(const T* S, const T* x, T* y) {
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        T s = S[pidx(r, 0)] * x[0];
#pragma unroll
        for (int c = 1; c < 6; ++c) s = v_fma(S[pidx(r, c)], x[c], s);
        y[r] = s;
    }
}

// What an identity factor (Eq. 5, J = +I for the receiver, -I for the sender)
// sends to the receiver, from the sender's variable-to-factor marginal
// V = W + u u^T, eta_v and the residual r. With A = W + lam I (well conditioned:
// its eigenvalues lie between lam and a few lam; the rank-one u u^T, which can be
// far larger, stays out of the inversion), z = A^-1 u and C = A + u u^T:
//   Lambda = lam C^-1 V: off its diagonal -lam^2 (C^-1)_rc, on it
//            lam (A^-1 W)_rr + lam^2 z_r^2 / (1 + u^T z), free of the cancellation
//            of lam - lam^2 (C^-1)_rr when W << lam;
//   eta    = lam C^-1 (eta_v - V r) = lam (h - z (u^T r + u^T h) / (1 + u^T z)),
//            h = A^-1 (eta_v - W r).
// One inverse and two matrix-vector products replace a Cholesky factor with eight
// pairs of triangular solves: fewer operations, in independent rows where each
// solve was one dependent chain (the sweep waits on its chains, not on a pipe),
// and a smaller rounding error (random W of up to seven messages with eigenvalues
// 1e-5..1 lam: 0.8-1.2e-7 normwise in Lambda against 0.9-1.4e-7 before).
// U false: no rank-one part (u = 0, a pose node as the sender; the same values).
template <typename T, bool U = true>
struct IdMsg {
    T Ai[21];      // A^-1
    T dg[6];       // (A^-1 W)_rr
    T z[6], zi[6]; // z and z / (1 + u^T z)
    T he[6];       // eta / lam
    // C^-1, entry (r, c); off the diagonal -Lambda / lam^2
    PV_HD T ci(int r, int c) const { return U ? v_fma(-zi[c], z[r], Ai[pidx(r, c)]) : Ai[pidx(r, c)]; }
    // w Lambda + b, entry (r, c), r >= c, with the products wl = w lam, wll = w lam^2
    PV_HD T lambda(int r, int c, T wl, T wll, T b) const {
        if (r != c) return v_fma(-wll, ci(r, c), b);
        return v_fma(wl, dg[r], U ? v_fma(wll * zi[r], z[r], b) : b);
    }
};

template <typename T, bool U>
PV_HD bool identity_msg(const T* W, const T* u, const T* etav, const T* r, T lam, IdMsg<T, U>& m) {
    T A[21], g[6], h[6];
#pragma unroll
    for (int q = 0; q < 21; ++q) A[q] = W[q];
#pragma unroll
    for (int q = 0; q < 6; ++q) A[pidx(q, q)] += lam;
    const bool ok = inverse6(A, m.Ai);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        g[q] = etav[q];
        // the small off-diagonal products first
        T s = T(0);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            g[q] = v_fma(-W[pidx(q, c)], r[c], g[q]);
            if (c != q) s = v_fma(m.Ai[pidx(q, c)], W[pidx(q, c)], s);
        }
        m.dg[q] = v_fma(m.Ai[pidx(q, q)], W[pidx(q, q)], s);
    }
    sym6_mv(m.Ai, g, h);
    if constexpr (!U) {
#pragma unroll
        for (int q = 0; q < 6; ++q) m.he[q] = h[q];
        return ok;
    }
    sym6_mv(m.Ai, u, m.z);
    T uz = u[0] * m.z[0], ur = u[0] * r[0], uh = u[0] * h[0];
#pragma unroll
    for (int q = 1; q < 6; ++q) {
        uz = v_fma(u[q], m.z[q], uz);
        ur = v_fma(u[q], r[q], ur);
        uh = v_fma(u[q], h[q], uh);
    }
    const T iuz = v_div(T(1), T(1) + uz);
    const T ec = (ur + uh) * iuz;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        m.zi[q] = iuz * m.z[q];
        m.he[q] = v_fma(-ec, m.z[q], h[q]);
    }
    return ok;
}

}  // namespace pv
