// SU(3) algebra on the device, templated on the real type (double for the
// plain FP64 path, float for the FP32 path).
//
// Matrices are held as separate real and imaginary 3x3 arrays so that every
// element lives in a register after unrolling.  The Lie algebra is spanned by
// T^a = lambda^a / 2 (Gell-Mann); an element is stored as its 8 real
// components X^a = 2 tr(X T^a) (App. B of arXiv:2303.05599).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace gl {

template <typename R>
struct M3 {
    R re[3][3];
    R im[3][3];
};

template <typename R>
struct A8 {
    R v[8];
};

template <typename R>
__host__ __device__ __forceinline__ R inv_sqrt3() { return R(0.57735026918962576451); }

// A product that the compiler does not fuse into a later sum.  The FP64 field
// step has two kernels (tiles of 128 and of 16 sites) whose results are the
// same bits: every operation whose fusion would depend on what surrounds it is
// either this or an explicit fma.  FP32 has one kernel body and lets it fuse.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return a * b; }

template <typename R>
__device__ __forceinline__ M3<R> m_zero() {
    M3<R> m;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { m.re[i][j] = R(0); m.im[i][j] = R(0); }
    return m;
}

template <typename R>
__device__ __forceinline__ M3<R> m_id() {
    M3<R> m = m_zero<R>();
    m.re[0][0] = m.re[1][1] = m.re[2][2] = R(1);
    return m;
}

// c = a b
template <typename R>
__device__ __forceinline__ M3<R> mul(const M3<R>& a, const M3<R>& b) {
    M3<R> c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                sr = fma(a.re[i][k], b.re[k][j], sr);
                sr = fma(-a.im[i][k], b.im[k][j], sr);
                si = fma(a.re[i][k], b.im[k][j], si);
                si = fma(a.im[i][k], b.re[k][j], si);
            }
            c.re[i][j] = sr;
            c.im[i][j] = si;
        }
    return c;
}

// c = a b^+
template <typename R>
__device__ __forceinline__ M3<R> mul_nd(const M3<R>& a, const M3<R>& b) {
    M3<R> c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                // a_ik conj(b_jk)
                sr = fma(a.re[i][k], b.re[j][k], sr);
                sr = fma(a.im[i][k], b.im[j][k], sr);
                si = fma(a.im[i][k], b.re[j][k], si);
                si = fma(-a.re[i][k], b.im[j][k], si);
            }
            c.re[i][j] = sr;
            c.im[i][j] = si;
        }
    return c;
}

// c = a^+ b
template <typename R>
__device__ __forceinline__ M3<R> mul_dn(const M3<R>& a, const M3<R>& b) {
    M3<R> c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                // conj(a_ki) b_kj
                sr = fma(a.re[k][i], b.re[k][j], sr);
                sr = fma(a.im[k][i], b.im[k][j], sr);
                si = fma(a.re[k][i], b.im[k][j], si);
                si = fma(-a.im[k][i], b.re[k][j], si);
            }
            c.re[i][j] = sr;
            c.im[i][j] = si;
        }
    return c;
}

template <typename R>
__device__ __forceinline__ M3<R> dag(const M3<R>& a) {
    M3<R> c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { c.re[i][j] = a.re[j][i]; c.im[i][j] = -a.im[j][i]; }
    return c;
}

template <typename R>
__device__ __forceinline__ M3<R> add(const M3<R>& a, const M3<R>& b) {
    M3<R> c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { c.re[i][j] = a.re[i][j] + b.re[i][j]; c.im[i][j] = a.im[i][j] + b.im[i][j]; }
    return c;
}

template <typename R>
__device__ __forceinline__ M3<R> sub(const M3<R>& a, const M3<R>& b) {
    M3<R> c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { c.re[i][j] = a.re[i][j] - b.re[i][j]; c.im[i][j] = a.im[i][j] - b.im[i][j]; }
    return c;
}

// Hermitian matrix X = sum_a x^a T^a
template <typename R>
__device__ __forceinline__ M3<R> alg_to_mat(const A8<R>& x) {
    const R h = R(0.5), s3 = inv_sqrt3<R>();
    M3<R> m;
    m.re[0][0] = h * (x.v[2] + x.v[7] * s3); m.im[0][0] = R(0);
    m.re[1][1] = h * (-x.v[2] + x.v[7] * s3); m.im[1][1] = R(0);
    m.re[2][2] = -x.v[7] * s3; m.im[2][2] = R(0);
    m.re[0][1] = h * x.v[0]; m.im[0][1] = -h * x.v[1];
    m.re[1][0] = h * x.v[0]; m.im[1][0] = h * x.v[1];
    m.re[0][2] = h * x.v[3]; m.im[0][2] = -h * x.v[4];
    m.re[2][0] = h * x.v[3]; m.im[2][0] = h * x.v[4];
    m.re[1][2] = h * x.v[5]; m.im[1][2] = -h * x.v[6];
    m.re[2][1] = h * x.v[5]; m.im[2][1] = h * x.v[6];
    return m;
}

// components x^a = 2 Re tr(X T^a) of the traceless part of a Hermitian X
template <typename R>
__device__ __forceinline__ A8<R> herm_to_alg(const M3<R>& X) {
    A8<R> x;
    x.v[0] = X.re[0][1] + X.re[1][0];
    x.v[1] = X.im[1][0] - X.im[0][1];
    x.v[2] = X.re[0][0] - X.re[1][1];
    x.v[3] = X.re[0][2] + X.re[2][0];
    x.v[4] = X.im[2][0] - X.im[0][2];
    x.v[5] = X.re[1][2] + X.re[2][1];
    x.v[6] = X.im[2][1] - X.im[1][2];
    x.v[7] = (X.re[0][0] + X.re[1][1] - R(2) * X.re[2][2]) * inv_sqrt3<R>();
    return x;
}

// components of the Hermitian traceless matrix i [M]_ah, with
// [M]_ah = (M - M^+)/2 - tr(M - M^+)/6  (anti-Hermitian traceless part)
template <typename R>
__device__ __forceinline__ A8<R> iah_to_alg(const M3<R>& M) {
    A8<R> x;
    x.v[0] = -(M.im[0][1] + M.im[1][0]);
    x.v[1] = M.re[1][0] - M.re[0][1];
    x.v[2] = M.im[1][1] - M.im[0][0];
    x.v[3] = -(M.im[0][2] + M.im[2][0]);
    x.v[4] = M.re[2][0] - M.re[0][2];
    x.v[5] = -(M.im[1][2] + M.im[2][1]);
    x.v[6] = M.re[2][1] - M.re[1][2];
    x.v[7] = (R(2) * M.im[2][2] - M.im[0][0] - M.im[1][1]) * inv_sqrt3<R>();
    return x;
}

template <typename R>
__device__ __forceinline__ void cmul(R ar, R ai, R br, R bi, R& cr, R& ci) {
    cr = ar * br - ai * bi;
    ci = ar * bi + ai * br;
}

template <typename R>
__device__ __forceinline__ A8<R> a_zero() {
    A8<R> x;
#pragma unroll
    for (int a = 0; a < 8; a++) x.v[a] = R(0);
    return x;
}

template <typename R>
__device__ __forceinline__ R a_dot(const A8<R>& p, const A8<R>& q) {
    R s = R(0);
#pragma unroll
    for (int a = 0; a < 8; a++) s = fma(p.v[a], q.v[a], s);
    return s;
}

// U X U^+ for Hermitian X, as algebra components
template <typename R>
__device__ __forceinline__ A8<R> adj(const M3<R>& U, const A8<R>& x) {
    return herm_to_alg(mul_nd(mul(U, alg_to_mat(x)), U));
}

// U^+ X U for Hermitian X, as algebra components
template <typename R>
__device__ __forceinline__ A8<R> adj_dag(const M3<R>& U, const A8<R>& x) {
    return herm_to_alg(mul(mul_dn(U, alg_to_mat(x)), U));
}

// 2 X for X = sum_a x^a T^a: the off-diagonal entries are the components
// themselves (no factor 1/2)
template <typename R>
__device__ __forceinline__ M3<R> alg_to_mat2(const A8<R>& x) {
    const R p = mul_rn(x.v[7], inv_sqrt3<R>());
    M3<R> m;
    m.re[0][0] = x.v[2] + p; m.im[0][0] = R(0);
    m.re[1][1] = p - x.v[2]; m.im[1][1] = R(0);
    m.re[2][2] = R(-2) * p; m.im[2][2] = R(0);
    m.re[0][1] = x.v[0]; m.im[0][1] = -x.v[1];
    m.re[1][0] = x.v[0]; m.im[1][0] = x.v[1];
    m.re[0][2] = x.v[3]; m.im[0][2] = -x.v[4];
    m.re[2][0] = x.v[3]; m.im[2][0] = x.v[4];
    m.re[1][2] = x.v[5]; m.im[1][2] = -x.v[6];
    m.re[2][1] = x.v[5]; m.im[2][1] = x.v[6];
    return m;
}

// components of V^+ X V for Hermitian X (only the upper triangle of the
// Hermitian result is formed).  The product is taken of 2 X, so that the
// off-diagonal components need no factor 2 and the diagonal ones a factor
// 1/2; scaling by powers of 2 is exact, so the result is bitwise that of X.
template <typename R>
__device__ __forceinline__ A8<R> conj_dn(const M3<R>& V, const A8<R>& x) {
    const M3<R> X = alg_to_mat2(x);
    M3<R> Y;  // X V, with X's diagonal real
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            R sr = X.re[i][i] * V.re[i][j], si = X.re[i][i] * V.im[i][j];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (k == i) continue;
                sr = fma(X.re[i][k], V.re[k][j], sr);
                sr = fma(-X.im[i][k], V.im[k][j], sr);
                si = fma(X.re[i][k], V.im[k][j], si);
                si = fma(X.im[i][k], V.re[k][j], si);
            }
            Y.re[i][j] = sr;
            Y.im[i][j] = si;
        }
    R zr[3][3], zi[3][3];  // V^+ Y, upper triangle
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                sr = fma(V.re[k][i], Y.re[k][j], sr);
                sr = fma(V.im[k][i], Y.im[k][j], sr);
                if (i != j) {
                    si = fma(V.re[k][i], Y.im[k][j], si);
                    si = fma(-V.im[k][i], Y.re[k][j], si);
                }
            }
            zr[i][j] = sr;
            zi[i][j] = si;
        }
    A8<R> o;
    o.v[0] = zr[0][1];
    o.v[1] = -zi[0][1];
    o.v[2] = R(0.5) * (zr[0][0] - zr[1][1]);
    o.v[3] = zr[0][2];
    o.v[4] = -zi[0][2];
    o.v[5] = zr[1][2];
    o.v[6] = -zi[1][2];
    o.v[7] = (zr[0][0] + zr[1][1] - R(2) * zr[2][2]) * (R(0.5) * inv_sqrt3<R>());
    return o;
}

// conj_dn for the field step, where the transports are the bulk of the
// arithmetic.  V^+ X V is traceless like X, so the (2, 2) entry is not formed:
// the eighth component follows from the first two diagonal entries (the same
// value up to rounding).  Rows 0 and 1 of the result, all that is left to
// form, are rows 0 and 1 of W = V^+ (2X) times V, so the product is
// associated that way and only two rows of W are formed: six entries instead
// of the nine of (2X) V, about 108 multiply-adds instead of 138.
template <typename R>
__device__ __forceinline__ A8<R> conj_dn_t(const M3<R>& V, const A8<R>& x) {
    const M3<R> X = alg_to_mat2(x);
    R wr[2][3], wi[2][3];  // W = V^+ X, rows 0 and 1, with X's diagonal real
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            // conj(V_ji) X_jj, then conj(V_ki) X_kj for k != j
            R sr = V.re[j][i] * X.re[j][j], si = -(V.im[j][i] * X.re[j][j]);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (k == j) continue;
                sr = fma(V.re[k][i], X.re[k][j], sr);
                sr = fma(V.im[k][i], X.im[k][j], sr);
                si = fma(V.re[k][i], X.im[k][j], si);
                si = fma(-V.im[k][i], X.re[k][j], si);
            }
            wr[i][j] = sr;
            wi[i][j] = si;
        }
    R zr[2][3], zi[2][3];  // Z = W V, upper triangle of rows 0 and 1
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                sr = fma(wr[i][k], V.re[k][j], sr);
                sr = fma(-wi[i][k], V.im[k][j], sr);
                if (i != j) {
                    si = fma(wr[i][k], V.im[k][j], si);
                    si = fma(wi[i][k], V.re[k][j], si);
                }
            }
            zr[i][j] = sr;
            zi[i][j] = si;
        }
    A8<R> o;
    o.v[0] = zr[0][1];
    o.v[1] = -zi[0][1];
    o.v[2] = mul_rn(R(0.5), zr[0][0] - zr[1][1]);
    o.v[3] = zr[0][2];
    o.v[4] = -zi[0][2];
    o.v[5] = zr[1][2];
    o.v[6] = -zi[1][2];
    // (Z00 + Z11 - 2 Z22) / sqrt 3 with Z22 = -(Z00 + Z11), halved for 2X
    o.v[7] = mul_rn(zr[0][0] + zr[1][1], R(0.86602540378443864676));
    return o;
}

// components of V X V^+ for Hermitian X
template <typename R>
__device__ __forceinline__ A8<R> conj_up(const M3<R>& V, const A8<R>& x) {
    return conj_dn(dag(V), x);
}
template <typename R>
__device__ __forceinline__ A8<R> conj_up_t(const M3<R>& V, const A8<R>& x) {
    return conj_dn_t(dag(V), x);
}

// X^2 for Hermitian X: the upper triangle is formed, the lower one mirrored
template <typename R>
__device__ __forceinline__ M3<R> sq_herm(const M3<R>& X) {
    M3<R> Z;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                // the diagonal entries are real
                sr = fma(X.re[i][k], X.re[k][j], sr);
                if (k != i && k != j) sr = fma(-X.im[i][k], X.im[k][j], sr);
                if (i != j) {
                    if (k != j) si = fma(X.re[i][k], X.im[k][j], si);
                    if (k != i) si = fma(X.im[i][k], X.re[k][j], si);
                }
            }
            Z.re[i][j] = sr;
            Z.im[i][j] = si;
            Z.re[j][i] = sr;
            Z.im[j][i] = -si;
        }
#pragma unroll
    for (int i = 0; i < 3; i++) Z.im[i][i] = R(0);
    return Z;
}

// components of i[A B^+]_ah without forming the whole product: only the
// imaginary parts of the diagonal and both triangles are needed
template <typename R>
__device__ __forceinline__ A8<R> iah_of_mul_nd(const M3<R>& A, const M3<R>& B) {
    R dr[3][3], di[3][3];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            R sr = R(0), si = R(0);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                // A_ik conj(B_jk)
                if (i != j) {
                    sr = fma(A.re[i][k], B.re[j][k], sr);
                    sr = fma(A.im[i][k], B.im[j][k], sr);
                }
                si = fma(A.im[i][k], B.re[j][k], si);
                si = fma(-A.re[i][k], B.im[j][k], si);
            }
            dr[i][j] = sr;
            di[i][j] = si;
        }
    A8<R> x;
    x.v[0] = -(di[0][1] + di[1][0]);
    x.v[1] = dr[1][0] - dr[0][1];
    x.v[2] = di[1][1] - di[0][0];
    x.v[3] = -(di[0][2] + di[2][0]);
    x.v[4] = dr[2][0] - dr[0][2];
    x.v[5] = -(di[1][2] + di[2][1]);
    x.v[6] = dr[2][1] - dr[1][2];
    x.v[7] = (R(2) * di[2][2] - di[0][0] - di[1][1]) * inv_sqrt3<R>();
    return x;
}

// cubic Casimir q3 = d_abc Q^a Q^b Q^c from the 16 independent nonzero
// symmetric structure constants of SU(3) (Table II), each weighted by the
// number of distinct index orderings
template <typename R>
__device__ __forceinline__ R casimir3(const A8<R>& q) {
    const R s3 = inv_sqrt3<R>();  // 1/sqrt(3)
    const R* Q = q.v;             // Q[0] = Q^1 ... Q[7] = Q^8
    const R h = R(0.5);
    R r = R(3) * s3 * (Q[0] * Q[0] + Q[1] * Q[1] + Q[2] * Q[2]) * Q[7]    // d118, d228, d338
        + R(6) * h * (Q[0] * Q[3] * Q[5] + Q[0] * Q[4] * Q[6]             // d146, d157
                      - Q[1] * Q[3] * Q[6] + Q[1] * Q[4] * Q[5])          // d247, d256
        + R(3) * h * Q[2] * (Q[3] * Q[3] + Q[4] * Q[4] - Q[5] * Q[5] - Q[6] * Q[6])  // d344 d355 d366 d377
        - R(3) * h * s3 * (Q[3] * Q[3] + Q[4] * Q[4] + Q[5] * Q[5] + Q[6] * Q[6]) * Q[7]  // d448..d778
        - s3 * Q[7] * Q[7] * Q[7];                                           // d888
    return r;
}

// The coefficients of exp(iX) = f0 + f1 X + f2 X^2 for Hermitian traceless X
// with X^3 = c1 X + c0 (Cayley-Hamilton: c1 = tr(X^2)/2, c0 = det X).
template <typename R>
struct ExpScale {
    int nsq;    // squarings: the series is summed for scl X, scl = 2^-nsq
    R scl;
    int terms;  // FP64: its last power
};

// FP32: the series to X^6 for |X| <= 0.2 (truncation error below 1e-8),
// reduced by X^3 = c1 X + c0 to one polynomial in (c0, c1) for each real
// coefficient: 11 operations, where the recurrence of the reduced powers takes
// about 48.  Two exponentials a site are 2 % of the field step's issue slots.
__device__ __forceinline__ void exp_coeffs(float c0, float c1, const ExpScale<float>&, float* fr, float* fi) {
    fr[0] = fmaf(-1.0f / 720, c0 * c0, 1.0f);
    fi[0] = c0 * fmaf(1.0f / 120, c1, -1.0f / 6);
    fr[1] = c0 * fmaf(-1.0f / 360, c1, 1.0f / 24);
    fi[1] = fmaf(c1, fmaf(1.0f / 120, c1, -1.0f / 6), 1.0f);
    fr[2] = fmaf(c1, fmaf(-1.0f / 720, c1, 1.0f / 24), -0.5f);
    fi[2] = c0 * (1.0f / 120);
}

// FP64: Horner's rule on the reduced series.  With P = p0 + p1 X + p2 X^2,
// 1/k! + iX P has the coefficients 1/k! + i c0 p2, i (p0 + c1 p2), i p1: four
// operations a term.  FP64 operations take 64 cycles of a scheduler per warp
// on GB300, so the number of terms follows the norm: 6 for |X| <= 0.01 (a
// field step late in the run, a Newton step), 12 for 0.25, 18 for 1, 24 for 2
// (one sheet of an MV nucleus), each with a truncation error below 3e-18.
__device__ __forceinline__ void exp_coeffs(double c0, double c1, const ExpScale<double>& s, double* fr, double* fi) {
    constexpr double F[25] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320,
                              1.0 / 362880, 1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0,
                              1.0 / 87178291200.0, 1.0 / 1307674368000.0, 1.0 / 20922789888000.0,
                              1.0 / 355687428096000.0, 1.0 / 6402373705728000.0, 1.0 / 121645100408832000.0,
                              1.0 / 2432902008176640000.0, 1.0 / 51090942171709440000.0,
                              1.0 / 1124000727777607680000.0, 1.0 / 25852016738884976640000.0,
                              1.0 / 620448401733239439360000.0};
    double r0 = s.terms == 24 ? F[24] : s.terms == 18 ? F[18] : s.terms == 12 ? F[12] : F[6];
    double i0 = 0, r1 = 0, i1 = 0, r2 = 0, i2 = 0;
#define GL_HORNER(k)                                         \
    {                                                        \
        const double n0r = fma(-c0, i2, F[k]), n0i = c0 * r2; \
        const double n1r = -fma(c1, i2, i0), n1i = fma(c1, r2, r0); \
        r2 = -i1;                                            \
        i2 = r1;                                             \
        r0 = n0r;                                            \
        i0 = n0i;                                            \
        r1 = n1r;                                            \
        i1 = n1i;                                            \
    }
#define GL_HORNER6(k) \
    GL_HORNER(k) GL_HORNER((k) - 1) GL_HORNER((k) - 2) GL_HORNER((k) - 3) GL_HORNER((k) - 4) GL_HORNER((k) - 5)
    if (s.terms > 18) { GL_HORNER6(23) }
    if (s.terms > 12) { GL_HORNER6(17) }
    if (s.terms > 6) { GL_HORNER6(11) }
    GL_HORNER6(5)
#undef GL_HORNER6
#undef GL_HORNER
    fr[0] = r0; fi[0] = i0;
    fr[1] = r1; fi[1] = i1;
    fr[2] = r2; fi[2] = i2;
}

__device__ __forceinline__ ExpScale<float> exp_scale(float nrm2) {
    ExpScale<float> s = {0, 1.0f, 6};
    while (nrm2 > 0.04f && s.nsq < 30) { nrm2 *= 0.25f; s.scl *= 0.5f; s.nsq++; }
    return s;
}
__device__ __forceinline__ ExpScale<double> exp_scale(double nrm2) {
    ExpScale<double> s = {0, 1.0, 24};
    while (nrm2 > 4.0 && s.nsq < 30) { nrm2 *= 0.25; s.scl *= 0.5; s.nsq++; }
    if (nrm2 <= 1.0) s.terms = nrm2 <= 1e-4 ? 6 : nrm2 <= 0.0625 ? 12 : 18;
    return s;
}

// exp(i s X) for Hermitian traceless X = x^a T^a (scaling and squaring beyond
// the series' range)
template <typename R>
__device__ __forceinline__ M3<R> exp_i_alg(const A8<R>& x, R s) {
    // s X: 2 X from the components, times s / 2 (exact: a power of 2), one
    // product per distinct entry
    M3<R> X = alg_to_mat2(x);
    const R hs = R(0.5) * s;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        X.re[i][i] *= hs;
#pragma unroll
        for (int j = i + 1; j < 3; j++) {
            X.re[i][j] *= hs;
            X.im[i][j] *= hs;
            X.re[j][i] = X.re[i][j];
            X.im[j][i] = -X.im[i][j];
        }
    }
    M3<R> X2 = sq_herm(X);
    R c1 = R(0.5) * (X2.re[0][0] + X2.re[1][1] + X2.re[2][2]);
    const ExpScale<R> sc = exp_scale(R(2) * c1);  // the squared Frobenius norm of X is 2 c1
    if (sc.nsq) {
        const R scl = sc.scl;
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) {
                X.re[i][j] *= scl; X.im[i][j] *= scl;
                X2.re[i][j] *= scl * scl; X2.im[i][j] *= scl * scl;
            }
        c1 *= scl * scl;
    }
    // det X = tr(X^3) / 3 of the traceless X, from X and X^2 (both Hermitian)
    R c0 = X.re[0][1] * X2.re[0][1];
    c0 = fma(X.im[0][1], X2.im[0][1], c0);
    c0 = fma(X.re[0][2], X2.re[0][2], c0);
    c0 = fma(X.im[0][2], X2.im[0][2], c0);
    c0 = fma(X.re[1][2], X2.re[1][2], c0);
    c0 = fma(X.im[1][2], X2.im[1][2], c0);
    c0 = fma(R(0.5) * X.re[0][0], X2.re[0][0], c0);
    c0 = fma(R(0.5) * X.re[1][1], X2.re[1][1], c0);
    c0 = fma(R(0.5) * X.re[2][2], X2.re[2][2], c0);
    c0 *= R(2.0 / 3.0);
    R fr[3], fi[3];
    exp_coeffs(c0, c1, sc, fr, fi);
    M3<R> U;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            // (f0 + f1 X + f2 X2)_ij, complex coefficients; X and X2 have real diagonals
            if (i == j) {
                U.re[i][j] = fma(fr[1], X.re[i][j], fma(fr[2], X2.re[i][j], fr[0]));
                U.im[i][j] = fma(fi[1], X.re[i][j], fma(fi[2], X2.re[i][j], fi[0]));
            } else {
                U.re[i][j] = fma(fr[1], X.re[i][j], fma(-fi[1], X.im[i][j], fma(fr[2], X2.re[i][j], -(fi[2] * X2.im[i][j]))));
                U.im[i][j] = fma(fr[1], X.im[i][j], fma(fi[1], X.re[i][j], fma(fr[2], X2.im[i][j], fi[2] * X2.re[i][j])));
            }
        }
    for (int k = 0; k < sc.nsq; k++) U = mul(U, U);
    return U;
}

// third row of an SU(3) matrix from the first two: u_2 = conj(u_0 x u_1)
template <typename R>
__device__ __forceinline__ void rebuild_row2(M3<R>& u) {
#define GL_CX(ar, ai, br, bi, cr, ci, dr, di) ((ar) * (br) - (ai) * (bi) - ((cr) * (dr) - (ci) * (di)))
#define GL_CY(ar, ai, br, bi, cr, ci, dr, di) ((ar) * (bi) + (ai) * (br) - ((cr) * (di) + (ci) * (dr)))
    // u20 = conj(u01 u12 - u02 u11)
    u.re[2][0] = GL_CX(u.re[0][1], u.im[0][1], u.re[1][2], u.im[1][2], u.re[0][2], u.im[0][2], u.re[1][1], u.im[1][1]);
    u.im[2][0] = -GL_CY(u.re[0][1], u.im[0][1], u.re[1][2], u.im[1][2], u.re[0][2], u.im[0][2], u.re[1][1], u.im[1][1]);
    // u21 = conj(u02 u10 - u00 u12)
    u.re[2][1] = GL_CX(u.re[0][2], u.im[0][2], u.re[1][0], u.im[1][0], u.re[0][0], u.im[0][0], u.re[1][2], u.im[1][2]);
    u.im[2][1] = -GL_CY(u.re[0][2], u.im[0][2], u.re[1][0], u.im[1][0], u.re[0][0], u.im[0][0], u.re[1][2], u.im[1][2]);
    // u22 = conj(u00 u11 - u01 u10)
    u.re[2][2] = GL_CX(u.re[0][0], u.im[0][0], u.re[1][1], u.im[1][1], u.re[0][1], u.im[0][1], u.re[1][0], u.im[1][0]);
    u.im[2][2] = -GL_CY(u.re[0][0], u.im[0][0], u.re[1][1], u.im[1][1], u.re[0][1], u.im[0][1], u.re[1][0], u.im[1][0]);
#undef GL_CX
#undef GL_CY
}

}  // namespace gl
