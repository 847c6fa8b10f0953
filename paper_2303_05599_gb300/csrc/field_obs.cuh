// The FP64 field checks of one site (Gauss constraint of Sec. 2, unitarity of
// the links, the squared site fields whose lattice means give the energy
// density) and the block reduction of their accumulators, shared by the
// single-event launch (obs.cu) and the one launch over all events of a batch.
// The maxima leave the kernels as squared norms; the host takes their roots.
#pragma once
#include "ff.cuh"
#include "internal.h"
#include "layout.cuh"
#include "obs_body.cuh"

namespace gl {

// an FP32 value in FP64, by integer operations: the conversion instruction runs
// at the FP64 pipe's rate (64 cycles a warp and scheduler), and the checks of an
// FP32 state convert about 70 values a site
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return (double)x;  // zero, denormal, infinite, NaN
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
template <typename R>
__device__ __forceinline__ A8<double> to_d(const A8<R>& a) {
    A8<double> o;
#pragma unroll
    for (int k = 0; k < 8; k++) o.v[k] = widen(a.v[k]);
    return o;
}
template <typename R>
__device__ __forceinline__ M3<double> to_d(const M3<R>& a) {
    M3<double> o;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { o.re[i][j] = widen(a.re[i][j]); o.im[i][j] = widen(a.im[i][j]); }
    return o;
}

// ||U U^+ - 1||_F^2 from the Gram matrix of the rows (Hermitian: upper
// triangle, off-diagonal twice; the diagonal is real)
__device__ __forceinline__ double gram_deviation(const M3<double>& u) {
    double n2 = 0;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            double gr = 0, gi = 0;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                gr = fma(u.re[i][k], u.re[j][k], gr);
                gr = fma(u.im[i][k], u.im[j][k], gr);
                if (i != j) {
                    gi = fma(u.im[i][k], u.re[j][k], gi);
                    gi = fma(-u.re[i][k], u.im[j][k], gi);
                }
            }
            const double r = gr - (i == j ? 1.0 : 0.0);
            n2 += (i == j ? 1.0 : 2.0) * (r * r + gi * gi);
        }
    return n2;
}

// sum of products of FP32 values in three FP32 parts (every product and every
// rounding of the sum and of its first correction is kept: the error is below
// 2^-68 of the largest product, against FP64's 2^-53)
struct Sum3 {
    float s, c, d;
    __device__ __forceinline__ Sum3(float a, float b) {
        s = __fmul_rn(a, b);
        c = fmaf(a, b, -s);
        d = 0.f;
    }
    __device__ __forceinline__ void add(float a, float b) {
        const float p = __fmul_rn(a, b), e = fmaf(a, b, -p);
        const ff t = ff_sum(s, p), u = ff_sum(c, t.l), v = ff_sum(u.h, e);
        s = t.h;
        c = v.h;
        d = __fadd_rn(d, __fadd_rn(u.l, v.l));
    }
    // the sum less `one` (0, or 1 with s within a factor 2 of it, else rounded)
    __device__ __forceinline__ ff less(float one) const {
        const ff t = ff_sum(s, -one), u = ff_sum(t.h, c);
        return ff_quick(u.h, __fadd_rn(t.l, __fadd_rn(u.l, d)));
    }
};
// the same of an FP32 link, on the FP32 pipe: the Gram matrix in three parts,
// its deviation and the sum of squares in pairs.  54 FP64 operations a link
// less, with a smaller error.  Links with entries whose products would leave
// the FP32 range, or that are not finite, take the FP64 form.
__device__ __forceinline__ double gram_deviation(const M3<float>& u) {
    float big = 0.f;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) big += fabsf(u.re[i][j]) + fabsf(u.im[i][j]);
    if (!(big < 1e9f)) return gram_deviation(to_d(u));
    ff n2{0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            Sum3 gr(u.re[i][0], u.re[j][0]);
            gr.add(u.im[i][0], u.im[j][0]);
#pragma unroll
            for (int k = 1; k < 3; k++) {
                gr.add(u.re[i][k], u.re[j][k]);
                gr.add(u.im[i][k], u.im[j][k]);
            }
            const ff r = gr.less(i == j ? 1.f : 0.f);
            ff q = r * r;
            if (i != j) {
                Sum3 gi(u.im[i][0], u.re[j][0]);
                gi.add(-u.re[i][0], u.im[j][0]);
#pragma unroll
                for (int k = 1; k < 3; k++) {
                    gi.add(u.im[i][k], u.re[j][k]);
                    gi.add(-u.re[i][k], u.im[j][k]);
                }
                const ff m = gi.less(0.f);
                q = ff_scale(ff_fma(m, m, q), 2.f);
            }
            n2 = n2 + q;
        }
    return (double)n2.h + (double)n2.l;
}

// Site s = (x, y) into the accumulators v[FO_N]:
//   G(x) = sum_i [e_i(x) - U_i(x-i)^+ e_i(x-i) U_i(x-i)] + i[phi(x), pi(x)]
// (with the full transport: for a link that is not unitary, which is what the
// check is for, U^+ e U has a trace) and ||U U^+ - 1||_F of the two links it
// transports by, U_i(x-i) (every link is that of one site); the maxima are kept
// as squared norms (the root, monotonic, is taken once of the maximum).  The
// Gauss residual is FP64 throughout; an FP32 link's unitarity takes three-part
// FP32 sums, which are more exact.  The sums of squares of the six site fields,
// whose halves are tr X^2 = X^a X^a / 2, are FP64 sums of site values; an FP32
// state's squares are exact as float pairs, and a site's 8 or 16 of them are
// summed as a pair (SquareSum) before they cost FP64 issue, two additions a
// value.  (As pairs over all sites of a thread and of a block they lost up to
// 2.5e-14 on 1024^2, against 1.5e-15, and overflowed at FP32's range: the
// additions cost 1 % of the call on 18 events of 64/128/256, 3 % on 1024^2.)
// Bound by the FP64 pipe (87 % of its cycles): 18 events of 64/128/256, FP32,
// 540 FP64 warp instructions a site, 559 us under ncu; with FP64 Gram matrices,
// converted inputs and one block reduction a site the call took 786 us, now 602.
// (The commutator and the first product of the transport in three-part sums,
// 107 FP64 operations fewer and 4,400 FP32 ones more: 663 us.)
template <typename R>
__device__ __forceinline__ void field_obs_site(const Fields<R>& f, const typename Prec<R>::V* __restrict__ site,
                                               int N, int64_t Vn, int64_t s, double* v) {
    constexpr int AP = Prec<R>::AP;
    const int x = (int)(s % N), y = (int)(s / N);
    const int64_t sb[2] = {(int64_t)y * N + (x == 0 ? N - 1 : x - 1), (int64_t)(y == 0 ? N - 1 : y - 1) * N + x};
    A8<double> G = icomm(to_d(load_alg(f.phi, s, Vn)), to_d(load_alg(f.pi, s, Vn)));
#pragma unroll
    for (int d = 0; d < 2; d++) {
        const typename Prec<R>::V* e = f.e + (size_t)d * AP * Vn;
        const A8<double> eh = to_d(load_alg(e, s, Vn));
        const M3<R> u = load_link(f.U, d, sb[d], Vn);
        const A8<double> eb = conj_dn(to_d(u), to_d(load_alg(e, sb[d], Vn)));
#pragma unroll
        for (int a = 0; a < 8; a++) G.v[a] += eh.v[a] - eb.v[a];
        v[FO_UMAX] = nanmax(v[FO_UMAX], gram_deviation(u));
    }
    const double g2 = a_dot(G, G);
    v[FO_GMAX] = nanmax(v[FO_GMAX], g2);
    v[FO_GSUM] += g2;
    double sum = SquareSum<R>::init();
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const A8<R> X = load_alg(site + (size_t)k * AP * Vn, s, Vn);
        const int slot = k < 2 ? FO_ET2 : k == 2 ? FO_EL2 : k < 5 ? FO_BT2 : FO_BL2;
        if constexpr (sizeof(R) == 8) {
#pragma unroll
            for (int a = 0; a < 8; a++) v[slot] = SquareSum<R>::add(v[slot], X.v[a]);
        } else {
#pragma unroll
            for (int a = 0; a < 8; a++) sum = SquareSum<R>::add(sum, X.v[a]);
            if (k == 0 || k == 3) continue;  // the second component of the same value follows
            v[slot] += widen(f2_lo(sum)) + widen(f2_hi(sum));
            sum = SquareSum<R>::init();
        }
    }
}

// the block's accumulators (maxima and sums, fixed order) into row[FO_N]; every
// thread of the block calls it.  Eight threads a value: each combines an eighth
// of the threads' accumulators in order, then three shuffles; the halves of the
// sums of squares are tr X^2.  (Five shuffle levels of all seven values took each
// warp 60 FP64 instructions.)
__device__ __forceinline__ void field_obs_block_reduce(const double* v, double* row) {
    __shared__ double acc[FO_N][FIELD_OBS_THREADS + 1];
    static_assert(FIELD_OBS_THREADS == 64 && FO_N <= 8, "eight threads a value");
#pragma unroll
    for (int k = 0; k < FO_N; k++) acc[k][threadIdx.x] = v[k];
    __syncthreads();
    const int k = threadIdx.x >> 3, part = threadIdx.x & 7;
    auto combine = [&](double a, double b) { return k == FO_GMAX || k == FO_UMAX ? nanmax(a, b) : a + b; };
    double a = 0.0;
    if (k < FO_N) {
        a = acc[k][part * 8];
        for (int j = 1; j < 8; j++) a = combine(a, acc[k][part * 8 + j]);
    }
    for (int o = 4; o > 0; o >>= 1) a = combine(a, __shfl_down_sync(0xffffffffu, a, o, 8));
    if (k < FO_N && part == 0) row[k] = k >= FO_ET2 ? 0.5 * a : a;
}

}  // namespace gl
