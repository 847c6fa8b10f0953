// Pairs of FP32 values (hi + lo, about 48 significant bits) on the FP32 pipe,
// for the parts of an FP32 event's initial conditions that the FP64 pipe
// bounded: GB300 issues an FP64 warp instruction in 76 cycles of a scheduler
// and an FP32 one in one.  Error-free sums (Knuth) and products (Dekker, by
// FMA), and dot products that carry the errors of their sums and products in
// one FP32 accumulator (Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26 (2005)).
#pragma once
#include <stdint.h>

#include "su3.cuh"

namespace gl {

struct ff {
    float h, l;
};

__host__ __device__ constexpr ff ff_of(double d) { return ff{(float)d, (float)(d - (double)(float)d)}; }
__device__ __forceinline__ double to_double(ff a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ ff ff_quick(float a, float b) {  // |a| >= |b| or a = 0
    const float s = __fadd_rn(a, b);
    return ff{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff ff_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return ff{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ ff operator-(ff a) { return ff{-a.h, -a.l}; }
__device__ __forceinline__ ff operator+(ff a, ff b) {
    const ff s = ff_sum(a.h, b.h);
    return ff_quick(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }
// a b + e, not normalised, with |e| far below |a b| or its rounding
__device__ __forceinline__ ff ff_prod(ff a, ff b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    return ff{p, e};
}
__device__ __forceinline__ ff operator*(ff a, ff b) {
    const ff p = ff_prod(a, b);
    return ff_quick(p.h, p.l);
}
__device__ __forceinline__ ff ff_scale(ff a, float s) { return ff{a.h * s, a.l * s}; }  // s a power of 2
__device__ __forceinline__ ff ff_times(ff a, float b) {
    const float p = __fmul_rn(a.h, b);
    return ff_quick(p, fmaf(a.l, b, fmaf(a.h, b, -p)));
}
// a b + c
__device__ __forceinline__ ff ff_fma(ff a, ff b, ff c) {
    const ff p = ff_prod(a, b);
    const ff s = ff_sum(p.h, c.h);
    return ff_quick(s.h, __fadd_rn(s.l, __fadd_rn(p.l, c.l)));
}

// sum of products
struct FDot {
    float s, c;
    __device__ __forceinline__ FDot(ff a, ff b) {
        const ff p = ff_prod(a, b);
        s = p.h;
        c = p.l;
    }
    __device__ __forceinline__ FDot& add(ff a, ff b) {
        const ff p = ff_prod(a, b);
        const ff t = ff_sum(s, p.h);
        s = t.h;
        c = __fadd_rn(c, __fadd_rn(t.l, p.l));
        return *this;
    }
    __device__ __forceinline__ FDot& sub(ff a, ff b) { return add(-a, b); }
    __device__ __forceinline__ ff get() const { return ff_quick(s, c); }
};

struct M3ff {
    ff re[3][3], im[3][3];
};

// rows 0 .. ROWS - 1 of a b
template <int ROWS>
__device__ __forceinline__ M3ff ff_mul(const M3ff& a, const M3ff& b) {
    M3ff c;
#pragma unroll
    for (int i = 0; i < ROWS; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            FDot r(a.re[i][0], b.re[0][j]), m(a.re[i][0], b.im[0][j]);
            r.sub(a.im[i][0], b.im[0][j]);
            m.add(a.im[i][0], b.re[0][j]);
#pragma unroll
            for (int k = 1; k < 3; k++) {
                r.add(a.re[i][k], b.re[k][j]).sub(a.im[i][k], b.im[k][j]);
                m.add(a.re[i][k], b.im[k][j]).add(a.im[i][k], b.re[k][j]);
            }
            c.re[i][j] = r.get();
            c.im[i][j] = m.get();
        }
    return c;
}

// exp(iX), X = x^a T^a, by the series of exp_i_alg: reduced by X^3 = c1 X + c0,
// Horner's rule.  The powers whose term is below 2^-22 of the sum run in plain
// FP32 (their rounding enters below 2^-46).
__device__ __forceinline__ M3ff ff_exp_i(const ff* v) {
    constexpr double F[25] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320,
                              1.0 / 362880, 1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0,
                              1.0 / 87178291200.0, 1.0 / 1307674368000.0, 1.0 / 20922789888000.0,
                              1.0 / 355687428096000.0, 1.0 / 6402373705728000.0, 1.0 / 121645100408832000.0,
                              1.0 / 2432902008176640000.0, 1.0 / 51090942171709440000.0,
                              1.0 / 1124000727777607680000.0, 1.0 / 25852016738884976640000.0,
                              1.0 / 620448401733239439360000.0};
    // X: real diagonal d, upper triangle a = X01, b = X02, c = X12
    const ff e8 = v[7] * ff_of(0.57735026918962576451);
    ff d0 = ff_scale(v[2] + e8, 0.5f), d1 = ff_scale(e8 - v[2], 0.5f), d2 = -e8;
    ff ar = ff_scale(v[0], 0.5f), ai = ff_scale(v[1], -0.5f);
    ff br = ff_scale(v[3], 0.5f), bi = ff_scale(v[4], -0.5f);
    ff cr = ff_scale(v[5], 0.5f), ci = ff_scale(v[6], -0.5f);
    const float n2 = d0.h * d0.h + d1.h * d1.h + d2.h * d2.h +
                     2.f * (ar.h * ar.h + ai.h * ai.h + br.h * br.h + bi.h * bi.h + cr.h * cr.h + ci.h * ci.h);
    float nrm2 = n2, scl = 1.f;
    int nsq = 0;
    while (nrm2 > 4.f && nsq < 30) { nrm2 *= 0.25f; scl *= 0.5f; nsq++; }
    if (nsq) {
        d0 = ff_scale(d0, scl); d1 = ff_scale(d1, scl); d2 = ff_scale(d2, scl);
        ar = ff_scale(ar, scl); ai = ff_scale(ai, scl);
        br = ff_scale(br, scl); bi = ff_scale(bi, scl);
        cr = ff_scale(cr, scl); ci = ff_scale(ci, scl);
    }
    // S = X^2; d0 + d1 + d2 = 0 leaves three products in each off-diagonal part
    const ff na = FDot(ar, ar).add(ai, ai).get(), nb = FDot(br, br).add(bi, bi).get(), nc = FDot(cr, cr).add(ci, ci).get();
    const ff s0 = ff_fma(d0, d0, na + nb), s1 = ff_fma(d1, d1, na + nc), s2 = ff_fma(d2, d2, nb + nc);
    const ff sar = FDot(br, cr).add(bi, ci).sub(d2, ar).get(), sai = FDot(bi, cr).sub(br, ci).sub(d2, ai).get();
    const ff sbr = FDot(ar, cr).sub(ai, ci).sub(d1, br).get(), sbi = FDot(ar, ci).add(ai, cr).sub(d1, bi).get();
    const ff scr = FDot(ar, br).add(ai, bi).sub(d0, cr).get(), sci = FDot(ar, bi).sub(ai, br).sub(d0, ci).get();
    const ff c1 = ff_scale(s0 + s1 + s2, 0.5f);
    // det X = tr(X^3) / 3
    const ff off = FDot(ar, sar).add(ai, sai).add(br, sbr).add(bi, sbi).add(cr, scr).add(ci, sci).get();
    const ff dia = FDot(d0, s0).add(d1, s1).add(d2, s2).get();
    const ff c0 = (ff_scale(off, 2.f) + dia) * ff_of(1.0 / 3.0);
    ff r0, i0, r1, i1, r2, i2;
    int k;
    {
        const int n = nrm2 <= 0.0625f ? 12 : nrm2 <= 1.f ? 18 : 24;
        const int last = n == 12 ? 6 : n == 18 ? 10 : 14;
        float p0 = n == 12 ? (float)F[12] : n == 18 ? (float)F[18] : (float)F[24];
        float q0 = 0.f, p1 = 0.f, q1 = 0.f, p2 = 0.f, q2 = 0.f;
#pragma unroll
        for (int j = 23; j >= 6; j--)
            if (j < n && j >= last) {
                const float a = fmaf(-c0.h, q2, (float)F[j]), b = c0.h * p2, c = -fmaf(c1.h, q2, q0), d = fmaf(c1.h, p2, p0);
                p2 = -q1; q2 = p1; p0 = a; q0 = b; p1 = c; q1 = d;
            }
        r0 = ff{p0, 0.f}; i0 = ff{q0, 0.f}; r1 = ff{p1, 0.f}; i1 = ff{q1, 0.f}; r2 = ff{p2, 0.f}; i2 = ff{q2, 0.f};
        k = last;
    }
#pragma unroll
    for (int j = 13; j >= 0; j--)
        if (j < k) {
            const ff a = ff_fma(-c0, i2, ff_of(F[j])), b = c0 * r2, c = -ff_fma(c1, i2, i0), d = ff_fma(c1, r2, r0);
            r2 = -i1; i2 = r1; r0 = a; i0 = b; r1 = c; i1 = d;
        }
    M3ff U;
    auto diag = [&](int i, ff d, ff s) {
        U.re[i][i] = r0 + FDot(r1, d).add(r2, s).get();
        U.im[i][i] = i0 + FDot(i1, d).add(i2, s).get();
    };
    diag(0, d0, s0);
    diag(1, d1, s1);
    diag(2, d2, s2);
    // (f1 X + f2 S) at (i, j) and, of the conjugate entries, at (j, i)
    auto pair = [&](int i, int j, ff xr, ff xi, ff sr, ff si) {
        const ff P = FDot(r1, xr).add(r2, sr).get(), Q = FDot(i1, xi).add(i2, si).get();
        const ff A = FDot(r1, xi).add(r2, si).get(), B = FDot(i1, xr).add(i2, sr).get();
        U.re[i][j] = P - Q;
        U.re[j][i] = P + Q;
        U.im[i][j] = A + B;
        U.im[j][i] = B - A;
    };
    pair(0, 1, ar, ai, sar, sai);
    pair(0, 2, br, bi, sbr, sbi);
    pair(1, 2, cr, ci, scr, sci);
#pragma unroll 1
    for (int q = 0; q < nsq; q++) U = ff_mul<3>(U, U);
    return U;
}

// Tables of the normal variates: (cos, sin) of 2 pi j / 256, j <= 256, and per
// 1/128 of [1, 2) a short reciprocal of the cell and minus its logarithm.
static constexpr int FF_ANGLES = 257, FF_LOGS = 128;
struct FFTables {
    float4 angle[FF_ANGLES];  // cos hi, lo, sin hi, lo
    float4 log[FF_LOGS];      // 1 / c, then -log(1 / c) hi, lo
};
// cells above sqrt 2 are taken at half their value, so that values next to a
// power of two have a reciprocal of exactly 1 and keep their relative accuracy
__device__ __forceinline__ bool ff_log_half(int i) { return i >= 53; }
__device__ __forceinline__ void ff_table_entry(FFTables* t, int i) {
    if (i < FF_ANGLES) {
        double s, c;
        sincospi(i / 128.0, &s, &c);
        const ff cf = ff_of(c), sf = ff_of(s);
        t->angle[i] = make_float4(cf.h, cf.l, sf.h, sf.l);
    }
    if (i < FF_LOGS) {
        const double f = (1.0 + (i + 0.5) / 128.0) * (ff_log_half(i) ? 0.5 : 1.0);
        // 11 bits
        double r = i == 0 || i == FF_LOGS - 1 ? 1.0 : rint(1024.0 / f) / 1024.0;
        const ff l = ff_of(-log(r));
        t->log[i] = make_float4((float)r, l.h, l.l, 0.f);
    }
}

// Box-Muller of u = (r + 1/2) 2^-32 for two 32-bit words: sqrt(-2 ln u1) times
// the cosine and sine of 2 pi u2.  Table-driven logarithm (Tang's method) and
// sine, with series in the remainder below 2^-7 and pi / 256.
__device__ __forceinline__ void ff_box_muller(uint32_t w1, uint32_t w2, const FFTables* __restrict__ tab, ff& z0, ff& z1) {
    // u1 = m 2^-33 = 2^(k - 33) f, f in [1, 2)
    const uint64_t m = 2 * (uint64_t)w1 + 1;
    const int k = 63 - __clzll((long long)m);
    const uint64_t f = m << (33 - k);          // 34 bits: leading one at bit 33
    const int i = (int)(f >> 26) & 127;
    const bool half = ff_log_half(i);
    const float4 e = __ldg(&tab->log[i]);
    const float sc = half ? 0x1p-34f : 0x1p-33f;
    const float fh = (float)(uint32_t)(f >> 10) * sc * 1024.f, fl = (float)((uint32_t)f & 1023u) * sc;
    const float p = __fmul_rn(fh, e.x);
    const ff t = ff_quick(__fsub_rn(p, 1.0f), fmaf(fl, e.x, fmaf(fh, e.x, -p)));
    // log1p(t) = t - t^2/2 + t^3/3 - t^4 (1/4 - t/5 + t^2/6)
    const ff t2 = t * t;
    const float t4 = -(t2.h * t2.h) * fmaf(t.h, fmaf(t.h, 1.f / 6, -1.f / 5), 1.f / 4);
    const float E = (float)(k - 33 + (half ? 1 : 0));
    const ff cu = t2 * t * ff_of(1.0 / 3.0);
    ff ln = ff_times(ff_of(0.69314718055994530942), E) + ff{e.y, e.z};
    ln = ln + (t + (ff_scale(t2, -0.5f) + ff_quick(cu.h, cu.l + t4)));
    // sqrt(-2 ln u1)
    const ff x = ff_scale(ln, -2.0f);
    const float y = rsqrtf(x.h), s = x.h * y;
    const ff rad = ff_quick(s, 0.5f * y * (fmaf(-s, s, x.h) + x.l));
    // 2 pi u2 = 2 pi j / 256 + d
    const uint64_t m2 = 2 * (uint64_t)w2 + 1;
    const int j = (int)((m2 + (1u << 24)) >> 25);
    const float rem = (float)(int)((int64_t)m2 - ((int64_t)j << 25));
    const ff d = ff_times(ff_of(6.28318530717958647693 / 8589934592.0), rem);
    const float d2 = d.h * d.h;
    const ff sd = ff_quick(d.h, d.l + d.h * d2 * fmaf(d2, 1.f / 120, -1.f / 6));
    const ff dd = d * d;
    const ff cm = ff_quick(-0.5f * dd.h, fmaf(d2 * d2, fmaf(d2, -1.f / 720, 1.f / 24), -0.5f * dd.l));  // cos d - 1
    const float4 cs = __ldg(&tab->angle[j]);
    const ff C{cs.x, cs.y}, S{cs.z, cs.w};
    z0 = rad * (C + FDot(C, cm).sub(S, sd).get());
    z1 = rad * (S + FDot(S, cm).add(C, sd).get());
}

}  // namespace gl
