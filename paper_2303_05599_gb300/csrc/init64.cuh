// The MV initial conditions of FP64 events (the quantities are init.cu's).
//
// The plain FP64 method keeps one order of roundings.  The unitarity that the
// field checks report for an FP64 state right after its initial conditions is
// made of these roundings alone (1e-15 a link), so any other order of the same
// sums reports another number.  Hence eight complex planes a sheet (one for
// each colour), transforms of radix 2 in bit-reversed order, rows before
// columns in both directions, the 20-term exponential series, whole matrices
// multiplied sheet after sheet, and a Newton step in FP64 with row exchanges.
//
// What bounds it: FP64 arithmetic (a warp instruction takes 76 cycles of its
// scheduler), on small lattices the chain of one thread.  So everything that
// does not depend on another sheet runs for a round of sheets of both nuclei
// and of every event at once, and only the products are made in order, a
// matrix row by each of three warps:
//   rows      rho of a few lattice rows and their forward transforms
//   columns   forward transforms, Green function
//   rows, columns  inverse transforms
//   exp       exp(-i alpha) of every site and sheet, in the place of alpha
//   products  the Wilson lines
// Twiddles come from a table of each sign, and the Jacobian of a Newton step
// from the entries of K that K T^b is made of (the other products are with 0).
// Measured: a 32^2 event of 50 sheets 10474 us with seven launches a sheet, a
// sincospi a butterfly and eight matrix products a Newton step, 900 us so, in three
// rounds of 17 sheets; all in one round 829 us (normal variates 60, transforms 170,
// exponentials 68, products 89, links 270); with init.cu's transforms and series in
// FP64 it was 550 us, in other roundings.
#pragma once
#include "internal.h"
#include "layout.cuh"
#include "philox.cuh"

namespace gl {

static constexpr int INIT64_PLANES = 9;  // a sheet's slot: 8 colour planes, then the 9 entries of its exponential

// a line's points are placed in bit-reversed order where the transform starts from it
__device__ __forceinline__ int line_place(const InitEv& d, int k) {
    return d.pow2 ? (int)(__brev((unsigned)k) >> (32 - d.log2N)) : k;
}

// `lines` lines of a power-of-two length, `ls` points apart, in place (a barrier after each pass)
__device__ __forceinline__ void radix2_lines(double2* sh, int lines, int ls, const InitEv& d,
                                             const double2* __restrict__ tw) {
    const int N = d.N, lh = d.log2N - 1;
    for (int l = 0; l <= lh; l++) {
        const int half = 1 << l;
        for (int b = threadIdx.x; b < lines << lh; b += blockDim.x) {
            const int j = b & ((N >> 1) - 1), k = j & (half - 1);
            double2* p = sh + (b >> lh) * ls + ((j >> l) << (l + 1)) + k;
            const double2 w = __ldg(tw + (k << (lh - l)));
            const double cs = w.x, sn = w.y;
            const double2 u = p[0], v = p[half];
            const double2 vw = make_double2(v.x * cs - v.y * sn, v.x * sn + v.y * cs);
            p[0] = make_double2(u.x + vw.x, u.y + vw.y);
            p[half] = make_double2(u.x - vw.x, u.y - vw.y);
        }
        __syncthreads();
    }
}

// point k of a line's transform: in place after radix2_lines, else the direct sum
__device__ __forceinline__ double2 line_point(const double2* sh, int k, const InitEv& d,
                                              const double2* __restrict__ tw) {
    if (d.pow2) return sh[k];
    const int N = d.N;
    double re = 0, im = 0;
    int m = 0;  // j k mod N
    for (int j = 0; j < N; j++) {
        const double2 w = __ldg(tw + m);
        const double cs = w.x, sn = w.y;
        re += sh[j].x * cs - sh[j].y * sn;
        im += sh[j].x * sn + sh[j].y * cs;
        m += k;
        if (m >= N) m -= N;
    }
    return make_double2(re, im);
}

// d.lines rows of two colour planes of a sheet: rho and its forward transforms, or the inverse ones
template <bool FIRST>
__global__ void __launch_bounds__(256) init64_rows_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    extern __shared__ __align__(16) unsigned char init_smem[];
    double2* sh = (double2*)init_smem;
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_ROWS, &blk);
    const int N = d.N, S = d.S, nb = (N + d.lines - 1) / d.lines;
    const int row0 = (blk % nb) * d.lines, pair = (blk / nb) & 3, slot = blk / (4 * nb);
    const int nucleus = slot / S, sheet = round * S + slot - nucleus * S;
    if (sheet >= d.Ns) return;
    const int nl = N - row0 < d.lines ? N - row0 : d.lines, np = nl * N;
    const int64_t Vn = (int64_t)N * N;
    double2* w = slot_at(d, (size_t)slot * INIT64_PLANES * Vn) + 2 * pair * Vn + (size_t)row0 * N;
    for (int idx = threadIdx.x; idx < np; idx += blockDim.x) {
        const int l = idx / N, at = l * N + line_place(d, idx - l * N);
        if (FIRST) {
            const U4 r = philox4x32_10(U4{(uint32_t)(row0 * N + idx),
                                          (uint32_t)((nucleus * d.Ns + sheet) * 2 + (pair >> 1)), 1u, 0u}, d.k0, d.k1);
            double z0, z1;
            box_muller(u01((pair & 1) ? r.z : r.x), u01((pair & 1) ? r.w : r.y), z0, z1);
            sh[at] = make_double2(d.sigma * z0, 0.0);
            sh[np + at] = make_double2(d.sigma * z1, 0.0);
        } else {
            sh[at] = w[idx];
            sh[np + at] = w[Vn + idx];
        }
    }
    __syncthreads();
    const double2* tw = FIRST ? d.tw + N : d.tw;
    if (d.pow2) radix2_lines(sh, 2 * nl, N, d, tw);
    for (int idx = threadIdx.x; idx < 2 * np; idx += blockDim.x) {
        const int l = idx / N, k = idx - l * N;
        w[idx < np ? idx : Vn + idx - np] = line_point(sh + l * N, k, d, tw);
    }
}

// a tile of columns of one plane; the forward transforms are multiplied by the Green function
template <bool FORWARD>
__global__ void __launch_bounds__(256) init64_cols_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    extern __shared__ __align__(16) unsigned char init_smem[];
    double2* sh = (double2*)init_smem;
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_COLS, &blk);
    const int N = d.N, S = d.S, nt = (N + d.cols - 1) / d.cols, ls = N + 1;
    const int c0 = (blk % nt) * d.cols, plane = (blk / nt) & 7, slot = blk / (8 * nt);
    if (round * S + slot % S >= d.Ns) return;
    const int nc = N - c0 < d.cols ? N - c0 : d.cols;
    double2* w = slot_at(d, (size_t)slot * INIT64_PLANES * N * N) + (size_t)plane * N * N + c0;
    for (int idx = threadIdx.x; idx < nc * N; idx += blockDim.x) {
        const int r = idx / nc, c = idx - r * nc;
        sh[c * ls + line_place(d, r)] = w[(size_t)r * N + c];
    }
    __syncthreads();
    const double2* tw = FORWARD ? d.tw + N : d.tw;
    if (d.pow2) radix2_lines(sh, nc, ls, d, tw);
    for (int idx = threadIdx.x; idx < nc * N; idx += blockDim.x) {
        const int r = idx / nc, c = idx - r * nc;
        double2 v = line_point(sh + c * ls, r, d, tw);
        if (FORWARD) {
            const double g = d.green[(size_t)r * N + c0 + c];
            v = make_double2(v.x * g, v.y * g);
        }
        w[(size_t)r * N + c] = v;
    }
}

// exp(i X) for Hermitian traceless X = x^a T^a by the first 20 powers of iX for |X| <= 1 (scaled and
// squared beyond), each a combination of 1, X, X^2 by X^3 = c1 X + c0
__device__ __forceinline__ M3<double> exp_series20(const A8<double>& x) {
    M3<double> X;
    const double s3 = inv_sqrt3<double>();
    X.re[0][0] = 0.5 * (x.v[2] + x.v[7] * s3);
    X.re[1][1] = 0.5 * (-x.v[2] + x.v[7] * s3);
    X.re[2][2] = 0.5 * (-2.0 * (x.v[7] * s3));
    X.im[0][0] = X.im[1][1] = X.im[2][2] = 0.0;
    X.re[0][1] = X.re[1][0] = 0.5 * x.v[0];
    X.im[0][1] = 0.5 * -x.v[1];
    X.im[1][0] = -X.im[0][1];
    X.re[0][2] = X.re[2][0] = 0.5 * x.v[3];
    X.im[0][2] = 0.5 * -x.v[4];
    X.im[2][0] = -X.im[0][2];
    X.re[1][2] = X.re[2][1] = 0.5 * x.v[5];
    X.im[1][2] = 0.5 * -x.v[6];
    X.im[2][1] = -X.im[1][2];
    M3<double> X2 = sq_herm(X);
    double c1 = 0.5 * (X2.re[0][0] + X2.re[1][1] + X2.re[2][2]);
    int nsq = 0;
    double scl = 1.0, nrm2 = 2.0 * c1;
    while (nrm2 > 1.0 && nsq < 30) { nrm2 *= 0.25; scl *= 0.5; nsq++; }
    if (nsq) {
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) {
                X.re[i][j] *= scl; X.im[i][j] *= scl;
                X2.re[i][j] *= scl * scl; X2.im[i][j] *= scl * scl;
            }
        c1 *= scl * scl;
    }
    const double pr = X.re[0][1] * X.re[1][2] - X.im[0][1] * X.im[1][2];
    const double pi_ = X.re[0][1] * X.im[1][2] + X.im[0][1] * X.re[1][2];
    const double n01 = X.re[0][1] * X.re[0][1] + X.im[0][1] * X.im[0][1];
    const double n02 = X.re[0][2] * X.re[0][2] + X.im[0][2] * X.im[0][2];
    const double n12 = X.re[1][2] * X.re[1][2] + X.im[1][2] * X.im[1][2];
    const double c0 = X.re[0][0] * (X.re[1][1] * X.re[2][2] - n12) - X.re[1][1] * n02 - X.re[2][2] * n01 +
                      2.0 * (pr * X.re[0][2] + pi_ * X.im[0][2]);
    // (iX)^k / k! = i^k (a + b X + g X^2)
    double a = 1.0, b = 0.0, g = 0.0;
    double f0r = 1.0, f0i = 0.0, f1r = 0.0, f1i = 0.0, f2r = 0.0, f2i = 0.0;
#pragma unroll
    for (int k = 1; k <= 20; k++) {
        const double inv = 1.0 / (double)k;
        const double na = c0 * g * inv, nb = (a + c1 * g) * inv, ng = b * inv;
        a = na; b = nb; g = ng;
        if ((k & 3) == 1) { f0i += a; f1i += b; f2i += g; }
        else if ((k & 3) == 2) { f0r -= a; f1r -= b; f2r -= g; }
        else if ((k & 3) == 3) { f0i -= a; f1i -= b; f2i -= g; }
        else { f0r += a; f1r += b; f2r += g; }
    }
    M3<double> U;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const double e = (i == j) ? 1.0 : 0.0;
            U.re[i][j] = f0r * e + f1r * X.re[i][j] - f1i * X.im[i][j] + f2r * X2.re[i][j] - f2i * X2.im[i][j];
            U.im[i][j] = f0i * e + f1r * X.im[i][j] + f1i * X.re[i][j] + f2r * X2.im[i][j] + f2i * X2.re[i][j];
        }
    for (int k = 0; k < nsq; k++) U = mul(U, U);
    return U;
}

__global__ void __launch_bounds__(128) init64_exp_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_SHEETS, &blk);
    const int64_t Vn = (int64_t)d.N * d.N, t = (int64_t)blk * 128 + threadIdx.x;
    const int slot = (int)(t / Vn);
    if (slot >= 2 * d.S || round * d.S + slot % d.S >= d.Ns) return;
    const int64_t s = t - slot * Vn;
    // only this thread reads and writes the site's slot
    double2* w = slot_at(d, (size_t)slot * INIT64_PLANES * Vn);
    A8<double> al;
#pragma unroll
    for (int a = 0; a < 8; a++) al.v[a] = -w[(size_t)a * Vn + s].x;
    store_link(w, 0, s, Vn, exp_series20(al));
}

// Wilson lines: warp r of a block has row r of its 32 sites' matrices
__global__ void __launch_bounds__(96) init64_products_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_PRODUCTS, &blk);
    const int64_t Vn = (int64_t)d.N * d.N;
    const int nb = (int)((Vn + 31) / 32), nucleus = blk / nb, r = threadIdx.x >> 5;
    const int64_t s = (int64_t)(blk - nucleus * nb) * 32 + (threadIdx.x & 31);
    if (s >= Vn) return;
    int n = d.Ns - round * d.S;
    if (n > d.S) n = d.S;
    double2* V = d.V + ((size_t)nucleus * 9 + 3 * r) * Vn + s;
    // this round's sheet k
    const size_t step = (size_t)INIT64_PLANES * Vn;
    auto sheet = [&](int k) { return slot_at(d, (size_t)(nucleus * d.S + k) * step); };
    double2 v[3];
    int first = 0;
    if (round == 0) {
        // the unit matrix times the first sheet
#pragma unroll
        for (int j = 0; j < 3; j++) v[j] = sheet(0)[(size_t)(3 * r + j) * Vn + s];
        first = 1;
    } else {
        if (n <= 0) return;
#pragma unroll
        for (int j = 0; j < 3; j++) v[j] = V[(size_t)j * Vn];
    }
    // the next sheet's exponential on its way while one is multiplied
    M3<double> next = m_zero<double>();
    if (first < n) next = load_link(sheet(first), 0, s, Vn);
#pragma unroll 1
    for (int k = first; k < n; k++) {
        const M3<double> m = next;
        if (k + 1 < n) next = load_link(sheet(k + 1), 0, s, Vn);
        double2 o[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double sr = 0, si = 0;
#pragma unroll
            for (int q = 0; q < 3; q++) {
                sr = fma(v[q].x, m.re[q][j], sr);
                sr = fma(-v[q].y, m.im[q][j], sr);
                si = fma(v[q].x, m.im[q][j], si);
                si = fma(v[q].y, m.re[q][j], si);
            }
            o[j] = make_double2(sr, si);
        }
#pragma unroll
        for (int j = 0; j < 3; j++) v[j] = o[j];
    }
#pragma unroll
    for (int j = 0; j < 3; j++) V[(size_t)j * Vn] = v[j];
}

// F^a = Im tr T^a W (1 + U^+) and its largest entry
__device__ __forceinline__ double residual64(const M3<double>& W, const M3<double>& U, double* F) {
    M3<double> ud = dag(U);
    ud.re[0][0] += 1; ud.re[1][1] += 1; ud.re[2][2] += 1;
    im_tr_T(mul(W, ud), F);
    double r = 0;
#pragma unroll
    for (int a = 0; a < 8; a++) r = fmax(r, fabs(F[a]));
    return r;
}

// column b of the Jacobian, -Re tr(T^a K T^b).  Columns p and q of K T^b are columns q and p of K times
// +-1/2 or +-i/2; those of T^3 and T^8, which are diagonal, times its entries.
template <int b>
__device__ __forceinline__ void jacobian_column(const M3<double>& K, double (&J)[8][8]) {
    M3<double> T = m_zero<double>();
    if (b == 2 || b == 7) {
        const double c = 0.5 * inv_sqrt3<double>();
        const double e[3] = {b == 2 ? 0.5 : c, b == 2 ? -0.5 : c, b == 2 ? 0.0 : -inv_sqrt3<double>()};
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < (b == 2 ? 2 : 3); j++) {
                T.re[i][j] = __dmul_rn(K.re[i][j], e[j]);
                T.im[i][j] = __dmul_rn(K.im[i][j], e[j]);
            }
    } else {
        constexpr int p = b < 5 ? 0 : 1, q = b < 2 ? 1 : 2;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if (b == 0 || b == 3 || b == 5) {  // T_pq = T_qp = 1/2
                T.re[i][p] = 0.5 * K.re[i][q]; T.im[i][p] = 0.5 * K.im[i][q];
                T.re[i][q] = 0.5 * K.re[i][p]; T.im[i][q] = 0.5 * K.im[i][p];
            } else {                           // T_pq = -i/2, T_qp = i/2
                T.re[i][p] = -0.5 * K.im[i][q]; T.im[i][p] = 0.5 * K.re[i][q];
                T.re[i][q] = 0.5 * K.im[i][p]; T.im[i][q] = -0.5 * K.re[i][p];
            }
        }
    }
    double re[8];
    re_tr_T(T, re);
#pragma unroll
    for (int a = 0; a < 8; a++) J[a][b] = -re[a];
}

// J x = b in place of b, rows exchanged for the largest pivot (by selects, so
// that J stays in registers); 1 if J is singular
template <int c>
__device__ __forceinline__ int eliminate8(double (&J)[8][8], double (&b)[8]) {
    int p = c;
    double most = fabs(J[c][c]);
#pragma unroll
    for (int r = c + 1; r < 8; r++)
        if (fabs(J[r][c]) > most) { most = fabs(J[r][c]); p = r; }
    int singular = most < 1e-300;
#pragma unroll
    for (int r = c + 1; r < 8; r++) {
        const bool swap = r == p;
#pragma unroll
        for (int k = c; k < 8; k++) {
            const double u = J[c][k], w = J[r][k];
            J[c][k] = swap ? w : u;
            J[r][k] = swap ? u : w;
        }
        const double u = b[c], w = b[r];
        b[c] = swap ? w : u;
        b[r] = swap ? u : w;
    }
#pragma unroll
    for (int r = c + 1; r < 8; r++) {
        const double f = J[r][c] / J[c][c];
#pragma unroll
        for (int k = c + 1; k < 8; k++) J[r][k] = fma(-f, J[c][k], J[r][k]);
        b[r] = fma(-f, b[c], b[r]);
    }
    if constexpr (c < 7) singular |= eliminate8<c + 1>(J, b);
#pragma unroll
    for (int k = c + 1; k < 8; k++) b[c] = fma(-J[c][k], b[k], b[c]);
    b[c] /= J[c][c];
    return singular;
}

// Newton solve for the Glasma link from the pure-gauge links of both nuclei
__device__ __forceinline__ int solve_link64(const M3<double>& UA, const M3<double>& UB, M3<double>& U) {
    const M3<double> W = add(UA, UB);
    U = mul(UA, UB);
    double F[8];
    double r = residual64(W, U, F);
#pragma unroll 1
    for (int it = 0; it < 100 && r > 1e-14; it++) {
        A8<double> dx;
        {
            const M3<double> K = mul_nd(W, U);
            double J[8][8];
            jacobian_column<0>(K, J); jacobian_column<1>(K, J); jacobian_column<2>(K, J); jacobian_column<3>(K, J);
            jacobian_column<4>(K, J); jacobian_column<5>(K, J); jacobian_column<6>(K, J); jacobian_column<7>(K, J);
#pragma unroll
            for (int a = 0; a < 8; a++) dx.v[a] = -F[a];
            if (eliminate8<0>(J, dx.v)) break;
        }
        double lam = 1.0;
#pragma unroll 1
        for (int k = 0; k < 30; k++) {
            A8<double> st;
#pragma unroll
            for (int a = 0; a < 8; a++) st.v[a] = lam * dx.v[a];
            const M3<double> Un = mul(exp_series20(st), U);
            double Fn[8];
            const double rn = residual64(W, Un, Fn);
            if (rn < r || k == 29) {
                U = Un;
                r = rn;
#pragma unroll
                for (int a = 0; a < 8; a++) F[a] = Fn[a];
                break;
            }
            lam *= 0.5;
        }
    }
    return r > 1e-12;
}

// the Glasma link (d, s) into the event's fields, and i[-i[U^A]_ah, -i[U^B]_ah] of the link
__global__ void __launch_bounds__(64) init64_links_kernel(const InitEv* evs, int ne, InitEv one) {
    int blk;
    const InitEv& ev = init_find(evs, ne, one, IK_LINKS, &blk);
    const int N = ev.N;
    const int64_t Vn = (int64_t)N * N, l = (int64_t)blk * 64 + threadIdx.x;
    if (l >= 2 * Vn) return;
    const int d = (int)(l / Vn);
    const int64_t s = l % Vn;
    const int x = (int)(s % N), y = (int)(s / N);
    const int64_t sn = d == 0 ? (int64_t)y * N + (x + 1 == N ? 0 : x + 1) : (int64_t)(y + 1 == N ? 0 : y + 1) * N + x;
    const double2* VB = ev.V + (size_t)9 * Vn;
    const M3<double> UA = mul_dn(load_link(ev.V, 0, s, Vn), load_link(ev.V, 0, sn, Vn));
    const M3<double> UB = mul_dn(load_link(VB, 0, s, Vn), load_link(VB, 0, sn, Vn));
    store_alg(ev.comm + (size_t)d * 4 * Vn, s, Vn, icomm(iah_to_alg(UA), iah_to_alg(UB)));
    M3<double> U;
    if (solve_link64(UA, UB, U)) atomicAdd(ev.bad, 1);
    store_link(carve_fields<double>(ev.fields, Vn).U, d, s, Vn, U);
}

}  // namespace gl
