// Fused Glasma leapfrog step and site E/B interpolation (Sec. 2.1 and 3.2 of
// arXiv:2303.05599) on shared-memory tiles.
//
// One CTA owns a TX x TY tile of sites (FP64; FP32 has strip_body.cuh).  Per
// step it computes, from U(n), phi(n), e(n-1/2), pi(n-1/2):
//   the momenta e(n+1/2), pi(n+1/2), the links U(n+1) and the scalar phi(n+1),
//   and the site fields E, B at t_n that the particle push gathers.
// Every cell plaquette is formed once per tile and shared.  With
//   A(c)  = components of i[P(c)]_ah,  P(c) = Ux(c) Uy(c+x) Ux(c+y)^+ Uy(c)^+,
//   Dn(s) = Uy(s-y)^+ A(s-y) Uy(s-y),   Lf(s) = Ux(s-x)^+ A(s-x) Ux(s-x),
// the plaquette forces and the clover are
//   F_x = t (A - Dn),  F_y = t (Lf - A),
//   B_eta = (A + Lf + Dn + Uy(s-y)^+ Lf(s-y) Uy(s-y)) / 4.
// E_x(s) needs e_x(n+1/2) at s - x and E_y(s) needs e_y(n+1/2) at s - y, so
// the tile also advances e_x on one halo column (x0 - 1) and e_y (with Lf) on
// one halo row (y0 - 1); nothing else of the halo is needed.
//
// The tile's inputs are copied to shared memory with cp.async in the storage
// layout of global memory (16-byte vectors).  Regions, in tile coordinates:
//   links, phi:                   x in [-1, TX],   y in [-1, TY]    (LW x LH)
//   plaquettes A, momenta, Lf:    x in [-1, TX-1], y in [-1, TY-1]  (EW x EH)
// pi(n-1/2) is read by each site's thread straight from global memory.
//
// Bound by the FP64 pipe, which a warp instruction keeps for 64 cycles however
// many of its lanes work, so the halo's work is packed: its plaquettes are
// spread a matrix row a thread, its two kinds of transports over two warps.  A
// 16x8 tile has 25 plaquettes and 24 momenta beyond its own 128 sites (32x4: 37
// and 36, which took two and a half warps' passes of their own, a momentum's
// both directions one after the other): nine events of 64/128/256 1283 -> 1164
// us, a 256^2 event 379 -> 336 us; 32x4 tiles with the packed halo 1322 and 375.
// Every operation whose fusion would depend on what surrounds it is explicit, so
// the results do not depend on the tile shape.  The links arrive in their own
// group of copies, so the plaquettes start while phi and e(n-1/2) are in flight.
#pragma once
#include "internal.h"
#include "layout.cuh"

namespace gl {

template <typename R, int TX, int TY>
struct Tile {
    using V = typename Prec<R>::V;
    static constexpr int LP = Prec<R>::LP, AP = Prec<R>::AP;
    static constexpr int LW = TX + 2, LH = TY + 2, LN = LW * LH;
    static constexpr int EW = TX + 1, EH = TY + 1, EN = EW * EH;
    static constexpr int NT = TX * TY;
    static constexpr int NH = TX + TY;  // halo momenta: left column (e_x), bottom row (e_y, Lf)
    static constexpr int REST = EN - NT;  // plaquettes beyond one a thread
    static_assert(9 * REST <= AP * EN, "their matrices wait in the place of Lf");
    // vectors: links 2 LP LN, phi AP LN, A AP EN, e sums 2 AP EN, Lf AP EN, halo items AP (NH + TY)
    static constexpr size_t vecs = (size_t)2 * LP * LN + (size_t)AP * LN + (size_t)4 * AP * EN + (size_t)AP * (NH + TY);
    static constexpr size_t bytes = vecs * sizeof(V);
};

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// link (d) of shared-memory site li, planes of LN vectors
__device__ __forceinline__ M3<double> s_link(const double2* sU, int d, int li, int LN) {
    const double2* b = sU + (size_t)d * 9 * LN + li;
    M3<double> m;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const double2 v = b[k * LN];
        m.re[k / 3][k % 3] = v.x;
        m.im[k / 3][k % 3] = v.y;
    }
    return m;
}

// links of the tile in shared memory
template <typename R>
struct SLinks;
template <>
struct SLinks<double> {
    const double2* u;
    int LN;
    __device__ __forceinline__ M3<double> operator()(int d, int li) const { return s_link(u, d, li, LN); }
};
__device__ __forceinline__ A8<double> s_alg(const double2* s, int i, int n) {
    A8<double> x;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const double2 v = s[k * n + i];
        x.v[2 * k] = v.x;
        x.v[2 * k + 1] = v.y;
    }
    return x;
}
__device__ __forceinline__ void s_alg_put(double2* s, int i, int n, const A8<double>& x) {
#pragma unroll
    for (int k = 0; k < 4; k++) s[k * n + i] = make_double2(x.v[2 * k], x.v[2 * k + 1]);
}

struct StepArgs {
    int N;
    int tiles_x;
    double t, dt, inv_t, dt_over_th, dt_th;
    int reunit;
};

// the step scalars in the kernel's precision (converted once per launch or
// block: double arithmetic costs far more than single on GPUs with slow FP64)
template <typename R>
struct StepR {
    int N, tiles_x, reunit;
    R t, dt, inv_t, dt_over_th, dt_th;
};
template <typename R>
__host__ __device__ inline StepR<R> step_r(const StepArgs& a) {
    StepR<R> r;
    r.N = a.N;
    r.tiles_x = a.tiles_x;
    r.reunit = a.reunit;
    r.t = (R)a.t;
    r.dt = (R)a.dt;
    r.inv_t = (R)a.inv_t;
    r.dt_over_th = (R)a.dt_over_th;
    r.dt_th = (R)a.dt_th;
    return r;
}

// e(n+1/2) = e(n-1/2) + dt (t F + c / t), F the plaquette force and c the scalar
// current (shared with the small tiles, one rounding order)
template <typename R>
__device__ __forceinline__ R next_e(R e, R F, R c, R t, R dt, R inv_t) {
    return fma(dt, fma(t, F, mul_rn(inv_t, c)), e);
}

// a row of a matrix product, q = p m and q = p m^+, in the order of mul and mul_nd
template <typename R>
__device__ __forceinline__ void row_mul(const R* pr, const R* pi, const M3<R>& m, R* qr, R* qi) {
#pragma unroll
    for (int j = 0; j < 3; j++) {
        R sr = 0, si = 0;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            sr = fma(pr[k], m.re[k][j], sr);
            sr = fma(-pi[k], m.im[k][j], sr);
            si = fma(pr[k], m.im[k][j], si);
            si = fma(pi[k], m.re[k][j], si);
        }
        qr[j] = sr;
        qi[j] = si;
    }
}
template <typename R>
__device__ __forceinline__ void row_mul_dag(const R* pr, const R* pi, const M3<R>& m, R* qr, R* qi) {
#pragma unroll
    for (int j = 0; j < 3; j++) {
        R sr = 0, si = 0;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            sr = fma(pr[k], m.re[j][k], sr);
            sr = fma(pi[k], m.im[j][k], sr);
            si = fma(pi[k], m.re[j][k], si);
            si = fma(-pr[k], m.im[j][k], si);
        }
        qr[j] = sr;
        qi[j] = si;
    }
}

// one tile (index `tile` of a lattice with tiles_x tiles per row); the caller
// provides the dynamic shared memory of Tile<R, TX, TY>::bytes
template <typename R, int TX, int TY>
__device__ __forceinline__ void fused_tile(const Fields<R>& in, const Fields<R>& out, typename Prec<R>::V* site,
                                           const StepR<R>& a, int tile) {
    using T = Tile<R, TX, TY>;
    using Vec = typename Prec<R>::V;
    constexpr int LP = T::LP, AP = T::AP;
    constexpr int LW = T::LW, LN = T::LN, EW = T::EW, EN = T::EN, NT = T::NT, NH = T::NH, REST = T::REST;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Vec* sU = (Vec*)smem_raw;          // [2][LP][LN]
    Vec* sPhi = sU + 2 * LP * LN;      // [AP][LN]
    Vec* sA = sPhi + AP * LN;          // [AP][EN]
    Vec* sEs = sA + AP * EN;           // [2][AP][EN]: e(n-1/2), then e(n-1/2) + e(n+1/2)
    Vec* sLf = sEs + 2 * AP * EN;      // [AP][EN]
    Vec* sHalo = sLf + AP * EN;        // [AP][NH] scalar currents, [AP][TY] transported plaquettes of the left column
    const SLinks<R> lk{sU, LN};

    const int N = a.N;
    const int64_t Vn = (int64_t)N * N;
    const int x0 = (tile % a.tiles_x) * TX, y0 = (tile / a.tiles_x) * TY;
    const int tid = threadIdx.x;
    const R t = a.t, dt = a.dt, inv_t = a.inv_t;
    // this thread's site in tile coordinates and its shared-memory indices
    const int ix = tid % TX, iy = tid / TX;
    const int ls = (iy + 1) * LW + (ix + 1), es = (iy + 1) * EW + (ix + 1);

    // ---- phase 1: asynchronous copies of the tile's inputs, in two groups:
    // the links (all phase 2 needs), then phi and e(n-1/2)
    for (int i = tid; i < LN; i += NT) {
        const int gx = wrapi(x0 + i % LW - 1, N), gy = wrapi(y0 + i / LW - 1, N);
        const int64_t g = (int64_t)gy * N + gx;
#pragma unroll
        for (int k = 0; k < 2 * LP; k++) cp_async16(sU + (size_t)k * LN + i, in.U + (size_t)k * Vn + g);
    }
    cp_async_commit();
    for (int i = tid; i < LN; i += NT) {
        const int gx = wrapi(x0 + i % LW - 1, N), gy = wrapi(y0 + i / LW - 1, N);
        const int64_t g = (int64_t)gy * N + gx;
#pragma unroll
        for (int k = 0; k < AP; k++) cp_async16(sPhi + (size_t)k * LN + i, in.phi + (size_t)k * Vn + g);
    }
    for (int i = tid; i < EN; i += NT) {
        const int gx = wrapi(x0 + i % EW - 1, N), gy = wrapi(y0 + i / EW - 1, N);
        const int64_t g = (int64_t)gy * N + gx;
#pragma unroll
        for (int k = 0; k < 2 * AP; k++) cp_async16(sEs + (size_t)k * EN + i, in.e + (size_t)k * Vn + g);
    }
    cp_async_commit();
    cp_async_wait_group<1>();
    __syncthreads();

    // ---- phase 2: plaquettes of the cells x in [-1, TX-1], y in [-1, TY-1]:
    // one a thread, and of the REST that are left a row of the matrix a thread
    // (in the place of Lf), so that they fill warps
    for (int i = tid; i < 3 * REST; i += NT) {
        const int r = i / REST, j = i - r * REST, c = NT + j, l = (c / EW) * LW + (c % EW);
        R pr[3], pi[3], qr[3], qi[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const Vec v = sU[(size_t)(r * 3 + k) * LN + l];
            pr[k] = v.x;
            pi[k] = v.y;
        }
        row_mul(pr, pi, lk(1, l + 1), qr, qi);
        row_mul_dag(qr, qi, lk(0, l + LW), pr, pi);
        row_mul_dag(pr, pi, lk(1, l), qr, qi);
#pragma unroll
        for (int k = 0; k < 3; k++) sLf[(size_t)(r * 3 + k) * REST + j] = Vec{qr[k], qi[k]};
    }
    {
        const int l = (tid / EW) * LW + (tid % EW);  // cell (tid % EW - 1, tid / EW - 1)
        const M3<R> C = mul(lk(0, l), lk(1, l + 1));
        s_alg_put(sA, tid, EN, iah_of_mul_nd(mul_nd(C, lk(0, l + LW)), lk(1, l)));
    }
    cp_async_wait_group<0>();
    __syncthreads();
    for (int j = tid; j < REST; j += NT) {
        M3<R> P;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const Vec v = sLf[(size_t)k * REST + j];
            P.re[k / 3][k % 3] = v.x;
            P.im[k / 3][k % 3] = v.y;
        }
        s_alg_put(sA, NT + j, EN, iah_to_alg(P));
    }
    __syncthreads();

    // ---- phase 3: momenta at n+1/2 of the tile site (kept in registers for
    // phase 4) and of the halo: bottom row (h, -1), e_y and Lf only, and left
    // column (-1, h), e_x only.  A halo item's transport of the plaquette and its
    // scalar current go to two warps, its update follows the barrier.  Each
    // operation rounds alike wherever it stands (explicit fused operations), so a
    // momentum is the same bits whether the site is a tile's own or another's halo.
    A8<R> my_ex, my_ey, my_tx, my_ty, my_b;
    const int gx = x0 + ix, gy = y0 + iy;
    const bool valid = gx < N && gy < N;
    const int64_t g = (int64_t)gy * N + gx;
    {
        const A8<R> A0 = s_alg(sA, es, EN);
        const A8<R> ph = s_alg(sPhi, ls, LN);
        A8<R> sum;
        const A8<R> Dn = conj_dn_t(lk(1, ls - LW), s_alg(sA, es - EW, EN));
        my_tx = conj_up_t(lk(0, ls), s_alg(sPhi, ls + 1, LN));
        const A8<R> cx = icomm(my_tx, ph);
        const A8<R> eox = s_alg(sEs, es, EN);
#pragma unroll
        for (int c = 0; c < 8; c++) {
            my_ex.v[c] = next_e(eox.v[c], A0.v[c] - Dn.v[c], cx.v[c], t, dt, inv_t);
            sum.v[c] = eox.v[c] + my_ex.v[c];
        }
        // only this thread reads site es of sEs before the barrier
        s_alg_put(sEs, es, EN, sum);
        const A8<R> Lf = conj_dn_t(lk(0, ls - 1), s_alg(sA, es - 1, EN));
        my_ty = conj_up_t(lk(1, ls), s_alg(sPhi, ls + LW, LN));
        const A8<R> cy = icomm(my_ty, ph);
        const A8<R> eoy = s_alg(sEs + AP * EN, es, EN);
#pragma unroll
        for (int c = 0; c < 8; c++) {
            my_ey.v[c] = next_e(eoy.v[c], Lf.v[c] - A0.v[c], cy.v[c], t, dt, inv_t);
            sum.v[c] = eoy.v[c] + my_ey.v[c];
            my_b.v[c] = A0.v[c] + Lf.v[c] + Dn.v[c];
        }
        s_alg_put(sEs + AP * EN, es, EN, sum);
        s_alg_put(sLf, es, EN, Lf);
    }
    constexpr int CH = (NH + 31) / 32;
    for (int u = tid >> 5; u < 2 * CH; u += NT / 32) {
        const int j = (u % CH) * 32 + (tid & 31);
        if (j >= NH) continue;
        const bool row = j < TX;  // bottom row, else left column
        const int l = row ? j + 1 : (j - TX + 1) * LW, e = row ? j + 1 : (j - TX + 1) * EW;
        if (u < CH) {
            const A8<R> b = conj_dn_t(row ? lk(0, l - 1) : lk(1, l - LW), s_alg(sA, row ? e - 1 : e - EW, EN));
            if (row) s_alg_put(sLf, e, EN, b);
            else s_alg_put(sHalo + AP * NH, j - TX, TY, b);
        } else {
            const A8<R> f = conj_up_t(lk(row ? 1 : 0, l), s_alg(sPhi, row ? l + LW : l + 1, LN));
            s_alg_put(sHalo, j, NH, icomm(f, s_alg(sPhi, l, LN)));
        }
    }
    __syncthreads();
    // by the warps that had no item
    for (int j = NT - 1 - tid; j < NH; j += NT) {
        const bool row = j < TX;
        const int e = row ? j + 1 : (j - TX + 1) * EW;
        const A8<R> A0 = s_alg(sA, e, EN), b = row ? s_alg(sLf, e, EN) : s_alg(sHalo + AP * NH, j - TX, TY);
        const A8<R> cur = s_alg(sHalo, j, NH);
        Vec* es_h = sEs + (row ? AP * EN : 0);
        const A8<R> eo = s_alg(es_h, e, EN);
        A8<R> sum;
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const R F = row ? b.v[c] - A0.v[c] : A0.v[c] - b.v[c];
            sum.v[c] = eo.v[c] + next_e(eo.v[c], F, cur.v[c], t, dt, inv_t);
        }
        s_alg_put(es_h, e, EN, sum);
    }
    __syncthreads();

    // ---- phase 4: the tile sites
    // sites of a ragged tile beyond the lattice do nothing (no early return:
    // persistent callers reach further barriers)
    if (valid) {
        const A8<R> p_old = load_alg(in.pi, g, Vn);
        const A8<R> ph = s_alg(sPhi, ls, LN);
        const M3<R> Ux_m = lk(0, ls - 1);
        const M3<R> Uy_m = lk(1, ls - LW);
        const A8<R> bx = conj_dn_t(Ux_m, s_alg(sPhi, ls - 1, LN));
        const A8<R> by = conj_dn_t(Uy_m, s_alg(sPhi, ls - LW, LN));
        A8<R> p_new, ph_new;
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const R lap = my_tx.v[c] + my_ty.v[c] + bx.v[c] + by.v[c] - R(4) * ph.v[c];
            p_new.v[c] = fma(mul_rn(dt, inv_t), lap, p_old.v[c]);
            ph_new.v[c] = fma(a.dt_th, p_new.v[c], ph.v[c]);
        }
        // the site fields of t_n, written by every field step (one code path for
        // every caller, so the fields evolve bitwise alike whether or not the
        // site fields are used)
        // E_i = (1/4t){e_i(s) + U_i(s-i)^+ e_i(s-i) U_i(s-i)}, e summed over n -+ 1/2
        const A8<R> sx = conj_dn_t(Ux_m, s_alg(sEs, es - 1, EN));
        const A8<R> sy = conj_dn_t(Uy_m, s_alg(sEs + AP * EN, es - EW, EN));
        const A8<R> hx = s_alg(sEs, es, EN), hy = s_alg(sEs + AP * EN, es, EN);
        const A8<R> cr = conj_dn_t(Uy_m, s_alg(sLf, es - EW, EN));
        A8<R> Ex, Ey, Ee, Bx, By, Be;
        const R q = R(0.25) * inv_t, hf = R(0.5) * inv_t;
#pragma unroll
        for (int c = 0; c < 8; c++) {
            Ex.v[c] = q * (hx.v[c] + sx.v[c]);
            Ey.v[c] = q * (hy.v[c] + sy.v[c]);
            Ee.v[c] = R(0.5) * (p_old.v[c] + p_new.v[c]);
            Bx.v[c] = -hf * (my_ty.v[c] - by.v[c]);
            By.v[c] = hf * (my_tx.v[c] - bx.v[c]);
            Be.v[c] = R(0.25) * (my_b.v[c] + cr.v[c]);
        }
        store_alg(site, g, Vn, Ex);
        store_alg(site + (size_t)1 * AP * Vn, g, Vn, Ey);
        store_alg(site + (size_t)2 * AP * Vn, g, Vn, Ee);
        store_alg(site + (size_t)3 * AP * Vn, g, Vn, Bx);
        store_alg(site + (size_t)4 * AP * Vn, g, Vn, By);
        store_alg(site + (size_t)5 * AP * Vn, g, Vn, Be);
        store_alg_cs(out.e, g, Vn, my_ex);
        store_alg_cs(out.e + (size_t)AP * Vn, g, Vn, my_ey);
        store_alg_cs(out.pi, g, Vn, p_new);
        store_alg_cs(out.phi, g, Vn, ph_new);
        M3<R> nx = mul(exp_i_alg<R>(my_ex, a.dt_over_th), lk(0, ls));
        store_link_cs(out.U, 0, g, Vn, nx);
        M3<R> ny = mul(exp_i_alg<R>(my_ey, a.dt_over_th), lk(1, ls));
        store_link_cs(out.U, 1, g, Vn, ny);
    }
}

// step scalars of t_n = n dt, computed the same way on the host and the device
__host__ __device__ inline StepArgs step_args(int N, int tiles_x, int64_t n, double dt, int reunit) {
    StepArgs a;
    a.N = N;
    a.tiles_x = tiles_x;
    const double t = n * dt, th = t + 0.5 * dt;
    a.t = t;
    a.dt = dt;
    a.inv_t = t > 0 ? 1.0 / t : 0.0;
    a.dt_over_th = dt / th;
    a.dt_th = dt * th;
    a.reunit = reunit;
    return a;
}

}  // namespace gl
