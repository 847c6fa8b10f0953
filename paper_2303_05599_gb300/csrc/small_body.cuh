// The FP64 field step of small lattices: 4x4-site tiles, one block of four warps
// each, with a site's work spread over the warps.
//
// Same quantities as fused_body.cuh.  What bounds a small FP64 lattice is the
// rate of one scheduler: an FP64 warp instruction takes 64 cycles of it however
// many lanes are active, and a thread of the large tile runs about 4,000 of them
// one after the other (127 us on a 32^2 lattice, 8 blocks on 152 SMs).  Here a
// thread runs about 650: the three rows of a plaquette product go to three
// warps, the transports and commutators of the two directions to four, the
// exponentials, the electric and magnetic fields and the scalar to four.  The
// arithmetic of a site is the same but for the halo (25 plaquettes and 40
// momenta for 16 sites), so lattices that fill the chip anyway keep the larger
// tiles.
// Measured: 32^2 127 -> 29 us, 64^2 127 -> 39 us, 128^2 129 -> 119 us.  Both kernels
// give the same bits (su3.cuh, mul_rn).
#pragma once
#include "fused_body.cuh"

namespace gl {

// The large tiles of an N x N lattice, and whether a launch of `tiles` of them in
// all takes the small tiles instead.  A large tile keeps an SM's FP64 pipe to
// itself, so the time goes in steps of one tile an SM, and the small tiles' with
// the sites: 140^2 (162 tiles) 146 us against 170, 152^2 (190) 163 against 170,
// 156^2 (200) 177 against 170; batches of 5 and 6 events of 64^2 (160 and 192
// tiles) 153 against 173 and 182 against 174 us.
constexpr int TILE64_X = 16, TILE64_Y = 8;
inline int64_t tiles64(int N) { return (int64_t)((N + TILE64_X - 1) / TILE64_X) * ((N + TILE64_Y - 1) / TILE64_Y); }
inline bool small64(int64_t tiles, int sms) { return 4 * tiles <= 5 * sms; }

struct SmallTile {
    static constexpr int T = 4, SITES = 16, LW = 6, LN = 36, EW = 5, EN = 25, ITEMS = 20, NT = 128;
    double2 U[18][LN];       // links of x, y in [-1, 4]
    double2 phi[4][LN];
    double2 e[2][4][EN];     // e(n-1/2) of x, y in [-1, 3]
    double2 P[9][EN];        // plaquette matrices
    double2 A[4][EN];        // i[P]_ah
    // items of direction d: the 16 own sites, then the left column (d = 0) or
    // the bottom row (d = 1)
    double2 back[2][4][ITEMS];  // Dn, Lf
    double2 com[2][4][ITEMS];   // i[t, phi], t the forward scalar
    double2 fwd[2][4][SITES];   // t of the own sites
    double2 bwd[2][4][SITES];   // the backward scalar
    double2 sum[2][4][ITEMS];   // e(n-1/2) + e(n+1/2)
    double2 en[2][4][SITES];    // e(n+1/2)
};

__device__ __forceinline__ void small_tile(const Fields<double>& in, const Fields<double>& out, double2* site,
                                           const StepR<double>& a, int tile) {
    using S_ = SmallTile;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S_& S = *(S_*)smem_raw;
    const int N = a.N;
    const int64_t Vn = (int64_t)N * N;
    const int x0 = (tile % a.tiles_x) * S_::T, y0 = (tile / a.tiles_x) * S_::T;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    for (int i = tid; i < 22 * S_::LN; i += S_::NT) {
        const int k = i / S_::LN, c = i - k * S_::LN;
        const int64_t g = (int64_t)wrapi(y0 + c / S_::LW - 1, N) * N + wrapi(x0 + c % S_::LW - 1, N);
        if (k < 18) cp_async16(&S.U[k][c], in.U + (size_t)k * Vn + g);
        else cp_async16(&S.phi[k - 18][c], in.phi + (size_t)(k - 18) * Vn + g);
    }
    for (int i = tid; i < 8 * S_::EN; i += S_::NT) {
        const int k = i / S_::EN, c = i - k * S_::EN;
        const int64_t g = (int64_t)wrapi(y0 + c / S_::EW - 1, N) * N + wrapi(x0 + c % S_::EW - 1, N);
        cp_async16(&S.e[k >> 2][k & 3][c], in.e + (size_t)k * Vn + g);
    }
    cp_async_wait_all();
    __syncthreads();
    auto link = [&](int d, int l) { return s_link(&S.U[0][0], d, l, S_::LN); };
    auto scalar = [&](int l) { return s_alg(&S.phi[0][0], l, S_::LN); };

    // plaquettes: row `warp` of Ux Uy(x+1) Ux(y+1)^+ Uy^+
    if (warp < 3 && lane < S_::EN) {
        const int l = (lane / S_::EW) * S_::LW + lane % S_::EW;
        double pr[3], pi[3], qr[3], qi[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const double2 v = S.U[warp * 3 + k][l];
            pr[k] = v.x;
            pi[k] = v.y;
        }
        row_mul(pr, pi, link(1, l + 1), qr, qi);
        row_mul_dag(qr, qi, link(0, l + S_::LW), pr, pi);
        row_mul_dag(pr, pi, link(1, l), qr, qi);
#pragma unroll
        for (int j = 0; j < 3; j++) S.P[warp * 3 + j][lane] = make_double2(qr[j], qi[j]);
    }
    __syncthreads();
    // their components, a pair of them a warp
    if (lane < S_::EN) {
        double2 v;
        if (warp == 0) {
            const double2 p = S.P[1][lane], q = S.P[3][lane];
            v = make_double2(-(p.y + q.y), q.x - p.x);
        } else if (warp == 1) {
            const double2 p = S.P[2][lane], q = S.P[6][lane];
            v = make_double2(S.P[4][lane].y - S.P[0][lane].y, -(p.y + q.y));
        } else if (warp == 2) {
            const double2 p = S.P[5][lane], q = S.P[7][lane];
            v = make_double2(S.P[6][lane].x - S.P[2][lane].x, -(p.y + q.y));
        } else {
            v = make_double2(S.P[7][lane].x - S.P[5][lane].x,
                             (2.0 * S.P[8][lane].y - S.P[0][lane].y - S.P[4][lane].y) * inv_sqrt3<double>());
        }
        S.A[warp][lane] = v;
    }
    __syncthreads();

    // item `lane` of direction d: its cell
    auto item_x = [&](int d, int i) { return i < S_::SITES ? i & 3 : (d == 0 ? -1 : i - S_::SITES); };
    auto item_y = [&](int d, int i) { return i < S_::SITES ? i >> 2 : (d == 0 ? i - S_::SITES : -1); };
    const int dir = warp >> 1;
    const int step_l = dir == 0 ? 1 : S_::LW;
    if (lane < S_::ITEMS) {
        const int ix = item_x(dir, lane), iy = item_y(dir, lane);
        const int l = (iy + 1) * S_::LW + ix + 1, e = (iy + 1) * S_::EW + ix + 1;
        if ((warp & 1) == 0) {
            // Dn = Uy(y-1)^+ A(y-1) Uy(y-1) for e_x; Lf by Ux(x-1) for e_y
            const int bl = dir == 0 ? l - S_::LW : l - 1, be = dir == 0 ? e - S_::EW : e - 1;
            s_alg_put(&S.back[dir][0][0], lane, S_::ITEMS, conj_dn_t(link(1 - dir, bl), s_alg(&S.A[0][0], be, S_::EN)));
        } else {
            const A8<double> t = conj_up_t(link(dir, l), scalar(l + step_l));
            s_alg_put(&S.com[dir][0][0], lane, S_::ITEMS, icomm(t, scalar(l)));
            if (lane < S_::SITES) s_alg_put(&S.fwd[dir][0][0], lane, S_::SITES, t);
        }
    }
    __syncthreads();

    // own site of this lane (lanes 0..15 for direction 0, 16..31 for direction 1)
    const int own = lane & 15, od = lane >> 4;
    const int ox = own & 3, oy = own >> 2;
    const int ol = (oy + 1) * S_::LW + ox + 1, oe = (oy + 1) * S_::EW + ox + 1;
    const int gx = x0 + ox, gy = y0 + oy;
    const bool valid = gx < N && gy < N;
    const int64_t g = (int64_t)gy * N + gx;
    const int bl = od == 0 ? ol - 1 : ol - S_::LW;                     // the site behind in direction od
    const int bi = od == 0 ? (ox == 0 ? S_::SITES + oy : own - 1) : (oy == 0 ? S_::SITES + ox : own - 4);
    const double t = a.t, dt = a.dt, inv_t = a.inv_t;
    const double q = 0.25 * inv_t, hf = 0.5 * inv_t;
    if (warp < 2) {
        if (lane < S_::ITEMS) {
            const int d = warp;
            const int e = (item_y(d, lane) + 1) * S_::EW + item_x(d, lane) + 1;
            const A8<double> A0 = s_alg(&S.A[0][0], e, S_::EN), B = s_alg(&S.back[d][0][0], lane, S_::ITEMS);
            const A8<double> c = s_alg(&S.com[d][0][0], lane, S_::ITEMS), eo = s_alg(&S.e[d][0][0], e, S_::EN);
            A8<double> n, m;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const double F = d == 0 ? A0.v[k] - B.v[k] : B.v[k] - A0.v[k];
                n.v[k] = next_e(eo.v[k], F, c.v[k], t, dt, inv_t);
                m.v[k] = eo.v[k] + n.v[k];
            }
            s_alg_put(&S.sum[d][0][0], lane, S_::ITEMS, m);
            if (lane < S_::SITES) s_alg_put(&S.en[d][0][0], lane, S_::SITES, n);
        }
    } else if (warp == 2) {
        s_alg_put(&S.bwd[od][0][0], own, S_::SITES, conj_dn_t(link(od, bl), scalar(bl)));
    } else if (lane < S_::SITES) {
        // the fourth clover leaf and B_eta
        const int lo = oy == 0 ? S_::SITES + ox : own - 4;
        const A8<double> cr = conj_dn_t(link(1, ol - S_::LW), s_alg(&S.back[1][0][0], lo, S_::ITEMS));
        const A8<double> A0 = s_alg(&S.A[0][0], oe, S_::EN);
        const A8<double> Dn = s_alg(&S.back[0][0][0], own, S_::ITEMS), Lf = s_alg(&S.back[1][0][0], own, S_::ITEMS);
        A8<double> Be;
#pragma unroll
        for (int k = 0; k < 8; k++) Be.v[k] = 0.25 * (A0.v[k] + Lf.v[k] + Dn.v[k] + cr.v[k]);
        if (valid) store_alg(site + (size_t)20 * Vn, g, Vn, Be);
    }
    __syncthreads();

    if (warp == 0) {
        // the links, a direction in each half of the warp
        const A8<double> en = s_alg(&S.en[od][0][0], own, S_::SITES);
        const M3<double> u = mul(exp_i_alg<double>(en, a.dt_over_th), link(od, ol));
        if (valid) store_link_cs(out.U, od, g, Vn, u);
    } else if (warp == 1) {
        const A8<double> b = conj_dn_t(link(od, bl), s_alg(&S.sum[od][0][0], bi, S_::ITEMS));
        const A8<double> h = s_alg(&S.sum[od][0][0], own, S_::ITEMS);
        A8<double> E;
#pragma unroll
        for (int k = 0; k < 8; k++) E.v[k] = q * (h.v[k] + b.v[k]);
        if (valid) store_alg(site + (size_t)(4 * od) * Vn, g, Vn, E);
    } else if (warp == 2) {
        // lanes 0..15: the scalar and its momentum; 16..31: B_x, B_y
        const A8<double> tx = s_alg(&S.fwd[0][0][0], own, S_::SITES), ty = s_alg(&S.fwd[1][0][0], own, S_::SITES);
        const A8<double> bx = s_alg(&S.bwd[0][0][0], own, S_::SITES), by = s_alg(&S.bwd[1][0][0], own, S_::SITES);
        if (valid && od == 0) {
            const A8<double> po = load_alg(in.pi, g, Vn), ph = scalar(ol);
            A8<double> pn, phn, Ee;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const double lap = tx.v[k] + ty.v[k] + bx.v[k] + by.v[k] - 4.0 * ph.v[k];
                pn.v[k] = fma(mul_rn(dt, inv_t), lap, po.v[k]);
                phn.v[k] = fma(a.dt_th, pn.v[k], ph.v[k]);
                Ee.v[k] = 0.5 * (po.v[k] + pn.v[k]);
            }
            store_alg(site + (size_t)8 * Vn, g, Vn, Ee);
            store_alg_cs(out.pi, g, Vn, pn);
            store_alg_cs(out.phi, g, Vn, phn);
        } else if (valid) {
            A8<double> Bx, By;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                Bx.v[k] = -hf * (ty.v[k] - by.v[k]);
                By.v[k] = hf * (tx.v[k] - bx.v[k]);
            }
            store_alg(site + (size_t)12 * Vn, g, Vn, Bx);
            store_alg(site + (size_t)16 * Vn, g, Vn, By);
        }
    } else if (valid) {
        store_alg_cs(out.e + (size_t)(4 * od) * Vn, g, Vn, s_alg(&S.en[od][0][0], own, S_::SITES));
    }
}

// tiles of an N x N lattice
__host__ __device__ inline int small_tiles_x(int N) { return (N + SmallTile::T - 1) / SmallTile::T; }

}  // namespace gl
