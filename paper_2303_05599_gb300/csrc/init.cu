// McLerran-Venugopalan initial conditions on the GPU (Sec. 2.1 of
// arXiv:2303.05599):
//   rho^a_n(x) ~ N(0, (g^2 mu a)^2 / Ns) per sheet n, colour a, site x
//   alpha_n = rho_n / (k^2 + m^2) in Fourier space (lattice k^2, zero mode
//             removed, modes with k > Lambda removed)
//   V^+(x) = prod_n exp(-i alpha_n(x)), sheet 1 leftmost
//   U^{A,B}_i(x) = V(x) V^+(x+i)
//   Glasma link U_i: tr T^a [(U^A + U^B)(1 + U^+) - h.c.] = 0, Newton iteration
//   E_eta(0) = -i [alpha_A^i, alpha_B^i] from the link algebra elements -i[U]_ah,
//              forward and backward links averaged (the backward one
//              transported with the Glasma link)
// The paper states only that the continuum conditions are discretised; the
// matching condition is the standard one of the boost-invariant Glasma
// literature it builds on.
#include <math.h>
#include <string.h>

#include "ff.cuh"
#include "internal.h"
#include "layout.cuh"
#include "philox.cuh"

namespace gl {

// Work per nucleus and sheet: four complex planes, each two real colour planes
// of rho (the Green function is real and even, so the two parts of a plane
// stay apart through both transforms), and three launches over all events:
//   rows      rho of a few lattice rows into shared memory, their forward
//             transforms, out to the sheet's slot
//   columns   a tile of columns in: forward transform, Green function, inverse
//             transform, out
//   sheets    rows in: inverse transform, then per site exp(-i alpha) and the
//             product with the Wilson line
// The transforms work in place: the forward ones (decimation in frequency)
// leave each line in digit-reversed order, the Green table is stored in that
// order, and the inverse ones (decimation in time) start from it, so nothing
// is permuted.  Powers of two take radix 4 (and one radix 2), other sizes one
// direct pass per prime factor; the twiddles come from one table per event.
//
// What bounds it: FP64 arithmetic (GB300 issues one FP64 warp instruction per
// 19 cycles of an SM), so the passes are arranged to do less of it: radix-2
// transforms of eight complex planes with a sincospi per butterfly, a
// 20-term exponential series and whole matrices took 105.7 ms for a 256^2
// event of 50 sheets, 223 us a transform pass; these kernels in FP64 16.3 ms.
// An FP32 event's fields keep 24 bits of the result, so its sheets (variates,
// transforms, exponentials, products) run on pairs of FP32 values (ff.cuh,
// about 48 bits) and only the links' matching in FP64.  FP64 events have
// kernels of their own, in one fixed order of roundings (init64.cuh).
//
// A sheet's planes wait in a slot of the workspace, as many sheets a round as
// there are slots.  Small lattices split each nucleus's product over groups of
// consecutive sheets (a round takes some of every group), whose partial products
// are multiplied at the end: 1024 sites alone would leave most of the chip idle.
// Groups depend on N and Ns only, and rounds do not change the order of a
// product, so an event's fields are bitwise the same alone and in a batch.

static constexpr int INIT_T = 256;                  // threads of the line kernels
static constexpr int INIT_MAX_N = 3072;             // longest line
static constexpr int INIT_GEN_OUT = 12;             // outputs a thread of a prime pass: 256 x 12 = 3072 points
static_assert(sizeof(FFTables) % 16 == 0, "alignment of the tables behind it");

// Where the slots are.  The scratch holds the Wilson lines, the tables and as many
// slots as fit 576 B a site (nine FP64 matrices of both nuclei and their lines) or, on
// lattices below 86 sites a side, INIT_SMALL_ROOM.  The others lie in buffers of
// the event that are idle until its first step: the slice of the fields that is
// not current and the two site-field buffers, which are cleared afterwards.  An
// FP32 event of 256^2 has 14 slots, 7 sheets a round, and takes 4.46 ms (2 sheets
// a round: 4.75 ms).  The scratch is each event's own for good and serves the start
// alone, so it stays small: with 32 MB more an event, nine events of 64/128/256
// take 15.21 ms in 595 MB, with this 15.33 ms in 343 MB; a single small event,
// which needs many sheets a round to fill the chip, pays more: FP64 32^2 0.65 ms in
// 17 MB, here 0.72 ms in 7 MB and within 576 B a site 1.39 ms in 3 MB; FP32 64^2 0.37
// ms in 32 MB and 0.59 ms in 7 MB (0.47 ms in 11 MB, twice the room).
static constexpr size_t INIT_SMALL_ROOM = (size_t)4 << 20;

struct InitPlan {
    int groups, per_group, K;        // groups of sheets, sheets a group, sheets of each group a round
    int n0, n1;                      // slots up to n0 in the scratch, up to n1 in the fields, the rest in the site fields
    size_t unit, tw, work, green, total;  // bytes of a slot; byte offsets in the scratch (the lines are first)
};

static InitPlan init_plan(int prec, int N, int Ns) {
    const size_t V = (size_t)N * N;
    // per site: a slot, a group's lines of both nuclei, the slots that fit the idle buffers (FP64 544 and 768 B, FP32 224 and 384 B)
    const size_t unit = (prec == 0 ? 144 : 64) * V, lines = (prec == 0 ? 288 : 192) * V;
    const int in_fields = 3, in_site = prec == 0 ? 5 : 6;
    const size_t line_tw = ((size_t)N * 16 * (prec == 0 ? 2 : 1) + 255) & ~(size_t)255;
    const size_t tables = line_tw + (prec == 0 ? 0 : sizeof(FFTables));
    const size_t base = 576 * V, room = base > INIT_SMALL_ROOM ? base : INIT_SMALL_ROOM;
    auto slots = [&](int groups) {
        const size_t head = groups * lines + tables + 8 * V;
        return (int)((room > head ? (room - head) / unit : 0) + in_fields + in_site);
    };
    InitPlan p;
    int g = prec == 0 ? 1 : (int)(16384 / V);
    g = g < 1 ? 1 : g > Ns ? Ns : g;
    // at least two sheets a round of each group (64^2: 0.63 -> 0.59 ms, 48^2: 1.20 -> 0.96 ms)
    while (g > 1 && slots(g) < 4 * g) g--;
    p.per_group = (Ns + g - 1) / g;
    p.groups = (Ns + p.per_group - 1) / p.per_group;
    const int fit = slots(p.groups) / (2 * p.groups);
    p.K = fit < p.per_group ? fit : p.per_group;
    const int need = 2 * p.groups * p.K;
    p.n0 = need > in_fields + in_site ? need - in_fields - in_site : 0;
    p.n1 = p.n0 + (need - p.n0 < in_fields ? need - p.n0 : in_fields);
    p.unit = unit;
    p.tw = p.groups * lines;
    p.work = p.tw + tables;
    p.green = p.work + p.n0 * unit;
    p.total = p.green + 8 * V;
    return p;
}

size_t init_scratch_bytes(int prec, int N, int Ns) { return init_plan(prec, N, Ns).total; }

// blocks of the kernels of one event
static inline int rows_lines(int N) { return N >= 1024 ? 1 : 1024 / N; }          // lines a block of `rows`
static inline int cols_tile(int N, bool pow2) {                                    // columns a block of `columns`
    int c = pow2 ? (N > 1024 ? 2 : (N >= 256 ? 4 : 1024 / N)) : (N <= 256 ? 1024 / N : INIT_MAX_N / N);
    return c < 1 ? 1 : (c > N ? N : c);
}
static inline int sheet_rows(int N) { return N >= 256 ? 1 : 256 / N; }             // rows a block of `sheets`

// FP64: lines of each of two planes a block of `rows`, columns a block of `columns`
static inline int rows64(int N) { return N >= 512 ? 1 : 512 / N; }
static inline int cols64(int N) {
    const int c = N >= 2048 ? 1 : N >= 512 ? 2 : N >= 256 ? 4 : 1024 / N;
    return c > N ? N : c;
}

InitEv init_event(int prec, void* fields, void* scratch, void* idle_fields, void* idle_site, int N, int Ns, double g2mu_a, double m_a, double Lambda_a,
                  uint64_t seed, int* bad) {
    InitEv e;
    memset(&e, 0, sizeof e);
    const InitPlan p = init_plan(prec, N, Ns);
    const int64_t V = (int64_t)N * N;
    e.N = N;
    e.Ns = Ns;
    e.groups = p.groups;
    e.per_group = p.per_group;
    e.K = p.K;
    e.S = p.groups * p.K;
    e.pow2 = (N & (N - 1)) == 0;
    if (e.pow2) {
        int l = 0;
        while ((1 << l) < N) l++;
        e.log2N = l;
        for (; l >= 2; l -= 2) e.rad[e.nrad++] = 4;
        if (l) e.rad[e.nrad++] = 2;
    } else {
        int r = N;
        for (int q = 2; q * q <= r; q++)
            while (r % q == 0) { e.rad[e.nrad++] = q; r /= q; }
        if (r > 1) e.rad[e.nrad++] = r;
    }
    e.lines = prec == 0 ? rows64(N) : rows_lines(N);
    e.cols = prec == 0 ? cols64(N) : cols_tile(N, e.pow2);
    e.rows = sheet_rows(N);
    e.sigma = g2mu_a / sqrt((double)Ns);
    const ff sg = ff_of(e.sigma);
    e.sigma_h = sg.h;
    e.sigma_l = sg.l;
    e.m2 = m_a * m_a;
    e.lam2 = Lambda_a > 0 ? Lambda_a * Lambda_a : 0.0;
    e.k0 = (uint32_t)seed;
    e.k1 = (uint32_t)(seed >> 32);
    char* s = (char*)scratch;
    e.V = (double2*)s;
    e.normal = (FFTables*)(s + p.tw);
    e.tw = (double2*)(s + p.tw + (prec == 0 ? 0 : sizeof(FFTables)));
    e.green = (double*)(s + p.green);
    e.work[0] = (double2*)(s + p.work);
    e.work[1] = (double2*)idle_fields;
    e.work[2] = (double2*)idle_site;
    e.end0 = p.n0 * p.unit / sizeof(double2);
    e.end1 = p.n1 * p.unit / sizeof(double2);
    // after the last sheet, in the site fields: FP32 192 B a site of links, 128 B of commutators
    e.U64 = e.work[2];
    e.comm = prec == 0 ? e.work[2] : e.U64 + (size_t)12 * V;
    e.fields = fields;
    e.prec = prec;
    e.bad = bad;
    return e;
}

// the block's event and its block index there, for launch `k` of the table
__device__ __forceinline__ const InitEv& init_find(const InitEv* evs, int ne, const InitEv& one, int k, int* blk) {
    int lo = 0, hi = ne - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (evs[mid].begin[k] <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const InitEv& d = evs ? evs[lo] : one;
    *blk = blockIdx.x - (evs ? d.begin[k] : 0);
    return d;
}
// element o of the slots, one after another
__device__ __forceinline__ double2* slot_at(const InitEv& d, size_t o) {
    return o < d.end0 ? d.work[0] + o : o < d.end1 ? d.work[1] + (o - d.end0) : d.work[2] + (o - d.end1);
}
// the sheet that slot j of a nucleus has in a round, -1 for none
__device__ __forceinline__ int slot_sheet(const InitEv& d, int j, int round) {
    const int g = j / d.K, l = round * d.K + j - g * d.K, sheet = g * d.per_group + l;
    return l < d.per_group && sheet < d.Ns ? sheet : -1;
}
enum { IK_TABLES = 0, IK_ROWS, IK_COLS, IK_SHEETS, IK_SITES, IK_LINKS, IK_PRODUCTS, IK_N };
static_assert(IK_N <= InitEv::KINDS, "block table");

// ------------------------------------------------------------ line transforms
// `lines` lines of N points in shared memory, `ls` points apart, transformed in
// place by the block (no barrier before, one after each pass).
struct __align__(16) ff2 {
    ff x, y;
};
__device__ __forceinline__ ff2 cxy(ff x, ff y) { return ff2{x, y}; }
__device__ __forceinline__ ff2 cmul(ff2 a, ff2 w) {
    return ff2{FDot(a.x, w.x).sub(a.y, w.y).get(), FDot(a.x, w.y).add(a.y, w.x).get()};
}
__device__ __forceinline__ ff2 cmulc(ff2 a, ff2 w) {  // a conj(w)
    return ff2{FDot(a.x, w.x).add(a.y, w.y).get(), FDot(a.y, w.x).sub(a.x, w.y).get()};
}
__device__ __forceinline__ ff2 ldg16(const ff2* p) {
    const float4 v = __ldg((const float4*)p);
    return ff2{ff{v.x, v.y}, ff{v.z, v.w}};
}
__device__ __forceinline__ ff2 cadd(ff2 a, ff2 b) { return cxy(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ ff2 csub(ff2 a, ff2 b) { return cxy(a.x - b.x, a.y - b.y); }

// powers of two: radix 4, and radix 2 on neighbours for odd log2 N
__device__ __forceinline__ void pow2_radix2(ff2* sh, int lines, int ls, int lN) {
    for (int b = threadIdx.x; b < lines << (lN - 1); b += blockDim.x) {
        ff2* p = sh + (b >> (lN - 1)) * ls + 2 * (b & ((1 << (lN - 1)) - 1));
        const ff2 u = p[0], v = p[1];
        p[0] = cadd(u, v);
        p[1] = csub(u, v);
    }
    __syncthreads();
}
__device__ __forceinline__ void pow2_forward(ff2* sh, int lines, int ls, int lN, const ff2* __restrict__ tw) {
    for (int lb = lN; lb >= 2; lb -= 2) {
        const int q = 1 << (lb - 2);
        for (int b = threadIdx.x; b < lines << (lN - 2); b += blockDim.x) {
            const int j = b & ((1 << (lN - 2)) - 1), n = j & (q - 1);
            ff2* p = sh + (b >> (lN - 2)) * ls + ((j >> (lb - 2)) << lb) + n;
            const ff2 a0 = p[0], a1 = p[q], a2 = p[2 * q], a3 = p[3 * q];
            const ff2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = csub(a1, a3);
            p[0] = cadd(t0, t2);
            // t1 -+ i t3
            const ff2 y1 = cxy(t1.x + t3.y, t1.y - t3.x), y2 = csub(t0, t2),
                          y3 = cxy(t1.x - t3.y, t1.y + t3.x);
            if (lb > 2) {
                const int w = n << (lN - lb);
                p[q] = cmulc(y1, ldg16(tw + w));
                p[2 * q] = cmulc(y2, ldg16(tw + 2 * w));
                p[3 * q] = cmulc(y3, ldg16(tw + 3 * w));
            } else {
                p[q] = y1;
                p[2 * q] = y2;
                p[3 * q] = y3;
            }
        }
        __syncthreads();
    }
    if (lN & 1) pow2_radix2(sh, lines, ls, lN);
}
__device__ __forceinline__ void pow2_inverse(ff2* sh, int lines, int ls, int lN, const ff2* __restrict__ tw) {
    if (lN & 1) pow2_radix2(sh, lines, ls, lN);
    for (int lb = 2 + (lN & 1); lb <= lN; lb += 2) {
        const int q = 1 << (lb - 2);
        for (int b = threadIdx.x; b < lines << (lN - 2); b += blockDim.x) {
            const int j = b & ((1 << (lN - 2)) - 1), n = j & (q - 1);
            ff2* p = sh + (b >> (lN - 2)) * ls + ((j >> (lb - 2)) << lb) + n;
            ff2 x1 = p[q], x2 = p[2 * q], x3 = p[3 * q];
            const ff2 x0 = p[0];
            if (lb > 2) {
                const int w = n << (lN - lb);
                x1 = cmul(x1, ldg16(tw + w));
                x2 = cmul(x2, ldg16(tw + 2 * w));
                x3 = cmul(x3, ldg16(tw + 3 * w));
            }
            const ff2 t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3), t3 = csub(x1, x3);
            p[0] = cadd(t0, t2);
            p[q] = cxy(t1.x - t3.y, t1.y + t3.x);
            p[2 * q] = csub(t0, t2);
            p[3 * q] = cxy(t1.x + t3.y, t1.y - t3.x);
        }
        __syncthreads();
    }
}

// any N: a direct transform of each prime factor in turn, one output point at
// a time (a block's points, at most 256 x INIT_GEN_OUT, wait in registers for
// the barrier before they replace the inputs)
template <bool FORWARD>
__device__ __noinline__ void prime_passes(ff2* sh, int lines, int ls, const InitEv& d) {
    const ff2* tw = (const ff2*)d.tw;
    const int N = d.N, total = lines * N;
    int B = N;
    if (!FORWARD)
        for (int s = 0; s + 1 < d.nrad; s++) B /= d.rad[s];
    for (int i = 0; i < d.nrad; i++) {
        const int s = FORWARD ? i : d.nrad - 1 - i;
        const int r = d.rad[s], m = B / r;
        const int wr = N / r, wB = N / B;
        ff2 out[INIT_GEN_OUT];
#pragma unroll
        for (int c = 0; c < INIT_GEN_OUT; c++) {
            const int idx = threadIdx.x + c * INIT_T;
            if (idx < total) {
                const int line = idx / N, p = idx - line * N, nb = p / B, k = (p - nb * B) / m, n = p % m;
                const ff2* x = sh + line * ls + nb * B + n;
                ff2 a = {};
                int w = 0;               // (q k mod r) N / r
                const int step = k * wr;
                int tn = 0;              // inverse: n q N / B
                for (int q = 0; q < r; q++) {
                    const ff2 v = x[q * m];
                    if (FORWARD) {
                        const ff2 t = cmulc(v, ldg16(tw + w));
                        a = cadd(a, t);
                    } else {
                        int u = w + tn;
                        if (u >= N) u -= N;
                        const ff2 t = cmul(v, ldg16(tw + u));
                        a = cadd(a, t);
                        tn += n * wB;
                        if (tn >= N) tn -= N;
                    }
                    w += step;
                    if (w >= N) w -= N;
                }
                if (FORWARD) a = cmulc(a, ldg16(tw + n * k * wB));
                out[c] = a;
            }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < INIT_GEN_OUT; c++) {
            const int idx = threadIdx.x + c * INIT_T;
            if (idx < total) {
                const int line = idx / N;
                sh[line * ls + idx - line * N] = out[c];
            }
        }
        __syncthreads();
        if (FORWARD) B = m;
        else B *= i + 1 < d.nrad ? d.rad[s - 1] : 1;
    }
}

__device__ __forceinline__ void lines_forward(ff2* sh, int lines, int ls, const InitEv& d) {
    if (d.pow2) pow2_forward(sh, lines, ls, d.log2N, (const ff2*)d.tw);
    else prime_passes<true>(sh, lines, ls, d);
}
__device__ __forceinline__ void lines_inverse(ff2* sh, int lines, int ls, const InitEv& d) {
    if (d.pow2) pow2_inverse(sh, lines, ls, d.log2N, (const ff2*)d.tw);
    else
        for (int l = 0; l < lines;) {  // at most INIT_T x INIT_GEN_OUT points at a time
            int c = INIT_T * INIT_GEN_OUT / d.N;
            if (c > lines - l) c = lines - l;
            prime_passes<false>(sh + (size_t)l * ls, c, ls, d);
            l += c;
        }
}

// ------------------------------------------------------------ kernels
// the frequency at position p of a transformed line
__device__ __forceinline__ int line_frequency(const InitEv& d, int p) {
    int B = d.N, f = 0, scale = 1;
    for (int s = 0; s < d.nrad; s++) {
        const int m = B / d.rad[s], k = p / m;
        p -= k * m;
        f += k * scale;
        scale *= d.rad[s];
        B = m;
    }
    return f;
}

// the event's twiddles and its Green function over the number of sites, in the
// order the transforms leave (FP64: the order of the frequencies, and the
// twiddles of either sign)
__global__ void __launch_bounds__(INIT_T) init_tables_kernel(const InitEv* evs, int ne, InitEv one) {
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_TABLES, &blk);
    const int N = d.N;
    const int64_t Vn = (int64_t)N * N, s = (int64_t)blk * INIT_T + threadIdx.x;
    if (s == 0) *d.bad = 0;
    if (s < N) {
        double sn, cs;
        sincospi(2.0 * (double)s / (double)N, &sn, &cs);
        if (d.prec == 0) {
            d.tw[s] = make_double2(cs, sn);
            sincospi(-2.0 * (double)s / (double)N, &sn, &cs);
            d.tw[N + s] = make_double2(cs, sn);
        } else {
            ((ff2*)d.tw)[s] = ff2{ff_of(cs), ff_of(sn)};
        }
    }
    if (d.prec != 0 && s < FF_ANGLES) ff_table_entry(d.normal, (int)s);
    if (s < Vn) {
        const int px = (int)(s % N), py = (int)(s / N);
        const int kx = d.prec == 0 ? px : line_frequency(d, px), ky = d.prec == 0 ? py : line_frequency(d, py);
        const double sx = sinpi((double)kx / N), sy = sinpi((double)ky / N);
        const double k2 = 4.0 * (sx * sx + sy * sy);
        double g = 1.0 / (k2 + d.m2);
        if (kx == 0 && ky == 0) g = 0.0;
        if (d.lam2 > 0 && k2 > d.lam2) g = 0.0;
        g *= 1.0 / (double)Vn;
        if (d.prec == 0) d.green[s] = g;
        else ((ff*)d.green)[s] = ff_of(g);
    }
}

// two independent normal variates of standard deviation sigma
__device__ __forceinline__ ff2 normal_pair(const InitEv& d, uint32_t w1, uint32_t w2) {
    ff z0, z1;
    ff_box_muller(w1, w2, d.normal, z0, z1);
    const ff sigma{d.sigma_h, d.sigma_l};
    return ff2{sigma * z0, sigma * z1};
}

// Blocks per SM of the line kernels: pairs are bound by latency and take as many
// registers as the compiler is given (2, 2 and 1 blocks of the three kernels
// without a cap, 5.4 ms a 256^2 event; 4, 4 and 2 take 4.7 ms in spite of a few
// spills, 3, 3 and 3 5.8 ms).

// rho of d.lines lattice rows of one or two planes and their forward transforms
__device__ __forceinline__ void init_rows(const InitEv& d, int blk, int round, ff2* sh) {
    const int N = d.N, S = d.S;
    const int64_t all = (int64_t)2 * S * 4 * N, line0 = (int64_t)blk * d.lines;
    const int nl = (int)(all - line0 < d.lines ? all - line0 : d.lines);
    // nothing to do beyond the last sheet (the other events of a batch may go on)
    const int slot0 = (int)(line0 / (4 * (int64_t)N)), slot1 = (int)((line0 + nl - 1) / (4 * (int64_t)N));
    if (slot1 - slot0 < 2 && slot_sheet(d, slot0 % S, round) < 0 && slot_sheet(d, slot1 % S, round) < 0) return;
    for (int idx = threadIdx.x; idx < nl * N; idx += INIT_T) {
        const int l = idx / N, x = idx - l * N;
        const int64_t line = line0 + l;
        const int row = (int)(line % N), plane = (int)(line / N) & 3, slot = (int)(line / (4 * (int64_t)N));
        const int nucleus = slot / S, sheet = slot_sheet(d, slot - nucleus * S, round);
        ff2 z = {};
        if (sheet >= 0) {
            const U4 w = philox4x32_10(U4{(uint32_t)(row * N + x), (uint32_t)((nucleus * d.Ns + sheet) * 2 + (plane >> 1)),
                                          1u, 0u}, d.k0, d.k1);
            z = normal_pair(d, (plane & 1) ? w.z : w.x, (plane & 1) ? w.w : w.y);
        }
        sh[idx] = z;
    }
    __syncthreads();
    lines_forward(sh, nl, N, d);
    // [slot][plane][row][position]
    for (int idx = threadIdx.x; idx < nl * N; idx += INIT_T) *(ff2*)slot_at(d, (size_t)line0 * N + idx) = sh[idx];
}
__global__ void __launch_bounds__(INIT_T, 4) init_rows_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    extern __shared__ __align__(16) unsigned char init_smem[];
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_ROWS, &blk);
    init_rows(d, blk, round, (ff2*)init_smem);
}

// alpha = rho / (k^2 + m^2) along the columns of one plane
__global__ void __launch_bounds__(INIT_T, 4) init_cols_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    extern __shared__ __align__(16) unsigned char init_smem[];
    ff2* sh = (ff2*)init_smem;
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_COLS, &blk);
    const int N = d.N, S = d.S, ls = N + 1;  // a point of padding: neighbouring columns in other banks
    const int nt = (N + d.cols - 1) / d.cols;
    const int c0 = (blk % nt) * d.cols, sp = blk / nt, slot = sp >> 2;
    if (slot_sheet(d, slot % S, round) < 0) return;
    const int nc = N - c0 < d.cols ? N - c0 : d.cols;
    ff2* w = (ff2*)slot_at(d, (size_t)sp * N * N) + c0;
    for (int idx = threadIdx.x; idx < nc * N; idx += INIT_T) {
        const int r = idx / nc, c = idx - r * nc;
        sh[c * ls + r] = w[(size_t)r * N + c];
    }
    __syncthreads();
    lines_forward(sh, nc, ls, d);
    const ff* g = (const ff*)d.green + c0;
    for (int idx = threadIdx.x; idx < nc * N; idx += INIT_T) {
        const int r = idx / nc, c = idx - r * nc;
        const ff f = g[(size_t)r * N + c];
        const ff2 v = sh[c * ls + r];
        sh[c * ls + r] = cxy(v.x * f, v.y * f);
    }
    __syncthreads();
    lines_inverse(sh, nc, ls, d);
    for (int idx = threadIdx.x; idx < nc * N; idx += INIT_T) {
        const int r = idx / nc, c = idx - r * nc;
        w[(size_t)r * N + c] = sh[c * ls + r];
    }
}

// an SU(3) matrix of the scratch: rows 0 and 1 in six planes, row 2 rebuilt
__device__ __forceinline__ M3<double> load_rows(const double2* V, int64_t s, int64_t Vn) {
    M3<double> m;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const double2 v = V[(size_t)k * Vn + s];
        m.re[k / 3][k % 3] = v.x;
        m.im[k / 3][k % 3] = v.y;
    }
    rebuild_row2(m);
    return m;
}
__device__ __forceinline__ void store_rows(double2* V, int64_t s, int64_t Vn, const M3<double>& m) {
#pragma unroll
    for (int k = 0; k < 6; k++) V[(size_t)k * Vn + s] = make_double2(m.re[k / 3][k % 3], m.im[k / 3][k % 3]);
}
__device__ __forceinline__ M3ff load_rows(const ff2* V, int64_t s, int64_t Vn) {  // row 2 is left alone
    M3ff m;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const ff2 v = V[(size_t)k * Vn + s];
        m.re[k / 3][k % 3] = v.x;
        m.im[k / 3][k % 3] = v.y;
    }
    return m;
}
__device__ __forceinline__ void store_rows(ff2* V, int64_t s, int64_t Vn, const M3ff& m) {
#pragma unroll
    for (int k = 0; k < 6; k++) V[(size_t)k * Vn + s] = ff2{m.re[k / 3][k % 3], m.im[k / 3][k % 3]};
}
// a line kept as pairs, in FP64
__device__ __forceinline__ M3<double> load_line(const double2* V, int64_t s, int64_t Vn) {
    const M3ff f = load_rows((const ff2*)V, s, Vn);
    M3<double> m;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        m.re[k / 3][k % 3] = to_double(f.re[k / 3][k % 3]);
        m.im[k / 3][k % 3] = to_double(f.im[k / 3][k % 3]);
    }
    rebuild_row2(m);
    return m;
}
// rows 0 and 1 of v m
__device__ __forceinline__ M3<double> mul_rows(const M3<double>& v, const M3<double>& m) {
    M3<double> c = m_zero<double>();
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 3; j++)
#pragma unroll
            for (int k = 0; k < 3; k++) {
                c.re[i][j] = fma(v.re[i][k], m.re[k][j], c.re[i][j]);
                c.re[i][j] = fma(-v.im[i][k], m.im[k][j], c.re[i][j]);
                c.im[i][j] = fma(v.re[i][k], m.im[k][j], c.im[i][j]);
                c.im[i][j] = fma(v.im[i][k], m.re[k][j], c.im[i][j]);
            }
    return c;
}

// the inverse transforms of d.rows rows of a nucleus and the product over its
// sheets of this round (of one group of them)
__global__ void __launch_bounds__(INIT_T, 2) init_sheets_kernel(const InitEv* evs, int ne, InitEv one, int round) {
    extern __shared__ __align__(16) unsigned char init_smem[];
    ff2* sh = (ff2*)init_smem;
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_SHEETS, &blk);
    const int N = d.N, S = d.S;
    const int64_t Vn = (int64_t)N * N;
    const int nrb = (N + d.rows - 1) / d.rows;
    const int r0 = (blk % nrb) * d.rows, g = (blk / nrb) % d.groups, nucleus = blk / (nrb * d.groups);
    const int nr = N - r0 < d.rows ? N - r0 : d.rows, np = nr * N;
    const int first = g * d.per_group;
    const int s0 = first + round * d.K;
    int s1 = s0 + d.K < first + d.per_group ? s0 + d.K : first + d.per_group;
    if (s1 > d.Ns) s1 = d.Ns;
    ff2* V = (ff2*)d.V + (size_t)(nucleus * d.groups + g) * 6 * Vn + (int64_t)r0 * N;
    for (int s = s0; s < s1; s++) {
        const ff2* w = (const ff2*)slot_at(d, (size_t)(nucleus * S + g * d.K + s - s0) * 4 * Vn) + (int64_t)r0 * N;
        for (int idx = threadIdx.x; idx < 4 * np; idx += INIT_T) {
            const int p = idx / np;
            sh[idx] = w[(size_t)p * Vn + idx - p * np];
        }
        __syncthreads();
        lines_inverse(sh, 4 * nr, N, d);
        for (int i = threadIdx.x; i < np; i += INIT_T) {
            A8<ff> al;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                const ff2 v = sh[p * np + i];
                al.v[2 * p] = -v.x;
                al.v[2 * p + 1] = -v.y;
            }
            const M3ff e = ff_exp_i(al.v);
            // only this thread reads and writes the site's line, sheet after sheet
            if (s == first) store_rows(V, i, Vn, e);
            else store_rows(V, i, Vn, ff_mul<2>(load_rows(V, i, Vn), e));
        }
        __syncthreads();
    }
}

// the groups' partial products, in order, into the first
__global__ void __launch_bounds__(128) init_groups_kernel(const InitEv* evs, int ne, InitEv one) {
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_SITES, &blk);
    const int64_t Vn = (int64_t)d.N * d.N, t = (int64_t)blk * 128 + threadIdx.x;
    if (d.groups < 2 || t >= 2 * Vn) return;
    const int64_t s = t % Vn;
    ff2* V = (ff2*)d.V + (size_t)(t / Vn) * d.groups * 6 * Vn;
    M3ff v = load_rows(V, s, Vn);
    for (int g = 1; g < d.groups; g++) {
        M3ff m = load_rows(V + (size_t)g * 6 * Vn, s, Vn);
        // row 2: the conjugate cross product of rows 0 and 1
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int p = (j + 1) % 3, q = (j + 2) % 3;
            m.re[2][j] = FDot(m.re[0][p], m.re[1][q]).sub(m.im[0][p], m.im[1][q]).sub(m.re[0][q], m.re[1][p])
                             .add(m.im[0][q], m.im[1][p]).get();
            m.im[2][j] = -FDot(m.re[0][p], m.im[1][q]).add(m.im[0][p], m.re[1][q]).sub(m.re[0][q], m.im[1][p])
                             .sub(m.im[0][q], m.re[1][p]).get();
        }
        v = ff_mul<2>(v, m);
    }
    store_rows(V, s, Vn, v);
}

// Im tr(T^a M)
template <typename R>
__device__ __forceinline__ void im_tr_T(const M3<R>& M, R* f) {
    const R h = R(0.5), s3 = R(0.5) * inv_sqrt3<R>();
    f[0] = h * (M.im[1][0] + M.im[0][1]);
    f[1] = h * (M.re[0][1] - M.re[1][0]);
    f[2] = h * (M.im[0][0] - M.im[1][1]);
    f[3] = h * (M.im[2][0] + M.im[0][2]);
    f[4] = h * (M.re[0][2] - M.re[2][0]);
    f[5] = h * (M.im[2][1] + M.im[1][2]);
    f[6] = h * (M.re[1][2] - M.re[2][1]);
    f[7] = s3 * (M.im[0][0] + M.im[1][1] - R(2) * M.im[2][2]);
}
// Re tr(T^a M)
template <typename R>
__device__ __forceinline__ void re_tr_T(const M3<R>& M, R* f) {
    const R h = R(0.5), s3 = R(0.5) * inv_sqrt3<R>();
    f[0] = h * (M.re[1][0] + M.re[0][1]);
    f[1] = h * (M.im[1][0] - M.im[0][1]);
    f[2] = h * (M.re[0][0] - M.re[1][1]);
    f[3] = h * (M.re[2][0] + M.re[0][2]);
    f[4] = h * (M.im[2][0] - M.im[0][2]);
    f[5] = h * (M.re[2][1] + M.re[1][2]);
    f[6] = h * (M.im[2][1] - M.im[1][2]);
    f[7] = s3 * (M.re[0][0] + M.re[1][1] - R(2) * M.re[2][2]);
}

}  // namespace gl

#include "init64.cuh"

namespace gl {

// Jacobian of F^a = Im tr T^a (W + K), K = W U^+, under U -> exp(i x.T) U:
// J_ab = -Re tr(T^a K T^b).  With T^b T^a = delta/6 + (d + i f)_bac T^c / 2,
// J_ab = -(delta_ab Re tr K / 6 + d_abc r^c / 2 + f_abc i^c / 2) for tr(T^c K)
// = r^c + i i^c: the sixteen independent d and nine f, instead of eight
// matrix products.
template <typename R>
__device__ __forceinline__ void match_jacobian(const M3<R>& K, R J[8][8]) {
    R r[8], q[8];
    re_tr_T(K, r);
    im_tr_T(K, q);
    const R t = -(K.re[0][0] + K.re[1][1] + K.re[2][2]) * R(1.0 / 6.0);
    const R h = R(0.25), s3 = R(0.5) * inv_sqrt3<R>();  // d / 2 for d = 1/2, 1/sqrt 3
    const R fh = R(0.25), fs = R(0.43301270189221932338);    // f / 2 for f = 1/2, sqrt(3)/2
#pragma unroll
    for (int a = 0; a < 8; a++)
#pragma unroll
        for (int b = 0; b < 8; b++) J[a][b] = R(0);
    // diagonal: delta term and d_aac r^c
    const R e8 = s3 * r[7], h8 = R(0.5) * e8, h3 = h * r[2];
    J[0][0] = J[1][1] = J[2][2] = t - e8;
    J[3][3] = J[4][4] = t - h3 + h8;
    J[5][5] = J[6][6] = t + h3 + h8;
    J[7][7] = t + e8;
#define GL_D(a, b, v) J[a][b] -= (v), J[b][a] -= (v)
    GL_D(0, 7, s3 * r[0]); GL_D(1, 7, s3 * r[1]); GL_D(2, 7, s3 * r[2]);         // d118 d228 d338
    GL_D(0, 3, h * r[5]); GL_D(0, 5, h * r[3]); GL_D(3, 5, h * r[0]);            // d146
    GL_D(0, 4, h * r[6]); GL_D(0, 6, h * r[4]); GL_D(4, 6, h * r[0]);            // d157
    GL_D(1, 3, -h * r[6]); GL_D(1, 6, -h * r[3]); GL_D(3, 6, -h * r[1]);         // d247
    GL_D(1, 4, h * r[5]); GL_D(1, 5, h * r[4]); GL_D(4, 5, h * r[1]);            // d256
    GL_D(2, 3, h * r[3]); GL_D(2, 4, h * r[4]);                                  // d344 d355
    GL_D(2, 5, -h * r[5]); GL_D(2, 6, -h * r[6]);                                // d366 d377
    const R m8 = R(0.5) * s3;
    GL_D(3, 7, -m8 * r[3]); GL_D(4, 7, -m8 * r[4]); GL_D(5, 7, -m8 * r[5]); GL_D(6, 7, -m8 * r[6]);  // d448..d778
#undef GL_D
#define GL_F(a, b, c, v)                             \
    {                                                \
        const R va = (v) * q[a], vb = (v) * q[b], vc = (v) * q[c]; \
        J[a][b] -= vc; J[b][a] += vc;                \
        J[b][c] -= va; J[c][b] += va;                \
        J[c][a] -= vb; J[a][c] += vb;                \
    }
    GL_F(0, 1, 2, R(0.5));
    GL_F(0, 3, 6, fh); GL_F(0, 4, 5, -fh); GL_F(1, 3, 5, fh); GL_F(1, 4, 6, fh); GL_F(2, 3, 4, fh);
    GL_F(2, 5, 6, -fh);
    GL_F(3, 4, 7, fs); GL_F(5, 6, 7, fs);
#undef GL_F
}

// The Newton step dx = -J^-1 F at K, false where it is not to be trusted.  Its
// direction needs no more than FP32 as long as the full step contracts: an
// error of 1e-6 in it leaves 1e-6 of the residual, where the iteration's own
// square would leave less only in its last step, so the Jacobian and its
// elimination (half of the operations of an iteration) run on the FP32 pipe
// and the residual, the step's exponential and the link in FP64.  J is close
// to -1 for links near the unit matrix, so the elimination runs in its own
// order, in registers; not where a pivot falls below 1/16 of the diagonal's scale.
__device__ __forceinline__ bool match_step(const M3<double>& K, const double* F, double* x) {
    float J[8][8], y[8], inv[8];
    M3<float> Kf;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { Kf.re[i][j] = (float)K.re[i][j]; Kf.im[i][j] = (float)K.im[i][j]; }
    match_jacobian(Kf, J);
#pragma unroll
    for (int a = 0; a < 8; a++) y[a] = -(float)F[a];
    bool small = false;
#pragma unroll
    for (int c = 0; c < 8; c++) {
        small = small || !(fabsf(J[c][c]) > 0.0625f);
        inv[c] = 1.0f / J[c][c];
#pragma unroll
        for (int r = c + 1; r < 8; r++) {
            const float f = J[r][c] * inv[c];
#pragma unroll
            for (int k = c + 1; k < 8; k++) J[r][k] = fmaf(-f, J[c][k], J[r][k]);
            y[r] = fmaf(-f, y[c], y[r]);
        }
    }
#pragma unroll
    for (int c = 7; c >= 0; c--) {
#pragma unroll
        for (int k = c + 1; k < 8; k++) y[c] = fmaf(-J[c][k], y[k], y[c]);
        y[c] *= inv[c];
        x[c] = (double)y[c];
    }
    return !small;
}

// F^a = Im tr T^a (W + K), K = W U^+, and its largest entry
__device__ __forceinline__ double match_residual(const M3<double>& K, const double* fw, double* F) {
    im_tr_T(K, F);
    double r = 0;
#pragma unroll
    for (int a = 0; a < 8; a++) {
        F[a] += fw[a];
        r = fmax(r, fabs(F[a]));
    }
    return r;
}

// the plain FP64 method of init64.cuh, which few links of few events need
__device__ __noinline__ int solve_link_plain(const M3<double>& UA, const M3<double>& UB, M3<double>& U) {
    return solve_link64(UA, UB, U);
}

// Newton solve for the Glasma link from the pure-gauge links of both nuclei, by
// full steps of FP32 directions while each leaves at most a quarter of the
// residual.  Iterations that do not contract (strong fields on coarse lattices,
// g^2 mu a of order 1) wander before they converge, or do not: there an error of
// 1e-6 in a direction ends at another solution of the matching condition, or
// at none, so such a link starts again with the plain method.
__device__ int solve_link(const M3<double>& UA, const M3<double>& UB, M3<double>& U) {
    const M3<double> W = add(UA, UB);
    double fw[8], F[8];
    im_tr_T(W, fw);
    U = mul(UA, UB);
    M3<double> K = mul_nd(W, U);
    double r = match_residual(K, fw, F);
    // a finite residual: quartered by every pass, so at most 522 passes follow
    bool contracts = r <= 1e300;
    while (contracts && r > 1e-14) {
        A8<double> dx;
        contracts = match_step(K, F, dx.v);
        if (!contracts) break;
        U = mul_rows(exp_i_alg<double>(dx, 1.0), U);
        rebuild_row2(U);
        K = mul_nd(W, U);
        const double rn = match_residual(K, fw, F);
        contracts = rn <= 0.25 * r;
        r = rn;
    }
    return contracts ? 0 : solve_link_plain(UA, UB, U);
}

// The Glasma link (d, s), as two rows, and i[-i[U^A]_ah, -i[U^B]_ah] of the
// link, which E_eta(0) of both its ends needs.
__global__ void __launch_bounds__(64) init_links_kernel(const InitEv* evs, int ne, InitEv one) {
    int blk;
    const InitEv& ev = init_find(evs, ne, one, IK_LINKS, &blk);
    const int N = ev.N;
    const int64_t Vn = (int64_t)N * N, l = (int64_t)blk * 64 + threadIdx.x;
    if (l >= 2 * Vn) return;
    const int d = (int)(l / Vn);
    const int64_t s = l % Vn;
    const int x = (int)(s % N), y = (int)(s / N);
    const int64_t sn = d == 0 ? (int64_t)y * N + (x + 1 == N ? 0 : x + 1) : (int64_t)(y + 1 == N ? 0 : y + 1) * N + x;
    const double2* VB = ev.V + (size_t)ev.groups * 6 * Vn;
    const M3<double> UA = mul_dn(load_line(ev.V, s, Vn), load_line(ev.V, sn, Vn));
    const M3<double> UB = mul_dn(load_line(VB, s, Vn), load_line(VB, sn, Vn));
    store_alg(ev.comm + (size_t)d * 4 * Vn, s, Vn, icomm(iah_to_alg(UA), iah_to_alg(UB)));
    M3<double> U;
    if (solve_link(UA, UB, U)) atomicAdd(ev.bad, 1);
    store_rows(ev.U64 + (size_t)d * 6 * Vn, s, Vn, U);
}

// the Glasma link: an FP64 event's is in its fields already, an FP32 event's in the scratch
__device__ __forceinline__ M3<double> matched_link(const InitEv&, const Fields<double>& f, int k, int64_t s, int64_t Vn) {
    return load_link(f.U, k, s, Vn);
}
__device__ __forceinline__ M3<double> matched_link(const InitEv& d, const Fields<float>&, int k, int64_t s, int64_t Vn) {
    return load_rows(d.U64 + (size_t)k * 6 * Vn, s, Vn);
}
__device__ __forceinline__ void put_link(const InitEv&, const Fields<double>&, int, int64_t, int64_t) {}
__device__ __forceinline__ void put_link(const InitEv& d, const Fields<float>& f, int k, int64_t s, int64_t Vn) {
    const M3<double> m = matched_link(d, f, k, s, Vn);
    M3<float> o;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) { o.re[i][j] = (float)m.re[i][j]; o.im[i][j] = (float)m.im[i][j]; }
    store_link(f.U, k, s, Vn, o);
}

// pi(-1/2) = E_eta(0) = -sum over the four links at the site of the link's
// commutator / 2 (the backward ones transported by the Glasma link), phi = e =
// 0, and the links
template <typename R>
__device__ __forceinline__ void initial_site(const InitEv& d, int64_t s) {
    const int N = d.N;
    const int64_t Vn = (int64_t)N * N;
    const Fields<R> f = carve_fields<R>(d.fields, Vn);
    const int x = (int)(s % N), y = (int)(s / N);
    A8<double> pi = a_zero<double>();
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int64_t sb = k == 0 ? (int64_t)y * N + (x == 0 ? N - 1 : x - 1) : (int64_t)(y == 0 ? N - 1 : y - 1) * N + x;
        const double2* cm = d.comm + (size_t)k * 4 * Vn;
        const A8<double> c = load_alg(cm, s, Vn);
        const A8<double> b = conj_dn_t(matched_link(d, f, k, sb, Vn), load_alg(cm, sb, Vn));
#pragma unroll
        for (int q = 0; q < 8; q++) pi.v[q] -= 0.5 * (c.v[q] + b.v[q]);
    }
    A8<R> pr;
#pragma unroll
    for (int a = 0; a < 8; a++) pr.v[a] = (R)pi.v[a];
    const A8<R> z = a_zero<R>();
    store_alg(f.pi, s, Vn, pr);
    store_alg(f.phi, s, Vn, z);
    store_alg(f.e, s, Vn, z);
    store_alg(f.e + (size_t)Prec<R>::AP * Vn, s, Vn, z);
#pragma unroll
    for (int k = 0; k < 2; k++) put_link(d, f, k, s, Vn);
}
__global__ void __launch_bounds__(128) init_fields_kernel(const InitEv* evs, int ne, InitEv one) {
    int blk;
    const InitEv& d = init_find(evs, ne, one, IK_SITES, &blk);
    const int64_t s = (int64_t)blk * 128 + threadIdx.x;
    if (s >= (int64_t)d.N * d.N) return;
    if (d.prec == 0) initial_site<double>(d, s);
    else initial_site<float>(d, s);
}

// the blocks of event e in launch k
static int64_t init_blocks(const InitEv& e, int k) {
    const int64_t V = (int64_t)e.N * e.N;
    if (e.prec == 0) switch (k) {
        case IK_ROWS: return (int64_t)8 * e.S * ((e.N + e.lines - 1) / e.lines);
        case IK_COLS: return (int64_t)16 * e.S * ((e.N + e.cols - 1) / e.cols);
        case IK_SHEETS: return (2 * e.S * V + 127) / 128;
        case IK_PRODUCTS: return 2 * ((V + 31) / 32);
        default: break;
    }
    switch (k) {
        case IK_TABLES: return ((V > FF_ANGLES ? V : FF_ANGLES) + INIT_T - 1) / INIT_T;
        case IK_ROWS: return ((int64_t)8 * e.S * e.N + e.lines - 1) / e.lines;
        case IK_COLS: return (int64_t)8 * e.S * ((e.N + e.cols - 1) / e.cols);
        case IK_SHEETS: return (int64_t)2 * e.groups * ((e.N + e.rows - 1) / e.rows);
        case IK_SITES: return (2 * V + 127) / 128;
        default: return (2 * V + 63) / 64;
    }
}

bool init_supported(int N) { return N <= INIT_MAX_N; }

void init_block_table(InitEv* evs, int ne) {
    for (int k = 0; k < IK_N; k++) {
        int64_t b = 0;
        for (int e = 0; e < ne; e++) {
            evs[e].begin[k] = (int)b;
            b += init_blocks(evs[e], k);
        }
    }
}

// The shared memory a launch may ask for is an attribute of the kernel on its
// device, which calls on other contexts and host threads set too: every call
// sets the most that any lattice needs (a row's four planes of the longest line).
static constexpr int INIT_MAX_SMEM = 4 * INIT_MAX_N * 16;
static_assert(INIT_MAX_SMEM <= 227 * 1024, "beyond a block's shared memory");
template <typename K>
static void line_smem(K* kernel, size_t bytes) {
    if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, INIT_MAX_SMEM);
}

void launch_mv_init(const InitEv* h, const InitEv* d_ev, int ne, cudaStream_t st) {
    const InitEv one = h[0];
    const InitEv* ev = ne > 1 ? d_ev : nullptr;
    const bool wide = one.prec == 0;  // the events of a launch have one precision
    unsigned nb[IK_N];
    size_t rows = 0, cols = 0, sheets = 0;
    int rounds = 1;
    bool grouped = false;
    for (int k = 0; k < IK_N; k++) nb[k] = (unsigned)(h[ne - 1].begin[k] + init_blocks(h[ne - 1], k));
    for (int e = 0; e < ne; e++) {
        const size_t r = (size_t)h[e].lines * h[e].N * (wide ? 32 : 16), c = (size_t)h[e].cols * (h[e].N + 1) * 16,
                     s = (size_t)4 * h[e].rows * h[e].N * 16;
        rows = r > rows ? r : rows;
        cols = c > cols ? c : cols;
        sheets = s > sheets ? s : sheets;
        const int n = (h[e].per_group + h[e].K - 1) / h[e].K;
        rounds = n > rounds ? n : rounds;
        grouped = grouped || h[e].groups > 1;
    }
    init_tables_kernel<<<nb[IK_TABLES], INIT_T, 0, st>>>(ev, ne, one);
    if (wide) {
        line_smem(init64_rows_kernel<true>, rows);
        line_smem(init64_rows_kernel<false>, rows);
        line_smem(init64_cols_kernel<true>, cols);
        line_smem(init64_cols_kernel<false>, cols);
        for (int r = 0; r < rounds; r++) {
            init64_rows_kernel<true><<<nb[IK_ROWS], 256, rows, st>>>(ev, ne, one, r);
            init64_cols_kernel<true><<<nb[IK_COLS], 256, cols, st>>>(ev, ne, one, r);
            init64_rows_kernel<false><<<nb[IK_ROWS], 256, rows, st>>>(ev, ne, one, r);
            init64_cols_kernel<false><<<nb[IK_COLS], 256, cols, st>>>(ev, ne, one, r);
            init64_exp_kernel<<<nb[IK_SHEETS], 128, 0, st>>>(ev, ne, one, r);
            init64_products_kernel<<<nb[IK_PRODUCTS], 96, 0, st>>>(ev, ne, one, r);
        }
        init64_links_kernel<<<nb[IK_LINKS], 64, 0, st>>>(ev, ne, one);
    } else {
        line_smem(init_rows_kernel, rows);
        line_smem(init_cols_kernel, cols);
        line_smem(init_sheets_kernel, sheets);
        for (int r = 0; r < rounds; r++) {
            init_rows_kernel<<<nb[IK_ROWS], INIT_T, rows, st>>>(ev, ne, one, r);
            init_cols_kernel<<<nb[IK_COLS], INIT_T, cols, st>>>(ev, ne, one, r);
            init_sheets_kernel<<<nb[IK_SHEETS], INIT_T, sheets, st>>>(ev, ne, one, r);
        }
        if (grouped) init_groups_kernel<<<nb[IK_SITES], 128, 0, st>>>(ev, ne, one);
        init_links_kernel<<<nb[IK_LINKS], 64, 0, st>>>(ev, ne, one);
    }
    init_fields_kernel<<<nb[IK_SITES], 128, 0, st>>>(ev, ne, one);
}

}  // namespace gl
