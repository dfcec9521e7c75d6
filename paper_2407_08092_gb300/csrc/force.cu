// Fermion force on the device: the gradient of the bilinear form
//   b(U) = Re( Y^+ D(U) X )
// with respect to every link, for full-lattice fields X and Y.  For the
// pseudofermion action S = phi^+ (D^+ D)^{-1} phi with X = (D^+ D)^{-1} phi and
// Y = D X, varying U gives dS = -2 Re(Y^+ dD X), so dS/dU = -2 grad b.  The
// paper has no force; the operator is the Wilson-clover D of Sec. 2.3.
//
// Convention: G = db/dRe U + i db/dIm U, so that db = Re sum conj(G) dU.
// For b = Re tr(U M) the gradient is M^+; for b = Re tr(U^+ M) it is M.
//
// Hopping term.  U_mu(x) enters row x as -1/2 s (1 - g_mu) U psi(x+mu) and row
// x+mu as -1/2 s (1 + g_mu) U^+ psi(x), s the fermion time-boundary sign:
//   G_hop(x, mu) = -1/2 s sum_spin [ Y(x) (P- X(x+mu))^+ + (P+ X(x)) Y(x+mu)^+ ]
// with colour outer products and P-+ = 1 -+ g_mu.
//
// Clover term.  C = (4 + m0) + c_sw (i/2) sum_{mu<nu} sigma_mu_nu F_mu_nu with
// F = (Q - Q^+)/8, so
//   Re(Y^+ C X) = const + sum_y sum_{mu<nu} Re tr( Q_mu_nu(y) Gam_mu_nu(y) ),
//   Gam = (i c_sw / 16)(Lam + Lam^+),  Lam_mu_nu = sum_{s,s'} sigma_mu_nu[s][s'] X_s' Y_s^+
// (colour matrices).  In the chiral basis sigma_jk = -eps_jkl diag(s_l, s_l)
// and sigma_j4 = diag(s_j, -s_j), so with, per chirality block (spins 0,1 and
// 2,3), u_1 = X_1 Y_0^+ + X_0 Y_1^+, u_2 = i (X_0 Y_1^+ - X_1 Y_0^+),
// u_3 = X_0 Y_0^+ - X_1 Y_1^+ (upper block u, lower block l):
//   Lam_xy = -(u_3 + l_3), Lam_xz = u_2 + l_2, Lam_yz = -(u_1 + l_1),
//   Lam_xt = u_1 - l_1,    Lam_yt = u_2 - l_2, Lam_zt = u_3 - l_3.
// The leaf sum over Q is a sum over plaquettes with one insertion per corner.
// For the plaquette of plane (m, n) at z, with links a = U_m(z), b = U_n(z+m),
// c = U_m(z+n), d = U_n(z) and corners z, z+m, z+m+n, z+n, it is
//   tr(Gam_z a b c^+ d^+) + tr(a Gam_{z+m} b c^+ d^+) + ...   (four corners).
// With the paths W = a b, W2 = d c, Z = b c^+, V = d^+ a and, per link of the
// plaquette, the insertions at its two ends E_u = Gam(start) u + u Gam(end)
// (Gam is anti-Hermitian, so E_u^+ = -(u^+ Gam(start) + Gam(end) u^+)), the four
// gradients of that sum are two products each:
//   G_a = W2 E_b^+ - E_d Z^+      G_b = E_a^+ W2 - V^+ E_c
//   G_c = V E_b - E_d^+ W         G_d = E_a Z - W E_c^+
// Per plaquette that is 4 products for the paths, 4 for E_m(z) and E_n(z) (E_b
// and E_c are those of the neighbouring plaquettes) and 8 for the gradients:
// 96 per site, where the 24 leaves of each link, formed one by one, take 288.
//
// Arithmetic is df64 (FP64-accurate on the FP32 units) throughout.
#include <type_traits>

#include "leaves.cuh"
#include "lq_kernels.h"

namespace lq {

// Resident blocks per SM asked of the two kernels.  The link kernel takes three (168
// registers, 74 KB of staged factors each): lq_force on 24^3 x 48 takes 4.93 ms (5.15
// with the matrices of each range made anew, 0.05 more at two blocks and 0.27 more with
// the factors read where they are used at four, 128 registers).  The plaquette kernel:
// four (some spills outside the products), 0.2 ms under three.
#ifndef LQ_FLINK_MINB
#define LQ_FLINK_MINB 3
#endif
#ifndef LQ_FLOOP_MINB
#define LQ_FLOOP_MINB 4
#endif

// gamma_mu psi: component s is i^k[mu][s] psi_perm[mu][s] (chiral basis)
__constant__ unsigned char c_gperm[4][4] = {{3, 2, 1, 0}, {3, 2, 1, 0}, {2, 3, 0, 1}, {2, 3, 0, 1}};
__constant__ unsigned char c_gipow[4][4] = {{3, 3, 1, 1}, {2, 0, 0, 2}, {3, 1, 1, 3}, {0, 0, 0, 0}};
// plane number of (mu, nu), mu < nu, in the numbering of leaves.cuh
__constant__ signed char c_plane[16] = {-1, 0, 1, 3, -1, -1, 2, 4, -1, -1, -1, 5, -1, -1, -1, -1};

__device__ __forceinline__ cx<df64> times_ipow(cx<df64> v, int k)
{
    switch (k & 3) {
    case 0: return v;
    case 1: return ti(v);
    case 2: return -v;
    default: return tmi(v);
    }
}

__device__ __forceinline__ cx<df64> ld_comp(const df2 *__restrict__ f, long long stride, int comp, long long cb)
{
    return df2_cx(ldg(f + (long long)comp * stride + cb));
}

// x or -x, as the sign bit `bit` says
__device__ __forceinline__ df64 flip_sign(df64 x, unsigned bit)
{
    return df64(__uint_as_float(__float_as_uint(x.hi) ^ bit), __uint_as_float(__float_as_uint(x.lo) ^ bit));
}

// Gam of the six planes at one site per thread, from X(x) and Y(x); k16 = c_sw / 16
__global__ void __launch_bounds__(128) force_insertion_kernel(Geom g, const df2 *__restrict__ Xe,
                                                              const df2 *__restrict__ Xo,
                                                              const df2 *__restrict__ Ye,
                                                              const df2 *__restrict__ Yo, df64 k16, float2 *Gam)
{
    const long long lex = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (lex >= g.V) return;
    int c[4];
    lex_coords(g, lex, c);
    const int parity = (c[0] + c[1] + c[2] + c[3]) & 1;
    const long long cb = lex >> 1;
    const df2 *X = parity ? Xo : Xe, *Y = parity ? Yo : Ye;
#pragma unroll 1
    for (int l = 1; l <= 3; l++) {
        // H_block = u_l + u_l^+ for the upper (blk 0) and lower (blk 1) chirality
        M3<df64> H[2];
#pragma unroll 1
        for (int blk = 0; blk < 2; blk++) {
            cx<df64> x0[3], x1[3], y0[3], y1[3];
#pragma unroll
            for (int a = 0; a < 3; a++) {
                x0[a] = ld_comp(X, g.stride, (2 * blk) * 3 + a, cb);
                x1[a] = ld_comp(X, g.stride, (2 * blk + 1) * 3 + a, cb);
                y0[a] = ld_comp(Y, g.stride, (2 * blk) * 3 + a, cb);
                y1[a] = ld_comp(Y, g.stride, (2 * blk + 1) * 3 + a, cb);
            }
            // entry (a, b) of X_s' Y_s^+ is X_s'[a] conj(Y_s[b]); u_1 and u_3 take
            // y0 with x1 resp. x0 and y1 with the other, u_2 = i (x0 y1^+ - x1 y0^+)
            const unsigned f0 = l == 2 ? 0x80000000u : 0u, f1 = l == 3 ? 0x80000000u : 0u;
            M3<df64> u;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const df64x2 p = dl2(l == 3 ? x0[a] : x1[a]), q = dl2(l == 3 ? x1[a] : x0[a]);
#pragma unroll
                for (int b = 0; b < 3; b++) {
                    dlrow t = dlrow_prod({flip_sign(y0[b].re, f0), flip_sign(y0[b].im, f0)}, p);
                    dlrow_fma(t, {flip_sign(y1[b].re, f1), flip_sign(y1[b].im, f1)}, q);
                    const cx<df64> v = dl2_cx(dl2_norm(dlrow_conj(t)));
                    u.a[a * 3 + b] = l == 2 ? ti(v) : v;
                }
            }
            H[blk] = u;
#pragma unroll
            for (int a = 0; a < 3; a++)
#pragma unroll
                for (int b = 0; b < 3; b++) H[blk].a[a * 3 + b] = u.a[a * 3 + b] + cconj(u.a[b * 3 + a]);
        }
        // the two planes built from l: (space plane, time plane) with the space
        // sign: l = 1 -> (yz, -; xt), l = 2 -> (xz, +; yt), l = 3 -> (xy, -; zt)
        const int ps = l == 1 ? 2 : l == 2 ? 1 : 0, pt = l == 1 ? 3 : l == 2 ? 4 : 5;
#pragma unroll 1
        for (int q = 0; q < 2; q++) {
            const int p = q == 0 ? ps : pt;
            const bool neg = q == 0 && l != 2;
            df64 v[9];
            auto h = [&](int a, int b) {
                cx<df64> t = q == 0 ? H[0].a[a * 3 + b] + H[1].a[a * 3 + b] : H[0].a[a * 3 + b] - H[1].a[a * 3 + b];
                return neg ? -t : t;
            };
            // Gam = i (c_sw/16) Hm: Im Gam_aa = (c_sw/16) Re Hm_aa; Gam_ab = i (c_sw/16) Hm_ab
#pragma unroll
            for (int a = 0; a < 3; a++) v[a] = k16 * h(a, a).re;
            const cx<df64> g01 = ti(h(0, 1)), g02 = ti(h(0, 2)), g12 = ti(h(1, 2));
            v[3] = k16 * g01.re;
            v[4] = k16 * g01.im;
            v[5] = k16 * g02.re;
            v[6] = k16 * g02.im;
            v[7] = k16 * g12.re;
            v[8] = k16 * g12.im;
            store_antiherm(Gam, g.V, lex, p, v);
        }
    }
}

// entry (i, k) of a 3x3 matrix stored component-major at m (distance `st` between
// components), or of its Hermitian conjugate
__device__ __forceinline__ M3<df64> load_mat(const df2 *__restrict__ m, long long st, bool dag)
{
    M3<df64> A;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const cx<df64> t = df2_cx(ldg(m + (dag ? k * 3 + i : i * 3 + k) * st));
            A.a[i * 3 + k] = dag ? cx<df64>{t.re, dl_neg(t.im)} : t;
        }
    return A;
}

// one row of a product added to a row of sums: s_j += sum_k r_k B_kj.  Each
// product and each sum is renormalised: twelve products summed with their low
// parts left to grow put the force 9.6e-15 from its 64-bit value, 6.2e-15 so
// (a twentieth of the time; renormalising a link's sums after every second product
// would save half of that, at 6.5e-15 and twice the largest error).
__device__ __forceinline__ void row_fma(cx<df64> s[3], const cx<df64> r[3], const M3<df64> &B)
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        dlrow t = dlrow_prod(r[0], dl2(B.a[j]));
        dlrow_fma(t, r[1], dl2(B.a[3 + j]));
        dlrow_fma(t, r[2], dl2(B.a[6 + j]));
        df64x2 u = dl2(s[j]);
        dl2_add(t.r, dlrow_rot(t));
        dl2_add(u, dl2_norm(t.r));
        s[j] = dl2_cx(dl2_norm(u));
    }
}

// entry (i, k) of the anti-Hermitian matrix of plane p at site lex
__device__ __forceinline__ cx<df64> antiherm_entry(const float2 *__restrict__ base, long long V, long long lex, int p,
                                                   int i, int k)
{
    auto ld = [&](int q) {
        const float2 t = __ldg(base + ((long long)p * 9 + q) * V + lex);
        return df64(t.x, t.y);
    };
    if (i == k) return {df64(0.0f, 0.0f), ld(i)};
    const int lo = i < k ? i : k, hi = i < k ? k : i, q = 3 + 2 * (lo + hi - 1);   // (0,1) (0,2) (1,2) at 3, 5, 7
    const df64 re = ld(q), im = ld(q + 1);
    return {i < k ? re : dl_neg(re), im};
}

// The plaquette matrices of some time slices, in a ring of `slots` slices:
// [plane][matrix][9][slot][site of the slice, x fastest] df2.  A slice's slot stands in
// the place of its time coordinate, with the extent `slots`; `head` is the slot of the
// first slice of a launch.
constexpr int F_W = 0, F_W2 = 1, F_Z = 2, F_V = 3, F_EM = 4, F_EN = 5, F_MATS = 6;
struct LoopMats {
    df2 *m;
    int head, slots;
    long long s3;    // sites of a slice
    long long n;     // sites of the ring
    __device__ __forceinline__ df2 *at(int p, int q, long long site) const
    {
        return m + ((long long)(p * F_MATS + q) * 9) * n + site;
    }
    // the slot of the launch's slice tl
    __device__ __forceinline__ int slot(int tl) const { return head + tl >= slots ? head + tl - slots : head + tl; }
    // the stored index of coordinates c, c[3] the slot
    __device__ __forceinline__ long long site(const Geom &g, const int c[4]) const
    {
        return LQ_IDX(c[3] * s3 + c[0] + (long long)g.L[0] * (c[1] + (long long)g.L[1] * c[2]), n, B_LEX);
    }
};

// coordinates c moved by +-1 along mu (mu uniform over a block); Lt, the extent of c[3]
__device__ __forceinline__ void step(const Geom &g, const int c[4], int mu, int s, int o[4], int Lt)
{
#pragma unroll
    for (int k = 0; k < 4; k++) {
        int v = c[k];
        if (k == mu) {
            v += s;
            const int L = k == 3 ? Lt : g.L[k];
            v = v < 0 ? v + L : (v >= L ? v - L : v);
        }
        o[k] = v;
    }
}

// One plaquette of plane p at z: its links a, b, c, d (0..3) and Gam at z, z+m, z+n
// (4..6), and the eight products that make its matrices, which share one copy of
// the product code, their operands picked by the step.
struct Plaquette {
    const df2 *Uz, *Un;
    const float2 *Gam;
    const Geom &g;
    long long lz, lm, ln;
    int p, m, n;
    __device__ __forceinline__ Plaquette(const Geom &geom, const df2 *Ue, const df2 *Uo, const float2 *gam, int plane,
                                         const int z[4])
        : Gam(gam), g(geom), p(plane), m(c_pmu[plane]), n(c_pnu[plane])
    {
        int zm[4], zn[4];
        step(g, z, m, +1, zm, g.L[3]);
        step(g, z, n, +1, zn, g.L[3]);
        lz = lex_of(g, z);
        lm = lex_of(g, zm);
        ln = lex_of(g, zn);
        const bool odd = (z[0] + z[1] + z[2] + z[3]) & 1;
        Uz = (odd ? Uo : Ue) + (lz >> 1);
        Un = odd ? Ue : Uo;   // z + m and z + n have the other parity
    }
    __device__ __forceinline__ const df2 *link(int code) const   // U_m(z), U_n(z+m), U_m(z+n), U_n(z)
    {
        const df2 *u = code == 0 || code == 3 ? Uz : Un + ((code == 1 ? lm : ln) >> 1);
        return u + (long long)(code == 0 || code == 2 ? m : n) * 9 * g.stride;
    }
    // acc = or, for the second product of an E, += product j of
    // a b | d c | b c^+ | d^+ a | Gam_z a, a Gam_{z+m} | Gam_z d, d Gam_{z+n}
    __device__ __forceinline__ void product(int j, M3<df64> &acc) const
    {
        const int lc = (0x34043130 >> (4 * j)) & 15, rc = (0x63500221 >> (4 * j)) & 15;
        const M3<df64> B = rc >= 4 ? load_antiherm(Gam, g.V, rc == 5 ? lm : ln, p) : load_mat(link(rc), g.stride, j == 2);
        if (j != 5 && j != 7)
#pragma unroll
            for (int k = 0; k < 9; k++) acc.a[k] = {df64(0.0f, 0.0f), df64(0.0f, 0.0f)};
        const df2 *A = link(lc);
        const bool gam = lc >= 4, dag = j == 3;
#pragma unroll
        for (int i = 0; i < 3; i++) {   // the left factor one row at a time
            cx<df64> r[3];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (gam) {
                    r[k] = antiherm_entry(Gam, g.V, lz, p, i, k);
                } else {
                    const cx<df64> t = df2_cx(ldg(A + (dag ? k * 3 + i : i * 3 + k) * g.stride));
                    r[k] = dag ? cx<df64>{t.re, dl_neg(t.im)} : t;
                }
            }
            row_fma(acc.a + 3 * i, r, B);
        }
    }
};

// W, W2, Z, V, E_m and E_n of one plaquette per thread (plane = blockIdx.y), for
// the n sites of the slices from t0 on (t0 may be Lt, the first slice again)
__global__ void __launch_bounds__(128, LQ_FLOOP_MINB) force_loop_kernel(Geom g, const df2 *__restrict__ Ue,
                                                         const df2 *__restrict__ Uo, const float2 *__restrict__ Gam,
                                                         LoopMats S, int t0, long long n)
{
    const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (id >= n) return;
    const int p = blockIdx.y;
    int z[4];
    long long site;
    {
        const int tl = (int)(id / S.s3);
        unsigned r = (unsigned)(id - tl * S.s3);
        z[0] = (int)(r % (unsigned)g.L[0]);
        r /= (unsigned)g.L[0];
        z[1] = (int)(r % (unsigned)g.L[1]);
        z[2] = (int)(r / (unsigned)g.L[1]);
        z[3] = t0 + tl >= g.L[3] ? t0 + tl - g.L[3] : t0 + tl;
        site = LQ_IDX(id + (long long)(S.slot(tl) - tl) * S.s3, S.n, B_LEX);
    }
    const Plaquette P(g, Ue, Uo, Gam, p, z);
    M3<df64> acc;
#pragma unroll 1
    for (int j = 0; j < 8; j++) {
        P.product(j, acc);
        if (j == 4 || j == 6) continue;
        df2 *o = S.at(p, j < 4 ? j : j == 5 ? F_EM : F_EN, site);
#pragma unroll
        for (int k = 0; k < 9; k++) o[(long long)k * S.n] = cx_df2(acc.a[k]);
    }
}

// G(x, mu) for one (site, direction) per thread, sites of the slices t0 ..
// (mu = blockIdx.y): the hopping term's outer products, then per plane that
// contains mu the link's two plaquettes, two products each.  FORM: without stored
// matrices, each formed where it is used: 192 products a site in the place of 96, the
// same values, 11.7 ms on 24^3 x 48 (4.93 with them).  It runs when no scratch can be had.
template <bool FORM>
__global__ void __launch_bounds__(128, FORM ? 2 : LQ_FLINK_MINB) force_link_kernel(Geom g, const df2 *__restrict__ Ue,
                                                         const df2 *__restrict__ Uo, const float2 *__restrict__ Gam,
                                                         const df2 *__restrict__ Xe,
                                                         const df2 *__restrict__ Xo, const df2 *__restrict__ Ye,
                                                         const df2 *__restrict__ Yo, LoopMats S, int t0, long long ns,
                                                         double coef, double2 *G)
{
    const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (id >= ns) return;
    const int mu = blockIdx.y;
    const long long lex = t0 * S.s3 + id;
    int c[4];
    lex_coords(g, lex, c);
    const int parity = (c[0] + c[1] + c[2] + c[3]) & 1;
    int cn[4];
    step(g, c, mu, +1, cn, g.L[3]);
    const long long cb = lex >> 1, cbn = lex_of(g, cn) >> 1;
    const df2 *Xx = parity ? Xo : Xe, *Yx = parity ? Yo : Ye;      // at x
    const df2 *Xn = parity ? Xe : Xo, *Yn = parity ? Ye : Yo;      // at x + mu

    // The clover term's products h: plane (h / 4), plaquette at x (0) or x - nu (1),
    // first or second product of the link's two,
    //   U_mu = a: W2 E'^+, E Z^+    = c: V E', E^+ W    = d: E Z, W E'^+    = b: E^+ W2, V^+ E'
    // (E: of the nu links; E' at z + mu).  Both factors are copied to shared memory
    // one product ahead, the first during the hopping term; each thread reads only
    // what it copied itself.
    struct Product {
        bool lower, down, second, efirst;   // lower: mu < nu; efirst: E is the left factor and sits at z
    };
    auto product = [&](int h) {
        const int q = h >> 2, nu = q < mu ? q : q + 1;
        Product r;
        r.lower = mu < nu;
        r.down = h & 2;
        r.second = h & 1;
        r.efirst = r.lower == r.second;
        return r;
    };
    extern __shared__ float4 force_stage[];
    float4 *stage = force_stage + threadIdx.x;
    auto entry = [&](int h, int e) { return stage + ((h & 1) * 18 + e) * 128; };   // left factor 0..8, right 9..17
    // the factors of product h into their entries, the left one first
    auto form_product = [&](int h) {
        const Product r = product(h);
        const int q = h >> 2, nu = q < mu ? q : q + 1;
        const int p = c_plane[r.lower ? mu * 4 + nu : nu * 4 + mu];
        int z[4], zu[4];
        step(g, c, nu, r.down ? -1 : 0, z, g.L[3]);
        step(g, z, mu, +1, zu, g.L[3]);
        const int other = r.down ? (r.efirst ? (r.lower ? F_W : F_W2) : F_V) : (r.efirst ? F_Z : (r.lower ? F_W2 : F_W));
#pragma unroll 1
        for (int f = 0; f < 2; f++) {
            const bool is_e = (f == 0) == r.efirst;
            int y[4];
#pragma unroll
            for (int k = 0; k < 4; k++) y[k] = is_e && !r.efirst ? zu[k] : z[k];
            const Plaquette P(g, Ue, Uo, Gam, p, y);
            const int j0 = is_e ? (r.lower ? 6 : 4) : other, j1 = is_e ? j0 + 2 : j0 + 1;
            M3<df64> t;
#pragma unroll 1
            for (int j = j0; j < j1; j++) P.product(j, t);
#pragma unroll
            for (int e = 0; e < 9; e++) {
                const df2 v = cx_df2(t.a[e]);
                *entry(h, 9 * f + e) = make_float4(v.rh, v.ih, v.rl, v.il);
            }
        }
    };
    const int cs[4] = {c[0], c[1], c[2], S.slot(c[3] - t0)};
    auto copy_product = [&](int h) {
        const Product r = product(h);
        const int q = h >> 2, nu = q < mu ? q : q + 1;
        const int p = c_plane[r.lower ? mu * 4 + nu : nu * 4 + mu];
        int z[4], zu[4];
        step(g, cs, nu, r.down ? -1 : 0, z, S.slots);
        step(g, z, mu, +1, zu, S.slots);
        const long long iz = S.site(g, z), iu = S.site(g, zu);
        const int other = r.down ? (r.efirst ? (r.lower ? F_W : F_W2) : F_V) : (r.efirst ? F_Z : (r.lower ? F_W2 : F_W));
        const df2 *E = S.at(p, r.lower ? F_EN : F_EM, r.efirst ? iz : iu), *O = S.at(p, other, iz);
        const df2 *A = r.efirst ? E : O, *B = r.efirst ? O : E;
#pragma unroll
        for (int e = 0; e < 9; e++) {
            copy_async(entry(h, e), A + e * S.n);
            copy_async(entry(h, 9 + e), B + e * S.n);
        }
        copy_commit();
    };
    if (!FORM) copy_product(0);

    M3<df64> acc;
#pragma unroll
    for (int k = 0; k < 9; k++) acc.a[k] = {df64(0.0f, 0.0f), df64(0.0f, 0.0f)};

    // ---- hopping term: sum_s Y_s(x) (P- X(x+mu))_s^+ + (P+ X(x))_s Y_s(x+mu)^+ ----
#pragma unroll 1
    for (int s = 0; s < 4; s++) {
        const int sp = c_gperm[mu][s], ip = c_gipow[mu][s];
        cx<df64> y[3], w[3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            y[a] = ld_comp(Yx, g.stride, s * 3 + a, cb);
            w[a] = ld_comp(Xn, g.stride, s * 3 + a, cbn) -
                   times_ipow(ld_comp(Xn, g.stride, sp * 3 + a, cbn), ip);   // (1 - g_mu) X(x+mu)
        }
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) {
                dl_cfmac(acc.a[a * 3 + b], w[b], y[a]);
                acc.a[a * 3 + b] = dl_cnorm(acc.a[a * 3 + b]);   // eight terms of one size
            }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            y[a] = ld_comp(Yn, g.stride, s * 3 + a, cbn);
            w[a] = ld_comp(Xx, g.stride, s * 3 + a, cb) +
                   times_ipow(ld_comp(Xx, g.stride, sp * 3 + a, cb), ip);    // (1 + g_mu) X(x)
        }
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) {
                dl_cfmac(acc.a[a * 3 + b], y[b], w[a]);
                acc.a[a * 3 + b] = dl_cnorm(acc.a[a * 3 + b]);   // eight terms of one size
            }
    }
    {
        const bool wrap = mu == 3 && c[3] == g.L[3] - 1;
        const float f = (wrap && g.tbc < 0) ? 0.5f : -0.5f;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const cx<df64> t = acc.a[k];
            acc.a[k] = {dl_scale2(t.re, f), dl_scale2(t.im, f)};
        }
    }

    // ---- clover term: the two plaquettes of each plane (mu, nu) that hold U_mu(x) ----
#pragma unroll 1
    for (int h = 0; h < 12; h++) {
        if (FORM) {
            form_product(h);
        } else if (h < 11) {
            copy_product(h + 1);
            copy_wait<1>();
        } else {
            copy_wait<0>();
        }
        const Product r = product(h);
        const bool dag = r.down && (r.efirst || !r.lower), dagb = !r.down && (r.efirst ? r.lower : true);
        const unsigned sre = r.second ? 0x80000000u : 0u, sim = (r.second != dag) ? 0x80000000u : 0u;
        const unsigned sb = dagb ? 0x80000000u : 0u;
        auto factor = [&](int at, bool t, int i, int k) {   // entry (i, k) of a factor as stored, or its transpose
            const float4 v = *entry(h, at + (t ? k * 3 + i : i * 3 + k));
            return cx<df64>{df64(v.x, v.z), df64(v.y, v.w)};
        };
        M3<df64> B;
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const cx<df64> t = factor(9, dagb, i, k);
                B.a[i * 3 + k] = {t.re, flip_sign(t.im, sb)};
            }
#pragma unroll
        for (int i = 0; i < 3; i++) {   // the left factor one row at a time, with the product's sign
            cx<df64> row[3];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const cx<df64> t = factor(0, dag, i, k);
                row[k] = {flip_sign(t.re, sre), flip_sign(t.im, sim)};
            }
            row_fma(acc.a + 3 * i, row, B);
        }
    }

    double2 *o = G + (lex * 4 + mu) * 9;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const cx<df64> v = acc.a[k];
        o[k] = make_double2(coef * df_join(v.re.hi, v.re.lo), coef * df_join(v.im.hi, v.im.lo));
    }
}

// out = g5 in on natural full spinors [V][4][3] complex double (spins 2, 3 negated)
__global__ void gamma5_nat_kernel(long long V, const double2 *in, double2 *out)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= V * 12) return;
    const double2 v = in[i];
    out[i] = ((i % 12) >= 6) ? make_double2(-v.x, -v.y) : v;
}

static inline unsigned blocks_of(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

void force_insertion(const Exec &e, const void *X[2], const void *Y[2], double csw, void *Gam)
{
    // reads X, Y (2 x 192 B df64), writes six anti-Hermitian 3x3 (6 x 72 B);
    // per site 6 blocks x (2 x 9 products + 9 additions) and the Hermitian parts
    Launch L_(e, K_FORCE, (double)e.g.V * (2 * 192 + 6 * 72), (double)e.g.V * 3 * 2 * (18 * 6 + 18 * 2 + 18 * 2));
    force_insertion_kernel<<<blocks_of(e.g.V, 128), 128, 0, e.st>>>(
        e.g, (const df2 *)X[0], (const df2 *)X[1], (const df2 *)Y[0], (const df2 *)Y[1], df64(csw / 16.0),
        (float2 *)Gam);
}

// The plaquette matrices take 5184 B a site, so the lattice goes through in ranges
// of time slices: the matrices of a range and of the slice on either side stand in
// a ring of slices, in which the next range finds the two that it shares with this
// one: 7.6 ns a site on 48^3 x 96 in ranges of one slice, 14.0 with the neighbours made
// anew for each, 7.4 on 24^3 x 48 in ranges of 27.  Bytes of a ring of `slots` slices.
size_t force_scratch_bytes(const Geom &g, int slots)
{
    return (size_t)slots * (g.V / g.L[3]) * 6 * F_MATS * 9 * sizeof(df2);
}

// slots: Lt (every slice at once), from 3 to Lt - 1 (ranges of slots - 2 slices), or
// 0 (no scratch)
void force_links(const Exec &e, const void *Udf[2], const void *X[2], const void *Y[2], const void *Gam, void *scratch,
                 int slots, double coef, void *G)
{
    const Geom &g = e.g;
    const int Lt = g.L[3];
    const df2 *Ue = (const df2 *)Udf[0], *Uo = (const df2 *)Udf[1];
    LoopMats S;
    S.m = (df2 *)scratch;
    S.s3 = g.V / Lt;
    S.slots = slots;
    S.n = slots * S.s3;
    S.head = 0;
    const int range = slots == 0 || slots == Lt ? Lt : slots - 2;
    auto links = [&](auto form, int t0, int nt) {
        constexpr bool FORM = decltype(form)::value;
        const long long ns = nt * S.s3;
        // X and Y, the matrices, the 4 gradients (c128); per link 12 products and
        // the hopping term's 2 x 4 x 9 outer-product entries
        Launch L_(e, K_FORCE, (double)ns * (2 * 192 + (FORM ? 4 * 144 + 6 * 72 : 36 * 144) + 4 * 144),
                  (double)ns * 4 * ((FORM ? 48 : 12) * (198 + 18) + 2 * 4 * (9 * 8 + 12)));
        constexpr int sm = 2 * 18 * 128 * (int)sizeof(float4);
        cudaFuncSetAttribute(force_link_kernel<FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        force_link_kernel<FORM><<<dim3(blocks_of(ns, 128), 4), 128, sm, e.st>>>(
            g, Ue, Uo, (const float2 *)Gam, (const df2 *)X[0], (const df2 *)X[1], (const df2 *)Y[0], (const df2 *)Y[1],
            S, t0, ns, coef, (double2 *)G);
    };
    if (slots == 0) return links(std::true_type(), 0, Lt);
    for (int t0 = 0; t0 < Lt; t0 += range) {
        const int nt = Lt - t0 < range ? Lt - t0 : range;
        int from = 0, count = Lt;   // the slices to make
        if (slots != Lt) {          // t0 - 1 .. t0 + nt, of which the first two are there from the second range on;
                                    // slice t has the slot (t + 1) mod slots
            from = t0 ? t0 + 1 : Lt - 1;
            count = t0 ? nt : nt + 2;
            S.head = t0 ? (t0 + 2) % slots : 0;
        }
        {
            // unique bytes per site: 4 df64 links and six Gam in, 36 matrices out; per
            // plane eight 3x3 products of 198 flops
            const long long n = count * S.s3;
            Launch L_(e, K_FORCE, (double)n * (4 * 144 + 6 * 72 + 36 * 144), (double)n * 6 * 8 * 198);
            force_loop_kernel<<<dim3(blocks_of(n, 128), 6), 128, 0, e.st>>>(g, Ue, Uo, (const float2 *)Gam, S, from, n);
        }
        if (slots != Lt) S.head = (t0 + 1) % slots;
        links(std::false_type(), t0, nt);
    }
}

void gamma5_nat(const Exec &e, const void *in, void *out)
{
    Launch L_(e, K_LAYOUT, (double)e.g.V * 2 * 192);
    gamma5_nat_kernel<<<blocks_of(e.g.V * 12, 256), 256, 0, e.st>>>(e.g.V, (const double2 *)in, (double2 *)out);
}

}  // namespace lq
