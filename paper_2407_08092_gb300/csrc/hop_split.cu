// The hopping kernels of small lattices: twelve threads per output site.
//
// With one thread per site (dslash.cu) a lattice of a few thousand sites leaves
// most SMs without a block, and its time is one thread's chain of eight hops and
// two clover blocks.  Here a block of twelve warps holds 32 sites, lane = site:
//   1. warp d < 8 forms the transported half spinor u of direction d;
//   2. warp c < 12 sums the eight contributions to component c;
//   3. warp c forms component c of the site term, one row of a 6x6 clover block,
//      whose entries it loaded before step 1.
// The operations are those of the larger lattices' kernels.
//
// lq_apply of D_S in us, twelve threads and the larger lattices' kernels (one thread
// a site in FP32 and BF16, two in df64 and FP64), at 2048 sites a parity: df64
// 14.5 / 22.6, FP32 12.3 / 18.4, FP64 34.8 / 47.2, BF16 12.4 / 24.7; at 24576: 53.4 / 40.5,
// 26.7 / 28.9, 158 / 138, 28.8 / 28.8.  The larger the lattice, the less it needs the
// extra threads, which pass the eight half spinors through shared memory and idle
// while others work.
// df64 takes one block an SM (168 registers; two: 8 us more at 2048 sites).
#include <type_traits>

#include "bf16.cuh"
#include "lq_kernels.h"
#include "nat.cuh"
#include "spin.cuh"

namespace lq {

constexpr int kSplitSites = 32, kSplitThreads = 12 * kSplitSites;

// component c of a field at site s
__device__ __forceinline__ cx<double> ld_comp(const double2 *f, long long st, long long s, int c)
{
    const double2 t = f[c * st + s];
    return {t.x, t.y};
}
__device__ __forceinline__ cx<df64> ld_comp(const df2 *f, long long st, long long s, int c) { return df2_cx(f[c * st + s]); }
__device__ __forceinline__ cx<float> ld_comp(const float4 *f, long long st, long long s, int c)
{
    const float2 t = reinterpret_cast<const float2 *>(f + (c >> 1) * st + s)[c & 1];
    return {t.x, t.y};
}
__device__ __forceinline__ cx<float> ld_comp(const BfS4 *f, long long st, long long s, int c)
{
    return bf_cx((f + (c >> 2) * st + s)->c[c & 3]);
}
__device__ __forceinline__ void st_comp(double2 *f, long long st, long long s, int c, cx<double> v)
{
    f[c * st + s] = make_double2(v.re, v.im);
}
__device__ __forceinline__ void st_comp(df2 *f, long long st, long long s, int c, cx<df64> v) { f[c * st + s] = cx_df2(v); }
__device__ __forceinline__ void st_comp(float4 *f, long long st, long long s, int c, cx<float> v)
{
    reinterpret_cast<float2 *>(f + (c >> 1) * st + s)[c & 1] = make_float2(v.re, v.im);
}
__device__ __forceinline__ void st_comp(BfS4 *f, long long st, long long s, int c, cx<float> v)
{
    (f + (c >> 2) * st + s)->c[c & 3] = cx_bf(v);
}

// Row r of a packed 6x6 clover block: its diagonal entry and the five others in
// column order, each as it stands in the lower triangle (the conjugate of the
// row's entry in the columns above r).
template <typename R>
struct CloverRow {
    R diag;
    cx<R> l[5];
};
__device__ __forceinline__ cx<double> clover_pair(const double2 *C, long long st, long long s, int blk, int k)
{
    const double2 t = ldg(C + (blk * 18 + (k >> 1)) * st + s);
    return {t.x, t.y};
}
__device__ __forceinline__ cx<df64> clover_pair(const df2 *C, long long st, long long s, int blk, int k)
{
    return df2_cx(ldg(C + (blk * 18 + (k >> 1)) * st + s));
}
__device__ __forceinline__ cx<float> clover_pair(const float4 *C, long long st, long long s, int blk, int k)
{
    const float2 t = __ldg(reinterpret_cast<const float2 *>(C + (blk * 9 + (k >> 2)) * st + s) + ((k >> 1) & 1));
    return {t.x, t.y};
}
template <typename R, typename CV>
__device__ __forceinline__ CloverRow<R> load_row(const CV *C, long long st, long long s, int blk, int r)
{
    CloverRow<R> w;
    const cx<R> d = clover_pair(C, st, s, blk, r & ~1);
    w.diag = (r & 1) ? d.im : d.re;
#pragma unroll
    for (int q = 0; q < 5; q++) w.l[q] = clover_pair(C, st, s, blk, 6 + 2 * (q < r ? tri(r, q) : tri(q + 1, r)));
    return w;
}

// y0 + (row of C) x, x[j * kSplitSites] the six components of the block; `y0`
// enters as the larger lattices' kernels add it: before the row in df64, not at all in
// the others, where the caller adds to the row's product
template <typename R>
__device__ __forceinline__ cx<R> row_apply(const CloverRow<R> &w, int r, const cx<R> *x, cx<R>)
{
    cx<R> y = w.diag * x[r * kSplitSites];
#pragma unroll
    for (int q = 0; q < 5; q++) {
        const int j = q < r ? q : q + 1;
        const cx<R> l = {w.l[q].re, q < r ? w.l[q].im : -w.l[q].im};
        y = cfma(l, x[j * kSplitSites], y);
    }
    return y;
}
template <>
__device__ __forceinline__ cx<df64> row_apply<df64>(const CloverRow<df64> &w, int r, const cx<df64> *x, cx<df64> y0)
{
    df64x2 y = dl2(y0), z;
    dl2_fma(y, dl2_both(w.diag), dl2(x[r * kSplitSites]));
#pragma unroll
    for (int q = 0; q < 5; q++) {
        const int j = q < r ? q : q + 1;
        const df64x2 xj = dl2(x[j * kSplitSites]), im = dl2_both(q < r ? w.l[q].im : dl_neg(w.l[q].im));
        dl2_fma(y, dl2_both(w.l[q].re), xj);
        if (q == 0) z = dl2_prod(im, xj);
        else dl2_fma(z, im, xj);
    }
    dl2_add(y, dlrow_rot({y, z}));
    return dl_cnorm(dl2_cx(y));
}

// the transported half spinor of direction D at the neighbour nb
template <int D, typename R, typename SV, typename LV>
__device__ __forceinline__ void half_hop(const SV *psi, const LV *U, long long st, long long link, long long nb, R sign,
                                         cx<R> u[6])
{
    constexpr int MU = D >> 1, SIGN = (D & 1) ? +1 : -1;
    cx<R> p[12], m[9], h[6];
    load_spinor_rw(psi, st, nb, p);
    load_link(U, st, MU, link, m);
    project<MU, SIGN>(p, h);
    transport<SIGN>(m, h, sign, u);
}
template <typename R, typename SV, typename LV>
struct HalfHop {
    static __device__ __forceinline__ void run(int d, const SV *psi, const LV *Uout, const LV *Uin, long long st,
                                               long long s, long long nb, R sign, cx<R> u[6])
    {
        switch (d) {
        case 0: half_hop<0>(psi, Uout, st, s, nb, sign, u); break;
        case 1: half_hop<1>(psi, Uin, st, nb, nb, sign, u); break;
        case 2: half_hop<2>(psi, Uout, st, s, nb, sign, u); break;
        case 3: half_hop<3>(psi, Uin, st, nb, nb, sign, u); break;
        case 4: half_hop<4>(psi, Uout, st, s, nb, sign, u); break;
        case 5: half_hop<5>(psi, Uin, st, nb, nb, sign, u); break;
        case 6: half_hop<6>(psi, Uout, st, s, nb, sign, u); break;
        default: half_hop<7>(psi, Uin, st, nb, nb, sign, u); break;
        }
    }
    static __device__ __forceinline__ void add(cx<R> &acc, cx<R> u) { acc = acc + u; }
    static __device__ __forceinline__ cx<R> norm(cx<R> acc) { return acc; }
    static __device__ __forceinline__ cx<R> scale(cx<R> a, float f) { return R(f) * a; }
};
// df64: one body for the eight directions, as in hop_df_kernel
template <>
struct HalfHop<df64, df2, df2> {
    static __device__ __forceinline__ void run(int d, const df2 *psi, const df2 *Uout, const df2 *Uin, long long st,
                                               long long s, long long nb, df64 sign, cx<df64> u[6])
    {
        const bool fwd = (d & 1) == 0;
        const int qa = (kHopQA >> (2 * d)) & 3, qb = (kHopQB >> (2 * d)) & 3;
        const df2 *Um = (fwd ? Uout + s : Uin + nb) + (long long)(d >> 1) * 9 * st;
        cx<df64> m[9], h[6];
#pragma unroll
        for (int k = 0; k < 9; k++) m[k] = df2_cx(ldg(Um + k * st));
#pragma unroll
        for (int a = 0; a < 3; a++) {
            h[a] = df2_cx(psi[a * st + nb]);
            dl_cadd(h[a], rot_i(df2_cx(psi[(d < 4 ? 9 + a : 6 + a) * st + nb]), qa));
            h[3 + a] = df2_cx(psi[(3 + a) * st + nb]);
            dl_cadd(h[3 + a], rot_i(df2_cx(psi[(d < 4 ? 6 + a : 9 + a) * st + nb]), qb));
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            cx<df64> e[3];
#pragma unroll
            for (int b = 0; b < 3; b++) e[b] = fwd ? m[a * 3 + b] : cx<df64>{m[b * 3 + a].re, dl_neg(m[b * 3 + a].im)};
#pragma unroll
            for (int q = 0; q < 2; q++) {
                dlrow r = dlrow_prod(e[0], dl2(h[3 * q]));
                dlrow_fma(r, e[1], dl2(h[3 * q + 1]));
                dlrow_fma(r, e[2], dl2(h[3 * q + 2]));
                dl2_add(r.r, dlrow_rot(r));
                const cx<df64> v = dl2_cx(r.r);
                u[3 * q + a] = sign.hi < 0.0f ? cx<df64>{dl_neg(v.re), dl_neg(v.im)} : v;
            }
        }
    }
    static __device__ __forceinline__ void add(cx<df64> &acc, cx<df64> u) { dl_cadd(acc, u); }
    static __device__ __forceinline__ cx<df64> norm(cx<df64> acc) { return dl_cnorm(acc); }
    static __device__ __forceinline__ cx<df64> scale(cx<df64> a, float f) { return {dl_scale2(a.re, f), dl_scale2(a.im, f)}; }
};
// t + a for the modes that add to a loaded field
template <typename R>
__device__ __forceinline__ cx<R> plus(cx<R> t, cx<R> a) { return t + a; }
template <>
__device__ __forceinline__ cx<df64> plus<df64>(cx<df64> t, cx<df64> a)
{
    dl_cadd(t, a);
    return dl_cnorm(t);
}

template <typename R, typename SV, typename LV, typename CV>
struct SplitArgs {
    const SV *in, *in2, *b;
    SV *out, *out2;
    const LV *Uout, *Uin;
    const CV *clov, *clov2;
    R omega;
    int pout, nrhs;
    long long fs;
    NatOut nat;
};

template <typename R, int MODE, typename SV, typename LV, typename CV>
__global__ void __launch_bounds__(kSplitThreads, std::is_same<R, df64>::value ? 1 : 2) hop_split_kernel(const __grid_constant__ Geom g,
                                                                  const __grid_constant__ SplitArgs<R, SV, LV, CV> k)
{
    typedef HalfHop<R, SV, LV> H;
    extern __shared__ __align__(16) unsigned char split_sm[];
    after_previous();
    cx<R> *U = reinterpret_cast<cx<R> *>(split_sm);        // [direction][6][site]
    cx<R> *X = U + 48 * kSplitSites;                       // [12][site]: what the clover blocks multiply
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned sb = blockIdx.x / (unsigned)k.nrhs;
    const long long o = (blockIdx.x - sb * k.nrhs) * k.fs, st = g.stride;
    const long long s0 = sb * (long long)kSplitSites + lane;
    const bool on = s0 < g.Vh;
    const long long s = LQ_IDX(on ? s0 : g.Vh - 1, g.Vh, B_HOP_SITE);   // idle lanes shadow the last site, without its stores
    constexpr bool CLOVER = MODE != HOP_PREP, SITE = MODE != HOP_K1;
    constexpr bool RECON = MODE == HOP_RECON || MODE == HOP_RECON_RES;
    const int blk = w >= 6 ? 1 : 0, row = w - 6 * blk;

    CloverRow<R> C;
    if constexpr (CLOVER) C = load_row<R>(k.clov, st, s, blk, row);
    cx<R> x;
    if constexpr (SITE) {
        x = ld_comp(k.in2 + o, st, s, w);
        if (!RECON && CLOVER) X[w * kSplitSites + lane] = x;
    }
    if (w < 8) {
        const Coords c = cb_coords(g, s, k.pout);
        bool cross;
        const long long nb = hop_neighbour(g, c, s, w, cross, B_HOP_NB);
        cx<R> u[6];
        H::run(w, k.in + o, k.Uout, k.Uin, st, s, nb, cross && g.tbc < 0 ? R(-1.0f) : R(1.0f), u);
#pragma unroll
        for (int q = 0; q < 6; q++) U[(w * 6 + q) * kSplitSites + lane] = u[q];
    }
    __syncthreads();

    // component w = 3 spin + colour of the sum over directions
    const int spin = w / 3, a = w - 3 * spin;
    cx<R> acc = {R(0.0f), R(0.0f)};
    const unsigned turn = spin < 2 ? 0u : spin == 2 ? kHopQC : kHopQD;
#pragma unroll
    for (int d = 0; d < 8; d++) {
        const int half = spin < 2 ? spin : (d < 4) == (spin == 2) ? 1 : 0;
        const cx<R> u = rot_i(U[(d * 6 + 3 * half + a) * kSplitSites + lane], (turn >> (2 * d)) & 3);
        if (d == 0 && std::is_same<R, double>::value) acc = u;
        else H::add(acc, u);
    }
    acc = H::norm(acc);

    const cx<R> zero = {R(0.0f), R(0.0f)};
    const cx<R> *Xb = X + 6 * blk * kSplitSites + lane;
    cx<R> v;
    if constexpr (MODE == HOP_K1) {
        X[w * kSplitSites + lane] = H::scale(acc, -0.5f);
        __syncthreads();
        v = row_apply<R>(C, row, Xb, zero);
    } else if constexpr (!RECON && CLOVER) {
        const cx<R> ha = H::scale(acc, MODE == HOP_FULL || MODE == HOP_RES ? -0.5f : 0.5f);
        v = row_apply<R>(C, row, Xb, ha);
        if constexpr (!std::is_same<R, df64>::value) v = v + ha;
        if constexpr (MODE == HOP_RICH) v = x + k.omega * (ld_comp(k.b + o, st, s, w) - v);
        if constexpr (MODE == HOP_RES) v = ld_comp(k.b + o, st, s, w) - v;
    } else {
        v = plus<R>(x, H::scale(acc, 0.5f));
        if constexpr (RECON) {
            const cx<R> y = v;
            X[w * kSplitSites + lane] = y;
            __syncthreads();
            v = row_apply<R>(C, row, Xb, zero);
            if constexpr (MODE == HOP_RECON_RES) {
                C = load_row<R>(k.clov2, st, s, blk, row);
                __syncthreads();
                X[w * kSplitSites + lane] = v;
                __syncthreads();
                const cx<R> z = row_apply<R>(C, row, Xb, zero);
                if (on) st_comp(k.out2 + o, st, s, w, y - z);
            }
        }
    }
    if (k.nat.p) {   // 32 natural rows through shared memory, one vector a thread
        double2 *tile = reinterpret_cast<double2 *>(split_sm);   // over U: 32 rows of 12 and a pad
        double2 d = nat_value((const SV *)nullptr, v);
        if (w >= 6) d = make_double2(flip_sign64(d.x, k.nat.flip), flip_sign64(d.y, k.nat.flip));
        __syncthreads();
        tile[lane * 13 + w] = d;
        __syncthreads();
        const int r = threadIdx.x / 12, c = threadIdx.x - 12 * r;
        const long long q = sb * (long long)kSplitSites + r;
        if (q < g.Vh) {
            const long long row = k.nat.full ? 2 * q + (cb_coords(g, q, k.pout).x & 1) : q;
            k.nat.p[LQ_IDX(row, k.nat.rows, B_NAT) * 12 + c] = tile[r * 13 + c];
        }
    } else if (on) {
        st_comp(k.out + o, st, s, w, v);
    }
}

template <typename R, int MODE, typename SV, typename LV, typename CV>
static void launch_split(const Exec &e, const HopCall &c)
{
    SplitArgs<R, SV, LV, CV> k;
    k.in = (const SV *)c.in;
    k.in2 = (const SV *)c.in2;
    k.b = (const SV *)c.b;
    k.out = (SV *)c.out;
    k.out2 = (SV *)c.out2;
    k.Uout = (const LV *)c.U[c.pout];
    k.Uin = (const LV *)c.U[1 - c.pout];
    k.clov = (const CV *)c.clov;
    k.clov2 = (const CV *)c.clov2;
    k.omega = R(c.omega);
    k.pout = c.pout;
    k.nrhs = c.nrhs;
    k.fs = (long long)(spinor_bytes(e.g, c.prec) / sizeof(SV));
    k.nat = nat_out(e.g, c.nat, c.nat_full, c.nat_g5);
    const unsigned blocks = (unsigned)((e.g.Vh + kSplitSites - 1) / kSplitSites) * (unsigned)c.nrhs;
    launch_after(e, c.after, hop_split_kernel<R, MODE, SV, LV, CV>, blocks, kSplitThreads, 60 * kSplitSites * sizeof(cx<R>), e.g, k);
}

bool hop_split_takes(const Geom &g, int prec, int nrhs)
{
    // Sites up to which twelve threads are the faster, in us with twelve and without:
    // D_S of df64 22.7 / 24.4 at 9216, 30.9 / 30.9 at 12096, 39.1 / 35.0 at 16384; of FP32
    // 20.6 / 27.0 at 18432, 26.7 / 28.9 at 24576, where Richardson(4) takes 118 / 111; of
    // BF16 22.6 / 26.8 at 18432, 28.8 / 28.8 at 24576.  FP64: D_S 34.9 / 47.2 at 4096 and
    // 84.0 / 69.8 at 12096, a GMRES solve 8.6 / 10.3 ms at 10368, 10.4 / 11.5 at 12096,
    // 14.6 / 14.8 at 24576.
    const long long most = prec == P32 || prec == P16 ? 20480 : 12288;
    return g.Vh * nrhs <= most;
}

template <int M>
static void split_mode(const Exec &e, const HopCall &c)
{
    if (c.prec == P64) return launch_split<double, M, double2, double2, double2>(e, c);
    if (c.prec == PDF) return launch_split<df64, M, df2, df2, df2>(e, c);
    if constexpr (hop_form(M, P32))
        if (c.prec == P32) return launch_split<float, M, float4, float4, float4>(e, c);
    if constexpr (hop_form(M, P16))
        if (c.prec == P16) return launch_split<float, M, BfS4, BfL2, float4>(e, c);
}

bool hop_split(const Exec &e, const HopCall &c)
{
    if (!hop_split_takes(e.g, c.prec, c.nrhs)) return false;
    switch (c.mode) {
    case HOP_K1: split_mode<HOP_K1>(e, c); break;
    case HOP_K2: split_mode<HOP_K2>(e, c); break;
    case HOP_RICH: split_mode<HOP_RICH>(e, c); break;
    case HOP_FULL: split_mode<HOP_FULL>(e, c); break;
    case HOP_PREP: split_mode<HOP_PREP>(e, c); break;
    case HOP_RECON: split_mode<HOP_RECON>(e, c); break;
    case HOP_RES: split_mode<HOP_RES>(e, c); break;
    case HOP_RECON_RES: split_mode<HOP_RECON_RES>(e, c); break;
    }
    return true;
}

}  // namespace lq
