// The fused hopping kernels of the odd-even Wilson-clover operator.
//
// One thread per output site of one parity (FP32 and BF16 storage; the df64 form
// below takes two, FP64 is hop_f64.cu and small lattices hop_split.cu).  For each
// of the eight directions the neighbour spinor is spin-projected onto a half spinor with
// (1 -+ g_mu), multiplied by the link (U_mu(x) forward, U_mu(x-mu)^+ backward)
// and reconstructed into the 12-component accumulator; the epilogue then
// applies the site-diagonal clover block (C or C^{-1}) and whatever BLAS-1
// step the mode fuses.  Together the two launches
//   K1: t_o = D_oo^{-1} D_oe x_e      (HOP_K1 on odd sites)
//   K2: y_e = D_ee x_e - D_eo t_o     (HOP_K2 on even sites)
// apply the Schur complement D_S of Eq. 3; HOP_RICH fuses the Richardson
// update x_e += omega (b_e - D_S x_e) of Algorithm 4 into K2.
// The spin projection and transport of one hop live in spin.cuh.
#include <type_traits>

#include "bf16.cuh"
#include "lq_kernels.h"
#include "nat.cuh"
#include "spin.cuh"

namespace lq {

#define LQ_HOP_THREADS 128
static_assert(LQ_HOP_THREADS == kHopBlock, "hopping block size");
// minimum resident blocks per SM asked of the single-right-hand-side kernels.
// Unset leaves the register allocation to the compiler's default for
// 128-thread blocks, which differs from an explicit 1 (that one lets the
// kernels grow to about 160 registers).
#ifdef LQ_HOP_MINB
#define LQ_HOP_BOUNDS __launch_bounds__(LQ_HOP_THREADS, LQ_HOP_MINB)
#else
#define LQ_HOP_BOUNDS __launch_bounds__(LQ_HOP_THREADS)
#endif

// one hop: acc += (1 -+ g_mu) W psi(nb), W = U_mu(x) (SIGN -1) or U_mu(x-mu)^+ (SIGN +1);
// `bsign` is the fermion boundary factor of this hop
template <int MU, int SIGN, typename R, typename SV, typename LV>
__device__ __forceinline__ void hop_dir(cx<R> acc[12], const SV *psi, const LV *__restrict__ U,
                                        long long link_site, long long nb, long long stride, R bsign)
{
    cx<R> p[12];
    load_spinor_rw(psi, stride, nb, p);   // the kernel before wrote it: not through the read-only path (after_previous)
    cx<R> m[9];
    load_link(U, stride, MU, link_site, m);
    hop_apply<MU, SIGN>(acc, p, m, bsign);
}

template <typename R>
struct HopArgs {
    typedef typename St<R>::vec V;
    const V *in;
    const V *in2;
    const V *b;
    V *out;
    const V *Uout;   // links of the output parity: forward links U_mu(x)
    const V *Uin;    // links of the input parity: backward links U_mu(x - mu)
    const V *clov;
    const V *clov2;  // HOP_RECON_RES: C of the output parity
    V *out2;         // HOP_RECON_RES: the residual
    R omega;
    int pout;
    int nrhs;        // right-hand sides sharing the links and clover of this launch
    long long fs;    // distance between consecutive right-hand sides' fields, in vectors
    NatOut nat;      // natural output in the place of `out`
};

// all twelve components of a warp's sites in natural form, six at a time: seven
// slots a row keep the shared-memory accesses free of bank conflicts
constexpr int kNatRow = 7;
template <typename SV, typename R>
__device__ __forceinline__ void store_nat(const NatOut &o, double2 *tile, const SV *, long long s0, int n, int xbit,
                                          const cx<R> v[12])
{
    const int lane = threadIdx.x & 31;
    auto at = [](int r, int k) { return r * kNatRow + k; };
#pragma unroll
    for (int half = 0; half < 2; half++) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 6; k++) {
            double2 d = nat_value((const SV *)nullptr, v[6 * half + k]);
            if (half) d = make_double2(flip_sign64(d.x, o.flip), flip_sign64(d.y, o.flip));
            tile[at(lane, k)] = d;
        }
        __syncwarp();
        nat_write6(o, tile, at, s0, n, xbit, half);
    }
}


// SV, LV, CV: storage vectors of the spinors, links and clover blocks (the same
// type for FP64, FP32 and df64; BF16 spinors and links with FP32 clover)
// (SCALED, for K1 and K2: omega is a factor of the input field)
template <typename R, int MODE, bool NAT = false, bool SCALED = false, typename SV, typename LV, typename CV>
__device__ __forceinline__ void hop_body(const Geom &g, const LV *Uout, const LV *Uin, const CV *clov, R omega,
                                         const SV *in, const SV *in2, const SV *bv, SV *out, long long s,
                                         const Coords &c, const NatOut &nat = NatOut(), double2 *tile = nullptr, int nvalid = 0)
{
    const long long st = g.stride;
    cx<R> acc[12];
#pragma unroll
    for (int i = 0; i < 12; i++) acc[i] = {R(0), R(0)};
    const R one = R(1);

    // x direction: the neighbour changes x, so its cb index is recomputed
    {
        const long long base = c.row * g.Lxh;
        const int xp = (c.x + 1 == g.L[0]) ? 0 : c.x + 1;
        const int xm = (c.x == 0) ? g.L[0] - 1 : c.x - 1;
        const long long nf = LQ_IDX(base + (xp >> 1), g.Vh, B_HOP_NB), nb = LQ_IDX(base + (xm >> 1), g.Vh, B_HOP_NB);
        hop_dir<0, -1>(acc, in, Uout, s, nf, st, one);
        hop_dir<0, +1>(acc, in, Uin, nb, nb, st, one);
    }
    // y, z, t: x is unchanged, so the cb index moves by a fixed stride
    {
        const long long d = g.Lxh;
        const long long nf = LQ_IDX((c.y + 1 == g.L[1]) ? s - (long long)(g.L[1] - 1) * d : s + d, g.Vh, B_HOP_NB);
        const long long nb = LQ_IDX((c.y == 0) ? s + (long long)(g.L[1] - 1) * d : s - d, g.Vh, B_HOP_NB);
        hop_dir<1, -1>(acc, in, Uout, s, nf, st, one);
        hop_dir<1, +1>(acc, in, Uin, nb, nb, st, one);
    }
    {
        const long long d = (long long)g.Lxh * g.L[1];
        const long long nf = LQ_IDX((c.z + 1 == g.L[2]) ? s - (long long)(g.L[2] - 1) * d : s + d, g.Vh, B_HOP_NB);
        const long long nb = LQ_IDX((c.z == 0) ? s + (long long)(g.L[2] - 1) * d : s - d, g.Vh, B_HOP_NB);
        hop_dir<2, -1>(acc, in, Uout, s, nf, st, one);
        hop_dir<2, +1>(acc, in, Uin, nb, nb, st, one);
    }
    {
        const long long d = (long long)g.Lxh * g.L[1] * g.L[2];
        const bool last = (c.t + 1 == g.L[3]), first = (c.t == 0);
        const long long nf = LQ_IDX(last ? s - (long long)(g.L[3] - 1) * d : s + d, g.Vh, B_HOP_NB);
        const long long nb = LQ_IDX(first ? s + (long long)(g.L[3] - 1) * d : s - d, g.Vh, B_HOP_NB);
        const R tb = R(g.tbc);
        hop_dir<3, -1>(acc, in, Uout, s, nf, st, last ? tb : one);
        hop_dir<3, +1>(acc, in, Uin, nb, nb, st, first ? tb : one);
    }

    cx<R> v[12];
    if (MODE == HOP_K1) {
#pragma unroll
        for (int i = 0; i < 12; i++) acc[i] = (SCALED ? R(-0.5) * omega : R(-0.5)) * acc[i];
        clover_apply<R>(clov, st, s, acc, v);
    } else {   // HOP_K2, HOP_RICH, HOP_FULL
        cx<R> x[12];
        load_spinor_rw(in2, st, s, x);
        clover_apply<R>(clov, st, s, x, v);
        const R f = MODE == HOP_FULL ? R(-0.5) : R(0.5);
#pragma unroll
        for (int i = 0; i < 12; i++) v[i] = (SCALED ? omega * v[i] : v[i]) + f * acc[i];
        if (MODE == HOP_RICH) {
            cx<R> bb[12];
            load_spinor(bv, st, s, bb);
#pragma unroll
            for (int i = 0; i < 12; i++) v[i] = x[i] + omega * (bb[i] - v[i]);
        }
    }
    if (NAT) store_nat(nat, tile, (const SV *)nullptr, s - min((int)(threadIdx.x & 31), nvalid - 1), nvalid, c.x & 1, v);
    else store_spinor(out, st, s, v);
}

// Two right-hand sides per thread (K1 and K2 of the batched hop): each link is
// loaded once and transports both neighbour spinors.
template <int MU, int SIGN>
__device__ __forceinline__ void hop_dir2(cx<float> acc0[12], cx<float> acc1[12], const float4 *__restrict__ psi0,
                                         const float4 *__restrict__ psi1, const float4 *__restrict__ U,
                                         long long link_site, long long nb, long long stride, float bsign)
{
    cx<float> m[9];
    load_link(U, stride, MU, link_site, m);
    cx<float> p[12];
    load_spinor(psi0, stride, nb, p);
    hop_apply<MU, SIGN>(acc0, p, m, bsign);
    load_spinor(psi1, stride, nb, p);
    hop_apply<MU, SIGN>(acc1, p, m, bsign);
}

template <int MODE>
__device__ __forceinline__ void hop_body2(const Geom &g, const float4 *Uout, const float4 *Uin, const float4 *clov,
                                          const float4 *in0, const float4 *in1, const float4 *in20,
                                          const float4 *in21, float4 *out0, float4 *out1, bool two, long long s,
                                          const Coords &c, float sc0, float sc1)
{
    const long long st = g.stride;
    cx<float> a0[12], a1[12];
#pragma unroll
    for (int i = 0; i < 12; i++) a0[i] = a1[i] = {0.0f, 0.0f};
    {
        const long long base = c.row * g.Lxh;
        const int xp = (c.x + 1 == g.L[0]) ? 0 : c.x + 1;
        const int xm = (c.x == 0) ? g.L[0] - 1 : c.x - 1;
        const long long nf = LQ_IDX(base + (xp >> 1), g.Vh, B_HOP_NB), nb = LQ_IDX(base + (xm >> 1), g.Vh, B_HOP_NB);
        hop_dir2<0, -1>(a0, a1, in0, in1, Uout, s, nf, st, 1.0f);
        hop_dir2<0, +1>(a0, a1, in0, in1, Uin, nb, nb, st, 1.0f);
    }
    {
        const long long d = g.Lxh;
        const long long nf = LQ_IDX((c.y + 1 == g.L[1]) ? s - (long long)(g.L[1] - 1) * d : s + d, g.Vh, B_HOP_NB);
        const long long nb = LQ_IDX((c.y == 0) ? s + (long long)(g.L[1] - 1) * d : s - d, g.Vh, B_HOP_NB);
        hop_dir2<1, -1>(a0, a1, in0, in1, Uout, s, nf, st, 1.0f);
        hop_dir2<1, +1>(a0, a1, in0, in1, Uin, nb, nb, st, 1.0f);
    }
    {
        const long long d = (long long)g.Lxh * g.L[1];
        const long long nf = LQ_IDX((c.z + 1 == g.L[2]) ? s - (long long)(g.L[2] - 1) * d : s + d, g.Vh, B_HOP_NB);
        const long long nb = LQ_IDX((c.z == 0) ? s + (long long)(g.L[2] - 1) * d : s - d, g.Vh, B_HOP_NB);
        hop_dir2<2, -1>(a0, a1, in0, in1, Uout, s, nf, st, 1.0f);
        hop_dir2<2, +1>(a0, a1, in0, in1, Uin, nb, nb, st, 1.0f);
    }
    {
        const long long d = (long long)g.Lxh * g.L[1] * g.L[2];
        const bool last = (c.t + 1 == g.L[3]), first = (c.t == 0);
        const long long nf = LQ_IDX(last ? s - (long long)(g.L[3] - 1) * d : s + d, g.Vh, B_HOP_NB);
        const long long nb = LQ_IDX(first ? s + (long long)(g.L[3] - 1) * d : s - d, g.Vh, B_HOP_NB);
        const float tb = (float)g.tbc;
        hop_dir2<3, -1>(a0, a1, in0, in1, Uout, s, nf, st, last ? tb : 1.0f);
        hop_dir2<3, +1>(a0, a1, in0, in1, Uin, nb, nb, st, first ? tb : 1.0f);
    }
    cx<float> v[12], x[12];
    if (MODE == HOP_K1) {
#pragma unroll
        for (int i = 0; i < 12; i++) a0[i] = -0.5f * sc0 * a0[i];
        clover_apply<float>(clov, st, s, a0, v);
        store_spinor(out0, st, s, v);
        if (two) {
#pragma unroll
            for (int i = 0; i < 12; i++) a1[i] = -0.5f * sc1 * a1[i];
            clover_apply<float>(clov, st, s, a1, v);
            store_spinor(out1, st, s, v);
        }
    } else {   // HOP_K2
        load_spinor_rw(in20, st, s, x);
        clover_apply<float>(clov, st, s, x, v);
#pragma unroll
        for (int i = 0; i < 12; i++) v[i] = sc0 * v[i] + 0.5f * a0[i];
        store_spinor(out0, st, s, v);
        if (two) {
            load_spinor_rw(in21, st, s, x);
            clover_apply<float>(clov, st, s, x, v);
#pragma unroll
            for (int i = 0; i < 12; i++) v[i] = sc1 * v[i] + 0.5f * a1[i];
            store_spinor(out1, st, s, v);
        }
    }
}

// The output site of a thread, and how many sites its warp has (its lanes from
// there on shadow the last one): with natural output a warp stays whole.
__device__ __forceinline__ long long warp_site(const Geom &g, int &nvalid)
{
    const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x, s0 = s - (threadIdx.x & 31);
    nvalid = (int)min(32LL, g.Vh - s0);
    return LQ_IDX(min(s, g.Vh - 1), g.Vh, B_HOP_SITE);
}
template <typename R, int MODE, bool NAT>
__device__ __forceinline__ void hop_site(const Geom &g, const HopArgs<R> &k)
{
    extern __shared__ __align__(16) double2 nat_tile[];
    int nv = 0;
    long long s;
    if (NAT) {
        s = warp_site(g, nv);
        if (nv <= 0) return;
    } else {
        s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        if (s >= g.Vh) return;
    }
    const Coords c = cb_coords(g, s, k.pout);
    double2 *tile = NAT ? nat_tile + (threadIdx.x >> 5) * 32 * kNatRow : nullptr;
    // links and clover read once: no L1 allocation
    hop_body<R, MODE, NAT>(g, (const F4S *)k.Uout, (const F4S *)k.Uin, (const F4S *)k.clov, k.omega, k.in, k.in2, k.b,
                           k.out, s, c, k.nat, tile, nv);
}
template <typename R, int MODE, bool NAT>
__global__ void LQ_HOP_BOUNDS hop_kernel(Geom g, HopArgs<R> k)
{
    after_previous();
    hop_site<R, MODE, NAT>(g, k);
}

// The same for FP32 K2 and its Richardson form, asked to fit six blocks per SM
// (80 registers, a few bytes of spills): measured on GB300 on 32^3 x 64, K2
// moves from 0.89 to 0.93 of the copy bandwidth this way, while K1 (78
// registers unbounded) gains nothing.
template <typename R, int MODE, bool NAT>
__global__ void __launch_bounds__(LQ_HOP_THREADS, 6) hop_kernel_occ(Geom g, HopArgs<R> k)
{
    after_previous();
    hop_site<R, MODE, NAT>(g, k);
}


// BF16 spinors and links, FP32 clover and arithmetic (K1, K2, Richardson)
struct HopArgsBF {
    const BfS4 *in, *in2, *b;
    BfS4 *out;
    const BfL2 *Uout, *Uin;
    const F4S *clov;   // FP32 clover blocks, read once
    float omega;
    int pout;
    NatOut nat;
};
template <int MODE, bool NAT>
__device__ __forceinline__ void hop_site_bf(const Geom &g, const HopArgsBF &k)
{
    extern __shared__ __align__(16) double2 nat_tile[];
    int nv = 0;
    long long s;
    if (NAT) {
        s = warp_site(g, nv);
        if (nv <= 0) return;
    } else {
        s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        if (s >= g.Vh) return;
    }
    const Coords c = cb_coords(g, s, k.pout);
    hop_body<float, MODE, NAT>(g, k.Uout, k.Uin, k.clov, k.omega, k.in, k.in2, k.b, k.out, s, c, k.nat,
                               NAT ? nat_tile + (threadIdx.x >> 5) * 32 * kNatRow : nullptr, nv);
}
template <int MODE>
__global__ void LQ_HOP_BOUNDS hop_kernel_bf(Geom g, HopArgsBF k)
{
    after_previous();
    hop_site_bf<MODE, false>(g, k);
}
// K2 with natural output: held to the registers of the plain one (104 without the bound)
__global__ void __launch_bounds__(LQ_HOP_THREADS, 6) hop_kernel_bf_nat(Geom g, HopArgsBF k)
{
    after_previous();
    hop_site_bf<HOP_K2, true>(g, k);
}

// shared memory of a block's natural output
constexpr size_t nat_smem(int threads) { return (size_t)threads * kNatRow * sizeof(double2); }
// the modes that end a call on natural fields (HOP_FULL always does)
constexpr bool nat_mode(int mode) { return mode == HOP_K2 || mode == HOP_FULL; }

template <int MODE>
static void launch_hop_bf(const Exec &e, const HopCall &c)
{
    HopArgsBF k;
    k.in = (const BfS4 *)c.in;
    k.in2 = (const BfS4 *)c.in2;
    k.b = (const BfS4 *)c.b;
    k.out = (BfS4 *)c.out;
    k.Uout = (const BfL2 *)c.U[c.pout];
    k.Uin = (const BfL2 *)c.U[1 - c.pout];
    k.clov = (const F4S *)c.clov;
    k.omega = (float)c.omega;
    k.pout = c.pout;
    k.nat = nat_out(e.g, c.nat, c.nat_full, c.nat_g5);
    const unsigned blocks = (unsigned)((e.g.Vh + LQ_HOP_THREADS - 1) / LQ_HOP_THREADS);
    // Blocks brought in early are not spread as evenly over the SMs, which costs more
    // than the gap between the launches while they are few.  D_S in us, overlapped and
    // not: 217 blocks 32.2 / 28.9, 288 33.0 / 30.7, 405 35.0 / 33.4, 512 37.2 / 37.1, 625
    // 39.7 / 42.2, 1000 55.1 / 58.2, 2592 112.5 / 118.
    const bool after = c.after && blocks > 512;
    if constexpr (MODE == HOP_K2)   // always natural (hop_refused)
        launch_after(e, after, hop_kernel_bf_nat, blocks, LQ_HOP_THREADS, nat_smem(LQ_HOP_THREADS), e.g, k);
    else
        launch_after(e, after, hop_kernel_bf<MODE>, blocks, LQ_HOP_THREADS, 0, e.g, k);
}

// The batched hop over the right-hand sides of several lattices of different
// sizes in one persistent launch: each block walks the work table, an entry
// naming a lattice, a block of blockDim.x consecutive sites and the first of
// blockDim.y right-hand sides.  Entries of the same sites follow one another, so
// a site's links and clover block reach L1/L2 once for all its right-hand sides.
#ifdef LQ_GROUP_MINB
#define LQ_GROUP_BOUNDS __launch_bounds__(LQ_HOP_THREADS, LQ_GROUP_MINB)
#else
#define LQ_GROUP_BOUNDS __launch_bounds__(LQ_HOP_THREADS)
#endif
// the factor of system r's input field (null: 1)
__device__ __forceinline__ float scale_of(const double *scale, int stride, int r)
{
    return scale ? (float)scale[(long long)r * stride] : 1.0f;
}
template <int MODE, int RPT>
__global__ void LQ_GROUP_BOUNDS hop_group_kernel(const LatDesc *__restrict__ d,
                                                                   const int4 *__restrict__ tiles, int ntiles,
                                                                   const float4 *in, const float4 *in2, float4 *out,
                                                                   const double *scale, int sstride)
{
    constexpr int pout = MODE == HOP_K1 ? 1 : 0;
    // consecutive entries, so that a site block's right-hand sides find its links in L1
    const int t0 = (int)((long long)ntiles * blockIdx.x / gridDim.x), t1 = (int)((long long)ntiles * (blockIdx.x + 1) / gridDim.x);
    for (int t = t0; t < t1; t++) {
        const int4 w = __ldg(tiles + t);
        const LatDesc *L = d + w.x;
        const Geom g = L->g;
        const long long s = (long long)w.y * blockDim.x + threadIdx.x;
        const int r = w.z + RPT * threadIdx.y;   // the thread's first right-hand side
        if (s >= g.Vh || r >= L->nrhs) continue;
        const Coords c = cb_coords(g, s, pout);
        const long long o = L->off + r * L->fs;
        const float sc = scale_of(scale, sstride, L->first + r);
        if (RPT == 1) {
            hop_body<float, MODE, false, true>(g, L->U[pout], L->U[1 - pout], L->clov[pout], sc, in + o,
                                               in2 ? in2 + o : nullptr, (const float4 *)nullptr, out + o, s, c);
        } else {
            // the second right-hand side, when it exists (else the first is read twice, stored once)
            const bool two = r + 1 < L->nrhs;
            const long long o1 = two ? o + L->fs : o;
            hop_body2<MODE>(g, L->U[pout], L->U[1 - pout], L->clov[pout], in + o, in + o1,
                            in2 ? in2 + o : nullptr, in2 ? in2 + o1 : nullptr, out + o, out + o1, two, s, c, sc,
                            two ? scale_of(scale, sstride, L->first + r + 1) : 0.0f);
        }
    }
}

// The batched hop with a site block's links and clover blocks staged in shared
// memory once for every right-hand side of its lattice.  A tile is (lattice,
// block of S consecutive sites); the block has S x (128 / S) threads, thread
// (x, y) owns site x of the block and walks right-hand sides y, y + 128/S, ...
// Staging: for every site of the block, the four forward links U_mu(x), the
// four backward links U_mu(x - mu) (read at the neighbour's index in the other
// parity's link array) and the two packed clover blocks of the output parity:
// 12 + 12 + 18 float4, laid out [entry][site] so that a warp's reads of one
// entry are consecutive.  The links and clover thus cross DRAM once per site,
// whatever the number of right-hand sides, and each right-hand side costs only
// its spinor traffic.
constexpr int kTileEntries = 42;   // float4 entries staged per site
constexpr int kTileFwd = 0, kTileBwd = 12, kTileClov = 24;

__device__ __forceinline__ void tile_link(const float4 *sm, int S, int e0, int x, cx<float> m[9])
{
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float4 t = sm[(e0 + k) * S + x];
        m[2 * k] = {t.x, t.y};
        m[2 * k + 1] = {t.z, t.w};
    }
    m[6] = cconj(cmul(m[1], m[5]) - cmul(m[2], m[4]));
    m[7] = cconj(cmul(m[2], m[3]) - cmul(m[0], m[5]));
    m[8] = cconj(cmul(m[0], m[4]) - cmul(m[1], m[3]));
}

// y = C x with both packed blocks of the site read from the staged entries
__device__ __forceinline__ void tile_clover(const float4 *sm, int S, int x, const cx<float> in[12], cx<float> y[12])
{
#pragma unroll
    for (int blk = 0; blk < 2; blk++) {
        float a[36];
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const float4 t = sm[(kTileClov + blk * 9 + k) * S + x];
            a[4 * k] = t.x;
            a[4 * k + 1] = t.y;
            a[4 * k + 2] = t.z;
            a[4 * k + 3] = t.w;
        }
        herm6_apply<float>(a, in + 6 * blk, y + 6 * blk);
    }
}

template <int MU, int SIGN>
__device__ __forceinline__ void tile_hop(cx<float> acc[12], const float4 *__restrict__ psi, long long st, int nb,
                                         const float4 *sm, int S, int x, float bsign)
{
    cx<float> p[12];
    load_spinor(psi, st, nb, p);
    cx<float> m[9];
    tile_link(sm, S, (SIGN < 0 ? kTileFwd : kTileBwd) + 3 * MU, x, m);
    hop_apply<MU, SIGN>(acc, p, m, bsign);
}

template <int MODE, int S>
__global__ void __launch_bounds__(LQ_HOP_THREADS, 5) hop_tile_kernel(const LatDesc *__restrict__ d,
                                                                     const int4 *__restrict__ tiles, int ntiles,
                                                                     const float4 *in, const float4 *in2, float4 *out,
                                                                     const double *scale, int sstride)
{
    static_assert(MODE == HOP_K1 || MODE == HOP_K2, "K1 or K2");
    constexpr int R = LQ_HOP_THREADS / S;   // right-hand-side lanes
    constexpr int pout = MODE == HOP_K1 ? 1 : 0;
    extern __shared__ float4 tile_sm[];
    // after the staged entries: the eight neighbour indices of each site and its
    // two time-boundary factors, [10][S] words (kept here rather than in
    // registers across the loop over right-hand sides)
    int *tile_nb = reinterpret_cast<int *>(tile_sm + kTileEntries * S);
    float *tile_bc = reinterpret_cast<float *>(tile_nb + 8 * S);
    const int x = threadIdx.x, y = threadIdx.y;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int4 w = __ldg(tiles + t);
        const LatDesc *L = d + w.x;
        const Geom g = L->g;
        const long long st = g.stride;
        const long long s = (long long)w.y * S + x;
        const bool valid = s < g.Vh;
        // neighbour checkerboard indices (forward, backward per direction) and
        // the time-boundary factors; Vh < 2^31, so they fit an int
        int nf[4], nb[4];
        float tf = 1.0f, tb = 1.0f;
        if (valid) {
            const Coords c = cb_coords(g, s, pout);
            const long long base = c.row * g.Lxh;
            const int xp = (c.x + 1 == g.L[0]) ? 0 : c.x + 1;
            const int xm = (c.x == 0) ? g.L[0] - 1 : c.x - 1;
            nf[0] = (int)LQ_IDX(base + (xp >> 1), g.Vh, B_TILE_NB);
            nb[0] = (int)LQ_IDX(base + (xm >> 1), g.Vh, B_TILE_NB);
            long long dd = g.Lxh;
            const int co[3] = {c.y, c.z, c.t};
#pragma unroll
            for (int mu = 1; mu < 4; mu++) {
                const int ext = g.L[mu], q = co[mu - 1];
                nf[mu] = (int)LQ_IDX((q + 1 == ext) ? s - (long long)(ext - 1) * dd : s + dd, g.Vh, B_TILE_NB);
                nb[mu] = (int)LQ_IDX((q == 0) ? s + (long long)(ext - 1) * dd : s - dd, g.Vh, B_TILE_NB);
                dd *= ext;
            }
            if (c.t + 1 == g.L[3]) tf = (float)g.tbc;
            if (c.t == 0) tb = (float)g.tbc;
        }
        __syncthreads();   // the previous tile's reads of the staged entries are done
        if (valid) {
            const F4S *Uo = (const F4S *)L->U[pout];
            const F4S *Ui = (const F4S *)L->U[1 - pout];
            const F4S *Cl = (const F4S *)L->clov[pout];
            for (int e = y; e < kTileEntries; e += R) {
                const F4S *src;
                if (e < kTileBwd) src = Uo + e * st + s;
                else if (e < kTileClov) {
                    const int mu = (e - kTileBwd) / 3;   // selected, not indexed: nb stays in registers
                    const int n = mu == 0 ? nb[0] : mu == 1 ? nb[1] : mu == 2 ? nb[2] : nb[3];
                    src = Ui + (long long)(e - kTileBwd) * st + n;
                } else {
                    src = Cl + (long long)(e - kTileClov) * st + s;
                }
                tile_sm[e * S + x] = ldg(src);
            }
            if (y == 0) {
#pragma unroll
                for (int mu = 0; mu < 4; mu++) {
                    tile_nb[(2 * mu) * S + x] = nf[mu];
                    tile_nb[(2 * mu + 1) * S + x] = nb[mu];
                }
                tile_bc[x] = tf;
                tile_bc[S + x] = tb;
            }
        }
        __syncthreads();
        if (!valid) continue;
        for (int r = y; r < L->nrhs; r += R) {
            const long long o = L->off + r * L->fs;
            const float4 *pin = in + o;
            cx<float> acc[12];
#pragma unroll
            for (int i = 0; i < 12; i++) acc[i] = {0.0f, 0.0f};
            tile_hop<0, -1>(acc, pin, st, tile_nb[0 * S + x], tile_sm, S, x, 1.0f);
            tile_hop<0, +1>(acc, pin, st, tile_nb[1 * S + x], tile_sm, S, x, 1.0f);
            tile_hop<1, -1>(acc, pin, st, tile_nb[2 * S + x], tile_sm, S, x, 1.0f);
            tile_hop<1, +1>(acc, pin, st, tile_nb[3 * S + x], tile_sm, S, x, 1.0f);
            tile_hop<2, -1>(acc, pin, st, tile_nb[4 * S + x], tile_sm, S, x, 1.0f);
            tile_hop<2, +1>(acc, pin, st, tile_nb[5 * S + x], tile_sm, S, x, 1.0f);
            tile_hop<3, -1>(acc, pin, st, tile_nb[6 * S + x], tile_sm, S, x, tile_bc[x]);
            tile_hop<3, +1>(acc, pin, st, tile_nb[7 * S + x], tile_sm, S, x, tile_bc[S + x]);
            cx<float> v[12];
            const float sc = scale_of(scale, sstride, L->first + r);
            if (MODE == HOP_K1) {
#pragma unroll
                for (int i = 0; i < 12; i++) acc[i] = -0.5f * sc * acc[i];
                tile_clover(tile_sm, S, x, acc, v);
            } else {
                cx<float> xs[12];
                load_spinor_rw(in2 + o, st, s, xs);
                tile_clover(tile_sm, S, x, xs, v);
#pragma unroll
                for (int i = 0; i < 12; i++) v[i] = sc * v[i] + 0.5f * acc[i];
            }
            store_spinor(out + o, st, s, v);
        }
    }
}

// ---------------------------------------------------------------------------
// df64 variant.  Each df64 operation is a chain of several FP32 instructions,
// so the fully unrolled eight-direction body of hop_kernel would not fit the
// instruction cache.  Here the eight hops share one loop body, the direction a
// table index of the spin projection and reconstruction (spin.cuh); the
// backward link enters as U^+.
// ---------------------------------------------------------------------------
// y += A x for one packed Hermitian 6x6 block A (reals 0..5 the diagonal,
// then the strictly lower entries), ld(k) its k-th vector, read as the product
// needs it; the six sums are lazily normalised (dl_*) and left unnormalised.
template <typename Ld>
__device__ __forceinline__ void herm6_fma_df(Ld ld, const cx<df64> x[6], cx<df64> y[6])
{
#pragma unroll
    for (int k = 0; k < 3; k++) {   // the diagonal: reals 2k, 2k+1
        const df2 t = ld(k);
        df64x2 y0 = dl2(y[2 * k]), y1 = dl2(y[2 * k + 1]);
        dl2_fma(y0, dl2_both(df64(t.rh, t.rl)), dl2(x[2 * k]));
        dl2_fma(y1, dl2_both(df64(t.ih, t.il)), dl2(x[2 * k + 1]));
        y[2 * k] = dl2_cx(y0);
        y[2 * k + 1] = dl2_cx(y1);
    }
    // the lower entries l_ij and their conjugates above the diagonal: the real
    // parts' products go straight into y, the imaginary parts' into z, whose
    // parts are exchanged once at the end
    df64x2 z[6];
#pragma unroll
    for (int i = 1; i < 6; i++)
#pragma unroll
        for (int j = 0; j < i; j++) {
            const cx<df64> l = df2_cx(ld(3 + tri(i, j)));
            const df64x2 re = dl2_both(l.re), im = dl2_both(l.im), xi = dl2(x[i]), xj = dl2(x[j]);
            df64x2 yi = dl2(y[i]), yj = dl2(y[j]);
            dl2_fma(yi, re, xj);
            dl2_fma(yj, re, xi);
            y[i] = dl2_cx(yi);
            y[j] = dl2_cx(yj);
            if (j == 0) z[i] = dl2_prod(im, xj);
            else dl2_fma(z[i], im, xj);
            const df64x2 mi = dl2_both(dl_neg(l.im));
            if (i == 1) z[j] = dl2_prod(mi, xi);
            else dl2_fma(z[j], mi, xi);
        }
#pragma unroll
    for (int i = 0; i < 6; i++) {
        df64x2 yi = dl2(y[i]);
        dl2_add(yi, dlrow_rot({yi, z[i]}));
        y[i] = dl2_cx(yi);
    }
}

// Operands staged ahead of their use (below): vectors of 16 bytes per thread,
// each thread reading only what it copied itself.
constexpr int kDfPsi = 0;        // the neighbour's 12 components
constexpr int kDfLink = 12;      // two buffers of 9 link entries
constexpr int kDfVecs = 30;
constexpr int kDfSites = LQ_HOP_THREADS / 2;   // sites of a block: two threads each
// a use of v that the compiler keeps before the copies that follow
__device__ __forceinline__ void used(cx<df64> v) { asm volatile("" ::"f"(v.re.hi), "f"(v.re.lo), "f"(v.im.hi), "f"(v.im.lo) : "memory"); }

// IO, how the fields stand: the output natural (kNat), the neighbours' field in
// FP32 (kIn32: its values are exact in df64, and a site reads half the bytes), the
// output rounded to FP32 (kOut32)
constexpr int kNat = 1, kIn32 = 2, kOut32 = 4;
template <int MODE, int IO>
__device__ __forceinline__ void hop_df_body(const Geom &g, const HopArgs<df64> &k, const df2 *in, const df2 *in2,
                                            const df2 *bv, df2 *out, df2 *out2, long long s, const Coords &c,
                                            float4 *stage, int nvalid)
{
    // The directions run through one loop body (the tables of spin.cuh).  The
    // neighbour's components and the link's entries are read as the
    // projection and the product use them, and every sum is lazily normalised
    // (dl_*): the two halves' sums are added and renormalised once.
    const long long st = g.stride;
    const int half = threadIdx.x / kDfSites, d0 = 4 * half, d1 = d0 + 4;
    const bool on = (int)(threadIdx.x & 31) < nvalid;   // shadowing lanes store nothing
    cx<df64> acc[12];
#pragma unroll
    for (int i = 0; i < 12; i++) acc[i] = {df64(0.0f, 0.0f), df64(0.0f, 0.0f)};

    // the neighbour in direction d, and whether the time boundary flips the hop's sign
    auto neighbour = [&](int d, bool &flip) {
        const long long nb = hop_neighbour(g, c, s, d, flip, B_DF_NB);
        flip = flip && g.tbc < 0;
        return nb;
    };

    // The kernel waits on its loads, not on its arithmetic, when each direction
    // reads its operands as it comes to them (long scoreboard the first stall,
    // the FMA pipe 60% busy at 12 warps an SM).  So they are copied to shared
    // memory ahead: the links of direction d + 1 while d runs (two buffers),
    // the neighbour of d + 1 as soon as d is projected, and the clover block
    // while the last direction is multiplied.
    auto vec = [&](int e) {
        const float4 t = stage[e * LQ_HOP_THREADS];
        return cx<df64>{df64(t.x, t.z), df64(t.y, t.w)};
    };
    auto copy_psi = [&](long long nb) {
#pragma unroll
        for (int e = 0; e < (IO & kIn32 ? 6 : 12); e++) copy_async(stage + (kDfPsi + e) * LQ_HOP_THREADS, in + nb + e * st);
        copy_commit();
    };
    auto psi = [&](int e) {   // component e of the neighbour
        if (!(IO & kIn32)) return vec(kDfPsi + e);
        const float4 t = stage[(kDfPsi + (e >> 1)) * LQ_HOP_THREADS];
        return cx<df64>{df64(e & 1 ? t.z : t.x, 0.0f), df64(e & 1 ? t.w : t.y, 0.0f)};
    };
    auto copy_link = [&](int d, long long nb) {
        const bool fwd = (d & 1) == 0;
        const df2 *Um = (fwd ? k.Uout : k.Uin) + (long long)(d >> 1) * 9 * st + (fwd ? s : nb);
#pragma unroll
        for (int e = 0; e < 9; e++) copy_async(stage + (kDfLink + (d & 1) * 9 + e) * LQ_HOP_THREADS, Um + e * st);
        copy_commit();
    };
    bool flip;
    long long nb = neighbour(d0, flip);
    copy_link(d0, nb);
    copy_psi(nb);
#pragma unroll 1
    for (int d = d0; d < d1; d++) {
        const bool fwd = (d & 1) == 0;
        bool flip1 = false;
        const long long nb1 = d + 1 < d1 ? neighbour(d + 1, flip1) : 0;
#pragma unroll
        for (int a = 0; a < 3; a++) used(acc[a]);   // the last direction's link entries are used up
        if (d + 1 < d1) {
            copy_link(d + 1, nb1);
            copy_wait<1>();
        } else {
            copy_wait<0>();
        }
        const int pa = d < 4 ? 3 : 2;
        const int qa = (kHopQA >> (2 * d)) & 3, qb = (kHopQB >> (2 * d)) & 3;
        cx<df64> h[6];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            h[a] = psi(a);
            dl_cadd(h[a], rot_i(psi(pa == 3 ? 9 + a : 6 + a), qa));
            h[3 + a] = psi(3 + a);
            dl_cadd(h[3 + a], rot_i(psi(pa == 3 ? 6 + a : 9 + a), qb));
        }
#pragma unroll
        for (int a = 0; a < 6; a++) used(h[a]);
        if (d + 1 < d1) {
            copy_psi(nb1);
        } else if (MODE != HOP_PREP) {   // the clover block, over the neighbour and the free link buffer
#pragma unroll
            for (int e = 0; e < 18; e++) copy_async(stage + e * LQ_HOP_THREADS, k.clov + (18 * half + e) * st + s);
            copy_commit();
        }
        const int ra = d < 4 ? 1 : 0;
        const int qc = (kHopQC >> (2 * d)) & 3, qd = (kHopQD >> (2 * d)) & 3;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            // row a of U (forward) or of U^+ (backward): entries m[a*3+b] or conj(m[b*3+a])
            cx<df64> e[3];
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const cx<df64> t = vec(kDfLink + (d & 1) * 9 + (fwd ? a * 3 + b : b * 3 + a));
                e[b] = fwd ? t : cx<df64>{t.re, dl_neg(t.im)};
            }
            dlrow r0 = dlrow_prod(e[0], dl2(h[0])), r1 = dlrow_prod(e[0], dl2(h[3]));
            dlrow_fma(r0, e[1], dl2(h[1]));
            dlrow_fma(r1, e[1], dl2(h[4]));
            dlrow_fma(r0, e[2], dl2(h[2]));
            dlrow_fma(r1, e[2], dl2(h[5]));
            dl2_add(r0.r, dlrow_rot(r0));
            dl2_add(r1.r, dlrow_rot(r1));
            cx<df64> u0 = dl2_cx(r0.r), u1 = dl2_cx(r1.r);
            if (flip) {
                u0 = {dl_neg(u0.re), dl_neg(u0.im)};
                u1 = {dl_neg(u1.re), dl_neg(u1.im)};
            }
            dl_cadd(acc[a], u0);
            dl_cadd(acc[3 + a], u1);
            dl_cadd(acc[6 + a], rot_i(ra ? u1 : u0, qc));
            dl_cadd(acc[9 + a], rot_i(ra ? u0 : u1, qd));
        }
        nb = nb1;
        flip = flip1;
    }
    // each half hands the other its sums of the other's spins, through the second
    // link buffer, which the last direction has left
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const cx<df64> v = half ? acc[i] : acc[6 + i];
        stage[(kDfLink + 9 + i) * LQ_HOP_THREADS] = make_float4(v.re.hi, v.im.hi, v.re.lo, v.im.lo);
    }
    __syncthreads();
    cx<df64> a6[6], y[6];
    const float4 *other = stage + (half ? -kDfSites : kDfSites);
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const float4 t = other[(kDfLink + 9 + i) * LQ_HOP_THREADS];
        a6[i] = half ? acc[6 + i] : acc[i];
        dl_cadd(a6[i], {df64(t.x, t.z), df64(t.y, t.w)});
        a6[i] = dl_cnorm(a6[i]);
    }
    if (MODE != HOP_PREP) copy_wait<0>();

    // the site term of the half's two spins, one 6x6 clover block
    const long long o = (long long)half * 6 * st + s;
    auto Cb = [&](int e) {   // vector e of the clover block
        const float4 t = stage[e * LQ_HOP_THREADS];
        return df2(t.x, t.z, t.y, t.w);
    };
    if (MODE == HOP_K1) {   // y = C (-1/2 acc)
#pragma unroll
        for (int i = 0; i < 6; i++) {
            a6[i] = {dl_scale2(a6[i].re, -0.5f), dl_scale2(a6[i].im, -0.5f)};
            y[i] = {df64(0.0f, 0.0f), df64(0.0f, 0.0f)};
        }
        herm6_fma_df(Cb, a6, y);
#pragma unroll
        for (int i = 0; i < 6; i++) y[i] = dl_cnorm(y[i]);
    } else if (MODE == HOP_K2 || MODE == HOP_RICH || MODE == HOP_FULL || MODE == HOP_RES) {   // y = C x +- 1/2 acc
        const float f = (MODE == HOP_FULL || MODE == HOP_RES) ? -0.5f : 0.5f;
        cx<df64> x6[6];
#pragma unroll
        for (int i = 0; i < 6; i++) {
            x6[i] = df2_cx(in2[o + i * st]);
            y[i] = {dl_scale2(a6[i].re, f), dl_scale2(a6[i].im, f)};
        }
        herm6_fma_df(Cb, x6, y);
#pragma unroll
        for (int i = 0; i < 6; i++) y[i] = dl_cnorm(y[i]);
        if (MODE == HOP_RICH) {   // x + omega (b - D x)
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = x6[i] + k.omega * (df2_cx(ldg(bv + o + i * st)) - y[i]);
        }
        if (MODE == HOP_RES) {   // b - D x
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = df2_cx(ldg(bv + o + i * st)) - y[i];
        }
    } else {   // y = in2 + 1/2 acc, and for the reconstruction C^{-1} of that
#pragma unroll
        for (int i = 0; i < 6; i++) {
            cx<df64> t = df2_cx(in2[o + i * st]);
            dl_cadd(t, {dl_scale2(a6[i].re, 0.5f), dl_scale2(a6[i].im, 0.5f)});
            a6[i] = dl_cnorm(t);
        }
        if (MODE == HOP_RECON || MODE == HOP_RECON_RES) {
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = {df64(0.0f, 0.0f), df64(0.0f, 0.0f)};
            herm6_fma_df(Cb, a6, y);
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = dl_cnorm(y[i]);
            if (MODE == HOP_RECON_RES) {   // the parity's residual u - C x_o of the x_o just formed
                cx<df64> z[6];
#pragma unroll
                for (int i = 0; i < 6; i++) z[i] = {df64(0.0f, 0.0f), df64(0.0f, 0.0f)};
                herm6_fma_df([&](int e) { return ldg(k.clov2 + ((long long)half * 18 + e) * st + s); }, y, z);
#pragma unroll
                for (int i = 0; i < 6; i++)
                    if (on) out2[o + i * st] = cx_df2(a6[i] - dl_cnorm(z[i]));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = a6[i];
        }
    }
    if (IO & kNat) {
        // through the vectors that the clover block has left (each
        // lane's column turned by the component, against bank conflicts)
        const int lane = threadIdx.x & 31;
        double2 *tile = reinterpret_cast<double2 *>(stage - lane);
        auto at = [](int r, int q) { return q * LQ_HOP_THREADS + ((r + q) & 31); };
        const unsigned flip = half ? k.nat.flip : 0u;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const double2 d = nat_value((const df2 *)nullptr, y[i]);
            tile[at(lane, i)] = make_double2(flip_sign64(d.x, flip), flip_sign64(d.y, flip));
        }
        __syncwarp();
        nat_write6(k.nat, tile, at, s - min(lane, nvalid - 1), nvalid, c.x & 1, half);
    } else if (IO & kOut32) {
        float4 *f = reinterpret_cast<float4 *>(out) + (long long)half * 3 * st + s;
#pragma unroll
        for (int i = 0; i < 3; i++)
            if (on) f[i * st] = make_float4(df_to_float(y[2 * i].re), df_to_float(y[2 * i].im), df_to_float(y[2 * i + 1].re),
                                    df_to_float(y[2 * i + 1].im));
    } else {
#pragma unroll
        for (int i = 0; i < 6; i++)
            if (on) out[o + i * st] = cx_df2(y[i]);
    }
}

// Two threads per output site and right-hand side: the first takes the directions
// along x and y and the site term of spins 0 and 1, the second those along z and t
// and spins 2 and 3.  One thread's chain is half as long so, which a lattice of
// about one wave of blocks waits for, and the sums need fewer registers: lq_apply of
// D_S takes 45.7 us on 18x10x14x22 and 350 on 24^3 x 48, against 56.3 and 367 with
// one thread a site (whose K1 / K2 took 158 / 171 us on 24^3 x 48, 187 / 193 before
// the staging and 214 / 215 with scalar arithmetic).  Three resident blocks per SM
// (61 KB of staging each).  The right-hand sides of a site block are consecutive
// blocks, so its links and clover come from L2 for all but the first.
#ifndef LQ_DF_MINB
#define LQ_DF_MINB 3
#endif
template <int MODE, int IO>
__global__ void __launch_bounds__(LQ_HOP_THREADS, LQ_DF_MINB) hop_df_kernel(const __grid_constant__ Geom g,
                                                                const __grid_constant__ HopArgs<df64> k)
{
    extern __shared__ float4 df_stage[];
    after_previous();
    const unsigned sb = blockIdx.x / (unsigned)k.nrhs;
    // blocks stay whole: threads beyond the last site shadow it
    long long s = sb * (long long)kDfSites + threadIdx.x % kDfSites;
    const int nv = (int)min(32LL, g.Vh - (s - (threadIdx.x & 31)));
    s = LQ_IDX(min(s, g.Vh - 1), g.Vh, B_HOP_SITE);
    const Coords c = cb_coords(g, s, k.pout);
    const long long o = (blockIdx.x - sb * k.nrhs) * k.fs;
    hop_df_body<MODE, IO>(g, k, k.in + o, k.in2 ? k.in2 + o : nullptr, k.b ? k.b + o : nullptr, k.out + o,
                           k.out2 ? k.out2 + o : nullptr, s, c, df_stage + threadIdx.x, nv);
}

// one parity's FP32 field as its rows of a natural full field
__global__ void __launch_bounds__(LQ_HOP_THREADS) export_parity_kernel(Geom g, const float4 *f, int parity, NatOut nat)
{
    extern __shared__ __align__(16) double2 nat_tile[];
    int nv;
    const long long s = warp_site(g, nv);
    if (nv <= 0) return;
    cx<float> v[12];
    load_spinor_rw(f, g.stride, s, v);
    store_nat(nat, nat_tile + (threadIdx.x >> 5) * 32 * kNatRow, f, s - min((int)(threadIdx.x & 31), nv - 1), nv,
              cb_coords(g, s, parity).x & 1, v);
}
void export_parity(const Exec &e, const void *f, int parity, void *nat)
{
    Launch L_(e, K_LAYOUT, (double)e.g.Vh * (96 + 192));
    const NatOut o = nat_out(e.g, nat, true, false);
    export_parity_kernel<<<(unsigned)((e.g.Vh + LQ_HOP_THREADS - 1) / LQ_HOP_THREADS), LQ_HOP_THREADS,
                           nat_smem(LQ_HOP_THREADS), e.st>>>(e.g, (const float4 *)f, parity, o);
}

template <typename R>
__global__ void __launch_bounds__(256) clover_mul_kernel(Geom g, const typename St<R>::vec *__restrict__ C,
                                                         const typename St<R>::vec *in, typename St<R>::vec *out)
{
    const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (s >= g.Vh) return;
    in += blockIdx.y * St<R>::SPINOR_VECS * g.stride;
    out += blockIdx.y * St<R>::SPINOR_VECS * g.stride;
    cx<R> x[12], y[12];
    load_spinor_rw(in, g.stride, s, x);
    clover_apply<R>(C, g.stride, s, x, y);
    store_spinor(out, g.stride, s, y);
}

template <typename R, int MODE>
static void launch_hop(const Exec &e, const HopCall &c)
{
    typedef typename St<R>::vec V;
    HopArgs<R> k;
    k.in = (const V *)c.in;
    k.in2 = (const V *)c.in2;
    k.b = (const V *)c.b;
    k.out = (V *)c.out;
    k.Uout = (const V *)c.U[c.pout];
    k.Uin = (const V *)c.U[1 - c.pout];
    k.clov = (const V *)c.clov;
    k.clov2 = (const V *)c.clov2;
    k.out2 = (V *)c.out2;
    k.omega = R(c.omega);
    k.pout = c.pout;
    k.nrhs = c.nrhs;
    k.fs = (long long)St<R>::SPINOR_VECS * e.g.stride;
    constexpr int threads = LQ_HOP_THREADS, sites = std::is_same<R, df64>::value ? kDfSites : threads;   // of a block
    const unsigned blocks = (unsigned)((e.g.Vh + sites - 1) / sites);
    k.nat = nat_out(e.g, c.nat, c.nat_full, c.nat_g5);
    if constexpr (std::is_same<R, df64>::value)
    {
        constexpr int sm = kDfVecs * LQ_HOP_THREADS * (int)sizeof(float4);
        auto launch = [&](auto io) {
            auto kernel = hop_df_kernel<MODE, decltype(io)::value>;
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
            launch_after(e, c.after, kernel, blocks * (unsigned)c.nrhs, LQ_HOP_THREADS, sm, e.g, k);
        };
        if constexpr (MODE == HOP_PREP)
            if (c.out32) return launch(std::integral_constant<int, kOut32>());
        if constexpr (MODE == HOP_RECON)
            if (c.in32) return launch(std::integral_constant<int, kNat | kIn32>());
        if constexpr (nat_mode(MODE))
            if (MODE == HOP_FULL || c.nat) return launch(std::integral_constant<int, kNat>());
        if constexpr (MODE != HOP_FULL) launch(std::integral_constant<int, 0>());
    }
    else
    {
        // several right-hand sides of FP32 fields: one launch each (the batched
        // solve uses the work-table kernel instead)
        for (int r = 0; r < c.nrhs; r++) {
            HopArgs<R> kr = k;
            const long long o = r * k.fs;
            kr.in = k.in + o;
            kr.in2 = k.in2 ? k.in2 + o : nullptr;
            kr.b = k.b ? k.b + o : nullptr;
            kr.out = k.out + o;
            const size_t sm = c.nat || MODE == HOP_FULL ? nat_smem(threads) : 0;
            auto launch = [&](auto nat) {
                constexpr bool NAT = decltype(nat)::value;
                if constexpr (std::is_same<R, float>::value && (MODE == HOP_K2 || MODE == HOP_RICH))
                    launch_after(e, c.after, hop_kernel_occ<R, MODE, NAT>, blocks, threads, sm, e.g, kr);
                else
                    launch_after(e, c.after, hop_kernel<R, MODE, NAT>, blocks, threads, sm, e.g, kr);
            };
            if constexpr (MODE == HOP_FULL) {
                launch(std::true_type());
            } else if constexpr (nat_mode(MODE)) {
                if (c.nat) launch(std::true_type());
                else launch(std::false_type());
            } else {
                launch(std::false_type());
            }
        }
    }
}

// algorithmic bytes per output site of one hopping launch (FP64 and df64 share
// the 8-byte-per-real layout)
static double hop_site_bytes(int mode, int prec, int nrhs)
{
    const bool wide = prec == P64 || prec == PDF;
    const double sp = wide ? 192.0 : prec == P16 ? 48.0 : 96.0;   // spinor
    const double lk = wide ? 144.0 : prec == P16 ? 24.0 : 48.0;   // link (18 / 12 reals)
    const double cl = wide ? 576.0 : 288.0;                       // 72-real clover pair (FP32 for BF16)
    double once = 8 * lk, per = sp + sp;            // links; neighbours and output per rhs
    switch (mode) {
    case HOP_K1: once += cl; break;
    case HOP_K2: case HOP_FULL: once += cl; per += sp; break;
    case HOP_RICH: once += cl; per += 2 * sp; break;
    case HOP_PREP: per += sp; break;
    case HOP_RECON: once += cl; per += sp; break;
    case HOP_RES: once += cl; per += 2 * sp; break;                  // x, b
    case HOP_RECON_RES: once += 2 * cl; per += 2 * sp; break;        // C^{-1} and C; b in, x and r out
    }
    return once + nrhs * per;
}

static int hop_class(int mode, int prec)
{
    if (prec == P16) return mode == HOP_K1 ? K_HOP_K1_BF16 : (mode == HOP_K2 || mode == HOP_RICH) ? K_HOP_K2_BF16 : K_HOP_OTHER;
    if (mode == HOP_K1) return prec == P64 ? K_HOP_K1_F64 : prec == P32 ? K_HOP_K1_F32 : K_HOP_K1_DF;
    if (mode == HOP_K2 || mode == HOP_RICH) return prec == P64 ? K_HOP_K2_F64 : prec == P32 ? K_HOP_K2_F32 : K_HOP_K2_DF;
    return K_HOP_OTHER;
}

// algorithmic flops per site: 1320 for the eight hops (projection 12, two
// SU(3) mat-vecs 132, accumulation 24, per direction, less the first
// accumulation), 552 per clover-block pair, 24 per spinor add / scale
static const double c_hop_flops[8] = {1320 + 552, 1320 + 552 + 24, 1320 + 552 + 24 + 48,
                                      1320 + 552 + 24, 1320 + 24, 1320 + 24 + 552,
                                      1320 + 552 + 48, 1320 + 24 + 2 * 552 + 24};

double hop_bytes(int mode, int prec, int nrhs, double sites) { return sites * hop_site_bytes(mode, prec, nrhs); }
double hop_flops(int mode, double site_rhs) { return site_rhs * c_hop_flops[mode]; }

// dynamic shared memory of the staged batched hop with S sites per tile
static size_t tile_smem(int S) { return (size_t)kTileEntries * S * sizeof(float4) + 10 * S * sizeof(int); }

int hop_group_resident(int rpt, int spt)
{
    int a = 0, b = 0;
    if (rpt == 0) {
        if (spt == 64) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hop_tile_kernel<HOP_K1, 64>, LQ_HOP_THREADS, tile_smem(64));
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, hop_tile_kernel<HOP_K2, 64>, LQ_HOP_THREADS, tile_smem(64));
        } else {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hop_tile_kernel<HOP_K1, 32>, LQ_HOP_THREADS, tile_smem(32));
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, hop_tile_kernel<HOP_K2, 32>, LQ_HOP_THREADS, tile_smem(32));
        }
    } else if (rpt == 2) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hop_group_kernel<HOP_K1, 2>, LQ_HOP_THREADS, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, hop_group_kernel<HOP_K2, 2>, LQ_HOP_THREADS, 0);
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hop_group_kernel<HOP_K1, 1>, LQ_HOP_THREADS, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, hop_group_kernel<HOP_K2, 1>, LQ_HOP_THREADS, 0);
    }
    const int r = a < b ? a : b;
    return r < 1 ? 1 : r;
}

void hop_group(const Exec &e, int mode, const LatDesc *desc, const int4 *tiles, int ntiles, int grid, int spt,
               int rpt, const void *in, const void *in2, void *out, const double *scale, int sstride, double bytes,
               double flops)
{
    Launch L_(e, mode == HOP_K1 ? K_HOP_K1_F32 : K_HOP_K2_F32, bytes, flops);
    const dim3 block(spt, LQ_HOP_THREADS / spt);
    const float4 *i1 = (const float4 *)in, *i2 = (const float4 *)in2;
    float4 *o = (float4 *)out;
    if (rpt == 0) {   // staged links and clover, every right-hand side of the tile's lattice
        const size_t sm = tile_smem(spt);
        if (spt == 64) {
            if (mode == HOP_K1) hop_tile_kernel<HOP_K1, 64><<<grid, block, sm, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
            else hop_tile_kernel<HOP_K2, 64><<<grid, block, sm, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
        } else {
            if (mode == HOP_K1) hop_tile_kernel<HOP_K1, 32><<<grid, block, sm, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
            else hop_tile_kernel<HOP_K2, 32><<<grid, block, sm, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
        }
        return;
    }
    if (mode == HOP_K1 && rpt == 2) hop_group_kernel<HOP_K1, 2><<<grid, block, 0, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
    else if (mode == HOP_K1) hop_group_kernel<HOP_K1, 1><<<grid, block, 0, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
    else if (rpt == 2) hop_group_kernel<HOP_K2, 2><<<grid, block, 0, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
    else hop_group_kernel<HOP_K2, 1><<<grid, block, 0, e.st>>>(desc, tiles, ntiles, i1, i2, o, scale, sstride);
}

template <int MODE>
static void launch_mode(const Exec &e, const HopCall &c)
{
    if (c.prec == PDF) return launch_hop<df64, MODE>(e, c);
    if constexpr (hop_form(MODE, P32))
        if (c.prec == P32) return launch_hop<float, MODE>(e, c);
    if constexpr (hop_form(MODE, P16))
        if (c.prec == P16) return launch_hop_bf<MODE>(e, c);
}

void hop(const Exec &e, const HopCall &c)
{
    if (const char *why = hop_refused(e.g, c)) throw Refused{why};
    // df64 and FP64 take all right-hand sides in one launch (links and clover
    // counted once for df64); FP32 launches once per right-hand side
    const double site_bytes = c.prec == PDF ? hop_site_bytes(c.mode, c.prec, c.nrhs)
                                            : c.nrhs * hop_site_bytes(c.mode, c.prec, 1);
    // natural rows are complex doubles whatever the precision
    const double nat_bytes = (c.nat ? 192.0 - (double)spinor_bytes(e.g, c.prec) / e.g.stride : 0.0) -
                             96.0 * (c.in32 + c.out32);
    Launch L_(e, hop_class(c.mode, c.prec), (double)e.g.Vh * (site_bytes + nat_bytes), (double)e.g.Vh * c_hop_flops[c.mode] * c.nrhs);
    if (hop_split(e, c)) return;
    if (c.prec == P64) return hop_f64(e, c);
    switch (c.mode) {
    case HOP_K1: launch_mode<HOP_K1>(e, c); break;
    case HOP_K2: launch_mode<HOP_K2>(e, c); break;
    case HOP_RICH: launch_mode<HOP_RICH>(e, c); break;
    case HOP_FULL: launch_mode<HOP_FULL>(e, c); break;
    case HOP_PREP: launch_mode<HOP_PREP>(e, c); break;
    case HOP_RECON: launch_mode<HOP_RECON>(e, c); break;
    case HOP_RES: launch_mode<HOP_RES>(e, c); break;
    case HOP_RECON_RES: launch_mode<HOP_RECON_RES>(e, c); break;
    }
}

void clover_mul(const Exec &e, int prec, const void *clov, const void *in, void *out, int nfields)
{
    if (prec == P16) throw Refused{"no clover multiply of BF16 fields"};
    Launch L_(e, K_HOP_OTHER,
              (double)e.g.Vh * (prec != P32 ? nfields * 192.0 * 2 + 576.0 : nfields * 96.0 * 2 + 288.0),
              (double)e.g.Vh * nfields * 552);
    const dim3 blocks((unsigned)((e.g.Vh + 255) / 256), nfields);
    if (prec == P64)
        clover_mul_kernel<double><<<blocks, 256, 0, e.st>>>(e.g, (const double2 *)clov, (const double2 *)in,
                                                           (double2 *)out);
    else if (prec == P32)
        clover_mul_kernel<float><<<blocks, 256, 0, e.st>>>(e.g, (const float4 *)clov, (const float4 *)in,
                                                          (float4 *)out);
    else
        clover_mul_kernel<df64><<<blocks, 256, 0, e.st>>>(e.g, (const df2 *)clov, (const df2 *)in, (df2 *)out);
}

}  // namespace lq
