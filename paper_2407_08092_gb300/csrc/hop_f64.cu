// The hopping kernels in native FP64, for the lattices beyond hop_split's sizes.
//
// The FP64 pipe is the bound: 1128 instructions a site at two lanes a clock and SM.
// Two threads per output site keep it fed: the first takes the directions along x
// and y and the site term of spins 0 and 1, the second those along z and t and
// spins 2 and 3; they hand each other the sums of the other's spins.  A block is
// the two warps of 32 sites, so that the sites spread evenly over the SMs.  D on
// 16^3 x 32 takes 287 us (1.9 of the two lanes busy) at eight blocks an SM (128
// registers), 288 at ten and unbounded seven, 333 with one thread a site and 344
// with blocks of 128 such threads; D_S on 12^3 x 16 70 us, 89 with one thread.
#include "lq_kernels.h"
#include "nat.cuh"
#include "spin.cuh"

namespace lq {

constexpr int kF64Sites = 32, kF64Blocks = 8;   // sites of a block, blocks of an SM

struct F64Args {
    const double2 *in, *in2, *b;
    double2 *out, *out2;
    const double2 *Uout, *Uin, *clov, *clov2;
    double omega;
    int pout, nrhs;
    long long fs;
    NatOut nat;
};

// one hop of direction D = 2 mu + (backward), as hop_dir of the other precisions
template <int D, bool FIRST>
__device__ __forceinline__ void hop_one(const Geom &g, const F64Args &k, const double2 *in, long long s, const Coords &c,
                                        cx<double> acc[12])
{
    constexpr int MU = D >> 1, SIGN = (D & 1) ? +1 : -1;
    bool cross;
    const long long nb = hop_neighbour(g, c, s, D, cross, B_HOP_NB);
    cx<double> p[12], m[9];
    load_spinor_rw(in, g.stride, nb, p);
    load_link(SIGN < 0 ? k.Uout : k.Uin, g.stride, MU, SIGN < 0 ? s : nb, m);
    hop_apply<MU, SIGN, FIRST>(acc, p, m, MU == 3 && cross ? (double)g.tbc : 1.0);
}

template <int MODE, bool NAT>
__global__ void __launch_bounds__(2 * kF64Sites, kF64Blocks) hop_f64_kernel(const __grid_constant__ Geom g,
                                                               const __grid_constant__ F64Args k)
{
    __shared__ double2 handed[2][6][kF64Sites];
    __shared__ double2 tile[2][NAT ? kF64Sites * 7 : 1];
    after_previous();
    const int lane = threadIdx.x & 31, half = threadIdx.x >> 5;
    const unsigned sb = blockIdx.x / (unsigned)k.nrhs;
    const long long o = (blockIdx.x - sb * k.nrhs) * k.fs, st = g.stride;
    const long long s0 = sb * (long long)kF64Sites;
    const int nv = (int)min((long long)kF64Sites, g.Vh - s0);
    const long long s = LQ_IDX(s0 + min(lane, nv - 1), g.Vh, B_HOP_SITE);   // lanes beyond the last site shadow it
    const bool on = lane < nv;
    const Coords c = cb_coords(g, s, k.pout);

    cx<double> acc[12];
    if (half == 0) {
        hop_one<0, true>(g, k, k.in + o, s, c, acc);
        hop_one<1, false>(g, k, k.in + o, s, c, acc);
        hop_one<2, false>(g, k, k.in + o, s, c, acc);
        hop_one<3, false>(g, k, k.in + o, s, c, acc);
    } else {
        hop_one<4, true>(g, k, k.in + o, s, c, acc);
        hop_one<5, false>(g, k, k.in + o, s, c, acc);
        hop_one<6, false>(g, k, k.in + o, s, c, acc);
        hop_one<7, false>(g, k, k.in + o, s, c, acc);
    }
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const cx<double> v = half ? acc[i] : acc[6 + i];
        handed[half][i][lane] = make_double2(v.re, v.im);
    }
    __syncthreads();
    cx<double> a6[6], y[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const double2 t = handed[1 - half][i][lane];
        a6[i] = (half ? acc[6 + i] : acc[i]) + cx<double>{t.x, t.y};
    }

    // the site term of the half's two spins, one 6x6 clover block
    const long long q = o + (long long)half * 6 * st + s;
    double C[36];
    if (MODE != HOP_PREP) load_block(k.clov, st, half, s, C);
    auto load6 = [&](const double2 *f, cx<double> x[6]) {
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const double2 t = f[q + i * st];
            x[i] = {t.x, t.y};
        }
    };
    auto store6 = [&](double2 *f, const cx<double> x[6]) {
#pragma unroll
        for (int i = 0; i < 6; i++)
            if (on) f[q + i * st] = make_double2(x[i].re, x[i].im);
    };
    if (MODE == HOP_K1) {
#pragma unroll
        for (int i = 0; i < 6; i++) a6[i] = -0.5 * a6[i];
        herm6_apply<double>(C, a6, y);
    } else if (MODE == HOP_K2 || MODE == HOP_RICH || MODE == HOP_FULL || MODE == HOP_RES) {
        const double f = (MODE == HOP_FULL || MODE == HOP_RES) ? -0.5 : 0.5;
        cx<double> x[6], b[6];
        load6(k.in2, x);
        herm6_apply<double>(C, x, y);
#pragma unroll
        for (int i = 0; i < 6; i++) y[i] = y[i] + f * a6[i];
        if (MODE == HOP_RICH || MODE == HOP_RES) load6(k.b, b);
        if (MODE == HOP_RICH)
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = x[i] + k.omega * (b[i] - y[i]);
        if (MODE == HOP_RES)
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = b[i] - y[i];
    } else {   // HOP_PREP, HOP_RECON, HOP_RECON_RES
        cx<double> u[6];
        load6(k.in2, u);
#pragma unroll
        for (int i = 0; i < 6; i++) u[i] = u[i] + 0.5 * a6[i];
        if (MODE == HOP_PREP) {
#pragma unroll
            for (int i = 0; i < 6; i++) y[i] = u[i];
        } else {
            herm6_apply<double>(C, u, y);
            if (MODE == HOP_RECON_RES) {   // the parity's residual u - C x_o of the x_o just formed
                cx<double> z[6];
                load_block(k.clov2, st, half, s, C);
                herm6_apply<double>(C, y, z);
#pragma unroll
                for (int i = 0; i < 6; i++) z[i] = u[i] - z[i];
                store6(k.out2, z);
            }
        }
    }
    if (NAT) {
        double2 *t = tile[half];
        auto at = [](int r, int i) { return r * 7 + i; };   // seven slots a row: no bank conflicts
        const unsigned flip = half ? k.nat.flip : 0u;
#pragma unroll
        for (int i = 0; i < 6; i++) t[at(lane, i)] = make_double2(flip_sign64(y[i].re, flip), flip_sign64(y[i].im, flip));
        __syncwarp();
        nat_write6(k.nat, t, at, s0, nv, c.x & 1, half);
    } else {
        store6(k.out, y);
    }
}

template <int MODE>
static void launch_f64(const Exec &e, const HopCall &c)
{
    F64Args k;
    k.in = (const double2 *)c.in;
    k.in2 = (const double2 *)c.in2;
    k.b = (const double2 *)c.b;
    k.out = (double2 *)c.out;
    k.out2 = (double2 *)c.out2;
    k.Uout = (const double2 *)c.U[c.pout];
    k.Uin = (const double2 *)c.U[1 - c.pout];
    k.clov = (const double2 *)c.clov;
    k.clov2 = (const double2 *)c.clov2;
    k.omega = c.omega;
    k.pout = c.pout;
    k.nrhs = c.nrhs;
    k.fs = (long long)St<double>::SPINOR_VECS * e.g.stride;
    k.nat = nat_out(e.g, c.nat, c.nat_full, c.nat_g5);
    const unsigned blocks = (unsigned)((e.g.Vh + kF64Sites - 1) / kF64Sites) * (unsigned)c.nrhs;
    // Blocks brought in early are not spread as evenly, which shows when they are most
    // of one wave, but not nearly all of it.  D_S in us, overlapped and not: 576 blocks
    // 86.4 / 90.5, 784 139.2 / 129.4, 867 139.7 / 131.0, 1024 160.4 / 158.0, 1152
    // 167.1 / 170.4, 1280 203.7 / 209.3, 4000 548 / 553.
    constexpr unsigned wave = kSMs * kF64Blocks;
    const bool after = c.after && (blocks <= wave * 5 / 8 || blocks > wave * 7 / 8);
    auto launch = [&](auto kernel) { launch_after(e, after, kernel, blocks, 2 * kF64Sites, 0, e.g, k); };
    if constexpr (MODE == HOP_FULL) {   // always natural
        launch(hop_f64_kernel<MODE, true>);
    } else if constexpr (MODE == HOP_K2) {
        if (c.nat) launch(hop_f64_kernel<MODE, true>);
        else launch(hop_f64_kernel<MODE, false>);
    } else {
        launch(hop_f64_kernel<MODE, false>);
    }
}

void hop_f64(const Exec &e, const HopCall &c)
{
    switch (c.mode) {
    case HOP_K1: launch_f64<HOP_K1>(e, c); break;
    case HOP_K2: launch_f64<HOP_K2>(e, c); break;
    case HOP_RICH: launch_f64<HOP_RICH>(e, c); break;
    case HOP_FULL: launch_f64<HOP_FULL>(e, c); break;
    case HOP_PREP: launch_f64<HOP_PREP>(e, c); break;
    case HOP_RECON: launch_f64<HOP_RECON>(e, c); break;
    case HOP_RES: launch_f64<HOP_RES>(e, c); break;
    case HOP_RECON_RES: launch_f64<HOP_RECON_RES>(e, c); break;
    }
}

}  // namespace lq
