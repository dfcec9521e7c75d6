// Natural output of the hopping kernels: the last hop of a call writes the
// caller's complex-double field itself, instead of an internal field that an
// export pass would read back (192 + 2 bytes-per-site fields of traffic and a
// launch).  The rows of a warp's 32 sites are turned in shared memory, so that
// they leave in whole 32-byte sectors.
#pragma once

#include "bf16.cuh"

namespace lq {

struct NatOut {
    double2 *p = nullptr;   // natural field, 12 complex numbers a row
    int full = 0;           // rows are the lattice's sites (else the sites of one parity)
    unsigned flip = 0;      // sign bit of spins 2 and 3 (gamma_5)
    long long rows = 0;     // rows of the field
};

static inline NatOut nat_out(const Geom &g, void *p, bool full, bool g5)
{
    NatOut o;
    o.p = (double2 *)p;
    o.full = full;
    o.rows = full ? g.V : g.Vh;
    o.flip = g5 ? 0x80000000u : 0u;
    return o;
}

__device__ __forceinline__ double flip_sign64(double d, unsigned bit)
{
    return __hiloint2double(__double2hiint(d) ^ (int)bit, __double2loint(d));
}
// the value that the export of a stored component gives: `store` names the
// storage type, whose rounding (BF16) applies
__device__ __forceinline__ double2 nat_value(const double2 *, cx<double> v) { return make_double2(v.re, v.im); }
__device__ __forceinline__ double2 nat_value(const df2 *, cx<df64> v)
{
    return make_double2(df_join(v.re.hi, v.re.lo), df_join(v.im.hi, v.im.lo));
}
__device__ __forceinline__ double2 nat_value(const float4 *, cx<float> v)
{
    return make_double2(f2d_bits(v.re), f2d_bits(v.im));
}
__device__ __forceinline__ double2 nat_value(const BfS4 *, cx<float> v)
{
    const cx<float> r = bf_cx(cx_bf(v));
    return make_double2(f2d_bits(r.re), f2d_bits(r.im));
}

// Components 6 half .. 6 half + 5 of the 32 sites s0 .. of a warp (those below
// n exist), component k of lane l at tile[at(l, k)] in shared memory.  xbit: the
// lane's x coordinate mod 2, which with its checkerboard index gives its row on a
// full lattice.  The whole warp calls it.
template <typename At>
__device__ __forceinline__ void nat_write6(const NatOut &o, const double2 *tile, At at, long long s0, int n, int xbit,
                                           int half)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const int e = i * 32 + lane, r = e / 6, k = e - 6 * r;
        const int b = __shfl_sync(0xffffffffu, xbit, r);
        const long long row = o.full ? 2 * (s0 + r) + b : s0 + r;
        if (r < n) o.p[LQ_IDX(row, o.rows, B_NAT) * 12 + 6 * half + k] = tile[at(r, k)];
    }
}

}  // namespace lq
