// Spin projection and colour transport of one hop of the Wilson operator,
// shared by the hopping kernels (global-memory neighbours) and the SAP block
// kernel (shared-memory neighbours).
//
// Projection identities (chiral basis, upper = spins 0,1):
//   (1 - s g_k) psi = (h, s(-i s_k) h)  with h = psi_u + s i s_k psi_l   (k = 1,2,3)
//   (1 - s g_4) psi = (h, -s h)         with h = psi_u - s psi_l
// where s = +1 for the forward and -1 for the backward hop.
#pragma once

#include "lq_internal.cuh"

namespace lq {

// half spinor h[hs*3 + a] from the full spinor p[s*3 + a]; SIGN = -1 projects
// with (1 - g_mu) (forward hop), SIGN = +1 with (1 + g_mu) (backward hop)
template <int MU, int SIGN, typename R>
__device__ __forceinline__ void project(const cx<R> p[12], cx<R> h[6])
{
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const cx<R> p0 = p[a], p1 = p[3 + a], p2 = p[6 + a], p3 = p[9 + a];
        if (MU == 0) {
            h[a] = SIGN < 0 ? p0 + ti(p3) : p0 - ti(p3);
            h[3 + a] = SIGN < 0 ? p1 + ti(p2) : p1 - ti(p2);
        } else if (MU == 1) {
            h[a] = SIGN < 0 ? p0 + p3 : p0 - p3;
            h[3 + a] = SIGN < 0 ? p1 - p2 : p1 + p2;
        } else if (MU == 2) {
            h[a] = SIGN < 0 ? p0 + ti(p2) : p0 - ti(p2);
            h[3 + a] = SIGN < 0 ? p1 - ti(p3) : p1 + ti(p3);
        } else {
            h[a] = SIGN < 0 ? p0 - p2 : p0 + p2;
            h[3 + a] = SIGN < 0 ? p1 - p3 : p1 + p3;
        }
    }
}

// acc += the full spinor reconstructed from the transported half spinor u; the
// FIRST direction of a sum sets acc instead (24 additions fewer, which count on
// the FP64 pipe)
template <int MU, int SIGN, bool FIRST = false, typename R>
__device__ __forceinline__ void reconstruct(cx<R> acc[12], const cx<R> u[6])
{
    if constexpr (FIRST) {
        static_assert(!FIRST || SIGN < 0, "the first direction of a sum is a forward one");
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const cx<R> u0 = u[a], u1 = u[3 + a];
            acc[a] = u0;
            acc[3 + a] = u1;
            acc[6 + a] = MU == 0 ? tmi(u1) : MU == 1 ? -u1 : MU == 2 ? tmi(u0) : -u0;
            acc[9 + a] = MU == 0 ? tmi(u0) : MU == 1 ? u0 : MU == 2 ? ti(u1) : -u1;
        }
    } else
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const cx<R> u0 = u[a], u1 = u[3 + a];
        acc[a] = acc[a] + u0;
        acc[3 + a] = acc[3 + a] + u1;
        if (MU == 0) {
            acc[6 + a] = SIGN < 0 ? acc[6 + a] + tmi(u1) : acc[6 + a] + ti(u1);
            acc[9 + a] = SIGN < 0 ? acc[9 + a] + tmi(u0) : acc[9 + a] + ti(u0);
        } else if (MU == 1) {
            acc[6 + a] = SIGN < 0 ? acc[6 + a] - u1 : acc[6 + a] + u1;
            acc[9 + a] = SIGN < 0 ? acc[9 + a] + u0 : acc[9 + a] - u0;
        } else if (MU == 2) {
            acc[6 + a] = SIGN < 0 ? acc[6 + a] + tmi(u0) : acc[6 + a] + ti(u0);
            acc[9 + a] = SIGN < 0 ? acc[9 + a] + ti(u1) : acc[9 + a] + tmi(u1);
        } else {
            acc[6 + a] = SIGN < 0 ? acc[6 + a] - u0 : acc[6 + a] + u0;
            acc[9 + a] = SIGN < 0 ? acc[9 + a] - u1 : acc[9 + a] + u1;
        }
    }
}

// b z for b = +-1: a sign bit for FP64, whose pipe is the bound of its kernels
template <typename R>
__device__ __forceinline__ cx<R> times_sign(R b, cx<R> z) { return b * z; }
template <>
__device__ __forceinline__ cx<double> times_sign<double>(double b, cx<double> z)
{
    const int m = __double2hiint(b) & (int)0x80000000u;
    return {__hiloint2double(__double2hiint(z.re) ^ m, __double2loint(z.re)),
            __hiloint2double(__double2hiint(z.im) ^ m, __double2loint(z.im))};
}

// u = bsign W h: W = m (SIGN -1, forward hop) or m^+ (SIGN +1, backward hop)
template <int SIGN, typename R>
__device__ __forceinline__ void transport(const cx<R> m[9], const cx<R> h[6], R bsign, cx<R> u[6])
{
#pragma unroll
    for (int hs = 0; hs < 2; hs++)
#pragma unroll
        for (int a = 0; a < 3; a++) {
            cx<R> t;
            if (SIGN < 0) {
                t = cmul(m[a * 3 + 0], h[hs * 3 + 0]);
                t = cfma(m[a * 3 + 1], h[hs * 3 + 1], t);
                t = cfma(m[a * 3 + 2], h[hs * 3 + 2], t);
            } else {
                t = cmulc(m[0 * 3 + a], h[hs * 3 + 0]);
                t = cfmac(m[1 * 3 + a], h[hs * 3 + 1], t);
                t = cfmac(m[2 * 3 + a], h[hs * 3 + 2], t);
            }
            u[hs * 3 + a] = times_sign(bsign, t);
        }
}

// acc += bsign (1 -+ g_mu) W p for a loaded neighbour spinor p and link m
template <int MU, int SIGN, bool FIRST = false, typename R>
__device__ __forceinline__ void hop_apply(cx<R> acc[12], const cx<R> p[12], const cx<R> m[9], R bsign)
{
    cx<R> h[6], u[6];
    project<MU, SIGN>(p, h);
    transport<SIGN>(m, h, bsign, u);
    reconstruct<MU, SIGN, FIRST>(acc, u);
}

// ---- the same hop with its direction d = 2 mu + (backward) as data ------------
// h0 = psi_0 + i^qa psi_pa, h1 = psi_1 + i^qb psi_(5-pa) with pa = 3 for x, y and
// 2 for z, t, and acc_0 += u_0, acc_1 += u_1, acc_2 += i^qc u_ra,
// acc_3 += i^qd u_(1-ra) with ra = 1 for x, y and 0 for z, t.  The powers
//   qa = {1,3,0,2,1,3,2,0}, qb = {1,3,2,0,3,1,2,0},
//   qc = {3,1,2,0,3,1,2,0}, qd = {3,1,0,2,1,3,2,0}
// are packed two bits per direction (no local-memory tables).
constexpr unsigned kHopQA = 11661u, kHopQB = 10029u, kHopQC = 10023u, kHopQD = 11655u;

template <typename R>
__device__ __forceinline__ cx<R> rot_i(cx<R> z, int q)   // i^q z
{
    const cx<R> a = (q & 1) ? cx<R>{-z.im, z.re} : z;
    return (q & 2) ? cx<R>{-a.re, -a.im} : a;
}

// the checkerboard index of the neighbour of site s (coordinates c) in
// direction d, and whether the hop crosses the lattice's time boundary
__device__ __forceinline__ long long hop_neighbour(const Geom &g, const Coords &c, long long s, int d, bool &cross,
                                                   unsigned code)
{
    const int mu = d >> 1;
    const bool fwd = (d & 1) == 0;
    cross = false;
    if (mu == 0) {
        const int xn = fwd ? (c.x + 1 == g.L[0] ? 0 : c.x + 1) : (c.x == 0 ? g.L[0] - 1 : c.x - 1);
        return LQ_IDX(c.row * g.Lxh + (xn >> 1), g.Vh, code);
    }
    const int coord = mu == 1 ? c.y : mu == 2 ? c.z : c.t;
    const int ext = g.L[mu];
    const long long dd = mu == 1 ? (long long)g.Lxh
                       : mu == 2 ? (long long)g.Lxh * g.L[1] : (long long)g.Lxh * g.L[1] * g.L[2];
    if (mu == 3) cross = fwd ? coord + 1 == ext : coord == 0;
    if (fwd) return LQ_IDX((coord + 1 == ext) ? s - (long long)(ext - 1) * dd : s + dd, g.Vh, code);
    return LQ_IDX((coord == 0) ? s + (long long)(ext - 1) * dd : s - dd, g.Vh, code);
}

}  // namespace lq
