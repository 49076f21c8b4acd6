// H_W(mu) with eight lanes per site and field, one per hop: the kernel of the FP64 stencil
// (stencil_f64.cu, which says why) and, on small lattices, of the FP32 one.
//
// The hop-dependent parts of the arithmetic (which spins are paired, the factors +-1, +-i, the
// link's dagger) are addresses, selects and sign-bit flips, so that the eight lanes run the same
// floating-point instructions: 12 additions (spin projection), 72 multiply-adds (link), the sum of
// the eight hops as a reduce-scatter over the lanes (12 + 6 + 3 multiply-adds) that leaves three of the
// site's 24 real numbers in each lane, and 6 for the diagonal and the coefficient: 888 per site and
// field, as in one thread.  The hop coefficients cost nothing of their own: a lane's sum is kept in
// units of its hop's coefficient and the partner's number enters with the ratio of the two
// (1, e^{+-mu} or e^{-+2 mu}).  Rounding of the FP64 form against extended precision, 4^4 to 8^4 at |mu|
// up to 0.9: 1.08e-16 to 1.16e-16 of the result, 1.38e-16 to 1.44e-16 for one thread's chain of eight hops.
// ROW: three warps share four sites, a colour of the result (a row of the link) each, so that a lane
// has 45 instead of 111 floating-point instructions (the projections are repeated): for the
// smallest lattices.
// Fields in natural [site][12] or packed order (sgn_internal.cuh): a lane's 12 loads of its
// neighbour touch the same 32-byte sectors either way.
#pragma once

#include "sgn_internal.cuh"

namespace sgn {
namespace hops {

constexpr int kMaxThreads = 128;

// Ratios of the time hops' coefficients to the space hops' (t: forward, backward), their
// inverses, and backward over forward and its inverse.
template <class R>
struct Ratios {
    R t[2], ti[2], bf, fb;
};

template <class R>
struct Cx2;
template <>
struct Cx2<double> {
    using T = double2;
};
template <>
struct Cx2<float> {
    using T = float2;
};
template <class R>
using C2 = typename Cx2<R>::T;

__device__ __forceinline__ double2 ld_link(const double2* p) { return __ldg(p); }
__device__ __forceinline__ float2 ld_link(const float2* p) { return __ldg(p); }
__device__ __forceinline__ float2 ld_link(const __nv_bfloat162* p) { return __bfloat1622float2(*p); }
__device__ __forceinline__ float2 ld_link(const __half2* p) { return __half22float2(__ldg(p)); }

// v with its sign flipped where mask is 0x80000000 (0: unchanged)
__device__ __forceinline__ double flip(double v, unsigned mask) {
    return __hiloint2double((int)((unsigned)__double2hiint(v) ^ mask), __double2loint(v));
}
__device__ __forceinline__ float flip(float v, unsigned mask) { return __uint_as_float(__float_as_uint(v) ^ mask); }
// c v (imag = false) or c i v (imag = true), c = +-1 given by its sign mask
template <class V>
__device__ __forceinline__ V phase(V v, bool imag, unsigned c) {
    const auto a = imag ? v.y : v.x, b = imag ? v.x : v.y;
    return V{flip(a, imag ? c ^ 0x80000000u : c), flip(b, c)};
}

// Offset of complex entry k of a site: natural order, or plane k/2 of the packed order.
template <bool NAT>
__device__ __forceinline__ int64_t entry(int64_t site, int k, int64_t vol) {
    return NAT ? site * 12 + k : (int64_t)(k >> 1) * 2 * vol + 2 * site + (k & 1);
}

// CTA b: site tile b / nrhs (blockDim.x / 8 sites, with ROW 4) of field b % nrhs (the fields of a site
// tile run together and share its links in L2).  Lane l of a site's eight: nu = l / 2, forward for even l.
// RATIO: the space hops' coefficients are equal and non-zero, so are the units of the sums; else
// every hop is scaled by its own coefficient (dH_W/dmu, whose space hops are zero).
template <class R, class LinkT, bool NAT, bool RATIO, bool ROW>
__global__ void __launch_bounds__(kMaxThreads, 4)
    k_hw_hops(C2<R>* out, const C2<R>* in, const LinkT* __restrict__ U, int nrhs,
              StencilParams P, Ratios<R> Q, const int* skip) {
    using V = C2<R>;
    const int64_t tile = blockIdx.x / (unsigned)nrhs;
    const int rhs = (int)(blockIdx.x - tile * nrhs);
    constexpr int NA = ROW ? 1 : 3;  // rows of the link per lane
    const int row = ROW ? threadIdx.x >> 5 : 0;
    const int64_t s0 = ROW ? tile * 4 + ((threadIdx.x & 31) >> 3) : tile * (blockDim.x >> 3) + (threadIdx.x >> 3);
    const bool act = s0 < P.vol;
    const int64_t site = act ? s0 : P.vol - 1;  // idle lanes take part in the shuffles
    const int l = threadIdx.x & 7, nu = l >> 1;
    const bool fwd = !(l & 1);
    const V* f = in + rhs * P.stride_rhs;

    // neighbour, and the hop's coefficient with the boundary sign
    int co, L;
    int64_t stride;
    {
        const uint32_t q0 = P.div[0].div((uint32_t)site);
        const uint32_t q1 = P.div[1].div(q0);
        const uint32_t q2 = P.div[2].div(q1);
        const int c0 = (int)((uint32_t)site - q0 * (uint32_t)P.L[0]), c1 = (int)(q0 - q1 * (uint32_t)P.L[1]),
                  c2 = (int)(q1 - q2 * (uint32_t)P.L[2]), c3 = (int)q2;
        co = nu < 2 ? (nu == 0 ? c0 : c1) : (nu == 2 ? c2 : c3);
        L = nu < 2 ? (nu == 0 ? P.L[0] : P.L[1]) : (nu == 2 ? P.L[2] : P.L[3]);
        const int64_t s1 = P.L[0], s2 = s1 * P.L[1], s3 = s2 * P.L[2];
        stride = nu < 2 ? (nu == 0 ? 1 : s1) : (nu == 2 ? s2 : s3);
    }
    R coef, diag;
    if constexpr (sizeof(R) == 8) {
        coef = fwd ? (nu == 3 ? P.cf[3] : nu == 2 ? P.cf[2] : nu == 1 ? P.cf[1] : P.cf[0])
                   : (nu == 3 ? P.cb[3] : nu == 2 ? P.cb[2] : nu == 1 ? P.cb[1] : P.cb[0]);
        diag = P.diag;
    } else {
        coef = fwd ? (nu == 3 ? P.cf32[3] : nu == 2 ? P.cf32[2] : nu == 1 ? P.cf32[1] : P.cf32[0])
                   : (nu == 3 ? P.cb32[3] : nu == 2 ? P.cb32[2] : nu == 1 ? P.cb32[1] : P.cb32[0]);
        diag = P.diag32;
    }
    const bool wrap = fwd ? co == L - 1 : co == 0;
    const int64_t nb = fwd ? (wrap ? site - (int64_t)(L - 1) * stride : site + stride)
                           : (wrap ? site + (int64_t)(L - 1) * stride : site - stride);
    const int apf = nu < 2 ? (nu == 0 ? P.ap[0] : P.ap[1]) : (nu == 2 ? P.ap[2] : P.ap[3]);

    // loads: the neighbour's four spins (the lower two in the order they pair with the upper ones),
    // the link (its transpose for a backward hop), and this lane's three numbers of the site itself
    const unsigned NEG = 0x80000000u;
    const unsigned bs = wrap && apf ? NEG : 0u;  // sign of a hop across an antiperiodic boundary
    const bool imag = !(nu & 1);
    const int ka = nu < 2 ? 9 : 6, kb = nu < 2 ? 6 : 9;
    V h0[3], h1[3], qa[3], qb[3], u[3 * NA];
    // the links belong to no kernel of the stream: their loads go out before the predecessor is done
    const int ra = fwd ? 3 : 1, rb = fwd ? 1 : 3;
    const LinkT* lb = U + (int64_t)(nu * 9 + ra * row) * P.vol + (fwd ? site : nb);
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) u[3 * a + b] = ld_link(lb + (int64_t)(ra * a + rb * b) * P.vol);
    pdl_begin();
    if (skip && skip[rhs]) return;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h0[c] = *(f + entry<NAT>(nb, c, P.vol));
        h1[c] = *(f + entry<NAT>(nb, 3 + c, P.vol));
        qa[c] = *(f + entry<NAT>(nb, ka + c, P.vol));
        qb[c] = *(f + entry<NAT>(nb, kb + c, P.vol));
    }
    const R* own = reinterpret_cast<const R*>(f);
    R psi[NA];
    int64_t at[NA];  // this lane's real numbers of the site: 3 l .. 3 l + 2, or number l % 2 of entry 3 (l / 2) + row
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        const int k = ROW ? 3 * nu + row : (3 * l + i) >> 1, c = ROW ? l & 1 : (3 * l + i) & 1;
        at[i] = 2 * entry<NAT>(site, k, P.vol) + c;
        psi[i] = own[at[i]];
    }
    // spin projection h = psi_up + S B psi_dn, S = -1 forward, +1 backward (see stencil.cu)
    const unsigned sS = fwd ? NEG : 0u;
    const unsigned c0 = nu == 3 ? sS : sS ^ NEG;  // factors of the paired spins: -S, -S, -S, S (times i for nu even)
    const unsigned c1 = nu == 0 ? sS ^ NEG : sS;  // -S, S, S, S
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        qa[c] = phase(qa[c], imag, c0);
        h0[c] = V{h0[c].x + qa[c].x, h0[c].y + qa[c].y};
        qb[c] = phase(qb[c], imag, c1);
        h1[c] = V{h1[c].x + qb[c].x, h1[c].y + qb[c].y};
    }
    // g = W h with the boundary sign (RATIO: in units of the coefficient)
    const unsigned cj = fwd ? 0u : NEG;
    R v[8 * NA];  // the hop's contribution: spins 0, 1 from g0, g1, spins 2, 3 by reconstruction
    const unsigned c3 = (nu == 1 || nu == 2) ? sS ^ NEG : sS;  // spin 3: S, -S, -S, S (times i for nu even)
#pragma unroll
    for (int a = 0; a < NA; ++a) {
        V g0 = V{0, 0}, g1 = V{0, 0};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R ux = u[3 * a + b].x, uy = flip(u[3 * a + b].y, cj);
            g0.x = fma(ux, h0[b].x, g0.x);
            g0.x = fma(-uy, h0[b].y, g0.x);
            g0.y = fma(ux, h0[b].y, g0.y);
            g0.y = fma(uy, h0[b].x, g0.y);
            g1.x = fma(ux, h1[b].x, g1.x);
            g1.x = fma(-uy, h1[b].y, g1.x);
            g1.y = fma(ux, h1[b].y, g1.y);
            g1.y = fma(uy, h1[b].x, g1.y);
        }
        if constexpr (!RATIO) {
            g0.x *= coef;
            g0.y *= coef;
            g1.x *= coef;
            g1.y *= coef;
        }
        g0 = V{flip(g0.x, bs), flip(g0.y, bs)};
        g1 = V{flip(g1.x, bs), flip(g1.y, bs)};
        const V e2 = nu < 2 ? g1 : g0, e3 = nu < 2 ? g0 : g1;
        const V l2 = phase(e2, imag, sS), l3 = phase(e3, imag, c3);
        const V e[4] = {g0, g1, l2, l3};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * (NA * k + a)] = e[k].x;
            v[2 * (NA * k + a) + 1] = e[k].y;
        }
    }
    // sum over the eight hops: at each level a lane keeps one half of its numbers and adds the
    // partner's same half; lane l ends with numbers NA l .. NA l + NA - 1
    R w[4 * NA], x[2 * NA], y[NA];
    // coefficient of the partner's hop over this lane's: the time hops (nu = 3) against nu = 1,
    // then against nu = 2 (whose sums are in units of a space hop), then forward against backward
    const R t = fwd ? Q.t[0] : Q.t[1], ti = fwd ? Q.ti[0] : Q.ti[1];
    const R one = 1, r4 = nu == 1 ? t : nu == 3 ? ti : one, r2 = nu == 2 ? t : nu == 3 ? ti : one,
            r1 = nu == 3 ? (fwd ? Q.bf : Q.fb) : one;
    {
        const bool up = l & 4;
#pragma unroll
        for (int i = 0; i < 4 * NA; ++i) {
            const R keep = up ? v[4 * NA + i] : v[i], send = up ? v[i] : v[4 * NA + i];
            const R got = __shfl_xor_sync(0xffffffffu, send, 4);
            w[i] = RATIO ? fma(r4, got, keep) : keep + got;
        }
    }
    {
        const bool up = l & 2;
#pragma unroll
        for (int i = 0; i < 2 * NA; ++i) {
            const R keep = up ? w[2 * NA + i] : w[i], send = up ? w[i] : w[2 * NA + i];
            const R got = __shfl_xor_sync(0xffffffffu, send, 2);
            x[i] = RATIO ? fma(r2, got, keep) : keep + got;
        }
    }
    {
        const bool up = l & 1;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const R keep = up ? x[NA + i] : x[i], send = up ? x[i] : x[NA + i];
            const R got = __shfl_xor_sync(0xffffffffu, send, 1);
            y[i] = RATIO ? fma(r1, got, keep) : keep + got;
        }
    }
    if (!act) return;
    const unsigned g5 = l & 4 ? NEG : 0u;  // gamma5 = diag(1, 1, -1, -1): lanes 4.. hold spins 2, 3
    R* o = reinterpret_cast<R*>(out + rhs * P.stride_rhs);
#pragma unroll
    for (int i = 0; i < NA; ++i)
        o[at[i]] = flip(RATIO ? fma(coef, y[i], diag * psi[i]) : fma(diag, psi[i], y[i]), g5);
}

// The coefficients' ratios, and whether they can be used: no hop zero, e^{2 |mu|} within range.
template <class R>
bool ratios(const StencilParams& p, Ratios<R>& q) {
    const double r[6] = {p.cf[3] / p.cf[0], p.cb[3] / p.cb[0], p.cf[0] / p.cf[3],
                         p.cb[0] / p.cb[3], p.cb[3] / p.cf[3], p.cf[3] / p.cb[3]};
    bool ok = true;
    for (int d = 0; d < 3; ++d) ok = ok && p.cf[d] == p.cf[0] && p.cb[d] == p.cf[0] && p.cf[0] != 0;
    const double far = sizeof(R) == 8 ? 1e100 : 1e15;
    for (double v : r) ok = ok && v > 1 / far && v < far;
    q = {{(R)r[0], (R)r[1]}, {(R)r[2], (R)r[3]}, (R)r[4], (R)r[5]};
    return ok;
}

template <class R, class LinkT, bool ROW>
cudaError_t launch(C2<R>* out, const C2<R>* in, const LinkT* U, int nrhs, const StencilParams& p, const int* skip,
                   cudaStream_t st, bool nat) {
    if (nrhs <= 0 || p.vol <= 0) return cudaSuccess;
    // one-warp CTAs (4 sites) while they fit in a few per SM: every SM gets the same number
    const int threads = ROW ? 96 : p.vol * nrhs < 4 * 16 * 152 ? 32 : kMaxThreads, sites = ROW ? 4 : threads / 8;
    const int64_t blocks = (p.vol + sites - 1) / sites * nrhs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    Ratios<R> q;
    const bool ratio = ratios(p, q);
    auto k = nat ? (ratio ? k_hw_hops<R, LinkT, true, true, ROW> : k_hw_hops<R, LinkT, true, false, ROW>)
                 : (ratio ? k_hw_hops<R, LinkT, false, true, ROW> : k_hw_hops<R, LinkT, false, false, ROW>);
    launch_pdl(k, (unsigned)blocks, threads, 0, st, out, in, U, nrhs, p, q, skip);
    count_launch();
    return cudaGetLastError();
}

}  // namespace hops
}  // namespace sgn
