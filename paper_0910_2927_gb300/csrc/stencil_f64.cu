// H_W(mu) = gamma5 D_W(mu) (Sec. 1 of the paper) in FP64, eight lanes per site and field: one
// lane per hop (direction nu = 0..3, forward or backward).
//
// What bounds it: the FP64 pipe.  An SM executes two FP64 operations per cycle, half a one in each
// of its four sub-partitions, so a warp's FP64 instruction takes 64 cycles of its sub-partition
// whatever its active lanes, and a site costs about 900 of them.  With a thread per site a 4^4
// lattice is eight warps of 900; with a lane per hop it is 64 warps of 114.  Measured, us per
// launch, thread per site -> lane per hop: 4^4 x 1 field 31.3 -> 6.5, 6^4 x 1 32.5 -> 6.8,
// 7x6x9x8 x 3 32.8 -> 18.9, 10^4 x 12 206 -> 189 (92 % of the FP64 rate), where natural-order
// fields also save the 24 us of packing and unpacking.
// The hop-dependent parts of the arithmetic (which spins are paired, the factors +-1, +-i, the
// link's dagger) are addresses, selects and sign-bit flips, so that the eight lanes run the same
// FP64 instructions: 12 additions (spin projection), 72 multiply-adds (link), the sum of the eight
// hops as a reduce-scatter over the lanes (12 + 6 + 3 multiply-adds) that leaves three of the site's
// 24 real numbers in each lane, and 6 for the diagonal and the coefficient: 888 per site and
// field, as in one thread.  The hop coefficients cost nothing of their own: a lane's sum is kept in
// units of its hop's coefficient and the partner's number enters with the ratio of the two
// (1, e^{+-mu} or e^{-+2 mu}).
// Fields in natural [site][12] or packed order (sgn_internal.cuh): a lane's 12 loads of its
// neighbour touch the same 32-byte sectors either way.
#include "sgn_internal.cuh"

namespace sgn {
namespace {

constexpr int kMaxThreads = 128;

// Ratios of the time hops' coefficients to the space hops' (t: forward, backward), their
// inverses, and backward over forward and its inverse.
struct HopRatios {
    double t[2], ti[2], bf, fb;
};

// v with its sign flipped where mask is 0x80000000 (0: unchanged)
__device__ __forceinline__ double flip(double v, unsigned mask) {
    return __hiloint2double((int)((unsigned)__double2hiint(v) ^ mask), __double2loint(v));
}
// c v (imag = false) or c i v (imag = true), c = +-1 given by its sign mask
__device__ __forceinline__ double2 phase(double2 v, bool imag, unsigned c) {
    const double a = imag ? v.y : v.x, b = imag ? v.x : v.y;
    return make_double2(flip(a, imag ? c ^ 0x80000000u : c), flip(b, c));
}

// Offset of complex entry k of a site: natural order, or plane k/2 of the packed order.
template <bool NAT>
__device__ __forceinline__ int64_t entry(int64_t site, int k, int64_t vol) {
    return NAT ? site * 12 + k : (int64_t)(k >> 1) * 2 * vol + 2 * site + (k & 1);
}

// CTA b: site tile b / nrhs (blockDim.x / 8 sites) of field b % nrhs (the fields of a site tile run
// together and share its links in L2).  Lane l of a site's eight: nu = l / 2, forward for even l.
// RATIO: the space hops' coefficients are equal and non-zero, so are the units of the sums; else
// every hop is scaled by its own coefficient (dH_W/dmu, whose space hops are zero).
template <bool NAT, bool RATIO>
__global__ void __launch_bounds__(kMaxThreads, 4)
    k_hw_hops(double2* out, const double2* in, const double2* __restrict__ U, int nrhs,
              StencilParams P, HopRatios Q, const int* skip) {
    pdl_begin();
    const int64_t tile = blockIdx.x / (unsigned)nrhs;
    const int rhs = (int)(blockIdx.x - tile * nrhs);
    if (skip && skip[rhs]) return;
    const int64_t s0 = tile * (blockDim.x >> 3) + (threadIdx.x >> 3);
    const bool act = s0 < P.vol;
    const int64_t site = act ? s0 : P.vol - 1;  // idle lanes take part in the shuffles
    const int l = threadIdx.x & 7, nu = l >> 1;
    const bool fwd = !(l & 1);
    const double2* f = in + rhs * P.stride_rhs;

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
    double coef = fwd ? (nu == 3 ? P.cf[3] : nu == 2 ? P.cf[2] : nu == 1 ? P.cf[1] : P.cf[0])
                      : (nu == 3 ? P.cb[3] : nu == 2 ? P.cb[2] : nu == 1 ? P.cb[1] : P.cb[0]);
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
    double2 h0[3], h1[3], qa[3], qb[3], u[9];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h0[c] = *(f + entry<NAT>(nb, c, P.vol));
        h1[c] = *(f + entry<NAT>(nb, 3 + c, P.vol));
        qa[c] = *(f + entry<NAT>(nb, ka + c, P.vol));
        qb[c] = *(f + entry<NAT>(nb, kb + c, P.vol));
    }
    const double2* lb = U + (int64_t)nu * 9 * P.vol + (fwd ? site : nb);
    const int ra = fwd ? 3 : 1, rb = fwd ? 1 : 3;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) u[3 * a + b] = __ldg(lb + (int64_t)(ra * a + rb * b) * P.vol);
    const double* own = reinterpret_cast<const double*>(f);
    double psi[3];
    int64_t at[3];  // this lane's real numbers 3 l .. 3 l + 2 of the site
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int r = 3 * l + i;
        at[i] = 2 * entry<NAT>(site, r >> 1, P.vol) + (r & 1);
        psi[i] = own[at[i]];
    }
    // spin projection h = psi_up + S B psi_dn, S = -1 forward, +1 backward (see stencil.cu)
    const unsigned sS = fwd ? NEG : 0u;
    const unsigned c0 = nu == 3 ? sS : sS ^ NEG;  // factors of the paired spins: -S, -S, -S, S (times i for nu even)
    const unsigned c1 = nu == 0 ? sS ^ NEG : sS;  // -S, S, S, S
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h0[c] = cadd(h0[c], phase(qa[c], imag, c0));
        h1[c] = cadd(h1[c], phase(qb[c], imag, c1));
    }
    // g = W h with the boundary sign (RATIO: in units of the coefficient)
    const unsigned cj = fwd ? 0u : NEG;
    double v[24];  // the hop's contribution: spins 0, 1 from g0, g1, spins 2, 3 by reconstruction
    const unsigned c3 = (nu == 1 || nu == 2) ? sS ^ NEG : sS;  // spin 3: S, -S, -S, S (times i for nu even)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double2 g0 = make_double2(0, 0), g1 = make_double2(0, 0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double ux = u[3 * a + b].x, uy = flip(u[3 * a + b].y, cj);
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
        g0 = make_double2(flip(g0.x, bs), flip(g0.y, bs));
        g1 = make_double2(flip(g1.x, bs), flip(g1.y, bs));
        const double2 e2 = nu < 2 ? g1 : g0, e3 = nu < 2 ? g0 : g1;
        const double2 l2 = phase(e2, imag, sS), l3 = phase(e3, imag, c3);
        v[2 * a] = g0.x;
        v[2 * a + 1] = g0.y;
        v[6 + 2 * a] = g1.x;
        v[6 + 2 * a + 1] = g1.y;
        v[12 + 2 * a] = l2.x;
        v[12 + 2 * a + 1] = l2.y;
        v[18 + 2 * a] = l3.x;
        v[18 + 2 * a + 1] = l3.y;
    }
    // sum over the eight hops: at each level a lane keeps one half of its numbers and adds the
    // partner's same half; lane l ends with numbers 3 l .. 3 l + 2
    double w[12], x[6], y[3];
    // coefficient of the partner's hop over this lane's: the time hops (nu = 3) against nu = 1,
    // then against nu = 2 (whose sums are in units of a space hop), then forward against backward
    const double t = fwd ? Q.t[0] : Q.t[1], ti = fwd ? Q.ti[0] : Q.ti[1];
    const double r4 = nu == 1 ? t : nu == 3 ? ti : 1.0, r2 = nu == 2 ? t : nu == 3 ? ti : 1.0,
                 r1 = nu == 3 ? (fwd ? Q.bf : Q.fb) : 1.0;
    {
        const bool up = l & 4;
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            const double keep = up ? v[12 + i] : v[i], send = up ? v[i] : v[12 + i];
            const double got = __shfl_xor_sync(0xffffffffu, send, 4);
            w[i] = RATIO ? fma(r4, got, keep) : keep + got;
        }
    }
    {
        const bool up = l & 2;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const double keep = up ? w[6 + i] : w[i], send = up ? w[i] : w[6 + i];
            const double got = __shfl_xor_sync(0xffffffffu, send, 2);
            x[i] = RATIO ? fma(r2, got, keep) : keep + got;
        }
    }
    {
        const bool up = l & 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double keep = up ? x[3 + i] : x[i], send = up ? x[i] : x[3 + i];
            const double got = __shfl_xor_sync(0xffffffffu, send, 1);
            y[i] = RATIO ? fma(r1, got, keep) : keep + got;
        }
    }
    if (!act) return;
    const unsigned g5 = l & 4 ? NEG : 0u;  // gamma5 = diag(1, 1, -1, -1): numbers 12.. are spins 2, 3
    double* o = reinterpret_cast<double*>(out + rhs * P.stride_rhs);
#pragma unroll
    for (int i = 0; i < 3; ++i)
        o[at[i]] = flip(RATIO ? fma(coef, y[i], P.diag * psi[i]) : fma(P.diag, psi[i], y[i]), g5);
}

}  // namespace

cudaError_t launch_hw_f64(double2* out, const double2* in, const double2* U, int nrhs, const StencilParams& p,
                          const int* skip, cudaStream_t st, bool nat) {
    if (nrhs <= 0 || p.vol <= 0) return cudaSuccess;
    // one-warp CTAs (4 sites) while they fit in a few per SM: every SM gets the same number
    const int threads = p.vol * nrhs < 4 * 16 * 152 ? 32 : kMaxThreads, sites = threads / 8;
    const int64_t blocks = (p.vol + sites - 1) / sites * nrhs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const HopRatios q = {{p.cf[3] / p.cf[0], p.cb[3] / p.cb[0]},
                         {p.cf[0] / p.cf[3], p.cb[0] / p.cb[3]},
                         p.cb[3] / p.cf[3],
                         p.cf[3] / p.cb[3]};
    bool ratio = true;  // e^{2 |mu|} within range, and no hop zero
    for (int d = 0; d < 3; ++d) ratio = ratio && p.cf[d] == p.cf[0] && p.cb[d] == p.cf[0] && p.cf[0] != 0;
    for (double r : {q.t[0], q.t[1], q.ti[0], q.ti[1], q.bf, q.fb}) ratio = ratio && r > 1e-100 && r < 1e100;
    const unsigned grid = (unsigned)blocks;
    if (nat && ratio)
        launch_pdl(k_hw_hops<true, true>, grid, threads, 0, st, out, in, U, nrhs, p, q, skip);
    else if (nat)
        launch_pdl(k_hw_hops<true, false>, grid, threads, 0, st, out, in, U, nrhs, p, q, skip);
    else if (ratio)
        launch_pdl(k_hw_hops<false, true>, grid, threads, 0, st, out, in, U, nrhs, p, q, skip);
    else
        launch_pdl(k_hw_hops<false, false>, grid, threads, 0, st, out, in, U, nrhs, p, q, skip);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sgn
