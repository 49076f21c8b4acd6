// H_W(mu) = gamma5 D_W(mu) (Sec. 1 of the paper) in float-float arithmetic on the FP32 units:
// every real quantity is an unevaluated sum hi + lo of two floats (about 48 significant bits),
// the arithmetic built from error-free transformations (Knuth's TwoSum, Dekker's FastTwoSum and
// the FMA form of TwoProd) and, for the link products, a compensated dot product in the style of
// Ogita, Rump and Oishi's Dot2 (the sum and the product errors carried in a second float).
//
// Use: the mixed form's true residuals r_i = b~ - (A^2 - sigma_i) x_i need A^2 x_i to far better
// than FP32 (they decide convergence at 1e-8 ||b~||), and GB300 executes FP64 at 1/64 of its FP32
// rate: the FP64 stencil is bound by the FP64 pipe.  The float-float stencil reaches ~1e-13 of the
// FP64 result with FP32 instructions only.
//
// Layout: a float4 (Re hi, Im hi, Re lo, Im lo) per complex number, in the place the complex128
// number has in the natural or the packed order, so that conversion is elementwise; links too.
// Eight lanes per site and field, one per hop, as in stencil_f64.cu (see there for the hop-dependent
// selects): about 1,500 instructions per lane.  One thread per site (11,000) needed 128 registers
// for its accumulators and waited for loads most of the time (FMA pipe 32 % busy).  Measured per
// launch: 16^4 x 4 fields 201 -> 179 us, 10^4 x 12 85 -> 76; 6^4 x 1 27.5 us per shift, now 20 us for
// twenty shifts together.  The conversions were bound by FP64 conversion instructions (cvt.cuh): split
// 47 -> 31 us on 16^4 x 4; the join (36 us) and the residual assembly are part of the stencil.
#include "cvt.cuh"
#include "sgn_internal.cuh"

namespace sgn {
namespace {

struct ff {
    float hi, lo;
};

// Knuth's TwoSum: s + e = a + b exactly.  Explicit _rn intrinsics keep the compiler from
// contracting or reassociating the error terms.
__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
// Dekker's FastTwoSum (exact when |a| >= |b|).
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }
// Sum of two float-float numbers, left unnormalised: hi is the rounded sum of the high parts, lo
// collects its error and the low parts (|lo| stays within a few units of 2^-24 |hi| unless the sum
// cancels, and hi + lo is the sum to about 2^-46 of the operands either way).  The stencil's
// intermediate sums and its accumulators use this form; the accumulators are normalised once,
// before the store.
__device__ __forceinline__ ff ff_add_u(ff a, ff b) {
    const ff s = two_sum(a.hi, b.hi);
    return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}
// a * b: TwoProd of the high parts by FMA, the cross terms in FP32 (their rounding is of
// order 2^-48 of the product), the small lo * lo term dropped.
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}

// Compensated dot-product accumulator: value s + c.  add(a, b) adds a * b: the product's
// rounding error (TwoProd) and the sum's (TwoSum) go into c.
struct Dot {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(ff a, ff b) {
        const float p = __fmul_rn(a.hi, b.hi);
        float e = __fmaf_rn(a.hi, b.hi, -p);
        e = __fmaf_rn(a.hi, b.lo, e);
        e = __fmaf_rn(a.lo, b.hi, e);
        const ff t = two_sum(s, p);
        s = t.hi;
        c = __fadd_rn(c, __fadd_rn(t.lo, e));
    }
    __device__ __forceinline__ ff value() const { return {s, c}; }  // unnormalised (see ff_add_u)
};

struct ffc {
    ff re, im;
};
__device__ __forceinline__ ffc cadd(ffc a, ffc b) { return {ff_add_u(a.re, b.re), ff_add_u(a.im, b.im)}; }
// x with its sign flipped where mask is 0x80000000 (0: unchanged)
__device__ __forceinline__ float flip(float x, unsigned mask) { return __uint_as_float(__float_as_uint(x) ^ mask); }
__device__ __forceinline__ ff flip(ff a, unsigned mask) { return {flip(a.hi, mask), flip(a.lo, mask)}; }
// c v (imag = false) or c i v (imag = true), c = +-1 given by its sign mask
__device__ __forceinline__ ffc phase(ffc v, bool imag, unsigned c) {
    const ff a = imag ? v.im : v.re, b = imag ? v.re : v.im;
    return {flip(a, imag ? c ^ 0x80000000u : c), flip(b, c)};
}
__device__ __forceinline__ ffc ld(const float4* p) {
    const float4 v = *p;
    return {{v.x, v.z}, {v.y, v.w}};
}
__device__ __forceinline__ ff shfl_xor(ff a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ ff sel(bool c, ff a, ff b) { return {c ? a.hi : b.hi, c ? a.lo : b.lo}; }

// Offset of entry k of a site: natural order, or plane k/2 of the packed order.
template <bool NAT>
__device__ __forceinline__ int64_t entry(int64_t site, int k, int64_t vol) {
    return NAT ? site * 12 + k : (int64_t)(k >> 1) * 2 * vol + 2 * site + (k & 1);
}

constexpr int kMaxThreads = 128;

// What becomes of H psi.
enum FfOut {
    FF_PAIRS,    // float-float field
    FF_DOUBLES,  // complex128 field
    FF_RESIDUAL  // r_f = b_c - H psi_f + sigma_i x_f (complex128) for field f = i ncol + c
};
struct FfResidual {
    const double2 *b, *x;
    const double* sigma;  // device, one per shift
    int ncol;
};

// CTA b: site tile b / nrhs (blockDim.x / 8 sites) of field b % nrhs.
template <bool NAT, FfOut OUT>
__global__ void __launch_bounds__(kMaxThreads, 4)
    k_hw_ff(void* out, const float4* in, const float4* Uf, int nrhs,
            StencilParams P, FfResidual R) {
    pdl_begin();
    const int64_t tile = blockIdx.x / (unsigned)nrhs;
    const int rhs = (int)(blockIdx.x - tile * nrhs);
    const int64_t s0 = tile * (blockDim.x >> 3) + (threadIdx.x >> 3);
    const bool act = s0 < P.vol;
    const int64_t site = act ? s0 : P.vol - 1;  // idle lanes take part in the shuffles
    const int l = threadIdx.x & 7, nu = l >> 1;
    const bool fwd = !(l & 1);
    const float4* f = in + rhs * P.stride_rhs;

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
    const bool wrap = fwd ? co == L - 1 : co == 0;
    const int64_t nb = fwd ? (wrap ? site - (int64_t)(L - 1) * stride : site + stride)
                           : (wrap ? site + (int64_t)(L - 1) * stride : site - stride);
    const int apf = nu < 2 ? (nu == 0 ? P.ap[0] : P.ap[1]) : (nu == 2 ? P.ap[2] : P.ap[3]);

    const unsigned NEG = 0x80000000u;
    const unsigned bs = wrap && apf ? NEG : 0u;  // sign of a hop across an antiperiodic boundary
    const bool imag = !(nu & 1);
    const int ka = nu < 2 ? 9 : 6, kb = nu < 2 ? 6 : 9;
    // spin projection h = psi_up + S B psi_dn, S = -1 forward, +1 backward
    const unsigned sS = fwd ? NEG : 0u;
    const unsigned c0 = nu == 3 ? sS : sS ^ NEG;  // factors of the paired spins: -S, -S, -S, S (times i for nu even)
    const unsigned c1 = nu == 0 ? sS ^ NEG : sS;  // -S, S, S, S
    ffc h0[3], h1[3], u[9];
    const float4* lb = Uf + (int64_t)nu * 9 * P.vol + (fwd ? site : nb);
    const int ra = fwd ? 3 : 1, rb = fwd ? 1 : 3;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) u[3 * a + b] = ld(lb + (int64_t)(ra * a + rb * b) * P.vol);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const ffc p0 = ld(f + entry<NAT>(nb, c, P.vol)), p1 = ld(f + entry<NAT>(nb, 3 + c, P.vol));
        const ffc qa = ld(f + entry<NAT>(nb, ka + c, P.vol)), qb = ld(f + entry<NAT>(nb, kb + c, P.vol));
        h0[c] = cadd(p0, phase(qa, imag, c0));
        h1[c] = cadd(p1, phase(qb, imag, c1));
    }
    const unsigned cj = fwd ? 0u : NEG;
    const ff tc = fwd ? ff{P.cf32[3], P.cf_lo[3]} : ff{P.cb32[3], P.cb_lo[3]};
    const float sc = fwd ? (nu == 0 ? P.cf32[0] : nu == 1 ? P.cf32[1] : P.cf32[2])
                         : (nu == 0 ? P.cb32[0] : nu == 1 ? P.cb32[1] : P.cb32[2]);  // -1/2: exact
    ff v[24];  // the hop's contribution: spins 0, 1 from g0, g1, spins 2, 3 by reconstruction
    const unsigned c3 = (nu == 1 || nu == 2) ? sS ^ NEG : sS;  // spin 3: S, -S, -S, S (times i for nu even)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Dot g0r, g0i, g1r, g1i;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const ff ur = u[3 * a + b].re, ui = flip(u[3 * a + b].im, cj), nui = flip(ui, NEG);
            g0r.add(ur, h0[b].re);
            g0r.add(nui, h0[b].im);
            g0i.add(ur, h0[b].im);
            g0i.add(ui, h0[b].re);
            g1r.add(ur, h1[b].re);
            g1r.add(nui, h1[b].im);
            g1i.add(ur, h1[b].im);
            g1i.add(ui, h1[b].re);
        }
        ff g[4] = {g0r.value(), g0i.value(), g1r.value(), g1i.value()};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            g[k] = nu == 3 ? ff_mul(g[k], tc) : ff{g[k].hi * sc, g[k].lo * sc};
            g[k] = flip(g[k], bs);
        }
        const ffc g0 = {g[0], g[1]}, g1 = {g[2], g[3]};
        const ffc e2 = {sel(nu < 2, g1.re, g0.re), sel(nu < 2, g1.im, g0.im)},
                  e3 = {sel(nu < 2, g0.re, g1.re), sel(nu < 2, g0.im, g1.im)};
        const ffc l2 = phase(e2, imag, sS), l3 = phase(e3, imag, c3);
        v[2 * a] = g0.re;
        v[2 * a + 1] = g0.im;
        v[6 + 2 * a] = g1.re;
        v[6 + 2 * a + 1] = g1.im;
        v[12 + 2 * a] = l2.re;
        v[12 + 2 * a + 1] = l2.im;
        v[18 + 2 * a] = l3.re;
        v[18 + 2 * a + 1] = l3.im;
    }
    // sum over the eight hops: at each level a lane keeps one half of its numbers and adds the
    // partner's same half; lane l ends with numbers 3 l .. 3 l + 2
    ff w[12], x[6], y[3];
#pragma unroll
    for (int i = 0; i < 12; ++i) {
        const bool up = l & 4;
        w[i] = ff_add_u(sel(up, v[12 + i], v[i]), shfl_xor(sel(up, v[i], v[12 + i]), 4));
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const bool up = l & 2;
        x[i] = ff_add_u(sel(up, w[6 + i], w[i]), shfl_xor(sel(up, w[i], w[6 + i]), 2));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const bool up = l & 1;
        y[i] = ff_add_u(sel(up, x[3 + i], x[i]), shfl_xor(sel(up, x[i], x[3 + i]), 1));
    }
    if (!act) return;
    const unsigned g5 = l & 4 ? NEG : 0u;  // gamma5 = diag(1, 1, -1, -1): numbers 12.. are spins 2, 3
    const float* own = reinterpret_cast<const float*>(f);
    const ff d = {P.diag32, P.diag_lo};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int r = 3 * l + i, im = r & 1;
        const int64_t e = entry<NAT>(site, r >> 1, P.vol);
        const ff psi = {own[4 * e + im], own[4 * e + 2 + im]};
        ff z = ff_add_u(ff_mul(psi, d), y[i]);
        z = flip(two_sum(z.hi, z.lo), g5);
        const int64_t o = rhs * P.stride_rhs + e;
        if constexpr (OUT == FF_PAIRS) {
            float* q = reinterpret_cast<float*>(out) + 4 * o;
            q[im] = z.hi;
            q[2 + im] = z.lo;
        } else {
            const double zd = f2d(z.hi) + f2d(z.lo);
            double* q = reinterpret_cast<double*>(out) + 2 * o + im;
            if constexpr (OUT == FF_DOUBLES) {
                *q = zd;
            } else {
                const int sh = rhs / R.ncol, col = rhs - sh * R.ncol;
                const double bv = reinterpret_cast<const double*>(R.b + col * P.stride_rhs + e)[im];
                const double xv = reinterpret_cast<const double*>(R.x + o)[im];
                *q = fma(R.sigma[sh], xv, bv - zd);
            }
        }
    }
}

// complex128 -> float-float, elementwise
__global__ void k_split_ff(const double2* in, float4* out, int64_t count) {
    pdl_begin();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 v = in[i];
        const float2 re = d2ff(v.x), im = d2ff(v.y);
        out[i] = make_float4(re.x, im.x, re.y, im.y);
    }
}

unsigned grid_of(int64_t count) {
    const int64_t b = (count + 255) / 256;
    return (unsigned)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

template <FfOut OUT>
cudaError_t launch_ff(void* out, const float4* in, const float4* Uf, int nrhs, const StencilParams& p, bool nat,
                      const FfResidual& r, cudaStream_t st) {
    if (nrhs <= 0 || p.vol <= 0) return cudaSuccess;
    // one-warp CTAs (4 sites) while they fit in a few per SM, as in stencil_f64.cu
    const int threads = p.vol * nrhs < 4 * 16 * 152 ? 32 : kMaxThreads, sites = threads / 8;
    const int64_t blocks = (p.vol + sites - 1) / sites * nrhs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    if (nat)
        launch_pdl(k_hw_ff<true, OUT>, (unsigned)blocks, threads, 0, st, out, in, Uf, nrhs, p, r);
    else
        launch_pdl(k_hw_ff<false, OUT>, (unsigned)blocks, threads, 0, st, out, in, Uf, nrhs, p, r);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t hw_ff(float4* out, const float4* in, const float4* Uf, int nrhs, const StencilParams& p, cudaStream_t st) {
    return launch_ff<FF_PAIRS>(out, in, Uf, nrhs, p, false, {}, st);
}
cudaError_t hw_ff_doubles(double2* out, const float4* in, const float4* Uf, int nrhs, const StencilParams& p, bool nat,
                          cudaStream_t st) {
    return launch_ff<FF_DOUBLES>(out, in, Uf, nrhs, p, nat, {}, st);
}
cudaError_t hw_ff_residual(double2* r, const float4* in, const float4* Uf, int nrhs, const StencilParams& p,
                           const double2* b, int ncol, const double2* x, const double* sigma, cudaStream_t st) {
    return launch_ff<FF_RESIDUAL>(r, in, Uf, nrhs, p, false, {b, x, sigma, ncol}, st);
}

cudaError_t split_ff(const double2* in, float4* out, int64_t count, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    launch_pdl(k_split_ff, grid_of(count), 256, 0, st, in, out, count);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sgn
