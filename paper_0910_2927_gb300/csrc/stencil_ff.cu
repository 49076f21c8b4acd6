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
// Layout: fields as twelve planes, one per spin-colour entry k = 3 spin + colour, of a float4
// (Re hi, Im hi, Re lo, Im lo) per site (entry k of site s at k vol + s), links as [dir][3][3][site]
// of the same float4: every load of a warp is 512 contiguous bytes.
// A CTA takes 32 sites of one field with a warp per hop (direction, forward or backward): a warp
// projects its neighbours, multiplies by its links and leaves the two colour vectors in shared
// memory (24 KB), then six warps add the eight hops, a colour and a spin half each, and write the
// result.  No thread holds a site's 48 accumulators: 80 registers, 24 warps per SM.
// What bounds it: about 3,000 warp instructions per 32 sites and field, nearly all of them FP32: the
// schedulers issue in 68 % of the cycles, FMA pipe 52 % busy, L1 35 %, DRAM 11 % (16^4 x 4 fields with a
// complex128 result, whose assembly keeps the FP64 pipe 23 % busy); 21.6 warps active per SM.
// Measured us per launch at 10^4 x 12 fields, thread per site (128 registers, waiting for loads: FMA
// pipe 32 % busy) / eight lanes per site, one per hop (L1 79 % busy with up to 32 lines per load) /
// now: 85 / 76 / 65; 6^4 x 1 27.5 per shift / 20 / 19 for twenty shifts together; a whole call on
// 16^4 x 4 fields 357 / 213 / 172.  The conversions were bound by FP64 conversion instructions
// (cvt.cuh): splitting 10^4 x 12 fields 23 -> 10 us; the join and the residual assembly (29 us) are
// part of the stencil.
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
// c v, or c i v with IMAG, c = +-1 given by its sign mask
template <bool IMAG>
__device__ __forceinline__ ffc phase(ffc v, unsigned c) {
    if constexpr (IMAG) return {flip(v.im, c ^ 0x80000000u), flip(v.re, c)};
    return {flip(v.re, c), flip(v.im, c)};
}
__device__ __forceinline__ ffc ffc_of(float4 v) { return {{v.x, v.z}, {v.y, v.w}}; }
__device__ __forceinline__ ffc ld(const float4* p) { return ffc_of(*p); }

constexpr int kSites = 32;
constexpr int kThreads = 8 * kSites;  // a warp per hop

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

// One hop of a warp's 32 sites: g = W (1 + S gamma_nu) psi(nb), boundary sign included, in units of
// -1/2; sm[4 a + {0..3}] = Re, Im of the two colour vectors' entry a.  IMAG: the projector pairs the
// spins with +-i (nu = 0, 2).  All other arguments are uniform over the warp: signs as masks, ka
// and kb the entries of the lower spins that pair with spins 0 and 1.
template <bool IMAG>
__device__ __forceinline__ void hop(float2 (*sm)[kSites], const float4* f,
                                    const float4* __restrict__ lb, int64_t vol, int ka, int kb, unsigned c0,
                                    unsigned c1, unsigned bs, unsigned cj, int ra, int rb, bool time, ff tc) {
    const int lane = threadIdx.x & 31;
    ffc h0[3], h1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const ffc p = cadd(ld(f + c * vol), phase<IMAG>(ld(f + (ka + c) * vol), c0));
        const ffc q = cadd(ld(f + (3 + c) * vol), phase<IMAG>(ld(f + (kb + c) * vol), c1));
        h0[c] = {flip(p.re, bs), flip(p.im, bs)};
        h1[c] = {flip(q.re, bs), flip(q.im, bs)};
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Dot g0r, g0i, g1r, g1i;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const ffc u = ffc_of(__ldg(lb + (int64_t)(ra * a + rb * b) * vol));
            const ff ui = flip(u.im, cj), nui = {-ui.hi, -ui.lo};
            g0r.add(u.re, h0[b].re);
            g0r.add(nui, h0[b].im);
            g0i.add(u.re, h0[b].im);
            g0i.add(ui, h0[b].re);
            g1r.add(u.re, h1[b].re);
            g1r.add(nui, h1[b].im);
            g1i.add(u.re, h1[b].im);
            g1i.add(ui, h1[b].re);
        }
        ff g[4] = {g0r.value(), g0i.value(), g1r.value(), g1i.value()};
        if (time)
#pragma unroll
            for (int k = 0; k < 4; ++k) g[k] = ff_mul(g[k], tc);
#pragma unroll
        for (int k = 0; k < 4; ++k) sm[4 * a + k][lane] = make_float2(g[k].hi, g[k].lo);
    }
}

// CTA b: 32 sites from 32 (b / nrhs) of field b % nrhs (the fields of a site tile run together and
// share its links in L2).  NAT: complex128 output in natural order, else packed.
template <FfOut OUT, bool NAT>
__global__ void __launch_bounds__(kThreads, 3)
    k_hw_ff(void* out, const float4* in, const float4* __restrict__ Uf, int nrhs,
            StencilParams P, FfResidual R) {
    pdl_begin();
    __shared__ float2 sm[8][12][kSites];  // [hop][colour a: g0 re, g0 im, g1 re, g1 im][site]
    const int64_t tile = blockIdx.x / (unsigned)nrhs;
    const int rhs = (int)(blockIdx.x - tile * nrhs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t s0 = tile * kSites + lane;
    const int64_t site = s0 < P.vol ? s0 : P.vol - 1;  // the last tile's idle lanes repeat a site
    const float4* f = in + rhs * P.stride_rhs;
    {
        const int nu = warp >> 1;
        const bool fwd = !(warp & 1);
        const uint32_t q0 = P.div[0].div((uint32_t)site);
        const uint32_t q1 = P.div[1].div(q0);
        const uint32_t q2 = P.div[2].div(q1);
        const int co = nu == 0   ? (int)((uint32_t)site - q0 * (uint32_t)P.L[0])
                       : nu == 1 ? (int)(q0 - q1 * (uint32_t)P.L[1])
                       : nu == 2 ? (int)(q1 - q2 * (uint32_t)P.L[2])
                                 : (int)q2;
        const int L = P.L[nu];
        const int64_t s1 = P.L[0], s2 = s1 * P.L[1], s3 = s2 * P.L[2];
        const int64_t stride = nu == 0 ? 1 : nu == 1 ? s1 : nu == 2 ? s2 : s3;
        const bool wrap = fwd ? co == L - 1 : co == 0;
        const int64_t nb = fwd ? (wrap ? site - (int64_t)(L - 1) * stride : site + stride)
                               : (wrap ? site + (int64_t)(L - 1) * stride : site - stride);
        const unsigned NEG = 0x80000000u;
        const unsigned bs = wrap && P.ap[nu] ? NEG : 0u;  // a hop across an antiperiodic boundary
        // spin projection h = psi_up + S B psi_dn, S = -1 forward, +1 backward (see stencil.cu)
        const unsigned sS = fwd ? NEG : 0u;
        const unsigned c0 = nu == 3 ? sS : sS ^ NEG;  // factors of the paired spins: -S, -S, -S, S
        const unsigned c1 = nu == 0 ? sS ^ NEG : sS;  // -S, S, S, S (times i for nu even)
        const int ka = nu < 2 ? 9 : 6, kb = nu < 2 ? 6 : 9;
        const float4* lb = Uf + (int64_t)nu * 9 * P.vol + (fwd ? site : nb);
        const unsigned cj = fwd ? 0u : NEG;
        const int ra = fwd ? 3 : 1, rb = fwd ? 1 : 3;  // U(site), or the transpose of U(nb), conjugated
        // the time hops' coefficient -1/2 e^{+-mu} over the space hops' -1/2
        const ff tc = fwd ? ff{-2.f * P.cf32[3], -2.f * P.cf_lo[3]} : ff{-2.f * P.cb32[3], -2.f * P.cb_lo[3]};
        if (nu & 1)
            hop<false>(sm[warp], f + nb, lb, P.vol, ka, kb, c0, c1, bs, cj, ra, rb, nu == 3, tc);
        else
            hop<true>(sm[warp], f + nb, lb, P.vol, ka, kb, c0, c1, bs, cj, ra, rb, false, tc);
    }
    __syncthreads();
    if (warp >= 6 || s0 >= P.vol) return;
    // warp: colour a, upper (spins 0, 1) or lower (2, 3) half
    const bool lower = warp >= 3;
    const int a = lower ? warp - 3 : warp, k0 = lower ? 6 + a : a;  // entries k0 and k0 + 3
    const ffc p0 = ld(f + k0 * P.vol + site), p1 = ld(f + (k0 + 3) * P.vol + site);
    ff z[4];  // Re, Im of the two entries: the sum over the hops
#pragma unroll
    for (int h = 0; h < 8; ++h) {
        ff g[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 v = sm[h][4 * a + k][lane];
            g[k] = {v.x, v.y};
        }
        ff e[4] = {g[0], g[1], g[2], g[3]};
        if (lower) {  // S B^dag g: (i g1, i g0), (g1, -g0), (i g0, -i g1), (g0, g1) for nu = 0..3
            const int nu = h >> 1;
            const int src0 = nu < 2 ? 2 : 0, src1 = nu < 2 ? 0 : 2;
            const bool im = !(nu & 1);
            const unsigned S = h & 1 ? 0u : 0x80000000u;                      // backward +, forward -
            const unsigned T = (nu == 1 || nu == 2) ? S ^ 0x80000000u : S;  // of the second entry
            e[0] = im ? flip(g[src0 + 1], S ^ 0x80000000u) : flip(g[src0], S);
            e[1] = im ? flip(g[src0], S) : flip(g[src0 + 1], S);
            e[2] = im ? flip(g[src1 + 1], T ^ 0x80000000u) : flip(g[src1], T);
            e[3] = im ? flip(g[src1], T) : flip(g[src1 + 1], T);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = h == 0 ? e[k] : ff_add_u(z[k], e[k]);
    }
    const unsigned g5 = lower ? 0x80000000u : 0u;  // gamma5 = diag(1, 1, -1, -1)
    const ff d = {P.diag32, P.diag_lo};
    const ff psi[4] = {p0.re, p0.im, p1.re, p1.im};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const ff v = ff_add_u(ff_mul(psi[k], d), {-0.5f * z[k].hi, -0.5f * z[k].lo});
        z[k] = flip(two_sum(v.hi, v.lo), g5);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int k = k0 + 3 * e;
        const ff re = z[2 * e], im = z[2 * e + 1];
        const int64_t base = rhs * P.stride_rhs;
        if constexpr (OUT == FF_PAIRS) {
            reinterpret_cast<float4*>(out)[base + k * P.vol + site] = make_float4(re.hi, im.hi, re.lo, im.lo);
        } else {
            const int64_t o = NAT ? site * 12 + k : (int64_t)(k >> 1) * 2 * P.vol + 2 * site + (k & 1);
            double2 v = make_double2(f2d(re.hi) + f2d(re.lo), f2d(im.hi) + f2d(im.lo));
            if constexpr (OUT == FF_RESIDUAL) {
                const int sh = rhs / R.ncol, col = rhs - sh * R.ncol;
                const double2 b = R.b[col * P.stride_rhs + o], x = R.x[base + o];
                const double sg = R.sigma[sh];
                v = make_double2(fma(sg, x.x, b.x - v.x), fma(sg, x.y, b.y - v.y));
            }
            reinterpret_cast<double2*>(out)[base + o] = v;
        }
    }
}

__device__ __forceinline__ float4 split1(double2 v) {
    const float2 re = d2ff(v.x), im = d2ff(v.y);
    return make_float4(re.x, im.x, re.y, im.y);
}
// complex128 -> float-float, elementwise
__global__ void k_split_ff(const double2* __restrict__ in, float4* __restrict__ out, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = split1(in[i]);
}
// complex128 fields (NAT: natural order, else packed) -> entry planes.  CTA: 32 sites of field blockIdx.y;
// natural-order entries turn through shared memory.
template <bool NAT>
__global__ void __launch_bounds__(128) k_split_fields_ff(const double2* __restrict__ in, float4* __restrict__ out,
                                                         int64_t vol) {
    const int64_t s0 = (int64_t)blockIdx.x * kSites;
    const int ns = (int)(vol - s0 < kSites ? vol - s0 : kSites);
    const double2* f = in + (int64_t)blockIdx.y * 12 * vol;
    float4* o = out + (int64_t)blockIdx.y * 12 * vol;
    __shared__ float4 sm[NAT ? 12 * (kSites + 1) : 1];
    if constexpr (NAT) {
        for (int i = threadIdx.x; i < 12 * ns; i += 128) sm[(i % 12) * (kSites + 1) + i / 12] = split1(f[s0 * 12 + i]);
        __syncthreads();
        for (int i = threadIdx.x; i < 12 * kSites; i += 128) {
            const int k = i / kSites, s = i % kSites;
            if (s < ns) o[k * vol + s0 + s] = sm[k * (kSites + 1) + s];
        }
    } else {
        for (int i = threadIdx.x; i < 12 * kSites; i += 128) {  // entries 2 p + j of site s: 2 p vol + 2 s + j
            const int p = i / (2 * kSites), r = i % (2 * kSites), s = r >> 1, k = 2 * p + (r & 1);
            if (s < ns) o[k * vol + s0 + s] = split1(f[(int64_t)p * 2 * vol + 2 * s0 + r]);
        }
    }
}

unsigned grid_of(int64_t count) {
    const int64_t b = (count + 255) / 256;
    return (unsigned)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

template <FfOut OUT, bool NAT>
cudaError_t launch_ff(void* out, const float4* in, const float4* Uf, int nrhs, const StencilParams& p,
                      const FfResidual& r, cudaStream_t st) {
    if (nrhs <= 0 || p.vol <= 0) return cudaSuccess;
    const int64_t blocks = (p.vol + kSites - 1) / kSites * nrhs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    launch_pdl(k_hw_ff<OUT, NAT>, (unsigned)blocks, kThreads, 0, st, out, in, Uf, nrhs, p, r);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t hw_ff(float4* out, const float4* in, const float4* Uf, int nrhs, const StencilParams& p, cudaStream_t st) {
    return launch_ff<FF_PAIRS, false>(out, in, Uf, nrhs, p, {}, st);
}
cudaError_t hw_ff_doubles(double2* out, const float4* in, const float4* Uf, int nrhs, const StencilParams& p, bool nat,
                          cudaStream_t st) {
    if (nat) return launch_ff<FF_DOUBLES, true>(out, in, Uf, nrhs, p, {}, st);
    return launch_ff<FF_DOUBLES, false>(out, in, Uf, nrhs, p, {}, st);
}
cudaError_t hw_ff_residual(double2* r, const float4* in, const float4* Uf, int nrhs, const StencilParams& p,
                           const double2* b, int ncol, const double2* x, const double* sigma, cudaStream_t st) {
    return launch_ff<FF_RESIDUAL, false>(r, in, Uf, nrhs, p, {b, x, sigma, ncol}, st);
}

cudaError_t split_ff(const double2* in, float4* out, int64_t count, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    k_split_ff<<<grid_of(count), 256, 0, st>>>(in, out, count);
    count_launch();
    return cudaGetLastError();
}
cudaError_t split_fields_ff(const double2* in, float4* out, int64_t vol, int nfield, bool nat, cudaStream_t st) {
    if (nfield <= 0 || vol <= 0) return cudaSuccess;
    for (int f0 = 0; f0 < nfield; f0 += 65535) {
        const dim3 grid((unsigned)((vol + kSites - 1) / kSites), nfield - f0 < 65535 ? nfield - f0 : 65535);
        const double2* i = in + (int64_t)f0 * 12 * vol;
        float4* o = out + (int64_t)f0 * 12 * vol;
        if (nat)
            k_split_fields_ff<true><<<grid, 128, 0, st>>>(i, o, vol);
        else
            k_split_fields_ff<false><<<grid, 128, 0, st>>>(i, o, vol);
        count_launch();
    }
    return cudaGetLastError();
}

}  // namespace sgn
