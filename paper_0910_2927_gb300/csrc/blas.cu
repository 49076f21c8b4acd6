// Tall-skinny vector kernels: multi-dot products with deterministic two-stage
// FP64 reductions, the fused passes of classical Gram-Schmidt with
// reorthogonalisation (CGS2) for the Arnoldi relation eq. (2.4), the basis
// update of Algorithm 1 and the LR projection r -> (I - R L^dag) r (Sec. 4).
//
// Element granularity is a 16-byte "pack": one complex128 or two complex64.
// A thread owns PKT packs of one column (PKT = 1, 2 or 4, a template
// parameter); a CTA of NT threads owns NT*PKT consecutive packs.  The number
// of CTAs per column is chosen so that the grid fills whole waves of the GPU
// (wave_blocks), and PKT follows from it.  Dot products: each thread forms its PKT pack products
// (in FP32 for complex64 storage, i.e. chunks of 8 complex products), promotes
// them to FP64 and the rest of the reduction -- warp shuffles, the CTA sum and
// the per-column sum over CTAs -- is FP64 in a fixed order (no atomics).  The FP64 inner products
// are in gs_f64.cu.
#include "blas.cuh"
#include "cvt.cuh"

#include <cooperative_groups.h>

#include <cstdlib>

#include <algorithm>

namespace sgn {
namespace {

constexpr int NT = 256;
constexpr int NWARP = NT / 32;
constexpr int PK = 4;  // default packs per thread (reduce_blocks)
constexpr int MAXSLOT = kMaxSlots;

template <class T>
struct Ops;

template <>
struct Ops<double2> {
    using P = double2;
    using C = double2;  // coefficient type used in the arithmetic
    static constexpr int CPX = 1;
    static __device__ __forceinline__ P ld_ro(const double2* b, int64_t pk) { return b[pk]; }
    static __device__ __forceinline__ P ld(const double2* b, int64_t pk) { return b[pk]; }
    static __device__ __forceinline__ void st(double2* b, int64_t pk, P v) { b[pk] = v; }
    static __device__ __forceinline__ P zero() { return make_double2(0, 0); }
    static __device__ __forceinline__ C coef(double2 c) { return c; }
    // conj(v) * w
    static __device__ __forceinline__ double2 dot(P v, P w) { return cconjmul(v, w); }
    static __device__ __forceinline__ double nrm2(P w) { return w.x * w.x + w.y * w.y; }
    // w -= c v
    static __device__ __forceinline__ void sub_cv(P& w, C c, P v) {
        w.x = fma(-c.x, v.x, w.x);
        w.x = fma(c.y, v.y, w.x);
        w.y = fma(-c.x, v.y, w.y);
        w.y = fma(-c.y, v.x, w.y);
    }
    // a += c v
    static __device__ __forceinline__ void add_cv(P& a, C c, P v) {
        a.x = fma(c.x, v.x, a.x);
        a.x = fma(-c.y, v.y, a.x);
        a.y = fma(c.x, v.y, a.y);
        a.y = fma(c.y, v.x, a.y);
    }
    static __device__ __forceinline__ P scal(P v, double s) { return make_double2(v.x * s, v.y * s); }
    // x (complex128 array, CPX entries per pack) += v
    static __device__ __forceinline__ void add_to(double2* x, int64_t pk, P v) {
        double2 a = x[pk];
        x[pk] = make_double2(a.x + v.x, a.y + v.y);
    }
    // x += c v computed in FP64
    static __device__ __forceinline__ void add_cv_f64(double2 acc[1], double2 c, P v) {
        acc[0].x = fma(c.x, v.x, acc[0].x);
        acc[0].x = fma(-c.y, v.y, acc[0].x);
        acc[0].y = fma(c.x, v.y, acc[0].y);
        acc[0].y = fma(c.y, v.x, acc[0].y);
    }
};

template <>
struct Ops<float2> {
    using P = float4;
    using C = float2;
    static constexpr int CPX = 2;
    static __device__ __forceinline__ P ld_ro(const float2* b, int64_t pk) { return reinterpret_cast<const float4*>(b)[pk]; }
    static __device__ __forceinline__ P ld(const float2* b, int64_t pk) { return reinterpret_cast<const float4*>(b)[pk]; }
    static __device__ __forceinline__ void st(float2* b, int64_t pk, P v) { reinterpret_cast<float4*>(b)[pk] = v; }
    static __device__ __forceinline__ P zero() { return make_float4(0, 0, 0, 0); }
    static __device__ __forceinline__ C coef(double2 c) { return make_float2((float)c.x, (float)c.y); }
    static __device__ __forceinline__ double2 dot(P v, P w) {
        float re = v.x * w.x;
        re = fmaf(v.y, w.y, re);
        re = fmaf(v.z, w.z, re);
        re = fmaf(v.w, w.w, re);
        float im = v.x * w.y;
        im = fmaf(-v.y, w.x, im);
        im = fmaf(v.z, w.w, im);
        im = fmaf(-v.w, w.z, im);
        return make_double2(re, im);
    }
    static __device__ __forceinline__ double nrm2(P w) {
        float a = w.x * w.x;
        a = fmaf(w.y, w.y, a);
        a = fmaf(w.z, w.z, a);
        a = fmaf(w.w, w.w, a);
        return a;
    }
    // FP32 results: no FP64 instruction in the inner loops (FP64 runs at 1/64 rate)
    static __device__ __forceinline__ void dot_acc(float& re, float& im, P v, P w) {
        re = fmaf(v.x, w.x, re);
        re = fmaf(v.y, w.y, re);
        re = fmaf(v.z, w.z, re);
        re = fmaf(v.w, w.w, re);
        im = fmaf(v.x, w.y, im);
        im = fmaf(-v.y, w.x, im);
        im = fmaf(v.z, w.w, im);
        im = fmaf(-v.w, w.z, im);
    }
    static __device__ __forceinline__ void nrm2_acc(float& a, P w) {
        a = fmaf(w.x, w.x, a);
        a = fmaf(w.y, w.y, a);
        a = fmaf(w.z, w.z, a);
        a = fmaf(w.w, w.w, a);
    }
    static __device__ __forceinline__ P scalf(P v, float f) { return make_float4(v.x * f, v.y * f, v.z * f, v.w * f); }
    static __device__ __forceinline__ void sub_cv(P& w, C c, P v) {
        w.x = fmaf(-c.x, v.x, w.x);
        w.x = fmaf(c.y, v.y, w.x);
        w.y = fmaf(-c.x, v.y, w.y);
        w.y = fmaf(-c.y, v.x, w.y);
        w.z = fmaf(-c.x, v.z, w.z);
        w.z = fmaf(c.y, v.w, w.z);
        w.w = fmaf(-c.x, v.w, w.w);
        w.w = fmaf(-c.y, v.z, w.w);
    }
    static __device__ __forceinline__ void add_cv(P& a, C c, P v) {
        a.x = fmaf(c.x, v.x, a.x);
        a.x = fmaf(-c.y, v.y, a.x);
        a.y = fmaf(c.x, v.y, a.y);
        a.y = fmaf(c.y, v.x, a.y);
        a.z = fmaf(c.x, v.z, a.z);
        a.z = fmaf(-c.y, v.w, a.z);
        a.w = fmaf(c.x, v.w, a.w);
        a.w = fmaf(c.y, v.z, a.w);
    }
    static __device__ __forceinline__ P scal(P v, double s) {
        float f = (float)s;
        return make_float4(v.x * f, v.y * f, v.z * f, v.w * f);
    }
    static __device__ __forceinline__ void add_to(double2* x, int64_t pk, P v) {
        double2 a = x[2 * pk], b = x[2 * pk + 1];
        x[2 * pk] = make_double2(a.x + f2d(v.x), a.y + f2d(v.y));
        x[2 * pk + 1] = make_double2(b.x + f2d(v.z), b.y + f2d(v.w));
    }
    static __device__ __forceinline__ void add_cv_f64(double2 acc[2], double2 c, P v) {
        const double x = f2d(v.x), y = f2d(v.y), z = f2d(v.z), w = f2d(v.w);
        acc[0].x = fma(c.x, x, acc[0].x);
        acc[0].x = fma(-c.y, y, acc[0].x);
        acc[0].y = fma(c.x, y, acc[0].y);
        acc[0].y = fma(c.y, x, acc[0].y);
        acc[1].x = fma(c.x, z, acc[1].x);
        acc[1].x = fma(-c.y, w, acc[1].x);
        acc[1].y = fma(c.x, w, acc[1].y);
        acc[1].y = fma(c.y, z, acc[1].y);
    }
};

__device__ __forceinline__ double2 warp_sum(double2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// Sum over the 32 lanes of an FP32 value kept as an unevaluated pair (hi, lo)
// (error-free TwoSum at every level): about FP64 accuracy for the tree at FP32
// instruction rates (FP64 runs at 1/64 of the FP32 rate on this part).
__device__ __forceinline__ float2 warp_sum_pair(float v) {
    float hi = v, lo = 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ohi = __shfl_xor_sync(0xffffffffu, hi, o);
        const float olo = __shfl_xor_sync(0xffffffffu, lo, o);
        // TwoSum(hi, ohi) = (s, e) exactly, then FastTwoSum(s, e + lo + olo).  Written
        // with __fsub_rn: the same algebra spelled as __fadd_rn(x, -__fadd_rn(..))
        // was measured to lose the error term on this toolchain.
        const float s = __fadd_rn(hi, ohi);
        const float bp = __fsub_rn(s, hi);
        const float ap = __fsub_rn(s, bp);
        const float e = __fadd_rn(__fsub_rn(hi, ap), __fsub_rn(ohi, bp));
        const float t = __fadd_rn(e, __fadd_rn(lo, olo));
        const float nh = __fadd_rn(s, t);
        lo = __fsub_rn(t, __fsub_rn(nh, s));
        hi = nh;
    }
    return make_float2(hi, lo);
}
// Warp sums of a per-thread FP32 complex partial (re, im); lane 0 stores the
// FP64 result in sm[slot][warp].
__device__ __forceinline__ void warp_store_f(double2 (*sm)[NWARP], int slot, float re, float im, int lane, int warp) {
    const float2 r = warp_sum_pair(re);
    const float2 i = warp_sum_pair(im);
    if (lane == 0) sm[slot][warp] = make_double2((double)r.x + (double)r.y, (double)i.x + (double)i.y);
}

// Store the per-warp values sm[slot][warp] summed over warps into the partials.
__device__ __forceinline__ void flush_partials(double2 (*sm)[NWARP], int nslot, const Reduce& rd, int col) {
    __syncthreads();
    for (int j = threadIdx.x; j < nslot; j += NT) {
        double2 a = sm[j][0];
#pragma unroll
        for (int w = 1; w < NWARP; ++w) a = cadd(a, sm[j][w]);
        rd.partial[((int64_t)col * rd.stride + j) * rd.nblk + blockIdx.x] = a;
    }
}

// ---------------------------------------------------------------- kernels --

// partial[j] = sum_e conj(V_j[e]) w[e], j < J; slot J: ||w||^2 if with_norm.
// FP32 storage (FP64: gs_f64.cu).
template <int PKT>
__global__ void __launch_bounds__(NT) k_mdot(Basis<float2> V, int J, const float2* w, int64_t wsr, int64_t npk,
                                             Reduce rd, int with_norm, const int* skip) {
    pdl_begin();
    using T = float2;
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    __shared__ double2 sm[MAXSLOT][NWARP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T* wc = w + col * wsr;
    const int64_t base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    typename O::P wv[PKT];
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        int64_t i = base + p * NT;
        wv[p] = i < npk ? O::ld_ro(wc, i) : O::zero();
    }
    const T* vb = V.base + col * V.sr;
    for (int j = 0; j < J; ++j) {
        const T* vj = vb + j * V.sj;
        float ax = 0.f, ay = 0.f;  // FP32 chunk of PKT packs (8 complex products)
#pragma unroll
        for (int p = 0; p < PKT; ++p) {
            int64_t i = base + p * NT;
            if (i < npk) O::dot_acc(ax, ay, O::ld_ro(vj, i), wv[p]);
        }
        warp_store_f(sm, j, ax, ay, lane, warp);
    }
    if (with_norm) {
        float a = 0.f;
#pragma unroll
        for (int p = 0; p < PKT; ++p) O::nrm2_acc(a, wv[p]);
        warp_store_f(sm, J, a, 0.f, lane, warp);
    }
    flush_partials(sm, J + (with_norm ? 1 : 0), rd, col);
}

// w -= sum_j c_j V_j; then partial[j] = V_j^dag w (j < J) and slot J = ||w||^2.
template <class T, int PKT>
__global__ void __launch_bounds__(NT) k_maxpy_mdot(Basis<T> V, int J, const double2* __restrict__ coef, int cstride,
                                                   T* w, int64_t wsr, int64_t npk, Reduce rd,
                                                   const int* __restrict__ skip) {
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    __shared__ double2 sm[MAXSLOT][NWARP];
    __shared__ typename O::C cs[MAXSLOT];
    for (int j = threadIdx.x; j < J; j += NT) cs[j] = O::coef(coef[(int64_t)col * cstride + j]);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T* wc = w + col * wsr;
    const int64_t base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    typename O::P wv[PKT];
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        int64_t i = base + p * NT;
        wv[p] = i < npk ? O::ld(wc, i) : O::zero();
    }
    const T* vb = V.base + col * V.sr;
    for (int j = 0; j < J; ++j) {
        const T* vj = vb + j * V.sj;
        const typename O::C c = cs[j];
#pragma unroll
        for (int p = 0; p < PKT; ++p) {
            int64_t i = base + p * NT;
            if (i < npk) O::sub_cv(wv[p], c, O::ld_ro(vj, i));
        }
    }
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        int64_t i = base + p * NT;
        if (i < npk) O::st(wc, i, wv[p]);
    }
    for (int j = 0; j < J; ++j) {
        const T* vj = vb + j * V.sj;
        if constexpr (O::CPX == 2) {
            float ax = 0.f, ay = 0.f;
#pragma unroll
            for (int p = 0; p < PKT; ++p) {
                int64_t i = base + p * NT;
                if (i < npk) O::dot_acc(ax, ay, O::ld_ro(vj, i), wv[p]);
            }
            warp_store_f(sm, j, ax, ay, lane, warp);
        } else {
            double2 acc = make_double2(0, 0);
#pragma unroll
            for (int p = 0; p < PKT; ++p) {
                int64_t i = base + p * NT;
                if (i < npk) acc = cadd(acc, O::dot(O::ld_ro(vj, i), wv[p]));
            }
            acc = warp_sum(acc);
            if (lane == 0) sm[j][warp] = acc;
        }
    }
    if constexpr (O::CPX == 2) {
        float a = 0.f;
#pragma unroll
        for (int p = 0; p < PKT; ++p) O::nrm2_acc(a, wv[p]);
        warp_store_f(sm, J, a, 0.f, lane, warp);
    } else {
        double a = 0;
#pragma unroll
        for (int p = 0; p < PKT; ++p) a += O::nrm2(wv[p]);
        double2 acc = warp_sum(make_double2(a, 0));
        if (lane == 0) sm[J][warp] = acc;
    }
    flush_partials(sm, J + 1, rd, col);
}

// out = (w - sum_j c_j V_j) * scale[col]   (out may alias w)
template <class T, int PKT>
__global__ void __launch_bounds__(NT) k_maxpy_scale(Basis<T> V, int J, const double2* coef, int cstride,
                                                    const T* w, int64_t wsr, T* out, int64_t osr,
                                                    const double* scale, int64_t npk,
                                                    const int* skip) {
    pdl_begin();
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    __shared__ typename O::C cs[MAXSLOT];
    for (int j = threadIdx.x; j < J; j += blockDim.x) cs[j] = O::coef(coef[(int64_t)col * cstride + j]);
    __syncthreads();
    const T* wc = w + col * wsr;
    T* oc = out + col * osr;
    const double sc = scale ? scale[col] : 1.0;
    const int64_t base = (int64_t)blockIdx.x * blockDim.x * PKT + threadIdx.x;
    typename O::P wv[PKT];
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        int64_t i = base + p * (int)blockDim.x;
        wv[p] = i < npk ? O::ld(wc, i) : O::zero();
    }
    const T* vb = V.base + col * V.sr;
    for (int j = 0; j < J; ++j) {
        const T* vj = vb + j * V.sj;
        const typename O::C c = cs[j];
#pragma unroll
        for (int p = 0; p < PKT; ++p) {
            int64_t i = base + p * (int)blockDim.x;
            if (i < npk) O::sub_cv(wv[p], c, O::ld_ro(vj, i));
        }
    }
    if constexpr (O::CPX == 2) {
        const float scf = (float)sc;
#pragma unroll
        for (int p = 0; p < PKT; ++p) {
            int64_t i = base + p * (int)blockDim.x;
            if (i < npk) O::st(oc, i, O::scalf(wv[p], scf));
        }
    } else {
#pragma unroll
        for (int p = 0; p < PKT; ++p) {
            int64_t i = base + p * (int)blockDim.x;
            if (i < npk) O::st(oc, i, O::scal(wv[p], sc));
        }
    }
}

// x += sum_j c_j V_j in FP64 (x complex128), j < min(J, kk[col]).
template <class T, int PKT>
__global__ void __launch_bounds__(NT) k_update_x(Basis<T> V, int J, const double2* coef, int cstride,
                                                 double2* x, int64_t xsr, int64_t npk,
                                                 const int* skip, const int* kk) {
    pdl_begin();
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    if (kk && kk[col] < J) J = kk[col];
    __shared__ double2 cs[MAXSLOT];
    for (int j = threadIdx.x; j < J; j += blockDim.x) cs[j] = coef[(int64_t)col * cstride + j];
    __syncthreads();
    double2* xc = x + col * xsr;
    const T* vb = V.base + col * V.sr;
    const int64_t base = (int64_t)blockIdx.x * blockDim.x * PKT + threadIdx.x;
    double2 acc[PKT][O::CPX];
#pragma unroll
    for (int p = 0; p < PKT; ++p)
#pragma unroll
        for (int q = 0; q < O::CPX; ++q) acc[p][q] = make_double2(0, 0);
    constexpr int UNR = 8 / PKT;
    for (int j0 = 0; j0 < J; j0 += UNR) {
        typename O::P q[UNR][PKT];
#pragma unroll
        for (int g = 0; g < UNR; ++g) {
            const T* vj = vb + (j0 + g) * V.sj;
#pragma unroll
            for (int p = 0; p < PKT; ++p) {
                const int64_t i = base + p * (int)blockDim.x;
                q[g][p] = (j0 + g < J && i < npk) ? O::ld_ro(vj, i) : O::zero();
            }
        }
#pragma unroll
        for (int g = 0; g < UNR; ++g)
            if (j0 + g < J)
#pragma unroll
                for (int p = 0; p < PKT; ++p) O::add_cv_f64(acc[p], cs[j0 + g], q[g][p]);
    }
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        const int64_t i = base + p * (int)blockDim.x;
        if (i >= npk) break;
#pragma unroll
        for (int q = 0; q < O::CPX; ++q) {
            double2 a = xc[i * O::CPX + q];
            xc[i * O::CPX + q] = make_double2(a.x + acc[p][q].x, a.y + acc[p][q].y);
        }
    }
}

// xs[i] += sum_j y_ij V_j for every shift i.  Each CTA takes one group of SG shifts for one
// tile of elements; the groups of a tile are consecutive CTAs (blockIdx.x = tile * ngrp + group),
// so they run together and the tile of V comes from HBM once, the other groups reading it from L2.
// SG = 2 by default (on the 10^4 workload 176 us per launch, against 193 us with SG = 4 and 253 us
// with SG = 8); with SG = 20 (all of the workloads' 20 poles in one CTA) the FP32 kernel needs 192
// registers and ran at half the speed.  Products and the sum over j in the
// storage precision; the add to xs in FP64.
template <class T, int SG>
__global__ void __launch_bounds__(NT) k_update_shifts(Basis<T> V, int J, const double2* y, int s,
                                                      int kmax, double2* xs, int64_t xs_shift,
                                                      int64_t xs_col, int64_t npk, const int* skip,
                                                      const int* kk) {
    pdl_begin();
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    if (kk && kk[col] < J) J = kk[col];
    const int ngrp = (s + SG - 1) / SG;
    const int64_t tile = blockIdx.x / (unsigned)ngrp;
    const int g0 = (int)(blockIdx.x - tile * ngrp) * SG;
    const int ng = (s - g0) < SG ? (s - g0) : SG;
    extern __shared__ unsigned char smraw[];
    typename O::C* ys = reinterpret_cast<typename O::C*>(smraw);  // [ng][J]: this CTA's shifts
    for (int t = threadIdx.x; t < ng * J; t += blockDim.x) {
        int i = t / J, j = t % J;
        ys[t] = O::coef(y[((int64_t)col * s + g0 + i) * kmax + j]);
    }
    __syncthreads();
    const int64_t i = tile * blockDim.x + threadIdx.x;
    if (i >= npk) return;
    const T* vb = V.base + col * V.sr;
    {
        typename O::P acc[SG];
#pragma unroll
        for (int g = 0; g < SG; ++g) acc[g] = O::zero();
        // loads of 4 basis vectors in flight together
        for (int j0 = 0; j0 < J; j0 += 4) {
            typename O::P v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = j0 + u < J ? O::ld_ro(vb + (j0 + u) * V.sj, i) : O::zero();
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j0 + u < J)
#pragma unroll
                    for (int g = 0; g < SG; ++g)
                        if (g < ng) O::add_cv(acc[g], ys[g * J + j0 + u], v[u]);
        }
#pragma unroll
        for (int g = 0; g < SG; ++g)
            if (g < ng) O::add_to(xs + (int64_t)(g0 + g) * xs_shift + col * xs_col, i, acc[g]);
    }
}

// Delayed CGS2, fused reduction of step j (Q = V_0..V_{J-1} orthonormal, u the
// once-orthogonalised candidate, z = A^2 u):  slots [0,J) s = Q^dag u,
// [J,2J) t = Q^dag z, 2J: u^dag u, 2J+1: u^dag z, 2J+2: z^dag z.  With z = null
// (the closing pass of a cycle) only s and u^dag u (slot J).
// FP32 storage (FP64: gs_f64.cu).
template <int PKT>
__global__ void __launch_bounds__(NT) k_dcgs_dots(Basis<float2> V, int J, const float2* u,
                                                  const float2* z, int64_t wsr, int64_t npk, Reduce rd,
                                                  const int* skip) {
    pdl_begin();
    using T = float2;
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T* uc = u + col * wsr;
    const T* zc = z ? z + col * wsr : nullptr;
    const int64_t base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    typename O::P uv[PKT], zv[PKT];
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        int64_t i = base + p * NT;
        uv[p] = i < npk ? O::ld(uc, i) : O::zero();
        zv[p] = (zc && i < npk) ? O::ld(zc, i) : O::zero();
    }
    const T* vb = V.base + col * V.sr;
    // FP32 storage: per-thread FP32 chunk partials are staged in shared memory
    // for a tile of TL basis vectors; each (vector, component) slot is then summed
    // over the whole CTA by one warp in double-float and written as this CTA's
    // FP64 partial.  Four values per vector: Re/Im of q^dag u and of q^dag z.
    constexpr int TL = 8;
    __shared__ float st[TL * 4][NT + 8];  // rows padded: the segmented sums below are bank-conflict free
    double* pd = reinterpret_cast<double*>(rd.partial);
    auto put = [&](int slot, int comp, double v) {
        pd[2 * (((int64_t)col * rd.stride + slot) * rd.nblk + blockIdx.x) + comp] = v;
    };
    const int nv = zc ? 4 : 2;
    // loads of GB basis vectors are issued together: 8 independent 16-byte
    // loads in flight per thread (4 with PKT = 4, whose registers hold 4 packs
    // of u and z already)
    constexpr int GB = PKT == 4 ? 1 : 8 / PKT;
    for (int l0 = 0; l0 < J; l0 += TL) {
        const int tl = (J - l0) < TL ? (J - l0) : TL;
#pragma unroll
        for (int g0 = 0; g0 < TL; g0 += GB) {
            if (g0 >= tl) break;
            typename O::P q[GB][PKT];
#pragma unroll
            for (int g = 0; g < GB; ++g) {
                const T* vl = vb + (l0 + g0 + g) * V.sj;
#pragma unroll
                for (int p = 0; p < PKT; ++p) {
                    const int64_t i = base + p * NT;
                    q[g][p] = (g0 + g < tl && i < npk) ? O::ld_ro(vl, i) : O::zero();
                }
            }
#pragma unroll
            for (int g = 0; g < GB; ++g) {
                if (g0 + g < tl) {
                    float sx = 0.f, sy = 0.f, tx = 0.f, ty = 0.f;
#pragma unroll
                    for (int p = 0; p < PKT; ++p) {
                        O::dot_acc(sx, sy, q[g][p], uv[p]);
                        if (zc) O::dot_acc(tx, ty, q[g][p], zv[p]);
                    }
                    st[(g0 + g) * 4 + 0][threadIdx.x] = sx;
                    st[(g0 + g) * 4 + 1][threadIdx.x] = sy;
                    st[(g0 + g) * 4 + 2][threadIdx.x] = tx;
                    st[(g0 + g) * 4 + 3][threadIdx.x] = ty;
                }
            }
        }
        __syncthreads();
        {
            // slot sl = tid / 8 (TL * 4 = 32 slots for 256 threads), summed by 8 lanes:
            // lane seg adds values seg, seg + 8, ... in FP32, then a 3-level shuffle
            // tree.  Every partial is a sum of at most a few hundred FP32 products
            // (error ~ eps_32 times the sum of their moduli, the rounding the FP32
            // products carry anyway); the sum over CTAs is FP64.
            static_assert(TL * 4 * 8 == NT, "one 8-lane group per slot");
            const int sl = threadIdx.x >> 3, seg = threadIdx.x & 7;
            float a = 0.f;
#pragma unroll
            for (int k = 0; k < NT / 8; ++k) a += st[sl][k * 8 + seg];
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            a += __shfl_xor_sync(0xffffffffu, a, 4);
            const int g = sl >> 2, v = sl & 3;
            if (seg == 0 && g < tl && v < nv) put(v < 2 ? l0 + g : J + l0 + g, v & 1, (double)a);
        }
        __syncthreads();
    }
    // norms and u^dag z
    float a = 0.f, bx = 0.f, by = 0.f, gz = 0.f;
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        O::nrm2_acc(a, uv[p]);
        if (zc) {
            O::dot_acc(bx, by, uv[p], zv[p]);
            O::nrm2_acc(gz, zv[p]);
        }
    }
    st[0][threadIdx.x] = a;
    st[1][threadIdx.x] = bx;
    st[2][threadIdx.x] = by;
    st[3][threadIdx.x] = gz;
    __syncthreads();
    const int bs = zc ? 2 * J : J;
    if (warp < (zc ? 4 : 1)) {
        const double r = cta_sum_df<NT>(st[warp], lane);
        if (lane == 0) {
            if (warp == 0) {
                put(bs, 0, r);
                put(bs, 1, 0.0);
            } else if (warp == 1) {
                put(bs + 1, 0, r);
            } else if (warp == 2) {
                put(bs + 1, 1, r);
            } else {
                put(bs + 2, 0, r);
                put(bs + 2, 1, 0.0);
            }
        }
    }
}

// Delayed CGS2, update of step j:  q_j = (u - Q s) / rho  (written over u), and
// the next candidate  u_{j+1} = z / rho - Q c - d q_j  (when next != null).
// Coefficients per column: [0,J) s, [J,2J) c, 2J: (1/rho, 0), 2J+1: d.
// FP32 storage (FP64: gs_f64.cu).
template <int PKT>
__global__ void __launch_bounds__(NT) k_dcgs_update(Basis<float2> V, int J, const double2* coef,
                                                    int cstride, float2* u, const float2* z, float2* next,
                                                    int64_t wsr, int64_t npk, double2* H, int km,
                                                    const int* skip) {
    pdl_begin();
    using T = float2;
    using O = Ops<T>;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    if (H && blockIdx.x == 0) {  // one CTA per column forms the Hessenberg column beside the update
        hess_column(H + (int64_t)col * (km + 1) * km, coef + (int64_t)col * cstride, J, km);
        return;
    }
    const int tile = H ? blockIdx.x - 1 : blockIdx.x;
    __shared__ typename O::C cs[MAXSLOT], cc[MAXSLOT];
    __shared__ double ex[2][2];
    const double2* cf = coef + (int64_t)col * cstride;
    for (int l = threadIdx.x; l < J; l += NT) {
        cs[l] = O::coef(cf[l]);
        cc[l] = O::coef(cf[J + l]);
    }
    if (threadIdx.x == 0) {
        ex[0][0] = cf[2 * J].x;
        ex[1][0] = cf[2 * J + 1].x;
        ex[1][1] = cf[2 * J + 1].y;
    }
    __syncthreads();
    const float inv_rho_f = (float)ex[0][0];
    const typename O::C dd = O::coef(make_double2(ex[1][0], ex[1][1]));
    T* uc = u + col * wsr;
    const T* zc = next ? z + col * wsr : nullptr;
    T* nc = next ? next + col * wsr : nullptr;
    const T* vb = V.base + col * V.sr;
    const int64_t base = (int64_t)tile * NT * PKT + threadIdx.x;
    // Q s and Q c with the basis loop outside: the loads of UNR basis vectors
    // (PKT packs each) are independent and in flight together
    typename O::P qs[PKT], qc[PKT];
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        qs[p] = O::zero();
        qc[p] = O::zero();
    }
    constexpr int UNR = 8 / PKT;
    for (int l0 = 0; l0 < J; l0 += UNR) {
        typename O::P q[UNR][PKT];
#pragma unroll
        for (int g = 0; g < UNR; ++g) {
            const T* vl = vb + (l0 + g) * V.sj;
#pragma unroll
            for (int p = 0; p < PKT; ++p) {
                const int64_t i = base + p * NT;
                q[g][p] = (l0 + g < J && i < npk) ? O::ld_ro(vl, i) : O::zero();
            }
        }
#pragma unroll
        for (int g = 0; g < UNR; ++g) {
            if (l0 + g < J) {
                const typename O::C a = cs[l0 + g], c = cc[l0 + g];
#pragma unroll
                for (int p = 0; p < PKT; ++p) {
                    O::add_cv(qs[p], a, q[g][p]);
                    if (nc) O::add_cv(qc[p], c, q[g][p]);
                }
            }
        }
    }
    const typename O::C one = make_float2(1.0f, 0.0f);
#pragma unroll
    for (int p = 0; p < PKT; ++p) {
        const int64_t i = base + p * NT;
        if (i >= npk) break;
        typename O::P uv = O::ld(uc, i);
        // q_j = (u - qs) / rho
        O::sub_cv(uv, one, qs[p]);
        const typename O::P qj = O::scalf(uv, inv_rho_f);
        O::st(uc, i, qj);
        if (nc) {
            typename O::P nv = O::scalf(O::ld(zc, i), inv_rho_f);
            O::sub_cv(nv, one, qc[p]);
            O::sub_cv(nv, dd, qj);
            O::st(nc, i, nv);
        }
    }
}

// ---- second stage of the reductions ------------------------------------------
// A latency chain of one to a few CTAs per column, in FP64 instructions of 64 cycles each: sums with
// eight lanes per slot and the Hessenberg column formed beside the update took a step's reduction
// from 12.6 to 6 us (4^4 FP64, 6^4 mixed), 15.3 to 7.6 (7x6x9x8 x 3 FP64), 18 to 12 (10^4 x 12 mixed).
// LPS lanes per slot (8 slots of 8 lanes would fill a warp's FP64 instructions; one slot per warp
// where there are few): FP64 additions over the CTAs' partial sums in a fixed order.  Valid in
// every lane of the slot's group.
template <int LPS>
__device__ __forceinline__ double2 slot_sum(const Reduce& rd, int col, int slot, bool act) {
    const int seg = threadIdx.x % LPS;
    double2 a = make_double2(0, 0);
    if (act) {
        const double2* p = rd.partial + ((int64_t)col * rd.stride + slot) * rd.nblk;
#pragma unroll 8
        for (int b = seg; b < rd.nblk; b += LPS) a = cadd(a, p[b]);
    }
#pragma unroll
    for (int o = LPS / 2; o > 0; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    }
    return a;
}

// RM_STORE and RM_SIGNED: every slot on its own.  Grid (column, NT / LPS slots).
template <int LPS>
__global__ void __launch_bounds__(NT) k_reduce_store(Reduce rd, int nslot, int mode, DevState S,
                                                     const double2* lambda) {
    pdl_begin();
    const int col = blockIdx.x;
    if (S.skip[col]) return;
    const int j = (blockIdx.y * NT + threadIdx.x) / LPS;
    double2 a = slot_sum<LPS>(rd, col, j, j < nslot);
    if (j >= nslot || threadIdx.x % LPS) return;
    if (mode == RM_SIGNED && !(lambda[j].x > 0)) a = make_double2(-a.x, -a.y);
    S.red[(int64_t)col * S.rstride + j] = a;
}

// The scalar work of a reduction once the slot sums of column col are known
// (sums: shared memory, nslot entries).  Called by every thread of one CTA.
__device__ void reduce_tail(const double2* sums, int col, int nslot, int mode, int colidx, const DevState& S) {
    const int64_t cr = (int64_t)col * S.rstride;
    switch (mode) {
        case RM_H1:
            for (int j = threadIdx.x; j < nslot - 1; j += NT) S.h1[cr + j] = sums[j];
            if (threadIdx.x == 0) S.norm0[col] = sqrt(sums[nslot - 1].x);
            break;
        case RM_P2: {
            const int J = nslot - 1;  // = colidx + 1
            const int64_t hb = (int64_t)col * (S.kmax + 1) * S.kmax;
            for (int l = threadIdx.x; l < J; l += NT) {
                S.red[cr + l] = sums[l];
                S.H[hb + (int64_t)l * S.kmax + colidx] = cadd(S.h1[cr + l], sums[l]);
            }
            if (threadIdx.x == 0) {
                double h2 = 0;
                for (int l = 0; l < J; ++l) h2 += cabs2(sums[l]);
                double hn2 = sums[J].x - h2;
                double hn = hn2 > 0 ? sqrt(hn2) : 0.0;
                S.H[hb + (int64_t)(colidx + 1) * S.kmax + colidx] = make_double2(hn, 0);
                if (!(hn > S.bd_tol * S.norm0[col])) {
                    S.kk[col] = colidx + 1;
                    S.skip[col] = 1;
                    S.scale[col] = 0;
                    if (!isfinite(hn2)) atomicOr(S.err, 2);
                } else {
                    S.scale[col] = 1.0 / hn;
                }
            }
            break;
        }
        case RM_DCGS:
        case RM_DCGS_FINAL: {
            // Delayed CGS2 bookkeeping of step j = colidx (see k_dcgs_dots for the slots).  Only
            // what the update of the step waits for is done here: rho, the coefficients s, c = t / rho
            // and d = (u^dag z - s^dag t) / rho^2, and s added to column j - 1 of H.  The tentative
            // column j, which takes j^2 / 2 products, is formed beside the update (hess_column).
            // FP64 instructions take 64 cycles each here, so the three sums over l share one
            // reduction, and rho and ||z|| one rsqrt (lanes 0 and 1).
            const int j = colidx;
            const bool fin = mode == RM_DCGS_FINAL;
            const int km = S.kmax;
            double2* H = S.H + (int64_t)col * (km + 1) * km;
            __shared__ double ir_sh;
            __shared__ int broke_sh;
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            if (warp == 0) {
                // sum_l |s_l|^2 and sum_l conj(s_l) t_l, l < j
                double a[4] = {0.0, 0.0, 0.0, 0.0};
                for (int l = lane; l < j; l += 32) {
                    const double2 sl = sums[l];
                    a[0] = fma(sl.x, sl.x, a[0]);
                    a[0] = fma(sl.y, sl.y, a[0]);
                    if (!fin) {
                        const double2 t = sums[j + l];
                        a[1] = fma(sl.x, t.x, a[1]);
                        a[1] = fma(sl.y, t.y, a[1]);
                        a[2] = fma(sl.x, t.y, a[2]);
                        a[2] = fma(-sl.y, t.x, a[2]);
                    }
                }
                const double mine = reduce_few<4>(a, lane);  // lane l: sum l mod 4
                const double stx = __shfl_sync(0xffffffffu, mine, 1), sty = __shfl_sync(0xffffffffu, mine, 2);
                const double v = lane == 0 ? sums[fin ? j : 2 * j].x - mine : fin ? 0.0 : sums[2 * j + 2].x;
                const double rs = v > 0 ? rsqrt(v) : 0.0;
                const double root = v > 0 ? v * rs : 0.0;  // lane 0: rho, lane 1: ||z||
                const double nz = __shfl_sync(0xffffffffu, root, 1);
                if (lane == 0) {
                    int broke = j == 0 ? !(root > 0) : !(root > S.bd_tol * S.norm0[col]);
                    if (j == 0)
                        S.beta[col] = root;
                    else
                        H[(int64_t)j * km + (j - 1)] = make_double2(root, 0);
                    if (!isfinite(v)) {
                        atomicOr(S.err, 2);
                        broke = 1;
                    }
                    // closing pass: q_k = (u - Q s) / rho; an invariant Krylov space (rho ~ 0) leaves
                    // q_k = 0, so the restart norm is 0 and the column converges
                    const double ir = broke ? 0.0 : rs;
                    S.red[cr + 2 * j] = make_double2(ir, 0);
                    if (!fin) {
                        if (broke) {  // the Krylov space is invariant: FOM on its j columns is exact
                            S.kk[col] = j;
                            S.skip[col] = 1;
                        } else {
                            const double2 b = sums[2 * j + 1];
                            S.red[cr + 2 * j + 1] = make_double2((b.x - stx) * ir * ir, (b.y - sty) * ir * ir);
                            S.norm0[col] = nz * ir;  // ~ ||A^2 q_j|| for the next breakdown test
                        }
                    }
                    ir_sh = ir;
                    broke_sh = broke;
                }
            } else if (threadIdx.x - 32 < j) {  // column j - 1: H[0:j, j-1] += s (j <= 64 < NT - 32)
                const int l = threadIdx.x - 32;
                double2* h = H + (int64_t)l * km + (j - 1);
                *h = cadd(*h, sums[l]);
                S.red[cr + l] = sums[l];
            }
            __syncthreads();
            if (fin || broke_sh) break;
            const double ir = ir_sh;
            for (int l = threadIdx.x; l < j; l += NT)
                S.red[cr + j + l] = make_double2(sums[j + l].x * ir, sums[j + l].y * ir);
            break;
        }
        case RM_BETA_FIRST: {
            const double beta = sqrt(sums[0].x);
            for (int i = threadIdx.x; i < S.s; i += NT) S.rho[(int64_t)col * S.s + i] = make_double2(1, 0);
            if (threadIdx.x == 0) {
                S.beta[col] = beta;
                S.bnorm[col] = beta;
                S.kk[col] = S.kmax;
                if (!isfinite(beta)) atomicOr(S.err, 2);
                if (beta > 0 && isfinite(beta)) {
                    S.scale[col] = 1.0 / beta;
                    S.resest[col] = 1.0;
                    S.skip[col] = 0;
                    S.done[col] = 0;
                } else {
                    S.scale[col] = 0;
                    S.resest[col] = 0;
                    S.skip[col] = 1;
                    S.done[col] = 1;
                }
            }
            break;
        }
        case RM_BETA_RESTART:
            if (threadIdx.x < 32) {
                // max_i |rho_i|^2, lanes over the shifts
                double m = 0;
                for (int i = threadIdx.x; i < S.s; i += 32) {
                    const double a = cabs2(S.rho[(int64_t)col * S.s + i]);
                    m = a > m ? a : m;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const double a = __shfl_xor_sync(0xffffffffu, m, o);
                    m = a > m ? a : m;
                }
                if (threadIdx.x != 0) break;
                if (S.kk[col] < S.kmax) {  // invariant subspace met: FOM is exact
                    S.resest[col] = 0;
                    S.done[col] = 1;
                    S.skip[col] = 1;
                    S.scale[col] = 0;
                    break;
                }
                const double beta = sqrt(sums[0].x);
                const double rmax = sqrt(m) * beta / S.bnorm[col];
                S.beta[col] = beta;
                S.resest[col] = rmax;
                if (!isfinite(rmax)) {
                    atomicOr(S.err, 2);
                    S.done[col] = 1;
                    S.skip[col] = 1;
                    S.scale[col] = 0;
                    break;
                }
                const int conv = rmax <= S.tol || beta == 0;
                S.done[col] = conv;
                S.skip[col] = conv;
                S.scale[col] = beta > 0 ? 1.0 / beta : 0.0;
            }
            break;
    }
}

// Slot sums, then the column's scalar work.  CTA (col, g) sums slots g * NT / LPS ...; the CTAs of a
// column form a cluster, write their sums into the shared memory of the first one, and that one
// does the scalar work after the cluster's barrier: latency bound (an arrival counter with fences
// and the sums through L2 instead: the 4^4 FP64 solve took 4.69 ms, now 4.59; CTAs of 128 threads,
// one warp of additions per SM sub-partition: 4.60).
template <int LPS>
__global__ void __launch_bounds__(NT) k_reduce(Reduce rd, int nslot, int mode, int colidx, DevState S) {
    pdl_begin();
    const int col = blockIdx.x;
    // RM_BETA_FIRST starts a solve; RM_BETA_RESTART must still see columns that
    // broke down in this cycle; every other mode is column work proper.
    if (mode == RM_BETA_RESTART && S.done[col]) return;
    if (mode != RM_BETA_FIRST && mode != RM_BETA_RESTART && S.skip[col]) return;
    __shared__ double2 sums[MAXSLOT];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const bool split = gridDim.y > 1;  // = the cluster
    double2* to = split ? cl.map_shared_rank(sums, 0) : sums;
    if (split) cl.barrier_arrive();
    const int j = blockIdx.y * (NT / LPS) + threadIdx.x / LPS;
    const double2 a = slot_sum<LPS>(rd, col, j, j < nslot);
    if (split) cl.barrier_wait();  // the first CTA is running
    if (j < nslot && threadIdx.x % LPS == 0) to[j] = a;
    if (split)
        cl.sync();
    else
        __syncthreads();
    if (blockIdx.y) return;
    reduce_tail(sums, col, nslot, mode, colidx, S);
}

// out = a x + b y + c z on whole blocks (real coefficients; z may be null).
template <class T>
__global__ void __launch_bounds__(NT) k_axpby3(T* __restrict__ out, double a, const T* __restrict__ x, double b,
                                               const T* __restrict__ y, double c, const T* __restrict__ z,
                                               int64_t npk) {
    using O = Ops<T>;
    const float af = (float)a, bf = (float)b, cf = (float)c;  // FP32 path: convert once
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < npk; i += (int64_t)gridDim.x * NT) {
        typename O::P r;
        if constexpr (O::CPX == 1) {
            typename O::P v = O::scal(O::ld(x, i), a);
            typename O::P w = O::scal(O::ld(y, i), b);
            r = make_double2(v.x + w.x, v.y + w.y);
            if (z) {
                typename O::P u = O::scal(O::ld(z, i), c);
                r = make_double2(r.x + u.x, r.y + u.y);
            }
        } else {
            typename O::P v = O::scalf(O::ld(x, i), af);
            typename O::P w = O::scalf(O::ld(y, i), bf);
            r = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
            if (z) {
                typename O::P u = O::scalf(O::ld(z, i), cf);
                r = make_float4(r.x + u.x, r.y + u.y, r.z + u.z, r.w + u.w);
            }
        }
        O::st(out, i, r);
    }
}

// Z_j = sum_i C[i][j] Y_i  (Y: q fields, Z: r fields, each n complex apart; C row-major q x r),
// SG output fields per sweep of Y.
constexpr int SG = 8;
template <class T>
__global__ void __launch_bounds__(NT) k_block_combine(const T* __restrict__ Y, int q, const double2* __restrict__ Cm,
                                                      int r, T* __restrict__ Z, int64_t n, int64_t npk) {
    using O = Ops<T>;
    __shared__ typename O::C cs[MAXSLOT * SG];
    const int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x;
    for (int g0 = 0; g0 < r; g0 += SG) {
        const int ng = (r - g0) < SG ? (r - g0) : SG;
        __syncthreads();
        for (int t = threadIdx.x; t < q * SG; t += NT) {
            int a = t / SG, g = t % SG;
            cs[t] = g < ng ? O::coef(Cm[(int64_t)a * r + g0 + g]) : O::coef(make_double2(0, 0));
        }
        __syncthreads();
        if (i < npk) {
            typename O::P acc[SG];
#pragma unroll
            for (int g = 0; g < SG; ++g) acc[g] = O::zero();
            for (int a = 0; a < q; ++a) {
                typename O::P v = O::ld_ro(Y + a * n, i);
#pragma unroll
                for (int g = 0; g < SG; ++g) O::add_cv(acc[g], cs[a * SG + g], v);
            }
#pragma unroll
            for (int g = 0; g < SG; ++g)
                if (g < ng) O::st(Z + (int64_t)(g0 + g) * n, i, acc[g]);
        }
    }
}

// Counter-based Gaussian start vectors: SplitMix64 of (seed, index), Box-Muller.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}
template <class T>
__global__ void k_random_fill(T* out, int64_t count, uint64_t seed) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t h1 = splitmix64(seed ^ (2 * (uint64_t)i)), h2 = splitmix64(seed ^ (2 * (uint64_t)i + 1));
        double u1 = ((h1 >> 11) + 1.0) * (1.0 / 9007199254740993.0);
        double u2 = (h2 >> 11) * (1.0 / 9007199254740992.0);
        double rr = sqrt(-2.0 * log(u1));
        double re = rr * cos(6.283185307179586 * u2), im = rr * sin(6.283185307179586 * u2);
        if constexpr (sizeof(T) == 16) {
            out[i] = T{re, im};
        } else {
            out[i] = T{(float)re, (float)im};
        }
    }
}

__global__ void k_f64_to_f32(const double2* __restrict__ in, float2* __restrict__ out, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = in[i];
        out[i] = make_float2(d2f(v.x), d2f(v.y));
    }
}
__global__ void k_f32_to_f64(const float2* __restrict__ in, double2* __restrict__ out, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        float2 v = in[i];
        out[i] = make_double2(f2d(v.x), f2d(v.y));
    }
}
__global__ void k_f64_to_bf16(const double2* __restrict__ in, __nv_bfloat162* __restrict__ out, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = in[i];
        out[i] = __floats2bfloat162_rn(d2f(v.x), d2f(v.y));
    }
}
// FP16 links: SU(3) entries have modulus <= 1, inside FP16's normal range (one rounding
// from FP32; entries below 6e-5 in modulus lose relative precision as subnormals, which
// costs at most 6e-8 absolute per entry)
__global__ void k_f64_to_f16(const double2* __restrict__ in, __half2* __restrict__ out, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = in[i];
        out[i] = __floats2half2_rn(d2f(v.x), d2f(v.y));
    }
}

// y_f = a_f + beta gamma5 s_f for nfield packed complex128 fields of vol sites: gamma5 =
// diag(1, 1, -1, -1) in spin negates spins 2 and 3, i.e. planes 3..5 of the packed
// field, its second half.
__global__ void k_gamma5_axpy(double2* __restrict__ y, const double2* __restrict__ a, const double2* __restrict__ sv,
                              double beta, int64_t half, int64_t total) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i % (2 * half);
        const double g = e < half ? beta : -beta;
        const double2 av = a[i], v = sv[i];
        y[i] = make_double2(av.x + g * v.x, av.y + g * v.y);
    }
}

inline unsigned grid_for(int64_t count) {
    int64_t g = (count + 255) / 256;
    if (g > 152 * 16) g = 152 * 16;
    if (g < 1) g = 1;
    return (unsigned)g;
}

}  // namespace

template <class T>
int reduce_blocks(int64_t n) {
    int64_t npk = n / Ops<T>::CPX;
    int64_t b = (npk + (int64_t)NT * PK - 1) / ((int64_t)NT * PK);
    return (int)(b < 1 ? 1 : b);
}

namespace {
int sm_count() {
    static const int n = [] {
        int d = 0, v = 0;
        if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d) != cudaSuccess)
            v = 0;
        return v > 0 ? v : 152;
    }();
    return n;
}

// Packs per thread that nblk CTAs per column need for npk packs (0: too few CTAs).
int pk_for(int64_t npk, int nblk) {
    for (int pk = 1; pk <= 4; pk *= 2)
        if ((int64_t)NT * pk * nblk >= npk) return pk;
    return 0;
}
}  // namespace

// The vector kernels hold 4 CTAs of NT threads per SM (64 registers, 32 KB of
// shared memory).  A grid of 1.16 waves runs as long as 2 waves, so the CTAs per
// column are picked from PKT = 4, 2, 1 (in that order of preference) for a grid
// that fills at least 85 % of its last wave, else the fullest.
template <class T>
int wave_blocks(int64_t n, int ncol) {
    const int64_t npk = n / Ops<T>::CPX;
    const int64_t slots = (int64_t)sm_count() * 4;
    int best = 1;
    double best_eff = -1.0;
    for (int pk = 4; pk >= 1; pk /= 2) {
        int64_t nb = (npk + (int64_t)NT * pk - 1) / ((int64_t)NT * pk);
        if (nb < 1) nb = 1;
        const double waves = (double)(nb * (ncol > 0 ? ncol : 1)) / (double)slots;
        const double eff = waves / std::ceil(waves);
        if (eff >= 0.85) return (int)nb;
        if (eff > best_eff) {
            best_eff = eff;
            best = (int)nb;
        }
    }
    return best;
}

namespace {
// CTAs per column, threads per CTA and packs per thread of the update kernels (one thread's
// elements, all basis vectors).  FP32: whole waves of 256 threads.  FP64: those kernels are bound
// by the two FP64 lanes of an SM, so what counts is that every SM gets the same number of warps:
// one element per thread in CTAs of two warps, or of one while that leaves SMs without a CTA.
struct Split {
    int nb, threads, pkt;
};
template <class T>
Split split_for(int64_t n, int ncol) {
    if constexpr (Ops<T>::CPX == 1) {
        const int threads = n * ncol < 64 * kFewWarps ? 32 : 64;
        return {(int)((n + threads - 1) / threads), threads, 1};
    } else {
        const int nb = wave_blocks<T>(n, ncol);
        return {nb, NT, pk_for(n / Ops<T>::CPX, nb)};
    }
}
}  // namespace

// Instantiate the kernel call for PKT = 1, 2 or 4.
#define SGN_PK_SWITCH(PKV, ...)               \
    switch (PKV) {                            \
        case 1: {                             \
            constexpr int PKT_ = 1;           \
            __VA_ARGS__;                      \
            break;                            \
        }                                     \
        case 2: {                             \
            constexpr int PKT_ = 2;           \
            __VA_ARGS__;                      \
            break;                            \
        }                                     \
        case 4: {                             \
            constexpr int PKT_ = 4;           \
            __VA_ARGS__;                      \
            break;                            \
        }                                     \
        default:                              \
            return cudaErrorInvalidValue;     \
    }

template <>
cudaError_t mdot<float2>(Basis<float2> V, int J, const float2* w, int64_t wsr, int64_t n, int ncol, const Reduce& rd,
                         int with_norm, const int* skip, cudaStream_t st) {
    if (J + 1 > MAXSLOT) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<float2>::CPX;
    dim3 grid(rd.nblk, ncol);
    SGN_PK_SWITCH(pk_for(npk, rd.nblk), launch_pdl(k_mdot<PKT_>, grid, NT, 0, st, V, J, w, wsr, npk, rd, with_norm, skip))
    count_launch();
    return cudaGetLastError();
}

cudaError_t reduce(const Reduce& rd, int nslot, int ncol, int mode, int colidx, const DevState& S,
                   const double2* lambda, cudaStream_t st) {
    if (nslot > MAXSLOT) return cudaErrorInvalidValue;
    const bool few = nslot <= NWARP;
    const int groups = few ? 1 : (nslot + NT / 8 - 1) / (NT / 8);
    if (mode == RM_STORE || mode == RM_SIGNED) {
        if (few)
            launch_pdl(k_reduce_store<32>, dim3(ncol, groups), NT, 0, st, rd, nslot, mode, S, lambda);
        else
            launch_pdl(k_reduce_store<8>, dim3(ncol, groups), NT, 0, st, rd, nslot, mode, S, lambda);
    } else {
        auto k = few ? k_reduce<32> : k_reduce<8>;
        launch_pdl_cluster(k, dim3(ncol, groups), NT, dim3(1, groups), st, rd, nslot, mode, colidx, S);
    }
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t maxpy_mdot(Basis<T> V, int J, const double2* coef, int cstride, T* w, int64_t wsr, int64_t n, int ncol,
                       const Reduce& rd, const int* skip, cudaStream_t st) {
    if (J + 1 > MAXSLOT) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<T>::CPX;
    dim3 grid(rd.nblk, ncol);
    SGN_PK_SWITCH(pk_for(npk, rd.nblk),
                  k_maxpy_mdot<T, PKT_><<<grid, NT, 0, st>>>(V, J, coef, cstride, w, wsr, npk, rd, skip))
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t maxpy_scale(Basis<T> V, int J, const double2* coef, int cstride, const T* w, int64_t wsr, T* out,
                        int64_t osr, const double* scale, int64_t n, int ncol, const int* skip, cudaStream_t st) {
    if (J > MAXSLOT) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<T>::CPX;
    const Split sp = split_for<T>(n, ncol);
    SGN_PK_SWITCH(sp.pkt, launch_pdl(k_maxpy_scale<T, PKT_>, dim3(sp.nb, ncol), sp.threads, 0, st, V, J, coef, cstride, w, wsr, out, osr,
                                                                              scale, npk, skip))
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t update_x(Basis<T> V, int J, const double2* coef, int cstride, double2* x, int64_t xsr, int64_t n,
                     int ncol, const int* skip, const int* kk, cudaStream_t st) {
    if (J > MAXSLOT) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<T>::CPX;
    const Split sp = split_for<T>(n, ncol);
    SGN_PK_SWITCH(sp.pkt,
                  launch_pdl(k_update_x<T, PKT_>, dim3(sp.nb, ncol), sp.threads, 0, st, V, J, coef, cstride, x, xsr, npk, skip, kk))
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t update_shifts(Basis<T> V, int J, const double2* y, int s, int kmax, double2* xs, int64_t xs_shift,
                          int64_t xs_col, int64_t n, int ncol, const int* skip, const int* kk, cudaStream_t st) {
    int64_t npk = n / Ops<T>::CPX;
    if (s <= 0 || npk <= 0) return cudaSuccess;
    // group size: SGN_SHIFT_GROUP = 1, 4, 8, 10 or 20 overrides the default 2 (measurements)
    static const int forced = [] {
        const char* e = getenv("SGN_SHIFT_GROUP");
        return e ? atoi(e) : 0;
    }();
    const int sg = (forced == 20 && s <= 20) || forced == 10 || forced == 8 || forced == 4 || forced == 1 ? forced : 2;
    size_t smem = sizeof(typename Ops<T>::C) * (size_t)(s < sg ? s : sg) * (size_t)J;
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    const int threads = split_for<T>(n, ncol).threads;
    const int64_t tiles = (npk + threads - 1) / threads;
    const int64_t nblk = tiles * ((s + sg - 1) / sg);
    if (nblk > 0x7fffffff) return cudaErrorInvalidValue;
    dim3 grid((unsigned)nblk, ncol);
    if (sg == 20)
        launch_pdl(k_update_shifts<T, 20>, grid, threads, smem, st, V, J, y, s, kmax, xs, xs_shift, xs_col, npk, skip, kk);
    else if (sg == 10)
        launch_pdl(k_update_shifts<T, 10>, grid, threads, smem, st, V, J, y, s, kmax, xs, xs_shift, xs_col, npk, skip, kk);
    else if (sg == 8)
        launch_pdl(k_update_shifts<T, 8>, grid, threads, smem, st, V, J, y, s, kmax, xs, xs_shift, xs_col, npk, skip, kk);
    else if (sg == 4)
        launch_pdl(k_update_shifts<T, 4>, grid, threads, smem, st, V, J, y, s, kmax, xs, xs_shift, xs_col, npk, skip, kk);
    else if (sg == 1)
        launch_pdl(k_update_shifts<T, 1>, grid, threads, smem, st, V, J, y, s, kmax, xs, xs_shift, xs_col, npk, skip, kk);
    else
        launch_pdl(k_update_shifts<T, 2>, grid, threads, smem, st, V, J, y, s, kmax, xs, xs_shift, xs_col, npk, skip, kk);
    count_launch();
    return cudaGetLastError();
}

template <>
cudaError_t dcgs_dots<float2>(Basis<float2> V, int J, const float2* u, const float2* z, int64_t wsr, int64_t n,
                              int ncol, const Reduce& rd, const int* skip, cudaStream_t st) {
    if (2 * J + 3 > MAXSLOT) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<float2>::CPX;
    dim3 grid(rd.nblk, ncol);
    SGN_PK_SWITCH(pk_for(npk, rd.nblk), launch_pdl(k_dcgs_dots<PKT_>, grid, NT, 0, st, V, J, u, z, wsr, npk, rd, skip))
    count_launch();
    return cudaGetLastError();
}

template <>
cudaError_t dcgs_update<float2>(Basis<float2> V, int J, const double2* coef, int cstride, float2* u, const float2* z,
                                float2* next, int64_t wsr, int64_t n, int ncol, double2* H, int km, const int* skip,
                                cudaStream_t st) {
    if (2 * J + 2 > MAXSLOT) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<float2>::CPX;
    const Split sp = split_for<float2>(n, ncol);
    const dim3 grid(sp.nb + (H ? 1 : 0), ncol);
    SGN_PK_SWITCH(sp.pkt, launch_pdl(k_dcgs_update<PKT_>, grid, sp.threads, 0, st, V, J, coef, cstride, u, z, next, wsr, npk, H,
                                                                          km, skip))
    count_launch();
    return cudaGetLastError();
}

cudaError_t gamma5_axpy(double2* y, const double2* a, const double2* s, double beta, int64_t vol, int nfield,
                        cudaStream_t st) {
    const int64_t total = (int64_t)nfield * 12 * vol;
    if (total <= 0) return cudaSuccess;
    k_gamma5_axpy<<<grid_for(total), NT, 0, st>>>(y, a, s, beta, 6 * vol, total);
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t axpby3(T* out, double a, const T* x, double b, const T* y, double c, const T* z, int64_t count,
                   cudaStream_t st) {
    int64_t npk = count / Ops<T>::CPX;
    k_axpby3<T><<<grid_for(npk), NT, 0, st>>>(out, a, x, b, y, c, z, npk);
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t block_combine(const T* Y, int q, const double2* Cm, int r, T* Z, int64_t n, cudaStream_t st) {
    if (q > MAXSLOT || r < 1) return cudaErrorInvalidValue;
    int64_t npk = n / Ops<T>::CPX;
    k_block_combine<T><<<(unsigned)((npk + NT - 1) / NT), NT, 0, st>>>(Y, q, Cm, r, Z, n, npk);
    count_launch();
    return cudaGetLastError();
}

template <class T>
cudaError_t random_fill(T* out, int64_t count, uint64_t seed, cudaStream_t st) {
    k_random_fill<T><<<grid_for(count), 256, 0, st>>>(out, count, seed);
    count_launch();
    return cudaGetLastError();
}

template cudaError_t axpby3<double2>(double2*, double, const double2*, double, const double2*, double,
                                     const double2*, int64_t, cudaStream_t);
template cudaError_t axpby3<float2>(float2*, double, const float2*, double, const float2*, double, const float2*,
                                    int64_t, cudaStream_t);
template cudaError_t block_combine<double2>(const double2*, int, const double2*, int, double2*, int64_t,
                                            cudaStream_t);
template cudaError_t block_combine<float2>(const float2*, int, const double2*, int, float2*, int64_t, cudaStream_t);
template cudaError_t random_fill<double2>(double2*, int64_t, uint64_t, cudaStream_t);
template cudaError_t random_fill<float2>(float2*, int64_t, uint64_t, cudaStream_t);

cudaError_t convert_f64_to_f32(const double2* in, float2* out, int64_t count, cudaStream_t st) {
    k_f64_to_f32<<<grid_for(count), 256, 0, st>>>(in, out, count);
    count_launch();
    return cudaGetLastError();
}
cudaError_t convert_f32_to_f64(const float2* in, double2* out, int64_t count, cudaStream_t st) {
    k_f32_to_f64<<<grid_for(count), 256, 0, st>>>(in, out, count);
    count_launch();
    return cudaGetLastError();
}
cudaError_t links_f64_to_bf16(const double2* in, __nv_bfloat162* out, int64_t count, cudaStream_t st) {
    k_f64_to_bf16<<<grid_for(count), 256, 0, st>>>(in, out, count);
    count_launch();
    return cudaGetLastError();
}
cudaError_t links_f64_to_f16(const double2* in, __half2* out, int64_t count, cudaStream_t st) {
    k_f64_to_f16<<<grid_for(count), 256, 0, st>>>(in, out, count);
    count_launch();
    return cudaGetLastError();
}

#define SGN_INST(T)                                                                                              \
    template int reduce_blocks<T>(int64_t);                                                                      \
    template int wave_blocks<T>(int64_t, int);                                                                   \
    template cudaError_t maxpy_mdot<T>(Basis<T>, int, const double2*, int, T*, int64_t, int64_t, int,           \
                                       const Reduce&, const int*, cudaStream_t);                                 \
    template cudaError_t maxpy_scale<T>(Basis<T>, int, const double2*, int, const T*, int64_t, T*, int64_t,     \
                                        const double*, int64_t, int, const int*, cudaStream_t);                  \
    template cudaError_t update_x<T>(Basis<T>, int, const double2*, int, double2*, int64_t, int64_t, int,       \
                                     const int*, const int*, cudaStream_t);                                      \
    template cudaError_t update_shifts<T>(Basis<T>, int, const double2*, int, int, double2*, int64_t, int64_t,  \
                                          int64_t, int, const int*, const int*, cudaStream_t);
SGN_INST(double2)
SGN_INST(float2)

}  // namespace sgn
