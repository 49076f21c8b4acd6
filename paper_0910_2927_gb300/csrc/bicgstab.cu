// Short-recurrence correction solves of the mixed form's refinement: (A^2 - sigma_c) d_c = r_c, one
// shifted system per column, by BiCGStab (van der Vorst 1992; complex arithmetic, shadow residual
// r_c) in FP32 fields with FP64 scalars.  The paper has no counterpart (it works in FP64); the
// multishift phase and the fallback of these solves are its restarted FOM.
//
// Why: the refinement's systems have different right-hand sides, so they share no Krylov space, and
// restarted FOM(16) reads and writes 28 fields per application of A^2 (16 + 8 of them for the
// orthogonalisation) and loses convergence at every restart.  BiCGStab moves 9 fields per
// application besides the two stencils' 4.5 and never restarts.  Every kernel below is bound by
// HBM (FP32, two complex numbers per 16-byte load), on small lattices by launch latency: 58 to 76 % of
// the DRAM rate on 120 systems of 8^4 (k_bi_t and k_bi_v wait for the CTA's sums between their loads).
// Measured: the refinement of the 10^4 x 12 solve (240 systems, tol 1e-10) 75 ms with FOM(16), about half
// of that now; the whole solve 133 -> 91 ms; the 6^4 x 1 solve 15.0 -> 11.2 ms when it came in.
//
// One iteration: w = A^2 p, k_bi_v, k_bi_s, t = A^2 s, k_bi_t, k_bi_x.  The shift enters as
// w - sigma p and t - sigma s where these are used.  Sums: FP32 within a thread (up to eight complex
// products), pairs of floats over a CTA, FP64 over the CTAs of a column, done by the column's last CTA to arrive (same sums whatever the order), which then forms
// the column's next coefficients: no kernel waits for another.
#include "blas.cuh"
#include "cvt.cuh"

namespace sgn {
namespace {

constexpr int NT = 256;
constexpr int MAXV = 7;  // real sums per kernel

__device__ __forceinline__ float4 ld(const float2* f, int64_t i) { return reinterpret_cast<const float4*>(f)[i]; }
__device__ __forceinline__ void st(float2* f, int64_t i, float4 v) { reinterpret_cast<float4*>(f)[i] = v; }
// w - sigma p
__device__ __forceinline__ float4 shifted(float4 w, float sigma, float4 p) {
    return make_float4(fmaf(-sigma, p.x, w.x), fmaf(-sigma, p.y, w.y), fmaf(-sigma, p.z, w.z), fmaf(-sigma, p.w, w.w));
}
// a + c b
__device__ __forceinline__ float4 axpy(float4 a, float2 c, float4 b) {
    return make_float4(fmaf(-c.y, b.y, fmaf(c.x, b.x, a.x)), fmaf(c.y, b.x, fmaf(c.x, b.y, a.y)),
                       fmaf(-c.y, b.w, fmaf(c.x, b.z, a.z)), fmaf(c.y, b.z, fmaf(c.x, b.w, a.w)));
}
// re, im += conj(a) b
__device__ __forceinline__ void dot(float& re, float& im, float4 a, float4 b) {
    re = fmaf(a.x, b.x, fmaf(a.y, b.y, re));
    re = fmaf(a.z, b.z, fmaf(a.w, b.w, re));
    im = fmaf(a.x, b.y, fmaf(-a.y, b.x, im));
    im = fmaf(a.z, b.w, fmaf(-a.w, b.z, im));
}
__device__ __forceinline__ void nrm(float& s, float4 a) {
    s = fmaf(a.x, a.x, fmaf(a.y, a.y, s));
    s = fmaf(a.z, a.z, fmaf(a.w, a.w, s));
}
__device__ __forceinline__ float2 to_f(double2 c) { return make_float2((float)c.x, (float)c.y); }
__device__ __forceinline__ bool fin(double2 c) { return isfinite(c.x) && isfinite(c.y); }
__device__ __forceinline__ double2 divc(double2 a, double2 b) {
    const double d = 1.0 / cabs2(b);
    return make_double2((a.x * b.x + a.y * b.y) * d, (a.y * b.x - a.x * b.y) * d);
}

// Adds v over the column's CTAs.  True in thread 0 of the last CTA to arrive, with the sums in tot.
template <int NV>
__device__ __forceinline__ bool column_sum(float (&v)[NV], const BiState& S, int col, double (&tot)[NV]) {
    __shared__ float sm[NV][NT];
    __shared__ double sd[NV];
    __shared__ int last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    static_assert(NV <= NT / 32, "a warp per sum");
#pragma unroll
    for (int k = 0; k < NV; ++k) sm[k][threadIdx.x] = v[k];
    __syncthreads();
    double* part = S.partial + (int64_t)col * MAXV * S.nblk;
    if (warp < NV) {
        const double a = cta_sum_df<NT>(sm[warp], lane);
        if (lane == 0) {
            part[warp * S.nblk + blockIdx.x] = a;
            __threadfence();  // visible device-wide before this CTA is counted
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&S.count[col], 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    if (warp < NV) {
        double a = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) a += __ldcg(part + warp * S.nblk + b);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) sd[warp] = a;
    }
    if (threadIdx.x == 0) S.count[col] = 0;  // ready for the next kernel
    __syncthreads();
    if (threadIdx.x != 0) return false;
#pragma unroll
    for (int k = 0; k < NV; ++k) tot[k] = sd[k];
    return true;
}

// 2^e, |e| <= 1022
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// fl32(2^-e v), two complex numbers
__device__ __forceinline__ float4 scaled_f32(const double2* f, int64_t i, double q) {
    const double2 a = f[2 * i], b = f[2 * i + 1];
    return make_float4(d2f(a.x * q), d2f(a.y * q), d2f(b.x * q), d2f(b.y * q));
}

// r = rt = p = fl32(2^-ex[col] src at off[col]), d = 0, rho = ||r||^2.  Columns from nb on are idle.
// The caller's 2^ex is the residual's size: the sums square FP32 numbers that go down to 1e-6 of it, so
// that unscaled residuals of right-hand sides of norm 1e-12 underflowed (three times the iterations,
// and at 1e-14 no convergence).
__global__ void __launch_bounds__(NT) k_bi_init(const double2* __restrict__ src, const long long* __restrict__ off,
                                                const int* __restrict__ ex, int nb, BiState S) {
    const int col = blockIdx.y;
    if (col >= nb) {
        if (blockIdx.x == 0 && threadIdx.x == 0) S.done[col] = BI_IDLE;
        return;
    }
    const double2* f = src + off[col];
    const double q = pow2(-ex[col]);
    const int64_t c = (int64_t)col * 2 * S.npk;
    float v[1] = {0.f};
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < S.npk; i += (int64_t)gridDim.x * NT) {
        const float4 r = scaled_f32(f, i, q);
        st(S.r + c, i, r);
        st(S.rt + c, i, r);
        st(S.p + c, i, r);
        st(S.d + c, i, make_float4(0.f, 0.f, 0.f, 0.f));
        nrm(v[0], r);
    }
    double tot[1];
    if (column_sum(v, S, col, tot)) {
        S.rho[col] = make_double2(tot[0], 0.0);
        S.lim[col] = S.tol[col] * S.tol[col] * tot[0];
        S.rn0[col] = tot[0];
        S.done[col] = !isfinite(tot[0]) ? BI_FAILED : tot[0] > 0 ? BI_RUN : BI_DONE;
    }
}

// alpha = rho / <rt, v>, v = w - sigma p
template <int PKT>
__global__ void __launch_bounds__(NT) k_bi_v(BiState S) {
    pdl_begin();
    const int col = blockIdx.y;
    if (S.done[col]) return;
    const int64_t c = (int64_t)col * 2 * S.npk, base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    const float sg = (float)S.sigma[col];
    float v[2] = {0.f, 0.f};
    float4 w[PKT], p[PKT], q[PKT];
#pragma unroll
    for (int k = 0; k < PKT; ++k) {
        const int64_t i = base + k * NT;
        if (i < S.npk) {
            w[k] = ld(S.w + c, i);
            p[k] = ld(S.p + c, i);
            q[k] = ld(S.rt + c, i);
        }
    }
#pragma unroll
    for (int k = 0; k < PKT; ++k)
        if (base + k * NT < S.npk) dot(v[0], v[1], q[k], shifted(w[k], sg, p[k]));
    double tot[2];
    if (column_sum(v, S, col, tot)) {
        const double2 rv = make_double2(tot[0], tot[1]);
        const double2 a = divc(S.rho[col], rv);
        S.alpha[col] = a;
        if (!fin(a)) S.done[col] = BI_FAILED;  // <rt, v> = 0, or not finite
    }
}

// s = r - alpha v
template <int PKT>
__global__ void __launch_bounds__(NT) k_bi_s(BiState S) {
    pdl_begin();
    const int col = blockIdx.y;
    if (S.done[col]) return;
    const int64_t c = (int64_t)col * 2 * S.npk, base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    const float sg = (float)S.sigma[col];
    const float2 al = to_f(S.alpha[col]), ma = make_float2(-al.x, -al.y);
    float4 w[PKT], p[PKT], r[PKT];
#pragma unroll
    for (int k = 0; k < PKT; ++k) {
        const int64_t i = base + k * NT;
        if (i < S.npk) {
            w[k] = ld(S.w + c, i);
            p[k] = ld(S.p + c, i);
            r[k] = ld(S.r + c, i);
        }
    }
#pragma unroll
    for (int k = 0; k < PKT; ++k)
        if (base + k * NT < S.npk) st(S.s + c, base + k * NT, axpy(r[k], ma, shifted(w[k], sg, p[k])));
}

// q = t - sigma s: omega = <q, s> / <q, q>, rho' = <rt, s> - omega <rt, q>, beta = rho' alpha / (rho omega)
template <int PKT>
__global__ void __launch_bounds__(NT) k_bi_t(BiState S) {
    pdl_begin();
    const int col = blockIdx.y;
    if (S.done[col]) return;
    const int64_t c = (int64_t)col * 2 * S.npk, base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    const float sg = (float)S.sigma[col];
    float v[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float4 t[PKT], s[PKT], h[PKT];
#pragma unroll
    for (int k = 0; k < PKT; ++k) {
        const int64_t i = base + k * NT;
        if (i < S.npk) {
            t[k] = ld(S.t + c, i);
            s[k] = ld(S.s + c, i);
            h[k] = ld(S.rt + c, i);
        }
    }
#pragma unroll
    for (int k = 0; k < PKT; ++k)
        if (base + k * NT < S.npk) {
            const float4 q = shifted(t[k], sg, s[k]);
            dot(v[0], v[1], q, s[k]);
            dot(v[2], v[3], h[k], s[k]);
            dot(v[4], v[5], h[k], q);
            nrm(v[6], q);
        }
    double tot[7];
    if (column_sum(v, S, col, tot)) {
        // q = 0 (with s = 0): r = s is the exact solution's residual, omega = 0 ends the column
        const double iq = tot[6] == 0 ? 0.0 : 1.0 / tot[6];
        const double2 om = make_double2(tot[0] * iq, tot[1] * iq);
        const double2 rho = csub(make_double2(tot[2], tot[3]), cmul(om, make_double2(tot[4], tot[5])));
        const double2 be = tot[6] == 0 ? make_double2(0, 0) : divc(cmul(rho, S.alpha[col]), cmul(S.rho[col], om));
        S.omega[col] = om;
        S.beta[col] = be;
        S.rho[col] = rho;
        if (!fin(om) || !fin(be)) S.done[col] = BI_FAILED;
    }
}

// d += alpha p + omega s, r = s - omega q, p = r + beta (p - omega v); convergence test on ||r||
template <int PKT>
__global__ void __launch_bounds__(NT) k_bi_x(BiState S) {
    pdl_begin();
    const int col = blockIdx.y;
    if (S.done[col]) return;
    const int64_t c = (int64_t)col * 2 * S.npk, base = (int64_t)blockIdx.x * NT * PKT + threadIdx.x;
    const float sg = (float)S.sigma[col];
    const float2 al = to_f(S.alpha[col]), om = to_f(S.omega[col]), be = to_f(S.beta[col]);
    const float2 mo = make_float2(-om.x, -om.y);
    float v[1] = {0.f};
    constexpr int H = PKT > 2 ? 2 : PKT;  // two packs' ten loads in flight at a time
#pragma unroll
    for (int k0 = 0; k0 < PKT; k0 += H) {
        float4 d[H], p[H], s[H], t[H], w[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const int64_t i = base + (k0 + k) * NT;
            if (i < S.npk) {
                d[k] = ld(S.d + c, i);
                p[k] = ld(S.p + c, i);
                s[k] = ld(S.s + c, i);
                t[k] = ld(S.t + c, i);
                w[k] = ld(S.w + c, i);
            }
        }
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const int64_t i = base + (k0 + k) * NT;
            if (i < S.npk) {
                st(S.d + c, i, axpy(axpy(d[k], al, p[k]), om, s[k]));
                const float4 r = axpy(s[k], mo, shifted(t[k], sg, s[k]));
                st(S.r + c, i, r);
                st(S.p + c, i, axpy(r, be, axpy(p[k], mo, shifted(w[k], sg, p[k]))));
                nrm(v[0], r);
            }
        }
    }
    double tot[1];
    if (column_sum(v, S, col, tot)) {
        const double rn = tot[0];
        if (rn <= S.lim[col])
            S.done[col] = BI_DONE;
        else if (!(rn < 1e6 * S.rn0[col]))  // diverging (or not finite): the caller's fallback
            S.done[col] = BI_FAILED;
    }
}

__device__ __forceinline__ double2 to_d(float2 v) { return make_double2(f2d(v.x), f2d(v.y)); }
__device__ __forceinline__ double2 to_d(double2 v) { return v; }
// x_j += 2^ex[j] d_j, x_j at x + off[j], d_j at j n; with done, for the converged systems.
template <class T>
__global__ void __launch_bounds__(NT) k_add_corrections(double2* __restrict__ x, const long long* __restrict__ off,
                                                        const int* __restrict__ ex, const int* __restrict__ done,
                                                        const T* __restrict__ d, int64_t n) {
    const int j = blockIdx.y;
    if (done && done[j] != BI_DONE) return;
    double2* xj = x + off[j];
    const T* dj = d + (int64_t)j * n;
    const double q = pow2(ex[j]);
    for (int64_t e = (int64_t)blockIdx.x * NT + threadIdx.x; e < n; e += (int64_t)gridDim.x * NT) {
        const double2 dv = to_d(dj[e]), xv = xj[e];
        xj[e] = make_double2(fma(q, dv.x, xv.x), fma(q, dv.y, xv.y));
    }
}
// out_j = fl32(2^-ex[j] src at off[j])
__global__ void __launch_bounds__(NT) k_scaled_residuals(const double2* __restrict__ src,
                                                         const long long* __restrict__ off,
                                                         const int* __restrict__ ex, float2* __restrict__ out,
                                                         int64_t npk) {
    const int j = blockIdx.y;
    const double q = pow2(-ex[j]);
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < npk; i += (int64_t)gridDim.x * NT)
        st(out + (int64_t)j * 2 * npk, i, scaled_f32(src + off[j], i, q));
}
dim3 field_grid(int64_t count, int nb) {
    const int64_t gx = (count + NT - 1) / NT;
    return dim3((unsigned)(gx < 1024 ? gx : 1024), nb);
}

template <class K1, class K2, class K4>
cudaError_t launch(const BiState& S, int ncol, cudaStream_t st, K1 k1, K2 k2, K4 k4) {
    const dim3 grid(S.nblk, ncol);
    switch (S.pkt) {
        case 1: launch_pdl(k1, grid, NT, 0, st, S); break;
        case 2: launch_pdl(k2, grid, NT, 0, st, S); break;
        case 4: launch_pdl(k4, grid, NT, 0, st, S); break;
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace

void bi_shape(BiState& S, int64_t n, int ncol) {
    S.npk = n / 2;
    S.nblk = wave_blocks<float2>(n, ncol);
    S.pkt = 1;
    while (S.pkt < 4 && (int64_t)NT * S.pkt * S.nblk < S.npk) S.pkt *= 2;
}
size_t bi_partial_bytes(const BiState& S, int ncol) { return sizeof(double) * MAXV * (size_t)S.nblk * ncol; }

cudaError_t bi_init(const BiState& S, int ncol, const double2* src, const long long* off, const int* ex, int nb,
                    cudaStream_t st) {
    k_bi_init<<<dim3(S.nblk, ncol), NT, 0, st>>>(src, off, ex, nb, S);
    count_launch();
    return cudaGetLastError();
}
cudaError_t bi_v(const BiState& S, int ncol, cudaStream_t st) {
    return launch(S, ncol, st, k_bi_v<1>, k_bi_v<2>, k_bi_v<4>);
}
cudaError_t bi_s(const BiState& S, int ncol, cudaStream_t st) {
    return launch(S, ncol, st, k_bi_s<1>, k_bi_s<2>, k_bi_s<4>);
}
cudaError_t bi_t(const BiState& S, int ncol, cudaStream_t st) {
    return launch(S, ncol, st, k_bi_t<1>, k_bi_t<2>, k_bi_t<4>);
}
cudaError_t bi_x(const BiState& S, int ncol, cudaStream_t st) {
    return launch(S, ncol, st, k_bi_x<1>, k_bi_x<2>, k_bi_x<4>);
}

template <class T>
cudaError_t add_corrections(double2* x, const long long* off, const int* ex, const int* done, const T* d, int64_t n,
                            int nb, cudaStream_t st) {
    if (nb < 1) return cudaSuccess;
    if (nb > 65535) return cudaErrorInvalidValue;
    k_add_corrections<T><<<field_grid(n, nb), NT, 0, st>>>(x, off, ex, done, d, n);
    count_launch();
    return cudaGetLastError();
}
template cudaError_t add_corrections<float2>(double2*, const long long*, const int*, const int*, const float2*,
                                             int64_t, int, cudaStream_t);
template cudaError_t add_corrections<double2>(double2*, const long long*, const int*, const int*, const double2*,
                                              int64_t, int, cudaStream_t);
cudaError_t scaled_residuals(const double2* src, const long long* off, const int* ex, float2* out, int64_t n, int nb,
                             cudaStream_t st) {
    if (nb < 1) return cudaSuccess;
    if (nb > 65535) return cudaErrorInvalidValue;
    k_scaled_residuals<<<field_grid(n / 2, nb), NT, 0, st>>>(src, off, ex, out, n / 2);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sgn
