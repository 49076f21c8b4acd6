// The FP64 Gram-Schmidt kernels: inner products of a basis with one or two fields per column (the
// coefficients of the Arnoldi relation eq. (2.4), the projection coefficients L^dag r of eq. (4.5),
// sgn_inner_products; first stage of the two-stage reductions of blas.cu) and the fused update of
// a delayed-CGS2 step.
//
// What bounds them: the FP64 pipe.  Each of an SM's four sub-partitions needs 64 cycles for a
// warp's FP64 instruction, and both kernels take 8 multiply-adds per basis entry of 16 bytes
// (1.25 TB/s of basis at the FP64 rate, a fifth of the HBM rate).  So (1) the sums over a warp must
// not cost more than the products: a warp keeps 32 sums (8 basis vectors x Re, Im x two fields,
// or 16 vectors x one field) over all its elements and adds them over the lanes by a
// reduce-scatter, 16 + 8 + 4 + 2 + 1 additions per lane that leave one finished sum in each (a
// butterfly per sum takes 5 each); (2) all 608 sub-partitions must get the same number of
// instructions: small lattices are split over CTAs by elements and by groups of basis vectors.
//
// Measured, us per launch averaged over the steps of a solve, before (one butterfly per sum, CTAs
// of 256 elements) and now.  Two-field products: 4^4 x 1 column 24.6 -> 7.0, 6^4 x 1 32.0 -> 16.6,
// 7x6x9x8 x 3 85.6 -> 42.5.  30 x 12 products on 16^4 (one field): 4472 -> 2055 (floor 1810: 8 flops
// per product at the FP64 rate; FP64 pipe 95 % busy).  Update: 4^4 x 1 10.8 -> 3.9, 6^4 x 1 13.4 -> 8.0.
#include "blas.cuh"

#include <algorithm>
#include <utility>

namespace sgn {
namespace {

constexpr int MAXW = 4;             // warps per CTA: one per sub-partition
constexpr int64_t PIPES = 4 * 152;  // sub-partitions of the chip

__device__ __forceinline__ void dot_acc(double& re, double& im, double2 v, double2 w) {  // += conj(v) w
    re = fma(v.x, w.x, re);
    re = fma(v.y, w.y, re);
    im = fma(v.x, w.y, im);
    im = fma(-v.y, w.x, im);
}

// NF = 2: slots [0, J) V^dag u, [J, 2J) V^dag z, 2J: u^dag u, 2J + 1: u^dag z, 2J + 2: z^dag z.
// NF = 1: slots [0, J) V^dag u and, with norm, J: u^dag u.
// CTA (b, col, part): elements [b per, (b + 1) per), vector groups part, part + gridDim.z, ...
// E elements per thread and chunk of the CTA's elements.
template <int NF, int E>
__global__ void __launch_bounds__(32 * MAXW, 3)
    k_dots_f64(Basis<double2> V, int J, const double2* u, const double2* z, int64_t wsr,
               int64_t n, int64_t per, Reduce rd, int norm, const int* skip) {
    pdl_begin();
    constexpr int VG = 16 / NF;
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    __shared__ double red[2][MAXW][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = b0 + per < n ? b0 + per : n;
    const int step = blockDim.x * E;
    const double2* uc = u + col * wsr;
    const double2* zc = NF == 2 ? z + col * wsr : nullptr;
    const double2* vb = V.base + col * V.sr;
    double* pd = reinterpret_cast<double*>(rd.partial);
    auto put = [&](int slot, int comp, double v) {
        pd[2 * (((int64_t)col * rd.stride + slot) * rd.nblk + blockIdx.x) + comp] = v;
    };
    auto load = [&](double2 (&q)[E], const double2* f, int64_t c0) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int64_t i = c0 + threadIdx.x + e * (int)blockDim.x;
            q[e] = i < b1 ? f[i] : make_double2(0, 0);
        }
    };
    auto cta_sum = [&](double r, int buf) {  // valid in warp 0
        if (W == 1) return r;
        red[buf][warp][lane] = r;
        __syncthreads();
        if (warp == 0)
            for (int w = 1; w < W; ++w) r += red[buf][w][lane];
        return r;
    };
    int buf = 0;
    for (int l0 = blockIdx.z * VG; l0 < J; l0 += gridDim.z * VG) {
        const int tl = J - l0 < VG ? J - l0 : VG;
        double a[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) a[i] = 0.0;
        for (int64_t c0 = b0; c0 < b1; c0 += step) {
            double2 uv[E], zv[E], q[E], nx[E];
            load(uv, uc, c0);
            if constexpr (NF == 2) load(zv, zc, c0);
            load(q, vb + l0 * V.sj, c0);
#pragma unroll
            for (int v = 0; v < VG; ++v) {
                if (v < tl) {
                    if (v + 1 < tl) load(nx, vb + (l0 + v + 1) * V.sj, c0);  // one vector ahead
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        dot_acc(a[2 * NF * v], a[2 * NF * v + 1], q[e], uv[e]);
                        if constexpr (NF == 2) dot_acc(a[4 * v + 2], a[4 * v + 3], q[e], zv[e]);
                    }
#pragma unroll
                    for (int e = 0; e < E; ++e) q[e] = nx[e];
                }
            }
        }
        const double r = cta_sum(reduce_scatter<32>(a, lane), buf);
        buf ^= 1;
        const int v = lane / (2 * NF), f = (lane >> 1) & (NF - 1);
        if (warp == 0 && v < tl) put(f * J + l0 + v, lane & 1, r);
    }
    if (norm && blockIdx.z == gridDim.z - 1) {
        double a[4] = {0.0, 0.0, 0.0, 0.0};  // u^dag u, Re and Im u^dag z, z^dag z
        for (int64_t c0 = b0; c0 < b1; c0 += step) {
            double2 uv[E], zv[E];
            load(uv, uc, c0);
            if constexpr (NF == 2) load(zv, zc, c0);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                a[0] = fma(uv[e].x, uv[e].x, a[0]);
                a[0] = fma(uv[e].y, uv[e].y, a[0]);
                if constexpr (NF == 2) {
                    dot_acc(a[1], a[2], uv[e], zv[e]);
                    a[3] = fma(zv[e].x, zv[e].x, a[3]);
                    a[3] = fma(zv[e].y, zv[e].y, a[3]);
                }
            }
        }
        const double r = cta_sum(reduce_few<4>(a, lane), buf);
        if (warp == 0 && lane < 4) {
            if (lane == 0) put(NF * J, 0, r);
            if (lane == 3) put(NF * J, 1, 0.0);
            if constexpr (NF == 2) {
                if (lane == 1 || lane == 2) put(2 * J + 1, lane - 1, r);
                if (lane == 3) put(2 * J + 2, 0, r);
                if (lane == 0) put(2 * J + 2, 1, 0.0);
            }
        }
    }
}

// Parts into which the vector groups are best split, and the groups that the busiest sub-partition
// then works through, for the given warps per part.
std::pair<int, int64_t> rounds(int64_t warps, int groups) {
    std::pair<int, int64_t> best{1, INT64_MAX};
    for (int p = 1; p <= groups; ++p) {
        const int64_t t = (warps * p + PIPES - 1) / PIPES * ((groups + p - 1) / p);
        if (t < best.second) best = {p, t};
    }
    return best;
}

template <int NF>
cudaError_t launch(Basis<double2> V, int J, const double2* u, const double2* z, int64_t wsr, int64_t n, int ncol,
                   const Reduce& rd, int norm, const int* skip, cudaStream_t st) {
    if (J * NF + (NF == 2 ? 3 : 1) > kMaxSlots) return cudaErrorInvalidValue;
    const int64_t per = (n + rd.nblk - 1) / rd.nblk;
    const int threads = per > 64 ? 128 : per > 32 ? 64 : 32;
    // vector groups as a grid dimension where that shortens the busiest sub-partition's work
    const int64_t warps = (int64_t)rd.nblk * ncol * (threads / 32);
    const int groups = std::max(1, (J * NF + 15) / 16);
    const dim3 grid(rd.nblk, ncol, rounds(warps, groups).first);
    if (per <= 128)
        launch_pdl(k_dots_f64<NF, 1>, grid, threads, 0, st, V, J, u, z, wsr, n, per, rd, norm, skip);
    else if (per <= 256)
        launch_pdl(k_dots_f64<NF, 2>, grid, threads, 0, st, V, J, u, z, wsr, n, per, rd, norm, skip);
    else
        launch_pdl(k_dots_f64<NF, 4>, grid, threads, 0, st, V, J, u, z, wsr, n, per, rd, norm, skip);
    count_launch();
    return cudaGetLastError();
}

// Update of a delayed-CGS2 step (see k_dcgs_update in blas.cu for the coefficients), S warps per
// 32 elements: warp w takes the basis vectors w, w + S, ..., and warp 0 adds their sums.
template <int S>
__global__ void __launch_bounds__(S == 1 ? 64 : 32 * S)
    k_dcgs_update_f64(Basis<double2> V, int J, const double2* coef, int cstride, double2* u,
                      const double2* z, double2* next, int64_t wsr, int64_t n, double2* H, int km,
                      const int* skip) {
    pdl_begin();
    const int col = blockIdx.y;
    if (skip && skip[col]) return;
    if (H && blockIdx.x == 0) {  // one CTA per column forms the Hessenberg column beside the update
        hess_column(H + (int64_t)col * (km + 1) * km, coef + (int64_t)col * cstride, J, km);
        return;
    }
    const int64_t tile = H ? blockIdx.x - 1 : blockIdx.x;
    __shared__ double2 cf[kMaxSlots];
    for (int l = threadIdx.x; l < 2 * J + 2; l += blockDim.x) cf[l] = coef[(int64_t)col * cstride + l];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = S == 1 ? tile * blockDim.x + threadIdx.x : tile * 32 + lane;
    const bool act = i < n;
    const double2* vb = V.base + col * V.sr + (act ? i : 0);
    double2* uc = u + col * wsr;
    double2* nc = next ? next + col * wsr : nullptr;
    double2 uv = make_double2(0, 0), zv = make_double2(0, 0);
    if (act && warp % S == 0) {
        uv = uc[i];
        if (nc) zv = z[col * wsr + i];
    }
    double2 qs = make_double2(0, 0), qc = make_double2(0, 0);
    constexpr int UNR = 8;
    const int w0 = S == 1 ? 0 : warp;
    for (int l0 = w0; l0 < J; l0 += UNR * S) {
        double2 q[UNR];
#pragma unroll
        for (int g = 0; g < UNR; ++g) q[g] = l0 + g * S < J ? vb[(l0 + g * S) * V.sj] : make_double2(0, 0);
#pragma unroll
        for (int g = 0; g < UNR; ++g) {
            const int l = l0 + g * S;
            if (l < J) {
                const double2 a = cf[l];
                qs.x = fma(a.x, q[g].x, qs.x);
                qs.x = fma(-a.y, q[g].y, qs.x);
                qs.y = fma(a.x, q[g].y, qs.y);
                qs.y = fma(a.y, q[g].x, qs.y);
                if (nc) {
                    const double2 c = cf[J + l];
                    qc.x = fma(c.x, q[g].x, qc.x);
                    qc.x = fma(-c.y, q[g].y, qc.x);
                    qc.y = fma(c.x, q[g].y, qc.y);
                    qc.y = fma(c.y, q[g].x, qc.y);
                }
            }
        }
    }
    if constexpr (S > 1) {
        __shared__ double sm[S][4][32];
        sm[warp][0][lane] = qs.x;
        sm[warp][1][lane] = qs.y;
        sm[warp][2][lane] = qc.x;
        sm[warp][3][lane] = qc.y;
        __syncthreads();
        if (warp != 0) return;
#pragma unroll
        for (int w = 1; w < S; ++w) {
            qs.x += sm[w][0][lane];
            qs.y += sm[w][1][lane];
            qc.x += sm[w][2][lane];
            qc.y += sm[w][3][lane];
        }
    }
    if (!act) return;
    const double inv_rho = cf[2 * J].x;
    const double2 qj = make_double2((uv.x - qs.x) * inv_rho, (uv.y - qs.y) * inv_rho);
    uc[i] = qj;
    if (nc) {
        const double2 d = cf[2 * J + 1];
        double2 nv = make_double2(fma(zv.x, inv_rho, -qc.x), fma(zv.y, inv_rho, -qc.y));
        nv.x = fma(-d.x, qj.x, nv.x);
        nv.x = fma(d.y, qj.y, nv.x);
        nv.y = fma(-d.x, qj.y, nv.y);
        nv.y = fma(-d.y, qj.x, nv.y);
        nc[i] = nv;
    }
}

}  // namespace

// CTAs per column of the inner products: of 128, 256, 512 or 1024 elements (1, 2, 4 or 8 per
// thread), whichever leaves the busiest sub-partition the fewest FP64 instructions (64 e + 31 per
// group of vectors) over the first five groups a basis grows through.
template <>
int dot_blocks<double2>(int64_t n, int ncol) {
    int64_t best = INT64_MAX, pick = 1;
    for (int e = 1; e <= 8; e *= 2) {
        const int64_t nb = std::max<int64_t>(1, (n + 128 * e - 1) / (128 * e));
        int64_t t = 0;
        for (int g = 1; g <= 5; ++g) t += rounds(4 * nb * ncol, g).second * (64 * e + 31);
        if (t < best) {
            best = t;
            pick = nb;
        }
    }
    return (int)pick;
}

template <>
cudaError_t mdot<double2>(Basis<double2> V, int J, const double2* w, int64_t wsr, int64_t n, int ncol,
                          const Reduce& rd, int with_norm, const int* skip, cudaStream_t st) {
    return launch<1>(V, J, w, nullptr, wsr, n, ncol, rd, with_norm, skip, st);
}
template <>
cudaError_t dcgs_dots<double2>(Basis<double2> V, int J, const double2* u, const double2* z, int64_t wsr, int64_t n,
                               int ncol, const Reduce& rd, const int* skip, cudaStream_t st) {
    if (z) return launch<2>(V, J, u, z, wsr, n, ncol, rd, 1, skip, st);
    return launch<1>(V, J, u, nullptr, wsr, n, ncol, rd, 1, skip, st);
}

template <>
cudaError_t dcgs_update<double2>(Basis<double2> V, int J, const double2* coef, int cstride, double2* u,
                                 const double2* z, double2* next, int64_t wsr, int64_t n, int ncol, double2* H, int km,
                                 const int* skip, cudaStream_t st) {
    if (2 * J + 2 > kMaxSlots) return cudaErrorInvalidValue;
    // four warps per 32 elements where that shortens the busiest sub-partition's work (the extra
    // sums cost about an eighth)
    const int64_t warps = (n + 31) / 32 * ncol;
    const bool split = J > 4 && 9 * ((4 * warps + PIPES - 1) / PIPES) < 32 * ((warps + PIPES - 1) / PIPES);
    const dim3 grid((unsigned)((split ? (n + 31) / 32 : (n + 63) / 64) + (H ? 1 : 0)), ncol);
    if (split)
        launch_pdl(k_dcgs_update_f64<4>, grid, 128, 0, st, V, J, coef, cstride, u, z, next, wsr, n, H, km, skip);
    else
        launch_pdl(k_dcgs_update_f64<1>, grid, 64, 0, st, V, J, coef, cstride, u, z, next, wsr, n, H, km, skip);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sgn
