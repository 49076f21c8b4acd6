// Tall-skinny vector kernels for the Arnoldi process (eq. (2.4)), the update
// of Algorithm 1 and the LR projection (Sec. 4).  Declarations.
#pragma once

#include "sgn_internal.cuh"

namespace sgn {

// Per-column solver state kept on the device, so that one restart cycle is a
// fixed sequence of launches with no host round trip (captured as a graph).
struct DevState {
    double2* H;        // [col][(kmax+1) * kmax] Hessenberg matrix, row-major (row i, col j)
    double2* red;      // [col][rstride] reduction results / coefficients of the next pass
    double2* h1;       // [col][rstride] first Gram-Schmidt coefficients of the current step
    double2* coef;     // [col][rstride] combined update coefficients sum_i omega_i y_i
    double2* y;        // [col][s][kmax] shifted solutions of the current cycle
    double2* rho;      // [col][s] collinearity factors (eq. (3.1))
    double* norm0;     // [col] ||A^2 v_j|| before orthogonalisation
    double* scale;     // [col] scale applied by the next normalising pass
    double* beta;      // [col] ||r|| of the restart vector
    double* bnorm;     // [col] ||b~||
    double* resest;    // [col] max_i |rho_i| ||r|| / ||b~||
    const double* sigma;  // [col][s] shifts (per column: the mixed refinement solves one shift per column)
    const double* omega;  // [col][s] weights
    const double* sigma_im = nullptr;  // [col][s] imaginary parts of the shifts (null: real shifts)
    double2* gres = nullptr;  // [col][kmax + 1] minimal-residual form: coefficients of the new residual in V_{k+1}
    int* kk;           // [col] Krylov dimension of the current cycle
    int* done;         // [col] converged (column work is skipped)
    int* skip;         // [col] done or broken down in this cycle
    int* err;          // [1] device error word (bit 0: singular shifted system; bit 1: non-finite)
    int kmax;
    int s;
    int rstride;
    double tol;
    double bd_tol;     // breakdown threshold relative to norm0
};

#ifdef __CUDACC__
// Sum over the lanes of N = 2^k <= 32 values per lane; lane l ends with the sum of value l mod N.
template <int N>
__device__ __forceinline__ double reduce_scatter(const double (&a)[N], int lane) {
    if constexpr (N == 1) {
        return a[0];
    } else {
        constexpr int H = N / 2;
        const bool up = lane & H;
        double h[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const double keep = up ? a[H + i] : a[i], send = up ? a[i] : a[H + i];
            h[i] = keep + __shfl_xor_sync(0xffffffffu, send, H);
        }
        return reduce_scatter<H>(h, lane);
    }
}
// The same for N < 32: the lanes beyond N are added first.
template <int N>
__device__ __forceinline__ double reduce_few(double (&a)[N], int lane) {
#pragma unroll
    for (int o = 16; o >= N; o >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) a[i] += __shfl_xor_sync(0xffffffffu, a[i], o);
    return reduce_scatter<N>(a, lane);
}

// Sum of the N FP32 values st[0..N) (one per thread of a CTA) by one warp as an unevaluated pair (hi,
// lo): N / 32 values per lane with TwoSum, then the lane butterfly.
template <int N>
__device__ __forceinline__ double cta_sum_df(const float* st, int lane) {
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int q = 0; q < N / 32; ++q) {
        const float v = st[lane + 32 * q];
        const float s = __fadd_rn(hi, v);
        const float bp = __fsub_rn(s, hi);
        const float ap = __fsub_rn(s, bp);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, ap), __fsub_rn(v, bp)));
        hi = s;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ohi = __shfl_xor_sync(0xffffffffu, hi, o);
        const float olo = __shfl_xor_sync(0xffffffffu, lo, o);
        const float s = __fadd_rn(hi, ohi);
        const float bp = __fsub_rn(s, hi);
        const float ap = __fsub_rn(s, bp);
        const float e = __fadd_rn(__fsub_rn(hi, ap), __fsub_rn(ohi, bp));
        const float t = __fadd_rn(e, __fadd_rn(lo, olo));
        const float nh = __fadd_rn(s, t);
        lo = __fsub_rn(t, __fsub_rn(nh, s));
        hi = nh;
    }
    return (double)hi + (double)lo;
}

// Tentative column j of the Hessenberg matrix in a delayed-CGS2 step, by one CTA:
//   H[i][j] = c_i - g_i / rho (i < j),  H[j][j] = d - g_j / rho,  g = H[0:j+1, 0:j] s,
// with the step's coefficients s = red[0, j), c = red[j, 2j), 1 / rho = red[2j], d = red[2j + 1].
// Four lanes per row.  Not inlined: in the FP32 update it would take that kernel from 80 to 107
// registers, a third of its resident warps (74 -> 87 us on 120 columns of 10^4).
__device__ __noinline__ static void hess_column(double2* H, const double2* red, int j, int km) {
    const int q = threadIdx.x & 3;
    const double ir = red[2 * j].x;
    for (int i0 = 0; i0 <= j; i0 += blockDim.x / 4) {
        const int i = i0 + threadIdx.x / 4;
        double gx = 0.0, gy = 0.0;
        if (i <= j)
            for (int l = (i > 0 ? i - 1 : 0) + q; l < j; l += 4) {
                const double2 h = H[(int64_t)i * km + l], s = red[l];
                gx = fma(h.x, s.x, gx);
                gx = fma(-h.y, s.y, gx);
                gy = fma(h.x, s.y, gy);
                gy = fma(h.y, s.x, gy);
            }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            gx += __shfl_xor_sync(0xffffffffu, gx, o);
            gy += __shfl_xor_sync(0xffffffffu, gy, o);
        }
        if (i <= j && q == 0) {
            const double2 c = red[i < j ? j + i : 2 * j + 1];
            H[(int64_t)i * km + j] = make_double2(fma(-gx, ir, c.x), fma(-gy, ir, c.y));
        }
    }
}
#endif

// Slots of one reduction: >= 2 kmax + 3 (delayed CGS2), >= deflation size + 1, >= eigensolver block + 1.
constexpr int kMaxSlots = 136;

enum ReduceMode {
    RM_STORE = 0,        // red[col][j] = sum_j
    RM_H1 = 1,           // h1[col][j] = sum_j (j < J), norm0 = sqrt(sum_J)
    RM_P2 = 2,           // second CGS pass: Hessenberg column, h_{j+1,j}, breakdown, scale
    RM_BETA_FIRST = 3,   // bnorm = beta = sqrt(sum_0), rho = 1, scale = 1/beta
    RM_BETA_RESTART = 4, // beta = sqrt(sum_0), residual estimate, convergence, scale = 1/beta
    RM_SIGNED = 5,       // red[col][j] = sign(Re lambda_j) * sum_j (x_P coefficients)
    RM_DCGS = 6,         // delayed CGS2 step j: rho, column j-1 correction, update coefficients
    RM_DCGS_FINAL = 7    // delayed CGS2 closing pass of a cycle (no new candidate)
};

template <class T>
cudaError_t mdot(Basis<T> V, int J, const T* w, int64_t wsr, int64_t n, int ncol, const Reduce& rd,
                 int with_norm, const int* skip, cudaStream_t st);
template <>
cudaError_t mdot<double2>(Basis<double2> V, int J, const double2* w, int64_t wsr, int64_t n, int ncol,
                          const Reduce& rd, int with_norm, const int* skip, cudaStream_t st);
template <>
cudaError_t mdot<float2>(Basis<float2> V, int J, const float2* w, int64_t wsr, int64_t n, int ncol,
                         const Reduce& rd, int with_norm, const int* skip, cudaStream_t st);
cudaError_t reduce(const Reduce& rd, int nslot, int ncol, int mode, int colidx, const DevState& S,
                   const double2* lambda, cudaStream_t st);
template <class T>
cudaError_t maxpy_mdot(Basis<T> V, int J, const double2* coef, int cstride, T* w, int64_t wsr, int64_t n,
                       int ncol, const Reduce& rd, const int* skip, cudaStream_t st);
template <class T>
cudaError_t maxpy_scale(Basis<T> V, int J, const double2* coef, int cstride, const T* w, int64_t wsr, T* out,
                        int64_t osr, const double* scale, int64_t n, int ncol, const int* skip, cudaStream_t st);
template <class T>
cudaError_t update_x(Basis<T> V, int J, const double2* coef, int cstride, double2* x, int64_t xsr, int64_t n,
                     int ncol, const int* skip, const int* kk, cudaStream_t st);
template <class T>
cudaError_t update_shifts(Basis<T> V, int J, const double2* y, int s, int kmax, double2* xs, int64_t xs_shift,
                          int64_t xs_col, int64_t n, int ncol, const int* skip, const int* kk, cudaStream_t st);

// Delayed CGS2 (one fused reduction and one fused update per Arnoldi step).  dcgs_update with
// H (the columns' Hessenberg matrices, row stride km; null: not) also forms column J of H from the
// step's coefficients (hess_column).
template <class T>
cudaError_t dcgs_dots(Basis<T> V, int J, const T* u, const T* z, int64_t wsr, int64_t n, int ncol, const Reduce& rd,
                      const int* skip, cudaStream_t st);
template <>
cudaError_t dcgs_dots<double2>(Basis<double2> V, int J, const double2* u, const double2* z, int64_t wsr, int64_t n,
                               int ncol, const Reduce& rd, const int* skip, cudaStream_t st);
template <>
cudaError_t dcgs_dots<float2>(Basis<float2> V, int J, const float2* u, const float2* z, int64_t wsr, int64_t n,
                              int ncol, const Reduce& rd, const int* skip, cudaStream_t st);
template <class T>
cudaError_t dcgs_update(Basis<T> V, int J, const double2* coef, int cstride, T* u, const T* z, T* next, int64_t wsr,
                        int64_t n, int ncol, double2* H, int km, const int* skip, cudaStream_t st);
template <>
cudaError_t dcgs_update<double2>(Basis<double2> V, int J, const double2* coef, int cstride, double2* u,
                                 const double2* z, double2* next, int64_t wsr, int64_t n, int ncol, double2* H, int km,
                                 const int* skip, cudaStream_t st);
template <>
cudaError_t dcgs_update<float2>(Basis<float2> V, int J, const double2* coef, int cstride, float2* u, const float2* z,
                                float2* next, int64_t wsr, int64_t n, int ncol, double2* H, int km, const int* skip,
                                cudaStream_t st);

// out = a x + b y + c z over `count` complex elements (z may be null).
template <class T>
cudaError_t axpby3(T* out, double a, const T* x, double b, const T* y, double c, const T* z, int64_t count,
                   cudaStream_t st);
// Z_j = sum_i C[i][j] Y_i for q input and r output fields of n complex (C: device, row-major q x r).
template <class T>
cudaError_t block_combine(const T* Y, int q, const double2* C, int r, T* Z, int64_t n, cudaStream_t st);
// Seeded complex Gaussian entries (counter-based, SplitMix64 + Box-Muller).
template <class T>
cudaError_t random_fill(T* out, int64_t count, uint64_t seed, cudaStream_t st);

// Type conversions of whole fields.
cudaError_t convert_f64_to_f32(const double2* in, float2* out, int64_t count, cudaStream_t st);
cudaError_t convert_f32_to_f64(const float2* in, double2* out, int64_t count, cudaStream_t st);
cudaError_t links_f64_to_bf16(const double2* in, __nv_bfloat162* out, int64_t count, cudaStream_t st);
cudaError_t links_f64_to_f16(const double2* in, __half2* out, int64_t count, cudaStream_t st);

// Small dense steps (hess.cu).  prepare_small_kernels sets launch attributes once
// per device (before any stream capture).
cudaError_t prepare_small_kernels();
cudaError_t shifted_solves(const DevState& S, int ncol, cudaStream_t st);
// Minimal-residual (GMRES) form for one shift per column: y, rho = 1 and the new
// residual's coefficients in S.gres (k_shifted_lsq).
cudaError_t shifted_lsq(const DevState& S, int ncol, cudaStream_t st);
cudaError_t combine_shifts(const DevState& S, int ncol, cudaStream_t st);

// y = a + beta gamma5 s for nfield packed complex128 fields (gamma5: spins 2, 3 negated).
cudaError_t gamma5_axpy(double2* y, const double2* a, const double2* s, double beta, int64_t vol, int nfield,
                        cudaStream_t st);

// BiCGStab correction solves of the refinement (bicgstab.cu): FP32 fields of ncol columns back to
// back, FP64 scalars per column.
enum BiStatus { BI_RUN = 0, BI_DONE = 1, BI_IDLE = 2, BI_FAILED = 3 };
struct BiState {
    float2 *r, *rt, *p, *w, *s, *t, *d;  // residual, shadow residual, direction, A^2 p, half step, A^2 s, solution
    double2 *rho, *alpha, *omega, *beta;
    double *lim, *rn0;    // ||r||^2 to reach, and of the start
    const double* tol;    // relative residual to reach
    const double* sigma;
    int* done;            // BiStatus (non-zero: skip)
    int* count;           // arrival counters of the sums
    double* partial;
    int64_t npk;          // packs of two complex numbers per column
    int nblk, pkt;        // CTAs per column, packs per thread
};
void bi_shape(BiState& S, int64_t n, int ncol);
size_t bi_partial_bytes(const BiState& S, int ncol);
cudaError_t bi_init(const BiState& S, int ncol, const double2* src, const long long* off, const int* ex, int nb,
                    cudaStream_t st);
cudaError_t bi_v(const BiState& S, int ncol, cudaStream_t st);
cudaError_t bi_s(const BiState& S, int ncol, cudaStream_t st);
cudaError_t bi_t(const BiState& S, int ncol, cudaStream_t st);
cudaError_t bi_x(const BiState& S, int ncol, cudaStream_t st);

// Corrections are solved for residuals scaled to about norm one, by an exact power of two: fl32(2^-ex[j] r_j)
// for nb systems, r_j at off[j] of src (bi_init takes the same), and x_j += 2^ex[j] d_j, x_j at
// off[j], d_j (float2 or double2) at j n; with done, only systems marked BI_DONE.  |ex| <= 1022.
cudaError_t scaled_residuals(const double2* src, const long long* off, const int* ex, float2* out, int64_t n, int nb,
                             cudaStream_t st);
template <class T>
cudaError_t add_corrections(double2* x, const long long* off, const int* ex, const int* done, const T* d, int64_t n,
                            int nb, cudaStream_t st);

// Tall-skinny products of a basis V (J <= 64 fields, stride sv) with N columns W
// (complex128, stride sw): tsmm_tn writes the partials of V^dag W into rd (then
// reduce(rd, J, N, RM_STORE, ...) gives red[col * rstride + j]); tsmm_nn does
// W_col += alpha sum_j V_j C[col * cstride + j].  FP32 products, FP64 sums over CTAs.
template <class TV>
cudaError_t tsmm_tn(const TV* V, int64_t sv, int J, const double2* W, int64_t sw, int N, int64_t n,
                    const Reduce& rd, cudaStream_t st);
template <class TV>
cudaError_t tsmm_nn(const TV* V, int64_t sv, int J, const double2* C, int cstride, double2* W, int64_t sw, int N,
                    int64_t n, double alpha, cudaStream_t st);

// Number of blocks per column used by the reductions for n complex elements.
template <class T>
int reduce_blocks(int64_t n);
// CTAs per column of the FP64 inner products of ncol columns (gs_f64.cu), at most ceil(n / 128).
// mdot and dcgs_dots on double2 take any Reduce::nblk >= 1.
template <class T>
int dot_blocks(int64_t n, int ncol);
template <>
int dot_blocks<double2>(int64_t n, int ncol);
// Two warps on each of 152 SMs: fewer warps than this leave FP64 pipes idle.
constexpr int64_t kFewWarps = 304;
// CTAs per column for a grid of ncol columns that fills whole waves (1, 2 or 4
// packs per thread); a Reduce built with it serves every kernel of the file.
template <class T>
int wave_blocks(int64_t n, int ncol);

}  // namespace sgn
