// The small dense steps of Algorithm 1, kept on the device:
//   y_i = beta rho_i (H_k - sigma_i I)^{-1} e_1          (one warp per column and shift)
//   rho_i <- -h_{k+1,k} e_k^T y_i                        (collinearity factor, eq. (3.1))
//   c = sum_i omega_i y_i                                (the combination of eq. (2.3))
#include "blas.cuh"

namespace sgn {
namespace {

constexpr int KMAX = 64;

// a / b, b scaled by a power of two so that |b|^2 neither overflows nor underflows
__device__ __forceinline__ double2 cdiv_scaled(double2 a, double2 b) {
    const int e = max((__double2hiint(b.x) >> 20) & 0x7ff, (__double2hiint(b.y) >> 20) & 0x7ff);
    const double f = e == 0 ? 0x1p1000 : e >= 2046 ? 0x1p-1020 : __hiloint2double((2046 - e) << 20, 0);  // ~ 1 / |b|
    const double x = b.x * f, y = b.y * f, d = f / fma(x, x, y * y);
    return make_double2(fma(a.x, x, a.y * y) * d, fma(a.y, x, -a.x * y) * d);
}
__device__ __forceinline__ double2 shfl(double2 v, int src) {
    return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// The shifted systems by Hyman's method: all rows of an upper Hessenberg system but the first fix
// the solution up to its scale, backwards from x_{q-1} = 1 by one division-free step per row,
//   x_{l-1} = -(sum_{i >= l} M_li x_i) / M_{l,l-1},
// and the first row gives the scale.  Each computed x_{l-1} satisfies its row exactly for
// coefficients perturbed by a few units in the last place, and so does the scaled first row: the
// solution is that of a system with rows perturbed componentwise by rounding (backward stable
// without pivoting).  The subdiagonal entries are the non-zero norms rho_l of the Arnoldi process.
//
// What bounds it: an FP64 instruction takes a warp 64 cycles, so the elimination with partial
// pivoting used before (35 of them per row, two divisions among them, and 30 per row of the back
// substitution) took 118 us at k = 30 and 180 us at k = 40 per cycle.  Here a step takes 6: lanes own
// rows, add the new x_l times column l to their row sums (4), and the owner of row l hands over
// x_{l-1} (2; the rows are divided by -M_{l,l-1} when they are staged).  Measured 29 us
// at k = 40 (17 averaged over the mixed form's k = 16 and 40).
//
// BORDER = false: FOM, (H_k - sigma_i I) y = beta rho_i e_1 (k x k), shift i.
// BORDER = true: the non-seed shifts of restarted multishift GMRES, shift i + 1:
// [Hbar_k - sigma_i I~ | z] (y, tau) = beta rho_i e_1, (k+1) x (k+1), z = gres the seed's
// residual coefficients; the new residual of shift i is tau times the seed's, so rho_i <- tau.
// Both matrices are upper Hessenberg (the bordered one has a full last column).  After a breakdown
// (kk < kmax, or a last norm of zero) FOM on the kk columns is exact and takes the bordered
// system's place.
// One warp per shift, SW shifts of a column per CTA sharing the staged matrix.
constexpr int SW = 4;
template <bool BORDER>
__global__ void __launch_bounds__(32 * SW) k_shifted_solve(DevState S) {
    pdl_begin();
    const int col = blockIdx.y;
    if (S.done[col]) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int km = S.kmax;
    const int kk = S.kk[col];
    const double2* H = S.H + (int64_t)col * (km + 1) * km;
    const bool border = BORDER && kk == km && H[(int64_t)kk * km + kk - 1].x > 0;
    const int q = border ? kk + 1 : kk;  // system size
    const int ld = q | 1;                // odd: the transposed stores meet no bank conflicts
    extern __shared__ double2 M[];       // [q][ld], column-major, row r >= 1 divided by -H[r][r-1]
    __shared__ double ninv[KMAX + 1];
    for (int r = threadIdx.x; r < q; r += blockDim.x) ninv[r] = r > 0 ? -1.0 / H[(int64_t)r * km + r - 1].x : 1.0;
    __syncthreads();
    for (int t = threadIdx.x; t < q * q; t += blockDim.x) {
        const int r = t / q, c = t - r * q;
        if (c < r) continue;
        const double2 h = border && c == kk ? S.gres[(int64_t)col * (km + 1) + r] : H[(int64_t)r * km + c];
        const double f = ninv[r];
        M[c * ld + r] = make_double2(h.x * f, h.y * f);
    }
    __syncthreads();
    const int slot = blockIdx.x * SW + warp;
    const int i = BORDER ? slot + 1 : slot;  // shift
    if (i >= S.s) return;
    const double sigma = S.sigma[(int64_t)col * S.s + i];
    const double sigma_im = S.sigma_im ? S.sigma_im[(int64_t)col * S.s + i] : 0.0;
    double2* y = S.y + ((int64_t)col * S.s + i) * km;
    const double2 zero = make_double2(0, 0);
    double2 acc[3] = {zero, zero, zero};  // row sums of rows lane, lane + 32, lane + 64
    double2 xo[3] = {zero, zero, zero};   // x of the same indices
    double2 x = make_double2(1.0, 0.0);
    for (int l = q - 1; l >= 0; --l) {
        if (lane == (l & 31)) {
            if (l < 32)
                xo[0] = x;
            else if (l < 64)
                xo[1] = x;
            else
                xo[2] = x;
        }
        const double2* mc = M + l * ld;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (32 * k > l) break;  // uniform
            const int r = lane + 32 * k;
            const double2 m = r <= l ? mc[r] : zero;
            acc[k].x = fma(m.x, x.x, acc[k].x);
            acc[k].x = fma(-m.y, x.y, acc[k].x);
            acc[k].y = fma(m.x, x.y, acc[k].y);
            acc[k].y = fma(m.y, x.x, acc[k].y);
        }
        // the row sum of row l, less its shift: x_{l-1} (the last, l = 0, is the first row's value).
        // The bordered system's last row has no shift.
        double2 v = shfl(l >= 64 ? acc[2] : l >= 32 ? acc[1] : acc[0], l & 31);
        if (l < kk) {
            const double sr = sigma * ninv[l];
            v.x = fma(-sr, x.x, v.x);
            v.y = fma(-sr, x.y, v.y);
            if (sigma_im != 0.0) {
                const double si = sigma_im * ninv[l];
                v.x = fma(si, x.y, v.x);
                v.y = fma(-si, x.x, v.y);
            }
        }
        x = v;
        // keep the running solution far from overflow (shifts of large modulus): scale by 2^-400
        const int big = max(__double2hiint(x.x) & 0x7fffffff, __double2hiint(x.y) & 0x7fffffff);
        if (l > 0 && big > 0x59000000 && big < 0x7ff00000) {  // above 2^401, finite
            const double f = __hiloint2double(0x26f00000, 0);  // 2^-400
            x = make_double2(x.x * f, x.y * f);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                acc[k] = make_double2(acc[k].x * f, acc[k].y * f);
                xo[k] = make_double2(xo[k].x * f, xo[k].y * f);
            }
        }
    }
    if (x.x == 0 && x.y == 0) {  // first row's value zero: the shift is an eigenvalue
        if (lane == 0) atomicOr(S.err, 1);
        for (int j = lane; j < km; j += 32) y[j] = zero;
        return;
    }
    const double2 rho = S.rho[(int64_t)col * S.s + i];
    const double beta = S.beta[col];
    const double2 sc = cdiv_scaled(make_double2(beta * rho.x, beta * rho.y), x);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int j = lane + 32 * k;
        const double2 v = cmul(xo[k], sc);
        if (j < km) y[j] = j < kk ? v : zero;
        if (j == q - 1) {  // the last component
            double2 rnew = zero;
            if (border) {
                rnew = v;  // tau
            } else if (!BORDER && kk == km) {
                const double2 h = H[(int64_t)kk * km + (kk - 1)];
                rnew = cmul(h, v);
                rnew = make_double2(-rnew.x, -rnew.y);
            }
            S.rho[(int64_t)col * S.s + i] = rnew;
        }
    }
}

__global__ void k_combine(DevState S) {
    pdl_begin();
    const int col = blockIdx.x;
    if (S.done[col]) return;
    const int km = S.kmax;
    for (int j = threadIdx.x; j < km; j += blockDim.x) {
        double2 c = make_double2(0, 0);
        for (int i = 0; i < S.s; ++i) {
            double2 y = S.y[((int64_t)col * S.s + i) * km + j];
            double w = S.omega[(int64_t)col * S.s + i];
            c.x = fma(w, y.x, c.x);
            c.y = fma(w, y.y, c.y);
        }
        S.coef[(int64_t)col * S.rstride + j] = c;
    }
}

// Minimal-residual form for one shift per column (restarted GMRES):  y = argmin
// || beta rho e_1 - (Hbar_k - sigma I~) y ||  by Givens rotations, with the
// coefficients of the new residual, c = beta rho e_1 - (Hbar_k - sigma I~) y, in
// gres[col][0..kk] (the next restart vector is V_{k+1} c) and rho = 1.  One CTA per column stages
// the matrix; one warp applies the rotations (lanes own columns, the right-hand side is column
// kk), back-substitutes and forms c (lanes own rows).
__global__ void __launch_bounds__(128) k_shifted_lsq(DevState S) {
    pdl_begin();
    const int col = blockIdx.x;
    if (S.done[col]) return;
    const int km = S.kmax;
    const int kk = S.kk[col];
    const double2* H = S.H + (int64_t)col * (km + 1) * km;
    const double sig = S.sigma[(int64_t)col * S.s];
    const double sig_im = S.sigma_im ? S.sigma_im[(int64_t)col * S.s] : 0.0;
    const double beta = S.beta[col];
    const double2 rho = S.rho[(int64_t)col * S.s];
    const double2 b0 = make_double2(beta * rho.x, beta * rho.y), zero = make_double2(0, 0);
    const int ld = kk + 2;           // row stride: columns 0..kk-1, the right-hand side, one of padding
    extern __shared__ double2 M[];   // [kk + 1][ld]
    __shared__ double inv[KMAX];     // 1 / diagonal after the rotations (0: zero column)
    for (int t = threadIdx.x; t < (kk + 1) * ld; t += blockDim.x) {
        const int r = t / ld, c = t - r * ld;
        double2 h = zero;
        if (c < kk && c >= r - 1) {
            h = H[(int64_t)r * km + c];
            if (r == c) {
                h.x -= sig;
                h.y -= sig_im;
            }
        } else if (c == kk && r == 0) {
            h = b0;
        }
        M[t] = h;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    // rows c and c+1: G = [[conj(cs), sn], [-sn, cs]] zeroes M[c+1][c] (real: an Arnoldi norm)
    for (int c = 0; c < kk; ++c) {
        const double2 a = M[c * ld + c];
        const double b = M[(c + 1) * ld + c].x;
        const double n2 = fma(b, b, cabs2(a));
        const double ir = n2 > 0 ? rsqrt(n2) : 0.0;
        if (lane == 0) inv[c] = ir;
        __syncwarp();
        if (!(n2 > 0)) continue;  // zero column (only at a breakdown): y_c = 0 below
        const double2 cs = make_double2(a.x * ir, a.y * ir);
        const double sn = b * ir;
        for (int j = c + lane; j <= kk; j += 32) {
            const double2 x = M[c * ld + j], w = M[(c + 1) * ld + j];
            double2 p = cconjmul(cs, x), r = cmul(cs, w);
            p.x = fma(sn, w.x, p.x);
            p.y = fma(sn, w.y, p.y);
            r.x = fma(-sn, x.x, r.x);
            r.y = fma(-sn, x.y, r.y);
            M[c * ld + j] = p;
            M[(c + 1) * ld + j] = r;
        }
        __syncwarp();
    }
    // back substitution; lane owns rows lane, lane + 32
    double2 z0 = lane < kk ? M[lane * ld + kk] : zero, z1 = lane + 32 < kk ? M[(lane + 32) * ld + kk] : zero;
    double2 y0 = zero, y1 = zero;
    for (int r = kk - 1; r >= 0; --r) {
        double2 yr = shfl(r >= 32 ? z1 : z0, r & 31);
        yr = make_double2(yr.x * inv[r], yr.y * inv[r]);
        if (lane == (r & 31)) {
            if (r < 32)
                y0 = yr;
            else
                y1 = yr;
        }
        if (lane < r) z0 = csub(z0, cmul(M[lane * ld + r], yr));
        if (r > 32 && lane + 32 < r) z1 = csub(z1, cmul(M[(lane + 32) * ld + r], yr));
    }
    double2* yv = S.y + (int64_t)col * S.s * km;
    if (lane < km) yv[lane] = lane < kk ? y0 : zero;
    if (lane + 32 < km) yv[lane + 32] = lane + 32 < kk ? y1 : zero;
    // c = beta rho e_1 - (Hbar - sigma I~) y, from the unrotated matrix; lane owns rows lane, + 32, + 64
    double2 acc[3] = {lane == 0 ? b0 : zero, zero, zero};
    for (int c = 0; c < kk; ++c) {
        const double2 yc = shfl(c >= 32 ? y1 : y0, c & 31);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int r = lane + 32 * k;
            if (32 * k > c + 1) break;  // uniform
            double2 h = r <= c + 1 ? H[(int64_t)r * km + c] : zero;
            if (r == c) {
                h.x -= sig;
                h.y -= sig_im;
            }
            acc[k] = csub(acc[k], cmul(h, yc));
        }
    }
    double2* cres = S.gres + (int64_t)col * (km + 1);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (lane + 32 * k <= km) cres[lane + 32 * k] = lane + 32 * k <= kk ? acc[k] : zero;
    if (lane == 0) S.rho[(int64_t)col * S.s] = make_double2(1, 0);
}

// Shared memory of a q x q system staged by k_shifted_solve.
constexpr size_t staged_bytes(int q) { return sizeof(double2) * (size_t)q * (q | 1); }

}  // namespace

cudaError_t shifted_lsq(const DevState& S, int ncol, cudaStream_t st) {
    if (S.s < 1 || !S.gres || S.kmax > KMAX) return cudaErrorInvalidValue;
    launch_pdl(k_shifted_lsq, ncol, 128, sizeof(double2) * (S.kmax + 1) * (S.kmax + 2), st, S);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || S.s == 1) return e;
    // the other shifts: bordered systems with the seed's residual coefficients
    launch_pdl(k_shifted_solve<true>, dim3((S.s - 1 + SW - 1) / SW, ncol), 32 * SW, staged_bytes(S.kmax + 1), st, S);
    count_launch();
    return cudaGetLastError();
}

cudaError_t prepare_small_kernels() {
    cudaError_t e = cudaFuncSetAttribute(k_shifted_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)staged_bytes(KMAX));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_shifted_solve<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)staged_bytes(KMAX + 1));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_shifted_lsq, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(double2) * (KMAX + 1) * (KMAX + 2)));
}

cudaError_t shifted_solves(const DevState& S, int ncol, cudaStream_t st) {
    if (S.kmax > KMAX) return cudaErrorInvalidValue;
    launch_pdl(k_shifted_solve<false>, dim3((S.s + SW - 1) / SW, ncol), 32 * SW, staged_bytes(S.kmax), st, S);
    count_launch();
    return cudaGetLastError();
}

cudaError_t combine_shifts(const DevState& S, int ncol, cudaStream_t st) {
    launch_pdl(k_combine, ncol, 64, 0, st, S);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sgn
