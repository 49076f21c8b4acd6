// The direct projection that the paper compares Algorithm 1 against (Sec. 6, eq. (6.3)):
//   x = x_P + ||r|| V_k sign(H_k) e_1,   r = (I - P) b,   x_P = R sign(Re Lambda) L^dag b,
// with V_k, H_k from k Arnoldi steps on A itself (no rational approximation, no restarts),
// and sign(H_k) by Roberts' Newton iteration X <- (X + X^{-1}) / 2 on the k x k matrix.
// The whole basis is kept (k + 1 FP64 fields per column, the method's memory cost); the
// Arnoldi steps use the FP64 stencil and two classical Gram-Schmidt passes, in blocks of at
// most 128 basis vectors per kernel (the reduction's slot limit).  The Newton iterations run
// on the GPU for all columns at once: X^{-1} by Gauss-Jordan elimination with partial
// pivoting on [X | I], one launch per pivot (captured once as a CUDA graph), with the
// matrices of shorter Krylov dimension padded by the identity (sign(I) = I).
//
// What bounds it: the Gram-Schmidt passes' FP64 products (16 multiply-adds per basis entry and step),
// so nothing else may hold them up: the Hessenberg matrix, the norms and the breakdown flags stay on
// the device, and the host only looks every 32 steps whether a column is still growing.  With four
// host round trips per step, a pair of launches per pivot and one CTA for the Newton update,
// k = 100 on 8^4 x 2 took 43 ms; now 28.
#include "ctx.cuh"
#include "dense_eig.h"

#include <algorithm>

namespace sgn {

namespace {
constexpr int GS_BLOCK = 128;
using cdd = std::complex<double>;

__device__ __forceinline__ double2 cdiv_d(double2 a, double2 b) {
    const double den = b.x * b.x + b.y * b.y;
    return make_double2((a.x * b.x + a.y * b.y) / den, (a.y * b.x - a.x * b.y) / den);
}

constexpr int GJ_COLS = 4;  // columns per CTA of an elimination step

// Gauss-Jordan step p on the augmented matrices A[col] = [X | I] (q rows, 2q columns, row-major).
// fac: column p before the step.  Every CTA finds the pivot row r (the first row i >= p of largest
// |fac[i]|) for itself, and on its columns j > p exchanges rows r and p, scales row p by 1 / pivot and
// subtracts fac[i] times it from the others; the CTA of column p + 1 leaves that column in next.  A zero
// pivot (singular X: an eigenvalue of H_k on the imaginary axis), or no finite one, sets bad[col].
// A latency chain: moduli are compared as bit patterns and one warp forms the reciprocal, as FP64
// instructions take 64 cycles.
__global__ void __launch_bounds__(256) k_gj_step(double2* A, int q, int p, const double2* fac, double2* next,
                                                 int* bad) {
    pdl_begin();
    const int col = blockIdx.y;
    if (bad[col]) return;
    double2* M = A + (size_t)col * q * 2 * q;
    const double2* f = fac + (size_t)col * q;
    const int ld = 2 * q, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ long long sv[8];
    __shared__ int si[8];
    __shared__ double2 pinv_sh;
    long long best = -1;
    int r = p;
    for (int i = p + tid; i < q; i += 256) {
        const double2 v = f[i];
        const double a2 = v.x * v.x + v.y * v.y;
        long long a = __double_as_longlong(a2);
        if (a >= 0x7ff0000000000000LL) a = -1;  // not finite
        if (a > best) {
            best = a;
            r = i;
        }
    }
    auto take = [&](long long o, int oi) {  // ties keep the lower row (first maximal pivot)
        if (o > best || (o == best && oi < r)) {
            best = o;
            r = oi;
        }
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, r, o));
    if (lane == 0) {
        sv[warp] = best;
        si[warp] = r;
    }
    __syncthreads();
    for (int w = 0; w < 8; ++w) take(sv[w], si[w]);
    if (!(best > 0)) {
        if (blockIdx.x == 0 && tid == 0) bad[col] = 1;
        return;
    }
    if (warp == 0) {
        const double2 pinv = cdiv_d(make_double2(1.0, 0.0), f[r]);
        if (lane == 0) pinv_sh = pinv;
    }
    const int j = p + 1 + blockIdx.x * GJ_COLS + tid % GJ_COLS;
    const bool act = j < ld;
    double2 ar = make_double2(0, 0), ap = ar;
    if (act) {
        ar = M[(size_t)r * ld + j];
        ap = M[(size_t)p * ld + j];
    }
    __syncthreads();  // rows r and p are read by all before any of them is written
    if (!act) return;
    const double2 prow = cmul(ar, pinv_sh);
    for (int i = tid / GJ_COLS; i < q; i += 256 / GJ_COLS) {
        double2 v = prow;
        if (i != p) {
            const double2 g = f[i == r ? p : i], o = i == r ? ap : M[(size_t)i * ld + j];
            v = make_double2(o.x - (g.x * prow.x - g.y * prow.y), o.y - (g.x * prow.y + g.y * prow.x));
        }
        M[(size_t)i * ld + j] = v;
        if (j == p + 1) next[(size_t)col * q + i] = v;
    }
}

// [X | I] and its first column from X (q x q per column), and after the inversion the Newton update
// X <- (X + X^{-1}) / 2 with the sums ||X_new - X||^2 and ||X_new||^2 of each CTA (gridDim.x per column).
__global__ void k_gj_load(const double2* X, double2* A, double2* fac, int q) {
    pdl_begin();
    const int col = blockIdx.y;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)q * 2 * q) return;
    const int i = (int)(e / (2 * q)), j = (int)(e - (int64_t)i * 2 * q);
    A[(size_t)col * q * 2 * q + e] =
        j < q ? X[(size_t)col * q * q + (size_t)i * q + j] : make_double2(j - q == i ? 1.0 : 0.0, 0.0);
    if (j == 0) fac[(size_t)col * q + i] = X[(size_t)col * q * q + (size_t)i * q];
}
__global__ void __launch_bounds__(256) k_newton_update(double2* X, const double2* A, int q, double* sums) {
    pdl_begin();
    const int col = blockIdx.y;
    __shared__ double sd[256], sx[256];
    double dn = 0, xn = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)q * q;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / q), j = (int)(e - (int64_t)i * q);
        const double2 xo = X[(size_t)col * q * q + e];
        const double2 xi = A[(size_t)col * q * 2 * q + (size_t)i * 2 * q + q + j];
        const double2 xn1 = make_double2(0.5 * (xo.x + xi.x), 0.5 * (xo.y + xi.y));
        dn += (xn1.x - xo.x) * (xn1.x - xo.x) + (xn1.y - xo.y) * (xn1.y - xo.y);
        xn += xn1.x * xn1.x + xn1.y * xn1.y;
        X[(size_t)col * q * q + e] = xn1;
    }
    sd[threadIdx.x] = dn;
    sx[threadIdx.x] = xn;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sd[threadIdx.x] += sd[threadIdx.x + s];
            sx[threadIdx.x] += sx[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        sums[2 * (col * gridDim.x + blockIdx.x)] = sd[0];
        sums[2 * (col * gridDim.x + blockIdx.x) + 1] = sx[0];
    }
}

// Second stage of a Gram-Schmidt pass over J basis vectors from i0: the coefficients go to red and are
// added to column j of H (k + 1 rows of k per column).  Eight lanes per coefficient.
__global__ void __launch_bounds__(256) k_direct_coef(Reduce rd, int J, int i0, int j, int k, double2* red, int rs,
                                                     double2* H) {
    pdl_begin();
    const int col = blockIdx.x, slot = blockIdx.y * 32 + threadIdx.x / 8, seg = threadIdx.x & 7;
    double2 a = make_double2(0, 0);
    if (slot < J) {
        const double2* p = rd.partial + ((int64_t)col * rd.stride + slot) * rd.nblk;
#pragma unroll 8
        for (int b = seg; b < rd.nblk; b += 8) a = cadd(a, p[b]);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    }
    if (slot >= J || seg) return;
    red[(int64_t)col * rs + slot] = a;
    double2* h = H + ((int64_t)col * (k + 1) + i0 + slot) * k + j;
    *h = cadd(*h, a);
}

// The norm of step j (j = -1: of the start vector, to beta): H[j+1][j] = ||w||, scale = 1 / ||w||; a column
// with ||w|| <= 1e-14 ||A v_j|| has an invariant subspace of dimension kk = j + 1, where the projection
// is exact: its further basis vectors are zero.
__global__ void __launch_bounds__(256) k_direct_norm(Reduce rd, int j, int k, double2* H, double* scale, double* beta,
                                                     int* kk, int* live) {
    pdl_begin();
    const int col = blockIdx.x, tid = threadIdx.x;
    __shared__ double s2[256], sh[256];
    double a = 0, h2 = 0;
    const double2* p = rd.partial + (int64_t)col * rd.stride * rd.nblk;
    for (int b = tid; b < rd.nblk; b += 256) a += p[b].x;
    for (int i = tid; i <= j; i += 256) h2 += cabs2(H[((int64_t)col * (k + 1) + i) * k + j]);
    s2[tid] = a;
    sh[tid] = h2;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (tid < s) {
            s2[tid] += s2[tid + s];
            sh[tid] += sh[tid + s];
        }
        __syncthreads();
    }
    if (tid != 0) return;
    const double n2 = s2[0] < 0 ? 0.0 : s2[0], nr = sqrt(n2);  // not finite stays so: the Newton iteration fails
    double sc = 0.0;
    if (j < 0) {
        beta[col] = nr;
        live[col] = nr > 0;
        kk[col] = nr > 0 ? k : 0;
        sc = nr > 0 ? 1.0 / nr : 0.0;
    } else if (live[col]) {
        if (nr <= 1e-14 * sqrt(n2 + sh[0])) {
            live[col] = 0;
            kk[col] = j + 1;
        } else {
            H[((int64_t)col * (k + 1) + j + 1) * k + j] = make_double2(nr, 0);
            sc = 1.0 / nr;
        }
    }
    scale[col] = sc;
}

// sign(X_col) for ncol matrices of size q (row-major, device) by Roberts' Newton iteration,
// every column until its update falls below 1e-12 of the iterate, then once more.  Returns
// 1 if a column met a singular iterate or did not converge in 100 steps.
int newton_sign_gpu(sgn_ctx* c, double2* X, int q, int ncol, int* failed) {
    cudaStream_t st = c->work;
    const size_t aug = (size_t)ncol * q * 2 * q;
    DevBuf buf;
    const int nu = (int)std::min<int64_t>(16, ((int64_t)q * q + 255) / 256);  // CTAs per matrix of the Newton update
    const size_t oA = 0, of = align256(sizeof(double2) * aug), ob = of + align256(sizeof(double2) * 2 * ncol * q),
                 os = ob + align256(sizeof(int) * ncol);
    SGN_CHECK(dev_alloc(c, buf, os + align256(sizeof(double) * 2 * ncol * nu)));
    char* base = reinterpret_cast<char*>(buf.p);
    double2* A = reinterpret_cast<double2*>(base + oA);
    double2* fac = reinterpret_cast<double2*>(base + of);
    int* bad = reinterpret_cast<int*>(base + ob);
    double* sums = reinterpret_cast<double*>(base + os);
    auto done_with = [&](int rc) {
        dev_free(c, buf);
        return rc;
    };
    // one inversion = q + 1 launches: captured once, replayed every Newton step
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const int64_t cells = (int64_t)q * 2 * q;
        launch_pdl(k_gj_load, dim3((unsigned)((cells + 255) / 256), ncol), 256, 0, st, X, A, fac, q);
        double2* two[2] = {fac, fac + (size_t)ncol * q};  // column p and column p + 1
        for (int p = 0; p < q && e == cudaSuccess; ++p) {
            launch_pdl(k_gj_step, dim3((2 * q - p - 1 + GJ_COLS - 1) / GJ_COLS, ncol), 256, 0, st, A, q, p, two[p & 1],
                       two[(p + 1) & 1], bad);
            e = cudaGetLastError();
        }
        launch_pdl(k_newton_update, dim3(nu, ncol), 256, 0, st, X, A, q, sums);
        cudaError_t ee = cudaStreamEndCapture(st, &g);
        if (e == cudaSuccess) e = ee;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        set_error(std::string("apply_direct: Newton graph: ") + cudaGetErrorString(e));
        return done_with(SGN_ERR_CUDA);
    }
    // per column: 0 iterating, 1 update below 1e-12 of the iterate (one more step to take),
    // 2 finished; every column steps with the others (a converged X is a fixed point)
    std::vector<double> hs(2 * (size_t)ncol * nu);
    std::vector<int> hb(ncol), state(ncol, 0);
    bool launch_ok = cudaMemsetAsync(bad, 0, sizeof(int) * ncol, st) == cudaSuccess;
    for (int it = 0; it < 100 && launch_ok; ++it) {
        if (cudaGraphLaunch(ge, st) != cudaSuccess ||
            cudaMemcpyAsync(hs.data(), sums, sizeof(double) * hs.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaMemcpyAsync(hb.data(), bad, sizeof(int) * ncol, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            launch_ok = false;
            break;
        }
        count_launch(2 + q);
        bool all = true;
        for (int col = 0; col < ncol; ++col) {
            if (hb[col] || state[col] == 2) continue;
            if (state[col] == 1) {
                state[col] = 2;
                continue;
            }
            double dn = 0, xn = 0;
            for (int u = 0; u < nu; ++u) {
                dn += hs[2 * (col * (size_t)nu + u)];
                xn += hs[2 * (col * (size_t)nu + u) + 1];
            }
            if (std::sqrt(dn) <= 1e-12 * std::sqrt(xn)) state[col] = 1;
            all = false;
        }
        if (all) break;
    }
    cudaGraphExecDestroy(ge);
    if (!launch_ok) {
        set_error("apply_direct: Newton iteration launch failed");
        return done_with(SGN_ERR_CUDA);
    }
    for (int col = 0; col < ncol; ++col)
        if (hb[col] || state[col] != 2) failed[col] = 1;
    return done_with(SGN_OK);
}

}  // namespace

int direct_projection(sgn_ctx* c, const double2* b, double2* x, int ncol, int k, bool adjoint, int* kk_out) {
    using cd = std::complex<double>;
    cudaStream_t st = c->work;
    const int64_t n = c->n;
    const int m = c->m;
    const size_t field = (size_t)n * sizeof(double2);
    const int rs = GS_BLOCK + 8;
    const int nblk = dot_blocks<double2>(n, ncol);
    const size_t oV = 0, ow = oV + align256(field * (size_t)(k + 1) * ncol);
    const size_t op = ow + align256(field * ncol);
    const size_t ored = op + align256(sizeof(double2) * (size_t)ncol * rs * nblk);
    const size_t ocoef = ored + align256(sizeof(double2) * (size_t)ncol * rs);
    const size_t oflag = ocoef + align256(sizeof(double2) * (size_t)ncol * rs);
    const size_t hcount = (size_t)ncol * (k + 1) * k;
    const size_t oH = oflag + align256(sizeof(int) * 4 * (size_t)ncol), osc = oH + align256(sizeof(double2) * hcount);
    const size_t total = osc + align256(sizeof(double) * 2 * (size_t)ncol);
    DevBuf buf;
    SGN_CHECK(dev_alloc(c, buf, total));
    char* base = reinterpret_cast<char*>(buf.p);
    double2* V = reinterpret_cast<double2*>(base + oV);
    double2* w = reinterpret_cast<double2*>(base + ow);
    double2* coef = reinterpret_cast<double2*>(base + ocoef);
    const Reduce rd{reinterpret_cast<double2*>(base + op), nblk, rs};
    DevState S{};
    S.red = reinterpret_cast<double2*>(base + ored);
    S.skip = reinterpret_cast<int*>(base + oflag);
    S.done = S.skip + ncol;
    S.rstride = rs;
    const int64_t sj = (int64_t)ncol * n;
    int *kk_dev = S.skip + 2 * ncol, *live_dev = kk_dev + ncol;
    double2* Hd = reinterpret_cast<double2*>(base + oH);
    double* scale = reinterpret_cast<double*>(base + osc);
    double* beta_dev = scale + ncol;
    auto bail = [&](int e) {
        dev_free(c, buf);
        return e;
    };
#define DC(call)                                                                     \
    do {                                                                             \
        cudaError_t e_ = (call);                                                     \
        if (e_ != cudaSuccess) {                                                     \
            set_error(std::string("apply_direct: ") + cudaGetErrorString(e_));      \
            return bail(SGN_ERR_CUDA);                                               \
        }                                                                            \
    } while (0)
    auto upload = [&](const std::vector<cd>& C, int J, int j0) -> cudaError_t {  // C[col][j0 .. j0+J) -> coef
        std::vector<double2> h((size_t)ncol * rs, make_double2(0, 0));
        const int ld = (int)(C.size() / ncol);
        for (int col = 0; col < ncol; ++col)
            for (int j = 0; j < J; ++j) {
                const cd v = C[(size_t)col * ld + j0 + j];
                h[(size_t)col * rs + j] = make_double2(v.real(), v.imag());
            }
        cudaError_t e = cudaMemcpyAsync(coef, h.data(), sizeof(double2) * h.size(), cudaMemcpyHostToDevice, st);
        return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
    };
    DC(cudaMemsetAsync(S.skip, 0, sizeof(int) * 2 * ncol, st));
    DC(cudaMemsetAsync(x, 0, field * ncol, st));
    // x_P and r = (I - P) b (eqs. (4.2), (4.3)); r goes to w
    const double2* Lb = reinterpret_cast<const double2*>(adjoint ? c->R64.p : c->L64.p);
    const double2* Rb = reinterpret_cast<const double2*>(adjoint ? c->L64.p : c->R64.p);
    const double2* lam = reinterpret_cast<const double2*>(adjoint ? c->lamc_dev.p : c->lam_dev.p);
    if (m > 0) {
        if (m > GS_BLOCK) {
            set_error("apply_direct: deflation size above 128");
            return bail(SGN_ERR_ARG);
        }
        const Basis<double2> LB{Lb, n, 0}, RB{Rb, n, 0};
        DC(mdot<double2>(LB, m, b, n, n, ncol, rd, 0, nullptr, st));
        DC(reduce(rd, m, ncol, RM_SIGNED, 0, S, lam, st));
        DC(update_x<double2>(RB, m, S.red, rs, x, n, n, ncol, nullptr, nullptr, st));
        DC(reduce(rd, m, ncol, RM_STORE, 0, S, nullptr, st));
        DC(maxpy_scale<double2>(RB, m, S.red, rs, b, n, w, n, nullptr, n, ncol, nullptr, st));
    } else {
        DC(cudaMemcpyAsync(w, b, field * ncol, cudaMemcpyDeviceToDevice, st));
    }
    // Arnoldi on A (eq. (2.4)) with two classical Gram-Schmidt passes; a column stops growing at its
    // first breakdown
    DC(cudaMemsetAsync(Hd, 0, sizeof(double2) * hcount, st));
    auto next_vector = [&](int j) -> cudaError_t {  // v_{j+1} = w / ||w||
        cudaError_t e = mdot<double2>(Basis<double2>{w, 0, n}, 0, w, n, n, ncol, rd, 1, nullptr, st);
        if (e != cudaSuccess) return e;
        launch_pdl(k_direct_norm, ncol, 256, 0, st, rd, j, k, Hd, scale, beta_dev, kk_dev, live_dev);
        count_launch();
        return maxpy_scale<double2>(Basis<double2>{w, 0, n}, 0, coef, rs, w, n, V + (size_t)(j + 1) * sj, n, scale, n,
                                    ncol, nullptr, st);
    };
    std::vector<double> beta(ncol);
    std::vector<int> flags(2 * (size_t)ncol);  // kk, live
    DC(next_vector(-1));
    for (int j = 0; j < k; ++j) {
        DC(apply_hw64(c, w, V + (size_t)j * sj, ncol, adjoint, nullptr, st));
        for (int pass = 0; pass < 2; ++pass)
            for (int i0 = 0; i0 <= j; i0 += GS_BLOCK) {
                const int J = std::min(GS_BLOCK, j + 1 - i0);
                const Basis<double2> VB{V + (size_t)i0 * sj, sj, n};
                DC(mdot<double2>(VB, J, w, n, n, ncol, rd, 0, nullptr, st));
                launch_pdl(k_direct_coef, dim3(ncol, (J + 31) / 32), 256, 0, st, rd, J, i0, j, k, S.red, rs, Hd);
                count_launch();
                DC(maxpy_scale<double2>(VB, J, S.red, rs, w, n, w, n, nullptr, n, ncol, nullptr, st));
            }
        DC(next_vector(j));
        if ((j + 1) % 32 == 0 || j + 1 == k) {
            DC(cudaMemcpyAsync(flags.data(), kk_dev, sizeof(int) * flags.size(), cudaMemcpyDeviceToHost, st));
            DC(cudaStreamSynchronize(st));
            if (std::none_of(flags.begin() + ncol, flags.end(), [](int v) { return v != 0; })) break;
        }
    }
    std::vector<cd> H(hcount);
    DC(cudaMemcpyAsync(beta.data(), beta_dev, sizeof(double) * ncol, cudaMemcpyDeviceToHost, st));
    DC(cudaMemcpyAsync(H.data(), Hd, sizeof(double2) * hcount, cudaMemcpyDeviceToHost, st));
    DC(cudaStreamSynchronize(st));
    const std::vector<int> kk(flags.begin(), flags.begin() + ncol);
    // y_col = beta sign(H_kk) e_1: Roberts' Newton iteration for all columns on the GPU,
    // each H_kk padded to the largest Krylov dimension with the identity
    const int kmaxu = *std::max_element(kk.begin(), kk.end());
    const int qd = std::max(kmaxu, 1);
    std::vector<cd> Y((size_t)ncol * qd, 0.0);
    std::vector<int> fail(ncol, 0);
    if (kmaxu > 0) {
        std::vector<double2> Xh((size_t)ncol * qd * qd, make_double2(0, 0));
        for (int col = 0; col < ncol; ++col) {
            const int q = kk[col];
            for (int r = 0; r < qd; ++r)
                for (int l = 0; l < qd; ++l) {
                    cd v = (r < q && l < q) ? H[((size_t)col * (k + 1) + r) * k + l] : cd(r == l ? 1.0 : 0.0, 0.0);
                    Xh[((size_t)col * qd + r) * qd + l] = make_double2(v.real(), v.imag());
                }
        }
        DevBuf xb;
        const int ra = dev_alloc(c, xb, sizeof(double2) * Xh.size());
        if (ra != SGN_OK) return bail(ra);
        double2* Xd = reinterpret_cast<double2*>(xb.p);
        auto xfail = [&](int code) {
            dev_free(c, xb);
            return bail(code);
        };
        if (cudaMemcpyAsync(Xd, Xh.data(), sizeof(double2) * Xh.size(), cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            set_error("apply_direct: copying H_k to the device failed");
            return xfail(SGN_ERR_CUDA);
        }
        const int rn = newton_sign_gpu(c, Xd, qd, ncol, fail.data());
        if (rn != SGN_OK) return xfail(rn);
        if (cudaMemcpyAsync(Xh.data(), Xd, sizeof(double2) * Xh.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            set_error("apply_direct: copying sign(H_k) to the host failed");
            return xfail(SGN_ERR_CUDA);
        }
        dev_free(c, xb);
        for (int col = 0; col < ncol; ++col)
            for (int r = 0; r < kk[col]; ++r) {
                const double2 v = Xh[((size_t)col * qd + r) * qd];  // first column of sign(H)
                Y[(size_t)col * qd + r] = beta[col] * cd(v.x, v.y);
            }
    }
    if (std::any_of(fail.begin(), fail.end(), [](int f) { return f != 0; })) {
        set_error("apply_direct: Newton iteration for sign(H_k) failed (singular iterate or no convergence)");
        return bail(SGN_ERR_NOT_CONVERGED);
    }
    // x += V_k y, in blocks
    for (int i0 = 0; i0 < kmaxu; i0 += GS_BLOCK) {
        const int J = std::min(GS_BLOCK, kmaxu - i0);
        DC(upload(Y, J, i0));
        DC(update_x<double2>(Basis<double2>{V + (size_t)i0 * sj, sj, n}, J, coef, rs, x, n, n, ncol, nullptr, nullptr,
                             st));
    }
    DC(cudaStreamSynchronize(st));
#undef DC
    if (kk_out) *kk_out = kmaxu;
    dev_free(c, buf);
    return SGN_OK;
}

}  // namespace sgn
