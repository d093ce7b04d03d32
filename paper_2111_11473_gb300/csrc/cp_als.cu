// Eigenvalue-weighted CP-ALS of the rank-reduced projectors (Eqs. 15-16,
// App. I): U_ia^P ~ sum_W y_i^W y_a^W tau^PW, minimising
//   f = sum_P eps_P^2 sum_ia (U_ia^P - sum_W y_i^W y_a^W tau^PW)^2
// by alternating least squares over y_o, y_v and tau, in float64 on the
// device.  The right-hand sides are products with the weighted factors
// (the MTTKRP of App. I's Eq. 46 as one GEMM plus a reduction over the
// other orbital index); the W x W normal equations (Eqs. 44-45) are solved
// by Cholesky factorisation instead of App. I's preconditioned CG.
// The large products run as exact integer slices on the tensor cores
// (gemm_tc.cu) where that is estimated to be faster and the operands allow it:
// slices are cut below one power of two per row, so that an output in which the
// large entries of a row of one operand meet small ones of the other's (U over
// eigenvalues of several decades) would lose what float64 sums keep.  Every
// product by slices is checked for that (k_slices_even); outputs that fail are done
// again as float64 sums, the whole product on the CUDA cores if they are more than
// a sixteenth.  With sums of |a b| at or above that scale the slices
// are the more accurate ones: rms error over the sum of |a b|, U of rank 200
// plus noise, 300 projectors, eigenvalues 1 .. 0.3: U te 2^-54.5 (float64 sums
// 2^-53.1), U^T KR 2^-55.9 (2^-51.4), KR tau^T 2^-54.4 (2^-53.8); without the
// check, eigenvalues over 6 decades and U large where they are small: 2^-33.8.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "common.cuh"
#include "gemm_tc.cuh"

namespace thc {

void set_thread_error(const std::string& msg);

namespace {

unsigned nblk(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 152 * 16); }

// te[P][X] = eps_P^2 tau[P][X]
__global__ void k_weight_rows(const double* tau, const double* eps, int N, int W, double* te) {
    grid_wait();
    const long long tot = (long long)N * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const double w = eps[e / W];
        te[e] = w * w * tau[e];
    }
}

// occ = 1: R[i][X] = sum_a M[(i,a)][X] yv[a][X];  occ = 0: R[a][X] = sum_i M[(i,a)][X] yo[i][X]
__global__ void k_reduce_other(const double* M, const double* f, int o, int v, int W, int occ,
                               double* R) {
    grid_wait();
    const int rows = occ ? o : v, other = occ ? v : o;
    const long long tot = (long long)rows * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(e / W), X = (int)(e % W);
        double s = 0;
        for (int q = 0; q < other; ++q) {
            const long long row = occ ? (long long)r * v + q : (long long)q * v + r;
            s += M[row * W + X] * f[(long long)q * W + X];
        }
        R[e] = s;
    }
}

// KR[(i,a)][X] = yo[i][X] yv[a][X]
__global__ void k_khatri_rao(const double* yo, const double* yv, int o, int v, int W, double* KR) {
    grid_wait();
    const long long tot = (long long)o * v * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const long long row = e / W;
        const int X = (int)(e % W), i = (int)(row / v), a = (int)(row % v);
        KR[e] = yo[(long long)i * W + X] * yv[(long long)a * W + X];
    }
}

__global__ void k_mul(double* a, const double* b, long long n) {
    grid_wait();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        a[e] *= b[e];
}

// part[block] = sum over its elements of (eps_P (U - rec))^2, U, rec: (ov) x N
__global__ void k_wsq(const double* U, const double* rec, const double* eps, long long rows,
                      int N, double* part) {
    grid_wait();
    __shared__ double red[32];
    double s = 0;
    const long long tot = rows * N;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const double d = eps[e % N] * (U[e] - rec[e]);
        s += d * d;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = s;
    __syncthreads();
    if (w == 0) {
        s = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) part[blockIdx.x] = s;
    }
}

// Cholesky factorisation and solve of the W x W normal equations.  Both are
// chains: W pivots, each a square root, a broadcast and a column update, and
// 2 W / 32 steps of every right-hand side; float64 units are few (two fused
// multiply-adds per clock and SM), so the updates between the chains are
// spread over as many SMs as possible.  32 columns at a time:
//   panel:  every block factors the 32 x 32 diagonal block for itself (cheaper
//           than handing it over) and solves 8 rows of the panel below it;
//   update: one 16 x 16 tile of the remaining lower triangle per block.
// The panel is also stored mirrored, so that both triangular solves read S
// along its rows.  Three solves of W = 200 with 40, 200 and 300 right-hand
// sides took 3.2 ms in the vendor's factorisation and solve, where the
// multiply-adds take 0.03 ms of all SMs.
constexpr int CB = 32;
// Per diagonal block: F[l][j] = L[j][l] / L[l][l] (j > l), B[l][j] =
// L[l][j] / L[l][l] (j < l) and 1 / L[l][l].
constexpr int kDiagDoubles = 2 * CB * CB + CB;
constexpr int kSolveSmem = 200 * 1024;   // rows of one block of the substitution

__global__ void __launch_bounds__(128) k_chol_panel(double* S, int W, int k0, double* D,
                                                    int* info) {
    grid_wait();
    __shared__ double L[CB][CB + 1];
    __shared__ double col[2][CB];
    __shared__ double rinv[CB];
    const int nb = min(CB, W - k0), r = threadIdx.x & 31, w = threadIdx.x >> 5;
    // thread (r, w) holds row r, columns 4 m + w; rows and columns beyond W are the identity's
    double a[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const int j = 4 * m + w;
        a[m] = r < nb && j <= r ? S[(long long)(k0 + r) * W + k0 + j] : (r == j ? 1.0 : 0.0);
    }
#pragma unroll
    for (int l = 0; l < CB; ++l) {
        if (w == (l & 3)) {
            const double p = __shfl_sync(0xffffffffu, a[l >> 2], l);
            const double ri = rsqrt(p);
            const double c = r >= l ? a[l >> 2] * ri : 0.0;
            col[l & 1][r] = c;
            L[r][l] = c;
            if (r == l) {
                rinv[l] = ri;
                if (!(p > 0.0) && blockIdx.x == 0) atomicCAS(info, 0, k0 + l + 1);
            }
        }
        __syncthreads();
        const double lr = col[l & 1][r];
#pragma unroll
        for (int m = 0; m < 8; ++m)
            if (4 * m + w > l) a[m] -= lr * col[l & 1][4 * m + w];
    }
    if (blockIdx.x == 0) {
        double* d = D + (long long)(k0 / CB) * kDiagDoubles;
        for (int e = threadIdx.x; e < CB * CB; e += 128) {
            const int l = e / CB, j = e % CB;
            d[e] = j > l ? L[j][l] * rinv[l] : 0.0;
            d[CB * CB + e] = j < l ? L[l][j] * rinv[l] : 0.0;
        }
        if (threadIdx.x < CB) d[2 * CB * CB + threadIdx.x] = rinv[threadIdx.x];
    }
    // rows below: 16 lanes per row, columns g and g + 16
    const int g = r & 15, i = k0 + CB + blockIdx.x * 8 + w * 2 + (r >> 4);
    const bool ok = i < W;
    double x0 = ok ? S[(long long)i * W + k0 + g] : 0.0;
    double x1 = ok ? S[(long long)i * W + k0 + g + 16] : 0.0;
#pragma unroll
    for (int l = 0; l < CB; ++l) {
        const double x = (l < 16 ? x0 : x1) * rinv[l];
        const double xl = __shfl_sync(0xffffffffu, x, (r & 16) | (l & 15));
        if (l < 16) {
            if (g == l) x0 = xl;
            if (g > l) x0 -= xl * L[g][l];
            x1 -= xl * L[g + 16][l];
        } else {
            if (g + 16 == l) x1 = xl;
            if (g + 16 > l) x1 -= xl * L[g + 16][l];
        }
    }
    if (ok) {
        S[(long long)i * W + k0 + g] = x0;
        S[(long long)i * W + k0 + g + 16] = x1;
        S[(long long)(k0 + g) * W + i] = x0;
        S[(long long)(k0 + g + 16) * W + i] = x1;
    }
}

// Lower triangle beyond the panel at k0, a 16 x 16 tile per block:
// S[i][j] -= sum_l X[i][l] X[j][l].
__global__ void __launch_bounds__(256) k_chol_update(double* S, int W, int k0) {
    grid_wait();
    __shared__ double xi[16][CB + 1], xj[16][CB + 1];
    int ti = (int)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
    while ((long long)ti * (ti + 1) / 2 > blockIdx.x) --ti;
    while ((long long)(ti + 1) * (ti + 2) / 2 <= blockIdx.x) ++ti;
    const int tj = (int)(blockIdx.x - (long long)ti * (ti + 1) / 2);
    const int i0 = k0 + CB + ti * 16, j0 = k0 + CB + tj * 16;
    for (int e = threadIdx.x; e < 16 * CB; e += 256) {
        const int q = e / CB, l = e % CB;
        xi[q][l] = i0 + q < W ? S[(long long)(i0 + q) * W + k0 + l] : 0.0;
        xj[q][l] = j0 + q < W ? S[(long long)(j0 + q) * W + k0 + l] : 0.0;
    }
    __syncthreads();
    const int i = i0 + threadIdx.x / 16, j = j0 + threadIdx.x % 16;
    if (i >= W || j > i) return;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int l = 0; l < CB; l += 2) {
        s0 += xi[threadIdx.x / 16][l] * xj[threadIdx.x % 16][l];
        s1 += xi[threadIdx.x / 16][l + 1] * xj[threadIdx.x % 16][l + 1];
    }
    S[(long long)i * W + j] -= s0 + s1;
}

// out = B S^-1 for RR rows of B per block, from the factor in S and D: the
// eight warps share the sums over the columns done before (or, backwards,
// after), one warp per row then runs the chain over a diagonal block.  The
// rows are worked on in shared memory, or in out itself if they do not fit.
template <int RR>
__global__ void __launch_bounds__(256) k_chol_solve(const double* S, int W, const double* D,
                                                    const double* B, int rows, double* out,
                                                    int in_smem) {
    grid_wait();
    extern __shared__ double ybuf[];
    __shared__ double red[8][RR][CB];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long row0 = (long long)blockIdx.x * RR;
    const int nr = (int)min((long long)RR, rows - row0);
    double* y = in_smem ? ybuf : out + row0 * W;
    for (long long e = threadIdx.x; e < (long long)nr * W; e += 256) y[e] = B[row0 * W + e];
    __syncthreads();
    const int nblk = (W + CB - 1) / CB;
    for (int step = 0; step < 2 * nblk; ++step) {
        const bool fwd = step < nblk;
        const int k = fwd ? step : 2 * nblk - 1 - step;
        const int k0 = k * CB, lo = fwd ? 0 : k0 + CB, hi = fwd ? k0 : W;
        const bool cok = k0 + lane < W;
        const double* d = D + (long long)k * kDiagDoubles;
        double f[CB];
        if (w < nr) {
#pragma unroll
            for (int l = 0; l < CB; ++l) f[l] = d[(fwd ? 0 : CB * CB) + l * CB + lane];
        }
        double acc[RR] = {};
#pragma unroll 4
        for (int l = lo + w; l < hi; l += 8) {
            const double sv = cok ? S[(long long)l * W + k0 + lane] : 0.0;
#pragma unroll
            for (int r = 0; r < RR; ++r)
                if (r < nr) acc[r] += sv * y[(long long)r * W + l];
        }
#pragma unroll
        for (int r = 0; r < RR; ++r) red[w][r][lane] = acc[r];
        __syncthreads();
        if (w < nr) {
            double* yr = y + (long long)w * W + k0;
            double t = cok ? yr[lane] : 0.0;
            double sum = 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) sum += red[q][w][lane];
            t -= sum;
#pragma unroll
            for (int e = 0; e < CB; ++e) {
                const int l = e;
                if (fwd) t -= f[l] * __shfl_sync(0xffffffffu, t, l);
                else t -= f[CB - 1 - l] * __shfl_sync(0xffffffffu, t, CB - 1 - l);
            }
            if (cok) yr[lane] = t * d[2 * CB * CB + lane];
        }
        __syncthreads();
    }
    if (in_smem)
        for (long long e = threadIdx.x; e < (long long)nr * W; e += 256) out[row0 * W + e] = y[e];
}

struct Dev {
    double* p = nullptr;
    ~Dev() { release(); }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
    }
    cudaError_t alloc(size_t n) { return cudaMalloc(&p, n * sizeof(double)); }
};

View<double> rmv(const double* p, long long ld) { return View<double>{p, ld, 1}; }
View<double> trv(const double* p, long long ld) { return View<double>{p, 1, ld}; }

struct Als {
    int o, v, N, W;
    long long ov;
    cudaStream_t st;
    Dev S, S2, SE, M, KR, R, te, rec, part, ws, diag, info;
    Dev slices, fpart, expo, list;
    static constexpr int kRedo = 1 << 16;   // outputs of a product done again
    F64TcWorkspace tc;
    bool expired = false;   // a bounded wait of a product
    std::string err;

    cudaError_t init() {
        cudaError_t e;
        const long long mx = std::max<long long>(std::max<long long>(o, v), N);
        if ((e = S.alloc((size_t)W * W)) || (e = S2.alloc((size_t)W * W)) ||
            (e = SE.alloc((size_t)W * W)) ||
            (e = M.alloc((size_t)ov * W)) || (e = KR.alloc((size_t)ov * W)) ||
            (e = R.alloc((size_t)mx * W)) || (e = te.alloc((size_t)N * W)) ||
            (e = rec.alloc((size_t)ov * N)) || (e = part.alloc(152 * 16)) ||
            (e = ws.alloc(1 << 22)) || (e = diag.alloc((size_t)cdiv(W, CB) * kDiagDoubles)) ||
            (e = info.alloc(2)))
            return e;
        return cudaMemsetAsync(info.p, 0, 2 * sizeof(double), st);
    }

    // Tensor-core products: room for the largest in one piece, at most 2 GiB of
    // slices and 512 MiB of partial sums (larger ones are cut).  Optional, hence
    // after everything else: without the memory the products stay on the CUDA cores.
    void init_slices() {
        size_t sl = 0, pt = 0, ex = 0;
        const long long shapes[][3] = {{ov, W, N}, {W, W, N}, {W, W, v}, {W, W, o},
                                       {N, W, ov}, {ov, N, W}};
        for (const auto& sh : shapes) {
            if (std::max({sh[0], sh[1], sh[2]}) > INT32_MAX ||
                !f64_tc_pays((int)sh[0], (int)sh[1], (int)sh[2], 1, false))
                continue;
            size_t a, b, c;
            gemm_f64_tc_sizes((int)sh[0], (int)sh[1], (int)sh[2], 1, false, &a, &b, &c);
            sl = std::max(sl, a);
            pt = std::max(pt, b);
            ex = std::max(ex, c);
        }
        if (sl > 0) {
            sl = std::min<size_t>(sl, 1ULL << 30);
            pt = std::min<size_t>(pt, 1ULL << 27);
            if (slices.alloc(sl / 4 + 1) || fpart.alloc(pt / 2 + 1) || expo.alloc(ex / 2 + 1) ||
                list.alloc(kRedo)) {
                cudaGetLastError();   // not enough memory
                for (Dev* d : {&slices, &fpart, &expo, &list}) d->release();
            } else {
                tc.slices = reinterpret_cast<__nv_bfloat16*>(slices.p);
                tc.slice_elems = sl;
                tc.part = reinterpret_cast<float*>(fpart.p);
                tc.part_elems = pt;
                tc.expo = reinterpret_cast<int*>(expo.p);
                tc.expo_elems = ex;
                tc.err = reinterpret_cast<int*>(info.p) + 1;
                tc.redo = tc.err + 1;
                tc.redo_list = reinterpret_cast<int2*>(list.p);
                tc.redo_cap = kRedo;
            }
        }
    }

    // C (M x N) = A B, row-major views.
    cudaError_t gemm(int m, int n, int k, View<double> A, View<double> B, double* C) {
        Gemm<double> g;
        g.M = m; g.N = n; g.K = k;
        g.A = A; g.B = B; g.C = C; g.ldc = n;
        g.ws = ws.p; g.ws_elems = 1 << 22;
        if (tc.slices && f64_tc_pays(m, n, k, 1, false)) {
            int flags[3] = {0, 0, 0};   // a wait expired; -; too many outputs to do again
            cudaError_t e = cudaMemsetAsync(tc.redo + 1, 0, sizeof(int), st);
            if (!e) e = gemm_f64_tc(g, tc, st);
            if (!e) e = cudaMemcpyAsync(flags, tc.err, sizeof(flags), cudaMemcpyDeviceToHost, st);
            if (!e) e = cudaStreamSynchronize(st);
            if (!e && flags[0]) {
                expired = true;
                return cudaErrorUnknown;
            }
            if (!e && !flags[2]) return cudaSuccess;
            if (e && e != cudaErrorMemoryAllocation) return e;
        }
        return gemm_simt(g, st);
    }

    // S = (Aᵀ A) o (Bᵀ B) for row-major A (na x W), B (nb x W)
    cudaError_t gram2(const double* A, int na, const double* B, int nb) {
        cudaError_t e;
        if ((e = gemm(W, W, na, trv(A, W), rmv(A, W), S.p))) return e;
        if ((e = gemm(W, W, nb, trv(B, W), rmv(B, W), S2.p))) return e;
        launch_chained(k_mul, nblk((long long)W * W), 256, 0, st, S.p, S2.p, (long long)W * W);
        count_launches(1);
        return cudaGetLastError();
    }

    // out (rows x W, row-major) = R S^-1 by Cholesky of the symmetric S.
    cudaError_t solve(int rows, double* out) {
        cudaError_t e;
        int hinfo = 0;
        if ((e = cudaMemcpyAsync(S2.p, S.p, sizeof(double) * W * W, cudaMemcpyDeviceToDevice, st)))
            return e;
        for (int attempt = 0; attempt < 2; ++attempt) {
            if ((e = factor())) return e;
            if ((e = cudaMemcpyAsync(&hinfo, info.p, sizeof(int), cudaMemcpyDeviceToHost, st)) ||
                (e = cudaStreamSynchronize(st)))
                return e;
            if (hinfo == 0) break;
            // Numerically singular: retry once with a ridge of 1e-12 of the largest diagonal.
            std::vector<double> hs((size_t)W * W);
            if ((e = cudaMemcpy(hs.data(), S2.p, sizeof(double) * W * W, cudaMemcpyDeviceToHost)))
                return e;
            double dmax = 0;
            for (int k = 0; k < W; ++k) dmax = std::max(dmax, std::fabs(hs[(size_t)k * W + k]));
            for (int k = 0; k < W; ++k) hs[(size_t)k * W + k] += 1e-12 * dmax;
            if ((e = cudaMemcpy(S.p, hs.data(), sizeof(double) * W * W, cudaMemcpyHostToDevice)))
                return e;
        }
        if (hinfo != 0) {
            err = "cp_als: normal equations are singular";
            return cudaErrorInvalidValue;
        }
        // Rows per block: as few as one block per SM takes, at most four (the
        // units' work is the same; more rows share the reads of the factor).
        int rr = (int)std::min<long long>(4, cdiv(rows, device_sms()));
        while (rr > 1 && sizeof(double) * rr * W > kSolveSmem) --rr;
        return rr <= 1 ? substitute<1>(rows, out)
                       : (rr <= 3 ? substitute<2>(rows, out) : substitute<4>(rows, out));
    }

    cudaError_t factor() {
        cudaError_t e = cudaMemsetAsync(info.p, 0, sizeof(int), st);
        for (int k0 = 0; k0 < W && !e; k0 += CB) {
            const int rest = std::max(0, W - k0 - CB);
            launch_chained(k_chol_panel, std::max(1u, cdiv(rest, 8)), 128, 0, st, S.p, W, k0,
                           diag.p, (int*)info.p);
            count_launches(1);
            if (rest > 0) {
                const long long T = cdiv(rest, 16);
                launch_chained(k_chol_update, (unsigned)(T * (T + 1) / 2), 256, 0, st, S.p, W, k0);
                count_launches(1);
            }
            e = cudaGetLastError();
        }
        return e;
    }

    template <int RR>
    cudaError_t substitute(int rows, double* out) {
        size_t smem = sizeof(double) * RR * W;
        const int fits = smem <= kSolveSmem;
        if (!fits) smem = 0;
        cudaError_t e = smem_optin((const void*)k_chol_solve<RR>, kSolveSmem);
        if (e) return e;
        launch_chained(k_chol_solve<RR>, cdiv(rows, RR), 256, smem, st, S.p, W, diag.p, R.p, rows,
                       out, fits);
        count_launches(1);
        return cudaGetLastError();
    }

    cudaError_t objective(const double* U, const double* eps, const double* yo, const double* yv,
                          const double* tau, double* f) {
        cudaError_t e;
        launch_chained(k_khatri_rao, nblk(ov * W), 256, 0, st, yo, yv, o, v, W, KR.p);
        count_launches(1);
        if ((e = cudaGetLastError())) return e;
        if ((e = gemm((int)ov, N, W, rmv(KR.p, W), trv(tau, W), rec.p)))
            return e;
        const unsigned nb = nblk(ov * N);
        launch_chained(k_wsq, nb, 256, 0, st, U, rec.p, eps, ov, N, part.p);
        count_launches(1);
        if ((e = cudaGetLastError())) return e;
        std::vector<double> hp(nb);
        if ((e = cudaMemcpyAsync(hp.data(), part.p, sizeof(double) * nb, cudaMemcpyDeviceToHost, st)) ||
            (e = cudaStreamSynchronize(st)))
            return e;
        double s = 0;
        for (double x : hp) s += x;
        *f = s;
        return cudaSuccess;
    }

    cudaError_t sweep(const double* U, const double* eps, double* yo, double* yv, double* tau) {
        cudaError_t e;
        // y_o and y_v share M = U diag(eps^2) tau (tau is fixed in both updates)
        launch_chained(k_weight_rows, nblk((long long)N * W), 256, 0, st, tau, eps, N, W, te.p);
        count_launches(1);
        if ((e = cudaGetLastError())) return e;
        if ((e = gemm((int)ov, W, N, rmv(U, N), rmv(te.p, W), M.p)))
            return e;
        // y_o: S = (y_v^T y_v) o (tau^T E tau)
        if ((e = gemm(W, W, N, trv(tau, W), rmv(te.p, W), SE.p))) return e;
        if ((e = gemm(W, W, v, trv(yv, W), rmv(yv, W), S.p))) return e;
        launch_chained(k_mul, nblk((long long)W * W), 256, 0, st, S.p, SE.p, (long long)W * W);
        launch_chained(k_reduce_other, nblk((long long)o * W), 256, 0, st, M.p, yv, o, v, W, 1, R.p);
        count_launches(2);
        if ((e = cudaGetLastError())) return e;
        if ((e = solve(o, yo))) return e;
        // y_v: S = (y_o^T y_o) o (tau^T E tau)
        if ((e = gemm(W, W, o, trv(yo, W), rmv(yo, W), S.p))) return e;
        launch_chained(k_mul, nblk((long long)W * W), 256, 0, st, S.p, SE.p, (long long)W * W);
        launch_chained(k_reduce_other, nblk((long long)v * W), 256, 0, st, M.p, yo, o, v, W, 0, R.p);
        count_launches(2);
        if ((e = cudaGetLastError())) return e;
        if ((e = solve(v, yv))) return e;
        // tau: S = (y_o^T y_o) o (y_v^T y_v), R = U^T KR(y_o, y_v)
        if ((e = gram2(yo, o, yv, v))) return e;
        launch_chained(k_khatri_rao, nblk(ov * W), 256, 0, st, yo, yv, o, v, W, KR.p);
        count_launches(1);
        if ((e = cudaGetLastError())) return e;
        if ((e = gemm(N, W, (int)ov, trv(U, N), rmv(KR.p, W), R.p)))
            return e;
        return solve(N, tau);
    }
};

}  // namespace
}  // namespace thc

extern "C" thc_status thc_cp_als(int n_occ, int n_vir, int n_rr, int rank, const double* U,
                                 const double* eps, double* y_o, double* y_v, double* tau,
                                 int iters, double* objective, void* stream) {
    using namespace thc;
    if (n_occ <= 0 || n_vir <= 0 || n_rr <= 0 || rank <= 0 || iters < 0 || !U || !eps || !y_o ||
        !y_v || !tau) {
        set_thread_error("thc_cp_als: non-positive size or NULL pointer");
        return THC_ERR_ARG;
    }
    Als a;
    a.o = n_occ; a.v = n_vir; a.N = n_rr; a.W = rank;
    a.ov = (long long)n_occ * n_vir;
    a.st = (cudaStream_t)stream;
    cudaError_t e = a.init();
    // Device copies of the inputs and of the factors (updated in place).
    Dev dU, de, dyo, dyv, dt;
    const size_t nU = (size_t)a.ov * n_rr;
    const size_t no = (size_t)n_occ * rank, nv = (size_t)n_vir * rank, nt = (size_t)n_rr * rank;
    if (!e) e = dU.alloc(nU);
    if (!e) e = de.alloc(n_rr);
    if (!e) e = dyo.alloc(no);
    if (!e) e = dyv.alloc(nv);
    if (!e) e = dt.alloc(nt);
    if (!e) a.init_slices();
    if (!e) e = cudaMemcpyAsync(dU.p, U, sizeof(double) * nU, cudaMemcpyDefault, a.st);
    if (!e) e = cudaMemcpyAsync(de.p, eps, sizeof(double) * n_rr, cudaMemcpyDefault, a.st);
    if (!e) e = cudaMemcpyAsync(dyo.p, y_o, sizeof(double) * no, cudaMemcpyDefault, a.st);
    if (!e) e = cudaMemcpyAsync(dyv.p, y_v, sizeof(double) * nv, cudaMemcpyDefault, a.st);
    if (!e) e = cudaMemcpyAsync(dt.p, tau, sizeof(double) * nt, cudaMemcpyDefault, a.st);
    for (int it = 0; it < iters && !e; ++it) {
        e = a.sweep(dU.p, de.p, dyo.p, dyv.p, dt.p);
        if (!e && objective) {
            double f = 0;
            e = a.objective(dU.p, de.p, dyo.p, dyv.p, dt.p, &f);
            if (!e) objective[it] = f;
        }
    }
    if (!e) e = cudaMemcpyAsync(y_o, dyo.p, sizeof(double) * no, cudaMemcpyDefault, a.st);
    if (!e) e = cudaMemcpyAsync(y_v, dyv.p, sizeof(double) * nv, cudaMemcpyDefault, a.st);
    if (!e) e = cudaMemcpyAsync(tau, dt.p, sizeof(double) * nt, cudaMemcpyDefault, a.st);
    if (!e) e = cudaStreamSynchronize(a.st);
    if (a.expired) {
        set_thread_error("thc_cp_als: a tensor-core kernel's bounded wait expired");
        return THC_ERR_TIMEOUT;
    }
    if (e) {
        set_thread_error(a.err.empty() ? std::string("thc_cp_als: ") + cudaGetErrorString(e)
                                       : "thc_cp_als: " + a.err);
        return a.err.empty() ? THC_ERR_CUDA : THC_ERR_NUMERIC;
    }
    return THC_OK;
}
