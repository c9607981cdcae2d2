// Row orthonormalisation of a complex m x n matrix (m <= n) by CholeskyQR2 on the FP64 GEMM.
//
// Gram-Schmidt of the rows in order is the LQ factorisation A = L Q with L lower triangular
// and a positive diagonal; so is CholeskyQR: G = A A^dag = L L^dag (Cholesky), Q = L^{-1} A.
// One pass loses orthogonality like u kappa(A)^2; a second pass on Q restores it to O(u)
// while kappa(A) stays well below u^{-1/2} (Yamamoto et al., ETNA 44, 2015).  Every O(m^2 n)
// and O(m^3) step is a complex GEMM spread over all SMs:
//   Gram           G = A A^dag (lower tiles);
//   Cholesky       right-looking in blocks of NB: the diagonal block is factored (and its
//                  factor inverted) by one CTA, the panel below is L21 = A21 L11^{-dag} and the
//                  trailing matrix is updated by G22 -= L21 L21^dag;
//   solve          Q = L^{-1} A by block rows: A_b -= L[b, <b] Q[<b], Q_b = L_bb^{-1} A_b.
// The second pass checks its Gram matrix first: if max |G - I| > 0.1 (or a pivot of either
// pass was not positive, or a value is not finite) the rows were too ill-conditioned -- or
// exactly dependent -- for CholeskyQR, and the original rows are orthonormalised again by the
// row-by-row Gram-Schmidt kernel, which keeps an exactly dependent row at zero.  Both branches
// are queued; a device flag selects which one acts, so nothing is read back to the host.
#include <algorithm>

#include "vtn_internal.cuh"

namespace vtn {
namespace {

constexpr int NB = 32;  // diagonal block of the blocked Cholesky and of the triangular solve

// 1 / x and 1 / sqrt(x) from an FP32 start by two Newton steps each: the serial chain of the factorisation is
// these, and an FP64 instruction takes about 30 ns whether or not others could run beside it.  x is scaled into
// FP32's range by the caller.
__device__ __forceinline__ double recip_newton(double x) {
    double r = (double)__frcp_rn((float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}
__device__ __forceinline__ double rsqrt_newton(double x) {
    double r = (double)rsqrtf((float)x);
#pragma unroll
    for (int i = 0; i < 2; ++i) r = fma(0.5 * r, fma(-x * r, r, 1.0), r);
    return r;
}

// Cholesky factor of the b x b diagonal block at G (leading dimension ld; lower triangle read
// and written) and the inverse of that factor into Linv (NB x NB, zero above the diagonal).
// One CTA, b <= NB.  flag[0] = 1 on a pivot that is not positive.
// FP64-issue bound (about 2 x 170 warp-wide element updates of 6 instructions), so the elements left of each step are
// dealt out densely to the lanes: L D L^dag with unit L, the update of column j and the same row operations on
// the growing inverse in one pass with one barrier, the square roots taken once at the end, the next pivot while
// the others still work.  168 -> 50 us for a block of 32 (three barriers a column and the inverse as 32 serial dot products before).
__global__ void __launch_bounds__(256) potrf_block(double2* __restrict__ G, int b, long long ld,
                                                  double2* __restrict__ Linv, int* __restrict__ flag) {
    __shared__ double2 S[NB][NB + 1];
    __shared__ double2 X[NB][NB + 1];
    __shared__ double D[NB];
    __shared__ int bad;
    const int tid = threadIdx.x;
    if (tid == 0) bad = 0;
    for (int t = tid; t < NB * NB; t += 256) {
        const int i = t / NB, j = t - (t / NB) * NB;
        S[i][j] = (i < b && j <= i) ? G[(long long)i * ld + j] : make_double2(0.0, 0.0);
        X[i][j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    if (tid < 32) {
        // row scaling by powers of two: D^-1/2 of the diagonal, so that every pivot is within [0, 4)
        int e = 0;
        if (tid < b) {
            const double d = S[tid][tid].x;
            e = d > 0.0 && d < 1e300 ? ilogb(d) / 2 : 0;
        }
        D[tid] = (double)e;
    }
    __syncthreads();
    for (int t = tid; t < NB * NB; t += 256) {
        const int i = t / NB, j = t - (t / NB) * NB;
        if (j <= i) {
            const int e = -(int)D[i] - (int)D[j];
            S[i][j].x = scalbn(S[i][j].x, e);
            S[i][j].y = scalbn(S[i][j].y, e);
        }
    }
    __shared__ int row_exp[NB];
    __shared__ double piv[NB], pinv[NB];
    __syncthreads();
    if (tid < NB) row_exp[tid] = (int)D[tid];
    // (row, column) of the t-th element of a lower triangle counted by rows: the same for every size
    __shared__ unsigned char ti[NB * (NB + 1) / 2], tl[NB * (NB + 1) / 2];
    for (int t = tid; t < NB * NB; t += 256) {
        const int i = t / NB, l = t - (t / NB) * NB;
        if (l <= i) {
            ti[i * (i + 1) / 2 + l] = (unsigned char)i;
            tl[i * (i + 1) / 2 + l] = (unsigned char)l;
        }
    }
    // pivot j and its reciprocal; the thread that updates S[j + 1][j + 1] takes the next one while the others work
    auto take_pivot = [&](int j, double d) {
        if (!(d > 1e-30)) {  // pivots are relative to their row's norm; the caller's fallback replaces the result
            bad = 1;
            d = 1.0;
        }
        piv[j] = d;
        pinv[j] = recip_newton(d);
    };
    if (tid == 0) take_pivot(0, S[0][0].x);
    __syncthreads();
    for (int j = 0; j < b; ++j) {
        const double inv = pinv[j];
        const int r = b - 1 - j;
        const int n_s = r * (r + 1) / 2, n_x = r * (j + 1);
        const float wi = 1.0f / (float)(j + 1);
        for (int t = tid; t < n_s + n_x; t += 256) {
            if (t < n_s) {  // S[i][l] -= S[i][j] conj(S[l][j]) / d, j < l <= i
                const int i = ti[t] + j + 1, l = tl[t] + j + 1;
                double2 a = S[i][j];
                const double2 c = S[l][j];
                a.x *= inv;
                a.y *= inv;
                double2 s = S[i][l];
                s.x = fma(-a.x, c.x, fma(-a.y, c.y, s.x));
                s.y = fma(-a.y, c.x, fma(a.x, c.y, s.y));
                S[i][l] = s;
                if (t == 0) take_pivot(j + 1, s.x);
            } else {  // X[i][l] -= S[i][j] / d X[j][l], i > j, l <= j
                const int u = t - n_s;
                int q = (int)((float)u * wi);
                q += (q + 1) * (j + 1) <= u;
                q -= q * (j + 1) > u;
                const int i = j + 1 + q, l = u - q * (j + 1);
                double2 a = S[i][j];
                const double2 x = X[j][l];
                a.x *= inv;
                a.y *= inv;
                double2 s = X[i][l];
                s.x = fma(-a.x, x.x, fma(a.y, x.y, s.x));
                s.y = fma(-a.x, x.y, fma(-a.y, x.x, s.y));
                X[i][l] = s;
            }
        }
        __syncthreads();
    }
    if (tid < NB) D[tid] = tid < b ? rsqrt_newton(piv[tid]) : 1.0;
    __syncthreads();
    // L = (unit L) D^1/2 and its inverse, with the row scaling undone
    for (int t = tid; t < NB * NB; t += 256) {
        const int i = t / NB, j = t - (t / NB) * NB;
        double2 x = make_double2(0.0, 0.0);
        if (i < b && j <= i) {
            const double2 s = i == j ? make_double2(piv[j], 0.0) : S[i][j];
            G[(long long)i * ld + j] = make_double2(scalbn(s.x * D[j], row_exp[i]), scalbn(s.y * D[j], row_exp[i]));
            x = make_double2(scalbn(X[i][j].x * D[i], -row_exp[j]), scalbn(X[i][j].y * D[i], -row_exp[j]));
        }
        Linv[t] = x;
    }
    if (tid == 0 && bad) flag[0] = 1;
}

// flag[0] = 1 if max over the lower triangle of |G - I| > tol or a value is not finite
__global__ void __launch_bounds__(256) gram_identity_check(const double2* __restrict__ G, int m, double tol,
                                                          int* __restrict__ flag) {
    double mx = 0.0;
    const long long total = (long long)m * m;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
        const long long i = t / m, j = t - (t / m) * m;
        if (j > i) continue;
        const double2 g = G[t];
        const double dev = fmax(fabs(g.x - (i == j ? 1.0 : 0.0)), fabs(g.y));
        mx = (dev == dev) ? fmax(mx, dev) : 1e300;
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx > tol) flag[0] = 1;
}

// dst = src (n elements) when *pred != 0
__global__ void copy_if(double2* __restrict__ dst, const double2* __restrict__ src, long long n,
                        const int* __restrict__ pred) {
    if (*pred == 0) return;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
        dst[t] = src[t];
}

// Lower Cholesky factor of the m x m Hermitian G in place (lower triangle), blocks of NB;
// Linv_all[c] = inverse of diagonal block c (NB x NB); tmp: at least (m - NB) x NB complex.
void cholesky_blocked(Ctx& ctx, double2* G, int m, double2* Linv_all, double2* tmp, int* flag) {
    for (int p = 0; p < m; p += NB) {
        const int b = std::min(NB, m - p);
        double2* Li = Linv_all + (size_t)(p / NB) * NB * NB;
        potrf_block<<<1, 256, 0, ctx.stream>>>(G + (size_t)p * m + p, b, m, Li, flag);
        ctx.count_launch();
        ctx.check_launch("potrf_block");
        const int rest = m - p - b;
        if (rest <= 0) break;
        double2* L21 = G + (size_t)(p + b) * m + p;
        GemmArgs t;  // tmp = A21 L11^{-dag}
        t.M = rest; t.N = b; t.K = b;
        t.A = L21; t.lda = m;
        t.opB = OP_C; t.B = Li; t.ldb = NB;
        t.C = tmp; t.ldc = b;
        gemm_c64(ctx, t);
        VTN_CUDA_TRY(cudaMemcpy2DAsync(L21, sizeof(double2) * (size_t)m, tmp, sizeof(double2) * (size_t)b,
                                       sizeof(double2) * (size_t)b, rest, cudaMemcpyDeviceToDevice, ctx.stream));
        GemmArgs u;  // G22 -= L21 L21^dag
        u.M = rest; u.N = rest; u.K = b;
        u.A = L21; u.lda = m;
        u.opB = OP_C; u.B = L21; u.ldb = m;
        u.C = L21 + b; u.ldc = m;
        u.accumulate = true;
        u.negate = true;
        u.herm_lower = true;  // (the strict upper tiles are never read)
        gemm_c64(ctx, u);
    }
}

// A (m x n) <- L^{-1} A with L the lower factor in G (leading dimension m); tmp: NB x n.
void solve_lower_rows(Ctx& ctx, const double2* G, const double2* Linv_all, int m, int n, double2* A, double2* tmp) {
    for (int r0 = 0; r0 < m; r0 += NB) {
        const int b = std::min(NB, m - r0);
        double2* Ab = A + (size_t)r0 * n;
        if (r0 > 0) {
            GemmArgs g;  // A_b -= L[b, <b] Q[<b]
            g.M = b; g.N = n; g.K = r0;
            g.A = G + (size_t)r0 * m; g.lda = m;
            g.B = A; g.ldb = n;
            g.C = Ab; g.ldc = n;
            g.accumulate = true;
            g.negate = true;
            gemm_c64(ctx, g);
        }
        GemmArgs h;  // Q_b = L_bb^{-1} A_b
        h.M = b; h.N = n; h.K = b;
        h.A = Linv_all + (size_t)(r0 / NB) * NB * NB; h.lda = NB;
        h.B = Ab; h.ldb = n;
        h.C = tmp; h.ldc = n;
        gemm_c64(ctx, h);
        VTN_CUDA_TRY(cudaMemcpyAsync(Ab, tmp, sizeof(double2) * (size_t)b * n, cudaMemcpyDeviceToDevice, ctx.stream));
    }
}

// before the factorisation: the Gram matrix' diagonal, after shift * trace is added to it
__global__ void __launch_bounds__(1024) gram_diagonal(double2* __restrict__ G, int m, double shift, double* __restrict__ d) {
    __shared__ double sh[32];
    double tr = 0.0;
    if (shift > 0.0) {
        for (int j = threadIdx.x; j < m; j += 1024) tr += G[(long long)j * m + j].x;
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = tr;
        __syncthreads();
        tr = 0.0;
        for (int w = 0; w < 32; ++w) tr += sh[w];
    }
    for (int j = threadIdx.x; j < m; j += 1024) {
        const double g = G[(long long)j * m + j].x + shift * tr;
        if (shift > 0.0) G[(long long)j * m + j].x = g;
        d[j] = g;
    }
}

// after it: pivots of rows 0, k - 1 and m - 1, the smallest pivot relative to its row's norm, the flag
__global__ void __launch_bounds__(1024) pivot_info(const double2* __restrict__ G, int m, int k, const double* __restrict__ d,
                                                   const int* __restrict__ flag, double* __restrict__ info) {
    __shared__ double sh[32];
    double mn = 2.0;
    for (int j = threadIdx.x; j < m; j += 1024) {
        const double r = G[(long long)j * m + j].x / sqrt(d[j]);
        mn = r == r ? fmin(mn, r) : -1.0;
    }
    for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mn;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 32; ++w) mn = fmin(mn, sh[w]);
    info[0] = G[0].x;
    info[1] = G[(long long)(k - 1) * m + k - 1].x;
    info[2] = G[(long long)(m - 1) * m + m - 1].x;
    info[3] = mn;
    info[4] = *flag;
}

}  // namespace

void cholqr_pass(Ctx& ctx, double2* A, int m, int n, int k, double* info, double shift) {
    const int nblk = (m + NB - 1) / NB;
    double2* G = (double2*)ctx.workspace(WS_CQR_G, sizeof(double2) * ((size_t)m * m + (size_t)nblk * NB * NB + m));
    double2* Linv = G + (size_t)m * m;
    double* diag = (double*)(Linv + (size_t)nblk * NB * NB);
    int* flag = (int*)(diag + m);
    double2* tmp = (double2*)ctx.workspace(WS_CQR_T, sizeof(double2) * (size_t)NB * std::max(n, m));
    VTN_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(int), ctx.stream));
    GemmArgs g;
    g.M = m; g.N = m; g.K = n;
    g.A = A; g.lda = n;
    g.opB = OP_C; g.B = A; g.ldb = n;
    g.C = G; g.ldc = m;
    g.herm_lower = true;
    gemm_c64(ctx, g);
    gram_diagonal<<<1, 1024, 0, ctx.stream>>>(G, m, shift, diag);
    cholesky_blocked(ctx, G, m, Linv, tmp, flag);
    pivot_info<<<1, 1024, 0, ctx.stream>>>(G, m, k, diag, flag, info);
    ctx.count_launch(2);
    ctx.check_launch("cholqr_pass");
    solve_lower_rows(ctx, G, Linv, m, n, A, tmp);
}

void orthonormalize_rows_cholqr(Ctx& ctx, double2* A, int m, int n) {
    VTN_REQUIRE(m >= 1 && m <= n && m <= 4096, "row orthonormalisation needs 1 <= rows <= min(cols, 4096)");
    const int nblk = (m + NB - 1) / NB;
    double2* G = (double2*)ctx.workspace(WS_CQR_G, sizeof(double2) * ((size_t)m * m + (size_t)nblk * NB * NB));
    double2* Linv = G + (size_t)m * m;
    double2* tmp = (double2*)ctx.workspace(WS_CQR_T, sizeof(double2) * (size_t)NB * std::max(n, m));
    double2* backup = (double2*)ctx.workspace(WS_CQR_B, sizeof(double2) * (size_t)m * n + 256);
    int* flag = (int*)(backup + (size_t)m * n);
    VTN_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(int), ctx.stream));
    VTN_CUDA_TRY(cudaMemcpyAsync(backup, A, sizeof(double2) * (size_t)m * n, cudaMemcpyDeviceToDevice, ctx.stream));
    for (int pass = 0; pass < 2; ++pass) {
        GemmArgs g;  // G = A A^dag (tiles on and below the diagonal)
        g.M = m; g.N = m; g.K = n;
        g.A = A; g.lda = n;
        g.opB = OP_C; g.B = A; g.ldb = n;
        g.C = G; g.ldc = m;
        g.herm_lower = true;
        gemm_c64(ctx, g);
        if (pass == 1) {
            gram_identity_check<<<std::min(1024, (m * m + 255) / 256), 256, 0, ctx.stream>>>(G, m, 0.1, flag);
            ctx.count_launch();
        }
        cholesky_blocked(ctx, G, m, Linv, tmp, flag);
        solve_lower_rows(ctx, G, Linv, m, n, A, tmp);
    }
    const long long cnt = (long long)m * n;
    copy_if<<<(unsigned)std::min<long long>(4096, (cnt + 255) / 256), 256, 0, ctx.stream>>>(A, backup, cnt, flag);
    ctx.count_launch();
    ctx.check_launch("copy_if");
    orthonormalize_rows_small(ctx, A, m, n, flag);
}

}  // namespace vtn
