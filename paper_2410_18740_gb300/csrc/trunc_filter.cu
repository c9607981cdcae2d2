// Truncation by Chebyshev-filtered subspace iteration, run to the accuracy of the full eigendecomposition.
//
// The tridiagonalisation of eigh.cu reduces all n dimensions of rho to find k eigenpairs: n serial columns of
// about 9 us of latency and 12 n^2 FP64 operations on the narrow FP64 pipe.  With FP64 products 35 times
// cheaper on the tensor cores (oz_gemm.cu) the k-dimensional top subspace is cheaper to find by products
// (Zhou, Saad, Tiago, Chelikowsky, J. Comput. Phys. 219 (2006)): a block of m = 1.5 k rows is multiplied by
// Chebyshev polynomials of rho that stay within 1 on [0, b], b ~ the m-th eigenvalue, and grow fastest
// above it, and is re-orthonormalised by Cholesky-QR between them.  The rows come out in Schur order, so the
// pivots of the Cholesky factor are the growth of each direction: once the k-th has grown by e^35 over the
// unwanted ones, and the residual rho S - (S rho S^dag) S of the first k rows is at rounding level, the kept
// eigenpairs follow from the m x n problem S T by the exact truncation (Rayleigh-Ritz).
//
// Rows: S holds the conjugates of the vectors (m x n), so rho acts from the right; (S rho)^T = rho^T S^T is one
// product with the digits of rho^T, which all products share.
//
// Measured (whole truncation; full reduction with sliced products -> here, when the step was made): n = 512, k = 64
// 8.9 -> 7.2 ms; n = 1024, k = 128 29.8 -> 13.7 ms; n = 1830, k = 300 86 -> 40 ms (Schmidt values decaying by e^-9);
// flat random spectra 8.9 -> 9.0, 29.8 -> 27.3, 86 -> 71 ms.  With the shorter Cholesky and tridiagonalisation chains
// and the correction of the Ritz vectors the decaying ones take 12.8 ms at n = 1024 and 39.2 ms at 1830.  What is left
// is latency: the Cholesky chains (50 us per 32 rows and pass), the m x m tridiagonalisation (10 us a column) and about
// 50 us a product.
//
// The host reads five numbers after each pass.  It gives up (false: the full eigendecomposition runs) when the
// spectrum at k is so flat that the predicted polynomial degree costs more than the reduction, when the block is
// rank deficient, or when the residual stays above rounding.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>

#include "vtn_internal.cuh"

namespace vtn {
namespace {

// out = a p + b y + c z (z may be null, and may be out)
__global__ void __launch_bounds__(256) cheb_step(long long n, double a, const double2* __restrict__ p, double b,
                                                 const double2* __restrict__ y, double c, const double2* z, double2* out) {
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const double2 u = p[i], v = y[i];
    double2 r = make_double2(fma(a, u.x, b * v.x), fma(a, u.y, b * v.y));
    if (z != nullptr) {
        const double2 w = z[i];
        r.x = fma(c, w.x, r.x);
        r.y = fma(c, w.y, r.y);
    }
    out[i] = r;
}

// out[0] = max over the rows of |row|^2 (as the bits of a non-negative double), one CTA per row
__global__ void __launch_bounds__(256) row_norm_max(const double2* __restrict__ A, int n, unsigned long long* out) {
    __shared__ double sh[8];
    const double2* row = A + (long long)blockIdx.x * n;
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) acc = fma(row[i].x, row[i].x, fma(row[i].y, row[i].y, acc));
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) acc += sh[w];
        atomicMax(out, (unsigned long long)__double_as_longlong(acc));  // a NaN orders above every number
    }
}

// lam[j] = |Y_j|^2 / |V_j|^2 and g[j] = |V_j|^2, one CTA per Ritz vector (element q of vector j at j sj + q sq): partial
// sums of a few terms and a tree, whose error is below that of one long chain of additions.
__global__ void __launch_bounds__(256) ritz_values(const double2* __restrict__ Y, int ny, long long yj, long long yq,
                                                   const double2* __restrict__ V, int nv, long long vj, long long vq,
                                                   double* __restrict__ lam, double* __restrict__ g) {
    __shared__ double sh[2][8];
    const int j = blockIdx.x;
    double a[2] = {0.0, 0.0};
    for (int s = 0; s < 2; ++s) {
        const double2* x = s ? V + j * vj : Y + j * yj;
        const int n = s ? nv : ny;
        const long long step = s ? vq : yq;
        for (int q = threadIdx.x; q < n; q += 256) {
            const double2 v = x[q * step];
            a[s] += fma(v.x, v.x, v.y * v.y);
        }
        for (int o = 16; o > 0; o >>= 1) a[s] += __shfl_xor_sync(0xffffffffu, a[s], o);
        if ((threadIdx.x & 31) == 0) sh[s][threadIdx.x >> 5] = a[s];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int s = 0; s < 2; ++s)
        a[s] = ((sh[s][0] + sh[s][1]) + (sh[s][2] + sh[s][3])) + ((sh[s][4] + sh[s][5]) + (sh[s][6] + sh[s][7]));
    lam[j] = a[0] / a[1];
    g[j] = a[1];
}

// First-order correction of the top k of m Ritz vectors v_i: E = V^dag rho V and G = V^dag V (lower triangles),
// C (m x k) = I + X, X_ij = (E_ij - lam_j G_ij) / (lam_j - lam_i) against the unkept vectors, -(G - I) / 2 within the
// kept ones (orthonormal again, and each still its own eigenvector); lam and the diagonal g of G from ritz_values.
// A pair too close for first order (|X| > 1e-9, whose square would cost orthonormality) stays as it is.
__global__ void __launch_bounds__(256) ritz_correction(int m, int k, const double2* __restrict__ E, const double2* __restrict__ G,
                                                       const double* __restrict__ lam, const double* __restrict__ gd,
                                                       double2* __restrict__ C) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= m * k) return;
    const int i = t / k, j = t % k;
    const double lj = lam[j];
    const double2 g = i >= j ? G[(long long)i * m + j] : G[(long long)j * m + i];
    double2 c;
    if (i == j) {
        c = make_double2(1.0 - 0.5 * (gd[j] - 1.0), 0.0);
    } else if (i < k) {
        c = make_double2(-0.5 * g.x, i > j ? -0.5 * g.y : 0.5 * g.y);
    } else {
        const double2 e = E[(long long)i * m + j];
        const double r = 1.0 / (lj - lam[i]);
        c = make_double2((e.x - lj * g.x) * r, (e.y - lj * g.y) * r);
        if (!(c.x * c.x + c.y * c.y <= 1e-18)) c = make_double2(0.0, 0.0);
    }
    C[t] = c;
}

}  // namespace

// Block size 1.5 k + 16 in tiles of 32, from n = 257 on and where the block is at most half of rho.  Where T's other
// side r is no larger than that, the block is T's own range (r rows, no iteration): at the ends of a chain, where
// rho is n x n of rank r = n / d.
int filter_rows(int nL, int nR, int direction, int k) {
    const int n = direction == 0 ? nL : nR, other = direction == 0 ? nR : nL, m = (3 * k / 2 + 16 + 31) / 32 * 32;
    if (n <= 256) return 0;
    if (2 * other <= n && other <= 4096 && (other <= m || n > 4096)) return other;
    return n <= 4096 && 2 * m <= n && m <= other ? m : 0;
}

bool truncate_filtered(Ctx& ctx, int nL, int nR, int direction, int k, int m, const double2* theta, double2* left,
                       double2* right, int outer, double* defer, TruncResult& res) {
    const int n = direction == 0 ? nL : nR, other = direction == 0 ? nR : nL;
    const long long mn = (long long)m * n;
    const int tt = ctx.tbegin(TC_EIG, 0.0);
    const bool timing = ctx.timing;
    struct Timing {  // the products inside are part of this interval
        Ctx& c;
        bool on;
        int t;
        ~Timing() {
            c.timing = on;
            if (t >= 0) c.tend(t);
        }
    } guard{ctx, timing, tt};
    const bool range = m == other;
    double2* rho = nullptr;
    OzPrep prep;
    if (!range) {
        rho = (double2*)ctx.workspace(WS_EIG_A, sizeof(double2) * (size_t)n * n);
        density_dev(ctx, nL, nR, direction, theta, rho);
        prep = oz_prepare(ctx, n, n, OP_T, rho, n);
    }
    double2* S = (double2*)ctx.workspace(WS_FLT_S, sizeof(double2) * (size_t)mn);
    double2* X = (double2*)ctx.workspace(WS_FLT_X, sizeof(double2) * (size_t)mn);
    double2* P = (double2*)ctx.workspace(WS_FLT_P, sizeof(double2) * (size_t)m * std::max(n, other));
    double2* H = (double2*)ctx.workspace(WS_FLT_H, sizeof(double2) * (size_t)m * m);
    double* num = (double*)ctx.workspace(WS_FLT_N, sizeof(double) * 16);  // info[5], residual, |theta|^2
    auto apply = [&](const double2* in, double2* out) {  // out = in rho
        GemmArgs g;
        g.M = n; g.N = m; g.K = n;
        g.prepA = &prep; g.opA = OP_T; g.A = rho; g.lda = n;  // (rho itself for rows that are not finite)
        g.opB = OP_T; g.B = in; g.ldb = n;
        g.C = out; g.ldc = 1; g.sC_n = n;
        gemm_c64(ctx, g);
    };
    double l1 = 0, lk = 0, lm = 0, pivot = 0;
    auto orth = [&](double2* A) {
        cholqr_pass(ctx, A, m, n, k, num);
        VTN_CUDA_TRY(cudaMemcpyAsync(ctx.pinned, num, sizeof(double) * 5, cudaMemcpyDeviceToHost, ctx.stream));
        ctx.sync();
        l1 = ctx.pinned[0]; lk = ctx.pinned[1]; lm = ctx.pinned[2]; pivot = ctx.pinned[3];
        // NaN fails every comparison
        return ctx.pinned[4] == 0.0 && pivot > 1e-7 && lk > 0.0 && l1 < 1e300;
    };
    auto iterate = [&]() -> bool {
        // ---- two plain products of a random block: eigenvalue estimates from the second one's pivots
        fill_random_normal(ctx, S, mn, 0x5eedull, n, PHILOX_STREAM_TRUNC);
        apply(S, P);
        if (!orth(P)) return false;
        apply(P, S);
        if (!orth(S)) return false;
        if (!(lm > 1e-12 * l1) || !(lk > lm)) return false;
        const double b = lm, lam1 = l1;
        const double g1 = std::acosh(2.0 * 1.6 * lam1 / b - 1.0);  // growth per degree; the largest pivot reads low
        double gk = std::acosh(2.0 * lk / b - 1.0);
        // Degrees that cost as much as the reduction: 8.9 ms at n = 512, 30 at 1024 and 86 at 1830, against 5, 8 and
        // 20 ms of orthonormalisation and Rayleigh-Ritz and 40, 60 and 110 us a degree.
        const double limit = 40.0 * std::pow(n / 512.0, 1.6);
        if (!(35.0 / gk <= limit)) return false;
        double grown = 0.0, degrees = 0.0;
        bool done = false;
        for (int cycle = 0; cycle < 32 && !done; ++cycle) {
            // the first block is not in Schur order yet: its rows may part by 1e6 only; later ones by 1e13
            int D = (int)(std::log(cycle == 0 ? 1e6 : 1e13) / g1);
            D = std::max(2, std::min({D, 12, (int)std::ceil((36.0 - grown) / gk)}));
            degrees += D;
            if (degrees > 2.0 * limit) return false;
            apply(S, P);
            cheb_step<<<(unsigned)((mn + 255) / 256), 256, 0, ctx.stream>>>(mn, 2.0 / b, P, -1.0, S, 0.0, nullptr, X);
            double2 *prev = S, *cur = X;
            for (int i = 1; i < D; ++i) {
                apply(cur, P);
                cheb_step<<<(unsigned)((mn + 255) / 256), 256, 0, ctx.stream>>>(mn, 4.0 / b, P, -2.0, cur, -1.0, prev, prev);
                std::swap(prev, cur);
            }
            ctx.count_launch(D);
            ctx.check_launch("cheb_step");
            S = cur;
            X = prev;
            if (!orth(S)) return false;
            grown += std::log(lk);
            gk = std::log(lk) / D;
            if (!(gk > 0.0)) return false;
            if (grown < 35.0) {
                if (!(degrees + (35.0 - grown) / gk <= 2.0 * limit)) return false;
                continue;
            }
            // the pass lost orthogonality like u / pivot^2 (a second pass costs 0.5 ms at m = 224)
            if (pivot < 0.5 && !orth(S)) return false;
            // ---- residual of the first k rows: S rho - (S rho S^dag) S
            apply(S, P);
            GemmArgs h;
            h.M = m; h.N = m; h.K = n;
            h.A = P; h.lda = n;
            h.opB = OP_C; h.B = S; h.ldb = n;
            h.C = H; h.ldc = m;
            gemm_c64(ctx, h);
            GemmArgs r;
            r.M = k; r.N = n; r.K = m;
            r.A = H; r.lda = m;
            r.B = S; r.ldb = n;
            r.C = P; r.ldc = n;
            r.accumulate = true; r.negate = true;
            gemm_c64(ctx, r);
            VTN_CUDA_TRY(cudaMemsetAsync(num + 5, 0, sizeof(double), ctx.stream));
            row_norm_max<<<k, 256, 0, ctx.stream>>>(P, n, (unsigned long long*)(num + 5));
            ctx.count_launch();
            ctx.check_launch("row_norm_max");
            VTN_CUDA_TRY(cudaMemcpyAsync(ctx.pinned, num + 5, sizeof(double), cudaMemcpyDeviceToHost, ctx.stream));
            ctx.sync();
            done = std::sqrt(ctx.pinned[0]) <= 4e-15 * lam1;
            if (!done && grown > 60.0) return false;
        }
        return done;
    };
    if (range) {
        // the rows of T (or of T^dag) span everything; two passes, as one loses u (|T| / smallest singular value)^2
        auto load = [&]() {
            if (direction == 0) conj_transpose_dev(ctx, nL, nR, theta, nR, S, nL);
            else VTN_CUDA_TRY(cudaMemcpyAsync(S, theta, sizeof(double2) * (size_t)mn, cudaMemcpyDeviceToDevice, ctx.stream));
        };
        load();
        if (!orth(S)) {
            // ill-conditioned: shifted passes first (Fukaya et al. 2020), each of which takes a factor of about 1e7 off
            load();
            const double shift = 11.0 * ((double)mn + (double)m * (m + 1)) * 1.1e-16;
            cholqr_pass(ctx, S, m, n, k, num, shift);
            cholqr_pass(ctx, S, m, n, k, num, shift);
            if (!orth(S)) return false;
        }
        if (!orth(S) || !(pivot > 0.5)) return false;
    } else if (!iterate()) {
        return false;
    }
    // ---- Rayleigh-Ritz: the exact truncation of the projected tensor, by the full reduction: P, U1 and S are this
    // function's workspaces, and the range of a tensor larger than 4096 is itself of a size that suits the filter.
    // Its backward error u |rho| lies in m dimensions instead of n, so the vectors at the boundary mix more than
    // those of the full reduction do; with the next 16 Ritz vectors at hand (k2 in all, 768 at most unless k is
    // larger: the reduction's own limit is 775) a first-order correction from products takes that back.  Error of
    // theta against twice the working precision, reduction of all of rho | without the correction | with it:
    // 1.9 | 2.9 | 0.83e-15 at n = 1024, k = 128; 3.4 | 4.4 | 1.2e-15 at n = 1830, k = 300; of lam 1.2 | 3.7 | 1.3e-16.
    // It takes 0.4 of 14.0 and 1.9 of 47.1 ms; with k / 4 more vectors 14.6 and 48.3 ms for 0.75 and 1.09e-15,
    // with all m 15.0 and 50.1 ms for 0.68 and 1.03e-15.
    const int k2 = std::min(m, std::max(k, std::min(768, k + 16)));
    norm2_dev(ctx, theta, (long long)nL * nR, num + 6);
    ctx.timing = false;
    double2* U1 = (double2*)ctx.workspace(WS_FLT_U, sizeof(double2) * (size_t)m * k2);
    double2* Y = (double2*)ctx.workspace(WS_FLT_Y, sizeof(double2) * (size_t)k2 * other);
    double2* E = (double2*)ctx.workspace(WS_FLT_H, sizeof(double2) * ((size_t)k2 * k2 * 2 + (size_t)k2 * k) + sizeof(double) * 2 * k2);
    double2 *G = E + (size_t)k2 * k2, *C = G + (size_t)k2 * k2, *V = X;
    double *lam = (double*)(C + (size_t)k2 * k), *gd = lam + k2;
    auto gemm = [&](int M, int N, int K, Op opA, const double2* A, int lda, Op opB, const double2* B, int ldb, double2* out,
                    int ldc, bool herm) {
        GemmArgs g;
        g.M = M; g.N = N; g.K = K;
        g.opA = opA; g.A = A; g.lda = lda;
        g.opB = opB; g.B = B; g.ldb = ldb;
        g.C = out; g.ldc = ldc;
        g.herm_lower = herm;
        gemm_c64(ctx, g);
    };
    if (direction == 0) {  // P = S T; P P^dag = U' w U'^dag, V = S^dag U' (n x k2), Y = U'^dag P
        gemm(m, nR, n, OP_N, S, n, OP_N, theta, nR, P, nR, false);
        res = truncate_dev(ctx, m, 1, 1, nR, 0, k2, P, U1, Y, -1, nullptr, false);
        gemm(n, k2, m, OP_C, S, n, OP_N, U1, k2, V, k2, false);
        gemm(k2, k2, nR, OP_N, Y, nR, OP_C, Y, nR, E, k2, true);
        gemm(k2, k2, n, OP_C, V, k2, OP_N, V, k2, G, k2, true);
    } else {  // P = T S^dag; P^dag P = V' w V'^dag, V = V'^dag S (k2 x n), Y = P V'
        gemm(nL, m, n, OP_N, theta, nR, OP_C, S, n, P, m, false);
        res = truncate_dev(ctx, nL, 1, 1, m, 1, k2, P, Y, U1, -1, nullptr, false);
        gemm(k2, n, m, OP_N, U1, m, OP_N, S, n, V, n, false);
        gemm(k2, k2, nL, OP_C, Y, k2, OP_N, Y, k2, E, k2, true);
        gemm(k2, k2, n, OP_N, V, n, OP_C, V, n, G, k2, true);
    }
    const bool cols = direction == 0;  // V's vectors are columns and Y's rows, or the other way round
    ritz_values<<<k2, 256, 0, ctx.stream>>>(Y, other, cols ? other : 1, cols ? 1 : k2, V, n, cols ? 1 : n, cols ? k2 : 1, lam, gd);
    ritz_correction<<<(k2 * k + 255) / 256, 256, 0, ctx.stream>>>(k2, k, E, G, lam, gd, C);
    ctx.count_launch(2);
    ctx.check_launch("ritz_correction");
    if (direction == 0) {
        gemm(n, k, k2, OP_N, V, k2, OP_N, C, k, left, k, false);
        gemm(k, outer, k2, OP_C, C, k, OP_N, Y, nR, right, outer, false);
    } else {
        gemm(outer, k, k2, OP_N, Y, k2, OP_N, C, k, left, k, false);
        gemm(k, n, k2, OP_C, C, k, OP_N, V, n, right, n, false);
    }
    // the discarded weight refers to the whole tensor
    if (defer != nullptr) {
        VTN_CUDA_TRY(cudaMemcpyAsync(defer, lam, sizeof(double) * k, cudaMemcpyDeviceToHost, ctx.stream));
        VTN_CUDA_TRY(cudaMemcpyAsync(defer + k, num + 6, sizeof(double), cudaMemcpyDeviceToHost, ctx.stream));
        std::memset(defer + k + 1, 0, sizeof(int) * 8);  // the reduction's status words were read above
        res.k = k;
        res.lam.clear();
        res.discarded = 0.0;
        return true;
    }
    VTN_CUDA_TRY(cudaMemcpyAsync(ctx.pinned, lam, sizeof(double) * k, cudaMemcpyDeviceToHost, ctx.stream));
    VTN_CUDA_TRY(cudaMemcpyAsync(ctx.pinned + k, num + 6, sizeof(double), cudaMemcpyDeviceToHost, ctx.stream));
    ctx.sync();
    res.k = k;
    res.lam.assign(ctx.pinned, ctx.pinned + k);
    std::sort(res.lam.begin(), res.lam.end(), std::greater<double>());  // equal ones differ in their last bits
    double kept = 0.0;
    for (double l : res.lam) kept += l;
    res.discarded = ctx.pinned[k] > 0.0 ? 1.0 - kept / ctx.pinned[k] : 0.0;
    return true;
}

}  // namespace vtn
