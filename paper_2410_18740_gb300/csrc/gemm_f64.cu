// Complex FP64 GEMM for the FP64 solver path:
//   C[batch] (=|+=) sum_{kb} op(A[batch, kb]) op(B[batch, kb]),  op in {X, X^dag}.
// Every contraction of the two-site effective Hamiltonian, the environment updates and
// the reduced density matrix is one call.
//
// Large products go to the tensor cores by exact integer slices (oz_gemm.cu).  The kernel here is for
// the small ones and for callers that cannot use a workspace: SIMT DFMA, of which GB300 issues one warp
// instruction per 64 cycles and SM sub-partition, so a call is bound by the number of SMs that work.
// Hence tiles of 16 x 16 outputs, one per thread of a 256-thread CTA (a 64 x 64 tile takes an SM 40 us per 8
// terms whatever part of it is used: the 454 products of a 4-mode chi = 16 solve took 103 us each, 5 us with
// these), and a summation that is split over CTAs while there are fewer than two per SM; the partial
// sums are added in a fixed order by a second kernel (deterministic).
#include <algorithm>

#include "vtn_internal.cuh"

namespace vtn {
namespace {

constexpr int BT = 16, BK = 16, NT = 256;  // output tile edge, summation step, threads

struct GemmP {
    int M, N, K, kb;
    int opA, opB;
    const double2* A; long long lda, sA_batch, sA_kb;
    const double2* B; long long ldb, sB_batch, sB_kb;
    double2* C; long long ldc, sC_batch;
    int accumulate;
    int herm_lower;
    int negate;
    int batch;
    int splits;          // S: CTAs per output tile along the summation range
    double2* part;       // S > 1: partial tiles [S][batch][M][N]
};

__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }

__global__ void __launch_bounds__(NT) gemm_c64_kernel(GemmP p) {
    __shared__ double2 As[BK][BT + 1];
    __shared__ double2 Bs[BK][BT + 1];
    const int tid = threadIdx.x;
    const int tx = tid % BT, ty = tid / BT;
    const int gx = (p.N + BT - 1) / BT, gy = (p.M + BT - 1) / BT;
    long long id = blockIdx.x;
    const int n0 = (int)(id % gx) * BT;
    id /= gx;
    const int m0 = (int)(id % gy) * BT;
    id /= gy;
    const int split = (int)(id % p.splits);
    const long long bz = id / p.splits;
    if (p.herm_lower && n0 > m0) return;  // tile strictly above the diagonal
    double2 acc = make_double2(0.0, 0.0);

    // this CTA's share [t0, t1) of the kb * ceil(K / BK) steps of the summation
    const int nk = (p.K + BK - 1) / BK;
    const long long T = (long long)nk * p.kb;
    const long long t0 = T * split / p.splits, t1 = T * (split + 1) / p.splits;
    int kb = (int)(t0 / nk), k0 = (int)(t0 % nk) * BK;
    // the staged element of each thread: along the contiguous index of its operand
    const int am = p.opA == OP_N ? ty : tx, ak = p.opA == OP_N ? tx : ty;
    const int bn = p.opB == OP_N ? tx : ty, bk = p.opB == OP_N ? ty : tx;
    auto load = [&](double2& a, double2& b) {
        const double2* A = p.A + bz * p.sA_batch + (long long)kb * p.sA_kb;
        const double2* B = p.B + bz * p.sB_batch + (long long)kb * p.sB_kb;
        const int m = m0 + am, n = n0 + bn, ka = k0 + ak, kk = k0 + bk;
        a = b = make_double2(0.0, 0.0);
        if (m < p.M && ka < p.K)
            a = p.opA == OP_N ? A[(long long)m * p.lda + ka] : cconj(A[(long long)ka * p.lda + m]);
        if (n < p.N && kk < p.K)
            b = p.opB == OP_N ? B[(long long)kk * p.ldb + n] : cconj(B[(long long)n * p.ldb + kk]);
    };
    double2 ra, rb;
    if (t0 < t1) load(ra, rb);
    for (long long t = t0; t < t1; ++t) {
        As[ak][am] = ra;
        Bs[bk][bn] = rb;
        __syncthreads();
        const int ke = min(BK, p.K - k0);
        k0 += BK;
        if (k0 >= p.K) { k0 = 0; ++kb; }
        if (t + 1 < t1) load(ra, rb);  // the next step's elements, in flight during this one
        for (int kk = 0; kk < ke; ++kk) {
            const double2 a = As[kk][ty], b = Bs[kk][tx];
            acc.x = fma(a.x, b.x, acc.x);
            acc.x = fma(-a.y, b.y, acc.x);
            acc.y = fma(a.x, b.y, acc.y);
            acc.y = fma(a.y, b.x, acc.y);
        }
        __syncthreads();
    }
    if (p.negate) acc = make_double2(-acc.x, -acc.y);
    const int m = m0 + ty, n = n0 + tx;
    if (m >= p.M || n >= p.N) return;
    if (p.splits > 1) {
        p.part[(((long long)split * p.batch + bz) * p.M + m) * p.N + n] = acc;
        return;
    }
    double2* c = p.C + bz * p.sC_batch + (long long)m * p.ldc + n;
    if (p.accumulate) {
        const double2 o = *c;
        acc.x += o.x;
        acc.y += o.y;
    }
    *c = acc;
}

// C[b][m][n] (=|+=) sum_{s < S} part[s][b][m][n], s ascending
__global__ void splitk_sum(GemmP p, int batch) {
    const long long mn = (long long)p.M * p.N;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= mn * batch) return;
    const long long b = t / mn, e = t % mn;
    const int m = (int)(e / p.N), n = (int)(e % p.N);
    if (p.herm_lower && n / BT > m / BT) return;
    double2 acc = p.part[t];
    for (int s = 1; s < p.splits; ++s) {
        const double2 v = p.part[(long long)s * mn * batch + t];
        acc.x += v.x;
        acc.y += v.y;
    }
    double2* c = p.C + b * p.sC_batch + (long long)m * p.ldc + n;
    if (p.accumulate) {
        const double2 o = *c;
        acc.x += o.x;
        acc.y += o.y;
    }
    *c = acc;
}

__global__ void mirror_kernel(double2* C, int n, long long ldc) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)n * n) return;
    const int i = (int)(t / n), j = (int)(t % n);
    if (j <= i) return;
    const double2 v = C[(long long)j * ldc + i];
    C[(long long)i * ldc + j] = make_double2(v.x, -v.y);
}

}  // namespace

void mirror_lower_to_upper(Ctx& ctx, double2* C, int n, long long ldc) {
    const long long cnt = (long long)n * n;
    if (cnt == 0) return;
    mirror_kernel<<<(unsigned)((cnt + 255) / 256), 256, 0, ctx.stream>>>(C, n, ldc);
    ctx.count_launch();
    ctx.check_launch("mirror_kernel");
}

void gemm_c64(Ctx& ctx, const GemmArgs& g, int timing_class) {
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return;
    VTN_REQUIRE(g.batch <= 65535, "gemm batch too large");
    GemmP p;
    p.M = g.M; p.N = g.N; p.K = g.K; p.kb = g.kb;
    p.opA = g.opA; p.opB = g.opB;
    p.A = g.A; p.lda = g.lda; p.sA_batch = g.sA_batch; p.sA_kb = g.sA_kb;
    p.B = g.B; p.ldb = g.ldb; p.sB_batch = g.sB_batch; p.sB_kb = g.sB_kb;
    p.C = g.C; p.ldc = g.ldc; p.sC_batch = g.sC_batch;
    p.accumulate = g.accumulate ? 1 : 0;
    p.herm_lower = g.herm_lower ? 1 : 0;
    p.negate = g.negate ? 1 : 0;
    VTN_REQUIRE(g.sC_n == 1 || (g.prepA != nullptr && g.ldc == 1 && !g.herm_lower), "column strides need a prepared operand");
    VTN_REQUIRE(!g.herm_lower || g.M == g.N, "Hermitian GEMM needs a square C");
    p.batch = g.batch;
    const long long gx = (g.N + BT - 1) / BT, gy = (g.M + BT - 1) / BT;
    VTN_REQUIRE(gy <= 4 * 65535LL, "gemm M too large");
    const double macs = (double)g.M * g.N * g.K * g.kb * g.batch * (g.herm_lower ? 0.5 : 1.0);
    // The sliced product costs four launches, about 48 us back to back, and then runs 35 times faster; the FP64 units
    // take a wave of 16 x 16 tiles after the other.  Measured, FP64 units | sliced: 128 x 128 x 256 (4.2e6) 43 | 48 us,
    // 160 x 128 x 256 (5.2e6) 76 | 48 us, 160 x 160 x 256 76 | 48 us; at 3072^3 200 ms against 6.2 ms.  The line counts what is
    // asked for, not the padding, which is the wrong way round at the worst by 1.5: 8 columns (padded to 16 and 32)
    // 2048 x 8 x 256 (4.2e6) 76 | 50 us, rows that fill an eighth of a tile 24 x 16 x 16 x 4096 (2.5e7) 195 | 281 us.
    // Its row sums fit 96-bit integers for summations of up to 2^19 terms.
    bool oz = g.prepA != nullptr || ctx.dstatus != nullptr && g.max_splits != 1 && macs >= 5.2e6 && (long long)g.K * g.kb <= (1LL << 19);
    int S = 1;
    if (oz) {
        S = oz_splits(ctx, g);
    } else {
        // output tiles that do work; split the summation when they leave SMs short of 2 CTAs
        const long long tiles = (g.herm_lower ? gy * (gy + 1) / 2 : gx * gy) * g.batch;
        // (a share of fewer than 128 terms costs more in the second pass than it saves)
        const long long slots = 2LL * std::max(ctx.num_sms, 1);
        if (tiles < slots) S = (int)std::min<long long>({slots / tiles, (long long)g.K * g.kb / 128, 32LL});
    }
    if (g.max_splits > 0) S = std::min(S, g.max_splits);
    S = std::max(S, 1);
    p.part = nullptr;
    if (S > 1) {
        try {
            p.part = (double2*)ctx.workspace(WS_GEMM_SPLIT, sizeof(double2) * (size_t)S * g.batch * g.M * g.N);
        } catch (const Error& e) {  // no memory for the sliced product's partial sums: the FP64 kernel, unsplit
            if (e.status != VTN_ENOMEM || !oz || g.prepA != nullptr) throw;
            oz = false;
            S = 1;
        }
    }
    p.splits = S;
    const long long ctas = gx * gy * g.batch * S;
    double flops = 8.0 * g.M * (double)g.N * g.K * g.kb * g.batch * (g.herm_lower ? 0.5 : 1.0);
    int t0 = ctx.tbegin(TC_GEMM, flops);
    int t1 = (timing_class != TC_GEMM) ? ctx.tbegin(timing_class, flops) : -1;
    if (!oz || !oz_gemm(ctx, g, S, p.part)) {
        if (g.prepA != nullptr) throw Error{VTN_ENOMEM, "no device memory for the digits of a prepared product"};
        VTN_REQUIRE(ctas < (1LL << 31), "gemm too large");
        gemm_c64_kernel<<<(unsigned)ctas, NT, 0, ctx.stream>>>(p);
        ctx.count_launch();
        ctx.check_launch("gemm_c64_kernel");
    }
    if (S > 1) {
        const long long cnt = (long long)g.batch * g.M * g.N;
        if (g.sC_n != 1) {  // C and the partials are stored column by column
            std::swap(p.M, p.N);
            p.ldc = g.sC_n;
        }
        splitk_sum<<<(unsigned)((cnt + 255) / 256), 256, 0, ctx.stream>>>(p, g.batch);
        ctx.count_launch();
        ctx.check_launch("splitk_sum");
    }
    ctx.tend(t1);
    ctx.tend(t0);
}

}  // namespace vtn
