// Complex FP64 GEMM on the tensor cores by error-free slicing (the splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012), with integer slices):
//   C[batch] (=|+=) (-) sum_kb op(A[batch, kb]) op(B[batch, kb]),   the contract of gemm_c64.
//
// GB300 issues about 1.2 TFLOP/s of FP64 multiply-adds and 1.9 PFLOP/s of bf16 ones, so a product of
// 64-bit fixed-point numbers is cheaper on the tensor cores than one DFMA per term:
//   * each row of A (column of B) is written as fixed point relative to its largest exponent, 63 bits
//     and a sign, cut into eight signed 8-bit digits (|digit| <= 128, exact in bf16);
//   * digit i of A times digit j of B contributes at weight 256^-(i+j).  The 36 pairs with i + j <= 7
//     are multiplied.  The 28 others (at most 1.76 2^-60 a real product) and the cut of both operands
//     to 63 bits (2^-60) leave out less than 6 2^-60 of (largest of the row) x (largest of the column)
//     a complex term;
//   * products of one weight s = i + j are summed in one FP32 tensor-memory accumulator while every
//     partial sum is an integer of at most 2^24 (128 products-of-pairs deep: exact), then drained into
//     64-bit integers.  The only roundings are the final conversion to double (of each part of a split
//     summation) and that of C += : one rounding of the sum where a DFMA chain has one per term.
// So the accuracy is relative to the largest entries of the row and the column (of the scaled operands: k_shift), not
// to the terms themselves: in [[1, e], [1, 1]] [[0, 1], [1, 1]] the e of the first output has a relative error of
// up to 2^-56 / e, where a DFMA chain gives it exactly.
// Complex products take the real 2 x 2 block form of the split-precision mode (A~ rows (re, im), B~ rows
// (re, -im) and (im, re)), so a real GEMM yields interleaved outputs.
//
// Three launches: the rows' largest exponents, the digits, the product.  The digit kernel writes the
// operands as ready-made shared-memory tiles (128 rows of A~ or 64 of B~, 32 columns, all eight slices;
// no-swizzle K-major core matrices), so a stage is two plain bulk copies with no tensor map.
//
// A row or column that holds an infinity or NaN is left out of the digits; its outputs are summed
// term by term in FP64 in the epilogue, with the results the FP64 kernel gives (sparse_b: zeros of B are no terms).
#include <algorithm>

#include "tc_ptx.cuh"
#include "vtn_internal.cuh"

namespace vtn {
namespace {

constexpr int SL = 8;                        // digits per number
constexpr int TM = 128, TN = 64, KB = 32;    // A~ rows, B~ rows (32 complex columns), real columns per stage
constexpr int TNC = TN / 2, KBC = KB / 2;    // the same in complex elements
constexpr int A_BYTES = SL * TM * KB * 2;    // 64 KiB
constexpr int B_BYTES = SL * TN * KB * 2;    // 32 KiB
constexpr int STAGE = A_BYTES + B_BYTES;
constexpr int NST = 2;
constexpr int A_SLICE = TM * KB * 2, B_SLICE = TN * KB * 2;
constexpr int NP = SL / 2;                   // accumulators are issued and drained in pairs of weights
constexpr int THREADS = 384;                 // warp 0 copies, warp 1 MMA + tensor memory, warps 4-11 drain
// registers per thread at launch (384 threads) and after the split: 128 * 40 + 256 * 224 <= 384 * 168
constexpr int REGS_ISSUE = 40, REGS_DRAIN = 224;
constexpr size_t SMEM = 1024 + (size_t)NST * STAGE + 256;

// Weight pair q holds weights 7 - 2q and 6 - 2q (q = 0 is issued first).  A weight w sums w + 1 digit pairs of at
// most 2^14 per column, so an accumulator stays within 2^24 for 1024 / (w + 1) columns: the pairs are drained
// every 4, 4, 8 and 16 stages of 32 columns, at different stages so that one drain overlaps the products of
// the other pairs; all of them after an item's last stage.  An item of at most eight stages is bound by its drains, so it
// has as few as are exact: weights 7 and 6 after four stages, 5 and 4 after five, the others at the end (eight
// stages of L theta at chi 128, d 8: six drains instead of eight; the three products of that H_eff
// application 766 -> 732 us each).
__device__ __forceinline__ bool drain_due(int q, int k, int nk) {
    if (k == nk - 1) return true;
    if (nk <= 8) return q == 0 ? k == 3 : q == 1 && k == 4;
    return q == 0 ? (k & 3) == 3 : q == 1 ? (k & 3) == 1 : q == 2 ? (k & 7) == 6 : (k & 15) == 8;
}

struct OzOperand {
    const double2* X;
    long long ld, s_batch, s_kb;
    int rows;        // rows of op(A) or columns of op(B)
    int nb;          // independent batches (1 when all share it)
    int kc;          // the summation index is the contiguous one
    int conj;
    int K, kbn;      // summation range: kbn blocks of K
    int tiles;       // row tiles per batch
    int* bx;         // [nb][tiles * tile rows] largest exponent of a row (offset EXP0; 0 = zero row; NONFINITE)
    int* kx;         // [kbn * K] largest biased exponent of the finite entries of a column of op(A) or row of op(B)
    uint4* out;      // tiles
};

struct OzParams {
    OzOperand a, b;
    int M, N, nkb;
    int tiles_m, tiles_n, batch, splits, kb_per;
    double2* C;
    long long ldc, sC_n, sC_batch;
    double2* part;
    long long part_m, part_n, part_batch, part_split;  // strides of the partials
    int accumulate, negate, herm_lower, sparse_b;
    int* status;
};

__device__ __forceinline__ double2 oz_load(const OzOperand& o, long long base, int row, int kb, int k) {
    const double2* p = o.X + base + (long long)kb * o.s_kb;
    double2 v = o.kc ? p[(long long)row * o.ld + k] : p[(long long)k * o.ld + row];
    if (o.conj) v.y = -v.y;
    return v;
}

__device__ __forceinline__ int biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

constexpr int EXP0 = 8192;           // stored row exponent = biased exponent (with its shift) + EXP0
constexpr int NONFINITE = 1 << 20;
// Binades that the row-times-column scaling may cost against the largest term of the sum before the summation
// index is scaled too: what is left out of a term then stays below 2^-51 of that largest one (mantissas add up to two
// binades), and typically 2^-56
constexpr int LOSS_BITS = 4;

struct OzShift {
    int on;          // the summation index is scaled
    unsigned done;   // blocks of the exponent kernel that have finished
    int pad[2];
};

// Power-of-two scaling of summation index k: A's column by 2^-shift, B's row by 2^+shift, so that both have
// the same largest exponent.  It cancels in the product and costs an addition per exponent.  An index that is
// zero in one operand adds nothing, so the other operand's entries go below all digits, and no row's or column's largest
// exponent is theirs.
constexpr int DEAD = 4096;
__device__ __forceinline__ int k_shift(const OzShift* sh, const int* kxa, const int* kxb, int kk) {
    if (!sh->on) return 0;
    const int x = kxa[kk], y = kxb[kk];
    if (x == 0 || y == 0) return x == y ? 0 : x == 0 ? -DEAD : DEAD;
    return (x - y) / 2;
}

constexpr int MAX_KS = 64;

// Largest exponent of each row: tiles of 32 rows x 64 summation indices, 8 warps (eight independent loads a
// thread: one memory latency), `reps` tiles of the same indices one after the other per block: as many as make
// the grid about eight blocks an SM, so that a large operand's blocks do not queue for the same 64 index
// maxima and the one counter.  PASS 0 takes the
// unscaled rows and the exponents kx of the summation indices; its last block decides whether the summation
// index needs scaling (OzShift::on) and clears the row exponents if it does.  PASS 1 then takes the
// scaled rows (and returns at once where no scaling is needed).
// Bound by its loads: comparisons of doubles cost more than a load on the FP64 pipe, and loads that wait behind
// an atomic come two at a time.  Without both, mean of the three products of an H_eff application at chi 256, d 4:
// 132 -> 71 us; of the products of a readout at chi 96 (mostly latency): 10.4 -> 6.2 us.
template <int PASS>
__global__ void __launch_bounds__(256) oz_max_kernel(OzOperand a, OzOperand b, OzShift* shift, int nblk_a, int kseg,
                                                     int reps, int n_bx) {
    if (PASS == 1 && !shift->on) return;
    const bool is_b = (int)blockIdx.x >= nblk_a;
    const OzOperand& o = is_b ? b : a;
    const int id = is_b ? (int)blockIdx.x - nblk_a : (int)blockIdx.x;
    const int rb = (o.rows + 31) / 32, rg = (rb + reps - 1) / reps;
    const int seg = id % kseg, rt0 = (id / kseg) % rg * reps, rt1 = min(rb, rt0 + reps), bt = id / (kseg * rg);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Kt = o.K * o.kbn;
    const int k0 = seg * MAX_KS, k1 = min(Kt, k0 + MAX_KS);
    const long long base = (long long)bt * o.s_batch;
    int* bx = o.bx + (long long)bt * o.tiles * (is_b ? TNC : TM);
    __shared__ int kmax[MAX_KS];
    __shared__ int sh[2][8][32];
    if (PASS == 0) {
        if (threadIdx.x < MAX_KS) kmax[threadIdx.x] = 0;
        __syncthreads();
    }
    auto load = [&](int row, int kk) {
        if (row >= o.rows || kk >= k1) return make_double2(0.0, 0.0);
        const int kb = o.kbn > 1 ? kk / o.K : 0;
        const double2* p = o.X + base + kb * o.s_kb;
        const long long k = kk - kb * o.K;
        return __ldg(o.kc ? p + row * o.ld + k : p + k * o.ld + row);
    };
    auto exp_of = [&](double2 v, int kk, int& raw) {
        raw = max(biased_exp(v.x), biased_exp(v.y));
        if (raw == 0x7ff) {  // flags its row; the other rows' scaling of the index is that without it
            raw = 0;
            return NONFINITE;
        }
        // by bits: two comparisons of doubles an element are longer than its load on the narrow FP64 pipe
        if (raw == 0 && ((unsigned)(__double2hiint(v.x) | __double2hiint(v.y)) << 1 | (unsigned)__double2loint(v.x) |
                         (unsigned)__double2loint(v.y)) == 0u) return 0;
        int e = max(raw, 1);
        if (PASS == 1) {
            const int sk = k_shift(shift, a.kx, b.kx, kk);
            e += is_b ? sk : -sk;
        }
        return e + EXP0;
    };
    // (all loads of a tile before the first maximum: none moves up over an atomic)
    constexpr int NL = MAX_KS / 8;
    if (o.kc) {
        // a warp per four rows, its lanes along the summation index
        int km[2] = {0, 0};
        for (int rt = rt0; rt < rt1; ++rt) {
            const int row = rt * 32 + warp * 4;
            double2 v[NL];
#pragma unroll
            for (int j = 0; j < NL; ++j) v[j] = load(row + j / 2, k0 + (j & 1) * 32 + lane);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                int raw0, raw1;
                int m = max(exp_of(v[2 * r], k0 + lane, raw0), exp_of(v[2 * r + 1], k0 + 32 + lane, raw1));
                km[0] = max(km[0], raw0);
                km[1] = max(km[1], raw1);
                m = __reduce_max_sync(0xffffffffu, m);
                if (lane == 0 && row + r < o.rows) atomicMax(&bx[row + r], m);
            }
        }
        if (PASS == 0) {
            atomicMax(&kmax[lane], km[0]);
            atomicMax(&kmax[32 + lane], km[1]);
        }
    } else {
        int km[NL];
#pragma unroll
        for (int j = 0; j < NL; ++j) km[j] = 0;
        for (int rt = rt0; rt < rt1; ++rt) {
            const int row = rt * 32 + lane;
            double2 v[NL];
#pragma unroll
            for (int j = 0; j < NL; ++j) v[j] = load(row, k0 + warp * NL + j);
            int m = 0;
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                int raw;
                m = max(m, exp_of(v[j], k0 + warp * NL + j, raw));
                km[j] = max(km[j], raw);
            }
            // two buffers: a warp is at most one tile ahead of the one that reads
            int(*part)[32] = sh[rt & 1];
            part[warp][lane] = m;
            __syncthreads();
            if (warp == (rt & 7) && row < o.rows) {
#pragma unroll
                for (int w = 0; w < 8; ++w) m = max(m, part[w][lane]);
                atomicMax(&bx[row], m);
            }
        }
        if (PASS == 0)
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                const int kk = warp * NL + j, raw = __reduce_max_sync(0xffffffffu, km[j]);
                if (lane == 0) kmax[kk] = raw;  // this warp alone has index kk in this block
            }
    }
    if (PASS == 1 || n_bx < 0) return;  // a prepared operand leaves no choice
    __syncthreads();
    if ((int)threadIdx.x < k1 - k0) atomicMax(&o.kx[k0 + threadIdx.x], kmax[threadIdx.x]);
    // the last block compares the largest term with (largest of A) x (largest of B)
    __shared__ bool last_sh;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last_sh = atomicAdd(&shift->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last_sh) return;
    __threadfence();
    int ma = 0, mb = 0, mt = 0;
    for (int kk0 = threadIdx.x; kk0 < Kt; kk0 += 8 * 256) {
        int x[8], y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int kk = kk0 + j * 256;
            x[j] = kk < Kt ? __ldcg(&a.kx[kk]) : 0;
            y[j] = kk < Kt ? __ldcg(&b.kx[kk]) : 0;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            ma = max(ma, x[j]);
            mb = max(mb, y[j]);
            if (x[j] > 0 && y[j] > 0) mt = max(mt, x[j] + y[j]);
        }
    }
    ma = __reduce_max_sync(0xffffffffu, ma);
    mb = __reduce_max_sync(0xffffffffu, mb);
    mt = __reduce_max_sync(0xffffffffu, mt);
    if (lane == 0) {
        sh[0][0][warp] = ma;
        sh[0][1][warp] = mb;
        sh[0][2][warp] = mt;
    }
    __syncthreads();
    for (int w = 0; w < 8; ++w) {
        ma = max(ma, sh[0][0][w]);
        mb = max(mb, sh[0][1][w]);
        mt = max(mt, sh[0][2][w]);
    }
    if (mt > 0 && ma + mb - mt > LOSS_BITS) {
        for (int i = threadIdx.x; i < n_bx; i += 256) a.bx[i] = 0;  // bx of A and B are contiguous
        if (threadIdx.x == 0) shift->on = 1;
    }
}

// 63-bit fixed point of x 2^-shift relative to the row's largest exponent e0
__device__ __forceinline__ long long fixed_point(double x, int e0, int shift) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    int e = (int)(bits >> 52) & 0x7ff;
    unsigned long long m = bits & 0xfffffffffffffull;
    if (e) m |= 1ull << 52;
    else e = 1;
    const int sh = e0 - (e - shift);
    m = (unsigned)sh < 64u ? (m << 10) >> sh : 0ull;
    return (bits >> 63) ? -(long long)m : (long long)m;
}

constexpr long long DIGIT_BIAS = 0x0080808080808080ll;

// digit i (0 = leading): the bytes of q + bias are the digits + 128; the leading one is signed, carries no
// bias and may be +128
__device__ __forceinline__ float digit(long long q, int i) {
    if (i == 0) return (float)(int)(((q >> 1) + (DIGIT_BIAS >> 1)) >> 55);
    const unsigned b = (unsigned)((unsigned long long)(q + DIGIT_BIAS) >> (8 * (7 - i))) & 0xffu;
    return __uint_as_float(0x4B000000u | b) - 8388736.0f;  // 2^23 + b - (2^23 + 128)
}

// bf16 pair (lo, hi halves) of two floats that are exact in bf16
__device__ __forceinline__ unsigned pack2(float lo, float hi) {
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// one tile per block: 128 rows of A (or 32 columns of B) x 16 complex summation indices.  A unit is one
// row and four indices: one 16-byte core-matrix row per slice (two rows per slice for B).
__global__ void __launch_bounds__(256) oz_slice_kernel(OzOperand a, OzOperand b, const OzShift* shift, int nblk_a, int nkb) {
    const bool is_b = (int)blockIdx.x >= nblk_a;
    const OzOperand& o = is_b ? b : a;
    const int id = is_b ? (int)blockIdx.x - nblk_a : (int)blockIdx.x;
    const int kblk = id % nkb, tile = (id / nkb) % o.tiles, bt = id / (nkb * o.tiles);
    const int trows = is_b ? TNC : TM;
    const long long base = (long long)bt * o.s_batch;
    const int* bx = o.bx + ((long long)bt * o.tiles + tile) * trows;
    uint4* out = o.out + (long long)id * ((is_b ? B_BYTES : A_BYTES) / 16);
    const int Kt = o.K * o.kbn;
    for (int u = threadIdx.x; u < trows * (KBC / 4); u += 256) {
        const int r = u % trows, ch = u / trows;
        const int row = tile * trows + r;
        const int e = row < o.rows ? bx[r] : 0;
        const bool use = row < o.rows && e != NONFINITE;
        long long re[4], im[4];
        const int kk0 = kblk * KBC + ch * 4;
        int kb = kk0 / o.K, k = kk0 - kb * o.K;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            double2 v = make_double2(0.0, 0.0);
            int sk = 0;
            if (use && kk0 + j < Kt) {
                v = oz_load(o, base, row, kb, k);
                sk = k_shift(shift, a.kx, b.kx, kk0 + j);
                if (is_b) sk = -sk;
            }
            re[j] = fixed_point(v.x, e - EXP0, sk);
            im[j] = fixed_point(v.y, e - EXP0, sk);
            if (++k == o.K) { k = 0; ++kb; }
        }
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            float x[4], y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[j] = digit(re[j], s);
                y[j] = digit(im[j], s);
            }
            if (!is_b) {
                out[s * (A_SLICE / 16) + ch * TM + r] =
                    make_uint4(pack2(x[0], y[0]), pack2(x[1], y[1]), pack2(x[2], y[2]), pack2(x[3], y[3]));
            } else {
                uint4* q = out + s * (B_SLICE / 16) + ch * TN + 2 * r;
                q[0] = make_uint4(pack2(x[0], -y[0]), pack2(x[1], -y[1]), pack2(x[2], -y[2]), pack2(x[3], -y[3]));
                q[1] = make_uint4(pack2(y[0], x[0]), pack2(y[1], x[1]), pack2(y[2], x[2]), pack2(y[3], x[3]));
            }
        }
    }
}

// shared-memory matrix descriptor: K-major, no swizzle; core matrices of 8 rows x 16 bytes are 128
// contiguous bytes, `lbo` bytes apart along K and 128 bytes apart along the rows
__device__ __forceinline__ uint64_t oz_desc(uint32_t addr, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)(lbo >> 4) << 16;
    d |= (uint64_t)(128 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

constexpr uint32_t OZ_IDESC =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);

// use: the A tile's way through the collector buffer (0 none, 1 fill, 2 use, 3 last use)
#define OZ_MMA(COLLECT)                                                                             \
    asm volatile(                                                                                   \
        "{\n\t.reg .pred p;\n\t"                                                                    \
        "setp.ne.b32 p, %4, 0;\n\t"                                                                 \
        "tcgen05.mma.cta_group::1.kind::f16" COLLECT " [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),    \
        "l"(adesc), "l"(bdesc), "r"(OZ_IDESC), "r"(accumulate)                                      \
        : "memory")

__device__ __forceinline__ void oz_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate, int use) {
    if (use == 1) OZ_MMA(".collector::a::fill");
    else if (use == 2) OZ_MMA(".collector::a::use");
    else if (use == 3) OZ_MMA(".collector::a::lastuse");
    else OZ_MMA("");
}

__device__ __forceinline__ bool elect_one() {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok));
    return ok != 0;
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"((uint64_t)__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// overflow and gradual underflow of (hi:lo, leading bit set) 2^(E - 1086)
__device__ __noinline__ double oz_scaled(unsigned hi, unsigned lo, int E) {
    return ldexp((double)(long long)((((unsigned long long)hi << 32) | lo) >> 11), E - 1075);
}

// double of (H 2^32 + L) 2^(x - 2114), rounded to nearest; x the sum of the operands' biased row exponents.
// In 32-bit integer instructions (about 30): conversions to and from 64-bit types run on the narrow FP64
// pipe, and 64-bit shifts by a variable amount made a one-stage call 10 us longer.
__device__ __forceinline__ double oz_value(long long H, long long L, int x) {
    const long long h = H + (L >> 32);
    unsigned w0 = (unsigned)L, w1 = (unsigned)h, w2 = (unsigned)(h >> 32);
    const unsigned s = (unsigned)((int)w2 >> 31);  // all ones when negative
    asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %6;\n\tsubc.u32 %2, %5, %6;"
        : "=r"(w0), "=r"(w1), "=r"(w2)
        : "r"(w0 ^ s), "r"(w1 ^ s), "r"(w2 ^ s), "r"(s));
    int E = x - 996;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool z = w2 == 0u;
        w2 = z ? w1 : w2;
        w1 = z ? w0 : w1;
        w0 = z ? 0u : w0;
        E -= z ? 32 : 0;
    }
    const int lz = __clz(w2);
    E -= lz;  // biased exponent of the leading bit
    unsigned hi = __funnelshift_l(w1, w2, lz), lo = __funnelshift_l(w0, w1, lz), carry;
    if ((unsigned)(E - 1) > 2043u && w2 != 0u) {
        const double r = oz_scaled(hi, lo, E);
        return s ? -r : r;
    }
    asm("add.cc.u32 %0, %3, 1024;\n\taddc.cc.u32 %1, %4, 0;\n\taddc.u32 %2, 0, 0;"
        : "=r"(lo), "=r"(hi), "=r"(carry)
        : "r"(lo), "r"(hi));
    const unsigned rl = __funnelshift_r(lo, hi, 11);
    const unsigned rh = ((hi >> 11) + (carry << 21) + ((unsigned)(E - 1) << 20)) | (s & 0x80000000u);
    return w2 == 0u ? 0.0 : __hiloint2double((int)rh, (int)rl);
}

// The output of a row or column with a non-finite entry, term by term in FP64: an infinity or a NaN, whatever the
// order of the terms.  By the whole warp, 128 terms a step of about a microsecond (one lane alone takes half of
// one a term): the other warps' waits end after a second.  The longest sums of an SM with more than one item are of
// 83,000 terms (digits of at most 1 GiB an operand, 16 splits), 0.3 s for all 512 outputs of a warp.
__device__ __noinline__ double2 oz_direct(const OzParams& p, int ba, int bb, int m, int n) {
    double2 acc = make_double2(0.0, 0.0);
    const int Kt = p.a.K * p.a.kbn;
    for (int k0 = threadIdx.x & 31; k0 - (int)(threadIdx.x & 31) < Kt; k0 += 128) {
        double2 x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int kk = k0 + 32 * u, kb = kk / p.a.K, k = kk - kb * p.a.K;
            x[u] = y[u] = make_double2(0.0, 0.0);
            if (kk < Kt) {
                x[u] = oz_load(p.a, (long long)ba * p.a.s_batch, m, kb, k);
                y[u] = oz_load(p.b, (long long)bb * p.b.s_batch, n, kb, k);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (p.sparse_b && y[u].x == 0.0 && y[u].y == 0.0) continue;
            acc.x = fma(x[u].x, y[u].x, acc.x);
            acc.x = fma(-x[u].y, y[u].y, acc.x);
            acc.y = fma(x[u].x, y[u].y, acc.y);
            acc.y = fma(x[u].y, y[u].x, acc.y);
        }
        // NaN in both parts stays
        if (__any_sync(0xffffffffu, acc.x != acc.x) && __any_sync(0xffffffffu, acc.y != acc.y)) break;
    }
    for (int o = 16; o > 0; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
    }
    return acc;
}

// Persistent: CTA c takes items c, c + gridDim.x, ...; an item is (split, batch, m tile, n tile).
// Eight accumulators of 64 columns (one per digit weight) fill the 512 tensor-memory columns.
__global__ void __launch_bounds__(THREADS, 1) oz_gemm_kernel(const __grid_constant__ OzParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + (size_t)NST * STAGE);
    uint64_t* empty = full + NST;
    uint64_t* acc_full = empty + NST;     // [NP]
    uint64_t* acc_empty = acc_full + NP;  // [SL]
    uint32_t* tmem_slot = (uint32_t*)(acc_empty + SL);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int per_split = p.batch * p.tiles_m * p.tiles_n;
    const int items = per_split * p.splits;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < NP; ++s) mbar_init(&acc_full[s], 1);
        for (int s = 0; s < SL; ++s) mbar_init(&acc_empty[s], 8);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(SL * TN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    // item -> (split, batch, m tile, n tile); false when the tile lies above the diagonal of a Hermitian result
    auto decode = [&](int t, int& z, int& bz, int& mt, int& nt) {
        z = t / per_split;
        int r = t - z * per_split;
        nt = r % p.tiles_n;
        r /= p.tiles_n;
        mt = r % p.tiles_m;
        bz = r / p.tiles_m;
        return !(p.herm_lower && nt * TNC >= mt * TM + TM);
    };
    bool ok = true;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ISSUE));
        if (warp == 0 && lane == 0) {
            uint32_t g = 0;
            for (int t = blockIdx.x; t < items && ok; t += gridDim.x) {
                int z, bz, mt, nt;
                if (!decode(t, z, bz, mt, nt)) continue;
                const int k0 = z * p.kb_per, nk = min(p.nkb - k0, p.kb_per);
                const uint8_t* ga = (const uint8_t*)p.a.out +
                                    ((long long)((p.a.nb > 1 ? bz : 0) * p.tiles_m + mt) * p.nkb + k0) * A_BYTES;
                const uint8_t* gb = (const uint8_t*)p.b.out +
                                    ((long long)((p.b.nb > 1 ? bz : 0) * p.tiles_n + nt) * p.nkb + k0) * B_BYTES;
                for (int k = 0; k < nk; ++k, ++g) {
                    const int s = g % NST;
                    const uint32_t round = g / NST;
                    if (g >= NST && !(ok = mbar_wait(&empty[s], (round & 1) ^ 1, p.status))) break;
                    uint8_t* dst = smem + (size_t)s * STAGE;
                    mbar_expect_tx(&full[s], STAGE);
                    bulk_load(dst, ga + (long long)k * A_BYTES, A_BYTES, &full[s]);
                    bulk_load(dst + A_BYTES, gb + (long long)k * B_BYTES, B_BYTES, &full[s]);
                }
            }
        } else if (warp == 1) {
            // the whole warp walks the loop, so that its operands are warp-uniform; one elected lane issues
            const bool leader = elect_one();
            uint32_t g = 0;                      // stages of this CTA
            uint32_t drains[NP] = {0, 0, 0, 0};  // drains of each pair so far
            uint32_t fresh = 0xf;                // pairs whose next product starts a new sum
            for (int t = blockIdx.x; t < items && ok; t += gridDim.x) {
                int z, bz, mt, nt;
                if (!decode(t, z, bz, mt, nt)) continue;
                const int k0 = z * p.kb_per, nk = min(p.nkb - k0, p.kb_per);
                for (int k = 0; k < nk && ok; ++k, ++g) {
                    const int s = g % NST;
                    if (!(ok = mbar_wait(&full[s], (g / NST) & 1, p.status))) break;
                    fence_after();
                    const uint32_t sa = smem_u32(smem + (size_t)s * STAGE), sb = sa + A_BYTES;
                    const uint64_t ad = oz_desc(sa, TM * 16), bd = oz_desc(sb, TN * 16);
#pragma unroll
                    for (int q = 0; q < NP; ++q) {
                        const int w0 = SL - 1 - 2 * q, w1 = w0 - 1;
                        const bool is_fresh = (fresh >> q) & 1u;
                        if (is_fresh && drains[q] > 0) {
                            if (ok) ok = mbar_wait(&acc_empty[w0], (drains[q] & 1) ^ 1, p.status);
                            if (ok) ok = mbar_wait(&acc_empty[w1], (drains[q] & 1) ^ 1, p.status);
                            fence_after();
                        }
                        const bool due = drain_due(q, k, nk);
                        if (leader) {
                            // digit i of A serves both weights from the collector buffer
#pragma unroll
                            for (int h = 0; h < KB / 16; ++h) {
#pragma unroll
                                for (int i = 0; i <= w0; ++i) {
                                    const uint64_t ai = ad + ((i * A_SLICE + h * 2 * TM * 16) >> 4);
                                    const uint64_t b0 = bd + (((w0 - i) * B_SLICE + h * 2 * TN * 16) >> 4);
                                    const uint64_t b1 = bd + (((w1 - i) * B_SLICE + h * 2 * TN * 16) >> 4);
                                    const uint32_t add = h == 0 && i == 0 ? (is_fresh ? 0u : 1u) : 1u;
                                    oz_mma(tmem + (uint32_t)(w0 * TN), ai, b0, add, i <= w1 ? 1 : 0);
                                    if (i <= w1) oz_mma(tmem + (uint32_t)(w1 * TN), ai, b1, add, 3);
                                }
                            }
                            if (due) mma_commit(&acc_full[q]);
                            if (q == NP - 1) mma_commit(&empty[s]);
                        }
                        __syncwarp();
                        fresh &= ~(1u << q);
                        if (due) {
                            ++drains[q];
                            fresh |= 1u << q;
                        }
                    }
                }
            }
        }
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_DRAIN));
        // drain: warp w reads TMEM lanes [32 (w % 4), +32) = tile rows, columns [32 half, +32)
        const int q = warp & 3, half = (warp - 4) >> 2;
        const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 32);
        uint32_t drains = 0;  // parity of the drains of each pair so far
        for (int t = blockIdx.x; t < items && ok; t += gridDim.x) {
            int z, bz, mt, nt;
            if (!decode(t, z, bz, mt, nt)) continue;
            const int k0 = z * p.kb_per, nk = min(p.nkb - k0, p.kb_per);
            const int ba = p.a.nb > 1 ? bz : 0, bb = p.b.nb > 1 ? bz : 0;
            const int m = mt * TM + q * 32 + lane, n0 = nt * TNC + half * 16;
            // exponents of this lane's row and (lane j < 16) of column n0 + j
            const int ea = m < p.M ? p.a.bx[(long long)ba * p.a.tiles * TM + m] : 0;
            const int eb = lane < 16 && n0 + lane < p.N ? p.b.bx[(long long)bb * p.b.tiles * TNC + n0 + lane] : 0;
            long long H[32], L[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) H[j] = L[j] = 0;
            for (int k = 0; k < nk && ok; ++k) {
                // weights 7..4 into L, then 3..0 into H (rolled: the kernel's code is a large part of a small call)
                auto drain = [&](int pr, long long (&acc)[32]) {
                    if (!ok || !drain_due(pr, k, nk)) return;
                    ok = mbar_wait(&acc_full[pr], (drains >> pr) & 1u, p.status);
                    drains ^= 1u << pr;
                    if (!ok) return;
                    fence_after();
#pragma unroll 1
                    for (int u = 0; u < 2; ++u) {
                        const int w = SL - 1 - 2 * pr - u;
                        uint32_t v[32];
                        TC_LD32(lane_addr + w * TN, v);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_empty[w]);
                        const int scale = 1 << (8 * (3 - (w & 3)));
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            acc[j] += (long long)__float2int_rn(__uint_as_float(v[j])) * scale;
                    }
                };
#pragma unroll 1
                for (int pr = 0; pr < NP / 2; ++pr) drain(pr, L);
#pragma unroll 1
                for (int pr = NP / 2; pr < NP; ++pr) drain(pr, H);
            }
            if (!ok) break;
            const bool to_part = p.splits > 1;
            double2* C = to_part ? p.part + z * p.part_split + bz * p.part_batch : p.C + (long long)bz * p.sC_batch;
            const long long cn = to_part ? p.part_n : p.sC_n;
            double2* dst = C + (long long)m * (to_part ? p.part_m : p.ldc) + n0 * cn;
            auto store = [&](int j, double2 r) {
                if (p.negate) r = make_double2(-r.x, -r.y);
                if (p.accumulate && !to_part) {
                    const double2 o = dst[j * cn];
                    r.x += o.x;
                    r.y += o.y;
                }
                dst[j * cn] = r;
            };
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int en = __shfl_sync(0xffffffffu, eb, j);
                if (m >= p.M || n0 + j >= p.N || ea == NONFINITE || en == NONFINITE) continue;
                const int x = ea + en - 2 * EXP0;  // of zero rows: the sums are zero
                store(j, make_double2(oz_value(H[2 * j], L[2 * j], x), oz_value(H[2 * j + 1], L[2 * j + 1], x)));
            }
            // (apart from the loop above, which is 4 % of a product longer with this inside)
            if (__any_sync(0xffffffffu, ea == NONFINITE || eb == NONFINITE)) {
#pragma unroll 1
                for (int j = 0; j < 16; ++j) {
                    const int en = __shfl_sync(0xffffffffu, eb, j);
                    unsigned todo = __ballot_sync(0xffffffffu, m < p.M && n0 + j < p.N && (ea == NONFINITE || en == NONFINITE));
                    for (; todo != 0u; todo &= todo - 1u) {
                        const int l = __ffs(todo) - 1;
                        double2 r = make_double2(0.0, 0.0);
                        if (z == 0) r = oz_direct(p, ba, bb, mt * TM + q * 32 + l, n0 + j);
                        if (lane == l) store(j, r);
                    }
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SL * TN));
    }
}

long long cdiv(long long a, long long b) { return (a + b - 1) / b; }

// tiles per block of the exponent kernel
int max_reps(const Ctx& ctx, long long tiles) { return (int)cdiv(tiles, 8ll * std::max(ctx.num_sms, 1)); }

}  // namespace

// Splits of the summation over the CTAs: the smallest number (<= 16) whose waves of equal items come within a
// tenth of the best; a split costs one more pass over the outputs.
int oz_splits(const Ctx& ctx, const GemmArgs& g) {
    const long long nkb = cdiv((long long)g.K * g.kb, KBC);
    const long long tiles = cdiv(g.M, TM) * cdiv(g.N, TNC) * g.batch / (g.herm_lower ? 2 : 1) + 1;
    const long long sms = std::max(ctx.num_sms, 1);
    auto cost = [&](int s) { return (double)cdiv(tiles * s, sms) * (double)(cdiv(nkb, s) + 2); };
    double best = cost(1);
    for (int s = 2; s <= 16 && s * 4 <= nkb; ++s) best = std::min(best, cost(s));
    for (int s = 1; s <= 16; ++s)
        if (s == 1 || s * 4 <= nkb) {
            if (cost(s) <= 1.1 * best) return s;
        }
    return 1;
}

// op(A) (or op(B)) rows [r0, r0 + rows) of batches [b0, b0 + nb)
static void fill_operand(OzOperand& o, const GemmArgs& g, bool is_b, long long b0, long long r0, int rows, int tiles, int nb) {
    const Op op = is_b ? g.opB : g.opA;
    o.K = g.K; o.kbn = g.kb;
    o.kc = is_b ? op != OP_N : op == OP_N;
    o.conj = op == OP_C;
    o.ld = is_b ? g.ldb : g.lda;
    o.s_batch = is_b ? g.sB_batch : g.sA_batch;
    o.s_kb = is_b ? g.sB_kb : g.sA_kb;
    o.X = (is_b ? g.B : g.A) + b0 * o.s_batch + (o.kc ? r0 * o.ld : r0);
    o.rows = rows; o.tiles = tiles; o.nb = nb;
}

// The digits of op(A) (M x K) once, for products that share it; without the scaling of the summation index,
// which depends on both operands.
OzPrep oz_prepare(Ctx& ctx, int M, int K, Op opA, const double2* A, long long lda) {
    GemmArgs g;
    g.M = M; g.N = 1; g.K = K;
    g.opA = opA; g.A = A; g.lda = lda;
    g.B = nullptr; g.ldb = 0; g.C = nullptr; g.ldc = 0;
    const int nkb = (int)cdiv(K, KBC), tiles = (int)cdiv(M, TM);
    const size_t digits = (size_t)tiles * nkb * A_BYTES, n_bx = (size_t)tiles * TM;
    char* w = (char*)ctx.workspace(WS_OZ_PREP, digits + sizeof(int) * n_bx + sizeof(OzShift));
    OzOperand a;
    fill_operand(a, g, false, 0, 0, M, tiles, 1);
    a.out = (uint4*)w;
    a.bx = (int*)(w + digits);
    OzShift* shift = (OzShift*)(a.bx + n_bx);
    a.kx = nullptr;
    VTN_CUDA_TRY(cudaMemsetAsync(a.bx, 0, sizeof(int) * n_bx + sizeof(OzShift), ctx.stream));
    const int kseg = (int)cdiv(K, MAX_KS), reps = max_reps(ctx, cdiv(M, 32) * kseg);
    const long long ma = cdiv(cdiv(M, 32), reps) * kseg, sa = (long long)tiles * nkb;
    oz_max_kernel<0><<<(unsigned)ma, 256, 0, ctx.stream>>>(a, a, shift, (int)ma, kseg, reps, -1);
    oz_slice_kernel<<<(unsigned)sa, 256, 0, ctx.stream>>>(a, a, shift, (int)sa, nkb);
    ctx.count_launch(2);
    ctx.check_launch("oz_prepare");
    OzPrep p;
    p.digits = w;
    p.bx = a.bx;
    p.M = M;
    p.K = K;
    return p;
}

// Returns false, with nothing launched, when there is no device memory for the digits (the first piece needs the
// most): the caller then takes the FP64 kernel, which needs none.
bool oz_gemm(Ctx& ctx, const GemmArgs& g, int splits, double2* part) {
    VTN_REQUIRE(ctx.dstatus != nullptr, "context has no device status word");
    VTN_REQUIRE(g.prepA == nullptr || (g.prepA->M == g.M && g.prepA->K == g.K && g.batch == 1 && g.kb == 1),
                "prepared operand of another shape");
    set_smem_attr_once(ctx, (const void*)oz_gemm_kernel, (int)SMEM);
    const int nkb = (int)cdiv((long long)g.K * g.kb, KBC);
    // At most 1 GiB of digit tiles per operand (one tile row at least, 128 rows and columns of a Hermitian result): larger
    // problems run in pieces, a Hermitian one in square ones of which those above the diagonal are left out.  A
    // prepared operand is the caller's; it comes whole.
    const long long cap = 1ll << 30;
    const bool a_shared = g.sA_batch == 0 || g.batch == 1, b_shared = g.sB_batch == 0 || g.batch == 1;
    const long long a_batch = cdiv(g.M, TM) * nkb * A_BYTES, b_batch = cdiv(g.N, TNC) * nkb * B_BYTES;
    long long bs = g.batch;
    if (!a_shared) bs = std::min(bs, std::max(1ll, cap / a_batch));
    if (!b_shared) bs = std::min(bs, std::max(1ll, cap / b_batch));
    long long ms = g.M, ns = g.N;
    if (a_batch > cap) ms = std::max(1ll, cap / ((long long)nkb * A_BYTES)) * TM;
    if (b_batch > cap) ns = std::max(1ll, cap / ((long long)nkb * B_BYTES)) * TNC;
    if (g.prepA) ms = g.M;
    if (g.herm_lower && (ms < g.M || ns < g.N)) ms = ns = std::max(1ll, std::min(ms, ns) / TM) * TM;
    const bool part_t = g.sC_n != 1;  // partials column by column
    const long long part_m = part_t ? 1 : g.N, part_n = part_t ? g.M : 1, part_batch = (long long)g.M * g.N;
    for (long long b0 = 0; b0 < g.batch; b0 += bs) {
        const int nb = (int)std::min(bs, g.batch - b0);
        for (long long n0 = 0; n0 < g.N; n0 += ns) {
            const int nn = (int)std::min(ns, g.N - n0);
            for (long long m0 = g.herm_lower ? n0 : 0; m0 < g.M; m0 += ms) {
                const int mm = (int)std::min(ms, g.M - m0);
                OzParams p;
                p.M = mm; p.N = nn; p.nkb = nkb;
                p.batch = nb; p.splits = splits; p.kb_per = (int)cdiv(nkb, splits);
                p.tiles_m = (int)cdiv(mm, TM);
                p.tiles_n = (int)cdiv(nn, TNC);
                const OzPrep* prep = g.prepA;
                fill_operand(p.a, g, false, b0, m0, mm, p.tiles_m, a_shared ? 1 : nb);
                fill_operand(p.b, g, true, b0, n0, nn, p.tiles_n, b_shared ? 1 : nb);
                const size_t na = prep ? 0 : (size_t)p.a.nb * p.tiles_m * TM, nbx = (size_t)p.b.nb * p.tiles_n * TNC;
                const size_t nk = (size_t)g.K * g.kb, n_exp = sizeof(OzShift) / sizeof(int) + na + nbx + 2 * nk;
                OzShift* shift;
                ctx.digits_busy = true;
                try {
                    shift = (OzShift*)ctx.workspace(WS_OZ_EXP, sizeof(int) * n_exp);
                    p.a.out = prep ? (uint4*)prep->digits
                                   : (uint4*)ctx.workspace(WS_OZ_A, (size_t)p.a.nb * p.tiles_m * nkb * A_BYTES);
                    p.b.out = (uint4*)ctx.workspace(WS_OZ_B, (size_t)p.b.nb * p.tiles_n * nkb * B_BYTES);
                } catch (const Error& e) {
                    ctx.digits_busy = false;
                    if (e.status != VTN_ENOMEM || b0 + n0 + m0 > 0) throw;
                    ctx.drop_digits();
                    return false;
                }
                ctx.digits_busy = false;
                p.a.bx = prep ? prep->bx : (int*)(shift + 1);
                p.b.bx = (int*)(shift + 1) + na;
                p.a.kx = p.b.bx + nbx;
                p.b.kx = p.a.kx + nk;
                p.C = g.C + b0 * g.sC_batch + m0 * g.ldc + n0 * g.sC_n;
                p.ldc = g.ldc; p.sC_n = g.sC_n; p.sC_batch = g.sC_batch;
                p.part = part + b0 * part_batch + m0 * part_m + n0 * part_n;
                p.part_m = part_m; p.part_n = part_n;
                p.part_batch = part_batch; p.part_split = part_batch * g.batch;
                p.accumulate = g.accumulate; p.negate = g.negate; p.herm_lower = g.herm_lower && m0 == n0; p.sparse_b = g.sparse_b;
                p.status = ctx.dstatus;
                VTN_CUDA_TRY(cudaMemsetAsync(shift, 0, sizeof(int) * n_exp, ctx.stream));
                const int kseg = (int)cdiv((long long)g.K * g.kb, MAX_KS);
                const long long ra = prep ? 0 : cdiv(mm, 32), rb = cdiv(nn, 32);
                const int reps = max_reps(ctx, (ra * p.a.nb + rb * p.b.nb) * kseg);
                const long long ma = cdiv(ra, reps) * kseg * p.a.nb, mb = cdiv(rb, reps) * kseg * p.b.nb;
                oz_max_kernel<0><<<(unsigned)(ma + mb), 256, 0, ctx.stream>>>(p.a, p.b, shift, (int)ma, kseg, reps,
                                                                              prep ? -1 : (int)(na + nbx));
                if (!prep) oz_max_kernel<1><<<(unsigned)(ma + mb), 256, 0, ctx.stream>>>(p.a, p.b, shift, (int)ma, kseg, reps, 0);
                const long long sa = prep ? 0 : (long long)p.a.nb * p.tiles_m * nkb, sb = (long long)p.b.nb * p.tiles_n * nkb;
                oz_slice_kernel<<<(unsigned)(sa + sb), 256, 0, ctx.stream>>>(p.a, p.b, shift, (int)sa, nkb);
                const long long items = (long long)p.tiles_m * p.tiles_n * nb * splits;
                VTN_REQUIRE(items < (1ll << 31) && ma + mb < (1ll << 31) && sa + sb < (1ll << 31), "GEMM too large");
                oz_gemm_kernel<<<(unsigned)std::min<long long>(items, std::max(ctx.num_sms, 1)), THREADS, SMEM, ctx.stream>>>(p);
                ctx.dstatus_due = true;
                ctx.count_launch(prep ? 3 : 4);
                ctx.check_launch("oz_gemm");
            }
        }
    }
    return true;
}

}  // namespace vtn
