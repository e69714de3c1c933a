// FP64 complex products on the tensor cores by digit splitting (the Ozaki scheme: K. Ozaki,
// T. Ogita, S. Oishi, S. M. Rump, Numer. Algorithms 59, 95 (2012)).
//
//   cn: C[m][n] = sum_k conj(A[m][k]) B[n][k]
//   tn: C[m][n] (+)= alpha sum_k A[k][m] d[k] B[k][n]
//
// This GPU's FP64 pipe does 1.2 TFLOP/s, its BF16 tensor cores 1956; the products above are the
// bulk of the plain FP64 form.  Every row x of an operand is scaled by a power of two of its
// largest component, |x| < 2^E, and rounded to the integer X = x 2^(55 - E) (the largest elements
// keep all their bits), written in seven balanced base-256 digits
//   X = sum_i D_i 256^(6-i),  D_i in [-128, 128],
// which BF16 holds exactly.  A product of two digits is at most 2^14, so a sum of them is an
// integer FP32 holds exactly below 2^24: the tensor core's FP32 accumulation commits no rounding.
// Digit products of equal weight i + j = d share one accumulator; the eight accumulators
// d = 0 ... 7 (34 of the 49 digit products; the dropped ones sum to at most 2^-59.7 of max|a| max|b| per
// real term) are read from tensor memory every kDgChunk K tiles and added to 64-bit integers,
// hi = S_0 2^24 + ... + S_3 and lo = S_4 2^24 + ... + S_7, so the sum over K is exact as well and
// does not depend on how K is split; one rounding makes the FP64 result.
// The error of a term is that of its operands' rounding, at most 2^-55 of the row's largest component,
// where FP64 multiply-adds round every partial sum: FP64 accuracy by norm.  It is not element by
// element: what lies below 2^-56 of its row's largest is lost, so a sum that such elements decide (rows
// that fall where the other operand's rise, |a_k| = e^(-20 k/K), |b_k| = e^(20 k/K - 20): error 7e-11 of
// sum |a| |b| at 200 x 60 x 4000, FP64 2e-17; e^-3: 8e-18, 2e-17) needs the FP64 kernels: qm_zgemm's arith 3, qm_davidson_opts.fp64_exact.
// Relative error (2-norm, against 80-bit sums) of rows that fall together, FP64
// multiply-adds / digits: 2.7e-15 / 1.3e-16 at 480 x 157 x 18232 (rows falling off 13-fold), 2.4e-15 /
// 8.9e-17 (200-fold), 3.8e-15 / 9.6e-17 at 640 x 100 x 40000, 8.6e-16 / 8.4e-17 at 512 x 64 x 400;
// tn 2.3e-16 / 7.2e-17 at 64 x 12000 x 17, 2.7e-15 / 1.2e-16 at 157 x 18232 x 480.
// (In one accumulator at most 7 x 256 digit products of at most 2^14 meet; should their sum pass
// 2^24, which needs nearly all digits of both rows at their extreme with one sign, FP32 rounds
// off units of the accumulator's weight.)
//
// Rows that hold a non-finite value, or nothing above 2^-960, are flagged in the exponent arrays
// and left to the FP64 kernels (zgemm.cu), which recompute exactly those outputs.
//
// Complex to real as in nonlocal_tc.cu: K' = 2K with re, im interleaved; the "plain" operand's
// rows as stored, the "expanded" operand's rows doubled (2r + t) so that the product of a plain
// and an expanded row is the real (t = 0) or imaginary (t = 1) part.
// cn: plain = A (rows m), expanded = conj pattern of B; tn: plain = B transposed (rows n: the
// long plane-wave dimension), expanded = alpha d A transposed.
//
// GEMM kernel (k_dg_gemm): 128 plain x 64 expanded rows per CTA, the eight accumulators in the
// 8 x 64 columns of tensor memory; a producer thread streams 16-term K tiles (both operands' seven
// planes, 43 KB, one bulk copy each) into a 5-stage mbarrier ring, one thread issues the
// tcgen05.mma of a tile, eight warps drain the accumulators.  The seven planes of the expanded
// operand lie one after another, i.e. as 448 rows of one operand, and the accumulators likewise, so
// the products of plain digit i with every digit j are one or two wide products (N up to 256,
// columns 64 i ...) instead of one of N = 64 per pair: each reads the plain plane from shared memory
// again (32 cycles), and 34 narrow products were bound by that (48 cycles each; 1.01 us per K tile
// for 28 of them, 0.81 us for 34 as 13 wide ones).  The drains do not overlap the products (the
// accumulators leave no second buffer): about 0.13 us per K tile.
// Every mbarrier wait is bounded; on expiry the kernel flags its rows for the FP64 kernels (an
// output that is accumulated onto gets NaN instead), sets the error word (when there is one),
// waits (bounded) for its own copies and products and returns.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "qm_internal.h"
#include "tc_util.cuh"

namespace qm {
namespace {

constexpr int kDg = 7;             // digits per operand
constexpr int kDgAcc = 8;          // accumulators: digit products of weight 0 ... 7
constexpr int kDgM = 128;          // plain rows per tile
constexpr int kDgN = 64;           // expanded rows per tile
constexpr int kDgK = 16;           // real terms per K tile
constexpr int kDgChunk = 16;       // K tiles between drains (256 terms)
constexpr int kDgStages = 5;
constexpr int kDgEpiWarps = 8;
constexpr int kDgThreads = 32 * (kDgEpiWarps + 2);
constexpr int kDgFlag = 0x7FF;     // exponent of a row left to the FP64 kernels
constexpr int kDgSegs = 4;         // partial maxima per row
constexpr int kDgSpin = 1 << 26;

__host__ __device__ constexpr size_t dg_plane(int R) { return (size_t)R * kDgK * 2; }
__host__ __device__ constexpr size_t dg_block(int R) { return kDg * dg_plane(R); }

__device__ __forceinline__ int hi_abs(double x) { return __double2hiint(x) & 0x7FFFFFFF; }

// exponent of a row from the largest high word of its components: the biased FP64 exponent, 0 for
// a zero row, kDgFlag for rows the integers do not serve
__device__ __forceinline__ int row_exponent(int hmax) {
    if (hmax >= 0x7FF00000) return kDgFlag;
    const int e = hmax >> 20;
    return hmax == 0 ? 0 : (e < 64 ? kDgFlag : e);
}
__device__ __forceinline__ int reduce_segs(const int* __restrict__ emax, int n, int r) {  // n: rows of the whole operand
    int h = 0;
#pragma unroll
    for (int s = 0; s < kDgSegs; ++s) h = max(h, __ldg(emax + (size_t)s * n + r));
    return row_exponent(h);
}

// x 2^(55 - E) rounded to an integer (|x| < 2^E, E the unbiased exponent of `e` plus one), plus the
// digit bias: bits 8p .. of the result are digit 6-p + 128 (nine bits for the leading one)
__device__ __forceinline__ unsigned long long digits_of(double x, int e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7FF;
    const int sh = e - 2 - ex;  // -2 for the row's largest exponent
    unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    if (sh < 0) m <<= -sh;
    else m = sh < 63 ? ((m + ((1ull << sh) >> 1)) >> sh) : 0;
    if (ex == 0 || e == 0 || e == kDgFlag) m = 0;
    const unsigned long long bias = 0x0080808080808080ull;
    return (b >> 63) ? bias - m : bias + m;
}
// digits p (from the low end) of two values as a pair of BF16
__device__ __forceinline__ uint32_t digit_pair(unsigned long long u, unsigned long long v, int p) {
    uint32_t a, b;  // 2^23 + digit + 128 as floats
    if (p == kDg - 1) {
        a = 0x4B000000u | (uint32_t)(u >> 48);
        b = 0x4B000000u | (uint32_t)(v >> 48);
    } else {
        a = __byte_perm((uint32_t)(p < 4 ? u : u >> 32), 0x4B000000u, 0x7650 | (p & 3));
        b = __byte_perm((uint32_t)(p < 4 ? v : v >> 32), 0x4B000000u, 0x7650 | (p & 3));
    }
    const float x = __uint_as_float(a) - 8388736.0f, y = __uint_as_float(b) - 8388736.0f;
    return __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
}
// write 8 consecutive K values of row r (k0 a multiple of 8) into the seven planes of a blocked operand
__device__ __forceinline__ void put_digits(unsigned char* blk, int R, int nkt, int r, int k0, const double* v, int e) {
    const int rt = r / R, rr = r - rt * R, kt = k0 / kDgK, kk = k0 - kt * kDgK;
    unsigned char* p = blk + ((size_t)rt * nkt + kt) * dg_block(R) + ((((rr >> 3) << 1) + (kk >> 3)) << 7) + ((rr & 7) << 4);
    unsigned long long u[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) u[j] = digits_of(v[j], e);
#pragma unroll
    for (int q = 0; q < kDg; ++q) {
        uint4 w;
        w.x = digit_pair(u[0], u[1], kDg - 1 - q);
        w.y = digit_pair(u[2], u[3], kDg - 1 - q);
        w.z = digit_pair(u[4], u[5], kDg - 1 - q);
        w.w = digit_pair(u[6], u[7], kDg - 1 - q);
        *reinterpret_cast<uint4*>(p + q * dg_plane(R)) = w;
    }
}
// the expanded row t of 4 complex values (interleaved): conj pattern (cn) (re, im), (im, -re);
// plain pattern (tn) (re, -im), (im, re)
__device__ __forceinline__ void expand4(double* v, int t, int conj) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const double re = v[2 * j], im = v[2 * j + 1];
        v[2 * j] = t ? im : re;
        v[2 * j + 1] = conj ? (t ? -re : im) : (t ? re : -im);
    }
}

// largest high word of each row over column segment blockIdx.y
// (any: the word that tells whether some row is flagged; cleared here by the first launch of a
// product and set by the digit kernels)
__global__ void __launch_bounds__(256) k_dg_rowmax(const double2* __restrict__ src, int ld, int rows, int cols,
                                                   int* __restrict__ emax, int* __restrict__ any) {
    __shared__ int red[8];
    if (any && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *any = 0;
    const int r = blockIdx.x, per = (cols + kDgSegs - 1) / kDgSegs;
    const int c0 = blockIdx.y * per, c1 = min(cols, c0 + per);
    const double2* p = src + (size_t)r * ld;
    int h = 0;
    for (int c = c0 + threadIdx.x; c < c1; c += 256) {
        const double2 v = __ldg(p + c);
        h = max(h, max(hi_abs(v.x), hi_abs(v.y)));
    }
    h = __reduce_max_sync(0xffffffffu, h);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) h = max(h, red[w]);
        emax[(size_t)blockIdx.y * rows + r] = h;
    }
}

// the same per column of src [K][cols] (optionally scaled by alpha d[k]) over K segment blockIdx.y
__global__ void __launch_bounds__(256) k_dg_colmax(const double2* __restrict__ src, int ld, int K, int cols,
                                                   const double* __restrict__ d, double alpha, int* __restrict__ emax,
                                                   int* __restrict__ any) {
    if (any && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *any = 0;
    const int c = blockIdx.x * 256 + threadIdx.x, per = (K + kDgSegs - 1) / kDgSegs;
    if (c >= cols) return;
    const int k0 = blockIdx.y * per, k1 = min(K, k0 + per);
    int h = 0;
#pragma unroll 8
    for (int k = k0; k < k1; ++k) {
        double2 v = __ldg(src + (size_t)k * ld + c);
        if (d || alpha != 1.0) {
            const double sc = d ? alpha * __ldg(d + k) : alpha;
            v.x *= sc;
            v.y *= sc;
        }
        h = max(h, max(hi_abs(v.x), hi_abs(v.y)));
    }
    emax[(size_t)blockIdx.y * cols + c] = h;
}

// rows of src (complex columns [0, cols)) -> digit planes; expanded: output row 2r + t.  CTA: 8
// output rows (one core-matrix row group) x 32 chunks of 8 real values.  eout: the rows' exponents, written
// for the first panel of K only (NULL later): a product that gives up marks its rows there, and a later panel
// must not take the mark off
__global__ void __launch_bounds__(256) k_dg_rows(const double2* __restrict__ src, int ld, int rows, int cols, int expand,
                                                 int R, int nkt, const int* __restrict__ emax, int* __restrict__ eout,
                                                 int* __restrict__ any, unsigned char* __restrict__ blk) {
    const int r = blockIdx.y * 8 + (threadIdx.x & 7);
    const int ch = blockIdx.x * 32 + (threadIdx.x >> 3);
    const int b = expand ? (r >> 1) : r;
    const int e = b < rows ? reduce_segs(emax, rows, b) : 0;
    if (eout && ch == 0 && b < rows && !(expand && (r & 1))) {
        eout[b] = e;
        if (e == kDgFlag) *any = 1;
    }
    if (ch >= nkt * (kDgK / 8)) return;
    double v[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        double2 x = make_double2(0.0, 0.0);
        if (b < rows && ch * 4 + j < cols) x = __ldg(src + (size_t)b * ld + ch * 4 + j);
        v[2 * j] = x.x;
        v[2 * j + 1] = x.y;
    }
    if (expand) expand4(v, r & 1, 1);
    put_digits(blk, R, nkt, r, ch * 8, v, e);
}

// columns of src [K][cols] (scaled by alpha d[k]) -> digit planes of its transpose: output row =
// column c (expanded: 2c + t), K = k.  CTA: 64 output rows x 16 values of k, transposed through
// shared memory so the global reads run along the columns.
__global__ void __launch_bounds__(256) k_dg_cols(const double2* __restrict__ src, int ld, int K, int cols,
                                                 const double* __restrict__ d, double alpha, int expand, int R, int nkt,
                                                 const int* __restrict__ emax, int nmax, int* __restrict__ eout,
                                                 int* __restrict__ any, unsigned char* __restrict__ blk) {
    __shared__ double2 t[16][65];
    const int r0 = blockIdx.x * 64, nc = expand ? 32 : 64, c0 = expand ? (r0 >> 1) : r0, k0 = blockIdx.y * 16;
    for (int i = threadIdx.x; i < 16 * nc; i += 256) {
        const int kk = i / nc, cc = i - kk * nc;
        double2 x = make_double2(0.0, 0.0);
        if (k0 + kk < K && c0 + cc < cols) {
            x = __ldg(src + (size_t)(k0 + kk) * ld + c0 + cc);
            if (d || alpha != 1.0) {
                const double sc = d ? alpha * __ldg(d + k0 + kk) : alpha;
                x.x *= sc;
                x.y *= sc;
            }
        }
        t[kk][cc] = x;
    }
    __syncthreads();
    const int rlo = threadIdx.x & 7, ch = (threadIdx.x >> 3) & 3, rg = threadIdx.x >> 5;
    const int rr = rg * 8 + rlo, cc = expand ? (rr >> 1) : rr, c = c0 + cc;
    const int e = c < cols ? reduce_segs(emax, nmax, c) : 0;
    if (blockIdx.y == 0 && ch == 0 && c < cols && !(expand && (rr & 1))) {
        eout[c] = e;
        if (e == kDgFlag) *any = 1;
    }
    if (blockIdx.y * 2 + (ch >> 1) >= nkt) return;
    double v[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const double2 x = t[ch * 4 + j][cc];
        v[2 * j] = x.x;
        v[2 * j + 1] = x.y;
    }
    if (expand) expand4(v, rr & 1, 0);
    put_digits(blk, R, nkt, r0 + rr, (k0 + ch * 4) * 2, v, e);
}

// (hi 2^32 + lo) 2^ex rounded to FP64 (to nearest, ties away from zero), by integer arithmetic: the
// conversions and additions of the FP64 pipe would cost several times as much
__device__ __forceinline__ double dg_value(long long hi, long long lo, int ex) {
    unsigned long long L = (unsigned long long)hi << 32;
    long long H = hi >> 32;
    L += (unsigned long long)lo;
    H += (lo >> 63) + (L < (unsigned long long)lo ? 1 : 0);
    const bool neg = H < 0;
    if (neg) {
        L = ~L + 1;
        H = ~H + (L == 0 ? 1 : 0);
    }
    if (H == 0 && L == 0) return 0.0;
    const int lz = H ? __clzll(H) : 64 + __clzll((long long)L);
    unsigned long long top = lz >= 64 ? L << (lz - 64) : (lz ? ((unsigned long long)H << lz) | (L >> (64 - lz)) : (unsigned long long)H);
    int e2 = ex + 127 - lz;  // exponent of the leading bit
    top += 1024;
    if (top < 1024) {  // carried out: the value is the next power of two
        top = 1ull << 63;
        ++e2;
    }
    const unsigned long long mant = (top >> 11) & 0xFFFFFFFFFFFFFull;
    const unsigned long long sgn = neg ? 0x8000000000000000ull : 0ull;
    if (e2 > -1022 && e2 < 1024) return __longlong_as_double((long long)(sgn | ((unsigned long long)(e2 + 1023) << 52) | mant));
    const double m = __longlong_as_double((long long)(sgn | (1023ull << 52) | mant));
    return scalbn(m, e2);
}
// exponent of the integer unit of a product of rows with exponents ea, eb
__device__ __forceinline__ int dg_unit(int ea, int eb) { return ea + eb - 2 * 1022 - 70; }

__device__ __forceinline__ bool dg_wait(uint32_t bar, uint32_t parity, volatile int* abort, int polls = kDgSpin) {
    for (int i = 0; i < polls; ++i) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 1023) == 1023 && abort && *abort) return false;
    }
    return false;
}

// Products of plain tile blockIdx.y and expanded tile blockIdx.x over the K tiles of split
// blockIdx.z.  EPI 0 (cn): the exact sums (hi, lo) of row m, real column n to
// part[(z * mpad + m) * npad + n] (add: on top of what an earlier panel of K left there).
// EPI 1 (tn): C[n / 2][plain row] of the complex FP64 output, component n % 2 (accumulate: added),
// except outputs of flagged rows.  kHold: waits give up after `polls` polls (as a run-time number in every
// launch it cost 5 us of 316 at 480 x 157 x 18232).
template <int EPI, bool kHold>
__global__ void __launch_bounds__(kDgThreads, 1)
k_dg_gemm(const unsigned char* __restrict__ P, const unsigned char* __restrict__ X, int nkt, int kt_per_split,
          longlong2* __restrict__ part, int mpad, int npad, int add, int* __restrict__ ep,
          const int* __restrict__ ex, int* __restrict__ any, int nplain, int nexp, double2* __restrict__ C, int ldc, int accumulate,
          int* __restrict__ err, int polls) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[kDgStages], empty[kDgStages], acc_full, acc_empty, done;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, s_used, s_issued;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kt0 = blockIdx.z * kt_per_split;
    const int nk = max(0, min(nkt, kt0 + kt_per_split) - kt0);
    const int nchunk = (nk + kDgChunk - 1) / kDgChunk;
    constexpr uint32_t a_bytes = (uint32_t)dg_block(kDgM), b_bytes = (uint32_t)dg_block(kDgN), st_bytes = a_bytes + b_bytes;
    if (warp == kDgEpiWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tc::smem_u32(&tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int s = 0; s < kDgStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&empty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&acc_full)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(tc::smem_u32(&acc_empty)), "r"(kDgEpiWarps));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&done)));
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        abort_flag = 0;
        s_used = s_issued = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = tmem_base, sbase = tc::smem_u32(smem);
    volatile int* abort = &abort_flag;
    const int limit = kHold ? polls : kDgSpin;
    if (warp == kDgEpiWarps) {
        if (lane == 0) {
            const unsigned char* a_src = P + ((size_t)blockIdx.y * nkt + kt0) * a_bytes;
            const unsigned char* b_src = X + ((size_t)blockIdx.x * nkt + kt0) * b_bytes;
            int it = 0;
            for (; it < nk; ++it) {
                const int s = it % kDgStages;
                if (it >= kDgStages && !dg_wait(tc::smem_u32(&empty[s]), ((it / kDgStages) & 1) ^ 1, abort, limit)) {
                    *abort = 1;
                    break;
                }
                const uint32_t fb = tc::smem_u32(&full[s]), dst = sbase + s * st_bytes;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(st_bytes) : "memory");
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                    "l"(a_src + (size_t)it * a_bytes), "r"(a_bytes), "r"(fb)
                    : "memory");
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                        dst + a_bytes),
                    "l"(b_src + (size_t)it * b_bytes), "r"(b_bytes), "r"(fb)
                    : "memory");
            }
            s_issued = it;
        }
    } else if (warp == kDgEpiWarps + 1) {
        if (lane == 0) {
            int it = 0;
            for (; it < nk; ++it) {
                const int s = it % kDgStages, c = it / kDgChunk;
                // the drains of the previous chunk must have read the accumulators
                if (it % kDgChunk == 0 && c > 0 && !dg_wait(tc::smem_u32(&acc_empty), (c - 1) & 1, abort, limit)) {
                    *abort = 1;
                    break;
                }
                if (!dg_wait(tc::smem_u32(&full[s]), (it / kDgStages) & 1, abort, limit)) {
                    *abort = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint32_t sa = sbase + s * st_bytes, sb = sa + a_bytes;
                // plain digit i times expanded digits j = 0 ... min(6, 7 - i), in at most 256 columns at once
                // from column 64 i on.  A chunk's first tile starts the accumulators: d < 7 with i = 0,
                // d = 7 with (i, j) = (1, 6), which is a product of its own.
                const uint32_t more = it % kDgChunk != 0 ? 1u : 0u;
#pragma unroll
                for (int i = 0; i < kDg; ++i) {
                    const uint64_t da = tc::sdesc(sa + i * (uint32_t)dg_plane(kDgM), 128, 256);
                    const int cols = kDgN * (i == 0 ? kDg : kDgAcc - i);
#pragma unroll
                    for (int n0 = 0, n = 0; n0 < cols; n0 += n) {
                        n = i == 1 ? (n0 == 0 ? 256 : n0 == 256 ? 128 : 64) : cols <= 256 ? cols : (n0 == 0 ? (cols / 2 + 15) / 16 * 16 : cols - n0);
                        const uint64_t db = tc::sdesc(sb + n0 * 32, 128, 256);
                        const uint32_t acc = i == 0 || (i == 1 && n0 == 384) ? more : 1u;
                        asm volatile(
                            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + i * kDgN + n0),
                            "l"(da), "l"(db), "r"(tc::idesc_bf16(kDgM, n)), "r"(acc));
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    tc::smem_u32(&empty[s])));
                if (it % kDgChunk == kDgChunk - 1 || it == nk - 1)
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                        tc::smem_u32(&acc_full)));
            }
            s_used = it;
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                tc::smem_u32(&done)));
        }
    } else {
        const int q = warp & 3, col0 = (warp >> 2) * 32;  // tensor-memory lanes 32 q.., columns col0..col0+31
        long long hi[32], lo[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) hi[j] = lo[j] = 0;
        bool ok = true;
        for (int c = 0; c < nchunk; ++c) {
            ok = dg_wait(tc::smem_u32(&acc_full), c & 1, abort, limit);
            if (!ok) *abort = 1;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += 4) {
                uint32_t v[kDgAcc][4];
#pragma unroll
                for (int d = 0; d < kDgAcc; ++d)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                                 : "=r"(v[d][0]), "=r"(v[d][1]), "=r"(v[d][2]), "=r"(v[d][3])
                                 : "r"(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(d * kDgN + col0 + c0)));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int S[kDgAcc];
#pragma unroll
                    for (int d = 0; d < kDgAcc; ++d) S[d] = __float2int_rn(__uint_as_float(v[d][j]));
                    hi[c0 + j] += (long long)S[0] * 16777216 + (long long)S[1] * 65536 + (long long)S[2] * 256 + S[3];
                    lo[c0 + j] += (long long)S[4] * 16777216 + (long long)S[5] * 65536 + (long long)S[6] * 256 + S[7];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_u32(&acc_empty)) : "memory");
        }
        const int row = blockIdx.y * kDgM + q * 32 + lane, n0 = blockIdx.x * kDgN + col0;
        if (EPI == 0) {
            longlong2* o = part + ((size_t)blockIdx.z * mpad + row) * npad + n0;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                longlong2 x = make_longlong2(hi[j], lo[j]);
                if (add) {
                    const longlong2 y = o[j];
                    x.x += y.x;
                    x.y += y.y;
                }
                o[j] = x;
            }
        } else if (row < nplain) {
            const int er = ep[row];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int m = (n0 >> 1) + j;
                if (m >= nexp) break;
                const int em = __ldg(ex + m);
                if (er == kDgFlag || em == kDgFlag) continue;
                double2 r = make_double2(dg_value(hi[2 * j], lo[2 * j], dg_unit(er, em)),
                                         dg_value(hi[2 * j + 1], lo[2 * j + 1], dg_unit(er, em)));
                if (!ok) r.x = r.y = __longlong_as_double(0x7FF8000000000000ll);
                double2* o = C + (size_t)m * ldc + row;
                if (accumulate) {
                    const double2 y = *o;
                    r.x += y.x;
                    r.y += y.y;
                }
                *o = r;
            }
        }
    }
    __syncthreads();
    if (*abort) {
        if (tid == 0 && err) atomicExch(err, 1);
        // the FP64 kernels recompute the tile's rows (an accumulated output holds NaN instead)
        if (tid < kDgM && !(EPI == 1 && accumulate) && (int)blockIdx.y * kDgM + tid < nplain) ep[blockIdx.y * kDgM + tid] = kDgFlag;
        if (tid == 0) *any = 1;
        // drain: copies issued but never consumed
        if (warp == kDgEpiWarps && lane == 0)
            for (int it = s_used; it < s_issued; ++it)
                dg_wait(tc::smem_u32(&full[it % kDgStages]), (it / kDgStages) & 1, nullptr);
    }
    if (warp == kDgEpiWarps + 1 && lane == 0) dg_wait(tc::smem_u32(&done), 0, nullptr);
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == kDgEpiWarps + 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
}

// cn: sum the splits' exact integers and round once: C[m][n]
__global__ void __launch_bounds__(128) k_dg_finish(const longlong2* __restrict__ part, int Z, int mpad, int npad, int M,
                                                   int N, const int* __restrict__ ea, const int* __restrict__ eb,
                                                   double2* __restrict__ C, int ldc) {
    const size_t total = (size_t)M * N;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / N), n = (int)(i - (size_t)m * N);
        const int xa = __ldg(ea + m), xb = __ldg(eb + n);
        if (xa == kDgFlag || xb == kDgFlag) continue;
        long long h0 = 0, l0 = 0, h1 = 0, l1 = 0;
        for (int z = 0; z < Z; ++z) {
            const longlong2* p = part + ((size_t)z * mpad + m) * npad + 2 * n;
            const longlong2 a = p[0], b = p[1];
            h0 += a.x;
            l0 += a.y;
            h1 += b.x;
            l1 += b.y;
        }
        C[(size_t)m * ldc + n] = make_double2(dg_value(h0, l0, dg_unit(xa, xb)), dg_value(h1, l1, dg_unit(xa, xb)));
    }
}

inline int cdiv(long a, long b) { return (int)((a + b - 1) / b); }

// Digit planes held at once: the K panel (cn) or the panel of plain rows (tn) is chosen so that
// they stay below this.  Larger is faster (a launch costs about 11 us of start, fill and partial
// sums, and the planes stream from HBM as well as from L2): 480 x 157 x 18232 takes 692, 654, 532 and
// 487 us with 64, 128, 256 and 512 MB, 1020 x 288 x 95885 9.06, 8.00, 7.41 and 7.12 ms.
constexpr size_t kDgBudget = 512ull << 20;
constexpr int kDgMaxSplits = 160;

struct DgLayout {
    int ptiles, xtiles, nkt;            // plain / expanded row tiles, K tiles of the whole product
    int panel, npanel;                  // cn: K tiles per panel; tn: plain tiles per panel
    int splits;                         // cn
    size_t emax_off, ep_off, ex_off, any_off, part_off, dig_off, total;
};

bool dg_layout_in(bool cn, int nplain, int nexp, int K, size_t budget, size_t* panel_bytes, DgLayout& L) {
    L = DgLayout{};
    L.ptiles = cdiv(nplain, kDgM);
    L.xtiles = cdiv(2L * nexp, kDgN);
    L.nkt = cdiv(2L * K, kDgK);
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t o = off;
        off = align_up(off + b, 256);
        return o;
    };
    L.any_off = take(sizeof(int));
    L.emax_off = take(sizeof(int) * (size_t)kDgSegs * ((size_t)nplain + nexp));
    L.ep_off = take(sizeof(int) * (size_t)nplain);
    L.ex_off = take(sizeof(int) * (size_t)nexp);
    const size_t pb = dg_block(kDgM), xb = dg_block(kDgN);
    if (cn) {
        const size_t per = (size_t)L.ptiles * pb + (size_t)L.xtiles * xb;  // one K tile of both operands
        const long tiles = (long)L.ptiles * L.xtiles, sms = device_sms();
        int most = (int)std::max<size_t>(32, std::min<size_t>(L.nkt, budget / per));
        const size_t fix = (size_t)L.ptiles * kDgM * L.xtiles * kDgN * sizeof(longlong2);
        L.npanel = cdiv(L.nkt, most);
        L.panel = cdiv(L.nkt, L.npanel);
        // splits of a panel: fewest waves of one CTA per SM x (products and drains of a CTA, about
        // 1900 cycles per K tile, + its start and the partial sums' write)
        long best = -1;
        for (int s = 1; s <= std::max(1, std::min(kDgMaxSplits, L.panel / 16)); ++s) {
            const long c = (tiles * s + sms - 1) / sms * (cdiv(L.panel, s) * 1900L + 8000);
            if (best < 0 || c < best) {
                best = c;
                L.splits = s;
            }
        }
        const int per_split = cdiv(L.panel, L.splits);
        L.splits = cdiv(L.panel, per_split);
        L.part_off = take(fix * L.splits);
        L.dig_off = take(*panel_bytes = per * L.panel);
    } else {
        const size_t xbytes = (size_t)L.xtiles * L.nkt * xb, row = (size_t)L.nkt * pb;
        int most = (int)std::max<size_t>(1, std::min<size_t>(L.ptiles, budget / row));
        most = std::min(most, 65535 * 8 / kDgM);
        L.npanel = cdiv(L.ptiles, most);
        L.panel = cdiv(L.ptiles, L.npanel);
        L.splits = 1;
        L.dig_off = take(xbytes + (*panel_bytes = row * L.panel));
    }
    L.total = off;
    // grid limits of the digit and product launches
    if (L.xtiles * (long)kDgN / 8 > 65535 || L.ptiles > 65535L * 8 || L.nkt > 2 * 65535L || (cn && L.ptiles * (long)kDgM / 8 > 65535))
        return false;
    return true;
}
// Panels of at most kDgBudget, smaller where a workspace sized for other shapes (a Davidson's, for its
// largest product) has less room: a product that takes more splits than that one needs more partial sums.
// 528 x 176 x 18232 in the workspace of 704 x 704: 0.6 ms, 10.9 ms on the FP64 kernels.  Splits and panels do
// not change the result (the partial sums are integers).
// `bytes` = 0: as much as the product can use (the layout's total is what to provide)
bool dg_layout(bool cn, int nplain, int nexp, int K, size_t bytes, DgLayout& L) {
    size_t budget = kDgBudget, panel = 0;
    for (int t = 0; t < 8; ++t) {
        if (!dg_layout_in(cn, nplain, nexp, K, budget, &panel, L)) return false;
        if (bytes == 0 || L.total <= bytes) return true;
        const size_t over = L.total - bytes;
        if (over >= panel) return false;
        budget = panel - over;
    }
    return false;
}

// Whether the digit products serve a shape: estimates of both paths' times.  FP64 kernels: 1.1
// TFLOP/s.  Digits: 45 us of launches and starts, the maxima and digit planes at 4 TB/s, then the
// rounds of product tiles over the SMs (1 us per K tile).  Measured on both sides of the line (us,
// FP64 / digits): cn 32 x 32 x 3000
// 38 / 68, 64 x 64 x 1500 59 / 64, 300 x 10 x 3000 117 / 76, 64 x 32 x 6000 99 / 76, 16 x 8 x 97000
// 126 / 314; tn (M x N x K) 16 x 4000 x 64 38 / 54, 48 x 3000 x 48 54 / 55, 32 x 6000 x 64 87 / 58.
bool dg_serves(bool cn, int M, int N, int K) {
    const double np = cn ? M : N, nx = cn ? N : M;
    const long pt = cdiv((long)np, kDgM), xt = cdiv(2 * (long)nx, kDgN), nkt = cdiv(2L * K, kDgK), tiles = pt * xt;
    const double t64 = 8.0 * (cn ? 64.0 * cdiv(M, 8) * cdiv(N, 8) : 256.0 * cdiv(M, 8) * cdiv(N, 32)) * K / 1.1e12;  // their 8 x 8, 8 x 32 tiles
    const double bytes = K * ((np + nx) * 32.0 + 28.0 * (pt * kDgM + xt * kDgN));
    const long split = cn ? std::max<long>(1, std::min<long>({device_sms() / tiles, nkt / 16, (long)kDgMaxSplits})) : 1;
    const double rounds = (double)cdiv(tiles * split, device_sms()) * cdiv(nkt, split);
    return t64 > 45e-6 + bytes / 4e12 + rounds * 1e-6;
}

template <int EPI>
qm_status dg_gemm(const unsigned char* P, const unsigned char* X, int nkt, int splits, int pt, int xt, longlong2* part, int mpad,
                  int npad, bool add, int* ep, const int* ex, int* any, int nplain, int nexp, double2* C, int ldc, bool accumulate,
                  int* err, int polls, cudaStream_t s) {
    const size_t smem = (size_t)kDgStages * (dg_block(kDgM) + dg_block(kDgN));
    const auto kern = polls < kDgSpin ? k_dg_gemm<EPI, true> : k_dg_gemm<EPI, false>;
    qm_status st = allow_dynamic_smem((const void*)kern, smem, "digit products: shared memory");
    if (st) return st;
    ProfScope pf(EPI ? PF_GEMM_TN : PF_GEMM_CN, s);
    kern<<<dim3(xt, pt, splits), kDgThreads, smem, s>>>(P, X, nkt, cdiv(nkt, splits), part, mpad, npad, add ? 1 : 0, ep, ex,
                                                                any, nplain, nexp, C, ldc, accumulate ? 1 : 0, err, polls);
    return cuda_check(cudaGetLastError(), "k_dg_gemm launch");
}

}  // namespace

size_t zdigits_bytes(bool cn, int M, int N, int K) {
    if (!dg_serves(cn, M, N, K)) return 0;
    DgLayout L;
    return dg_layout(cn, cn ? M : N, cn ? N : M, K, 0, L) ? L.total : 0;
}

int zdigits_panels(bool cn, int M, int N, int K, size_t bytes) {
    DgLayout L;
    return dg_serves(cn, M, N, K) && dg_layout(cn, cn ? M : N, cn ? N : M, K, bytes, L) ? L.npanel : 0;
}

// Both return false in *done when the product is left to the FP64 kernels (small, or not enough
// workspace); flags: what the FP64 kernels must recompute (see GemmFlags).
qm_status zdigits_cn(int M, int N, int K, const double2* A, int lda, const double2* B, int ldb, double2* C, int ldc, const GemmWork& w,
                     cudaStream_t s, GemmFlags* flags, bool* done) {
    *done = false;
    DgLayout L;
    if (!w.ptr || !dg_serves(true, M, N, K) || !dg_layout(true, M, N, K, w.bytes, L)) return QM_OK;
    char* base = (char*)w.ptr;
    int *any = (int*)(base + L.any_off), *ma = (int*)(base + L.emax_off), *mb = ma + (size_t)kDgSegs * M;
    int *ea = (int*)(base + L.ep_off), *eb = (int*)(base + L.ex_off);
    longlong2* part = (longlong2*)(base + L.part_off);
    unsigned char* P = (unsigned char*)base + L.dig_off;
    unsigned char* X = P + (size_t)L.ptiles * L.panel * dg_block(kDgM);
    {
        ProfScope pf(PF_SPLIT, s);
        k_dg_rowmax<<<dim3(M, kDgSegs), 256, 0, s>>>(A, lda, M, K, ma, any);
    }
    {
        ProfScope pf(PF_SPLIT, s);
        k_dg_rowmax<<<dim3(N, kDgSegs), 256, 0, s>>>(B, ldb, N, K, mb, nullptr);
    }
    const int mpad = L.ptiles * kDgM, npad = L.xtiles * kDgN, percol = kDgK / 2;
    int Z = 1;
    for (int p = 0; p < L.npanel; ++p) {
        const int t0 = p * L.panel, nkt = std::min(L.panel, L.nkt - t0);
        if (nkt <= 0) break;
        const int c0 = t0 * percol, cols = std::min(nkt * percol, K - c0);
        // every panel uses the first one's splits, so that each partial sum has one place
        const int per = cdiv(L.panel, L.splits), splits = p == 0 ? cdiv(nkt, per) : Z;
        if (p == 0) Z = splits;
        {
            ProfScope pf(PF_SPLIT, s);
            k_dg_rows<<<dim3(cdiv(nkt * 2, 32), mpad / 8), 256, 0, s>>>(A + c0, lda, M, cols, 0, kDgM, nkt, ma, p ? nullptr : ea, any, P);
        }
        {
            ProfScope pf(PF_SPLIT, s);
            k_dg_rows<<<dim3(cdiv(nkt * 2, 32), npad / 8), 256, 0, s>>>(B + c0, ldb, N, cols, 1, kDgN, nkt, mb, p ? nullptr : eb, any, X);
        }
        qm_status st = dg_gemm<0>(P, X, nkt, splits, L.ptiles, L.xtiles, part, mpad, npad, p > 0, ea, eb, any, M, N, nullptr, 0, false,
                                  w.err, p == w.hold_panel ? w.hold_polls : kDgSpin, s);
        if (st) return st;
    }
    {
        ProfScope pf(PF_REDUCE, s);
        k_dg_finish<<<grid_stride_blocks((size_t)M * N, 128, 16), 128, 0, s>>>(part, Z, mpad, npad, M, N, ea, eb, C, ldc);
    }
    *flags = GemmFlags{any, ea, eb, kDgFlag};
    *done = true;
    return cuda_check(cudaGetLastError(), "digit products launch");
}

qm_status zdigits_tn(int M, int N, int K, const double2* A, int lda, const double* d, double alpha, const double2* B, int ldb, double2* C,
                     int ldc, bool accumulate, const GemmWork& w, cudaStream_t s, GemmFlags* flags, bool* done) {
    *done = false;
    DgLayout L;
    if (!w.ptr || !dg_serves(false, M, N, K) || !dg_layout(false, N, M, K, w.bytes, L)) return QM_OK;
    char* base = (char*)w.ptr;
    int *any = (int*)(base + L.any_off), *mb = (int*)(base + L.emax_off), *ma = mb + (size_t)kDgSegs * N;
    int *eb = (int*)(base + L.ep_off), *ea = (int*)(base + L.ex_off);
    unsigned char* X = (unsigned char*)base + L.dig_off;
    unsigned char* P = X + (size_t)L.xtiles * L.nkt * dg_block(kDgN);
    {
        ProfScope pf(PF_SPLIT, s);
        k_dg_colmax<<<dim3(cdiv(N, 256), kDgSegs), 256, 0, s>>>(B, ldb, K, N, nullptr, 1.0, mb, any);
    }
    {
        ProfScope pf(PF_SPLIT, s);
        k_dg_colmax<<<dim3(cdiv(M, 256), kDgSegs), 256, 0, s>>>(A, lda, K, M, d, alpha, ma, nullptr);
    }
    {
        ProfScope pf(PF_SPLIT, s);
        k_dg_cols<<<dim3(L.xtiles, cdiv(L.nkt, 2)), 256, 0, s>>>(A, lda, K, M, d, alpha, 1, kDgN, L.nkt, ma, M, ea, any, X);
    }
    for (int p = 0; p < L.npanel; ++p) {
        const int r0 = p * L.panel * kDgM, pt = std::min(L.panel, L.ptiles - p * L.panel);
        if (pt <= 0) break;
        const int rows = std::min(pt * kDgM, N - r0);
        {
            ProfScope pf(PF_SPLIT, s);
            k_dg_cols<<<dim3(pt * kDgM / 64, cdiv(L.nkt, 2)), 256, 0, s>>>(B + r0, ldb, K, rows, nullptr, 1.0, 0, kDgM, L.nkt, mb + r0,
                                                                        N, eb + r0, any, P);
        }
        qm_status st = dg_gemm<1>(P, X, L.nkt, 1, pt, L.xtiles, nullptr, 0, 0, false, eb + r0, ea, any, rows, M, C + r0, ldc, accumulate,
                                  w.err, p == w.hold_panel ? w.hold_polls : kDgSpin, s);
        if (st) return st;
    }
    *flags = GemmFlags{any, ea, eb, kDgFlag};
    *done = true;
    return cuda_check(cudaGetLastError(), "digit products launch");
}

}  // namespace qm
