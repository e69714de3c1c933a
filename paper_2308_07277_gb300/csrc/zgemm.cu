// Complex GEMMs of the nonlocal projector step (Sec. 2.3, KB form: P = beta^H psi, then
// beta D P) and of the Davidson subspace products (<V_i|H V_j>, rotations by the Ritz
// coefficients, Gram-Schmidt projections).
//
//   cn : C[m][n] = sum_k conj(A[m][k]) B[n][k]                 (k contiguous in A and B)
//        split over K into partial sums reduced in a fixed order (deterministic)
//   tn : C[m][n] = alpha sum_k A[k][m] d[k] B[k][n]  (+ C[m][n])  (m, n contiguous)
//
// FP64: long products as digit products on the tensor cores (zdigits.cu), the others, and the rows those
// leave, on small tiles with one output per thread (k_cn, k_tn; the FP64 pipe bounds them).  FP32: the same
// small tiles for the precision form's small projector products (csmall_*), and register tiles for
// qm_hpsi_noalloc (cgemm_*): 16 x 16 threads per CTA, each owning a TM x TN block of outputs (tile
// 16TM x 16TN), the tile chosen per call so that the M and N edges waste as little as possible (160
// bands -> TM = 5, 256 projectors -> TM = 4); the products of one K tile (16 terms) are summed in FP32 and
// the tile sums in FP64, so the rounding error does not grow with K (inner products over 10^4 - 10^5 plane
// waves keep ~1e-7 relative accuracy).
#include <algorithm>

#include "qm_internal.h"

namespace qm {

namespace {

constexpr int BK = 16, NTH = 256;

template <class C>
__device__ __forceinline__ C czero() {
    C z;
    z.x = 0;
    z.y = 0;
    return z;
}

template <int TM, int TN>
__device__ __forceinline__ void flush_tile(float (&acc)[TM][TN][2], double (&hi)[TM][TN][2]) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                hi[i][j][c] += (double)acc[i][j][c];
                acc[i][j][c] = 0.f;
            }
}

// FP32 products (complex): the products of one K tile are summed in FP32 and the tile
// sums in FP64
template <int TM, int TN>
__global__ void __launch_bounds__(NTH)
k_gemm_cn(int M, int N, int K, const float2* __restrict__ A, int lda, const float2* __restrict__ B, int ldb,
          float2* __restrict__ out, int ldo, int kchunk) {
    constexpr int BM = 16 * TM, BN = 16 * TN;
    __shared__ float2 As[BK][BM + 1];
    __shared__ float2 Bs[BK][BN + 1];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int kb = blockIdx.z * kchunk;
    const int ke = min(K, kb + kchunk);
    float acc[TM][TN][2];
    double hi[TM][TN][2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j][0] = acc[i][j][1] = 0.f, hi[i][j][0] = hi[i][j][1] = 0.0;
    for (int k0 = kb; k0 < ke; k0 += BK) {
        for (int e = tid; e < BM * BK; e += NTH) {
            int row = e / BK, kk = e % BK;
            int gm = m0 + row, gk = k0 + kk;
            As[kk][row] = (gm < M && gk < ke) ? A[(size_t)gm * lda + gk] : czero<float2>();
        }
        for (int e = tid; e < BN * BK; e += NTH) {
            int row = e / BK, kk = e % BK;
            int gn = n0 + row, gk = k0 + kk;
            Bs[kk][row] = (gn < N && gk < ke) ? B[(size_t)gn * ldb + gk] : czero<float2>();
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            float2 a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {  // conj(a) * b
                    acc[i][j][0] = fma(a[i].x, b[j].x, fma(a[i].y, b[j].y, acc[i][j][0]));
                    acc[i][j][1] = fma(a[i].x, b[j].y, fma(-a[i].y, b[j].x, acc[i][j][1]));
                }
        }
        flush_tile<TM, TN>(acc, hi);
        __syncthreads();
    }
    float2* o = out + (size_t)blockIdx.z * M * ldo;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int gm = m0 + ty + 16 * i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            int gn = n0 + tx + 16 * j;
            if (gn < N) o[(size_t)gm * ldo + gn] = make_float2((float)hi[i][j][0], (float)hi[i][j][1]);
        }
    }
}

// kParts threads add the splits of one output (z = part, part + kParts, ...), then each other's sums: few
// outputs with many splits are a chain of dependent loads otherwise (8 x 24 outputs: 2.8 us, 6 us with one)
template <class C, int kParts = 1>
__global__ void k_reduce_splits(int M, int N, const C* __restrict__ part, int splits, C* __restrict__ Cout, int ldc) {
    const size_t total = (size_t)M * N;
    constexpr int kOut = 32 / kParts;  // outputs of a warp
    const int lane = threadIdx.x & 31, q = lane / kOut;
    const size_t warps = (size_t)gridDim.x * (blockDim.x >> 5);
    for (size_t i0 = (blockIdx.x * (size_t)(blockDim.x >> 5) + (threadIdx.x >> 5)) * kOut; i0 < total; i0 += warps * kOut) {
        const size_t i = i0 + lane % kOut;
        C s = czero<C>();
        if (i < total)
#pragma unroll 4
            for (int z = q; z < splits; z += kParts) {
                C v = part[(size_t)z * total + i];
                s.x += v.x;
                s.y += v.y;
            }
#pragma unroll
        for (int o = kOut; o < 32; o <<= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (i < total && q == 0) Cout[(size_t)(i / N) * ldc + i % N] = s;
    }
}

template <int TM, int TN>
__global__ void __launch_bounds__(NTH)
k_gemm_tn(int M, int N, int K, const float2* __restrict__ A, int lda, const double* __restrict__ d, double alpha,
          const float2* __restrict__ B, int ldb, float2* __restrict__ Cm, int ldc, int accumulate) {
    constexpr int BM = 16 * TM, BN = 16 * TN;
    __shared__ float2 As[BK][BM + 1];
    __shared__ float2 Bs[BK][BN + 1];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    float acc[TM][TN][2];
    double hi[TM][TN][2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j][0] = acc[i][j][1] = 0.f, hi[i][j][0] = hi[i][j][1] = 0.0;
    for (int k0 = 0; k0 < K; k0 += BK) {
        for (int e = tid; e < BM * BK; e += NTH) {
            int kk = e / BM, col = e % BM;
            int gk = k0 + kk, gm = m0 + col;
            float2 v = czero<float2>();
            if (gk < K && gm < M) {
                v = A[(size_t)gk * lda + gm];
                const float sc = (float)(d ? alpha * d[gk] : alpha);
                v.x *= sc;
                v.y *= sc;
            }
            As[kk][col] = v;
        }
        for (int e = tid; e < BN * BK; e += NTH) {
            int kk = e / BN, col = e % BN;
            int gk = k0 + kk, gn = n0 + col;
            Bs[kk][col] = (gk < K && gn < N) ? B[(size_t)gk * ldb + gn] : czero<float2>();
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            float2 a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    acc[i][j][0] = fma(a[i].x, b[j].x, fma(-a[i].y, b[j].y, acc[i][j][0]));
                    acc[i][j][1] = fma(a[i].x, b[j].y, fma(a[i].y, b[j].x, acc[i][j][1]));
                }
        }
        flush_tile<TM, TN>(acc, hi);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int gm = m0 + ty + 16 * i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            int gn = n0 + tx + 16 * j;
            if (gn < N) {
                float2* p = Cm + (size_t)gm * ldc + gn;
                float2 v = make_float2((float)hi[i][j][0], (float)hi[i][j][1]);
                if (accumulate) {
                    const float2 o = *p;
                    v.x += o.x;
                    v.y += o.y;
                }
                *p = v;
            }
        }
    }
}

// ---------------------------------------------------------------- FP64
// FP64 multiply-adds issue at two lanes per clock per SM here (a warp instruction takes 16
// cycles), so an FP64 product is bound by that pipe whatever the operands cost: one output per
// thread with both factors read from shared memory for every term (two 128-bit loads beside four
// multiply-adds) keeps the pipe full, and what counts is that no lane works on padding and that
// every SM gets a share.  Tiles are therefore small (8 x 8 with four K groups for cn, 8 x 32 for
// tn) and cn is split over K until the CTAs fill the SMs.  The register-tiled 80 x 80 ... 32 x 32
// tiles these replace padded 8 bands to 32 and ran a small product on one SM: 900 us for a 32 x 8
// product of 1060 terms, 85 % of the self-consistency of an 8-atom cell.  Measured: that run's first
// two steps 1249 -> 164 ms, H psi of the two-atom cell (8 x 8 x 411) 518 -> 65 us, and at large
// sizes 1.22 instead of 1.01 TFLOP/s (480 x 157 x 18232, 10.9 -> 9.0 ms).
constexpr int kCnTile = 8, kCnK = 32, kCnGroups = 4;
// hi + lo <- hi + lo + a, hi the rounded sum (the error of the addition by Knuth's two-sum goes to lo)
__device__ __forceinline__ void add_comp(float& hi, float& lo, float a) {
    const float s = hi + a, t = s - hi;
    lo += (hi - (s - t)) + (a - t);
    hi = s;
}
template <class C>
__global__ void __launch_bounds__(NTH)
k_cn(int M, int N, int K, const C* __restrict__ A, int lda, const C* __restrict__ B, int ldb, C* __restrict__ out, int ldo, int kchunk, const GemmFlags f) {
    if (f.any && !*f.any) return;
    __shared__ C As[kCnK][kCnTile + 1], Bs[kCnK][kCnTile + 1];
    const int tid = threadIdx.x, tx = tid & 7, ty = (tid >> 3) & 7, kg = tid >> 6;
    const int m0 = blockIdx.y * kCnTile, n0 = blockIdx.x * kCnTile;
    const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
    const int lrow = tid / kCnK, lk = tid % kCnK;  // this thread's element of a tile (one row per warp)
    C acc = czero<C>(), hi = acc, lo = acc;
    const bool va = m0 + lrow < M, vb = n0 + lrow < N;
    const C* pa = A + (size_t)(va ? m0 + lrow : 0) * lda + lk;
    const C* pb = B + (size_t)(vb ? n0 + lrow : 0) * ldb + lk;
    C ra = czero<C>(), rb = ra;
    if (kb + lk < ke) {
        if (va) ra = pa[kb];
        if (vb) rb = pb[kb];
    }
    for (int k0 = kb; k0 < ke; k0 += kCnK) {
        As[lk][lrow] = ra;
        Bs[lk][lrow] = rb;
        __syncthreads();
        ra = rb = czero<C>();
        if (k0 + kCnK + lk < ke) {  // the next tile's loads are in flight during this tile's products
            if (va) ra = pa[k0 + kCnK];
            if (vb) rb = pb[k0 + kCnK];
        }
#pragma unroll
        for (int q = 0; q < kCnK / kCnGroups; ++q) {
            const C a = As[kg + kCnGroups * q][ty], b = Bs[kg + kCnGroups * q][tx];
            acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
            acc.y = fma(a.x, b.y, fma(-a.y, b.x, acc.y));
        }
        if constexpr (sizeof(C) == sizeof(float2)) {  // the tiles' sums compensated: K / 32 of them without their rounding
            add_comp(hi.x, lo.x, acc.x);
            add_comp(hi.y, lo.y, acc.y);
            acc = czero<C>();
        }
        __syncthreads();
    }
    if constexpr (sizeof(C) == sizeof(float2)) {
        acc.x = hi.x + lo.x;
        acc.y = hi.y + lo.y;
    }
    C* red = &As[0][0];  // 3 x 64 partial sums of the K groups, added in group order
    if (kg) red[(kg - 1) * 64 + ty * 8 + tx] = acc;
    __syncthreads();
    if (kg == 0 && m0 + ty < M && n0 + tx < N && (!f.any || f.em[m0 + ty] == f.flag || f.en[n0 + tx] == f.flag)) {
        for (int g = 0; g < kCnGroups - 1; ++g) {
            const C v = red[g * 64 + ty * 8 + tx];
            acc.x += v.x;
            acc.y += v.y;
        }
        out[((size_t)blockIdx.z * M + m0 + ty) * ldo + n0 + tx] = acc;
    }
}

constexpr int kTnN = 32, kTnK = 16;
template <class T, int kTnM>  // a warp per row
__global__ void __launch_bounds__(32 * kTnM)
k_tn(int M, int N, int K, const T* __restrict__ A, int lda, const double* __restrict__ d, double alpha,
     const T* __restrict__ B, int ldb, T* __restrict__ C, int ldc, int accumulate, const GemmFlags f) {
    if (f.any && !*f.any) return;
    __shared__ T As[kTnK][kTnM], Bs[kTnK][kTnN];
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int n0 = blockIdx.x * kTnN, m0 = blockIdx.y * kTnM;
    T acc = czero<T>();
    for (int k0 = 0; k0 < K; k0 += kTnK) {
        if (tid < kTnK * kTnM) {
            const int kk = tid / kTnM, m = m0 + tid % kTnM, k = k0 + kk;
            T v = czero<T>();
            if (k < K && m < M) {
                v = A[(size_t)k * lda + m];
                const auto sc = (decltype(v.x))(d ? alpha * d[k] : alpha);
                v.x *= sc;
                v.y *= sc;
            }
            As[kk][tid % kTnM] = v;
        }
#pragma unroll
        for (int q = 0; q < kTnK / kTnM; ++q) {
            const int kk = ty + q * kTnM, k = k0 + kk, n = n0 + tx;
            Bs[kk][tx] = (k < K && n < N) ? B[(size_t)k * ldb + n] : czero<T>();
        }
        __syncthreads();
        const int kn = m0 + ty < M ? min(kTnK, K - k0) : 0;  // (warps past the last row leave the FP64 pipe alone)
        for (int kk = 0; kk < kn; ++kk) {
            const T a = As[kk][ty], b = Bs[kk][tx];
            acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
            acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
        }
        __syncthreads();
    }
    const int m = m0 + ty, n = n0 + tx;
    if (m < M && n < N && (!f.any || f.em[m] == f.flag || f.en[n] == f.flag)) {
        T* p = C + (size_t)m * ldc + n;
        if (accumulate) {
            const T o = *p;
            acc.x += o.x;
            acc.y += o.y;
        }
        *p = acc;
    }
}

// Splits of cn over K: the count that minimises (waves of one CTA per SM) x (cycles per CTA) plus
// the reduction of the partial sums, 128 pipe cycles per term of an 8 x 8 tile in FP64, about 12 in FP32; the fixed costs
// (1500 cycles of start and loads, 4000 of the second launch) are estimates of launch latency.
int zcn_splits(int M, int N, int K, long cap, int per_term = 128) {
    const long tiles = (long)((M + kCnTile - 1) / kCnTile) * ((N + kCnTile - 1) / kCnTile), sms = device_sms();
    const int smax = (int)std::max<long>(1, std::min<long>({(long)((K + kCnK - 1) / kCnK), cap, 64L}));
    int best = 1;
    long cost = -1;
    for (int s = 1; s <= smax; ++s) {
        const long kc = ((K + s - 1) / s + kCnK - 1) / kCnK * kCnK;
        const long c = (tiles * s + sms - 1) / sms * (kc * per_term + 1500) + (s > 1 ? 4000 + 40L * s : 0);
        if (cost < 0 || c < cost) {
            cost = c;
            best = s;
        }
    }
    return best;
}

// a launch's row tiles are its y blocks, at most 65535: more rows take several launches
constexpr int kMaxRowTiles = 65535;
GemmFlags flags_from(GemmFlags f, int row) {
    if (f.em) f.em += row;
    return f;
}

template <class T>
qm_status cn_small(int M, int N, int K, const T* A, int lda, const T* B, int ldb, T* C, int ldc, T* partial, size_t partial_bytes, const GemmFlags& f, cudaStream_t s) {
    constexpr int most = kMaxRowTiles * kCnTile;
    if (M > most) {
        qm_status st = cn_small(most, N, K, A, lda, B, ldb, C, ldc, partial, partial_bytes, f, s);
        return st ? st : cn_small(M - most, N, K, A + (size_t)most * lda, lda, B, ldb, C + (size_t)most * ldc, ldc, partial,
                                  partial_bytes, flags_from(f, most), s);
    }
    const long cap = partial ? (long)(partial_bytes / sizeof(T)) / ((long)M * N) : 1;
    int splits = zcn_splits(M, N, K, std::max<long>(1, cap), sizeof(T) == 8 ? 12 : 128);
    int kchunk = std::max(kCnK, ((K + splits - 1) / splits + kCnK - 1) / kCnK * kCnK);
    splits = std::max(1, (K + kchunk - 1) / kchunk);
    const dim3 grid((N + kCnTile - 1) / kCnTile, (M + kCnTile - 1) / kCnTile, splits);
    {
        ProfScope pf(PF_GEMM_CN, s);
        k_cn<T><<<grid, NTH, 0, s>>>(M, N, K, A, lda, B, ldb, splits > 1 ? partial : C, splits > 1 ? N : ldc, kchunk, f);
    }
    if (splits > 1) {
        ProfScope pf(PF_REDUCE, s);
        k_reduce_splits<T, 8><<<grid_stride_blocks((size_t)M * N, 8, 16), 64, 0, s>>>(M, N, partial, splits, C, ldc);
    }
    return cuda_check(cudaGetLastError(), "gemm_cn launch");
}

template <class T>
qm_status tn_small(int M, int N, int K, const T* A, int lda, const double* d, double alpha, const T* B, int ldb, T* C,
                   int ldc, bool accumulate, const GemmFlags& f, cudaStream_t s) {
    // Rows per CTA, 8 or 4, in FP64: a warp's FP64 instruction holds one of the SM's four partitions, so eight
    // rows take twice the time of four and are worth it only where the tiles fill the SMs that often anyway
    // (8 x 1500 outputs, K up to 32: 5.2 us with 4 rows on 94 SMs, 6.9 us with 8 on 47)
    const auto tiles = [&](int rows) { return (long)((N + kTnN - 1) / kTnN) * ((M + rows - 1) / rows); };
    const long sms = device_sms(), load8 = (tiles(8) + sms - 1) / sms * 2, load4 = (tiles(4) + sms - 1) / sms;
    const int rows = sizeof(T) == sizeof(double2) && load4 < load8 ? 4 : 8;
    if (M > kMaxRowTiles * rows) {
        const int most = kMaxRowTiles * rows;
        qm_status st = tn_small(most, N, K, A, lda, d, alpha, B, ldb, C, ldc, accumulate, f, s);
        return st ? st : tn_small(M - most, N, K, A + most, lda, d, alpha, B, ldb, C + (size_t)most * ldc, ldc, accumulate,
                                  flags_from(f, most), s);
    }
    const dim3 grid((N + kTnN - 1) / kTnN, (M + rows - 1) / rows);
    ProfScope pf(PF_GEMM_TN, s);
    if (rows == 4) k_tn<T, 4><<<grid, 128, 0, s>>>(M, N, K, A, lda, d, alpha, B, ldb, C, ldc, accumulate ? 1 : 0, f);
    else k_tn<T, 8><<<grid, 256, 0, s>>>(M, N, K, A, lda, d, alpha, B, ldb, C, ldc, accumulate ? 1 : 0, f);
    return cuda_check(cudaGetLastError(), "gemm_tn launch");
}

// thread-tile size for one dimension: the T in {5, 4, 2} (BM = 16 T) that pads n least
int pick_t(int n) {
    int best = 4;
    long bestpad = 1L << 60;
    for (int t : {5, 4, 2}) {
        long b = 16L * t;
        long pad = (n + b - 1) / b * b;
        if (pad < bestpad) {
            bestpad = pad;
            best = t;
        }
    }
    return best;
}

constexpr int kMaxSlots = 4 * 152;

// resident CTAs of a kernel on the current device (occupancy x SM count), cached per kernel
template <class F>
int resident_slots(F* kernel) {
    static thread_local int cached = 0;
    if (cached) return cached;
    int dev = 0, sms = 152, occ = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, NTH, 0) != cudaSuccess || occ < 1) occ = 1;
    cached = std::min(kMaxSlots, occ * sms);
    return cached;
}

template <int TM, int TN>
qm_status cn_launch(int M, int N, int K, const float2* A, int lda, const float2* B, int ldb, float2* Cm, int ldc, float2* partial,
                    int max_splits, cudaStream_t s) {
    constexpr int BM = 16 * TM, BN = 16 * TN;
    const int tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    const int kSlots = resident_slots(k_gemm_cn<TM, TN>);
    // splits: each at least 128 deep, within the caller's partial-sum buffer (max_splits, and
    // the size gemm_cn_partial_bytes guarantees), chosen so that the CTAs fill the resident
    // slots in nearly whole waves: the fewest splits whose last wave is not more than 10 %
    // emptier than the best choice (a grid of 160 tiles on 304 slots otherwise leaves half
    // of them idle)
    const long cap = (long)(gemm_cn_partial_bytes(true) / sizeof(float2)) / std::max<long>(1, (long)M * N);
    const int smax = (int)std::max<long>(1, std::min<long>({(long)std::max(1, K / 128), (long)max_splits, cap, 64L}));
    auto fill = [&](int sp) {
        const long ctas = (long)tiles * sp, waves = (ctas + kSlots - 1) / kSlots;
        return (double)ctas / (double)(waves * kSlots);
    };
    double best = 0.0;
    for (int sp = 1; sp <= smax; ++sp) best = std::max(best, fill(sp));
    int splits = 1;
    while (splits < smax && fill(splits) < best - 0.1) ++splits;
    if (!partial) splits = 1;
    int kchunk = (K + splits - 1) / splits;
    kchunk = std::max(BK, (kchunk + BK - 1) / BK * BK);
    splits = std::max(1, (K + kchunk - 1) / kchunk);
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, splits);
    if (splits == 1) {
        ProfScope pf(PF_GEMM_CN, s);
        k_gemm_cn<TM, TN><<<grid, NTH, 0, s>>>(M, N, K, A, lda, B, ldb, Cm, ldc, kchunk);
    } else {
        {
            ProfScope pf(PF_GEMM_CN, s);
            k_gemm_cn<TM, TN><<<grid, NTH, 0, s>>>(M, N, K, A, lda, B, ldb, partial, N, kchunk);
        }
        size_t total = (size_t)M * N;
        const int blocks = grid_stride_blocks(total, 256, 8);
        ProfScope pf(PF_REDUCE, s);
        k_reduce_splits<float2><<<blocks, 256, 0, s>>>(M, N, partial, splits, Cm, ldc);
    }
    return cuda_check(cudaGetLastError(), "gemm_cn launch");
}

qm_status gemm_cn_impl(int M, int N, int K, const float2* A, int lda, const float2* B, int ldb, float2* Cm, int ldc,
                       float2* partial, int max_splits, cudaStream_t s) {
    if (M <= 0 || N <= 0) return QM_OK;
    const int tm = pick_t(M), tn = pick_t(N);
#define QM_CN(a, b) \
if (tm == a && tn == b) return cn_launch<a, b>(M, N, K, A, lda, B, ldb, Cm, ldc, partial, max_splits, s);
    QM_CN(5, 5) QM_CN(5, 4) QM_CN(4, 5) QM_CN(4, 4) QM_CN(2, 4) QM_CN(4, 2) QM_CN(2, 5) QM_CN(5, 2) QM_CN(2, 2)
#undef QM_CN
    return fail(QM_ERR_UNSUPPORTED, "gemm_cn: no tile");
}

template <int TM, int TN>
qm_status tn_launch(int M, int N, int K, const float2* A, int lda, const double* d, double alpha, const float2* B, int ldb,
                    float2* Cm, int ldc, bool accumulate, cudaStream_t s) {
    constexpr int BM = 16 * TM, BN = 16 * TN;
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, 1);
    ProfScope pf(PF_GEMM_TN, s);
    k_gemm_tn<TM, TN><<<grid, NTH, 0, s>>>(M, N, K, A, lda, d, alpha, B, ldb, Cm, ldc, accumulate ? 1 : 0);
    return cuda_check(cudaGetLastError(), "gemm_tn launch");
}

qm_status gemm_tn_impl(int M, int N, int K, const float2* A, int lda, const double* d, double alpha, const float2* B,
                       int ldb, float2* Cm, int ldc, bool accumulate, cudaStream_t s) {
    if (M <= 0 || N <= 0) return QM_OK;
    const int tm = pick_t(M);
    // the N dimension (plane waves) is long: TN = 4 keeps 256-wide rows of whole tiles
#define QM_TN(a) \
if (tm == a) return tn_launch<a, 4>(M, N, K, A, lda, d, alpha, B, ldb, Cm, ldc, accumulate, s);
    QM_TN(5) QM_TN(4) QM_TN(2)
#undef QM_TN
    return fail(QM_ERR_UNSUPPORTED, "gemm_tn: no tile");
}

}  // namespace

size_t gemm_cn_partial_bytes(bool fp32) {
    // splits * tiles <= resident slots, so splits * M * N <= kMaxSlots * (80 x 80 largest tile)
    return (size_t)kMaxSlots * 80 * 80 * (fp32 ? sizeof(float2) : sizeof(double2));
}

int zgemm_cn_splits(int K) { return std::max(1, std::min(64, (K + kCnK - 1) / kCnK)); }

size_t zgemm_cn_bytes(int M, int N, int K, bool digits) {
    if (M <= 0 || N <= 0) return 0;
    const int splits = zcn_splits(M, N, K, 64);
    return std::max(digits ? zdigits_bytes(true, M, N, K) : 0, splits > 1 ? (size_t)splits * M * N * sizeof(double2) : 0);
}
size_t zgemm_tn_bytes(int M, int N, int K, bool digits) { return M <= 0 || N <= 0 || !digits ? 0 : zdigits_bytes(false, M, N, K); }

size_t zgemm_lean_bytes(size_t bytes) { return std::min(bytes, gemm_cn_partial_bytes(false)); }

qm_status zgemm_cn(int M, int N, int K, const double2* A, int lda, const double2* B, int ldb, double2* C, int ldc,
                   const GemmWork& w, cudaStream_t s) {
    if (M <= 0 || N <= 0) return QM_OK;
    GemmFlags f{};
    bool done = false;
    qm_status st = w.digits ? zdigits_cn(M, N, K, A, lda, B, ldb, C, ldc, w, s, &f, &done) : QM_OK;
    if (st) return st;
    return done ? cn_small(M, N, K, A, lda, B, ldb, C, ldc, (double2*)nullptr, 0, f, s)
                : cn_small(M, N, K, A, lda, B, ldb, C, ldc, (double2*)w.ptr, w.bytes, f, s);
}
qm_status zgemm_tn(int M, int N, int K, const double2* A, int lda, const double* d, const double2* B, int ldb,
                   double2* C, int ldc, bool accumulate, const GemmWork& w, cudaStream_t s, double alpha) {
    if (M <= 0 || N <= 0) return QM_OK;
    GemmFlags f{};
    bool done = false;
    qm_status st = w.digits ? zdigits_tn(M, N, K, A, lda, d, alpha, B, ldb, C, ldc, accumulate, w, s, &f, &done) : QM_OK;
    if (st) return st;
    return tn_small(M, N, K, A, lda, d, alpha, B, ldb, C, ldc, accumulate, f, s);
}
// FP32 products on the same small tiles (the precision form's nonlocal part of small cells).  cn: chains of eight
// multiply-adds per thread, the sums of K / 32 of them compensated, then four groups and at most 64 splits in FP32;
// without the compensation a split of several hundred terms showed (8 x 200 x 401: 4.86e-8 of H psi, now 4.54e-8).
// tn: one chain of K multiply-adds
size_t csmall_cn_bytes(int M, int N, int K) {
    const int splits = zcn_splits(M, N, K, 64, 12);
    return splits > 1 ? (size_t)splits * M * N * sizeof(float2) : 0;
}
qm_status csmall_cn(int M, int N, int K, const float2* A, int lda, const float2* B, int ldb, float2* C, int ldc,
                    const GemmWork& w, cudaStream_t s) {
    return cn_small(M, N, K, A, lda, B, ldb, C, ldc, (float2*)w.ptr, w.bytes, GemmFlags{}, s);
}
qm_status csmall_tn(int M, int N, int K, const float2* A, int lda, const double* d, const float2* B, int ldb, float2* C,
                    int ldc, cudaStream_t s) {
    return tn_small(M, N, K, A, lda, d, 1.0, B, ldb, C, ldc, true, GemmFlags{}, s);
}
qm_status cgemm_cn(int M, int N, int K, const float2* A, int lda, const float2* B, int ldb, float2* C, int ldc,
                   float2* partial, int splits, cudaStream_t s) {
    return gemm_cn_impl(M, N, K, A, lda, B, ldb, C, ldc, partial, splits, s);
}
qm_status cgemm_tn(int M, int N, int K, const float2* A, int lda, const double* d, const float2* B, int ldb,
                   float2* C, int ldc, bool accumulate, cudaStream_t s, double alpha) {
    return gemm_tn_impl(M, N, K, A, lda, d, alpha, B, ldb, C, ldc, accumulate, s);
}

}  // namespace qm

using namespace qm;

static qm_status check_zgemm(int op, int M, int N, int K, const void* A, int lda, const void* B, int ldb, const void* C,
                             int ldc) {
    if (M < 1 || N < 1 || K < 1 || !A || !B || !C) return fail(QM_ERR_ARG, "qm_zgemm: bad sizes or NULL operand");
    if (op == 0 ? (lda < K || ldb < K || ldc < N) : (lda < M || ldb < N || ldc < N))
        return fail(QM_ERR_ARG, "qm_zgemm: leading dimension too small");
    return QM_OK;
}

extern "C" qm_status qm_zgemm(int op, int arith, int M, int N, int K, const void* A, int lda, const void* B, int ldb,
                              void* C, int ldc, void* stream) {
    clear_error();
    if ((op != 0 && op != 1) || arith < 0 || arith > 3) return fail(QM_ERR_ARG, "qm_zgemm: op not 0/1 or arith not 0..2 or 3");
    if (qm_status st = check_zgemm(op, M, N, K, A, lda, B, ldb, C, ldc)) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const double2* a = (const double2*)A;
    const double2* b = (const double2*)B;
    double2* c = (double2*)C;
    if (arith == 2) {  // BF16x3 split products on the tensor cores (the Davidson's FP32 phase)
        const size_t wbytes = op == 0 ? subspace_bf16x3_bytes(M, N)
                                      : std::max(subspace_bf16x3_bytes(M, 1), (size_t)M * K * sizeof(float2));
        void* work = nullptr;
        int* err = nullptr;
        if (cudaMallocAsync(&work, wbytes, s) != cudaSuccess || cudaMallocAsync((void**)&err, sizeof(int), s) != cudaSuccess) {
            cudaGetLastError();
            if (work) cudaFreeAsync(work, s);
            return fail(QM_ERR_OOM, "qm_zgemm: tensor-core workspace");
        }
        qm_status st = cuda_check(cudaMemsetAsync(err, 0, sizeof(int), s), "memset");
        if (!st)
            st = op == 0 ? zgemm_cn_bf16x3(M, N, K, a, lda, b, ldb, c, ldc, work, wbytes, err, s)
                         : zgemm_tn_bf16x3(M, N, K, a, lda, b, ldb, c, ldc, false, 1.0, work, wbytes, err, s);
        int e = 0;
        if (!st) st = cuda_check(cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, s), "D2H error word");
        if (!st) st = cuda_check(cudaStreamSynchronize(s), "stream sync");
        cudaFreeAsync(work, s);
        cudaFreeAsync(err, s);
        if (!st && e) st = fail(QM_ERR_TIMEOUT, "qm_zgemm: a bounded tensor-core wait expired");
        return st;
    }
    GemmWork w;
    w.digits = arith != 3;
    w.bytes = op == 0 ? zgemm_cn_bytes(M, N, K, w.digits) : zgemm_tn_bytes(M, N, K, w.digits);
    if (w.bytes && cudaMallocAsync(&w.ptr, w.bytes, s) != cudaSuccess) {
        cudaGetLastError();
        w.ptr = nullptr;
        w.bytes = zgemm_lean_bytes(w.bytes);
        if (cudaMallocAsync(&w.ptr, w.bytes, s) != cudaSuccess) {
            cudaGetLastError();
            return fail(QM_ERR_OOM, "qm_zgemm: workspace");
        }
    }
    qm_status st = op == 0 ? zgemm_cn(M, N, K, a, lda, b, ldb, c, ldc, w, s)
                           : zgemm_tn(M, N, K, a, lda, nullptr, b, ldb, c, ldc, false, w, s, 1.0);
    if (w.ptr) cudaFreeAsync(w.ptr, s);
    return st;
}

extern "C" qm_status qm_zgemm_hold(int op, int M, int N, int K, const void* A, int lda, const void* B, int ldb, void* C,
                                   int ldc, size_t scratch, int panel, long long polls, int* panels, void* stream) {
    clear_error();
    if (op != 0 && op != 1) return fail(QM_ERR_ARG, "qm_zgemm_hold: op not 0/1");
    if (panel < -1 || polls < 0 || !panels) return fail(QM_ERR_ARG, "qm_zgemm_hold: bad panel or polls, or NULL panels");
    qm_status st = check_zgemm(op, M, N, K, A, lda, B, ldb, C, ldc);
    if (st) return st;
    *panels = 0;
    cudaStream_t s = (cudaStream_t)stream;
    GemmWork w;
    w.bytes = scratch;
    w.hold_panel = panel;
    w.hold_polls = (int)std::min<long long>(polls, 1 << 26);
    if (scratch && (st = cuda_check(cudaMallocAsync(&w.ptr, scratch, s), "qm_zgemm_hold: workspace"))) return st;
    if (scratch) *panels = zdigits_panels(op == 0, M, N, K, scratch);
    st = op == 0 ? zgemm_cn(M, N, K, (const double2*)A, lda, (const double2*)B, ldb, (double2*)C, ldc, w, s)
                 : zgemm_tn(M, N, K, (const double2*)A, lda, nullptr, (const double2*)B, ldb, (double2*)C, ldc, false, w, s, 1.0);
    if (w.ptr) cudaFreeAsync(w.ptr, s);
    return st;
}
