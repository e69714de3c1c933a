// Nonlocal part of the precision form on the tensor cores: the projection P = beta^H psi and
// the application beta (D P) of the Kleinman-Bylander term (Sec. 2.3) as split products of FP16
// pairs accumulated in FP32 (tcgen05, accumulators in tensor memory).
//
// Splitting: every operand row is scaled by a power of two that brings its largest component to
// [2^14, 2^15), and a scaled value x is written x = x0 + x1 with x0 = fp16(x), x1 = fp16(x - x0):
// 23 significant bits (a quarter of the values lose the last bit of their 24, 2^-24 rms) down to
// 2^-17 of the row's largest, an absolute error of 2^-40 of it below.  A product keeps x0 y0 + x0 y1 +
// x1 y0 (x1 y1 is 2^-24.6 rms of the product).  Three BF16 pieces hold all 24 bits but take six
// products; what limits the result is neither, it is the accumulation: the tensor core truncates
// every sum it adds to an accumulator, 12 sums per 32 terms with six products, 6 with three (and
// the projection's K is split twice as often).  Measured error of H psi against 64 bits, six BF16
// products / these: 3.5e-6 / 1.4e-6 (255 atoms), 5.3e-6 / 2.2e-6 (216 atoms), 3.1e-7 / 1.5e-7 (64 atoms),
// 8.9e-8 / 8.0e-8 (32 atoms).  With fewer projectors the six were ahead: 7.4e-8 / 9.1e-8 with 32 of them (1060
// plane waves, 56 to 90 bands; FP32 arithmetic 4.6e-8).  Up to kFewProj projectors the two small products
// therefore go to accumulators of their own, so that the large one is truncated once per K tile instead of three
// times, and both are added in the epilogue: 5.7e-8.  It halves the error of larger ones too, but doubles the tensor
// memory and the drain (propagation step of 32 atoms 1046 -> 1066 us), and their error is below the six
// products' as it is.  (x1 y1 as a fourth product on top: 5.6e-8, no difference.)  Up to 16 projectors the 23 bits
// themselves show beside the FFT path's error (4.95e-8, six products 4.77e-8): hpsi.cu keeps those in FP32.
//
// Operands are split ONCE into FP16 planes stored in global memory in a tile-blocked order:
// block (row tile, K tile) holds, for both planes, the R x 16 tile in the canonical no-swizzle
// K-major shared-memory layout of the tensor core (8-row x 16-byte core matrices; element (r, k) at
// ((r/8)*2 + k/8)*128 + (r%8)*16 + (k%8)*2).  A K tile of one operand is therefore one contiguous
// run of 64 R bytes, which a single bulk copy (cp.async.bulk, completion counted on an mbarrier)
// lands in shared memory ready for the MMA.
//
// Complex products as real GEMMs over K' = 2K (re, im interleaved or (p, u) pairs):
//   projection  C[p][2b+t] = sum_(g,u) betaK[p][(g,u)] psiX[2b+t][(g,u)]
//               betaK = beta as stored (K = (g, u) interleaved), psiX row 2b = psi_b as stored,
//               row 2b+1 = (im, -re) of psi_b, so C[p][2b] = Re<beta_p|psi_b>, C[p][2b+1] = Im.
//   application C[2b+t][g] = sum_(p,u) E[2b+t][(p,u)] betaT[g][(p,u)]
//               betaT[g][(p,u)] = component u of beta[p][g] (beta transposed, not expanded),
//               E = D P expanded: E[2b][(p,0)] = ar, E[2b][(p,1)] = -ai, E[2b+1][(p,0)] = ai,
//               E[2b+1][(p,1)] = ar (a = D_p P[p][b]), so C[2b][g] = Re(beta D P)[b][g], C[2b+1] = Im.
//
// GEMM kernel (k_nl_gemm): one CTA per (128 or 256 rows of A, N tile of BN <= 256, K range): one or two
// M = 128 accumulators side by side in tensor memory.  A 128-row CTA would read 48 KB of operands per 768
// tensor cycles, more than L2 delivers to 152 SMs at once (48 bytes per clock and SM are what the
// six-product kernel drew at 0.94 of the tensor peak); 256 rows need 43.  Where that
// leaves SMs without work the tiles shrink (gemm_shape).  Twelve warps: warp 0 issues
// the bulk copies into a ring of kNlStages stages of one K tile, one thread of warp 1 issues the
// 3 or 6 tcgen05.mma of a K tile (M = 128, N = BN, K = 16) and commits the stage back to the producer,
// warps 4-11 drain the accumulators.  Every mbarrier wait is bounded: on expiry the kernel sets the
// error word, waits (bounded) for its own copies and products in flight, frees its tensor memory and
// returns.
#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>

#include "qm_internal.h"
#include "tc_util.cuh"

namespace qm {
namespace {

constexpr int KT = 16;          // K tile (real elements): 2 chunks of 8 FP16
constexpr int TM = 128;         // rows of an A tile (M of the MMA)
constexpr int kNlStages = 4;    // K tiles in flight: at most 128 KB, which leaves room for an FFT CTA (77 to 87 KB) on the SM
constexpr int kGemmThreads = 384;
constexpr int kNlSegs = 8;      // partial maxima per row
constexpr long kSpin = 1L << 26;

__host__ __device__ constexpr size_t plane_bytes(int R) { return (size_t)R * KT * 2; }
__host__ __device__ constexpr size_t block_bytes(int R) { return 2 * plane_bytes(R); }

// byte offset of element (r, k) inside one plane of a tile
__device__ __forceinline__ int cm_off(int r, int k) {
    return ((((r >> 3) << 1) + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1);
}

// split two scaled FP32 values into their FP16 components, packed in pairs
__device__ __forceinline__ void split2(float x, float y, uint32_t& c0, uint32_t& c1) {
    const __half2 h = __floats2half2_rn(x, y);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
    c0 = *reinterpret_cast<const uint32_t*>(&h);
    c1 = *reinterpret_cast<const uint32_t*>(&l);
}

// write the 8 consecutive K values v[0..7], scaled by sc, of row r (k0 a multiple of 8) into the blocked array
__device__ __forceinline__ void put8(unsigned char* blk, int R, int nkt, int r, int k0, const float* v, float sc) {
    const int rt = r / R, rr = r - rt * R, kt = k0 / KT, kk = k0 - kt * KT;
    unsigned char* p = blk + ((size_t)rt * nkt + kt) * block_bytes(R) + cm_off(rr, kk);
    uint4 c[2];
    split2(v[0] * sc, v[1] * sc, c[0].x, c[1].x);
    split2(v[2] * sc, v[3] * sc, c[0].y, c[1].y);
    split2(v[4] * sc, v[5] * sc, c[0].z, c[1].z);
    split2(v[6] * sc, v[7] * sc, c[0].w, c[1].w);
#pragma unroll
    for (int q = 0; q < 2; ++q) *reinterpret_cast<uint4*>(p + q * plane_bytes(R)) = c[q];
}

// the power of two that brings values below 2^(e - 126) (e: biased exponent of the row's largest) below
// 2^15, limited to FP32's range (rows below 2^-112 or with nothing in them; a row with a non-finite value
// keeps scale 1 and gives NaN), and its inverse
__device__ __forceinline__ float row_scale(int hmax) {
    const int e = hmax >> 23;
    const int k = e >= 255 ? 0 : min(126, 141 - e);
    return __uint_as_float((uint32_t)(k + 127) << 23);
}
__device__ __forceinline__ float inv_scale(float s) { return __uint_as_float((254u << 23) - __float_as_uint(s)); }
// a product of scaled operands times both inverse scales, the smaller first: large rows against small ones
// give an ordinary number, but the larger scale alone could take it past FP32's range
__device__ __forceinline__ float unscale(float a, float s, float t) { return a * fminf(s, t) * fmaxf(s, t); }
__device__ __forceinline__ int f_abs(float x) { return __float_as_int(x) & 0x7FFFFFFF; }
// The kernels of one call form a chain whose members are launched while the one before still runs
// (launch_chained) and wait for its results here.  What the kernel before wrote is read by volatile loads:
// a load through the read-only path could be moved above the wait.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;\n"); }
__device__ __forceinline__ int ld_dep(const int* p) {
    int v;
    asm volatile("ld.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float ld_dep(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];\n" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_dep(const float2* p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int max_segs(const int* __restrict__ emax, int n, int r) {
    int h = 0;
#pragma unroll
    for (int s = 0; s < kNlSegs; ++s) h = max(h, ld_dep(emax + (size_t)s * n + r));
    return h;
}

// largest magnitude (bits) of row r of src over column segment seg (one CTA)
__device__ __forceinline__ void nl_rowmax(const float2* __restrict__ src, int ld, int rows, int cols, int* __restrict__ emax, int r,
                                          int seg) {
    __shared__ int red[8];
    const int per = (cols + kNlSegs - 1) / kNlSegs;
    const int c0 = seg * per, c1 = min(cols, c0 + per);
    const float2* p = src + (size_t)r * ld;
    int h = 0;
#pragma unroll 4
    for (int c = c0 + threadIdx.x; c < c1; c += 256) {
        const float2 v = __ldg(p + c);
        h = max(h, max(f_abs(v.x), f_abs(v.y)));
    }
    h = __reduce_max_sync(0xffffffffu, h);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) h = max(h, red[w]);
        emax[(size_t)seg * rows + r] = h;
    }
}
// the same per column of src [K][cols] over K segment seg, columns from 256 cb on
__device__ __forceinline__ void nl_colmax(const float2* __restrict__ src, int ld, int K, int cols, int* __restrict__ emax, int cb,
                                          int seg) {
    const int c = cb * 256 + threadIdx.x, per = (K + kNlSegs - 1) / kNlSegs;
    if (c >= cols) return;
    const int k0 = seg * per, k1 = min(K, k0 + per);
    int h = 0;
#pragma unroll 8
    for (int k = k0; k < k1; ++k) {
        const float2 v = __ldg(src + (size_t)k * ld + c);
        h = max(h, max(f_abs(v.x), f_abs(v.y)));
    }
    emax[(size_t)seg * cols + c] = h;
}
__global__ void __launch_bounds__(256) k_nl_rowmax(const float2* __restrict__ src, int ld, int rows, int cols,
                                                   int* __restrict__ emax) {
    chain_next();
    nl_rowmax(src, ld, rows, cols, emax, blockIdx.x, blockIdx.y);
}
// both of the projectors: the first `rows` blocks of x the rows, the others the columns
__global__ void __launch_bounds__(256) k_nl_maxima(const float2* __restrict__ src, int ld, int rows, int cols,
                                                   int* __restrict__ erow, int* __restrict__ ecol) {
    chain_next();
    if ((int)blockIdx.x < rows) nl_rowmax(src, ld, rows, cols, erow, blockIdx.x, blockIdx.y);
    else nl_colmax(src, ld, rows, cols, ecol, blockIdx.x - rows, blockIdx.y);
}

// Rows of complex src (K = 2 ncols interleaved reals) -> blocked split operand.  expand = 0:
// row r is src row r as stored; expand = 1: rows 2b, 2b+1 are src row b as stored and its
// rotation (im, -re).  Rows >= nsrc (resp. 2 nsrc) and K beyond 2 ncols are written as zeros.
// CTA: 8 rows (one core-matrix row group, by) x 32 chunks of 8 K values (bx);
// the 8 rows of a core matrix on consecutive threads (one 128-byte run per plane), the 2
// chunks of a K tile on consecutive thread octets.  inv: the source rows' inverse scales.
constexpr int kSplitChunks = 32;
constexpr int kFoldReduce = 1024;  // projectors x splits up to which the expansion sums the splits (one CTA per 4 bands)
constexpr int kSelfScale = 2048;  // plane waves up to which a row's scale is found in its splitting CTA
__device__ __forceinline__ void split_rows(const float2* __restrict__ src, int ld, int nsrc, int ncols, int expand, int R, int nkt,
                                           const int* __restrict__ emax, float* __restrict__ inv, unsigned char* __restrict__ blk,
                                           int bx, int by) {
    const int r = by * 8 + (threadIdx.x & 7);
    int ch = bx * kSplitChunks + (threadIdx.x >> 3);
    const int b = expand ? (r >> 1) : r;
    float sc = 1.f;
    if (!emax) {  // short rows, one CTA per row group: the rows' largest values are found here
        __shared__ int smax[8];
        const int nrow = expand ? 4 : 8, l = threadIdx.x & 31, b0 = by * nrow;
        for (int q = threadIdx.x >> 5; q < nrow; q += 8) {
            int h = 0;
            if (b0 + q < nsrc)
                for (int c = l; c < ncols; c += 32) {
                    const float2 x = __ldg(src + (size_t)(b0 + q) * ld + c);
                    h = max(h, max(f_abs(x.x), f_abs(x.y)));
                }
            h = __reduce_max_sync(0xffffffffu, h);
            if (l == 0) smax[q] = h;
        }
        __syncthreads();
        sc = row_scale(smax[b - b0]);
    } else if (b < nsrc) {
        sc = row_scale(max_segs(emax, nsrc, b));
    }
    if (ch == 0 && b < nsrc && !(expand && (r & 1))) inv[b] = inv_scale(sc);
    for (; ch < nkt * (KT / 8); ch += emax ? nkt * (KT / 8) : kSplitChunks) {
        const int c0 = ch * 4;  // first complex column of the chunk
        float v[8];
        if (b < nsrc && c0 + 3 < ncols) {
            const float2* s2 = src + (size_t)b * ld + c0;
            if (((uintptr_t)s2 & 15) == 0) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(s2)), bb = __ldg(reinterpret_cast<const float4*>(s2) + 1);
                v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = bb.x; v[5] = bb.y; v[6] = bb.z; v[7] = bb.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 x = __ldg(s2 + j);
                    v[2 * j] = x.x;
                    v[2 * j + 1] = x.y;
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 x = make_float2(0.f, 0.f);
                if (b < nsrc && c0 + j < ncols) x = __ldg(src + (size_t)b * ld + c0 + j);
                v[2 * j] = x.x;
                v[2 * j + 1] = x.y;
            }
        }
        if (expand && (r & 1)) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float re = v[2 * j], im = v[2 * j + 1];
                v[2 * j] = im;
                v[2 * j + 1] = -re;
            }
        }
        put8(blk, R, nkt, r, ch * 8, v, sc);
    }
}

// beta [P][G] (complex, ld) -> blocked split betaT: row g, K = (p, u) (u = re/im of beta[p][g]).
// CTA tile: 64 rows g x 16 projectors (two K tiles), transposed through shared memory so the
// global reads run along g.  Rows g >= G (up to rows_pad) and p >= P are zeros.
constexpr int kTG = 64, kTP = 16;
__device__ __forceinline__ void split_t(const float2* __restrict__ beta, int ld, int P, int G, int R, int nkt,
                                        const int* __restrict__ emax, float* __restrict__ inv, unsigned char* __restrict__ blk,
                                        int bx, int by) {
    __shared__ float2 t[kTP][kTG + 1];
    const int g0 = bx * kTG, p0 = by * kTP;
    for (int i = threadIdx.x; i < kTP * kTG; i += blockDim.x) {
        const int pp = i / kTG, gg = i - pp * kTG;
        const int p = p0 + pp, g = g0 + gg;
        t[pp][gg] = (p < P && g < G) ? __ldg(beta + (size_t)p * ld + g) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    // 64 rows x 4 chunks of 4 projectors; the 8 rows of a core matrix on consecutive threads
    const int rlo = threadIdx.x & 7, ch = (threadIdx.x >> 3) & 3, rg = threadIdx.x >> 5;
    const int gg = rg * 8 + rlo, g = g0 + gg;
    const float sc = g < G ? row_scale(max_segs(emax, G, g)) : 1.f;
    if (by == 0 && ch == 0 && g < G) inv[g] = inv_scale(sc);
    if (by * 2 + (ch >> 1) >= nkt) return;
    float v[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 x = t[ch * 4 + j][gg];
        v[2 * j] = x.x;
        v[2 * j + 1] = x.y;
    }
    put8(blk, R, nkt, g, p0 * 2 + ch * 8, v, sc);
}

__global__ void __launch_bounds__(256) k_split_rows(const float2* __restrict__ src, int ld, int nsrc, int ncols,
                                                    int expand, int R, int nkt, const int* __restrict__ emax,
                                                    float* __restrict__ inv, unsigned char* __restrict__ blk) {
    chain_wait();
    split_rows(src, ld, nsrc, ncols, expand, R, nkt, emax, inv, blk, blockIdx.x, blockIdx.y);
}
// both layouts of the projectors beta [P][G]: the first nxk * nyk blocks betaK (nxk blocks per row group), the
// others betaT (nxt blocks of columns)
__global__ void __launch_bounds__(256) k_split_beta(const float2* __restrict__ beta, int ld, int P, int G, int nxk, int nyk, int nktk,
                                                    const int* __restrict__ ek, float* __restrict__ invk,
                                                    unsigned char* __restrict__ blkk, int nxt, int Rt, int nktt,
                                                    const int* __restrict__ et, float* __restrict__ invt,
                                                    unsigned char* __restrict__ blkt) {
    chain_wait();
    int b = blockIdx.x;
    if (b < nxk * nyk) {
        split_rows(beta, ld, P, G, 0, TM, nktk, ek, invk, blkk, b % nxk, b / nxk);
    } else {
        b -= nxk * nyk;
        split_t(beta, ld, P, G, Rt, nktt, et, invt, blkt, b % nxt, b / nxt);
    }
}

// sum the split-K partials of the projection C[z][p][c] (FP32, ldc; c = 2b + t) in a fixed order,
// undo the rows' scales and multiply by D_p: Pd[p][c].  CTA: 32 consecutive outputs x 8 parts of the
// splits (one thread per output took 7 us for 64 splits of a few thousand outputs, all of it latency).
__global__ void __launch_bounds__(256) k_reduce_p(const float* __restrict__ part, int Z, size_t zstride, int ldc, int P,
                                                  int ncol, const double* __restrict__ D, const float* __restrict__ inv_p,
                                                  const float* __restrict__ inv_b, float* __restrict__ Pd) {
    __shared__ float red[8][32];
    const size_t total = (size_t)P * ncol, e = blockIdx.x * (size_t)32 + (threadIdx.x & 31);
    const int w = threadIdx.x >> 5, p = (int)(e / ncol), c = (int)(e - (size_t)p * ncol);
    float a = 0.f;
    chain_next();
    chain_wait();
    if (e < total) {
        const float* q = part + (size_t)p * ldc + c;
#pragma unroll 8
        for (int z = w; z < Z; z += 8) a += ld_dep(q + (size_t)z * zstride);
    }
    red[w][threadIdx.x & 31] = a;
    __syncthreads();
    if (w == 0 && e < total) {
#pragma unroll
        for (int i = 1; i < 8; ++i) a += red[i][threadIdx.x];
        Pd[e] = unscale(a, __ldg(inv_p + p), ld_dep(inv_b + (c >> 1))) * (float)__ldg(D + p);
    }
}

// the application's A operand E = D P expanded, blocked and split (rows 2b + t, K = (p, u)):
// E[2b][(p,0)] = ar, E[2b][(p,1)] = -ai, E[2b+1][(p,0)] = ai, E[2b+1][(p,1)] = ar with
// a = Pd[p][2b] + i Pd[p][2b+1]; rows >= 2 nb and p >= P are zeros.  One CTA per core-matrix row
// group (four bands): their largest values first, then one thread per (row, 4 projectors).
// part != NULL (few partial sums): the sums of k_reduce_p are taken here instead of read from Pd, through
// shared memory (P x 4 bands).
__global__ void __launch_bounds__(256) k_expand_e(const float* __restrict__ Pd, const float* __restrict__ part, int Z,
                                                  size_t zstride, int ldc, const double* __restrict__ D,
                                                  const float* __restrict__ inv_p, const float* __restrict__ inv_b, int P, int nb,
                                                  int nkt, float* __restrict__ inv, unsigned char* __restrict__ blk) {
    extern __shared__ __align__(16) unsigned char esm[];
    chain_next();
    float2* sp = reinterpret_cast<float2*>(esm);  // [P][4] when part
    __shared__ int smax[4];
    const int tid = threadIdx.x, q4 = tid & 3, b4 = blockIdx.x * 4 + q4;
    if (tid < 4) smax[tid] = 0;
    __syncthreads();
    chain_wait();
    int h = 0;
    const float ib = part && b4 < nb ? ld_dep(inv_b + b4) : 0.f;
    if (!part && b4 < nb) {
#pragma unroll 8
        for (int p = tid >> 2; p < P; p += 64) {
            const float2 a = ld_dep(reinterpret_cast<const float2*>(Pd + (size_t)p * 2 * nb) + b4);
            h = max(h, max(f_abs(a.x), f_abs(a.y)));
        }
    }
    for (int p = tid >> 2; part && p < P; p += 64) {
        float2 a = make_float2(0.f, 0.f);
        if (b4 < nb) {
            const float* q = part + (size_t)p * ldc + 2 * b4;
#pragma unroll 8
            for (int z = 0; z < Z; ++z) {
                const float2 v = ld_dep(reinterpret_cast<const float2*>(q + (size_t)z * zstride));
                a.x += v.x;
                a.y += v.y;
            }
            const float ip = __ldg(inv_p + p), d = (float)__ldg(D + p);
            a.x = unscale(a.x, ip, ib) * d;
            a.y = unscale(a.y, ip, ib) * d;
        }
        sp[p * 4 + q4] = a;
        h = max(h, max(f_abs(a.x), f_abs(a.y)));
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    if ((tid & 31) < 4) atomicMax(&smax[q4], h);
    __syncthreads();
    const int nchunk = nkt * (KT / 8), rlo = tid & 7, r = blockIdx.x * 8 + rlo, b = r >> 1, t = r & 1;
    const float sc = row_scale(smax[rlo >> 1]);
    if (tid < 8 && !t && b < nb && blockIdx.y == 0) inv[b] = inv_scale(sc);
    for (int ch = blockIdx.y * 32 + (tid >> 3); ch < nchunk; ch += 32 * gridDim.y) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = ch * 4 + j;
            float2 a = make_float2(0.f, 0.f);
            if (b < nb && p < P) a = part ? sp[p * 4 + (rlo >> 1)] : ld_dep(reinterpret_cast<const float2*>(Pd + (size_t)p * 2 * nb) + b);
            v[2 * j] = t ? a.y : a.x;
            v[2 * j + 1] = t ? a.x : -a.y;
        }
        put8(blk, TM, nkt, r, ch * 8, v, sc);
    }
}

__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort) {
    for (long i = 0; i < kSpin; ++i) {
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

// C (+)= A B^T over the K tiles [kt0, kt1) of this split.  A: blocked, 128-row tiles (mtiles of them), nkt K
// tiles per row tile, msub (1 or 2) row tiles per CTA; B: blocked in tiles of bsub x BN rows, one of the
// bsub parts per CTA.  EPI 0: C is FP32 [m][n] (ldc) at
// C + z*zstride (split-K partials, operands' scales not undone); EPI 1: row m = 2b + t, column g -> complex
// out[b][g] component t (ldc = complex row stride) times inv_m[b] inv_n[g], accumulate: add to out.
template <int EPI, bool kDual>
__global__ void __launch_bounds__(kGemmThreads, 1)
k_nl_gemm(const unsigned char* __restrict__ A, const unsigned char* __restrict__ B, int nkt, int BN, int bsub, int msub, int M,
          int N, int mtiles, int kt_per_split, float* __restrict__ C, size_t ldc, size_t zstride, int accumulate,
          const float* __restrict__ inv_m, const float* __restrict__ inv_n, int* __restrict__ err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[kNlStages], empty[kNlStages], accf;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, s_used, s_issued;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // projection: N tiles fastest (the few N tiles of one M tile share its beta tiles in L2);
    // application: M tiles fastest (the M tiles of one N tile share its betaT tiles, which are
    // then read from HBM once instead of once per M tile)
    const int nt = EPI == 0 ? blockIdx.x : blockIdx.y, mt = msub * (EPI == 0 ? blockIdx.y : blockIdx.x);
    const int nsub = min(msub, mtiles - mt);
    const int kt0 = blockIdx.z * kt_per_split;
    const int kt1 = min(nkt, kt0 + kt_per_split);
    const int nk = max(0, kt1 - kt0);
    const uint32_t a_bytes = (uint32_t)block_bytes(TM), b_bytes = (uint32_t)block_bytes(BN), b_src_bytes = b_bytes * bsub;
    const uint32_t stage_bytes = msub * a_bytes + b_bytes, tx_bytes = nsub * a_bytes + b_bytes;
    const uint32_t acols = BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256;  // columns between the accumulators
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tc::smem_u32(&tmem_base)),
                     "r"(kDual ? 2 * msub * acols : msub * acols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int s = 0; s < kNlStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&empty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc::smem_u32(&accf)));
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        abort_flag = 0;
        s_used = s_issued = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    chain_wait();  // (barriers and tensor memory are set up beside the kernel before)
    const uint32_t tmem = tmem_base;
    volatile int* abort = &abort_flag;
    const unsigned char* a_src = A + ((size_t)mt * nkt + kt0) * a_bytes;
    const unsigned char* b_src = B + ((size_t)(nt / bsub) * nkt + kt0) * b_src_bytes + (nt % bsub) * (b_bytes / 2);
    const uint32_t sbase = tc::smem_u32(smem);
    int issued = 0;  // producer: K tiles whose copies were issued
    int used = 0;    // MMA issuer: K tiles consumed
    if (warp == 0 && lane == 0) {
        for (int it = 0, s = 0, ph = 0; it < nk; ++it) {
            if (it >= kNlStages && !wait_bar(tc::smem_u32(&empty[s]), ph ^ 1, abort)) {
                *abort = 1;
                break;
            }
            const uint32_t fb = tc::smem_u32(&full[s]);
            const uint32_t dst = sbase + s * stage_bytes;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(tx_bytes) : "memory");
            for (int u = 0; u < nsub; ++u)
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                        dst + u * a_bytes),
                    "l"(a_src + ((size_t)u * nkt + it) * a_bytes), "r"(a_bytes), "r"(fb)
                    : "memory");
            for (int q = 0; q < 2; ++q)  // the two planes of this CTA's part of the source's row tile
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                        dst + msub * a_bytes + q * (b_bytes / 2)),
                    "l"(b_src + (size_t)it * b_src_bytes + q * (b_src_bytes / 2)), "r"(b_bytes / 2), "r"(fb)
                    : "memory");
            issued = it + 1;
            if (++s == kNlStages) s = 0, ph ^= 1;
        }
    } else if (warp == 1 && lane == 0) {
        const uint32_t idesc = tc::idesc_f16(TM, BN);
        const int pa[3] = {1, 0, 0}, pb[3] = {0, 1, 0};  // smallest terms first
        for (int it = 0, s = 0, ph = 0; it < nk; ++it) {
            if (!wait_bar(tc::smem_u32(&full[s]), ph, abort)) {
                *abort = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint32_t sa = sbase + s * stage_bytes, sb = sa + msub * a_bytes;
            for (int u = 0; u < nsub; ++u) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const uint64_t da = tc::sdesc(sa + u * a_bytes + pa[q] * (uint32_t)plane_bytes(TM), 128, 256);
                    const uint64_t db = tc::sdesc(sb + pb[q] * (uint32_t)plane_bytes(BN), 128, 256);
                    const uint32_t acc = (it > 0 || q == 1 || (q == 2 && !kDual)) ? 1u : 0u;
                    const uint32_t td = tmem + (kDual && q < 2 ? u + msub : u) * acols;
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(td),
                        "l"(da), "l"(db), "r"(idesc), "r"(acc));
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                tc::smem_u32(&empty[s])));
            used = it + 1;
            if (++s == kNlStages) s = 0, ph ^= 1;
        }
        // the accumulators are final once every product issued so far has completed
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
            tc::smem_u32(&accf)));
    }
    if (warp == 1 && lane == 0) s_used = used;
    if (warp == 0 && lane == 0) s_issued = issued;
    if (warp >= 4) {
        const bool ok = wait_bar(tc::smem_u32(&accf), 0, nullptr);
        if (!ok) *abort = 1;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const int q = warp & 3, u = (warp - 4) >> 2;  // tensor-memory lanes 32 q .., accumulator u
        // warp-uniform decision (tcgen05.ld and the shuffles below need the whole warp)
        if (__all_sync(0xffffffffu, ok && nk > 0 && !*abort) && u < nsub) {
            const int mrow = (mt + u) * TM + q * 32 + lane;  // this thread's accumulator row
            const float im = EPI == 1 && mrow < M ? ld_dep(inv_m + (mrow >> 1)) : 1.f;
            // (as unscale: the row's scale before the column's if it is below one, else after it)
            const float im_lo = fminf(im, 1.f), im_hi = fmaxf(im, 1.f);
            const bool low = __all_sync(0xffffffffu, im <= 1.f);
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += 16) {
                uint32_t v[16];
                const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)u * acols + (uint32_t)c0;
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                    "%13, %14, %15}, [%16];\n"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                      "=r"(v[15])
                    : "r"(taddr));
                if (!kDual) {
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                } else {
                    uint32_t x[16];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                        "%13, %14, %15}, [%16];\n"
                        : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]),
                          "=r"(x[8]), "=r"(x[9]), "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]), "=r"(x[14]),
                          "=r"(x[15])
                        : "r"(taddr + msub * acols));
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(x[j]));
                }
                const int n0 = nt * BN + c0;
                if (EPI == 0) {
                    if (mrow < M) {
                        float* crow = C + (size_t)blockIdx.z * zstride + (size_t)mrow * ldc;
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (n0 + j < N) crow[n0 + j] = __uint_as_float(v[j]);
                    }
                } else {
                    // lanes 2j, 2j+1 hold Re and Im of band mrow/2: swap halves so that each lane
                    // owns 8 complex values (64 contiguous bytes) of the band's row
                    const int t = lane & 1;
                    float y[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        y[j] = __shfl_xor_sync(0xffffffffu, __uint_as_float(t ? v[j] : v[8 + j]), 1);
                    if (mrow < M) {
                        const int g0 = n0 + (t ? 8 : 0);
                        float2* orow = reinterpret_cast<float2*>(C) + (size_t)(mrow >> 1) * ldc;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int g = g0 + j;
                            if (g < N) {
                                const float in = __ldg(inv_n + g) * im_lo;
                                float2 o = t ? make_float2(y[j], __uint_as_float(v[8 + j]))
                                             : make_float2(__uint_as_float(v[j]), y[j]);
                                o.x *= in;
                                o.y *= in;
                                if (!low) {
                                    o.x *= im_hi;
                                    o.y *= im_hi;
                                }
                                if (accumulate) {
                                    const float2 a = orow[g];
                                    o.x += a.x;
                                    o.y += a.y;
                                }
                                orow[g] = o;
                            }
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    if (*abort) {
        if (tid == 0) atomicExch(err, 1);
        // drain: the copies issued but never consumed, then every product issued
        if (warp == 0 && lane == 0) {
            for (int it = s_used; it < s_issued; ++it) {
                const int s = it % kNlStages;
                wait_bar(tc::smem_u32(&full[s]), (it / kNlStages) & 1, nullptr);
            }
        }
        if (warp == 1 && lane == 0) wait_bar(tc::smem_u32(&accf), 0, nullptr);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kDual ? 2 * msub * acols : msub * acols));
}

inline size_t rup(size_t x, size_t a) { return (x + a - 1) / a * a; }

// N tile of the projection: the 2 nb columns in the fewest tiles of at most 256, rounded to 16
int proj_bn(int nb) {
    const int n = 2 * nb;
    const int tiles = (n + 255) / 256;
    return (int)rup((size_t)((n + tiles - 1) / tiles), 16);
}
constexpr int kAppBN = 256;

// Tile shape of a GEMM (row tiles per CTA, parts of a B tile, splits of K): the cheapest by rounds of CTAs
// over the SMs times the cycles of a CTA's K tiles (3 products of 128 x BN x 16 per row tile, or their
// operands at 45 bytes per clock, at least the 400 a step takes), plus start, fill and drain.
struct GemmShape {
    int msub, bsub, splits;
    bool dual;  // the small terms in accumulators of their own
};
constexpr int kFewProj = 48;  // projectors up to which they are (64: 1.3e-7 with six products, 9.9e-8 in one accumulator)
GemmShape gemm_shape(int mtiles, int ntiles, int BN, int nkt, int max_bsub, int max_splits, bool few) {
    GemmShape best{1, 1, 1, few};
    double cost = -1;
    const int sms = device_sms();
    for (int msub = std::min(2, mtiles); msub >= 1; --msub)
        for (int bsub = 1; bsub <= max_bsub; bsub *= 2) {
            const long tiles = (long)((mtiles + msub - 1) / msub) * ntiles * bsub;
            const int sp = (int)std::max<long>(1, std::min<long>({(long)max_splits, (long)std::max(1, nkt / 8), sms / tiles}));
            const int per = (nkt + sp - 1) / sp, m = std::min(msub, mtiles), bn = BN / bsub;
            const double tile = std::max(1.5 * m * bn, (m * 8192.0 + bn * 64.0) / 45.0);
            if (few && 2 * msub * (bn <= 32 ? 32 : bn <= 64 ? 64 : bn <= 128 ? 128 : 256) > 512) continue;  // (bn and msub halve)
            // CTAs an SM holds, by shared memory and tensor memory; more than one share its throughput
            const int cols = (few ? 2 : 1) * msub * (bn <= 32 ? 32 : bn <= 64 ? 64 : bn <= 128 ? 128 : 256);
            const long occ = std::min<long>((226 << 10) / (long)(kNlStages * (msub * block_bytes(TM) + block_bytes(bn))), 512 / cols);
            const long n = tiles * sp;
            const double load = occ > 1 ? std::max(1.0, (double)n / sms) : (double)((n + sms - 1) / sms);
            const double c = std::max(load * per * tile, (double)((n + sms * occ - 1) / (sms * occ)) * per * std::max(tile, 400.0)) + 6000.0;
            if (cost < 0 || c < cost) {
                cost = c;
                best = GemmShape{msub, bsub, (nkt + per - 1) / per, few};
            }
        }
    return best;
}

struct NlLayout {
    GemmShape sp, sa;                   // shapes of the projection and the application
    int bn_p, ntile_p, mtile_p, nkt_p;  // projection: N tile, tiles, K tiles (of 2 npw)
    int mtile_a, ntile_a, nkt_a;        // application
    int splits;
    size_t betaK_off, betaT_off, inv_off, psiX_off, part_off, pd_off, e_off, emax_off, invb_off, total;
    size_t zstride;
};

NlLayout nl_layout(int nproj, int nb, int npw, bool with_beta) {
    NlLayout L{};
    L.bn_p = proj_bn(nb);
    L.ntile_p = (2 * nb + L.bn_p - 1) / L.bn_p;
    L.mtile_p = (nproj + TM - 1) / TM;
    L.nkt_p = (int)(rup(2 * (size_t)npw, KT) / KT);
    L.mtile_a = (2 * nb + TM - 1) / TM;
    L.ntile_a = (npw + kAppBN - 1) / kAppBN;
    L.nkt_a = (int)(rup(2 * (size_t)nproj, KT) / KT);
    const bool few = nproj <= kFewProj;
    L.sp = gemm_shape(L.mtile_p, L.ntile_p, L.bn_p, L.nkt_p, 1, kMaxUmmaSplits, few);
    L.sa = gemm_shape(L.mtile_a, L.ntile_a, kAppBN, L.nkt_a, 4, 1, few);
    L.splits = L.sp.splits;
    L.zstride = (size_t)L.mtile_p * TM * L.ntile_p * L.bn_p;
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t o = off;
        off = rup(off + b, 256);
        return o;
    };
    L.betaK_off = take(with_beta ? (size_t)L.mtile_p * L.nkt_p * block_bytes(TM) : 0);
    L.betaT_off = take(with_beta ? (size_t)L.ntile_a * L.nkt_a * block_bytes(kAppBN) : 0);
    // inverse scales: betaK rows, betaT rows; then the partial maxima of both
    L.inv_off = take(with_beta ? sizeof(float) * ((size_t)nproj + npw) * (1 + kNlSegs) : 0);
    L.psiX_off = take((size_t)L.ntile_p * L.nkt_p * block_bytes(L.bn_p));
    L.part_off = take((size_t)L.splits * L.zstride * sizeof(float));
    L.pd_off = take((size_t)nproj * 2 * nb * sizeof(float));
    L.e_off = take((size_t)L.mtile_a * L.nkt_a * block_bytes(TM));
    L.emax_off = take(sizeof(int) * (size_t)kNlSegs * nb);
    L.invb_off = take(sizeof(float) * 2 * (size_t)nb);  // inverse scales of psi's and of E's bands
    L.total = off;
    return L;
}

// grid-dimension limits of the split and GEMM launches (y and z of a grid are below 65536)
qm_status check_limits(const NlLayout& L) {
    if ((long)L.mtile_p * TM / 8 > 65535 || (long)L.ntile_p * L.bn_p / 8 > 65535 || (L.nkt_a + 1) / 2 > 65535 ||
        L.ntile_a * L.sa.bsub > 65535 || L.mtile_p > 65535)
        return fail(QM_ERR_UNSUPPORTED, "tensor-core nonlocal part: too many bands, projectors or plane waves");
    return QM_OK;
}

// Launch while the kernel before in the stream still runs (programmatic dependent launch): its last CTAs, the
// launch and the set-up of this one overlap, 1 to 2 us at each link of the chain (64 atoms: 2 bands 73.6 ->
// 64.6 us, 24 bands 107 -> 98; 160 bands 427 -> 420).  The kernel calls chain_wait before it uses or
// overwrites anything.  chain_next in the kernel before lets this one's CTAs take their places early; the
// products and k_split_rows do not call it: projection CTAs that wait beside the split keep FFT CTAs of the
// other stream off the SMs (propagation of 32 atoms: 1107 us with it, 1044 without).
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

qm_status split_beta(int nproj, int npw, const float2* beta, int ld_beta, const NlLayout& L, unsigned char* base, cudaStream_t s) {
    float* invk = (float*)(base + L.inv_off);
    float* invt = invk + nproj;
    int* ek = (int*)(invt + npw);
    int* et = ek + (size_t)kNlSegs * nproj;
    {
        ProfScope pf(PF_SPLIT, s);
        k_nl_maxima<<<dim3((unsigned)(nproj + (npw + 255) / 256), kNlSegs), 256, 0, s>>>(beta, ld_beta, nproj, npw, ek, et);
    }
    const int nxk = (L.nkt_p * (KT / 8) + kSplitChunks - 1) / kSplitChunks, nyk = L.mtile_p * TM / 8;
    const int nxt = L.ntile_a * kAppBN / kTG, nyt = (L.nkt_a + 1) / 2;
    ProfScope pf(PF_SPLIT, s);
    return cuda_check(launch_chained(k_split_beta, dim3((unsigned)((long)nxk * nyk + (long)nxt * nyt)), 256, 0, s, beta, ld_beta, nproj,
                                     npw, nxk, nyk, L.nkt_p, ek, invk, base + L.betaK_off, nxt, kAppBN, L.nkt_a, et, invt,
                                     base + L.betaT_off), "k_split_beta launch");
}

template <int EPI>
qm_status gemm_launch(const unsigned char* A, const unsigned char* B, int nkt, int BN, const GemmShape& sh, int M, int N, int mt,
                      int ntl, float* C, size_t ldc, size_t zstride, bool accumulate, const float* inv_m, const float* inv_n,
                      int* err, cudaStream_t s) {
    const int per = (nkt + sh.splits - 1) / sh.splits, bn = BN / sh.bsub;
    const size_t stage = sh.msub * block_bytes(TM) + block_bytes(bn);
    const int mg = (mt + sh.msub - 1) / sh.msub, ng = ntl * sh.bsub;
    const size_t smem = kNlStages * stage;
    const auto kern = sh.dual ? k_nl_gemm<EPI, true> : k_nl_gemm<EPI, false>;
    qm_status st = allow_dynamic_smem((const void*)kern, smem, "tensor-core nonlocal GEMM shared memory");
    if (st) return st;
    ProfScope pf(PF_UMMA, s);
    const dim3 grid = EPI == 0 ? dim3(ng, mg, sh.splits) : dim3(mg, ng, sh.splits);
    st = cuda_check(launch_chained(kern, grid, kGemmThreads, smem, s, A, B, nkt, bn, sh.bsub, sh.msub, M, N, mt, per, C,
                                   ldc, zstride, accumulate ? 1 : 0, inv_m, inv_n, err), "k_nl_gemm launch");
    if (st) return st;
    return cuda_check(cudaGetLastError(), "k_nl_gemm launch");
}

}  // namespace

size_t nonlocal_tc_bytes(int nproj, int nb, int npw, bool with_beta) {
    return nl_layout(nproj, nb, npw, with_beta).total;
}

size_t nonlocal_tc_beta_bytes(int nproj, int nb, int npw) {
    const NlLayout L = nl_layout(nproj, nb, npw, true);
    return L.psiX_off;  // betaK, betaT and their scales come first
}

qm_status nonlocal_tc_prepare(int nproj, int nb, int npw, const float2* beta, int ld_beta, void* beta_work,
                              cudaStream_t s) {
    if (nproj <= 0) return QM_OK;
    const NlLayout L = nl_layout(nproj, nb, npw, true);
    if (qm_status st0 = check_limits(L)) return st0;
    unsigned char* w = (unsigned char*)beta_work;
    return split_beta(nproj, npw, beta, ld_beta, L, w, s);
}

qm_status nonlocal_tc(int nproj, int nb, int npw, const float2* beta, int ld_beta, const void* beta_prepared,
                      const float2* psi, int ld_psi, const double* D, float2* out, int ld_out, void* work, int* err,
                      cudaStream_t s, bool accumulate) {
    if (nproj <= 0 || nb <= 0) return QM_OK;
    const bool own_beta = beta_prepared == nullptr;
    const NlLayout L = nl_layout(nproj, nb, npw, own_beta);
    if (qm_status st0 = check_limits(L)) return st0;
    unsigned char* w = (unsigned char*)work;
    qm_status st;
    const unsigned char* bw = w;  // the split projectors: in the workspace or prepared
    NlLayout Lb = L;
    if (own_beta) {
        if ((st = split_beta(nproj, npw, beta, ld_beta, L, w, s))) return st;
    } else {
        Lb = nl_layout(nproj, nb, npw, true);
        bw = (const unsigned char*)beta_prepared;
    }
    const unsigned char *betaK = bw + Lb.betaK_off, *betaT = bw + Lb.betaT_off;
    const float *invk = (const float*)(bw + Lb.inv_off), *invt = invk + nproj;
    unsigned char* psiX = w + L.psiX_off;
    float* part = (float*)(w + L.part_off);
    unsigned char* E = w + L.e_off;
    int* emax = (int*)(w + L.emax_off);
    float *invb = (float*)(w + L.invb_off), *inve = invb + nb;
    // short rows find their scale in the splitting kernel (one launch less, one CTA per four bands)
    const bool self = npw <= kSelfScale;
    if (!self) {
        ProfScope pf(PF_SPLIT, s);
        k_nl_rowmax<<<dim3((unsigned)nb, kNlSegs), 256, 0, s>>>(psi, ld_psi, nb, npw, emax);
    }
    {
        ProfScope pf(PF_SPLIT, s);
        const dim3 grid(self ? 1u : (unsigned)((L.nkt_p * (KT / 8) + kSplitChunks - 1) / kSplitChunks),
                        (unsigned)(L.ntile_p * L.bn_p / 8));
        if (self) k_split_rows<<<grid, 256, 0, s>>>(psi, ld_psi, nb, npw, 1, L.bn_p, L.nkt_p, nullptr, invb, psiX);
        else if ((st = cuda_check(launch_chained(k_split_rows, grid, 256, 0, s, psi, ld_psi, nb, npw, 1, L.bn_p, L.nkt_p, emax, invb,
                                                 psiX), "k_split_rows launch")))
            return st;
    }
    if ((st = cuda_check(cudaGetLastError(), "k_split_rows launch"))) return st;
    // projection C[p][2b + t] = <beta_p | psi_b>, split over K
    const size_t ldc_p = (size_t)L.ntile_p * L.bn_p;
    if ((st = gemm_launch<0>(betaK, psiX, L.nkt_p, L.bn_p, L.sp, nproj, 2 * nb, L.mtile_p, L.ntile_p, part, ldc_p, L.zstride,
                             false, nullptr, nullptr, err, s)))
        return st;
    const int Z = [&] {
        const int per = (L.nkt_p + L.splits - 1) / L.splits;
        return (L.nkt_p + per - 1) / per;
    }();
    float* Pd = (float*)(w + L.pd_off);
    // few projectors: the split-K sums are taken in the expansion (one launch less)
    const bool fold = (long)nproj * Z <= kFoldReduce;
    if (!fold) {
        ProfScope pf(PF_SPLIT, s);
        if ((st = cuda_check(launch_chained(k_reduce_p, dim3((unsigned)(((size_t)nproj * 2 * nb + 31) / 32)), 256, 0, s, part, Z,
                                            L.zstride, (int)ldc_p, nproj, 2 * nb, D, invk, invb, Pd), "k_reduce_p launch")))
            return st;
    }
    {
        ProfScope pf(PF_SPLIT, s);
        // the chunks of a row group over up to eight CTAs (each finds the bands' largest values for itself)
        const dim3 grid((unsigned)(L.mtile_a * TM / 8), fold ? 1u : (unsigned)std::min(8, (L.nkt_a + 15) / 16));
        if ((st = cuda_check(launch_chained(k_expand_e, grid, 256, fold ? (size_t)nproj * 4 * sizeof(float2) : 0, s, Pd,
                                            fold ? part : nullptr, Z, L.zstride, (int)ldc_p, D, invk, invb, nproj, nb, L.nkt_a, inve, E),
                             "k_expand_e launch")))
            return st;
    }
    // application out[b][g] (+)= sum_p beta[p][g] D_p P[p][b]
    return gemm_launch<1>(E, betaT, L.nkt_a, kAppBN, L.sa, 2 * nb, npw, L.mtile_a, L.ntile_a, (float*)out, (size_t)ld_out, 0, accumulate,
                          inve, invt, err, s);
}

}  // namespace qm
