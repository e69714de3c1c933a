// Lowest eigenpairs of a complex Hermitian matrix in FP64, for the Rayleigh-Ritz step of the
// Davidson solver (and the Loewdin orthonormalisation).  Classical dense algorithms, written
// for a GPU whose FP64 rate is low: the O(m^3) work is done once (Householder reduction), and
// only the wanted eigenpairs are computed from the tridiagonal matrix.
//
//   1. k_tridiag_rows Householder reduction Q^H A Q = T, T real symmetric tridiagonal
//                     (Golub & Van Loan, Matrix Computations, Sec. 8.3.1; the complex
//                     reflector makes every subdiagonal element real).  One cooperative
//                     launch, one grid barrier per column, rows resident in shared memory
//                     (k_tridiag: two barriers per column, for matrices beyond that).
//                     (k_tridiag_small: one CTA, matrices up to kTriSmall.)
//   2. k_multisect    the j-th smallest eigenvalue of T by multisection on Sturm counts
//                     (Sec. 8.4.1): a CTA tests 128 points per round, 8 or 9 rounds.
//   3. k_inviter      eigenvectors of T by inverse iteration (LU with partial pivoting of the
//                     tridiagonal, three solves), one warp per eigenvalue; k_cluster_orth
//                     then orthonormalises the vectors of each cluster of close eigenvalues
//                     by Gram-Schmidt (Sec. 8.4.2, 8.2.2).
//   4. k_backtransf   y <- Q y by applying the reflectors in reverse order, one CTA per
//                     eigenvector (no grid barrier needed: the columns are independent).
#include <cooperative_groups.h>

#include <algorithm>

#include <map>
#include <mutex>

#include "qm_internal.h"

namespace cg = cooperative_groups;

namespace qm {
namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {  // conj(a) * b
    return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

// block-wide sum of a double2 (every thread gets the result); sh >= 32 entries
__device__ double2 block_sum2(double2 v, double2* sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double2 t = make_double2(0.0, 0.0);
    for (int i = 0; i < nw; ++i) {  // fixed order: identical result in every block
        t.x += sh[i].x;
        t.y += sh[i].y;
    }
    return t;
}

__global__ void __launch_bounds__(256)
k_tridiag(double2* __restrict__ A, int lda, int m, double2* __restrict__ Vh, double2* __restrict__ tau,
          double* __restrict__ d, double* __restrict__ e, double2* __restrict__ wbuf) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ double2 sm[];
    double2* sv = sm;       // reflector v (length n)
    double2* sw = sm + m;   // w
    __shared__ double2 red[32];
    const int tid = threadIdx.x, bs = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int gw = blockIdx.x * (bs >> 5) + warp, nwg = gridDim.x * (bs >> 5);
    for (int k = 0; k < m - 1; ++k) {
        const int n = m - k - 1;
        for (int i = tid; i < n; i += bs) sv[i] = A[(size_t)(k + 1 + i) * lda + k];
        __syncthreads();
        double part = 0.0;
        for (int i = 1 + tid; i < n; i += bs) part += sv[i].x * sv[i].x + sv[i].y * sv[i].y;
        const double xn2 = block_sum2(make_double2(part, 0.0), red).x;
        const double2 alpha = sv[0];
        double2 t = make_double2(0.0, 0.0), scale = make_double2(0.0, 0.0);
        double beta = alpha.x;
        if (xn2 > 0.0 || alpha.y != 0.0) {
            // complex reflector H = I - t v v^H with H^H (alpha, x) = (beta, 0), beta real
            beta = -copysign(sqrt(alpha.x * alpha.x + alpha.y * alpha.y + xn2), alpha.x);
            t = make_double2((beta - alpha.x) / beta, -alpha.y / beta);
            const double2 den = make_double2(alpha.x - beta, alpha.y);  // 1 / (alpha - beta)
            const double dd = den.x * den.x + den.y * den.y;
            scale = make_double2(den.x / dd, -den.y / dd);
        }
        __syncthreads();
        for (int i = tid; i < n; i += bs) sv[i] = (i == 0) ? make_double2(1.0, 0.0) : cmul(sv[i], scale);
        __syncthreads();
        if (blockIdx.x == 0) {
            for (int i = tid; i < n; i += bs) Vh[(size_t)k * m + k + 1 + i] = sv[i];
            if (tid == 0) {
                tau[k] = t;
                e[k] = beta;
                d[k] = A[(size_t)k * lda + k].x;
            }
        }
        if (t.x == 0.0 && t.y == 0.0) continue;  // uniform: every block computed the same t
        // w = t * A22 v, one warp per row
        for (int r = gw; r < n; r += nwg) {
            const double2* row = A + (size_t)(k + 1 + r) * lda + (k + 1);
            double2 acc = make_double2(0.0, 0.0);
            for (int j = lane; j < n; j += 32) {
                const double2 a = row[j], v = sv[j];
                acc.x += a.x * v.x - a.y * v.y;
                acc.y += a.x * v.y + a.y * v.x;
            }
            for (int o = 16; o > 0; o >>= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            }
            if (lane == 0) wbuf[r] = cmul(t, acc);
        }
        grid.sync();
        for (int i = tid; i < n; i += bs) sw[i] = wbuf[i];
        __syncthreads();
        double2 dp = make_double2(0.0, 0.0);
        for (int i = tid; i < n; i += bs) {
            const double2 c = cmulc(sw[i], sv[i]);  // w^H v
            dp.x += c.x;
            dp.y += c.y;
        }
        dp = block_sum2(dp, red);
        const double2 a2 = cmul(make_double2(-0.5 * t.x, -0.5 * t.y), dp);
        for (int i = tid; i < n; i += bs) {
            const double2 av = cmul(a2, sv[i]);
            sw[i].x += av.x;
            sw[i].y += av.y;
        }
        __syncthreads();
        // A22 -= v w^H + w v^H, one row per block iteration
        for (int i = blockIdx.x; i < n; i += gridDim.x) {
            double2* row = A + (size_t)(k + 1 + i) * lda + (k + 1);
            const double2 vi = sv[i], wi = sw[i];
            for (int j = tid; j < n; j += bs) {
                const double2 vj = sv[j], wj = sw[j];
                double2 a = row[j];
                // v_i conj(w_j) + w_i conj(v_j)
                a.x -= vi.x * wj.x + vi.y * wj.y + wi.x * vj.x + wi.y * vj.y;
                a.y -= vi.y * wj.x - vi.x * wj.y + wi.y * vj.x - wi.x * vj.y;
                row[j] = a;
            }
        }
        grid.sync();
    }
    if (blockIdx.x == 0 && tid == 0) d[m - 1] = A[(size_t)(m - 1) * lda + (m - 1)].x;
}

// The same reduction with one grid barrier per column.  Row i of A is owned by CTA i mod G
// and, when the rows fit (kSmemRows), lives in that CTA's shared memory for the whole
// reduction.  Step k needs row k of A^(k) (A after the first k reflections): its owner
// publishes row k of A^(k-1) one step early, and every CTA applies the rank-2 update of step
// k-1 to that copy itself, so the pivot row costs no extra barrier.  Per step, every CTA:
//   1. forms the pivot row and the reflector (v_k, t_k) redundantly (same data, same order:
//      bitwise identical in every CTA);
//   2. applies the update of step k-1 to its own rows (columns > k) and multiplies them by
//      v_k, writing its entries of w_k = t_k A22 v_k; the owner of row k+1 publishes it;
//   3. grid barrier;
//   4. reads w_k and applies the symmetric correction w_k -= (t_k/2)(w_k^H v_k) v_k.
// w and the published row are double-buffered by step parity: a CTA may already write step
// k+1's entries while another still reads step k's (the barrier of step k+1 orders step k+2).
// The arithmetic per element is that of k_tridiag (same reflector, same update formula).
template <bool kSmemRows>
__global__ void __launch_bounds__(256)
k_tridiag_rows(double2* __restrict__ A, int lda, int m, double2* __restrict__ Vh, double2* __restrict__ tau,
               double* __restrict__ d, double* __restrict__ e, double2* __restrict__ wbuf, double2* __restrict__ prow) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ double2 sm[];
    double2* sv = sm;             // v_k (indices k+1..m-1)
    double2* svp = sm + m;        // v_{k-1}
    double2* sw = sm + 2 * m;     // w_{k-1}
    double2* sr = sm + 3 * m;     // pivot row of step k
    double2* srows = sm + 4 * m;  // own rows (kSmemRows)
    __shared__ double2 red[32];
    __shared__ double2 s_sc[3];          // t, scale, beta of the current reflector
    __shared__ double2 s_part[8][8];     // per-warp partial products of up to 8 own rows
    const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, b = blockIdx.x;
    const int nr = b < m ? (m - b + G - 1) / G : 0;  // own rows i = b + G r, r < nr
    if (kSmemRows)
        for (int r = 0; r < nr; ++r)
            for (int j = tid; j < m; j += bs) srows[(size_t)r * m + j] = A[(size_t)(b + G * r) * lda + j];
    __syncthreads();
    bool have_prev = false;  // svp, sw hold the update of the previous step
    for (int k = 0; k < m - 1; ++k) {
        // 1. pivot row r_j = A^(k)[k][j], j >= k
        const double2* P = k == 0 ? A : prow + (size_t)(k & 1) * m;
        for (int j = k + tid; j < m; j += bs) {
            double2 a = P[j];
            if (have_prev) {  // a -= v_k conj(w_j) + w_k conj(v_j)   (update of step k-1)
                const double2 vk = svp[k], wk = sw[k], vj = svp[j], wj = sw[j];
                a.x -= vk.x * wj.x + vk.y * wj.y + wk.x * vj.x + wk.y * vj.y;
                a.y -= vk.y * wj.x - vk.x * wj.y + wk.y * vj.x - wk.x * vj.y;
            }
            sr[j] = a;
        }
        __syncthreads();
        // reflector of the column below the diagonal, x_j = conj(r_j), j > k
        double part = 0.0;
        for (int j = k + 2 + tid; j < m; j += bs) part += sr[j].x * sr[j].x + sr[j].y * sr[j].y;
        const double xn2 = block_sum2(make_double2(part, 0.0), red).x;
        if (tid == 0) {  // the reflector's scalars once per CTA (FP64 divisions are costly)
            const double2 alpha = make_double2(sr[k + 1].x, -sr[k + 1].y);
            double2 t = make_double2(0.0, 0.0), scale = make_double2(0.0, 0.0);
            double beta = alpha.x;
            if (xn2 > 0.0 || alpha.y != 0.0) {
                beta = -copysign(sqrt(alpha.x * alpha.x + alpha.y * alpha.y + xn2), alpha.x);
                t = make_double2((beta - alpha.x) / beta, -alpha.y / beta);
                const double2 den = make_double2(alpha.x - beta, alpha.y);
                const double dd = den.x * den.x + den.y * den.y;
                scale = make_double2(den.x / dd, -den.y / dd);
            }
            s_sc[0] = t;
            s_sc[1] = scale;
            s_sc[2] = make_double2(beta, 0.0);
        }
        __syncthreads();
        const double2 t = s_sc[0], scale = s_sc[1];
        const double beta = s_sc[2].x;
        for (int j = k + 1 + tid; j < m; j += bs) {
            const double2 v = j == k + 1 ? make_double2(1.0, 0.0) : cmul(make_double2(sr[j].x, -sr[j].y), scale);
            sv[j] = v;
            if (b == 0) Vh[(size_t)k * m + j] = v;
        }
        if (b == 0 && tid == 0) {
            tau[k] = t;
            e[k] = beta;
            d[k] = sr[k].x;
        }
        __syncthreads();
        // 2. own rows i > k, 8 at a time: update of step k-1 (columns > k), then
        //    w_k[i] = t (A22 v_k)_i.  The threads stride over the columns (every warp busy on
        //    every row); the owner of row k+1 publishes its updated entries.
        const int r_first = k + 1 > b ? (k + 1 - b + G - 1) / G : 0;
        double2* pub = prow + (size_t)((k + 1) & 1) * m;
        for (int r0 = r_first; r0 < nr; r0 += 8) {
            const int rn = min(8, nr - r0);
            double2 acc[8], vi[8], wi[8];
            double2* rowp[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                acc[q] = make_double2(0.0, 0.0);
                const int i = b + G * (r0 + (q < rn ? q : 0));
                vi[q] = have_prev ? svp[i] : make_double2(0.0, 0.0);
                wi[q] = have_prev ? sw[i] : make_double2(0.0, 0.0);
                rowp[q] = kSmemRows ? srows + (size_t)(r0 + (q < rn ? q : 0)) * m : A + (size_t)i * lda;
            }
            const int q_pub = (k + 1 - b) % G == 0 ? (k + 1 - b) / G - r0 : -1;  // row k+1 in this chunk
            for (int j = k + 1 + tid; j < m; j += bs) {
                const double2 v = sv[j];
                const double2 vj = have_prev ? svp[j] : make_double2(0.0, 0.0);
                const double2 wj = have_prev ? sw[j] : make_double2(0.0, 0.0);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (q < rn) {
                        double2 a = rowp[q][j];
                        if (have_prev) {
                            a.x -= vi[q].x * wj.x + vi[q].y * wj.y + wi[q].x * vj.x + wi[q].y * vj.y;
                            a.y -= vi[q].y * wj.x - vi[q].x * wj.y + wi[q].y * vj.x - wi[q].x * vj.y;
                            rowp[q][j] = a;
                        }
                        if (q == q_pub) pub[j] = a;
                        acc[q].x += a.x * v.x - a.y * v.y;
                        acc[q].y += a.x * v.y + a.y * v.x;
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (q < rn) {
                    for (int o = 16; o > 0; o >>= 1) {
                        acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, o);
                        acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, o);
                    }
                    if (lane == 0) s_part[warp][q] = acc[q];
                }
            }
            __syncthreads();
            if (tid < rn) {
                double2 sum = make_double2(0.0, 0.0);
                for (int w8 = 0; w8 < 8; ++w8) {  // fixed order
                    sum.x += s_part[w8][tid].x;
                    sum.y += s_part[w8][tid].y;
                }
                wbuf[(size_t)(k & 1) * m + b + G * (r0 + tid)] = cmul(t, sum);
            }
            __syncthreads();
        }
        grid.sync();
        // 4. w_k with the symmetric correction; (v_k, w_k) become the previous update
        double2 dp = make_double2(0.0, 0.0);
        for (int j = k + 1 + tid; j < m; j += bs) {
            const double2 wj = wbuf[(size_t)(k & 1) * m + j];
            sw[j] = wj;
            const double2 c = cmulc(wj, sv[j]);
            dp.x += c.x;
            dp.y += c.y;
        }
        dp = block_sum2(dp, red);
        const double2 a2 = cmul(make_double2(-0.5 * t.x, -0.5 * t.y), dp);
        for (int j = k + 1 + tid; j < m; j += bs) {
            const double2 v = sv[j], av = cmul(a2, v);
            sw[j].x += av.x;
            sw[j].y += av.y;
            svp[j] = v;
        }
        __syncthreads();
        have_prev = true;
    }
    if (b == 0 && tid == 0) {
        double2 a = m == 1 ? A[0] : prow[(size_t)((m - 1) & 1) * m + (m - 1)];
        if (have_prev) {
            const double2 v = svp[m - 1], w = sw[m - 1];
            a.x -= 2.0 * (v.x * w.x + v.y * w.y);
        }
        d[m - 1] = a.x;
    }
}

// The reduction of a small matrix (m <= kTriSmall) in one CTA, the matrix in shared memory: a column of the
// grid-wide reduction costs 8 us of barriers and launch-wide latency whatever its length.  What bounds it is
// the chain of FP64 instructions: each holds its warp and its partition's pipe for 64 cycles, independent or
// not, and a root or a division is six to ten of them.  So the reflector stays unscaled (v = x - beta e_1,
// tau = -1 / (beta conj(v_0))): the product A v needs only the root, and the division for tau runs on the
// last warp beside it.  v^H A v is real, so the correction of w = tau A v is one real sum.  Warp 0 updates the
// next column first and builds its reflector while the others update the rest (lower triangle, mirrored).
// Eight-band solves (m up to 32): 80 us on average, 248 us with the grid-wide kernel.
// Unscaled, |tau|^2 is of the order of |x|^-4, so the range of x has to be bounded: a matrix whose largest
// component lies outside 2^-50 ... 2^50 is scaled by a power of two into it (T is scaled back; v and tau belong
// together at either scale), and a column whose norm is below 2^-120 of that component counts as eliminated
// (its coupling is zero: a change of 1e-36 |A|).  Then |x| is within 2^-171 ... 2^57, |tau|^2 below 2^685.
constexpr int kTriSmall = 64;
constexpr int kTriRange = 50, kTriDrop = 120;
__global__ void __launch_bounds__(256)
k_tridiag_small(const double2* __restrict__ A, int lda, int m, double2* __restrict__ Vh, double2* __restrict__ tau,
                double* __restrict__ d, double* __restrict__ e) {
    extern __shared__ double2 smt[];
    const int ld = m + 1;
    double2 *a = smt, *vb = smt + m * ld, *w = vb + 2 * m;  // [m][ld], reflectors of two columns, product
    __shared__ double s_beta[2], s_half;  // beta (0: no reflection), -|tau|^2 / 2
    __shared__ double2 s_t;
    __shared__ int s_max[8];
    const int tid = threadIdx.x, lane = tid & 31;
    int h = 0;  // largest high word of a component, compared as integers
    for (int i = tid; i < m * m; i += 256) {
        const double2 x = A[(size_t)(i / m) * lda + i % m];
        h = max(h, max(__double2hiint(x.x) & 0x7FFFFFFF, __double2hiint(x.y) & 0x7FFFFFFF));
        a[(i / m) * ld + i % m] = x;
    }
    h = __reduce_max_sync(0xffffffffu, h);
    if (lane == 0) s_max[tid >> 5] = h;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) h = max(h, s_max[i]);
    // (a non-finite matrix is left as it is; a zero one has nothing to scale)
    int ex = (h >> 20) - 1023;  // the largest component is in [2^ex, 2^(ex+1))
    const bool scaled = (ex < -kTriRange || ex > kTriRange) && ex < 1024 && h > 0;
    const int shift = scaled ? max(-1000, min(1000, -ex)) : 0;
    if (scaled) {
        const double up = __hiloint2double((1023 + shift) << 20, 0);
        for (int i = tid; i < m * m; i += 256) {
            double2& x = a[(i / m) * ld + i % m];
            x.x *= up;
            x.y *= up;
        }
        ex = 0;
    }
    // high word of the bound on the square of a column's norm (compared as integers: a comparison of doubles
    // holds the pipe like any other FP64 instruction)
    const int drop = max(0, min(2046, 1023 + 2 * (ex - kTriDrop))) << 20;
    // the reflector of column k but for tau (one warp)
    auto reflector = [&](int k) {
        const int n = m - k - 1;
        double2* v = vb + (k & 1) * m;
        double part = 0.0;
        bool below = false;  // anything to eliminate
        for (int i = lane; i < n; i += 32) {
            const double2 x = a[(k + 1 + i) * ld + k];
            part = fma(x.x, x.x, fma(x.y, x.y, part));
            below = below || x.y != 0.0 || (i > 0 && x.x != 0.0);
        }
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        const double2 alpha = a[(k + 1) * ld + k];
        const bool none = __double2hiint(part) < drop;
        double beta = 0.0;
        if (__any_sync(0xffffffffu, below) && !none) beta = -copysign(sqrt(part), alpha.x);
        for (int i = lane; i < n; i += 32) {
            double2 x = a[(k + 1 + i) * ld + k];
            if (i == 0) x.x -= beta;
            v[i] = x;
        }
        if (lane == 0) {
            s_beta[k & 1] = beta;
            e[k] = none ? 0.0 : beta != 0.0 ? beta : alpha.x;
            d[k] = a[k * ld + k].x;
        }
    };
    if (scaled) __syncthreads();
    if (tid < 32) reflector(0);
    for (int k = 0; k < m - 1; ++k) {
        __syncthreads();
        const int n = m - k - 1;
        double2* a22 = a + (k + 1) * ld + k + 1;
        const double2* v = vb + (k & 1) * m;
        const double beta = s_beta[k & 1];
        const bool any = beta != 0.0;  // (uniform)
        if (tid >= 224) {
            const double2 v0 = v[0];
            double2 t = make_double2(0.0, 0.0);
            if (any) {
                // the two reciprocals on two lanes
                const double inv = 1.0 / (lane & 1 ? fma(v0.x, v0.x, v0.y * v0.y) : beta);
                const double ib = __shfl_sync(0xffffffffu, inv, 0), in = __shfl_sync(0xffffffffu, inv, 1);
                t = make_double2(-(v0.x * in) * ib, -(v0.y * in) * ib);
                if (lane == 0) {
                    s_t = t;
                    s_half = -0.5 * ib * (ib * in);
                }
            }
            if (lane == 0) tau[k] = t;
            for (int i = lane; i < n; i += 32) Vh[(size_t)k * m + k + 1 + i] = v[i];
        }
        if (any) {
            // w = A22 v, four lanes a row; the pairs of lanes sum a component each
            for (int r0 = 0; r0 < n; r0 += 64) {
                const int r = r0 + (tid >> 2);
                double2 acc = make_double2(0.0, 0.0);
                if (r < n)
                    for (int j = tid & 3; j < n; j += 4) {
                        const double2 x = a22[r * ld + j], y = v[j];
                        acc.x = fma(x.x, y.x, fma(-x.y, y.y, acc.x));
                        acc.y = fma(x.x, y.y, fma(x.y, y.x, acc.y));
                    }
                if (r0 + ((tid & ~31) >> 2) < n) {  // (warps without a row skip the sums)
                    const bool up = tid & 1;
                    double h = (up ? acc.y : acc.x) + __shfl_xor_sync(0xffffffffu, up ? acc.x : acc.y, 1);
                    h += __shfl_xor_sync(0xffffffffu, h, 2);
                    if (r < n && (tid & 3) < 2) reinterpret_cast<double*>(w + r)[tid & 1] = h;
                }
            }
            __syncthreads();
            if (tid < 32) {  // w <- tau w - |tau|^2 (v^H w) / 2 v
                double dp = 0.0;
                for (int i = lane; i < n; i += 32) dp = fma(w[i].x, v[i].x, fma(w[i].y, v[i].y, dp));
                for (int o = 16; o > 0; o >>= 1) dp += __shfl_xor_sync(0xffffffffu, dp, o);
                const double g = s_half * dp;
                const double2 t = s_t;
                for (int i = lane; i < n; i += 32) {
                    const double2 x = w[i], y = v[i];
                    w[i] = make_double2(fma(t.x, x.x, fma(-t.y, x.y, g * y.x)), fma(t.x, x.y, fma(t.y, x.x, g * y.y)));
                }
            }
            __syncthreads();
        }
        // A22 -= v w^H + w v^H
        auto update = [&](int i, int j) {
            const double2 vi = v[i], wi = w[i], vj = v[j], wj = w[j];
            double2 x = a22[i * ld + j];
            x.x = fma(-vi.x, wj.x, fma(-vi.y, wj.y, fma(-wi.x, vj.x, fma(-wi.y, vj.y, x.x))));
            x.y = fma(-vi.y, wj.x, fma(vi.x, wj.y, fma(-wi.y, vj.x, fma(wi.x, vj.y, x.y))));
            if (i == j) x.y = 0.0;
            a22[i * ld + j] = x;
            if (j > 0 && i != j) a22[j * ld + i] = make_double2(x.x, -x.y);
        };
        if (tid < 32) {
            if (any)
                for (int i = lane; i < n; i += 32) update(i, 0);
            __syncwarp();
            if (k + 1 < m - 1) reflector(k + 1);
        } else if (any) {
            for (int q = tid - 32; q < n * (n - 1) / 2; q += 224) {  // rows and columns 1 .. n-1
                int i = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
                while ((i + 1) * (i + 2) / 2 <= q) ++i;
                while (i * (i + 1) / 2 > q) --i;
                update(i + 1, q - i * (i + 1) / 2 + 1);
            }
        }
    }
    __syncthreads();
    if (tid == 0) d[m - 1] = a[(m - 1) * ld + m - 1].x;
    if (scaled) {  // (in a loop of its own: beside each column's stores the products would be taken in any case)
        const double back = __hiloint2double((1023 - shift) << 20, 0);
        __syncthreads();
        for (int i = tid; i < m; i += 256) {
            d[i] *= back;
            if (i < m - 1) e[i] *= back;
        }
    }
}

// number of eigenvalues of T smaller than x: sign changes of the leading minors' determinants by their
// three-term recurrence p_i = (d_i - x) p_(i-1) - e_(i-1)^2 p_(i-2) (Wilkinson, The Algebraic Eigenvalue
// Problem, Ch. 5, Sec. 37), T scaled below 2 in magnitude.
// (Eight-band solves: 41 us, 150 us with
// quotients and one warp.)  A ratio p_i / p_(i-1) below 2^-100 is replaced
// by -2^-100 (a shift of d_i by less than 2^-99, and a zero counts as negative), so eight rows change the
// pair by factors between 2^-900 and 2^40 and its rescaling every eight rows keeps it in range.  The
// quotient form has a division in the chain of every row, about 430 cycles on this GPU; a
// multiply-add is 64, and eight unrolled rows keep the loads and differences off the chain.
__device__ __forceinline__ int sturm_count(const double* __restrict__ d, const double* __restrict__ e2, int m, double x) {
    int c = 0;
    double p0 = 1.0, p1 = d[0] - x;
    if (fabs(p1) < 0x1p-100) p1 = -0x1p-100;
    if (p1 < 0.0) ++c;
    for (int i0 = 1; i0 < m; i0 += 8) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {  // (rows m .. of the last group are padding: d = 4, e = 0, no sign change)
            const int i = i0 + q;
            double p = fma(d[i] - x, p1, -e2[i - 1] * p0);
            const int hp = __double2hiint(p), h1 = __double2hiint(p1);
            if ((hp & 0x7FF00000) < (h1 & 0x7FF00000) - (100 << 20))  // -2^-100 p1, without the FP64 pipe
                p = __hiloint2double((h1 - (100 << 20)) ^ (int)0x80000000, __double2loint(p1));
            c += (int)((unsigned)(__double2hiint(p) ^ h1) >> 31);
            p0 = p1;
            p1 = p;
        }
        // divide the pair by the power of two of the larger one
        const int ex = max(__double2hiint(p0) & 0x7FF00000, __double2hiint(p1) & 0x7FF00000);
        const double sc = __hiloint2double(max(0x7FE00000 - ex, 0x00100000), 0);
        p0 *= sc;
        p1 *= sc;
    }
    return c;
}

// one CTA per wanted eigenvalue j < nev, 128 points per round: a warp on each of the SM's four partitions (an
// FP64 instruction holds a partition for 64 cycles, whatever its warp's lanes do); d and e^2, scaled, in
// shared memory (2 (m + 8) doubles)
__global__ void __launch_bounds__(128) k_multisect(const double* __restrict__ d, const double* __restrict__ e, int m, int nev,
                                                  double* __restrict__ evals) {
    extern __shared__ double sms[];
    double *sd = sms, *se = sms + m + 8;
    const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    if (j >= nev) return;
    __shared__ int first[2][4];  // each warp's first point above eigenvalue j, rounds alternating
    // Gershgorin interval (every warp)
    double lo = 1e300, hi = -1e300;
    for (int i = lane; i < m; i += 32) {
        const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < m - 1 ? fabs(e[i]) : 0.0);
        lo = fmin(lo, d[i] - r);
        hi = fmax(hi, d[i] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double span = fmax(hi - lo, 1e-300);
    lo -= 1e-14 * span + 1e-300;
    hi += 1e-14 * span + 1e-300;
    // a power of two near 1 / max(|lo|, |hi|): scaled entries below 2
    int ex = 0;
    frexp(fmax(fabs(lo), fabs(hi)), &ex);
    const double scale = ldexp(1.0, -ex), back = ldexp(1.0, ex);
    for (int i = tid; i < m; i += 128) {
        sd[i] = d[i] * scale;
        const double t = i < m - 1 ? e[i] * scale : 0.0;
        se[i] = t * t;
    }
    if (tid < 8) {
        sd[m + tid] = 4.0;
        se[m + tid] = 0.0;
    }
    lo *= scale;
    hi *= scale;
    __syncthreads();
    for (int round = 0; round < 11; ++round) {
        const auto point = [&](int q) { return fma(hi - lo, (double)(q + 1) * (1.0 / 129.0), lo); };
        const int c = sturm_count(sd, se, m, point(tid));
        const unsigned above = __ballot_sync(0xffffffffu, c > j);
        if (lane == 0) first[round & 1][tid >> 5] = above ? (tid & ~31) + __ffs(above) - 1 : 128;
        __syncthreads();
        const int *fr = first[round & 1], f = min(min(fr[0], fr[1]), min(fr[2], fr[3]));
        const double nlo = f > 0 ? point(f - 1) : lo;
        if (f < 128) hi = point(f);
        lo = nlo;
        if (hi - lo <= 4.0e-16 * fmax(fabs(lo), fabs(hi)) + 1e-300) break;
    }
    if (tid == 0) evals[j] = 0.5 * (lo + hi) * back;
}

// LU with partial pivoting of T - lam, T = tridiag(e, d, e): row i of U is (1 / r[i], c[i], c2[i]), the
// multiplier f[i] eliminates row i + 1, sw[i] = 1 marks a swap of rows i and i + 1 before it.
// The row being eliminated is carried in registers.  Pivots below cut are raised to tiny = eps |T|.
__device__ __forceinline__ void tri_factor(const double* __restrict__ d, const double* __restrict__ e, int m, double lam, double tiny, double cut,
                                           double* __restrict__ r, double* __restrict__ c, double* __restrict__ c2,
                                           double* __restrict__ f, unsigned char* __restrict__ sw) {
    double ai = d[0] - lam, ci = (m > 1) ? e[0] : 0.0;
    for (int i = 0; i < m - 1; ++i) {
        const double sub = e[i];
        double an = d[i + 1] - lam, cn = (i + 1 < m - 1) ? e[i + 1] : 0.0;
        const bool keep = fabs(ai) >= fabs(sub) || fabs(sub) < cut;
        if (keep && fabs(ai) < cut) ai = copysign(tiny, ai);
        const double piv = keep ? ai : sub, inv = 1.0 / piv, fi = (keep ? sub : ai) * inv;
        r[i] = inv;
        f[i] = fi;
        sw[i] = keep ? 0 : 1;
        if (keep) {
            c[i] = ci;
            c2[i] = 0.0;
            an -= fi * ci;
        } else {  // rows i and i+1 swapped
            c[i] = an;
            c2[i] = cn;
            an = ci - fi * an;
            cn = -fi * cn;
        }
        ai = an;
        ci = cn;
    }
    if (fabs(ai) < cut) ai = copysign(tiny, ai);
    r[m - 1] = 1.0 / ai;
}
// solve with that factorisation in place (b -> x): no division in the chains
__device__ __forceinline__ void tri_apply(int m, const double* __restrict__ r, const double* __restrict__ c,
                                          const double* __restrict__ c2, const double* __restrict__ f,
                                          const unsigned char* __restrict__ sw, double* __restrict__ b) {
    double bi = b[0];
#pragma unroll 4
    for (int i = 0; i < m - 1; ++i) {
        double bn = b[i + 1];
        if (sw[i]) {
            const double t = bi;
            bi = bn;
            bn = t;
        }
        b[i] = bi;
        bi = fma(-f[i], bi, bn);
    }
    double x1 = bi * r[m - 1], x2 = 0.0;  // x[i+1], x[i+2]
    b[m - 1] = x1;
#pragma unroll 4
    for (int i = m - 2; i >= 0; --i) {
        const double xi = fma(-c2[i], x2, fma(-c[i], x1, b[i])) * r[i];
        b[i] = xi;
        x2 = x1;
        x1 = xi;
    }
}

// infinity norm of T.  Eigenvalues closer than a part ctol of it form a cluster whose vectors are
// orthogonalised explicitly; outside clusters inverse iteration alone leaves a non-orthogonality of about
// eps |T| / gap: 1e-13 where the chain of dot products is short (m <= 128, ctol = 1e-3), 1e-11 (1e-5) above
__device__ double tri_norm(const double* __restrict__ d, const double* __restrict__ e, int m) {
    double tn = 0.0;
    for (int i = threadIdx.x & 31; i < m; i += 32)
        tn = fmax(tn, fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < m - 1 ? fabs(e[i]) : 0.0));
    for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    return tn;
}

// deterministic pseudo-random start vector (a counter hash of (j, i))
__device__ __forceinline__ double start_entry(int j, int i) {
    unsigned h = 2654435761u * (unsigned)(j + 1) ^ (2246822519u * (unsigned)(i + 1));
    h ^= h >> 15;
    h *= 2246822519u;
    h ^= h >> 13;
    return ((double)(h >> 8) / 16777216.0) - 0.5;
}

// one warp per eigenvalue j: lane 0 factors T - lambda_j once and runs the (sequential) solves of three
// inverse iterations from a deterministic start, the warp shares the O(m) vector work; the normalised
// vector is left in x_j = work + (4 j + 3) m.  Vectors of one cluster are orthogonalised
// afterwards (k_cluster_orth), so every eigenvalue's iterations run in parallel.  kSmem: the factors, T
// and the vector live in shared memory (57 m bytes), else in work and wf.
__host__ __device__ constexpr size_t inviter_smem(int m) { return (size_t)m * (7 * sizeof(double) + 1); }
template <bool kSmem>
__global__ void __launch_bounds__(32)
k_inviter(const double* __restrict__ dg, const double* __restrict__ eg, int m, int nev,
          const double* __restrict__ evals, double* __restrict__ work, double* __restrict__ wf, unsigned char* __restrict__ wsw) {
    extern __shared__ double smi[];
    const int j = blockIdx.x, lane = threadIdx.x;
    if (j >= nev) return;
    const double tn = tri_norm(dg, eg, m);
    double* xg = work + ((size_t)j * 4 + 3) * m;
    double *r = kSmem ? smi : work + (size_t)j * 4 * m, *c = r + m, *c2 = c + m;
    double* f = kSmem ? smi + 3 * m : wf + (size_t)j * m;
    double* x = kSmem ? smi + 4 * m : xg;
    const double *d = dg, *e = eg;
    unsigned char* sw = kSmem ? (unsigned char*)(smi + 7 * m) : wsw + (size_t)j * m;
    if (kSmem) {
        double *sd = smi + 5 * m, *se = smi + 6 * m;
        for (int i = lane; i < m; i += 32) {
            sd[i] = dg[i];
            se[i] = i < m - 1 ? eg[i] : 0.0;
        }
        d = sd;
        e = se;
    }
    const double tiny = 2.2e-16 * fmax(tn, 1e-200);
    const double lam = evals[j];
    for (int i = lane; i < m; i += 32) x[i] = start_entry(j, i);
    __syncwarp();
    if (lane == 0) tri_factor(d, e, m, lam, tiny, 0x1p-100 * fmax(tn, 1e-200), r, c, c2, f, sw);
    for (int it = 0; it < 3; ++it) {
        if (lane == 0) tri_apply(m, r, c, c2, f, sw, x);
        __syncwarp();
        double xm = 0.0;  // rescale before any sum of squares can overflow
        for (int i = lane; i < m; i += 32) xm = fmax(xm, fabs(x[i]));
        for (int o = 16; o > 0; o >>= 1) xm = fmax(xm, __shfl_xor_sync(0xffffffffu, xm, o));
        const double rs = (xm > 0.0 && xm < 1e300) ? 1.0 / xm : 1.0;
        double nrm = 0.0;
        for (int i = lane; i < m; i += 32) {
            x[i] *= rs;
            nrm += x[i] * x[i];
        }
        for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        nrm = 1.0 / sqrt(nrm);
        for (int i = lane; i < m; i += 32) x[i] *= nrm;
        __syncwarp();
    }
    if (kSmem)
        for (int i = lane; i < m; i += 32) xg[i] = x[i];
}

// One CTA per cluster leader (eigenvalue j0 not within ctol of j0-1): the cluster's vectors
// j0..j1-1 are orthonormalised in order by two classical Gram-Schmidt passes against the
// earlier ones (dot products split over the warps), then written as columns of Y (imag 0).
// A vector that loses more than nine tenths of its length (graded couplings beside equal diagonal
// entries make the iterates of several eigenvalues agree) is started afresh, then iterated from what the
// orthogonalisation leaves, at most 8 times, with pivots of at least eps |T| so that eigenvalues that agree
// to rounding count alike; factors in work, wf, wsw.
__global__ void __launch_bounds__(256)
k_cluster_orth(const double* __restrict__ d, const double* __restrict__ e, int m, int nev,
               const double* __restrict__ evals, double* work, double* wf, unsigned char* wsw,
               double2* __restrict__ Y, int ldy) {
    __shared__ double dots[256];
    __shared__ double red[32];
    const int j0 = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (j0 >= nev) return;
    const double tn = tri_norm(d, e, m), ctol = (m <= 128 ? 1e-3 : 1e-5) * tn;  // every warp computes the same value
    if (j0 > 0 && evals[j0] - evals[j0 - 1] <= ctol) return;  // not a cluster leader
    int j1 = j0 + 1;
    while (j1 < nev && evals[j1] - evals[j1 - 1] <= ctol) ++j1;
    auto X = [&](int q) { return work + ((size_t)q * 4 + 3) * m; };
    auto sum = [&](const double* x) {  // |x|^2, the same value in every thread
        double s = 0.0;
        for (int i = tid; i < m; i += 256) s += x[i] * x[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        __syncthreads();
        return t;
    };
    auto scale_by = [&](double* x, double f) {
        for (int i = tid; i < m; i += 256) x[i] *= f;
        __syncthreads();
    };
    for (int j = j0 + 1; j < j1; ++j) {
        double* x = X(j);
        for (int again = 0;; ++again) {
            for (int pass = 0; pass < 2; ++pass) {
                for (int q0 = j0; q0 < j; q0 += 256) {  // coefficients against up to 256 earlier vectors
                    const int nq = min(256, j - q0);
                    for (int q = warp; q < nq; q += 8) {
                        const double* y = X(q0 + q);
                        double s = 0.0;
                        for (int i = lane; i < m; i += 32) s += y[i] * x[i];
                        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                        if (lane == 0) dots[q] = s;
                    }
                    __syncthreads();
                    for (int i = tid; i < m; i += 256) {
                        double v = x[i];
                        for (int q = 0; q < nq; ++q) v -= dots[q] * X(q0 + q)[i];
                        x[i] = v;
                    }
                    __syncthreads();
                }
            }
            const double t = sum(x);
            scale_by(x, t > 0.0 ? 1.0 / sqrt(t) : 0.0);
            if (t > 1e-2 || again == 8) break;
            if (!again || t == 0.0)
                for (int i = tid; i < m; i += 256) x[i] = start_entry(j + nev, i);
            __syncthreads();
            if (tid == 0) {
                double *r = work + (size_t)j * 4 * m, *c = r + m, *c2 = c + m, *f = wf + (size_t)j * m;
                unsigned char* sw = wsw + (size_t)j * m;
                const double tiny = 2.2e-16 * fmax(tn, 1e-200);
                if (!again) tri_factor(d, e, m, evals[j], tiny, tiny, r, c, c2, f, sw);
                tri_apply(m, r, c, c2, f, sw, x);
                double xm = 0.0;
                for (int i = 0; i < m; ++i) xm = fmax(xm, fabs(x[i]));
                red[0] = (xm > 0.0 && xm < 1e300) ? 1.0 / xm : 1.0;
            }
            __syncthreads();
            scale_by(x, red[0]);
            scale_by(x, 1.0 / sqrt(sum(x)));
        }
    }
    for (int j = j0; j < j1; ++j)
        for (int i = tid; i < m; i += 256) Y[(size_t)i * ldy + j] = make_double2(X(j)[i], 0.0);
}

// y <- H_0 H_1 ... H_{m-2} y for column j of Y (one CTA per column)
__global__ void __launch_bounds__(256)
k_backtransf(const double2* __restrict__ Vh, const double2* __restrict__ tau, int m, double2* __restrict__ Y, int ldy) {
    extern __shared__ double2 sy[];
    __shared__ double2 red[32];
    const int j = blockIdx.x, tid = threadIdx.x, bs = blockDim.x;
    for (int i = tid; i < m; i += bs) sy[i] = Y[(size_t)i * ldy + j];
    __syncthreads();
    for (int k = m - 2; k >= 0; --k) {
        const double2 t = tau[k];
        if (t.x == 0.0 && t.y == 0.0) continue;
        const int n = m - k - 1;
        const double2* v = Vh + (size_t)k * m + (k + 1);
        double2 sp = make_double2(0.0, 0.0);
        for (int i = tid; i < n; i += bs) {
            const double2 c = cmulc(v[i], sy[k + 1 + i]);
            sp.x += c.x;
            sp.y += c.y;
        }
        const double2 s = cmul(t, block_sum2(sp, red));
        for (int i = tid; i < n; i += bs) {
            const double2 c = cmul(v[i], s);
            sy[k + 1 + i].x -= c.x;
            sy[k + 1 + i].y -= c.y;
        }
        __syncthreads();
    }
    for (int i = tid; i < m; i += bs) Y[(size_t)i * ldy + j] = sy[i];
}

// the same for m <= 32 kRows: one warp per column, the column in registers (rows lane, lane + 32), the next
// reflector loaded while the present one is applied.  Bound by the chain of FP64 instructions, 64 cycles
// each: the two components of the dot product are summed by half a warp each.  Eight-band solves: 21 us, 74 us
// with the general kernel.
template <int kRows>
__global__ void __launch_bounds__(32)
k_backtransf_small(const double2* __restrict__ Vh, const double2* __restrict__ tau, int m, double2* __restrict__ Y, int ldy) {
    const int j = blockIdx.x, lane = threadIdx.x;
    const bool upper = lane >= 16;
    const double2 z = make_double2(0.0, 0.0);
    double2 y[kRows], v[kRows], nv[kRows];
    const auto ref = [&](int k, int r) { return k >= 0 && r > k && r < m ? Vh[(size_t)k * m + r] : z; };
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
        const int r = lane + 32 * q;
        y[q] = r < m ? Y[(size_t)r * ldy + j] : z;
        v[q] = ref(m - 2, r);
    }
    double2 t = tau[m - 2];
    for (int k = m - 2; k >= 0; --k) {
#pragma unroll
        for (int q = 0; q < kRows; ++q) nv[q] = ref(k - 1, lane + 32 * q);
        const double2 nt = k > 0 ? tau[k - 1] : z;
        if (t.x != 0.0 || t.y != 0.0) {
            double2 sp = cmulc(v[0], y[0]);
#pragma unroll
            for (int q = 1; q < kRows; ++q) {
                sp.x = fma(v[q].x, y[q].x, fma(v[q].y, y[q].y, sp.x));
                sp.y = fma(v[q].x, y[q].y, fma(-v[q].y, y[q].x, sp.y));
            }
            double h = (upper ? sp.y : sp.x) + __shfl_xor_sync(0xffffffffu, upper ? sp.x : sp.y, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
            // s = t (v^H y), a component per half
            const double other = __shfl_xor_sync(0xffffffffu, h, 16);
            const double sh = fma(t.x, h, (upper ? t.y : -t.y) * other);
            const double2 s = make_double2(__shfl_sync(0xffffffffu, sh, 0), __shfl_sync(0xffffffffu, sh, 16));
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                y[q].x = fma(-v[q].x, s.x, fma(v[q].y, s.y, y[q].x));
                y[q].y = fma(-v[q].x, s.y, fma(-v[q].y, s.x, y[q].y));
            }
        }
#pragma unroll
        for (int q = 0; q < kRows; ++q) v[q] = nv[q];
        t = nt;
    }
#pragma unroll
    for (int q = 0; q < kRows; ++q)
        if (lane + 32 * q < m) Y[(size_t)(lane + 32 * q) * ldy + j] = y[q];
}

// the same for 64 < m <= 128 kRows: four warps, one on each partition; rows 32 w + lane + 128 q of the column in
// warp w's registers, so that a reflector costs one barrier; a warp skips its rows above the reflector.
// 176 vectors of 528 to 704 rows: 2.6 ms, 3.8 ms with the general kernel, whose eight warps repeat the sums.
template <int kRows>
__global__ void __launch_bounds__(128)
k_backtransf_rows(const double2* __restrict__ Vh, const double2* __restrict__ tau, int m, double2* __restrict__ Y, int ldy) {
    __shared__ double red[2][4][2];
    const int j = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, last = tid | 31;
    const bool upper = lane >= 16;
    const double2 z = make_double2(0.0, 0.0);
    double2 y[kRows], v[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
        const int r = tid + 128 * q;
        y[q] = r < m ? Y[(size_t)r * ldy + j] : z;
        v[q] = r == m - 1 ? Vh[(size_t)(m - 2) * m + r] : z;
    }
    double2 t = tau[m - 2];
    int buf = 0;
    for (int k = m - 2; k >= 0; --k) {
        double2 nv[kRows];  // the next reflector
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            const int r = tid + 128 * q;
            nv[q] = k > 0 && r >= k && r < m ? Vh[(size_t)(k - 1) * m + r] : z;
        }
        const double2 nt = k > 0 ? tau[k - 1] : z;
        if (t.x != 0.0 || t.y != 0.0) {  // (uniform)
            double2 sp = z;
#pragma unroll
            for (int q = 0; q < kRows; ++q)
                if (last + 128 * q > k) {
                    sp.x = fma(v[q].x, y[q].x, fma(v[q].y, y[q].y, sp.x));
                    sp.y = fma(v[q].x, y[q].y, fma(-v[q].y, y[q].x, sp.y));
                }
            double h = (upper ? sp.y : sp.x) + __shfl_xor_sync(0xffffffffu, upper ? sp.x : sp.y, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
            if ((lane & 15) == 0) red[buf][warp][upper] = h;
            __syncthreads();
            const double(*rd)[2] = red[buf];
            buf ^= 1;  // (not k & 1: skipped reflectors have no barrier)
            h = (rd[0][upper] + rd[1][upper]) + (rd[2][upper] + rd[3][upper]);
            const double other = __shfl_xor_sync(0xffffffffu, h, 16);
            const double sh = fma(t.x, h, (upper ? t.y : -t.y) * other);
            const double2 s = make_double2(__shfl_sync(0xffffffffu, sh, 0), __shfl_sync(0xffffffffu, sh, 16));
#pragma unroll
            for (int q = 0; q < kRows; ++q)
                if (last + 128 * q > k) {
                    y[q].x = fma(-v[q].x, s.x, fma(v[q].y, s.y, y[q].x));
                    y[q].y = fma(-v[q].x, s.y, fma(-v[q].y, s.x, y[q].y));
                }
        }
#pragma unroll
        for (int q = 0; q < kRows; ++q) v[q] = nv[q];
        t = nt;
    }
#pragma unroll
    for (int q = 0; q < kRows; ++q)
        if (tid + 128 * q < m) Y[(size_t)(tid + 128 * q) * ldy + j] = y[q];
}

}  // namespace

size_t heev_work_bytes(int m, int nev) {
    size_t b = 0;
    b += align_up((size_t)m * m * sizeof(double2), 256);      // Vh
    b += align_up((size_t)m * sizeof(double2), 256);          // tau
    b += align_up((size_t)2 * m * sizeof(double2), 256) * 2;  // wbuf, published rows (double-buffered)
    b += align_up((size_t)m * sizeof(double), 256) * 2;       // d, e
    b += align_up((size_t)nev * 4 * m * sizeof(double), 256); // inverse-iteration scratch
    b += align_up((size_t)nev * m * sizeof(double), 256) + align_up((size_t)nev * m, 256);
    return b;
}

// Lowest nev eigenpairs of the Hermitian m x m matrix A (lda; destroyed).  evals: nev
// doubles (device, increasing); Y: m x nev (device, row-major, ld ldy) eigenvectors as columns.
// the process-wide stream of a device for cooperative launches (created on first use)
static qm_status cooperative_stream(int dev, cudaStream_t* out) {
    static std::mutex mu;
    static std::map<int, cudaStream_t> streams;
    std::lock_guard<std::mutex> lk(mu);
    auto it = streams.find(dev);
    if (it == streams.end()) {
        cudaStream_t cs = nullptr;
        qm_status st = cuda_check(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "cooperative stream");
        if (st) return st;
        it = streams.emplace(dev, cs).first;
    }
    *out = it->second;
    return QM_OK;
}

qm_status heev_lowest(double2* A, int lda, int m, int nev, double* evals, double2* Y, int ldy, void* work,
                      cudaStream_t s) {
    if (m <= 0 || nev <= 0) return QM_OK;
    if (nev > m) return fail(QM_ERR_ARG, "heev_lowest: nev > m");
    char* w = (char*)work;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = w + off;
        off += align_up(bytes, 256);
        return p;
    };
    double2* Vh = (double2*)take((size_t)m * m * sizeof(double2));
    double2* tau = (double2*)take((size_t)m * sizeof(double2));
    double2* wbuf = (double2*)take((size_t)2 * m * sizeof(double2));
    double2* prow = (double2*)take((size_t)2 * m * sizeof(double2));
    double* d = (double*)take((size_t)m * sizeof(double));
    double* e = (double*)take((size_t)m * sizeof(double));
    double* iw = (double*)take((size_t)nev * 4 * m * sizeof(double));
    double* wf = (double*)take((size_t)nev * m * sizeof(double));  // multipliers and swaps beyond shared memory
    unsigned char* wsw = (unsigned char*)take((size_t)nev * m);
    qm_status st;
    if (m == 1) {
        // T = (a11): copy the real diagonal, eigenvector 1
        cudaMemcpy2DAsync(evals, sizeof(double), A, sizeof(double2), sizeof(double), 1, cudaMemcpyDeviceToDevice, s);
        const double2 one = make_double2(1.0, 0.0);
        cudaMemcpyAsync(Y, &one, sizeof(double2), cudaMemcpyHostToDevice, s);
        return cuda_check(cudaGetLastError(), "heev m=1");
    }
    if (m <= kTriSmall) {
        const size_t smem = ((size_t)m * (m + 1) + 3 * m) * sizeof(double2);
        if ((st = allow_dynamic_smem((const void*)k_tridiag_small, smem, "heev_lowest: reduction kernel"))) return st;
        ProfScope pf(PF_TRIDIAG, s);
        k_tridiag_small<<<1, 256, smem, s>>>(A, lda, m, Vh, tau, d, e);
    } else {
        int dev = 0, sms = 152;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        // one-barrier reduction: one CTA per SM (the FP64 work of a column is spread over the
        // whole GPU); rows in shared memory when they fit, else updated in place in A.  Beyond
        // 4 m vectors of shared memory, the two-barrier kernel (shared memory for 2 vectors only).
        const int G = std::max(1, std::min(sms, m));
        const size_t vec = 4 * (size_t)m * sizeof(double2);
        const size_t rows = (size_t)((m + G - 1) / G) * m * sizeof(double2);
        const void* kern = nullptr;
        size_t smem = 0;
        int blocks = G;
        if (vec + rows <= 200 * 1024) {
            kern = (const void*)k_tridiag_rows<true>;
            smem = vec + rows;
        } else if (vec <= 200 * 1024) {
            kern = (const void*)k_tridiag_rows<false>;
            smem = vec;
        } else {
            kern = (const void*)k_tridiag;
            smem = 2 * (size_t)m * sizeof(double2);
            if (smem > 200 * 1024) return fail(QM_ERR_UNSUPPORTED, "heev_lowest: m too large for the reduction kernel");
        }
        if ((st = allow_dynamic_smem(kern, smem, "heev_lowest: reduction kernel"))) return st;
        int occ = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 256, smem);
        if (occ < 1) return fail(QM_ERR_UNSUPPORTED, "heev_lowest: reduction kernel does not fit an SM");
        if (kern == (const void*)k_tridiag)  // fewer CTAs: two barriers per column
            blocks = std::min(std::min(occ * sms, std::max(1, (m + 7) / 8)), 64);
        blocks = std::min(blocks, occ * sms);
        if (kern != (const void*)k_tridiag && blocks != G)
            return fail(QM_ERR_UNSUPPORTED, "heev_lowest: reduction grid not resident");
        void* args_old[] = {(void*)&A, (void*)&lda, (void*)&m, (void*)&Vh, (void*)&tau, (void*)&d, (void*)&e,
                            (void*)&wbuf};
        void* args_new[] = {(void*)&A, (void*)&lda, (void*)&m, (void*)&Vh, (void*)&tau, (void*)&d, (void*)&e,
                            (void*)&wbuf, (void*)&prow};
        void** args = kern == (const void*)k_tridiag ? args_old : args_new;
        // Cooperative grids of concurrent callers (other host threads, other streams) must not
        // be resident at the same time: two partly resident grids could each wait at a grid
        // barrier for CTAs the other holds.  Every cooperative launch therefore goes through
        // one stream per device, joined to the caller's stream by events.
        cudaStream_t cs = nullptr;
        if ((st = cooperative_stream(dev, &cs))) return st;
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        if ((st = cuda_check(cudaEventCreateWithFlags(&e0, cudaEventDisableTiming), "event")) ||
            (st = cuda_check(cudaEventCreateWithFlags(&e1, cudaEventDisableTiming), "event")))
            return st;
        st = cuda_check(cudaEventRecord(e0, s), "event record");
        if (!st) st = cuda_check(cudaStreamWaitEvent(cs, e0, 0), "cooperative stream wait");
        if (!st) {
            ProfScope pf(PF_TRIDIAG, cs);
            st = cuda_check(cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3(256), args, smem, cs),
                            "k_tridiag cooperative launch");
        }
        if (!st) st = cuda_check(cudaEventRecord(e1, cs), "event record");
        if (!st) st = cuda_check(cudaStreamWaitEvent(s, e1, 0), "stream wait");
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        if (st) return st;
    }
    {
        const size_t smem = 2 * (size_t)(m + 8) * sizeof(double);
        if ((st = allow_dynamic_smem((const void*)k_multisect, smem, "heev_lowest: multisection"))) return st;
        ProfScope pf(PF_MULTISECT, s);
        k_multisect<<<nev, 128, smem, s>>>(d, e, m, nev, evals);
    }
    {
        // shared memory while every eigenvalue's CTA is resident at once (1 KB of it is the system's)
        int dev = 0, sms = 152;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const size_t per = inviter_smem(m) + 1024;
        const bool fits = per <= 200 * 1024 && nev <= sms * (int)(224 * 1024 / per);
        const size_t smem = fits ? inviter_smem(m) : 0;
        const void* kern = fits ? (const void*)k_inviter<true> : (const void*)k_inviter<false>;
        if ((st = allow_dynamic_smem(kern, smem, "heev_lowest: inverse iteration"))) return st;
        ProfScope pf(PF_INVITER, s);
        (fits ? k_inviter<true> : k_inviter<false>)<<<nev, 32, smem, s>>>(d, e, m, nev, evals, iw, wf, wsw);
    }
    {
        ProfScope pf(PF_INVITER, s);
        k_cluster_orth<<<nev, 256, 0, s>>>(d, e, m, nev, evals, iw, wf, wsw, Y, ldy);
    }
    {
        const size_t smem = (size_t)m * sizeof(double2);
        if ((st = allow_dynamic_smem((const void*)k_backtransf, smem, "heev_lowest: back-transformation"))) return st;
        ProfScope pf(PF_BACKTR, s);
        if (m <= 32) k_backtransf_small<1><<<nev, 32, 0, s>>>(Vh, tau, m, Y, ldy);
        else if (m <= 64) k_backtransf_small<2><<<nev, 32, 0, s>>>(Vh, tau, m, Y, ldy);
        else if (m <= 256) k_backtransf_rows<2><<<nev, 128, 0, s>>>(Vh, tau, m, Y, ldy);
        else if (m <= 512) k_backtransf_rows<4><<<nev, 128, 0, s>>>(Vh, tau, m, Y, ldy);
        else if (m <= 768) k_backtransf_rows<6><<<nev, 128, 0, s>>>(Vh, tau, m, Y, ldy);
        else k_backtransf<<<nev, 256, smem, s>>>(Vh, tau, m, Y, ldy);
    }
    return cuda_check(cudaGetLastError(), "heev launches");
}

}  // namespace qm

using namespace qm;

extern "C" qm_status qm_eigh_lowest(int m, int nev, const void* A, int lda, double* evals, void* Y, int ldy,
                                    void* stream) {
    clear_error();
    if (m <= 0 || nev <= 0 || nev > m) return fail(QM_ERR_ARG, "qm_eigh_lowest: need 0 < nev <= m");
    if (!A || !evals || !Y || lda < m || ldy < nev) return fail(QM_ERR_ARG, "qm_eigh_lowest: bad pointer or ld");
    if ((uintptr_t)A % 16 || (uintptr_t)Y % 16) return fail(QM_ERR_ARG, "qm_eigh_lowest: A, Y not 16-byte aligned");
    if (2 * (size_t)m * sizeof(double2) > 200 * 1024) return fail(QM_ERR_UNSUPPORTED, "qm_eigh_lowest: m > 6400");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t a_bytes = align_up((size_t)m * m * sizeof(double2), 256);
    void* work = nullptr;
    qm_status st = cuda_check(cudaMallocAsync(&work, a_bytes + heev_work_bytes(m, nev), s), "qm_eigh_lowest alloc");
    if (st) return st;
    double2* Aw = (double2*)work;
    st = cuda_check(cudaMemcpy2DAsync(Aw, (size_t)m * sizeof(double2), A, (size_t)lda * sizeof(double2),
                                      (size_t)m * sizeof(double2), m, cudaMemcpyDeviceToDevice, s),
                    "qm_eigh_lowest copy");
    if (!st) st = heev_lowest(Aw, m, m, nev, evals, (double2*)Y, ldy, (char*)work + a_bytes, s);
    cudaFreeAsync(work, s);
    return st;
}
