// FP32 FFT path on two transforms at once (the precision form's H psi and GW kernels).
//
// The same data flow as fft_kernels.cuh (x sticks -> yz planes -> x sticks, digit-reversed
// positions, V laid out in that order); what differs is what bounds it.  The single-transform
// kernels spent two thirds of their issue slots on other things than butterflies (index arithmetic,
// twiddle loads, shared-memory accesses) and a third of their shared-memory traffic on clearing
// planes, scattering into them and transforming rows that hold nothing.  Here
//  * every value is a pair of transforms (two bands, two band pairs at Gamma, two right-hand states
//    in GW) held as packed pairs (re, re'), (im, im'): one index computation, one twiddle, one
//    16-byte shared-memory access and one packed instruction (add/mul/fma.f32x2) serve both;
//  * the first pass of an axis reads global memory and the last one writes it (x: the sphere itself,
//    by the run of plane waves of a stick; y: the sticks of a row by a (row, y) -> stick table), so
//    nothing is cleared, scattered or gathered in between;
//  * rows of the plane that hold no stick are neither transformed nor touched: the z passes know the
//    active rows [0, lo) and [hi, N3).
// Measured (us, single / paired): GW 32 x 64 pairs of the 64-atom cell, product kernel 2375 / 1525; plane
// kernel 1253 / 1165 (96 x 96 x 48, 288 bands), 252 / 200 (72^3, 160 bands), 83 / 72 (72 x 72 x 36, 81
// bands), 943 / 959 (90^3, 240 transforms, one CTA per SM); x passes 335 + 292 / 308 + 278, 12 + 14 /
// 11 + 14, Gamma 135 + 315 / 111 + 225.  What bounds the plane kernel now: 0.69 of the shared-memory
// wavefronts and 0.46 of the issue slots at 24 warps per SM, a quarter of them waiting at the passes'
// barriers (two planes are what shared memory holds); packed instructions take two issue cycles, so
// they save index and twiddle work but no FP32 time.
// Every axis takes two register passes (strided groups of the first stages of the plan, contiguous
// blocks of the rest, see Fused in fft_kernels.cuh), the z axis three with V in the middle one.
// Stick buffer: T[pair][p1][s], 16 bytes per entry.
#pragma once
#include <algorithm>
#include <type_traits>

#include "fft_kernels.cuh"

namespace qm {
namespace pr {

using f2 = unsigned long long;  // two FP32 values
__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 dup(float a) { return pk(a, a); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// a complex value of each of the two transforms
struct __align__(16) c2 {
    f2 x, y;
};
__device__ __forceinline__ c2 zero2() { return c2{0ull, 0ull}; }
__device__ __forceinline__ c2 operator+(const c2& a, const c2& b) { return c2{add2(a.x, b.x), add2(a.y, b.y)}; }
__device__ __forceinline__ c2 operator-(const c2& a, const c2& b) { return c2{sub2(a.x, b.x), sub2(a.y, b.y)}; }
// a + SG i b
template <int SG> __device__ __forceinline__ c2 addi(const c2& a, const c2& b) {
    return SG > 0 ? c2{sub2(a.x, b.y), add2(a.y, b.x)} : c2{add2(a.x, b.y), sub2(a.y, b.x)};
}
// a (w.x + SG i w.y), w the twiddle of both transforms
template <int SG> __device__ __forceinline__ c2 cmulw(const c2& a, const c2& w) {
    return SG > 0 ? c2{sub2(mul2(a.x, w.x), mul2(a.y, w.y)), fma2(a.x, w.y, mul2(a.y, w.x))}
                  : c2{fma2(a.y, w.y, mul2(a.x, w.x)), sub2(mul2(a.y, w.x), mul2(a.x, w.y))};
}

template <int SG, int R> struct Dft;
template <int SG> struct Dft<SG, 2> {
    static __device__ __forceinline__ void run(c2* u) {
        const c2 a = u[0], b = u[1];
        u[0] = a + b;
        u[1] = a - b;
    }
};
template <int SG> struct Dft<SG, 3> {
    static __device__ __forceinline__ void run(c2* u) {
        const c2 t = u[1] + u[2], d = u[1] - u[2];
        const f2 mh = dup(-0.5f), p = dup(SG * 0.86602540378443864676f), n = dup(-SG * 0.86602540378443864676f);
        const c2 m = c2{fma2(t.x, mh, u[0].x), fma2(t.y, mh, u[0].y)};
        u[0] = u[0] + t;
        u[1] = c2{fma2(d.y, n, m.x), fma2(d.x, p, m.y)};
        u[2] = c2{fma2(d.y, p, m.x), fma2(d.x, n, m.y)};
    }
};
template <int SG> struct Dft<SG, 4> {
    static __device__ __forceinline__ void run(c2* u) {
        const c2 a = u[0] + u[2], b = u[0] - u[2], c = u[1] + u[3], d = u[1] - u[3];
        u[0] = a + c;
        u[2] = a - c;
        u[1] = addi<SG>(b, d);
        u[3] = addi<-SG>(b, d);
    }
};
template <int SG> struct Dft<SG, 5> {
    static __device__ __forceinline__ void run(c2* u) {
        const f2 c1 = dup(0.30901699437494742410f), c2_ = dup(-0.80901699437494742410f);
        const f2 s1 = dup(0.95105651629515357212f), s2 = dup(0.58778525229247312917f), m1 = dup(-0.95105651629515357212f);
        const c2 t1 = u[1] + u[4], t2 = u[2] + u[3], d1 = u[1] - u[4], d2 = u[2] - u[3];
        const c2 a1 = c2{fma2(t2.x, c2_, fma2(t1.x, c1, u[0].x)), fma2(t2.y, c2_, fma2(t1.y, c1, u[0].y))};
        const c2 a2 = c2{fma2(t2.x, c1, fma2(t1.x, c2_, u[0].x)), fma2(t2.y, c1, fma2(t1.y, c2_, u[0].y))};
        const c2 b1 = c2{fma2(d2.x, s2, mul2(d1.x, s1)), fma2(d2.y, s2, mul2(d1.y, s1))};
        const c2 b2 = c2{fma2(d2.x, m1, mul2(d1.x, s2)), fma2(d2.y, m1, mul2(d1.y, s2))};
        u[0] = u[0] + (t1 + t2);
        u[1] = addi<SG>(a1, b1);
        u[4] = addi<-SG>(a1, b1);
        u[2] = addi<SG>(a2, b2);
        u[3] = addi<-SG>(a2, b2);
    }
};
template <int SG> struct Dft<SG, 8> {
    static __device__ __forceinline__ void run(c2* u) {
        c2 a[4] = {u[0], u[2], u[4], u[6]}, b[4] = {u[1], u[3], u[5], u[7]};
        Dft<SG, 4>::run(a);
        Dft<SG, 4>::run(b);
        const f2 h = dup(0.70710678118654752440f), g = dup(-0.70710678118654752440f);
        // (1 + SG i) b1 and (1 - SG i) b3; w8 b1 = h p, w8^3 b3 = -h q
        const c2 p = addi<SG>(b[1], b[1]), q = addi<-SG>(b[3], b[3]);
        u[0] = a[0] + b[0];
        u[4] = a[0] - b[0];
        u[1] = c2{fma2(p.x, h, a[1].x), fma2(p.y, h, a[1].y)};
        u[5] = c2{fma2(p.x, g, a[1].x), fma2(p.y, g, a[1].y)};
        u[2] = addi<SG>(a[2], b[2]);
        u[6] = addi<-SG>(a[2], b[2]);
        u[3] = c2{fma2(q.x, g, a[3].x), fma2(q.y, g, a[3].y)};
        u[7] = c2{fma2(q.x, h, a[3].x), fma2(q.y, h, a[3].y)};
    }
};
template <int SG> struct Dft<SG, 9> {
    static __device__ __forceinline__ void run(c2* u) {
        c2 a0[3] = {u[0], u[3], u[6]}, a1[3] = {u[1], u[4], u[7]}, a2[3] = {u[2], u[5], u[8]};
        Dft<SG, 3>::run(a0);
        Dft<SG, 3>::run(a1);
        Dft<SG, 3>::run(a2);
        const c2 w1 = c2{dup(0.76604444311897803520f), dup(0.64278760968653932632f)};
        const c2 w2 = c2{dup(0.17364817766693034885f), dup(0.98480775301220805936f)};
        const c2 w4 = c2{dup(-0.93969262078590838405f), dup(0.34202014332566873304f)};
        a1[1] = cmulw<SG>(a1[1], w1);
        a1[2] = cmulw<SG>(a1[2], w2);
        a2[1] = cmulw<SG>(a2[1], w2);
        a2[2] = cmulw<SG>(a2[2], w4);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c2 col[3] = {a0[k], a1[k], a2[k]};
            Dft<SG, 3>::run(col);
            u[k] = col[0];
            u[k + 3] = col[1];
            u[k + 6] = col[2];
        }
    }
};

// Lengths served, by the larger of their two groups (the split is Fused's, also for plans of two
// stages): up to 12 values, which leaves 24 warps on an SM (80 registers), and 15 to 20 (128 registers).
#define QM_PAIR_SMALL(X) \
    X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) X(72) X(80) X(81) X(90) \
    X(96) X(108)
#define QM_PAIR_BIG(X) X(75) X(100) X(120) X(128) X(144)
inline int pair_class(int n) {  // 0: small groups, 1: big ones, -1: not served
    switch (n) {
#define QM_CASE(n) case n:
        QM_PAIR_SMALL(QM_CASE)
        return 0;
        QM_PAIR_BIG(QM_CASE)
#undef QM_CASE
        return 1;
        default: return -1;
    }
}

// ---------------------------------------------------------------- stages of a group in registers
template <int SG, bool DIF, int R, bool UNIT>
__device__ __forceinline__ void butterfly(c2* v, const c2* tw, int step) {  // twiddle of element k: tw[k * step]
    if constexpr (DIF) Dft<SG, R>::run(v);
    if constexpr (!UNIT) {
#pragma unroll
        for (int k = 1; k < R; ++k) v[k] = cmulw<SG>(v[k], tw[k * step]);
    }
    if constexpr (!DIF) Dft<SG, R>::run(v);
}
template <int SG, bool DIF, int N, int S>
__device__ __forceinline__ void stage_strided(c2* u, int n, const c2* tw) {
    constexpr CPlan P = make_cplan(N);
    constexpr int MB = Fused<N>::MB, R = P.r[S], L = P.L[S], M = L / R, STEP = N / L;
#pragma unroll
    for (int blk = 0; blk < N / L; ++blk)
#pragma unroll
        for (int q = 0; q < M / MB; ++q) {
            c2 v[R];
#pragma unroll
            for (int j = 0; j < R; ++j) v[j] = u[blk * (L / MB) + q + j * (M / MB)];
            butterfly<SG, DIF, R, M == 1>(v, tw, (n + q * MB) * STEP);
#pragma unroll
            for (int j = 0; j < R; ++j) u[blk * (L / MB) + q + j * (M / MB)] = v[j];
        }
}
template <int SG, bool DIF, int N, int S>
__device__ __forceinline__ void stage_block(c2* u, const c2* tw) {
    constexpr CPlan P = make_cplan(N);
    constexpr int MB = Fused<N>::MB, R = P.r[S], L = P.L[S], M = L / R, STEP = N / L;
#pragma unroll
    for (int blk = 0; blk < MB / L; ++blk)
#pragma unroll
        for (int n1 = 0; n1 < M; ++n1) {
            c2 v[R];
#pragma unroll
            for (int j = 0; j < R; ++j) v[j] = u[blk * L + n1 + j * M];
            if (n1 == 0) butterfly<SG, DIF, R, true>(v, tw, 0);
            else butterfly<SG, DIF, R, false>(v, tw, n1 * STEP);
#pragma unroll
            for (int j = 0; j < R; ++j) u[blk * L + n1 + j * M] = v[j];
        }
}
template <int SG, bool DIF, int N, int S, int S1>
__device__ __forceinline__ void strided_stages(c2* u, int n, const c2* tw) {
    if constexpr (S < S1) {
        if constexpr (DIF) stage_strided<SG, DIF, N, S>(u, n, tw);
        strided_stages<SG, DIF, N, S + 1, S1>(u, n, tw);
        if constexpr (!DIF) stage_strided<SG, DIF, N, S>(u, n, tw);
    }
}
template <int SG, bool DIF, int N, int S, int S1>
__device__ __forceinline__ void block_stages(c2* u, const c2* tw) {
    if constexpr (S < S1) {
        if constexpr (DIF) stage_block<SG, DIF, N, S>(u, tw);
        block_stages<SG, DIF, N, S + 1, S1>(u, tw);
        if constexpr (!DIF) stage_block<SG, DIF, N, S>(u, tw);
    }
}

// ---------------------------------------------------------------- element access
// open(line, e0) -> cursor of a line from element e0; get(j) / put(j, v): element e0 + j
__device__ __forceinline__ c2* smem2() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<c2*>(smem_raw);
}
__device__ __forceinline__ c2 ldcg2(const c2* p) {
    const longlong2 v = __ldcg(reinterpret_cast<const longlong2*>(p));
    return c2{(f2)v.x, (f2)v.y};
}
__device__ __forceinline__ void stcg2(c2* p, const c2& v) {
    __stcg(reinterpret_cast<longlong2*>(p), make_longlong2((long long)v.x, (long long)v.y));
}

struct SmemRow {  // line l is row (l < lo ? l : l + skip) of the plane, unit stride
    int ld, lo, skip;
    struct Cur {
        c2* p;
        __device__ __forceinline__ c2 get(int j) const { return p[j]; }
        __device__ __forceinline__ void put(int j, const c2& v) const { p[j] = v; }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{smem2() + (l < lo ? l : l + skip) * ld + e0}; }
};
struct SmemCol {  // line l is column l, stride ld
    int ld;
    struct Cur {
        c2* p;
        int ld;
        __device__ __forceinline__ c2 get(int j) const { return p[j * ld]; }
        __device__ __forceinline__ void put(int j, const c2& v) const { p[j * ld] = v; }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{smem2() + e0 * ld + l, ld}; }
};
struct SmemColAct {  // columns of which only the rows [0, lo) and [hi, N) exist
    int ld, lo, hi;
    struct Cur {
        c2* p;
        int ld, z, lo;
        unsigned gap;
        __device__ __forceinline__ bool act(int j) const { return (unsigned)(z + j - lo) >= gap; }
        __device__ __forceinline__ c2 get(int j) const { return act(j) ? p[j * ld] : zero2(); }
        __device__ __forceinline__ void put(int j, const c2& v) const {
            if (act(j)) p[j * ld] = v;
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{smem2() + e0 * ld + l, ld, e0, lo, (unsigned)(hi - lo)}; }
};
struct StickRow {  // row l of a plane in the stick buffer: element y is stick map[l * n2 + y] (-1: none, zero)
    c2* t;
    const int* map;
    int n2;
    struct Cur {
        c2* t;
        const int* m;
        __device__ __forceinline__ c2 get(int j) const {
            const int s = __ldg(m + j);
            return s >= 0 ? ldcg2(t + s) : zero2();
        }
        __device__ __forceinline__ void put(int j, const c2& v) const {
            const int s = __ldg(m + j);
            if (s >= 0) stcg2(t + s, v);
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{t, map + l * n2 + e0}; }
};
struct StickLines {  // line l is stick l of a tile, element p at t[p * pad + l]
    c2* t;
    int pad;
    struct Cur {
        c2* t;
        int pad;
        __device__ __forceinline__ c2 get(int j) const { return ldcg2(t + (size_t)j * pad); }
        __device__ __forceinline__ void put(int j, const c2& v) const { stcg2(t + (size_t)j * pad, v); }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{t + (size_t)e0 * pad + l, pad}; }
};
struct SlotLines {  // line l is the stick of slot l (shared array of kGammaTile; -1: none)
    c2* t;
    int pad;
    const int2* slot;
    struct Cur {
        c2* t;
        int pad;
        bool on;
        __device__ __forceinline__ c2 get(int j) const { return on ? ldcg2(t + (size_t)j * pad) : zero2(); }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const {
        const int s = slot[l].x;
        return Cur{t + (size_t)e0 * pad + max(s, 0), pad, s >= 0};
    }
};
// The plane waves of a stick: x in [q.y, q.y + q.z) is plane wave q.x + (x - q.y), x in [q.w, q.w + cb)
// is q.x + q.z + (x - q.w), cb the stick's other plane waves (the runs of non-negative and negative G_1)
struct Run {
    int g0, xa, ca, xb, cb;
    __device__ __forceinline__ int find(int x) const {  // plane wave, or -1
        const unsigned d = (unsigned)(x - xa), e = (unsigned)(x - xb);
        return d < (unsigned)ca ? g0 + (int)d : (e < (unsigned)cb ? g0 + ca + (int)e : -1);
    }
};
__device__ __forceinline__ Run run_of(const int4* runs, int s) {
    const int4 q = __ldg(runs + s);
    return Run{q.x, q.y, q.z, q.w, __ldg(&runs[s + 1].x) - q.x - q.z};
}
struct SphereIn {  // two bands (b1 may be NULL: zero)
    const float2 *b0, *b1;
    const int4* runs;
    struct Cur {
        const float2 *b0, *b1;
        Run r;
        int x;
        __device__ __forceinline__ c2 get(int j) const {
            const int g = r.find(x + j);
            if (g < 0) return zero2();
            const float2 a = __ldg(b0 + g), b = b1 ? __ldg(b1 + g) : make_float2(0.f, 0.f);
            return c2{pk(a.x, b.x), pk(a.y, b.y)};
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{b0, b1, run_of(runs, l), e0}; }
};
struct SphereIn4 {  // Gamma: four bands as two transforms psi_a + i psi_b (missing bands zero)
    const float2* b;
    int ld, n;  // bands there are
    const int4* runs;
    struct Cur {
        const float2* b;
        size_t ld;
        int n;
        Run r;
        int x;
        __device__ __forceinline__ c2 get(int j) const {
            const int g = r.find(x + j);
            if (g < 0) return zero2();
            const float2 z = make_float2(0.f, 0.f);
            const float2 p = __ldg(b + g), q = n > 1 ? __ldg(b + ld + g) : z;
            const float2 s = n > 2 ? __ldg(b + 2 * ld + g) : z, t = n > 3 ? __ldg(b + 3 * ld + g) : z;
            return c2{pk(p.x - q.y, s.x - t.y), pk(p.y + q.x, s.y + t.x)};
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{b, (size_t)ld, n, run_of(runs, l), e0}; }
};
struct SphereOut {  // out = F + 1/2|k+G|^2 psi (+ out), two bands (o1 may be NULL)
    const float2 *p0, *p1;
    float2 *o0, *o1;
    const float* kin;
    const int4* runs;
    int acc;
    struct Cur {
        const SphereOut* s;
        Run r;
        int x;
        // the elements of a group four at a time: their loads first, then their stores (a store between
        // them would keep the later loads waiting)
        template <int NA, int STEP, int H>
        __device__ __forceinline__ void band(const c2* u, const float2* p, float2* o) const {
#pragma unroll
            for (int m0 = 0; m0 < NA; m0 += 4) {
                float2 y[4], a[4];
                float k[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (m0 + q >= NA) break;
                    const int g = r.find(x + (m0 + q) * STEP);
                    y[q] = g >= 0 ? __ldg(p + g) : make_float2(0.f, 0.f);
                    k[q] = g >= 0 ? __ldg(s->kin + g) : 0.f;
                    a[q] = g >= 0 && s->acc ? __ldcg(o + g) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (m0 + q >= NA) break;
                    const int g = r.find(x + (m0 + q) * STEP);
                    float re[2], im[2];
                    upk(u[m0 + q].x, re[0], re[1]);
                    upk(u[m0 + q].y, im[0], im[1]);
                    if (g >= 0) o[g] = make_float2(fmaf(k[q], y[q].x, re[H]) + a[q].x, fmaf(k[q], y[q].y, im[H]) + a[q].y);
                }
            }
        }
        template <int NA, int STEP>
        __device__ __forceinline__ void put_all(const c2* u) const {
            band<NA, STEP, 0>(u, s->p0, s->o0);
            if (s->o1) band<NA, STEP, 1>(u, s->p1, s->o1);
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{this, run_of(runs, l), e0}; }
};
struct MelOut {  // conj(F) / N_r, two rows of M (o1 may be NULL)
    float2 *o0, *o1;
    const int4* runs;
    float s;
    struct Cur {
        float2 *o0, *o1;
        float s;
        Run r;
        int x;
        __device__ __forceinline__ void put(int j, const c2& v) const {
            const int g = r.find(x + j);
            if (g < 0) return;
            float a, b, c, d;
            upk(v.x, a, b);
            upk(v.y, c, d);
            o0[g] = make_float2(a * s, -c * s);
            if (o1) o1[g] = make_float2(b * s, -d * s);
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const { return Cur{o0, o1, s, run_of(runs, l), e0}; }
};
struct PlaneOut {  // whole plane in real space, element (z, column) at z * n2 + column: packed, or as two boxes
    c2* u;
    float2 *u0, *u1;  // u NULL: the two transforms apart (u1 may be NULL)
    int n2;
    struct Cur {
        c2* u;
        float2 *u0, *u1;
        int n2;
        __device__ __forceinline__ void put(int j, const c2& v) const {
            if (u) {
                stcg2(u + j * n2, v);
            } else {
                float a, b, c, d;
                upk(v.x, a, b);
                upk(v.y, c, d);
                u0[j * n2] = make_float2(a, c);
                if (u1) u1[j * n2] = make_float2(b, d);
            }
        }
    };
    __device__ __forceinline__ Cur open(int l, int e0) const {
        const int o = e0 * n2 + l;
        return Cur{u ? u + o : nullptr, u ? nullptr : u0 + o, !u && u1 ? u1 + o : nullptr, n2};
    }
};
struct ProductIn {  // u_n conj(u_m) of a left state and the two right states of a packed plane
    const float2* l;
    const c2* r;
    int n2;
    struct Cur {
        const float2* l;
        const c2* r;
        int n2;
        __device__ __forceinline__ c2 get(int j) const {
            const float2 a = __ldg(l + j * n2);
            const longlong2 q = __ldg(reinterpret_cast<const longlong2*>(r + j * n2));
            const f2 ax = dup(a.x), ay = dup(a.y), x = (f2)q.x, y = (f2)q.y;
            return c2{fma2(ay, y, mul2(ax, x)), sub2(mul2(ay, x), mul2(ax, y))};
        }
    };
    __device__ __forceinline__ Cur open(int l_, int e0) const { return Cur{l + e0 * n2 + l_, r + e0 * n2 + l_, n2}; }
};

// ---------------------------------------------------------------- passes
// GF: consecutive threads take consecutive groups of a line (global runs of consecutive elements),
// else consecutive lines (conflict-free: odd row lengths, unit column stride)
template <int SG, bool DIF, bool GF, int N, class Ld, class St>
__device__ __forceinline__ void pass_strided(int nlines, const Ld& ld, const St& st, const c2* tw) {
    using F = Fused<N>;
    const RDiv dl{nlines, 1.0f / (float)nlines};
    for (int t = threadIdx.x; t < nlines * F::MB; t += blockDim.x) {
        int line, n;
        if (GF) {
            line = t / F::MB;
            n = t - line * F::MB;
        } else {
            n = dl.div(t);
            line = t - n * nlines;
        }
        c2 u[F::NA];
        const auto in = ld.open(line, n);
#pragma unroll
        for (int m = 0; m < F::NA; ++m) u[m] = in.get(m * F::MB);
        strided_stages<SG, DIF, N, 0, F::K>(u, n, tw);
        const auto out = st.open(line, n);
        if constexpr (std::is_same_v<St, SphereOut>) {
            out.template put_all<F::NA, F::MB>(u);
        } else {
#pragma unroll
            for (int m = 0; m < F::NA; ++m) out.put(m * F::MB, u[m]);
        }
    }
    __syncthreads();
}
template <int SG, bool DIF, int N, class Ld, class St>
__device__ __forceinline__ void pass_block(int nlines, const Ld& ld, const St& st, const c2* tw) {
    using F = Fused<N>;
    const RDiv dl{nlines, 1.0f / (float)nlines};
    for (int t = threadIdx.x; t < nlines * F::NA; t += blockDim.x) {
        const int b = dl.div(t), line = t - b * nlines;
        c2 u[F::MB];
        const auto in = ld.open(line, b * F::MB);
#pragma unroll
        for (int i = 0; i < F::MB; ++i) u[i] = in.get(i);
        block_stages<SG, DIF, N, F::K, F::P.nst>(u, tw);
        const auto out = st.open(line, b * F::MB);
#pragma unroll
        for (int i = 0; i < F::MB; ++i) out.put(i, u[i]);
    }
    __syncthreads();
}

// whole-axis steps of one length
template <int N>
__device__ __forceinline__ void y_inverse(StickRow in, SmemRow row, int nrow, int tw) {
    pass_strided<+1, true, true, N>(nrow, in, row, smem2() + tw);
    pass_block<+1, true, N>(nrow, row, row, smem2() + tw);
}
template <int N>
__device__ __forceinline__ void y_forward(SmemRow row, StickRow out, int nrow, int tw) {
    pass_block<-1, false, N>(nrow, row, row, smem2() + tw);
    pass_strided<-1, false, true, N>(nrow, row, out, smem2() + tw);
}
// inverse z on every column, multiplication by the real V (element (z, column) at v[z * n2 + column],
// digit-reversed positions), forward z
template <int N>
__device__ __forceinline__ void z_vmul(SmemColAct act, int n2, const float* v, int twi) {
    using F = Fused<N>;
    const c2* tw = smem2() + twi;
    const SmemCol col{act.ld};
    pass_strided<+1, true, false, N>(n2, act, col, tw);
    const RDiv dl{n2, 1.0f / (float)n2};
    for (int t = threadIdx.x; t < n2 * F::NA; t += blockDim.x) {
        const int b = dl.div(t), line = t - b * n2;
        float sc[F::MB];
#pragma unroll
        for (int i = 0; i < F::MB; ++i) sc[i] = __ldg(v + (b * F::MB + i) * n2 + line);
        c2 u[F::MB];
        const auto p = col.open(line, b * F::MB);
#pragma unroll
        for (int i = 0; i < F::MB; ++i) u[i] = p.get(i);
        block_stages<+1, true, N, F::K, F::P.nst>(u, tw);
#pragma unroll
        for (int i = 0; i < F::MB; ++i) {
            const f2 s = dup(sc[i]);
            u[i] = c2{mul2(u[i].x, s), mul2(u[i].y, s)};
        }
        block_stages<-1, false, N, F::K, F::P.nst>(u, tw);
#pragma unroll
        for (int i = 0; i < F::MB; ++i) p.put(i, u[i]);
    }
    __syncthreads();
    pass_strided<-1, false, false, N>(n2, col, act, tw);
}
template <int N>
__device__ __forceinline__ void z_real(SmemColAct act, PlaneOut out, int n2, int tw) {
    pass_strided<+1, true, false, N>(n2, act, SmemCol{act.ld}, smem2() + tw);
    pass_block<+1, true, N>(n2, SmemCol{act.ld}, out, smem2() + tw);
}
template <int N>
__device__ __forceinline__ void z_product(ProductIn in, SmemColAct act, int n2, int tw) {
    pass_block<-1, false, N>(n2, in, SmemCol{act.ld}, smem2() + tw);
    pass_strided<-1, false, false, N>(n2, SmemCol{act.ld}, act, smem2() + tw);
}
template <int N, class In>
__device__ __forceinline__ void x_inverse(In in, StickLines out, int ld, int ns, int tw) {
    const SmemRow row{ld, ns, 0};
    pass_strided<+1, true, true, N>(ns, in, row, smem2() + tw);
    pass_block<+1, true, N>(ns, row, out, smem2() + tw);
}
template <int N, class In, class Out>
__device__ __forceinline__ void x_forward(In in, Out out, int ld, int ns, int tw) {
    const SmemRow row{ld, ns, 0};
    pass_block<-1, false, N>(ns, in, row, smem2() + tw);
    pass_strided<-1, false, true, N>(ns, row, out, smem2() + tw);
}

__device__ __forceinline__ void stage_tw(int at, const float2* tw, int n) {
    c2* dst = smem2() + at;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float2 w = __ldg(tw + i);
        dst[i] = c2{dup(w.x), dup(w.y)};
    }
}

// call with n_ the length (a compile-time constant); the kernels of class 0 hold the small lengths only
template <int N> struct Len {
    static constexpr int n = N;
};
template <int BIG, class F>
__device__ __forceinline__ void dispatch(int n, const F& f) {
    switch (n) {
#define QM_CASE(k) \
    case k: f(Len<k>()); return;
        QM_PAIR_SMALL(QM_CASE)
        default: break;
    }
    if constexpr (BIG) {
        switch (n) {
            QM_PAIR_BIG(QM_CASE)
            default: break;
        }
    }
#undef QM_CASE
}
#define QM_PAIR_DISPATCH(len, call)          \
    dispatch<BIG>(len, [&](auto l_) {        \
        constexpr int n_ = decltype(l_)::n;  \
        call;                                \
    });

constexpr int kPairTile = 32;      // sticks per CTA of the x passes
constexpr int kPairStick = 256;    // their threads at most (see stick_nt)

// ---------------------------------------------------------------- kernels
// x: sphere -> sticks.  gamma: two band pairs per packed pair, nb = bands there are
template <int BIG>
__global__ void __launch_bounds__(kPairStick, BIG ? 2 : 3)
k_pair_x_inverse(const float2* __restrict__ psi, int ld_psi, int nb, int gamma, const int4* __restrict__ runs, int nstick,
                 int nstick_pad, int N1, const float2* __restrict__ tw_x, int ldx, c2* __restrict__ T) {
    const int tw = kPairTile * ldx;
    stage_tw(tw, tw_x, N1);
    __syncthreads();
    const int s0 = blockIdx.x * kPairTile, ns = min(kPairTile, nstick - s0);
    const StickLines out{T + (size_t)blockIdx.y * N1 * nstick_pad + s0, nstick_pad};
    if (gamma) {
        const int b = 4 * blockIdx.y;
        const SphereIn4 in{psi + (size_t)b * ld_psi, ld_psi, nb - b, runs + s0};
        QM_PAIR_DISPATCH(N1, x_inverse<n_>(in, out, ldx, ns, tw))
    } else {
        const int b = 2 * blockIdx.y;
        const float2* p = psi + (size_t)b * ld_psi;
        const SphereIn in{p, b + 1 < nb ? p + ld_psi : nullptr, runs + s0};
        QM_PAIR_DISPATCH(N1, x_inverse<n_>(in, out, ldx, ns, tw))
    }
}

// y and z of one yz plane per (pair, p1): inverse, V, forward, in place in the stick buffer
template <int BIG>
__global__ void __launch_bounds__(BIG ? 512 : 768, 1)
k_pair_plane(c2* __restrict__ T, int nstick_pad, const int* __restrict__ ymap, int lo, int hi, int N1, int N2, int N3,
             const float2* __restrict__ tw_y, const float2* __restrict__ tw_z, int ldy, const float* __restrict__ Vt) {
    const int twy = N3 * ldy, twz = twy + N2, nrow = lo + N3 - hi;
    stage_tw(twy, tw_y, N2);
    stage_tw(twz, tw_z, N3);
    __syncthreads();
    const StickRow sticks{T + ((size_t)blockIdx.y * N1 + blockIdx.x) * nstick_pad, ymap, N2};
    const SmemRow row{ldy, lo, hi - lo};
    const SmemColAct act{ldy, lo, hi};
    QM_PAIR_DISPATCH(N2, y_inverse<n_>(sticks, row, nrow, twy))
    const float* v = Vt + (size_t)blockIdx.x * N3 * N2;
    QM_PAIR_DISPATCH(N3, z_vmul<n_>(act, N2, v, twz))
    QM_PAIR_DISPATCH(N2, y_forward<n_>(row, sticks, nrow, twy))
}

// x: sticks -> sphere, kinetic term (and what is already in out when acc)
template <int BIG>
__global__ void __launch_bounds__(kPairStick, BIG ? 2 : 3)
k_pair_x_forward(c2* __restrict__ T, int nb, const int4* __restrict__ runs, int nstick, int nstick_pad, int N1,
                 const float2* __restrict__ tw_x, int ldx, const float* __restrict__ kin, const float2* __restrict__ psi,
                 int ld_psi, float2* __restrict__ out, int ld_out, int acc) {
    const int tw = kPairTile * ldx;
    stage_tw(tw, tw_x, N1);
    __syncthreads();
    const int s0 = blockIdx.x * kPairTile, ns = min(kPairTile, nstick - s0), b = 2 * blockIdx.y;
    const StickLines in{T + (size_t)blockIdx.y * N1 * nstick_pad + s0, nstick_pad};
    const float2* p = psi + (size_t)b * ld_psi;
    float2* o = out + (size_t)b * ld_out;
    const bool two = b + 1 < nb;
    const SphereOut so{p, two ? p + ld_psi : nullptr, o, two ? o + ld_out : nullptr, kin, runs + s0, acc};
    QM_PAIR_DISPATCH(N1, x_forward<n_>(in, so, ldx, ns, tw))
}

// the same at Gamma for two band pairs: each tile holds every stick beside the stick of -G, so that
// the two bands of a transform separate as in k_stick_forward_gamma
template <int BIG>
__global__ void __launch_bounds__(kPairStick, BIG ? 2 : 3)
k_pair_x_forward_gamma(c2* __restrict__ T, int nb, const int2* __restrict__ gtile, const int* __restrict__ stick_g0,
                       const int2* __restrict__ g_code, int nstick_pad, int N1, const float2* __restrict__ tw_x, int ldx,
                       const float* __restrict__ kin, const float2* __restrict__ psi, int ld_psi, float2* __restrict__ out,
                       int ld_out, int acc) {
    __shared__ int2 slot[kGammaTile];
    __shared__ int gstart[kGammaTile], goff[kGammaTile + 1];
    const int tid = threadIdx.x, tw = kGammaTile * ldx;
    stage_tw(tw, tw_x, N1);
    if (tid < kGammaTile) {
        const int2 sl = __ldg(gtile + (size_t)blockIdx.x * kGammaTile + tid);
        const int g0 = sl.x >= 0 ? __ldg(stick_g0 + sl.x) : 0;
        const int c = sl.x >= 0 ? __ldg(stick_g0 + sl.x + 1) - g0 : 0;
        slot[tid] = sl;
        gstart[tid] = g0;
        int sum = c;  // inclusive scan over the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, sum, o);
            if (tid >= o) sum += y;
        }
        goff[tid + 1] = sum;
        if (tid == 0) goff[0] = 0;
    }
    __syncthreads();
    const SlotLines in{T + (size_t)blockIdx.y * N1 * nstick_pad, nstick_pad, slot};
    const SmemRow row{ldx, kGammaTile, 0};
    QM_PAIR_DISPATCH(N1, x_forward<n_>(in, row, ldx, kGammaTile, tw))
    const c2* lines = smem2();
    const int total = goff[kGammaTile];
    for (int t = tid; t < total; t += blockDim.x) {
        int l = 0, h = kGammaTile;  // slot with goff[l] <= t < goff[l + 1]
        while (h - l > 1) {
            const int mid = (l + h) >> 1;
            if (goff[mid] <= t) l = mid;
            else h = mid;
        }
        const int g = gstart[l] + (t - goff[l]);
        const int x = __ldg(g_code + g).y, xm = x ? N1 - x : 0;
        const c2 F = lines[l * ldx + x], M = lines[slot[l].y * ldx + xm];
        const float k = __ldg(kin + g);
        float fx[2], fy[2], mx[2], my[2];
        upk(F.x, fx[0], fx[1]);
        upk(F.y, fy[0], fy[1]);
        upk(M.x, mx[0], mx[1]);
        upk(M.y, my[0], my[1]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int b = 4 * blockIdx.y + q, j = q >> 1;
            if (b >= nb) break;
            const float re = (q & 1) ? fy[j] + my[j] : fx[j] + mx[j], im = (q & 1) ? mx[j] - fx[j] : fy[j] - my[j];
            const float2 y = __ldg(psi + (size_t)b * ld_psi + g);
            float2* o = out + (size_t)b * ld_out + g;
            float2 r = make_float2(fmaf(k, y.x, 0.5f * re), fmaf(k, y.y, 0.5f * im));
            if (acc) {
                const float2 a = *o;
                r.x += a.x;
                r.y += a.y;
            }
            *o = r;
        }
    }
}

// GW: one real-space plane per (pair, p1), packed (U) or as single boxes (U0: box of each state)
template <int BIG>
__global__ void __launch_bounds__(BIG ? 512 : 768, 1)
k_pair_real(c2* __restrict__ T, int nstick_pad, const int* __restrict__ ymap, int lo, int hi, int N1, int N2, int N3,
            const float2* __restrict__ tw_y, const float2* __restrict__ tw_z, int ldy, c2* __restrict__ U,
            float2* __restrict__ U0, int nst) {
    const int twy = N3 * ldy, twz = twy + N2, nrow = lo + N3 - hi;
    stage_tw(twy, tw_y, N2);
    stage_tw(twz, tw_z, N3);
    __syncthreads();
    const StickRow sticks{T + ((size_t)blockIdx.y * N1 + blockIdx.x) * nstick_pad, ymap, N2};
    const SmemRow row{ldy, lo, hi - lo};
    const SmemColAct act{ldy, lo, hi};
    QM_PAIR_DISPATCH(N2, y_inverse<n_>(sticks, row, nrow, twy))
    const size_t np = (size_t)N2 * N3;
    PlaneOut po{nullptr, nullptr, nullptr, N2};
    if (U) {
        po.u = U + ((size_t)blockIdx.y * N1 + blockIdx.x) * np;
    } else {
        po.u0 = U0 + ((size_t)(2 * blockIdx.y) * N1 + blockIdx.x) * np;
        po.u1 = 2 * (int)blockIdx.y + 1 < nst ? po.u0 + (size_t)N1 * np : nullptr;
    }
    QM_PAIR_DISPATCH(N3, z_real<n_>(act, po, N2, twz))
}

// GW: plane p1 of the products of left state n with the right states 2m, 2m + 1 (job = n * nrp + m),
// forward z, forward y on the rows of the q sphere, onto its sticks.  The jobs are the fast grid dimension: all
// jobs of a plane read the same few planes of U from L2 (plane-fastest streams every right box per left state).
template <int BIG>
__global__ void __launch_bounds__(BIG ? 512 : 768, 1)
k_pair_product(const float2* __restrict__ UL, const c2* __restrict__ UR, int nrp, int job0, c2* __restrict__ Te, int nstick_pad,
               const int* __restrict__ ymap, int lo, int hi, int N1, int N2, int N3, const float2* __restrict__ tw_y,
               const float2* __restrict__ tw_z, int ldy) {
    const int twy = N3 * ldy, twz = twy + N2, nrow = lo + N3 - hi;
    stage_tw(twy, tw_y, N2);
    stage_tw(twz, tw_z, N3);
    __syncthreads();
    const int job = job0 + blockIdx.x, n = job / nrp, m = job - n * nrp;
    const size_t np = (size_t)N2 * N3;
    const ProductIn in{UL + ((size_t)n * N1 + blockIdx.y) * np, UR + ((size_t)m * N1 + blockIdx.y) * np, N2};
    QM_PAIR_DISPATCH(N3, z_product<n_>(in, SmemColAct{ldy, lo, hi}, N2, twz))
    const StickRow sticks{Te + ((size_t)blockIdx.x * N1 + blockIdx.y) * nstick_pad, ymap, N2};
    QM_PAIR_DISPATCH(N2, y_forward<n_>(SmemRow{ldy, lo, hi - lo}, sticks, nrow, twy))
}

// GW: forward x on the q sphere's sticks, M rows of the job's two pairs
template <int BIG>
__global__ void __launch_bounds__(kPairStick, BIG ? 2 : 3)
k_pair_mel(c2* __restrict__ Te, int nr, int nrp, int job0, const int4* __restrict__ runs, int nstick, int nstick_pad, int N1,
           const float2* __restrict__ tw_x, int ldx, float inv_nr, float2* __restrict__ M, int ld_m) {
    const int tw = kPairTile * ldx;
    stage_tw(tw, tw_x, N1);
    __syncthreads();
    const int s0 = blockIdx.x * kPairTile, ns = min(kPairTile, nstick - s0);
    const int job = job0 + blockIdx.y, n = job / nrp, m = 2 * (job - n * nrp);
    const StickLines in{Te + (size_t)blockIdx.y * N1 * nstick_pad + s0, nstick_pad};
    float2* o = M + ((size_t)n * nr + m) * ld_m;
    const MelOut mo{o, m + 1 < nr ? o + ld_m : nullptr, runs + s0, inv_nr};
    QM_PAIR_DISPATCH(N1, x_forward<n_>(in, mo, ldx, ns, tw))
}

// ---------------------------------------------------------------- launch shapes
inline size_t plane_smem(qm_gspace g) { return (size_t)(g->n[2] * g->ldy + g->n[1] + g->n[2]) * sizeof(c2); }
inline size_t stick_smem(qm_gspace g) { return (size_t)(kPairTile * g->ldx + g->n[0]) * sizeof(c2); }
// threads of a stick CTA: 192; 256 where the outgoing pass of long axes wants the loads in flight.  us for
// 128 / 192 / 256: 96-point axis of the 255-atom cell in 347 / 308 / 339, out 364 / 345 / 278; 90 points
// (Gamma, 216 atoms) in 136 / 111 / 131, out 276 / 225 / 229; 72 points in 93 / 86 / 120, out 126 / 109 / 148
inline int stick_nt(int n1, bool out) { return out && n1 > 81 ? 256 : 192; }
constexpr size_t kPairSmem = 226 * 1024;  // dynamic shared memory a CTA may have (227 KB less the static part)

// threads of a plane CTA: the register budget's 768 (big groups: 512) on an SM, in two CTAs where their
// shared memory fits twice (one CTA's barriers then overlap with the other's passes), else in one
inline int plane_nt(const void* kernel, size_t smem, int big) {
    const int all = big ? 512 : 768;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, all / 2, smem) != cudaSuccess) cudaGetLastError();
    return occ >= 2 ? all / 2 : all;
}

}  // namespace pr
}  // namespace qm
