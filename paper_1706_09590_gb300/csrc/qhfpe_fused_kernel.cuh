// Fused right-hand-side stage: one launch evaluates the whole of Eq. (heom) (linear coupling, Sec. II)
// for a tile of TQ q-rows of one (replica, hierarchy element) -- all S x S electronic blocks, all p --
// and applies the Horner update of the RK4 step.
//
//   phase A  potential term, Eq. (quantum-liouvillian): the tile's p-rows are loaded into shared
//            memory, transformed by a two-pass in-place FFT (radix NP/16, then 16; sign +, digit-reversed
//            output), mixed per r-mode across the S x S blocks with the tables
//            D = UL_jj - UR_kk, L = UL_js, R = UR_sk (pre-scaled by 1/np, stored in the same
//            digit-reversed order), multiplied by -i, and transformed back (sign -, natural order).
//   phase B  one warp per p-row: upwind q-stencil (rows i-3..i+3 through L1/L2), damping and
//            delta-term, tier-up/-down couplings (neighbour elements' rows), terminator, the
//            potential term from shared memory, and out = base + h * L (row_wide: FP32 rows that fill a warp).
// The FP64 form runs phase A and most of phase B on 64-bit integers (potential_fixed, rows_fixed).
//
// Grid order: the hierarchy element varies fastest, then the replica, then the q-tile, so the blocks
// in flight cover all elements of a few q-tiles and the neighbour tiers and q-halos they re-read are
// L2-resident.
#pragma once
// (the fused stage kernel template; included by qhfpe_fused.cu, which instantiates the single-model
// kernel, and by qhfpe_fused_multi.cu, which instantiates the heterogeneous-batch kernel, so that the
// two compile in parallel)
#include "qhfpe.h"
#include "qhfpe_fixed.cuh"
#include "qhfpe_internal.cuh"

namespace {

constexpr int FTHREADS = 128;

template <typename T> struct V2;
template <> struct V2<float> { using type = float2; };
template <> struct V2<double> { using type = double2; };

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return {a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return {a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
template <typename C> __device__ __forceinline__ C cconjmul(C a, C w) { return {a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y}; }
// multiply by s*i, s = +1 or -1
template <int SG, typename C> __device__ __forceinline__ C cmul_si(C a) { return SG > 0 ? C{-a.y, a.x} : C{a.y, -a.x}; }

// a + SG i b and a - SG i b
template <int SG, typename C> __device__ __forceinline__ C cadd_si(C a, C b) { return {a.x - SG * b.y, a.y + SG * b.x}; }
template <int SG, typename C> __device__ __forceinline__ C csub_si(C a, C b) { return {a.x + SG * b.y, a.y - SG * b.x}; }

// ---- packed FP32x2 arithmetic (sm_100 and later) ---------------------------------------------------
// An FP32 complex value occupies a register pair, so one packed instruction adds or subtracts both of
// its parts; the lanes' runs of consecutive p values pair up the same way.  Each component is rounded
// exactly as the scalar instruction would round it.  The FP64 form keeps scalar arithmetic.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b)
{
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pd;\n\tmov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
        "sub.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// y += a x (a broadcast), y += u x (elementwise), y += x over N values
template <int N> __device__ __forceinline__ void v_axpy(float *y, float a, const float *x)
{
    if constexpr (N % 2 == 0) {
        const float2 a2 = make_float2(a, a);
#pragma unroll
        for (int v = 0; v < N; v += 2) {
            const float2 r = __ffma2_rn(a2, make_float2(x[v], x[v + 1]), make_float2(y[v], y[v + 1]));
            y[v] = r.x;
            y[v + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int v = 0; v < N; ++v) y[v] = fmaf(a, x[v], y[v]);
    }
}
template <int N> __device__ __forceinline__ void v_axpy(double *y, double a, const double *x)
{
#pragma unroll
    for (int v = 0; v < N; ++v) y[v] = fma(a, x[v], y[v]);
}
template <int N> __device__ __forceinline__ void v_fma(float *y, const float *u, const float *x)
{
    if constexpr (N % 2 == 0) {
#pragma unroll
        for (int v = 0; v < N; v += 2) {
            const float2 r = __ffma2_rn(make_float2(u[v], u[v + 1]), make_float2(x[v], x[v + 1]), make_float2(y[v], y[v + 1]));
            y[v] = r.x;
            y[v + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int v = 0; v < N; ++v) y[v] = fmaf(u[v], x[v], y[v]);
    }
}
template <int N> __device__ __forceinline__ void v_fma(double *y, const double *u, const double *x)
{
#pragma unroll
    for (int v = 0; v < N; ++v) y[v] = fma(u[v], x[v], y[v]);
}
template <int N> __device__ __forceinline__ void v_add(float *y, const float *x)
{
    if constexpr (N % 2 == 0) {
#pragma unroll
        for (int v = 0; v < N; v += 2) {
            const float2 r = __fadd2_rn(make_float2(x[v], x[v + 1]), make_float2(y[v], y[v + 1]));
            y[v] = r.x;
            y[v + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int v = 0; v < N; ++v) y[v] += x[v];
    }
}
template <int N> __device__ __forceinline__ void v_add(double *y, const double *x)
{
#pragma unroll
    for (int v = 0; v < N; ++v) y[v] += x[v];
}

// In-register DFTs of length 2, 4, 8 with sign SG (y_u = sum_t x_t e^{SG 2 pi i t u / R}), natural order.
template <int SG, typename C> __device__ __forceinline__ void dft2(C &a, C &b)
{
    C t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
template <int SG, typename C> __device__ __forceinline__ void dft4(C &x0, C &x1, C &x2, C &x3)
{
    const C t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3), d = csub(x1, x3);
    x0 = cadd(t0, t2);
    x2 = csub(t0, t2);
    x1 = cadd_si<SG>(t1, d);
    x3 = csub_si<SG>(t1, d);
}
template <int SG, typename C> __device__ __forceinline__ void dft8(C *x)
{
    using R = decltype(x[0].x);
    C e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    C o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
    dft4<SG>(e0, e1, e2, e3);
    dft4<SG>(o0, o1, o2, o3);
    const R h = (R)0.70710678118654752440;
    // w8^u, w8 = e^{SG 2 pi i / 8}
    C w1o = {(o1.x - SG * o1.y) * h, (o1.y + SG * o1.x) * h};    // o1 * (1 + SG i)/sqrt2
    C w3o = {(-o3.x - SG * o3.y) * h, (-o3.y + SG * o3.x) * h};  // o3 * (-1 + SG i)/sqrt2
    x[0] = cadd(e0, o0);
    x[4] = csub(e0, o0);
    x[1] = cadd(e1, w1o);
    x[5] = csub(e1, w1o);
    x[2] = cadd_si<SG>(e2, o2);  // e2 +- o2 * SG i
    x[6] = csub_si<SG>(e2, o2);
    x[3] = cadd(e3, w3o);
    x[7] = csub(e3, w3o);
}
// Length 16 as 4 x 4 (index n = 4 n1 + n2, frequency k = k1 + 4 k2): length-4 DFTs over n1, the
// twiddles w16^(n2 k1), length-4 DFTs over n2.
template <int SG, typename C> __device__ __forceinline__ void dft16(C *x)
{
    using R = decltype(x[0].x);
    const R c1 = (R)0.92387953251128675613;  // cos(pi/8)
    const R s1 = (R)0.38268343236508977173;  // sin(pi/8)
    const R h = (R)0.70710678118654752440;   // cos(pi/4)
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4<SG>(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);  // y[n2][k1] at x[4 k1 + n2]
    // w16^m = cos(2 pi m / 16) + SG i sin(2 pi m / 16) for m = n2 k1 in {1, 2, 3, 4, 6, 9}
    auto rot = [](C a, R c, R s) { return C{a.x * c - a.y * s, a.x * s + a.y * c}; };
    x[5] = rot(x[5], c1, SG * s1);    // n2 = 1, k1 = 1
    x[9] = rot(x[9], h, SG * h);      // n2 = 1, k1 = 2
    x[13] = rot(x[13], s1, SG * c1);  // n2 = 1, k1 = 3
    x[6] = rot(x[6], h, SG * h);      // n2 = 2, k1 = 1
    x[10] = cmul_si<SG>(x[10]);       // n2 = 2, k1 = 2
    x[14] = rot(x[14], -h, SG * h);   // n2 = 2, k1 = 3
    x[7] = rot(x[7], s1, SG * c1);    // n2 = 3, k1 = 1
    x[11] = rot(x[11], -h, SG * h);   // n2 = 3, k1 = 2
    x[15] = rot(x[15], -c1, -SG * s1); // n2 = 3, k1 = 3
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4<SG>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);  // -> X[k1 + 4 k2] at x[4 k1 + k2]
    C t[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) t[k1 + 4 * k2] = x[4 * k1 + k2];
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = t[k];
}
template <int R, int SG, typename C> __device__ __forceinline__ void dft_small(C *x)
{
    if constexpr (R == 2) dft2<SG>(x[0], x[1]);
    else if constexpr (R == 4) dft4<SG>(x[0], x[1], x[2], x[3]);
    else if constexpr (R == 8) dft8<SG>(x);
    else dft16<SG>(x);
}

// Radix sequence (first pass = longest span): a first pass of span NP with stride 16 and a last pass
// of radix 16.  With the padding below, the 16 threads of a half-warp then touch 16 distinct bank
// pairs in both passes.
template <int NP> struct Radices;
template <> struct Radices<32> { static constexpr int n = 2; static constexpr int r[2] = {2, 16}; };
template <> struct Radices<64> { static constexpr int n = 2; static constexpr int r[2] = {4, 16}; };
template <> struct Radices<128> { static constexpr int n = 2; static constexpr int r[2] = {8, 16}; };
template <> struct Radices<256> { static constexpr int n = 2; static constexpr int r[2] = {16, 16}; };

// Shared-memory index with one padding slot per 16 complex values (breaks the power-of-two strides of
// the FFT passes across banks).
__device__ __forceinline__ int pad16(int i) { return i + (i >> 4); }

// One DIF pass (forward, sign +) or DIT pass (inverse, sign -) of radix R at sub-length M over
// n_tr transforms of length NP stored contiguously in X.
template <int NP, int R, int M, bool FWD, typename C>
__device__ __forceinline__ void fft_pass(C *X, int n_tr, const C *__restrict__ tw)
{
    constexpr int S = M / R;
    constexpr int PER = NP / R;  // butterflies per transform
    // padded stride between the R inputs of a butterfly: exact when S is a multiple of 16, or when
    // S = 1 and every butterfly starts on a multiple of 16 (M a multiple of 16, R <= 16)
    static_assert(S % 16 == 0 || (S == 1 && M % 16 == 0 && R <= 16), "padding");
    // a thread keeps the same butterfly position (and twiddles) in every transform it visits
    static_assert(FTHREADS % PER == 0, "butterfly positions");
    constexpr int PS = S + S / 16;
    constexpr int PNP = NP + NP / 16;  // padded length of one transform
    const int jl = threadIdx.x % PER;
    const int grp = jl / S, j = jl - grp * S;
    const int off = pad16(grp * M + j);
    C w[R];
    if constexpr (S > 1) {  // the last pass (sub-length R) has only unit twiddles
#pragma unroll
        for (int u = 1; u < R; ++u) w[u] = tw[(j * u) * (NP / M)];
    }
    for (int tr = threadIdx.x / PER; tr < n_tr; tr += FTHREADS / PER) {
        C *xb = X + tr * PNP + off;
        C x[R];
#pragma unroll
        for (int t = 0; t < R; ++t) x[t] = xb[t * PS];
        if (FWD) {
            dft_small<R, +1>(x);
            if constexpr (S > 1) {
#pragma unroll
                for (int u = 1; u < R; ++u) x[u] = cmul(x[u], w[u]);
            }
        } else {
            if constexpr (S > 1) {
#pragma unroll
                for (int u = 1; u < R; ++u) x[u] = cconjmul(x[u], w[u]);
            }
            dft_small<R, -1>(x);
        }
#pragma unroll
        for (int t = 0; t < R; ++t) xb[t * PS] = x[t];
    }
    __syncthreads();
}

template <int NP, bool FWD, typename C>
__device__ __forceinline__ void fft_all(C *X, int n_tr, const C *tw)
{
    using RD = Radices<NP>;
    constexpr int R0 = RD::r[0], R1 = RD::r[1];
    static_assert(R0 * R1 == NP, "radices");
    if (FWD) {
        fft_pass<NP, R0, NP, true>(X, n_tr, tw);
        fft_pass<NP, R1, R1, true>(X, n_tr, tw);
    } else {
        fft_pass<NP, R1, R1, false>(X, n_tr, tw);
        fft_pass<NP, R0, NP, false>(X, n_tr, tw);
    }
}

// VEC consecutive reals through 16-byte vector accesses where the size allows (rows are 16-byte
// aligned); the vector is unpacked member by member so that the destination stays in registers.
template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; };
template <> struct Vec16<double> { using type = double2; };

__device__ __forceinline__ void unpack(const float4 &q, float *o) { o[0] = q.x; o[1] = q.y; o[2] = q.z; o[3] = q.w; }
__device__ __forceinline__ void unpack(const double2 &q, double *o) { o[0] = q.x; o[1] = q.y; }
__device__ __forceinline__ float4 pack(const float *i) { return make_float4(i[0], i[1], i[2], i[3]); }
__device__ __forceinline__ double2 pack(const double *i) { return make_double2(i[0], i[1]); }

template <typename T, int VEC>
__device__ __forceinline__ void ldv(const T *__restrict__ p, T *out)
{
    constexpr int N = 16 / (int)sizeof(T);
    if constexpr (VEC % N == 0) {
#pragma unroll
        for (int c = 0; c < VEC / N; ++c) unpack(reinterpret_cast<const typename Vec16<T>::type *>(p)[c], out + c * N);
    } else if constexpr (sizeof(T) == 4 && VEC == 2) {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        out[0] = q.x;
        out[1] = q.y;
    } else {
#pragma unroll
        for (int v = 0; v < VEC; ++v) out[v] = p[v];
    }
}

template <typename T, int VEC>
__device__ __forceinline__ void stv(T *p, const T *in)
{
    constexpr int N = 16 / (int)sizeof(T);
    if constexpr (VEC % N == 0) {
#pragma unroll
        for (int c = 0; c < VEC / N; ++c) reinterpret_cast<typename Vec16<T>::type *>(p)[c] = pack(in + c * N);
    } else if constexpr (sizeof(T) == 4 && VEC == 2) {
        *reinterpret_cast<float2 *>(p) = make_float2(in[0], in[1]);
    } else {
#pragma unroll
        for (int v = 0; v < VEC; ++v) p[v] = in[v];
    }
}

// The same for rows of the state in global memory: 32-byte accesses where a lane has that much (FP32 np 256, FP64
// np >= 128; rows are 32-byte aligned there).  Two 16-byte accesses of stride 32 touch every sector twice: np 256
// with three states spent two thirds of its L1 wavefronts on them.  256 x 256, depth 10, three states: 8.60 -> 7.78
// ms a step; 96 x 128, depth 8 in FP64: 1 %.
template <typename T, int VEC>
__device__ __forceinline__ void ldrow(const T *p, T *o)
{
    if constexpr (VEC * sizeof(T) % 32 == 0) {
        constexpr int N = 32 / (int)sizeof(T);
#pragma unroll
        for (int c = 0; c < VEC; c += N) {
            const size_t a = __cvta_generic_to_global(p + c);
            if constexpr (sizeof(T) == 4)
                asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=f"(o[c]), "=f"(o[c + 1]), "=f"(o[c + 2]), "=f"(o[c + 3]), "=f"(o[c + 4]), "=f"(o[c + 5]),
                               "=f"(o[c + 6]), "=f"(o[c + 7])
                             : "l"(a));
            else
                asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                             : "=d"(o[c]), "=d"(o[c + 1]), "=d"(o[c + 2]), "=d"(o[c + 3])
                             : "l"(a));
        }
    } else {
        ldv<T, VEC>(p, o);
    }
}
template <typename T, int VEC>
__device__ __forceinline__ void strow(T *p, const T *i)
{
    if constexpr (VEC * sizeof(T) % 32 == 0) {
        constexpr int N = 32 / (int)sizeof(T);
#pragma unroll
        for (int c = 0; c < VEC; c += N) {
            const size_t a = __cvta_generic_to_global(p + c);
            if constexpr (sizeof(T) == 4)
                asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(a), "f"(i[c]), "f"(i[c + 1]),
                             "f"(i[c + 2]), "f"(i[c + 3]), "f"(i[c + 4]), "f"(i[c + 5]), "f"(i[c + 6]), "f"(i[c + 7])
                             : "memory");
            else
                asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(a), "d"(i[c]), "d"(i[c + 1]), "d"(i[c + 2]),
                             "d"(i[c + 3])
                             : "memory");
        }
    } else {
        stv<T, VEC>(p, i);
    }
}

// 128-thread blocks (measured faster than 256: more independent blocks per SM keep phase A and phase B
// of different blocks overlapping, and each barrier stalls four warps).  The kernel waits mostly on L2
// loads, so resident warps count: FP32 with one or two states runs seven blocks per SM (72 registers;
// measured 5 % faster than six at 80), three states six (seven would spill), NP = 256 four (wider rows; 256 x 256 with
// three states took 34.4 ms for four steps with four, 35.7 with three, 43.2 with five, which spill).
// FP64 (integer arithmetic, latency-bound below 16 warps) runs four at 128 registers: on 96 x 128 at depth 8
// three, four and five blocks took within 3 % of each other, two 25 % longer.
// Its np 256 spills at four (1200 to 3800 bytes stored, at three 440 to 1140, at two none); us a step with two, three
// and four blocks: two states, 100 x 256, depth 4 1139, 1105, 1090; 24 x 256, depth 2 158, 178, 213; three states, 80 x
// 256, depth 4 3081, 3086, 3260; one state, 150 x 256, depth 40 583, 419, 431; c2 != 0, 100 x 256 1781, 1730, 1776.
template <typename T, int NP, int S>
struct FusedOcc {
    static constexpr int blocks = sizeof(T) == 4 ? (NP >= 256 ? 4 : (S >= 3 ? 6 : 7)) : (NP >= 256 ? 3 : 4);
};

// Phase A of the fused stage kernels: the potential term of Eq. (quantum-liouvillian) in place on the
// block's rows * S^2 p-rows in X (padded, complex): forward FFT (sign +, digit-reversed), per r-mode
// mixing across the S x S blocks with the tables D, L, R (pre-scaled by 1/NP) times -i, plus the
// p-diagonal bath terms (f_pp lambda_pp(m) - ngam) / NP (damping, delta-term, terminator d2/dp2, which
// are circulants along p), and the inverse FFT (sign -, natural order).  Called by all threads of the
// block after a barrier that makes X complete; ends with the inverse FFT's barrier.
// c2 != 0 (nonlinear coupling V = q + c2 q^2): the d2/dp2 coefficient of row i is fpp phi(q_i)^2,
// phi = 1 + 2 c2 q (Phi^2 = phi^2 d2/dp2); q_i = q_min + i dq.
template <typename T, int NP, int S>
__device__ __forceinline__ void potential_in_place(typename V2<T>::type *X, const typename V2<T>::type *tw,
                                                   const FusedTables<T> &tab, int nq, int i0, int rows, T fpp,
                                                   T ngam, const T *s_lpp, double c2 = 0.0, double q_min = 0.0,
                                                   double dq = 0.0)
{
    using C = typename V2<T>::type;
    constexpr int S2 = S * S;
    fft_all<NP, true>(X, rows * S2, tw);
    constexpr int MV = S >= 3 ? (NP > FTHREADS ? 2 : 1) : (S == 2 ? 2 : 4);  // modes per thread (vector table loads)
    static_assert(FTHREADS % (NP / MV) == 0, "mixing positions");
    const int pos0 = (threadIdx.x % (NP / MV)) * MV;
    // r-space coefficient of the bath terms diagonal in p (already over NP, like the tables):
    // (f_pp lambda_pp(m) - sum n_k gamma_k) / NP
    T cf[MV];
    {
        const T ng_a = ngam / (T)NP;
#pragma unroll
        for (int v = 0; v < MV; ++v) cf[v] = fpp * s_lpp[pos0 + v] - ng_a;
    }
    for (int r = threadIdx.x / (NP / MV); r < rows; r += FTHREADS / (NP / MV)) {
        const int i = i0 + r;
        if (c2 != 0.0) {  // block-uniform
            const T ph = (T)(1.0 + 2.0 * c2 * (q_min + i * dq));
            const T ng_a = ngam / (T)NP;
#pragma unroll
            for (int v = 0; v < MV; ++v) cf[v] = fpp * ph * ph * s_lpp[pos0 + v] - ng_a;
        }
        C rho[S2][MV];
#pragma unroll
        for (int a = 0; a < S2; ++a)
#pragma unroll
            for (int v = 0; v < MV; ++v) rho[a][v] = X[pad16((r * S2 + a) * NP + pos0 + v)];
#pragma unroll
        for (int j = 0; j < S; ++j)
#pragma unroll
            for (int k = 0; k < S; ++k) {
                T d[MV];
                ldv<T, MV>(tab.D + ((size_t)(j * S + k) * nq + i) * NP + pos0, d);
                C acc[MV];
#pragma unroll
                for (int v = 0; v < MV; ++v) acc[v] = C{d[v] * rho[j * S + k][v].x, d[v] * rho[j * S + k][v].y};
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    if (s != j) {
                        T u[MV];
                        ldv<T, MV>(tab.L + ((size_t)(j * S + s) * nq + i) * NP + pos0, u);
#pragma unroll
                        for (int v = 0; v < MV; ++v) {
                            acc[v].x += u[v] * rho[s * S + k][v].x;
                            acc[v].y += u[v] * rho[s * S + k][v].y;
                        }
                    }
                    if (s != k) {
                        T u[MV];
                        ldv<T, MV>(tab.R + ((size_t)(s * S + k) * nq + i) * NP + pos0, u);
#pragma unroll
                        for (int v = 0; v < MV; ++v) {
                            acc[v].x -= u[v] * rho[j * S + s][v].x;
                            acc[v].y -= u[v] * rho[j * S + s][v].y;
                        }
                    }
                }
#pragma unroll
                for (int v = 0; v < MV; ++v) {  // times -i, plus the p-diagonal bath terms
                    const C w = rho[j * S + k][v];
                    X[pad16((r * S2 + j * S + k) * NP + pos0 + v)] = C{acc[v].y + cf[v] * w.x, cf[v] * w.y - acc[v].x};
                }
            }
    }
    __syncthreads();
    fft_all<NP, false>(X, rows * S2, tw);
}

// Phase A of the FP64 form on block fixed-point integers (qhfpe_fixed.cuh), in place in X: the rows * S^2
// p-rows as integers of one exponent each, on entry (fill_fixed) and on return.  The same passes as
// potential_in_place.  The real and imaginary parts of the mixed values are exchanged, which turns the
// inverse transform into a forward one, so that the radix-16 pass is one function for both directions: with
// every pass and conversion unrolled twice the instruction cache missed on 39 % of the issue slots.
// Exponents stand in the padding slots of a transform, as 16-bit values: the row's (before the forward
// transform, and again after the inverse) at FWD_EXP, those of the runs of 16 modes between at 0 .. R0 - 1.
template <int NP> struct FixedRows {
    static constexpr int R0 = Radices<NP>::r[0];
    static constexpr int PNP = NP + NP / 16;
    static constexpr int FWD_EXP = R0 == 16 ? 16 : 15;
    static __device__ __forceinline__ short &exp_slot(double2 *X, int tr, int b)
    {
        return reinterpret_cast<short *>(X + tr * PNP + 17 * (b >> 3) + 16)[b & 7];
    }
};

// rows * S2 p-rows of the tile into X as integers below 2^bits of their row's exponent
template <int NP, int S2>
__device__ __forceinline__ void fill_fixed(double2 *X, const double *__restrict__ v, size_t blk, int i0, int rows)
{
    using namespace qhfx;
    using F = FixedRows<NP>;
    constexpr int LV = NP >= 128 ? NP / 32 : 4, PL = NP / LV;  // p values per lane, lanes per row
    constexpr int B = Scale<F::R0>::bits;
    const int l = (threadIdx.x % PL) * LV;
#pragma unroll 1
    for (int base = 0; base < rows * S2; base += FTHREADS / PL) {
        const int rp = base + threadIdx.x / PL;
        const bool act = rp < rows * S2;
        const int pr = act ? rp % S2 : 0, r = act ? rp / S2 : 0;
        const double *src = v + (size_t)pr * 2 * blk + (size_t)(i0 + r) * NP + l;
        double re[LV], im[LV];
        ldrow<double, LV>(src, re);
        ldrow<double, LV>(src + blk, im);
        unsigned top = 0, low = 0;  // the row's largest upper half; zero for a row of zeros only
#pragma unroll
        for (int q = 0; q < LV; ++q) {
            top = max(top, max((unsigned)__double2hiint(re[q]) & 0x7fffffffu, (unsigned)__double2hiint(im[q]) & 0x7fffffffu));
            low |= (unsigned)__double2loint(re[q]) | (unsigned)__double2loint(im[q]);
        }
        top |= low != 0u;
#pragma unroll
        for (int o = PL / 2; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        const int E = top >= 0x00100000u ? (int)(top >> 20) : (top ? 1 : EXP_NONE);
        if (act) {
            I2 *x = reinterpret_cast<I2 *>(X + pad16(rp * NP + l));
            if (E >= EXP_SMALL) {
#pragma unroll
                for (int q = 0; q < LV; ++q) x[q] = I2{to_fixed<B>(re[q], E), to_fixed<B>(im[q], E)};
            } else if (E == EXP_NONE) {
#pragma unroll
                for (int q = 0; q < LV; ++q) x[q] = I2{0, 0};
            } else {
#pragma unroll
                for (int q = 0; q < LV; ++q) x[q] = I2{to_fixed_any<B>(re[q], E), to_fixed_any<B>(im[q], E)};
            }
            if (l == 0) F::exp_slot(X, rp, F::FWD_EXP) = (short)(E < 2047 ? E : EXP_BAD);
        }
    }
}

// the radix-16 pass over the 16-point runs of n_tr transforms, sign +
template <int NP> __device__ __noinline__ void pass16_fixed(double2 *X, int n_tr)
{
    using namespace qhfx;
    using F = FixedRows<NP>;
#pragma unroll 1
    for (int b = threadIdx.x; b < n_tr * F::R0; b += FTHREADS) {
        I2 *xb = reinterpret_cast<I2 *>(X) + 17 * b;
        I2 x[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) x[t] = xb[t];
        dft16<+1>(x);
#pragma unroll
        for (int t = 0; t < 16; ++t) xb[t] = x[t];
    }
    __syncthreads();
}

template <int NP, int S>
__device__ __forceinline__ void potential_fixed(double2 *X, const double2 *tw, const FusedTables<double> &tab, int nq, int i0,
                                                int rows, double fpp, double ngam, const double *s_lpp, int &s_far,
                                                double c2, double q_min, double dq)
{
    using namespace qhfx;
    using F = FixedRows<NP>;
    constexpr int S2 = S * S, R0 = F::R0, PNP = F::PNP;
    I2 *XI = reinterpret_cast<I2 *>(X);
    const I2 *w62 = reinterpret_cast<const I2 *>(tw);
    const int n_tr = rows * S2;
    const int j = threadIdx.x % 16;  // butterfly of the radix-R0 passes: points j, j + 16, ...
#pragma unroll 1
    for (int tr = threadIdx.x / 16; tr < n_tr; tr += FTHREADS / 16) {
        I2 *xb = XI + tr * PNP + j;
        I2 x[R0];
#pragma unroll
        for (int t = 0; t < R0; ++t) x[t] = xb[17 * t];
        forward_butterfly<R0>(x, w62, j);
#pragma unroll
        for (int u = 0; u < R0; ++u) xb[17 * u] = x[u];
    }
    __syncthreads();
    pass16_fixed<NP>(X, n_tr);

    // mixing: the tables are integers c of one exponent k per pair and row (value c 2^(k - 62)).  A run of 16
    // modes (a butterfly of the next pass) is brought to the top of the word before the products and again
    // after their sum, with an exponent of its own: bounds that hold for any row would leave 10 bits unused
    constexpr int MV = NP > FTHREADS ? 2 : (S == 1 && NP >= 64 ? 2 : 1);  // modes per thread (few: code size)
    static_assert(FTHREADS % (NP / MV) == 0 && 16 % MV == 0, "mixing positions");
    constexpr int RS = FTHREADS / (NP / MV);  // rows at once
    constexpr int RUN = 16 / MV;              // lanes of a run
    const unsigned run = (RUN == 32 ? 0xffffffffu : ((1u << RUN) - 1)) << (threadIdx.x & 31 & ~(RUN - 1));
    const int pos0 = (threadIdx.x % (NP / MV)) * MV;
    const size_t tn = (size_t)nq * NP;
    const long long *tD = reinterpret_cast<const long long *>(tab.D) + pos0, *tL = reinterpret_cast<const long long *>(tab.L) + pos0,
                    *tR = reinterpret_cast<const long long *>(tab.R) + pos0;
    const int *kD = tab.kx, *kL = kD + S2 * nq, *kR = kL + S2 * nq;
    // the p-diagonal bath terms cf = (f_pp lambda_pp(m) - ngam) / NP, |lambda_pp| <= 64 / NP
    Half cf[MV];
    int kcf;
    const auto bath = [&](double f) {
        const double bound = (64.0 * fabs(f) + fabs(ngam)) * (1.0 / NP);
        const int Eb = max(exponent_of(bound) + 1, EXP_MIN);
        kcf = bound > 0.0 ? Eb - 1022 : EXP_NO_TABLE;
#pragma unroll
        for (int v = 0; v < MV; ++v) cf[v] = halves(to_fixed<62>(f * s_lpp[pos0 + v] - ngam * (1.0 / NP), Eb));
    };
    bath(fpp);
#pragma unroll 1
    for (int base = 0; base < rows; base += RS) {
        const int r = base + threadIdx.x / (NP / MV), i = i0 + r;
        if (r >= rows) break;  // (a run's lanes share their row)
        if (c2 != 0.0) {       // block-uniform
            const double ph = 1.0 + 2.0 * c2 * (q_min + i * dq);
            bath(fpp * ph * ph);
        }
        Half xr[S2][MV], xi[S2][MV];
        int E[S2], big = 0;
#pragma unroll
        for (int a = 0; a < S2; ++a) {
            const int tr = r * S2 + a;
            E[a] = F::exp_slot(X, tr, F::FWD_EXP);
            big = max(big, E[a]);
            I2 q[MV];
            unsigned o = 0;
#pragma unroll
            for (int v = 0; v < MV; ++v) {
                q[v] = XI[tr * PNP + pad16(pos0 + v)];
                o |= magnitude(q[v]);
            }
            const int n = norm_shift<61>(__reduce_or_sync(run, o));
            E[a] -= n;
#pragma unroll
            for (int v = 0; v < MV; ++v) {
                q[v] = shift(q[v], n);
                xr[a][v] = halves(q[v].x);
                xi[a][v] = halves(q[v].y);
            }
        }
#pragma unroll
        for (int j_ = 0; j_ < S; ++j_)
#pragma unroll
            for (int k = 0; k < S; ++k) {
                const int jk = j_ * S + k;
                int M = max(E[jk] + kD[jk * nq + i], E[jk] + kcf);
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    if (s != j_) M = max(M, E[s * S + k] + kL[(j_ * S + s) * nq + i]);
                    if (s != k) M = max(M, E[j_ * S + s] + kR[(s * S + k) * nq + i]);
                }
                long long ar[MV], ai[MV];  // the commutator: at most six products below 2^60
                {
                    const int sh = M - (E[jk] + kD[jk * nq + i]);
#pragma unroll
                    for (int v = 0; v < MV; ++v) {
                        const Half c = halves(tD[jk * tn + (size_t)i * NP + v]);
                        ar[v] = shr_s(mul_hi(xr[jk][v], c), sh);
                        ai[v] = shr_s(mul_hi(xi[jk][v], c), sh);
                    }
                }
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    if (s != j_) {
                        const int a = s * S + k, t = j_ * S + s, sh = M - (E[a] + kL[t * nq + i]);
#pragma unroll
                        for (int v = 0; v < MV; ++v) {
                            const Half c = halves(tL[t * tn + (size_t)i * NP + v]);
                            ar[v] += shr_s(mul_hi(xr[a][v], c), sh);
                            ai[v] += shr_s(mul_hi(xi[a][v], c), sh);
                        }
                    }
                    if (s != k) {
                        const int a = j_ * S + s, t = s * S + k, sh = M - (E[a] + kR[t * nq + i]);
#pragma unroll
                        for (int v = 0; v < MV; ++v) {
                            const Half c = halves(tR[t * tn + (size_t)i * NP + v]);
                            ar[v] -= shr_s(mul_hi(xr[a][v], c), sh);
                            ai[v] -= shr_s(mul_hi(xi[a][v], c), sh);
                        }
                    }
                }
                const int sc = M - (E[jk] + kcf), tr = r * S2 + jk;
                I2 q[MV];
                unsigned o = 0;
#pragma unroll
                for (int v = 0; v < MV; ++v) {  // times -i, plus the bath terms; parts exchanged
                    q[v] = I2{shr_s(mul_hi(xi[jk][v], cf[v]), sc) - ar[v], shr_s(mul_hi(xr[jk][v], cf[v]), sc) + ai[v]};
                    o |= magnitude(q[v]);
                }
                const int n = norm_shift<59>(__reduce_or_sync(run, o));
#pragma unroll
                for (int v = 0; v < MV; ++v) XI[tr * PNP + pad16(pos0 + v)] = shift(q[v], n);
                if (pos0 % 16 == 0) F::exp_slot(X, tr, pos0 / 16) = (short)(big >= EXP_BAD ? EXP_BAD : M - n);
            }
    }
    __syncthreads();
    pass16_fixed<NP>(X, n_tr);
#pragma unroll 1
    for (int tr = threadIdx.x / 16; tr < n_tr; tr += FTHREADS / 16) {
        I2 *xb = XI + tr * PNP + j;
        I2 x[R0];
        int e[R0];
#pragma unroll
        for (int t = 0; t < R0; ++t) {
            x[t] = xb[17 * t];
            e[t] = F::exp_slot(X, tr, t);
        }
        const int E = align<R0>(x, e);
        inverse_butterfly<R0>(x, w62, j);
#pragma unroll
        for (int t = 0; t < R0; ++t) xb[17 * t] = I2{x[t].y, x[t].x};
        if (j == 0) {
            F::exp_slot(X, tr, F::FWD_EXP) = (short)E;
            if (exp_far(E)) s_far = 1;
        }
    }
    __syncthreads();
}
// the potential term in X is v 2^(E + fixed_pot_exponent), E at the transform's FWD_EXP (EXP_BAD: NaN)
template <int NP, int S> constexpr int fixed_pot_exponent()
{
    constexpr int R0 = Radices<NP>::r[0];
    return qhfx::Scale<R0>::K_fwd + 4 + 2 + qhfx::Scale<R0>::inv + qhfx::Scale<R0>::down;
}
// ... as doubles, for the phase B in FP64
template <int NP, int S> __device__ __forceinline__ void potential_to_double(double2 *X, int n_tr)
{
    using namespace qhfx;
    for (int t = threadIdx.x; t < n_tr * NP; t += FTHREADS) {
        const int tr = t / NP, M = FixedRows<NP>::exp_slot(X, tr, FixedRows<NP>::FWD_EXP);
        const I2 v = reinterpret_cast<const I2 *>(X)[pad16(t)];
        const double bad = bitsd(0x7ff8000000000000ull);
        const int K = M + fixed_pot_exponent<NP, S>();
        X[pad16(t)] = M >= EXP_BAD ? double2{bad, bad} : double2{from_fixed_any(v.x, K), from_fixed_any(v.y, K)};
    }
}

// A factor for fixed-point products: w = c 2^(k - 62), |c| in [2^61, 2^62).
struct FixedWeight {
    qhfx::Half c;
    int k;
};
__device__ __forceinline__ FixedWeight fixed_weight(double w)
{
    const int ex = qhfx::exponent_of(w);
    if (ex == 0) return FixedWeight{{0, 0}, -4096};  // far below every other term
    const long long m = qhfx::to_fixed<62>(w, ex);
    return FixedWeight{qhfx::halves(m), ex - 1022};
}

// weight of the t-th of the six rows of the upwind q difference
__device__ __forceinline__ int upwind_weight(bool neg, int t)
{
    const int s = neg ? 5 - t : t;
    const int w = s == 0 ? -2 : s == 1 ? 15 : s == 2 ? -60 : s == 3 ? 20 : s == 4 ? 30 : -3;
    return neg ? -w : w;
}

// A value's q difference times pk, in FP64, and its potential term pot 2^K: the column V, window rows from ii on
__device__ __forceinline__ double far_value(const double *V, int np, int ii, int nq, int periodic, bool neg, double pk,
                                         long long pot, int K)
{
    double kin = 0.0;
#pragma unroll 1
    for (int t = 0; t < 6; ++t) {
        int i = ii + t;
        const bool ok = i >= 0 && i < nq;
        if (!ok && periodic) i = wrap_q(i, nq);
        kin = fma((double)upwind_weight(neg, t), ok || periodic ? V[(size_t)i * np] : 0.0, kin);
    }
    return fma(pk, kin, qhfx::from_fixed_any(pot, K));
}

template <int VEC> __device__ __forceinline__ bool nonzero(const double *x)
{
    unsigned long long any = 0;
#pragma unroll
    for (int v = 0; v < VEC; ++v) any |= qhfx::dbits(x[v]) << 1;
    return any != 0;
}

// e: a p row's values x with two on each side (periodic p), a warp a row
template <int VEC, typename T> __device__ __forceinline__ void with_neighbours(const T *x, T *e, int lane)
{
    const unsigned all = 0xffffffffu;
#pragma unroll
    for (int v = 0; v < VEC; ++v) e[v + 2] = x[v];
    if constexpr (VEC == 1) {
        e[0] = __shfl_sync(all, x[0], (lane + 30) & 31);
        e[1] = __shfl_sync(all, x[0], (lane + 31) & 31);
        e[3] = __shfl_sync(all, x[0], (lane + 1) & 31);
        e[4] = __shfl_sync(all, x[0], (lane + 2) & 31);
    } else {
        e[0] = __shfl_sync(all, x[VEC - 2], (lane + 31) & 31);
        e[1] = __shfl_sync(all, x[VEC - 1], (lane + 31) & 31);
        e[VEC + 2] = __shfl_sync(all, x[0], (lane + 1) & 31);
        e[VEC + 3] = __shfl_sync(all, x[1], (lane + 1) & 31);
    }
}

// Phase B of the FP64 form (linear coupling, all terms, the potential and the p-diagonal bath terms already
// in X): kinetic term, tier couplings and update of the block's rows.  As in the transforms
// (qhfpe_fixed.cuh) the FP64 pipe would bound it, so it is left with the tier sums:
//   kinetic  the q differences have small integer weights (sum of sizes 130).  A warp takes four rows of one
//            pair; for each of its p columns the nine rows read are brought to the column's largest exponent
//            (62 bits below it) once, and the four sums of six are exact.  Where the rows' own exponents are
//            more than eight apart each of the four takes its own.  The four are rows 4 n .. 4 n + 3 of the grid
//            (or three, np >= 128: GridInfo::q_group): a unit that holds only some of them, at the edge of a tile or in a small one,
//            reads all nine rows all the same, so that results don't depend on the tile.  (With an exponent for each row
//            everywhere four steps of 96 x 128 at depth 8 took 9.26 ms where this way they took 8.1.)
//   tiers    G = sum of the neighbours' rows, weighted, in FP64 (one instruction per value and neighbour, on a
//            pipe that has room for them; in integers the conversions alone took twenty); its row is brought
//            to the largest exponent, 58 bits below it, and the p difference (weights 1, 8) is exact.
// Quantising at 2^-54 to 2^-62 of the largest term is below the rounding of the FP64 sums, whose partial sums of
// up to 100 times the values round at 2^-53.
// Rows whose differences or potential term are near the ends of the range of doubles (exp_plain) have their q differences
// in FP64, values by value, and so do the p differences of such rows: subnormal values, infinities and NaN as in FP64 sums.
template <int NP, int S>
__device__ __forceinline__ void
rows_fixed(const GridInfo &g, const StageScalars<double> &sc, const double *__restrict__ v_in, const double *y, double *v_out,
           int mode, size_t ebase, int i0, int rows, const long long *nb_off, const double *nb_wg, const double *nb_wa,
           int n_d0, int n_nb, bool term, bool any_far, double2 *X, const double *pgrid)
{
    using namespace qhfx;
    constexpr int S2 = S * S;
    constexpr int VEC = NP / 32;              // a warp holds a p row
    constexpr int RG = 4;                     // q rows per unit, at most
    constexpr int BITS = 58;                  // of G below its row's largest value: 18 x 2^58 stays below 2^63
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t blk = g.blk;
    const int nq = g.nq;
    const int l0 = lane * VEC;
    const bool neg = pgrid[l0] < 0.0;  // one sign per lane (caller's check)
    int ck[6];                         // p < 0: offsets -2..+3, p >= 0: -3..+2
#pragma unroll
    for (int t = 0; t < 6; ++t) ck[t] = upwind_weight(neg, t);
    const int first = neg ? -2 : -3;
    const double bad = bitsd(0x7ff8000000000000ull);
    const int gr = NP >= 128 ? g.q_group : RG;
    int rg = min(gr, (rows * S2 + FTHREADS / 32 - 1) / (FTHREADS / 32));  // fewer where warps would idle
    if (2 * rg > gr) rg = gr;
    const int u0 = i0 / rg, n_u = (i0 + rows - 1) / rg - u0 + 1;  // units of rg rows, aligned on the grid
#pragma unroll 1
    for (int u = warp; u < n_u * S2; u += FTHREADS / 32) {
        const int pr = u % S2, us = (u0 + u / S2) * rg;
        const int ia = max(us, i0), r0 = ia - i0;
        const int nr = min(us + rg, i0 + rows) - ia;
        const int gs = NP < 128 ? ia & ~(RG - 1) : ia - ia % gr, k0 = ia - gs;  // the group of grid rows that the unit's are among
        const size_t poff = ebase + (size_t)pr * 2 * blk;
        // the unit's rows in the group, by the exponent of their potential term
        unsigned near = ((1u << nr) - 1) << k0, far = 0;
        if (any_far) {
#pragma unroll 1
            for (int r = 0; r < nr; ++r)
                if (exp_far(FixedRows<NP>::exp_slot(X, (r0 + r) * S2 + pr, FixedRows<NP>::FWD_EXP))) far |= 1u << (k0 + r);
            near &= ~far;
        }
#pragma unroll 1
        for (int plane = 0; plane < 2; ++plane) {
            const double *V = v_in + poff + plane * blk;
            // (each lane reads and writes only its own values of X from here on)
            const auto Xat = [&](int r, int v) -> double & {
                return reinterpret_cast<double *>(X + pad16(((r0 + r) * S2 + pr) * NP + l0 + v))[plane];
            };
#pragma unroll 1
            for (int v = 0; v < VEC; ++v) {  // (one p column at a time: more in flight would only lengthen the code)
                const FixedWeight pk = fixed_weight(-(pgrid[l0 + v] * sc.fkin));
                const auto value = [&](int t) {  // window row t of the column
                    int ii = gs + first + t;
                    bool ok = ii >= 0 && ii < nq;
                    if (!ok && g.periodic_q) {
                        ii = wrap_q(ii, nq);
                        ok = true;
                    }
                    return ok ? V[(size_t)ii * NP + l0 + v] : 0.0;
                };
                // row r from its six window rows x (below 2^62) of exponent E: -p dW/dq and the potential term, each
                // an integer, at the larger unit
                const auto emit = [&](int r, const Half *x, int E) {
                    double &xv = Xat(r, v);
                    const long long pot = (long long)dbits(xv);
                    const int M = FixedRows<NP>::exp_slot(X, (r0 + r) * S2 + pr, FixedRows<NP>::FWD_EXP);
                    long long lo = 0, hi = 0;
#pragma unroll
                    for (int t = 0; t < 6; ++t) {
                        lo = madw(x[t].l, ck[t], lo);
                        hi = madw(x[t].h, ck[t], hi);
                    }
                    const long long kin = mul_hi(halves((long long)((unsigned long long)hi << 24) + (lo >> 8)), pk.c);
                    const int uk = E + pk.k - 1022 - 62 + 8 + 2, up = M + fixed_pot_exponent<NP, S>();
                    const int U = max(uk, up);  // (below 2^60 and 2^62: the sum fits)
                    const long long fine = uk < up ? kin : pot, coarse = uk < up ? pot : kin;
                    xv = from_fixed(coarse + shr_round(fine, U - min(uk, up)), U);
                };
                double raw[RG + 5];
                int ex[RG + 5], E = EXP_MIN;
#pragma unroll
                for (int t = 0; t < RG + 5; ++t) raw[t] = value(t);
#pragma unroll
                for (int t = 0; t < RG + 5; ++t) {
                    ex[t] = exponent_of(raw[t]);
                    E = max(E, ex[t]);
                }
                int least = E;  // smallest of the rows' own exponents
#pragma unroll
                for (int r = 0; r < RG; ++r) {
                    const int er = max(max(max(ex[r], ex[r + 1]), max(ex[r + 2], ex[r + 3])), max(ex[r + 4], ex[r + 5]));
                    if (r < gr && gs + r < nq) least = min(least, er);
                }
                unsigned odd = far;  // rows left to FP64
                bool zero = false;  // nothing but zeros in the window
                if (!exp_plain(E)) {
                    unsigned long long any = 0;
#pragma unroll
                    for (int t = 0; t < RG + 5; ++t) any |= dbits(raw[t]) << 1;
                    zero = any == 0;
                    if (!zero) least = -EXP_BIG;  // each row by itself
                }
                if (!__any_sync(0xffffffffu, E - least > 8)) {
                    Half x[RG + 5];
#pragma unroll
                    for (int t = 0; t < RG + 5; ++t) x[t] = halves(to_fixed<62>(raw[t], E));
#pragma unroll
                    for (int r = 0; r < RG; ++r)
                        if (near >> r & 1) emit(r - k0, x + r, E);
                } else {  // steep in q: an exponent for each row
#pragma unroll
                    for (int r = 0; r < RG; ++r) {
                        if (!(near >> r & 1)) continue;
                        int er = EXP_MIN;
#pragma unroll
                        for (int t = 0; t < 6; ++t) er = max(er, ex[r + t]);
                        Half x[6];
#pragma unroll
                        for (int t = 0; t < 6; ++t) x[t] = halves(to_fixed<62>(raw[r + t], er));
                        if (exp_plain(er) || zero) emit(r - k0, x, er);
                        else odd |= 1u << r;
                    }
                }
#pragma unroll 1
                for (int r = -k0; odd; ++r, odd >>= 1) {
                    if (!(odd & 1)) continue;
                    double &xv = Xat(r, v);
                    const int M = FixedRows<NP>::exp_slot(X, (r0 + r) * S2 + pr, FixedRows<NP>::FWD_EXP);
                    xv = M >= EXP_BAD ? bad
                                      : far_value(V + l0 + v, NP, gs + first + k0 + r, nq, g.periodic_q, neg,
                                                  -(pgrid[l0 + v] * sc.fkin), (long long)dbits(xv),
                                                  M + fixed_pot_exponent<NP, S>());
                }
            }
            double p[VEC], pw[VEC];  // p, and times the weight of the (first) neighbour with a p term
            ldv<double, VEC>(pgrid + l0, p);
            if (n_d0 < n_nb) {
                const double wa = nb_wa[n_d0];
#pragma unroll
                for (int v = 0; v < VEC; ++v) pw[v] = p[v] * wa;
            }
#pragma unroll 1
            for (int r = 0; r < nr; ++r) {
                const int i = ia + r;
                const size_t o = poff + plane * blk + (size_t)i * NP + l0;
                double a[VEC];
#pragma unroll
                for (int v = 0; v < VEC; ++v) a[v] = Xat(r, v);  // potential and kinetic terms
                // tier couplings: G = sum of the neighbours, weighted, in FP64
                double G[VEC];
#pragma unroll
                for (int v = 0; v < VEC; ++v) G[v] = 0.0;
                {
                    double next[VEC];
                    if (n_nb > 0) ldrow<double, VEC>(v_in + (long long)o + nb_off[0], next);
#pragma unroll 1
                    for (int n = 0; n < n_nb; ++n) {
                        double w[VEC];
                        const double wg = nb_wg[n];
#pragma unroll
                        for (int v = 0; v < VEC; ++v) w[v] = next[v];
                        if (n + 1 < n_nb) ldrow<double, VEC>(v_in + (long long)o + nb_off[n + 1], next);
#pragma unroll
                        for (int v = 0; v < VEC; ++v) G[v] = fma(wg, w[v], G[v]);
                        if (n >= n_d0) {  // warp-uniform; (the barrier keeps it a branch: FP64 instructions that
                                          // are only predicated off take their 64 clocks all the same)
                            __syncwarp();
                            const double wa = nb_wa[n];
#pragma unroll
                            for (int v = 0; v < VEC; ++v) a[v] = fma(n == n_d0 ? pw[v] : p[v] * wa, w[v], a[v]);
                        }
                    }
                }
                if (term) {  // r_0 p W of the Eq. (GMFP) terminator
                    __syncwarp();
                    double w[VEC];
                    ldrow<double, VEC>(v_in + o, w);
#pragma unroll
                    for (int v = 0; v < VEC; ++v) G[v] = fma(sc.r0 * p[v], w[v], G[v]);
                }
                if (n_nb > 0 || term) {  // 4th-order central d/dp of G, periodic p, neighbours through the warp
                    int E = EXP_MIN;
#pragma unroll
                    for (int v = 0; v < VEC; ++v) E = max(E, exponent_of(G[v]));
                    E = __reduce_max_sync(0xffffffffu, E);
                    if (exp_plain(E)) {
                        long long Gi[VEC], e[VEC + 4];
#pragma unroll
                        for (int v = 0; v < VEC; ++v) Gi[v] = to_fixed<BITS>(G[v], E);
                        with_neighbours<VEC>(Gi, e, lane);
#pragma unroll
                        for (int v = 0; v < VEC; ++v) {
                            const long long d = (e[v] - e[v + 4]) + ((e[v + 3] - e[v + 1]) << 3);
                            a[v] = fma(sc.inv12dp, from_fixed(d, E - 1022 - BITS), a[v]);
                        }
                    } else if (__any_sync(0xffffffffu, nonzero<VEC>(G))) {  // (warp-uniform)
                        double e[VEC + 4];
                        with_neighbours<VEC>(G, e, lane);
#pragma unroll
                        for (int v = 0; v < VEC; ++v)
                            a[v] = fma(sc.inv12dp, e[v] - 8.0 * e[v + 1] + 8.0 * e[v + 3] - e[v + 4], a[v]);
                    }
                }
                if (mode != 0) {
                    double b[VEC];
                    ldrow<double, VEC>(y + o, b);
#pragma unroll
                    for (int v = 0; v < VEC; ++v) a[v] = fma(sc.h, a[v], b[v]);
                }
                strow<double, VEC>(v_out + o, a);
            }
        }
    }
}

// Phase B of one p-row that fills a warp (FP32, np 128 and 256): linear coupling, every term, lanes of one p sign, the
// potential and the p-diagonal bath terms in xp (this lane's place of the row in X).  Bound by load latency at 16 to
// 28 warps an SM.  The general loop below keeps the centre row and the p part of the tier coupling in registers
// and has one neighbour in flight; here the p part goes straight to the sum, the centre row is read again where the
// terminator needs it, and the neighbours come three at a time.  256 x 256, depth 10, three states: 7.78 -> 7.03 ms
// a step (one neighbour at a time: 7.71; the base row loaded ahead of the p-stencil spills: 7.65).  np 128: 512 x
// 128, two states 86 -> 83 us, 96 x 128, three states, depth 4 196 -> 187 us.
template <int NP, bool MIXED>
__device__ __forceinline__ void row_wide(const GridInfo &g, const StageScalars<float> &sc, const float *__restrict__ v_in,
                                         const float *y, const double *y0, float *v_out, double *y0_out, double h, int mode,
                                         bool tier0, size_t o, size_t o0, int i, const float *pcol, bool interior,
                                         const long long *nb_off, const float *nb_wg, const float *nb_wa, int n_d0, int n_nb, bool term, const float2 *xp)
{
    constexpr int VEC = NP / 32, NB = 3;
    const size_t blk = g.blk;
    const int nq = g.nq;
    const bool neg = pcol[0] < 0.f;
    float ar[VEC], ai[VEC];
    {  // -p dW/dq, 5th-order upwind
        const float cneg[6] = {3, -30, -20, 60, -15, 2};  // p < 0: offsets -2..+3
        const float cpos[6] = {-2, 15, -60, 20, 30, -3};  // p >= 0: offsets -3..+2
        const int first = i - 3 + (neg ? 1 : 0);
        const float *row = v_in + o - (size_t)i * NP;  // row 0
        float kr[VEC], ki[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) kr[v] = ki[v] = 0.f;
#pragma unroll
        for (int t0 = 0; t0 < 6; t0 += 3) {
            float sr[3][VEC], si[3][VEC];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                int ii = first + t0 + b;
                bool ok = interior || (ii >= 0 && ii < nq);
                if (!ok && g.periodic_q) {
                    ii = wrap_q(ii, nq);
                    ok = true;
                }
                if (ok) {
                    ldrow<float, VEC>(row + (size_t)ii * NP, sr[b]);
                    ldrow<float, VEC>(row + (size_t)ii * NP + blk, si[b]);
                } else {
#pragma unroll
                    for (int v = 0; v < VEC; ++v) sr[b][v] = si[b][v] = 0.f;
                }
            }
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const float c = neg ? cneg[t0 + b] : cpos[t0 + b];
                v_axpy<VEC>(kr, c, sr[b]);
                v_axpy<VEC>(ki, c, si[b]);
            }
        }
        float pk[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) pk[v] = -(pcol[v] * sc.fkin);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            ar[v] = pk[v] * kr[v];
            ai[v] = pk[v] * ki[v];
        }
    }
    {
        float gr[VEC], gi[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) gr[v] = gi[v] = 0.f;
        const auto add = [&](int a, const float *xr, const float *xi) {
            const float wg = nb_wg[a];
            v_axpy<VEC>(gr, wg, xr);
            v_axpy<VEC>(gi, wg, xi);
            if (a >= n_d0) {
                const float wa = nb_wa[a];
                float q[VEC];
#pragma unroll
                for (int v = 0; v < VEC; ++v) q[v] = wa * pcol[v];
                v_fma<VEC>(ar, q, xr);
                v_fma<VEC>(ai, q, xi);
            }
        };
        int a = 0;
#pragma unroll 1
        for (; a + NB <= n_nb; a += NB) {
            float xr[NB][VEC], xi[NB][VEC];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const float *u = v_in + (long long)o + nb_off[a + b];
                ldrow<float, VEC>(u, xr[b]);
                ldrow<float, VEC>(u + blk, xi[b]);
            }
#pragma unroll
            for (int b = 0; b < NB; ++b) add(a + b, xr[b], xi[b]);
        }
#pragma unroll 1
        for (; a < n_nb; ++a) {
            float xr[VEC], xi[VEC];
            const float *u = v_in + (long long)o + nb_off[a];
            ldrow<float, VEC>(u, xr);
            ldrow<float, VEC>(u + blk, xi);
            add(a, xr, xi);
        }
        if (term) {  // d/dp (r_0 p W) of the terminator
            float wr[VEC], wi[VEC], r0p[VEC];
            ldrow<float, VEC>(v_in + o, wr);
            ldrow<float, VEC>(v_in + o + blk, wi);
#pragma unroll
            for (int v = 0; v < VEC; ++v) r0p[v] = sc.r0 * pcol[v];
            v_fma<VEC>(gr, r0p, wr);
            v_fma<VEC>(gi, r0p, wi);
        }
        if (n_nb > 0 || term) {  // 4th-order central d/dp, neighbours along p through the warp
            const int left = (threadIdx.x + 31) & 31, right = (threadIdx.x + 1) & 31;
            const auto ddp = [&](const float *x, float *acc) {
                float er[VEC + 4];
#pragma unroll
                for (int v = 0; v < VEC; ++v) er[v + 2] = x[v];
                er[0] = __shfl_sync(0xffffffffu, x[VEC - 2], left);
                er[1] = __shfl_sync(0xffffffffu, x[VEC - 1], left);
                er[VEC + 2] = __shfl_sync(0xffffffffu, x[0], right);
                er[VEC + 3] = __shfl_sync(0xffffffffu, x[1], right);
#pragma unroll
                for (int v = 0; v < VEC; ++v)
                    acc[v] += sc.inv12dp * (er[v] - 8.f * er[v + 1] + 8.f * er[v + 3] - er[v + 4]);
            };
            ddp(gr, ar);
            ddp(gi, ai);
        }
    }
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        ar[v] += xp[v].x;
        ai[v] += xp[v].y;
    }
    if (mode == 0) {
        strow<float, VEC>(v_out + o, ar);
        strow<float, VEC>(v_out + o + blk, ai);
    } else if (tier0) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            const double nr = y0[o0 + v] + h * (double)ar[v];
            const double ni = y0[o0 + v + blk] + h * (double)ai[v];
            v_out[o + v] = (float)nr;
            v_out[o + v + blk] = (float)ni;
            if (mode == 2) {
                y0_out[o0 + v] = nr;
                y0_out[o0 + v + blk] = ni;
            }
        }
    } else {
        float br[VEC], bi[VEC];
        ldrow<float, VEC>(y + o, br);
        ldrow<float, VEC>(y + o + blk, bi);
        v_axpy<VEC>(br, sc.h, ar);
        v_axpy<VEC>(bi, sc.h, ai);
        strow<float, VEC>(v_out + o, br);
        strow<float, VEC>(v_out + o + blk, bi);
    }
}

// MULTI: one Horner stage of several propagators at once (heterogeneous batch: members differ in q
// grid, surfaces, bath, hierarchy depth, closure, dt and replica count, and share NP, S and the
// precision).  Blocks are numbered member by member; a block finds its member (first block numbers
// ascending), copies the member's description into shared memory and does that member's block of stage
// k = 4..1 of the Horner form.  The other arguments are then taken from the member.
// The block `bid` of a fused stage launch (see fused_stage_kernel below); also called in a loop by the
// persistent kernel (a barrier must separate two calls of one block: shared memory is reused).
// NL: the terms of the nonlinear coupling (GridInfo::c2 != 0) are compiled in; NL = false requires
// c2 = 0 (the linear coupling keeps their registers free).
template <typename T, int NP, int S, bool MIXED, bool MULTI, bool NL>
__device__ __forceinline__ void
fused_stage_body(unsigned bid, GridInfo g, const ElemInfo *__restrict__ elems, FusedTables<T> tab, StageScalars<T> sc,
                 const T *__restrict__ v_in, const T *y, const double *y0, T *v_out, double *y0_out, double h, int mode,
                 int terms, int rep0, int n_rep, int tq, const T *__restrict__ Pg, const MultiMember<T> *__restrict__ mem,
                 int n_mem, int k, bool warm = false)
{
    // warm: this block's previous call was for the same member and tile height (the persistent kernel's
    // one-member loop), so the member's description, twiddles, p grid and r-space eigenvalues are still
    // in shared memory
    if constexpr (MULTI) {
        __shared__ MultiMember<T> M;
        __shared__ int s_m;
        if (!warm) {
            if (threadIdx.x == 0) {
                int m = 0;
                while (m + 1 < n_mem && mem[m + 1].block0 <= (long)bid) ++m;
                s_m = m;
            }
            __syncthreads();
            static_assert(sizeof(MultiMember<T>) % sizeof(int) == 0, "member size");
            const int *src = reinterpret_cast<const int *>(mem + s_m);
            int *dst = reinterpret_cast<int *>(&M);
            for (int w = threadIdx.x; w < (int)(sizeof(MultiMember<T>) / sizeof(int)); w += FTHREADS) dst[w] = src[w];
            __syncthreads();
        }
        g = M.g;
        elems = M.elems;
        tab = M.tab;
        sc = M.sc[k];
        v_in = k == 4 ? M.y : (k == 2 ? M.vB : M.vA);
        y = M.y;
        y0 = M.y0;
        v_out = k == 1 ? M.y : (k == 3 ? M.vB : M.vA);
        y0_out = k == 1 ? M.y0 : nullptr;
        h = M.dt / k;
        mode = k == 1 ? 2 : 1;
        terms = QHFPE_TERM_ALL;
        rep0 = 0;
        n_rep = M.g.n_rep;
        Pg = nullptr;
        bid -= (unsigned)M.block0;
    }
    using C = typename V2<T>::type;
    constexpr int S2 = S * S;
    // phase B: a lane holds VEC consecutive p values of one row, a row spans LPR lanes, and a warp
    // covers RPW rows (several for NP < 128, so that short rows still fill a warp with 16-byte loads)
    constexpr int VEC = NP >= 128 ? NP / 32 : 4;
    constexpr int LPR = NP / VEC;
    constexpr int RPW = 32 / LPR;
    static_assert(LPR * VEC == NP && RPW * LPR == 32, "lane layout");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *X = reinterpret_cast<C *>(smem_raw);          // [tq * S2][NP], padded (pad16)
    C *tw = X + pad16(tq * S2 * NP) + 1;             // [NP]

    const int nq = g.nq;
    const int e = bid % g.n_elem;
    const int rep = rep0 + (bid / g.n_elem) % n_rep;
    const int tile = bid / (g.n_elem * n_rep);
    const int i0 = tile * tq;
    const int rows = min(tq, nq - i0);
    const size_t blk = g.blk;
    const size_t ebase = (size_t)rep * g.rep_stride + (size_t)e * g.elem_stride;

    __shared__ long long nb_off[3 * QH_MAX_MODES];
    __shared__ T nb_wg[3 * QH_MAX_MODES], nb_wa[3 * QH_MAX_MODES];
    __shared__ long long mx_off[QH_MAX_MODES];  // nonlinear coupling: mixed-derivative neighbours
    __shared__ T mx_w[QH_MAX_MODES];
    __shared__ int s_nmx;
    __shared__ int s_far;  // FP64: a row whose potential term's exponent is far from doubles'
    __shared__ int s_cnt[4];
    __shared__ T s_ngam;
    __shared__ __align__(16) T pgrid[NP];
    __shared__ __align__(16) T s_lpp[NP];
    if (threadIdx.x == 0) {
        const ElemInfo &E = elems[e];
        int n = 0;
        const int n_up = (terms & 8) ? E.n_up : 0;
        for (int a = 0; a < n_up; ++a, ++n) {
            nb_off[n] = (long long)(E.up[a] - e) * (long long)g.elem_stride;
            nb_wg[n] = (T)1;
            nb_wa[n] = (T)0;
        }
        const int n_dn = (terms & 16) ? E.n_dn : 0;
        for (int pass = 0; pass < 2; ++pass) {
            if (NL && pass == 0 && (terms & 16)) {  // |m| = 2 couplings of the nonlinear coupling: G only
                for (int a = 0; a < E.n_d2; ++a, ++n) {
                    nb_off[n] = (long long)(E.d2[a] - e) * (long long)g.elem_stride;
                    nb_wg[n] = (T)E.w2[a];
                    nb_wa[n] = (T)0;
                }
            }
            for (int a = 0; a < n_dn; ++a) {
                if ((E.wr[a] != 0.0) != (pass == 1)) continue;
                nb_off[n] = (long long)(E.dn[a] - e) * (long long)g.elem_stride;
                nb_wg[n] = (T)E.wc[a];
                nb_wa[n] = (T)E.wr[a];
                ++n;
            }
            if (pass == 0) s_cnt[1] = n;
        }
        const int n_mx = NL && (terms & 16) ? E.n_mx : 0;
        for (int a = 0; a < n_mx; ++a) {
            mx_off[a] = (long long)(E.mx[a] - e) * (long long)g.elem_stride;
            mx_w[a] = (T)(E.wmx[a] / (12.0 * g.dq));
        }
        s_nmx = n_mx;
        s_far = 0;
        s_cnt[0] = n_up;
        s_cnt[2] = n;
        s_cnt[3] = (terms & 8) && E.terminator;
        s_ngam = (terms & 4) ? (T)E.ngam : (T)0;
    }
    if (!warm)
        for (int t = threadIdx.x; t < NP; t += FTHREADS) {
            tw[t] = C{tab.tw[2 * t], tab.tw[2 * t + 1]};
            pgrid[t] = (T)(g.p_min + t * g.dp);
            s_lpp[t] = tab.lpp[t];
        }

    // the previous launch on the stream (the stage whose output this one reads) has completed and its
    // writes are visible
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- phase A: potential term -------------------------------------------------------------
    // With the potential term computed here, the p-diagonal parts of the bath terms ride along in
    // r-space: the damping -(sum n_k gamma_k) W and the 5-point d2/dp2 of the delta-term and of the
    // terminator are circulants along p, i.e. products with their eigenvalues after the FFT.
    const bool want_pot = (terms & 2) != 0;
    const bool fold = want_pot && !Pg;
    if constexpr (sizeof(T) == sizeof(double)) {
        if (fold) {
            fill_fixed<NP, S2>(X, v_in + ebase, blk, i0, rows);
            __syncthreads();
            potential_fixed<NP, S>(X, tw, tab, nq, i0, rows,
                                   ((terms & 4) ? sc.fdelta : (T)0) + ((s_cnt[3] != 0) ? sc.fterm : (T)0), s_ngam, s_lpp,
                                   s_far, NL ? g.c2 : 0.0, g.q_min, g.dq);
        }
    } else if (fold) {
        constexpr int LV = 4;  // p values per load
        constexpr int PL = NP / LV;
        static_assert(FTHREADS % PL == 0, "load positions");
        const int l = (threadIdx.x % PL) * LV;
        for (int rp = threadIdx.x / PL; rp < rows * S2; rp += FTHREADS / PL) {
            const int pr = rp % S2, r = rp / S2;
            const T *src = v_in + ebase + (size_t)pr * 2 * blk + (size_t)(i0 + r) * NP + l;
            T re[LV], im[LV];
            ldv<T, LV>(src, re);
            ldv<T, LV>(src + blk, im);
            const int base = (r * S2 + pr) * NP + l;
#pragma unroll
            for (int v = 0; v < LV; ++v) X[pad16(base + v)] = C{re[v], im[v]};
        }
        __syncthreads();
        potential_in_place<T, NP, S>(X, tw, tab, nq, i0, rows,
                                     ((terms & 4) ? sc.fdelta : (T)0) + ((s_cnt[3] != 0) ? sc.fterm : (T)0), s_ngam,
                                     s_lpp, NL ? g.c2 : 0.0, g.q_min, g.dq);
    }

    // ---- phase B: one warp per p-row ------------------------------------------------------------
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_up = s_cnt[0], n_d0 = s_cnt[1], n_nb = s_cnt[2];
    const bool term = s_cnt[3] != 0;
    // (folded into phase A when it ran)
    const T ngam = fold ? (T)0 : s_ngam;
    const T inv12dp = sc.inv12dp;
    const T fkin = sc.fkin;
    const T fpp = fold ? (T)0 : ((terms & 4) ? sc.fdelta : (T)0) + (term ? sc.fterm : (T)0);
    const int lr = lane / LPR;            // this lane's row among the warp's RPW rows
    const int l0 = (lane % LPR) * VEC;    // its first p index
    T pcol[VEC];
    ldv<T, VEC>(pgrid + l0, pcol);
    const bool neg0 = pcol[0] < (T)0;
    const bool uni_warp = __all_sync(0xffffffffu, neg0 == (pcol[VEC - 1] < (T)0));
    const int sh = neg0 ? 1 : 0;
    const bool interior = i0 >= 3 && i0 + rows + 3 <= nq;  // no q-stencil row outside the grid
    if constexpr (sizeof(T) == sizeof(double) && !NL) {
        // the fixed-point form: all terms, the potential in X, every lane's p values of one sign
        const bool one_sign = __all_sync(0xffffffffu, (pgrid[lane * (NP / 32)] < (T)0) == (pgrid[lane * (NP / 32) + NP / 32 - 1] < (T)0));
        if (fold && terms == QHFPE_TERM_ALL && one_sign) {
            rows_fixed<NP, S>(g, sc, v_in, y, v_out, mode, ebase, i0, rows, nb_off, nb_wg, nb_wa, n_d0, n_nb, term,
                              s_far != 0, X, pgrid);
            return;
        }
    }
    if constexpr (sizeof(T) == sizeof(double)) {
        if (fold) {
            potential_to_double<NP, S>(X, rows * S2);
            __syncthreads();
        }
    }
    T pk[VEC];  // -p / (60 dq)
#pragma unroll
    for (int v = 0; v < VEC; ++v) pk[v] = -(pcol[v] * fkin);

    // work unit: RPW consecutive rows of one pair; lanes past the tile's last row compute a copy of it
    // (their shuffles are needed) and store nothing
    const int n_units = RPW == 1 ? rows * S2 : ((rows + RPW - 1) / RPW) * S2;
    for (int rp = warp; rp < n_units; rp += FTHREADS / 32) {
        int pr, r;
        bool act = true;
        if constexpr (RPW == 1) {
            pr = rp % S2;
            r = rp / S2;
        } else {
            pr = rp % S2;
            const int r_lane = (rp / S2) * RPW + lr;
            act = r_lane < rows;
            r = act ? r_lane : rows - 1;
        }
        const int i = i0 + r;
        const size_t poff = ebase + (size_t)pr * 2 * blk;
        const T *Vre = v_in + poff, *Vim = Vre + blk;
        const size_t o = poff + (size_t)i * NP + l0;
        if constexpr (sizeof(T) == 4 && NP >= 128 && !NL) {
            if (uni_warp && fold && terms == QHFPE_TERM_ALL) {
                row_wide<NP, MIXED>(g, sc, v_in, y, y0, v_out, y0_out, h, mode, MIXED && e == 0, o,
                                    (size_t)rep * g.tier0_rep_stride + (size_t)pr * 2 * blk + (size_t)i * NP + l0, i, pcol,
                                    interior, nb_off, nb_wg, nb_wa, n_d0, n_nb, term,
                                    X + pad16((r * S2 + pr) * NP + l0));
                continue;
            }
        }
        T ar[VEC], ai[VEC], wr[VEC], wi[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) ar[v] = ai[v] = (T)0;

        if (uni_warp) {
            // the six stencil rows in two batches of three (loads of a batch issued before use); the
            // centre row is among them
            const T cneg[6] = {3, -30, -20, 60, -15, 2};  // p < 0: offsets -2..+3
            const T cpos[6] = {-2, 15, -60, 20, 30, -3};  // p >= 0: offsets -3..+2
            const int tc = neg0 ? 2 : 3;                  // centre row
            T kr[VEC], ki[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) kr[v] = ki[v] = (T)0;
            // interior tiles: the six rows lie inside the grid, at fixed offsets from row i - 3 + sh
            const T *rre = interior ? Vre + (size_t)(i - 3 + sh) * NP + l0 : Vre;
            const T *rim = rre + blk;
#pragma unroll
            for (int t0 = 0; t0 < 6; t0 += 3) {
                T sr[3][VEC], si[3][VEC];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    if (interior) {
                        ldrow<T, VEC>(rre + (t0 + b) * NP, sr[b]);
                        ldrow<T, VEC>(rim + (t0 + b) * NP, si[b]);
                        continue;
                    }
                    int ii = i + t0 + b - 3 + sh;
                    bool ok = ii >= 0 && ii < nq;
                    if (!ok && g.periodic_q) {
                        ii = wrap_q(ii, nq);
                        ok = true;
                    }
                    if (ok) {
                        ldrow<T, VEC>(Vre + (size_t)ii * NP + l0, sr[b]);
                        ldrow<T, VEC>(Vim + (size_t)ii * NP + l0, si[b]);
                    } else {
#pragma unroll
                        for (int v = 0; v < VEC; ++v) sr[b][v] = si[b][v] = (T)0;
                    }
                }
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const T c = neg0 ? cneg[t0 + b] : cpos[t0 + b];
                    v_axpy<VEC>(kr, c, sr[b]);
                    v_axpy<VEC>(ki, c, si[b]);
                    if (t0 + b == tc) {
#pragma unroll
                        for (int v = 0; v < VEC; ++v) {
                            wr[v] = sr[b][v];
                            wi[v] = si[b][v];
                        }
                    }
                }
            }
            if (terms & 1) {
                v_fma<VEC>(ar, pk, kr);
                v_fma<VEC>(ai, pk, ki);
            }
        } else {
            if (terms & 1) {
                const T cneg[7] = {0, 3, -30, -20, 60, -15, 2};
                const T cpos[7] = {-2, 15, -60, 20, 30, -3, 0};
                T kr[VEC], ki[VEC];
#pragma unroll
                for (int v = 0; v < VEC; ++v) kr[v] = ki[v] = (T)0;
#pragma unroll
                for (int d = -3; d <= 3; ++d) {
                    int ii = i + d;
                    if (ii < 0 || ii >= nq) {
                        if (!g.periodic_q) continue;
                        ii = wrap_q(ii, nq);
                    }
                    T rr[VEC], ri[VEC];
                    ldrow<T, VEC>(Vre + (size_t)ii * NP + l0, rr);
                    ldrow<T, VEC>(Vim + (size_t)ii * NP + l0, ri);
#pragma unroll
                    for (int v = 0; v < VEC; ++v) {
                        const T c = pcol[v] < (T)0 ? cneg[d + 3] : cpos[d + 3];
                        kr[v] += c * rr[v];
                        ki[v] += c * ri[v];
                    }
                }
                v_fma<VEC>(ar, pk, kr);
                v_fma<VEC>(ai, pk, ki);
            }
            ldrow<T, VEC>(Vre + (size_t)i * NP + l0, wr);
            ldrow<T, VEC>(Vim + (size_t)i * NP + l0, wi);
        }
        if (ngam != (T)0) {
            v_axpy<VEC>(ar, -ngam, wr);
            v_axpy<VEC>(ai, -ngam, wi);
        }
        // G = sum_up W^(n+e_k) + sum_dn wc W^(n-e_k) [+ r_0 p W at the terminator]; d/dp of G below
        T gr[VEC], gi[VEC], hr[VEC], hi[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) gr[v] = gi[v] = hr[v] = hi[v] = (T)0;
        for (int a = 0; a < n_up; ++a) {
            const T *u = v_in + (long long)o + nb_off[a];
            T xr[VEC], xi[VEC];
            ldrow<T, VEC>(u, xr);
            ldrow<T, VEC>(u + blk, xi);
            v_add<VEC>(gr, xr);
            v_add<VEC>(gi, xi);
        }
        for (int a = n_up; a < n_d0; ++a) {
            const T *u = v_in + (long long)o + nb_off[a];
            T xr[VEC], xi[VEC];
            ldrow<T, VEC>(u, xr);
            ldrow<T, VEC>(u + blk, xi);
            const T wg = nb_wg[a];
            v_axpy<VEC>(gr, wg, xr);
            v_axpy<VEC>(gi, wg, xi);
        }
        // nonlinear coupling V = q + c2 q^2: phi = 1 + 2 c2 q_i multiplies Phi = -phi d/dp and the
        // p phi part of Lambda^(1); its d2/dp dq part enters G below (block-uniform branches)
        const T phi = NL && g.c2 != 0.0 ? (T)(1.0 + 2.0 * g.c2 * (g.q_min + i * g.dq)) : (T)1;
        if (n_d0 < n_nb) {
            for (int a = n_d0; a < n_nb; ++a) {
                const T *u = v_in + (long long)o + nb_off[a];
                T xr[VEC], xi[VEC];
                ldrow<T, VEC>(u, xr);
                ldrow<T, VEC>(u + blk, xi);
                const T wg = nb_wg[a], wa = nb_wa[a];
                v_axpy<VEC>(gr, wg, xr);
                v_axpy<VEC>(gi, wg, xi);
                v_axpy<VEC>(hr, wa, xr);
                v_axpy<VEC>(hi, wa, xi);
            }
            if (NL && g.c2 != 0.0) {
#pragma unroll
                for (int v = 0; v < VEC; ++v) {
                    hr[v] *= phi;
                    hi[v] *= phi;
                }
            }
            v_fma<VEC>(ar, pcol, hr);
            v_fma<VEC>(ai, pcol, hi);
        }
        const int n_mx = NL ? s_nmx : 0;
        if (NL && g.c2 != 0.0) {
            // G' = phi G + sum_a wmx_a d/dq W^(mx_a) (4th-order central in q, rows i-2..i+2), so that
            // d/dp G' = phi dG/dp + wmx d2/dp dq W: the p-stencil below covers both
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                gr[v] *= phi;
                gi[v] *= phi;
            }
            for (int a = 0; a < n_mx; ++a) {
                const T *Ere = v_in + poff + mx_off[a];
                const T w = mx_w[a];
                const T cq[4] = {(T)1, (T)-8, (T)8, (T)-1};
                const int dqo[4] = {-2, -1, 1, 2};
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    int ii = i + dqo[b];
                    if (ii < 0 || ii >= nq) {
                        if (!g.periodic_q) continue;
                        ii = wrap_q(ii, nq);
                    }
                    T xr[VEC], xi[VEC];
                    ldrow<T, VEC>(Ere + (size_t)ii * NP + l0, xr);
                    ldrow<T, VEC>(Ere + blk + (size_t)ii * NP + l0, xi);
                    v_axpy<VEC>(gr, w * cq[b], xr);
                    v_axpy<VEC>(gi, w * cq[b], xi);
                }
            }
        }
        const bool have_g = n_nb > 0 || term || n_mx > 0;
        if (term) {
            T r0p[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) r0p[v] = sc.r0 * pcol[v];
            v_fma<VEC>(gr, r0p, wr);
            v_fma<VEC>(gi, r0p, wi);
        }
        // neighbours along p (periodic) through the warp: ext[k] = value at l0 - 2 + k
        auto stencil = [&](const T *xr, const T *xi, T *er, T *ei) {
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                er[v + 2] = xr[v];
                ei[v + 2] = xi[v];
            }
            // lanes of one row form a shuffle segment of width LPR; source lanes are relative to it
            static_assert(VEC >= 2, "two p values per lane");
            int left, right;
            if constexpr (LPR == 32) {
                left = (lane + 31) & 31;
                right = (lane + 1) & 31;
            } else {
                const int li = lane % LPR;
                left = (li + LPR - 1) & (LPR - 1);
                right = (li + 1) & (LPR - 1);
            }
            er[0] = __shfl_sync(0xffffffffu, xr[VEC - 2], left, LPR);
            er[1] = __shfl_sync(0xffffffffu, xr[VEC - 1], left, LPR);
            ei[0] = __shfl_sync(0xffffffffu, xi[VEC - 2], left, LPR);
            ei[1] = __shfl_sync(0xffffffffu, xi[VEC - 1], left, LPR);
            er[VEC + 2] = __shfl_sync(0xffffffffu, xr[0], right, LPR);
            er[VEC + 3] = __shfl_sync(0xffffffffu, xr[1], right, LPR);
            ei[VEC + 2] = __shfl_sync(0xffffffffu, xi[0], right, LPR);
            ei[VEC + 3] = __shfl_sync(0xffffffffu, xi[1], right, LPR);
        };
        if (have_g) {  // uniform across the block (same element)
            T er[VEC + 4], ei[VEC + 4];
            stencil(gr, gi, er, ei);
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                ar[v] += inv12dp * (er[v] - (T)8 * er[v + 1] + (T)8 * er[v + 3] - er[v + 4]);
                ai[v] += inv12dp * (ei[v] - (T)8 * ei[v + 1] + (T)8 * ei[v + 3] - ei[v + 4]);
            }
        }
        if (fpp != (T)0) {
            T er[VEC + 4], ei[VEC + 4];
            stencil(wr, wi, er, ei);
            const T f = fpp * phi * phi;
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                ar[v] += f * (-er[v] + (T)16 * er[v + 1] - (T)30 * er[v + 2] + (T)16 * er[v + 3] - er[v + 4]);
                ai[v] += f * (-ei[v] + (T)16 * ei[v + 1] - (T)30 * ei[v + 2] + (T)16 * ei[v + 3] - ei[v + 4]);
            }
        }
        if (want_pot && Pg) {  // potential term computed by another kernel
            T pr_[VEC], pi_[VEC];
            ldrow<T, VEC>(Pg + poff + (size_t)i * NP + l0, pr_);
            ldrow<T, VEC>(Pg + poff + blk + (size_t)i * NP + l0, pi_);
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                ar[v] += pr_[v];
                ai[v] += pi_[v];
            }
        } else if (want_pot) {
            const int pb = (r * S2 + pr) * NP + l0;
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                const C pv = X[pad16(pb + v)];
                ar[v] += pv.x;
                ai[v] += pv.y;
            }
        }
        // ---- update -------------------------------------------------------------------------------
        if (!act) {
        } else if (mode == 0) {
            strow<T, VEC>(v_out + o, ar);
            strow<T, VEC>(v_out + o + blk, ai);
        } else if (MIXED && e == 0) {
            const size_t o0 = (size_t)rep * g.tier0_rep_stride + (size_t)pr * 2 * blk + (size_t)i * NP + l0;
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                const double nr = y0[o0 + v] + h * (double)ar[v];
                const double ni = y0[o0 + v + blk] + h * (double)ai[v];
                v_out[o + v] = (T)nr;
                v_out[o + v + blk] = (T)ni;
                if (mode == 2) {
                    y0_out[o0 + v] = nr;
                    y0_out[o0 + v + blk] = ni;
                }
            }
        } else {
            const T hh = sc.h;
            T br[VEC], bi[VEC];
            ldrow<T, VEC>(y + o, br);
            ldrow<T, VEC>(y + o + blk, bi);
            v_axpy<VEC>(br, hh, ar);
            v_axpy<VEC>(bi, hh, ai);
            strow<T, VEC>(v_out + o, br);
            strow<T, VEC>(v_out + o + blk, bi);
        }
    }
}

template <typename T, int NP, int S, bool MIXED, bool MULTI, bool NL>
__global__ void __launch_bounds__(FTHREADS, FusedOcc<T, NP, S>::blocks - (MULTI && FusedOcc<T, NP, S>::blocks > 3 ? 1 : 0))
fused_stage_kernel(GridInfo g, const ElemInfo *__restrict__ elems, FusedTables<T> tab, StageScalars<T> sc, const T *__restrict__ v_in,
                   const T *y, const double *y0, T *v_out, double *y0_out, double h, int mode, int terms, int rep0,
                   int n_rep, int tq, const T *__restrict__ Pg, const MultiMember<T> *__restrict__ mem, int n_mem, int k)
{
    // Programmatic dependent launch: the next stage may start its blocks (prologue only) once every
    // block of this one has started; the body waits (griddepcontrol.wait) for this grid's completion
    // before touching the state.  Both are no-ops for a plain launch.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    fused_stage_body<T, NP, S, MIXED, MULTI, NL>(blockIdx.x, g, elems, tab, sc, v_in, y, y0, v_out, y0_out, h, mode, terms,
                                             rep0, n_rep, tq, Pg, mem, n_mem, k);
}


// One stage of the single-model kernel at tile height tq_req (0: default), launched with programmatic
// stream serialisation: its blocks may be scheduled while the previous kernel drains (the kernel waits
// for it before reading the state).
template <typename T, int NP, int S, bool MIXED, bool NL>
cudaError_t launch_general_t(const GridInfo &g, const ElemInfo *elems, const FusedTables<T> &tab, const T *v_in,
                             const T *y, const double *y0, T *v_out, double *y0_out, double h, int mode, int terms,
                             int rep0, int n_rep, cudaStream_t st, const T *Pg, int tq_req)
{
    int tq = tq_req > 0 ? tq_req : fused_rows_per_tile(NP, S, sizeof(T));
    const int tmax = fused_max_rows(NP, S, sizeof(T));  // the shared-memory limit set at preparation
    if (tq > tmax) tq = tmax;
    if (tq > g.nq) tq = g.nq;
    const size_t smem = fused_smem_bytes(tq, NP, S, sizeof(T));
    const int tiles = (g.nq + tq - 1) / tq;
    const long blocks = (long)tiles * n_rep * g.n_elem;
    if (blocks <= 0) return cudaSuccess;
    const StageScalars<T> sc = stage_scalars<T>(g, h);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(FTHREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fused_stage_kernel<T, NP, S, MIXED, false, NL>, g, elems, tab, sc, v_in, y, y0,
                              v_out, y0_out, h, mode, terms, rep0, n_rep, tq, Pg, (const MultiMember<T> *)nullptr, 0, 0);
}

template <typename T, int NP, int S, bool MIXED, bool NL>
cudaError_t prepare_general_t()
{
    const size_t smem = fused_smem_bytes(fused_max_rows(NP, S, sizeof(T)), NP, S, sizeof(T));
    return cudaFuncSetAttribute(fused_stage_kernel<T, NP, S, MIXED, false, NL>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace
