// Cluster-resident propagation: whole runs of RK4 steps of small propagators with the state in shared memory.
//
// A replica of the two-state models at np = 32 or 64 is a few hundred KB (four elements on 32 x 32: 131 KB
// in FP32), so the launch-per-stage form spends its time on launches, L2 latency and half-empty SMs (27 us a
// step for one such propagation) or, for hundreds of replicas, on re-reading neighbour tiers and q halos
// through L2.  Here one thread-block cluster holds one replica: block c of the cluster owns `rows`
// consecutive q rows of every hierarchy element and electronic pair.  Everything but the q difference is
// local to a row, so the blocks exchange only their edge rows (three on each side, written into the
// neighbours' shared memory) and one cluster barrier separates two Horner stages.  Two stage buffers
// live in shared memory; the step's base y (8 B per cell and stage, coalesced) and the FP64 zeroth tier
// stay in global memory, L2-resident.
//
// Inside a block there is no barrier at all: a row of one pair belongs to eight lanes with np/8 consecutive p
// values each (res_lane), the four pairs of a row to neighbouring lane groups of one warp.
//   FFT along p  length-8 transform across the lanes (radix 2, shuffles), twiddles, length np/8 in registers;
//                the inverse runs back the same way, so every lane ends with its own p values
//   mixing       the r-space products with the other pairs' values by shuffles; tables per lane, shared by the
//                elements of a row
//   the rest     q rows by 16-byte shared-memory loads, the p difference with two values from each
//                neighbouring lane
// The arithmetic is the fused stage kernel's: FP32 stages, the zeroth tier's base and update in FP64 at every stage.
#include "qhfpe.h"
#include "qhfpe_fused_kernel.cuh"

namespace {

// consecutive p values of a lane, and threads of a block: four values at np = 32 (128 registers, 16 warps
// per SM: 37 us a step for 76 replicas of four elements on 32 x 32, 13.5 us for one; eight values at 248
// registers and 8 warps took 10 and 50 % longer)
constexpr int res_lane(int np) { return np == 32 ? 4 : 8; }
constexpr int res_threads(int np) { return np == 32 ? 512 : 256; }
constexpr int RES_MAXNB = 2 * QH_MAX_MODES;

struct ResElem {  // couplings of one element
    int n_up, n_d0, n_nb, term;
    float ng, fpp;      // the p-diagonal bath terms: sum n_k gamma_k / np, coefficient of d2/dp2
    int nb[RES_MAXNB];  // neighbours' places in a stage buffer (bytes): up, down without a p term, down with one
    float wg[RES_MAXNB], wa[RES_MAXNB];
};

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 lds4(unsigned a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts4(unsigned a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// the shared-memory address that `a` has in block `rank` of the cluster, and a store to such an address
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned rank)
{
    unsigned b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
    return b;
}
__device__ __forceinline__ void stc4(unsigned a, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// floats of one stage buffer: [elem][pair] slabs of two planes of rows + 6 q rows; slabs are offset by four
// banks so that the two pairs of a quarter-warp's 16-byte accesses (np = 32) fall on different banks
__host__ __device__ constexpr int res_slab(int np, int rows) { return 2 * (rows + 6) * np + 4; }

// transform of length LPR across the lanes (positions l), in place, bit-reversed frequencies; sign +
template <int LPR, int VL> __device__ __forceinline__ void lanes_forward(float2 (&x)[VL], int l, float2 w8)
{
#pragma unroll
    for (int half = LPR / 2; half >= 1; half >>= 1) {
        const float s = (l & half) ? -1.f : 1.f;
#pragma unroll
        for (int b = 0; b < VL; ++b) {
            const float2 p = make_float2(__shfl_xor_sync(0xffffffffu, x[b].x, half), __shfl_xor_sync(0xffffffffu, x[b].y, half));
            x[b] = __ffma2_rn(x[b], make_float2(s, s), p);
        }
        if (half == 4) {  // e^{2 pi i (l mod 4) / 8} on the upper lanes
#pragma unroll
            for (int b = 0; b < VL; ++b) x[b] = cmul(x[b], w8);
        }
        if (half == 2) {  // i on lanes 3 mod 4
            const bool r = (l & 3) == 3;
#pragma unroll
            for (int b = 0; b < VL; ++b) x[b] = r ? make_float2(-x[b].y, x[b].x) : x[b];
        }
    }
}
template <int LPR, int VL> __device__ __forceinline__ void lanes_inverse(float2 (&x)[VL], int l, float2 w8)
{
#pragma unroll
    for (int half = 1; half <= LPR / 2; half <<= 1) {
        if (half == 4) {
#pragma unroll
            for (int b = 0; b < VL; ++b) x[b] = cconjmul(x[b], w8);
        }
        if (half == 2) {
            const bool r = (l & 3) == 3;
#pragma unroll
            for (int b = 0; b < VL; ++b) x[b] = r ? make_float2(x[b].y, -x[b].x) : x[b];
        }
        const float s = (l & half) ? -1.f : 1.f;
#pragma unroll
        for (int b = 0; b < VL; ++b) {
            const float2 p = make_float2(__shfl_xor_sync(0xffffffffu, x[b].x, half), __shfl_xor_sync(0xffffffffu, x[b].y, half));
            x[b] = __ffma2_rn(x[b], make_float2(s, s), p);
        }
    }
}

// Conversions by integer operations (GB300 converts two values a clock and SM); the instruction serves floats below
// 2^-126, values beyond the floats, infinities and NaN.  double to float, to nearest even:
__device__ __forceinline__ float narrow(double w)
{
    const unsigned h = (unsigned)__double2hiint(w), l = (unsigned)__double2loint(w);
    const unsigned ex = (h >> 20) & 2047u;
    if (ex - 897u > 253u && (h << 1 | l) != 0u) return (float)w;
    const unsigned rest = l & 0x1fffffffu;
    const unsigned f = __funnelshift_l(l, (h & 0x7fffffffu) - 0x38000000u, 3);
    const unsigned up = (rest > 0x10000000u || (rest == 0x10000000u && (f & 1u))) ? 1u : 0u;
    const unsigned s = h & 0x80000000u;
    return __uint_as_float(ex == 0u ? s : ((f + up) | s));
}
__device__ __forceinline__ double widen(float a)
{
    const unsigned u = __float_as_uint(a), m = u & 0x7fffffffu;
    if (m - 0x00800000u > 0x7effffffu && m != 0u) return (double)a;
    const unsigned h = (u & 0x80000000u) | (m == 0u ? 0u : (m >> 3) + 0x38000000u);
    return __hiloint2double((int)h, (int)(u << 29));
}

template <int NP>
__global__ void __launch_bounds__(res_threads(NP), 1)
resident_kernel(const ResidentMember *__restrict__ members, int n_mem, int n_steps)
{
    constexpr int VL = res_lane(NP);   // consecutive p values of a lane
    constexpr int LPR = NP / VL;       // lanes of a row
    constexpr int UNIT = 4 * LPR;      // lanes of the four pairs of a row
    static_assert(32 % UNIT == 0, "a row's pairs within a warp");
    extern __shared__ __align__(16) float smem[];
    const unsigned rank = cluster_rank(), csize = cluster_size();
    const int cluster = blockIdx.x / csize;
    int m = 0;
    while (m + 1 < n_mem && members[m + 1].cluster0 <= cluster) ++m;
    const ResidentMember &M = members[m];
    const GridInfo &g = M.g;
    const int rep = cluster - M.cluster0;
    const int E = g.n_elem, nq = g.nq, R = M.rows;
    const int lo = (int)rank * R;                          // first own row
    const int nloc = max(0, min(R, nq - lo));              // own rows
    const int RH = R + 6;
    const int PL = RH * NP, SLAB = res_slab(NP, R);
    float *A = smem, *B = smem + (size_t)E * 4 * SLAB;
    ResElem *el = reinterpret_cast<ResElem *>(B + (size_t)E * 4 * SLAB);

    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const ElemInfo &I = M.elems[e];
        ResElem &o = el[e];
        int n = 0;
        for (int a = 0; a < I.n_up; ++a, ++n) {
            o.nb[n] = I.up[a] * 16 * SLAB;
            o.wg[n] = 1.f;
            o.wa[n] = 0.f;
        }
        o.n_up = n;
        for (int pass = 0; pass < 2; ++pass) {
            for (int a = 0; a < I.n_dn; ++a) {
                if ((I.wr[a] != 0.0) != (pass == 1)) continue;
                o.nb[n] = I.dn[a] * 16 * SLAB;
                o.wg[n] = (float)I.wc[a];
                o.wa[n] = (float)I.wr[a];
                ++n;
            }
            if (pass == 0) o.n_d0 = n;
        }
        o.n_nb = n;
        o.term = I.terminator;
        o.ng = (float)I.ngam / (float)NP;
        o.fpp = M.sc[0].fdelta + (I.terminator ? M.sc[0].fterm : 0.f);
    }
    float *yrep = M.y + (size_t)rep * g.rep_stride;
    double *y0rep = M.y0 + (size_t)rep * g.tier0_rep_stride;
    const size_t blk = g.blk;

    // the swizzle of a row's 16-byte quads (np = 64: the quads of lanes 4-7 swapped, so that a
    // quarter-warp's accesses cover all banks)
    const auto quad = [](int q) { return NP == 64 ? q ^ ((q >> 3) & 1) : q; };
    // state with halos into A, zeros into B
    for (int t = threadIdx.x; t < E * 4 * SLAB; t += blockDim.x) B[t] = 0.f;
    for (int t = threadIdx.x; t < E * 4 * 2 * RH * (NP / 4); t += blockDim.x) {
        const int q = t % (NP / 4), r = (t / (NP / 4)) % RH, pp = t / (NP / 4) / RH;  // pp: (elem, pair, plane)
        int i = lo + r - 3;
        if (g.periodic_q) i = wrap_q(i, nq);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= 0 && i < nq && r < nloc + 6)
            v = *reinterpret_cast<const float4 *>(yrep + (size_t)(pp / 2) * 2 * blk + (size_t)(pp & 1) * blk + (size_t)i * NP + 4 * q);
        *reinterpret_cast<float4 *>(A + (size_t)(pp / 2) * SLAB + (pp & 1) * PL + r * NP + 4 * quad(q)) = v;
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l = lane % LPR, pair = (lane / LPR) & 3;
    const int group = threadIdx.x / UNIT, groups = blockDim.x / UNIT;
    const int EG = max(1, min(E, groups / max(R, 1)));  // element groups working on a row at once
    const int trips = (R * EG + groups - 1) / groups;   // rows per thread
    const int l0 = VL * l;
    // byte offsets of this lane's quads in a row
    const unsigned o0 = 16 * (VL == 8 ? quad(2 * l) : l), od = 16 * quad(2 * l + 1) - o0;
    const unsigned PL4 = 4u * PL, ES4 = 16u * SLAB;  // plane and element strides in bytes
    const auto lds = [&](unsigned a, float *v) {
        unpack(lds4(a), v);
        if constexpr (VL == 8) unpack(lds4(a + od), v + 4);
    };
    float pcol[VL];
    const float fkin = M.sc[0].fkin, r0 = M.sc[0].r0, inv12dp = M.sc[0].inv12dp;
#pragma unroll
    for (int v = 0; v < VL; ++v) pcol[v] = (float)(g.p_min + (l0 + v) * g.dp);
    const bool neg = pcol[0] < 0.f;
    float ck[6];
    {
        const float cneg[6] = {3, -30, -20, 60, -15, 2}, cpos[6] = {-2, 15, -60, 20, 30, -3};
#pragma unroll
        for (int t = 0; t < 6; ++t) ck[t] = neg ? cneg[t] : cpos[t];
    }
    const unsigned first = (neg ? -2 : -3) * NP * 4;  // byte offset of the stencil's first row
    int k1 = 0;  // frequency of this lane after the lane transform
#pragma unroll
    for (int b = 1; b < LPR; b <<= 1) k1 = 2 * k1 + ((l & b) ? 1 : 0);
    float2 tw[VL];
#pragma unroll
    for (int b = 1; b < VL; ++b) tw[b] = make_float2(M.tw[2 * (b * k1)], M.tw[2 * (b * k1) + 1]);
    const int t8 = (l & 4) ? (l & 3) * (NP / 8) : 0;  // e^{2 pi i (l mod 4) / 8} on the upper lanes
    const float2 w8 = make_float2(M.tw[2 * t8], M.tw[2 * t8 + 1]);
    const size_t tabn = (size_t)4 * blk;
    const float *tD = M.tab + (size_t)pair * blk + l0;                                            // D_jk
    const float *tL = M.tab + tabn + (size_t)((pair & 2) + 1 - (pair >> 1)) * blk + l0;           // L_j,1-j
    const float *tR = M.tab + 2 * tabn + (size_t)((1 - (pair & 1)) * 2 + (pair & 1)) * blk + l0;  // R_1-k,k
    const float *tP = M.tab + 3 * tabn + l0;                                                      // eigenvalues of d2/dp2
    const double mud = M.mu[(pair & 1) * 2 + (pair >> 1)];                                        // Tr{mu W}: mu_kj
    const bool traced = M.part != nullptr && mud != 0.0;

    // what depends on the thread's row: tables, places, and where the row is a halo (the same byte offset in
    // the other blocks' buffers, by rank)
    constexpr int NT = 6;
    float dD[VL], dL[VL], dR[VL];
    unsigned own = 0, halo[NT];
    int n_halo = 0;
    float *yrow = yrep;
    double *y0row = y0rep;
    const unsigned Ab = (unsigned)__cvta_generic_to_shared(A), Bb = (unsigned)__cvta_generic_to_shared(B);
    const auto set_row = [&](int rl) {
        const int i = lo + rl;
        ldv<float, VL>(tD + (size_t)i * NP, dD);
        ldv<float, VL>(tL + (size_t)i * NP, dL);
        ldv<float, VL>(tR + (size_t)i * NP, dR);
        own = (unsigned)(pair * SLAB + (rl + 3) * NP) * 4u + o0;
        const size_t c = (size_t)pair * 2 * blk + (size_t)i * NP + l0;
        yrow = yrep + c;
        y0row = y0rep + c;
        n_halo = 0;
        // the row on the unwrapped axis (periodic q: also whole periods away, as far as the three rows beyond either
        // edge reach: one where nq >= 3); block t holds t R - 3 .. t R + R + 2, so at most six others hold a row
        // (three on each side at one row a block)
        const int blocks = (nq + R - 1) / R;
        const int periods = g.periodic_q ? (nq + 2) / nq : 0;
        for (int w = -periods; w <= periods; ++w) {
            const int pos = i + w * nq;
            for (int t = 0; t < blocks; ++t) {
                const int at = pos - t * R + 3;
                if (at < 0 || at >= R + 6 || (t == (int)rank && w == 0)) continue;
                const unsigned h = map_rank(Ab + (unsigned)(pair * SLAB + at * NP) * 4u + o0, (unsigned)t);
#pragma unroll
                for (int q = 0; q < NT; ++q)
                    if (q == n_halo) halo[q] = h;
                ++n_halo;
            }
        }
    };
    {
        const int row = group / EG;
        if (nloc > 0) set_row(row < nloc ? row : 0);
    }
    cluster_sync();

    for (int step = 0; step < n_steps; ++step) {
#pragma unroll 1
        for (int k = 4; k >= 1; --k) {
            // stage 4: y in A -> B, 3: B -> A, 2: A -> B, 1: B -> A, the new y
            const unsigned in = (k & 1) ? Bb : Ab, out = (k & 1) ? Ab : Bb;
            const float h = M.sc[k].h;
            const double hd = M.hd[k];
            double trr = 0.0, tri = 0.0;
            if (nloc > 0) {
#pragma unroll 1
                for (int trip = 0; trip < trips; ++trip) {
                    const int item = trip * groups + group;
                    const int row = item / EG;
                    const bool act_row = item < R * EG && row < nloc;
                    // where all passes over the elements are full, each row starts at another one: the zeroth tier's
                    // FP64 instructions, 64 clocks of a quarter of the SM each, then don't meet (2D spectrum 198 -> 170 ms)
                    const int eg = item - row * EG + (E % EG == 0 ? row % E : 0);
                    if (trips > 1) set_row(act_row ? row : 0);
#pragma unroll 1
                    for (int e0 = 0; e0 < E; e0 += EG) {
                        const int et = e0 + eg;
                        const bool act = act_row && (E % EG == 0 || et < E);
                        const int e = act ? (et < E ? et : et - E) : 0;
                        const ResElem &I = el[e];
                        const unsigned pe = in + own + e * ES4;  // this lane's values of the row (real part)
                        const size_t go = (size_t)e * g.elem_stride;
                        float2 x[VL];
                        {
                            float a[VL], c[VL];
                            lds(pe, a);
                            lds(pe + PL4, c);
#pragma unroll
                            for (int v = 0; v < VL; ++v) x[v] = make_float2(a[v], c[v]);
                        }
                        // the step's base, asked for early: y (at the first stage the input itself), for the zeroth tier
                        // its FP64 value, whose parts take the registers of both planes
                        float base[4 * VL];
                        if (e == 0) {
                            const float *w = reinterpret_cast<const float *>(y0row);
                            ldrow<float, 2 * VL>(w, base);
                            ldrow<float, 2 * VL>(w + 2 * blk, base + 2 * VL);
                        } else if (k != 4) {
                            ldrow<float, VL>(yrow + go, base);
                            ldrow<float, VL>(yrow + go + blk, base + VL);
                        } else {
                            lds(pe, base);
                            lds(pe + PL4, base + VL);
                        }
                        lanes_forward<LPR, VL>(x, l, w8);
#pragma unroll
                        for (int b = 1; b < VL; ++b) x[b] = cmul(x[b], tw[b]);
                        dft_small<VL, +1>(x);
                        {
                            const float fpp = I.fpp, ng = I.ng;
                            float lpp[VL];
                            ldv<float, VL>(tP, lpp);
#pragma unroll
                            for (int v = 0; v < VL; ++v) {
                                const float2 a = make_float2(__shfl_xor_sync(0xffffffffu, x[v].x, 2 * LPR),
                                                             __shfl_xor_sync(0xffffffffu, x[v].y, 2 * LPR));
                                const float2 c = make_float2(__shfl_xor_sync(0xffffffffu, x[v].x, LPR),
                                                             __shfl_xor_sync(0xffffffffu, x[v].y, LPR));
                                const float2 s = __ffma2_rn(make_float2(-dR[v], -dR[v]), c,
                                                            __ffma2_rn(make_float2(dL[v], dL[v]), a,
                                                                       __fmul2_rn(make_float2(dD[v], dD[v]), x[v])));
                                const float cf = fmaf(fpp, lpp[v], -ng);
                                x[v] = __ffma2_rn(make_float2(cf, cf), x[v], make_float2(s.y, -s.x));
                            }
                        }
                        dft_small<VL, -1>(x);
#pragma unroll
                        for (int b = 1; b < VL; ++b) x[b] = cconjmul(x[b], tw[b]);
                        lanes_inverse<LPR, VL>(x, l, w8);
                        // kinetic term: six rows
                        float ar[VL], ai[VL];
                        {
                            float kr[VL], ki[VL], r8[VL];
#pragma unroll
                            for (int v = 0; v < VL; ++v) kr[v] = ki[v] = 0.f;
                            const unsigned pr = pe + first, pi = pr + PL4;
#pragma unroll
                            for (int t = 0; t < 6; ++t) {
                                lds(pr + t * NP * 4, r8);
                                v_axpy<VL>(kr, ck[t], r8);
                                lds(pi + t * NP * 4, r8);
                                v_axpy<VL>(ki, ck[t], r8);
                            }
#pragma unroll
                            for (int v = 0; v < VL; ++v) {
                                const float pk = -(pcol[v] * fkin);
                                ar[v] = fmaf(kr[v], pk, x[v].x);
                                ai[v] = fmaf(ki[v], pk, x[v].y);
                            }
                        }
                        // tier couplings
                        float gr[VL], gi[VL];
#pragma unroll
                        for (int v = 0; v < VL; ++v) gr[v] = gi[v] = 0.f;
                        const int n_d0 = I.n_d0, n_nb = act ? I.n_nb : 0;
                        const unsigned pn = in + own;
#pragma unroll 1
                        for (int n = 0; n < n_nb; ++n) {
                            const unsigned u = pn + (unsigned)I.nb[n];
                            float xr[VL], xi[VL];
                            lds(u, xr);
                            lds(u + PL4, xi);
                            const float wg = I.wg[n];
                            v_axpy<VL>(gr, wg, xr);
                            v_axpy<VL>(gi, wg, xi);
                            if (n >= n_d0) {
                                const float wa = I.wa[n];
                                float pw[VL];
#pragma unroll
                                for (int v = 0; v < VL; ++v) pw[v] = wa * pcol[v];
                                v_fma<VL>(ar, pw, xr);
                                v_fma<VL>(ai, pw, xi);
                            }
                        }
                        if (I.term) {  // r_0 p W of the Eq. (GMFP) terminator
                            float r0p[VL], w0[VL], w1[VL];
                            lds(pe, w0);
                            lds(pe + PL4, w1);
#pragma unroll
                            for (int v = 0; v < VL; ++v) r0p[v] = r0 * pcol[v];
                            v_fma<VL>(gr, r0p, w0);
                            v_fma<VL>(gi, r0p, w1);
                        }
                        __syncwarp();
                        {  // 4th-order central d/dp of the tier sum, periodic p
                            const int left = (l + LPR - 1) % LPR, right = (l + 1) % LPR;
                            const auto ddp = [&](const float *G, float *a) {
                                float ex[VL + 4];
#pragma unroll
                                for (int v = 0; v < VL; ++v) ex[v + 2] = G[v];
                                ex[0] = __shfl_sync(0xffffffffu, G[VL - 2], left, LPR);
                                ex[1] = __shfl_sync(0xffffffffu, G[VL - 1], left, LPR);
                                ex[VL + 2] = __shfl_sync(0xffffffffu, G[0], right, LPR);
                                ex[VL + 3] = __shfl_sync(0xffffffffu, G[1], right, LPR);
#pragma unroll
                                for (int v = 0; v < VL; ++v)
                                    a[v] += inv12dp * (ex[v] - 8.f * ex[v + 1] + 8.f * ex[v + 3] - ex[v + 4]);
                            };
                            ddp(gr, ar);
                            ddp(gi, ai);
                        }
                        if (!act) continue;
                        // ---- update: base + h L
                        float br[VL], bi[VL];
                        if (e != 0) {
#pragma unroll
                            for (int v = 0; v < VL; ++v) {
                                br[v] = base[v];
                                bi[v] = base[VL + v];
                            }
                            v_axpy<VL>(br, h, ar);
                            v_axpy<VL>(bi, h, ai);
                            if (k == 1) {
                                strow<float, VL>(yrow + go, br);
                                strow<float, VL>(yrow + go + blk, bi);
                            }
                        } else {
                            const auto accumulate = [&](const float (&a)[VL], float (&b)[VL], const float *w0, size_t off, double &sum) {
                                double w[VL], tr = 0.0;
#pragma unroll
                                for (int v = 0; v < VL; ++v) {
                                    w[v] = __hiloint2double(__float_as_int(w0[2 * v + 1]), __float_as_int(w0[2 * v]));
                                    w[v] = fma(hd, widen(a[v]), w[v]);
                                    b[v] = narrow(w[v]);
                                    if (traced && k == 1) tr += w[v];
                                }
                                if (k == 1) {
                                    strow<double, VL>(y0row + off, w);
                                    strow<float, VL>(yrow + off, b);
                                    if (traced) sum += mud * tr;
                                }
                            };
                            accumulate(ar, br, base, 0, trr);
                            accumulate(ai, bi, base + 2 * VL, blk, tri);
                        }
                        // own buffer, and the halos of the blocks within three rows
                        const unsigned po = out + own + e * ES4;
                        sts4(po, pack(br));
                        sts4(po + PL4, pack(bi));
                        if constexpr (VL == 8) {
                            sts4(po + od, pack(br + 4));
                            sts4(po + PL4 + od, pack(bi + 4));
                        }
                        const unsigned he = out - Ab + e * ES4;
#pragma unroll
                        for (int q = 0; q < NT; ++q) {
                            if (q < n_halo) {
                                const unsigned a = halo[q] + he;
                                stc4(a, pack(br));
                                stc4(a + PL4, pack(bi));
                                if constexpr (VL == 8) {
                                    stc4(a + od, pack(br + 4));
                                    stc4(a + PL4 + od, pack(bi + 4));
                                }
                            }
                        }
                    }
                }
            }
            if (k == 1 && M.part) {  // this warp's part of Tr{mu W^(0)}
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    trr += __shfl_xor_sync(0xffffffffu, trr, off);
                    tri += __shfl_xor_sync(0xffffffffu, tri, off);
                }
                if (lane == 0) {
                    const int warps = blockDim.x >> 5;
                    double *p = M.part + 2 * ((((size_t)rep * n_steps + step) * csize + rank) * warps + warp);
                    p[0] = trr;
                    p[1] = tri;
                }
            }
            cluster_sync();
        }
    }
}

// traces of n_steps steps: the n_part warps' parts added in a fixed order (a warp per step: strided sums, then
// a butterfly over the lanes), into slots slot0.. of each replica
__global__ void resident_trace_kernel(const double *__restrict__ part, int n_rep, int n_steps, int n_part, double scale,
                                      double *out, long stride, long slot0)
{
    const long total = (long)n_rep * n_steps;
    const int lane = threadIdx.x & 31;
    for (long t = (blockIdx.x * (long)blockDim.x + threadIdx.x) >> 5; t < total; t += ((long)gridDim.x * blockDim.x) >> 5) {
        double a = 0.0, b = 0.0;
        for (int c = lane; c < n_part; c += 32) {
            const double2 v = reinterpret_cast<const double2 *>(part)[t * n_part + c];
            a += v.x;
            b += v.y;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, off);
            b += __shfl_xor_sync(0xffffffffu, b, off);
        }
        if (lane) continue;
        double *o = out + 2 * ((t / n_steps) * stride + slot0 + t % n_steps);
        o[0] = a * scale;
        o[1] = b * scale;
    }
}

constexpr size_t resident_smem_limit() { return 220 * 1024; }

template <int NP>
cudaError_t configure(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int clusters, int csize, int threads, size_t smem,
                      cudaStream_t st)
{
    // (always the same limit: handles on other threads launch the same kernel)
    cudaError_t e = cudaFuncSetAttribute(resident_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)resident_smem_limit());
    if (!e) e = cudaFuncSetAttribute(resident_kernel<NP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e) return e;
    cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * csize));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)csize;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaSuccess;
}

}  // namespace

bool resident_supported(int np, int S) { return (np == 32 || np == 64) && S == 2; }

int resident_frequency(int np, int pos)
{
    const int vl = res_lane(np), lpr = np / vl, l = pos / vl;
    int k1 = 0;
    for (int b = 1; b < lpr; b <<= 1) k1 = 2 * k1 + ((l & b) ? 1 : 0);
    return k1 + lpr * (pos % vl);
}

size_t resident_smem(int np, int n_elem, int rows)  // 0: more than a block can have
{
    const size_t n = (size_t)2 * n_elem * 4 * res_slab(np, rows) * sizeof(float) + (size_t)n_elem * sizeof(ResElem);
    return n <= resident_smem_limit() ? n : 0;
}

int resident_threads(int np, int n_elem, int rows)
{
    const int want = rows * n_elem * (4 * np / res_lane(np));  // lanes of the pairs of a row
    return std::min(res_threads(np), (want + 31) / 32 * 32);
}

cudaError_t resident_capacity(int np, int csize, int threads, size_t smem, int *clusters)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    *clusters = 0;
    cudaError_t e = np == 32 ? configure<32>(cfg, attr, 1, csize, threads, smem, nullptr)
                             : configure<64>(cfg, attr, 1, csize, threads, smem, nullptr);
    if (e) return e;
    return np == 32 ? cudaOccupancyMaxActiveClusters(clusters, resident_kernel<32>, &cfg)
                    : cudaOccupancyMaxActiveClusters(clusters, resident_kernel<64>, &cfg);
}

cudaError_t launch_resident(int np, const ResidentMember *members, int n_mem, int clusters, int csize, int threads,
                            size_t smem, int n_steps, cudaStream_t st)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cudaError_t e = np == 32 ? configure<32>(cfg, attr, clusters, csize, threads, smem, st)
                             : configure<64>(cfg, attr, clusters, csize, threads, smem, st);
    if (e) return e;
    return np == 32 ? cudaLaunchKernelEx(&cfg, resident_kernel<32>, members, n_mem, n_steps)
                    : cudaLaunchKernelEx(&cfg, resident_kernel<64>, members, n_mem, n_steps);
}

cudaError_t launch_resident_trace(const double *part, int n_rep, int n_steps, int n_part, double scale, double *out,
                                  long stride, long slot0, cudaStream_t st)
{
    const long total = (long)n_rep * n_steps;
    resident_trace_kernel<<<(unsigned)std::min<long>((total + 3) / 4, 152 * 16), 128, 0, st>>>(part, n_rep, n_steps, n_part,
                                                                                     scale, out, stride, slot0);
    return cudaGetLastError();
}
