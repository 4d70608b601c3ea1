// kernels_ang.cu -- the operator apply A_+- x (Eq. solPsi with the coupling of Eq. fullH) in
// factorised form, angular sums first: the coupling values are never formed.
//
// In the frame of the output channel a every partner b = (kappa_b, mu +- 1) contributes
//   sign sum_l [ alpha_l(a,b) K_l(ka, kb) + beta_l(a,b) KT_l(kb, ka) ] x_b
// with K_l(k', k) = G0 + k' G1 + k G2 + k' k G3 (the pulse bands of multipole l at the current time),
// KT the block transpose, and alpha, beta the angular coefficients.  The dual-kinetic-balance
// functions make most of the 2 x 2 entries of the G bands zero: P = p0 + kappa p1 has p1 = 0 for type
// 0, Q = q0 + kappa q1 has q1 = 0 for type 1, so G1 = int p1 F q0 has only type-1 rows, G2 = int p0 F q1
// only type-0 columns and G3 = int p1 F q1 the single entry (1, 0).  Collecting what the partners enter
// with, six sums per (channel a, multipole l, slot) carry all of them:
//   s1 = sum alpha x0   s2 = sum alpha kb x0   s3 = sum alpha x1
//   s4 = sum beta x0    s5 = sum beta x1       s6 = sum beta kb x1     (x0, x1: the two DKB types of x_b)
// and the rows of a follow from twelve bands that depend on (l, kappa_a) only:
//   y0 += G0[00] s1 + G2[00] s2 + G0[01] s3 + T(G0[00] + ka G2[00]) s4 + T(G0[10] + ka G2[10]) s5
//         + T(G1[10] + ka G3[10]) s6
//   y1 += (G0[10] + ka G1[10]) s1 + (G2[10] + ka G3[10]) s2 + (G0[11] + ka G1[11]) s3 + T(G0[01]) s4
//         + T(G0[11]) s5 + T(G1[11]) s6
// (T: the value at the transposed band position).  Per apply that is 12 real multiply-adds per
// directed (pair, multipole) and slot and 24 per (channel, multipole, band position): 2.3e9 + 4.1e9
// at 1860 channels, 1001 slots and seven multipoles, against 8.5e9 for the stored coupling, whose
// 2.1e9 values also have to be formed and read.
//
// Two launches:
//   k_ang  block = a few output channels of one mu at 128 slots, a thread per slot: a partner's x at the
//          slot is loaded once for the block's outputs; the six sums of each (a, l) go to the buffer S,
//          [a][l][6][slot].
//   k_rad  block = up to two kappa chunks of together <= 32 channels on the lanes of a warp x 8 warps
//          of consecutive slots.  Stage by stage (one of the six sums of one l, then the diagonal
//          block) the channels' windows arrive by cp.async one stage ahead, the stage's two band rows
//          are formed for each kappa in shared memory, and every lane applies them, read as
//          broadcasts, to its channel's window in registers.  The result leaves through shared memory
//          with the BiCGSTAB epilogues.
// S is written once and read 1.2 to 1.4 times (the windows' halo); 0.65 GB in complex64 at the size
// above.  Precision policies: float (the complex64 operator), double-float (the refinement residual and
// the accurate apply of precision 2) and double (precision 0).
//
// Times at 1860 channels, 1001 slots, seven multipoles (k_ang + k_rad; band entries 0.03 ms once per
// time), against the stored form (its values once per time: 4.4 ms double-float):
//   complex64      0.24 + 0.33 ms   subgroup form 1.03 ms, stored owner/gather form 1.56 ms
//   double-float   0.93 + 1.50 ms   owner + gather passes 3.12 + 0.61 ms
//   FP64           3.95 + 8.14 ms   row kernel 15.6 ms
// Counters at 420 channels and 601 slots: the FP64 one holds the FP64 pipe at 97 % in both passes.  The
// double-float one has the FMA pipe at 46 (k_ang) and 54 % (k_rad) with the offsets, 64 and 71 % as Dot2 sums, and
// latency for the rest: k_rad's 2 x RSL complex accumulators and window in registers leave two blocks an
// SM.  The complex64 one is bound by latency (FMA pipe 23 and 29 %): 6.4e9 multiply-adds of FP32 alone
// would take 0.17 ms at the size above.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "device.h"
#include "df64.cuh"
#include "kernels.h"
#include "mbar.cuh"

namespace dg {

namespace {
constexpr int BDG = 13, HG = (BDG - 1) / 2;   // block diagonals (order-7 splines)
constexpr int NS = 6;                         // angular sums per (channel, multipole)
constexpr int RWP = 8;                        // warps per radial block
constexpr int MARGIN = 8;                     // zero slots before and (at least) after the n1 slots of a row
constexpr int RT = 32 * RWP;

// ---- packed pairs of floats (one instruction of the FMA pipe for two lanes' worth of work) ----
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 up(f2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)   // a - b, exact negation folded into the FMA
{
    return fma2(b, pk(-1.f, -1.f), a);
}

// ---- double-float on packed pairs: two independent accumulators in one instruction stream ----
struct D2 { f2 s, c; };   // running sums and corrections

// df_fma (Dot2 form, ten operations): a += (kh + kl) (xh + xl) in both halves.  The rounded products
// are formed by scalar multiplications: a packed one was contracted into the sum that follows it (the
// residues were then wrong by an ulp of the product where it exceeds the sum).
__device__ __forceinline__ void d2_fma(D2& a, f2 kh, f2 kl, f2 xh, f2 xl)
{
    const float2 k = up(kh), x = up(xh);
    const f2 p = pk(__fmul_rn(k.x, x.x), __fmul_rn(k.y, x.y));
    const f2 t = add2(a.s, p);
    const f2 nz = sub2(a.s, t);               // -(t - s)
    const f2 r1 = sub2(a.s, add2(t, nz));     // s - (t - z)
    const f2 r2 = fma2(kh, xh, nz);           // product - z, rounded once
    const f2 c = fma2(kl, xh, fma2(kh, xl, a.c));
    a.s = t;
    a.c = add2(c, add2(r1, r2));
}
// df_fma_off (fixed-binade form, six operations): a.s carries an offset
__device__ __forceinline__ void d2_fma_off(D2& a, f2 kh, f2 kl, f2 xh, f2 xl)
{
    const f2 t = fma2(kh, xh, a.s);
    const f2 nd = sub2(a.s, t);
    const f2 e = fma2(kh, xh, nd);
    a.c = fma2(kl, xh, fma2(kh, xl, add2(a.c, e)));
    a.s = t;
}
__device__ __forceinline__ void d2_add(D2& a, const D2& b)   // df_add
{
    const f2 t = add2(a.s, b.s);
    const f2 nz = sub2(a.s, t);
    const f2 r1 = sub2(a.s, add2(t, nz));
    const f2 r2 = add2(b.s, nz);
    a.s = t;
    a.c = add2(a.c, add2(b.c, add2(r1, r2)));
}
// offset 1.5 * 2^k with 2^(k-2) above the bound B of a sum of |products|
__device__ __forceinline__ float off_of(float B) { return df_offset(df_offset_byte(B)); }

// ---- precision policies --------------------------------------------------------------------------
// C: a complex element in memory; R: a real band value or coefficient in memory.
//  angular pass: AG outputs per thread, ACH items staged at a time; K: a coefficient; Acc: one complex sum.
//  radial pass: RSL slots per thread, XW the staged window stride (C; 16-byte rows, conflict-free
//  16-byte lane reads), E: the (row 0, row 1) factors of a band position; RAcc: both rows of one slot.
struct PF {
    typedef float2 C;
    typedef float R;
    static constexpr int AG = 4, ACH = 64;
    static constexpr bool SPLIT = false;
    typedef float K;
    struct Acc { float x, y; };
    static __device__ __forceinline__ Acc zero() { return {0.f, 0.f}; }
    static __device__ __forceinline__ void fma(Acc& a, K c, C x) { a.x = fmaf(c, x.x, a.x); a.y = fmaf(c, x.y, a.y); }
    static __device__ __forceinline__ C get(const Acc& a) { return make_float2(a.x, a.y); }
    static __device__ __forceinline__ C czero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ R rzero() { return 0.f; }

    static constexpr int RSL = 8, XW = 78, EW = 14;
    static __device__ __forceinline__ int place(int ls, int d) { return ls * EW + (ls & 1) + d; }   // see the radial pass
    typedef float2 E;
    struct RAcc { f2 re, im; };   // (row 0, row 1) packed
    static __device__ __forceinline__ R comb(R a, float k, R b) { return fmaf(k, b, a); }   // a + k b
    static __device__ __forceinline__ R scale(double s, R a) { return (float)s * a; }
    static __device__ __forceinline__ E pair(R e0, R e1) { return make_float2(e0, e1); }
    static __device__ __forceinline__ void rzero(RAcc& a) { a.re = a.im = 0ull; }
    static __device__ __forceinline__ C rot(C x) { return make_float2(-x.y, x.x); }   // i x
    static __device__ __forceinline__ void times(RAcc& a, float r0, float r1)
    {
        a.re = fma2(a.re, pk(r0, r1), 0ull);
        a.im = fma2(a.im, pk(r0, r1), 0ull);
    }
    static __device__ __forceinline__ float4 rows(const RAcc& a)   // (y0, y1)
    {
        const float2 r = up(a.re), i = up(a.im);
        return make_float4(r.x, i.x, r.y, i.y);
    }
};

struct PD {
    typedef double2 C;
    typedef double R;
    static constexpr int AG = 4, ACH = 64;
    static constexpr bool SPLIT = false;
    typedef double K;
    struct Acc { double x, y; };
    static __device__ __forceinline__ Acc zero() { return {0.0, 0.0}; }
    static __device__ __forceinline__ void fma(Acc& a, K c, C x) { a.x = ::fma(c, x.x, a.x); a.y = ::fma(c, x.y, a.y); }
    static __device__ __forceinline__ C get(const Acc& a) { return make_double2(a.x, a.y); }
    static __device__ __forceinline__ C czero() { return make_double2(0, 0); }
    static __device__ __forceinline__ R rzero() { return 0.0; }

    static constexpr int RSL = 4, XW = 45, EW = 13;
    static __device__ __forceinline__ int place(int ls, int d) { return ls * EW + d; }
    typedef double2 E;
    struct RAcc { double r0, i0, r1, i1; };
    static __device__ __forceinline__ R comb(R a, float k, R b) { return ::fma((double)k, b, a); }
    static __device__ __forceinline__ R scale(double s, R a) { return s * a; }
    static __device__ __forceinline__ E pair(R e0, R e1) { return make_double2(e0, e1); }
    static __device__ __forceinline__ void rzero(RAcc& a) { a.r0 = a.i0 = a.r1 = a.i1 = 0.0; }
    static __device__ __forceinline__ C rot(C x) { return make_double2(-x.y, x.x); }
    static __device__ __forceinline__ void times(RAcc& a, float r0, float r1)
    {
        a.r0 *= r0; a.i0 *= r0; a.r1 *= r1; a.i1 *= r1;
    }
    static __device__ __forceinline__ double2 row(const RAcc& a, int t)
    {
        return t ? make_double2(a.r1, a.i1) : make_double2(a.r0, a.i0);
    }
};

// double-float: C = (re hi, im hi, re lo, im lo), R = (hi, lo).  The angular pass packs real and
// imaginary part (its coefficients are kept with each word doubled), the radial pass the two rows (the
// x words are doubled once per window element and used by all its slots).
struct PX {
    typedef float4 C;
    typedef float2 R;
    static constexpr int AG = AGX, ACH = 32;
    static constexpr bool SPLIT = true;
    typedef ulonglong2 K;   // (hi, hi), (lo, lo)
    typedef D2 Acc;
    static __device__ __forceinline__ Acc zero() { return {0ull, 0ull}; }
    static __device__ __forceinline__ void fma(Acc& a, const K& k, const C& x) { d2_fma(a, k.x, k.y, pk(x.x, x.y), pk(x.z, x.w)); }
    static __device__ __forceinline__ void fma_off(Acc& a, const K& k, const C& x)
    {
        d2_fma_off(a, k.x, k.y, pk(x.x, x.y), pk(x.z, x.w));
    }
    static __device__ __forceinline__ Acc offset(float sg) { return {pk(sg, sg), 0ull}; }
    static __device__ __forceinline__ void unoffset(Acc& a, float sg) { a.s = sub2(a.s, pk(sg, sg)); }   // exact
    static __device__ __forceinline__ C get(const Acc& a)   // normalised words
    {
        const f2 h = add2(a.s, a.c), l = add2(sub2(a.s, h), a.c);
        const float2 hh = up(h), ll = up(l);
        return make_float4(hh.x, hh.y, ll.x, ll.y);
    }
    static __device__ __forceinline__ C czero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
    static __device__ __forceinline__ R rzero() { return make_float2(0.f, 0.f); }

    static constexpr int RSL = 4, XW = 45, EW = 13;
    static __device__ __forceinline__ int place(int ls, int d) { return ls * EW + d; }
    typedef float4 E;   // (row 0 hi, row 1 hi, row 0 lo, row 1 lo)
    struct RAcc { D2 re, im; };
    static __device__ __forceinline__ R comb(R a, float k, R b)   // a + k b, k a small integer
    {
        DfAcc v = {a.x, a.y};
        df_fma(v, k, 0.f, b.x, b.y);
        const float h = v.s + v.c;
        return make_float2(h, (v.s - h) + v.c);
    }
    static __device__ __forceinline__ R scale(double s, R a) { const float f = (float)s; return make_float2(f * a.x, f * a.y); }   // s = +-1
    static __device__ __forceinline__ E pair(R e0, R e1) { return make_float4(e0.x, e1.x, e0.y, e1.y); }
    static __device__ __forceinline__ void rzero(RAcc& a) { a.re.s = a.re.c = a.im.s = a.im.c = 0ull; }
    static __device__ __forceinline__ C rot(C x) { return make_float4(-x.y, x.x, -x.w, x.z); }
    static __device__ __forceinline__ void times(RAcc& a, float r0, float r1)
    {
        const f2 f = pk(r0, r1);
        a.re.s = fma2(a.re.s, f, 0ull); a.re.c = fma2(a.re.c, f, 0ull);
        a.im.s = fma2(a.im.s, f, 0ull); a.im.c = fma2(a.im.c, f, 0ull);
    }
    static __device__ __forceinline__ double2 row(const RAcc& a, int t)
    {
        const float2 rs = up(a.re.s), rc = up(a.re.c), is = up(a.im.s), ic = up(a.im.c);
        return t ? make_double2((double)rs.y + (double)rc.y, (double)is.y + (double)ic.y)
                 : make_double2((double)rs.x + (double)rc.x, (double)is.x + (double)ic.x);
    }
};

// x of one channel at one slot, both types
__device__ __forceinline__ void load_x(const float2* x, int ch, int n1, int, int r, float2& a, float2& b)
{
    const float4 v = __ldg(reinterpret_cast<const float4*>(x) + (int64_t)ch * n1 + r);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load_x(const double2* x, int ch, int n1, int, int r, double2& a, double2& b)
{
    const double2* p = x + ((int64_t)ch * n1 + r) * 2;
    a = __ldg(p);
    b = __ldg(p + 1);
}
__device__ __forceinline__ void load_x(const float4* x, int ch, int, int NP, int r, float4& a, float4& b)
{
    const float4* p = x + (int64_t)ch * 2 * NP + MARGIN + r;   // split vector, type-major with margins
    a = __ldg(p);
    b = __ldg(p + NP);
}
}  // namespace

// ---------------------------------------------------------------------------------------------
// Angular pass.  Block = a list of AG output channels of one mu and one parity of the orbital l
// (neighbours in |kappa|, which share most partners) at AT row positions, a thread per position: a
// partner's x is loaded once for the AG outputs.  Per multipole the list's items are the partners of any
// of its outputs, each with a mask of the outputs that use it (uniform branches: no multiply-add with a
// zero) and (alpha, alpha kb, beta, beta kb) per output; the block stages ACH of them at a time.  The x
// of the next pair of items is loaded while a pair is used.  Positions outside the grid (the margins)
// are written as zeros.
// OFF (double-float): the sums take the fixed-binade form, their offsets from the coefficients'
// absolute sums and the largest |x| (xmax, per channel and position) among the multipole's partners.
// ---------------------------------------------------------------------------------------------
constexpr int AT = 128;     // row positions (threads) per angular block

template <class P, bool OFF>
__global__ void __launch_bounds__(AT)
    k_ang(int n1, AngList G, const typename P::K* __restrict__ coef, const typename P::C* __restrict__ x,
          const float* __restrict__ xmax, typename P::C* __restrict__ S, int NC, int NP, const KState* skip,
          const int* gate)
{
    typedef typename P::C C;
    typedef typename P::K K;
    constexpr int AG = P::AG, ACH = P::ACH;
    if (skip && skip->done) return;   // uniform over the grid
    if (gate && !*gate) return;
    __shared__ __align__(16) K sc[ACH][AG][4];
    __shared__ int sb[ACH + 2];
    const int g = blockIdx.y, tid = threadIdx.x;
    const int pos = blockIdx.x * AT + tid, r = pos - MARGIN, rc = min(max(r, 0), n1 - 1);
    const bool in = r >= 0 && r < n1, act = pos < NP;
    int out[AG];
#pragma unroll
    for (int j = 0; j < AG; j++) out[j] = G.out[g * AG + j];
    if (NC > G.L * NS && act) {   // the channels' own x, for the diagonal stages
#pragma unroll
        for (int j = 0; j < AG; j++) {
            if (out[j] < 0) continue;
            C a = P::czero(), b = P::czero();
            if (in) load_x(x, out[j], n1, NP, r, a, b);
            C* o = S + ((int64_t)out[j] * NC + G.L * NS) * NP + pos;
            o[0] = a;
            o[NP] = b;
        }
    }
    int i0 = G.start[g * G.L], se = i0, base = i0;   // items base .. se - 1 are staged
    const int iend = G.start[(g + 1) * G.L];
    C xa[2][2], xb[2][2];
    auto stage = [&](int i) {
        base = i;
        se = min(i + ACH, iend);
        __syncthreads();   // the previous items are no longer read
        for (int e = tid; e < (se - base) * AG * 4; e += AT) (&sc[0][0][0])[e] = coef[(int64_t)base * AG * 4 + e];
        if (tid < ACH + 2 && base + tid < iend) sb[tid] = G.item[base + tid];   // the next pair's partners too
        __syncthreads();
    };
    static_assert(ACH + 2 <= AT && ACH % 4 == 0, "one item word per thread, whole groups");
    // the sums over the list's multipoles; EDGE: the block holds slot 0, where functions that the
    // partner's kappa leaves unused count as zero
    auto sweep = [&](auto edge) {
        constexpr bool EDGE = decltype(edge)::value;
        auto load = [&](int buf, int i) {   // items i, i + 1
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int b = sb[i - base + q];
                load_x(x, b & ITEM_CH, n1, NP, rc, xa[buf][q], xb[buf][q]);
                if (EDGE && rc == 0) {
                    if (b & ITEM_NO0) xa[buf][q] = P::czero();
                    if (b & ITEM_NO1) xb[buf][q] = P::czero();
                }
            }
        };
        if (iend > i0) {
            stage(i0);
            load(0, i0);
        }
        for (int l = 0; l < G.L; l++) {
            const int i1 = G.start[g * G.L + l + 1];
            typename P::Acc acc[AG][NS];
            float M = 0.f;
            if constexpr (OFF) {
#pragma unroll 4
                for (int i = i0; i < i1; i++) M = fmaxf(M, __ldg(xmax + (int64_t)(G.item[i] & ITEM_CH) * NP + MARGIN + rc));
            }
#pragma unroll
            for (int j = 0; j < AG; j++) {
                if constexpr (OFF) {
                    const float4 cs = G.csum[(g * G.L + l) * AG + j];   // sums of |alpha|, |alpha kb|, |beta|, |beta kb|
                    const float o0 = off_of(cs.x * M), o1 = off_of(cs.y * M), o2 = off_of(cs.z * M), o3 = off_of(cs.w * M);
                    acc[j][0] = P::offset(o0); acc[j][1] = P::offset(o1); acc[j][2] = P::offset(o0);
                    acc[j][3] = P::offset(o2); acc[j][4] = P::offset(o2); acc[j][5] = P::offset(o3);
                } else {
#pragma unroll
                    for (int q = 0; q < NS; q++) acc[j][q] = P::zero();
                }
            }
            auto pair = [&](int buf, int i) {   // items i, i + 1, in buffer buf
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const int b = sb[i - base + q];
#pragma unroll
                    for (int j = 0; j < AG; j++) {
                        if (!(b & (ITEM_USE << j))) continue;   // uniform over the block
                        const K* c = sc[i - base + q][j];
                        const K ca = c[0], cak = c[1], cb = c[2], cbk = c[3];
                        typename P::Acc* a = acc[j];
                        if constexpr (OFF) {
                            P::fma_off(a[0], ca, xa[buf][q]);
                            P::fma_off(a[1], cak, xa[buf][q]);
                            P::fma_off(a[2], ca, xb[buf][q]);
                            P::fma_off(a[3], cb, xa[buf][q]);
                            P::fma_off(a[4], cb, xb[buf][q]);
                            P::fma_off(a[5], cbk, xb[buf][q]);
                        } else {
                            P::fma(a[0], ca, xa[buf][q]);
                            P::fma(a[1], cak, xa[buf][q]);
                            P::fma(a[2], ca, xb[buf][q]);
                            P::fma(a[3], cb, xa[buf][q]);
                            P::fma(a[4], cb, xb[buf][q]);
                            P::fma(a[5], cbk, xb[buf][q]);
                        }
                    }
                }
            };
            for (; i0 < i1; i0 += 4) {   // item counts are multiples of 4
                if (i0 == se) stage(i0);   // its x is in buffer 0 already
                load(1, i0 + 2);
                pair(0, i0);
                if (i0 + 4 < iend) load(0, i0 + 4);
                pair(1, i0 + 2);
            }
            if (!act) continue;   // the barriers are reached by every thread of the block
#pragma unroll
            for (int j = 0; j < AG; j++) {
                if (out[j] < 0) continue;
                if constexpr (OFF) {
                    const float4 cs = G.csum[(g * G.L + l) * AG + j];
                    const float o0 = off_of(cs.x * M), o1 = off_of(cs.y * M), o2 = off_of(cs.z * M), o3 = off_of(cs.w * M);
                    P::unoffset(acc[j][0], o0); P::unoffset(acc[j][1], o1); P::unoffset(acc[j][2], o0);
                    P::unoffset(acc[j][3], o2); P::unoffset(acc[j][4], o2); P::unoffset(acc[j][5], o3);
                }
                C* o = S + ((int64_t)out[j] * NC + l * NS) * NP + pos;
#pragma unroll
                for (int q = 0; q < NS; q++) o[(int64_t)q * NP] = in ? P::get(acc[j][q]) : P::czero();
            }
        }
    };
    if (blockIdx.x == 0) sweep(std::true_type{});
    else sweep(std::false_type{});
}

// ---------------------------------------------------------------------------------------------
// Band entries of the radial pass, each time the field changes: for (l, stage c) the three values
// (a0, a1, b) per band position with row factors e0 = a0, e1 = a1 + ka b (c < 3) or e0 = a0 + ka b,
// e1 = a1 (c >= 3), the transposed ones read at the transposed position (zero outside the grid).
// E[l][c][3][n1 x BDG].  The time factors multiply the static pulse matrices in FP64.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_rad_entries(PulseView P, int n1, const double* __restrict__ s,
                                                     float* __restrict__ Ef, float2* __restrict__ Ex,
                                                     double* __restrict__ Ed)
{
    const int nrd = n1 * BDG, be = nrd * 4;
    const int idx = blockIdx.x * 256 + threadIdx.x, l = blockIdx.y / NS, c = blockIdx.y % NS;
    if (idx >= nrd) return;
    const int r = idx / BDG, d = idx - r * BDG, rr = r + d - HG;
    const bool in = rr >= 0 && rr < n1;
    // (n, 2 x 2 entry) of a0, a1, b for each c, and whether read at the transposed position
    const int nn[NS][3] = {{0, 0, 1}, {2, 2, 3}, {0, 0, 1}, {0, 0, 2}, {0, 0, 2}, {1, 1, 3}};
    const int ee[NS][3] = {{0, 2, 2}, {0, 2, 2}, {1, 3, 3}, {0, 1, 0}, {2, 3, 2}, {2, 3, 2}};
    const int pos = c < 3 ? idx : rr * BDG + (2 * HG - d);
#pragma unroll
    for (int k = 0; k < 3; k++) {
        double v = 0;
        if (in) {
            int n = 0, e = 0;
#pragma unroll
            for (int q = 0; q < NS; q++)
                if (q == c) { n = nn[q][k]; e = ee[q][k]; }
            const int64_t o = (int64_t)n * be + (int64_t)pos * 4 + e;
            for (int cc = 0; cc < 3; cc++) v += s[l * 3 + cc] * P.M[((int64_t)l * 3 + cc) * 4 * be + o];
        }
        const int64_t w = ((int64_t)(l * NS + c) * 3 + k) * nrd + idx;
        const float2 h = df_split(v);
        if (Ef) Ef[w] = h.x;
        if (Ex) Ex[w] = h;
        if (Ed) Ed[w] = v;
    }
}

// row sums of |a0|, |a1|, |b| over the band, rounded up: the bounds of the fixed-binade form
__global__ void __launch_bounds__(256) k_rad_rowsums(int n1, int rows, const float2* __restrict__ Ex,
                                                     float* __restrict__ rs)
{
    const int i = blockIdx.x * 256 + threadIdx.x;   // (l, c, k) x slot
    if (i >= rows * n1) return;
    const float2* e = Ex + (int64_t)i * BDG;
    float t = 0.f;
    for (int d = 0; d < BDG; d++) t += fabsf(e[d].x);
    rs[i] = t * 1.000002f;
}

// ---------------------------------------------------------------------------------------------
// Radial pass.  A warp copies the windows of four lanes (channels), 16 bytes a copy; row margins make
// every copy whole.  The thread's share of the bands (positions tid, tid + RT, ..) keeps its places in
// global and shared memory from stage to stage.  The sign of the apply and the rows that a kappa
// leaves unused (the coupling is zero there) are applied to the accumulators once the sums are in; the
// diagonal stages come last, so that the large diagonal part is not what the many small terms are
// added to.
// ---------------------------------------------------------------------------------------------
template <class P>
struct RadCfg {
    static constexpr int SB = RWP * P::RSL;            // slots per block
    static constexpr int ROWS = SB + 2 * HG;           // window rows
    static constexpr int UNIT = 16 / (int)sizeof(typename P::C);   // slots per 16-byte copy
    static constexpr int UNITS = ROWS / UNIT, EXTRA = UNITS - 32;  // copies per lane's window
    static constexpr int EPT = (SB * BDG + RT - 1) / RT;   // band positions formed per thread
    static constexpr size_t XB = (size_t)FLANE * P::XW * sizeof(typename P::C);   // one window buffer
    static constexpr size_t EB1 = (size_t)SB * P::EW * sizeof(typename P::E) + 16;   // one chunk's bands (+16: other banks)
    static constexpr size_t EB = 2 * EB1;
    static constexpr size_t OUT = (size_t)FLANE * (SB + 1) * (sizeof(typename P::C) == 8 ? 16 : 32);
    static constexpr size_t SMEM = 2 * XB + 2 * EB > OUT ? 2 * XB + 2 * EB : OUT;
    static_assert(ROWS % UNIT == 0 && P::XW * sizeof(typename P::C) % 16 == 0, "16-byte copies");
    static_assert(EXTRA >= 0 && EXTRA <= 16 && FLANE == 4 * RWP, "a warp copies four lanes' windows");
    static_assert(P::RSL % UNIT == 0, "aligned windows");
};

struct RadOut {          // what leaves the pass
    void* y;
    const void* bsub;
    const void* dv;
    double2* part_dot;
    double* part_nrm;
};

template <class P, bool OFF>
__global__ void __launch_bounds__(RT, 2)
    k_rad(OpView A, const RadPack* __restrict__ rp, int npack, int L, const typename P::R* __restrict__ E,
          const float* __restrict__ rs, const typename P::R* __restrict__ Sb, const typename P::R* __restrict__ Hb,
          double htau, int sign, const typename P::C* __restrict__ S, int NC, int NP,
          const typename P::C* __restrict__ dS, const typename P::C* __restrict__ dH, RadOut o, const KState* skip,
          const int* gate)
{
    typedef typename P::C C;
    typedef typename P::R R;
    typedef typename P::E EP;
    typedef typename P::RAcc Acc;
    typedef RadCfg<P> F;
    constexpr int SB = F::SB, RSL = P::RSL, XW = P::XW, EW = P::EW, EPT = F::EPT;
    if (skip && skip->done) return;   // uniform over the grid
    if (gate && !*gate) return;
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ int s_ch[FLANE];
    __shared__ float2 s_bd[2][2][SB];       // [buffer][chunk][slot]: the two rows' sums of |band| (OFF)
    const int pack = blockIdx.x % npack, tile = blockIdx.x / npack;
    const int n1 = A.n1, s0 = tile * SB, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const RadChunk c0 = rp[pack].c[0], c1 = rp[pack].c[1];
    const int n0 = c0.count, nl = n0 + c1.count, nchunk = c1.count ? 2 : 1;
    const int nss = L * NS, nst = nss + 4;   // stages: the sums, then S x0, S x1, H (i x0), H (i x1)
    if (tid < FLANE) {   // lanes beyond the pack repeat its first channel (their results are not stored)
        const int i = tid < nl ? tid : 0;
        s_ch[tid] = A.prec_order[i < n0 ? c0.first + i : c1.first + i - n0];
    }
    __syncthreads();
    auto xbuf = [&](int b) { return reinterpret_cast<C*>(rsm + b * F::XB); };
    auto ebuf = [&](int b, int ck) { return reinterpret_cast<EP*>(rsm + 2 * F::XB + b * F::EB + ck * F::EB1); };
    // this thread's copies of a sum's windows: four lanes' first 32 units, then its share of the rest.
    // The places move one row of S per stage and are kept in registers where there is room for them.
    constexpr int NX = (4 * F::EXTRA + 31) / 32;
    constexpr bool KEEP = !P::SPLIT;
    auto lane_of = [&](int c) { return w * 4 + (c < 4 ? c : (lane + 32 * (c - 4)) / F::EXTRA); };
    auto unit_of = [&](int c) { return c < 4 ? lane : 32 + (lane + 32 * (c - 4)) % F::EXTRA; };
    auto copies = [&](int c) { return c < 4 || lane + 32 * (c - 4) < 4 * F::EXTRA; };
    auto place_of = [&](int c) {
        return S + (int64_t)s_ch[copies(c) ? lane_of(c) : 0] * NC * NP + MARGIN + s0 - HG + unit_of(c) * F::UNIT;
    };
    const C* src[KEEP ? 4 + NX : 1];
    if constexpr (KEEP) {
#pragma unroll
        for (int c = 0; c < 4 + NX; c++) src[c] = place_of(c);
    }
    auto issue = [&](int st) {   // stages 0, 1, .. in turn
        C* xs = xbuf(st & 1);
#pragma unroll
        for (int c = 0; c < 4 + NX; c++) {
            const C* from = KEEP ? src[KEEP ? c : 0] : place_of(c) + (int64_t)st * NP;
            if (copies(c)) cp_async16(xs + lane_of(c) * XW + unit_of(c) * F::UNIT, from);
            if constexpr (KEEP) src[c] += NP;
        }
    };
    auto issue_diag = [&](int st) {   // the diagonal's vectors: after the sums in S, or apart
        const int t = (st - nss) & 1;
        const C* base = dS ? (st < nss + 2 ? dS : dH) : S;
        const int rows = dS ? 2 : NC, row = dS ? t : nss + t;
        C* xs = xbuf(st & 1);
        for (int i = tid; i < FLANE * F::UNITS; i += RT) {
            const int ln = i / F::UNITS, q = i % F::UNITS;
            cp_async16(xs + ln * XW + q * F::UNIT,
                       base + ((int64_t)s_ch[ln] * rows + row) * NP + MARGIN + s0 - HG + q * F::UNIT);
        }
    };
    const int ntot = min(SB, n1 - s0) * BDG;   // band positions of the block inside the grid
    R pre[EPT][3];
    float prs[3] = {0.f, 0.f, 0.f};
    const int eb13 = n1 * BDG;
    const R* Es = E + s0 * BDG + tid;
    auto fetch = [&](int st) {   // this thread's share of a sum's band values, stages in turn
#pragma unroll
        for (int q = 0; q < EPT; q++)
#pragma unroll
            for (int k = 0; k < 3; k++) pre[q][k] = tid + q * RT < ntot ? __ldg(Es + k * eb13 + q * RT) : P::rzero();
        Es += 3 * eb13;
        if constexpr (OFF) {
            if (tid < SB)
#pragma unroll
                for (int k = 0; k < 3; k++)
                    prs[k] = s0 + tid < n1 ? rs[((int64_t)st * 3 + k) * n1 + s0 + tid] : 0.f;
        }
    };
    int dst[EPT];
#pragma unroll
    for (int q = 0; q < EPT; q++) {
        const int i = tid + q * RT;
        dst[q] = P::place(i / BDG, i % BDG);
    }
    auto form = [&](int st) {   // the two row factors of every band position, per kappa
        const bool direct = st % NS < 3;
        for (int ck = 0; ck < nchunk; ck++) {
            const float kap = (float)(ck ? c1.kappa : c0.kappa);
            EP* e = ebuf(st & 1, ck);
#pragma unroll
            for (int q = 0; q < EPT; q++) {
                if (tid + q * RT >= SB * BDG) break;
                const R m = P::comb(direct ? pre[q][1] : pre[q][0], kap, pre[q][2]);
                e[dst[q]] = direct ? P::pair(pre[q][0], m) : P::pair(m, pre[q][1]);
            }
        }
        if constexpr (OFF) {
            if (tid < SB) {
                for (int ck = 0; ck < nchunk; ck++) {
                    const float ak = fabsf((float)(ck ? c1.kappa : c0.kappa));
                    s_bd[st & 1][ck][tid] = make_float2(direct ? prs[0] : fmaf(ak, prs[2], prs[0]),
                                                        direct ? fmaf(ak, prs[2], prs[1]) : prs[1]);
                }
            }
        }
    };
    auto form_diag = [&](int st) {   // straight from the kappa's bands
        const R* B = st < nss + 2 ? Sb : Hb;
        for (int ck = 0; ck < nchunk; ck++) {
            const R* b = B + ((int64_t)(ck ? c1.ks : c0.ks) * n1 + s0) * BDG * 4 + ((st - nss) & 1);
            EP* e = ebuf(st & 1, ck);
            for (int q = 0; q < EPT; q++) {
                const int i = tid + q * RT;
                if (i >= SB * BDG) break;
                R e0 = P::rzero(), e1 = P::rzero();
                if (i < ntot) {
                    e0 = b[i * 4];
                    e1 = b[i * 4 + 2];
                }
                if (st >= nss + 2) {
                    e0 = P::scale(htau, e0);
                    e1 = P::scale(htau, e1);
                }
                e[P::place(i / BDG, i % BDG)] = P::pair(e0, e1);
            }
        }
    };
    Acc acc[RSL];
#pragma unroll
    for (int s = 0; s < RSL; s++) P::rzero(acc[s]);
    const int ck = lane < n0 || lane >= nl ? 0 : 1;
    // stage st on the thread's slots; TURN: the diagonal stages, whose H part takes i x
    auto use = [&](int st, auto diag) {
        constexpr bool DIAG = decltype(diag)::value;
        const bool turn = DIAG && st >= nss + 2;
        const C* xr = xbuf(st & 1) + lane * XW + w * RSL;
        const EP* eb = ebuf(st & 1, ck) + w * RSL * EW;
        // window element j meets band position j - s of slot s
        if constexpr (sizeof(R) == 4) {
            // two window elements at a time: slot s takes its bands d, d + 1, d = j0 - s, in one 16-byte
            // read (odd slots are stored one element further, so that d is aligned)
#pragma unroll
            for (int j0 = 0; j0 < RSL + 2 * HG; j0 += 2) {
                const float4 v = *reinterpret_cast<const float4*>(xr + j0);
                C x0 = make_float2(v.x, v.y), x1 = make_float2(v.z, v.w);
                if (turn) {
                    x0 = P::rot(x0);
                    x1 = P::rot(x1);
                }
                const f2 re0 = pk(x0.x, x0.x), im0 = pk(x0.y, x0.y), re1 = pk(x1.x, x1.x), im1 = pk(x1.y, x1.y);
#pragma unroll
                for (int s = 0; s < RSL; s++) {
                    const int d = j0 - s;
                    if (d < -1 || d >= BDG) continue;
                    const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(eb + s * EW + (s & 1) + d);
                    if (d >= 0) {
                        acc[s].re = fma2(e.x, re0, acc[s].re);
                        acc[s].im = fma2(e.x, im0, acc[s].im);
                    }
                    if (d + 1 < BDG) {
                        acc[s].re = fma2(e.y, re1, acc[s].re);
                        acc[s].im = fma2(e.y, im1, acc[s].im);
                    }
                }
            }
        } else if constexpr (!P::SPLIT) {
#pragma unroll
            for (int j = 0; j < RSL + 2 * HG; j++) {
                C x = xr[j];
                if (turn) x = P::rot(x);
#pragma unroll
                for (int s = 0; s < RSL; s++) {
                    const int d = j - s;
                    if (d < 0 || d >= BDG) continue;
                    const EP e = eb[s * EW + d];
                    acc[s].r0 = fma(e.x, x.x, acc[s].r0);
                    acc[s].i0 = fma(e.x, x.y, acc[s].i0);
                    acc[s].r1 = fma(e.y, x.x, acc[s].r1);
                    acc[s].i1 = fma(e.y, x.y, acc[s].i1);
                }
            }
        } else {
            // double-float: the stage's sums in accumulators of their own, added at the end
            constexpr bool off = OFF && !DIAG;
            Acc t[RSL];
            f2 sg[RSL];
            float M = 0.f;
            if (off) {
#pragma unroll
                for (int j = 0; j < RSL + 2 * HG; j++) {
                    const float2 h = *reinterpret_cast<const float2*>(xr + j);   // the hi words
                    M = fmaxf(M, fmaxf(fabsf(h.x), fabsf(h.y)));
                }
            }
#pragma unroll
            for (int s = 0; s < RSL; s++) {
                P::rzero(t[s]);
                sg[s] = 0ull;
                if (off) {
                    const float2 b = s_bd[st & 1][ck][w * RSL + s];
                    sg[s] = pk(off_of(b.x * M), off_of(b.y * M));
                    t[s].re.s = t[s].im.s = sg[s];
                }
            }
            if constexpr (off) {
#pragma unroll
                for (int j = 0; j < RSL + 2 * HG; j++) {
                    const C x = xr[j];
                    const f2 rh = pk(x.x, x.x), rl = pk(x.z, x.z), ih = pk(x.y, x.y), il = pk(x.w, x.w);
#pragma unroll
                    for (int s = 0; s < RSL; s++) {
                        const int d = j - s;
                        if (d < 0 || d >= BDG) continue;
                        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(eb + s * EW + d);
                        d2_fma_off(t[s].re, e.x, e.y, rh, rl);
                        d2_fma_off(t[s].im, e.x, e.y, ih, il);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < RSL + 2 * HG; j++) {
                    C x = xr[j];
                    if (turn) x = P::rot(x);
                    const f2 rh = pk(x.x, x.x), rl = pk(x.z, x.z), ih = pk(x.y, x.y), il = pk(x.w, x.w);
#pragma unroll
                    for (int s = 0; s < RSL; s++) {
                        const int d = j - s;
                        if (d < 0 || d >= BDG) continue;
                        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(eb + s * EW + d);
                        d2_fma(t[s].re, e.x, e.y, rh, rl);
                        d2_fma(t[s].im, e.x, e.y, ih, il);
                    }
                }
            }
#pragma unroll
            for (int s = 0; s < RSL; s++) {
                if (off) {
                    t[s].re.s = sub2(t[s].re.s, sg[s]);   // exact
                    t[s].im.s = sub2(t[s].im.s, sg[s]);
                }
                d2_add(acc[s].re, t[s].re);
                d2_add(acc[s].im, t[s].im);
            }
        }
    };
    issue(0);
    fetch(0);
    form(0);
#pragma unroll 1
    for (int st = 0; st < nss; st++) {
        cp_async_wait_all();
        __syncthreads();   // stage st's windows and bands are in; stage st - 1 is no longer read
        if (st + 1 < nss) {
            issue(st + 1);
            fetch(st + 1);
        } else {
            issue_diag(st + 1);
        }
        use(st, std::false_type{});
        if (st + 1 < nss) form(st + 1);
        else form_diag(st + 1);
    }
    {   // the coupling is in: its sign, and zero at functions a kappa leaves unused
        const int kap = ck ? c1.kappa : c0.kappa;
#pragma unroll
        for (int s = 0; s < RSL; s++) {
            const bool edge = s0 + w * RSL + s == 0;
            P::times(acc[s], edge && kap != -1 ? 0.f : (float)sign, edge && kap != 1 ? 0.f : (float)sign);
        }
    }
#pragma unroll 1
    for (int st = nss; st < nst; st++) {
        cp_async_wait_all();
        __syncthreads();
        if (st + 1 < nst) issue_diag(st + 1);
        use(st, std::true_type{});
        if (st + 1 < nst) form_diag(st + 1);
    }
    __syncthreads();   // the staging space is free: it takes the outputs
    double2 dsum = make_double2(0, 0);
    double nsum = 0;
    if constexpr (sizeof(C) == 8) {
        float4* out = reinterpret_cast<float4*>(rsm);
        if (lane < nl)
#pragma unroll
            for (int s = 0; s < RSL; s++) out[lane * (SB + 1) + w * RSL + s] = P::rows(acc[s]);
        __syncthreads();
        for (int i = tid; i < nl * SB; i += RT) {
            const int ln = i / SB, j = i - ln * SB, r = s0 + j;
            if (r >= n1) continue;
            float4 v = out[ln * (SB + 1) + j];
            const int64_t q = (int64_t)s_ch[ln] * n1 + r;
            if (o.bsub) {
                const float4 b = static_cast<const float4*>(o.bsub)[q];
                v = make_float4(b.x - v.x, b.y - v.y, b.z - v.z, b.w - v.w);
            }
            static_cast<float4*>(o.y)[q] = v;
            if (o.dv) {
                const float4 d = static_cast<const float4*>(o.dv)[q];
                dsum.x += (double)d.x * v.x + (double)d.y * v.y + (double)d.z * v.z + (double)d.w * v.w;
                dsum.y += (double)d.x * v.y - (double)d.y * v.x + (double)d.z * v.w - (double)d.w * v.z;
            }
            if (o.part_nrm)
                nsum += (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z + (double)v.w * v.w;
        }
    } else {
        double2* out = reinterpret_cast<double2*>(rsm);   // [lane][slot][row]
        if (lane < nl)
#pragma unroll
            for (int s = 0; s < RSL; s++)
#pragma unroll
                for (int t = 0; t < 2; t++) out[(lane * (SB + 1) + w * RSL + s) * 2 + t] = P::row(acc[s], t);
        __syncthreads();
        for (int i = tid; i < nl * SB * 2; i += RT) {
            const int ln = i / (SB * 2), j = i - ln * SB * 2, r = s0 + (j >> 1);
            if (r >= n1) continue;
            double2 v = out[ln * (SB + 1) * 2 + j];
            const int64_t q = ((int64_t)s_ch[ln] * n1 + s0) * 2 + j;
            if (o.bsub) {
                const double2 b = static_cast<const double2*>(o.bsub)[q];
                v = make_double2(b.x - v.x, b.y - v.y);
            }
            static_cast<double2*>(o.y)[q] = v;
            if (o.dv) {
                const double2 d = static_cast<const double2*>(o.dv)[q];
                dsum.x += d.x * v.x + d.y * v.y;
                dsum.y += d.x * v.y - d.y * v.x;
            }
            if (o.part_nrm) nsum += v.x * v.x + v.y * v.y;
        }
    }
    if (o.part_dot || o.part_nrm) block_reduce_store(dsum, nsum, o.part_dot, o.part_nrm, blockIdx.x);
}

// ---- launchers ---------------------------------------------------------------------------------

// row stride of S and of the split vectors: margins, 16-byte rows of complex64
int ang_np(int n1) { return (n1 + 2 * MARGIN + 1) & ~1; }
// elements past the last row that the windows of the last tile may reach
int ang_tail() { return RadCfg<PF>::SB + 2 * HG; }
// u = psi + x, v = psi - x (or u = x alone) split into double-float words (re hi, im hi, re lo, im lo),
// type-major with zero margins, psi rounded to FP32 in the state's order, and the largest |u| word of each
// position.  The sums are FP64 additions, the words taken from their bit patterns.
__global__ void __launch_bounds__(256) k_split_rows(int n1, int NP, const double2* __restrict__ psi,
                                                    const double2* __restrict__ x, float4* __restrict__ u,
                                                    float4* __restrict__ v, float2* __restrict__ psi32,
                                                    float* __restrict__ umax)
{
    const int q = blockIdx.x * 256 + threadIdx.x, ch = blockIdx.y, r = q - MARGIN;
    if (q >= NP) return;
    const bool in = r >= 0 && r < n1;
    float m = 0.f;
#pragma unroll
    for (int t = 0; t < 2; t++) {
        const int64_t o = ((int64_t)ch * 2 + t) * NP + q, i = ((int64_t)ch * n1 + r) * 2 + t;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (in) {
            const double2 p = psi[i];
            if (v) {
                const double2 y = x[i];
                const float2 c = df_split_bits(p.x - y.x), d = df_split_bits(p.y - y.y);
                b = make_float4(c.x, d.x, c.y, d.y);
                const float2 e = df_split_bits(p.x + y.x), f = df_split_bits(p.y + y.y);
                a = make_float4(e.x, f.x, e.y, f.y);
                // rounded to nearest: the truncated hi words alone would lower ||b|| by a part of their error
                const float2 pr = df_split_bits(p.x), pi = df_split_bits(p.y);
                psi32[i] = make_float2(pr.x + pr.y, pi.x + pi.y);
            } else {
                const float2 e = df_split_bits(p.x), f = df_split_bits(p.y);
                a = make_float4(e.x, f.x, e.y, f.y);
            }
        }
        u[o] = a;
        if (v) v[o] = b;
        m = fmaxf(m, fmaxf(fabsf(a.x), fabsf(a.y)));
    }
    umax[(int64_t)ch * NP + q] = m;
}

void launch_split_rows(cudaStream_t st, int nch, int n1, const double2* psi, const double2* x, float4* u, float4* v,
                       float2* psi32, float* umax)
{
    const int NP = ang_np(n1);
    k_split_rows<<<dim3((NP + 255) / 256, nch), 256, 0, st>>>(n1, NP, psi, x, u, v, psi32, umax);
}

int rad_parts(int prec, int n1, int npack)
{
    const int sb = prec == 1 ? RadCfg<PF>::SB : RadCfg<PD>::SB;
    return ((n1 + sb - 1) / sb) * npack;
}

template <class K>
static cudaError_t shared_limit(K* kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t ang_prepare()
{
    cudaError_t e[] = {shared_limit(k_rad<PF, false>, RadCfg<PF>::SMEM), shared_limit(k_rad<PD, false>, RadCfg<PD>::SMEM),
                       shared_limit(k_rad<PX, false>, RadCfg<PX>::SMEM), shared_limit(k_rad<PX, true>, RadCfg<PX>::SMEM)};
    for (cudaError_t x : e)
        if (x != cudaSuccess) return x;
    return cudaSuccess;
}

void launch_rad_entries(cudaStream_t st, const PulseView& P, int n1, const double* s, float* Ef, float2* Ex, double* Ed,
                        float* rs)
{
    k_rad_entries<<<dim3((n1 * BDG + 255) / 256, P.L * NS), 256, 0, st>>>(P, n1, s, Ef, Ex, Ed);
    if (rs) {
        const int rows = P.L * NS * 3;
        k_rad_rowsums<<<(rows * n1 + 255) / 256, 256, 0, st>>>(n1, rows, Ex, rs);
    }
}

template <class P, bool OFF>
static void ang_pass(cudaStream_t st, int n1, const AngList& G, const void* coef, const void* x, const float* xmax, void* S,
                     int NC, const KState* skip, const int* gate)
{
    const int NP = ang_np(n1);
    k_ang<P, OFF><<<dim3((NP + AT - 1) / AT, G.nlist), AT, 0, st>>>(
        n1, G, (const typename P::K*)coef, (const typename P::C*)x, xmax, (typename P::C*)S, NC, NP, skip, gate);
}

void launch_ang32(cudaStream_t st, const OpView& A, const AngList& G, const float* coef, const RadPack* rp, int npack,
                  const float* E, const float* Sb, const float* Hb, int sign, const void* x, void* S, void* y,
                  const void* bsub, const void* dv, double2* pdot, double* pnrm, const KState* skip, const int* gate)
{
    const int NC = G.L * NS + 2, NP = ang_np(A.n1);
    ang_pass<PF, false>(st, A.n1, G, coef, x, nullptr, S, NC, skip, gate);
    RadOut o = {y, bsub, dv, pdot, pnrm};
    k_rad<PF, false><<<rad_parts(1, A.n1, npack), RT, RadCfg<PF>::SMEM, st>>>(
        A, rp, npack, G.L, E, nullptr, Sb, Hb, sign * A.tau, sign, (const float2*)S, NC, NP, nullptr, nullptr, o, skip,
        gate);
}

void launch_ang64(cudaStream_t st, const OpView& A, const AngList& G, const double* coef, const RadPack* rp, int npack,
                  const double* E, const double* Sb, const double* Hb, int sign, const void* x, void* S, void* y,
                  const void* bsub, const void* dv, double2* pdot, double* pnrm, const KState* skip)
{
    const int NC = G.L * NS + 2, NP = ang_np(A.n1);
    ang_pass<PD, false>(st, A.n1, G, coef, x, nullptr, S, NC, skip, nullptr);
    RadOut o = {y, bsub, dv, pdot, pnrm};
    k_rad<PD, false><<<rad_parts(0, A.n1, npack), RT, RadCfg<PD>::SMEM, st>>>(
        A, rp, npack, G.L, E, nullptr, Sb, Hb, sign * A.tau, sign, (const double2*)S, NC, NP, nullptr, nullptr, o, skip,
        nullptr);
}

void launch_ang_df(cudaStream_t st, const OpView& A, const AngList& G, bool offsets, const float4* coef,
                   const RadPack* rp, int npack, const float2* E, const float* rs, const float2* Sb, const float2* Ht,
                   int sign, const float4* u, const float* umax, const float4* v, void* S, double2* y, double* pnrm)
{
    const int NC = G.L * NS, NP = ang_np(A.n1);
    const int gr = rad_parts(2, A.n1, npack);
    RadOut o = {y, nullptr, nullptr, nullptr, pnrm};
    if (offsets) {
        ang_pass<PX, true>(st, A.n1, G, coef, u, umax, S, NC, nullptr, nullptr);
        k_rad<PX, true><<<gr, RT, RadCfg<PX>::SMEM, st>>>(A, rp, npack, G.L, E, rs, Sb, Ht, (double)sign, sign,
                                                        (const float4*)S, NC, NP, v, u, o, nullptr, nullptr);
    } else {
        ang_pass<PX, false>(st, A.n1, G, coef, u, umax, S, NC, nullptr, nullptr);
        k_rad<PX, false><<<gr, RT, RadCfg<PX>::SMEM, st>>>(A, rp, npack, G.L, E, rs, Sb, Ht, (double)sign, sign,
                                                         (const float4*)S, NC, NP, v, u, o, nullptr, nullptr);
    }
}

}  // namespace dg
