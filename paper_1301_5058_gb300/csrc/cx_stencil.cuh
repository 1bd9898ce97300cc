// cx_stencil.cuh -- the per-thread stencil machinery shared by the
// single-grid and batched step kernels: vector loads, the face fluxes of the
// scaled scheme, per-step noise, and the row march (see cx_step.cu).
#pragma once

#include <type_traits>

#include "cx_internal.h"
#include "cx_philox.cuh"

namespace cx {
namespace stencil {


constexpr int kThreads = 128;  // 4 warps side by side along x
// Threads of a block of the one-stage march: one warp in FP64.  Its warps share
// nothing; a warp's FP64 instruction holds its scheduler's FP64 unit for 64
// cycles, so what counts is that every scheduler gets the same number of warp
// rows, and blocks of 128 columns cut a grid finer than blocks of 512 (with the
// faces evaluated once and the heights chosen for it, 256^2 18.7 -> 10.4 us per
// step, 1024^2 113.4 -> 92.7, 4096^2 1477 -> 1304).
template <typename T> constexpr int step_threads() { return sizeof(T) == 4 ? kThreads : 32; }
constexpr int kCells = 4;      // cells per thread along x
constexpr unsigned kFull = 0xffffffffu;

template <typename T> struct Vec;
template <> struct Vec<float> {
    // A coherent load: the kernel may have been launched before the array was
    // written (launch_pass).  volatile keeps it behind pass_wait(); that it
    // clobbers no memory lets the march issue a row's loads ahead of the stores
    // of the row before, to other arrays (as plain loads, held behind the
    // stores, 2048^2 took 10.3 instead of 9.9 us per step).
    static __device__ __forceinline__ void load(const float *p, float (&v)[4])
    {
        asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                     : "l"(p));
    }
    static __device__ __forceinline__ float load1(const float *p)
    {
        float v;
        asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
        return v;
    }
    // L2 path (bypasses L1): for a persistent launch, where the arrays a
    // block reads were written by other blocks earlier in the same launch
    static __device__ __forceinline__ void load_cg(const float *p, float (&v)[4])
    {
        const float4 q = __ldcg(reinterpret_cast<const float4 *>(p));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
    static __device__ __forceinline__ void store(float *p, const float (&v)[4])
    {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct Vec<double> {
    static __device__ __forceinline__ void load(const double *p, double (&v)[4])
    {
        asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "l"(p));
        asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v[2]), "=d"(v[3]) : "l"(p + 2));
    }
    static __device__ __forceinline__ double load1(const double *p)
    {
        double v;
        asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ void load_cg(const double *p, double (&v)[4])
    {
        const double2 q0 = __ldcg(reinterpret_cast<const double2 *>(p));
        const double2 q1 = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
        v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    }
    static __device__ __forceinline__ void store(double *p, const double (&v)[4])
    {
        reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
    }
};

// ---------------------------------------------------------------------------
// Arithmetic with every rounding explicit, on one cell (float, double) or on
// a pair of cells (float2, double2).  The FP32 pair forms are Blackwell's
// paired FP32 instructions (one issue slot for two cells); each component
// rounds exactly as the scalar form, so a pair and two scalars give the same
// bits.  No operation is contracted by the compiler, so a face value or an
// update is the same bits in every kernel that evaluates it.

template <typename T> struct PairOf;
template <> struct PairOf<float> { using type = float2; };
template <> struct PairOf<double> { using type = double2; };
template <typename T> using P2 = typename PairOf<T>::type;

__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 add_rn(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 add_rn(double2 a, double2 b)
{
    return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float2 mul_rn(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 mul_rn(double2 a, double2 b)
{
    return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y));
}
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 fma_rn(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma_rn(double2 a, double2 b, double2 c)
{
    return make_double2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
}
// a - b; the pair form is fma(b, -1, a), which rounds the exact difference
// once, as the scalar subtraction does (m1 holds -1)
__device__ __forceinline__ float sub_rn(float a, float b, float) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b, double) { return __dsub_rn(a, b); }
__device__ __forceinline__ float2 sub_rn(float2 a, float2 b, float2 m1) { return __ffma2_rn(b, m1, a); }
__device__ __forceinline__ double2 sub_rn(double2 a, double2 b, double2)
{
    return make_double2(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y));
}
// 1 / q for the receptor-law weight.  FP32: the hardware's approximate
// reciprocal (the FP32 path is judged by tolerance).  rcp.approx.ftz, not
// __fdividef: the range handling around __fdividef (scalings of numerator and
// denominator, predicated off for every q that occurs but issued all the same)
// was a quarter of the march's instructions.  16384^2 two-stage pass
// 0.919 -> 0.847 ms, which is 0.94 of the measured HBM bandwidth and no longer
// bound by instruction issue; paper's scheme 1.226 -> 1.133 ms; 2048^2
// 12.3 -> 11.3 and 45.6 -> 39.4 us per step.
// FP64: the hardware's approximate FP64 reciprocal x (rcp.approx.ftz.f64; q is
// never subnormal) and one third-order correction: with e = 1 - q x,
// 1 / q = x / (1 - e) = x (1 + e + e^2 + ...), so x + x (e + e^2) is off by
// e^3, far below FP64 rounding for any seed within 2^-19.  Three operations on
// GB300's narrow FP64 pipe where two Newton steps took four.
__device__ __forceinline__ float rcp_w(float q)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(q));
    return r;
}
__device__ __forceinline__ double rcp_w(double q)
{
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(q));
    const double e = __fma_rn(-q, x, 1.0);
    return __fma_rn(x, __fma_rn(e, e, e), x);
}
__device__ __forceinline__ float2 rcp_w(float2 q) { return make_float2(rcp_w(q.x), rcp_w(q.y)); }
__device__ __forceinline__ double2 rcp_w(double2 q) { return make_double2(rcp_w(q.x), rcp_w(q.y)); }
// donor-cell b: the side with the lower n (dm = nL - nR)
__device__ __forceinline__ float donor(float dm, float bL, float bR) { return dm <= 0.f ? bL : bR; }
__device__ __forceinline__ double donor(double dm, double bL, double bR) { return dm <= 0.0 ? bL : bR; }
__device__ __forceinline__ float2 donor(float2 dm, float2 bL, float2 bR)
{
    return make_float2(donor(dm.x, bL.x, bR.x), donor(dm.y, bL.y, bR.y));
}
__device__ __forceinline__ double2 donor(double2 dm, double2 bL, double2 bR)
{
    return make_double2(donor(dm.x, bL.x, bR.x), donor(dm.y, bL.y, bR.y));
}
__host__ __device__ __forceinline__ float2 pair(float x, float y) { return make_float2(x, y); }
__host__ __device__ __forceinline__ double2 pair(double x, double y) { return make_double2(x, y); }

// The scaled flux coefficients (dt folded in) as stored per grid.
template <typename T> struct CoefT {
    T cA, cChi, cG, cR, cN;
};
template <typename T> CoefT<T> coef_t(const Coef &k)
{
    return CoefT<T>{(T)k.cA, (T)k.cChi, (T)k.cG, (T)k.cR, (T)k.cN};
}

// The coefficients and constants of the face and update arithmetic, for
// one cell (V = T) or a pair (V = P2<T>): signs are folded in so that every
// subtraction of a product is one multiply-add.
template <typename V> struct KV {
    V cA;     // scale of the bacterial flux divergence
    V chi;    // constant law: hc; receptor law: FP32 its numerator, FP64 the scale of q
    V two;    // receptor law: FP32 2, FP64 twice chi
    V ncG;    // -scale of the nutrient flux divergence
    V cR;     // growth
    V ncN;    // -consumption
    V m1, half;
};
template <typename T> __host__ __device__ __forceinline__ KV<P2<T>> make_kv(const CoefT<T> &k)
{
    KV<P2<T>> v;
    v.cA = pair(k.cA, k.cA);
    v.chi = pair(k.cChi, k.cChi);
    v.two = sizeof(T) == 4 ? pair(T(2), T(2)) : pair(T(2) * k.cChi, T(2) * k.cChi);
    v.ncG = pair(-k.cG, -k.cG);
    v.cR = pair(k.cR, k.cR);
    v.ncN = pair(-k.cN, -k.cN);
    v.m1 = pair(T(-1), T(-1));
    v.half = pair(T(0.5), T(0.5));
    return v;
}
template <typename T> __device__ __forceinline__ KV<T> scalar_kv(const KV<P2<T>> &k)
{
    return KV<T>{k.cA.x, k.chi.x, k.two.x, k.ncG.x, k.cR.x, k.ncN.x, k.m1.x, k.half.x};
}

// The receptor law's weight at a face (see face()).
template <typename V> __device__ __forceinline__ V weight(V n2, const KV<V> &k)
{
    if constexpr (std::is_same<V, float>::value || std::is_same<V, float2>::value) {
        const V q = add_rn(n2, k.two);
        return mul_rn(k.chi, rcp_w(mul_rn(q, q)));
    } else {
        const V q = fma_rn(n2, k.chi, k.two);
        return rcp_w(mul_rn(q, q));
    }
}

// Unscaled fluxes (phi, g) through the face between L (left/lower) and R,
// for one face or a pair of faces:
//   phi = s2 n2 b2 (db + hc b2 dm)      (central b^2 mobility)
//   phi = s2 n2 (b2 db + hc bd^2 dm)    (donor-cell b^2)
//   g   = dm
// with s2 = sL + sR (likewise n2, b2), db = bR - bL, dm = nL - nR and, under
// the constant law, hc = chi.  The receptor law's weight is in FP32
// hc = chi / (2 + n2)^2.  In FP64 its strength is folded into the scale of the
// denominator, hc = 1 / q^2 with q = chi n2 + 2 chi, so that no face multiplies
// by it: the FP64 kernels are bound by the FP64 pipe and take 15 operations per
// face instead of 17 (with rcp_w), 4096^2 1630 -> 1476 us per step, 1024^2
// 125.6 -> 113.4.  In FP32 the second constant of that multiply-add costs the
// marches a register pair that they do not have (16384^2 422 -> 428 us per
// step, the paper's scheme 1118 -> 1171).  The constant factors cA and cG are
// applied once per cell, to the divergence (cell_update), not once per face.
// face_s2 takes s2 itself, for a caller that keeps it from stage to stage.
template <int LAW, int MOB, typename V>
__device__ __forceinline__ void face_s2(V s2, V nL, V nR, V bL, V bR, const KV<V> &k, V &phi, V &g)
{
    const V n2 = add_rn(nL, nR), b2 = add_rn(bL, bR);
    const V db = sub_rn(bR, bL, k.m1), dm = sub_rn(nL, nR, k.m1);
    V hc = k.chi;
    if (LAW == CX_CHEMO_RECEPTOR) hc = weight(n2, k);
    const V a = mul_rn(s2, n2);
    if (MOB == CX_MOBILITY_CENTRAL) {
        phi = mul_rn(mul_rn(a, b2), fma_rn(mul_rn(hc, b2), dm, db));
    } else {
        const V bd = donor(dm, bL, bR);
        phi = mul_rn(a, fma_rn(mul_rn(mul_rn(hc, bd), bd), dm, mul_rn(b2, db)));
    }
    g = dm;
}
template <int LAW, int MOB, typename V>
__device__ __forceinline__ void face(V sL, V sR, V nL, V nR, V bL, V bR, const KV<V> &k, V &phi,
                                     V &g)
{
    face_s2<LAW, MOB>(add_rn(sL, sR), nL, nR, bL, bR, k, phi, g);
}

// Four adjacent cells x0..x0+3 of one field, held as the pairs
// E = (x0, x0+2) and O = (x0+1, x0+3), so that the x-faces pair up too.
template <typename T> struct Cells {
    P2<T> E, O;
};
// A vector as loaded from (or stored to) a device array in pair order
// (cx_internal.h): (x0, x0+2, x0+1, x0+3), i.e. E then O.
template <typename T> __device__ __forceinline__ Cells<T> split4(const T (&v)[4])
{
    return Cells<T>{pair(v[0], v[1]), pair(v[2], v[3])};
}
template <typename T> __device__ __forceinline__ void join4(const Cells<T> &c, T (&v)[4])
{
    v[0] = c.E.x; v[1] = c.E.y; v[2] = c.O.x; v[3] = c.O.y;
}
// Four values in natural cell order x0 .. x0+3 (values made in registers,
// such as per-step sigma, and the element-wise edge stores).
template <typename T> __device__ __forceinline__ Cells<T> split4_nat(const T (&v)[4])
{
    return Cells<T>{pair(v[0], v[2]), pair(v[1], v[3])};
}
template <typename T> __device__ __forceinline__ void join4_nat(const Cells<T> &c, T (&v)[4])
{
    v[0] = c.E.x; v[1] = c.O.x; v[2] = c.E.y; v[3] = c.O.y;
}
template <typename T> __device__ __forceinline__ Cells<T> zero_cells()
{
    return Cells<T>{pair(T(0), T(0)), pair(T(0), T(0))};
}

// y-faces of four cells (between a row and the next one), as E / O pairs.
template <typename T> struct YFaces {
    P2<T> phE, phO, gE, gO;
};
template <typename T> __device__ __forceinline__ YFaces<T> zero_yfaces()
{
    const P2<T> z = pair(T(0), T(0));
    return YFaces<T>{z, z, z, z};
}
template <typename T, int LAW, int MOB>
__device__ __forceinline__ YFaces<T> row_yfaces(const Cells<T> &sL, const Cells<T> &nL,
                                                const Cells<T> &bL, const Cells<T> &sU,
                                                const Cells<T> &nU, const Cells<T> &bU,
                                                const KV<P2<T>> &k)
{
    YFaces<T> y;
    face<LAW, MOB>(sL.E, sU.E, nL.E, nU.E, bL.E, bU.E, k, y.phE, y.gE);
    face<LAW, MOB>(sL.O, sU.O, nL.O, nU.O, bL.O, bU.O, k, y.phO, y.gO);
    return y;
}

// The same with the face sums of sigma given.
template <typename T, int LAW, int MOB>
__device__ __forceinline__ YFaces<T> row_yfaces_s2(const Cells<T> &s2, const Cells<T> &nL,
                                                   const Cells<T> &bL, const Cells<T> &nU,
                                                   const Cells<T> &bU, const KV<P2<T>> &k)
{
    YFaces<T> y;
    face_s2<LAW, MOB>(s2.E, nL.E, nU.E, bL.E, bU.E, k, y.phE, y.gE);
    face_s2<LAW, MOB>(s2.O, nL.O, nU.O, bL.O, bU.O, k, y.phO, y.gO);
    return y;
}
template <typename T>
__device__ __forceinline__ Cells<T> y_sums(const Cells<T> &sL, const Cells<T> &sU)
{
    return Cells<T>{add_rn(sL.E, sU.E), add_rn(sL.O, sU.O)};
}

// x-faces of four cells: f_c lies between cells x0+c-1 and x0+c.  They are
// computed as A = (f0, f2), B = (f1, f3) and f4; (l*, r*) are the cells
// x0-1 and x0+4.  Faces on the walls (and past the row's end) carry zero
// flux unless INTERIOR (no wall within reach).
template <typename T> struct XFaces {
    P2<T> phA, gA, phB, gB;
    T ph4, g4;
};
template <typename T, int LAW, int MOB, bool INTERIOR>
__device__ __forceinline__ XFaces<T> row_xfaces(const Cells<T> &s, const Cells<T> &n,
                                                const Cells<T> &b, T ls, T ln, T lb, T rs, T rn,
                                                T rb, const KV<P2<T>> &k, int x0, int nx)
{
    XFaces<T> f;
    face<LAW, MOB>(pair(ls, s.O.x), s.E, pair(ln, n.O.x), n.E, pair(lb, b.O.x), b.E, k, f.phA, f.gA);
    face<LAW, MOB>(s.E, s.O, n.E, n.O, b.E, b.O, k, f.phB, f.gB);
    face<LAW, MOB>(s.O.y, rs, n.O.y, rn, b.O.y, rb, scalar_kv<T>(k), f.ph4, f.g4);
    if (!INTERIOR) {
        if (x0 == 0) f.phA.x = f.gA.x = T(0);           // west wall
        if (x0 + 1 >= nx) f.phB.x = f.gB.x = T(0);      // east wall and padding
        if (x0 + 2 >= nx) f.phA.y = f.gA.y = T(0);
        if (x0 + 3 >= nx) f.phB.y = f.gB.y = T(0);
        if (x0 + 4 >= nx) f.ph4 = f.g4 = T(0);
    }
    return f;
}

// The same x-faces when the lanes hold the row's cells four by four (the
// two-stage march, the register tiles): f4 is the right lane's f0, so each
// face is evaluated once and no right-hand neighbour is needed.  A row lies in
// WIDTH consecutive lanes; the last of them takes its own f0 for f4, and the
// caller discards what depends on it.  s2: the face sums of sigma, (f0, f2)
// and (f1, f3).
template <typename T, int LAW, int MOB, bool INTERIOR, int WIDTH>
__device__ __forceinline__ XFaces<T> row_xfaces_s2(const Cells<T> &s2, const Cells<T> &n,
                                                   const Cells<T> &b, T ln, T lb,
                                                   const KV<P2<T>> &k, int x0, int nx)
{
    XFaces<T> f;
    face_s2<LAW, MOB>(s2.E, pair(ln, n.O.x), n.E, pair(lb, b.O.x), b.E, k, f.phA, f.gA);
    face_s2<LAW, MOB>(s2.O, n.E, n.O, b.E, b.O, k, f.phB, f.gB);
    f.ph4 = __shfl_down_sync(kFull, f.phA.x, 1, WIDTH);
    f.g4 = __shfl_down_sync(kFull, f.gA.x, 1, WIDTH);
    if (!INTERIOR) {
        if (x0 == 0) f.phA.x = f.gA.x = T(0);           // west wall
        if (x0 + 1 >= nx) f.phB.x = f.gB.x = T(0);      // east wall and padding
        if (x0 + 2 >= nx) f.phA.y = f.gA.y = T(0);
        if (x0 + 3 >= nx) f.phB.y = f.gB.y = T(0);
        if (x0 + 4 >= nx) f.ph4 = f.g4 = T(0);
    }
    return f;
}
template <typename T> __device__ __forceinline__ Cells<T> x_sums(const Cells<T> &s, T ls)
{
    return Cells<T>{add_rn(pair(ls, s.O.x), s.E), add_rn(s.E, s.O)};
}
template <typename T, int LAW, int MOB, bool INTERIOR, int WIDTH = 32>
__device__ __forceinline__ XFaces<T> row_xfaces_shfl(const Cells<T> &s, const Cells<T> &n,
                                                     const Cells<T> &b, T ls, T ln, T lb,
                                                     const KV<P2<T>> &k, int x0, int nx)
{
    return row_xfaces_s2<T, LAW, MOB, INTERIOR, WIDTH>(x_sums(s, ls), n, b, ln, lb, k, x0, nx);
}

// u + reaction + div for one pair of cells: faces west/east and, in march
// order, behind/ahead (DIR +1: ahead is north):
//   b' = b + cR n b + cA div(phi),   n' = n - cN n b - cG div(g).
template <typename T, int DIR>
__device__ __forceinline__ void cell_update(P2<T> b, P2<T> n, P2<T> phW, P2<T> gW, P2<T> phE,
                                            P2<T> gE, P2<T> phB, P2<T> gB, P2<T> phA, P2<T> gA,
                                            const KV<P2<T>> &k, P2<T> &ob, P2<T> &on)
{
    const P2<T> phN = DIR > 0 ? phA : phB, phS = DIR > 0 ? phB : phA;
    const P2<T> gN = DIR > 0 ? gA : gB, gS = DIR > 0 ? gB : gA;
    const P2<T> r = mul_rn(n, b);
    const P2<T> divb = add_rn(sub_rn(phE, phW, k.m1), sub_rn(phN, phS, k.m1));
    const P2<T> divn = add_rn(sub_rn(gE, gW, k.m1), sub_rn(gN, gS, k.m1));
    ob = fma_rn(k.cA, divb, fma_rn(k.cR, r, b));
    on = fma_rn(k.ncG, divn, fma_rn(k.ncN, r, n));
}
// the four cells: even cells lie between A (west) and B (east), odd cells
// between B and (f2, f4)
template <typename T, int DIR>
__device__ __forceinline__ void row_update(const Cells<T> &b, const Cells<T> &n,
                                           const XFaces<T> &x, const YFaces<T> &yB,
                                           const YFaces<T> &yA, const KV<P2<T>> &k, Cells<T> &ob,
                                           Cells<T> &on)
{
    cell_update<T, DIR>(b.E, n.E, x.phA, x.gA, x.phB, x.gB, yB.phE, yB.gE, yA.phE, yA.gE, k, ob.E,
                        on.E);
    cell_update<T, DIR>(b.O, n.O, x.phB, x.gB, pair(x.phA.y, x.ph4), pair(x.gA.y, x.g4), yB.phO,
                        yB.gO, yA.phO, yA.gO, k, ob.O, on.O);
}
// Heun's second stage: (u0 + u) / 2
template <typename T>
__device__ __forceinline__ Cells<T> heun_mean(const Cells<T> &u0, const Cells<T> &u,
                                              const KV<P2<T>> &k)
{
    return Cells<T>{mul_rn(k.half, add_rn(u0.E, u.E)), mul_rn(k.half, add_rn(u0.O, u.O))};
}

// Per-step noise: the sigma recipe of the state's precision.
template <typename T> struct NoiseT;
template <> struct NoiseT<float> {
    uint64_t seed, step;
    int dist;
    float sigma0, amp;
    uint32_t kx[10], ky[10];  // the key schedule of seed (set_keys)
    __host__ __device__ void set_keys()
    {
        uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
        for (int r = 0; r < 10; ++r) {
            kx[r] = a;
            ky[r] = b;
            a += 0x9E3779B9u;
            b += 0xBB67AE85u;
        }
    }
    __device__ __forceinline__ uint4 block(uint64_t q) const
    {
        return philox4x32_10_ks(
            make_uint4((uint32_t)q, (uint32_t)(q >> 32), (uint32_t)step, (uint32_t)(step >> 32)), kx,
            ky);
    }
    __device__ __forceinline__ float at(long long idx) const
    {
        const uint4 w = block((uint64_t)idx >> 2);
        return sigma_from_word(block_word(w, (int)(idx & 3)), dist, sigma0, amp);
    }
    // cells idx0 .. idx0+3: one Philox block when idx0 is a multiple of 4
    // (always, in rows whose width is), two otherwise (the offset is the same
    // for all threads of a row)
    __device__ __forceinline__ void four(long long idx0, float (&s)[4]) const
    {
        const uint64_t q = (uint64_t)idx0 >> 2;
        const int h = (int)(idx0 & 3);
        const uint4 w0 = block(q);
        if (h == 0) {
            s[0] = sigma_from_word(w0.x, dist, sigma0, amp);
            s[1] = sigma_from_word(w0.y, dist, sigma0, amp);
            s[2] = sigma_from_word(w0.z, dist, sigma0, amp);
            s[3] = sigma_from_word(w0.w, dist, sigma0, amp);
        } else {
            const uint4 w1 = block(q + 1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int k = h + c;
                s[c] = sigma_from_word(k < 4 ? block_word(w0, k) : block_word(w1, k - 4), dist,
                                       sigma0, amp);
            }
        }
    }
};
template <> struct NoiseT<double> {
    uint64_t seed, step;
    int dist;
    double sigma0, amp;
    __device__ __forceinline__ double at(long long idx) const
    {
        return sigma_f64(seed, (uint64_t)idx, step, dist, sigma0, amp);
    }
    __device__ __forceinline__ void four(long long idx0, double (&s)[4]) const
    {
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] = at(idx0 + c);
    }
};

// Before a launch: the FP32 recipe's Philox key schedule from the seed (the
// FP64 recipe derives its keys as it goes).
inline void set_noise_keys(NoiseT<float> &nz) { nz.set_keys(); }
inline void set_noise_keys(NoiseT<double> &) {}

template <typename T> struct Ptrs {
    const T *__restrict__ b;
    const T *__restrict__ n;
    const T *__restrict__ s;
    const T *bu;  // may alias bo (in-place Heun combine)
    const T *nu;
    T *bo;
    T *no;
};

// Both marches ask L2, once per iteration, for the state row kPrefetchRows
// ahead of the one they load.  A loaded row feeds the iteration's whole
// dependence chain, so without the hint each iteration waits a full DRAM
// latency; with it the load finds the row in L2.  On the 16384^2 FP32
// workload, 1 to 3 rows ahead all gain about 18 % for the two-stage march
// (6 rows ahead gains less) and 5 % for the one-stage march.  Only rows the
// tile itself loads are asked for (a row past the tile's end would be read
// by the neighbouring tile, usually long after), at the thread's in-row
// vector offset `off` (row * pitch + in-row column).
constexpr int kPrefetchRows = 2;
template <typename T, int NOISE>
__device__ __forceinline__ void prefetch_row(const Ptrs<T> &P, long long off)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(P.b + off));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(P.n + off));
    if (NOISE == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(P.s + off));
}

template <typename T> struct Row {
    Cells<T> b, n, s;
    T hb, hn, hs;     // lane 0: cell x0-1; lane 31: cell x0+4 (FP32)
    Cells<T> ub, un;  // STAGE 1: the state at the start of the step
};

// One thread's march over rows j0..jend-1 in direction DIR (+1: increasing j,
// -1: decreasing j).  The y-faces shared with the row processed before
// ("behind") are carried in registers; the y-faces with the next row in
// march order ("ahead") are computed from the row loaded in this iteration.
// Face values do not depend on DIR (a face is always evaluated with L the
// lower row), so both directions give bit-identical results.  CG: read
// through L2 only (a persistent launch whose blocks read what other blocks
// wrote earlier in the same launch).  A lane's fifth x-face is the right
// lane's first.  In FP32 every lane evaluates it again (the pass is bound by
// HBM).  In FP64 it comes by shuffle, and the warp's last lane takes it from
// faces that the warp evaluates once per 32 rows, each lane one row's: the
// FP64 pipe, which bounds the pass, spends as much on an instruction with one
// active lane as with 32.  INTERIOR: the caller guarantees that
// every thread's cells and both x-neighbours of the warp lie inside the grid
// (0 < x0 and x0 + 4 < nx for all threads), so the x-wall tests drop out.
template <typename T, int LAW, int MOB, int NOISE, int STAGE, int DIR, bool CG = false,
          bool INTERIOR = false>
__device__ __forceinline__ void march(const Ptrs<T> &P, int nx, int ny, long long pitch,
                                      const KV<P2<T>> &k, const NoiseT<T> &nz, int x0, int j0,
                                      int jend)
{
    const int lane = threadIdx.x & 31;
    // threads past the right edge keep running (they take part in the
    // shuffles) but load an in-row vector and store nothing
    const long long xv = INTERIOR ? (long long)x0 : min((long long)x0, pitch - kCells);
    const bool halo_l = (lane == 0) && (INTERIOR || ((x0 > 0) && (x0 < nx)));
    constexpr bool kRightOnce = sizeof(T) == 8;
    const bool halo_r = !kRightOnce && (lane == 31) && (INTERIOR || (x0 + kCells < nx));
    const bool halo = halo_l || halo_r;
    const long long xh = halo_l ? (long long)x0 - 1 : (long long)x0 + kCells;

    auto vload = [](const T *p) -> Cells<T> {
        T v[kCells];
        if (CG) Vec<T>::load_cg(p, v);
        else Vec<T>::load(p, v);
        return split4(v);
    };
    auto sload = [](const T *p) -> T { return CG ? __ldcg(p) : Vec<T>::load1(p); };
    auto load_row = [&](int r, Row<T> &R, bool own) {
        const long long off = (long long)r * pitch;
        R.b = vload(P.b + off + xv);
        R.n = vload(P.n + off + xv);
        if (NOISE == 0) {
            R.s = vload(P.s + off + xv);
        } else {
            T v[kCells];
            nz.four((long long)r * nx + x0, v);
            if (!INTERIOR) {
#pragma unroll
                for (int c = 0; c < kCells; ++c)
                    if (x0 + c >= nx) v[c] = T(0);  // past the row's end
            }
            R.s = split4_nat(v);
        }
        R.hb = R.hn = R.hs = T(0);
        if (halo) {
            R.hb = sload(P.b + off + xh);
            R.hn = sload(P.n + off + xh);
            R.hs = NOISE == 0 ? sload(P.s + off + xh) : nz.at((long long)r * nx + xh);
        }
        if (STAGE == 1 && own) {
            T v[kCells];
            if (CG) Vec<T>::load_cg(P.bu + off + xv, v);
            else Vec<T>::load(P.bu + off + xv, v);
            R.ub = split4(v);
            if (CG) Vec<T>::load_cg(P.nu + off + xv, v);
            else Vec<T>::load(P.nu + off + xv, v);
            R.un = split4(v);
        }
    };
    // the face right of the warp's last column in the row `it + lane` rows
    // after the tile's first, in march order
    T phR = T(0), gR = T(0);
    auto right_faces = [&](int jfirst, int it, int rows) {
        const int xe = x0 + (32 - lane) * kCells;
        phR = gR = T(0);
        if (it + lane < rows && (INTERIOR || xe < nx)) {
            const int j = jfirst + DIR * (it + lane);
            const long long off = (long long)j * pitch + xe;
            T sL, sR;
            if (NOISE == 0) {
                sL = sload(P.s + off - 1);
                sR = sload(P.s + off);
            } else {
                sL = nz.at((long long)j * nx + xe - 1);
                sR = nz.at((long long)j * nx + xe);
            }
            face<LAW, MOB>(sL, sR, sload(P.n + off - 1), sload(P.n + off), sload(P.b + off - 1),
                           sload(P.b + off), scalar_kv<T>(k), phR, gR);
        }
    };
    // y-faces between a lower row lo and an upper row hi
    auto yfaces = [&](const Row<T> &lo, const Row<T> &hi) {
        return row_yfaces<T, LAW, MOB>(lo.s, lo.n, lo.b, hi.s, hi.n, hi.b, k);
    };

    const int jfirst = DIR > 0 ? j0 : jend - 1;
    const int jbehind = jfirst - DIR;
    Row<T> cur, nxt;
    YFaces<T> yB;
    load_row(jfirst, cur, true);
    if (jbehind >= 0 && jbehind < ny) {
        Row<T> prv;
        load_row(jbehind, prv, false);
        yB = DIR > 0 ? yfaces(prv, cur) : yfaces(cur, prv);
    } else {
        yB = zero_yfaces<T>();  // wall behind
    }

    // the last row this tile loads, in march order (the row beyond its last
    // written row, or the grid's edge)
    const int plast = DIR > 0 ? min(jend, ny - 1) : max(j0 - 1, 0);
    const int rows = jend - j0;
    for (int it = 0; it < rows; ++it) {
        const int j = jfirst + DIR * it;
        const int ja = j + DIR;
        const bool has_a = (ja >= 0 && ja < ny);  // uniform across the block
        {
            const int jp = ja + DIR * kPrefetchRows;
            if (DIR > 0 ? jp <= plast : jp >= plast)
                prefetch_row<T, NOISE>(P, (long long)jp * pitch + xv);
        }
        if (has_a) load_row(ja, nxt, it + 1 < rows);

        // x-neighbours of this thread's 4 cells
        T lb = __shfl_up_sync(kFull, cur.b.O.y, 1);
        T ln = __shfl_up_sync(kFull, cur.n.O.y, 1);
        T ls = __shfl_up_sync(kFull, cur.s.O.y, 1);
        if (lane == 0) { lb = cur.hb; ln = cur.hn; ls = cur.hs; }
        XFaces<T> xf;
        if (kRightOnce) {
            if ((it & 31) == 0) right_faces(jfirst, it, rows);
            xf = row_xfaces_shfl<T, LAW, MOB, INTERIOR>(cur.s, cur.n, cur.b, ls, ln, lb, k, x0, nx);
            const T ph = __shfl_sync(kFull, phR, it & 31), g = __shfl_sync(kFull, gR, it & 31);
            if (lane == 31) { xf.ph4 = ph; xf.g4 = g; }
        } else {
            T rb = __shfl_down_sync(kFull, cur.b.E.x, 1);
            T rn = __shfl_down_sync(kFull, cur.n.E.x, 1);
            T rs = __shfl_down_sync(kFull, cur.s.E.x, 1);
            if (lane == 31) { rb = cur.hb; rn = cur.hn; rs = cur.hs; }
            xf = row_xfaces<T, LAW, MOB, INTERIOR>(cur.s, cur.n, cur.b, ls, ln, lb, rs, rn, rb, k, x0,
                                                   nx);
        }

        // y-faces with the row ahead (a wall past the grid's first/last row)
        YFaces<T> yA;
        if (has_a) yA = DIR > 0 ? yfaces(cur, nxt) : yfaces(nxt, cur);
        else yA = zero_yfaces<T>();

        Cells<T> ob, on;
        row_update<T, DIR>(cur.b, cur.n, xf, yB, yA, k, ob, on);
        if (STAGE == 1) {
            ob = heun_mean(cur.ub, ob, k);
            on = heun_mean(cur.un, on, k);
        }
        T vb[kCells], vn[kCells];
        const long long off = (long long)j * pitch;
        if (INTERIOR || x0 + kCells <= nx) {
            join4(ob, vb);
            join4(on, vn);
            Vec<T>::store(P.bo + off + x0, vb);
            Vec<T>::store(P.no + off + x0, vn);
        } else {
            // the row's last group: cell x0 + c lives at column x0 + pair_col(c)
            join4_nat(ob, vb);
            join4_nat(on, vn);
#pragma unroll
            for (int c = 0; c < kCells; ++c)
                if (x0 + c < nx) {
                    P.bo[off + x0 + pair_col(c)] = vb[c];
                    P.no[off + x0 + pair_col(c)] = vn[c];
                }
        }

        cur = nxt;
        yB = yA;
    }
}


}  // namespace stencil
}  // namespace cx
