// Per-node arithmetic of the two-population compressible LB step, for sm_103a.
//
// Everything here acts on the 2Q populations of ONE node held in registers:
// moments (Eqs. density, momentum, energy, P), temperature from the total energy
// (Eqs. U, E with constant Cv = 1/(gamma-1), R = 1), the anomaly Q~_aaa
// (Eq. anomalya), the relaxation rates (Eqs. mu, Pr), the extended f-equilibrium
// (Eqs. productform, extf, Pa_star), the operator product-form g-equilibrium
// (Eq. geq_i) in closed form, the quasi-equilibrium g* (Eqs. gstar, qstar1) and
// the BGK relaxation (Eqs. fLBGK, gLBGK).
//
// Direction i = a + 3b + 9c with (c_x, c_y, c_z) = (a-1, b-1, c-1); D2Q9 uses
// i = a + 3b.  All loops over directions are fully unrolled, so every index is a
// compile-time constant and the populations stay in registers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "elbm_powtab.h"

namespace elbm {

enum StoreKind { ST_F64 = 0, ST_F32 = 1, ST_F16DEV = 2, ST_BF16DEV = 3 };

// Kernel parameters, passed by value (__grid_constant__).
struct KParams {
    int nx, ny, nz;
    int per_x, per_y, per_z;     // 1: periodic axis, 0: zero-gradient (clamped)
    long long N;                 // nx * ny * nz
    double gm1;                  // gamma - 1  (so Cv = 1 / gm1)
    double Pr, mu0, T0, mu_exp;
    int deriv;                   // 0 upwind, 1 central
    int tz;                      // segment length of the fused kernels (D3Q27: z planes, D2Q9: rows)
    int sched;                   // what the default fused schedule runs: 0 the marching kernel, 1 (D2Q9) one
                                 // tile per CTA, 2 (D2Q9) one strip per CTA, 3 the two passes
    int sms;                     // SMs of the device that the rules of the launches go by
    int aa;                      // layout of the store read by the diagnostics: 0 in place; AA single
                                 // store: 1 swapped at the node, 2 pushed to the neighbour
    float2 rest2[27];            // rest-state pair (f_i, g_i) of every direction, deviation stores
    float rest_rho, rest_Pxx, rest_Pyy, rest_Pzz, rest_E;   // their moment sums
    // The same parameters precomputed in both arithmetic types, so that no kernel
    // converts or divides a double per node (the FP64 pipe of GB300 is narrow).
    // fixed-state faces (D2Q9): flags per axis face and the ghost values
    int has_fixed, fix_lo[3], fix_hi[3];
    double fixd[9][2];           // ghost pair (f_i, g_i), FP64 store representation
    float2 fixf[9];              // the same as raw stored values of the FP32 path
    double fixQd[3];             // Q~_aaa of the fixed state
    float fixQf[3];
    // caloric equation of state: 0 constant Cv (d_Cv, gm1); 1 Cv(T) cubic, U(T) quartic
    int eos;
    double cvd[4], Ud[4];        // Cv(T) = sum cvd[k] T^k, U(T) = T sum Ud[k] T^k (Ud[k] = cvd[k]/(k+1))
    float cvf[4], Uf[4];
    int powlaw;                                            // mu_exp != 0
    unsigned inject_tx;          // fault injection: extra bytes each TMA plane announces (0 in use)
    double d_Cv, d_invT0;
    float f_gm1, f_Cv, f_Pr, f_mu0, f_invT0, f_mu_exp;
};

// Parameter in the arithmetic type R.
template <typename R> __device__ __forceinline__ R par(double d, float f);
template <> __device__ __forceinline__ double par<double>(double d, float) { return d; }
template <> __device__ __forceinline__ float par<float>(double, float f) { return f; }

// ---------------------------------------------------------------------------
// Storage codecs.  The store keeps, for every direction i and node n, the pair
// (f_i, g_i) in one element P (double2 / float2 / half2 / bfloat162): both values
// are pulled from the same source node, so one access moves both.  The deviation
// stores (DEV) hold (f_i - f_i^rest, g_i - g_i^rest) rounded to nearest even; the
// kernels keep working on these raw stored values (see node_moments and collide),
// so decoding is a conversion only.
// ---------------------------------------------------------------------------
template <int ST> struct Codec;

template <> struct Codec<ST_F64> {
    using P = double2;
    using R = double;
    static constexpr bool DEV = false;
    __device__ __forceinline__ static void dec(P v, R& f, R& g) { f = v.x; g = v.y; }
    __device__ __forceinline__ static P enc(R f, R g) { return make_double2(f, g); }
};
template <> struct Codec<ST_F32> {
    using P = float2;
    using R = float;
    static constexpr bool DEV = false;
    __device__ __forceinline__ static void dec(P v, R& f, R& g) { f = v.x; g = v.y; }
    __device__ __forceinline__ static P enc(R f, R g) { return make_float2(f, g); }
};
// Mixed-precision add and subtract (sm_100 and later): a 16-bit operand a, exact in
// FP32, combined with an FP32 operand c and rounded once to FP32 — the same result as
// converting a first, in one instruction.  The deviation stores use them to sum moments
// straight from the stored pairs.
__device__ __forceinline__ float mixed_add_f16(unsigned short a, float c) {
    float d;
    asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(a), "f"(c));
    return d;
}
__device__ __forceinline__ float mixed_sub_f16(unsigned short a, float c) {
    float d;
    asm("sub.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(a), "f"(c));
    return d;
}
__device__ __forceinline__ float mixed_add_bf16(unsigned short a, float c) {
    float d;
    asm("add.rn.f32.bf16 %0, %1, %2;" : "=f"(d) : "h"(a), "f"(c));
    return d;
}
__device__ __forceinline__ float mixed_sub_bf16(unsigned short a, float c) {
    float d;
    asm("sub.rn.f32.bf16 %0, %1, %2;" : "=f"(d) : "h"(a), "f"(c));
    return d;
}

template <> struct Codec<ST_F16DEV> {
    using P = __half2;
    using R = float;
    static constexpr bool DEV = true;
    __device__ __forceinline__ static void dec(P v, R& f, R& g) {
        const float2 d = __half22float2(v);
        f = d.x;
        g = d.y;
    }
    __device__ __forceinline__ static P enc(R f, R g) { return __floats2half2_rn(f, g); }
    // f or g component of a stored pair: to FP32, plus / minus an FP32 value
    __device__ __forceinline__ static float f32(P v, int k) { return __half2float(k ? __high2half(v) : __low2half(v)); }
    __device__ __forceinline__ static float add(P v, int k, float c) {
        return mixed_add_f16(__half_as_ushort(k ? __high2half(v) : __low2half(v)), c);
    }
    __device__ __forceinline__ static float sub(P v, int k, float c) {
        return mixed_sub_f16(__half_as_ushort(k ? __high2half(v) : __low2half(v)), c);
    }
};
template <> struct Codec<ST_BF16DEV> {
    using P = __nv_bfloat162;
    using R = float;
    static constexpr bool DEV = true;
    __device__ __forceinline__ static void dec(P v, R& f, R& g) {
        const float2 d = __bfloat1622float2(v);
        f = d.x;
        g = d.y;
    }
    __device__ __forceinline__ static P enc(R f, R g) { return __floats2bfloat162_rn(f, g); }
    __device__ __forceinline__ static float f32(P v, int k) {
        return __bfloat162float(k ? __high2bfloat16(v) : __low2bfloat16(v));
    }
    __device__ __forceinline__ static float add(P v, int k, float c) {
        return mixed_add_bf16(__bfloat16_as_ushort(k ? __high2bfloat16(v) : __low2bfloat16(v)), c);
    }
    __device__ __forceinline__ static float sub(P v, int k, float c) {
        return mixed_sub_bf16(__bfloat16_as_ushort(k ? __high2bfloat16(v) : __low2bfloat16(v)), c);
    }
};

// ---------------------------------------------------------------------------
// Lattice
// ---------------------------------------------------------------------------
template <int D> struct Lat {
    static constexpr int Q = (D == 3) ? 27 : 9;
    static constexpr int NC = (D == 3) ? 3 : 1;      // number of c_z values
};
__host__ __device__ constexpr int cx_of(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int cy_of(int i) { return (i / 3) % 3 - 1; }
template <int D> __host__ __device__ constexpr int cz_of(int i) { return D == 3 ? i / 9 - 1 : 0; }

// Index mapping of one axis: periodic wrap or zero-gradient clamp (the ghost is a
// copy of the adjacent interior node).  Valid for x in [-1, n].
__device__ __forceinline__ int map_axis(int x, int n, int periodic) {
    if (x < 0) return periodic ? x + n : 0;
    if (x >= n) return periodic ? x - n : n - 1;
    return x;
}

// Division in the arithmetic type: exact for FP64, the fast hardware form for FP32
// (a few ulp; every quotient here is of moderate magnitude).
__device__ __forceinline__ double qdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float qdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double qpow(double a, double b) { return pow(a, b); }
__device__ __forceinline__ float qpow(float a, float b) { return __powf(a, b); }

// 1 / x in FP64: the hardware's approximation (about 20 bits) and one step of Householder's
// third-order iteration x <- x (1 + e + e^2), e = 1 - d x, three FP64 instructions where the
// compiler's division takes about ten; within 1 ulp.  Outside 2^(+-1000) the division.
__device__ __forceinline__ double recip(double d) {
    const int ex = (__double2hiint(d) >> 20) & 0x7ff;
    if ((unsigned)(ex - 23) >= 2000u) return 1.0 / d;
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(d));
    const double e = fma(-d, x, 1.0);
    return fma(x, fma(e, e, e), x);
}
// Tests of an FP64 value on its bits: comparisons would take the FP64 pipe.
__device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool positive64(double x) {   // x > 0 (NaN: by its sign bit)
    const int hi = __double2hiint(x);
    return hi >= 0 && (hi | __double2loint(x)) != 0;
}

// x^e in FP64 for the viscosity law: 2^(e log2 x) from two 128-entry tables and Taylor
// polynomials of log2(1 + r), |r| < 0.0049, and 2^f - 1, |f| <= 2^-8 (truncation below
// 2^-60), after Tang's table-driven method; log2 x and its product with e are carried as sums
// of two doubles.  About 27 FP64 instructions where pow() takes several times as many; on
// GB300's FP64 pipe (one warp instruction per 16 cycles and SM) that is what a node's
// viscosity costs.  The remaining error is the rounding of 2^(j/128) and of the result (rms
// 0.4 ulp; pow() 0.3).  Arguments outside [2^-100, 2^100], non-finite ones and exponents of 2 beyond 60 go
// to pow().
__device__ __forceinline__ double pow_pos(double x, double e) {
    const int hi = __double2hiint(x);
    if ((unsigned)(hi - 0x39b00000) >= 0x0c800000u) return pow(x, e);
    const int k = (hi >> 20) - 1023, j = (hi >> 13) & 127;
    const double2 tab = kLogTab[j];
    const double m = __hiloint2double(hi - (k << 20), __double2loint(x));
    const double r = fma(m, tab.x, -1.0);
    double q = fma(r, 0x1.a61762a7aded9p-3, -0x1.ec709dc3a03fdp-3);
    q = fma(r, q, 0x1.2776c50ef9bfep-2);
    q = fma(r, q, -0x1.71547652b82fep-2);
    q = fma(r, q, 0x1.ec709dc3a03fdp-2);
    q = fma(r, q, -0x1.71547652b82fep-1);
    q = fma(r, q, 0x1.71547652b82fep+0);
    // log2 x = L + l; k + h_j is exact, and not below |r q| in size unless that is tiny
    const double A = (double)k + tab.y, L = fma(r, q, A), l = fma(r, q, A - L) + kLogLo[j];
    const double t = e * L, tl = fma(e, l, fma(e, L, -t));
    if ((__double2hiint(t) & 0x7fffffff) >= 0x404e0000 /* 60 */) return pow(x, e);
    const double tn = fma(t, 128.0, 0x1.8p52);   // nearest multiple of 1/128 in the low bits
    const int n = __double2loint(tn);
    const double f = fma(tn - 0x1.8p52, -0x1p-7, t) + tl;
    double s = fma(f, 0x1.5d87fe78a6731p-10, 0x1.3b2ab6fba4e77p-7);
    s = fma(f, s, 0x1.c6b08d704a0c0p-5);
    s = fma(f, s, 0x1.ebfbdff82c58fp-3);
    s = fma(f, s, 0x1.62e42fefa39efp-1);
    const double c = kExpTab[n & 127];
    const double y = fma(c, f * s, c);
    return __hiloint2double(__double2hiint(y) + ((n >> 7) << 20), __double2loint(y));
}

// ---------------------------------------------------------------------------
// Error-free FP32 sums.  Two floats at a time (FADD2/FFMA2, sm_100 and later): the sums that
// the diagnostics take over FP32 values run as unevaluated sums of three floats (Knuth's
// TwoSum; relative error about 2^-70), since one FP64 addition costs as much of the SM as 64
// FP32 ones.
// ---------------------------------------------------------------------------
// (V = float2; templates, so that host programs which include this header for another
// architecture need not know the two-lane instructions)
template <class V> __device__ __forceinline__ V add2(V a, V b) { return __fadd2_rn(a, b); }
template <class V> __device__ __forceinline__ V mul2(V a, V b) { return __fmul2_rn(a, b); }
template <class V> __device__ __forceinline__ V fma2(V a, V b, V c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 both(float c) { return make_float2(c, c); }
template <class V> __device__ __forceinline__ V sub2(V a, V b) { return __ffma2_rn(b, V{-1.f, -1.f}, a); }
// a + b = s + err exactly, in both lanes
template <class V> __device__ __forceinline__ V two_sum2(V a, V b, V& err) {
    const V s = __fadd2_rn(a, b);
    const V bb = sub2(s, a);
    err = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}
template <class V> struct TriOf {   // two running sums s + e1 + e2
    V s, e1, e2;
    __device__ __forceinline__ void zero() { s = e1 = e2 = V{0.f, 0.f}; }
    __device__ __forceinline__ void add(V v) {
        V r, r1;
        s = two_sum2(s, v, r);
        e1 = two_sum2(e1, r, r1);
        e2 = __fadd2_rn(e2, r1);
    }
    // adds v + lo, lo a correction of v
    __device__ __forceinline__ void add(V v, V lo) {
        V r;
        add(v);
        e1 = two_sum2(e1, lo, r);
        e2 = __fadd2_rn(e2, r);
    }
    __device__ __forceinline__ void add(const TriOf& o) {
        add(o.s, o.e1);
        e2 = __fadd2_rn(e2, o.e2);
    }
    // sum over the lanes of a warp, in every lane
    __device__ __forceinline__ void warp_sum() {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            TriOf o;
            o.s = V{__shfl_xor_sync(0xffffffffu, s.x, d), __shfl_xor_sync(0xffffffffu, s.y, d)};
            o.e1 = V{__shfl_xor_sync(0xffffffffu, e1.x, d), __shfl_xor_sync(0xffffffffu, e1.y, d)};
            o.e2 = V{__shfl_xor_sync(0xffffffffu, e2.x, d), __shfl_xor_sync(0xffffffffu, e2.y, d)};
            add(o);
        }
    }
};
using Tri2 = TriOf<float2>;
// FP64 running sum s + c (TwoSum)
__device__ __forceinline__ void dd_add(double& s, double& c, double v) {
    const double t = s + v, b = t - s;
    c += (s - (t - b)) + (v - b);
    s = t;
}

// Unevaluated sum h + l of two floats (|l| <= ulp(h)/2): differences and products of FP32
// values are exact in this form, sums are rounded to about 2^-47.
struct Df {
    float h, l;
};
__device__ __forceinline__ Df df_diff(float a, float b) {   // a - b, exact
    const float s = a - b, bb = s - a;
    return {s, (a - (s - bb)) - (b + bb)};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
    const float s = a.h + b.h, bb = s - a.h;
    const float e = ((a.h - (s - bb)) + (b.h - bb)) + (a.l + b.l);
    const float h = s + e;
    return {h, e - (h - s)};
}
// The same, adding what is rounded away to rest: a sum of squares needs it, whose low bits are not random (an
// odd number's square ends in 001) and whose roundings have a sign.
__device__ __forceinline__ Df df_add(Df a, Df b, float& rest) {
    const float s = a.h + b.h, bb = s - a.h, e1 = (a.h - (s - bb)) + (b.h - bb);
    const float q = a.l + b.l, qb = q - a.l, e2 = (a.l - (q - qb)) + (b.l - qb);
    const float e = e1 + q, eb = e - e1;
    rest += e2 + ((e1 - (e - eb)) + (q - eb));
    const float h = s + e;
    return {h, e - (h - s)};
}
__device__ __forceinline__ Df df_neg(Df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Df df_prod(float a, float b) {   // a b, exact
    const float p = __fmul_rn(a, b);
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ Df df_sq(Df a) {
    const float p = __fmul_rn(a.h, a.h);
    return {p, fmaf(2.f * a.h, a.l, fmaf(a.h, a.h, -p))};
}
__device__ __forceinline__ Df df_mul(Df a, Df b) {
    const float p = __fmul_rn(a.h, b.h);
    return {p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)))};
}
__device__ __forceinline__ Df df_scale(Df a, float b) {
    const float p = __fmul_rn(a.h, b);
    return {p, fmaf(a.l, b, fmaf(a.h, b, -p))};
}

// pow_pos of an FP32 x over 2^base, base a multiple of 2^-8, as a sum of two floats: the same steps in
// pairs of floats, about 100 FP32 instructions where one FP64 instruction keeps the SM as busy
// as 64.  Relative error about 2^-44, or 2^-47 |e (log2 x - base)| and 2^-49 where that is less; what many
// x share (the tables' and the exponent's third floats) is carried beside, so that sums have
// no more error than FP64 ones.  False (and no value) for an x or an exponent of 2 that pow_pos leaves to pow().
__device__ __forceinline__ bool pow_pos_df(float x, Df e, Df& y, float base = 0.f) {
    const int b = __float_as_int(x);
    if ((unsigned)(b - 0x0d800000) >= 0x64000000u) return false;   // 2^-100 <= x < 2^100
    const int k = (b >> 23) - 127;
    const float4 tab = kLogTabF[(b >> 16) & 127];
    const Df m = df_prod(__int_as_float(b - (k << 23)), tab.x);
    const float rh = m.h - 1.f;   // exact
    const float r0 = rh + m.l;
    const Df r = {r0, m.l - (r0 - rh)};
    // log2(1 + r) = r (c1 + r (c2 + r q))
    float q = fmaf(r.h, -0x1.ec709ep-3f, 0x1.2776c6p-2f);
    q = fmaf(r.h, q, -0x1.715476p-2f);
    q = fmaf(r.h, q, 0x1.ec709ep-2f);
    const Df c1 = {0x1.715476p+0f, 0x1.4ae0c0p-26f}, c2 = {-0x1.715476p-1f, -0x1.4ae0c0p-27f};
    const Df s = df_mul(r, df_add(c1, df_mul(r, df_add(c2, df_prod(r.h, q)))));
    float rest = tab.w;
    const Df L = df_add(df_add({(float)k - base, 0.f}, {tab.y, tab.z}, rest), s, rest);
    const Df t = df_mul(e, L);
    if (!(fabsf(t.h) < 60.f)) return false;
    const float n = rintf(t.h * 128.f);
    const float f0 = fmaf(n, -0x1p-7f, t.h), fh = f0 + t.l;
    const Df f = {fh, fmaf(e.h, rest, t.l - (fh - f0))};
    // 2^f - 1 = f (d1 + f (d2 + f (d3 + f d4)))
    const Df d1 = {0x1.62e430p-1f, -0x1.05c610p-29f}, d2 = {0x1.ebfbe0p-3f, -0x1.f4e9c6p-33f};
    const float d = fmaf(f.h, 0x1.3b2ab6p-7f, 0x1.c6b08ep-5f);
    const Df w = df_mul(f, df_add(d1, df_mul(f, df_add(d2, df_prod(f.h, d)))));
    const int ni = (int)n;
    const float2 c = kExpTabF[ni & 127];
    Df cw = df_mul({c.x, c.y}, w);
    cw.l += kExpTabL[ni & 127];
    const Df z = df_add({c.x, c.y}, cw);
    const float two = __int_as_float(((ni >> 7) + 127) << 23);
    y = {z.h * two, z.l * two};
    return true;
}

// ---------------------------------------------------------------------------
// Caloric equation of state (Eqs. U, E; R = 1): U(T) = int_0^T Cv dT and its inverse
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ R cubic(const double* cd, const float* cf, R T) {
    return par<R>(cd[0], cf[0]) + T * (par<R>(cd[1], cf[1]) + T * (par<R>(cd[2], cf[2]) + T * par<R>(cd[3], cf[3])));
}
// CAL = false compiles the constant-Cv model only (the kernels launch that form when
// the handle's model is constant gamma); CAL = true branches on the handle's model.
template <typename R, bool CAL = true>
__device__ __forceinline__ R U_of_T(R T, const KParams& p) {
    if (!CAL || !p.eos) return T * par<R>(p.d_Cv, p.f_Cv);
    return T * cubic<R>(p.Ud, p.Uf, T);
}
// T from U: constant Cv directly; otherwise Newton's method on the increasing U(T)
// from T = U / Cv(0), a fixed 8 iterations (enough for T <= 1 with the stated Cv).
template <typename R, bool CAL = true>
__device__ __forceinline__ R T_of_U(R U, const KParams& p) {
    if (!CAL || !p.eos) return U * par<R>(p.gm1, p.f_gm1);
    R T = U / par<R>(p.cvd[0], p.cvf[0]);
#pragma unroll
    for (int k = 0; k < 8; ++k) T -= (T * cubic<R>(p.Ud, p.Uf, T) - U) / cubic<R>(p.cvd, p.cvf, T);
    return T;
}

// ---------------------------------------------------------------------------
// Moments
// ---------------------------------------------------------------------------
template <typename R> struct Moments {
    R rho, ux, uy, uz, T, rE;
    R Pxx, Pyy, Pzz, Pxy, Pxz, Pyz;   // sum c c f (pre-collision)
};

// Moments of f: rho, rho u and (FULL) the pressure tensor sum c c f.  f holds the raw
// stored values; for the deviation stores (DEV) the moment sums of the rest state are
// added (the rest state carries no momentum and no off-diagonal stress, by symmetry).
template <int D, typename R, bool FULL, bool DEV>
__device__ __forceinline__ void f_moments(const R* f, const KParams& p, R& rho, R& jx, R& jy, R& jz,
                                          R P6[6]) {
    constexpr int NC = Lat<D>::NC;
    // per (b, c) row sums over c_x
    R t[3][3], d[3][3], e[3][3];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int i0 = 3 * b + 9 * c;
            R lo = f[i0], mid = f[i0 + 1], hi = f[i0 + 2];
            e[b][c] = hi + lo;
            d[b][c] = hi - lo;
            t[b][c] = e[b][c] + mid;
        }
    // sums over c_z first (columns b), then over c_y: depth 2 + 2
    R tb[3], db[3], eb[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        tb[b] = t[b][0];
        db[b] = d[b][0];
        eb[b] = e[b][0];
        if (D == 3) {
            tb[b] = (t[b][0] + t[b][2]) + t[b][1];
            db[b] = (d[b][0] + d[b][2]) + d[b][1];
            eb[b] = (e[b][0] + e[b][2]) + e[b][1];
        }
    }
    rho = (tb[0] + tb[2]) + tb[1];
    jx = (db[0] + db[2]) + db[1];
    jy = tb[2] - tb[0];
    jz = 0;
    R Pxx = (eb[0] + eb[2]) + eb[1], Pyy = tb[2] + tb[0], Pxy = db[2] - db[0];
    R Pzz = 0, Pxz = 0, Pyz = 0;
    if (D == 3) {
        const R tzh = (t[0][2] + t[2][2]) + t[1][2], tzl = (t[0][0] + t[2][0]) + t[1][0];
        const R dzh = (d[0][2] + d[2][2]) + d[1][2], dzl = (d[0][0] + d[2][0]) + d[1][0];
        jz = tzh - tzl;
        Pzz = tzh + tzl;
        Pxz = dzh - dzl;
        Pyz = (t[2][2] - t[0][2]) - (t[2][0] - t[0][0]);
    }
    if constexpr (DEV) {
        rho += R(p.rest_rho);
        Pxx += R(p.rest_Pxx);
        Pyy += R(p.rest_Pyy);
        Pzz += R(p.rest_Pzz);
    }
    if (FULL) {
        P6[0] = Pxx; P6[1] = Pyy; P6[2] = Pzz;
        P6[3] = Pxy; P6[4] = Pxz; P6[5] = Pyz;
    }
}

// rho E = sum of g, as a balanced tree (short dependency chains).
template <int D, typename R, bool DEV>
__device__ __forceinline__ R g_energy(const R* g, const KParams& p) {
    R gs[Lat<D>::Q];
#pragma unroll
    for (int i = 0; i < Lat<D>::Q; ++i) gs[i] = g[i];
#pragma unroll
    for (int w = 1; w < Lat<D>::Q; w *= 2)
#pragma unroll
        for (int i = 0; i + w < Lat<D>::Q; i += 2 * w) gs[i] += gs[i + w];
    R rE = gs[0];
    if constexpr (DEV) rE += R(p.rest_E);
    return rE;
}

// u = j / rho and T from E = Cv T + u^2/2.
template <typename R, bool CAL = true>
__device__ __forceinline__ void finish_moments(R rho, R jx, R jy, R jz, R rE, const KParams& p, Moments<R>& m) {
    R inv;
    if constexpr (sizeof(R) == 8) inv = recip(rho);
    else inv = qdiv(R(1), rho);
    m.rho = rho;
    m.rE = rE;
    m.ux = jx * inv;
    m.uy = jy * inv;
    m.uz = jz * inv;
    const R u2 = m.ux * m.ux + m.uy * m.uy + m.uz * m.uz;
    m.T = T_of_U<R, CAL>(rE * inv - R(0.5) * u2, p);
}

// The same moments straight from the stored pairs of a deviation store: pair(i) returns
// the stored (f_i, g_i) of direction i.  Per (c_y, c_z) row one component is converted and
// the other two enter through mixed-precision adds (hi + lo, hi - lo, mid + (hi + lo));
// the energy is the sum of the nine row sums of g.  The rounding is that of f_moments
// and g_energy on the converted values, up to the order of the energy sum.
template <int D, int ST, bool FULL, bool CAL = true, class Pair>
__device__ __forceinline__ void node_moments_stored(Pair pair, const KParams& p, Moments<float>& m) {
    using Cd = Codec<ST>;
    using R = float;
    constexpr int NC = Lat<D>::NC;
    R t[3][3], d[3][3], e[3][3], gr[3][3];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int i0 = 3 * b + 9 * c;
            const auto lo = pair(i0), mid = pair(i0 + 1), hi = pair(i0 + 2);
            const R lo32 = Cd::f32(lo, 0);
            e[b][c] = Cd::add(hi, 0, lo32);
            d[b][c] = Cd::sub(hi, 0, lo32);
            t[b][c] = Cd::add(mid, 0, e[b][c]);
            gr[b][c] = Cd::add(hi, 1, Cd::add(mid, 1, Cd::f32(lo, 1)));
        }
    R tb[3], db[3], eb[3], gb[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        tb[b] = t[b][0];
        db[b] = d[b][0];
        eb[b] = e[b][0];
        gb[b] = gr[b][0];
        if (D == 3) {
            tb[b] = (t[b][0] + t[b][2]) + t[b][1];
            db[b] = (d[b][0] + d[b][2]) + d[b][1];
            eb[b] = (e[b][0] + e[b][2]) + e[b][1];
            gb[b] = (gr[b][0] + gr[b][2]) + gr[b][1];
        }
    }
    R rho = (tb[0] + tb[2]) + tb[1];
    const R jx = (db[0] + db[2]) + db[1];
    const R jy = tb[2] - tb[0];
    R jz = 0;
    R Pxx = (eb[0] + eb[2]) + eb[1], Pyy = tb[2] + tb[0], Pxy = db[2] - db[0];
    R Pzz = 0, Pxz = 0, Pyz = 0;
    if (D == 3) {
        const R tzh = (t[0][2] + t[2][2]) + t[1][2], tzl = (t[0][0] + t[2][0]) + t[1][0];
        const R dzh = (d[0][2] + d[2][2]) + d[1][2], dzl = (d[0][0] + d[2][0]) + d[1][0];
        jz = tzh - tzl;
        Pzz = tzh + tzl;
        Pxz = dzh - dzl;
        Pyz = (t[2][2] - t[0][2]) - (t[2][0] - t[0][0]);
    }
    rho += R(p.rest_rho);
    const R rE = ((gb[0] + gb[2]) + gb[1]) + R(p.rest_E);
    finish_moments<R, CAL>(rho, jx, jy, jz, rE, p, m);
    if (FULL) {
        m.Pxx = Pxx + R(p.rest_Pxx);
        m.Pyy = Pyy + R(p.rest_Pyy);
        m.Pzz = Pzz + R(p.rest_Pzz);
        m.Pxy = Pxy; m.Pxz = Pxz; m.Pyz = Pyz;
    }
}

// Shifts that clamp: 0 from 64 on.
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned n) {
    asm("shr.b64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(n));
    return v;
}
__device__ __forceinline__ unsigned long long shl64(unsigned long long v, unsigned n) {
    asm("shl.b64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(n));
    return v;
}
// m 2^(e - 1086), sign bit of hi `sign`, for 0 < m < 2^63 within the normal range, rounded to nearest, ties
// to even (EVEN) or up; z leading zeros of m.
template <bool EVEN>
__device__ __forceinline__ double round64(unsigned long long m, int z, int e, unsigned sign) {
    unsigned long long b;   // 53 bits, or 2^53
    if (EVEN) {
        const unsigned long long s = m << (z - 1 & 63);   // first bit at 62
        b = (s + (0x1ffu + (((unsigned)s >> 10) & 1u))) >> 10;
    } else {
        b = (((m << z) >> 10) + 1ull) >> 1;
    }
    return __hiloint2double((int)(((unsigned)(b >> 32) + ((unsigned)(e - z - 1) << 20)) | sign), (int)(unsigned)b);
}

// Sums of FP64 values in 64-bit integers.  An FP64 instruction holds a quarter of an SM for 64 cycles
// and an integer one for one or two, so the moments, which only add and subtract populations, are
// summed as integers: fixed(x, top) is x in units of 2^-57 of the power of two of the
// largest |x| (biased exponent + 6: top); the sums are exact and 26 values fit.  The value at
// rest, part of rho and rho E alone and 16 times the next, is added in FP64.  A value that has bits
// below the unit is rounded to the odd one of its neighbours (von Neumann's rounding), others are
// exact, and the sum is rounded to nearest, ties to even: no step has a sign on the average, where a floor and
// half a unit added moved the mass of a periodic sheet by 2e-14 in 10,000 steps.  Each value is off by less
// than a unit, about 2^-55 of the largest in a sum of 26, where an FP64 tree
// rounds each partial sum by up to 2^-53 of it.  D3Q27 moments 243 -> 123 us (96^3; 141 -> 50 FP64
// instructions a warp), D2Q9 127 -> 83 (1024^2).
struct FixedSum {
    static __device__ __forceinline__ int top_of(int top, double x) { return max(top, __double2hiint(x) & 0x7fffffff); }
    // exponents that keep clear of infinities, NaN and the subnormal range
    static __device__ __forceinline__ bool usable(int top) { return top >= 128 << 20 && top < 2040 << 20; }
    static __device__ __forceinline__ long long fixed(double x, int top) {
        const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
        const unsigned h = __funnelshift_l(lo, hi, 11) | 0x80000000u, l = lo << 11;   // the significand, first bit set
        const unsigned n = (unsigned)top - ((hi >> 20) & 0x7ffu);                      // top = exponent + 6
        const unsigned long long sig = ((unsigned long long)h << 32) | l;
        unsigned long long v = shr64(sig, n);
        if (__funnelshift_rc(0u, l, n) != 0u) v |= 1ull;   // the low word's bits below the unit
        const long long neg = (int)hi >> 31;
        return ((long long)v ^ neg) - neg;
    }
    static __device__ __forceinline__ double value(long long v, int top) {
        const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
        return v == 0 ? 0.0 : round64<true>(m, __clzll((long long)m), top, (unsigned)(v >> 32) & 0x80000000u);
    }
};
template <int D, bool FULL>
__device__ __forceinline__ bool fixed_sums(const double* f, const double* g, const KParams& p, double& rho, double& jx,
                                           double& jy, double& jz, double P6[6], double& rE) {
    constexpr int Q = Lat<D>::Q, REST = Q / 2;
    int tf = 0, tg = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i)
        if (i != REST) {
            tf = FixedSum::top_of(tf, f[i]);
            tg = FixedSum::top_of(tg, g[i]);
        }
    if (!FixedSum::usable(tf) || !FixedSum::usable(tg)) return false;
    tf = (tf >> 20) + 6;
    tg = (tg >> 20) + 6;
    long long s[Q], n[4], P[6], E = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        s[i] = i == REST ? 0 : FixedSum::fixed(f[i], tf);
        if (i != REST) E += FixedSum::fixed(g[i], tg);
    }
    f_moments<D, long long, true, false>(s, p, n[0], n[1], n[2], n[3], P);
    rho = f[REST] + FixedSum::value(n[0], tf);
    rE = g[REST] + FixedSum::value(E, tg);
    jx = FixedSum::value(n[1], tf);
    jy = FixedSum::value(n[2], tf);
    jz = D == 3 ? FixedSum::value(n[3], tf) : 0.0;
    if (FULL)
#pragma unroll
        for (int k = 0; k < 6; ++k) P6[k] = D == 2 && (k == 2 || k > 3) ? 0.0 : FixedSum::value(P[k], tf);
    return true;
}

// All moments of one node: f_moments, g_energy, finish_moments.
template <int D, typename R, bool FULL, bool DEV, bool CAL = true>
__device__ __forceinline__ void node_moments(const R* f, const R* g, const KParams& p, Moments<R>& m) {
    R rho, jx, jy, jz, P6[6], rE;
    bool done = false;
    if constexpr (sizeof(R) == 8 && !DEV) done = fixed_sums<D, FULL>(f, g, p, rho, jx, jy, jz, P6, rE);
    if (!done) {
        f_moments<D, R, FULL, DEV>(f, p, rho, jx, jy, jz, P6);
        rE = g_energy<D, R, DEV>(g, p);
    }
    finish_moments<R, CAL>(rho, jx, jy, jz, rE, p, m);
    if (FULL) {
        m.Pxx = P6[0]; m.Pyy = P6[1]; m.Pzz = P6[2];
        m.Pxy = P6[3]; m.Pxz = P6[4]; m.Pyz = P6[5];
    }
}

// Q~_aaa = rho u_a (1 - 3T - u_a^2)  (Eq. anomalya, R = 1)
template <typename R>
__device__ __forceinline__ R anomaly(R rho, R ua, R T) {
    return rho * ua * (R(1) - R(3) * T - ua * ua);
}

// Discrete derivative of Q~_aaa at a node from its own value and the two axis
// neighbours: upwind by the sign of u_a at the node (strict '>'), or central.
template <typename R>
__device__ __forceinline__ R dQ(int deriv, R ua, R qm, R q0, R qp) {
    if (deriv) return R(0.5) * (qp - qm);
    if constexpr (sizeof(R) == 8) {   // one subtraction, the operands chosen on the sign bit
        const bool up = positive64(ua);
        return (up ? q0 : qp) - (up ? qm : q0);
    }
    return ua > R(0) ? (q0 - qm) : (qp - q0);
}

// Unphysical-state test used to latch ELBM_ERR_NONPHYSICAL.
template <typename R>
__device__ __forceinline__ bool nonphysical(const Moments<R>& m) {
    if constexpr (sizeof(R) == 8)
        return !positive64(m.rho) || !positive64(m.T) || !finite64(m.rho) || !finite64(m.T) || !finite64(m.ux) ||
               !finite64(m.uy) || !finite64(m.uz);
    return !(m.rho > R(0)) || !(m.T > R(0)) || !isfinite(m.rho) || !isfinite(m.T) ||
           !isfinite(m.ux) || !isfinite(m.uy) || !isfinite(m.uz);
}

// ---------------------------------------------------------------------------
// Equilibria and collision
// ---------------------------------------------------------------------------
// Psi triplet at (xi, P), indexed a = c + 1 (Eqs. phi0S, phiPlusS, phiMinusS).
template <typename R>
__device__ __forceinline__ void psi3(R xi, R P, R out[3]) {
    out[0] = R(0.5) * (P - xi);
    out[1] = R(1) - P;
    out[2] = R(0.5) * (P + xi);
}

// Per-axis factors of g^eq.  Applying Psi_c(O, O^2) (Eq. Operator) to functions of
// one velocity component u gives
//   on 1:       phi_c = Psi_c(u, T + u^2)                      (as f^eq)
//   on u^2/2:   psi_0 = u^2/2 - s,  psi_{+-1} = (s +- o)/2,
//   with o = O(u^2/2) = T u + u^3/2 and s = O^2(u^2/2) = T^2 + (5/2) T u^2 + u^4/2.
// With E = Cv T + sum_b u_b^2/2 this gives
//   g^eq_i = rho [ Cv T phi_x phi_y phi_z + psi_x phi_y phi_z + phi_x psi_y phi_z
//                  + phi_x phi_y psi_z ].
template <typename R>
__device__ __forceinline__ void gfactors(R u, R T, R phi[3], R ps[3]) {
    const R u2 = u * u;
    psi3(u, T + u2, phi);
    const R o = T * u + R(0.5) * u2 * u;
    const R s = T * T + R(2.5) * T * u2 + R(0.5) * u2 * u2;
    ps[0] = R(0.5) * (s - o);
    ps[1] = R(0.5) * u2 - s;
    ps[2] = R(0.5) * (s + o);
}

// Equilibria f^eq and g^eq of (rho, u, T) into f, g (full populations; used for
// initialisation).
template <int D, typename R>
__device__ __forceinline__ void equilibria(R rho, R ux, R uy, R uz, R T, R U, R* f, R* g) {
    R X[3], Y[3], Z[3], sx[3], sy[3], sz[3];
    gfactors(ux, T, X, sx);
    gfactors(uy, T, Y, sy);
    if (D == 3) gfactors(uz, T, Z, sz);
    else { Z[0] = Z[2] = 0; Z[1] = 1; sz[0] = sz[1] = sz[2] = 0; }
    const R CvT = U;   // U(T): Cv T for constant Cv
#pragma unroll
    for (int c = 0; c < Lat<D>::NC; ++c) {
        const int cc = (D == 3) ? c : 1;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R A = Y[b] * Z[cc];
            const R B = sy[b] * Z[cc] + Y[b] * sz[cc];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int i = a + 3 * b + 9 * c;
                f[i] = rho * X[a] * A;
                g[i] = rho * ((CvT * X[a] + sx[a]) * A + X[a] * B);
            }
        }
    }
}

// Relaxation rate omega (Eqs. mu, Pr) from the local pressure P = rho T, and omega_1.
template <typename R>
__device__ __forceinline__ R rate_w(R rho, R T, const KParams& p) {
    R mu = par<R>(p.mu0, p.f_mu0);
    if (p.powlaw) mu = mu * qpow(T * par<R>(p.d_invT0, p.f_invT0), par<R>(p.mu_exp, p.f_mu_exp));
    const R P = rho * T;
    return qdiv(R(2) * P, R(2) * mu + P);
}
template <typename R>
__device__ __forceinline__ R rate_w1(R w, const KParams& p) {
    const R Pr = par<R>(p.Pr, p.f_Pr);
    return qdiv(R(2) * Pr * w, R(2) - w + Pr * w);
}

// One collision, direction by direction.  init() evaluates the per-node factors;
// f(i, f_i) and g(i, g_i) return the post-collision values of direction i from the raw
// stored values (populations, or their deviations from the rest state when DEV).
//   f_i <- (1 - w) f_i + w f^ex_i            (Eqs. fLBGK, extf, Pa_star)
//   g_i <- (1 - w1) g_i + w1 g^eq_i + corr_i (Eqs. gLBGK, geq_i, gstar, qstar1)
// with w and w1 folded into the row factors of the product forms.  For DEV the rest
// state r_i is carried as (1 - w)(r_i + d_i) + w f^ex_i - r_i = (1 - w) d_i +
// w (f^ex_i - r_i).  corr_i is the quasi-equilibrium term, nonzero only for |c_i| = 1:
// q* - q^eq = u.(P - P^eq + div Q~ / 2) with P^eq = rho T I + rho u u and
// div Q~ = diag(D), and g_i += (omega - omega_1)(g^eq_i - g*_i) =
// -(omega - omega_1) c_i.(q* - q^eq) / 2.  m must carry the pressure tensor.
template <int D, typename R, bool DEV, bool CAL = true>
struct Relax {
    R omw, omw1, w, w1;
    R X[3], Y[3], Z[3], wr;                      // f^ex factors
    R gx[3], gy[3], gz[3], sy[3], sz[3], ax[3];  // g^eq factors
    R w1r;
    R h, dq[3];                                  // (omega - omega_1)/2 and q* - q^eq

    __device__ __forceinline__ void init(const Moments<R>& m, R Dx, R Dy, R Dz, const KParams& p) {
        const R rho = m.rho, T = m.T, ux = m.ux, uy = m.uy, uz = m.uz;
        w = rate_w(rho, T, p);
        w1 = rate_w1(w, p);
        // extended f-equilibrium
        const R k = qdiv(R(2) - w, R(2) * rho * w);
        psi3(ux, T + ux * ux + k * Dx, X);
        psi3(uy, T + uy * uy + k * Dy, Y);
        if (D == 3) psi3(uz, T + uz * uz + k * Dz, Z);
        else { Z[0] = Z[2] = 0; Z[1] = 1; }
        omw = R(1) - w;
        wr = w * rho;
        // g-equilibrium
        R sx[3];
        gfactors(ux, T, gx, sx);
        gfactors(uy, T, gy, sy);
        if (D == 3) gfactors(uz, T, gz, sz);
        else { gz[0] = gz[2] = 0; gz[1] = 1; sz[0] = sz[1] = sz[2] = 0; }
        const R CvT = U_of_T<R, CAL>(T, p);   // U(T) (Cv T for constant Cv)
#pragma unroll
        for (int a = 0; a < 3; ++a) ax[a] = CvT * gx[a] + sx[a];
        omw1 = R(1) - w1;
        w1r = w1 * rho;
        // quasi-equilibrium
        const R rT = rho * T;
        const R dxx = m.Pxx - rT - rho * ux * ux, dyy = m.Pyy - rT - rho * uy * uy;
        const R dxy = m.Pxy - rho * ux * uy;
        R dqx = ux * dxx + uy * dxy + R(0.5) * ux * Dx;
        R dqy = ux * dxy + uy * dyy + R(0.5) * uy * Dy;
        R dqz = 0;
        if (D == 3) {
            const R dzz = m.Pzz - rT - rho * uz * uz;
            const R dxz = m.Pxz - rho * ux * uz, dyz = m.Pyz - rho * uy * uz;
            dqx += uz * dxz;
            dqy += uz * dyz;
            dqz = ux * dxz + uy * dyz + uz * dzz + R(0.5) * uz * Dz;
        }
        h = R(0.5) * (w - w1);
        dq[0] = dqx;
        dq[1] = dqy;
        dq[2] = dqz;
    }

    // i is a compile-time constant after unrolling, so every branch below folds away
    __device__ __forceinline__ R f(int i, R fi, const KParams& p) const {
        const int a = cx_of(i) + 1, b = cy_of(i) + 1, c = (D == 3) ? cz_of<D>(i) + 1 : 1;
        const R yz = wr * Y[b] * Z[c];
        R t = X[a] * yz;
        if constexpr (DEV) t = fma(-w, R(p.rest2[i].x), t);
        return fma(omw, fi, t);
    }
    // Both updates of direction i at once, as two-lane FP32 arithmetic (FFMA2, sm_100 and
    // later): the same operations in the same order as f() and g(), so the same results.
    __device__ __forceinline__ float2 fg(int i, float2 v, const KParams& p) const {
        static_assert(sizeof(R) == 4, "two-lane form of the FP32 arithmetic");
        const int a = cx_of(i) + 1, b = cy_of(i) + 1, c = (D == 3) ? cz_of<D>(i) + 1 : 1;
        const R yz = wr * Y[b] * Z[c];
        const R A = w1r * gy[b] * gz[c];
        const R B = w1r * (sy[b] * gz[c] + gy[b] * sz[c]);
        float2 t = make_float2(X[a] * yz, fma(ax[a], A, gx[a] * B));
        if constexpr (DEV) t = __ffma2_rn(make_float2(-w, -w1), p.rest2[i], t);
        float2 o = __ffma2_rn(make_float2(omw, omw1), v, t);
        const int cx = cx_of(i), cy = cy_of(i), cz = cz_of<D>(i);
        if (cx * cx + cy * cy + cz * cz == 1) {
            const R q = cx != 0 ? dq[0] : (cy != 0 ? dq[1] : dq[2]);
            if (cx + cy + cz < 0) o.y += h * q;
            else o.y -= h * q;
        }
        return o;
    }
    __device__ __forceinline__ R g(int i, R gi, const KParams& p) const {
        constexpr int Q = Lat<D>::Q;
        const int a = cx_of(i) + 1, b = cy_of(i) + 1, c = (D == 3) ? cz_of<D>(i) + 1 : 1;
        const R A = w1r * gy[b] * gz[c];
        const R B = w1r * (sy[b] * gz[c] + gy[b] * sz[c]);
        R t = fma(ax[a], A, gx[a] * B);
        if constexpr (DEV) t = fma(-w1, R(p.rest2[i].y), t);
        R v = fma(omw1, gi, t);
        // unit-speed directions: the correction enters with the sign of -c_i
        const int cx = cx_of(i), cy = cy_of(i), cz = cz_of<D>(i);
        if (cx * cx + cy * cy + cz * cz == 1) {
            const R q = cx != 0 ? dq[0] : (cy != 0 ? dq[1] : dq[2]);
            if (cx + cy + cz < 0) v += h * q;
            else v -= h * q;
        }
        return v;
    }
};

// Sums of products of FP64 values in integers: a product of significands of 62 and 63 bits, the upper
// half of it (three multiplications of 32 bits), up to four such terms shifted to the exponent of the
// largest, added, and rounded once.  Every product has some 45 bits below the unit, so a floor
// takes half a unit from it on the average, and the product of the low words, which is left out, is a
// quarter of the last place before the shift on the average: both are added.  Of three terms' one and a half units
// the last half is what rounding ties up adds.  A term is off by less than 2^-57 of the largest, where FP64
// rounds every product and partial sum by up to 2^-53.  Zero counts as 2^-1023.
// Terms must keep clear of infinity; results below the normal range are zero.
struct FixedProd {
    struct Sig { unsigned hi, lo, es; };              // significand; biased exponent, sign in bit 31
    struct Term { unsigned long long r; unsigned es; };   // value r 2^-59 2^(e - 2046)
    template <int S>   // 64 - S bits of significand: S = 1 and 2 multiply
    static __device__ __forceinline__ Sig sig(double x) {
        const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
        return {(__funnelshift_l(l, h, 11 - S) & ((0x80000000u >> S) - 1u)) | (0x80000000u >> S), l << (11 - S),
                ((h >> 20) & 0x7ffu) | (h & 0x80000000u)};
    }
    static __device__ __forceinline__ Term mul(const Sig& a, const Sig& b) {   // sig<2> by sig<1>
        const unsigned long long t = (unsigned long long)a.hi * b.lo + 0x40000000ull + (unsigned long long)a.lo * b.hi;
        return {(unsigned long long)a.hi * b.hi + (t >> 32), a.es + b.es};     // the signs add without carry
    }
    static __device__ __forceinline__ Term term(const Sig& b) {   // sig<1>, times one
        return {(((unsigned long long)b.hi << 32) | b.lo) >> 3, b.es + 1023u};
    }
    template <int N>
    static __device__ __forceinline__ double sum(const Term (&t)[N], int terms = N) {   // terms: those that are not zero
        int top = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) top = max(top, (int)(t[k].es & 0x7fffffffu));
        long long v = terms >> 1;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const unsigned long long r = shr64(t[k].r, (unsigned)(top - (int)(t[k].es & 0x7fffffffu)));
            v += (long long)r ^ (long long)((int)t[k].es >> 31);
        }
        if (N == 4 && terms == 3) v |= 1;   // half a unit, and no ties
        const long long neg = v >> 63;
        const unsigned long long m = (unsigned long long)((v ^ neg) - neg);
        const int z = __clzll((long long)m);
        return top - 1019 - z < 1 || m == 0 ? 0.0 : round64<N != 3>(m, z, top - 1019, (unsigned)neg & 0x80000000u);
    }
};

// The same collision in FP64, arranged for the fewest FP64 instructions (the pipe takes one warp
// instruction per 16 cycles and SM, so their number is the time: D2Q9 about 320 -> 190 a node,
// D3Q27 about 860 -> 430 with the two passes below).
//   - every per-axis factor is carried as twice its value (Psi_{+-1} = P +- xi, Psi_0 = 2 - 2 P),
//     and 1/8 (D2Q9: 1/4) goes into the density factors;
//   - the rates are written over P = rho T: w = 2 P / (2 mu + P), w1 = 2 Pr P / (2 mu + Pr P),
//     (2 - w) / (2 rho w) = mu / (rho P), three reciprocals;
//   - mu(T) by pow_pos.
// With u = 0 the factors of opposite directions are equal bit for bit, as in Relax: a gas at
// rest stays at rest exactly.
template <int D, bool CAL>
struct Relax<D, double, false, CAL> {
    using R = double;
    double omw, omw1;
    double X[3], wY[3], Z[3];                 // 2 Psi(u, T + u^2 + k D); wY with the density factor
    double gx[3], ax[3], A[3], B[3], gz[3], sz[3];
    double hq[3];                             // (omega - omega_1)/2 (q* - q^eq)

    static __device__ __forceinline__ void phi2(double u, double P, double out[3]) {
        out[0] = P - u;
        out[1] = fma(-2.0, P, 2.0);
        out[2] = P + u;
    }
    // q* - q^eq without its derivative part: u . (P - rho T I - rho u u)
    static __device__ __forceinline__ void flux(const Moments<double>& m, double dq[3]) {
        const double P = m.rho * m.T, jx = m.rho * m.ux, jy = m.rho * m.uy;
        const double dxx = fma(-jx, m.ux, m.Pxx - P), dyy = fma(-jy, m.uy, m.Pyy - P), dxy = fma(-jx, m.uy, m.Pxy);
        dq[0] = fma(m.uy, dxy, m.ux * dxx);
        dq[1] = fma(m.uy, dyy, m.ux * dxy);
        dq[2] = 0.0;
        if (D == 3) {
            const double jz = m.rho * m.uz;
            const double dxz = fma(-jx, m.uz, m.Pxz), dyz = fma(-jy, m.uz, m.Pyz), dzz = fma(-jz, m.uz, m.Pzz - P);
            dq[0] = fma(m.uz, dxz, dq[0]);
            dq[1] = fma(m.uz, dyz, dq[1]);
            dq[2] = fma(m.uz, dzz, fma(m.uy, dyz, m.ux * dxz));
        }
    }
    __device__ __forceinline__ void init(const Moments<double>& m, double Dx, double Dy, double Dz, const KParams& p) {
        double dq[3];
        flux(m, dq);
        init(m.rho, m.T, m.ux, m.uy, m.uz, dq, Dx, Dy, Dz, p);
    }
    // k = (2 - w)/(2 rho w), 1 - w, 1 - w1, the density factors of f^ex and g^eq (w and w1 times
    // rho over the scale of the doubled factors) and (w - w1)/2
    static __device__ __forceinline__ void rates(double rho, double T, const KParams& p, double& k, double& omw,
                                                 double& omw1, double& wr, double& w1r, double& h) {
        double mu = p.mu0;
        if (p.powlaw) mu *= pow_pos(T * p.d_invT0, p.mu_exp);
        const double P = rho * T, PrP = p.Pr * P;
        const double t = P * recip(fma(2.0, mu, P)), t1 = PrP * recip(fma(2.0, mu, PrP));   // w/2, w1/2
        k = mu * recip(rho * P);
        omw = fma(-2.0, t, 1.0);
        omw1 = fma(-2.0, t1, 1.0);
        const double rs = (D == 3 ? 0.25 : 0.5) * rho;
        wr = t * rs;
        w1r = t1 * rs;
        h = t - t1;
    }
    __device__ __forceinline__ void init(double rho, double T, double ux, double uy, double uz, const double dq[3],
                                         double Dx, double Dy, double Dz, const KParams& p) {
        double k, wr, w1r, h;
        rates(rho, T, p, k, omw, omw1, wr, w1r, h);
        const double T25 = 2.5 * T, TT = T * T;
        double Y[3], sx[3], gy[3], sy[3];
        axis(ux, T, T25, TT, k, Dx, X, gx, sx);
        axis(uy, T, T25, TT, k, Dy, Y, gy, sy);
        if (D == 3) {
            axis(uz, T, T25, TT, k, Dz, Z, gz, sz);
        }
        const double U = U_of_T<double, CAL>(T, p);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ax[a] = fma(U, gx[a], sx[a]);
            wY[a] = wr * Y[a];
            A[a] = w1r * gy[a];
            B[a] = w1r * sy[a];
        }
        hq[0] = h * fma(ux, 0.5 * Dx, dq[0]);
        hq[1] = h * fma(uy, 0.5 * Dy, dq[1]);
        hq[2] = D == 3 ? h * fma(uz, 0.5 * Dz, dq[2]) : 0.0;
    }
    // factors of one axis: 2 Psi of f^ex, 2 phi and 2 psi of g^eq (gfactors)
    static __device__ __forceinline__ void axis(double u, double T, double T25, double TT, double k, double Da,
                                                double F[3], double phi[3], double ps[3]) {
        const double u2 = u * u, P = T + u2;
        phi2(u, fma(k, Da, P), F);
        phi2(u, P, phi);
        psi2(u, u2, T, T25, TT, ps);
    }
    static __device__ __forceinline__ void psi2(double u, double u2, double T, double T25, double TT, double ps[3]) {
        const double o = u * fma(0.5, u2, T), s = fma(u2, fma(0.5, u2, T25), TT);
        ps[0] = s - o;
        ps[1] = fma(-2.0, s, u2);
        ps[2] = s + o;
    }
    // f and g of all directions with the products in integers (in(i, f, g) loads, out(i, f, g)
    // stores); usable: every factor is finite and moderate.  A direction's f takes two FP64
    // instructions or some 55 integer ones, g three or four or some 80: all in integers D2Q9 keeps the FP64
    // pipe 80 % busy (1680 x 1440: 765 us a step all FP64, 644 with g, 580 with both), on D3Q27 a
    // third of f stays FP64 (128^3: 1330; g 1122, a third of f too 1115, two thirds 1070, all 1129; that
    // was with floors, whose sign the mass followed: with the present roundings 1680 x 1440 588, 128^3 1197).
    __device__ __forceinline__ bool usable() const {
        int top = 0;
        auto see = [&](double x) { top = max(top, __double2hiint(x) & 0x7fffffff); };
        see(omw);
        see(omw1);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            see(X[a]);
            see(wY[a]);
            see(gx[a]);
            see(ax[a]);
            see(A[a]);
            see(B[a]);
            see(hq[a]);
            if (D == 3) {
                see(Z[a]);
                see(gz[a]);
                see(sz[a]);
            }
        }
        return top < (1023 + 200) << 20;
    }
    template <class In, class Out>
    __device__ __forceinline__ void all(In in, Out out) const {
        using FP = FixedProd;
        const FP::Sig o = FP::sig<2>(omw), o1 = FP::sig<2>(omw1);
        FP::Sig x[3], s[3], h[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            x[a] = FP::sig<2>(X[a]);
            s[a] = FP::sig<2>(ax[a]);
            h[a] = FP::sig<2>(gx[a]);
        }
#pragma unroll
        for (int bc = 0; bc < (D == 3 ? 9 : 3); ++bc) {
            const int b = bc % 3, c = bc / 3;
            const double yzd = D == 3 ? wY[b] * Z[c] : wY[b];
            const FP::Sig yz = FP::sig<1>(yzd), q1 = FP::sig<1>(D == 3 ? A[b] * gz[c] : A[b]),
                          q2 = FP::sig<1>(D == 3 ? fma(A[b], sz[c], B[b] * gz[c]) : B[b]);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int i = a + 3 * bc;
                double f, g;
                in(i, f, g);
                const FP::Term tf[2] = {FP::mul(o, FP::sig<1>(f)), FP::mul(x[a], yz)};
                const FP::Term g0 = FP::mul(o1, FP::sig<1>(g)), g1 = FP::mul(s[a], q1), g2 = FP::mul(h[a], q2);
                f = (D == 2 || a != 1) ? FP::sum(tf) : fma(omw, f, X[a] * yzd);
                const int cx = cx_of(i), cy = cy_of(i), cz = cz_of<D>(i);
                if (cx * cx + cy * cy + cz * cz == 1) {
                    FP::Sig q = FP::sig<1>(cx != 0 ? hq[0] : (cy != 0 ? hq[1] : hq[2]));
                    if (cx + cy + cz > 0) q.es ^= 0x80000000u;
                    if ((q.es & 0x7fffffffu) == 0u) q.es = 0u;   // no unit for the sign of a zero
                    const FP::Term tg[4] = {g0, g1, g2, FP::term(q)};
                    g = FP::sum(tg, q.es ? 4 : 3);
                } else {
                    const FP::Term tg[3] = {g0, g1, g2};
                    g = FP::sum(tg);
                }
                out(i, f, g);
            }
        }
    }
    // i is a compile-time constant after unrolling; the row products are common subexpressions
    __device__ __forceinline__ double f(int i, double fi, const KParams&) const {
        const int a = i % 3, b = (i / 3) % 3, c = i / 9;
        const double yz = D == 3 ? wY[b] * Z[c] : wY[b];
        return fma(omw, fi, X[a] * yz);
    }
    __device__ __forceinline__ double g(int i, double gi, const KParams&) const {
        const int a = i % 3, b = (i / 3) % 3, c = i / 9;
        const double q1 = D == 3 ? A[b] * gz[c] : A[b];
        const double q2 = D == 3 ? fma(A[b], sz[c], B[b] * gz[c]) : B[b];
        double v = fma(omw1, gi, fma(ax[a], q1, gx[a] * q2));
        const int cx = cx_of(i), cy = cy_of(i), cz = cz_of<D>(i);
        if (cx * cx + cy * cy + cz * cz == 1) {
            const double q = cx != 0 ? hq[0] : (cy != 0 ? hq[1] : hq[2]);
            v = cx + cy + cz < 0 ? v + q : v - q;
        }
        return v;
    }
};

// One collision in place on the raw stored values f, g.
template <int D, typename R, bool DEV, bool CAL = true>
__device__ __forceinline__ void collide(R* f, R* g, const Moments<R>& m, R Dx, R Dy, R Dz,
                                        const KParams& p) {
    Relax<D, R, DEV, CAL> r;
    r.init(m, Dx, Dy, Dz, p);
#pragma unroll
    for (int i = 0; i < Lat<D>::Q; ++i) {
        f[i] = r.f(i, f[i], p);
        g[i] = r.g(i, g[i], p);
    }
}

}  // namespace elbm
