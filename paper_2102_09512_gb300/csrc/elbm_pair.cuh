// Arithmetic of TWO neighbouring nodes of a 16-bit deviation store on D2Q9 in one thread, as two-lane
// FP32 instructions (FADD2/FMUL2/FFMA2, sm_100 and later): lane .x is the node at x, lane .y the
// one at x + 1.  The march of these stores is bound by instruction issue, and these halve the
// arithmetic's instructions; conversions stay one instruction a value.
//
// Every operation is written out with the rounding that it has where a thread marches one node
// (node_moments_stored, Relax, with the products that the compiler fuses there), so a node's new
// pairs are the same bits in either form: an FP32 last bit more or less is now and then one of the
// 16-bit store (formulas arranged for fewer instructions moved 7 % of the values of 4096^2 nodes in 8 steps, rel.
// 4.8e-4).  4096^2, FP16, us a step: one node a thread 309, arranged 254, this 262.
#pragma once

#include "elbm_node.cuh"

namespace elbm {

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 div2(float2 a, float2 b) { return make_float2(qdiv(a.x, b.x), qdiv(a.y, b.y)); }

struct MomentsPair {
    float2 rho, ux, uy, T, rE;
    float2 Pxx, Pyy, Pxy;
};

// Moments of both nodes from the stored pairs: pair(i, k) is the stored (f_i, g_i) of node k.  The
// sums over c_x take one converted component and mixed-precision additions, as
// node_moments_stored; the rest runs on both nodes at once.  ALT: of u^2 = u_x^2 + u_y^2 the other
// square is rounded by itself.
template <int ST, bool CAL, bool ALT, class Pair>
__device__ __forceinline__ void node_moments_pair(Pair pair, const KParams& p, MomentsPair& m) {
    using Cd = Codec<ST>;
    float2 t[3], d[3], e[3], gr[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int i0 = 3 * b;
        float v[2][4];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const auto lo = pair(i0, k), mid = pair(i0 + 1, k), hi = pair(i0 + 2, k);
            const float lo32 = Cd::f32(lo, 0);
            v[k][0] = Cd::add(hi, 0, lo32);
            v[k][1] = Cd::sub(hi, 0, lo32);
            v[k][2] = Cd::add(mid, 0, v[k][0]);
            v[k][3] = Cd::add(hi, 1, Cd::add(mid, 1, Cd::f32(lo, 1)));
        }
        e[b] = make_float2(v[0][0], v[1][0]);
        d[b] = make_float2(v[0][1], v[1][1]);
        t[b] = make_float2(v[0][2], v[1][2]);
        gr[b] = make_float2(v[0][3], v[1][3]);
    }
    m.rho = add2(add2(add2(t[0], t[2]), t[1]), both(p.rest_rho));
    m.Pyy = add2(add2(t[2], t[0]), both(p.rest_Pyy));
    m.Pxx = add2(add2(add2(e[0], e[2]), e[1]), both(p.rest_Pxx));
    m.Pxy = sub2(d[2], d[0]);
    m.rE = add2(add2(add2(gr[0], gr[2]), gr[1]), both(p.rest_E));
    const float2 jx = add2(add2(d[0], d[2]), d[1]), jy = sub2(t[2], t[0]);
    const float2 inv = div2(both(1.f), m.rho);
    m.ux = mul2(jx, inv);
    m.uy = mul2(jy, inv);
    const float2 u2 = ALT ? fma2(m.uy, m.uy, mul2(m.ux, m.ux)) : fma2(m.ux, m.ux, mul2(m.uy, m.uy));
    const float2 U = fma2(m.rE, inv, mul2(both(-0.5f), u2));
    if (CAL) m.T = make_float2(T_of_U<float, true>(U.x, p), T_of_U<float, true>(U.y, p));
    else m.T = mul2(U, both(p.f_gm1));
}

// Q~_aaa = rho u_a (1 - 3 T - u_a^2); c = 1 - 3 T.  ALT: u_a^2 is rounded by itself.
__device__ __forceinline__ float2 anomaly_c(float2 T) { return fma2(both(-3.f), T, both(1.f)); }
template <bool ALT>
__device__ __forceinline__ float2 anomaly2(float2 rho, float2 u, float2 c) {
    return mul2(mul2(rho, u), ALT ? sub2(c, mul2(u, u)) : fma2(neg2(u), u, c));
}
// As dQ, lane by lane.
__device__ __forceinline__ float2 dQ2(int deriv, float2 u, float2 qm, float2 q0, float2 qp) {
    return make_float2(dQ<float>(deriv, u.x, qm.x, q0.x, qp.x), dQ<float>(deriv, u.y, qm.y, q0.y, qp.y));
}

// w, w1 and k = (2 - w)/(2 rho w)
__device__ __forceinline__ void pair_rates(float2 rho, float2 T, float2 mu, const KParams& p, float2& w, float2& w1, float2& k) {
    const float2 two = both(2.f), P = mul2(rho, T);
    w = div2(mul2(two, P), fma2(two, mu, P));
    const float2 w2 = sub2(two, w);
    w1 = div2(mul2(both(2.f * p.f_Pr), w), fma2(both(p.f_Pr), w, w2));
    k = div2(w2, mul2(mul2(two, rho), w));
}
// Twice the factors of one axis: F of f^ex, phi and ps of g^eq.  (Powers of two move through every
// product exactly; the density factors take them back.)
__device__ __forceinline__ void pair_axis(float2 u, float2 T, float2 k, float2 Da, float2 F[3], float2 phi[3], float2 ps[3]) {
    const float2 u2 = mul2(u, u), P = add2(T, u2), Pe = fma2(k, Da, P), m2 = both(-2.f), two = both(2.f);
    F[0] = sub2(Pe, u);
    F[1] = fma2(m2, Pe, two);
    F[2] = add2(Pe, u);
    phi[0] = sub2(P, u);
    phi[1] = fma2(m2, P, two);
    phi[2] = add2(P, u);
    const float2 hu = mul2(both(0.5f), u2);
    const float2 o = fma2(T, u, mul2(hu, u));
    const float2 s = fma2(hu, u2, fma2(T, T, mul2(mul2(both(2.5f), T), u2)));
    ps[0] = sub2(s, o);
    ps[1] = fma2(m2, s, u2);
    ps[2] = add2(s, o);
}

// The collision of both nodes: Relax in its deviation form.
template <bool CAL>
struct RelaxPair {
    float2 omw, omw1, nw, nw1;                  // 1 - w, 1 - w1, -w, -w1
    float2 X[3], wY[3];                         // twice the factors of f^ex, wY with the density factor
    float2 gx[3], ax[3], A[3], B[3];
    float2 hq[2];                               // (omega - omega_1)/2 (q* - q^eq)

    __device__ __forceinline__ void init(const MomentsPair& m, float2 Dx, float2 Dy, const KParams& p) {
        const float2 rho = m.rho, T = m.T, ux = m.ux, uy = m.uy;
        float2 mu = both(p.f_mu0);
        if (p.powlaw) {
            const float2 t = mul2(T, both(p.f_invT0));
            mu = mul2(mu, make_float2(qpow(t.x, p.f_mu_exp), qpow(t.y, p.f_mu_exp)));
        }
        float2 w, w1, k;
        pair_rates(rho, T, mu, p, w, w1, k);
        omw = sub2(both(1.f), w);
        omw1 = sub2(both(1.f), w1);
        nw = neg2(w);
        nw1 = neg2(w1);
        const float2 wr = mul2(mul2(w, rho), both(0.25f)), w1r = mul2(mul2(w1, rho), both(0.25f));
        float2 Y[3], sx[3], gy[3], sy[3];
        pair_axis(ux, T, k, Dx, X, gx, sx);
        pair_axis(uy, T, k, Dy, Y, gy, sy);
        float2 U;
        if (CAL) U = make_float2(U_of_T<float, true>(T.x, p), U_of_T<float, true>(T.y, p));
        else U = mul2(T, both(p.f_Cv));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ax[a] = fma2(U, gx[a], sx[a]);
            wY[a] = mul2(wr, Y[a]);
            A[a] = mul2(w1r, gy[a]);
            B[a] = mul2(w1r, sy[a]);
        }
        // q* - q^eq = u . (P - rho T I - rho u u + div Q~ / 2)
        const float2 P = mul2(rho, T), nrx = neg2(mul2(rho, ux)), nry = neg2(mul2(rho, uy));
        const float2 dxx = fma2(nrx, ux, sub2(m.Pxx, P)), dyy = fma2(nry, uy, sub2(m.Pyy, P)), dxy = fma2(nrx, uy, m.Pxy);
        const float2 qx = fma2(mul2(both(0.5f), ux), Dx, fma2(ux, dxx, mul2(uy, dxy)));
        const float2 qy = fma2(mul2(both(0.5f), uy), Dy, fma2(ux, dxy, mul2(uy, dyy)));
        const float2 h = mul2(both(0.5f), sub2(w, w1));
        hq[0] = mul2(h, qx);
        hq[1] = mul2(h, qy);
    }
    // i is a compile-time constant after unrolling
    __device__ __forceinline__ float2 f(int i, float2 d, const KParams& p) const {
        return fma2(omw, d, fma2(nw, both(p.rest2[i].x), mul2(X[i % 3], wY[i / 3])));
    }
    __device__ __forceinline__ float2 g(int i, float2 d, const KParams& p) const {
        const int a = i % 3, b = i / 3;
        float2 v = fma2(omw1, d, fma2(nw1, both(p.rest2[i].y), fma2(ax[a], A[b], mul2(gx[a], B[b]))));
        if (i == 3) v = add2(v, hq[0]);
        if (i == 5) v = sub2(v, hq[0]);
        if (i == 1) v = add2(v, hq[1]);
        if (i == 7) v = sub2(v, hq[1]);
        return v;
    }
};

}  // namespace elbm
