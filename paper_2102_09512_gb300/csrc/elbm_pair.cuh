// Arithmetic of TWO neighbouring nodes of a 16-bit deviation store in one thread, as two-lane
// FP32 instructions (FADD2/FMUL2/FFMA2, sm_100 and later): lane .x is the node at x, lane .y the
// one at x + 1.  The kernels of the 16-bit stores are bound by instruction issue (ncu: 1250
// instructions a node on D3Q27, 615 on D2Q9), and these halve the arithmetic's; conversions stay
// one instruction a value.
//
// The formulas are those of elbm_node.cuh in the arrangement of its FP64 collision: per-axis
// factors as twice their value, the rates over P = rho T with three reciprocals.
#pragma once

#include "elbm_node.cuh"

namespace elbm {

__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(qdiv(1.f, a.x), qdiv(1.f, a.y)); }

struct MomentsPair {
    float2 rho, ux, uy, uz, T, rE;
    float2 Pxx, Pyy, Pzz, Pxy, Pxz, Pyz;
};

// Moments of both nodes from the stored pairs: pair(i, k) is the stored (f_i, g_i) of node k.  The
// sums over c_x take one converted component and mixed-precision additions, as
// node_moments_stored; the rest runs on both nodes at once.
template <int D, int ST, bool CAL, class Pair>
__device__ __forceinline__ void node_moments_pair(Pair pair, const KParams& p, MomentsPair& m) {
    using Cd = Codec<ST>;
    constexpr int NC = Lat<D>::NC;
    float2 t[3][3], d[3][3], e[3][3], gr[3][3];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int i0 = 3 * b + 9 * c;
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
            e[b][c] = make_float2(v[0][0], v[1][0]);
            d[b][c] = make_float2(v[0][1], v[1][1]);
            t[b][c] = make_float2(v[0][2], v[1][2]);
            gr[b][c] = make_float2(v[0][3], v[1][3]);
        }
    float2 tb[3], db[3], eb[3], gb[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        tb[b] = t[b][0];
        db[b] = d[b][0];
        eb[b] = e[b][0];
        gb[b] = gr[b][0];
        if (D == 3) {
            tb[b] = add2(add2(t[b][0], t[b][2]), t[b][1]);
            db[b] = add2(add2(d[b][0], d[b][2]), d[b][1]);
            eb[b] = add2(add2(e[b][0], e[b][2]), e[b][1]);
            gb[b] = add2(add2(gr[b][0], gr[b][2]), gr[b][1]);
        }
    }
    const float2 yp = add2(tb[0], tb[2]);
    m.rho = add2(add2(yp, tb[1]), both(p.rest_rho));
    m.Pyy = add2(yp, both(p.rest_Pyy));
    m.Pxx = add2(add2(add2(eb[0], eb[2]), eb[1]), both(p.rest_Pxx));
    m.Pxy = sub2(db[2], db[0]);
    m.rE = add2(add2(add2(gb[0], gb[2]), gb[1]), both(p.rest_E));
    const float2 jx = add2(add2(db[0], db[2]), db[1]), jy = sub2(tb[2], tb[0]);
    const float2 inv = rcp2(m.rho);
    m.ux = mul2(jx, inv);
    m.uy = mul2(jy, inv);
    m.uz = both(0.f);
    float2 u2 = fma2(m.uy, m.uy, mul2(m.ux, m.ux));
    if (D == 3) {
        const float2 tzh = add2(add2(t[0][2], t[2][2]), t[1][2]), tzl = add2(add2(t[0][0], t[2][0]), t[1][0]);
        const float2 dzh = add2(add2(d[0][2], d[2][2]), d[1][2]), dzl = add2(add2(d[0][0], d[2][0]), d[1][0]);
        m.uz = mul2(sub2(tzh, tzl), inv);
        m.Pzz = add2(add2(tzh, tzl), both(p.rest_Pzz));
        m.Pxz = sub2(dzh, dzl);
        m.Pyz = sub2(sub2(t[2][2], t[0][2]), sub2(t[2][0], t[0][0]));
        u2 = fma2(m.uz, m.uz, u2);
    }
    const float2 U = fma2(u2, both(-0.5f), mul2(m.rE, inv));
    if (CAL) m.T = make_float2(T_of_U<float, true>(U.x, p), T_of_U<float, true>(U.y, p));
    else m.T = mul2(U, both(p.f_gm1));
}

// Q~_aaa = rho u_a (1 - 3 T - u_a^2); c = 1 - 3 T.
__device__ __forceinline__ float2 anomaly_c(float2 T) { return make_float2(fmaf(-3.f, T.x, 1.f), fmaf(-3.f, T.y, 1.f)); }
template <class V> __device__ __forceinline__ V anomaly2(V rho, V u, V c) {
    return mul2(mul2(rho, u), sub2(c, mul2(u, u)));
}
// As dQ, lane by lane.
__device__ __forceinline__ float2 dQ2(int deriv, float2 u, float2 qm, float2 q0, float2 qp) {
    return make_float2(dQ<float>(deriv, u.x, qm.x, q0.x, qp.x), dQ<float>(deriv, u.y, qm.y, q0.y, qp.y));
}

// The collision of both nodes (as Relax in its deviation form).
template <int D, bool CAL>
struct RelaxPair {
    float2 omw, omw1;                           // 1 - w, 1 - w1
    float2 X[3], wY[3], Z[3];                   // twice the factors of f^ex, wY with the density factor
    float2 gx[3], ax[3], A[3], B[3], gz[3], sz[3];
    float2 hq[3], nhq[3];                       // (omega - omega_1)/2 (q* - q^eq) and its negative
    // -w and -w1 times the rest state's pair: it depends on the number of zero components of c_i alone
    float2 rf[4], rg[4];

    __device__ __forceinline__ void axis(float2 u, float2 T, float2 T25, float2 TT, float2 k, float2 Da, float2 F[3],
                                         float2 phi[3], float2 ps[3]) {
        const float2 u2 = mul2(u, u), P = add2(T, u2), Pe = fma2(k, Da, P);
        F[0] = sub2(Pe, u);
        F[1] = fma2(Pe, both(-2.f), both(2.f));
        F[2] = add2(Pe, u);
        phi[0] = sub2(P, u);
        phi[1] = fma2(P, both(-2.f), both(2.f));
        phi[2] = add2(P, u);
        const float2 o = mul2(u, fma2(u2, both(0.5f), T)), s = fma2(u2, fma2(u2, both(0.5f), T25), TT);
        ps[0] = sub2(s, o);
        ps[1] = fma2(s, both(-2.f), u2);
        ps[2] = add2(s, o);
    }
    __device__ __forceinline__ void init(const MomentsPair& m, float2 Dx, float2 Dy, float2 Dz, const KParams& p) {
        const float2 rho = m.rho, T = m.T, ux = m.ux, uy = m.uy, uz = m.uz;
        float2 mu = both(p.f_mu0);
        if (p.powlaw)
            mu = mul2(mu, make_float2(qpow(T.x * p.f_invT0, p.f_mu_exp), qpow(T.y * p.f_invT0, p.f_mu_exp)));
        const float2 P = mul2(rho, T), PrP = mul2(both(p.f_Pr), P);
        const float2 t = mul2(P, rcp2(fma2(mu, both(2.f), P))), t1 = mul2(PrP, rcp2(fma2(mu, both(2.f), PrP)));
        const float2 k = mul2(mu, rcp2(mul2(rho, P)));
        const float2 mw = mul2(t, both(-2.f)), mw1 = mul2(t1, both(-2.f));
#pragma unroll
        for (int z = 0; z < (D == 3 ? 4 : 3); ++z) {
            constexpr int rep[4] = {0, 1, 4, 13};   // a direction with z zero components
            rf[z] = mul2(mw, both(p.rest2[rep[z]].x));
            rg[z] = mul2(mw1, both(p.rest2[rep[z]].y));
        }
        omw = add2(mw, both(1.f));
        omw1 = add2(mw1, both(1.f));
        const float2 rs = mul2(rho, both(D == 3 ? 0.25f : 0.5f)), wr = mul2(t, rs), w1r = mul2(t1, rs);
        const float2 T25 = mul2(T, both(2.5f)), TT = mul2(T, T);
        float2 Y[3], sx[3], gy[3], sy[3];
        axis(ux, T, T25, TT, k, Dx, X, gx, sx);
        axis(uy, T, T25, TT, k, Dy, Y, gy, sy);
        if (D == 3) axis(uz, T, T25, TT, k, Dz, Z, gz, sz);
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
        const float2 nrho = mul2(rho, both(-1.f)), njx = mul2(nrho, ux), njy = mul2(nrho, uy);
        const float2 dxx = fma2(njx, ux, fma2(Dx, both(0.5f), sub2(m.Pxx, P)));
        const float2 dyy = fma2(njy, uy, fma2(Dy, both(0.5f), sub2(m.Pyy, P)));
        const float2 dxy = fma2(njx, uy, m.Pxy);
        float2 qx = fma2(uy, dxy, mul2(ux, dxx)), qy = fma2(uy, dyy, mul2(ux, dxy));
        const float2 h = sub2(t, t1);
        if (D == 3) {
            const float2 dxz = fma2(njx, uz, m.Pxz), dyz = fma2(njy, uz, m.Pyz);
            const float2 dzz = fma2(mul2(nrho, uz), uz, fma2(Dz, both(0.5f), sub2(m.Pzz, P)));
            qx = fma2(uz, dxz, qx);
            qy = fma2(uz, dyz, qy);
            hq[2] = mul2(h, fma2(uz, dzz, fma2(uy, dyz, mul2(ux, dxz))));
        } else {
            hq[2] = both(0.f);
        }
        hq[0] = mul2(h, qx);
        hq[1] = mul2(h, qy);
#pragma unroll
        for (int a = 0; a < 3; ++a) nhq[a] = mul2(hq[a], both(-1.f));
    }
    static __device__ __forceinline__ constexpr int zeros(int i) {
        return (cx_of(i) == 0) + (cy_of(i) == 0) + (D == 3 && cz_of<D>(i) == 0);
    }
    // i is a compile-time constant after unrolling; the row products are common subexpressions
    __device__ __forceinline__ float2 f(int i, float2 d) const {
        const int a = i % 3, b = (i / 3) % 3, c = i / 9;
        const float2 yz = D == 3 ? mul2(wY[b], Z[c]) : wY[b];
        return fma2(omw, d, fma2(X[a], yz, rf[zeros(i)]));
    }
    __device__ __forceinline__ float2 g(int i, float2 d) const {
        const int a = i % 3, b = (i / 3) % 3, c = i / 9;
        const float2 q1 = D == 3 ? mul2(A[b], gz[c]) : A[b];
        const float2 q2 = D == 3 ? fma2(A[b], sz[c], mul2(B[b], gz[c])) : B[b];
        float2 v = fma2(omw1, d, fma2(ax[a], q1, fma2(gx[a], q2, rg[zeros(i)])));
        const int cx = cx_of(i), cy = cy_of(i), cz = cz_of<D>(i);
        if (cx * cx + cy * cy + cz * cz == 1) {
            const int k = cx != 0 ? 0 : (cy != 0 ? 1 : 2);
            v = add2(v, cx + cy + cz < 0 ? hq[k] : nhq[k]);
        }
        return v;
    }
};

}  // namespace elbm
