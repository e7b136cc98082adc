// far_bary.cuh -- the far-pair Galerkin quadrature in barycentric moments
// (paper Sec. II-B, Eqs. (K), (T), (Z)): the same 7 x 7 point sums as
// far_entries (far_math.cuh) with fewer operations.
//
// With p_j, p'_k the vertices of the two triangles relative to their centroids
// and lambda_j the barycentric coordinates, every entry is linear in the nine
// moments per kernel
//   M_jk = sum_pq w_p w_q lambda_j(p) lambda_k(q) G,   N_jk: the same of g,
// g = -(1 + j k R) G / R^2:
//   T: sum_jk M_jk [(p_j - p_a).(p'_k - p'_b) - 4/k^2]
//        = X - Y_a - Z_b + (D_ab - 4/k^2) M0,   D_jk = p_j . p'_k,
//   K: sum_jk N_jk (p_j - p_a).(d x (p'_k - p'_b)),  d = r - r',
// and in K only d's part e_ab between the vertices a and b survives, the terms
// j = a or k = b vanish, and e_ab.((p'_k - p'_b) x (p_j - p_a)) is the same for
// both ends of an edge: nine reals t_ik (edge i of one triangle, k of the other)
// serve all entries.  The 7-point rule's two orbits put their points at
// multiples of the vertices, so the trial points come from nine reals and the
// inner sums cost two multiply-adds per point.
//
// Bound: the FMA pipe, with the special-function unit close behind (five
// evaluations per point pair).  FP32 runs the two media as one packed pair
// (fma.rn.f32x2), which leaves issue slots for the latter: about 3.9e3 FMA-pipe
// cycles and 3.2e3 issue slots per 32 pairs against 4.9e3 of both before.  In FP64
// the pipe is the bound and the shorter sums are the gain.  Far pairs of the
// 9216-unknown cube by themselves 1.2 -> 0.8 ms, with the near pairs beside them
// 2.15 -> 1.80 ms (1.51 with the near pairs' present form); FP64, 2304 unknowns: 4.8 -> 3.4 ms.
#pragma once

#include "far_math.cuh"

namespace cbfm {
namespace fm {


// a pair of values, one per medium
struct PF {
    unsigned long long v;
};
struct PD {
    double a, b;
};
template <typename T> struct PairOf;
template <> struct PairOf<float> { using type = PF; };
template <> struct PairOf<double> { using type = PD; };

__device__ __forceinline__ PF pmk(float a, float b) {
    PF r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ PD pmk(double a, double b) { return PD{a, b}; }
__device__ __forceinline__ float plo(PF x) {
    float a;
    asm("{\n .reg .f32 t;\n mov.b64 {%0, t}, %1;\n}" : "=f"(a) : "l"(x.v));
    return a;
}
__device__ __forceinline__ float phi(PF x) {
    float b;
    asm("{\n .reg .f32 t;\n mov.b64 {t, %0}, %1;\n}" : "=f"(b) : "l"(x.v));
    return b;
}
__device__ __forceinline__ double plo(PD x) { return x.a; }
__device__ __forceinline__ double phi(PD x) { return x.b; }
__device__ __forceinline__ PF pfma(PF a, PF b, PF c) {
    PF r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ PF pmul(PF a, PF b) {
    PF r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ PF padd(PF a, PF b) {
    PF r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ PD pfma(PD a, PD b, PD c) { return PD{fma(a.a, b.a, c.a), fma(a.b, b.b, c.b)}; }
__device__ __forceinline__ PD pmul(PD a, PD b) { return PD{a.a * b.a, a.b * b.b}; }
__device__ __forceinline__ PD padd(PD a, PD b) { return PD{a.a + b.a, a.b + b.b}; }

// sine and cosine of both media's k R: FP32 with the two-term reduction of
// sincos_red (common.cuh) on the pair
__device__ __forceinline__ void psincos(PF x, PF &s, PF &c) {
    const PF n = padd(pfma(x, pmk(0.159154943091895335768883763372514362f, 0.159154943091895335768883763372514362f),
                           pmk(12582912.0f, 12582912.0f)),
                      pmk(-12582912.0f, -12582912.0f));
    PF r = pfma(n, pmk(-6.28318548202514648437500f, -6.28318548202514648437500f), x);
    r = pfma(n, pmk(1.7484555314695172e-7f, 1.7484555314695172e-7f), r);
    float s0, c0, s1, c1;
    __sincosf(plo(r), &s0, &c0);
    __sincosf(phi(r), &s1, &c1);
    s = pmk(s0, s1);
    c = pmk(c0, c1);
}
__device__ __forceinline__ void psincos(PD x, PD &s, PD &c) {
    f64::sincos64(x.a, &s.a, &c.a);
    f64::sincos64(x.b, &s.b, &c.b);
}
__device__ __forceinline__ float brsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double brsqrt(double x) { return f64::rsqrt64(x); }

// The rule of k_geom.cu: centroid (weight 9/40) and the orbits (a, b, b),
// b = (6 -/+ sqrt 15)/21, weights (155 -/+ sqrt 15)/1200.
constexpr double Q7_S15 = 3.87298334620741688517926539978;
constexpr double Q7_B1 = (6.0 - Q7_S15) / 21.0, Q7_B2 = (6.0 + Q7_S15) / 21.0;
constexpr double Q7_W0 = 9.0 / 40.0, Q7_W1 = (155.0 - Q7_S15) / 1200.0, Q7_W2 = (155.0 + Q7_S15) / 1200.0;

// barycentric coordinates of point p, plain and weighted; per orbit: distance factor T, weight times b, weight times T
template <typename T>
struct Q7Tab {
    T l[7][3], wl[7][3], orb[2][3];
};
template <typename T>
constexpr Q7Tab<T> q7_tab() {
    Q7Tab<T> t{};
    for (int p = 0; p < 7; ++p)
        for (int j = 0; j < 3; ++j) {
            const int o = p == 0 ? 0 : p < 4 ? 1 : 2, k = p == 0 ? -1 : (p - 1) % 3;
            const double b = o == 1 ? Q7_B1 : Q7_B2, w = o == 0 ? Q7_W0 : o == 1 ? Q7_W1 : Q7_W2;
            const double l = o == 0 ? 1.0 / 3.0 : j == k ? 1.0 - 2.0 * b : b;
            t.l[p][j] = (T)l;
            t.wl[p][j] = (T)(w * l);
        }
    for (int o = 0; o < 2; ++o) {
        const double b = o == 0 ? Q7_B1 : Q7_B2, w = o == 0 ? Q7_W1 : Q7_W2;
        t.orb[o][0] = (T)(1.0 - 3.0 * b);
        t.orb[o][1] = (T)(w * b);
        t.orb[o][2] = (T)(w * (1.0 - 3.0 * b));
    }
    return t;
}
static __constant__ Q7Tab<float> q7f = q7_tab<float>();
static __constant__ Q7Tab<double> q7d = q7_tab<double>();
template <typename T> __device__ __forceinline__ const Q7Tab<T> &q7();
template <> __device__ __forceinline__ const Q7Tab<float> &q7<float>() { return q7f; }
template <> __device__ __forceinline__ const Q7Tab<double> &q7<double>() { return q7d; }

// Near test of far records rt, rs (is_near_t's), leaving the centroid difference in dc.
template <typename T>
__device__ __forceinline__ bool is_near_b(const T *rt, const T *rs, const double *rt64, const double *rs64,
                                          const int32_t *vt, const int32_t *vs, double alpha, T dc[3]) {
    T d2 = 0;
    for (int d = 0; d < 3; ++d) {
        dc[d] = rt[FB_CEN + d] - rs[FB_CEN + d];
        if constexpr (sizeof(T) == 4) dc[d] += rt[FB_CLO + d] - rs[FB_CLO + d];
        d2 += dc[d] * dc[d];
    }
    if (shares_vertex(vt, vs)) return true;
    const T thr = (T)alpha * (rt[FB_H] > rs[FB_H] ? rt[FB_H] : rs[FB_H]), thr2 = thr * thr;
    if (d2 < thr2 * (T)(1.0 - 1e-5)) return true;
    if (d2 > thr2 * (T)(1.0 + 1e-5)) return false;
    return is_near(rt64, rs64, vt, vs, alpha);
}

// The 27 local entries (op x 3 x 3, op = Ks, Ta, Tb) of a far pair: pt, ps the
// vertices of the test and trial triangle relative to their centroids, at, as
// the coefficients c_a times the area, dc the centroid difference.  ROLL keeps the
// two orbits in one loop body (fewer instructions to fetch, a few more to execute):
// the FP32 far kernel is faster without (0.85 against 0.96 ms on the 9216-unknown
// cube), FP64 (3.37 against 3.44 ms) and the fused kernel, whose warps run in
// different places of a longer program (31 against 38 ms), with it.
template <typename T, bool ROLL>
__device__ __forceinline__ void far_bary(const T *pt, const T *at, const T *ps, const T *as, const T dc[3],
                                         const MediaT<T> &md, cx<T> *out) {
    using P = typename PairOf<T>::type;
    const bool lossy2 = md.ki[1] != (T)0;
    const P kk = pmk(md.kr[0], md.kr[1]), nk = pmk(-md.kr[0], -md.kr[1]);
    P M[4][3][3];   // Re G, -Im G, -Re g, Im g
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) M[x][j][k] = pmk((T)0, (T)0);
    const Q7Tab<T> &tab = q7<T>();
#pragma unroll 1
    for (int p = 0; p < 7; ++p) {
        T Dp[3];
#pragma unroll
        for (int d = 0; d < 3; ++d)
            Dp[d] = dc[d] + (tab.l[p][0] * pt[d] + tab.l[p][1] * pt[3 + d] + tab.l[p][2] * pt[6 + d]);
        P U[4][3], S[4];   // sums of w G lambda_k, w g lambda_k; the part common to the three k
        auto point = [&](const T d[3], P G[4]) {
            const T R2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
            const T iR = brsqrt(R2), R = R2 * iR, h = iR * iR;
            const P RR = pmk(R, R), hh = pmk(h, h);
            const P kR = pmul(RR, kk), nkR = pmul(RR, nk);
            P sn, cs;
            psincos(kR, sn, cs);
            if (lossy2) {
                const P aa = pmk(iR, iR * exp_t(md.ki[1] * R));
                const P o = pmk((T)1, (T)1 - md.ki[1] * R);
                G[0] = pmul(aa, cs);
                G[1] = pmul(aa, sn);
                G[2] = pmul(hh, pfma(kR, G[1], pmul(o, G[0])));
                G[3] = pmul(hh, pfma(nkR, G[0], pmul(o, G[1])));
            } else {
                const P aa = pmk(iR, iR);
                G[0] = pmul(aa, cs);
                G[1] = pmul(aa, sn);
                G[2] = pmul(hh, pfma(kR, G[1], G[0]));
                G[3] = pmul(hh, pfma(nkR, G[0], G[1]));
            }
        };
        {
            P G[4];
            point(Dp, G);
            const P wc = pmk((T)(Q7_W0 / 3.0), (T)(Q7_W0 / 3.0));
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                S[x] = pmul(wc, G[x]);
                U[x][0] = U[x][1] = U[x][2] = pmk((T)0, (T)0);
            }
        }
        // ROLL: the two orbits share one body
#pragma unroll(ROLL ? 1 : 2)
        for (int o = 0; o < 2; ++o) {
            const T tau = ROLL ? tab.orb[o][0] : (T)(1.0 - 3.0 * (o == 0 ? Q7_B1 : Q7_B2));
            const T wcs = ROLL ? tab.orb[o][1] : (T)(o == 0 ? Q7_W1 * Q7_B1 : Q7_W2 * Q7_B2);
            const T wks = ROLL ? tab.orb[o][2] : (T)(o == 0 ? Q7_W1 * (1.0 - 3.0 * Q7_B1) : Q7_W2 * (1.0 - 3.0 * Q7_B2));
            const P wc = pmk(wcs, wcs), wk = pmk(wks, wks);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                P G[4];
                const T d[3] = {Dp[0] - tau * ps[3 * k], Dp[1] - tau * ps[3 * k + 1], Dp[2] - tau * ps[3 * k + 2]};
                point(d, G);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    S[x] = pfma(wc, G[x], S[x]);
                    U[x][k] = !ROLL && o == 0 ? pmul(wk, G[x]) : pfma(wk, G[x], U[x][k]);
                }
            }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int k = 0; k < 3; ++k) U[x][k] = padd(U[x][k], S[x]);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const T wl = tab.wl[p][j];
            const P w2 = pmk(wl, wl);
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int k = 0; k < 3; ++k) M[x][j][k] = pfma(w2, U[x][k], M[x][j][k]);
        }
    }
    const T inv4pi = (T)(1.0 / (4.0 * PI));
    T cc[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) cc[a][b] = at[a] * as[b] * inv4pi;
    // ---- K, both media together
    {
        T t[3][3];   // t_ik = (dc + p_i - p'_k).(S_k x T_i), T_i = p_{i+1} - p_i, S_k = p'_{k+1} - p'_k
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            T Ti[3], ei[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                Ti[d] = pt[3 * ((i + 1) % 3) + d] - pt[3 * i + d];
                ei[d] = dc[d] + pt[3 * i + d];
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                T s[3], e[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    s[d] = ps[3 * ((k + 1) % 3) + d] - ps[3 * k + d];
                    e[d] = ei[d] - ps[3 * k + d];
                }
                t[i][k] = e[0] * (s[1] * Ti[2] - s[2] * Ti[1]) + e[1] * (s[2] * Ti[0] - s[0] * Ti[2]) +
                          e[2] * (s[0] * Ti[1] - s[1] * Ti[0]);
            }
        }
        T nr[3][3], ni[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                nr[j][k] = -(plo(M[2][j][k]) + phi(M[2][j][k]));
                ni[j][k] = plo(M[3][j][k]) + phi(M[3][j][k]);
            }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const int a1 = (a + 1) % 3, a2 = (a + 2) % 3, b1 = (b + 1) % 3, b2 = (b + 2) % 3;
                const T kr = t[a][b] * nr[a1][b1] - t[a][b2] * nr[a1][b2] - t[a2][b] * nr[a2][b1] + t[a2][b2] * nr[a2][b2];
                const T ki = t[a][b] * ni[a1][b1] - t[a][b2] * ni[a1][b2] - t[a2][b] * ni[a2][b1] + t[a2][b2] * ni[a2][b2];
                out[3 * a + b] = cx<T>(cc[a][b] * kr, cc[a][b] * ki);
            }
    }
    // ---- T: X, Y_a, Z_b, M0 per medium, then the weights -j k (-eta) and -j k / eta
    {
        T D[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                D[j][k] = pt[3 * j] * ps[3 * k] + pt[3 * j + 1] * ps[3 * k + 1] + pt[3 * j + 2] * ps[3 * k + 2];
        P q[2][8];   // [re, -im][X, Y_0..2, Z_0..2, M0]
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            P r[3], c[3], X = pmk((T)0, (T)0);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                r[j] = padd(padd(M[x][j][0], M[x][j][1]), M[x][j][2]);
                c[j] = padd(padd(M[x][0][j], M[x][1][j]), M[x][2][j]);
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                P y = pmk((T)0, (T)0), z = y;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const P djk = pmk(D[j][k], D[j][k]);
                    X = pfma(djk, M[x][j][k], X);
                    y = pfma(djk, c[k], y);
                    z = pfma(pmk(D[k][j], D[k][j]), r[k], z);
                }
                q[x][1 + j] = y;
                q[x][4 + j] = z;
            }
            q[x][0] = X;
            q[x][7] = padd(padd(r[0], r[1]), r[2]);
        }
        cx<T> A[8], B[8];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const cx<T> mjk(md.ki[i], -md.kr[i]);
            const cx<T> wa = cx<T>(md.wTar[i], md.wTai[i]) * mjk, wb = cx<T>(md.wTbr[i], md.wTbi[i]) * mjk;
            cx<T> v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = i == 0 ? cx<T>(plo(q[0][u]), -plo(q[1][u])) : cx<T>(phi(q[0][u]), -phi(q[1][u]));
            v[0] -= cx<T>(md.fk2r[i], md.fk2i[i]) * v[7];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (i == 0) {
                    A[u] = wa * v[u];
                    B[u] = wb * v[u];
                } else {
                    cfma(A[u], wa, v[u]);
                    cfma(B[u], wb, v[u]);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const cx<T> xa = A[0] - A[1 + a], xb = B[0] - B[1 + a];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                out[9 + 3 * a + b] = cc[a][b] * (xa - A[4 + b] + D[a][b] * A[7]);
                out[18 + 3 * a + b] = cc[a][b] * (xb - B[4 + b] + D[a][b] * B[7]);
            }
        }
    }
}

}  // namespace fm
}  // namespace cbfm
