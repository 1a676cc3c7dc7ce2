// D3Q19 building blocks: the three-dimensional extension the paper lists as
// future work (Sec. 6), with the method of Sec. 3.1 (Eq. 1 BGK, Eq. 2
// incompressible equilibrium with v = sum f c) on the 19 velocities of
// {-1,0,1}^3 with |c|^2 <= 2, ordered lexicographically in (c_z, c_y, c_x):
// opposite(i) = 18 - i, rest at i = 9, weights 1/3, 1/18 (faces), 1/36 (edges).
#pragma once

#include "lbm_device.cuh"

namespace lbm {
namespace d3 {

constexpr int Q = 19;
constexpr int REST = 9;
constexpr uint32_t SOLID = 0x3FFFFu;  // all 18 pulls bounce: solid (or isolated) node

__host__ __device__ constexpr int cx(int i) {
    return i == 0 || i == 4 || i == 14 || i == 18 ? 0
         : (i == 1 || i == 5 || i == 8 || i == 11 || i == 15) ? -1
         : (i == 3 || i == 7 || i == 10 || i == 13 || i == 17) ? 1 : 0;
}
__host__ __device__ constexpr int cy(int i) {
    return (i == 0 || (i >= 5 && i <= 7) || i == 14) ? -1 : ((i == 4 || (i >= 11 && i <= 13) || i == 18) ? 1 : 0);
}
__host__ __device__ constexpr int cz(int i) { return i <= 4 ? -1 : (i >= 14 ? 1 : 0); }
__host__ __device__ constexpr int opp(int i) { return 18 - i; }
__host__ __device__ constexpr int bit(int i) { return i < REST ? i : i - 1; }
__host__ __device__ constexpr int sq(int i) { return cx(i) * cx(i) + cy(i) * cy(i) + cz(i) * cz(i); }

// Bundles: directions with the same (c_y, c_z) (the same source row), in
// order; first direction and size of the bundle that holds direction i.
__host__ __device__ constexpr int bundle_first(int i) {
    return i == 0 ? 0 : i <= 3 ? 1 : i == 4 ? 4 : i <= 7 ? 5 : i <= 10 ? 8 : i <= 13 ? 11 : i == 14 ? 14 : i <= 17 ? 15 : 18;
}
__host__ __device__ constexpr int bundle_size(int i) { return (i == 0 || i == 4 || i == 14 || i == 18) ? 1 : 3; }

// Element offset of population i of node n (N nodes): stream i N + n,
// collision 19 n + i, bundle first N + size n + (i - first).
template <int L>
__host__ __device__ __forceinline__ int64_t addr(int64_t N, int64_t n, int i) {
    if (L == STREAM) return (int64_t)i * N + n;
    if (L == COLLISION) return n * 19 + i;
    return (int64_t)bundle_first(i) * N + (int64_t)bundle_size(i) * n + (i - bundle_first(i));
}

// Constants of the collision: as in 2-D, one operation order per storage
// class (FP32, FP64, 16-bit).
template <class C> struct Relax3;
template <> struct Relax3<float> {
    float omega;
    float hf[3];        // F/2
    float f[3];         // F
    float cF[Q];        // c_i . F
    float w0, w1, w2;   // 1/3, 1/18, 1/36
    float wl0, wl1, wl2;  // w - (float)w: rounding residuals of the weights
    float kw0, kw1, kw2;  // (1 - omega/2) w
};
template <> struct Relax3<double> {
    double om1, hom;           // 1 - omega, omega/4
    double hf[3], k[3], c[3];  // F/2, (1 - omega/2) F / 2, (1 - omega/2) F / 6
    double o6, o18;            // omega/6, omega/18
};
// T = float or f2 (each value duplicated).
template <class T> struct NarrowRelax3 {
    T nomega;                  // -omega
    T nw[3], nwl[3], kw[3];    // by weight (rest, axis, diagonal): -w, rounded value and residual; (1 - omega/2) w
    T hf[3], f[3], cF[Q];      // F/2, F, c_i . F
    T c45, c9, c3, cm3, cm15, cm1;   // 4.5, 9, 3, -3, -1.5, -1
};

template <class C, bool NARROW> struct Consts3 {
    std::conditional_t<NARROW, NarrowRelax3<C>, Relax3<C>> r;
    int force;            // F != 0
};

// Host: FP64 constants rounded once.
inline void make_relax3(double omega, const double *F, Relax3<float> &k) {
    const double kf = 1.0 - 0.5 * omega;
    k.omega = (float)omega;
    for (int d = 0; d < 3; ++d) {
        k.hf[d] = (float)(0.5 * F[d]);
        k.f[d] = (float)F[d];
    }
    k.w0 = (float)(1.0 / 3.0);
    k.w1 = (float)(1.0 / 18.0);
    k.w2 = (float)(1.0 / 36.0);
    k.wl0 = (float)(1.0 / 3.0 - (double)k.w0);
    k.wl1 = (float)(1.0 / 18.0 - (double)k.w1);
    k.wl2 = (float)(1.0 / 36.0 - (double)k.w2);
    k.kw0 = (float)(kf / 3.0);
    k.kw1 = (float)(kf / 18.0);
    k.kw2 = (float)(kf / 36.0);
    for (int i = 0; i < Q; ++i) k.cF[i] = (float)(cx(i) * F[0] + cy(i) * F[1] + cz(i) * F[2]);
}
inline void make_relax3(double omega, const double *F, Relax3<double> &q) {
    q.om1 = 1.0 - omega;
    const double om = 1.0 - q.om1;
    q.hom = 0.25 * om;
    for (int a = 0; a < 3; ++a) {
        q.hf[a] = 0.5 * F[a];
        q.k[a] = 0.5 * (1.0 - 0.5 * om) * F[a];
        q.c[a] = q.k[a] / 3.0;
    }
    q.o6 = om / 6.0;
    q.o18 = om / 18.0;
}
inline void make_relax3(double omega, const double *F, NarrowRelax3<float> &q) {
    const double w[3] = {1.0 / 3.0, 1.0 / 18.0, 1.0 / 36.0}, per[3] = {3.0, 18.0, 36.0}, kf = 1.0 - 0.5 * omega;
    q.nomega = (float)-omega;
    for (int s = 0; s < 3; ++s) {
        q.nw[s] = (float)-w[s];
        q.nwl[s] = (float)(-w[s] - (double)q.nw[s]);
        q.kw[s] = (float)(kf / per[s]);
        q.hf[s] = (float)(0.5 * F[s]);
        q.f[s] = (float)F[s];
    }
    for (int i = 0; i < Q; ++i) q.cF[i] = (float)(cx(i) * F[0] + cy(i) * F[1] + cz(i) * F[2]);
    q.c45 = 4.5f;
    q.c9 = 9.0f;
    q.c3 = 3.0f;
    q.cm3 = -3.0f;
    q.cm15 = -1.5f;
    q.cm1 = -1.0f;
}

// Moments, Eq. 2 equilibrium (deviation form) and Eq. 1 BGK relaxation with
// the Guo source in the fixed operation order of 32-bit storage:
//   P_i  = drho - 3/2 u^2 + cu_i (3 + 9/2 cu_i),  h*_i = g_i + omega (w_i P_i - g_i)
//          + (1 - omega/2) w_i [cF_i (3 + 9 cu_i) - 3 u.F]
// with cu_i formed from the one or two nonzero components of c_i, and in
// FP32 w_i P_i formed with w_i as the rounded weight plus its residual (the
// rounded weights alone miss sum_i w_i c_i c_i = 1/3 by ~1e-8, which would
// make the relaxation a momentum source proportional to u).
__device__ __forceinline__ void collide3_ops(const Relax3<float> &k, int force, float *g, float &drho, float &ux,
                                             float &uy, float &uz) {
    using C = float;
    using A = Ar<C>;
    C r = g[0];
#pragma unroll
    for (int i = 1; i < Q; ++i) r = A::add(r, g[i]);
    drho = r;
    // momentum: signed sums in direction order, starting from the first term
    C j[3];
    bool started[3] = {false, false, false};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int c[3] = {cx(i), cy(i), cz(i)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!c[a]) continue;
            if (!started[a]) {
                j[a] = c[a] > 0 ? g[i] : -g[i];
                started[a] = true;
            } else {
                j[a] = c[a] > 0 ? A::add(j[a], g[i]) : A::sub(j[a], g[i]);
            }
        }
    }
    ux = A::add(j[0], k.hf[0]);
    uy = A::add(j[1], k.hf[1]);
    uz = A::add(j[2], k.hf[2]);
    const C usq = A::fma(ux, ux, A::fma(uy, uy, A::mul(uz, uz)));
    const C base = A::fma(C(-1.5), usq, drho);
    const C m3uF = A::mul(C(-3), A::fma(ux, k.f[0], A::fma(uy, k.f[1], A::mul(uz, k.f[2]))));
    const C u[3] = {ux, uy, uz};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int c[3] = {cx(i), cy(i), cz(i)};
        C cu = C(0);
        bool any = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!c[a]) continue;
            const C t = c[a] > 0 ? u[a] : -u[a];
            cu = any ? A::add(cu, t) : t;
            any = true;
        }
        const C w = sq(i) == 0 ? k.w0 : (sq(i) == 1 ? k.w1 : k.w2);
        const C P = any ? A::fma(cu, A::fma(C(4.5), cu, C(3)), base) : base;
        C t = A::fma(w, P, -g[i]);
        t = A::fma(sq(i) == 0 ? k.wl0 : (sq(i) == 1 ? k.wl1 : k.wl2), P, t);
        C o = A::fma(k.omega, t, g[i]);
        if (force && any) {
            const C kw = sq(i) == 1 ? k.kw1 : k.kw2;
            o = A::fma(kw, A::fma(k.cF[i], A::fma(C(9), cu, C(3)), m3uF), o);
        } else if (force) {
            o = A::fma(k.kw0, m3uF, o);
        }
        g[i] = o;
    }
}

// 16-bit storage, one node or a packed pair: the update above, written without
// run-time negations as h* = g - omega (g - w P) + ... (t = g - w P), a
// negative first term of a sum being an exact product with -1. 157 operations
// without a force (NF), 215 with one.
template <bool NF, class T>
__device__ __forceinline__ void collide3_narrow(const NarrowRelax3<T> &q, T *g, T &drho, T *u) {
    using A = Op<T>;
    const T cm1 = A::lit(q.cm1, -1.0), cm15 = A::lit(q.cm15, -1.5), c45 = A::lit(q.c45, 4.5), c9 = A::lit(q.c9, 9.0),
            c3 = A::lit(q.c3, 3.0), cm3 = A::lit(q.cm3, -3.0);
    T r = g[0];
#pragma unroll
    for (int i = 1; i < Q; ++i) r = A::add(r, g[i]);
    drho = r;
    // momentum: signed sums in direction order, starting from the first term
    bool started[3] = {false, false, false};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int c[3] = {cx(i), cy(i), cz(i)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!c[a]) continue;
            if (!started[a]) u[a] = c[a] > 0 ? g[i] : A::mul(g[i], cm1);
            else u[a] = c[a] > 0 ? A::add(u[a], g[i]) : A::sub(u[a], g[i]);
            started[a] = true;
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = A::add(u[a], q.hf[a]);
    const T base = A::fma(cm15, A::fma(u[0], u[0], A::fma(u[1], u[1], A::mul(u[2], u[2]))), drho);
    T m3uF = cm3;
    if constexpr (!NF) m3uF = A::mul(cm3, A::fma(u[0], q.f[0], A::fma(u[1], q.f[1], A::mul(u[2], q.f[2]))));
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int c[3] = {cx(i), cy(i), cz(i)};
        T cu = base;
        bool any = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!c[a]) continue;
            if (!any) cu = c[a] > 0 ? u[a] : A::mul(u[a], cm1);
            else cu = c[a] > 0 ? A::add(cu, u[a]) : A::sub(cu, u[a]);
            any = true;
        }
        const int s = sq(i);
        const T P = any ? A::fma(cu, A::fma(c45, cu, c3), base) : base;
        const T t = A::fma(q.nwl[s], P, A::fma(q.nw[s], P, g[i]));   // g - w P
        T o = A::fma(q.nomega, t, g[i]);
        if constexpr (!NF) o = A::fma(q.kw[s], any ? A::fma(q.cF[i], A::fma(c9, cu, c3), m3uF) : m3uF, o);
        g[i] = o;
    }
}

// Density and momentum of the populations (without the force's half) from the
// sums and differences of opposite directions: 39 operations instead of 45.
__device__ __forceinline__ void moments3(const double *g, double &drho, double *u) {
    using A = Ar<double>;
    double r = g[REST];
    bool started[3] = {false, false, false};
#pragma unroll
    for (int i = REST + 1; i < Q; ++i) {
        r = A::add(r, A::add(g[i], g[opp(i)]));
        const double d = A::sub(g[i], g[opp(i)]);
        const int c[3] = {cx(i), cy(i), cz(i)};
        // the first term of each component has c_a = +1 (directions 10, 11, 14)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!c[a]) continue;
            u[a] = !started[a] ? d : (c[a] > 0 ? A::add(u[a], d) : A::sub(u[a], d));
            started[a] = true;
        }
    }
    drho = r;
}

// FP64: h* = (1 - omega) g + H with omega w folded into the shared parts,
//   b = omega/4 u + (1 - omega/2) F/2,  B = omega/18 drho - (b.u)/3,
//   O_a = omega/6 u_a + (1 - omega/2) F_a/6:
// the axis directions take E_a = B + b_a u_a and +-O_a, the rest direction
// 6 B, the diagonal ones of the axes a, e the even part
// (E_a + b_e u_e)/2 +- (b_a u_e + b_e u_a)/2 and (O_a +- O_e)/2: 119
// operations, where it was 216 with and 160 without a force.
__device__ __forceinline__ void collide3_ops64(const Relax3<double> &q, double *g, double &drho, double *u) {
    using A = Ar<double>;
    moments3(g, drho, u);
    double b[3], O[3], E[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = A::add(u[a], q.hf[a]);
        b[a] = A::fma(q.hom, u[a], q.k[a]);
        O[a] = A::fma(q.o6, u[a], q.c[a]);
    }
    const double t = A::fma(b[0], u[0], A::fma(b[1], u[1], A::mul(b[2], u[2])));
    const double B = A::fma(-1.0 / 3.0, t, A::mul(q.o18, drho));
    g[REST] = A::fma(q.om1, g[REST], A::mul(6.0, B));
#pragma unroll
    for (int a = 0; a < 3; ++a) E[a] = A::fma(b[a], u[a], B);
#pragma unroll
    for (int i = REST + 1; i < Q; ++i) {   // axis directions: +x = 10, +y = 12, +z = 16
        if (sq(i) != 1) continue;
        const int a = cx(i) ? 0 : (cy(i) ? 1 : 2);
        g[i] = A::fma(q.om1, g[i], A::add(E[a], O[a]));
        g[opp(i)] = A::fma(q.om1, g[opp(i)], A::sub(E[a], O[a]));
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) {   // pairs of axes a < e: c = (+1, +1) and (+1, -1)
        const int a = m == 2 ? 1 : 0, e = m == 0 ? 1 : 2;
        const double G = A::mul(0.5, A::fma(b[e], u[e], E[a]));
        const double X = A::fma(b[a], u[e], A::mul(b[e], u[a]));
        const double Es = A::fma(0.5, X, G), Ed = A::fma(-0.5, X, G);
        const double os = A::add(O[a], O[e]), od = A::sub(O[a], O[e]);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int c[3] = {cx(i), cy(i), cz(i)};
            if (sq(i) != 2 || c[a] != 1 || c[e] == 0) continue;
            const double Ei = c[e] > 0 ? Es : Ed, Oi = c[e] > 0 ? os : od;
            g[i] = A::fma(q.om1, g[i], A::fma(0.5, Oi, Ei));
            g[opp(i)] = A::fma(q.om1, g[opp(i)], A::fma(-0.5, Oi, Ei));
        }
    }
}

// The collision of a storage class.
template <class C, bool NARROW>
__device__ __forceinline__ void collide3(const Consts3<C, NARROW> &k, C *g, C &drho, C &ux, C &uy, C &uz) {
    if constexpr (NARROW || sizeof(C) == 8) {
        C u[3];
        if constexpr (!NARROW) collide3_ops64(k.r, g, drho, u);
        else if (k.force) collide3_narrow<false>(k.r, g, drho, u);
        else collide3_narrow<true>(k.r, g, drho, u);
        ux = u[0];
        uy = u[1];
        uz = u[2];
    } else {
        collide3_ops(k.r, k.force, g, drho, ux, uy, uz);
    }
}

// Two nodes of 16-bit storage at once: each lane equals the one-node form bit for bit.
__device__ __forceinline__ void collide3_2(const NarrowRelax3<f2> &q, int force, f2 *g, f2 &drho, f2 &ux, f2 &uy,
                                           f2 &uz) {
    f2 u[3];
    if (force) collide3_narrow<false>(q, g, drho, u);
    else collide3_narrow<true>(q, g, drho, u);
    ux = u[0];
    uy = u[1];
    uz = u[2];
}

}  // namespace d3
}  // namespace lbm
