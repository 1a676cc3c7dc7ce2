// Device-side building blocks of the D2Q9I BGK update (PortLBM, Sec. 3):
// direction set, the three population layouts, storage codecs, the pull
// mapping at domain edges, and the collision routine every kernel of a
// storage type calls.
#pragma once

#include <cstdint>
#include <cstring>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <type_traits>

namespace lbm {

enum Layout : int { STREAM = 0, BUNDLE = 1, COLLISION = 2 };
enum Algo : int { LPTL = 0, NPTL = 1, NPOL = 2, NSOL = 3, AA = 4 };
enum Bc : int {
    PERIODIC = 0, WALL = 1, FREESLIP = 2, INLET_ZOUHE = 3, INLET_EQ = 4, OUTFLOW_ZG = 5,
    INLET_EQ_NEUMANN = 6, OUTLET_PRESSURE = 7
};
enum Pull : int { PULL_NODE = 0, PULL_BOUNCE = 1, PULL_UNKNOWN = 2 };

// Per-node link byte: bit b(i) set when the value pulled in direction i is
// bounced back (source solid or a wall edge); 0xFF marks a solid node.
constexpr uint8_t SOLID_LINKS = 0xFF;

// Fig. 2 order: i = 0..8 = SW, S, SE, W, rest, E, NW, N, NE.
__host__ __device__ constexpr int cx(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int cy(int i) { return i / 3 - 1; }
__host__ __device__ constexpr int opp(int i) { return 8 - i; }
__host__ __device__ constexpr int mir_y(int i) { return (i % 3) + 3 * (2 - i / 3); }
__host__ __device__ constexpr int link_bit(int i) { return i < 4 ? i : i - 1; }

// Layouts of Fig. 2 (element offsets, N nodes).
template <int L>
__host__ __device__ __forceinline__ int64_t addr(int64_t N, int64_t n, int i) {
    if (L == STREAM) return (int64_t)i * N + n;
    if (L == COLLISION) return n * 9 + i;
    return (int64_t)(i / 3) * 3 * N + n * 3 + (i % 3);
}

// ------------------------------------------------------------ arithmetic
// Explicitly rounded operations: no contraction or reassociation, so every
// kernel that calls collide() produces the same bits.
template <class C> struct Ar;
template <> struct Ar<float> {
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
};
template <> struct Ar<double> {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
};

// ------------------------------------------------------------ chained launches
// Update kernels are launched so that the next update's blocks may become
// resident, and load what no update writes (node indices, link bytes, case
// records), while the last blocks of this one still run (programmatic
// dependent launch). chain_next() lets the next grid start once every block
// of this one has; chain_wait() returns when the previous grid has completed
// and its stores are visible, and comes before the first access to the
// lattice, the buffer grid, the moments or the update counter.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------ hashing
// 32-bit integer finaliser "lowbias32" (C. Wellons, hash-prospector).
__host__ __device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352dU;
    x ^= x >> 15;
    x *= 0x846ca68bU;
    x ^= x >> 16;
    return x;
}
__host__ __device__ __forceinline__ uint32_t step_key(uint64_t seed, uint32_t t) {
    return mix32((uint32_t)seed ^ mix32((uint32_t)(seed >> 32) ^ mix32(t)));
}
__host__ __device__ __forceinline__ uint32_t node_key(uint32_t skey, uint32_t n) {
    return mix32(n ^ skey);
}
// Random word of population i of a node: the node's hashed key with a
// per-direction constant folded in, multiplied by an odd constant (a
// multiplicative hash); the stochastic rounding below uses its top bits.
__host__ __device__ __forceinline__ uint32_t pop_rand(uint32_t nkey, int i) {
    return (nkey ^ ((uint32_t)i * 0x9E3779B9U)) * 0x85EBCA6BU;
}

// ------------------------------------------------------------ codecs
// Stochastic rounding of FP32 values to 16 bits with the stochastic-rounding
// conversion of the sm_100 family (cvt.rs): a random integer, the top bits of
// the value's random word r (13 for FP16, 16 for BF16), is added to the top
// bits the conversion drops and the sum truncated, so the kept part
// increments exactly when those dropped bits plus the draw carry: away from
// zero with probability (|x| - |lo|) / ulp, lo the value rounded toward zero
// and ulp the gap to the next magnitude. BF16 drops 16 bits and FP16 13 in
// its normal range (|x| >= 2^-14), where this is exact; below 2^-14 FP16
// drops more than 13 bits and the probability is the dropped fraction cut to
// 13 bits (at most 2^-13 ulp low). The packed forms round two values: hi to
// the upper half (its draw in bits 28..16 for FP16, 31..16 for BF16), lo to
// the lower half (bits 12..0, 15..0), each exactly as the one-value form.
__device__ __forceinline__ uint32_t sr_half2(float hi, float lo, uint32_t r_hi, uint32_t r_lo) {
    const uint32_t draw = ((r_hi >> 19) << 16) | (r_lo >> 19);
    uint32_t d;
    asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(draw));
    return d;
}
__device__ __forceinline__ uint32_t sr_bf162(float hi, float lo, uint32_t r_hi, uint32_t r_lo) {
    const uint32_t draw = (r_hi & 0xFFFF0000u) | (r_lo >> 16);
    uint32_t d;
    asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(draw));
    return d;
}
__device__ __forceinline__ __half sr_half(float x, uint32_t r) {
    return __ushort_as_half((unsigned short)(sr_half2(0.0f, x, 0u, r) & 0xFFFFu));
}
__device__ __forceinline__ __nv_bfloat16 sr_bf16(float x, uint32_t r) {
    return __ushort_as_bfloat16((unsigned short)(sr_bf162(0.0f, x, 0u, r) & 0xFFFFu));
}

template <class S> struct Codec;
template <> struct Codec<double> {
    using C = double;
    static constexpr bool narrow = false;
    static __device__ __forceinline__ double dec(double v) { return v; }
    static __device__ __forceinline__ double enc(double v, bool, uint32_t) { return v; }
};
template <> struct Codec<float> {
    using C = float;
    static constexpr bool narrow = false;
    static __device__ __forceinline__ float dec(float v) { return v; }
    static __device__ __forceinline__ float enc(float v, bool, uint32_t) { return v; }
};
template <> struct Codec<__half> {
    using C = float;
    static constexpr bool narrow = true;
    static __device__ __forceinline__ float dec(__half v) { return __half2float(v); }
    static __device__ __forceinline__ __half enc(float v, bool sr, uint32_t r) {
        return sr ? sr_half(v, r) : __float2half_rn(v);
    }
};
template <> struct Codec<__nv_bfloat16> {
    using C = float;
    static constexpr bool narrow = true;
    static __device__ __forceinline__ float dec(__nv_bfloat16 v) { return __bfloat162float(v); }
    static __device__ __forceinline__ __nv_bfloat16 enc(float v, bool sr, uint32_t r) {
        return sr ? sr_bf16(v, r) : __float2bfloat16_rn(v);
    }
};

// ------------------------------------------------------------ tensor copies
// Tensor copy (TMA) of a tile into shared memory with an mbarrier that
// counts the bytes: one thread initialises the barrier, announces the bytes
// and issues the copy; every thread then waits on the barrier's phase 0 with
// an iteration limit.
constexpr int kTmaSpin = 1 << 20;

__device__ __forceinline__ void tma_issue_3d(const void *tm, void *dst, uint64_t *bar, int c0, int c1, int c2,
                                             uint32_t bytes) {
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar), d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(d),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(b)
        : "memory");
}

__device__ __forceinline__ bool tma_wait(uint64_t *bar) {
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    for (int it = 0; it < kTmaSpin; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(b)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// ------------------------------------------------------------ NSOL
// One lattice, swap streaming: populations are stored in opposite slots
// (slot s of node x holds f*_{8-s}(x)). Tiles are staged in shared memory;
// for each of the four positive directions i, slot 8-i of x is exchanged
// with slot i of x + c_i when both are fluid (no exchange = bounce-back).
// Values that enter through domain edges or from other tiles (buffer grid)
// are substituted afterwards.
// Two block barriers: after the staging (and the substitutions, read from
// the lattice and the buffer grid), and after the exchanges.
// smem_raw: 9 * tx * ty compute values.
// ------------------------------------------------------------ edges
struct Geo {
    int nx, ny;
    int bw, be, bs, bn;
};

// Where the value pulled by node (x, y) in direction i comes from: first the
// y edge (periodic wrap, wall, or free-slip mirror onto the node's own row
// with direction mir_y(i)), then the x edge (wrap, wall, outflow clamp, or
// inlet = unknown).
__host__ __device__ __forceinline__ int map_pull(const Geo &g, int x, int y, int i, int &xs,
                                                 int &ys, int &j) {
    int sx = x - cx(i), sy = y - cy(i), d = i;
    if (sy < 0 || sy >= g.ny) {
        int bc = sy < 0 ? g.bs : g.bn;
        if (bc == PERIODIC) {
            sy = sy < 0 ? sy + g.ny : sy - g.ny;
        } else if (bc == FREESLIP) {
            sy = y;
            d = mir_y(i);
        } else {
            return PULL_BOUNCE;
        }
    }
    if (sx < 0 || sx >= g.nx) {
        int bc = sx < 0 ? g.bw : g.be;
        if (bc == PERIODIC) {
            sx = sx < 0 ? sx + g.nx : sx - g.nx;
        } else if (bc == OUTFLOW_ZG) {
            sx = sx < 0 ? 0 : g.nx - 1;
        } else if (bc == INLET_ZOUHE || bc == INLET_EQ || bc == INLET_EQ_NEUMANN || bc == OUTLET_PRESSURE) {
            return PULL_UNKNOWN;
        } else {
            return PULL_BOUNCE;
        }
    }
    xs = sx;
    ys = sy;
    j = d;
    return PULL_NODE;
}

// ------------------------------------------------------------ packed pairs
// Two FP32 values (lanes: first node, second node) in one 64-bit register
// pair, operated on by sm_100-family packed FP32 instructions. Each lane is
// rounded exactly like the scalar __fadd_rn / __fmul_rn / __fmaf_rn.
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void up2(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__host__ __device__ inline f2 dup2(float v) {
    uint32_t b;
    memcpy(&b, &v, 4);
    return ((f2)b << 32) | (f2)b;
}

// Arithmetic of the collision: one node (float, double) or a pair (f2). lit()
// gives a literal: an immediate for one node, a duplicated constant of the
// argument block for a pair.
template <class T> struct Op : Ar<T> {
    static __device__ __forceinline__ T lit(T, double v) { return (T)v; }
};
template <> struct Op<f2> {
    static __device__ __forceinline__ f2 lit(f2 c, double) { return c; }
    static __device__ __forceinline__ f2 add(f2 a, f2 b) { return add2(a, b); }
    static __device__ __forceinline__ f2 sub(f2 a, f2 b) { return sub2(a, b); }
    static __device__ __forceinline__ f2 mul(f2 a, f2 b) { return mul2(a, b); }
    static __device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) { return fma2(a, b, c); }
};

// ------------------------------------------------------------ collision
// Constants of the collision. Each storage class has its own operation order,
// which all of its kernels share (layouts, algorithms and batches agree bit
// for bit): FP32 storage (Relax<float>), FP64 storage (Relax<double>) and
// 16-bit storage (NarrowRelax, one node or a packed pair).
template <class C> struct Relax;
template <> struct Relax<float> {
    float omega;              // 1/tau
    float hfx, hfy;           // F/2
    float fx, fy, sF, dF;     // F, fx+fy, fx-fy
    float w0, w1, w4;         // 1/36, 1/9, 4/9
    float wl0, wl1, wl4;      // w - (float)w: the weights' rounding residuals
    float kw0, kw1, kw4;      // (1 - omega/2) * w
};
template <> struct Relax<double> {
    double om1, hom;           // 1 - omega, omega/2
    double hfx, hfy;           // F/2
    double k[2], c[2];         // (1 - omega/2) F, (1 - omega/2) F / 3
    double o3, o36;            // omega/3, omega/36
};
// T = float or f2 (each value duplicated).
template <class T> struct NarrowRelax {
    T nomega;                  // -omega
    T nw[3], nwl[3], kw[3];    // by weight (diagonal, axis, rest): -w, rounded value and residual; (1 - omega/2) w
    T hfx, hfy;                // F/2
    T fx, fy, sF, dF;          // F, fx+fy, fx-fy
    T c45, c9, c3, cm3, cm15;  // 4.5, 9, 3, -3, -1.5
};

struct NoPairs {};   // stands for the pair constants of storage types without node pairs

template <class C, bool NARROW> struct Consts {
    std::conditional_t<NARROW, NarrowRelax<C>, Relax<C>> r;
    C w0, w1, w4;         // 1/36, 1/9, 4/9
    C zh5, zh8, zh2;      // Zou-He: 2/3 Ux, Ux/6 + Uy/2, Ux/6 - Uy/2
    C drho_out;           // pressure outlet: rho_out - 1
    C heq_in[9];          // equilibrium inlet populations
    int force;            // F != 0
};

// Host: FP64 constants rounded once.
inline void make_relax(double omega, double fx, double fy, Relax<float> &k) {
    const double kf = 1.0 - 0.5 * omega;
    k.omega = (float)omega;
    k.hfx = (float)(0.5 * fx);
    k.hfy = (float)(0.5 * fy);
    k.fx = (float)fx;
    k.fy = (float)fy;
    k.sF = (float)(fx + fy);
    k.dF = (float)(fx - fy);
    k.w0 = (float)(1.0 / 36.0);
    k.w1 = (float)(1.0 / 9.0);
    k.w4 = (float)(4.0 / 9.0);
    k.wl0 = (float)(1.0 / 36.0 - (double)k.w0);
    k.wl1 = (float)(1.0 / 9.0 - (double)k.w1);
    k.wl4 = (float)(4.0 / 9.0 - (double)k.w4);
    k.kw0 = (float)(kf / 36.0);
    k.kw1 = (float)(kf / 9.0);
    k.kw4 = (float)(4.0 * kf / 9.0);
}
inline void make_relax(double omega, double fx, double fy, Relax<double> &q) {
    const double F[2] = {fx, fy};
    q.om1 = 1.0 - omega;
    const double om = 1.0 - q.om1;   // what the relaxation removes, to the last bit
    q.hom = 0.5 * om;
    q.hfx = 0.5 * fx;
    q.hfy = 0.5 * fy;
    for (int a = 0; a < 2; ++a) {
        q.k[a] = (1.0 - 0.5 * om) * F[a];
        q.c[a] = q.k[a] / 3.0;
    }
    q.o3 = om / 3.0;
    q.o36 = om / 36.0;
}
inline void make_relax(double omega, double fx, double fy, NarrowRelax<float> &q) {
    const double w[3] = {1.0 / 36.0, 1.0 / 9.0, 4.0 / 9.0}, kf = 1.0 - 0.5 * omega;
    q.nomega = (float)-omega;
    for (int s = 0; s < 3; ++s) {
        q.nw[s] = (float)-w[s];
        q.nwl[s] = (float)(-w[s] - (double)q.nw[s]);
        q.kw[s] = (float)(s == 1 ? kf / 9.0 : (s == 0 ? kf / 36.0 : 4.0 * kf / 9.0));
    }
    q.hfx = (float)(0.5 * fx);
    q.hfy = (float)(0.5 * fy);
    q.fx = (float)fx;
    q.fy = (float)fy;
    q.sF = (float)(fx + fy);
    q.dF = (float)(fx - fy);
    q.c45 = 4.5f;
    q.c9 = 9.0f;
    q.c3 = 3.0f;
    q.cm3 = -3.0f;
    q.cm15 = -1.5f;
}
// A block of float constants with each duplicated into both lanes.
template <template <class> class R>
inline R<f2> duplicate(const R<float> &r) {
    R<f2> q;
    static_assert(sizeof(R<f2>) == 2 * sizeof(R<float>), "the block holds values of its type only");
    float from[sizeof(R<float>) / sizeof(float)];
    f2 to[sizeof(from) / sizeof(float)];
    memcpy(from, &r, sizeof(from));
    for (size_t i = 0; i < sizeof(from) / sizeof(float); ++i) to[i] = dup2(from[i]);
    memcpy(&q, to, sizeof(q));
    return q;
}

// Zou-He velocity inlet: the three populations entering from the west are
// fixed by sum_i g_i c_i = U and bounce-back of the normal non-equilibrium part.
template <class K, class C>
__device__ __forceinline__ void zou_he(const K &k, C *g) {
    using A = Ar<C>;
    C g1 = g[1], g7 = g[7];
    g[5] = A::add(g[3], k.zh5);
    g[8] = A::fma(C(0.5), A::sub(g1, g7), A::add(g[0], k.zh8));
    g[2] = A::fma(C(0.5), A::sub(g7, g1), A::add(g[6], k.zh2));
}

// Zou-He pressure outlet: rho = rho_out and v_y = 0, with bounce-back of the
// normal non-equilibrium part, fix the three populations entering from the east.
template <class K, class C>
__device__ __forceinline__ void zou_he_pressure(const K &k, C *g) {
    using A = Ar<C>;
    const C g1 = g[1], g7 = g[7];
    const C ux = A::sub(A::fma(C(2), A::add(A::add(g[2], g[5]), g[8]), A::add(A::add(g1, g[4]), g7)), k.drho_out);
    const C u6 = A::mul(ux, C(1.0 / 6.0));
    g[3] = A::fma(C(-2.0 / 3.0), ux, g[5]);
    g[6] = A::sub(A::fma(C(0.5), A::sub(g1, g7), g[2]), u6);
    g[0] = A::sub(A::fma(C(0.5), A::sub(g7, g1), g[8]), u6);
}

// Moments, Eq. (2) equilibrium in deviation form and Eq. (1) BGK relaxation
// with the Guo source, in the fixed operation order of 32-bit storage:
//   P_i   = drho - 3/2 u^2 + cu_i (3 + 9/2 cu_i)          (h_i^eq = w_i P_i)
//   h*_i  = g_i + omega (w_i P_i - g_i)                    (w P - g in one fma)
//           + (1 - omega/2) w_i [cF_i (3 + 9 cu_i) - 3 u.F]
// with cu_i = c_i.u, cF_i = c_i.F. g (pulled h values) is replaced by h*.
// In FP32, w_i P_i uses w_i as the rounded weight plus its residual: with
// the rounded weights alone, sum_i w_i c_i c_i misses 1/3 by ~1e-8, and the
// relaxation then adds or removes momentum omega * 1e-8 * u at every node
// and update, a drift that reaches 1e-3 in lift and drag over 25,000 updates.
__device__ __forceinline__ void collide_ops(const Relax<float> &k, int force, float *g, float &drho, float &ux,
                                            float &uy) {
    using C = float;
    using A = Ar<C>;
    const C cw = A::add(A::add(g[0], g[3]), g[6]);   // c_x = -1 column
    const C cm = A::add(A::add(g[1], g[4]), g[7]);   // c_x =  0
    const C ce = A::add(A::add(g[2], g[5]), g[8]);   // c_x = +1
    const C rs = A::add(A::add(g[0], g[1]), g[2]);   // c_y = -1 row
    const C rn = A::add(A::add(g[6], g[7]), g[8]);   // c_y = +1
    drho = A::add(A::add(cw, cm), ce);
    ux = A::add(A::sub(ce, cw), k.hfx);
    uy = A::add(A::sub(rn, rs), k.hfy);
    const C usq = A::fma(ux, ux, A::mul(uy, uy));
    const C base = A::fma(C(-1.5), usq, drho);
    const C s = A::add(ux, uy), d = A::sub(ux, uy);
    const C cu[9] = {-s, -uy, d, -ux, C(0), ux, -d, uy, s};
    const C cF[9] = {-k.sF, -k.fy, k.dF, -k.fx, C(0), k.fx, -k.dF, k.fy, k.sF};
    const C m3uF = A::mul(C(-3), A::fma(ux, k.fx, A::mul(uy, k.fy)));
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const C w = i == 4 ? k.w4 : ((i & 1) ? k.w1 : k.w0);
        const C P = A::fma(cu[i], A::fma(C(4.5), cu[i], C(3)), base);
        C t = A::fma(w, P, -g[i]);
        t = A::fma(i == 4 ? k.wl4 : ((i & 1) ? k.wl1 : k.wl0), P, t);
        C o = A::fma(k.omega, t, g[i]);
        if (force) {
            const C kw = i == 4 ? k.kw4 : ((i & 1) ? k.kw1 : k.kw0);
            o = A::fma(kw, A::fma(cF[i], A::fma(C(9), cu[i], C(3)), m3uF), o);
        }
        g[i] = o;
    }
}

// 16-bit storage, one node or a packed pair: the update above as
//   h*_i = g_i - omega (g_i - w_i P_i) + (1 - omega/2) w_i [cF_i (3 + 9 cu_i) - 3 u.F]
// Every direction is written through the signed velocity c of its pair (u_x, u_y,
// u_x + u_y, u_x - u_y) and the sign sg of cu_i = sg c:
//   cu_i (3 + 9/2 cu_i) = c (9/2 c + 3 sg),  cF_i (3 + 9 cu_i) = cF+ (9 c + 3 sg)
// with cF+ = sg cF_i, so no operand is negated at run time and one node and a
// packed pair perform the same rounded operations. 92 operations, 64 without a
// force (NF). The force enters after the relaxation: with (1 - omega/2)/omega F in P
// and shared even parts, 73 operations, an update is 1 to 5 % faster (8192 x 4096 porous
// nodes, FP16, us, this order / that: node pairs 32 x 8 205 / 203, LPTL 221 / 211, one
// node 253 / 243, NPOL 367 / 352, AA 267 / 260), but that form moves stored 16-bit values to
// their neighbours and overflows where tau F does.
template <bool NF, class T>
__device__ __forceinline__ void collide_narrow(const NarrowRelax<T> &q, T *g, T &drho, T &ux, T &uy) {
    using A = Op<T>;
    const T cw = A::add(A::add(g[0], g[3]), g[6]);   // c_x = -1 column
    const T cm = A::add(A::add(g[1], g[4]), g[7]);   // c_x =  0
    const T ce = A::add(A::add(g[2], g[5]), g[8]);   // c_x = +1
    const T rs = A::add(A::add(g[0], g[1]), g[2]);   // c_y = -1 row
    const T rn = A::add(A::add(g[6], g[7]), g[8]);   // c_y = +1
    drho = A::add(A::add(cw, cm), ce);
    ux = A::add(A::sub(ce, cw), q.hfx);
    uy = A::add(A::sub(rn, rs), q.hfy);
    const T cm15 = A::lit(q.cm15, -1.5), c45 = A::lit(q.c45, 4.5), c9 = A::lit(q.c9, 9.0), c3 = A::lit(q.c3, 3.0),
            cm3 = A::lit(q.cm3, -3.0);
    const T base = A::fma(cm15, A::fma(ux, ux, A::mul(uy, uy)), drho);
    T m3uF = cm3;
    if constexpr (!NF) m3uF = A::mul(cm3, A::fma(ux, q.fx, A::mul(uy, q.fy)));
    // pairs (0, 8), (1, 7), (6, 2), (3, 5); c points to the second
    const T c[4] = {A::add(ux, uy), uy, A::sub(ux, uy), ux};
    const T cF[4] = {q.sF, q.fy, q.dF, q.fx};
    const int lo[4] = {0, 1, 6, 3};
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int s = p & 1;   // axis directions
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = e ? opp(lo[p]) : lo[p];
            const T sg3 = e ? c3 : cm3;
            const T P = A::fma(c[p], A::fma(c45, c[p], sg3), base);
            const T t = A::fma(q.nwl[s], P, A::fma(q.nw[s], P, g[i]));   // g - w P
            T o = A::fma(q.nomega, t, g[i]);
            if constexpr (!NF) o = A::fma(q.kw[s], A::fma(cF[p], A::fma(c9, c[p], sg3), m3uF), o);
            g[i] = o;
        }
    }
    const T t = A::fma(q.nwl[2], base, A::fma(q.nw[2], base, g[4]));
    T o = A::fma(q.nomega, t, g[4]);
    if constexpr (!NF) o = A::fma(q.kw[2], m3uF, o);
    g[4] = o;
}

// Density and momentum of the populations (without the force's half).
__device__ __forceinline__ void moments2(const double *g, double &drho, double &mx, double &my) {
    using A = Ar<double>;
    const double cw = A::add(A::add(g[0], g[6]), g[3]);   // c_x = -1 column
    const double cm = A::add(A::add(g[1], g[7]), g[4]);   // c_x =  0
    const double ce = A::add(A::add(g[2], g[8]), g[5]);   // c_x = +1
    drho = A::add(A::add(cw, ce), cm);
    mx = A::sub(ce, cw);
    my = A::add(A::add(A::sub(g[6], g[0]), A::sub(g[8], g[2])), A::sub(g[7], g[1]));
}

// FP64 (its arithmetic bounds every FP64 kernel, and its rounding is no
// concern): h* = (1 - omega) g + H with omega w folded into the shared parts,
//   a = omega/2 u + (1 - omega/2) F,  T = a.u,  B = omega/9 drho - T/3,
//   E_x = B + a_x u_x,  E_y = B + a_y u_y,  rest = 4 B,
//   E_diag = omega/36 drho + T/6 +- (a_x u_y + a_y u_x)/4,
//   O_x = omega/3 u_x + (1 - omega/2) F_x/3 (y alike),  O_diag = (O_x +- O_y)/4:
// 52 operations, 47 without a force (NF), where it was 88 and 61.
template <bool NF>
__device__ __forceinline__ void collide_ops64(const Relax<double> &q, double *g, double &drho, double &ux,
                                              double &uy) {
    using A = Ar<double>;
    moments2(g, drho, ux, uy);
    double ax, ay;
    if constexpr (NF) {
        ax = A::mul(q.hom, ux);
        ay = A::mul(q.hom, uy);
    } else {
        ux = A::add(ux, q.hfx);
        uy = A::add(uy, q.hfy);
        ax = A::fma(q.hom, ux, q.k[0]);
        ay = A::fma(q.hom, uy, q.k[1]);
    }
    const double ny = A::mul(-1.0 / 3.0, A::fma(ax, ux, A::mul(ay, uy)));   // -T/3
    const double z = A::mul(q.o36, drho);
    const double B = A::fma(4.0, z, ny), D = A::fma(-0.5, ny, z);
    const double Ex = A::fma(ax, ux, B), Ey = A::fma(ay, uy, B);
    double h[9];
    if constexpr (NF) {
        const double p = A::mul(ax, uy), o12 = 0.25 * q.o3;
        const double Es = A::fma(0.5, p, D), Ed = A::fma(-0.5, p, D);
        const double s = A::add(ux, uy), d = A::sub(ux, uy);
        h[5] = A::fma(q.o3, ux, Ex);
        h[3] = A::fma(-q.o3, ux, Ex);
        h[7] = A::fma(q.o3, uy, Ey);
        h[1] = A::fma(-q.o3, uy, Ey);
        h[8] = A::fma(o12, s, Es);
        h[0] = A::fma(-o12, s, Es);
        h[2] = A::fma(o12, d, Ed);
        h[6] = A::fma(-o12, d, Ed);
    } else {
        const double p = A::fma(ax, uy, A::mul(ay, ux));
        const double Es = A::fma(0.25, p, D), Ed = A::fma(-0.25, p, D);
        const double Ox = A::fma(q.o3, ux, q.c[0]), Oy = A::fma(q.o3, uy, q.c[1]);
        const double os = A::add(Ox, Oy), od = A::sub(Ox, Oy);
        h[5] = A::add(Ex, Ox);
        h[3] = A::sub(Ex, Ox);
        h[7] = A::add(Ey, Oy);
        h[1] = A::sub(Ey, Oy);
        h[8] = A::fma(0.25, os, Es);
        h[0] = A::fma(-0.25, os, Es);
        h[2] = A::fma(0.25, od, Ed);
        h[6] = A::fma(-0.25, od, Ed);
    }
    h[4] = A::mul(4.0, B);
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = A::fma(q.om1, g[i], h[i]);
}

// The collision of a storage class.
template <class C, bool NARROW>
__device__ __forceinline__ void collide(const Consts<C, NARROW> &k, C *g, C &drho, C &ux, C &uy) {
    if constexpr (NARROW) {
        if (k.force) collide_narrow<false>(k.r, g, drho, ux, uy);
        else collide_narrow<true>(k.r, g, drho, ux, uy);
    } else if constexpr (sizeof(C) == 8) {
        if (k.force) collide_ops64<false>(k.r, g, drho, ux, uy);
        else collide_ops64<true>(k.r, g, drho, ux, uy);
    } else {
        collide_ops(k.r, k.force, g, drho, ux, uy);
    }
}

// Two nodes of 16-bit storage at once: each lane performs collide()'s rounded
// operations, so it is bit-identical to the one-node form.
__device__ __forceinline__ void collide2(const NarrowRelax<f2> &q, int force, f2 *g, f2 &drho, f2 &ux, f2 &uy) {
    if (force) collide_narrow<false>(q, g, drho, ux, uy);
    else collide_narrow<true>(q, g, drho, ux, uy);
}

}  // namespace lbm
