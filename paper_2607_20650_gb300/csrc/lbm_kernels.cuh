// Kernel templates of the D2Q9I BGK update (PortLBM Sec. 3.3), instantiated
// once per storage type by lbm_ops_*.cu. Every update kernel pulls the nine
// incoming values of a node (Sec. 3.3, one-step pull), substitutes boundary
// values, and calls the same collide() so that all layouts and algorithms
// produce the same bits.
#pragma once

#include <cuda_runtime.h>

#include <cstring>
#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

constexpr int kMaxTileThreads = 512;

template <class S>
struct Step {
    using C = typename Codec<S>::C;
    Geo geo;
    uint32_t N;
    Consts<C, Codec<S>::narrow> k;
    const uint8_t *links;
    const S *src;
    S *dst;
    const S *halo_rd;
    S *halo_wr;
    C *mom;
    unsigned int *err;
    const long long *tctr;
    int toff;
    int sr;
    uint64_t seed;
    int tx, ty, ntx, nty;
    uint64_t nx_magic;
    int off32;  // 9N < 2^32: element offsets fit 32 bits
    int near32; // NPOL: and so do the buffer grid's, from the lattice's start
    int aos16;  // nx % 16 == 0: warp segments of 32 records start on 16-byte boundaries
    uint32_t pf;  // L2 prefetch distance of the two-lattice kernel: nodes (LPTL), rows (NPTL); 0 = off
    // 16-bit storage: k.r with every constant duplicated for the packed node pairs
    std::conditional_t<Codec<S>::narrow, NarrowRelax<f2>, NoPairs> k2;
};

// Host: FP64 constants rounded once to the compute type.
template <class S>
Step<S> make_step(const HostArgs &h, const StepCall &c) {
    using C = typename Codec<S>::C;
    Step<S> a;
    a.geo = Geo{h.nx, h.ny, h.bw, h.be, h.bs, h.bn};
    a.N = (uint32_t)h.N;
    Consts<C, Codec<S>::narrow> &k = a.k;
    make_relax(h.omega, h.fx, h.fy, k.r);
    k.w0 = (C)(1.0 / 36.0);
    k.w1 = (C)(1.0 / 9.0);
    k.w4 = (C)(4.0 / 9.0);
    k.zh5 = (C)(2.0 / 3.0 * h.ux_in);
    k.zh8 = (C)(h.ux_in / 6.0 + h.uy_in / 2.0);
    k.zh2 = (C)(h.ux_in / 6.0 - h.uy_in / 2.0);
    k.drho_out = (C)(h.rho_out - 1.0);
    const double W[9] = {1.0 / 36, 1.0 / 9, 1.0 / 36, 1.0 / 9, 4.0 / 9,
                         1.0 / 9, 1.0 / 36, 1.0 / 9, 1.0 / 36};
    for (int i = 0; i < 9; ++i) {
        double cu = cx(i) * h.ux_in + cy(i) * h.uy_in;
        double usq = h.ux_in * h.ux_in + h.uy_in * h.uy_in;
        k.heq_in[i] = (C)(W[i] * (3.0 * cu + 4.5 * cu * cu - 1.5 * usq));
    }
    k.force = (h.fx != 0.0 || h.fy != 0.0) ? 1 : 0;
    a.links = h.links;
    a.src = (const S *)h.pop[c.src];
    a.dst = (S *)(h.pop[1] ? h.pop[c.src ^ 1] : h.pop[0]);
    S *halo = (S *)h.halo;
    a.halo_rd = halo ? halo + (int64_t)c.rd_parity * h.halo_parity_elems : nullptr;
    a.halo_wr = halo ? halo + (int64_t)(c.rd_parity ^ 1) * h.halo_parity_elems : nullptr;
    a.mom = c.want_moments ? (C *)h.mom : nullptr;
    a.err = h.err;
    a.tctr = h.tctr;
    a.toff = c.toff;
    a.sr = h.rounding;
    a.seed = h.seed;
    a.tx = h.tile_x;
    a.ty = h.tile_y;
    a.ntx = h.ntx;
    a.nty = h.nty;
    a.nx_magic = h.nx_magic;
    a.off32 = (9 * h.N) < (int64_t(1) << 32) ? 1 : 0;
    // (flag 8: LBM_FLAG_WIDE_OFFSETS)
    a.near32 = halo && !(h.flags & 8u) && halo + 2 * h.halo_parity_elems - a.dst < (int64_t(1) << 32) ? 1 : 0;
    a.aos16 = (h.nx % 16 == 0) ? 1 : 0;
    a.pf = h.pf;
    if constexpr (Codec<S>::narrow) a.k2 = duplicate(a.k.r);
    return a;
}

template <class S, int L>
__device__ __forceinline__ typename Codec<S>::C ldp(const S *base, uint32_t N, uint32_t n, int i) {
    return Codec<S>::dec(base[addr<L>(N, n, i)]);
}

#ifndef LBM_ST_HINT
#define LBM_ST_HINT 0
#endif
// Loads of the source lattice are plain loads, never read-only (non-coherent)
// ones, and its pointer is not __restrict__: in a chained launch the previous
// update may still be writing it when this grid starts, and only a plain load
// is sure to stay behind chain_wait(). (The read-only path made no difference
// in time.)
// Stores of the destination lattice of the two-lattice update default to plain
// stores, which measured 1 % faster than evict-first (st.global.cs) for the
// bundle layout at 32 registers; LBM_ST_HINT=1 makes every store evict-first, 2
// only the bundle layout's.
template <class S, int L>
__device__ __forceinline__ void st_dst(S *p, S v) {
#if LBM_ST_HINT == 1
    __stcs(p, v);
#elif LBM_ST_HINT == 2
    if (L == BUNDLE)
        __stcs(p, v);
    else
        *p = v;
#else
    *p = v;
#endif
}

// Density deviation of node n + 1 (the Neumann inlet's east neighbour) in a
// stored state, summed in canonical direction order; 0 if it is solid.
template <class S, int L>
__device__ __forceinline__ typename Codec<S>::C neighbour_drho(const Step<S> &a, const S *lat, uint32_t n,
                                                               int rev) {
    using C = typename Codec<S>::C;
    if (a.links[n + 1] == SOLID_LINKS) return C(0);
    C d = C(0);
#pragma unroll
    for (int i = 0; i < 9; ++i) d = Ar<C>::add(d, ldp<S, L>(lat, a.N, n + 1, rev ? opp(i) : i));
    return d;
}

// Inlet substitution, collision, divergence flag, moments, and encoding of
// the nine post-collision values (canonical direction order) into e.
// drho_nb: density deviation of node (1, y) in the previous state, used by
// the Neumann equilibrium inlet only.
// Inlet (x = 0) and outlet (x = nx - 1) substitutions of the pulled values.
// drho_nb: density deviation of node (1, y) in the previous state, used by
// the Neumann equilibrium inlet only.
template <class S>
__device__ __forceinline__ void edge_substitute(const Step<S> &a, uint32_t x, typename Codec<S>::C *g,
                                                typename Codec<S>::C drho_nb) {
    using C = typename Codec<S>::C;
    using A = Ar<C>;
    if (x == 0) {
        if (a.geo.bw == INLET_ZOUHE) {
            zou_he(a.k, g);
        } else if (a.geo.bw == INLET_EQ) {
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = a.k.heq_in[i];
        } else if (a.geo.bw == INLET_EQ_NEUMANN) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const C w = i == 4 ? a.k.w4 : ((i & 1) ? a.k.w1 : a.k.w0);
                g[i] = A::fma(w, drho_nb, a.k.heq_in[i]);
            }
        }
    }
    if (x == (uint32_t)a.geo.nx - 1 && a.geo.be == OUTLET_PRESSURE) zou_he_pressure(a.k, g);
}

// Edge substitutions (EDGE = true; false when the caller has applied them or
// guarantees 0 < x < nx - 1, which keeps them out of the interior hot path),
// collision, divergence flag, moments, and encoding of the nine
// post-collision values (canonical direction order) into e.
template <class S, bool EDGE = true>
__device__ __forceinline__ void collide_encode(const Step<S> &a, uint32_t x, uint32_t n,
                                               typename Codec<S>::C *g, S *e,
                                               typename Codec<S>::C drho_nb = 0) {
    using C = typename Codec<S>::C;
    using A = Ar<C>;
    if (EDGE) edge_substitute(a, x, g, drho_nb);
    C drho, ux, uy;
    collide(a.k, g, drho, ux, uy);
    if (!isfinite(drho)) atomicOr(a.err, 1u);
    if (a.mom) {
        a.mom[n] = A::add(C(1), drho);
        a.mom[a.N + n] = ux;
        a.mom[2 * a.N + n] = uy;
    }
    const bool sr = Codec<S>::narrow && a.sr;
    uint32_t nk = 0;
    if (sr) nk = node_key(step_key(a.seed, (uint32_t)(*a.tctr + a.toff)), n);
#pragma unroll
    for (int i = 0; i < 9; ++i) e[i] = Codec<S>::enc(g[i], sr, sr ? pop_rand(nk, i) : 0u);
}

// ------------------------------------------------------------ two lattices
// Element offset of population i of node 0 in layout L; the offset of node n
// is lay_mul<L>() * n + lay_base<L>(N, i) for every layout.
template <int L> __host__ __device__ constexpr uint32_t lay_mul() {
    return L == STREAM ? 1u : (L == BUNDLE ? 3u : 9u);
}
template <int L> __device__ __forceinline__ uint32_t lay_base(uint32_t N, int i) {
    return L == STREAM ? (uint32_t)i * N
                       : (L == BUNDLE ? (uint32_t)(i / 3) * 3u * N + (uint32_t)(i % 3) : (uint32_t)i);
}

// Whether a solid node rewrites its (zero) record because it shares a
// 32-byte DRAM sector with a fluid node's record, from the warp's fluid
// ballot F (lanes = consecutive nodes). Only the stream layout does it
// (aligned groups of 32/sizeof(S) lanes): measured +9 % for the stream
// two-lattice kernels on the porous medium, but -6 % (FP32) / -10 % (FP16)
// for the bundle layout, -27 % for the AA pattern on it and -2 % for the
// collision layout, where the partial-sector writes cost less than the
// extra zeros.
template <class S, int L>
__device__ __forceinline__ bool shares_sector(unsigned F, int lane) {
    if (L != STREAM) return false;
    constexpr int G = (int)(32 / sizeof(S)) < 32 ? (int)(32 / sizeof(S)) : 32;
    const unsigned m = G >= 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane & ~(G - 1));
    return (F & m) != 0u;
}

template <class S, int L>
__device__ __forceinline__ void store_zero(S *dst, uint32_t N, uint32_t n, int off32) {
    const S z = Codec<S>::enc(typename Codec<S>::C(0), false, 0u);
    if (off32) {
        const uint32_t base = lay_mul<L>() * n;
#pragma unroll
        for (int i = 0; i < 9; ++i) st_dst<S, L>(dst + base + lay_base<L>(N, i), z);
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[addr<L>(N, n, i)] = z;
    }
}

// Pulls of an interior node (requires 9N < 2^32); each picks the pulled
// neighbour or, for a bounced link, the node's opposite slot. IDX: by 32-bit
// indices, one select a pull, else by pointers with constant offsets. us an update
// of FP32 lattices, pointers / indices: 2048 x 512 stream 9.63 / 9.22, bundle
// 9.81 / 9.97 (porous 9.31 / 9.10), 16384 x 8192 porous bundle 1192 / 1186.
template <class S, int L, bool IDX>
__device__ __forceinline__ void pull_interior(const S *src, uint32_t n, uint32_t nx, uint32_t N, uint32_t lk,
                                              typename Codec<S>::C *g) {
    constexpr uint32_t m = lay_mul<L>();
    if constexpr (IDX) {
        const uint32_t own = m * n;
        const uint32_t row[3] = {own + m * nx, own, own - m * nx};   // of c_y = -1, 0, +1
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            uint32_t p = row[cy(i) + 1] + (lay_base<L>(N, i) - m * (uint32_t)cx(i));
            if (i != 4 && ((lk >> link_bit(i)) & 1u)) p = own + lay_base<L>(N, opp(i));
            g[i] = Codec<S>::dec(src[p]);
        }
    } else {
        const S *own = src + m * n;
        const S *row[3] = {own + (ptrdiff_t)m * nx, own, own - (ptrdiff_t)m * nx};
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const S *p = row[cy(i) + 1] + ((ptrdiff_t)lay_base<L>(N, i) - (ptrdiff_t)m * cx(i));
            if (i != 4 && ((lk >> link_bit(i)) & 1u)) p = own + (ptrdiff_t)lay_base<L>(N, opp(i));
            g[i] = Codec<S>::dec(*p);
        }
    }
}

// The same for warps without a bounced link.
template <class S, int L>
__device__ __forceinline__ void pull_inner(const S *src, uint32_t n, uint32_t nx, uint32_t N,
                                           typename Codec<S>::C *g) {
    constexpr uint32_t m = lay_mul<L>();
    const S *own = src + m * n;
    const S *row[3] = {own + (ptrdiff_t)m * nx, own, own - (ptrdiff_t)m * nx};
#pragma unroll
    for (int i = 0; i < 9; ++i)
        g[i] = Codec<S>::dec(row[cy(i) + 1][(ptrdiff_t)lay_base<L>(N, i) - (ptrdiff_t)m * cx(i)]);
}

template <class S, int L>
__device__ __forceinline__ void store_node(S *dst, uint32_t n, uint32_t N, int off32, const S *e) {
    if (off32) {
        S *od = dst + lay_mul<L>() * n;
#pragma unroll
        for (int i = 0; i < 9; ++i) st_dst<S, L>(od + (ptrdiff_t)lay_base<L>(N, i), e[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[addr<L>(N, n, i)] = e[i];
    }
}

// Pulls of a node anywhere in the domain (requires 9N < 2^32). An edge changes
// the source by an amount that depends on the sign of c_x or c_y alone: across
// a periodic edge it wraps, at a zero-gradient outflow the column is clamped, at
// a free-slip edge the row stays and the population is the mirrored one, six
// directions on. Pulls over a wall bounce and those over an inlet or a
// pressure outlet are replaced afterwards; they read their own column. So an
// edge node costs a few selects more than an inner one, and the warps that
// hold edge nodes run this code for all their lanes. (With the general edge
// mapping per direction, beside the interior path, FP32: 256 x 64 nodes 2.43 ->
// 1.64 us an update, 2048 x 512 10.8 -> 9.7, 48 channels in a batch 133 -> 123.)
template <class S, int L>
__device__ __forceinline__ void pull_edge(const Step<S> &a, uint32_t x, uint32_t y, uint32_t n, uint32_t lk,
                                          typename Codec<S>::C *g) {
    // element indices modulo 2^32: every index read is below 9N
    constexpr uint32_t m = lay_mul<L>();
    const uint32_t nx = (uint32_t)a.geo.nx, N = a.N;
    const uint32_t mirror = L == COLLISION ? 6u : 6u * N;   // from direction i to i + 6
    const uint32_t own = m * n;
    uint32_t rn = 0u - m * nx, rs = m * nx;   // to the source row of c_y = +1, -1
    if (y == 0) rn = a.geo.bs == FREESLIP ? 0u - mirror : m * (N - nx);
    if (y == (uint32_t)a.geo.ny - 1) rs = a.geo.bn == FREESLIP ? mirror : m * (nx - N);
    uint32_t cw = 0u - m, ce = m;             // to the source column of c_x = +1, -1
    if (x == 0) cw = a.geo.bw == PERIODIC ? m * (nx - 1u) : 0u;
    if (x == nx - 1u) ce = a.geo.be == PERIODIC ? m * (1u - nx) : 0u;
    const uint32_t row[3] = {own + rs, own, own + rn};
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        uint32_t p = row[cy(i) + 1] + (cx(i) > 0 ? cw : (cx(i) < 0 ? ce : 0u)) + lay_base<L>(N, i);
        if (i != 4 && ((lk >> link_bit(i)) & 1u)) p = own + lay_base<L>(N, opp(i));
        g[i] = Codec<S>::dec(a.src[p]);
    }
}

// Pull, collide and store one fluid node of the two-lattice update. Interior
// nodes take a path with 32-bit element offsets. EDGES: warps that hold a node on the domain edge take pull_edge for all their
// lanes; without it (large lattices, where such warps are rare and the vote
// costs 0.3 %) and beyond 32-bit offsets, edge nodes take the general mapping.
// BATCH (arguments in shared memory): warps of inner nodes without a bounced link
// choose no source at all. 48 channels, us an update: FP32 124.3 -> 120.6, FP16
// 125.3 -> 115.4; single lattices gained nothing by it.
template <class S, int L, bool EDGES = true, bool BATCH = false>
__device__ __forceinline__ void two_lattice_fluid(const Step<S> &a, uint32_t x, uint32_t y, uint32_t n,
                                                  uint32_t lk) {
    using C = typename Codec<S>::C;
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    S *dst = a.dst;
    const S *src = a.src;
    const bool interior = (x - 1u < nx - 2u) && (y - 1u < ny - 2u);
    C g[9];
    if (BATCH && a.off32 && __all_sync(__activemask(), interior && lk == 0u)) {
        pull_inner<S, L>(src, n, nx, a.N, g);
    } else if (a.off32 && (EDGES ? __all_sync(__activemask(), interior) != 0 : interior)) {
        pull_interior<S, L, BATCH || L == STREAM || (L == BUNDLE && !EDGES)>(src, n, nx, a.N, lk, g);
    } else {
        if (EDGES && a.off32) {
            pull_edge<S, L>(a, x, y, n, lk, g);
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                if (i == 4) {
                    g[i] = ldp<S, L>(src, a.N, n, 4);
                    continue;
                }
                if ((lk >> link_bit(i)) & 1u) {
                    g[i] = ldp<S, L>(src, a.N, n, opp(i));
                } else if (interior) {
                    g[i] = ldp<S, L>(src, a.N, n - (uint32_t)(cy(i) * (int)nx + cx(i)), i);
                } else {
                    int xs, ys, j;
                    if (map_pull(a.geo, (int)x, (int)y, i, xs, ys, j) == PULL_NODE)
                        g[i] = ldp<S, L>(src, a.N, (uint32_t)ys * nx + (uint32_t)xs, j);
                    else
                        g[i] = C(0);  // inlet unknown, reconstructed by edge_substitute
                }
            }
        }
        const C dnb = (x == 0 && a.geo.bw == INLET_EQ_NEUMANN) ? neighbour_drho<S, L>(a, src, n, 0) : C(0);
        edge_substitute(a, x, g, dnb);
    }
    S e[9];
    collide_encode<S, false>(a, x, n, g, e);
    store_node<S, L>(dst, n, a.N, a.off32, e);
}

// One node of the two-lattice pull update (LPTL and NPTL). lane: the
// thread's lane (the zero fill below votes over the warp).
template <class S, int L, bool CHAIN, bool BATCH>
__device__ __forceinline__ void two_lattice_known(const Step<S> &a, uint32_t x, uint32_t y, uint32_t n, uint32_t lk,
                                                  int lane) {
    const bool fluid = lk != SOLID_LINKS;
    const unsigned F = __ballot_sync(__activemask(), fluid);
    if (!fluid) {
        // Solid nodes hold h = 0 and are never read. Where a solid node's
        // record shares a DRAM sector with a fluid node's, store the zeros
        // again so the sector is written whole (no read-modify-write).
        if (shares_sector<S, L>(F, lane)) store_zero<S, L>(a.dst, a.N, n, a.off32);
        return;
    }
    two_lattice_fluid<S, L, CHAIN, BATCH>(a, x, y, n, lk);
}
template <class S, int L, bool CHAIN = true, bool BATCH = false>
__device__ __forceinline__ void two_lattice_node(const Step<S> &a, uint32_t x, uint32_t y, int lane) {
    const uint32_t n = y * (uint32_t)a.geo.nx + x;
    const uint32_t lk = a.links[n];
    if (CHAIN) chain_wait();
    two_lattice_known<S, L, CHAIN, BATCH>(a, x, y, n, lk, lane);
}

// NPTL with two nodes per thread, rows y and y + ty/2 of a tx x ty tile:
// both link bytes, then all eighteen pulls of interior nodes are issued
// before either collision, so one thread keeps twice the loads in flight.
template <class S, int L>
__global__ void __launch_bounds__(kMaxTileThreads) k_two_lattice2(const Step<S> a) {
    using C = typename Codec<S>::C;
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    const uint32_t x = blockIdx.x * a.tx + threadIdx.x;
    chain_next();
    const uint32_t ya = blockIdx.y * a.ty + threadIdx.y, yb = ya + (uint32_t)(a.ty >> 1);
    if (x >= nx || ya >= ny) return;
    const int lane = (int)((threadIdx.y * blockDim.x + threadIdx.x) & 31u);
    const bool hb = yb < ny;
    const uint32_t na = ya * nx + x, nb = yb * nx + x;
    const uint32_t lka = a.links[na];
    const uint32_t lkb = hb ? (uint32_t)a.links[nb] : SOLID_LINKS;
    chain_wait();
    const bool fa = lka != SOLID_LINKS, fb = lkb != SOLID_LINKS;
    const unsigned act = __activemask();
    const unsigned Fa = __ballot_sync(act, fa), Fb = __ballot_sync(act, hb && fb);
    if (!fa && shares_sector<S, L>(Fa, lane)) store_zero<S, L>(a.dst, a.N, na, a.off32);
    if (hb && !fb && shares_sector<S, L>(Fb, lane)) store_zero<S, L>(a.dst, a.N, nb, a.off32);
    const bool fast_a = fa && a.off32 && (x - 1u < nx - 2u) && (ya - 1u < ny - 2u);
    const bool fast_b = fb && a.off32 && (x - 1u < nx - 2u) && (yb - 1u < ny - 2u);
    C ga[9], gb[9];
    if (fast_a) pull_interior<S, L, false>(a.src, na, nx, a.N, lka, ga);
    if (fast_b) pull_interior<S, L, false>(a.src, nb, nx, a.N, lkb, gb);
    S e[9];
    if (fast_a) {
        collide_encode<S, false>(a, x, na, ga, e);
        store_node<S, L>(a.dst, na, a.N, a.off32, e);
    } else if (fa) {
        two_lattice_fluid<S, L>(a, x, ya, na, lka);
    }
    if (fast_b) {
        collide_encode<S, false>(a, x, nb, gb, e);
        store_node<S, L>(a.dst, nb, a.N, a.off32, e);
    } else if (fb) {
        two_lattice_fluid<S, L>(a, x, yb, nb, lkb);
    }
}

// Collision layout (9 contiguous values per node), NPTL: a warp owns 32
// consecutive nodes of a row. For warps of 32 fluid nodes away from the domain
// edges, the three source row spans (nodes x0-1 .. x0+32 of rows y+1, y, y-1)
// are staged in shared memory with 16-byte loads, the pulls read shared
// memory, and the 32 output records are written back with 16-byte stores.
// Other warps use the per-node path.
template <class S>
struct AosSpan {
    static constexpr int R = 9 * (int)sizeof(S);                    // record bytes
    static constexpr int CHUNKS = (34 * R + 15) / 16 + 1;           // 16-byte chunks per row span
    static constexpr int ROW_BYTES = CHUNKS * 16;
    static constexpr int WARP_BYTES = 3 * ROW_BYTES;
};

template <class S, bool CHAIN = true>
__global__ void __launch_bounds__(kMaxTileThreads, sizeof(S) == 8 ? 1 : 4) k_two_lattice_aos(const Step<S> a) {
    using C = typename Codec<S>::C;
    using SP = AosSpan<S>;
    extern __shared__ __align__(16) unsigned char smem_aos[];
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const uint32_t x = blockIdx.x * a.tx + threadIdx.x;
    const uint32_t y = blockIdx.y * a.ty + threadIdx.y;
    if (CHAIN) chain_next();
    if (x >= nx || y >= ny) return;
    const uint32_t n = y * nx + x;
    const uint32_t lk = a.links[n];
    if (CHAIN) chain_wait();
    const bool fluid = lk != SOLID_LINKS;
    const unsigned act = __activemask();
    const unsigned F = __ballot_sync(act, fluid);
    const uint32_t x0 = x - (uint32_t)lane;   // first node of this warp's row segment
    // Staging pays off for warps of fluid nodes only (measured): with solid
    // nodes in the warp the spans carry unused records and the stores stay scalar.
    const bool staged = F == 0xffffffffu && a.off32 && a.aos16 && x0 >= 1u && x0 + 33u <= nx &&
                        y >= 1u && y + 2u <= ny;
    if (!staged) {
        if (!fluid) {
            if (shares_sector<S, COLLISION>(F, lane)) store_zero<S, COLLISION>(a.dst, a.N, n, a.off32);
            return;
        }
        two_lattice_fluid<S, COLLISION, CHAIN>(a, x, y, n, lk);
        return;
    }
    unsigned char *wbuf = smem_aos + (size_t)warp * SP::WARP_BYTES;
    const uint32_t n0 = y * nx + x0;
    const unsigned char *srcb = reinterpret_cast<const unsigned char *>(a.src);
    int shift[3];   // bytes from each staged span start to record (n0 - 1 - c_y nx)
#pragma unroll
    for (int r = 0; r < 3; ++r) {       // r = c_y + 1: source row y - c_y
        const uint64_t first = (uint64_t)SP::R * (uint64_t)(n0 - 1u - (uint32_t)((r - 1) * (int)nx));
        const uint64_t base = first & ~(uint64_t)15;
        shift[r] = (int)(first - base);
        const uint4 *g4 = reinterpret_cast<const uint4 *>(srcb + base);
        uint4 *s4 = reinterpret_cast<uint4 *>(wbuf + r * SP::ROW_BYTES);
#pragma unroll
        for (int k = lane; k < SP::CHUNKS; k += 32) s4[k] = g4[k];
    }
    __syncwarp();
    C g[9];
    if (fluid) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const S *pp = reinterpret_cast<const S *>(wbuf + (cy(i) + 1) * SP::ROW_BYTES + shift[cy(i) + 1]) +
                          (lane + 1 - cx(i)) * 9 + i;
            const S *pb = reinterpret_cast<const S *>(wbuf + SP::ROW_BYTES + shift[1]) + (lane + 1) * 9 + opp(i);
            g[i] = Codec<S>::dec(((lk >> link_bit(i)) & 1u) ? *pb : *pp);
        }
    }
    S e[9];
    if (fluid) collide_encode(a, x, n, g, e);
    if (F != 0xffffffffu) {
        if (fluid) {
            store_node<S, COLLISION>(a.dst, n, a.N, a.off32, e);
        } else if (shares_sector<S, COLLISION>(F, lane)) {
            store_zero<S, COLLISION>(a.dst, a.N, n, a.off32);
        }
        return;
    }
    __syncwarp();   // every lane has read its inputs; reuse the first span for the output
    S *out = reinterpret_cast<S *>(wbuf);
#pragma unroll
    for (int i = 0; i < 9; ++i) out[lane * 9 + i] = e[i];
    __syncwarp();
    uint4 *d4 = reinterpret_cast<uint4 *>(reinterpret_cast<unsigned char *>(a.dst) + (uint64_t)SP::R * n0);
    const uint4 *o4 = reinterpret_cast<const uint4 *>(wbuf);
    constexpr int OUT_CHUNKS = 32 * SP::R / 16;
#pragma unroll
    for (int k = lane; k < OUT_CHUNKS; k += 32) d4[k] = o4[k];
}

// L2 prefetch of one node's source record (stream and bundle layouts): one
// address per DRAM sector the record occupies, every value of the stream
// layout and the first value of each bundle (a bundle straddling two sectors
// has its second one fetched by the neighbour's prefetch).
template <class S, int L>
__device__ __forceinline__ void prefetch_record(const S *src, uint32_t N, uint32_t n) {
#pragma unroll
    for (int i = 0; i < 9; ++i)
        if (L == STREAM || i % 3 == 0)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(src + addr<L>(N, n, i)));
}

// LPTL (LINEAR: one node per thread over n, block size from the runtime) and
// NPTL (2-D tiles of tx x ty nodes over a padded grid).
//
// Blocks start in index order, so the node a.pf nodes (LPTL) or a.pf rows
// (NPTL) ahead belongs to a block that starts a few microseconds later. Each
// thread loads that node's link byte first and, once its own node is stored,
// prefetches the node's source record into L2 when it is fluid: the pulls of
// the later block then hit L2 instead of waiting on DRAM, and the prefetches
// keep more DRAM requests in flight than the pulls alone at full occupancy.
// Solid records are not fetched, so DRAM traffic does not grow. Only 32-bit
// storage in the stream and bundle layouts has it: the 16-bit update is bound
// by instruction issue (the prefetch cost 3 %), and the collision layout's
// LPTL form spills at 32 registers with it (its NPTL form is the staged
// kernel above).
// CHAIN: a chained launch (launch_update). Off for large lattices, where the
// gap between updates is nothing and the wait between the loads costs 0.9 %
// (134M nodes, FP32 bundle: 1.199 against 1.210 ms).
constexpr int64_t kChainNodes = 4 << 20;
template <class S, int L, bool LINEAR, bool CHAIN = true>
__global__ void __launch_bounds__(kMaxTileThreads, sizeof(S) == 8 ? 1 : 4) k_two_lattice(const Step<S> a) {
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    constexpr bool PF = sizeof(S) == 4 && L != COLLISION;
    uint32_t x, y, np = 0;
    bool ahead;
    if (CHAIN) chain_next();
    if (LINEAR) {
        const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
        if (n >= a.N) return;
        y = a.nx_magic ? (uint32_t)__umul64hi((unsigned long long)n, a.nx_magic) : n;
        x = n - y * nx;
        ahead = PF && a.pf != 0u && a.N - n > a.pf;
        np = n + a.pf;
    } else {
        x = blockIdx.x * a.tx + threadIdx.x;
        y = blockIdx.y * a.ty + threadIdx.y;
        if (x >= nx || y >= ny) return;
        ahead = PF && a.pf != 0u && ny - y > a.pf;
        np = (y + a.pf) * nx + x;
    }
    const uint32_t lkp = ahead ? (uint32_t)a.links[np] : SOLID_LINKS;
    two_lattice_node<S, L, CHAIN>(a, x, y, (int)((threadIdx.y * blockDim.x + threadIdx.x) & 31u));
    if (PF && lkp != SOLID_LINKS) prefetch_record<S, L>(a.src, a.N, np);
}

// ------------------------------------------------------------ node pairs
// Two-lattice update (LPTL, NPTL) for 16-bit storage with two horizontally
// adjacent nodes per thread, x even (nx even, so a pair never wraps a row).
// The 16-bit update is bound by instruction issue, not by DRAM, so the pair
// shares what one node per thread repeats: one 16-bit load brings both link
// bytes, the collision runs on packed FP32 pairs (collide2: each lane is the
// scalar collide() bit for bit), two results are rounded to 16 bits by one
// packed conversion, and the stores are 32-bit words: in the bundle layout a
// pair's bundle is six adjacent values (3n even), three words. A solid node of a pair holding a fluid one stores its zeros in
// the same words, so the pair's sector is written whole. Pairs touching the
// domain edge take the per-node path.
template <class S>
__device__ __forceinline__ uint32_t pack_rne(float lo, float hi) {
    uint32_t r;
    if constexpr (sizeof(S) == 2 && std::is_same<S, __half>::value)
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    else
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Encoded 16-bit pair words for the nine directions: word i holds direction i
// of node a (low half) and node b (high half). A node with keep = false
// contributes +0.
template <class S>
__device__ __forceinline__ void encode_pair(const Step<S> &a, uint32_t n, const f2 *g, bool ka, bool kb,
                                            uint32_t *w) {
    const bool sr = a.sr != 0;
    if (!sr) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float lo, hi;
            up2(g[i], lo, hi);
            w[i] = pack_rne<S>(ka ? lo : 0.0f, kb ? hi : 0.0f);
        }
    } else {
        // one packed stochastic conversion per direction: node a in the low
        // half, node b in the high half, each with its own draw (a solid
        // node's lane converts +0, which no draw changes)
        const uint32_t sk = step_key(a.seed, (uint32_t)(*a.tctr + a.toff));
        const uint32_t nka = node_key(sk, n), nkb = node_key(sk, n + 1);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float lo, hi;
            up2(g[i], lo, hi);
            lo = ka ? lo : 0.0f;
            hi = kb ? hi : 0.0f;
            if constexpr (std::is_same<S, __half>::value)
                w[i] = sr_half2(hi, lo, pop_rand(nkb, i), pop_rand(nka, i));
            else
                w[i] = sr_bf162(hi, lo, pop_rand(nkb, i), pop_rand(nka, i));
        }
    }
}

// Store the pair words of nodes n, n + 1 (n even).
template <class S>
__device__ __forceinline__ void store_pair(S *dst, uint32_t N, uint32_t n, const uint32_t *w) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        uint32_t *p = reinterpret_cast<uint32_t *>(dst + (uint32_t)b * 3u * N + 3u * n);
        const uint32_t w0 = w[3 * b], w1 = w[3 * b + 1], w2 = w[3 * b + 2];
        p[0] = (w0 & 0xFFFFu) | (w1 << 16);            // (a, 3b), (a, 3b+1)
        p[1] = (w2 & 0xFFFFu) | (w0 & 0xFFFF0000u);    // (a, 3b+2), (b, 3b)
        p[2] = (w1 >> 16) | (w2 & 0xFFFF0000u);        // (b, 3b+1), (b, 3b+2)
    }
}

// L2 prefetch of a pair's source records (both nodes): one address per bundle.
template <class S>
__device__ __forceinline__ void prefetch_pair(const S *src, uint32_t N, uint32_t n) {
#pragma unroll
    for (int i = 0; i < 9; i += 3) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + addr<BUNDLE>(N, n, i)));
}

// The lower / upper 16-bit value of a word.
template <class S>
__device__ __forceinline__ float lower(uint32_t w) {
    if constexpr (std::is_same<S, __half>::value) return __half2float(__ushort_as_half((unsigned short)(w & 0xFFFFu)));
    else return __uint_as_float(w << 16);
}
template <class S>
__device__ __forceinline__ float upper(uint32_t w) {
    if constexpr (std::is_same<S, __half>::value) return __half2float(__ushort_as_half((unsigned short)(w >> 16)));
    else return __uint_as_float(w & 0xFFFF0000u);
}

// Pulls of an interior pair in the bundle layout, by 32-bit words: the six
// values of one bundle that both nodes pull lie in the eight elements from one
// before to six after the source row's node n (3n is even), so five words per
// bundle bring them; where a lane of the warp bounces, the pair's own nine words
// (three of them are among the others) hold the values that replace them. No
// address is selected per direction and node, and a solid node, all of whose
// links bounce, yields the zeros it holds. FP16, 8192 x 4096 porous nodes, 16
// updates: 3.91 -> 3.59 ms (eighteen 16-bit loads through selected addresses before).
template <class S>
__device__ __forceinline__ void pull_pair(const Step<S> &a, uint32_t n, uint32_t lka, uint32_t lkb, f2 *g) {
    const uint32_t N3 = 3u * a.N, nx3 = 3u * (uint32_t)a.geo.nx;
    const S *own = a.src + 3u * n;
    const uint32_t *c[3] = {reinterpret_cast<const uint32_t *>(own + nx3),
                            reinterpret_cast<const uint32_t *>(own + N3),
                            reinterpret_cast<const uint32_t *>(own + 2 * (size_t)N3 - nx3)};
    uint32_t w[3][5], o[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int k = 0; k < 5; ++k) w[b][k] = c[b][k - 1];
    const bool bounces = __any_sync(__activemask(), (lka | lkb) != 0u);
    if (bounces) {
        const uint32_t *o0 = reinterpret_cast<const uint32_t *>(own);
        const uint32_t *o2 = reinterpret_cast<const uint32_t *>(own + 2 * (size_t)N3);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            o[0][k] = o0[k];
            o[1][k] = w[1][k + 1];
            o[2][k] = o2[k];
        }
    }
    float va[9], vb[9];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        va[3 * b] = upper<S>(w[b][2]);       // element 3: node n + 1
        vb[3 * b] = lower<S>(w[b][4]);       // element 6: node n + 2
        va[3 * b + 1] = upper<S>(w[b][1]);   // element 1: node n
        vb[3 * b + 1] = lower<S>(w[b][3]);   // element 4: node n + 1
        va[3 * b + 2] = upper<S>(w[b][0]);   // element -1: node n - 1
        vb[3 * b + 2] = lower<S>(w[b][2]);   // element 2: node n
    }
    if (bounces) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if (i == 4) continue;
            const uint32_t *r = o[opp(i) / 3];
            const int k = opp(i) % 3;
            if ((lka >> link_bit(i)) & 1u) va[i] = k == 0 ? lower<S>(r[0]) : (k == 1 ? upper<S>(r[0]) : lower<S>(r[1]));
            if ((lkb >> link_bit(i)) & 1u) vb[i] = k == 0 ? upper<S>(r[1]) : (k == 1 ? lower<S>(r[2]) : upper<S>(r[2]));
        }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = pk2(va[i], vb[i]);
}

// One pair: both link bytes in lk2 (node n in the low byte).
template <class S>
__device__ __forceinline__ void pair_update(const Step<S> &a, uint32_t x, uint32_t y, uint32_t n, uint32_t lk2) {
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    const uint32_t lka = lk2 & 0xFFu, lkb = lk2 >> 8;
    const bool fa = lka != SOLID_LINKS, fb = lkb != SOLID_LINKS;
    if (!fa && !fb) return;
    const bool interior = (x - 1u < nx - 3u) && (y - 1u < ny - 2u);
    if (!interior || !a.off32) {
        if (fa) two_lattice_fluid<S, BUNDLE>(a, x, y, n, lka);
        if (fb) two_lattice_fluid<S, BUNDLE>(a, x + 1u, y, n + 1u, lkb);
        return;
    }
    f2 g[9];
    pull_pair<S>(a, n, lka, lkb, g);
    f2 drho2, ux2, uy2;
    collide2(a.k2, a.k.force, g, drho2, ux2, uy2);
    float da, db;
    up2(drho2, da, db);
    if ((fa && !isfinite(da)) || (fb && !isfinite(db))) atomicOr(a.err, 1u);
    if (a.mom) {
        const f2 r2 = add2(dup2(1.0f), drho2);
        if (fa && fb) {
            *reinterpret_cast<f2 *>(a.mom + n) = r2;
            *reinterpret_cast<f2 *>(a.mom + a.N + n) = ux2;
            *reinterpret_cast<f2 *>(a.mom + 2 * a.N + n) = uy2;
        } else {
            float r0, r1, u0, u1, v0, v1;
            up2(r2, r0, r1);
            up2(ux2, u0, u1);
            up2(uy2, v0, v1);
            const uint32_t m = fa ? n : n + 1u;
            a.mom[m] = fa ? r0 : r1;
            a.mom[a.N + m] = fa ? u0 : u1;
            a.mom[2 * a.N + m] = fa ? v0 : v1;
        }
    }
    if (fa && fb && !a.sr) {
        // both fluid, nearest rounding: each 32-bit word of a bundle pair is
        // one packed conversion of the two values it holds
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            float a0, b0, a1, b1, a2, b2;
            up2(g[3 * b], a0, b0);
            up2(g[3 * b + 1], a1, b1);
            up2(g[3 * b + 2], a2, b2);
            uint32_t *p = reinterpret_cast<uint32_t *>(a.dst + (uint32_t)b * 3u * a.N + 3u * n);
            p[0] = pack_rne<S>(a0, a1);
            p[1] = pack_rne<S>(a2, b0);
            p[2] = pack_rne<S>(b1, b2);
        }
        return;
    }
    uint32_t w[9];
    encode_pair<S>(a, n, g, fa, fb, w);
    store_pair<S>(a.dst, a.N, n, w);
}

// a.pf: L2 prefetch distance as for the 32-bit kernel (pairs of nodes for
// LPTL, rows for NPTL; 0 = off): the link bytes of the pair that far ahead
// are loaded first, and after the pair is stored its source records are
// prefetched into L2 when either node is fluid.
// Measured on the 134M-node porous lattice (FP16, bundle, NPTL 32 x 8): 72
// registers unbounded gives 119 GLUPS, 48 (five blocks of 256) 144, 40 with
// spills 143; one node per thread 126.
#ifndef LBM_PAIR_MINB
#define LBM_PAIR_MINB 5
#endif
template <class S, bool LINEAR>
__global__ void __launch_bounds__(kMaxTileThreads / 2, LBM_PAIR_MINB) k_two_lattice_pair(const Step<S> a) {
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    uint32_t x, y, n, np;
    bool ahead;
    chain_next();
    if (LINEAR) {
        n = 2u * (blockIdx.x * blockDim.x + threadIdx.x);
        if (n >= a.N) return;
        y = a.nx_magic ? (uint32_t)__umul64hi((unsigned long long)n, a.nx_magic) : n;
        x = n - y * nx;
        ahead = a.pf != 0u && a.N - n > 2u * a.pf;
        np = n + 2u * a.pf;
    } else {
        x = blockIdx.x * (uint32_t)a.tx + 2u * threadIdx.x;
        y = blockIdx.y * (uint32_t)a.ty + threadIdx.y;
        if (x >= nx || y >= ny) return;
        n = y * nx + x;
        ahead = a.pf != 0u && ny - y > a.pf;
        np = n + a.pf * nx;
    }
    const uint32_t lkp = ahead ? (uint32_t)*reinterpret_cast<const unsigned short *>(a.links + np) : 0xFFFFu;
    const uint32_t lk2 = *reinterpret_cast<const unsigned short *>(a.links + n);
    chain_wait();
    pair_update<S>(a, x, y, n, lk2);
    if (lkp != 0xFFFFu) prefetch_pair<S>(a.src, a.N, np);
}

// ------------------------------------------------------------ buffer grid
// Per parity, in triples of the three populations that leave a tile through
// one of its edges: for each tile column the column of nodes on its east edge
// (2, 5, 8), triple bx ny + y; then those of the west edges (0, 3, 6); then for
// each tile row the row of nodes on its north edge (6, 7, 8), triple
// by nx + x, and those of the south edges (0, 1, 2). Global coordinates along
// the edge: a node finds a crossing value by the same shift from its own
// position as in the lattice, with no division into source tile and local
// position, and in the bundle layout a row of triples replaces the lattice's
// own row. 6 (ntx ny + nty nx) elements, at most the 6 (tx + ty) per tile that
// are allocated.
template <class S> __device__ __forceinline__ int64_t halo_cols(const Step<S> &a) { return (int64_t)a.ntx * a.geo.ny; }
template <class S> __device__ __forceinline__ int64_t halo_rows(const Step<S> &a) { return (int64_t)a.nty * a.geo.nx; }
// First triple elements of node (., y) of tile column bx and of node (x, .) of tile row by.
template <class S>
__device__ __forceinline__ int64_t halo_col(const Step<S> &a, bool west, int bx, int y) {
    return 3 * ((west ? halo_cols(a) : 0) + (int64_t)bx * a.geo.ny + y);
}
template <class S>
__device__ __forceinline__ int64_t halo_row(const Step<S> &a, bool south, int by, int x) {
    return 6 * halo_cols(a) + 3 * ((south ? halo_rows(a) : 0) + (int64_t)by * a.geo.nx + x);
}

// Value S[(xs, ys)][j] of a node in another tile, as that tile published it.
template <class S>
__device__ __forceinline__ typename Codec<S>::C halo_read(const Step<S> &a, int xs, int ys, int j, int bx) {
    const int bxs = xs / a.tx;
    const int64_t s = bxs != bx ? halo_col(a, cx(j) < 0, bxs, ys) + j / 3 : halo_row(a, cy(j) < 0, ys / a.ty, xs) + j % 3;
    return Codec<S>::dec(a.halo_rd[s]);
}

// Publish the populations of an edge node that leave its tile.
template <class S>
__device__ __forceinline__ void halo_publish(const Step<S> &a, S *hw, int bx, int by, int x, int y, int x0, int y0,
                                             int x1, int y1, const S *e) {
    if (x == x1 || x == x0) {
        S *p = hw + halo_col(a, false, bx, y);
        if (x == x1) {
#pragma unroll
            for (int k = 0; k < 3; ++k) p[k] = e[3 * k + 2];
        }
        if (x == x0) {
            p += 3 * halo_cols(a);
#pragma unroll
            for (int k = 0; k < 3; ++k) p[k] = e[3 * k];
        }
    }
    if (y == y1 || y == y0) {
        S *p = hw + halo_row(a, false, by, x);
        if (y == y1) {
#pragma unroll
            for (int k = 0; k < 3; ++k) p[k] = e[6 + k];
        }
        if (y == y0) {
            p += 3 * halo_rows(a);
#pragma unroll
            for (int k = 0; k < 3; ++k) p[k] = e[k];
        }
    }
}

// What the pulls of a node (x, y) of tile (bx, by) off the domain edge read
// where they leave the tile: triples of the adjacent tile columns and rows, at
// the node's own y and x.
template <class S>
struct HaloPull {
    const S *w, *e, *s, *n;   // east edges of the column before, west edges of the one after; rows alike
    bool x0, x1, y0, y1;      // the node lies on its tile's west, east, south, north edge
    __device__ __forceinline__ HaloPull(const Step<S> &a, int bx, int by, int x, int y, int tx0, int tx1, int ty0,
                                        int ty1) {
        w = a.halo_rd + halo_col(a, false, bx - 1, y);
        e = a.halo_rd + halo_col(a, true, bx + 1, y);
        s = a.halo_rd + halo_row(a, false, by - 1, x);
        n = a.halo_rd + halo_row(a, true, by + 1, x);
        x0 = x == tx0;
        x1 = x == tx1;
        y0 = y == ty0;
        y1 = y == ty1;
    }
    // Does the pull of direction i cross the south or north edge (crosses_y),
    // or only the west or east one (crosses_x)? Through a corner it reads the
    // diagonal tile's row.
    __device__ __forceinline__ bool crosses_y(int i) const { return cy(i) > 0 ? y0 : (cy(i) < 0 ? y1 : false); }
    __device__ __forceinline__ bool crosses_x(int i) const {
        return (cx(i) > 0 ? x0 : (cx(i) < 0 ? x1 : false)) && !crosses_y(i);
    }
    __device__ __forceinline__ const S *at_x(int i) const { return (cx(i) > 0 ? w : e) + (i / 3 - 3 * cy(i)); }
    __device__ __forceinline__ const S *at_y(int i) const { return (cy(i) > 0 ? s : n) + (i % 3 - 3 * cx(i)); }
};

// ------------------------------------------------------------ NPOL
// One lattice, pull: every node reads its nine incoming values (in-tile
// sources from the lattice, cross-tile sources from the buffer grid of the
// previous update), the block barrier separates all reads from the in-place
// writes, and edge nodes publish their outgoing values for the next update.

// Pulls of a node off the domain edge: every lane runs the same code, the
// interior pull (neighbour value, or the own opposite value of a bounced link)
// reading the source tile's publication of the previous update where the source
// lies across a tile edge. In the bundle layout a row of the buffer grid has the
// lattice's own format, so crossing the south or north edge only changes the
// two rows (for whole warps, tile_x being a multiple of 32).
// Lattice and buffer grid lie in one workspace, and I is an element's index from
// the lattice's start: 32 bits where that reaches the grid's end (Step::near32),
// so that choosing a source is one select, 64 otherwise. 6000 x 3001 porous nodes,
// us an update, pointers before / 32-bit indices: FP32 stream 32 x 8 242 / 233,
// collision 64 x 4 294 / 277, bundle 64 x 4 230 / 226 (220 with the prefetch
// below), FP16 bundle 64 x 4 229 / 190. (A select avoided by issuing the pulled
// and the bounced load, each under its own predicate, costs 9 %.)
template <class S, int L, class I>
__device__ __forceinline__ void npol_pull(const Step<S> &a, int bx, int by, int x, int y, int x0, int x1, int y0,
                                          int y1, uint32_t n, uint32_t lk, typename Codec<S>::C *g) {
    constexpr I m = lay_mul<L>();
    // direction i from the lattice's start
    auto base = [N = (I)a.N](int i) -> I {
        return L == STREAM ? (I)i * N : (L == BUNDLE ? (I)(i / 3) * 3 * N + (I)(i % 3) : (I)i);
    };
    const I nx = (I)a.geo.nx, ny = (I)a.geo.ny;
    const I ncol = (I)a.ntx * ny, nrow = (I)a.nty * nx, grid = (I)(a.halo_rd - a.dst);
    const I w = grid + 3 * ((I)(bx - 1) * ny + (I)y);                     // east edges of the column before
    const I e = grid + 3 * (ncol + (I)(bx + 1) * ny + (I)y);              // west edges of the column after
    const I s = grid + 6 * ncol + 3 * ((I)(by - 1) * nx + (I)x);          // rows alike
    const I t = grid + 6 * ncol + 3 * (nrow + (I)(by + 1) * nx + (I)x);
    const bool xl = x == x0, xh = x == x1, yl = y == y0, yh = y == y1;
    const I own = m * (I)n;
    I rs = own + m * nx, rn = own - m * nx;   // rows y + 1 and y - 1: sources of c_y = -1 and +1
    if (L == BUNDLE) {
        rn += base(6);
        if (yh) rs = t;
        if (yl) rn = s;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (i == 4) {
            g[i] = Codec<S>::dec(a.dst[own + base(4)]);
            continue;
        }
        const bool cross_y = cy(i) > 0 ? yl : (cy(i) < 0 ? yh : false);
        I p;
        if (L == BUNDLE) {
            p = (cy(i) < 0 ? rs : (cy(i) > 0 ? rn : own + base(3))) + (I)(i % 3 - 3 * cx(i));
        } else {
            p = (cy(i) < 0 ? rs : (cy(i) > 0 ? rn : own)) + (base(i) - m * (I)cx(i));
            if (cross_y) p = (cy(i) > 0 ? s : t) + (I)(i % 3 - 3 * cx(i));
        }
        if ((cx(i) > 0 ? xl : (cx(i) < 0 ? xh : false)) && !cross_y)
            p = (cx(i) > 0 ? w : e) + (I)(i / 3 - 3 * cy(i));
        if ((lk >> link_bit(i)) & 1u) p = own + base(opp(i));
        g[i] = Codec<S>::dec(a.dst[p]);
    }
}

// PF: L2 prefetch of the record a.pf rows ahead, as in the two-lattice kernel.
// FP32 in the bundle layout: 3 % (in the stream layout, nine addresses a node, 2 %,
// left out); a kernel of its own, as the test for it costs a lattice that fits
// the L2 cache 5 %.
template <class S, int L, bool PF = false>
__device__ __forceinline__ void npol_tile(const Step<S> &a, int bx, int by, int lx, int ly, int lane) {
    using C = typename Codec<S>::C;
    const int nx = a.geo.nx, ny = a.geo.ny;
    const int x0 = bx * a.tx, y0 = by * a.ty;
    const int x1 = min(x0 + a.tx, nx) - 1, y1 = min(y0 + a.ty, ny) - 1;
    const int x = x0 + lx, y = y0 + ly;
    const bool valid = lx < a.tx && ly < a.ty && x <= x1 && y <= y1;
    S *lat = a.dst;
    uint32_t n = 0, lk = SOLID_LINKS;
    if (valid) {
        n = (uint32_t)y * (uint32_t)nx + (uint32_t)x;
        lk = a.links[n];
    }
    const bool ahead = PF && valid && (uint32_t)(ny - y) > a.pf;
    const uint32_t np = n + a.pf * (uint32_t)nx;
    const uint32_t lkp = ahead ? (uint32_t)a.links[np] : SOLID_LINKS;
    chain_wait();
    const bool fluid = lk != SOLID_LINKS;
    const unsigned F = __ballot_sync(__activemask(), fluid);
    (void)F;
    const bool zero_fill = false;   // measured: NPOL is 5 % faster without the sector zero fill
    const bool inner = x > x0 && x < x1 && y > y0 && y < y1;
    const bool dom_inner = x > 0 && x < nx - 1 && y > 0 && y < ny - 1;
    C g[9];
    if (fluid && dom_inner && a.near32) {
        npol_pull<S, L, uint32_t>(a, bx, by, x, y, x0, x1, y0, y1, n, lk, g);
    } else if (fluid && dom_inner) {
        npol_pull<S, L, int64_t>(a, bx, by, x, y, x0, x1, y0, y1, n, lk, g);
    } else if (fluid) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if (i == 4) {
                g[i] = ldp<S, L>(lat, a.N, n, 4);
            } else if ((lk >> link_bit(i)) & 1u) {
                g[i] = ldp<S, L>(lat, a.N, n, opp(i));
            } else {
                int xs, ys, j;
                if (map_pull(a.geo, x, y, i, xs, ys, j) != PULL_NODE)
                    g[i] = C(0);
                else if (xs >= x0 && xs <= x1 && ys >= y0 && ys <= y1)
                    g[i] = ldp<S, L>(lat, a.N, (uint32_t)ys * (uint32_t)nx + (uint32_t)xs, j);
                else
                    g[i] = halo_read(a, xs, ys, j, bx);
            }
        }
    }
    const C dnb = (fluid && x == 0 && a.geo.bw == INLET_EQ_NEUMANN) ? neighbour_drho<S, L>(a, lat, n, 0) : C(0);
    if (PF && lkp != SOLID_LINKS) prefetch_record<S, L>(lat, a.N, np);
    __syncthreads();
    if (fluid) {
        S e[9];
        collide_encode(a, (uint32_t)x, n, g, e, dnb);
        store_node<S, L>(lat, n, a.N, a.off32, e);
        if (!inner) halo_publish(a, a.halo_wr, bx, by, x, y, x0, y0, x1, y1, e);
    } else if (zero_fill) {
        store_zero<S, L>(lat, a.N, n, a.off32);  // whole-sector writes, as in two_lattice_node
    }
}

// LARGE: the lattice exceeds the L2 cache. Registers: 40 (three 512-thread
// blocks), 32 (four, spills) for 16-bit storage and large lattices in the stream
// layout, where that measured faster; us an update, 32 / 40 registers: stream 32 x 8
// 6000 x 3001 nodes 233 / 251, 1501 x 777 17.0 / 16.0; with the pulls by pointers
// 6000 x 3001 FP32 bundle 64 x 4 243 / 244 and 128 x 4 272 / 256, collision
// 338 / 305, FP16 241 / 247.
template <class S, int L, bool LARGE>
__global__ void __launch_bounds__(kMaxTileThreads, sizeof(S) == 8 ? 1
                                                   : L == COLLISION || (sizeof(S) == 4 && !(L == STREAM && LARGE)) ? 3 : 4)
    k_npol(const Step<S> a) {
    chain_next();
    npol_tile<S, L, LARGE && sizeof(S) == 4 && L == BUNDLE>(
        a, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y,
        (int)((threadIdx.y * blockDim.x + threadIdx.x) & 31u));
}

// TMA: the tile's populations arrive by one tensor copy (FP32 storage, stream
// or bundle layout; tm is the kernel's tensor-map parameter) and keep the
// bundle interleave in shared memory; otherwise every fluid node stages its
// own nine values.
template <class S, int L, bool TMA = false>
__device__ __forceinline__ void nsol_tile(const Step<S> &a, int bx, int by, int lx, int ly, int lane,
                                          unsigned char *smem_raw, const TmaDesc *tm = nullptr) {
    using C = typename Codec<S>::C;
    const int T = a.tx * a.ty;
    C *sm = reinterpret_cast<C *>(smem_raw);
    // slot of direction s of tile node t among the staged values
    auto si = [T](int s, int t) { return (TMA && L == BUNDLE) ? (s / 3) * 3 * T + 3 * t + s % 3 : s * T + t; };
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + sizeof(C) * 9 * T);
    chain_wait();
    if constexpr (TMA) {
        if (lx == 0 && ly == 0)
            tma_issue_3d(tm, sm, bar, L == BUNDLE ? 3 * bx * a.tx : bx * a.tx, by * a.ty, 0,
                         (uint32_t)(sizeof(C) * 9 * T));
        __syncthreads();   // the barrier is initialised before anyone waits on it
    }
    const int nx = a.geo.nx, ny = a.geo.ny;
    const int x0 = bx * a.tx, y0 = by * a.ty;
    const int x1 = min(x0 + a.tx, nx) - 1, y1 = min(y0 + a.ty, ny) - 1;
    const bool member = lx < a.tx && ly < a.ty;  // thread has a slot in this tile
    const int tid = member ? ly * a.tx + lx : 0;
    const int x = x0 + lx, y = y0 + ly;
    const bool valid = member && x <= x1 && y <= y1;
    S *lat = a.dst;
    uint32_t n = 0, lk = SOLID_LINKS;
    if (valid) {
        n = (uint32_t)y * (uint32_t)nx + (uint32_t)x;
        lk = a.links[n];
    }
    const bool fluid = lk != SOLID_LINKS;
    const unsigned F = __ballot_sync(__activemask(), fluid);
    (void)F;
    const bool zero_fill = false;   // measured: NSOL is 2 % faster without the sector zero fill
    if (!TMA && fluid) {
#pragma unroll
        for (int s = 0; s < 9; ++s) sm[si(s, tid)] = ldp<S, L>(lat, a.N, n, s);
    }
    const C dnb = (fluid && x == 0 && a.geo.bw == INLET_EQ_NEUMANN) ? neighbour_drho<S, L>(a, lat, n, 1) : C(0);
    // Substitutions for pulls the in-tile exchange does not cover, read
    // before the first barrier: the lattice holds the previous state until
    // the stores after the last barrier, and other tiles' values come from
    // the buffer grid.
    C fix[9];
    unsigned fixmask = 0;
    const bool dom_inner = x > 0 && x < nx - 1 && y > 0 && y < ny - 1;
    if (fluid && dom_inner && !(x > x0 && x < x1 && y > y0 && y < y1)) {
        // Tile edge inside the domain: values from other tiles come from their
        // buffer grid (same slots as NPOL); in-tile sources are exchanged.
        const HaloPull<S> H(a, bx, by, x, y, x0, x1, y0, y1);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            fix[i] = C(0);
            if (i == 4 || ((lk >> link_bit(i)) & 1u)) continue;
            if (!H.crosses_y(i) && !H.crosses_x(i)) continue;
            fixmask |= 1u << i;
            fix[i] = Codec<S>::dec(H.crosses_y(i) ? *H.at_y(i) : *H.at_x(i));
        }
    } else if (fluid && !(x > x0 && x < x1 && y > y0 && y < y1)) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            fix[i] = C(0);
            if (i == 4 || ((lk >> link_bit(i)) & 1u)) continue;
            int xs, ys, j;
            const int kind = map_pull(a.geo, x, y, i, xs, ys, j);
            const bool in_tile = kind == PULL_NODE && xs >= x0 && xs <= x1 && ys >= y0 && ys <= y1;
            if (in_tile && j == i && xs == x - cx(i) && ys == y - cy(i)) continue;  // exchanged
            fixmask |= 1u << i;
            if (kind != PULL_NODE) continue;  // inlet unknown
            if (in_tile)
                fix[i] = ldp<S, L>(lat, a.N, (uint32_t)ys * (uint32_t)nx + (uint32_t)xs, opp(j));
            else
                fix[i] = halo_read(a, xs, ys, j, bx);
        }
    }
    if constexpr (TMA) {
        bool done = tma_wait(bar);
        if (!__syncthreads_and(done)) {
            // let a late copy land before the block's shared memory is released
            if (!done) done = tma_wait(bar);
            if (lx == 0 && ly == 0) atomicOr(a.err, 2u);
            return;
        }
    } else {
        __syncthreads();
    }
    if (fluid) {
        // partner x + c_i fluid <=> the pull of direction 8-i from it does not bounce
#pragma unroll
        for (int i = 5; i < 9; ++i) {
            const int px = lx + cx(i), py = ly + cy(i);
            if (px >= 0 && px < a.tx && py < a.ty && x0 + px <= x1 && y0 + py <= y1) {
                const int pt = py * a.tx + px;
                if (!((lk >> link_bit(opp(i))) & 1u)) {
                    C t = sm[si(opp(i), tid)];
                    sm[si(opp(i), tid)] = sm[si(i, pt)];
                    sm[si(i, pt)] = t;
                }
            }
        }
    }
    __syncthreads();
    if (fluid) {
        C g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = ((fixmask >> i) & 1u) ? fix[i] : sm[si(i, tid)];
        S e[9];
        collide_encode(a, (uint32_t)x, n, g, e, dnb);
#pragma unroll
        for (int i = 0; i < 9; ++i) lat[addr<L>(a.N, n, opp(i))] = e[i];
        if (!(x > x0 && x < x1 && y > y0 && y < y1))
            halo_publish(a, a.halo_wr, bx, by, x, y, x0, y0, x1, y1, e);
    } else if (zero_fill) {
        store_zero<S, L>(lat, a.N, n, a.off32);
    }
}

// Registers: 40 (three 512-thread blocks), 32 (four) where the tile is staged by
// a tensor copy and in the collision layout. us an update of 8192 x 4096 porous
// nodes, 32 / 40 registers: FP32 bundle 64 x 4 without the copy 553 / 522, with it
// 443 / 477, stream 32 x 8 558 / 540, collision 608 / 731, FP16 bundle 575 / 574.
template <class S, int L>
__global__ void __launch_bounds__(kMaxTileThreads, sizeof(S) == 8 ? 1 : (L == COLLISION ? 4 : 3)) k_nsol(const Step<S> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_next();
    nsol_tile<S, L>(a, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y,
                    (int)((threadIdx.y * blockDim.x + threadIdx.x) & 31u), smem_raw);
}

// NSOL with the tile staged by a tensor copy; shared memory: the tile's
// 9 T values, then the copy's mbarrier.
template <class S, int L>
__global__ void __launch_bounds__(kMaxTileThreads, 4)
    k_nsol_tma(const Step<S> a, const __grid_constant__ TmaDesc tm) {
    extern __shared__ __align__(128) unsigned char smem_tma[];
    chain_next();
    nsol_tile<S, L, true>(a, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y,
                          (int)((threadIdx.y * blockDim.x + threadIdx.x) & 31u), smem_tma, &tm);
}

// ------------------------------------------------------------ AA pattern
// In-place streaming with one lattice and no buffer grid (the AA pattern of
// Bailey et al., which Sec. 3.3 names as a state-of-the-art scheme). Updates
// alternate between two phases on the same array:
//  phase 0 (state: post-collision values in opposite slots, slot 8-i of x
//           holds S[x]_i): pull every value through the edge mapping,
//           collide, and store each result in the slot its puller reads next,
//           i.e. slot i of x + c_i (slot 8-i of x itself for a bounced link);
//  phase 1 (state: every node's pulled values in its own slots): read them,
//           collide, store the results in the node's opposite slots.
// Each slot is read and written by the same node within a phase, so no
// synchronisation is needed. Zero-gradient outflow reads one slot from two
// nodes and is not supported here.
template <class S, int L, int PHASE, bool CHAIN>
__device__ __forceinline__ void aa_node(const Step<S> &a, uint32_t x, uint32_t y, int lane) {
    constexpr int phase = PHASE;
    using C = typename Codec<S>::C;
    const uint32_t nx = (uint32_t)a.geo.nx, ny = (uint32_t)a.geo.ny;
    const uint32_t n = y * nx + x;
    const uint32_t lk = a.links[n];
    if (CHAIN) chain_wait();
    S *lat = a.dst;
    const bool fluid = lk != SOLID_LINKS;
    const unsigned F = __ballot_sync(__activemask(), fluid);
    if (!fluid) {
        if (shares_sector<S, L>(F, lane)) store_zero<S, L>(lat, a.N, n, a.off32);
        return;
    }
    C g[9];
    S e[9];
    if (phase == 1) {
        if (a.off32) {
            S *own = lat + lay_mul<L>() * n;
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = Codec<S>::dec(own[(ptrdiff_t)lay_base<L>(a.N, i)]);
            collide_encode(a, x, n, g, e);
#pragma unroll
            for (int i = 0; i < 9; ++i) own[(ptrdiff_t)lay_base<L>(a.N, opp(i))] = e[i];
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = ldp<S, L>(lat, a.N, n, i);
            collide_encode(a, x, n, g, e);
#pragma unroll
            for (int i = 0; i < 9; ++i) lat[addr<L>(a.N, n, opp(i))] = e[i];
        }
        return;
    }
    const bool interior = (x - 1u < nx - 2u) && (y - 1u < ny - 2u);
    if (interior && a.off32) {
        // 32-bit element indices with constant offsets: pull slot 8-i of
        // x - c_i (or own slot i when bounced), push to slot i of x + c_i (or
        // own slot 8-i). Each access is one select between two indices and one
        // widening address computation (measured 2 % faster than selecting
        // between 64-bit row pointers, at the same 40 registers).
        const uint32_t own = lay_mul<L>() * n;
        const uint32_t ra = own + lay_mul<L>() * nx;  // row y+1
        const uint32_t rb = own - lay_mul<L>() * nx;  // row y-1
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if (i == 4) {
                g[i] = Codec<S>::dec(lat[own + lay_base<L>(a.N, 4)]);
                continue;
            }
            const uint32_t row = cy(i) < 0 ? ra : (cy(i) > 0 ? rb : own);
            const uint32_t ip = row + lay_base<L>(a.N, opp(i)) - (uint32_t)((int)lay_mul<L>() * cx(i));
            const uint32_t ib = own + lay_base<L>(a.N, i);
            g[i] = Codec<S>::dec(lat[((lk >> link_bit(i)) & 1u) ? ib : ip]);
        }
        collide_encode(a, x, n, g, e);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if (i == 4) {
                lat[own + lay_base<L>(a.N, 4)] = e[4];
                continue;
            }
            const uint32_t row = cy(i) > 0 ? ra : (cy(i) < 0 ? rb : own);
            const uint32_t ip = row + lay_base<L>(a.N, i) + (uint32_t)((int)lay_mul<L>() * cx(i));
            const uint32_t ib = own + lay_base<L>(a.N, opp(i));
            lat[((lk >> link_bit(opp(i))) & 1u) ? ib : ip] = e[i];
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (i == 4) {
            g[i] = ldp<S, L>(lat, a.N, n, 4);
        } else if ((lk >> link_bit(i)) & 1u) {
            g[i] = ldp<S, L>(lat, a.N, n, i);  // slot i of x holds S[x]_{8-i}
        } else if (interior) {
            g[i] = ldp<S, L>(lat, a.N, n - (uint32_t)(cy(i) * (int)nx + cx(i)), opp(i));
        } else {
            int xs, ys, j;
            if (map_pull(a.geo, (int)x, (int)y, i, xs, ys, j) == PULL_NODE)
                g[i] = ldp<S, L>(lat, a.N, (uint32_t)ys * nx + (uint32_t)xs, opp(j));
            else
                g[i] = C(0);  // inlet unknown
        }
    }
    collide_encode(a, x, n, g, e);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (i == 4) {
            lat[addr<L>(a.N, n, 4)] = e[4];
        } else if ((lk >> link_bit(opp(i))) & 1u) {
            lat[addr<L>(a.N, n, opp(i))] = e[i];  // bounced back into this node
        } else if (interior) {
            lat[addr<L>(a.N, n + (uint32_t)(cy(i) * (int)nx + cx(i)), i)] = e[i];
        } else {
            // The neighbour x + c_i (wrapped across periodic edges) pulls
            // S[x]_i into slot i whenever it lies in the domain; otherwise the
            // puller is found through the edge mapping: every fluid node
            // within one cell whose mapped pull reads S[x]_i receives it.
            int tx_ = (int)x + cx(i), ty_ = (int)y + cy(i);
            bool in = true;
            if (tx_ < 0 || tx_ >= (int)nx) {
                if (a.geo.bw == PERIODIC) tx_ = tx_ < 0 ? tx_ + (int)nx : tx_ - (int)nx;
                else in = false;
            }
            if (ty_ < 0 || ty_ >= (int)ny) {
                if (a.geo.bs == PERIODIC) ty_ = ty_ < 0 ? ty_ + (int)ny : ty_ - (int)ny;
                else in = false;
            }
            if (in) {
                lat[addr<L>(a.N, (uint32_t)ty_ * nx + (uint32_t)tx_, i)] = e[i];
                continue;
            }
#pragma unroll 1
            for (int dy = -1; dy <= 1; ++dy)
#pragma unroll 1
                for (int dx = -1; dx <= 1; ++dx) {
                    int ux = (int)x + dx, uy = (int)y + dy;
                    if (ux < 0 || ux >= (int)nx) {
                        if (a.geo.bw != PERIODIC) continue;
                        ux = ux < 0 ? ux + (int)nx : ux - (int)nx;
                    }
                    if (uy < 0 || uy >= (int)ny) {
                        if (a.geo.bs != PERIODIC) continue;
                        uy = uy < 0 ? uy + (int)ny : uy - (int)ny;
                    }
                    const uint32_t m = (uint32_t)uy * nx + (uint32_t)ux;
                    const uint32_t ml = a.links[m];
                    if (ml == SOLID_LINKS) continue;
#pragma unroll 1
                    for (int k = 0; k < 9; ++k) {
                        if (k == 4 || ((ml >> link_bit(k)) & 1u)) continue;
                        int xs, ys, j;
                        if (map_pull(a.geo, ux, uy, k, xs, ys, j) == PULL_NODE && xs == (int)x &&
                            ys == (int)y && j == i)
                            lat[addr<L>(a.N, m, k)] = e[i];
                    }
                }
        }
    }
}

// CHAIN: as for k_two_lattice (134M nodes, bundle 64 x 2: 1.158 ms an update with
// the wait).
template <class S, int L, int PHASE, bool CHAIN = true>
__global__ void __launch_bounds__(kMaxTileThreads, sizeof(S) == 8 ? 1 : (PHASE == 0 || L == STREAM ? 3 : 4)) k_aa(const Step<S> a) {
    if (CHAIN) chain_next();
    const uint32_t x = blockIdx.x * a.tx + threadIdx.x;
    const uint32_t y = blockIdx.y * a.ty + threadIdx.y;
    if (x >= (uint32_t)a.geo.nx || y >= (uint32_t)a.geo.ny) return;
    // L2 prefetch of the record a.pf rows ahead, as in the two-lattice kernel
    constexpr bool PF = sizeof(S) == 4 && L != COLLISION;
    const bool ahead = PF && a.pf != 0u && (uint32_t)a.geo.ny - y > a.pf;
    const uint32_t np = (y + a.pf) * (uint32_t)a.geo.nx + x;
    const uint32_t lkp = ahead ? (uint32_t)a.links[np] : SOLID_LINKS;
    aa_node<S, L, PHASE, CHAIN>(a, x, y, (int)((threadIdx.y * blockDim.x + threadIdx.x) & 31u));
    if (PF && lkp != SOLID_LINKS) prefetch_record<S, L>(a.dst, a.N, np);
}

// ------------------------------------------------------------ batches
// Many independent lattices advanced by one persistent launch per update.
// The work list holds one entry per work item of every case: four tiles of
// a two-lattice case (LPTL tile = 256 consecutive nodes), one tile of a
// one-lattice case. Blocks take entries round-robin, so that neighbouring rows
// are updated at about the same time and share L2. A block's next case record
// is copied into the other of two shared-memory buffers while it updates the
// present item (one barrier per change of case, no exposed latency), and in a
// two-lattice item the records of the next tile are prefetched into L2 when
// the batch exceeds the L2 cache. Bound by memory latency at 75 % occupancy (40
// registers; 48 and fewer blocks were slower) and, reading a case's constants
// from shared memory, by instruction issue: 48 channels of 8.7M nodes, FP32,
// 100 updates 13.70 ms with one buffer and three barriers per change of case,
// 13.26 with two, 0.24 of it by the prefetch.
constexpr int kBatchThreads = 256;
constexpr int kBatchSuper = 4;  // tiles per work item of a two-lattice case

// One record per case, lattice parity (source lattice, buffer-grid parity) and
// whether moments are stored: index (2 moments + parity) ncases + case.
template <class S>
struct BatchCase {
    Step<S> st;                    // constants, links, pointers, tile shape of the case
    unsigned long long ntx_magic;  // ceil(2^64 / ntx), 0 when ntx == 1
    int layout, algo;
    int pf;                        // L2 prefetch of the next tile's records
};

struct BatchTile {
    uint32_t c;                 // case index
    uint32_t t;                 // work item within the case
};

// stage(): called once during the item, by every thread.
template <class S, int L, class Stage>
__device__ __forceinline__ void batch_item(const BatchCase<S> &bc, int algo, uint32_t t, int tid,
                                           unsigned char *smem, Stage stage) {
    const Step<S> &a = bc.st;
    const int lane = tid & 31;
    const bool ahead = sizeof(S) == 4 && L != COLLISION && bc.pf != 0;
    if (algo == LPTL) {
        // each tile's link bytes are loaded one tile ahead (256 channels 74.3 ->
        // 77.7 GLUPS, 71.8 before the pulls above)
        constexpr uint32_t T = kBatchThreads;
        uint32_t n = t * kBatchSuper * T + (uint32_t)tid;
        bool in = n < a.N;
        uint32_t lk = in ? (uint32_t)a.links[n] : SOLID_LINKS;
        chain_wait();
#pragma unroll 1
        for (int k = 0; k < kBatchSuper; ++k, n += T) {
            const bool more = k + 1 < kBatchSuper && in && a.N - n > T;
            const uint32_t lkn = more ? (uint32_t)a.links[n + T] : SOLID_LINKS;
            if (in) {
                if (ahead && more) prefetch_record<S, L>(a.src, a.N, n + T);
                const uint32_t y = a.nx_magic ? (uint32_t)__umul64hi((unsigned long long)n, a.nx_magic) : n;
                two_lattice_known<S, L, true, true>(a, n - y * (uint32_t)a.geo.nx, y, n, lk, lane);
            }
            in = more;
            lk = lkn;
            if (k == 0) stage();
        }
        return;
    }
    const int lx = tid % a.tx, ly = tid / a.tx;
    if (algo == NPTL) {
        const uint32_t ntiles = (uint32_t)a.ntx * (uint32_t)((a.geo.ny + a.ty - 1) / a.ty);
#pragma unroll 1
        for (int k = 0; k < kBatchSuper; ++k) {
            const uint32_t tt = t * kBatchSuper + k;
            if (tt < ntiles) {
                const uint32_t by = bc.ntx_magic ? (uint32_t)__umul64hi((unsigned long long)tt, bc.ntx_magic) : tt;
                const uint32_t bx = tt - by * (uint32_t)a.ntx;
                const int x = (int)bx * a.tx + lx, y = (int)by * a.ty + ly;
                if (ahead && k + 1 < kBatchSuper && ly < a.ty && y < a.geo.ny && x + a.tx < a.geo.nx)
                    prefetch_record<S, L>(a.src, a.N, (uint32_t)y * (uint32_t)a.geo.nx + (uint32_t)(x + a.tx));
                if (ly < a.ty && x < a.geo.nx && y < a.geo.ny) two_lattice_node<S, L, true, true>(a, x, y, lane);
            }
            if (k == 0) stage();
        }
        return;
    }
    stage();
    const int by = (int)(t / (uint32_t)a.ntx), bx = (int)(t - (uint32_t)by * (uint32_t)a.ntx);
    if (algo == NPOL)
        npol_tile<S, L>(a, bx, by, lx, ly, lane);
    else
        nsol_tile<S, L>(a, bx, by, lx, ly, lane, smem);
}

// LK / AK: the layout / algorithm shared by every case, or -1 (any).
// rec0: first record of the update's parity and moments flag (all cases start
// together at update 0, so they share the parity).
template <class S, int LK, int AK>
__global__ void __launch_bounds__(kBatchThreads, LK < 0 ? 2 : (AK <= NPTL ? (sizeof(S) == 8 ? 4 : 6) : 3))
    k_batch(const BatchCase<S> *recs, const BatchTile *tiles, uint32_t ntiles, int toff) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(16) BatchCase<S> buf[2];
    constexpr int kWords = (int)(sizeof(BatchCase<S>) / 4);
    constexpr int kToff = (int)(offsetof(BatchCase<S>, st.toff) / 4);
    static_assert(kWords <= kBatchThreads, "one word per thread");
    const int tid = threadIdx.x;
    chain_next();
    int cur = 0;
    uint32_t w = blockIdx.x;
    BatchTile bt = tiles[w];
    auto fetch = [&](int b, uint32_t c) {   // asynchronous copy of record c into buffer b
        if (tid < kWords) {
            uint32_t *to = reinterpret_cast<uint32_t *>(&buf[b]) + tid;
            const uint32_t *from = reinterpret_cast<const uint32_t *>(recs + c) + tid;
            if (tid == kToff)
                *to = (uint32_t)toff;
            else
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(to)),
                             "l"(from)
                             : "memory");
        }
    };
    auto arrive = [] { asm volatile("cp.async.wait_all;" ::: "memory"); };
    fetch(0, bt.c);
    arrive();
    __syncthreads();
    for (;;) {
        const uint32_t wn = w + gridDim.x;
        BatchTile next = bt;
        if (wn < ntiles) next = tiles[wn];
        const bool change = next.c != bt.c;   // the same in every thread
        auto stage = [&] {
            if (change) fetch(cur ^ 1, next.c);
        };
        const BatchCase<S> &bc = buf[cur];
        const int algo = AK >= 0 ? AK : bc.algo;
        const int layout = LK >= 0 ? LK : bc.layout;
        switch (layout) {
            case STREAM: batch_item<S, STREAM>(bc, algo, bt.t, tid, smem, stage); break;
            case BUNDLE: batch_item<S, BUNDLE>(bc, algo, bt.t, tid, smem, stage); break;
            default: batch_item<S, COLLISION>(bc, algo, bt.t, tid, smem, stage); break;
        }
        if (wn >= ntiles) return;
        if (change) arrive();
        // the next record is complete, and an NSOL tile's shared memory is free again
        if (change || algo == NSOL) __syncthreads();
        if (change) cur ^= 1;
        bt = next;
        w = wn;
    }
}

template <class S>
size_t batch_smem_bytes(bool nsol) {   // NSOL stages its tile
    return nsol ? sizeof(typename Codec<S>::C) * 9 * kBatchThreads : 0;
}

// kind = layout * 4 + algo when every case shares them, else -1.
#define LBM_BATCH_KINDS(X, S)                                                              \
    X(S, -1, -1) X(S, 0, 0) X(S, 0, 1) X(S, 0, 2) X(S, 0, 3) X(S, 1, 0) X(S, 1, 1) X(S, 1, 2) \
        X(S, 1, 3) X(S, 2, 0) X(S, 2, 1) X(S, 2, 2) X(S, 2, 3)

template <class S>
cudaError_t op_batch_step(int kind, const void *recs, int ncases, const void *tiles, uint32_t ntiles, int grid, int cur,
                          int toff, int want_moments, cudaStream_t st) {
    const size_t sm = batch_smem_bytes<S>(kind < 0 || kind % 4 == NSOL);
    const auto *c = (const BatchCase<S> *)recs + (size_t)((want_moments ? 2 : 0) + cur) * ncases;
    const auto *t = (const BatchTile *)tiles;
    cudaError_t e = cudaErrorInvalidValue;
#define LBM_BATCH_LAUNCH(S_, L_, A_)                                                       \
    if (kind == ((L_) < 0 ? -1 : (L_) * 4 + (A_)))                                        \
        e = launch_update(sizeof(S) < 8, k_batch<S_, L_, A_>, dim3(grid), dim3(kBatchThreads), sm, st, c, t, ntiles, toff);
    LBM_BATCH_KINDS(LBM_BATCH_LAUNCH, S)
#undef LBM_BATCH_LAUNCH
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

template <class S, int LK, int AK>
int batch_grid_of() {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch<S, LK, AK>, kBatchThreads,
                                                      batch_smem_bytes<S>(LK < 0 || AK == NSOL)) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms * (per_sm > 0 ? per_sm : 1);
}

template <class S>
int op_batch_grid(int kind) {
#define LBM_BATCH_GRID(S_, L_, A_) \
    if (kind == ((L_) < 0 ? -1 : (L_) * 4 + (A_))) return batch_grid_of<S_, L_, A_>();
    LBM_BATCH_KINDS(LBM_BATCH_GRID, S)
#undef LBM_BATCH_GRID
    return 0;
}

// Host: the device record of one case for a lattice parity, with or without
// moments (pointers from its HostArgs).
template <class S>
void op_batch_case(const HostArgs &h, int parity, int moments, int pf, void *out) {
    BatchCase<S> c;
    memset(&c, 0, sizeof(c));
    c.st = make_step<S>(h, StepCall{h.pop[1] ? parity : 0, parity, 0, moments});
    c.ntx_magic = h.ntx > 1 ? (~0ull / (unsigned long long)h.ntx) + 1ull : 0ull;
    c.layout = h.layout;
    c.algo = h.algo;
    c.pf = pf;
    memcpy(out, &c, sizeof(c));
}

// ------------------------------------------------------------ state kernels
template <class S, int L>
__global__ void k_init(const Step<S> a, const double *rho, const double *ux, const double *uy,
                       uint32_t n0, uint32_t count, int rev) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count) return;
    const uint32_t n = n0 + t;
    if (a.links[n] == SOLID_LINKS) return;
    const double dr = rho ? rho[t] - 1.0 : 0.0;
    const double vx = ux ? ux[t] : 0.0, vy = uy ? uy[t] : 0.0;
    const double usq = vx * vx + vy * vy;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const double w = i == 4 ? 4.0 / 9.0 : ((i & 1) ? 1.0 / 9.0 : 1.0 / 36.0);
        const double cu = cx(i) * vx + cy(i) * vy;
        const double h = w * (dr + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq);
        typename Codec<S>::C hc = (typename Codec<S>::C)h;
        a.dst[addr<L>(a.N, n, rev ? opp(i) : i)] = Codec<S>::enc(hc, false, 0u);
    }
}

// Solid nodes hold h = 0 (restored after host writes of the state).
template <class S, int L>
__global__ void k_zero_solid(const Step<S> a, S *lat) {
    const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= a.N || a.links[n] != SOLID_LINKS) return;
    store_zero<S, L>(lat, a.N, n, a.off32);
}

// Copy every tile-edge node's outgoing values into one buffer-grid parity.
template <class S, int L>
__global__ void k_publish(const Step<S> a, S *hw, int rev) {
    const int nx = a.geo.nx, ny = a.geo.ny;
    const int bx = blockIdx.x, by = blockIdx.y;
    const int x0 = bx * a.tx, y0 = by * a.ty;
    const int x1 = min(x0 + a.tx, nx) - 1, y1 = min(y0 + a.ty, ny) - 1;
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x > x1 || y > y1) return;
    if (x > x0 && x < x1 && y > y0 && y < y1) return;
    const uint32_t n = (uint32_t)y * (uint32_t)nx + (uint32_t)x;
    if (a.links[n] == SOLID_LINKS) return;
    S e[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) e[i] = a.src[addr<L>(a.N, n, rev ? opp(i) : i)];
    halo_publish(a, hw, bx, by, x, y, x0, y0, x1, y1, e);
}

// Nodes n0 .. n0 + count - 1 of the stored state to / from rows of canonical
// order, rows[i stride + n - n0], in page-locked, mapped host memory; H = double or
// float; rev: populations are stored in opposite slots. The host side of the copy
// is the coalesced one, and it alone bounds these kernels (the CPU-GPU link).
// Solid nodes are stored as zeros.
template <class S, int L, class H>
__global__ void __launch_bounds__(256) k_export(const S *lat, uint32_t N, int rev, H *rows, uint32_t n0,
                                                uint32_t count, size_t stride) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
#pragma unroll
    for (int i = 0; i < 9; ++i) rows[i * stride + k] = (H)ldp<S, L>(lat, N, n0 + k, rev ? opp(i) : i);
}
template <class S, int L, class H>
__global__ void __launch_bounds__(256) k_import(S *lat, const uint8_t *links, uint32_t N, int rev, const H *rows,
                                                uint32_t n0, uint32_t count, size_t stride) {
    using C = typename Codec<S>::C;
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    const uint32_t n = n0 + k;
    const bool solid = links[n] == SOLID_LINKS;
#pragma unroll
    for (int i = 0; i < 9; ++i)
        lat[addr<L>(N, n, rev ? opp(i) : i)] = Codec<S>::enc(solid ? C(0) : (C)rows[i * stride + k], false, 0u);
}

// Moments from a stored state: rho = 1 + sum h, v = sum h c (- F/2 for a
// post-collision state, since the collision adds F to sum f c), in the
// arithmetic type (used for the moments reported after lbm_init).
template <class S, int L>
__global__ void k_state_moments(const Step<S> a, int rev, int post) {
    using C = typename Codec<S>::C;
    using A = Ar<C>;
    const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= a.N) return;
    C *m = (C *)a.mom;
    if (a.links[n] == SOLID_LINKS) {
        m[n] = C(1);
        m[a.N + n] = C(0);
        m[2 * a.N + n] = C(0);
        return;
    }
    C h[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = ldp<S, L>(a.src, a.N, n, rev ? opp(i) : i);
    C r = C(0), jx = C(0), jy = C(0);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        r = A::add(r, h[i]);
        if (cx(i) != 0) jx = cx(i) > 0 ? A::add(jx, h[i]) : A::sub(jx, h[i]);
        if (cy(i) != 0) jy = cy(i) > 0 ? A::add(jy, h[i]) : A::sub(jy, h[i]);
    }
    if (post) {
        jx = A::sub(jx, a.k.r.hfx);
        jy = A::sub(jy, a.k.r.hfy);
    }
    m[n] = A::add(C(1), r);
    m[a.N + n] = jx;
    m[2 * a.N + n] = jy;
}

// Deterministic FP64 block reduction (fixed grid and tree).
template <int W>
__device__ __forceinline__ void block_reduce_store(double (&v)[W], double *partials) {
    __shared__ double red[W][kReduceThreads];
    for (int w = 0; w < W; ++w) red[w][threadIdx.x] = v[w];
    __syncthreads();
    for (int s = kReduceThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
            for (int w = 0; w < W; ++w) red[w][threadIdx.x] += red[w][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int w = 0; w < W; ++w) partials[blockIdx.x * W + w] = red[w][0];
}

template <class S, int L>
__global__ void __launch_bounds__(kReduceThreads) k_mass(const Step<S> a, int rev, double *partials) {
    double acc[1] = {0.0};
    for (uint64_t n64 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; n64 < a.N;
         n64 += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t n = (uint32_t)n64;
        if (a.links[n] == SOLID_LINKS) continue;
        double r = 1.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) r += (double)ldp<S, L>(a.src, a.N, n, rev ? opp(i) : i);
        acc[0] += r;
    }
    block_reduce_store<1>(acc, partials);
}

template <class S, int L>
__global__ void __launch_bounds__(kReduceThreads) k_force(const Step<S> a, int rev, const uint8_t *body,
                                                          double *partials) {
    double acc[2] = {0.0, 0.0};
    const int nx = a.geo.nx, ny = a.geo.ny;
    for (uint64_t n64 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; n64 < a.N;
         n64 += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t n = (uint32_t)n64;
        if (a.links[n] == SOLID_LINKS) continue;
        const int y = a.nx_magic ? (int)__umul64hi((unsigned long long)n, a.nx_magic) : (int)n;
        const int x = (int)n - y * nx;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if (i == 4) continue;
            int bx = x + cx(i), by = y + cy(i);
            if (bx < 0 || bx >= nx) {
                if (a.geo.bw != PERIODIC) continue;
                bx = bx < 0 ? bx + nx : bx - nx;
            }
            if (by < 0 || by >= ny) {
                if (a.geo.bs != PERIODIC) continue;
                by = by < 0 ? by + ny : by - ny;
            }
            const uint32_t m = (uint32_t)by * (uint32_t)nx + (uint32_t)bx;
            const bool hit = body ? body[m] != 0 : a.links[m] == SOLID_LINKS;
            if (!hit) continue;
            const double w = (i & 1) ? 1.0 / 9.0 : 1.0 / 36.0;
            const double f = w + (double)ldp<S, L>(a.src, a.N, n, rev ? opp(i) : i);
            acc[0] += 2.0 * cx(i) * f;
            acc[1] += 2.0 * cy(i) * f;
        }
    }
    block_reduce_store<2>(acc, partials);
}

template <class C>
__global__ void k_moments_f32(const C *mom, uint32_t N, float *r, float *u, float *v) {
    const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    r[n] = (float)mom[n];
    u[n] = (float)mom[N + n];
    v[n] = (float)mom[2 * (size_t)N + n];
}

// ------------------------------------------------------------ launchers
template <class S, int L>
int lptl_block() {
    static int block = [] {
        int minGrid = 0, b = 256;
        if (cudaOccupancyMaxPotentialBlockSize(&minGrid, &b, k_two_lattice<S, L, true>, 0,
                                               kMaxTileThreads) != cudaSuccess) {
            cudaGetLastError();
            b = 256;
        }
        return b;
    }();
    return block;
}

// Node pairs: 16-bit storage in the bundle layout, nx even, 32-bit offsets,
// unless LBM_FLAG_NO_PAIRS asks for one node per thread. (The stream layout
// measured 7 % slower with pairs than with one node per thread: nine
// separate arrays give each pair nine 32-bit stores and nine prefetches.)
template <class S, int L>
bool pairs_ok(const HostArgs &h) {
    return sizeof(S) == 2 && L == BUNDLE && (h.nx % 2) == 0 && (9 * h.N) < (int64_t(1) << 32) &&
           !(h.flags & 0x20u);
}

// Rows of a tile that one block of the per-node kernels (no exchange within a
// tile) updates: a lattice of few tiles is cut into smaller blocks, so that
// its nodes spread over all SMs. 256 x 64 nodes in 32 x 8 tiles are 64 blocks on
// 152 SMs, and the FP64 lanes of 88 SMs are idle; in blocks of 32 x 1 an FP64
// update takes 3.9 instead of 6.6 us, an FP32 one (chained) 1.65 instead of 1.87.
inline int rows_per_block(const HostArgs &h) {
    int ty = h.tile_y;
    int64_t blocks = (int64_t)h.ntx * h.nty;
    while (blocks < 4 * (int64_t)h.sms && ty % 2 == 0 && h.tile_x * ty >= 64) {
        ty /= 2;
        blocks = (int64_t)h.ntx * ((h.ny + ty - 1) / ty);
    }
    return ty;
}

template <class S, int L>
cudaError_t step_layout(const HostArgs &h, const Step<S> &a0, int phase, cudaStream_t st) {
    using C = typename Codec<S>::C;
    const dim3 tile(h.tile_x, h.tile_y), grid(h.ntx, h.nty);
    const bool chain = chained_updates(sizeof(S), h.N);
    Step<S> a = a0;
    if (h.algo == LPTL) {
        if constexpr (sizeof(S) == 2 && L == BUNDLE) {
            if (pairs_ok<S, L>(h)) {
                const dim3 b(128), g((unsigned)((h.N / 2 + 127) / 128));
                return launch_update(chain && spread_evenly(g, b, h.sms), k_two_lattice_pair<S, true>, g, b, 0, st, a);
            }
        }
        const int b = h.block_1d;
        const dim3 blocks((unsigned)((h.N + b - 1) / b));
        if (h.N > kChainNodes) {
            k_two_lattice<S, L, true, false><<<blocks, b, 0, st>>>(a);
            return cudaGetLastError();
        }
        return launch_update(chain, k_two_lattice<S, L, true>, blocks, dim3(b), 0, st, a);
    }
    const bool chain_tiles = chain && spread_evenly(grid, tile, h.sms);
    if (h.algo == NPOL) {
        if constexpr (sizeof(S) == 4 && L != COLLISION) {
            const bool large = L == BUNDLE ? h.pf != 0 : h.beyond_l2;
            if (large) return launch_update(chain_tiles, k_npol<S, L, true>, grid, tile, 0, st, a);
        }
        return launch_update(chain_tiles, k_npol<S, L, false>, grid, tile, 0, st, a);
    }
    if (h.algo == NSOL) {
        const size_t sm = sizeof(C) * 9 * h.tile_x * h.tile_y;
        if constexpr (std::is_same<S, float>::value && L != COLLISION) {
            if (h.tma) return launch_update(chain_tiles, k_nsol_tma<S, L>, grid, tile, sm + 16, st, a, h.tmap);
        }
        return launch_update(chain_tiles, k_nsol<S, L>, grid, tile, sm, st, a);
    }
    if (h.algo == NPTL) {
        if (L == COLLISION && h.tile_x % 32 == 0 && !(h.flags & 4u)) {
            const size_t sm = (size_t)AosSpan<S>::WARP_BYTES * ((h.tile_x * h.tile_y + 31) / 32);
            if (h.N > kChainNodes) {
                k_two_lattice_aos<S, false><<<grid, tile, sm, st>>>(a);
                return cudaGetLastError();
            }
            return launch_update(chain_tiles, k_two_lattice_aos<S>, grid, tile, sm, st, a);
        }
        if constexpr (sizeof(S) == 2 && L == BUNDLE) {
            if (pairs_ok<S, L>(h) && !(h.tile_x & 1))
                return launch_update(chain && spread_evenly(grid, dim3(h.tile_x / 2, h.tile_y), h.sms),
                                     k_two_lattice_pair<S, false>, grid, dim3(h.tile_x / 2, h.tile_y), 0, st, a);
        }
        // Two nodes per thread on request (4- and 8-byte storage): one node
        // per thread at 32 registers keeps full occupancy and measured faster.
        if (sizeof(S) >= 4 && h.tile_y >= 2 && !(h.tile_y & 1) && (h.flags & 2u))
            return launch_update(chain_tiles, k_two_lattice2<S, L>, grid, dim3(h.tile_x, h.tile_y / 2), 0, st, a);
    }
    if (h.algo == NPTL && h.N > kChainNodes) {
        k_two_lattice<S, L, false, false><<<grid, tile, 0, st>>>(a);
        return cudaGetLastError();
    }
    a.ty = rows_per_block(h);
    const dim3 cut(h.tile_x, a.ty), cuts(h.ntx, (h.ny + a.ty - 1) / a.ty);
    if (h.algo == NPTL) return launch_update(chain, k_two_lattice<S, L, false>, cuts, cut, 0, st, a);
    if (h.algo != AA) return cudaErrorInvalidValue;
    // (bundle: 256 x 64 3.0 unchained / 2.8 chained, 500 x 333 3.9 / 4.1, 1501 x 777
    // 11.0 / 11.4 us an update; stream 3.2 / 2.9, 4.9 / 4.9, 18.1 / 17.4)
    if (h.N > (L == BUNDLE ? kChainNodes >> 5 : kChainNodes)) {
        if (phase) k_aa<S, L, 1, false><<<cuts, cut, 0, st>>>(a);
        else k_aa<S, L, 0, false><<<cuts, cut, 0, st>>>(a);
        return cudaGetLastError();
    }
    return phase ? launch_update(chain, k_aa<S, L, 1>, cuts, cut, 0, st, a)
                 : launch_update(chain, k_aa<S, L, 0>, cuts, cut, 0, st, a);
}

template <class S>
cudaError_t op_step(const HostArgs &h, const StepCall &c, cudaStream_t st) {
    const Step<S> a = make_step<S>(h, c);
    cudaError_t e = cudaErrorInvalidValue;
    switch (h.layout) {
        case STREAM: e = step_layout<S, STREAM>(h, a, c.rd_parity, st); break;
        case BUNDLE: e = step_layout<S, BUNDLE>(h, a, c.rd_parity, st); break;
        case COLLISION: e = step_layout<S, COLLISION>(h, a, c.rd_parity, st); break;
    }
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

#define LBM_LAYOUT_SWITCH(h, CALL)                          \
    switch ((h).layout) {                                   \
        case STREAM: { constexpr int L_ = STREAM; CALL; break; }       \
        case BUNDLE: { constexpr int L_ = BUNDLE; CALL; break; }       \
        case COLLISION: { constexpr int L_ = COLLISION; CALL; break; } \
        default: return cudaErrorInvalidValue;              \
    }

template <class S>
cudaError_t op_init(const HostArgs &h, const double *rho, const double *ux, const double *uy,
                    int64_t n0, int64_t count, cudaStream_t st) {
    const Step<S> a = make_step<S>(h, StepCall{1, 0, 0, 0});  // dst = pop[0]
    if (count <= 0) return cudaSuccess;
    const unsigned g = (unsigned)((count + 255) / 256);
    const int rev = h.algo == NSOL || h.algo == AA;
    LBM_LAYOUT_SWITCH(h, (k_init<S, L_><<<g, 256, 0, st>>>(a, rho, ux, uy, (uint32_t)n0,
                                                             (uint32_t)count, rev)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_publish(const HostArgs &h, int src, int parity, cudaStream_t st) {
    const Step<S> a = make_step<S>(h, StepCall{src, 0, 0, 0});
    S *hw = (S *)h.halo + (int64_t)parity * h.halo_parity_elems;
    const int rev = h.algo == NSOL || h.algo == AA;
    const dim3 tile(h.tile_x, h.tile_y), grid(h.ntx, h.nty);
    LBM_LAYOUT_SWITCH(h, (k_publish<S, L_><<<grid, tile, 0, st>>>(a, hw, rev)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_zero_solid(const HostArgs &h, int src, cudaStream_t st) {
    const Step<S> a = make_step<S>(h, StepCall{src, 0, 0, 0});
    const unsigned g = (unsigned)((h.N + 255) / 256);
    S *lat = (S *)h.pop[src];
    LBM_LAYOUT_SWITCH(h, (k_zero_solid<S, L_><<<g, 256, 0, st>>>(a, lat)));
    return cudaGetLastError();
}

// f64: the host values are doubles, else floats.
template <class S>
cudaError_t op_export(const HostArgs &h, int src, void *rows, bool f64, int64_t n0, int64_t count, int64_t stride,
                      cudaStream_t st) {
    const unsigned g = (unsigned)((count + 255) / 256);
    const uint32_t N = (uint32_t)h.N, b = (uint32_t)n0, c = (uint32_t)count;
    const int rev = h.algo == NSOL || h.algo == AA;
    const S *lat = (const S *)h.pop[src];
    LBM_LAYOUT_SWITCH(h, (f64 ? k_export<S, L_, double><<<g, 256, 0, st>>>(lat, N, rev, (double *)rows, b, c, stride)
                              : k_export<S, L_, float><<<g, 256, 0, st>>>(lat, N, rev, (float *)rows, b, c, stride)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_import(const HostArgs &h, int dst, const void *rows, bool f64, int64_t n0, int64_t count,
                      int64_t stride, cudaStream_t st) {
    const unsigned g = (unsigned)((count + 255) / 256);
    const uint32_t N = (uint32_t)h.N, b = (uint32_t)n0, c = (uint32_t)count;
    const int rev = h.algo == NSOL || h.algo == AA;
    S *lat = (S *)h.pop[dst];
    LBM_LAYOUT_SWITCH(
        h, (f64 ? k_import<S, L_, double><<<g, 256, 0, st>>>(lat, h.links, N, rev, (const double *)rows, b, c, stride)
                : k_import<S, L_, float><<<g, 256, 0, st>>>(lat, h.links, N, rev, (const float *)rows, b, c, stride)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_state_moments(const HostArgs &h, int src, int post, cudaStream_t st) {
    Step<S> a = make_step<S>(h, StepCall{src, 0, 0, 1});
    const unsigned g = (unsigned)((h.N + 255) / 256);
    const int rev = h.algo == NSOL || h.algo == AA;
    LBM_LAYOUT_SWITCH(h, (k_state_moments<S, L_><<<g, 256, 0, st>>>(a, rev, post)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_mass(const HostArgs &h, int src, double *partials, int nblocks, cudaStream_t st) {
    const Step<S> a = make_step<S>(h, StepCall{src, 0, 0, 0});
    const int rev = h.algo == NSOL || h.algo == AA;
    LBM_LAYOUT_SWITCH(h, (k_mass<S, L_><<<nblocks, kReduceThreads, 0, st>>>(a, rev, partials)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_force(const HostArgs &h, int src, const uint8_t *body, double *partials, int nblocks,
                     cudaStream_t st) {
    const Step<S> a = make_step<S>(h, StepCall{src, 0, 0, 0});
    const int rev = h.algo == NSOL || h.algo == AA;
    LBM_LAYOUT_SWITCH(h, (k_force<S, L_><<<nblocks, kReduceThreads, 0, st>>>(a, rev, body, partials)));
    return cudaGetLastError();
}

template <class S>
cudaError_t op_moments_f32(const HostArgs &h, float *r, float *u, float *v, cudaStream_t st) {
    using C = typename Codec<S>::C;
    const unsigned g = (unsigned)((h.N + 255) / 256);
    k_moments_f32<C><<<g, 256, 0, st>>>((const C *)h.mom, (uint32_t)h.N, r, u, v);
    return cudaGetLastError();
}

template <class S>
int op_lptl_block(int layout) {
    switch (layout) {
        case STREAM: return lptl_block<S, STREAM>();
        case BUNDLE: return lptl_block<S, BUNDLE>();
        default: return lptl_block<S, COLLISION>();
    }
}

// Allow the staged collision-layout kernel more than the default 48 KB of
// dynamic shared memory (FP64: 7.4 KB per warp). Called at lattice creation.
template <class S>
void op_prepare() {
    static const bool done = [] {
        cudaFuncSetAttribute(k_two_lattice_aos<S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             AosSpan<S>::WARP_BYTES * (kMaxTileThreads / 32));
        cudaFuncSetAttribute(k_two_lattice_aos<S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             AosSpan<S>::WARP_BYTES * (kMaxTileThreads / 32));
        cudaGetLastError();
        return true;
    }();
    (void)done;
}

template <class S>
Ops make_ops() {
    Ops o;
    o.step = op_step<S>;
    o.init = op_init<S>;
    o.publish = op_publish<S>;
    o.zero_solid = op_zero_solid<S>;
    o.state_moments = op_state_moments<S>;
    o.export_state = op_export<S>;
    o.import_state = op_import<S>;
    o.mass = op_mass<S>;
    o.force = op_force<S>;
    o.moments_f32 = op_moments_f32<S>;
    o.lptl_block = op_lptl_block<S>;
    o.prepare = op_prepare<S>;
    o.batch_step = op_batch_step<S>;
    o.batch_grid = op_batch_grid<S>;
    o.batch_case = op_batch_case<S>;
    o.batch_case_bytes = sizeof(BatchCase<S>);
    o.elem = sizeof(S);
    o.compute = sizeof(typename Codec<S>::C);
    return o;
}

}  // namespace lbm
