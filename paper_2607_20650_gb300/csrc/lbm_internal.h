// Host-side interface between the C ABI (lbm_capi.cu) and the kernel
// translation units (one per storage type). No device types appear here.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace lbm {

// An opaque tensor-map descriptor for the tensor copies (the 128-byte,
// 64-byte aligned object the CUDA driver encodes), passed to kernels by value.
struct alignas(64) TmaDesc {
    unsigned char bytes[128];
};

// Launch of an update kernel (one that calls chain_wait before it touches what
// updates write). chained: its blocks may start before the previous kernel on
// the stream has ended.
// Small FP64 lattices are not chained: blocks placed beside the previous grid's
// end up unevenly over the SMs, and where FP64 arithmetic is the bound the
// fullest SM sets the time. Porous nodes, us an update, unchained / chained:
// FP64 431 x 77 5.7 / 12.1, 512 x 300 17.7 / 21.1, 1024 x 512 48.6 / 48.3; FP32
// 3.1 / 1.9, 3.8 / 2.6, 6.5 / 5.2.
inline bool chained_updates(size_t elem, int64_t nodes) { return elem < 8 || nodes >= (int64_t)1 << 19; }
// Nor are kernels with blocks of a tile's size, or of one node a thread in three
// dimensions, while their blocks neither fill the device's SMs (1,536 threads each,
// what these kernels keep resident at 40 registers) nor leave three quarters of
// them empty, for the same reason. D3Q19 FP32 on 152 SMs, us an update, unchained /
// chained: NPOL 8 x 8 x 8, 30 x 28 x 33 nodes (80 blocks) 4.7 / 8.1, 48 x 40 x 44 (180)
// 5.4 / 8.4, 64 x 64 x 64 (512) 11.1 / 10.7; LPTL (256 nodes a block) 4.0 / 4.9,
// 5.9 / 6.5 and 8.9 / 8.4; 12 x 12 x 12 (7 blocks) 3.7 / 3.2.
inline bool spread_evenly(dim3 grid, dim3 block, int sms) {
    const int64_t blocks = (int64_t)grid.x * grid.y * grid.z;
    return blocks * block.x * block.y * block.z >= (int64_t)sms * 1536 || blocks <= sms / 4;
}

// (A failure also stands as the runtime's last error, as after <<< >>>; the entry
// points of Ops and Ops3 take it from there, so that no later call reports it.)
template <class... P, class... A>
inline cudaError_t launch_update(bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t st, A &&...a) {
    cudaLaunchConfig_t c = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = at;
    c.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(a)...);
}

// What the launch rules ask of the current device (lbm_common.cu).
struct DeviceSize {
    int sms;          // 152 where there is no device to ask
    int sm_threads;   // the same: 0
    int64_t l2;       // bytes; the same: 0
};
DeviceSize device_size();

// Everything a kernel launch needs, in host types.
struct HostArgs {
    int nx, ny;
    int64_t N;
    int bw, be, bs, bn;
    int layout, algo, storage, rounding;
    double omega, fx, fy, ux_in, uy_in, rho_out;
    uint64_t seed;
    int tile_x, tile_y, ntx, nty;
    int block_1d;              // LPTL block size
    int sms;                   // SMs of the device
    bool beyond_l2;            // a lattice's populations exceed the L2 cache
    uint32_t flags;            // lbm_params.flags
    uint64_t nx_magic;         // ceil(2^64 / nx) for n -> (x, y); 0 when nx == 1
    uint32_t pf;               // L2 prefetch distance: nodes (LPTL) or rows (NPTL); 0 = off
    const uint8_t *links;
    void *pop[2];              // pop[1] == nullptr for one-lattice algorithms
    void *halo;                // one-lattice buffer grid (2 parities)
    int64_t halo_parity_elems; // elements per parity
    void *mom;                 // 3N compute-type values
    unsigned int *err;
    long long *tctr;           // device update counter (stochastic rounding keys)
    int tma;                   // NSOL, FP32: the tile is staged by one tensor copy (tmap)
    TmaDesc tmap;
};

// One update: which lattice is the source, the halo parity that is read,
// offset added to the device update counter, and whether moments are stored.
struct StepCall {
    int src;
    int rd_parity;
    int toff;
    int want_moments;
};

struct Ops {
    cudaError_t (*step)(const HostArgs &, const StepCall &, cudaStream_t);
    // Equilibrium from FP64 rho/ux/uy (device, count nodes from n0; NULL -> 1/0).
    cudaError_t (*init)(const HostArgs &, const double *rho, const double *ux, const double *uy,
                        int64_t n0, int64_t count, cudaStream_t);
    // Copy tile-edge populations of lattice `src` into halo parity `parity`.
    cudaError_t (*publish)(const HostArgs &, int src, int parity, cudaStream_t);
    // Store h = 0 at every solid node of lattice `src`.
    cudaError_t (*zero_solid)(const HostArgs &, int src, cudaStream_t);
    // Nodes n0 .. n0 + count - 1 of lattice src / dst to / from rows[i stride + n - n0] in mapped
    // host memory (doubles or floats).
    cudaError_t (*export_state)(const HostArgs &, int src, void *rows, bool f64, int64_t n0, int64_t count,
                                int64_t stride, cudaStream_t);
    cudaError_t (*import_state)(const HostArgs &, int dst, const void *rows, bool f64, int64_t n0, int64_t count,
                                int64_t stride, cudaStream_t);
    // rho = 1 + sum h, v = sum h c (- F/2 if post_collision) into mom.
    cudaError_t (*state_moments)(const HostArgs &, int src, int post_collision, cudaStream_t);
    // FP64 block partial sums: mass (1 value) or force (2 values) per block.
    cudaError_t (*mass)(const HostArgs &, int src, double *partials, int nblocks, cudaStream_t);
    cudaError_t (*force)(const HostArgs &, int src, const uint8_t *body, double *partials,
                         int nblocks, cudaStream_t);
    // Moments buffer (compute type) -> FP32 device arrays.
    cudaError_t (*moments_f32)(const HostArgs &, float *r, float *u, float *v, cudaStream_t);
    int (*lptl_block)(int layout);  // occupancy-chosen LPTL block size
    void (*prepare)();              // one-time kernel attributes (called at create)
    // Batches: one persistent launch over the packed tile list.
    // kind = layout * 4 + algo shared by every case, or -1 for a mixed batch.
    // recs: 4 ncases records (two lattice parities without, then with moments);
    // cur: the parity.
    cudaError_t (*batch_step)(int kind, const void *recs, int ncases, const void *tiles, uint32_t ntiles, int grid,
                              int cur, int toff, int want_moments, cudaStream_t);
    int (*batch_grid)(int kind);                           // resident blocks on the device
    // One device record; pf: L2 prefetch of the next tile's records.
    void (*batch_case)(const HostArgs &, int parity, int moments, int pf, void *out);
    size_t batch_case_bytes;
    size_t elem;               // bytes per stored population
    size_t compute;            // bytes per compute value
};

const Ops &ops_f64();
const Ops &ops_f32();
const Ops &ops_f16();
const Ops &ops_bf16();

// Shared kernels (lbm_common.cu).
cudaError_t launch_links(int nx, int ny, int bw, int be, int bs, int bn, const uint8_t *mask,
                         uint8_t *links, cudaStream_t);
cudaError_t launch_count_fluid(const uint8_t *links, int64_t N, unsigned long long *out,
                               cudaStream_t);
// out: width sums, then the bits of the error word.
cudaError_t launch_sum_partials(const double *partials, int nblocks, int width, double *out,
                                const unsigned int *err, cudaStream_t);
cudaError_t launch_bump_counter(long long *ctr, long long by, cudaStream_t);
cudaError_t launch_quantize(int storage, int rounding, uint64_t seed, int64_t t, const float *in,
                            void *out, float *back, int64_t count, cudaStream_t);

constexpr int kReduceBlocks = 1024;
constexpr int kReduceThreads = 256;
constexpr int kBatchTileNodes = 256;  // threads per batch block = nodes per LPTL tile
constexpr int kBatchSuperHost = 4;    // tiles per work item of a two-lattice case

}  // namespace lbm
