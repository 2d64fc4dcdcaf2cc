// lbm_aux.h -- host-side entry points of the kernel translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_common.cuh"

namespace lbm {

// Conservation reduction: instance i is split into P_i <= CONS_PARTIALS
// partial sums, partial b over the rows y = b mod P_i, each summed by
// cons_split(nodes) CTAs of CONS_THREADS threads (a cluster); the split is a
// function of the instance alone, so the FP64 summation order never depends
// on the device or on the other instances.
constexpr int CONS_PARTIALS = 64;
constexpr int CONS_THREADS = 256;
// one partial per 1024 nodes, at most one per row (with 64 for every
// lattice the smallest ones' CTAs are mostly tail: 121 us on 64 lattices of
// 64^2 to 1024^2, FP16, now 93 us); per 512 with FP64 storage, whose additions
// take an SM 5 ns a node
__host__ __device__ inline int cons_partials(int nx, int ny, int bytes) {
    const int nodes = bytes == 8 ? 512 : 1024;
    const int64_t want = ((int64_t)nx * ny + nodes - 1) / nodes;
    const int most = ny < CONS_PARTIALS ? ny : CONS_PARTIALS;
    return want < most ? (int)want : most;
}
// 1, 2, 4 or 8: some 2^14 nodes per CTA, which take it longer than its tail
// of FP64 additions (8 CTAs for 2^20 nodes: 787 us on 64 cavities of up to
// 1024^2, FP16, where one takes 351 us)
__host__ __device__ inline int cons_split(int64_t nodes) {
    return nodes <= (1 << 20) ? 1 : nodes <= (1 << 21) ? 2 : nodes <= (1 << 22) ? 4 : 8;
}

// Words of a context's error block: the error word, and from TILE_COUNTERS on
// the two counters of the TMA kernel's drawn tiles.
constexpr int TILE_COUNTERS = 8, ERROR_WORDS = 16;

enum class AuxOp { Init, SetF, CollideInPlace, Moments, GatherF, StreamFunction, Conservation, ClearPadding };

struct AuxArgs {
    int lattice;   // 1 = D1Q3, 2 = D2Q9
    int storage;   // DT_*
    int compute;   // DT_F64 or DT_F32
    int collision; // COLL_*
    int count;     // instances
    int64_t max_nodes, max_ny;  // of the largest / tallest instance
    int64_t total_nodes;
    const InstDesc* inst;  // device
    double rho0;
    bool pulled;           // stored field is post-collision (pull to read f(t_n))
    unsigned long long* status;
    unsigned int* error = nullptr;  // Init: ERROR_WORDS words cleared with the status counters unless null
    cudaStream_t stream;
    const int2* cons_items;  // device: (instance, partial) of each conservation block
    int32_t cons_nitems;
    int64_t node_base = 0;   // host-array index of the first node the call covers (Init,
                             // Moments, StreamFunction): arrays start at that node
};

// Init:           dst <- f^eq(rho=p0, ux=p1, uy=p2) deviations
// SetF:           dst <- p0 (FP64 populations, [inst][a][y][x])
// CollideInPlace: dst <- collide(src) without streaming
// Moments:        o0, o1, o2 <- rho, ux, uy of f(t_n) read from src
// GatherF:        o0 <- FP64 populations of f(t_n)
// ClearPadding:   columns of dst beyond each instance's own to deviation 0
// StreamFunction: o0 <- stream function of f(t_n) (D2Q9), [inst][y][x]
// Conservation:   o0 <- per-instance totals (3 doubles each), o1 = partials scratch
//                 (count * CONS_PARTIALS * 3 doubles; partial b of instance i at
//                 (i * CONS_PARTIALS + b) * 3)
cudaError_t run_aux(AuxOp op, const AuxArgs& a, const void* src, void* dst, const double* p0,
                    const double* p1, const double* p2, double* o0, double* o1, double* o2);

// Fused step kernels, one translation unit per storage type.  Each returns
// the __global__ function for (lattice, collision, V), or nullptr.
const void* step_kernel_f64(int lattice, int collision, int V);
const void* step_kernel_f32(int lattice, int collision, int V);
const void* step_kernel_f16(int lattice, int collision, int V);
const void* step_kernel_bf16(int lattice, int collision, int V);

// D1Q3 kernels of one step per launch (4 nodes a thread for FP32 storage, 8 for
// 2-byte storage).
const void* step_kernel_single_tube_f32();
const void* step_kernel_single_tube_f16();
const void* step_kernel_single_tube_bf16();

// D2Q9 step kernels that take several steps per launch on overlapping regions
// (lbm_step_block.cuh; FP32 arithmetic): regions of 64 columns and at most
// block_max_rows rows, CTAs of at most BLOCK_WARPS warps.
const void* step_kernel_block_f32(int collision, int rows);
const void* step_kernel_block_f16(int collision, int rows);
const void* step_kernel_block_bf16(int collision, int rows);
constexpr int BLOCK_WARPS = 16;
constexpr int BLOCK_COLS = 64;
// two buffers of nine planes of 64-node rows within 221 KB (storage 1: FP32)
constexpr int block_max_rows(int storage) { return storage == 1 ? 48 : 96; }
constexpr int BLOCK_SMALL_ROWS = 24;  // regions up to this height take buffers of it (two CTAs per SM)
constexpr size_t block_smem_bytes(int storage, int rows) {
    return (size_t)2 * 9 * BLOCK_COLS * (storage == 1 ? 4 : 2) *
           (rows <= BLOCK_SMALL_ROWS ? BLOCK_SMALL_ROWS : block_max_rows(storage));
}

// D2Q9 step kernels with shared-memory tile staging (FP32 arithmetic), tiles
// dealt out or (two-stage rings) drawn; also return the dynamic shared memory
// they need.
const void* step_kernel_smem_f32(int collision, int variant, bool draws, size_t* smem_bytes);
const void* step_kernel_smem_f16(int collision, int variant, bool draws, size_t* smem_bytes);
const void* step_kernel_smem_bf16(int collision, int variant, bool draws, size_t* smem_bytes);
// Geometries of the TMA-staged kernel (variant = launch-shape kind - 1).
// Every CTA has one copy warp, which writes finished tiles out and issues
// the copies of the next ones, besides its colliding warps; a tile holds
// 64 nodes per unit x the units of each colliding warp:
//   0  large tiles: 8 warps, 7 colliding with 4 units each (2-byte storage;
//      2 for FP32): 1792 / 896 nodes, two-stage ring;
//   1  small tiles: 8 warps, 2 / 1 units each: 896 / 448 nodes, three-stage
//      ring (more copies in flight per node);
//   2  wide CTAs: 10 warps, 4 / 2 units each: 2304 / 1152 nodes, two stages;
//   3  deep ring: one CTA of 16 warps per SM, 2 / 1 units each: 1920 / 960
//      nodes on a five- / four-stage ring, so a stage is refilled four /
//      three tiles before it is needed.
// Two CTAs of the 8- and 10-warp geometries fit an SM (registers and
// shared memory); the 16-warp one keeps all 128 registers per thread.
#ifndef LBM_SMEM_STAGES_DEEP
#define LBM_SMEM_STAGES_DEEP 4   // FP32 storage
#endif
#ifndef LBM_SMEM_STAGES_DEEP2
#define LBM_SMEM_STAGES_DEEP2 5  // 2-byte storage
#endif
#ifndef LBM_DEEP_WARPS
#define LBM_DEEP_WARPS 15  // colliding warps of the deep-ring CTA
#endif
#ifndef LBM_SMEM_STAGES
#define LBM_SMEM_STAGES 2        // ring depth, large tiles
#endif
#ifndef LBM_SMEM_STAGES_SMALL
#define LBM_SMEM_STAGES_SMALL 3  // ring depth, small tiles
#endif
// ring depth (storage 1: FP32)
constexpr int smem_stages(int storage, int variant) {
    return variant == 1   ? LBM_SMEM_STAGES_SMALL
           : variant == 3 ? (storage == 1 ? LBM_SMEM_STAGES_DEEP : LBM_SMEM_STAGES_DEEP2)
                          : LBM_SMEM_STAGES;
}
// colliding threads of a CTA (the copy warp comes on top)
constexpr int smem_threads(int variant) {
    return variant == 2 ? 288 : (variant == 3 ? 32 * LBM_DEEP_WARPS : 224);
}
constexpr int smem_block_threads(int variant) { return smem_threads(variant) + 32; }
// units of 32 node pairs per colliding warp and tile (storage 1: FP32)
#ifndef LBM_DEEP_UNITS
#define LBM_DEEP_UNITS 2  // units per colliding warp and tile of the deep ring (2-byte storage)
#endif
constexpr int smem_units(int storage, int variant) {
    return (variant == 0 || variant == 2 ? 4 : (variant == 3 ? LBM_DEEP_UNITS : 2)) /
           (storage == 1 ? 2 : 1);
}
constexpr int smem_tile_nodes(int storage, int variant) {
    return 64 * smem_units(storage, variant) * (smem_threads(variant) / 32);
}
// Tile width X of an nx x ny instance: 64, 128 or 256 nodes (at most nx
// unless 64), at most 32 tile_nodes / threads so that each warp's units
// (tile_nodes / (2 threads) units of 64 nodes) cover whole tile rows.  Of
// those, the widest (fewest halo columns and tile copies per node: what
// the bandwidth-bound rules want), or with least_padding the one whose
// tiles (X by tile_nodes / X rows) cover the instance with the fewest
// padding nodes (what arithmetic-bound rules want: a padding lane collides
// for nothing); ties go to the wider tile.
inline int smem_tile_width(int64_t nx, int64_t ny, int tile_nodes, int threads,
                           bool least_padding) {
    int best = 64;
    int64_t best_cells = -1;
    for (int w = 256; w >= 64; w /= 2) {
        if ((int64_t)w * threads > 32LL * tile_nodes) continue;
        if (w > 64 && nx < w) continue;
        if (!least_padding) return w;
        const int64_t R = tile_nodes / w;
        const int64_t cells = ((nx + w - 1) / w) * w * (((ny + R - 1) / R) * R);
        if (best_cells < 0 || cells < best_cells) {
            best_cells = cells;
            best = w;
        }
    }
    return best;
}
// The MinxEnt rules are arithmetic-bound on the TMA kernel, the others
// bandwidth-bound.
constexpr bool smem_least_padding(int collision) {
    return collision == COLL_MINXENT4 || collision == COLL_MINXENT2;
}

}  // namespace lbm
