// lbm_api.cu -- the C ABI of liblbm (declared in include/lbm.h): context
// lifetime, device memory layout, tile tables, the launch-shape autotuner,
// CUDA-graph replay of the step loop, and host I/O.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_aux.h"
#include "lbm_step_block.cuh"

using namespace lbm;

namespace {

constexpr int64_t ROW_ALIGN = 8;       // row pitch multiple (nodes)
constexpr int64_t PLANE_ALIGN = 128;   // plane / instance alignment (elements)
constexpr int GRAPH_STEPS = 16;        // steps per captured graph (even)
constexpr int BLOCK_WHOLE_STEPS = 32;  // steps per launch on uncut regions

size_t dtype_bytes(int dt) { return dt == DT_F64 ? 8 : (dt == DT_F32 ? 4 : 2); }

// Launch shape.  kind 0: register-chunk kernel (V nodes per thread, tiles of
// tw x th chunks); kind 1 / 2 / 3 / 4: TMA-staged D2Q9 kernel with node
// pairs (V = 2) in the large-tile / small-tile / wide-CTA / deep-ring
// geometry (smem_tile_nodes variant kind - 1), tile width per instance.
// Kind 5: overlapping regions (lbm_step_block.cuh), tw steps per launch on
// regions of th rows.
// Kind 0 with V = 1 on D2Q9 is the FP64 kernel with one node per thread
// (warps of 32 consecutive nodes: tw = 32, th = 1).  On D1Q3 kind 0 is the
// tube kernel: V nodes per lane, tw x th threads per CTA.  Kind 6: the
// register-chunk kernel on D1Q3, for single steps beside the tube kernel.
struct Shape {
    int V, tw, th;
    int kind = 0;
    bool tma() const { return kind >= 1 && kind <= 4; }
    bool block() const { return kind == 5; }
    bool single_tube() const { return kind == 6; }
};

// A step kernel ready to launch: its shape, and its tiles' place in the
// context's tile table.
struct StepPlan {
    Shape shape{};
    const void* kern = nullptr;
    int grid = 0;
    size_t smem = 0;  // dynamic shared memory
    int32_t tile0 = 0, ntiles = 0;
    bool draws = false;   // TMA kernel: tiles beyond the CTAs' first two are drawn
    int flat_nodes = 0;   // one-node-per-thread kernel: nodes per tile-table entry
    int halo = 0;         // tube and region kernels: halo nodes, steps per launch
    int block_warps = 0;  // region kernel: warps of a CTA
};

Shape default_shape_d2q9(int storage) {
    if (storage == DT_F64) return {1, 32, 1};
    if (storage == DT_F32) return {4, 16, 8};
    return {8, 8, 16};
}

// Launch-shape candidates of the autotuner on D2Q9.  FP32 arithmetic: the
// TMA-staged kernel in its four geometries and the default register-chunk
// shape (which wins only on small, cache-resident lattices).  FP64: one node
// per thread (measured ahead of every register-chunk shape from 800 x 4 to
// 2048^2 nodes, so nothing is timed).
std::vector<Shape> candidate_shapes(int storage) {
    std::vector<Shape> out;
    if (storage != DT_F64)
        for (int kind = 1; kind <= 4; ++kind) out.push_back({2, 0, 0, kind});
    out.push_back(default_shape_d2q9(storage));
    return out;
}

// Tiles of the TMA kernel's geometry `variant` (kind - 1).
int64_t count_smem_tiles(const std::vector<std::pair<int64_t, int64_t>>& dims, int variant, int storage,
                         bool least_padding) {
    int64_t n = 0;
    for (auto& d : dims) {
        const int tn = smem_tile_nodes(storage, variant);
        const int64_t X = smem_tile_width(d.first, d.second, tn, smem_threads(variant), least_padding);
        const int64_t R = tn / X;
        n += ((d.first + X - 1) / X) * ((d.second + R - 1) / R);
    }
    return n;
}

struct Layout {
    std::vector<InstDesc> inst;
    int64_t elems = 0;       // elements per population buffer
    int64_t total_nodes = 0;
    int64_t max_nodes = 0, max_nx = 0, max_ny = 0;
    int64_t max_tiles = 0;
};

Layout make_layout(int lattice, int storage, const std::vector<std::pair<int64_t, int64_t>>& dims) {
    Layout L;
    const int Q = lattice == 2 ? 9 : 3;
    int64_t off = 0, node0 = 0;
    for (auto& d : dims) {
        InstDesc in;
        std::memset(&in, 0, sizeof in);
        in.nx = (int32_t)d.first;
        in.ny = (int32_t)d.second;
        in.pitch = (int32_t)round_up(d.first, ROW_ALIGN);
        in.plane = round_up((int64_t)in.pitch * in.ny, PLANE_ALIGN);
        in.off = off;
        in.node0 = node0;
        off += Q * in.plane;
        node0 += d.first * d.second;
        L.max_nodes = std::max(L.max_nodes, d.first * d.second);
        L.max_nx = std::max(L.max_nx, d.first);
        L.max_ny = std::max(L.max_ny, d.second);
        L.inst.push_back(in);
    }
    L.elems = off;
    L.total_nodes = node0;
    // Tile-table capacity: a bound that holds for every register-chunk shape
    // (V >= 2, tw >= 4, tw * th >= 128 threads) and the shared-memory kernel's
    // tiling, so any shape the autotuner or LBM_SHAPE selects fits.
    int64_t bound = 0;
    for (auto& d : dims) {
        const int64_t chunks = (d.first + 1) / 2;
        bound += chunks * d.second / 128 + chunks / 4 + d.second + 1;
    }
    L.max_tiles = bound;
    for (int variant = 0; variant < 4; ++variant)
        for (bool lp : {false, true})
            L.max_tiles = std::max(L.max_tiles, count_smem_tiles(dims, variant, storage, lp));
    return L;
}

struct Carve {
    size_t buf_bytes, inst_off, tiles_off, status_off, partials_off, cons_off, stage_off, tmap_off,
        err_off, total;
};

Carve carve(const Layout& L, int lattice, int storage, int count) {
    const int Q = lattice == 2 ? 9 : 3;
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    Carve c;
    c.buf_bytes = al((size_t)L.elems * dtype_bytes(storage));
    size_t p = 2 * c.buf_bytes;
    c.inst_off = p;
    p += al(sizeof(InstDesc) * count);
    c.tiles_off = p;
    p += al(sizeof(TileDesc) * (size_t)std::max<int64_t>(L.max_tiles, 1));
    c.status_off = p;
    p += al(sizeof(unsigned long long) * 2 * count);
    c.partials_off = p;
    p += al(sizeof(double) * 3 * (size_t)CONS_PARTIALS * count);
    c.cons_off = p;  // (instance, partial) work list of the conservation reduction
    p += al(sizeof(int2) * (size_t)CONS_PARTIALS * count);
    c.stage_off = p;
    p += al(sizeof(double) * std::max<int64_t>(3 * L.total_nodes, Q * L.total_nodes));
    c.tmap_off = p;  // four TMA tensor maps per instance: [buffer][tile | halo]
    p += al(4 * sizeof(CUtensorMapOpaque) * count);
    c.err_off = p;  // ERROR_WORDS words (256 bytes are kept for them)
    p += 256;
    c.total = p;
    return c;
}

}  // namespace

struct lbm_ctx {
    int lattice = 2, Q = 9, count = 0, bc = 0, compute = DT_F64, storage = DT_F64;
    int collision = COLL_MINXENT4;
    double rho0 = 1.0;
    cudaStream_t stream = nullptr;
    cudaStream_t capture_stream = nullptr;
    int num_sms = 0;
    bool own_mem = false;
    char* mem = nullptr;
    Layout layout;
    Carve cv{};
    char* buf[2] = {nullptr, nullptr};
    int cur = 0;  // buffer holding the current state
    InstDesc* d_inst = nullptr;
    TileDesc* d_tiles = nullptr;
    unsigned long long* d_status = nullptr;
    double* d_partials = nullptr;
    int2* d_cons = nullptr;  // conservation work list
    int n_cons = 0;
    double* d_stage = nullptr;
    CUtensorMapOpaque* d_tmaps = nullptr;  // [buffer][tile | halo][instance]
    unsigned int* d_error = nullptr;
    int tmaps_variant = -1;  // tile variant the TMA tensor maps were built for
    bool initialized = false;
    std::vector<uint8_t> inst_init;  // per-instance initial fields set (lbm_init_batch)
    bool post = false;  // stored field is post-collision
    int64_t steps = 0;
    StepPlan plan;
    // One step per launch, beside a plan that takes several (kern = null where
    // there is none): launches of less than `plan_from` steps go to it.
    StepPlan single;
    int plan_from = 1;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    bool failed = false;
    int spin_limit = 1 << 20;  // polls of one bounded mbarrier wait in the TMA kernel
    int lost_tile = -1;        // timeout-path test hook (LBM_TEST_LOST_TILE)
};

namespace {

#define LBM_CK(call)                                                                   \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) {                                                       \
            if (getenv("LBM_DEBUG"))                                                   \
                fprintf(stderr, "liblbm: %s failed: %s (%s:%d)\n", #call,              \
                        cudaGetErrorString(e_), __FILE__, __LINE__);                   \
            if (ctx) ctx->failed = true;                                               \
            return LBM_ERR_CUDA;                                                       \
        }                                                                              \
    } while (0)

const void* find_step_kernel(int lattice, int storage, int collision, int V) {
    switch (storage) {
        case DT_F64: return step_kernel_f64(lattice, collision, V);
        case DT_F32: return step_kernel_f32(lattice, collision, V);
        case DT_F16: return step_kernel_f16(lattice, collision, V);
        case DT_BF16: return step_kernel_bf16(lattice, collision, V);
    }
    return nullptr;
}

const void* find_smem_kernel(const lbm_ctx* ctx, int variant, bool draws, size_t* smem) {
    switch (ctx->storage) {
        case DT_F32: return step_kernel_smem_f32(ctx->collision, variant, draws, smem);
        case DT_F16: return step_kernel_smem_f16(ctx->collision, variant, draws, smem);
        case DT_BF16: return step_kernel_smem_bf16(ctx->collision, variant, draws, smem);
    }
    return nullptr;
}

AuxArgs aux_args(const lbm_ctx* ctx) {
    AuxArgs a;
    a.lattice = ctx->lattice;
    a.storage = ctx->storage;
    a.compute = ctx->compute;
    a.collision = ctx->collision;
    a.count = ctx->count;
    a.max_nodes = ctx->layout.max_nodes;
    a.max_ny = ctx->layout.max_ny;
    a.total_nodes = ctx->layout.total_nodes;
    a.inst = ctx->d_inst;
    a.rho0 = ctx->rho0;
    a.pulled = ctx->post;
    a.status = ctx->d_status;
    a.stream = ctx->stream;
    a.cons_items = ctx->d_cons;
    a.cons_nitems = ctx->n_cons;
    return a;
}

// One-node-per-thread kernel: colliding nodes of an instance, and nodes per
// tile-table entry (the fewest, from one warp up, whose entries fit the
// table).
int64_t flat_fluid(int64_t nx, int64_t ny, int bc) {
    return bc == LBM_BC_CAVITY ? (nx - 2) * (ny - 2) : nx * ny;
}
int flat_nodes(const lbm_ctx* ctx) {
    for (int e = 32;; e *= 2) {
        int64_t n = 0;
        for (const InstDesc& in : ctx->layout.inst) {
            n += (flat_fluid(in.nx, in.ny, ctx->bc) + e - 1) / e;
        }
        if (n <= ctx->layout.max_tiles) return e;
    }
}
bool is_flat(const lbm_ctx* ctx, const Shape& s) {
    return ctx->lattice == 2 && s.kind == 0 && s.V == 1;
}
int block_threads(const lbm_ctx* ctx, const StepPlan& p) {
    const Shape& s = p.shape;
    if (s.tma()) return smem_block_threads(s.kind - 1);
    if (s.block()) return 32 * p.block_warps;
    if (s.single_tube()) return s.tw;
    if (ctx->lattice == 1) return std::max(32, std::min(s.tw * s.th, 256) / 32 * 32);
    return is_flat(ctx, s) ? 32 : s.tw * s.th;
}

// Tube kernel: nodes per lane V and halo (= steps per launch) of a context,
// the pair with the least modelled time per step
//     latency + (ceil(segments / schedulers) - 1) x throughput + launch / halo.
// A long halo spares launches and memory traffic, which is what single tubes
// are bound by, and costs redundant nodes, which ensembles are bound by; a
// small V spreads a short tube over more schedulers.  The constants (us per
// step of one segment alone on its scheduler / of one segment among many,
// and per launch) are fits of measurements, V and halo swept over single
// tubes of 800 to 20000 nodes and ensembles of 200 to 4096 tubes:
//   800 nodes FP64: V 1, halo 12: 0.78 us a step (V 2, halo 8: 1.45);
//   800 nodes FP32: V 2, halo 24: 0.19 us (V 4, halo 8: 0.43);
//   4096 tubes (18.0 M nodes) FP32: V 8, halo 8..16: 21.0 us (V 2: 32.2).
// V_pinned != 0 (LBM_SHAPE) fixes V.
void tube_plan(const lbm_ctx* ctx, int V_pinned, int* V, int* halo) {
    struct Cost {
        int V;
        double latency, throughput;
    };
    static const Cost f64[] = {{1, 0.62, 0.50}, {2, 1.22, 1.0}, {4, 2.4, 2.0}};
    static const Cost f32[] = {{2, 0.12, 0.045}, {4, 0.17, 0.079}, {8, 0.31, 0.151}};
    static const Cost b16[] = {{4, 0.20, 0.090}, {8, 0.36, 0.175}};
    const Cost* costs = ctx->storage == DT_F64 ? f64 : ctx->storage == DT_F32 ? f32 : b16;
    const int n = ctx->storage == DT_F64 || ctx->storage == DT_F32 ? 3 : 2;
    const double copy_us = 6.0 * dtype_bytes(ctx->storage) * ctx->layout.total_nodes / 6.8e6;
    double best = 1e30;
    *V = V_pinned;
    *halo = std::max(V_pinned, 8);
    for (int c = 0; c < n; ++c) {
        if (V_pinned && costs[c].V != V_pinned) continue;
        const int v = costs[c].V;
        for (int h = std::max(v, 4); h <= 48 && 32 * v - 2 * h >= 8; h += v) {
            const int64_t u = 32 * v - 2 * h;
            int64_t segs = 0;
            for (const InstDesc& in : ctx->layout.inst) segs += (in.nx + u - 1) / u;
            const double rounds = std::ceil((double)segs / (4.0 * ctx->num_sms));
            const double t = costs[c].latency + (rounds - 1.0) * costs[c].throughput +
                             (1.7 + 0.27 * copy_us) / h;
            if (t < best) {
                best = t;
                *V = v;
                *halo = h;
            }
        }
    }
}

// Regions of the kernel of lbm_step_block.cuh with K steps per launch and
// regions of `rows` rows: their number, and the table (t may be null).  An
// instance that fits a region along an axis with boundary rules of its own at
// both ends is not cut there; *whole = no instance is cut at all, so that the
// steps of a launch are not limited by the overlap.
int64_t block_tiles(const lbm_ctx* ctx, int K, int rows, bool* whole, std::vector<TileDesc>* t) {
    int64_t n = 0;
    *whole = true;
    for (int i = 0; i < ctx->count; ++i) {
        const InstDesc& in = ctx->layout.inst[i];
        const bool wide = ctx->bc == LBM_BC_PERIODIC || in.nx > BLOCK_COLS;
        const bool high = ctx->bc != LBM_BC_CAVITY || in.ny > rows;
        *whole = *whole && !wide && !high;
        const int U = wide ? BLOCK_COLS - 2 * K : BLOCK_COLS, V = high ? rows - 2 * K : rows;
        n += (int64_t)((in.nx + U - 1) / U) * ((in.ny + V - 1) / V);
        if (!t) continue;
        const int hx = wide ? K : 0, hy = high ? K : 0;
        for (int y = 0; y < in.ny; y += V)
            for (int x = 0; x < in.nx; x += U)
                t->push_back({(int32_t)i, x - hx, y - hy,
                              pack_part(hx, hx + std::min(U, in.nx - x), hy, hy + std::min(V, in.ny - y), !high)});
    }
    return n;
}

// Steps per launch and region height of a context with their modelled time per
// step, or false where the regions are too many for this kernel to be ahead of the TMA kernel (more
// than four per SM).  The modelled time per step, in us: a row of a region
// holds its scheduler for `unit` (16 warps take 16 rows at a time), a launch
// adds a region's loads and stores and the launch itself.  The constants fit
// 512 x 512, 64 x 64, 200 x 200 and 17 x 17 lattices with K = 2 .. 8 and 12 ..
// 64 rows within 15 %; over 60 lattices of all rules and types the measured
// time was 0.95 to 1.9 of the modelled one.  Whether the TMA kernel is ahead
// is timed, unless the model is already behind it.
bool block_plan(const lbm_ctx* ctx, int* K, int* rows, double* us) {
    const int64_t most = std::min<int64_t>(4 * ctx->num_sms, ctx->layout.max_tiles);
    if (ctx->count > most) return false;
    const int cap = block_max_rows(ctx->storage);
    const double unit = ctx->collision == LBM_MINXENT4 ? 0.41 : 0.28;
    *us = 1e30;
    auto consider = [&](int r, int steps, double live, int64_t n) {
        const double turns = std::ceil(live / BLOCK_WARPS);
        const double units = std::max(std::ceil(live / 4), turns > 1 ? 4 * (turns - 1) + 2.4 : 0.0);
        const double rounds = std::ceil((double)n / ctx->num_sms);
        const double t = rounds * (units * unit + 0.15 + 2.5 / steps) + 2.0 / steps;
        if (n <= most && t < *us) {
            *us = t;
            *K = steps;
            *rows = r;
        }
    };
    bool whole;
    const int tall = (int)std::min<int64_t>(ctx->layout.max_ny, cap);
    const int64_t n = block_tiles(ctx, 0, tall, &whole, nullptr);
    if (whole) consider(tall, BLOCK_WHOLE_STEPS, tall, n);
    for (int k = 2; k <= 8; k += 2) {
        // from the highest regions down, until there are too many
        std::vector<int64_t> cut(cap + 1, -1);  // by rows; -1: uncut or too many
        int r = cap;
        for (; r > 2 * k; --r) {
            const int64_t m = block_tiles(ctx, k, r, &whole, nullptr);
            if (m > most) break;
            if (!whole) cut[r] = m;
        }
        for (++r; r <= cap; ++r)
            if (cut[r] >= 0) consider(r, k, r - k - 1, cut[r]);  // (rows computed, on average)
    }
    return *us < 1e30;
}

std::vector<TileDesc> build_tiles(const lbm_ctx* ctx, const StepPlan& p) {
    const Shape& s = p.shape;
    std::vector<TileDesc> t;
    if (s.block()) {
        bool whole;
        block_tiles(ctx, s.tw, s.th, &whole, &t);
        return t;
    }
    if (s.tma()) {
        for (int i = 0; i < ctx->count; ++i) {
            const InstDesc& in = ctx->layout.inst[i];
            const int tn = smem_tile_nodes(ctx->storage, s.kind - 1);
            const int X = smem_tile_width(in.nx, in.ny, tn, smem_threads(s.kind - 1),
                                          smem_least_padding(ctx->collision));
            const int R = tn / X;
            for (int64_t y0 = 0; y0 < in.ny; y0 += R)
                for (int64_t x0 = 0; x0 < in.nx; x0 += X)
                    t.push_back({(int32_t)i, (int32_t)x0, (int32_t)y0, (int32_t)X});
        }
        return t;
    }
    if (ctx->lattice == 1 && !s.single_tube()) {
        const int u = 32 * s.V - 2 * p.halo;
        for (int i = 0; i < ctx->count; ++i)
            for (int32_t x = 0; x < ctx->layout.inst[i].nx; x += u) t.push_back({(int32_t)i, x, 0, 0});
        return t;
    }
    if (is_flat(ctx, s)) {
        // flat_nodes consecutive (fluid) nodes per entry
        for (int i = 0; i < ctx->count; ++i) {
            const InstDesc& in = ctx->layout.inst[i];
            const int64_t n = flat_fluid(in.nx, in.ny, ctx->bc);
            for (int64_t k = 0; k < n; k += p.flat_nodes)
                t.push_back({(int32_t)i, (int32_t)k, (int32_t)std::min<int64_t>(k + p.flat_nodes, n), 0});
        }
        return t;
    }
    for (int i = 0; i < ctx->count; ++i) {
        const InstDesc& in = ctx->layout.inst[i];
        const int64_t chunks = (in.nx + s.V - 1) / s.V;
        for (int64_t y0 = 0; y0 < in.ny; y0 += s.th)
            for (int64_t c0 = 0; c0 < chunks; c0 += s.tw)
                t.push_back({(int32_t)i, (int32_t)c0, (int32_t)y0, 0});
    }
    return t;
}

int ilog2(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}

int build_tensor_maps(lbm_ctx* ctx, int variant);

// The plan of shape s: kernel, grid size, and its tiles to the device's table
// from entry tile0 on.  halo: tube kernel's.
int make_plan(lbm_ctx* ctx, const Shape& s, int halo, int32_t tile0, StepPlan* out) {
    StepPlan p;
    p.shape = s;
    p.halo = halo;
    p.tile0 = tile0;
    const void* k = nullptr;
    size_t smem = 0;
    if (s.block()) {
        if (ctx->lattice != 2 || ctx->compute != DT_F32) return LBM_ERR_ARG;
        bool whole;
        if (s.th < 1 || s.th > block_max_rows(ctx->storage) || s.tw < 1 || s.tw > 64) return LBM_ERR_ARG;
        const bool cut = s.tw % 2 == 0 && 2 * s.tw < std::min(s.th, BLOCK_COLS);  // halos fit, words stay aligned
        block_tiles(ctx, cut ? s.tw : 0, s.th, &whole, nullptr);
        if (!whole && !cut) return LBM_ERR_ARG;
        if (ctx->storage == DT_F32) k = step_kernel_block_f32(ctx->collision, s.th);
        else if (ctx->storage == DT_F16) k = step_kernel_block_f16(ctx->collision, s.th);
        else if (ctx->storage == DT_BF16) k = step_kernel_block_bf16(ctx->collision, s.th);
        if (!k) return LBM_ERR_ARG;
        smem = block_smem_bytes(ctx->storage, s.th);
        p.halo = s.tw;
        LBM_CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    } else if (s.single_tube()) {
        if (ctx->lattice != 1) return LBM_ERR_ARG;
        if (ctx->storage == DT_F32) k = step_kernel_single_tube_f32();
        else if (ctx->storage == DT_F16) k = step_kernel_single_tube_f16();
        else if (ctx->storage == DT_BF16) k = step_kernel_single_tube_bf16();
    } else if (s.kind >= 1) {
        if (ctx->lattice != 2 || ctx->compute != DT_F32 || !s.tma()) return LBM_ERR_ARG;
        k = find_smem_kernel(ctx, s.kind - 1, false, &smem);
        if (!k) return LBM_ERR_ARG;
        LBM_CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const int rc = build_tensor_maps(ctx, s.kind - 1);
        if (rc != LBM_OK) return rc;
    } else {
        if (is_flat(ctx, s) && (s.tw != 32 || s.th != 1)) return LBM_ERR_ARG;
        k = find_step_kernel(ctx->lattice, ctx->storage, ctx->collision, s.V);
    }
    if (!k) return LBM_ERR_ARG;
    if (is_flat(ctx, s)) p.flat_nodes = flat_nodes(ctx);
    const std::vector<TileDesc> t = build_tiles(ctx, p);
    if (tile0 + (int64_t)t.size() > ctx->layout.max_tiles) return LBM_ERR_ARG;
    LBM_CK(cudaMemcpyAsync(ctx->d_tiles + tile0, t.data(), sizeof(TileDesc) * t.size(),
                           cudaMemcpyHostToDevice, ctx->stream));
    LBM_CK(cudaMemcpyAsync(ctx->d_inst, ctx->layout.inst.data(), sizeof(InstDesc) * ctx->count,
                           cudaMemcpyHostToDevice, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    // two CTAs of 8 warps on an SM where there are more regions than SMs
    if (s.block())
        p.block_warps = (int64_t)t.size() > ctx->num_sms && 2 * smem <= 220 * 1024 ? BLOCK_WARPS / 2 : BLOCK_WARPS;
    const int block = block_threads(ctx, p);
    if (is_flat(ctx, s)) {
        // An SM takes as many CTAs as it has room for, so a grid of a few
        // CTAs per SM is dealt unevenly: claim the shared memory that leaves
        // room for an equal share and no more.  Up to four warps per SM, one
        // per scheduler, gain nothing (40 lattices of 17 x 17: 12.6 us either
        // way), and leave their SMs free for other streams' work.
        const int64_t ctas = (int64_t)t.size() * (p.flat_nodes / block);
        const int64_t share = (ctas + ctx->num_sms - 1) / ctx->num_sms;
        if (share > 4 && share <= 32) smem = (size_t)(227 * 1024 / share - 1024) / 1024 * 1024;
        LBM_CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024));
    }
    int per_sm = 0;
    LBM_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, smem));
    per_sm = std::max(per_sm, 1);
    int64_t g = s.block() ? (int64_t)t.size()
                : ctx->lattice == 1 && !s.single_tube() ? ((int64_t)t.size() * 32 + block - 1) / block
                : is_flat(ctx, s) ? (int64_t)t.size() * (p.flat_nodes / block)
                                  : std::min<int64_t>((int64_t)per_sm * ctx->num_sms, (int64_t)t.size());
    if (s.tma() && smem_stages(ctx->storage, s.kind - 1) == 2 && 2 * g < (int64_t)t.size()) {
        // more tiles than the CTAs' first two: the others are drawn
        const void* kd = find_smem_kernel(ctx, s.kind - 1, true, &smem);
        LBM_CK(cudaFuncSetAttribute(kd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        LBM_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kd, block, smem));
        const int64_t gd = (int64_t)std::max(per_sm, 1) * ctx->num_sms;
        if (2 * gd < (int64_t)t.size()) {
            k = kd;
            g = gd;
            p.draws = true;
        }
    }
    p.kern = k;
    p.smem = smem;
    p.grid = (int)std::max<int64_t>(g, 1);
    p.ntiles = (int32_t)t.size();
    *out = p;
    return LBM_OK;
}

// Make shape s the context's plan, alone.
int apply_shape(lbm_ctx* ctx, const Shape& s, int halo = 0) {
    const int rc = make_plan(ctx, s, halo, 0, &ctx->plan);
    if (rc != LBM_OK) return rc;
    ctx->single.kern = nullptr;
    ctx->plan_from = 1;
    for (int p = 0; p < 2; ++p) {
        if (ctx->graph[p]) cudaGraphExecDestroy(ctx->graph[p]);
        ctx->graph[p] = nullptr;
    }
    return LBM_OK;
}

// Shape s for single steps beside the plan; launches of `from` steps on stay
// with the plan.  Where the tile table has no room for both the plan remains
// alone.
int add_single(lbm_ctx* ctx, const Shape& s, int from) {
    const int rc = make_plan(ctx, s, 0, ctx->plan.ntiles, &ctx->single);
    if (rc == LBM_OK) ctx->plan_from = from;
    return rc == LBM_ERR_ARG ? LBM_OK : rc;
}

// TMA tensor maps of both population buffers: per instance a 3-D view
// (x < nx, row, plane) of the populations, once with the box of one plane
// of a tile of the staged kernel (loads and stores: x beyond nx reads as
// zero and is not written) and once with a 16-byte-wide box of the tile's
// rows (the x halo loads).
int build_tensor_maps(lbm_ctx* ctx, int variant) {
    if (ctx->tmaps_variant == variant) return LBM_OK;
    using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    LBM_CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                            &q));
    if (!fn || q != cudaDriverEntryPointSuccess) return LBM_ERR_CUDA;
    EncodeFn encode = reinterpret_cast<EncodeFn>(fn);
    const size_t es = dtype_bytes(ctx->storage);
    const int E = (int)(16 / es);
    const int tile_nodes = smem_tile_nodes(ctx->storage, variant);
    std::vector<CUtensorMap> maps(4 * (size_t)ctx->count);
    for (int m = 0; m < 4; ++m) {
        const int b = m >> 1;
        const bool halo = (m & 1) != 0;
        for (int i = 0; i < ctx->count; ++i) {
            const InstDesc& in = ctx->layout.inst[i];
            const int X = smem_tile_width(in.nx, in.ny, tile_nodes, smem_threads(variant),
                                          smem_least_padding(ctx->collision));
            const int R = tile_nodes / X;
            void* base = ctx->buf[b] + (size_t)in.off * es;
            cuuint64_t dims[3] = {(cuuint64_t)in.nx, (cuuint64_t)in.ny, 9};
            cuuint64_t strides[2] = {(cuuint64_t)in.pitch * es, (cuuint64_t)in.plane * es};
            cuuint32_t box[3] = {(cuuint32_t)(halo ? E : X), (cuuint32_t)R, 1};
            cuuint32_t estr[3] = {1, 1, 1};
            CUresult r = encode(&maps[(size_t)m * ctx->count + i],
                                es == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                                3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) {
                if (getenv("LBM_DEBUG")) fprintf(stderr, "liblbm: tensor map encode failed (%d)\n", (int)r);
                return LBM_ERR_CUDA;
            }
        }
    }
    static_assert(sizeof(CUtensorMap) == sizeof(CUtensorMapOpaque), "tensor map size");
    LBM_CK(cudaMemcpyAsync(ctx->d_tmaps, maps.data(), sizeof(CUtensorMap) * maps.size(),
                           cudaMemcpyHostToDevice, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    ctx->tmaps_variant = variant;
    return LBM_OK;
}

StepArgs step_args(const lbm_ctx* ctx, const StepPlan& p, int src) {
    StepArgs a;
    a.src = ctx->buf[src];
    a.dst = ctx->buf[1 - src];
    a.inst = ctx->d_inst;
    a.tiles = ctx->d_tiles + p.tile0;
    a.ntiles = p.ntiles;
    a.tw = is_flat(ctx, p.shape) ? p.flat_nodes : p.shape.tw;
    a.tw_log2 = p.shape.tw > 0 ? ilog2(p.shape.tw) : 0;
    a.th = p.shape.th;
    a.rho0 = ctx->rho0;
    a.status = ctx->d_status;
    a.tmaps = ctx->d_tmaps + (size_t)src * 2 * ctx->count;
    a.tmaps_halo = ctx->d_tmaps + (size_t)(src * 2 + 1) * ctx->count;
    a.tmaps_dst = ctx->d_tmaps + (size_t)(1 - src) * 2 * ctx->count;
    a.error = ctx->d_error;
    a.tile_counters = ctx->d_error + TILE_COUNTERS;
    a.spin_limit = ctx->spin_limit;
    a.lost_tile = ctx->lost_tile;
    a.inplace = 0;
    a.steps = 1;
    a.halo = p.halo;
    return a;
}

// One step launch.  It is a programmatic dependent launch: the kernel may be
// scheduled while the previous kernel in the stream drains, and waits for its
// completion (griddepcontrol.wait) before touching device state.
// inplace: the (first) step collides without streaming (one-node-per-thread
// and tube kernels only); steps: time steps of the launch (tube and region
// kernels only).
cudaError_t launch_step(lbm_ctx* ctx, const StepPlan& p, int src, cudaStream_t s, bool inplace = false,
                        int steps = 1) {
    StepArgs a = step_args(ctx, p, src);
    a.inplace = inplace ? 1 : 0;
    a.steps = steps;
    void* params[] = {&a};
    const int block = block_threads(ctx, p);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, p.kern, params);
}

// Time of a launch of `steps` steps of the current plan in milliseconds, on
// the rest-state buffers: after an untimed launch three back-to-back
// launches (as the step loop runs them: a launch's tail overlaps the next
// one's start), for single steps the faster of two such runs; < 0 on a CUDA
// error.
float time_current_shape(lbm_ctx* ctx, cudaEvent_t* ev, int steps = 1) {
    // (several steps make a launch long enough for one run to do)
    const int runs = steps == 1 ? 2 : 1;
    if (launch_step(ctx, ctx->plan, 0, ctx->stream, false, steps) != cudaSuccess) return -1.f;
    int src = 1;
    float t[2] = {1e30f, 1e30f};
    for (int r = 0; r < runs; ++r) {
        if (cudaEventRecord(ev[2 * r], ctx->stream) != cudaSuccess) return -1.f;
        for (int k = 0; k < 3; ++k, src ^= 1)
            if (launch_step(ctx, ctx->plan, src, ctx->stream, false, steps) != cudaSuccess) return -1.f;
        if (cudaEventRecord(ev[2 * r + 1], ctx->stream) != cudaSuccess) return -1.f;
    }
    if (cudaEventSynchronize(ev[2 * runs - 1]) != cudaSuccess) return -1.f;
    for (int r = 0; r < runs; ++r)
        if (cudaEventElapsedTime(&t[r], ev[2 * r], ev[2 * r + 1]) != cudaSuccess) return -1.f;
    return std::min(t[0], t[1]) / 3.f;
}

// Time per step over some 12 steps of back-to-back launches of `steps` steps
// of the current plan, the faster of two trains: long enough that the first
// launch, which three launches are mostly, does not count.
float time_current_train(lbm_ctx* ctx, cudaEvent_t* ev, int steps = 1) {
    const int n = std::max(2, 12 / steps);
    int src = 0;
    float t[2];
    for (int r = 0; r < 2; ++r) {
        if (cudaEventRecord(ev[2 * r], ctx->stream) != cudaSuccess) return -1.f;
        for (int k = 0; k < n; ++k, src ^= 1)
            if (launch_step(ctx, ctx->plan, src, ctx->stream, false, steps) != cudaSuccess) return -1.f;
        if (cudaEventRecord(ev[2 * r + 1], ctx->stream) != cudaSuccess) return -1.f;
    }
    if (cudaEventSynchronize(ev[3]) != cudaSuccess) return -1.f;
    for (int r = 0; r < 2; ++r)
        if (cudaEventElapsedTime(&t[r], ev[2 * r], ev[2 * r + 1]) != cudaSuccess) return -1.f;
    return std::min(t[0], t[1]) / (float)(n * steps);
}

// The same timing through a captured graph of four launches, as the step
// loop replays them: one warm-up replay, then the faster of two, per launch.
// The deep ring with FP32 storage ran 5 % slower in graphs than as single
// launches (the 10-warp CTAs did not), so close calls are decided here.
float time_current_shape_graph(lbm_ctx* ctx, cudaEvent_t* ev) {
    cudaGraph_t graph;
    if (cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
        return -1.f;
    bool ok = true;
    for (int k = 0; k < 4; ++k)
        ok = ok && launch_step(ctx, ctx->plan, k & 1, ctx->capture_stream) == cudaSuccess;
    if (cudaStreamEndCapture(ctx->capture_stream, &graph) != cudaSuccess || !ok) return -1.f;
    cudaGraphExec_t g = nullptr;
    const cudaError_t e = cudaGraphInstantiate(&g, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return -1.f;
    float t[2] = {-1.f, -1.f};
    ok = cudaGraphLaunch(g, ctx->stream) == cudaSuccess;
    for (int r = 0; r < 2 && ok; ++r)
        ok = cudaEventRecord(ev[2 * r], ctx->stream) == cudaSuccess &&
             cudaGraphLaunch(g, ctx->stream) == cudaSuccess &&
             cudaEventRecord(ev[2 * r + 1], ctx->stream) == cudaSuccess;
    ok = ok && cudaEventSynchronize(ev[3]) == cudaSuccess;
    for (int r = 0; r < 2 && ok; ++r)
        ok = cudaEventElapsedTime(&t[r], ev[2 * r], ev[2 * r + 1]) == cudaSuccess;
    cudaGraphExecDestroy(g);
    return ok ? std::min(t[0], t[1]) / 4.f : -1.f;
}

// Autotuner cache: the chosen shape per (device, lattice, types, rule,
// boundary, instance sizes).  Kept for the life of the process, and in the
// text file named by LBM_AUTOTUNE_CACHE when that variable is set (one line
// per key: "<key> V tw th kind"; for the region kernel also "<key>/single" with
// the shape beside it and "<key>/from" with its shortest launch), so that a later process -- a profiler run,
// for instance -- takes the same shape without timing anything.
std::mutex g_tune_mu;
std::map<std::string, Shape>& tune_cache() {
    static std::map<std::string, Shape> m;
    return m;
}

std::string tune_key(const lbm_ctx* ctx) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceProp prop;
    std::string name = "?";
    if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) name = prop.name;
    for (char& c : name)
        if (c == ' ') c = '_';
    // sizes as a sorted histogram, hashed (FNV-1a)
    std::vector<std::pair<int64_t, int64_t>> d;
    for (const InstDesc& in : ctx->layout.inst) d.push_back({in.nx, in.ny});
    std::sort(d.begin(), d.end());
    uint64_t h = 1469598103934665603ull;
    for (auto& p : d)
        for (int64_t v : {p.first, p.second}) {
            h ^= (uint64_t)v;
            h *= 1099511628211ull;
        }
    char buf[256];
    // "k2": the set of kernels that were timed
    snprintf(buf, sizeof buf, "%s/k2/sm%d/lat%d/st%d/cp%d/co%d/bc%d/n%d/%016llx", name.c_str(),
             ctx->num_sms, ctx->lattice, ctx->storage, ctx->compute, ctx->collision, ctx->bc,
             ctx->count, (unsigned long long)h);
    return buf;
}

bool tune_lookup(const std::string& key, Shape* s) {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = tune_cache().find(key);
    if (it != tune_cache().end()) {
        *s = it->second;
        return true;
    }
    const char* path = getenv("LBM_AUTOTUNE_CACHE");
    if (!path || !*path) return false;
    FILE* f = fopen(path, "r");
    if (!f) return false;
    char k[256];
    Shape t{};
    bool found = false;
    while (fscanf(f, "%255s %d %d %d %d", k, &t.V, &t.tw, &t.th, &t.kind) == 5) {
        if (key == k) {
            *s = t;
            found = true;  // the last entry for a key wins
        }
    }
    fclose(f);
    if (found) tune_cache()[key] = *s;
    return found;
}

void tune_store(const std::string& key, const Shape& s) {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    tune_cache()[key] = s;
    const char* path = getenv("LBM_AUTOTUNE_CACHE");
    if (!path || !*path) return;
    FILE* f = fopen(path, "a");
    if (!f) return;
    fprintf(f, "%s %d %d %d %d\n", key.c_str(), s.V, s.tw, s.th, s.kind);
    fclose(f);
}

// Keep the fastest candidate shape: each is timed over back-to-back
// launches on the rest-state buffers (the collision's instruction stream
// does not depend on the data); close ones are
// timed again in a captured graph, which decides.  Where the region kernel
// takes less for its steps, it becomes the plan, and the fastest shape
// with one step per launch stays beside it for calls and remainders of fewer
// steps than pay for a region's loads and stores.  Then the buffers and
// counters are cleared.  Shapes found in the cache are applied without
// timing.
int autotune(lbm_ctx* ctx) {
    const std::string key = tune_key(ctx);
    Shape best_s{}, one{}, from{};  // from.V: steps of the shortest launch of the region kernel
    if (tune_lookup(key, &best_s) &&
        (!best_s.block() || (tune_lookup(key + "/single", &one) && tune_lookup(key + "/from", &from))) &&
        apply_shape(ctx, best_s) == LBM_OK)
        return best_s.block() ? add_single(ctx, one, std::min(std::max(from.V, 1), ctx->plan.halo)) : LBM_OK;
    const std::vector<Shape> cands = candidate_shapes(ctx->storage);
    if (cands.size() == 1) return apply_shape(ctx, cands[0]);
    cudaEvent_t ev[6];
    for (int i = 0; i < 6; ++i) LBM_CK(cudaEventCreate(&ev[i]));
    float best = 1e30f;
    best_s = default_shape_d2q9(ctx->storage);
    int rc = LBM_OK;
    std::vector<float> t(cands.size(), -1.f);
    for (size_t c = 0; c < cands.size(); ++c) {
        if (apply_shape(ctx, cands[c]) != LBM_OK) continue;
        const float ms = time_current_shape(ctx, ev);
        if (ms < 0.f) {
            rc = LBM_ERR_CUDA;
            break;
        }
        t[c] = ms;
        best = std::min(best, ms);
    }
    // The region kernel, unless its model leaves it no chance: a launch of k
    // steps takes t1 + (k - 1) slope.
    int K = 0, rows = 0;
    double us = 0.0;
    float tK = -1.f, t1 = -1.f;
    if (rc == LBM_OK && block_plan(ctx, &K, &rows, &us) && us < 1e3 * best &&
        apply_shape(ctx, Shape{2, K, rows, 5}) == LBM_OK) {
        tK = time_current_shape(ctx, ev, K);
        if (tK < 0.f) rc = LBM_ERR_CUDA;
    }
    // Candidates within 5 % of the fastest are timed once more, after the
    // others, through a captured graph as the step loop runs them, and
    // that time decides between them.
    int near = 0;
    for (size_t c = 0; c < cands.size(); ++c) {
        near += t[c] >= 0.f && t[c] <= 1.05f * best;
        if (t[c] == best) best_s = cands[c];
    }
    if (near > 1) {
        float fastest = 1e30f;
        for (size_t c = 0; c < cands.size() && rc == LBM_OK; ++c) {
            if (t[c] < 0.f || t[c] > 1.05f * best) continue;
            if (apply_shape(ctx, cands[c]) != LBM_OK) continue;
            const float ms = time_current_shape_graph(ctx, ev);
            if (ms < 0.f) {
                rc = LBM_ERR_CUDA;
                break;
            }
            if (getenv("LBM_DEBUG"))
                fprintf(stderr, "liblbm: autotune kind %d: %.4f ms in a graph\n", cands[c].kind, ms);
            if (ms < fastest) {
                fastest = ms;
                best_s = cands[c];
            }
        }
    }
    one = best_s;
    // Where the region kernel comes close to it, trains of both decide
    // (1001 x 333 FP32 TRT: 6.1 us a step against 7.0 by three launches or a
    // graph, and 6.1 against 5.8 in trains and in the step loop).
    bool region = rc == LBM_OK && tK >= 0.f && tK < K * best;
    if (region && tK >= 0.7f * K * best) {
        float step[2] = {-1.f, -1.f};
        if (apply_shape(ctx, Shape{2, K, rows, 5}) == LBM_OK) step[0] = time_current_train(ctx, ev, K);
        if (apply_shape(ctx, one) == LBM_OK) step[1] = time_current_train(ctx, ev);
        if (step[0] < 0.f || step[1] < 0.f) rc = LBM_ERR_CUDA;
        region = step[0] < step[1];
        if (getenv("LBM_DEBUG"))
            fprintf(stderr, "liblbm: autotune trains: regions %.4f ms a step, kind %d %.4f\n", step[0], one.kind, step[1]);
    }
    if (rc == LBM_OK && region) {
        // The region kernel takes launches of the steps from which on it is
        // ahead by a tenth of single steps, whose time in a row is
        // 0.8 of what was timed.
        best_s = {2, K, rows, 5};
        if (apply_shape(ctx, best_s) == LBM_OK) t1 = time_current_shape(ctx, ev, 1);
        if (t1 < 0.f) rc = LBM_ERR_CUDA;
        const float slope = (tK - t1) / (K - 1);
        from = {1, 0, 0};
        while (from.V < K && t1 + (from.V - 1) * slope > 0.9f * 0.8f * from.V * best) ++from.V;
    }
    if (getenv("LBM_DEBUG")) {
        for (size_t c = 0; c < cands.size(); ++c)
            fprintf(stderr, "liblbm: autotune kind %d V %d tw %d th %d: %.4f ms per launch\n", cands[c].kind,
                    cands[c].V, cands[c].tw, cands[c].th, t[c]);
        if (tK >= 0.f)
            fprintf(stderr, "liblbm: autotune regions of %d rows: 1 step %.4f ms, %d steps %.4f ms (%.4f modelled), "
                    "used from %d\n", rows, t1, K, tK, 1e-3 * K * us, best_s.block() ? from.V : 0);
    }
    for (int i = 0; i < 6; ++i) cudaEventDestroy(ev[i]);
    if (rc != LBM_OK) {
        ctx->failed = true;
        return rc;
    }
    // undo the tuning steps: back to the rest state, counters cleared
    LBM_CK(cudaMemsetAsync(ctx->buf[0], 0, 2 * ctx->cv.buf_bytes, ctx->stream));
    LBM_CK(cudaMemsetAsync(ctx->d_status, 0, sizeof(unsigned long long) * 2 * ctx->count,
                           ctx->stream));
    rc = apply_shape(ctx, best_s);
    if (rc == LBM_OK && best_s.block()) {
        rc = add_single(ctx, one, from.V);
        tune_store(key + "/single", one);
        tune_store(key + "/from", from);
    }
    if (rc == LBM_OK) tune_store(key, best_s);
    return rc;
}

// Capture the step loop of GRAPH_STEPS launches for both buffer parities and
// upload the executable graphs, so that no capture or first-launch upload
// happens inside a later lbm_step.
int capture_graphs(lbm_ctx* ctx) {
    if (ctx->plan.shape.block()) return LBM_OK;  // several steps per launch: no graph
    for (int p = 0; p < 2; ++p) {
        cudaGraphExec_t& g = ctx->graph[p];
        if (g) continue;
        cudaGraph_t graph;
        LBM_CK(cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal));
        int src = p;
        for (int k = 0; k < GRAPH_STEPS; ++k) {
            cudaError_t e = launch_step(ctx, ctx->plan, src, ctx->capture_stream);
            if (e != cudaSuccess) {
                cudaStreamEndCapture(ctx->capture_stream, &graph);
                LBM_CK(e);
            }
            src = 1 - src;
        }
        LBM_CK(cudaStreamEndCapture(ctx->capture_stream, &graph));
        cudaError_t e = cudaGraphInstantiate(&g, graph, 0);
        cudaGraphDestroy(graph);
        LBM_CK(e);
        LBM_CK(cudaGraphUpload(g, ctx->stream));
    }
    return LBM_OK;
}

// The plan takes several steps per launch (tube and region kernels).
bool takes_several(const lbm_ctx* ctx) { return ctx->lattice == 1 || ctx->plan.shape.block(); }

// The next launch of a call with n steps left, of *k steps (post: the stored
// field is post-collision).
const StepPlan& next_launch(const lbm_ctx* ctx, bool post, int64_t n, int* k) {
    *k = 1;
    if (!takes_several(ctx) || (!post && ctx->lattice == 2)) return ctx->plan;
    if (post && n < ctx->plan_from) return ctx->single;
    *k = (int)std::min<int64_t>(n, ctx->plan.halo);
    return ctx->plan;
}

bool parse_shape_env(Shape* s) {
    const char* e = getenv("LBM_SHAPE");
    if (!e) return false;
    if (strcmp(e, "smem") == 0 || strcmp(e, "smem2") == 0) {
        *s = {2, 0, 0, 1};
        return true;
    }
    if (strcmp(e, "smems") == 0) {
        *s = {2, 0, 0, 2};
        return true;
    }
    if (strcmp(e, "smemw") == 0) {
        *s = {2, 0, 0, 3};
        return true;
    }
    if (strcmp(e, "smemd") == 0) {
        *s = {2, 0, 0, 4};
        return true;
    }
    int v, tw, th;
    if (sscanf(e, "block,%d,%d", &tw, &th) == 2) {
        *s = {2, tw, th, 5};
        return true;
    }
    if (sscanf(e, "%d,%d,%d", &v, &tw, &th) != 3) return false;
    *s = {v, tw, th};
    return true;
}

void lid_deviation(double rho0, double u, double* dev) {
    // f^eq_a(rho0, (u, 0)) - W_a rho0, Eq. (numerical-plyeqm); D2Q9 in T's column order.
    static const int vx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
    for (int a = 0; a < 9; ++a) {
        const double w = a == 0 ? 4.0 / 9.0 : (a < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
        const double vu = vx[a] * u;
        dev[a] = w * rho0 * (3.0 * vu + 4.5 * vu * vu - 1.5 * u * u);
    }
}

int validate_opts(const lbm_opts* o) {
    if (o->compute != DT_F64 && o->compute != DT_F32) return LBM_ERR_ARG;
    if (o->storage < DT_F64 || o->storage > DT_BF16) return LBM_ERR_ARG;
    if (o->compute == DT_F64 && o->storage != DT_F64) return LBM_ERR_ARG;
    if (o->compute == DT_F32 && o->storage == DT_F64) return LBM_ERR_ARG;
    if (o->collision < COLL_MINXENT4 || o->collision > COLL_TRT) return LBM_ERR_ARG;
    if (o->tau2_reading != TAU2_PRINTED && o->tau2_reading != TAU2_MAGIC) return LBM_ERR_ARG;
    if (o->reserved != 0) return LBM_ERR_ARG;
    if (!(o->rho0 > 0.0) || !std::isfinite(o->rho0)) return LBM_ERR_ARG;
    return LBM_OK;
}

int validate_dims(int lat, int32_t count, const int64_t* dims,
                  std::vector<std::pair<int64_t, int64_t>>* out) {
    if (lat != 1 && lat != 2) return LBM_ERR_ARG;
    if (count < 1 || count > 65535 || !dims) return LBM_ERR_ARG;
    for (int i = 0; i < count; ++i) {
        const int64_t nx = dims[2 * i], ny = dims[2 * i + 1];
        if (nx < 1 || ny < 1 || nx > (1 << 26) || ny > (1 << 26)) return LBM_ERR_ARG;
        if (lat == 1 && ny != 1) return LBM_ERR_ARG;
        if (nx * ny > ((int64_t)1 << 31)) return LBM_ERR_ARG;
        out->push_back({nx, ny});
    }
    return LBM_OK;
}

// Device address of a host array the GPU can read and write in place
// (page-locked memory registered with CUDA: cudaHostAlloc, cudaHostRegister,
// torch's pin_memory), or nullptr.  A null array counts as addressable.
// Host I/O with such arrays runs its kernels straight on them, without
// staging copies: on a GB300 the kernel streams them over the CPU-GPU link.
template <typename P> bool device_view(P* host, P** dev) {
    if (!host) {
        *dev = nullptr;
        return true;
    }
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, host) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (at.type != cudaMemoryTypeHost || !at.devicePointer) return false;
    *dev = static_cast<P*>(at.devicePointer);
    return true;
}

// Auxiliary-kernel arguments that cover instance i alone, with host arrays
// indexed from its first node.
AuxArgs aux_args_instance(const lbm_ctx* ctx, int i) {
    AuxArgs a = aux_args(ctx);
    const InstDesc& in = ctx->layout.inst[i];
    a.inst = ctx->d_inst + i;
    a.count = 1;
    a.max_nodes = a.total_nodes = (int64_t)in.nx * in.ny;
    a.max_ny = in.ny;
    a.node_base = in.node0;
    return a;
}

// Header of a saved state (lbm_save_state): the layout it fits and the
// context's position in its run, followed by the status counters and the
// raw population buffer.
struct StateHeader {
    char magic[8];
    uint32_t version;
    int32_t lattice, storage, count;
    int32_t post, reserved;
    int64_t steps;
    uint64_t layout_hash, buf_bytes, status_bytes;
    uint64_t pad[8];
};
static_assert(sizeof(StateHeader) == 128, "state header is 128 bytes");
constexpr char STATE_MAGIC[8] = {'L', 'B', 'M', 'S', 'T', 'A', 'T', 'E'};

uint64_t layout_hash(const lbm_ctx* ctx) {
    uint64_t h = 1469598103934665603ull;
    auto mix = [&](uint64_t v) {
        h ^= v;
        h *= 1099511628211ull;
    };
    mix((uint64_t)ctx->lattice);
    mix((uint64_t)ctx->storage);
    for (const InstDesc& in : ctx->layout.inst) {
        mix((uint64_t)in.nx);
        mix((uint64_t)in.ny);
        mix((uint64_t)in.pitch);
        mix((uint64_t)in.plane);
        mix((uint64_t)in.off);
    }
    return h;
}

// The counters of the TMA kernel's drawn tiles are 0 between launches; a
// launch that timed out may leave them otherwise, so every entry point that
// sets a state clears them (the sticky error word is another matter).
cudaError_t clear_tile_counters(lbm_ctx* ctx) {
    if (!ctx->plan.draws && !ctx->single.draws) return cudaSuccess;
    return cudaMemsetAsync(ctx->d_error + TILE_COUNTERS, 0, 2 * sizeof(unsigned int), ctx->stream);
}

// LBM_ERR_UNSTABLE when instance i has flagged an unstable node (sticky
// error word first); syncs.
int instance_status(lbm_ctx* ctx, int32_t instance) {
    int64_t c[3];
    int rc = lbm_status_instance(ctx, instance, c);
    if (rc != LBM_OK) return rc;
    unsigned int err = 0;
    LBM_CK(cudaMemcpyAsync(&err, ctx->d_error, sizeof err, cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    if (err) return LBM_ERR_TIMEOUT;
    return c[1] ? LBM_ERR_UNSTABLE : LBM_OK;
}

uint64_t state_bytes(const lbm_ctx* ctx) {
    return sizeof(StateHeader) + sizeof(unsigned long long) * 2 * (uint64_t)ctx->count +
           (uint64_t)ctx->cv.buf_bytes;
}

}  // namespace

namespace lbm {
// Inputs of the conservation reduction of a context, for entry points that
// live in other translation units.  Returns LBM_OK, or the code the public
// conservation call would return for this context.
int ctx_conservation_inputs(const lbm_ctx* ctx, AuxArgs* args, const void** src, int* count) {
    if (!ctx) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    *args = aux_args(ctx);
    *src = ctx->buf[ctx->cur];
    *count = ctx->count;
    return LBM_OK;
}
}  // namespace lbm

extern "C" {

void lbm_default_opts(lbm_opts* o) {
    if (!o) return;
    std::memset(o, 0, sizeof *o);
    o->compute = DT_F64;
    o->storage = DT_F64;
    o->collision = COLL_MINXENT4;
    o->autotune = 1;
    o->rho0 = 1.0;
}

int lbm_required_bytes(lbm_lattice lat, int32_t count, const int64_t* dims, const lbm_opts* opts,
                       uint64_t* bytes) {
    if (!bytes) return LBM_ERR_ARG;
    lbm_opts o;
    if (opts) o = *opts;
    else lbm_default_opts(&o);
    if (validate_opts(&o) != LBM_OK) return LBM_ERR_ARG;
    std::vector<std::pair<int64_t, int64_t>> d;
    if (validate_dims(lat, count, dims, &d) != LBM_OK) return LBM_ERR_ARG;
    Layout L = make_layout(lat, o.storage, d);
    *bytes = carve(L, lat, o.storage, count).total;
    return LBM_OK;
}

int lbm_create_batch(lbm_ctx** out, lbm_lattice lat, int32_t count, const int64_t* dims,
                     const double* nu, const double* u_lid, lbm_bc bc, const lbm_opts* opts) {
    lbm_ctx* ctx = nullptr;
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    lbm_opts o;
    if (opts) o = *opts;
    else lbm_default_opts(&o);
    if (validate_opts(&o) != LBM_OK) return LBM_ERR_ARG;
    std::vector<std::pair<int64_t, int64_t>> d;
    if (validate_dims(lat, count, dims, &d) != LBM_OK || !nu) return LBM_ERR_ARG;
    if (bc != LBM_BC_PERIODIC && bc != LBM_BC_ZERO_GRADIENT && bc != LBM_BC_CAVITY)
        return LBM_ERR_ARG;
    if (bc == LBM_BC_CAVITY) {
        if (lat != LBM_D2Q9) return LBM_ERR_ARG;
        for (auto& p : d)
            if (p.first < 3 || p.second < 3) return LBM_ERR_ARG;
    }
    for (int i = 0; i < count; ++i) {
        // Eq. (visco-tau): tau = 3 nu + 1/2 must exceed 1/2
        if (!(nu[i] > 0.0) || !std::isfinite(nu[i])) return LBM_ERR_ARG;
        if (u_lid && !std::isfinite(u_lid[i])) return LBM_ERR_ARG;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBM_ERR_NODEV;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return LBM_ERR_NODEV;
    if (prop.major != 10 || prop.minor != 3) return LBM_ERR_NODEV;

    ctx = new lbm_ctx();
    ctx->lattice = lat;
    ctx->Q = lat == LBM_D2Q9 ? 9 : 3;
    ctx->count = count;
    ctx->bc = bc;
    ctx->compute = o.compute;
    ctx->storage = o.storage;
    ctx->collision = o.collision;
    ctx->rho0 = o.rho0;
    ctx->stream = static_cast<cudaStream_t>(o.stream);
    ctx->num_sms = prop.multiProcessorCount;
    // Test hooks of the bounded-wait timeout path (TMA kernel): a smaller
    // spin limit, and one tile whose copies are never issued.
    if (const char* e = getenv("LBM_SPIN_LIMIT")) {
        const long v = strtol(e, nullptr, 10);
        if (v >= 1 && v <= (1 << 20)) ctx->spin_limit = (int)v;
    }
    if (const char* e = getenv("LBM_TEST_LOST_TILE")) ctx->lost_tile = (int)strtol(e, nullptr, 10);
    ctx->layout = make_layout(lat, o.storage, d);
    ctx->cv = carve(ctx->layout, lat, o.storage, count);
    for (int i = 0; i < count; ++i) {
        InstDesc& in = ctx->layout.inst[i];
        const double tau = 3.0 * nu[i] + 0.5;
        in.bc = bc;
        in.omega = 1.0 / tau;
        // Eq. (tau2), as printed or in the magic-parameter reading
        const double tau2 = (8.0 * tau - 1.0) /
                            ((o.tau2_reading == TAU2_MAGIC ? 8.0 : 1.0) * (2.0 * tau - 1.0));
        in.omega2 = 1.0 / tau2;
        // Table III: MRT fixes the energy rates, TRT uses 1/tau for them
        in.s_e = o.collision == COLL_MRT ? 1.64 : in.omega;
        in.s_eps = o.collision == COLL_MRT ? 1.54 : in.omega;
        in.u_lid = u_lid ? u_lid[i] : 0.0;
        in.rates_f[0] = (float)in.omega;
        in.rates_f[1] = (float)in.omega2;
        in.rates_f[2] = (float)in.s_e;
        in.rates_f[3] = (float)in.s_eps;
        if (bc == LBM_BC_CAVITY) {
            lid_deviation(o.rho0, in.u_lid, in.lid_dev);
            for (int a = 0; a < 9; ++a) in.lid_dev_f[a] = (float)in.lid_dev[a];
        }
    }
    int rc = LBM_OK;
    if (o.device_mem) {
        if (o.device_mem_bytes < ctx->cv.total || ((uintptr_t)o.device_mem & 255u)) {
            delete ctx;
            return LBM_ERR_ARG;
        }
        ctx->mem = static_cast<char*>(o.device_mem);
    } else {
        void* p = nullptr;
        if (cudaMalloc(&p, ctx->cv.total) != cudaSuccess) {
            cudaGetLastError();
            delete ctx;
            return LBM_ERR_ALLOC;
        }
        ctx->mem = static_cast<char*>(p);
        ctx->own_mem = true;
    }
    ctx->buf[0] = ctx->mem;
    ctx->buf[1] = ctx->mem + ctx->cv.buf_bytes;
    ctx->d_inst = reinterpret_cast<InstDesc*>(ctx->mem + ctx->cv.inst_off);
    ctx->d_tiles = reinterpret_cast<TileDesc*>(ctx->mem + ctx->cv.tiles_off);
    ctx->d_status = reinterpret_cast<unsigned long long*>(ctx->mem + ctx->cv.status_off);
    ctx->d_partials = reinterpret_cast<double*>(ctx->mem + ctx->cv.partials_off);
    ctx->d_cons = reinterpret_cast<int2*>(ctx->mem + ctx->cv.cons_off);
    ctx->d_stage = reinterpret_cast<double*>(ctx->mem + ctx->cv.stage_off);
    ctx->d_tmaps = reinterpret_cast<CUtensorMapOpaque*>(ctx->mem + ctx->cv.tmap_off);
    ctx->d_error = reinterpret_cast<unsigned int*>(ctx->mem + ctx->cv.err_off);
    auto fail = [&](int code) {
        lbm_destroy(ctx);
        return code;
    };
    if (cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
        return fail(LBM_ERR_CUDA);
    if (cudaMemsetAsync(ctx->mem, 0, ctx->cv.total, ctx->stream) != cudaSuccess)
        return fail(LBM_ERR_CUDA);
    {
        std::vector<int2> items;
        for (int i = 0; i < count; ++i)
            for (int b = 0; b < cons_partials(ctx->layout.inst[i].nx, ctx->layout.inst[i].ny, (int)dtype_bytes(o.storage)); ++b)
                items.push_back({i, b});
        ctx->n_cons = (int)items.size();
        if (cudaMemcpyAsync(ctx->d_cons, items.data(), sizeof(int2) * items.size(),
                            cudaMemcpyHostToDevice, ctx->stream) != cudaSuccess ||
            cudaStreamSynchronize(ctx->stream) != cudaSuccess)
            return fail(LBM_ERR_CUDA);
    }
    Shape s;
    if (lat == 1) {
        // nothing to time: the plan follows from the sizes (LBM_SHAPE pins V
        // and the CTA size)
        int V = 0;
        const bool pinned = parse_shape_env(&s);
        int halo = 0;
        tube_plan(ctx, pinned ? s.V : 0, &V, &halo);
        rc = apply_shape(ctx, pinned ? s : Shape{V, 128, 1}, halo);
        if (rc == LBM_OK && !pinned && o.compute == DT_F32) {
            // CTAs of 128 threads, of fewer where the tubes do not fill them
            // (5000 tubes of 100 nodes, one step: FP32 7.9 us with 128, FP16 10.7)
            const int per = o.storage == DT_F32 ? 4 : 8;
            int threads = 32;
            while (threads < 128 && threads * per < ctx->layout.max_nx) threads *= 2;
            rc = add_single(ctx, Shape{per, threads, 1, 6}, 2);
        }
    } else if (parse_shape_env(&s)) rc = apply_shape(ctx, s);
    else if (o.autotune && !getenv("LBM_NO_AUTOTUNE")) rc = autotune(ctx);
    else rc = apply_shape(ctx, default_shape_d2q9(o.storage));
    if (rc != LBM_OK) return fail(rc);
    if (lat == 2) rc = capture_graphs(ctx);  // the tube kernel takes several steps per launch
    if (rc != LBM_OK) return fail(rc);
    *out = ctx;
    return LBM_OK;
}

int lbm_create(lbm_ctx** out, lbm_lattice lat, const int64_t* dims, double nu, lbm_bc bc,
               double u_lid, const lbm_opts* opts) {
    return lbm_create_batch(out, lat, 1, dims, &nu, &u_lid, bc, opts);
}

int lbm_destroy(lbm_ctx* ctx) {
    if (!ctx) return LBM_OK;
    for (int p = 0; p < 2; ++p)
        if (ctx->graph[p]) cudaGraphExecDestroy(ctx->graph[p]);
    if (ctx->capture_stream) cudaStreamDestroy(ctx->capture_stream);
    if (ctx->own_mem && ctx->mem) {
        cudaStreamSynchronize(ctx->stream);
        cudaFree(ctx->mem);
    }
    delete ctx;
    return LBM_OK;
}

int lbm_init_device(lbm_ctx* ctx, const double* rho, const double* ux, const double* uy) {
    if (!ctx || !rho) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    AuxArgs a = aux_args(ctx);
    a.error = ctx->d_error;  // the kernel clears the status counters and the error block
    LBM_CK(run_aux(AuxOp::Init, a, nullptr, ctx->buf[ctx->cur], rho, ux, uy, nullptr, nullptr,
                   nullptr));
    ctx->post = false;
    ctx->initialized = true;
    ctx->inst_init.assign(ctx->count, 1);
    ctx->steps = 0;
    return LBM_OK;
}

int lbm_init(lbm_ctx* ctx, const double* rho, const double* ux, const double* uy) {
    if (!ctx || !rho) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    const double *dr, *dx, *dy;
    if (device_view(rho, &dr) && device_view(ux, &dx) && device_view(uy, &dy)) {
        // page-locked arrays: the init kernel reads them in place
        int rc = lbm_init_device(ctx, dr, dx, ctx->Q == 9 ? dy : nullptr);
        if (rc != LBM_OK) return rc;
        LBM_CK(cudaStreamSynchronize(ctx->stream));
        return LBM_OK;
    }
    const size_t n = (size_t)ctx->layout.total_nodes;
    double* r = ctx->d_stage;
    double* x = ux ? ctx->d_stage + n : nullptr;
    double* y = (uy && ctx->Q == 9) ? ctx->d_stage + 2 * n : nullptr;
    LBM_CK(cudaMemcpyAsync(r, rho, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    if (x) LBM_CK(cudaMemcpyAsync(x, ux, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    if (y) LBM_CK(cudaMemcpyAsync(y, uy, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    int rc = lbm_init_device(ctx, r, x, y);
    if (rc != LBM_OK) return rc;
    // the caller may reuse its arrays once we return
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return LBM_OK;
}

int lbm_step(lbm_ctx* ctx, int64_t n) {
    if (!ctx || n < 0) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    if (n == 0) return LBM_OK;
    while (n > 0) {
        if (ctx->lattice == 2 && ctx->post && !takes_several(ctx) && n >= GRAPH_STEPS) {
            cudaGraphExec_t& g = ctx->graph[ctx->cur];
            if (!g) {
                const int rc = capture_graphs(ctx);
                if (rc != LBM_OK) return rc;
            }
            LBM_CK(cudaGraphLaunch(g, ctx->stream));
            n -= GRAPH_STEPS;
            ctx->steps += GRAPH_STEPS;
            continue;
        }
        int k;
        const StepPlan& p = next_launch(ctx, ctx->post, n, &k);
        if (!ctx->post && ctx->lattice == 2 && !is_flat(ctx, p.shape)) {
            AuxArgs a = aux_args(ctx);
            LBM_CK(run_aux(AuxOp::CollideInPlace, a, ctx->buf[ctx->cur], ctx->buf[1 - ctx->cur],
                           nullptr, nullptr, nullptr, nullptr, nullptr, nullptr));
        } else {
            LBM_CK(launch_step(ctx, p, ctx->cur, ctx->stream, !ctx->post, k));
        }
        ctx->cur = 1 - ctx->cur;
        ctx->post = true;
        ctx->steps += k;
        n -= k;
    }
    return LBM_OK;
}

int lbm_step_launches(lbm_ctx* ctx, int64_t n, int64_t* out) {
    if (!ctx || n < 0 || !out) return LBM_ERR_ARG;
    out[0] = out[1] = 0;
    bool post = ctx->post;
    while (n > 0) {
        int k;
        const StepPlan& p = next_launch(ctx, post, n, &k);
        // the same launch again and again, but for the first one and the remainder
        const int64_t m = post ? n / k : 1;
        out[0] += m;
        if (takes_several(ctx) && &p == &ctx->plan && (post || ctx->lattice == 1)) out[1] += m;
        post = true;
        n -= m * k;
    }
    return LBM_OK;
}

int lbm_moments_device(lbm_ctx* ctx, double* rho, double* ux, double* uy) {
    if (!ctx || !rho) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    AuxArgs a = aux_args(ctx);
    LBM_CK(run_aux(AuxOp::Moments, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr, rho,
                   ux, ctx->Q == 9 ? uy : nullptr));
    return LBM_OK;
}

int lbm_stream_function_device(lbm_ctx* ctx, double* psi) {
    if (!ctx || !psi) return LBM_ERR_ARG;
    if (ctx->Q != 9) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    AuxArgs a = aux_args(ctx);
    LBM_CK(run_aux(AuxOp::StreamFunction, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr, psi,
                   nullptr, nullptr));
    return LBM_OK;
}

int lbm_stream_function(lbm_ctx* ctx, double* psi) {
    if (!ctx || !psi) return LBM_ERR_ARG;
    const size_t n = (size_t)ctx->layout.total_nodes;
    double* dpsi = ctx->d_stage;
    int rc = lbm_stream_function_device(ctx, dpsi);
    if (rc != LBM_OK) return rc;
    LBM_CK(cudaMemcpyAsync(psi, dpsi, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    int64_t c[3];
    rc = lbm_status(ctx, c);
    if (rc != LBM_OK) return rc;
    return c[1] ? LBM_ERR_UNSTABLE : LBM_OK;
}

int lbm_status_instance(lbm_ctx* ctx, int32_t instance, int64_t* counters) {
    if (!ctx || !counters || instance < 0 || instance >= ctx->count) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    unsigned long long h[2];
    LBM_CK(cudaMemcpyAsync(h, ctx->d_status + 2 * instance, sizeof h, cudaMemcpyDeviceToHost,
                           ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    counters[0] = (int64_t)h[0];
    counters[1] = (int64_t)h[1];
    counters[2] = ctx->steps;
    return LBM_OK;
}

int lbm_status(lbm_ctx* ctx, int64_t* counters) {
    if (!ctx || !counters) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    std::vector<unsigned long long> h(2 * (size_t)ctx->count);
    LBM_CK(cudaMemcpyAsync(h.data(), ctx->d_status, sizeof(unsigned long long) * h.size(),
                           cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    counters[0] = counters[1] = 0;
    for (int i = 0; i < ctx->count; ++i) {
        counters[0] += (int64_t)h[2 * i];
        counters[1] += (int64_t)h[2 * i + 1];
    }
    counters[2] = ctx->steps;
    unsigned int err = 0;
    LBM_CK(cudaMemcpyAsync(&err, ctx->d_error, sizeof err, cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return err ? LBM_ERR_TIMEOUT : LBM_OK;
}

int lbm_moments(lbm_ctx* ctx, double* rho, double* ux, double* uy) {
    if (!ctx || !rho) return LBM_ERR_ARG;
    double *hr, *hx, *hy;
    if (device_view(rho, &hr) && device_view(ux, &hx) && device_view(uy, &hy)) {
        // page-locked arrays: the moments kernel writes them in place
        int rc = lbm_moments_device(ctx, hr, hx, hy);
        if (rc != LBM_OK) return rc;
    } else {
        const size_t n = (size_t)ctx->layout.total_nodes;
        double* r = ctx->d_stage;
        double* x = ctx->d_stage + n;
        double* y = ctx->d_stage + 2 * n;
        int rc = lbm_moments_device(ctx, r, x, y);
        if (rc != LBM_OK) return rc;
        LBM_CK(cudaMemcpyAsync(rho, r, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
        if (ux)
            LBM_CK(cudaMemcpyAsync(ux, x, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
        if (uy && ctx->Q == 9)
            LBM_CK(cudaMemcpyAsync(uy, y, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    }
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    int rc;
    int64_t c[3];
    rc = lbm_status(ctx, c);
    if (rc != LBM_OK) return rc;
    return c[1] ? LBM_ERR_UNSTABLE : LBM_OK;
}

int lbm_get_populations(lbm_ctx* ctx, double* f) {
    if (!ctx || !f) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    const size_t n = (size_t)ctx->layout.total_nodes * ctx->Q;
    AuxArgs a = aux_args(ctx);
    LBM_CK(run_aux(AuxOp::GatherF, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr,
                   ctx->d_stage, nullptr, nullptr));
    LBM_CK(cudaMemcpyAsync(f, ctx->d_stage, n * sizeof(double), cudaMemcpyDeviceToHost,
                           ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return LBM_OK;
}

int lbm_set_populations(lbm_ctx* ctx, const double* f) {
    if (!ctx || !f) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    const size_t n = (size_t)ctx->layout.total_nodes * ctx->Q;
    LBM_CK(cudaMemcpyAsync(ctx->d_stage, f, n * sizeof(double), cudaMemcpyHostToDevice,
                           ctx->stream));
    AuxArgs a = aux_args(ctx);
    LBM_CK(run_aux(AuxOp::SetF, a, nullptr, ctx->buf[ctx->cur], ctx->d_stage, nullptr, nullptr,
                   nullptr, nullptr, nullptr));
    LBM_CK(clear_tile_counters(ctx));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    ctx->post = false;
    ctx->initialized = true;
    ctx->inst_init.assign(ctx->count, 1);
    return LBM_OK;
}

int lbm_conservation(lbm_ctx* ctx, double* out) {
    if (!ctx || !out) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    AuxArgs a = aux_args(ctx);
    LBM_CK(run_aux(AuxOp::Conservation, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr,
                   ctx->d_stage, ctx->d_partials, nullptr));
    LBM_CK(cudaMemcpyAsync(out, ctx->d_stage, sizeof(double) * 3 * ctx->count,
                           cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return LBM_OK;
}

int lbm_conservation_device(lbm_ctx* ctx, double* out) {
    if (!ctx || !out) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    AuxArgs a = aux_args(ctx);
    LBM_CK(run_aux(AuxOp::Conservation, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr,
                   out, ctx->d_partials, nullptr));
    return LBM_OK;
}

int lbm_init_batch(lbm_ctx* ctx, int32_t instance, const double* rho, const double* ux,
                   const double* uy) {
    if (!ctx || !rho || instance < 0 || instance >= ctx->count) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (ctx->post) return LBM_ERR_STATE;  // mid-run: the stored field is post-collision
    const InstDesc& in = ctx->layout.inst[instance];
    const size_t n = (size_t)in.nx * in.ny;
    double* r = ctx->d_stage;
    double* x = ux ? ctx->d_stage + n : nullptr;
    double* y = (uy && ctx->Q == 9) ? ctx->d_stage + 2 * n : nullptr;
    LBM_CK(cudaMemcpyAsync(r, rho, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    if (x) LBM_CK(cudaMemcpyAsync(x, ux, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    if (y) LBM_CK(cudaMemcpyAsync(y, uy, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    AuxArgs a = aux_args_instance(ctx, instance);
    LBM_CK(run_aux(AuxOp::Init, a, nullptr, ctx->buf[ctx->cur], r, x, y, nullptr, nullptr,
                   nullptr));
    LBM_CK(cudaMemsetAsync(ctx->d_status + 2 * instance, 0, 2 * sizeof(unsigned long long),
                           ctx->stream));
    LBM_CK(clear_tile_counters(ctx));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    if (ctx->inst_init.size() != (size_t)ctx->count) ctx->inst_init.assign(ctx->count, 0);
    ctx->inst_init[instance] = 1;
    if (!ctx->initialized &&
        std::all_of(ctx->inst_init.begin(), ctx->inst_init.end(), [](uint8_t v) { return v; })) {
        LBM_CK(cudaMemsetAsync(ctx->d_error, 0, ERROR_WORDS * sizeof(unsigned int), ctx->stream));
        LBM_CK(cudaStreamSynchronize(ctx->stream));
        ctx->initialized = true;
        ctx->steps = 0;
    }
    return LBM_OK;
}

int lbm_moments_batch_device(lbm_ctx* ctx, int32_t instance, double* rho, double* ux, double* uy) {
    if (!ctx || !rho || instance < 0 || instance >= ctx->count) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    AuxArgs a = aux_args_instance(ctx, instance);
    LBM_CK(run_aux(AuxOp::Moments, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr, rho,
                   ux, ctx->Q == 9 ? uy : nullptr));
    return LBM_OK;
}

int lbm_moments_batch(lbm_ctx* ctx, int32_t instance, double* rho, double* ux, double* uy) {
    if (!ctx || !rho || instance < 0 || instance >= ctx->count) return LBM_ERR_ARG;
    const InstDesc& in = ctx->layout.inst[instance];
    const size_t n = (size_t)in.nx * in.ny;
    double* r = ctx->d_stage;
    double* x = ctx->d_stage + n;
    double* y = ctx->d_stage + 2 * n;
    int rc = lbm_moments_batch_device(ctx, instance, r, x, y);
    if (rc != LBM_OK) return rc;
    LBM_CK(cudaMemcpyAsync(rho, r, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    if (ux) LBM_CK(cudaMemcpyAsync(ux, x, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    if (uy && ctx->Q == 9)
        LBM_CK(cudaMemcpyAsync(uy, y, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return instance_status(ctx, instance);
}

int lbm_stream_function_batch(lbm_ctx* ctx, int32_t instance, double* psi) {
    if (!ctx || !psi || instance < 0 || instance >= ctx->count) return LBM_ERR_ARG;
    if (ctx->Q != 9) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    const InstDesc& in = ctx->layout.inst[instance];
    const size_t n = (size_t)in.nx * in.ny;
    AuxArgs a = aux_args_instance(ctx, instance);
    LBM_CK(run_aux(AuxOp::StreamFunction, a, ctx->buf[ctx->cur], nullptr, nullptr, nullptr, nullptr,
                   ctx->d_stage, nullptr, nullptr));
    LBM_CK(cudaMemcpyAsync(psi, ctx->d_stage, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return instance_status(ctx, instance);
}

int lbm_state_bytes(lbm_ctx* ctx, uint64_t* bytes) {
    if (!ctx || !bytes) return LBM_ERR_ARG;
    *bytes = state_bytes(ctx);
    return LBM_OK;
}

int lbm_save_state(lbm_ctx* ctx, void* host_buf) {
    if (!ctx || !host_buf) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    if (!ctx->initialized) return LBM_ERR_STATE;
    StateHeader h;
    std::memset(&h, 0, sizeof h);
    std::memcpy(h.magic, STATE_MAGIC, sizeof h.magic);
    h.version = 1;
    h.lattice = ctx->lattice;
    h.storage = ctx->storage;
    h.count = ctx->count;
    h.post = ctx->post ? 1 : 0;
    h.steps = ctx->steps;
    h.layout_hash = layout_hash(ctx);
    h.status_bytes = sizeof(unsigned long long) * 2 * (uint64_t)ctx->count;
    h.buf_bytes = ctx->cv.buf_bytes;
    char* out = static_cast<char*>(host_buf);
    std::memcpy(out, &h, sizeof h);
    // Nothing reads the columns [nx, pitch), but the TMA kernel's stores,
    // clipped at 16 bytes, leave values there where the region kernel does
    // not, and the saved state is to be the same whichever took the steps.
    if (ctx->plan.shape.block() && std::any_of(ctx->layout.inst.begin(), ctx->layout.inst.end(),
                                               [](const InstDesc& in) { return in.pitch != in.nx; })) {
        AuxArgs a = aux_args(ctx);
        LBM_CK(run_aux(AuxOp::ClearPadding, a, nullptr, ctx->buf[ctx->cur], nullptr, nullptr, nullptr,
                       nullptr, nullptr, nullptr));
    }
    LBM_CK(cudaMemcpyAsync(out + sizeof h, ctx->d_status, h.status_bytes, cudaMemcpyDeviceToHost,
                           ctx->stream));
    LBM_CK(cudaMemcpyAsync(out + sizeof h + h.status_bytes, ctx->buf[ctx->cur], h.buf_bytes,
                           cudaMemcpyDeviceToHost, ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    return LBM_OK;
}

int lbm_load_state(lbm_ctx* ctx, const void* host_buf) {
    if (!ctx || !host_buf) return LBM_ERR_ARG;
    if (ctx->failed) return LBM_ERR_CUDA;
    StateHeader h;
    std::memcpy(&h, host_buf, sizeof h);
    if (std::memcmp(h.magic, STATE_MAGIC, sizeof h.magic) != 0 || h.version != 1 ||
        h.lattice != ctx->lattice || h.storage != ctx->storage || h.count != ctx->count ||
        h.layout_hash != layout_hash(ctx) || h.buf_bytes != ctx->cv.buf_bytes ||
        h.status_bytes != sizeof(unsigned long long) * 2 * (uint64_t)ctx->count)
        return LBM_ERR_ARG;
    const char* in = static_cast<const char*>(host_buf);
    LBM_CK(cudaMemcpyAsync(ctx->d_status, in + sizeof h, h.status_bytes, cudaMemcpyHostToDevice,
                           ctx->stream));
    LBM_CK(cudaMemcpyAsync(ctx->buf[0], in + sizeof h + h.status_bytes, h.buf_bytes,
                           cudaMemcpyHostToDevice, ctx->stream));
    LBM_CK(cudaMemsetAsync(ctx->d_error, 0, ERROR_WORDS * sizeof(unsigned int), ctx->stream));
    LBM_CK(cudaStreamSynchronize(ctx->stream));
    ctx->cur = 0;
    ctx->post = h.post != 0;
    ctx->steps = h.steps;
    ctx->initialized = true;
    ctx->inst_init.assign(ctx->count, 1);
    return LBM_OK;
}

int lbm_launch_shape(lbm_ctx* ctx, int32_t* out) {
    if (!ctx || !out) return LBM_ERR_ARG;
    out[0] = ctx->plan.shape.V;
    out[1] = ctx->plan.shape.tw;
    out[2] = ctx->plan.shape.th;
    out[3] = ctx->plan.grid;
    out[4] = ctx->plan.shape.kind;
    return LBM_OK;
}

const char* lbm_status_string(int code) {
    switch (code) {
        case LBM_OK: return "ok";
        case LBM_ERR_ARG: return "invalid argument";
        case LBM_ERR_ALLOC: return "device memory allocation failed";
        case LBM_ERR_CUDA: return "CUDA runtime error";
        case LBM_ERR_UNSTABLE: return "unstable: negative or non-finite population";
        case LBM_ERR_STATE: return "call out of order (context not initialised)";
        case LBM_ERR_NODEV: return "no sm_103 CUDA device";
        case LBM_ERR_TIMEOUT: return "a bounded device-side wait ran out (data copy never completed)";
    }
    return "unknown status code";
}

}  // extern "C"
