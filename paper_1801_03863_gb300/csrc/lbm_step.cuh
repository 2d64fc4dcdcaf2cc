// lbm_step.cuh -- fused pull-stream + collide + boundary kernels that work in
// registers: the register-chunk kernel (below), the FP64 kernel with one node
// per thread and the D1Q3 kernel that takes several steps per launch.
//
// A launch of the register-chunk kernel performs one time step of Eq. (2) for
// every instance of a context.  Populations are stored SoA (one plane per velocity, rows of
// `pitch` elements, pitch a multiple of 8) as deviations from W_a rho0, and
// the stored state is the post-collision field of the previous step, so the
// step is a pull:
//     f~_a(x) = f^post_a(x - v_a)  (with the boundary rules),
//     f^post(x) = collide(f~(x))   (or the wall / lid rule),
// reading each plane once and writing each plane once, both aligned.
//
// Work decomposition: a thread owns a chunk of V consecutive nodes of one
// row; a CTA owns a tile of tw x th chunks of one instance (tile table
// built on the host, walked with a grid-stride loop: one persistent launch
// covers an ensemble of uneven instances).  Each plane's chunk is one
// 8/16/32-byte vector load from row y - v_y; the x-shift of +-1 is served by
// a warp shuffle of the neighbouring lane's edge element, or by one scalar
// load (with the boundary rule) at tile, warp and row edges.
#pragma once
#include "lbm_collide.cuh"

namespace lbm {

template <typename S> __device__ __forceinline__ S bits_to(uint32_t lo, uint32_t hi);
template <> __device__ __forceinline__ double bits_to<double>(uint32_t lo, uint32_t hi) {
    return __hiloint2double((int)hi, (int)lo);
}
template <> __device__ __forceinline__ float bits_to<float>(uint32_t lo, uint32_t) {
    return __uint_as_float(lo);
}
template <> __device__ __forceinline__ __half bits_to<__half>(uint32_t lo, uint32_t) {
    return __ushort_as_half((unsigned short)(lo & 0xffffu));
}
template <> __device__ __forceinline__ __nv_bfloat16 bits_to<__nv_bfloat16>(uint32_t lo, uint32_t) {
    return __ushort_as_bfloat16((unsigned short)(lo & 0xffffu));
}

template <typename S> __device__ __forceinline__ uint32_t lo_bits(S v);
template <typename S> __device__ __forceinline__ uint32_t hi_bits(S v) { return 0u; }
template <> __device__ __forceinline__ uint32_t lo_bits<double>(double v) {
    return (uint32_t)__double2loint(v);
}
template <> __device__ __forceinline__ uint32_t hi_bits<double>(double v) {
    return (uint32_t)__double2hiint(v);
}
template <> __device__ __forceinline__ uint32_t lo_bits<float>(float v) { return __float_as_uint(v); }
template <> __device__ __forceinline__ uint32_t lo_bits<__half>(__half v) {
    return (uint32_t)__half_as_ushort(v);
}
template <> __device__ __forceinline__ uint32_t lo_bits<__nv_bfloat16>(__nv_bfloat16 v) {
    return (uint32_t)__bfloat16_as_ushort(v);
}

// V consecutive elements of type S held as 32-bit words.
template <typename S, int V> struct Chunk {
    static constexpr int BYTES = V * (int)sizeof(S);
    static constexpr int WORDS = BYTES / 4;
    static_assert(BYTES == 8 || BYTES == 16 || BYTES == 32, "chunk must be 8, 16 or 32 bytes");
    uint32_t w[WORDS];

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < WORDS; ++k) w[k] = 0u;
    }
    __device__ __forceinline__ void load(const S* p) {
        if constexpr (BYTES == 8) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
            w[0] = v.x; w[1] = v.y;
        } else {
#pragma unroll
            for (int k = 0; k < BYTES / 16; ++k) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(p) + k);
                w[4 * k + 0] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
            }
        }
    }
    __device__ __forceinline__ void store(S* p) const {
        if constexpr (BYTES == 8) {
            *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
        } else {
#pragma unroll
            for (int k = 0; k < BYTES / 16; ++k)
                reinterpret_cast<uint4*>(p)[k] =
                    make_uint4(w[4 * k + 0], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
        }
    }
    // i must be a compile-time constant after unrolling
    __device__ __forceinline__ S get(int i) const {
        if constexpr (sizeof(S) == 2) {
            const uint32_t x = w[i >> 1];
            return bits_to<S>((i & 1) ? (x >> 16) : (x & 0xffffu), 0u);
        } else if constexpr (sizeof(S) == 4) {
            return bits_to<S>(w[i], 0u);
        } else {
            return bits_to<S>(w[2 * i], w[2 * i + 1]);
        }
    }
    __device__ __forceinline__ void set(int i, S v) {
        if constexpr (sizeof(S) == 2) {
            const uint32_t b = lo_bits<S>(v);
            w[i >> 1] = (i & 1) ? ((w[i >> 1] & 0xffffu) | (b << 16)) : ((w[i >> 1] & 0xffff0000u) | b);
        } else if constexpr (sizeof(S) == 4) {
            w[i] = lo_bits<S>(v);
        } else {
            w[2 * i] = lo_bits<S>(v);
            w[2 * i + 1] = hi_bits<S>(v);
        }
    }
};

// Warp shuffles of one element.
template <typename S> __device__ __forceinline__ S shfl_up1(S v) {
    const uint32_t lo = __shfl_up_sync(0xffffffffu, lo_bits<S>(v), 1);
    uint32_t hi = 0u;
    if constexpr (sizeof(S) == 8) hi = __shfl_up_sync(0xffffffffu, hi_bits<S>(v), 1);
    return bits_to<S>(lo, hi);
}
template <typename S> __device__ __forceinline__ S shfl_down1(S v) {
    const uint32_t lo = __shfl_down_sync(0xffffffffu, lo_bits<S>(v), 1);
    uint32_t hi = 0u;
    if constexpr (sizeof(S) == 8) hi = __shfl_down_sync(0xffffffffu, hi_bits<S>(v), 1);
    return bits_to<S>(lo, hi);
}

template <typename S> __device__ __forceinline__ S ldg_elem(const S* p) {
    if constexpr (sizeof(S) == 2) {
        return bits_to<S>((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p)), 0u);
    } else {
        return __ldg(p);
    }
}
template <typename S> __device__ __forceinline__ S zero_elem() { return bits_to<S>(0u, 0u); }

// Element xs of a source row, with the x boundary rule for xs = -1 or nx.
// row_ok = false: the row lies outside a cavity (fill: deviation 0).
template <typename S>
__device__ __forceinline__ S edge_elem(const S* rowp, bool row_ok, int xs, int nx, int bc) {
    if (!row_ok) return zero_elem<S>();
    if (xs < 0 || xs >= nx) {
        if (bc == BC_PERIODIC) xs = (xs < 0) ? xs + nx : xs - nx;
        else if (bc == BC_ZERO_GRADIENT) xs = (xs < 0) ? 0 : nx - 1;
        else return zero_elem<S>();  // cavity: outside the lattice
    }
    return ldg_elem<S>(rowp + xs);
}

template <typename T, typename S> __device__ __forceinline__ T to_compute(S v) {
    if constexpr (std::is_same<T, double>::value) return Store<S>::to_f64(v);
    else return Store<S>::to_f32(v);
}

template <class Lat, typename S, typename T, int V, int COLL>
__global__ void __launch_bounds__(256) step_kernel(const StepArgs args) {
    constexpr int Q = Lat::Q;
    const S* __restrict__ src = static_cast<const S*>(args.src);
    S* __restrict__ dst = static_cast<S*>(args.dst);
    const int tid = threadIdx.x;
    const int cx = tid & (args.tw - 1);
    const int cy = tid >> args.tw_log2;
    const int lane = tid & 31;
    const T rho0 = (T)args.rho0;
    wait_previous_grid();
    allow_next_grid();

    for (int t = blockIdx.x; t < args.ntiles; t += gridDim.x) {
        const TileDesc tile = args.tiles[t];
        const InstDesc& in = args.inst[tile.inst];
        const int nx = in.nx, ny = in.ny, bc = in.bc;
        const int64_t pitch = in.pitch, plane = in.plane;
        const int x0 = (tile.cx0 + cx) * V;
        const int y = tile.y0 + cy;
        const bool active = (x0 < nx) && (y < ny);
        const S* base = src + in.off;

        Chunk<S, V> raw[Q];
        S left[Q], right[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const int vxa = Lat::vx(a), vya = Lat::vy(a);
            int sy = y - vya;
            bool row_ok = true;
            if (vya != 0) {
                if (bc == BC_CAVITY) row_ok = (sy >= 0) && (sy < ny);
                else sy = (sy < 0) ? sy + ny : ((sy >= ny) ? sy - ny : sy);
            }
            const S* rowp = base + a * plane + (int64_t)(row_ok ? sy : 0) * pitch;
            if (active && row_ok) raw[a].load(rowp + x0);
            else raw[a].zero();
            if (vxa == 1) {
                // node x0 pulls from x0 - 1: last element of the left neighbour chunk
                S nb = shfl_up1<S>(raw[a].get(V - 1));
                const bool use_shfl = (x0 > 0) && (cx > 0) && (lane > 0);
                if (active && !use_shfl) nb = edge_elem<S>(rowp, row_ok, x0 - 1, nx, bc);
                left[a] = nb;
            } else if (vxa == -1) {
                // node x0+V-1 pulls from x0 + V: first element of the right chunk
                S nb = shfl_down1<S>(raw[a].get(0));
                const bool use_shfl = (x0 + V < nx) && (cx < args.tw - 1) && (lane < 31);
                if (active && !use_shfl) nb = edge_elem<S>(rowp, row_ok, min(x0 + V, nx), nx, bc);
                right[a] = nb;
            } else {
                left[a] = right[a] = zero_elem<S>();
            }
        }
        // Inactive threads fall through to the next tile without returning
        // early, so every lane reaches the shuffles of the next iteration.
        if (active) {
        // Ragged last chunk of a row: node nx-1 sits before the chunk's end and
        // must see the boundary value fetched into right[] instead of padding.
        const bool ragged = (x0 + V > nx);
        const int jr = nx - 1 - x0;  // last valid position in a ragged chunk
        if (ragged) {
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                if (Lat::vx(a) == -1) {
#pragma unroll
                    for (int k = 1; k < V; ++k) {
                        // unconditional set of a selected value keeps raw[] in registers
                        const S v = raw[a].get(k);
                        raw[a].set(k, (k == jr + 1) ? right[a] : v);
                    }
                }
            }
        }

        // Collide nodes one at a time (FP64) or two at a time (FP32, packed
        // FP32x2 arithmetic).
        using CT = typename std::conditional<std::is_same<T, float>::value, F2, T>::type;
        using N = Num<CT>;
        constexpr int P = N::LANES;
        using LT = typename LaneOf<CT>::type;
        const Rates<CT> rates{CT((LT)in.omega), CT((LT)in.omega2), CT((LT)in.s_e), CT((LT)in.s_eps)};
        const CT rho0v = CT((LT)rho0);
        const bool cavity_edge =
            (bc == BC_CAVITY) && (y == 0 || y == ny - 1 || x0 == 0 || x0 + V >= nx);
        Chunk<S, V> out[Q];
        uint32_t n_skip = 0, n_unst = 0;
#pragma unroll
        for (int i = 0; i < V; i += P) {
            CT d[Q], o[Q];
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const int vxa = Lat::vx(a);
#pragma unroll
                for (int l = 0; l < P; ++l) {
                    const int j = i + l;
                    S s;
                    if (vxa == 0) s = raw[a].get(j);
                    else if (vxa == 1) s = (j == 0) ? left[a] : raw[a].get(j - 1);
                    else s = (j == V - 1) ? right[a] : raw[a].get(j + 1);
                    if constexpr (std::is_same<CT, double>::value) d[a] = to_compute<T, S>(s);
                    else N::set_lane(d[a], l, to_compute<float, S>(s));
                }
            }
            uint32_t st = Collide<Lat, COLL, CT, (int)sizeof(S)>::run(d, rho0v, rates, o);
            if constexpr (Q == 3) st = bgk_suspect(st) ? bgk_status(o[0], o[1], o[2], rho0v) : 0u;
            if (cavity_edge) {
#pragma unroll
                for (int l = 0; l < P; ++l) {
                    const int x = x0 + i + l;
                    const bool wall = (x == 0) || (x == nx - 1) || (y == 0);
                    const bool lid = !wall && (y == ny - 1);
                    if (wall) {
                        // full-way bounce-back: reverse every population (W_opp = W_a)
#pragma unroll
                        for (int a = 0; a < Q; ++a)
                            N::set_lane(o[a], l, N::lane(d[Lat::opp(a)], l));
                        st &= ~(3u << (2 * l));
                    } else if (lid) {
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
                            if constexpr (std::is_same<T, double>::value)
                                N::set_lane(o[a], l, in.lid_dev[a]);
                            else
                                N::set_lane(o[a], l, in.lid_dev_f[a]);
                        }
                        st &= ~(3u << (2 * l));
                    }
                }
            }
#pragma unroll
            for (int l = 0; l < P; ++l) {
                if (x0 + i + l < nx) {
                    n_skip += (st >> (2 * l)) & ST_NEWTON_SKIPPED;
                    n_unst += ((st >> (2 * l)) & ST_UNSTABLE) >> 1;
                }
            }
#pragma unroll
            for (int a = 0; a < Q; ++a)
#pragma unroll
                for (int l = 0; l < P; ++l) out[a].set(i + l, Store<S>::from(N::lane(o[a], l)));
        }
        if (ragged) {
            // keep the row padding at deviation 0
#pragma unroll
            for (int a = 0; a < Q; ++a)
#pragma unroll
                for (int k = 1; k < V; ++k) {
                    const S v = out[a].get(k);
                    out[a].set(k, (k > jr) ? zero_elem<S>() : v);
                }
        }
        S* obase = dst + in.off + (int64_t)y * pitch + x0;
#pragma unroll
        for (int a = 0; a < Q; ++a) out[a].store(obase + a * plane);

        if (n_skip | n_unst) {
            atomicAdd(args.status + 2 * tile.inst + 0, (unsigned long long)n_skip);
            atomicAdd(args.status + 2 * tile.inst + 1, (unsigned long long)n_unst);
        }
        }  // active
    }
}

// ---------------------------------------------------------------------------
// The FP64 D2Q9 step with one node per thread and one warp per CTA.
//
// FP64 arithmetic bounds this step on GB300 (lbm_f64.cuh): a warp
// instruction holds its scheduler's FP64 unit for 64 cycles, whatever the
// number of active lanes, so what counts is that every scheduler gets the
// same number of full warps, down to the smallest lattices.  Nodes are
// numbered linearly, without tile padding; in a cavity only the fluid nodes
// are, and every CTA takes an equal share of the outer ring (walls and lid,
// which do not collide) along.  A CTA is one warp; an entry of the tile table
// covers up to args.tw nodes, [cx0, y0) of one instance, and args.tw / 32 CTAs.
// (42.6 us a step on 257 x 257 with one warp per CTA against 52.8 with two or
// four, ring nodes in colliding warps.)
//
// The hardware deals CTAs to SMs unevenly while some still have room, so the
// launch claims shared memory that leaves each SM room for its equal share
// and no more (257 x 257: 37.2 -> 34.2 us a step, then; at most 128 registers, so
// that 16 warps fit an SM: with more, 38.9).
//
// Measured, MinxEnt4, per step, against the register-chunk kernel with log1p
// and IEEE divisions: 120 lattices of 17 x 17: 122.4 -> 18.8 us; 257 x 257:
// 110 -> 34.5 us; 800 x 4: 52.6 -> 12.2 us; 2048 x 2048: 3680 -> 1920 us (252
// FP64 instructions per node against 485; 0.87 of the FP64 issue rate).  The
// smallest lattices are bound by one warp's instructions (252 x 64 cycles =
// 7.8 us) and the launch.
//
// inplace: the first step after a state was loaded collides f(x, t_n) itself,
// without streaming.
// ---------------------------------------------------------------------------
// Populations a cavity's or another lattice's node (x, y) pulls (or holds, inplace).
__device__ __forceinline__ void flat_pull(const double* base, const InstDesc& in, uint32_t x, uint32_t y,
                                          bool inplace, double (&d)[9]) {
    const int64_t pitch = in.pitch, plane = in.plane;
    if (inplace) {
        const double* p = base + (int64_t)y * pitch + x;
#pragma unroll
        for (int a = 0; a < 9; ++a) d[a] = p[a * plane];
        return;
    }
    // columns x - 1, x + 1 and rows y - 1, y + 1 under the boundary rule;
    // a cavity node pulls deviation 0 from outside the lattice
    const uint32_t nx = (uint32_t)in.nx, ny = (uint32_t)in.ny;
    const bool cav = in.bc == BC_CAVITY, per = in.bc == BC_PERIODIC;
    const bool l = x > 0u, r = x + 1u < nx, b = y > 0u, t = y + 1u < ny;
    const uint32_t xs[3] = {l ? x - 1u : (per ? nx - 1u : 0u), x, r ? x + 1u : (per ? 0u : nx - 1u)};
    const uint32_t ys[3] = {b ? y - 1u : ny - 1u, y, t ? y + 1u : 0u};
    const bool xok[3] = {l || !cav, true, r || !cav}, yok[3] = {b || !cav, true, t || !cav};
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int i = 1 - D2Q9::vx(a), j = 1 - D2Q9::vy(a);
        d[a] = (xok[i] && yok[j]) ? __ldg(base + a * plane + (int64_t)ys[j] * pitch + xs[i]) : 0.0;
    }
}

// Node j of a cavity's ring: bottom row, top row, then the two sides, row by row.
__device__ __forceinline__ void ring_node(uint32_t j, uint32_t nx, uint32_t ny, uint32_t& x, uint32_t& y) {
    if (j < 2u * nx) {
        y = j < nx ? 0u : ny - 1u;
        x = j < nx ? j : j - nx;
    } else {
        const uint32_t s = j - 2u * nx;
        y = 1u + (s >> 1);
        x = (s & 1u) ? nx - 1u : 0u;
    }
}

template <int COLL>
__global__ void __launch_bounds__(32, 16) step_flat_kernel(const StepArgs args) {
    constexpr int Q = 9;
    const double* src = static_cast<const double*>(args.src);
    double* __restrict__ dst = static_cast<double*>(args.dst);
    const uint32_t per = (uint32_t)args.tw / 32u, sub = blockIdx.x & (per - 1u);  // CTAs per entry: 2^n
    const uint32_t lane = threadIdx.x;
    const TileDesc tile = args.tiles[blockIdx.x / per];
    const InstDesc& in = args.inst[tile.inst];
    const uint32_t nx = (uint32_t)in.nx, ny = (uint32_t)in.ny;
    const bool cav = in.bc == BC_CAVITY;
    const uint32_t k = (uint32_t)tile.cx0 + sub * 32u + lane;
    const bool active = k < (uint32_t)tile.y0;
    const uint32_t mx = cav ? nx - 2u : nx;
    const uint32_t row = k / mx;
    const uint32_t x = k - row * mx + (cav ? 1u : 0u), y = row + (cav ? 1u : 0u);
    // this CTA's share of the cavity's ring
    uint32_t ring = 0u, ring_end = 0u;
    if (cav) {
        const uint32_t fluid = mx * (ny - 2u), all = 2u * (nx + ny) - 4u;
        const uint64_t ctas = (uint64_t)((fluid + (uint32_t)args.tw - 1u) / (uint32_t)args.tw) * per;
        const uint64_t me = (uint64_t)((uint32_t)tile.cx0 / (uint32_t)args.tw) * per + sub;
        ring = (uint32_t)(me * all / ctas) + lane;
        ring_end = (uint32_t)((me + 1u) * all / ctas);
    }
    wait_previous_grid();
    allow_next_grid();

    const double* base = src + in.off;
    double* obase = dst + in.off;
    const bool inplace = args.inplace != 0;
    double d[Q], rd[Q];
    if (active) flat_pull(base, in, x, y, inplace, d);
    // ring node: bounce-back of the pulled populations, or the lid's equilibrium;
    // its loads are issued before the collision and stored after it
    uint32_t rx = 0u, ry = 0u;
    auto ring_load = [&]() {
        ring_node(ring, nx, ny, rx, ry);
        if (ry == ny - 1u && rx > 0u && rx < nx - 1u) {
#pragma unroll
            for (int a = 0; a < Q; ++a) rd[D2Q9::opp(a)] = in.lid_dev[a];
        } else {
            flat_pull(base, in, rx, ry, inplace, rd);
        }
    };
    auto ring_store = [&]() {
        double* p = obase + (int64_t)ry * in.pitch + rx;
#pragma unroll
        for (int a = 0; a < Q; ++a) p[a * in.plane] = rd[D2Q9::opp(a)];
    };
    const bool first = ring < ring_end;
    if (first) ring_load();
    if (active) {
        double o[Q];
        const Rates<double> rates{in.omega, in.omega2, in.s_e, in.s_eps};
        const uint32_t st = Collide<D2Q9, COLL, double, 8>::run(d, args.rho0, rates, o);
        double* op = obase + (int64_t)y * in.pitch + x;
#pragma unroll
        for (int a = 0; a < Q; ++a) op[a * in.plane] = o[a];
        if (st & ST_NEWTON_SKIPPED) atomicAdd(args.status + 2 * tile.inst + 0, 1ull);
        if (st & ST_UNSTABLE) atomicAdd(args.status + 2 * tile.inst + 1, 1ull);
    }
    if (first) ring_store();
    for (ring += 32u; ring < ring_end; ring += 32u) {  // thin cavities: more ring than fluid
        ring_load();
        ring_store();
    }
}

inline const void* pick_step_flat_kernel(int collision) {
    switch (collision) {
        case COLL_MINXENT4: return (const void*)&step_flat_kernel<COLL_MINXENT4>;
        case COLL_SRT: return (const void*)&step_flat_kernel<COLL_SRT>;
        case COLL_MINXENT2: return (const void*)&step_flat_kernel<COLL_MINXENT2>;
        case COLL_MRT:
        case COLL_TRT: return (const void*)&step_flat_kernel<COLL_MRT>;
    }
    return nullptr;
}

// ---------------------------------------------------------------------------
// D1Q3: several time steps per launch, one warp per segment of a tube.
//
// A warp holds 32 V consecutive nodes in registers (V per lane) and advances
// them args.steps <= args.halo steps: streaming is a register shift within a
// lane and one shuffle per moving plane between lanes, so a step needs no
// memory and no barrier.  Each step the outermost node on either side of the
// segment loses its neighbour, so the outer `halo` nodes are carried along
// only to feed the inner ones and the segment's 32 V - 2 halo inner nodes
// are written back.  One step per launch moved 24 bytes a node and step (FP32)
// and was bound by HBM on ensembles and by the launch on single tubes; with a
// halo of 8 steps the traffic falls to 3 bytes and the arithmetic bounds it.
//
// Node i of a lane sits in half i / NP of pair i % NP (NP = V / 2 pairs), so
// that shifting by one node is taking the neighbouring pair, and only the
// end pairs are put together from two registers.
//
// Tube ends: a periodic segment loads its nodes modulo nx; at a zero-gradient
// end the entering population is the end node's own (the nodes beyond are
// never read by the lattice).  Each node's arithmetic is that of one step per
// launch, rounding to the storage type included.
// ---------------------------------------------------------------------------
template <typename CT, typename S> __device__ __forceinline__ CT round_to_storage(CT v) {
    if constexpr (std::is_same<S, double>::value || std::is_same<S, float>::value) {
        return v;
    } else {
        using N = Num<CT>;
#pragma unroll
        for (int l = 0; l < N::LANES; ++l)
            N::set_lane(v, l, Store<S>::to_f32(Store<S>::from(N::lane(v, l))));
        return v;
    }
}

template <typename S, typename T, int V>
__global__ void __launch_bounds__(256) step_tube_kernel(const StepArgs args) {
    using CT = typename std::conditional<std::is_same<T, float>::value, F2, T>::type;
    using N = Num<CT>;
    using LT = typename LaneOf<CT>::type;
    constexpr int P = N::LANES, NP = V / P;
    static_assert(V % P == 0, "whole pairs per lane");
    const int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = (int)(threadIdx.x & 31u);
    const bool some = t < args.ntiles;  // the same for the whole warp
    const TileDesc tile = args.tiles[some ? t : 0];
    const InstDesc& in = args.inst[tile.inst];
    const int nx = in.nx, halo = args.halo;
    const bool periodic = in.bc == BC_PERIODIC;
    const int x = tile.cx0 - halo + lane * V;  // first node of this lane
    const Rates<CT> rates{CT((LT)in.omega), CT((LT)in.omega2), CT((LT)in.s_e), CT((LT)in.s_eps)};
    const CT rho0 = CT((LT)args.rho0);
    wait_previous_grid();
    allow_next_grid();
    if (!some) return;

    // populations of node p + l NP: lane l of f[a][p]
    CT f[3][NP];
    const S* src = static_cast<const S*>(args.src) + in.off;
    const bool whole = x >= 0 && x + V <= nx;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Chunk<S, V> c;
        if (whole) {
            c.load(src + a * in.plane + x);
        } else {
            c.zero();
#pragma unroll
            for (int i = 0; i < V; ++i) {
                int xi = x + i;
                if (periodic) {
                    xi %= nx;
                    if (xi < 0) xi += nx;
                }
                if (xi >= 0 && xi < nx) c.set(i, ldg_elem<S>(src + a * in.plane + xi));
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int l = 0; l < P; ++l) N::set_lane(f[a][p], l, to_compute<T, S>(c.get(p + l * NP)));
    }

    const bool mine = lane * V >= halo && lane * V < 32 * V - halo;  // lanes written back
    const bool left_end = !periodic && x == 0;  // x = 0 is the first node of its lane
    // warp-uniform: the segment holds the last node of a zero-gradient tube
    const bool has_right = !periodic && tile.cx0 - halo < nx && tile.cx0 - halo + 32 * V >= nx;
    uint32_t n_unst = 0;
    for (int s = 0; s < args.steps; ++s) {
        CT from_l[NP], from_r[NP];  // plane 1 pulled from x - 1, plane 2 from x + 1
        if (s > 0 || !args.inplace) {
            const LT in_l = __shfl_up_sync(0xffffffffu, N::lane(f[1][NP - 1], P - 1), 1);
            const LT in_r = __shfl_down_sync(0xffffffffu, N::lane(f[2][0], 0), 1);
#pragma unroll
            for (int p = 1; p < NP; ++p) from_l[p] = f[1][p - 1];
#pragma unroll
            for (int p = 0; p < NP - 1; ++p) from_r[p] = f[2][p + 1];
            N::set_lane(from_l[0], 0, left_end ? N::lane(f[1][0], 0) : in_l);
            if constexpr (P == 2) N::set_lane(from_l[0], 1, N::lane(f[1][NP - 1], 0));
            if constexpr (P == 2) N::set_lane(from_r[NP - 1], 0, N::lane(f[2][0], 1));
            N::set_lane(from_r[NP - 1], P - 1, in_r);
            if (has_right) {
#pragma unroll
                for (int p = 0; p < NP; ++p)
#pragma unroll
                    for (int l = 0; l < P; ++l)
                        if (x + p + l * NP == nx - 1) N::set_lane(from_r[p], l, N::lane(f[2][p], l));
            }
        } else {
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                from_l[p] = f[1][p];
                from_r[p] = f[2][p];
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const CT d[3] = {f[0][p], from_l[p], from_r[p]};
            CT o[3];
            const uint32_t bits = Collide<D1Q3, COLL_MINXENT4, CT, (int)sizeof(S)>::run(d, rho0, rates, o);
#pragma unroll
            for (int a = 0; a < 3; ++a) f[a][p] = round_to_storage<CT, S>(o[a]);
            if (bgk_suspect(bits) && mine) {  // rare: a population is negative or not finite
                const uint32_t st = bgk_status(o[0], o[1], o[2], rho0);
#pragma unroll
                for (int l = 0; l < P; ++l)
                    if (x + p + l * NP < nx) n_unst += ((st >> (2 * l)) & ST_UNSTABLE) >> 1;
            }
        }
    }

    if (!mine || x >= nx) return;
    S* dst = static_cast<S*>(args.dst) + in.off + x;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Chunk<S, V> c;
        c.zero();
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int l = 0; l < P; ++l) c.set(p + l * NP, Store<S>::from(N::lane(f[a][p], l)));
        if (whole) {
            c.store(dst + a * in.plane);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (x + i < nx) dst[a * in.plane + i] = c.get(i);
        }
    }
    if (n_unst) atomicAdd(args.status + 2 * tile.inst + 1, (unsigned long long)n_unst);
}

// The register-chunk kernel on D1Q3 (FP32 arithmetic), for single steps: a
// launch of the tube kernel's is mostly a warp's wait for its tile's descriptor and
// nodes, which one step does not make up for (18.0 M nodes, one step: 84 us
// against 73 in FP32, 73 against 50 in FP16; two steps 90 against 146).  FP64
// stays with the tube kernel (1000 tubes: 135 against 300 us).
template <typename S, int V> const void* pick_step_single_tube_kernel() {
    return (const void*)&step_kernel<D1Q3, S, float, V, COLL_MINXENT4>;
}

// The D2Q9 register-chunk kernel for a collision rule with storage S,
// arithmetic T and V nodes per thread.  TRT shares the MRT kernel (its rates
// come from the instance table).
template <typename S, typename T, int V> const void* pick_step_kernel(int collision) {
    switch (collision) {
        case COLL_MINXENT4: return (const void*)&step_kernel<D2Q9, S, T, V, COLL_MINXENT4>;
        case COLL_SRT: return (const void*)&step_kernel<D2Q9, S, T, V, COLL_SRT>;
        case COLL_MINXENT2: return (const void*)&step_kernel<D2Q9, S, T, V, COLL_MINXENT2>;
        case COLL_MRT:
        case COLL_TRT: return (const void*)&step_kernel<D2Q9, S, T, V, COLL_MRT>;
    }
    return nullptr;
}

}  // namespace lbm
