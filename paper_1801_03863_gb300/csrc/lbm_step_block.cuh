// lbm_step_block.cuh -- several D2Q9 steps per launch on lattices that do not
// fill the GPU (FP32 collide arithmetic, FP32 / FP16 / BF16 storage).
//
// A small lattice's step is all latency: launch, loads, one or two units of
// collision per warp, stores.  512 x 512 nodes in FP32 take 8.2 us a step on
// the TMA kernel, where the collisions alone take 2.2 us.  Here a CTA loads a
// region of 64 nodes by up to 96 rows into shared memory, advances it K steps
// there and writes back what is still valid: each step invalidates one more
// node along the region's artificial edges (not along a cavity's own walls),
// so neighbouring regions overlap by 2 K nodes and recompute each other's
// margins.  The redundant collisions run on schedulers that would idle.
//
// A row of the region is one unit of 32 node pairs, one pair per lane, as in
// the TMA kernel; two shared-memory buffers alternate, with one barrier per
// step.  Every node's arithmetic, storage rounding included, is that of the
// other step kernels.
//
// Periodic images are loaded modulo the lattice and evolve like the nodes
// they repeat; nodes outside a cavity stay at deviation 0; at a zero-gradient
// end (x) the entering populations are the end column's own.
#pragma once
#include "lbm_aux.h"
#include "lbm_collide.cuh"
#include "lbm_step.cuh"

namespace lbm {

// TileDesc of this kernel: region origin (cx0, y0) and, packed in pad, the
// part it writes back: columns [x0, x1) and rows [y0, y1) of the region, and
// whether the region ends at the lattice's own top and bottom rows.
struct BlockPart {
    int x0, x1, y0, y1;
    bool whole_height;
};
__host__ __device__ inline int32_t pack_part(int x0, int x1, int y0, int y1, bool whole_height) {
    return x0 | (x1 << 7) | (y0 << 14) | (y1 << 21) | (whole_height ? 1 << 28 : 0);
}
__host__ __device__ inline BlockPart unpack_part(int32_t p) {
    return {p & 127, (p >> 7) & 127, (p >> 14) & 127, (p >> 21) & 127, ((p >> 28) & 1) != 0};
}

template <typename S> struct PairWord {
    using type = typename std::conditional<sizeof(S) == 2, uint32_t, float2>::type;
};

template <typename S> __device__ __forceinline__ float2 pair_floats(typename PairWord<S>::type w) {
    if constexpr (std::is_same<S, __half>::value)
        return __half22float2(*reinterpret_cast<const __half2*>(&w));
    else if constexpr (std::is_same<S, __nv_bfloat16>::value)
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
    else
        return w;
}
template <typename S> __device__ __forceinline__ typename PairWord<S>::type pair_word(float a, float b) {
    typename PairWord<S>::type w;
    if constexpr (std::is_same<S, __half>::value)
        *reinterpret_cast<__half2*>(&w) = __floats2half2_rn(a, b);
    else if constexpr (std::is_same<S, __nv_bfloat16>::value)
        *reinterpret_cast<__nv_bfloat162*>(&w) = __floats2bfloat162_rn(a, b);
    else
        w = make_float2(a, b);
    return w;
}

// ROWS: rows that a buffer has room for (a constant plane stride)
template <typename S, int COLL, int ROWS>
__global__ void __launch_bounds__(32 * BLOCK_WARPS, 1) step_block_kernel(const StepArgs args) {
    constexpr int Q = 9;
    using N = Num<F2>;
    using W = typename PairWord<S>::type;
    extern __shared__ __align__(16) unsigned char block_smem[];
    constexpr int plane = ROWS * 32, buffer = Q * plane;  // words
    W* buf = reinterpret_cast<W*>(block_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const TileDesc tile = args.tiles[blockIdx.x];
    const InstDesc& in = args.inst[tile.inst];
    const BlockPart part = unpack_part(tile.pad);
    const int nx = in.nx, ny = in.ny, bc = in.bc, K = args.steps;
    const bool cav = bc == BC_CAVITY, per = bc == BC_PERIODIC;
    const int rows = part.whole_height ? part.y1 : part.y1 + args.halo;
    const int x = tile.cx0 + 2 * lane;  // this lane's pair of columns
    const F2 rho0 = F2((float)args.rho0);
    const Rates<F2> rates{F2(in.rates_f[0]), F2(in.rates_f[1]), F2(in.rates_f[2]), F2(in.rates_f[3])};
    // columns of the pair as the lattice stores them, < 0: outside
    int xa = x, xb = x + 1;
    if (per) {
        xa %= nx;
        xa = xa < 0 ? xa + nx : xa;
        xb = xa + 1 == nx ? 0 : xa + 1;
    } else {
        xa = xa >= 0 && xa < nx ? xa : -1;
        xb = xb >= 0 && xb < nx ? xb : -1;
    }
    const bool pair_ok = xa >= 0 && xb == xa + 1 && (xa & 1) == 0;  // one aligned word in memory
    wait_previous_grid();
    allow_next_grid();

    const S* src = static_cast<const S*>(args.src) + in.off;
    for (int r = warp; r < rows; r += nwarps) {
        int y = tile.y0 + r;
        bool yok = true;
        if (cav) {
            yok = y >= 0 && y < ny;
        } else {
            y %= ny;
            y = y < 0 ? y + ny : y;
        }
        W w[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const S* row = src + a * in.plane + (int64_t)(yok ? y : 0) * in.pitch;
            if (yok && pair_ok) {
                w[a] = __ldg(reinterpret_cast<const W*>(row + xa));
            } else {
                const float lo = yok && xa >= 0 ? Store<S>::to_f32(ldg_elem<S>(row + xa)) : 0.f;
                const float hi = yok && xb >= 0 ? Store<S>::to_f32(ldg_elem<S>(row + xb)) : 0.f;
                w[a] = pair_word<S>(lo, hi);
            }
        }
#pragma unroll
        for (int a = 0; a < Q; ++a) buf[a * plane + r * 32 + lane] = w[a];
    }
    __syncthreads();

    uint32_t n_skip = 0, n_unst = 0;
    const bool mine_a = 2 * lane >= part.x0 && 2 * lane < part.x1;
    const bool mine_b = 2 * lane + 1 >= part.x0 && 2 * lane + 1 < part.x1;
    // all 64 columns of the region inside the lattice's outer ring
    const bool mid = per || (tile.cx0 >= 1 && tile.cx0 + 63 <= nx - 2);
    const int to_left = lane > 0 ? -1 : 0, to_right = lane < 31 ? 1 : 0;  // (edge columns are not valid)
    for (int s = 0; s < K; ++s) {
        const W* from = buf + (s & 1) * buffer;
        W* to = buf + ((s + 1) & 1) * buffer;
        const bool last = s == K - 1;
        // rows still valid after this step
        const int r0 = part.whole_height ? 0 : s + 1, r1 = rows - r0;
        for (int r = r0 + warp; r < r1; r += nwarps) {
            const int y = tile.y0 + r;
            // rows pulled with v_y = -1, 0, 1 (at a cavity's own first and last
            // row some row of the region: see below)
            const int row_of[3] = {part.whole_height ? min(r + 1, rows - 1) : r + 1, r,
                                   part.whole_height ? max(r - 1, 0) : r - 1};
            const W *own[3], *lft[3], *rgt[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                own[j] = from + row_of[j] * 32 + lane;
                lft[j] = own[j] + to_left;
                rgt[j] = own[j] + to_right;
            }
            F2 d[Q], o[Q];
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const int vx = D2Q9::vx(a), j = D2Q9::vy(a) + 1;
                const float2 v = pair_floats<S>(own[j][a * plane]);
                if (vx == 0) {
                    d[a] = F2(v);
                } else if (vx == 1) {
                    const float2 l = pair_floats<S>(lft[j][a * plane]);
                    d[a] = F2(l.y, v.x);
                } else {
                    const float2 h = pair_floats<S>(rgt[j][a * plane]);
                    d[a] = F2(v.y, h.x);
                }
            }
            const bool inner = mid && (!cav || (y >= 1 && y <= ny - 2));  // the same for the warp
            if (!inner) {
                // pulls that leave the lattice
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    const int vx = D2Q9::vx(a), vy = D2Q9::vy(a);
                    if (a == 0) continue;
#pragma unroll
                    for (int l = 0; l < 2; ++l) {
                        const int sx = x + l - vx;
                        const bool xout = sx < 0 || sx >= nx;
                        if (cav) {
                            if (xout || y - vy < 0 || y - vy >= ny) N::set_lane(d[a], l, 0.f);
                        } else if (xout && vx != 0) {
                            // zero gradient: the end column's own value
                            const float2 v = pair_floats<S>(own[vy + 1][a * plane]);
                            N::set_lane(d[a], l, l == 0 ? v.x : v.y);
                        }
                    }
                }
            }
            uint32_t st = Collide<D2Q9, COLL, F2, (int)sizeof(S)>::run(d, rho0, rates, o);
            if (!inner && cav) {
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const int xl = x + l;
                    const bool out = xl < 0 || xl >= nx || y < 0 || y >= ny;
                    const bool wall = xl == 0 || xl == nx - 1 || y == 0;
                    const bool lid = !wall && y == ny - 1;
                    if (out || wall || lid) {
                        if (out) {
#pragma unroll
                            for (int a = 0; a < Q; ++a) N::set_lane(o[a], l, 0.f);
                        } else if (wall) {
#pragma unroll
                            for (int a = 0; a < Q; ++a) N::set_lane(o[a], l, N::lane(d[D2Q9::opp(a)], l));
                        } else {
#pragma unroll
                            for (int a = 0; a < Q; ++a) N::set_lane(o[a], l, in.lid_dev_f[a]);
                        }
                        st &= ~(3u << (2 * l));
                    }
                }
            }
            const bool row_mine = r >= part.y0 && r < part.y1;
            if (st && row_mine) {  // rare: a lane skipped its Newton step or is unstable
                if (!mine_a) st &= ~3u;
                if (!mine_b) st &= ~(3u << 2);
                n_skip += __popc(st & (ST_NEWTON_SKIPPED * 5u));
                n_unst += __popc(st & (ST_UNSTABLE * 5u));
            }
            if (!last) {
#pragma unroll
                for (int a = 0; a < Q; ++a) to[a * plane + r * 32 + lane] = pair_word<S>(o[a].v.x, o[a].v.y);
            } else if (row_mine && (mine_a || mine_b)) {
                S* p = static_cast<S*>(args.dst) + in.off + (int64_t)y * in.pitch + x;
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    const W w = pair_word<S>(o[a].v.x, o[a].v.y);
                    if (mine_a && mine_b && (x & 1) == 0) {
                        *reinterpret_cast<W*>(p + a * in.plane) = w;
                    } else {
                        const S* e = reinterpret_cast<const S*>(&w);
                        if (mine_a) p[a * in.plane] = e[0];
                        if (mine_b) p[a * in.plane + 1] = e[1];
                    }
                }
            }
        }
        if (!last) __syncthreads();
    }
    if (n_skip | n_unst) {
        atomicAdd(args.status + 2 * tile.inst + 0, (unsigned long long)n_skip);
        atomicAdd(args.status + 2 * tile.inst + 1, (unsigned long long)n_unst);
    }
}

template <typename S, int ROWS> const void* pick_step_block_kernel_rows(int collision) {
    switch (collision) {
        case COLL_MINXENT4: return (const void*)&step_block_kernel<S, COLL_MINXENT4, ROWS>;
        case COLL_SRT: return (const void*)&step_block_kernel<S, COLL_SRT, ROWS>;
        case COLL_MINXENT2: return (const void*)&step_block_kernel<S, COLL_MINXENT2, ROWS>;
        case COLL_MRT:
        case COLL_TRT: return (const void*)&step_block_kernel<S, COLL_MRT, ROWS>;
    }
    return nullptr;
}
template <typename S> const void* pick_step_block_kernel(int collision, int rows) {
    constexpr int MOST = block_max_rows(sizeof(S) == 4 ? 1 : 2);
    return rows <= BLOCK_SMALL_ROWS ? pick_step_block_kernel_rows<S, BLOCK_SMALL_ROWS>(collision)
                                    : pick_step_block_kernel_rows<S, MOST>(collision);
}

}  // namespace lbm
