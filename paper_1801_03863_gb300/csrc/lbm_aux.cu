// lbm_aux.cu -- the kernels around the time step: initial equilibrium,
// the first (in-place) collision after a state is loaded, moments and
// population read-out, population load, the stream function and the FP64
// conservation reduction.
//
// Their results are FP64 and GB300's FP64 pipe issues one warp instruction
// per scheduler in 64 cycles, so FP64 instructions, not bytes, bound what is
// written plainly: moments of 33 M nodes took 2.26 ms where their 42 bytes a
// node take 0.21 ms.  Conversions between FP64 and the storage types are
// done on the integer pipe (exactly), sums of FP16 values exactly in FP32 or
// integers, and 1 / rho by three FP64 instructions.
//
// One thread per node; a block takes `per` consecutive nodes of one instance
// (grid = (blocks of the largest instance, instance)).
//
// 33.4 M nodes in 64 cavities, FP16: init 2.81 -> 0.28 ms (at rest; 1.1 GB,
// 0.6 of the copy bandwidth), moments 2.26 -> 0.34 ms (FP64 issue: 6
// instructions a node).  18.0 M nodes in 4096 tubes, FP32: init 0.78 -> 0.12,
// moments 0.55 -> 0.22 ms.  12.2 M nodes D2Q9 FP32: moments 0.99 -> 0.25 ms
// (sums in fixed point: 6 FP64 instructions a node instead of 22).
#include <cooperative_groups.h>

#include <algorithm>

#include "lbm_aux.h"
#include "lbm_collide.cuh"

namespace lbm {
namespace {

constexpr int AUX_THREADS = 256;

// ---------------------------------------------------------------------------
// Conversions without the FP64 pipe.  Zeros and normal numbers are converted
// by their bits; what is left (FP32 subnormals and overflow, infinities, NaN)
// goes through the conversion instruction.
// ---------------------------------------------------------------------------
__device__ __noinline__ double widen_slow(float v) { return (double)v; }
__device__ __noinline__ float narrow_slow(double v) { return (float)v; }
__device__ __noinline__ __half half_slow(double v) { return __double2half(v); }
__device__ __noinline__ __nv_bfloat16 bf16_slow(double v) { return __double2bfloat16(v); }

__device__ __forceinline__ double widen(float v) {
    const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)  // normal
        return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
    if (m == 0u) return __hiloint2double((int)b, 0);
    return widen_slow(v);
}
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(__half v) { return widen(__half2float(v)); }
__device__ __forceinline__ double widen(__nv_bfloat16 v) { return widen(__bfloat162float(v)); }

// The double with this high word lies in [2^-126, 2^127) by magnitude: FP32's
// normal range but for its last binade, from which a rounding might overflow.
__device__ __forceinline__ bool in_f32_range(uint32_t hi) {
    return ((hi >> 20) & 0x7ffu) - 897u < 1150u - 897u;
}
// FP32 nearest to v, ties to even
__device__ __forceinline__ float narrow(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    if (in_f32_range(hi)) {
        const uint64_t u = ((uint64_t)(hi & 0x7fffffffu) << 32) | lo;
        const uint64_t r = u + 0x0fffffffull + ((u >> 29) & 1ull);
        return __uint_as_float((hi & 0x80000000u) | ((uint32_t)(r >> 29) - 0x38000000u * 8u));
    }
    if (((hi & 0x7fffffffu) | lo) == 0u) return __uint_as_float(hi);
    return narrow_slow(v);
}
// v to FP32 rounded to odd (truncated, with a sticky last bit), so that a
// second rounding to 16 bits rounds as once
__device__ __forceinline__ float narrow_odd(uint32_t hi, uint32_t lo) {
    const uint32_t m = (hi << 3) | (lo >> 29);  // the low 32 bits of |v| >> 29
    const uint32_t bits = (m - 0xc0000000u) & 0x7fffffffu;
    return __uint_as_float((hi & 0x80000000u) | bits | ((lo & 0x1fffffffu) != 0u ? 1u : 0u));
}
template <typename S> __device__ __forceinline__ S to_storage(double v);
template <> __device__ __forceinline__ double to_storage<double>(double v) { return v; }
template <> __device__ __forceinline__ float to_storage<float>(double v) { return narrow(v); }
template <> __device__ __forceinline__ __half to_storage<__half>(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    if (in_f32_range(hi)) return __float2half_rn(narrow_odd(hi, lo));
    if (((hi >> 20) & 0x7ffu) < 897u) return __ushort_as_half((unsigned short)((hi >> 16) & 0x8000u));
    return half_slow(v);
}
template <> __device__ __forceinline__ __nv_bfloat16 to_storage<__nv_bfloat16>(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    if (in_f32_range(hi)) return __float2bfloat16_rn(narrow_odd(hi, lo));
    if (((hi & 0x7fffffffu) | lo) == 0u) return __ushort_as_bfloat16((unsigned short)(hi >> 16));
    return bf16_slow(v);
}

// ---------------------------------------------------------------------------
// Populations of one node.
// ---------------------------------------------------------------------------
template <class Lat, typename S>
__device__ __forceinline__ const S* elem_ptr(const S* base, const InstDesc& in, int a, int x, int y) {
    return base + in.off + (int64_t)a * in.plane + (int64_t)y * in.pitch + x;
}

template <typename S> __device__ __forceinline__ S zero_value() { return S(0.0f); }

// Stored deviations of f(x, t_n) at one node.  pulled = true: the stored
// field is post-collision and the node pulls f_a from x - v_a with the
// boundary rules of the step; pulled = false: the stored field is f(x, t_n).
template <class Lat, typename S>
__device__ __forceinline__ void node_state(const S* src, const InstDesc& in, int x, int y, bool pulled,
                                           S (&d)[Lat::Q]) {
    if (!pulled) {
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) d[a] = *elem_ptr<Lat, S>(src, in, a, x, y);
        return;
    }
    const bool cav = in.bc == BC_CAVITY, per = in.bc == BC_PERIODIC;
    const int nx = in.nx, ny = in.ny;
    const bool l = x > 0, r = x + 1 < nx, b = y > 0, t = y + 1 < ny;
    const int xs[3] = {l ? x - 1 : (per ? nx - 1 : 0), x, r ? x + 1 : (per ? 0 : nx - 1)};
    const int ys[3] = {b ? y - 1 : ny - 1, y, t ? y + 1 : 0};
    const bool xok[3] = {l || !cav, true, r || !cav}, yok[3] = {b || !cav, true, t || !cav};
#pragma unroll
    for (int a = 0; a < Lat::Q; ++a) {
        const int i = 1 - Lat::vx(a), j = 1 - Lat::vy(a);
        d[a] = (xok[i] && yok[j]) ? *elem_ptr<Lat, S>(src, in, a, xs[i], ys[j]) : zero_value<S>();
    }
}

// sum d, sum d v_x, sum d v_y in the number type V
template <class Lat, typename V>
__device__ __forceinline__ void moment_sums(const V (&d)[Lat::Q], V& m, V& jx, V& jy) {
    if constexpr (Lat::Q == 9) {
        const V a57 = d[5] - d[7], a86 = d[8] - d[6];
        m = (d[0] + ((d[1] + d[3]) + (d[2] + d[4]))) + ((d[5] + d[7]) + (d[6] + d[8]));
        jx = (d[1] - d[3]) + a57 + a86;
        jy = (d[2] - d[4]) + a57 - a86;
    } else {
        m = d[0] + (d[1] + d[2]);
        jx = d[1] - d[2];
        jy = V(0);
    }
}

// v 2^(e - 1023) rounded to FP64 (to nearest, ties to even), 64 < e < 1983
__device__ __forceinline__ double fixed_to_f64(long long v, int e) {
    const uint64_t sign = (uint64_t)v & 0x8000000000000000ull;
    const uint64_t a = (uint64_t)(v < 0 ? -v : v);
    if (a == 0u) return 0.0;
    const int lz = __clzll((long long)a);
    const uint64_t n = a << lz;  // leading bit at 63: it adds one to the exponent field below
    const uint64_t up = ((n & 0x7ffu) + 0x3ffu + ((n >> 11) & 1u)) >> 11;
    const uint64_t bits = sign | (((uint64_t)(e + 62 - lz) << 52) + (n >> 11) + up);
    return __longlong_as_double((long long)bits);
}

// moment_sums of FP32 values in 64-bit fixed point, the largest value at bit
// 58: exact, so that each sum rounds once, and the work of the integer pipe.
// False where a value is not finite, the largest is below 2^-80, or the
// smallest (but for zeros) has bits more than 58 places below the largest's
// first: FP64 additions then lose less where the largest is not in the sum.
template <class Lat>
__device__ __forceinline__ bool fixed_sums(const float (&d)[Lat::Q], double& m, double& jx, double& jy) {
    uint32_t top = 0u, low = 0xffffffffu;  // low: smallest magnitude's bits less 1, zeros apart
#pragma unroll
    for (int a = 0; a < Lat::Q; ++a) {
        const uint32_t b = __float_as_uint(d[a]) & 0x7fffffffu;
        top = max(top, b);
        low = min(low, b - 1u);
    }
    const int emax = (int)(top >> 23);
    if (top == 0u) {
        m = jx = jy = 0.0;
        return true;
    }
    if (emax == 255 || emax < 47 || emax - (int)((low + 1u) >> 23) > 35) return false;
    long long v[Lat::Q];
#pragma unroll
    for (int a = 0; a < Lat::Q; ++a) {
        const uint32_t b = __float_as_uint(d[a]);  // (no subnormals here)
        const uint64_t mant = (b & 0x7fffffffu) ? (b & 0x7fffffu) | 0x800000u : 0u;
        const long long u = (long long)(mant << (((b >> 23) & 0xffu) + 35u - (uint32_t)emax & 63u));
        v[a] = (int)b < 0 ? -u : u;
    }
    long long im, ix, iy;
    moment_sums<Lat, long long>(v, im, ix, iy);
    // units of 2^(emax - 150 - 35)
    const int e = 1023 + emax - 185;
    m = fixed_to_f64(im, e);
    jx = fixed_to_f64(ix, e);
    jy = Lat::Q == 9 ? fixed_to_f64(iy, e) : 0.0;
    return true;
}

// The same in FP64 from stored values.  FP16 values are multiples of 2^-24:
// where all are below 1/16 in magnitude, their sums (below 1) are exact in
// FP32.  FP32 and BF16 values add in fixed point.
template <class Lat, typename S>
__device__ __forceinline__ void node_sums(const S (&raw)[Lat::Q], double& m, double& jx, double& jy) {
    if constexpr (std::is_same<S, __half>::value) {
        float d[Lat::Q], big = 0.f;
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) {
            d[a] = __half2float(raw[a]);
            big = fmaxf(big, fabsf(d[a]));  // (drops a NaN:)
        }
        float fm, fx, fy;
        moment_sums<Lat, float>(d, fm, fx, fy);
        if (big < 0.0625f && fm == fm) {
            m = widen(fm);
            jx = widen(fx);
            jy = widen(fy);
            return;
        }
    }
    if constexpr (std::is_same<S, float>::value || std::is_same<S, __nv_bfloat16>::value) {
        float d[Lat::Q];
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) d[a] = Store<S>::to_f32(raw[a]);
        if (fixed_sums<Lat>(d, m, jx, jy)) return;
    }
    double d[Lat::Q];
#pragma unroll
    for (int a = 0; a < Lat::Q; ++a) d[a] = widen(raw[a]);
    moment_sums<Lat, double>(d, m, jx, jy);
}

// f^eq(rho, u) - W rho0 (Eq. numerical-plyeqm),
//   W_a [(rho - rho0) + rho (3 v.u + 9/2 (v.u)^2 - 3/2 u^2)],
// with A = rho u_x^2, B = rho u_y^2, C = rho u_x u_y: 30 FP64 instructions.
// A warp whose nodes are all at rest takes W_a (rho - rho0) alone.
template <class Lat>
__device__ __forceinline__ void eq_dev(double rho, double ux, double uy, double rho0, bool rest,
                                       double (&d)[Lat::Q]) {
    const double dr = rho - rho0;
    if (rest) {
        const double w0 = Lat::w(0) * dr, w1 = Lat::w(1) * dr;
        const double w2 = Lat::Q == 9 ? Lat::w(Lat::Q - 1) * dr : 0.0;
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) d[a] = a == 0 ? w0 : (a < 5 ? w1 : w2);
        return;
    }
    const double jx = rho * ux, A = jx * ux;
    if constexpr (Lat::Q == 9) {
        const double jy = rho * uy, B = jy * uy, C = jx * uy, S = A + B, D = A - B;
        const double t = fma(0.75, S, dr), e = fma(3.0, S, dr);
        const double ex = fma(2.25, D, t) * (1.0 / 9.0), ey = fma(-2.25, D, t) * (1.0 / 9.0);
        const double ep = fma(9.0, C, e) * (1.0 / 36.0), em = fma(-9.0, C, e) * (1.0 / 36.0);
        const double jp = jx + jy, jm = jy - jx;
        d[0] = fma(-1.5, S, dr) * (4.0 / 9.0);
        d[1] = fma(1.0 / 3.0, jx, ex);
        d[3] = fma(-1.0 / 3.0, jx, ex);
        d[2] = fma(1.0 / 3.0, jy, ey);
        d[4] = fma(-1.0 / 3.0, jy, ey);
        d[5] = fma(1.0 / 12.0, jp, ep);
        d[7] = fma(-1.0 / 12.0, jp, ep);
        d[6] = fma(1.0 / 12.0, jm, em);
        d[8] = fma(-1.0 / 12.0, jm, em);
    } else {
        const double e = fma(3.0, A, dr) * (1.0 / 6.0);
        d[0] = fma(-1.5, A, dr) * (2.0 / 3.0);
        d[1] = fma(0.5, jx, e);
        d[2] = fma(-0.5, jx, e);
    }
}

// Node k of instance `in` (row-major, x fastest) as (x, y): 32-bit index
// arithmetic (nx * ny <= 2^31 for every instance).
__device__ __forceinline__ void node_xy(uint32_t k, uint32_t nx, int& x, int& y) {
    const uint32_t yy = k / nx;
    y = (int)yy;
    x = (int)(k - yy * nx);
}

// This block's nodes of an instance of n: [first, last)
__device__ __forceinline__ void block_range(uint32_t n, uint32_t per, uint32_t& first, uint32_t& last) {
    const uint64_t f = (uint64_t)blockIdx.x * per;
    first = f < n ? (uint32_t)f : n;
    last = n - first < per ? n : first + per;
}

// Host arrays are indexed from the first node of the instances the launch
// covers: node0 - node_base (node_base = 0 for whole-context calls, the
// instance's node0 for single-instance calls).
template <class Lat, typename S>
__global__ void __launch_bounds__(AUX_THREADS)
init_kernel(S* dst, const InstDesc* insts, const double* rho, const double* ux, const double* uy,
            double rho0, int64_t node_base, uint32_t per, unsigned long long* status, unsigned int* error) {
    const InstDesc& in = insts[blockIdx.y];
    if (error && blockIdx.x == 0) {  // (whole-context calls: two launches of memsets less)
        if (threadIdx.x < 2) status[2 * blockIdx.y + threadIdx.x] = 0ull;
        if (blockIdx.y == 0 && threadIdx.x >= 32 && threadIdx.x < 32 + ERROR_WORDS) error[threadIdx.x - 32] = 0u;
    }
    const uint32_t nx = (uint32_t)in.nx;
    uint32_t first, last;
    block_range(nx * (uint32_t)in.ny, per, first, last);
    const int64_t g0 = in.node0 - node_base;
    for (uint32_t w = first + (threadIdx.x & ~31u); w < last; w += AUX_THREADS) {  // whole warps
        const uint32_t k = w + (threadIdx.x & 31u);
        const bool some = k < last;
        double r = 0.0, vx = 0.0, vy = 0.0;
        if (some) {
            r = rho[g0 + k];
            if (ux) vx = ux[g0 + k];
            if (uy && Lat::Q == 9) vy = uy[g0 + k];
        }
        // at rest: both velocities are zero (of either sign)
        const uint32_t v = (uint32_t)__double2hiint(vx) << 1 | (uint32_t)__double2loint(vx) |
                           (uint32_t)__double2hiint(vy) << 1 | (uint32_t)__double2loint(vy);
        const bool rest = __all_sync(0xffffffffu, v == 0u);
        if (!some) continue;
        double d[Lat::Q];
        eq_dev<Lat>(r, vx, vy, rho0, rest, d);
        int x, y;
        node_xy(k, nx, x, y);
        S* p = dst + in.off + (int64_t)y * in.pitch + x;
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) p[a * in.plane] = to_storage<S>(d[a]);
    }
}

template <class Lat, typename S>
__global__ void __launch_bounds__(AUX_THREADS)
set_f_kernel(S* dst, const InstDesc* insts, const double* f, double rho0, uint32_t per) {
    const InstDesc& in = insts[blockIdx.y];
    const uint32_t nx = (uint32_t)in.nx, n = nx * (uint32_t)in.ny;
    uint32_t first, last;
    block_range(n, per, first, last);
    for (uint32_t k = first + threadIdx.x; k < last; k += AUX_THREADS) {
        int x, y;
        node_xy(k, nx, x, y);
        const double* fk = f + in.node0 * Lat::Q + k;
        S* p = dst + in.off + (int64_t)y * in.pitch + x;
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a)
            p[a * in.plane] = to_storage<S>(fk[(int64_t)a * n] - Lat::w(a) * rho0);
    }
}

// First step after a state was loaded: collide in place, no streaming
// (the loaded field is f(x, t_n) itself, Eq. 2's collision input).  The
// arithmetic is that of the step kernels -- FP64, or node pairs in packed
// FP32x2 for FP32 -- with the same rates and boundary rules, so this step
// rounds exactly like a step kernel colliding the same pulled values: a
// state saved from a running context and loaded into a new one continues
// bit for bit.  One thread per node pair (x, x + 1) of a row, read and
// written as one word per plane; at an odd width the second lane collides
// the row's padding and is discarded.
template <class Lat, typename S, typename T, int COLL>
__global__ void __launch_bounds__(AUX_THREADS)
collide_inplace_kernel(const S* src, S* dst, const InstDesc* insts, double rho0,
                       unsigned long long* status, uint32_t per) {
    using Word = typename std::conditional<sizeof(S) == 2, uint32_t, typename std::conditional<
        sizeof(S) == 4, uint2, double>::type>::type;  // P elements
    using CT = typename std::conditional<std::is_same<T, float>::value, F2, T>::type;
    using N = Num<CT>;
    using LT = typename LaneOf<CT>::type;
    constexpr int P = N::LANES;
    const int inst = blockIdx.y;
    const InstDesc& in = insts[inst];
    const uint32_t groups = ((uint32_t)in.nx + P - 1) / P;  // node groups per row
    const uint32_t n = groups * (uint32_t)in.ny;
    const Rates<CT> rates{CT((LT)in.omega), CT((LT)in.omega2), CT((LT)in.s_e), CT((LT)in.s_eps)};
    const CT rho0v = CT((LT)rho0);
    uint32_t first, last;
    block_range(n, per, first, last);
    unsigned long long n_skip = 0, n_unst = 0;
    for (uint32_t k = first + threadIdx.x; k < last; k += AUX_THREADS) {
        int g, y;
        node_xy(k, groups, g, y);
        const int x0 = g * P;
        const int64_t at = in.off + (int64_t)y * in.pitch + x0;
        CT d[Lat::Q], o[Lat::Q];
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) {
            union {
                Word w;
                S v[P];
            } e;
            e.w = *reinterpret_cast<const Word*>(src + at + a * in.plane);
#pragma unroll
            for (int l = 0; l < P; ++l) {
                if constexpr (std::is_same<T, double>::value) d[a] = Store<S>::to_f64(e.v[l]);
                else N::set_lane(d[a], l, Store<S>::to_f32(e.v[l]));
            }
        }
        uint32_t st = Collide<Lat, COLL, CT, (int)sizeof(S)>::run(d, rho0v, rates, o);
        if (in.bc == BC_CAVITY) {
#pragma unroll
            for (int l = 0; l < P; ++l) {
                const int x = x0 + l;
                const bool wall = (x == 0) || (x == in.nx - 1) || (y == 0);
                const bool lid = !wall && (y == in.ny - 1);
                if (wall) {
#pragma unroll
                    for (int a = 0; a < Lat::Q; ++a) N::set_lane(o[a], l, N::lane(d[Lat::opp(a)], l));
                    st &= ~(3u << (2 * l));
                } else if (lid) {
#pragma unroll
                    for (int a = 0; a < Lat::Q; ++a) {
                        if constexpr (std::is_same<T, double>::value) N::set_lane(o[a], l, in.lid_dev[a]);
                        else N::set_lane(o[a], l, in.lid_dev_f[a]);
                    }
                    st &= ~(3u << (2 * l));
                }
            }
        }
#pragma unroll
        for (int l = 0; l < P; ++l) {
            if (x0 + l >= in.nx) continue;
            n_skip += (st >> (2 * l)) & ST_NEWTON_SKIPPED;
            n_unst += ((st >> (2 * l)) & ST_UNSTABLE) >> 1;
        }
        const bool whole = x0 + P <= in.nx;
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) {
            union {
                Word w;
                S v[P];
            } e;
#pragma unroll
            for (int l = 0; l < P; ++l) e.v[l] = Store<S>::from(N::lane(o[a], l));
            S* p = dst + at + a * in.plane;
            if (whole) *reinterpret_cast<Word*>(p) = e.w;
            else *p = e.v[0];
        }
    }
    if (n_skip) atomicAdd(status + 2 * inst + 0, n_skip);
    if (n_unst) atomicAdd(status + 2 * inst + 1, n_unst);
}

template <class Lat, typename S>
__global__ void __launch_bounds__(AUX_THREADS)
moments_kernel(const S* src, const InstDesc* insts, bool pulled, double rho0, double* rho, double* ux,
               double* uy, int64_t node_base, uint32_t per) {
    const InstDesc& in = insts[blockIdx.y];
    const uint32_t nx = (uint32_t)in.nx;
    uint32_t first, last;
    block_range(nx * (uint32_t)in.ny, per, first, last);
    const int64_t g0 = in.node0 - node_base;
    for (uint32_t k = first + threadIdx.x; k < last; k += AUX_THREADS) {
        int x, y;
        node_xy(k, nx, x, y);
        S raw[Lat::Q];
        node_state<Lat, S>(src, in, x, y, pulled, raw);
        double m, jx, jy;
        node_sums<Lat, S>(raw, m, jx, jy);
        const double r = rho0 + m;
        rho[g0 + k] = r;
        if (ux || uy) {
            const double ir = rcp_f64(r);
            if (ux) ux[g0 + k] = jx * ir;
            if (uy) uy[g0 + k] = jy * ir;
        }
    }
}

template <class Lat, typename S>
__global__ void __launch_bounds__(AUX_THREADS)
gather_f_kernel(const S* src, const InstDesc* insts, bool pulled, double rho0, double* f, uint32_t per) {
    const InstDesc& in = insts[blockIdx.y];
    const uint32_t nx = (uint32_t)in.nx, n = nx * (uint32_t)in.ny;
    uint32_t first, last;
    block_range(n, per, first, last);
    for (uint32_t k = first + threadIdx.x; k < last; k += AUX_THREADS) {
        int x, y;
        node_xy(k, nx, x, y);
        S raw[Lat::Q];
        node_state<Lat, S>(src, in, x, y, pulled, raw);
        double* fk = f + in.node0 * Lat::Q + k;
#pragma unroll
        for (int a = 0; a < Lat::Q; ++a) fk[(int64_t)a * n] = Lat::w(a) * rho0 + widen(raw[a]);
    }
}

// The columns [nx, pitch) of every row and plane to zero.  Nothing reads them,
// but the TMA kernel's stores, clipped at 16 bytes, leave values there where
// the other step kernels do not, and a saved state is to be the same whichever
// kernels took its steps.
template <class Lat, typename S>
__global__ void __launch_bounds__(AUX_THREADS) clear_padding_kernel(S* dst, const InstDesc* insts) {
    const InstDesc& in = insts[blockIdx.y];
    const int pad = in.pitch - in.nx;
    const int64_t n = (int64_t)pad * in.ny * Lat::Q;
    for (int64_t k = (int64_t)blockIdx.x * AUX_THREADS + threadIdx.x; k < n; k += (int64_t)gridDim.x * AUX_THREADS) {
        const int64_t row = k / pad, a = row / in.ny, y = row - a * in.ny;
        dst[in.off + a * in.plane + y * in.pitch + in.nx + (k - row * pad)] = zero_value<S>();
    }
}

// Stream function of the LDAS post-processing (Sec. IV.I) along each row of
// each instance: psi(x, y) = - integral_0^x u_y dx in lattice units, with
// the composite Simpson rule over pairs of unit intervals from the left
// wall and the trapezoidal rule on the last interval when x is odd.
//
// A warp takes a row in stretches of 256 nodes (128 or 64 at its end): u_y of the stretch straight
// from the populations (no density or velocity field goes through memory)
// into shared memory, then each lane integrates its 8 (4, 2) consecutive nodes, a
// warp scan adds up the lanes, and the results go back through shared memory
// so that they are stored in order.  4 FP64 instructions a node besides
// u_y's own.  8.9 M nodes in 64 lattices, FP16: 0.72 ms of moments and 0.29
// ms of one thread per row walking its row in memory, now 0.20 ms; 257 x 257
// FP64: 68 -> 20 us.  Rows of up to 32 nodes share a warp (4 x 100000 FP64: 205
// -> 22 us; with one thread per row 41 us).
constexpr int PSI_WARPS = 4, PSI_NODES = 256;
template <typename S>
__global__ void __launch_bounds__(PSI_WARPS * 32)
stream_function_kernel(const S* src, const InstDesc* insts, bool pulled, double rho0, double* psi,
                       int64_t node_base) {
    __shared__ double buf[PSI_WARPS][PSI_NODES + 2];  // u_y of nodes x - 2 .. x + 255
    const InstDesc& in = insts[blockIdx.y];
    const int nx = in.nx, lane = (int)(threadIdx.x & 31u);
    double* u = buf[threadIdx.x >> 5];
    auto velocity = [&](int x, int y) {  // u_y
        S raw[9];
        node_state<D2Q9, S>(src, in, x, y, pulled, raw);
        double m, jx, jy;
        node_sums<D2Q9, S>(raw, m, jx, jy);
        return jy * rcp_f64(rho0 + m);
    };
    if (nx <= 32) {
        // rows that 16 lanes or fewer hold, 2 nodes each, share a warp
        int log_lanes = 0;
        while ((2 << log_lanes) < nx) ++log_lanes;
        const int lanes = 1 << log_lanes, l = lane & (lanes - 1), x = 2 * l;
        const int64_t rows = 32 >> log_lanes, all = (int64_t)gridDim.x * PSI_WARPS * rows;
        for (int64_t y0 = ((int64_t)blockIdx.x * PSI_WARPS + (threadIdx.x >> 5)) * rows; y0 < in.ny; y0 += all) {
            const int64_t y = y0 + (lane >> log_lanes);
            const bool a = y < in.ny && x < nx, b = y < in.ny && x + 1 < nx;
            const double v0 = a ? velocity(x, (int)y) : 0.0, v1 = b ? velocity(x + 1, (int)y) : 0.0;
            const double w0 = __shfl_up_sync(0xffffffffu, v0, 1), w1 = __shfl_up_sync(0xffffffffu, v1, 1);
            const double inc = l == 0 ? 0.0 : fma(4.0, w1, w0 + v0) * (1.0 / 3.0);
            double sum = inc;
            for (int d = 1; d < lanes; d <<= 1) {
                const double o = __shfl_up_sync(0xffffffffu, sum, d);
                if (l >= d) sum += o;
            }
            const double left = __shfl_up_sync(0xffffffffu, sum, 1);
            const double e = (l == 0 ? 0.0 : left) + inc;
            double* p = psi + (in.node0 - node_base) + y * nx + x;
            if (a) p[0] = -e;
            if (b) p[1] = -fma(0.5, v0 + v1, e);
        }
        return;
    }
    for (int y = blockIdx.x * PSI_WARPS + (int)(threadIdx.x >> 5); y < in.ny; y += gridDim.x * PSI_WARPS) {
        double* p = psi + (in.node0 - node_base) + (int64_t)y * nx;
        double carry = 0.0;  // integral over [0, x0 - 2]
        double last = 0.0;   // lanes 30, 31: u_y of nodes x0 - 2, x0 - 1
        // one stretch of 32 L nodes from x0, L consecutive nodes per lane
        auto stretch = [&](auto length, int x0) {
            constexpr int L = decltype(length)::value;
            if (lane >= 30) u[lane - 30] = last;
#pragma unroll 2
            for (int i = 0; i < 32 * L; i += 32) {
                const int x = x0 + i + lane;
                double v = 0.0;
                if (x < nx) v = velocity(x, y);
                u[2 + i + lane] = v;
                last = v;
            }
            __syncwarp();
            // own nodes x0 + L lane + 0 .. L - 1 are v[2 ..]
            double v[L + 2], s[L / 2];  // s: integral from the lane's second node back to each even node
#pragma unroll
            for (int i = 0; i < L + 2; ++i) v[i] = u[L * lane + i];
#pragma unroll
            for (int j = 0; j < L / 2; ++j) {
                double inc = fma(4.0, v[2 * j + 1], v[2 * j] + v[2 * j + 2]) * (1.0 / 3.0);
                if (j == 0 && x0 + lane == 0) inc = 0.0;  // nothing left of node 0
                s[j] = j == 0 ? inc : s[j - 1] + inc;
            }
            double sum = s[L / 2 - 1];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const double o = __shfl_up_sync(0xffffffffu, sum, d);
                if (lane >= d) sum += o;
            }
            double base = __shfl_up_sync(0xffffffffu, sum, 1);
            base = lane == 0 ? carry : base + carry;
            carry += __shfl_sync(0xffffffffu, sum, 31);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < L / 2; ++j) {
                const double e = base + s[j];
                u[2 + L * lane + 2 * j] = -e;
                u[2 + L * lane + 2 * j + 1] = -fma(0.5, v[2 * j + 2] + v[2 * j + 3], e);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 32 * L; i += 32)
                if (x0 + i + lane < nx) p[x0 + i + lane] = u[2 + i + lane];
            __syncwarp();
        };
        // the shortest stretch that holds the rest of the row: a padding node
        // costs as much FP64 issue as any other
        for (int x0 = 0; x0 < nx;) {
            if (nx - x0 > 128) {
                stretch(std::integral_constant<int, 8>{}, x0);
                x0 += 256;
            } else if (nx - x0 > 64) {
                stretch(std::integral_constant<int, 4>{}, x0);
                x0 += 128;
            } else {
                stretch(std::integral_constant<int, 2>{}, x0);
                x0 += 64;
            }
        }
    }
}

// Conservation, pass 1.  Node x pulls f_a from x - v_a, so summed over an
// instance every stored value counts as often as nodes pull it: once, but
// for values on the outer ring (a cavity's are not pulled by a node when they
// leave the lattice; at a zero-gradient end the leaving ones are not pulled
// and the entering ones are pulled twice).  The reduction therefore reads the
// stored planes as they lie, 16 bytes per load, and weighs ring values.
//
// Partial b of instance i sums its rows y = b mod P_i (P_i = cons_partials),
// in a cluster of CTAs; of these, C_i = cons_split(nodes) CTAs take the
// rows' 16-byte chunks in turn (the others of the launch's cluster add zero),
// and the first CTA of the cluster adds the CTAs' sums in order.  The order
// of all additions is fixed by the instance alone.
//
// FP64 storage sums in FP64.  FP32 and BF16 storage sum a thread's nodes in
// compensated FP32 pairs (Knuth's two-sum; about twice FP32's precision,
// converted to FP64 once per thread), which spares the slow FP64 pipe.  FP16 storage sums
// exactly in integers: every FP16 value is a multiple of 2^-24 below 2^16 in
// magnitude; a chunk whose values are all below 2^-7 adds exactly in FP32
// (its sums stay below 1) and is converted to integers once, a node below
// 2^-4 likewise, others add in 64-bit integers, and a warp's total is
// converted to FP64.
// Nodes with a non-finite value take FP64, so that it propagates.
//
// Bound by the latency of a thread's few chunks and its CTA's tail, at 0.4 of
// the copy bandwidth.  64 cavities (33.4 M nodes) FP16: 324 us with shifted
// loads per node, now 214 us; 2048^2 FP16: 134 -> 51 us (clusters of 4);
// 4096 tubes FP32: 343 -> 84 us.  Pass 2 with one thread per instance took
// 17 us, now 6 us.
template <class Lat>
__device__ __forceinline__ int pull_count(const InstDesc& in, int a, int x, int y) {
    const int tx = x + Lat::vx(a), ty = y + Lat::vy(a);
    const bool xin = tx >= 0 && tx < in.nx, yin = ty >= 0 && ty < in.ny;
    if (in.bc == BC_CAVITY) return xin && yin ? 1 : 0;
    if (in.bc == BC_PERIODIC) return 1;
    // zero gradient (y wraps): the end node's entering value is its own
    const bool entering = (Lat::vx(a) == 1 && x == 0) || (Lat::vx(a) == -1 && x == in.nx - 1);
    return (xin ? 1 : 0) + (entering ? 1 : 0);
}

struct ConsSums {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    long long i0 = 0, i1 = 0, i2 = 0;                   // FP16: exact sums in units of 2^-24
    F2 h0 = 0.f, c0 = 0.f, h1 = 0.f, c1 = 0.f, h2 = 0.f, c2 = 0.f;  // FP32 / BF16: (sum, error)
};

// h + v = s + e exactly (Knuth's two-sum); the error joins the running c
__device__ __forceinline__ void add2(F2& h, F2& c, F2 v) {
    const F2 sum = h + v;
    const F2 bv = sum - h;
    const F2 e = (h - (sum - bv)) + (v - bv);
    h = sum;
    c = c + e;
}

template <class Lat> __device__ __forceinline__ void cons_add_f64(ConsSums& t, const double (&d)[Lat::Q]) {
    double m, jx, jy;
    moment_sums<Lat, double>(d, m, jx, jy);
    t.s0 += m;
    t.s1 += jx;
    t.s2 += jy;
}

// Sums of an FP16 node in units of 2^-24: exact in FP32 where all values are
// below 1/16 (the sums stay below 1), else in 64-bit integers; false if some
// value is not finite.
template <class Lat>
__device__ __forceinline__ bool half_sums(const float (&d)[Lat::Q], long long (&r)[3]) {
    float big = 0.f, m, jx, jy;
#pragma unroll
    for (int a = 0; a < Lat::Q; ++a) big = fmaxf(big, fabsf(d[a]));
    moment_sums<Lat, float>(d, m, jx, jy);
    if (big < 0.0625f && m == m) {
        r[0] = __float2int_rn(m * 16777216.f);
        r[1] = __float2int_rn(jx * 16777216.f);
        r[2] = __float2int_rn(jy * 16777216.f);
        return true;
    }
    bool finite = true;
#pragma unroll
    for (int a = 0; a < Lat::Q; ++a) {
        finite = finite && fabsf(d[a]) <= 131008.f;  // twice FP16's largest (a value pulled twice)
        const long long v = __float2ll_rn(d[a] * 16777216.f);
        r[0] += v;
        r[1] += Lat::vx(a) * v;
        r[2] += Lat::vy(a) * v;
    }
    return finite;
}

__device__ __noinline__ double add_slow(long long a, long long b) { return (double)a + (double)b; }

// CLUSTER: launched in clusters of several CTAs.  totals (null: none): every
// instance is one partial, and pass 2 is spared (5000 tubes of 100 nodes, FP32
// 33 us with it).
template <class Lat, typename S, bool CLUSTER>
__global__ void __launch_bounds__(CONS_THREADS, 3)
cons_partial_kernel(const S* src, const InstDesc* insts, const int2* items, bool pulled, double* partials,
                    double rho0, double* totals) {
    constexpr int Q = Lat::Q, E = 16 / (int)sizeof(S);  // nodes per chunk
    const int2 it = items[blockIdx.x];
    const InstDesc& in = insts[it.x];
    const int nx = in.nx, ny = in.ny, P = cons_partials(nx, ny, (int)sizeof(S));
    const uint32_t C = (uint32_t)cons_split((int64_t)nx * ny), rank = blockIdx.y;
    const uint32_t chunks = (uint32_t)(nx + E - 1) / E;       // per row
    const uint64_t total = (uint64_t)((ny - it.y + P - 1) / P) * chunks;
    const S* base = src + in.off;
    ConsSums t;
    if (rank < C)
        for (uint64_t k = rank * CONS_THREADS + threadIdx.x; k < total; k += (uint64_t)C * CONS_THREADS) {
            const uint32_t row = (uint32_t)(total <= 0xffffffffull ? (uint32_t)k / chunks : k / chunks);
            const int y = it.y + (int)row * P, x0 = (int)(k - (uint64_t)row * chunks) * E;
            union {
                uint4 w;
                S v[E];
                __half2 h[4];
            } raw[Q];
#pragma unroll
            for (int a = 0; a < Q; ++a)
                raw[a].w = __ldg(reinterpret_cast<const uint4*>(base + a * in.plane + (int64_t)y * in.pitch + x0));
            const bool ring = x0 == 0 || x0 + E >= nx || (Q == 9 && (y == 0 || y == ny - 1));
            if (ring) {
#pragma unroll
                for (int a = 0; a < Q; ++a)
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int n = x0 + e >= nx ? 0 : pulled ? pull_count<Lat>(in, a, x0 + e, y) : 1;
                        if (n == 0) raw[a].v[e] = zero_value<S>();
                    }
            }
            // values pulled twice (zero-gradient ends) count once more
            auto node = [&](int e, auto&& value) {
                const int x = x0 + e;
                if (ring && pulled && in.bc == BC_ZERO_GRADIENT && (x == 0 || x == nx - 1)) {
#pragma unroll
                    for (int a = 0; a < Q; ++a)
                        if (pull_count<Lat>(in, a, x, y) == 2) value(a) = value(a) + value(a);
                }
            };
            if constexpr (std::is_same<S, double>::value) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    double d[Q];
#pragma unroll
                    for (int a = 0; a < Q; ++a) d[a] = raw[a].v[e];
                    node(e, [&](int a) -> double& { return d[a]; });
                    cons_add_f64<Lat>(t, d);
                }
            } else if constexpr (std::is_same<S, __half>::value) {
                // largest magnitude of the chunk, NaN if there is one
                __half2 big2 = __habs2(raw[0].h[0]);
#pragma unroll
                for (int a = 0; a < Q; ++a)
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) big2 = __hmax2_nan(big2, __habs2(raw[a].h[e]));
                const float big = __half2float(__hmax_nan(__low2half(big2), __high2half(big2)));
                const bool twice = ring && pulled && in.bc == BC_ZERO_GRADIENT;
                if (big < 0.0078125f && !twice) {
                    // exact in FP32 over the whole chunk: 8 nodes of 9 values below 2^-7
                    F2 m = 0.f, jx = 0.f, jy = 0.f;
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) {
                        F2 d[Q], mm, jjx, jjy;
#pragma unroll
                        for (int a = 0; a < Q; ++a) d[a] = F2(__half22float2(raw[a].h[e]));
                        moment_sums<Lat, F2>(d, mm, jjx, jjy);
                        m = m + mm;
                        jx = jx + jjx;
                        if (Q == 9) jy = jy + jjy;
                    }
                    t.i0 += __float2int_rn((m.v.x + m.v.y) * 16777216.f);
                    t.i1 += __float2int_rn((jx.v.x + jx.v.y) * 16777216.f);
                    if (Q == 9) t.i2 += __float2int_rn((jy.v.x + jy.v.y) * 16777216.f);
                } else {
#pragma unroll 1
                    for (int e = 0; e < E; ++e) {
                        float d[Q];
                        long long r[3] = {0, 0, 0};
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
                            // element e by shifts: no indexing of registers
                            const uint32_t lo = e < 4 ? (e < 2 ? raw[a].w.x : raw[a].w.y) : (e < 6 ? raw[a].w.z : raw[a].w.w);
                            d[a] = __half2float(__ushort_as_half((unsigned short)(e & 1 ? lo >> 16 : lo & 0xffffu)));
                        }
                        node(e, [&](int a) -> float& { return d[a]; });
                        if (half_sums<Lat>(d, r)) {
                            t.i0 += r[0];
                            t.i1 += r[1];
                            t.i2 += r[2];
                        } else {
                            double f[Q];
#pragma unroll
                            for (int a = 0; a < Q; ++a) f[a] = (double)d[a];
                            cons_add_f64<Lat>(t, f);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; e += 2) {
                    float2 d[Q];
                    uint32_t big = 0u;
#pragma unroll
                    for (int a = 0; a < Q; ++a)
                        d[a] = make_float2(Store<S>::to_f32(raw[a].v[e]), Store<S>::to_f32(raw[a].v[e + 1]));
                    node(e, [&](int a) -> float& { return d[a].x; });
                    node(e + 1, [&](int a) -> float& { return d[a].y; });
#pragma unroll
                    for (int a = 0; a < Q; ++a)
                        big = max(big, max(__float_as_uint(d[a].x) & 0x7fffffffu, __float_as_uint(d[a].y) & 0x7fffffffu));
                    if (big < 0x7f800000u) {
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
                            const F2 v = d[a];
                            add2(t.h0, t.c0, v);
                            if (Lat::vx(a) != 0) add2(t.h1, t.c1, Lat::vx(a) > 0 ? v : -v);
                            if (Lat::vy(a) != 0) add2(t.h2, t.c2, Lat::vy(a) > 0 ? v : -v);
                        }
                    } else {
#pragma unroll 1
                        for (int l = 0; l < 2; ++l) {
                            double f[Q];
#pragma unroll
                            for (int a = 0; a < Q; ++a) f[a] = (double)(l ? d[a].y : d[a].x);
                            cons_add_f64<Lat>(t, f);
                        }
                    }
                }
            }
        }
    // fixed trees: threads, then the CTAs of the cluster in order; the terms of
    // threads and warps without nodes, zeros, are left out
    __shared__ double cta[3];
    const uint64_t before = (uint64_t)rank * CONS_THREADS;
    const uint32_t threads = rank < C && total > before ? (uint32_t)min(total - before, (uint64_t)CONS_THREADS) : 0u;
    const uint32_t warps = (threads + 31u) / 32u, lanes = min(threads, 32u);  // with nodes
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    if constexpr (std::is_same<S, __half>::value) {
        // integers add exactly within a warp; FP64 only holds nodes with non-finite values.
        // A lane has some 2^15 nodes at most (2^31 nodes of an instance, of at least 1 in 8 CTAs
        // of 256 threads; a row has at most 2^26), so its sums stay below
        // 2^15 x 9 x 2^40 < 2^58.2 and those of 16 lanes below 2^62.2; those of
        // two such halves may not fit.
        __shared__ double sh[3][CONS_THREADS / 32];
        if (warp < warps) {
            double s[3] = {t.s0, t.s1, t.s2};
            long long i[3] = {t.i0, t.i1, t.i2};
            const bool in_f64 = __any_sync(0xffffffffu, !(s[0] == 0.0 && s[1] == 0.0 && s[2] == 0.0));
#pragma unroll
            for (int c = 0; c < (Q == 3 ? 2 : 3); ++c) {
#pragma unroll
                for (int h = 16; h > 1; h >>= 1) i[c] += __shfl_down_sync(0xffffffffu, i[c], h);
                const long long o = __shfl_down_sync(0xffffffffu, i[c], 1);
                const long long sum = (long long)((uint64_t)i[c] + (uint64_t)o);
                if (lane == 0u) {
                    const bool wraps = ((i[c] ^ sum) & (o ^ sum)) < 0;
                    s[c] += (wraps ? add_slow(i[c], o) : (double)sum) * (1.0 / 16777216.0);
                }
                if (in_f64) {
#pragma unroll
                    for (int h = 16; h > 0; h >>= 1) s[c] += __shfl_down_sync(0xffffffffu, s[c], h);
                }
                if (lane == 0u) sh[c][warp] = s[c];
            }
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            double v = 0.0;
            if (threadIdx.x < (Q == 3 ? 2 : 3))
                for (uint32_t w = 0; w < warps; ++w) v = w == 0u ? sh[threadIdx.x][0] : v + sh[threadIdx.x][w];
            cta[threadIdx.x] = v;
        }
    } else {
        // A thread's sums in FP64, then one warp per sum adds them: 8 of every lane and a shuffle
        // tree, 36 FP64 warp instructions a CTA where a tree in each warp takes 120
        __shared__ double sh[3][CONS_THREADS];
        if (warp < warps) {
            double s[3] = {t.s0, t.s1, t.s2};
            if constexpr (!std::is_same<S, double>::value) {
                const F2 h[3] = {t.h0, t.h1, t.h2}, e[3] = {t.c0, t.c1, t.c2};
#pragma unroll
                for (int c = 0; c < (Q == 3 ? 2 : 3); ++c) {
                    // the thread's two node lanes as one pair
                    const float x = h[c].v.x, y = h[c].v.y;
                    const float sum = __fadd_rn(x, y), bv = __fsub_rn(sum, x);
                    const float r = __fadd_rn(__fadd_rn(e[c].v.x, e[c].v.y),
                                              __fadd_rn(__fsub_rn(x, __fsub_rn(sum, bv)), __fsub_rn(y, bv)));
                    const double v = widen(sum) + widen(r);
                    s[c] = __double_as_longlong(s[c]) == 0 ? v : s[c] + v;  // (FP64 part: nodes that are not finite)
                }
            }
#pragma unroll
            for (int c = 0; c < (Q == 3 ? 2 : 3); ++c) sh[c][threadIdx.x] = s[c];
        }
        __syncthreads();
        if (warp < 3u) {
            double v = 0.0;
            if (warp < (Q == 3 ? 2u : 3u) && warps > 0u) {
                v = sh[warp][lane];
                for (uint32_t w = 1; w < warps; ++w) v += sh[warp][lane + 32u * w];
#pragma unroll
                for (uint32_t h = 16; h > 0; h >>= 1)
                    if (lanes > h) v += __shfl_down_sync(0xffffffffu, v, h);
            }
            if (lane == 0u) cta[warp] = v;
        }
    }
    double* out = partials + ((int64_t)it.x * CONS_PARTIALS + it.y) * 3;
    if constexpr (CLUSTER) {
        const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
        cluster.sync();
        if (rank == 0 && threadIdx.x < 3) {
            double v = 0.0;
            for (uint32_t r = 0; r < C; ++r) v += *cluster.map_shared_rank(&cta[threadIdx.x], r);
            out[threadIdx.x] = v;
        }
        cluster.sync();  // a CTA's shared memory stays until the first has read it
    } else {
        __syncthreads();
        if (threadIdx.x < 3) {
            const double v = cta[threadIdx.x];
            if (totals) {  // one partial an instance: its totals
                totals[3 * it.x + threadIdx.x] = threadIdx.x == 0 ? (double)nx * (double)ny * rho0 + v : v;
            } else {
                out[threadIdx.x] = v;
            }
        }
    }
}

// Conservation, pass 2: one warp per instance adds its partials in a fixed
// tree; total mass = N rho0 + sum d (sum_a W_a = 1).
__global__ void cons_final_kernel(const double* partials, const InstDesc* insts, int count, int bytes,
                                  double rho0, double* out) {
    const int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = (int)(threadIdx.x & 31u);
    if (i >= count) return;
    const int P = cons_partials(insts[i].nx, insts[i].ny, bytes);
    double s[3] = {0.0, 0.0, 0.0};
    for (int b = lane; b < P; b += 32)
        for (int c = 0; c < 3; ++c) s[c] += partials[((int64_t)i * CONS_PARTIALS + b) * 3 + c];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int h = 16; h > 0; h >>= 1)
            if (P > h) s[c] += __shfl_down_sync(0xffffffffu, s[c], h);  // (others' terms are zeros)
    if (lane != 0) return;
    const double nodes = (double)insts[i].nx * (double)insts[i].ny;
    out[3 * i + 0] = nodes * rho0 + s[0];
    out[3 * i + 1] = s[1];
    out[3 * i + 2] = s[2];
}

// Nodes of a block: at most 2048 (8 per thread), fewer while that leaves
// less than 8 blocks per SM for the whole launch.  Beside a large instance
// (of max_items) the others' blocks are mostly empty ones, so an ensemble's
// instances get at most 4096 each (one 12000 x 12000 lattice beside 5000 of 20 x
// 20, FP16: init 179 -> 7.5 ms).
uint32_t nodes_per_block(int64_t total, int64_t max_items, int count) {
    uint32_t per = 2048;
    while (per > AUX_THREADS && total / per < 8 * 152) per /= 2;
    while (count > 1 && (max_items + per - 1) / per > 4096) per *= 2;
    return per;
}
dim3 aux_grid(int64_t max_items, int count, uint32_t per) {
    return dim3((unsigned)std::max<int64_t>((max_items + per - 1) / per, 1), (unsigned)count);
}

template <class Lat, typename S, typename T, int COLL>
cudaError_t collide_inplace_dispatch(const AuxArgs& a, const void* src, void* dst) {
    // node pairs of a row, rounded up per row
    const int P = std::is_same<T, float>::value ? 2 : 1;
    const int64_t most = a.max_nodes / P + a.max_ny;
    const uint32_t per = nodes_per_block(a.total_nodes / P, most, a.count);
    collide_inplace_kernel<Lat, S, T, COLL>
        <<<aux_grid(most, a.count, per), AUX_THREADS, 0, a.stream>>>(
            static_cast<const S*>(src), static_cast<S*>(dst), a.inst, a.rho0, a.status, per);
    return cudaGetLastError();
}

// TRT shares the MRT kernel.  D1Q3 collides in its step kernel.
template <class Lat, typename S, typename T>
cudaError_t collide_inplace_by_rule(const AuxArgs& a, const void* src, void* dst) {
    if constexpr (Lat::Q == 3) {
        return cudaErrorInvalidValue;
    } else {
        switch (a.collision) {
            case COLL_MINXENT4: return collide_inplace_dispatch<Lat, S, T, COLL_MINXENT4>(a, src, dst);
            case COLL_SRT: return collide_inplace_dispatch<Lat, S, T, COLL_SRT>(a, src, dst);
            case COLL_MINXENT2: return collide_inplace_dispatch<Lat, S, T, COLL_MINXENT2>(a, src, dst);
            case COLL_MRT:
            case COLL_TRT: return collide_inplace_dispatch<Lat, S, T, COLL_MRT>(a, src, dst);
        }
        return cudaErrorInvalidValue;
    }
}

template <class Lat, typename S>
cudaError_t aux_dispatch(AuxOp op, const AuxArgs& a, const void* src, void* dst, const double* p0,
                         const double* p1, const double* p2, double* o0, double* o1, double* o2) {
    const uint32_t per = nodes_per_block(a.total_nodes, a.max_nodes, a.count);
    const dim3 g = aux_grid(a.max_nodes, a.count, per);
    switch (op) {
        case AuxOp::Init:
            init_kernel<Lat, S><<<g, AUX_THREADS, 0, a.stream>>>(static_cast<S*>(dst), a.inst, p0, p1,
                                                                 p2, a.rho0, a.node_base, per, a.status,
                                                                 a.error);
            break;
        case AuxOp::SetF:
            set_f_kernel<Lat, S><<<g, AUX_THREADS, 0, a.stream>>>(static_cast<S*>(dst), a.inst, p0,
                                                                  a.rho0, per);
            break;
        case AuxOp::Moments:
            moments_kernel<Lat, S><<<g, AUX_THREADS, 0, a.stream>>>(static_cast<const S*>(src), a.inst,
                                                                    a.pulled, a.rho0, o0, o1, o2,
                                                                    a.node_base, per);
            break;
        case AuxOp::GatherF:
            gather_f_kernel<Lat, S><<<g, AUX_THREADS, 0, a.stream>>>(static_cast<const S*>(src), a.inst,
                                                                     a.pulled, a.rho0, o0, per);
            break;
        case AuxOp::ClearPadding: {
            const int64_t most = (int64_t)7 * a.max_ny * Lat::Q;  // rows are padded to a multiple of 8
            const dim3 blocks((unsigned)std::min<int64_t>((most + AUX_THREADS - 1) / AUX_THREADS, 1024), (unsigned)a.count);
            clear_padding_kernel<Lat, S><<<blocks, AUX_THREADS, 0, a.stream>>>(static_cast<S*>(dst), a.inst);
            break;
        }
        case AuxOp::StreamFunction:
            if constexpr (Lat::Q == 9) {
                // a warp per row
                const dim3 rows((unsigned)std::max<int64_t>((a.max_ny + PSI_WARPS - 1) / PSI_WARPS, 1),
                                (unsigned)a.count);
                stream_function_kernel<S><<<rows, PSI_WARPS * 32, 0, a.stream>>>(
                    static_cast<const S*>(src), a.inst, a.pulled, a.rho0, o0, a.node_base);
                break;
            }
            return cudaErrorInvalidValue;
        case AuxOp::Conservation: {
            if (a.cons_nitems < 1 || !a.cons_items) return cudaErrorInvalidValue;
            // clusters of as many CTAs as the largest instance splits into
            const unsigned C = (unsigned)cons_split(a.max_nodes);
            const S* planes = static_cast<const S*>(src);
            if (C == 1) {
                cons_partial_kernel<Lat, S, false>
                    <<<a.cons_nitems, CONS_THREADS, 0, a.stream>>>(planes, a.inst, a.cons_items, a.pulled, o1, a.rho0,
                                                                   a.cons_nitems == a.count ? o0 : nullptr);
                if (a.cons_nitems == a.count) break;
            } else {
                cudaLaunchAttribute attr[1];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = 1;
                attr[0].val.clusterDim.y = C;
                attr[0].val.clusterDim.z = 1;
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)a.cons_nitems, C);
                cfg.blockDim = dim3(CONS_THREADS);
                cfg.stream = a.stream;
                cfg.attrs = attr;
                cfg.numAttrs = 1;
                const cudaError_t e = cudaLaunchKernelEx(&cfg, &cons_partial_kernel<Lat, S, true>, planes, a.inst,
                                                         a.cons_items, a.pulled, o1, a.rho0, (double*)nullptr);
                if (e != cudaSuccess) return e;
            }
            cons_final_kernel<<<(a.count + 3) / 4, 128, 0, a.stream>>>(o1, a.inst, a.count, (int)sizeof(S), a.rho0, o0);
            break;
        }
        case AuxOp::CollideInPlace: {
            if (a.compute == DT_F64) {
                if constexpr (std::is_same<S, double>::value)
                    return collide_inplace_by_rule<Lat, S, double>(a, src, dst);
                return cudaErrorInvalidValue;
            }
            return collide_inplace_by_rule<Lat, S, float>(a, src, dst);
        }
    }
    return cudaGetLastError();
}

template <class Lat>
cudaError_t aux_by_storage(AuxOp op, const AuxArgs& a, const void* src, void* dst, const double* p0,
                           const double* p1, const double* p2, double* o0, double* o1, double* o2) {
    switch (a.storage) {
        case DT_F64: return aux_dispatch<Lat, double>(op, a, src, dst, p0, p1, p2, o0, o1, o2);
        case DT_F32: return aux_dispatch<Lat, float>(op, a, src, dst, p0, p1, p2, o0, o1, o2);
        case DT_F16: return aux_dispatch<Lat, __half>(op, a, src, dst, p0, p1, p2, o0, o1, o2);
        case DT_BF16:
            return aux_dispatch<Lat, __nv_bfloat16>(op, a, src, dst, p0, p1, p2, o0, o1, o2);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t run_aux(AuxOp op, const AuxArgs& a, const void* src, void* dst, const double* p0,
                    const double* p1, const double* p2, double* o0, double* o1, double* o2) {
    if (a.lattice == 2) return aux_by_storage<D2Q9>(op, a, src, dst, p0, p1, p2, o0, o1, o2);
    return aux_by_storage<D1Q3>(op, a, src, dst, p0, p1, p2, o0, o1, o2);
}

}  // namespace lbm
