// lbm_f64.cuh -- FP64 building blocks of the collision rules: reciprocal,
// logarithm, sign / finiteness tests, and the MinxEnt rules written for
// GB300's narrow FP64 pipe.
//
// GB300 issues two FP64 lane operations per clock and SM (629 G/s at
// 2.07 GHz x 152), so an FP64 step costs its FP64 instruction count and
// little else: everything that can run on the integer pipe does, and the
// functions below spend as few FP64 instructions as their precision allows.
#pragma once
#include "lbm_common.cuh"
#include "lbm_num.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// Natural logarithm, table driven (P. T. P. Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point
// arithmetic", ACM TOMS 16, 1990) with accurate tables (S. Gal, "Computing
// elementary functions: a new approach for achieving high accuracy and good
// performance", LNCS 235, 1986): for y = 1 + delta in [1/4, 4) the leading
// 10 mantissa bits select a rational rc close to 1/y, then
//     ln y = ln(1/rc) + ln(1 + r),  r = y rc - 1 = delta rc + (rc - 1),
// |r| <= 2^-10, by the Taylor series to r^6 (remainder below 2^-62 of r).
// Of the rc near 1/y the table holds the one whose ln(1/rc) lies closest to
// an FP64 number (0.04 ulp off on average instead of 0.25), which costs nothing
// here and leaves one rounding where |ln y| is large against r.  rc is 1 in
// the two intervals that touch y = 1, so ln y keeps its relative precision
// for small delta.  The terms from r^4 on, r^4 (-1/4 + r/5 - r^2/6), have
// their bracket in FP32: its rounding is below 2^-56 of r.  rc and rc - 1
// have at most 17 significant bits, so that their high words alone are
// stored.  6 FP64 instructions and one 16-byte table read, where the
// library's log1p takes about 25.
//
// Relative error in units of 2^-53, largest / rms over 2^20 values (the
// library's log1p in brackets): delta in (-3/4, 3) 2.0 / 0.445 (2.6 / 0.608),
// [1/4, 1/2] 1.4 / 0.442 (1.5 / 0.482), [2^-5, 2^-4] 1.06 / 0.414
// (1.06 / 0.416); worst in the binade that meets the intervals of rc = 1,
// [2^-10, 2^-9] 2.0 / 0.482 (1.0 / 0.408), where the rounding of r counts.  With rc at
// the intervals' centres it was 2.8 / 0.6 to 0.7 nearly everywhere.
// ---------------------------------------------------------------------------
constexpr int LOG_BITS = 10, LOG_HALF = 1 << LOG_BITS;  // intervals of an octave
constexpr int LOG_GRID = 1 << 14;                        // rc = j / (2^(k + 1) LOG_GRID), k: octave of y
struct alignas(16) LogEntry {
    double lc;           // ln(1 / rc)
    uint32_t rc, rm;     // high words of rc and rc - 1 (low words are 0)
};
struct LogTable {
    LogEntry e[4 * LOG_HALF];  // octaves [1/4, 1/2), [1/2, 1), [1, 2), [2, 4) of y
};

// High word of j / 2^sh as a double (|j| < 2^20).
constexpr uint32_t ratio_high_word(int j, int sh) {
    if (j == 0) return 0u;
    uint32_t m = (uint32_t)(j < 0 ? -j : j);
    int top = 0;
    while ((m >> top) > 1u) ++top;
    return (j < 0 ? 0x80000000u : 0u) | ((uint32_t)(1023 + top - sh) << 20) | ((m << (20 - top)) & 0xfffffu);
}

// a + b as hi + lo exactly (Knuth's two-sum)
struct DoubleDouble {
    double hi, lo;
};
constexpr DoubleDouble two_sum(double a, double b) {
    const double s = a + b, v = s - a;
    return {s, (a - (s - v)) + (b - v)};
}

// ln(2 G / j), j = G .. 2 G (G = LOG_GRID), as sums of ln((k + 1) / k) =
// 2 atanh(1 / (2 k + 1)), each term a short series, summed in double-double.
struct LogGrid {
    DoubleDouble v[LOG_GRID + 1];  // index j - G
};
constexpr LogGrid make_log_grid() {
    constexpr int G = LOG_GRID;
    LogGrid t{};
    for (int k = 2 * G - 1; k >= G; --k) {
        const double n = 2.0 * k + 1.0, z = 1.0 / n, z2 = z * z;
        // z = fl(1 / n); its rounding error is (1 - n z) / n, with n z split
        // exactly: n < 2^17, z cut to its upper 26 bits
        const double big = z * 134217729.0;  // Veltkamp split, 2^27 + 1
        const double zh = big - (big - z), zl = z - zh;
        const double ze = ((1.0 - n * zh) - n * zl) * z;
        // z^3 / 3 + z^5 / 5 + z^7 / 7 (z < 2^-15: the next term is below 2^-120 z)
        const double s = ((1.0 / 7.0 * z2 + 1.0 / 5.0) * z2 + 1.0 / 3.0) * z2 * z;
        const DoubleDouble p = t.v[k + 1 - G];
        const DoubleDouble q = two_sum(p.hi, 2.0 * z);
        t.v[k - G] = two_sum(q.hi, q.lo + (p.lo + 2.0 * (ze + s)));
    }
    return t;
}

constexpr LogTable make_log_table() {
    constexpr int H = LOG_HALF, G = LOG_GRID;
    const LogGrid ln = make_log_grid();
    LogTable t{};
    for (int i = 0; i < H; ++i) {
        const double c = 1.0 + (i + 0.5) / H;  // centre of the interval of m, y = 2^k m
        const int centre = (int)(2.0 * G / c + 0.5);
        for (int o = 0; o < 4; ++o) {
            const int k = o - 2;
            // rc = 1 right of y = 1 and left of it
            const bool at_one = (k == 0 && i == 0) || (k == -1 && i == H - 1);
            int best = at_one ? (k == 0 ? 2 * G : G) : centre;
            // others within 2^-12 of the centre: |r| stays below 2^-10
            const int reach = at_one ? 0 : centre >> 12;
            double least = 1e300, lc = 0.0;
            for (int j = centre - reach; j <= centre + reach; ++j) {
                const int jj = at_one ? best : j;
                if (jj < G || jj > 2 * G) continue;
                const DoubleDouble a = two_sum(ln.v[jj - G].hi, k * ln.v[0].hi);
                const DoubleDouble b = two_sum(a.hi, a.lo + (ln.v[jj - G].lo + k * ln.v[0].lo));
                // in units of the logarithm itself
                const double off = b.hi == 0.0 ? 0.0 : (b.lo < 0 ? -b.lo : b.lo) / (b.hi < 0 ? -b.hi : b.hi);
                if (off < least) {
                    least = off;
                    best = jj;
                    lc = b.hi;
                }
            }
            LogEntry& u = t.e[o * H + i];
            u.lc = lc;
            u.rc = ratio_high_word(best, 15 + k);
            u.rm = ratio_high_word(best - (k >= 0 ? (2 * G) << k : (2 * G) >> -k), 15 + k);
        }
    }
    return t;
}

static __device__ const LogTable LOG_TABLE = make_log_table();

// ln(1/rc) + ln(1 + r) of table entry i, for the deviation of a y in its interval
__device__ __forceinline__ double log_entry(uint32_t i, double delta) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(&LOG_TABLE.e[i]));
    const double r = fma(delta, __hiloint2double(e.z, 0), __hiloint2double(e.w, 0));
    // r in FP32 from its high word (2^-20 relative): the upper exponent bits
    // of |r| < 1 are dropped; a tiny r maps to some value below 2, which its
    // factor r^4 makes irrelevant
    const uint32_t rh = (uint32_t)__double2hiint(r);
    const float rf = __uint_as_float(((rh << 3) & 0x3fffffffu) | (rh & 0x80000000u));
    // t = 1/4 - r/5 + r^2/6, positive and near 1/4: widened by its bits
    const uint32_t tb = __float_as_uint(__fmaf_rn(rf, __fmaf_rn(rf, 1.f / 6.f, -0.2f), 0.25f));
    const double t = __hiloint2double((int)((tb >> 3) + 0x38000000u), (int)(tb << 29));
    const double q = fma(r, fma(-r, t, 1.0 / 3.0), -0.5);
    return __hiloint2double(e.y, e.x) + fma(r * r, q, r);
}

// Outside [1/4, 4): the library's.  Not inlined: FP64 instructions hold the
// pipe even where their predicate is off.
__device__ __noinline__ static double log1p_outside(double delta) { return log1p(delta); }

// ln(1 + delta), given delta and y = 1 + delta rounded
__device__ __forceinline__ double log1p_f64(double delta, double y) {
    const uint32_t i = ((uint32_t)__double2hiint(y) - 0x3fd00000u) >> (20 - LOG_BITS);
    if (i >= 4u * LOG_HALF) return log1p_outside(delta);
    return log_entry(i, delta);
}

// ---------------------------------------------------------------------------
// Tests on the high words (integer pipe); a test that cannot decide there
// falls back to the FP64 comparison it stands for.
// ---------------------------------------------------------------------------
// min over the finite numbers y of y > 0, as fmin and a compare decide it
template <int N> __device__ __forceinline__ bool all_positive(const double (&y)[N]) {
    int lo = 0x7fffffff, hi = 0;
#pragma unroll
    for (int a = 0; a < N; ++a) {
        lo = min(lo, __double2hiint(y[a]));
        hi = max(hi, __double2hiint(y[a]));
    }
    if (lo > 0 && hi < 0x7ff00000) return true;  // positive, finite
    double mn = y[0];
#pragma unroll
    for (int a = 1; a < N; ++a) mn = fmin(mn, y[a]);
    return mn > 0.0;
}

// Stability criterion of Sec. IV.H on f^post_a = W_a rho0 + out_a: every
// population >= 0 and the sum of the deviations below 1e30 in magnitude.
// A negative double orders as an unsigned integer by magnitude, so a high
// word below that of -W_a rho0 (unsigned) means out_a > -W_a rho0, and high
// words below 2^96's (signed) bound the sum.
template <int Q>
__device__ __forceinline__ bool finite_nonneg_f64(const double (&out)[Q], const double (&w)[Q],
                                                  double rho0) {
    bool ok = true;
    int big = 0;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const int h = __double2hiint(out[a]);
        ok = ok && ((uint32_t)h < (uint32_t)__double2hiint(-w[a] * rho0));
        big = max(big, h);
    }
    if (ok && big < 0x45f00000 && rho0 < 0x1p90) return true;
    bool good = true;
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        good = good && (out[a] >= -w[a] * rho0);
        s += out[a];
    }
    return good && (fabs(s) < 1e30);
}

// ---------------------------------------------------------------------------
// D2Q9 MinxEnt collision of one node in FP64 (NFREE = 4: MinxEnt4 with free
// M2, M3, M5, M7; NFREE = 2: MinxEnt2 with free M2, M3).  Start point and
// deviation variables as in lbm_collide.cuh; the Newton system is set up in
// the basis
//     n2 = (-2 | 0 0 0 0 | 1/2 1/2 1/2 1/2),   n3 = (-4 | 1 1 1 1 | 0 0 0 0),
//     nx = (0 | -1 0 1 0 | 1/2 -1/2 -1/2 1/2), ny = (0 | 0 -1 0 1 | 1/2 1/2 -1/2 -1/2)
// (rest | axis | diagonal) of the free subspace, which spans the same space
// as the rows e, eps, q_x, q_y of T and couples rest, axis and diagonal
// populations as little as possible: with y_a = p_a / W_a = c +- h for the
// opposite pairs and r = 1 / (y_a y_opp(a)), the half sum and half
// difference of 1/y over a pair are c r and -+ h r, and A / 18 is
//     [ q0/2 + Sd   q0         X57 - X68    X57 + X68 ]
//     [ q0          2 q0 + Sa  -X13         -X24      ]
//     [ .           .          C13 + Sd     C57 - C68 ]
//     [ .           .          .            C24 + Sd  ],
// C = c r, X = -h r, Sa = C13 + C24, Sd = C57 + C68, q0 = 1 / y_0.
// 252 FP64 instructions per node (MinxEnt4), against 485 with log1p, IEEE
// divisions and the system in the rows of T.
// ---------------------------------------------------------------------------
template <int NFREE>
__device__ __forceinline__ uint32_t minxent_f64(const double (&d)[9], double rho0, double omega,
                                                double omega2, double (&out)[9]) {
    using N = Num<double>;
    constexpr double W[9] = {4.0 / 9.0,  1.0 / 9.0,  1.0 / 9.0,  1.0 / 9.0, 1.0 / 9.0,
                             1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0};
    const double n13 = d[1] + d[3], n24 = d[2] + d[4], n57 = d[5] + d[7], n68 = d[6] + d[8];
    const double drho = (d[0] + (n13 + n24)) + (n57 + n68);
    const double a57 = d[5] - d[7], a86 = d[8] - d[6];
    const double m13 = d[1] - d[3], m24 = d[2] - d[4];
    const double jx = m13 + a57 + a86, jy = m24 + a57 - a86;
    const double rho = rho0 + drho;
    const double ir = N::rcp(rho);
    const double ux = jx * ir, uy = jy * ir;
    const double uyy = uy * uy, uxy = ux * uy;
    const double U2 = fma(ux, ux, uyy), D2 = fma(ux, ux, -uyy);
    // relaxed stress, even parts s of the pairs (mean of delta), odd parts h
    const double k = 1.0 - omega;
    const double G = fma(k, fma(n13 - n24, ir, -D2), D2);
    const double P = fma(k, fma(n57 - n68, ir, -uxy), uxy);
    const double F = 0.75 * U2, E = 3.0 * U2;
    const double sx = fma(2.25, G, F), sy = fma(-2.25, G, F);
    const double sp = fma(9.0, P, E), sm = fma(-9.0, P, E);
    // (odd parts 3 l, so that delta = s +- 3 l rounds once: with 3 l rounded
    // before the sum the collision's error against exact arithmetic was 5 %
    // above that of the plain rule, now it is 1 % below)
    double lx = ux, ly = uy, lp = ux + uy, lm = uy - ux;
    if constexpr (NFREE == 2) {
        // relaxed heat flux g = (omega2 - 1) Q / rho on the odd parts
        const double g = (omega2 - 1.0) * ir;
        const double gx = g * fma(-2.0, a57 + a86, m13), gy = g * fma(-2.0, a57 - a86, m24);
        lx = fma(-0.5, gx, lx);
        ly = fma(-0.5, gy, ly);
        lp += gx + gy;
        lm += gy - gx;
    }
    const double del[9] = {-1.5 * U2,          fma(3.0, lx, sx),  fma(3.0, ly, sy),
                           fma(-3.0, lx, sx),  fma(-3.0, ly, sy), fma(3.0, lp, sp),
                           fma(3.0, lm, sm),   fma(-3.0, lp, sp), fma(-3.0, lm, sm)};
    double y[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) y[a] = 1.0 + del[a];
    const bool ok = all_positive(y);  // the logarithms exist (reading C-NEG)

    const double r13 = N::rcp(y[1] * y[3]), r24 = N::rcp(y[2] * y[4]);
    const double r57 = N::rcp(y[5] * y[7]), r68 = N::rcp(y[6] * y[8]);
    const double q0 = N::rcp(y[0]);
    const double C13 = fma(sx, r13, r13), C24 = fma(sy, r24, r24);
    const double C57 = fma(sp, r57, r57), C68 = fma(sm, r68, r68);
    const double Sd = C57 + C68;
    const double a22 = fma(0.5, q0, Sd), a33 = fma(2.0, q0, C13 + C24);
    const double L0 = log1p_f64(del[0], y[0]);
    double x2, x3, xx = 0.0, xy = 0.0;
    if constexpr (NFREE == 4) {
        double L[9];
#pragma unroll
        for (int a = 1; a < 9; ++a) L[a] = log1p_f64(del[a], y[a]);
        const double l57 = L[5] - L[7], l68 = L[6] - L[8];
        const double b2 = fma(-2.0, L0, 0.5 * ((L[5] + L[7]) + (L[6] + L[8])));
        const double b3 = fma(-4.0, L0, (L[1] + L[3]) + (L[2] + L[4]));
        const double bx = fma(0.5, l57 - l68, L[3] - L[1]);
        const double by = fma(0.5, l57 + l68, L[4] - L[2]);
        const double X57 = (-3.0 * lp) * r57, X68 = (-3.0 * lm) * r68;
        spd4_solve<double>(a22, q0, a33, X57 - X68, (3.0 * lx) * r13, C13 + Sd, X57 + X68, (3.0 * ly) * r24,
                           C57 - C68, C24 + Sd, b2, b3, bx, by, x2, x3, xx, xy);
    } else {
        // logarithms of the axis and diagonal products: y_a y_opp - 1 =
        // s (2 + s) - h^2 = m, and (1 + m)(1 + m') - 1 = m + m' + m m'
        const double hx = 3.0 * lx, hy = 3.0 * ly, hp = 3.0 * lp, hm = 3.0 * lm;
        const double e13 = fma(sx, 2.0 + sx, -(hx * hx)), e24 = fma(sy, 2.0 + sy, -(hy * hy));
        const double e57 = fma(sp, 2.0 + sp, -(hp * hp)), e68 = fma(sm, 2.0 + sm, -(hm * hm));
        const double ma = fma(e13, e24, e13 + e24), md = fma(e57, e68, e57 + e68);
        const double b2 = fma(-2.0, L0, 0.5 * log1p_f64(md, 1.0 + md));
        const double b3 = fma(-4.0, L0, log1p_f64(ma, 1.0 + ma));
        const double idet = N::rcp(fma(a22, a33, -(q0 * q0)));
        x2 = fma(a33, b2, -(q0 * b3)) * idet;
        x3 = fma(a22, b3, -(q0 * b2)) * idet;
    }
    if (!ok) x2 = x3 = xx = xy = 0.0;  // keep p^start
    // f^post_a - W_a rho0 = W_a [drho + rho (delta_a - v_a)], v = (-(x2 + 2 x3)/4 |
    // (x3 -+ xx)/2, (x3 -+ xy)/2 | x2 +- (xx + xy), x2 -+ (xx - xy))
    double e[9];
    e[0] = fma(0.25, fma(2.0, x3, x2), del[0]);
    if constexpr (NFREE == 4) {
        const double p = xx + xy, m = xx - xy;
        e[1] = fma(-0.5, x3 - xx, del[1]);
        e[3] = fma(-0.5, x3 + xx, del[3]);
        e[2] = fma(-0.5, x3 - xy, del[2]);
        e[4] = fma(-0.5, x3 + xy, del[4]);
        e[5] = del[5] - (x2 + p);
        e[7] = del[7] - (x2 - p);
        e[6] = del[6] - (x2 - m);
        e[8] = del[8] - (x2 + m);
    } else {
#pragma unroll
        for (int a = 1; a < 5; ++a) e[a] = fma(-0.5, x3, del[a]);
#pragma unroll
        for (int a = 5; a < 9; ++a) e[a] = del[a] - x2;
    }
#pragma unroll
    for (int a = 0; a < 9; ++a) out[a] = fma(W[a] * rho, e[a], W[a] * drho);
    return (ok ? 0u : ST_NEWTON_SKIPPED) |
           (finite_nonneg_f64<9>(out, W, rho0) ? 0u : ST_UNSTABLE);
}

}  // namespace lbm
