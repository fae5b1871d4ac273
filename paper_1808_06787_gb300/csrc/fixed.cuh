// The FP64 collision of binary and ternary mixtures in 64-bit fixed point.
//
// GB300 issues one FP64 warp instruction in 16 clocks per SM, as long as 64 integer or
// FP32 ones, and the collision takes 116 (D2Q5) to 150 (D3Q7) of them per node, which
// bounded every FP64 step.  Sums of fixed-point numbers cost two integer instructions and
// are exact, and a product of two 60-bit numbers takes three 32 x 32 -> 64 multiplies, so
// the same arithmetic runs on the integer pipes several times faster, and with half the
// error (rms 0.9e-16 of a population against 1.8e-16).  Measured, us per step, FP64 ->
// fixed point: ternary D2Q5 128^2 5.77 -> 3.02, 200^2 12.35 -> 4.48, 1024^2 232 -> 56;
// D3Q7 101 x 96 x 67 189 -> 45.5; D2Q9 300^2 42 -> 11.4; binary D2Q5 240 x 40 3.18 -> 1.87.
// The large grids are bound by the integer and FP64 pipes together (D3Q7 101 x 96 x 67: ALU 69 %,
// FP64 50 % busy, 64 % of the issue slots), the small ones by the latency of a step.
//
//   populations  each species' populations at a node are integers X in units of 2^-58 of
//                the power of two above the largest of them (a block exponent M), so a
//                trace species keeps its relative precision; those down to 2^-5 of the
//                largest are exact, and every sum is exact
//   matrices     all entries are linear in the mole fractions (below), taken in units of
//                2^-57; the reciprocals come from an FP32 seed and two Newton steps
//   products     rounded to about half a unit (2^-59; a double's half ulp is 2^-53 to 2^-54)
//   results      rounded once to double, ties to even
//
// Ternary matrices.  With a = 1/(2 D_13), b = 1/(2 D_23), c = 1/(2 D_12), k = 1/c_s^2 and
// A = a + k, B = b + k, C = c + k, Eqs. 2-10 and 3-26 give for xi_1 + xi_2 + xi_3 = 1
//   det K = A B xi_3 + A C xi_1 + B C xi_2,
//   N_11  = a B xi_3 + a C xi_1 + c B xi_2,   N_12 = k (a - c) xi_1,
//   N_22  = A b xi_3 + A c xi_1 + b C xi_2,   N_21 = k (b - c) xi_2,
//   Lambda_1/2 = N / det K =: h,  lambda_2/2 = (1 - h_ii) / (1 - h_ii / 4)  (Eq. 3-16),
// sums of positive terms without cancellation.  For binary mixtures both matrices are
// constants.
//
// A node whose numbers do not fit (a population of one or more, in ternary mixtures a
// moving one of a half or more, a mole fraction outside [-1/16, 17/16], a magnitude below
// 2^-900, infinities, NaN) takes the FP64 arithmetic of node.cuh; so does a solver whose diffusivities spread too far for the bits above
// (fixed_table).  The functions are plain integer C++, the same on the host.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "lbms.h"

namespace lbms {

#ifdef __CUDACC__
#define LBMS_HD __host__ __device__ __forceinline__
#else
#define LBMS_HD inline
#endif

namespace fx {

constexpr int kUnit = 57;                       // fraction bits of the mole fractions
constexpr int64_t kOne = int64_t(1) << kUnit;
constexpr int64_t kLimit = int64_t(1) << 61;    // of the first factor of a product (X)

LBMS_HD uint64_t bits_of(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t b;
    memcpy(&b, &v, 8);
    return b;
#endif
}
LBMS_HD double double_of(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}
LBMS_HD int clz64(uint64_t v)  // 64 for zero
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
LBMS_HD float seed(float d)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
#else
    return 1.0f / d;
#endif
}
LBMS_HD int64_t wide(int32_t a, int32_t b) { return (int64_t)a * b; }
LBMS_HD int32_t hi32(int64_t v) { return (int32_t)(v >> 32); }

// The two factors of a product: x (|x| < 2^61) in 30-bit halves, and a coefficient c
// (|c| < 2^59) in 28-bit ones, so that
//   x c / 2^58 = h ch + (h cl4 + l ch) / 2^30 + (less than one)
struct X {
    int32_t h, l;
};
struct Cf {
    int32_t h, l4;
};
LBMS_HD X split(int64_t x) { return {(int32_t)(x >> 30), (int32_t)((uint32_t)x & 0x3fffffffu)}; }
LBMS_HD Cf coef(int64_t c) { return {(int32_t)(c >> 28), (int32_t)(((uint32_t)c << 2) & 0x3fffffffu)}; }

// half a unit to round to nearest, and the mean of what is dropped
constexpr int64_t kHalf = (int64_t(1) << 29) + (int64_t(1) << 28);
LBMS_HD int64_t mul(X a, Cf p) { return wide(a.h, p.h) + ((kHalf + wide(a.h, p.l4) + wide(a.l, p.h)) >> 30); }
LBMS_HD int64_t dot(X a, Cf p, X b, Cf q)
{
    return wide(a.h, p.h) + wide(b.h, q.h) + ((kHalf + wide(a.h, p.l4) + wide(a.l, p.h) + wide(b.h, q.l4) + wide(b.l, q.h)) >> 30);
}
LBMS_HD int64_t dot(X a, Cf p, X b, Cf q, X c, Cf r)
{
    return wide(a.h, p.h) + wide(b.h, q.h) + wide(c.h, r.h) +
           ((kHalf + wide(a.h, p.l4) + wide(a.l, p.h) + wide(b.h, q.l4) + wide(b.l, q.h) + wide(c.h, r.l4) + wide(c.l, r.h)) >> 30);
}

// 2^120 / d for d in [2^61, 2^62): 1/d of d in units of 2^-62, in units of 2^-58 (at most
// 2^59 - 1), to about one unit.
LBMS_HD int64_t reciprocal(int64_t d)
{
    const int32_t dh = hi32(d);                       // [2^29, 2^30)
    const uint32_t dl = (uint32_t)d;
    const float s = seed((float)dh) * 0x1p59f;        // y0 in units of 2^-29: (2^29, 2^30]
    const int32_t y0 = (int32_t)s;
    // 1 - d y0 in units of 2^-59, |.| < 2^38
    const int64_t e0 = (int64_t(1) << 59) - (wide(dh, y0) + (int64_t)(((uint64_t)dl * (uint32_t)y0) >> 32));
    // y1 = y0 + y0 e0 in units of 2^-61
    const int64_t y1 = ((int64_t)y0 << 32) + (wide(y0, (int32_t)(e0 >> 8)) >> 19);
    // 1 - d y1 modulo 2^-27, in units of 2^-91, then of 2^-71
    const uint32_t yl = (uint32_t)y1, yh = (uint32_t)((uint64_t)y1 >> 32);
    uint64_t p = (((uint64_t)dl * yl) >> 32) + (uint64_t)dl * yh + (uint64_t)(uint32_t)dh * yl;
    p += (uint64_t)((uint32_t)dh * yh) << 32;
    const int32_t e1 = (int32_t)((int64_t)(0 - p) >> 20);
    const int64_t y2 = y1 + (wide((int32_t)yh, e1) >> 39);
    const int64_t y = (y2 + 4) >> 3;
    const int64_t top = (int64_t(1) << 59) - 1;
    return y < top ? y : top;
}

// A species' populations: X_k = f_k 2^(1022 + bits - M), M the largest exponent field: the
// largest is 2^(bits - 1) to 2^bits.  bits is 58, or 59 on D2Q9, whose smallest equilibrium
// is a sixteenth of the largest.
struct Block {
    int M;        // exponent field of the largest population (0: all are zero)
    uint32_t up;  // what the scaling adds to the upper word of a double
    int right;    // shift from these units to units of 2^-57
};
template <typename L>
constexpr int block_bits()
{
    return L::Q == 9 ? 59 : 58;
}

// Bounds of a ternary node's numbers.  The departures of one species enter the other's
// results as coefficients, below two in magnitude in units of 2^-58 of one, and every result
// has to stay below 2^63.  With moving populations below a half (exponent field 1021) the even
// and odd departures are below 1 + 2 w (17/16) <= 1.54 and 1, and with the sum below 2^62 and
// Lambda_12/2 below 2^61 in the species' units, for the weights of each lattice
//   |f_k| + |even| lambda_2/2 + |odd| Lambda_1/2 + |Lambda_12/2| (1.54 + 1)  < 7.5 2^60,
//   |f_0| + 2 |w_0 sum - f_0| lambda_2/2 + 2 |Lambda_12/2| |w_0 xi - f_0|    < 7.5 2^60
// (f_0: the rest population).  On D2Q9, whose numbers have one bit more, the rest
// population takes part in the limit and the sum is below 2^61 (at equilibrium it is 2.25 of
// the largest population, 2^60.2).
template <typename L>
LBMS_HD bool fits_pair(uint32_t rest, uint32_t moving, int64_t half)
{
    if (block_bits<L>() == 58) return (int)(moving >> 20) <= 1021;
    return (int)((rest > moving ? rest : moving) >> 20) <= 1021 && half < kLimit / 2 && half > -kLimit / 2;
}

// Whether a species' largest exponent field serves as its block exponent; 0 where every
// population is zero, but not where some are subnormal.
template <int Q>
LBMS_HD bool fits_block(int M, const double (&f)[Q])
{
    if (M != 0) return M >= 120 && M <= 1022;
    uint64_t any = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) any |= bits_of(f[k]);
    return (any << 1) == 0;
}

LBMS_HD Block block(int M, int bits)
{
    const int r = 965 + bits - M;
    return {M, M == 0 ? 0u : (uint32_t)(1022 + bits - M) << 20, r < 63 ? r : 63};
}
// Conversions, by an instruction of the FP64 pipe (16 clocks per SM; scaling by a power of
// two is an integer addition to the exponent, and a zero's exponent field stays below
// that of 1/2, for M >= 120 or M = 0) or by some 14 integer instructions.  Ternary nodes
// convert every second population either way, so that the pipes share the work (D3Q7
// 101 x 96 x 67: all by the first 46.1 us per step, all by the second 48.9, shared 45.5;
// D2Q9 300^2 12.6, 12.4 and 11.4); binary nodes, whose steps wait rather than work, take the
// integer form (D2Q5 240 x 40: 2.14 and 1.87).
LBMS_HD int64_t to_fixed(double f, const Block& s, int bits, bool integer)
{
    if (integer) {
        const uint64_t b = bits_of(f);
        const uint32_t h = (uint32_t)(b >> 32);
        const uint64_t m = ((uint64_t)((h & 0xfffffu) | 0x100000u) << 32 | (uint32_t)b) << 9;
        // from 61, where the leading bit is, to bits - 1 - (M - e)
        int r = (s.M == 0 ? 63 : s.M + 62 - bits) - (int)((h >> 20) & 0x7ffu);
        r = r < 63 ? r : 63;
        const int64_t x = (int64_t)((m + ((uint64_t(1) << r) >> 1)) >> r);  // to nearest
        const int64_t neg = (int64_t)b >> 63;
        return (x ^ neg) - neg;
    }
    const double v = double_of(bits_of(f) + ((uint64_t)s.up << 32));
#ifdef __CUDA_ARCH__
    return __double2ll_rn(v);
#else
    return llrint(v);
#endif
}
LBMS_HD int64_t to_abs(int64_t x, const Block& s) { return x >> s.right; }
// The same as a coefficient, in units of 2^-58 (right is at least 1, as M <= 1022).
LBMS_HD Cf coef_of_abs(int64_t x, const Block& s) { return coef(x >> (s.right - 1)); }
// The double nearest to x; delta receives (that double - x), in units of x.
LBMS_HD double to_double(int64_t x, const Block& s, int32_t& delta)
{
#ifdef __CUDA_ARCH__
    const double v = __ll2double_rn(x);
#else
    const double v = (double)x;
#endif
    const uint64_t b = bits_of(v);
    // |v| = (53-bit mantissa) 2^sh, rounded where sh > 0 (sh <= 10): the lower words tell by how much
    const int sh = (int)((uint32_t)(b >> 52) & 0x7ffu) - 1075;
    const int32_t neg = (int32_t)(x >> 63);
    const int32_t t = (int32_t)((uint32_t)b << (sh & 31));
    delta = sh > 0 ? ((t ^ neg) - neg) - (int32_t)x : 0;
    return double_of(x != 0 ? b - ((uint64_t)s.up << 32) : 0);
}

}  // namespace fx

// Coefficients of a solver's matrices (see the header comment); on == 0: not applicable.
struct FixedTable {
    int on;
    int srt;
    fx::Cf det[3], n11[3], n22[3];  // of (xi_3, xi_1, xi_2), over a common scale
    fx::Cf g1, g2;                  // k (a - c) / 4 and k (b - c) / 4 over the same scale
    fx::Cf l1, l2;                  // binary mixtures: Lambda_1/2 and Lambda_2/2
};

// invD: 1/D_ij of the n = S + 1 species.
inline FixedTable fixed_table(int n, const double (&invD)[LBMS_MAX_SPECIES][LBMS_MAX_SPECIES], double cs2, int relax)
{
    FixedTable t;
    memset(&t, 0, sizeof(t));
    if (n > 3 || (relax != LBMS_RELAX_MAGIC && relax != LBMS_RELAX_SRT)) return t;
    t.srt = relax == LBMS_RELAX_SRT;
    const double q = 288230376151711744.0;  // 2^58
    auto cf = [&](long double v) { return fx::coef((int64_t)(v * q + (v < 0 ? -0.5L : 0.5L))); };
    const long double k = 1.0L / cs2;
    if (n == 2) {
        const long double c = 0.5L * invD[0][1], h = c / (c + k);
        if (!(h >= 0x1p-4L)) return t;
        t.l1 = cf(h);
        t.l2 = t.srt ? t.l1 : cf((1.0L - h) / (1.0L - h / 4.0L));
        t.on = 1;
        return t;
    }
    const long double a = 0.5L * invD[0][2], b = 0.5L * invD[1][2], c = 0.5L * invD[0][1];
    const long double A = a + k, B = b + k, C = c + k;
    const long double det[3] = {A * B, A * C, B * C};
    const long double n11[3] = {a * B, a * C, c * B}, n22[3] = {A * b, A * c, b * C};
    long double top = 0.0L, low = 1e300L;
    for (int i = 0; i < 3; ++i) {
        top = det[i] > top ? det[i] : top;
        low = det[i] < low ? det[i] : low;
    }
    // det K keeps 53 bits (its smallest coefficient at least 2^-4 of the largest), and
    // Lambda_1 is not small (1/(2 D) at least k/8)
    const long double least = a < b ? (a < c ? a : c) : (b < c ? b : c);
    if (!(low * 16.0L >= top) || !(least * 8.0L >= k)) return t;
    const long double s = 1.875L / top;
    for (int i = 0; i < 3; ++i) {
        t.det[i] = cf(det[i] * s);
        t.n11[i] = cf(n11[i] * s);
        t.n22[i] = cf(n22[i] * s);
    }
    const long double g1 = k * (a - c) * s / 4.0L, g2 = k * (b - c) * s / 4.0L;
    if (!(g1 < 0.5L && g1 > -0.5L && g2 < 0.5L && g2 > -0.5L)) return t;
    t.g1 = cf(g1);
    t.g2 = cf(g2);
    t.on = 1;
    return t;
}

// One node's collision: f in the lattice's device order (K0 rest populations, then opposite
// pairs; weights w).  False where the node does not fit (f unchanged).
template <typename L, int S>
LBMS_HD bool collide_fixed(double (&f)[S][L::Q], const FixedTable& t)
{
    using namespace fx;
    constexpr int Q = L::Q;
    static_assert(S == 1 || S == 2, "binary and ternary mixtures");
    Block e[S];
    int64_t x[S][Q], sum[S], half[S], xi[S];
    bool fits = true;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        uint32_t rest = 0, moving = 0;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const uint32_t h = (uint32_t)(bits_of(f[s][k]) >> 32) & 0x7fffffffu;
            uint32_t& most = k < L::K0 ? rest : moving;
            most = h > most ? h : most;
        }
        const uint32_t top = rest > moving ? rest : moving;
        e[s] = block((int)(top >> 20), block_bits<L>());
        fits &= fits_block(e[s].M, f[s]);
        int64_t a = 0;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            x[s][k] = to_fixed(f[s][k], e[s], block_bits<L>(), S == 1 || (k & 1) != 0);
            a += x[s][k];
        }
        half[s] = a >> 1;
        sum[s] = a;
        xi[s] = to_abs(a, e[s]);
        fits &= half[s] < kLimit && half[s] > -kLimit;
        if (S == 2) fits &= fits_pair<L>(rest, moving, half[s]);
        fits &= (uint64_t)(xi[s] + kOne / 16) <= (uint64_t)(kOne + kOne / 8);
    }
    Cf l1[S], l2[S];
    X q1, q2;  // Lambda_12 / 2 and Lambda_21 / 2 in the units of species 1 and 2
    if (S == 1) {
        l1[0] = t.l1;
        l2[0] = t.l2;
    } else {
        const int64_t x3 = kOne - xi[0] - xi[S - 1];
        fits &= (uint64_t)(x3 + kOne / 16) <= (uint64_t)(kOne + kOne / 8);
        const X a = split(x3), b = split(xi[0]), c = split(xi[S - 1]);
        const int64_t det = dot(a, t.det[0], b, t.det[1], c, t.det[2]);
        const int64_t n1 = dot(a, t.n11[0], b, t.n11[1], c, t.n11[2]);
        const int64_t n2 = dot(a, t.n22[0], b, t.n22[1], c, t.n22[2]);
        fits &= det > kOne / 32 && n1 > 0 && n2 > 0 && n1 < det && n2 < det;
        if (!fits) return false;
        const int up = clz64((uint64_t)det) - 2;  // det to [2^61, 2^62)
        const int64_t y = reciprocal(det << up);
        const Cf yc = coef(y);
        // h in units of 2^-60: n 2^up in units of 2^-62, taken at 2^-60
        const int64_t h1 = mul(split((n1 << up) >> 2), yc), h2 = mul(split((n2 << up) >> 2), yc);
        l1[0] = coef(h1 >> 2);
        l1[S - 1] = coef(h2 >> 2);
        if (t.srt) {
            l2[0] = l1[0];
            l2[S - 1] = l1[S - 1];
        } else {
            const int64_t unit = int64_t(1) << 60;
            l2[0] = coef(mul(split(unit - h1), coef(reciprocal(4 * unit - h1))) >> 2);
            l2[S - 1] = coef(mul(split(unit - h2), coef(reciprocal(4 * unit - h2))) >> 2);
        }
        // G = k (a - c) / det K = g1 (y / 2^58) 2^(up - 3) from the scales above; q = 2 G (sum / 2)
        const X y2 = split(y << 1);
        const int64_t p1 = mul(split(half[0]), coef(mul(y2, t.g1))), p2 = mul(split(half[S - 1]), coef(mul(y2, t.g2)));
        const int more = up > 3 ? up - 3 : 0;  // (det is below 2^59, so up is at least 3)
        const int64_t lim = kLimit >> more;
        fits &= p1 < lim && p1 > -lim && p2 < lim && p2 > -lim;
        q1 = split((int64_t)((uint64_t)p1 << more));
        q2 = split((int64_t)((uint64_t)p2 << more));
    }
    if (!fits) return false;
    uint64_t rest[S];  // what the moving populations leave of the sums (modulo 2^64 on the way)
    int32_t off[S];
    int64_t even[S];  // 2 w xi of the current weight
#pragma unroll
    for (int s = 0; s < S; ++s) {
        rest[s] = (uint64_t)sum[s];
        off[s] = 0;
    }
#pragma unroll
    for (int pr = 0; pr < L::NPAIR; ++pr) {
        const int ka = L::K0 + 2 * pr, kb = ka + 1;
        int64_t sym[S], asym[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if (pr == 0 || L::w(ka) != L::w(ka - 1))
                even[s] = mul(split(half[s]), coef((int64_t)(4.0 * L::w(ka) * 288230376151711744.0 + 0.5)));
            sym[s] = x[s][ka] + x[s][kb] - even[s];
            asym[s] = x[s][ka] - x[s][kb];
        }
        int64_t ds[S], da[S];
        if (S == 1) {
            ds[0] = mul(split(sym[0]), l2[0]);
            da[0] = mul(split(asym[0]), l1[0]);
        } else {
            const Cf s1 = coef_of_abs(sym[0], e[0]), s2 = coef_of_abs(sym[S - 1], e[S - 1]);
            const Cf a1 = coef_of_abs(asym[0], e[0]), a2 = coef_of_abs(asym[S - 1], e[S - 1]);
            ds[0] = dot(split(sym[0]), l2[0], q1, s2);
            ds[S - 1] = dot(split(sym[S - 1]), l2[S - 1], q2, s1);
            da[0] = dot(split(asym[0]), l1[0], q1, a2);
            da[S - 1] = dot(split(asym[S - 1]), l1[S - 1], q2, a1);
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            int32_t d;
            if (ka != 0) {
                const int64_t na = x[s][ka] - (ds[s] + da[s]);
                f[s][ka] = to_double(na, e[s], d);
                rest[s] -= (uint64_t)na;
                off[s] += d;
            }
            const int64_t nb = x[s][kb] - (ds[s] - da[s]);
            f[s][kb] = to_double(nb, e[s], d);
            rest[s] -= (uint64_t)nb;
            off[s] += d;
        }
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
        int32_t d;
        f[s][0] = to_double((int64_t)rest[s] - off[s], e[s], d);
    }
    return true;
}

#ifdef __CUDACC__
// collide_fixed of a ternary node by two lanes, one per species (own: this lane's, 0 or 1):
// f holds that species' populations, and the lane 16 away holds the other's.  The same
// integer operations per species, so the same results; the lanes exchange mole fractions
// and departures by shuffles.  All lanes of the warp take part; false (in both lanes of
// the node, f unchanged) where the node does not fit or is not active.
template <typename L>
__device__ __forceinline__ bool collide_fixed_lane(double (&f)[L::Q], const FixedTable& t, int own, bool active)
{
    using namespace fx;
    constexpr int Q = L::Q;
    constexpr unsigned all = 0xffffffffu;
    uint32_t still = 0, moving = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const uint32_t h = (uint32_t)(bits_of(f[k]) >> 32) & 0x7fffffffu;
        uint32_t& most = k < L::K0 ? still : moving;
        most = h > most ? h : most;
    }
    const uint32_t top = still > moving ? still : moving;
    const Block e = block((int)(top >> 20), block_bits<L>());
    bool fits = fits_block(e.M, f) && active;
    int64_t x[Q], sum = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        x[k] = to_fixed(f[k], e, block_bits<L>(), (k & 1) != 0);
        sum += x[k];
    }
    const int64_t half = sum >> 1, mine = to_abs(sum, e);
    fits &= (uint64_t)(mine + kOne / 16) <= (uint64_t)(kOne + kOne / 8) && half < kLimit && half > -kLimit;
    fits &= fits_pair<L>(still, moving, half);
    const int64_t other = __shfl_xor_sync(all, (long long)mine, 16);
    const int64_t x3 = kOne - mine - other;
    fits &= (uint64_t)(x3 + kOne / 16) <= (uint64_t)(kOne + kOne / 8);
    const X a = split(x3), b = split(own ? other : mine), c = split(own ? mine : other);
    const int64_t det = dot(a, t.det[0], b, t.det[1], c, t.det[2]);
    const Cf n0 = own ? t.n22[0] : t.n11[0], n1 = own ? t.n22[1] : t.n11[1], n2 = own ? t.n22[2] : t.n11[2];
    const int64_t n = dot(a, n0, b, n1, c, n2);
    fits &= det > kOne / 32 && n > 0 && n < det;
    const int up = fits ? clz64((uint64_t)det) - 2 : 0;
    const int64_t y = reciprocal(fits ? det << up : int64_t(1) << 61);
    const int64_t h = mul(split((n << up) >> 2), coef(y));
    const Cf l1 = coef(h >> 2);
    Cf l2 = l1;
    if (!t.srt) {
        const int64_t unit = int64_t(1) << 60;
        l2 = coef(mul(split(unit - h), coef(reciprocal(4 * unit - h))) >> 2);
    }
    const int64_t p = mul(split(half), coef(mul(split(y << 1), own ? t.g2 : t.g1)));
    const int more = up > 3 ? up - 3 : 0;
    const int64_t lim = kLimit >> more;
    fits &= p < lim && p > -lim;
    const X q = split((int64_t)((uint64_t)p << more));
    const unsigned votes = __ballot_sync(all, fits);
    const int lane = (int)(threadIdx.x & 31u);
    fits = ((votes >> lane) & (votes >> (lane ^ 16)) & 1u) != 0;
    if (votes == 0) return false;
    uint64_t rest = (uint64_t)sum;  // modulo 2^64 on the way
    int64_t even = 0;
    int32_t off = 0;
    double out[Q];
#pragma unroll
    for (int pr = 0; pr < L::NPAIR; ++pr) {
        const int ka = L::K0 + 2 * pr, kb = ka + 1;
        if (pr == 0 || L::w(ka) != L::w(ka - 1))
            even = mul(split(half), coef((int64_t)(4.0 * L::w(ka) * 288230376151711744.0 + 0.5)));
        const int64_t sym = x[ka] + x[kb] - even, asym = x[ka] - x[kb];
        const Cf s1 = coef_of_abs(sym, e), a1 = coef_of_abs(asym, e);
        const Cf s2 = {__shfl_xor_sync(all, s1.h, 16), __shfl_xor_sync(all, s1.l4, 16)};
        const Cf a2 = {__shfl_xor_sync(all, a1.h, 16), __shfl_xor_sync(all, a1.l4, 16)};
        const int64_t ds = dot(split(sym), l2, q, s2), da = dot(split(asym), l1, q, a2);
        int32_t d;
        if (ka != 0) {
            const int64_t na = x[ka] - (ds + da);
            out[ka] = to_double(na, e, d);
            rest -= (uint64_t)na;
            off += d;
        }
        const int64_t nb = x[kb] - (ds - da);
        out[kb] = to_double(nb, e, d);
        rest -= (uint64_t)nb;
        off += d;
    }
    int32_t d;
    out[0] = to_double((int64_t)rest - off, e, d);
    if (fits)
#pragma unroll
        for (int k = 0; k < Q; ++k) f[k] = out[k];
    return fits;
}
#endif

}  // namespace lbms
