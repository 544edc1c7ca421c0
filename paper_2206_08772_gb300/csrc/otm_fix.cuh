// otm_fix.cuh -- fixed-point arithmetic of the LME solve (Eq. 14), its force products and the node sums.
//
// Why: an FP64 instruction occupies an SM of this GPU for 16 cycles per warp (2 lanes per cycle), a
// 32x32->64-bit integer multiply-add for 1 and a 32-bit integer operation for 0.5. The exponents,
// the weights and the ten sums of one evaluation (Z, r = sum w d, A = sum w d d^T) cost 18 FP64
// instructions a pair; here they are formed in 64-bit integers, with errors at or below those of
// the FP64 form (bounds beside each step), and the FP64 pipe is left to the per-MP scalars and the
// force contributions.
//
// Coordinates: X = round(x 2^fb) modulo 2^64 per axis (a wrapped 64-bit integer, so positions have
// no range limit; only differences matter). fb is chosen so that the support radius is 2^63/4.4 to
// 2^63/2.2 units ("LSB" below, between 2^-60 and 2^-58 of the node spacing at the default support
// tolerance), below the FP64 spacing of positions a node spacing away from the origin.
//
// Completing the square, -beta |d|^2 + lambda . d = -beta |T|^2 + |lambda|^2 / (4 beta) with
// T_a = x_c - x_a, x_c = x_p - lambda / (2 beta): one evaluation needs the nodes' X and the centre
// X_c only. The exponent y = (|lambda|^2/(4 beta) - shift - beta |T|^2) 256/ln 2 has 46 fraction
// bits (half a unit is 2e-17 of a weight).
//
// Host and device code, so that the arithmetic can be checked without a GPU.
#pragma once

#include <stdint.h>
#include <string.h>

namespace otm {

typedef long long i64;
typedef unsigned long long u64;

#ifdef __CUDA_ARCH__
#define OTM_HD __host__ __device__ __forceinline__
// c + a b in 64 bits. As a low / high pair with carry it becomes one instruction (4 cycles of an SM
// quarter for a warp); mad.wide with a 64-bit addend becomes three (6.7 cycles), and a 64-bit product
// of sign-extended halves written in C four or more (measured).
__device__ __forceinline__ i64 fx_madw(int a, int b, i64 c)
{
    asm("{.reg .u32 l, h;\n mov.b64 {l, h}, %0;\n mad.lo.cc.u32 l, %1, %2, l;\n madc.hi.s32 h, %1, %2, h;\n mov.b64 %0, {l, h};}"
        : "+l"(c) : "r"(a), "r"(b));
    return c;
}
__device__ __forceinline__ u64 fx_umadw(uint32_t a, uint32_t b, u64 c)
{
    asm("{.reg .u32 l, h;\n mov.b64 {l, h}, %0;\n mad.lo.cc.u32 l, %1, %2, l;\n madc.hi.u32 h, %1, %2, h;\n mov.b64 %0, {l, h};}"
        : "+l"(c) : "r"(a), "r"(b));
    return c;
}
__device__ __forceinline__ int fx_mulhi(int a, int b) { return __mulhi(a, b); }
__device__ __forceinline__ uint32_t fx_umulhi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
__device__ __forceinline__ uint32_t fx_shf_r(uint32_t lo, uint32_t hi, int s) { return __funnelshift_r(lo, hi, s); }
__device__ __forceinline__ int fx_log2(uint32_t v) { return (int)(__float_as_uint(__uint2float_rz(v)) >> 23) - 127; }
__device__ __forceinline__ int fx_rint(float v) { return __float2int_rn(v); }
__device__ __forceinline__ double fx_bits_d(u64 b) { return __longlong_as_double((i64)b); }
__device__ __forceinline__ u64 fx_d_bits(double v) { return (u64)__double_as_longlong(v); }
__device__ __forceinline__ uint32_t fx_f_bits(float v) { return __float_as_uint(v); }
// shifts by any amount: 64 and more (as unsigned) give 0
__device__ __forceinline__ u64 fx_shr(u64 v, unsigned n)
{
    u64 r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}
__device__ __forceinline__ u64 fx_shl(u64 v, unsigned n)
{
    u64 r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}
#else
#ifdef __CUDACC__
#define OTM_HD __host__ __device__ inline
#else
#define OTM_HD inline
#endif
OTM_HD i64 fx_madw(int a, int b, i64 c) { return (i64)((u64)((i64)a * (i64)b) + (u64)c); }
OTM_HD u64 fx_umadw(uint32_t a, uint32_t b, u64 c) { return (u64)a * (u64)b + c; }
OTM_HD int fx_mulhi(int a, int b) { return (int)(((i64)a * (i64)b) >> 32); }
OTM_HD uint32_t fx_umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((u64)a * (u64)b) >> 32); }
OTM_HD uint32_t fx_shf_r(uint32_t lo, uint32_t hi, int s) { return (uint32_t)((((u64)hi << 32) | lo) >> (s & 31)); }
OTM_HD int fx_log2(uint32_t v)
{
    if (!v) return -127;   // as the device's
    int l = -1;
    while (v) { v >>= 1; l++; }
    return l;
}
OTM_HD int fx_rint(float v) { return (int)(v + (v < 0.f ? -0.5f : 0.5f)); }
OTM_HD double fx_bits_d(u64 b)
{
    double v;
    memcpy(&v, &b, 8);
    return v;
}
OTM_HD u64 fx_d_bits(double v)
{
    u64 b;
    memcpy(&b, &v, 8);
    return b;
}
OTM_HD uint32_t fx_f_bits(float v)
{
    uint32_t b;
    memcpy(&b, &v, 4);
    return b;
}
OTM_HD u64 fx_shr(u64 v, unsigned n) { return n < 64 ? v >> n : 0; }
OTM_HD u64 fx_shl(u64 v, unsigned n) { return n < 64 ? v << n : 0; }
#endif

// constants of a problem (host-derived, see make_fix_const)
struct FixConst {
    int on;            // 1: the fixed-point evaluation covers this problem's support radius
    int fb;            // X = round(x 2^fb)
    uint32_t near;     // high word of r_s (1 + 1e-9)
    u64 bq;            // beta 256/ln2 a^2 2^46 2^63, a = 2^(32 - fb): y units per unit of a^2, halved
    double i2b;        // 2^fb / (2 beta): lambda to the centre offset in LSB
    double cy;         // 256 / (4 beta ln 2): |lambda|^2 to the exponent's constant
    double vmax;       // largest centre offset per axis in LSB (0.66 2^63 minus the support radius)
    double r_unit;     // 2^-fb
    double a_unit;     // a^2 / 16
};

constexpr double kFixYScale = 0x1.71547652b82fep+8;   // 256 / ln 2
constexpr double kFixYOne = 0x1p46;
constexpr double kFixT = 0.66 * 0x1p63;               // |T| per axis stays below this

// x 2^fb rounded to an integer, modulo 2^64 (integer operations on the bits of x)
OTM_HD i64 fix_from_double(double x, int fb)
{
    const u64 b = fx_d_bits(x);
    const int ef = (int)((b >> 52) & 0x7ff);
    const u64 m = (b & 0xfffffffffffffULL) | (ef ? 0x10000000000000ULL : 0ULL);
    const int s = (ef ? ef : 1) - 1075 + fb;
    u64 r;
    if (s >= 0) r = s < 64 ? m << s : 0ULL;
    else r = s >= -54 ? (m + (1ULL << (-s - 1))) >> -s : 0ULL;
    return (b >> 63) ? -(i64)r : (i64)r;
}

// the same without losing the high words: the value is hi 2^64 + (u64)lo (for points whose distances are
// not known to fit 64 bits); false for |x| 2^fb of 2^116 or more and for non-finite x
OTM_HD bool fix_from_double_wide(double x, int fb, i64 &lo, i64 &hi)
{
    const u64 b = fx_d_bits(x);
    const int ef = (int)((b >> 52) & 0x7ff);
    const u64 m = (b & 0xfffffffffffffULL) | (ef ? 0x10000000000000ULL : 0ULL);
    const int s = (ef ? ef : 1) - 1075 + fb;
    const u64 sg = 0ULL - (b >> 63);
    lo = fix_from_double(x, fb);
    const u64 h = (s > 11 && s < 64) ? m >> (64 - s) : 0ULL;      // high word of the magnitude
    hi = (i64)((h ^ sg) + ((sg && lo == 0) ? 1ULL : 0ULL));       // two's complement of (h, |lo|)
    return s < 64;
}

// exp: 2^(j/1024) (j = 0..1023) as 64-bit mantissas in [2^63, 2^64) come from a table; the rest
// s = fraction of the 1024th, 44 bits in [0, 1), goes through exp(s ln2/1024) - 1 by its Taylor
// polynomial of degree 4 (truncation below 2e-18) in fixed point.
constexpr uint32_t kFxC4 = 161365u;          // C^4/24 2^64, C = ln2/1024
constexpr uint32_t kFxC3 = 953553326u;       // C^3/6 2^64
constexpr uint32_t kFxC2 = 4127059964u;      // C^2/2 2^54
constexpr u64 kFxC1 = 0xB17217F7D1CF79ACULL; // C 2^74

// the weight of exponent y (y < 0, fraction bits 46): mantissa W in [2^63, 2^64) and exponent e <= -1,
// w = W 2^(e - 63)
OTM_HD void fix_exp(i64 y, const u64 *T, u64 &W, int &e)
{
    const int yh = (int)(y >> 32);
    const uint32_t yl = (uint32_t)y;
    e = yh >> 22;
    const u64 Tj = T[(yh >> 12) & 1023];
    const uint32_t sh = fx_shf_r(yl, (uint32_t)yh, 12), sl = yl & 0xfffu;   // s = sh 2^-32 + sl 2^-44
    const uint32_t a3 = kFxC3 + fx_umulhi(sh, kFxC4);                        // 2^-64
    const uint32_t a2 = kFxC2 + (fx_umulhi(sh, a3) >> 10);                   // 2^-54
    const u64 a1 = kFxC1 + (fx_umadw(sh, a2, 0) >> 12);                           // 2^-74
    const uint32_t a1h = (uint32_t)(a1 >> 32);
    const u64 p = fx_umadw(sh, a1h, (u64)(fx_umulhi(sh, (uint32_t)a1)) + sl * (a1h >> 12));   // 2^-74, below 2^-10
    const uint32_t ph = (uint32_t)(p >> 32), Th = (uint32_t)(Tj >> 32);
    const u64 q = fx_umadw(Th, ph, (u64)fx_umulhi(Th, (uint32_t)p) + fx_umulhi((uint32_t)Tj, ph));   // T p, 2^-73
    W = Tj + (q >> 10);
}

// w = W 2^(e - 63) in FP64, truncated (the sums use all of W)
OTM_HD double fix_weight_double(u64 W, int e)
{
    const u64 b = W >> 11;
    return fx_bits_d(((u64)((uint32_t)(b >> 32) + ((uint32_t)(e + 1022) << 20)) << 32) | (uint32_t)b);
}

// the ten sums of one lane's pairs. Accumulators in limbs; no overflow for up to 12 pairs with every
// |T_i| < 0.66 2^63 and a sum of weights below 1:
//   w = wh 2^-31 + wl 2^-63 (wh < 2^31, wl signed 32 bits), wa = wl/4 rounded to odd (29 bits, the
//   mean of the dropped part is zero), T = th 2^32 + tl (th below 2^30.4, tl signed 32 bits),
//   M = T_i T_j 2^-64 = mh 2^32 + ml (mh below 2^28.8, ml unsigned)
struct FixSums {
    u64 z;             // sum w, 2^-63
    uint32_t zc;       // sum wh >> 5 (window check: z itself may wrap)
    int top;           // high words of all y or'ed by max: >= 0 means a weight of 1 or more
    i64 rh[3], r1[3], r2[3];
    i64 ah[6], a2[6];
    u64 a1[6];
    float a3[6];
};

OTM_HD void fix_sums_zero(FixSums &s)
{
    s.z = 0;
    s.zc = 0;
    s.top = -1;
    // the low limbs start at half of what fix_combine shifts out: its shifts then round to nearest
#pragma unroll
    for (int i = 0; i < 3; i++) {
        s.rh[i] = 0;
        s.r1[i] = 1LL << 30;
        s.r2[i] = 1LL << 28;
    }
#pragma unroll
    for (int i = 0; i < 6; i++) {
        s.ah[i] = 0;
        s.a1[i] = 1ULL << 26;
        s.a2[i] = 1LL << 24;
        s.a3[i] = 0.f;
    }
}

// one pair: node X (three coordinates), centre c, constant cst (46 fraction bits); returns the weight.
// LOLO: with the product of the low limbs in A, in FP32 (A to about 1e-16 of its trace; without it to 6e-16)
template <bool LOLO>
OTM_HD double fix_pair(const i64 X0, const i64 X1, const i64 X2, const i64 c0, const i64 c1, const i64 c2,
                       const i64 cst, const u64 bq, const u64 *T, FixSums &s)
{
    const i64 t0 = c0 - X0, t1 = c1 - X1, t2 = c2 - X2;
    const int h0 = (int)((t0 + 0x80000000LL) >> 32), h1 = (int)((t1 + 0x80000000LL) >> 32),
              h2 = (int)((t2 + 0x80000000LL) >> 32);
    const int l0 = (int)t0, l1 = (int)t1, l2 = (int)t2;
    // M = T T^T 2^-64: the low halves' product is dropped, the cross terms rounded
    i64 M[6];
    M[0] = fx_madw(h0, h0, fx_madw(h0, l0, 1LL << 30) >> 31);
    M[1] = fx_madw(h1, h1, fx_madw(h1, l1, 1LL << 30) >> 31);
    M[2] = fx_madw(h2, h2, fx_madw(h2, l2, 1LL << 30) >> 31);
    M[3] = fx_madw(h0, h1, fx_madw(h0, l1, fx_madw(l0, h1, 1LL << 31)) >> 32);
    M[4] = fx_madw(h1, h2, fx_madw(h1, l2, fx_madw(l1, h2, 1LL << 31)) >> 32);
    M[5] = fx_madw(h0, h2, fx_madw(h0, l2, fx_madw(l0, h2, 1LL << 31)) >> 32);
    // y = cst - beta |T|^2
    const u64 S = (u64)(M[0] + M[1] + M[2]) << 1;
    const uint32_t Sh = (uint32_t)(S >> 32), bh = (uint32_t)(bq >> 32);
    const i64 y = cst - (i64)fx_umadw(Sh, bh, (u64)fx_umulhi(Sh, (uint32_t)bq) + fx_umulhi((uint32_t)S, bh));
    const int yh = (int)(y >> 32);
    s.top = s.top > yh ? s.top : yh;
    u64 W;
    int e;
    fix_exp(y, T, W, e);
    const int sft = e < -63 ? 63 : -e;
    const u64 w = (W >> (sft & 63)) | 1ULL;      // 2^-63; odd: truncation without a mean error
    const int wh = (int)((w + 0x80000000ULL) >> 32);
    const int wl = (int)w;
    const int wa = (wl >> 2) | 1;                // 2^-61
    s.z += w;
    s.zc += (uint32_t)wh >> 5;
    s.rh[0] = fx_madw(wh, h0, s.rh[0]); s.rh[1] = fx_madw(wh, h1, s.rh[1]); s.rh[2] = fx_madw(wh, h2, s.rh[2]);   // 2 LSB
    s.r1[0] = fx_madw(wh, l0, s.r1[0]); s.r1[1] = fx_madw(wh, l1, s.r1[1]); s.r1[2] = fx_madw(wh, l2, s.r1[2]);   // 2^-31 LSB
    s.r2[0] = fx_madw(wa, h0, s.r2[0]); s.r2[1] = fx_madw(wa, h1, s.r2[1]); s.r2[2] = fx_madw(wa, h2, s.r2[2]);   // 2^-29 LSB
    const float fw = LOLO ? (float)wl : 0.f;
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const int mh = (int)(M[i] >> 32);        // floor; the low word unsigned
        const uint32_t ml = (uint32_t)M[i];
        s.ah[i] = fx_madw(wh, mh, s.ah[i]);                // 2 (units of 2^64 LSB^2)
        s.a1[i] = fx_umadw((uint32_t)wh, ml, s.a1[i]);   // 2^-31
        s.a2[i] = fx_madw(wa, mh, s.a2[i]);                // 2^-29
        if (LOLO) s.a3[i] += fw * (float)ml;     // 2^-63
    }
    return fix_weight_double(W, e);
}

// a lane's share of the window check on A: its trace in units of 2^27 (of 2^64 LSB^2). The warp total
// stays below kFixTraceMax so that A fits 64 bits in units of 2^60 LSB^2, fine enough for the 32
// lanes' roundings to vanish beside FP64's
constexpr uint32_t kFixTraceMax = 1u << 31;
OTM_HD uint32_t fix_trace(const FixSums &s)
{
    const i64 t = (s.ah[0] + s.ah[1] + s.ah[2]) >> 26;
    return t > 0x7fffffffLL ? 0x7fffffffu : (t < 0 ? 0u : (uint32_t)t);
}

// one lane's sums as ten 64-bit integers: Z (2^-63), r (LSB), A (2^60 LSB^2)
OTM_HD void fix_combine(const FixSums &s, i64 (&v)[10])
{
    v[0] = (i64)s.z;
#pragma unroll
    for (int i = 0; i < 3; i++) v[1 + i] = 2 * s.rh[i] + (s.r1[i] >> 31) + (s.r2[i] >> 29);
#pragma unroll
    for (int i = 0; i < 6; i++)
        v[4 + i] = 32 * s.ah[i] + (i64)(s.a1[i] >> 27) + (s.a2[i] >> 25) + (i64)fx_rint(s.a3[i] * 0x1p-59f);
}

// sums of T about the centre -> sums of d = T + v about the material point (v the centre offset):
// r_d = r + Z v;  A_d = A + v r_d^T + r v^T
OTM_HD i64 fix_r_about(i64 z, i64 r, i64 v) { return r + (i64)(((__int128)z * v) >> 63); }
OTM_HD i64 fix_a_about(i64 a, i64 ri, i64 rdj, i64 vi, i64 vj)
{
    return a + (i64)(((__int128)vi * rdj + (__int128)ri * vj) >> 60);
}

// floor(v 2^f) for normal or zero v with |v| 2^f < 2^63 (the kinematics gather's row values); whole numbers
// below zero come out one lower
OTM_HD i64 fix_floor(double v, int f)
{
    const u64 b = fx_d_bits(v);
    const int s = 1085 - f - (int)((b >> 52) & 0x7ff);       // right shift of the significand 2^10, >= 0
    const u64 m = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
    return (i64)(m >> (s < 63 ? s : 63)) ^ ((i64)b >> 63);
}

// N D 2^-fb as FP64 for N > 0 given by its significand nm (in [2^63, 2^64)) and biased exponent en, inside
// fix_mul_in_range: the leading 64 bits of the product (rounded: half a unit is at most one unit
// of D), normalised and rounded to nearest
OTM_HD double fix_mul_double(u64 nm, int en, i64 D, int fb)
{
    const u64 sg = (u64)(D >> 63);
    const u64 m = ((u64)D ^ sg) - sg;
    const uint32_t nh = (uint32_t)(nm >> 32), nl = (uint32_t)nm, mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
    const u64 c1 = fx_umadw(nl, mh, (u64)fx_umulhi(nl, ml) + 0x80000000ULL), c2 = fx_umadw(nh, ml, 0);
    const u64 c = (c1 >> 32) + (c2 >> 32) + (((c1 & 0xffffffffULL) + (c2 & 0xffffffffULL)) >> 32);
    u64 p = fx_umadw(nh, mh, c);
    const int lz = 30 - fx_log2((uint32_t)(p >> 32));    // leading bit to 62
    p = ((p << lz) + 512ULL) >> 10;                      // 53 bits, the leading one adds to the exponent
    const uint32_t hi = (uint32_t)(p >> 32) + ((uint32_t)(en + 62 - fb - lz) << 20);
    return fx_bits_d(((u64)(hi | ((uint32_t)sg & 0x80000000u)) << 32) | (uint32_t)p);
}

// Whether N, of biased exponent en, times each of a, b, c is in fix_mul_double's range: 2^33 <= |D| < 2^63, so
// that the high word of the product is not zero (it is normalised by that word), and N large enough
// for a normal result with any fb in [-60, 540]. By the high words, floors: 3 and above, -3 and below.
OTM_HD bool fix_mul_in_range(int en, i64 a, i64 b, i64 c)
{
    const int ah = (int)(a >> 32), bh = (int)(b >> 32), ch = (int)(c >> 32);
    const int am = ah < 0 ? -ah : ah, bm = bh < 0 ? -bh : bh, cm = ch < 0 ? -ch : ch;
    const int m = am < bm ? am : bm;
    return (m < cm ? m : cm) > 2 && en > 600;
}

// the significand of a normal v > 0 in [2^63, 2^64)
OTM_HD u64 fix_significand(double v) { return ((fx_d_bits(v) & 0xfffffffffffffULL) | 0x10000000000000ULL) << 11; }

// e = N d from the fixed-point separation; in FP64 where a component is within 2^-30 of the range or N is tiny
OTM_HD void fix_nd(double N, i64 d0, i64 d1, i64 d2, int fb, double unit, double &ex, double &ey, double &ez)
{
    const u64 nm = fix_significand(N);
    const int en = (int)(fx_d_bits(N) >> 52);
    if (fix_mul_in_range(en, d0, d1, d2)) {
        ex = fix_mul_double(nm, en, d0, fb);
        ey = fix_mul_double(nm, en, d1, fb);
        ez = fix_mul_double(nm, en, d2, fb);
    } else {
        ex = N * ((double)d0 * unit);
        ey = N * ((double)d1 * unit);
        ez = N * ((double)d2 * unit);
    }
}

// D 2^-fb rounded to FP32 (nearest, ties away from zero; |D| < 2^63)
OTM_HD float fix_to_float(i64 D, int fb)
{
    const u64 sg = (u64)(D >> 63);
    u64 m = ((u64)D ^ sg) - sg;
    if (m == 0) return 0.f;
    const uint32_t hi = (uint32_t)(m >> 32);
    const int lz = hi ? 31 - fx_log2(hi) : 63 - fx_log2((uint32_t)m);
    m <<= lz;
    const int E = 63 - lz - fb + 127;
    if (E < 1) return 0.f;
    const uint32_t t = (uint32_t)(m >> 40) + ((uint32_t)(m >> 39) & 1u);
    const uint32_t b = (((uint32_t)(E - 1) << 23) + t) | ((uint32_t)sg << 31);
    float f;
#ifdef __CUDA_ARCH__
    f = __uint_as_float(b);
#else
    memcpy(&f, &b, 4);
#endif
    return f;
}

// ------------------------------------------------------------------ force contributions (Eq. 5)
// f = N Q D 2^-fb of fixed-point separations D (|D| < 2^62) and an FP64 matrix Q per material point. Rows of Q
// as 60-bit integers of the row's own exponent, in limbs q = qh 2^32 + ql; what is dropped (ql dl and the
// rounding of Q) stays below 5 units of F: 2^-56 of the row's largest entry times 2^62.
struct FixRows {
    int qh[9], ql[9], fb[3];   // fb: the exponent of F in fix_mul_double
    bool ok;                   // false if a row is zero, not finite or far out of range: FP64 then
};

OTM_HD void fix_rows(const double (&Q)[9], int fb, FixRows &R)
{
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        int e = 0;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int ej = (int)(fx_d_bits(Q[3 * i + j]) >> 52) & 0x7ff;
            e = e > ej ? e : ej;
        }
        ok = ok && e > 600 && e < 1450;
        const int s = 60 - (e - 1022);                        // |Q_ij| < 2^(e - 1022)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const i64 q = fix_from_double(Q[3 * i + j], s);
            R.qh[3 * i + j] = (int)((q + 0x80000000LL) >> 32);
            R.ql[3 * i + j] = (int)q;
        }
        R.fb[i] = fb + s - 62;
    }
    R.ok = ok;
}

// row i: F = sum_j q_ij D_j in units of 2^62, below 2^62
OTM_HD i64 fix_row_dot(const FixRows &R, int i, const int (&dh)[3], const int (&dl)[3])
{
    i64 hh = 0, hl = 1LL << 29;
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int qh = R.qh[3 * i + j];
        hh = fx_madw(qh, dh[j], hh);
        hl = fx_madw(qh, dl[j], fx_madw(R.ql[3 * i + j], dh[j], hl));
    }
    return (hh << 2) + (hl >> 30);
}

// f = Q e from the fixed-point separation; false: out of range, FP64 then
OTM_HD bool force_fix(const FixRows &R, double N, i64 d0, i64 d1, i64 d2, double &fx, double &fy, double &fz)
{
    const int dh[3] = {(int)((d0 + 0x80000000LL) >> 32), (int)((d1 + 0x80000000LL) >> 32), (int)((d2 + 0x80000000LL) >> 32)};
    const int dl[3] = {(int)d0, (int)d1, (int)d2};
    const i64 F0 = fix_row_dot(R, 0, dh, dl), F1 = fix_row_dot(R, 1, dh, dl), F2 = fix_row_dot(R, 2, dh, dl);
    const u64 nm = fix_significand(N);
    const int en = (int)(fx_d_bits(N) >> 52);
    if (!R.ok || !fix_mul_in_range(en, F0, F1, F2)) return false;
    fx = fix_mul_double(nm, en, F0, R.fb[0]);
    fy = fix_mul_double(nm, en, F1, R.fb[1]);
    fz = fix_mul_double(nm, en, F2, R.fb[2]);
    return true;
}

// ------------------------------------------------------------------ kinematics gather (Eq. 9, 11)
// Not on a step's path: the step gathers in FP64 (k_kin_search), because the units here are fixed by the node
// spacing and the sums' error does not shrink with the increments. Used by the host tests alone.
// The products of a pair's row (N, e) with its node's increment du, summed over the support:
// sum N du (3) and G = sum du (x) e (9). Limbs: du = uh 2^28 + ul (|du| < 2^57 units; uh 29 bits, ul signed 28
// bits, kept as 8 ul) and row = rh 2^31 + rl (61 bits; rh 30 bits, rl signed 31 bits), so that both cross
// products share the unit 2^28. hh += uh rh (2^59), hl += uh rl + ul rh, and ul rl, at most 2^-60 of the largest
// product, in FP32. With sum N = 1 and |e| <= N r_s the sums of uh rh and ul rh are those of one pair with
// N = 1; uh rl reaches 12 2^59 in a lane of up to 12 pairs.
constexpr int kKinDuBits = 57;
struct KinFixSums {
    i64 hh[12], hl[12];
    float ll[12];
};

// an increment's limbs (uh, 8 ul)
OTM_HD void kin_fix_split(i64 du, int &uh, int &ul8)
{
    uh = (int)((du + (1LL << 27)) >> 28);
    ul8 = (int)((du - ((i64)uh << 28)) * 8);
}

// row values in half units: N by fix_floor(N, 62), e by fix_floor(e, fe); rounded here
OTM_HD void kin_fix_pair(i64 N, i64 e0, i64 e1, i64 e2, const int (&uh)[3], const int (&ul)[3], KinFixSums &s)
{
    const i64 r[4] = {N + 1, e0 + 1, e1 + 1, e2 + 1};
    const float uf[3] = {(float)ul[0], (float)ul[1], (float)ul[2]};
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int rh = (int)((r[c] + 0x80000000LL) >> 32), rl = (int)r[c] >> 1;
        const float rf = (float)rl;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const int j = c == 0 ? i : 3 + 3 * i + (c - 1);   // 0-2: sum N du_i, 3-11: G row-major
            s.hh[j] = fx_madw(uh[i], rh, s.hh[j]);
            s.hl[j] = fx_madw(uh[i], rl, fx_madw(ul[i], rh, s.hl[j]));
            s.ll[j] += uf[i] * rf;
        }
    }
}

// one lane's sums in units of 2^56 (du unit times row unit); the warp's total stays at most 2^62
OTM_HD i64 kin_fix_combine(const KinFixSums &s, int j)
{
    return (s.hh[j] << 3) + ((s.hl[j] + (1LL << 27)) >> 28) + (int)rintf(s.ll[j] * 0x1p-59f);
}

// the exponent of the combined sums' unit: du 2^fu, row 2^fr (62 for N, fe for e)
OTM_HD int kin_fix_exponent(int fu, int fr) { return 56 - fu - (fr - 1); }

// ------------------------------------------------------------------ node sums (Eq. 5)
// Signed fixed-point sums. A term enters as the magnitude's bits, complemented if it is negative; each
// negative term is short of its two's complement by one unit, which `neg` counts.
using u128 = unsigned __int128;
template <typename U>
struct FixedSum {
    U v;
    int neg;
};
using Sum128 = FixedSum<u128>;
using Sum64 = FixedSum<u64>;

// adds v / 2^(emax - 110), truncated toward zero. Branch-free: the significand, left-aligned in 128 bits, moves
// right by 17 + emax - e; zero, subnormal (negligible) and non-finite values (caught elsewhere) move out.
OTM_HD void add_fixed(Sum128 &a, double v, int emax)
{
    const u64 b = fx_d_bits(v);
    const u64 m = (b | 0x0010000000000000ULL) << 11;
    const unsigned ef = (unsigned)(b >> 52) & 0x7ffu;
    const unsigned r = ef - 1u >= 0x7feu ? 128u : (unsigned)(emax + 1023 + 17) - ef;
    const u64 sg = (u64)((long long)b >> 63);
    const u64 h = fx_shr(m, r) ^ sg;
    const u64 l = (fx_shl(m, 64u - r) | fx_shr(m, r - 64u)) ^ sg;
    a.v += ((u128)h << 64) | l;
    a.neg -= (int)sg;
}

// adds v / 2^(emax - 46), truncated toward zero
OTM_HD void add_fixed(Sum64 &a, float v, int emax)
{
    const uint32_t b = fx_f_bits(v);
    const u64 m = (u64)((b | 0x00800000u) << 8) << 32;
    const unsigned ef = (b >> 23) & 0xffu;
    const unsigned r = ef - 1u >= 0xfeu ? 64u : (unsigned)(emax + 127 + 17) - ef;
    const int sg = (int)b >> 31;
    a.v += fx_shr(m, r) ^ (u64)(long long)sg;
    a.neg -= sg;
}

}  // namespace otm
