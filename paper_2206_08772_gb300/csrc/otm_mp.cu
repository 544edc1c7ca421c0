// otm_mp.cu -- material-point kernels (sm_103a):
//   k_search     : Algorithm 3 steps 2-3, warp per MP: candidates of the linked-cell stencil
//                  tested in FP32 against an error band; only candidates inside the band take
//                  the exact FP64 test, so the support (d^2 <= r_s^2 in FP64) is bit-exact.
//                  Ascending-ID sort, influence counting (integer atomics -> rank).
//   k_lme        : Eq. 14, warp per MP: damped Newton for lambda (warm start, exponent shift from
//                  the previous log Z), N and grad N = -N J^-1 d, per-pair contributions
//                  (m_p N, -v sigma grad N) written straight into node-major order. k_lme_fix: the same
//                  with the pair sums in fixed point (the FP64 path; k_lme is the mixed path's).
//   k_kinematics : Eq. 9-13, warp per MP: x_p = sum N x_I, dF = 1 + sum du_I (x) grad N_I,
//                  F <- dF F, v <- det(dF) v
//   k_return_map : Sec. 4.1 / 4.2, thread per MP: Hencky exponential-map radial return (J2
//                  linear hardening closed form, Johnson-Cook safeguarded Newton), heating,
//                  fracture flag, sigma = tau / J
#include <cmath>
#include <mutex>

#include "otm_dev.cuh"
#include "otm_fix.cuh"
#include "otm_rm.cuh"

namespace otm {

// ======================================================================== double-float arithmetic
// FP32 pairs hi + lo, about 2^-47 relative (the exp's polynomial, the mixed path's Hessian sums)
// An FP64 value split into two FP32 values with integer operations on its bits (GB300 charges a
// conversion instruction an FP64-pipe slot): hi = the leading 24 significant bits, lo = the next
// 24 of the remaining 29 (truncated), so v = hi + lo to 2^-47 relative. Values outside the normal
// FP32 range give hi = lo = 0 (the Hessian sums only see weights in [1e-30, 1e30], checked by the
// caller, and differences of about h).
__device__ __forceinline__ void df_split(double v, float &hi, float &lo)
{
    const int vh = __double2hiint(v);
    const unsigned vl = (unsigned)__double2loint(v);
    const int e = ((vh >> 20) & 0x7ff) - 1023;
    const unsigned sgn = (unsigned)vh & 0x80000000u;
    const bool ok = e > -126 && e < 128;
    hi = ok ? __uint_as_float(sgn | ((unsigned)(e + 127) << 23) | ((unsigned)(vh & 0xfffff) << 3) | (vl >> 29))
            : 0.f;
    const unsigned r = vl & 0x1fffffffu;   // significand bits 28..0 below hi, weight 2^(e - 52)
    const int lz = __clz(r);               // >= 3 when r != 0
    const int el = e - 52 + (31 - lz);     // exponent of r's leading bit
    lo = (ok && r != 0 && el > -126) ? __uint_as_float(sgn | ((unsigned)(el + 127) << 23) | (((r << lz) << 1) >> 9))
                                     : 0.f;
}

// exact widening of an FP32 value to FP64 with integer operations (zero and normal values)
__device__ __forceinline__ double df_widen(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned ef = (b >> 23) & 0xff;
    if (ef == 0) return 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | ((ef - 127 + 1023) << 20) | ((b & 0x7fffffu) >> 3)),
                            (int)(b << 29));
}

// (p, e) ~ (ah + al)(bh + bl): the product and its error, the al bl term dropped
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float &p, float &e)
{
    p = ah * bh;
    e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
}

// (sh, sl) += (q, f) with an error-free sum of the leading parts
__device__ __forceinline__ void df_add(float &sh, float &sl, float q, float f)
{
    const float s = sh + q;
    const float t = s - sh;
    const float err = (sh - (s - t)) + (q - t);
    sl = sl + (err + f);
    sh = s;
}

// ======================================================================== FP64 exponential
// exp(f) by a table-driven method after P. T. P. Tang ("Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15(2), 1989), with the
// argument scaling folded into the caller: the argument arrives as y = f * 1024 / ln 2 (the LME
// scales lambda and the prior term instead of every exponent), and
//   y = n + s, n = round(y), |s| <= 1/2 and exact (integer operations on y's bits, see below),
//   exp(f) = 2^(n >> 10) * 2^((n & 1023) / 1024) * exp(s ln2 / 1024),
// with exp(t) - 1 for |t| <= ln2/2048 by its Taylor polynomial of degree 3 (truncation below
// 5.5e-16 relative). The 1024-entry table 2^(j/1024) is computed once on the host (C library
// exp2) into g_exp2_table; the kernels read it through L1. Valid for f in about
// [-707, 708]; below it returns 0 (a weight below 1e-307 of the largest), above +inf (the caller
// then re-shifts). The scaling rounds y like any FP64 argument, so the result carries
// |f| * 2^-53 relative error from it, plus about 3 ulps.
constexpr int kExpTable = 1024;
constexpr double kExpScale = 0x1.71547652b82fep+10;   // 1024 / ln 2
constexpr double kExpC1 = 0x1.62e42fefa39efp-11;      // ln 2 / 1024
constexpr double kExpC1lo = 0x1.abc9e3b39803fp-66;    // ln 2 / 1024 - kExpC1
constexpr double kExpC2 = 0x1.ebfbdff82c58fp-23;      // kExpC1^2 / 2
constexpr double kExpC3 = 0x1.c6b08d704a0c0p-35;      // kExpC1^3 / 6
constexpr double kExpShifter = 0x1.8p52;
constexpr int kExpNmin = -1020 * 1024;                 // 2^(n >> 10) stays normal with margin
constexpr int kExpNmax = 1021 * 1024 + 1023;

static __device__ double g_exp2_table[kExpTable];
static __device__ u64 g_exp2_mant[kExpTable];          // 2^(j/1024) as 64-bit mantissas (fix_exp)
static __device__ double2 g_log_table[kExpTable];      // (r, -log r), see log_pos

// Upload the three tables to the current device in a stream of its own. A synchronous copy belongs before any
// stream capture, but the stand-alone entries may be called first under one (this thread's or another's):
// a non-blocking stream has no part in a capture, and relaxed mode lets this thread use it meanwhile.
static cudaError_t upload_tables(const double *exp2, const u64 *mant, const double2 *lg)
{
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    cudaStream_t s = nullptr;
    e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
        const cudaMemcpyKind k = cudaMemcpyHostToDevice;
        e = cudaMemcpyToSymbolAsync(g_exp2_mant, mant, kExpTable * sizeof(u64), 0, k, s);
        if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(g_log_table, lg, kExpTable * sizeof(double2), 0, k, s);
        if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(g_exp2_table, exp2, kExpTable * sizeof(double), 0, k, s);
        const cudaError_t es = cudaStreamSynchronize(s), ed = cudaStreamDestroy(s);
        if (e == cudaSuccess) e = es != cudaSuccess ? es : ed;
    }
    const cudaError_t em = cudaThreadExchangeStreamCaptureMode(&mode);
    return e != cudaSuccess ? e : em;
}

// Fill the tables on the current device (first call per device: otm_init and every stand-alone entry whose
// kernels read them). With
// `verify`, a device whose table was already filled is checked again (a synchronous 8-byte read
// of 2^0 = 1): module data is lost when the device or its primary context is reset, and the
// tables are then filled anew. otm_init verifies; the stand-alone entries, which must stay free of
// synchronisation once set up, do not.
cudaError_t exp_table_setup(bool verify)
{
    static std::mutex mu;
    static bool done[64];
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev] && verify) {
        double t0 = 0.0;
        e = cudaMemcpyFromSymbol(&t0, g_exp2_table, sizeof(double));
        if (e != cudaSuccess) return e;
        if (t0 != 1.0) done[dev] = false;
    }
    if (done[dev]) return cudaSuccess;
    double host[kExpTable];
    for (int j = 0; j < kExpTable; j++) host[j] = std::exp2((double)j / (double)kExpTable);
    u64 mant[kExpTable];
    for (int j = 0; j < kExpTable; j++)
        mant[j] = (u64)std::floor(std::ldexp(std::exp2((long double)j / (long double)kExpTable), 63) + 0.5L);
    double2 lg[kExpTable];   // (r, -log r), r ~ 1/m at the middle of the interval (1 exactly about m = 1)
    for (int j = 0; j < kExpTable; j++) {
        double m = 1.0 + (j + 0.5) / kExpTable;
        if (j >= 424) m *= 0.5;
        const double r = (j == 0 || j == kExpTable - 1) ? 1.0 : 1.0 / m;
        lg[j] = make_double2(r, (double)-std::log((long double)r));
    }
    e = upload_tables(host, mant, lg);
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

// copy the table into shared memory (block-wide; ends with a barrier)
__device__ __forceinline__ void exp_table_load(double *T)
{
    for (int j = threadIdx.x; j < kExpTable; j += blockDim.x) T[j] = g_exp2_table[j];
    __syncthreads();
}

// the polynomial's coefficients as double-float pairs (C3 needs FP32 only: its term is below 7e-12)
constexpr float kExpC1h = (float)kExpC1;
constexpr float kExpC1l = (float)((kExpC1 - (double)kExpC1h) + kExpC1lo);
constexpr float kExpC2h = (float)kExpC2;
constexpr float kExpC2l = (float)(kExpC2 - (double)kExpC2h);
constexpr float kExpC3f = (float)kExpC3;

// The polynomial p(s) = exp(s ln2/1024) - 1 (|s| <= 1/2, |p| <= 3.4e-4) runs in double-float on
// the FP32 pipe: s split into two FP32 values with integer operations (2^-48 of |s|), Horner in
// error-free FP32 products and sums (p to about 2^-46 of itself: below 5e-18 absolute, against the
// cubic's own truncation of 5.5e-16), then v = T + T p_hi + T p_lo in two FMAs. The result is as
// accurate as the same cubic in FP64 Horner form, with two FP64 instructions instead of four.
__device__ __forceinline__ double exp_scaled(double y, const double *T)
{
    // y = n + s with n = round(y) and s exact, |s| <= 1/2. For 1 <= |y| < 2^20 (every weight of the
    // LME sums: y <= 0, and |y| < 1 only for a single node that carries nearly all the weight)
    // n and s are formed from y's bits with integer operations, which leaves the FP64 pipe to the
    // polynomial; other arguments take the 1.5 * 2^52 shifter (three FP64 additions).
    const int hi = __double2hiint(y);
    const int E = ((hi >> 20) & 0x7ff) - 1023;
    int n;
    double sr;
    if (E >= 0 && E < 20) {
        // significand M (53 bits) = |y| 2^(52 - E); f = 52 - E fraction bits (33..52)
        const unsigned long long M =
            ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(y);
        const int f = 52 - E;
        const unsigned long long na = (M + (1ULL << (f - 1))) >> f;   // |n|, rounded half up
        const long long rem = (long long)(M - (na << f));             // |rem| <= 2^(f-1) < 2^52
        const bool neg = hi < 0;
        n = neg ? -(int)na : (int)na;
        // s = rem 2^-f (sign of y applied): normalised with integer operations, exactly (|rem| has
        // at most 52 significant bits, so the 12 or more leading zeros cover the 11 dropped bits)
        const unsigned long long a = (unsigned long long)(rem < 0 ? -rem : rem);
        if (a == 0) {
            sr = 0.0;
        } else {
            const int lz = __clzll((long long)a);
            const unsigned long long m = (a << lz) >> 11;          // 1.xxx in bits 52..0
            const long long ex = 1023 + 63 - lz - f;
            const bool sneg = (rem < 0) != neg;
            sr = __longlong_as_double((long long)((sneg ? 0x8000000000000000ULL : 0ULL) |
                                                  ((unsigned long long)ex << 52) | (m & 0xFFFFFFFFFFFFFULL)));
        }
    } else {
        const double t = y + kExpShifter;
        const int thi = __double2hiint(t);
        n = __double2loint(t);
        // the high word of t is 0x43380000 for round(y) in [0, 2^32) and 0x4337ffff for
        // [-2^32, 0); a mismatch with the sign of the low word means |y| >= 2^31 (or y is not finite)
        if (thi != (n < 0 ? 0x4337ffff : 0x43380000)) return (y > 0.0) ? INFINITY : 0.0;
        sr = y - (t - kExpShifter);
    }
    if (n < kExpNmin || n > kExpNmax) return (y > 0.0) ? INFINITY : 0.0;
    const double Tj = T[n & (kExpTable - 1)];
    float sh, sl;
    df_split(sr, sh, sl);
    float ah = kExpC2h, al = kExpC2l;
    df_add(ah, al, kExpC3f * sh, 0.f);            // C2 + C3 s
    float bh, bl;
    df_mul(ah, al, sh, sl, bh, bl);               // (C2 + C3 s) s
    float ch = kExpC1h, cl = kExpC1l;
    df_add(ch, cl, bh, bl);                       // C1 + (C2 + C3 s) s
    float ph, pl;
    df_mul(ch, cl, sh, sl, ph, pl);               // p
    const double v = fma(Tj, df_widen(pl), fma(Tj, df_widen(ph), Tj));
    return __hiloint2double(__double2hiint(v) + ((n >> 10) << 20), __double2loint(v));
}

// ======================================================================== LME (Eq. 14)
// Sums of one evaluation at lambda with weights w_a = exp(f_a - shift), f_a = q_a + lambda . d_a:
// Z = sum w, r = sum w d, A = sum w d d^T (unnormalised). Then N = w / Z, the residual of the
// consistency condition is r / Z and the Hessian of log Z is J = A / Z - (r/Z)(r/Z)^T = J' / Z
// with J' = A - r r^T / Z.
struct LmeSums {
    double Z, r0, r1, r2, a00, a11, a22, a01, a12, a02;
    double shift;
};

__device__ __forceinline__ double rn2(const LmeSums &E) { return E.r0 * E.r0 + E.r1 * E.r1 + E.r2 * E.r2; }

// log Z(trial) < log Z(current)
__device__ __forceinline__ bool logz_less(const LmeSums &t, const LmeSums &c)
{
    if (t.shift == c.shift) return t.Z < c.Z;
    return t.shift + log(t.Z) < c.shift + log(c.Z);
}

// ======================================================================== support search
// Search of one MP over the linked-cell rows that cover [x_p - r_s, x_p + r_s] (with a 1e-4
// relative margin), rows of contiguous cells along x. Each candidate is first tested in FP32 on
// coordinates relative to the grid origin; the FP32 value d2f of |x_p - x_a|^2 differs from the
// FP64 value that defines the support by less than `band` (derived below), so a candidate with
// d2f < rs2 - band is inside, one with d2f > rs2 + band is outside, and only the rest take the
// exact FP64 test on the double coordinates. Accepted IDs go to list[0..min(count, S)); returns
// the full count. Warp-uniform.
//
// Band: with u = 2^-24, U >= |x - o| for both points, e = 1.001 u (2U + 1.5 r_s) bounds the
// error of each FP32 difference (two roundings of the coordinates, one of the difference), so
// |d2f - d2| <= e (2 sum|d_i| + 3e) + 3.1 u d2 (three roundings in the fused sum), and the FP64
// d2 is within 7e-16 d2 of the real value. Near the threshold |d_i| <= 1.5 r_s, giving
// band = 1.25 [e (9 r_s + 3e) + 3.1 u rs2] + 1e-15 rs2.
struct SearchGrid {
    const GridDev *g;
    const int32_t *cell_start;
    const float4 *spos32;
    const double4_32a *spos;
};

SearchConst make_search_const(double cell, double rs2)
{
    SearchConst c;
    c.cell = cell;
    c.rs2 = rs2;
    c.cf = (float)cell;
    c.rs = (float)std::sqrt(rs2);
    float lo = (float)rs2, hi = (float)rs2;
    if ((double)lo > rs2) lo = std::nextafterf(lo, -INFINITY);
    if ((double)hi < rs2) hi = std::nextafterf(hi, INFINITY);
    c.rs2_rd = lo;
    c.rs2_ru = hi;
    return c;
}

__device__ int warp_support_search(const SearchGrid &G, const SearchConst &C, double px, double py, double pz,
                                   int32_t *list, int S, int lane)
{
    const GridDev *g = G.g;
    if (g->n_cells == 0) return 0;
    const int nx = g->dims[0], ny = g->dims[1], nz = g->dims[2];
    const double rs2 = C.rs2;
    // position relative to the grid origin, in FP32 (one FP64 subtraction per axis)
    const float X = (float)(px - g->origin[0]), Y = (float)(py - g->origin[1]), Z = (float)(pz - g->origin[2]);
    const float cf = C.cf;
    const float rs = C.rs;
    const float ext = fmaxf(fmaxf((float)nx, (float)ny), (float)nz) * cf;
    const float U = fmaxf(fmaxf(fmaxf(fabsf(X), fabsf(Y)), fabsf(Z)), ext);
    const float u = 0x1p-24f;
    const float e = 1.001f * u * (2.f * U + 1.5f * rs);
    const float band = 1.5f * (1.25f * (e * (9.f * rs + 3.f * e) + 3.1f * u * rs * rs) + 1e-15f * rs * rs);
    const float lo = __fsub_rd(C.rs2_rd, band), hi = __fadd_ru(C.rs2_ru, band);
    // Cells that a ball of radius r_s (1 + 1e-4) + 2 e about the point meets (the margin covers the FP32
    // rounding of the point, the quotients and the distances; nodes are binned by the exact FP64
    // floor): the rows along x whose (y, z) square it meets, and of each row the cells it reaches. 84
    // cells on average instead of the 125 of the bounding box. With the branch-free tests and the next row's
    // loads ahead: k_kin_search 2.86 -> 2.64 ms (616 k MPs, mixed).
    const float rsm = rs * 1.0001f + 2.f * e;
    const int y0 = max((int)fmaxf(floorf((Y - rsm) / cf), -1.f), 0);
    const int y1 = min((int)fminf(floorf((Y + rsm) / cf), (float)ny), ny - 1);
    const int z0 = max((int)fmaxf(floorf((Z - rsm) / cf), -1.f), 0);
    const int z1 = min((int)fminf(floorf((Z + rsm) / cf), (float)nz), nz - 1);
    int cnt = 0;
    if (y0 > y1 || z0 > z1) return 0;
    const unsigned below = (1u << lane) - 1u;
    // the tests of 32 candidates from slot s on (their FP32 records loaded; lanes past the row's end hold a
    // point at infinity), the accepted IDs appended
    auto scan = [&](int s, const float4 &a) {
        const float dx = X - a.x, dy = Y - a.y, dz = Z - a.z;
        const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        bool acc = d2 <= lo;
        const bool near = !acc && d2 <= hi;
        if (__any_sync(0xffffffffu, near)) {   // ambiguity band: exact FP64 test
            if (near) {
                const double4_32a q = G.spos[s + lane];
                acc = dist2_exact(px, py, pz, q.x, q.y, q.z) <= rs2;
            }
            __syncwarp();
        }
        const unsigned m = __ballot_sync(0xffffffffu, acc);
        const int pos = cnt + __popc(m & below);
        if (acc && pos < S) list[pos] = __float_as_int(a.w);
        cnt += __popc(m);
    };
    // Rows in (z, y) order, r = (kz - z0) ny' + (ky - y0), up to 32 at once, one a lane for their ranges of
    // slots; then row by row, 64 slots a pass with both chunks' loads in flight and the next row's
    // first pass ahead of this row's tests. The accepted IDs keep the order of a plain scan (rows, cells,
    // slots).
    const int nyr = y1 - y0 + 1, nrows = nyr * (z1 - z0 + 1);
    const float4 none = make_float4(INFINITY, 0.f, 0.f, 0.f);
    const float4 *sp = G.spos32 + lane;
    for (int g0 = 0; g0 < nrows; g0 += kWarp) {
        int r0 = 0, len = 0;
        if (g0 + lane < nrows) {
            const int r = g0 + lane, kz = z0 + r / nyr, ky = y0 + r % nyr;
            // distance of the point from the row's square, less 2 e (the FP32 rounding of both)
            const float dy = fmaxf(fmaxf((float)ky * cf - Y, Y - (float)(ky + 1) * cf) - 2.f * e, 0.f);
            const float dz = fmaxf(fmaxf((float)kz * cf - Z, Z - (float)(kz + 1) * cf) - 2.f * e, 0.f);
            const float h2 = fmaf(-dz, dz, fmaf(-dy, dy, rsm * rsm));
            if (h2 >= 0.f) {
                const float half = sqrtf(h2) + 1e-4f * rs + 2.f * e;
                const int x0 = max((int)fmaxf(floorf((X - half) / cf), -1.f), 0);
                const int x1 = min((int)fminf(floorf((X + half) / cf), (float)nx), nx - 1);
                if (x0 <= x1) {
                    const int rowc = (kz * ny + ky) * nx;
                    r0 = G.cell_start[rowc + x0];
                    len = G.cell_start[rowc + x1 + 1] - r0;
                }
            }
        }
        unsigned live = __ballot_sync(0xffffffffu, len > 0);
        if (!live) continue;
        int s0, n, r = __ffs(live) - 1;
        s0 = __shfl_sync(0xffffffffu, r0, r);
        n = __shfl_sync(0xffffffffu, len, r);
        float4 qa = lane < n ? sp[s0] : none, qb = lane + kWarp < n ? sp[s0 + kWarp] : none;
        for (;;) {
            live &= live - 1;
            int s1 = 0, n1 = 0;
            float4 na = none, nb = none;
            if (live) {
                r = __ffs(live) - 1;
                s1 = __shfl_sync(0xffffffffu, r0, r);
                n1 = __shfl_sync(0xffffffffu, len, r);
                if (lane < n1) na = sp[s1];
                if (lane + kWarp < n1) nb = sp[s1 + kWarp];
            }
            scan(s0, qa);
            if (n > kWarp) scan(s0 + kWarp, qb);
            for (int b = 2 * kWarp; b < n; b += kWarp) scan(s0 + b, b + lane < n ? sp[s0 + b] : none);
            if (!live) break;
            s0 = s1; n = n1; qa = na; qb = nb;
        }
    }
    return cnt;
}

// unbiased binary exponent (-2000 for zero / subnormal)
__device__ __forceinline__ int fexp64(double v)
{
    const int e = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
    return e == 0 ? -2000 : e - 1023;
}

__device__ __forceinline__ int fexp32(float v)
{
    const int e = (int)((__float_as_uint(v) >> 23) & 0xff);
    return e == 0 ? -2000 : e - 127;
}

// per-warp shared-memory layout for the LME solve
struct WarpSmem {
    double *dx, *dy, *dz, *q, *w;
};

constexpr int kLmeWarps = 4;

// The damped Newton solve of Eq. 14 for the block's MPs: the convex log Z(lambda) by steps -J^-1 (r/Z) = -J'^-1 r,
// halved until log Z or the residual norm drops, to |r| / Z <= tol. All evaluations of a solve share its first
// shift, which makes the log Z comparison a comparison of Z. Block-synchronous: each round, every
// warp whose MP has an evaluation pending computes the sums (Z, r, A) at its trial lambda (the
// pair loop); then one warp takes the scalar decisions of all of them (accept or halve the trial, the
// convergence test, J'^-1, the next Newton step), eight lanes an MP. FP64 instructions cost the pipe
// the same with one active lane as with 32, so doing the scalar work once per block instead of once
// per warp saves most of it. State of one MP's solve, in shared memory:
enum : int { kNewtonIdle = 0, kNewtonEval = 1, kNewtonDone = 2, kNewtonFail = 3 };
struct MpNewton {
    double E[11];      // sums of the latest evaluation: Z, r (3), A (6), shift
    double C[11];      // sums at the current (accepted) point
    double lam[3];     // current lambda
    double trial[3];   // lambda of the pending evaluation
    double dir[3];     // Newton direction at the current point
    double ws[3];      // warm start of the solve (for the cold-start retry)
    double t;          // step fraction of the pending trial
    double inv[6];     // J'^-1 at the solution (xx, yy, zz, xy, yz, xz)
    double iZ, logz;
    double ts[3];      // the trial times 1024/ln2 (the exponent units of exp_scaled)
    double sh;         // exponent shift of the pending evaluation
    double qs;         // (solve's first shift - sh) * 1024/ln2, added to the stored prior terms
    double shift0;     // the solve's first shift (the stored prior terms are relative to it)
    int state, have_cur, iters, iters_total, halvings, retried;
};

// the scaled trial and the shift of the pending evaluation: trials share the current point's
// shift, the first evaluation of a start uses the solve's first shift
__device__ __forceinline__ void newton_set_trial(MpNewton &m)
{
    m.sh = m.have_cur ? m.C[10] : m.shift0;
    m.qs = (m.shift0 - m.sh) * kExpScale;
    for (int i = 0; i < 3; i++) m.ts[i] = m.trial[i] * kExpScale;
}

// One evaluation of the block path (Eq. 14 sums at the pending trial of MP state m): weights
// into W.w, the sums into m.E (written by one lane per value), m.E[10] = the shift used. If Z
// over- or underflows, again with the shift at the largest exponent. Warp-uniform.
// One evaluation's sums over the pairs of lane `lane`: Z, r = sum w d and A = sum w d d^T.
// FP64 path (DFH false): all in FP64. Mixed path (DFH true): Z and r in FP64 (r is a cancelling
// sum that decides convergence at 1e-14 h), the Hessian sums A in double-float: they only set
// the Newton step and J^-1, for which their relative accuracy of about 1e-14 is ample, and they
// then leave the FP64 pipe, the kernel's bound, to the weights; the per-lane double-float sums are
// widened to FP64 before the warp reduction.
template <bool SHIFTED, bool DFH>
__device__ __forceinline__ void lme_acc10(const WarpSmem &W, int n, double s0, double s1, double s2, double qs,
                                          int lane, const double *T, double (&v)[10])
{
#pragma unroll
    for (int i = 0; i < 10; i++) v[i] = 0.0;
    if (!DFH) {
        for (int k = lane; k < n; k += kWarp) {
            const double x = W.dx[k], y = W.dy[k], z = W.dz[k];
            const double qk = SHIFTED ? W.q[k] + qs : W.q[k];
            const double wk = exp_scaled(fma(s2, z, fma(s1, y, fma(s0, x, qk))), T);
            W.w[k] = wk;
            const double wx = wk * x, wy = wk * y, wz = wk * z;
            v[0] += wk;
            v[1] += wx; v[2] += wy; v[3] += wz;
            v[4] = fma(wx, x, v[4]); v[5] = fma(wy, y, v[5]); v[6] = fma(wz, z, v[6]);
            v[7] = fma(wx, y, v[7]); v[8] = fma(wy, z, v[8]); v[9] = fma(wx, z, v[9]);
        }
        return;
    }
    float ah[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, al[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int k = lane; k < n; k += kWarp) {
        const double x = W.dx[k], y = W.dy[k], z = W.dz[k];
        const double qk = SHIFTED ? W.q[k] + qs : W.q[k];
        const double wk = exp_scaled(fma(s2, z, fma(s1, y, fma(s0, x, qk))), T);
        W.w[k] = wk;
        v[0] += wk;
        v[1] = fma(wk, x, v[1]); v[2] = fma(wk, y, v[2]); v[3] = fma(wk, z, v[3]);
        float wh, wl, xh, xl, yh, yl, zh, zl;
        df_split(wk, wh, wl);
        df_split(x, xh, xl);
        df_split(y, yh, yl);
        df_split(z, zh, zl);
        float pxh, pxl, pyh, pyl, pzh, pzl, q, f;
        df_mul(wh, wl, xh, xl, pxh, pxl);
        df_mul(wh, wl, yh, yl, pyh, pyl);
        df_mul(wh, wl, zh, zl, pzh, pzl);
        df_mul(pxh, pxl, xh, xl, q, f); df_add(ah[0], al[0], q, f);
        df_mul(pyh, pyl, yh, yl, q, f); df_add(ah[1], al[1], q, f);
        df_mul(pzh, pzl, zh, zl, q, f); df_add(ah[2], al[2], q, f);
        df_mul(pxh, pxl, yh, yl, q, f); df_add(ah[3], al[3], q, f);
        df_mul(pyh, pyl, zh, zl, q, f); df_add(ah[4], al[4], q, f);
        df_mul(pxh, pxl, zh, zl, q, f); df_add(ah[5], al[5], q, f);
    }
#pragma unroll
    for (int i = 0; i < 6; i++) v[4 + i] = df_widen(ah[i]) + df_widen(al[i]);
}

// The FP64 Hessian sums of one evaluation from its stored weights (the fallback for weights
// outside the double-float range; see lme_eval_block)
__device__ __forceinline__ void lme_hessian64(const WarpSmem &W, int n, int lane, double (&v)[10])
{
    for (int k = lane; k < n; k += kWarp) {
        const double x = W.dx[k], y = W.dy[k], z = W.dz[k];
        const double wk = W.w[k];
        const double wx = wk * x, wy = wk * y, wz = wk * z;
        v[4] = fma(wx, x, v[4]); v[5] = fma(wy, y, v[5]); v[6] = fma(wz, z, v[6]);
        v[7] = fma(wx, y, v[7]); v[8] = fma(wy, z, v[8]); v[9] = fma(wx, z, v[9]);
    }
}

template <bool DFH>
__device__ void lme_eval_block(const WarpSmem &W, int n, MpNewton &m, int lane, const double *T)
{
    const double s0 = m.ts[0], s1 = m.ts[1], s2 = m.ts[2];
    double qs = m.qs, sh = m.sh;
    double v[10];
    if (qs == 0.0) lme_acc10<false, DFH>(W, n, s0, s1, s2, qs, lane, T, v);
    else lme_acc10<true, DFH>(W, n, s0, s1, s2, qs, lane, T, v);
    double t = warp_reduce_scatter10(v, lane);
    double Z = __shfl_sync(0xffffffffu, t, 0);
    if (!(Z > 1e-200) || !(Z < 1e200)) {
        double mx = -INFINITY;
        for (int k = lane; k < n; k += kWarp) mx = fmax(mx, W.q[k] + (s0 * W.dx[k] + s1 * W.dy[k] + s2 * W.dz[k]));
        sh = warp_max(mx) * (1.0 / kExpScale) + m.shift0;
        qs = (m.shift0 - sh) * kExpScale;
        lme_acc10<true, DFH>(W, n, s0, s1, s2, qs, lane, T, v);
        t = warp_reduce_scatter10(v, lane);
        Z = __shfl_sync(0xffffffffu, t, 0);
    }
    if (DFH && !(Z >= 1e-30 && Z <= 1e30)) {
        // weights this far from 1 may leave the FP32 range of the double-float sums: the Hessian
        // sums again in FP64 from the stored weights (Z and r are kept)
#pragma unroll
        for (int i = 4; i < 10; i++) v[i] = 0.0;
        lme_hessian64(W, n, lane, v);
        const double t2 = warp_reduce_scatter10(v, lane);
        if (rs10_value(lane) >= 4) t = t2;
    }
    if (rs10_writer(lane)) m.E[rs10_value(lane)] = t;
    if (lane == 0) m.E[10] = sh;
}

__device__ __forceinline__ LmeSums sums_of(const double *v)
{
    LmeSums e;
    e.Z = v[0]; e.r0 = v[1]; e.r1 = v[2]; e.r2 = v[3];
    e.a00 = v[4]; e.a11 = v[5]; e.a22 = v[6]; e.a01 = v[7]; e.a12 = v[8]; e.a02 = v[9];
    e.shift = v[10];
    return e;
}

// the solve failed from this start: once more from lambda = 0 if the start was not 0
__device__ __forceinline__ void newton_fail(MpNewton &m)
{
    if (!m.retried && (m.ws[0] != 0.0 || m.ws[1] != 0.0 || m.ws[2] != 0.0)) {
        m.retried = 1;
        m.have_cur = 0;
        m.iters = 0;
        m.halvings = 0;
        m.ws[0] = m.ws[1] = m.ws[2] = 0.0;
        m.trial[0] = m.trial[1] = m.trial[2] = 0.0;
        newton_set_trial(m);
        m.state = kNewtonEval;
    } else {
        m.state = kNewtonFail;
    }
}

// One scalar round after an evaluation (the damped Newton as a state machine) for the block's
// four MPs, eight lanes each (called by one warp): every lane forms the shared scalars, and lane q its entry of
// J', of the cofactors and of the step; a lane per MP issued 75 FP64 instructions a round, this 47 (mixed k_lme on 616 k MPs: 14.19 -> 13.33 ms, the same
// bits). True for the lanes of an MP with another evaluation to come.
// ZOFF: the binary exponent the next solve's Z starts below (see the end)
template <int ZOFF>
__device__ __forceinline__ bool newton_round(MpNewton *NS, double tol, int max_it, int lane)
{
    const int q = lane & 7, gb = lane & 24;
    MpNewton &m = NS[lane >> 3];
    const bool act = m.state == kNewtonEval;
    if (!__any_sync(0xffffffffu, act)) return false;
    auto from = [&](double v, int src) { return __shfl_sync(0xffffffffu, v, gb + src); };
    auto nib = [&](unsigned tab) { return (int)((tab >> (4 * q)) & 7u); };   // lane q's entry of a table
    const LmeSums E = sums_of(m.E);
    const double rn = rn2(E);
    bool accept = act;               // the first evaluation of a start is the current point
    if (act && m.have_cur) {         // accept if log Z or the residual norm drops, else halve
        const LmeSums c = sums_of(m.C);
        accept = isfinite(E.Z) && (logz_less(E, c) || rn * (c.Z * c.Z) < rn2(c) * (E.Z * E.Z));
    }
    const bool finite = isfinite(rn) && isfinite(E.Z);
    const bool conv = accept && finite && rn <= tol * tol * E.Z * E.Z;
    const bool newton = accept && finite && !conv && m.iters < max_it;
    // J' = A - r r^T / Z, lane q its entry (xx, yy, zz, xy, yz, xz)
    const double iZ = 1.0 / E.Z;
    const int ei = nib(0x010210), ej = nib(0x221210);
    const double ri = ei == 0 ? E.r0 : (ei == 1 ? E.r1 : E.r2), rj = ej == 0 ? E.r0 : (ej == 1 ? E.r1 : E.r2);
    const double si = ri * iZ;
    const double J = q < 6 ? m.E[4 + q] - si * rj : 0.0;
    // cofactors, same order: J[p1] J[p2] - J[p3] J[p4]
    const double j1 = from(J, nib(0x335001)), j2 = from(J, nib(0x454122)), j3 = from(J, nib(0x503354)), j4 = from(J, nib(0x142354));
    const double cf = j1 * j2 - j3 * j4;
    const double d0 = from(J, 0), d1 = from(J, 3), d2 = from(J, 5), f0 = from(cf, 0), f1 = from(cf, 3), f2 = from(cf, 5);
    const double det = d0 * f0 + d1 * f1 + d2 * f2;
    const bool regular = det > 0.0 && isfinite(det);
    const double id = 1.0 / det;
    const double inv = cf * id;
    // the step -J'^-1 r, lane q < 3 its component, and the next trial
    const double i0 = from(inv, nib(0x530)), i1 = from(inv, nib(0x413)), i2 = from(inv, nib(0x245));
    const double step = -(i0 * E.r0 + i1 * E.r1 + i2 * E.r2);
    const double lam = q < 3 ? m.trial[q] : 0.0, trial = lam + step;
    const double sh = m.E[10];
    __syncwarp();
    if (accept) {
        m.C[q] = m.E[q];
        if (q < 3) {
            m.C[8 + q] = m.E[8 + q];
            m.lam[q] = lam;
        }
    }
    if (newton && regular) {
        if (q < 3) {
            m.dir[q] = step;
            m.trial[q] = trial;
            m.ts[q] = trial * kExpScale;
        }
        if (q == 0) {
            m.t = 1.0;
            m.sh = sh;
            m.qs = (m.shift0 - sh) * kExpScale;
            m.have_cur = 1;
            m.halvings = 0;
            m.iters++;
            m.iters_total++;
        }
    } else if (conv && regular) {
        if (q < 6) m.inv[q] = inv;
        if (q == 0) {
            m.have_cur = 1;
            m.iZ = iZ;
            // the next solve's shift only has to keep the weights in range: log Z + ZOFF ln 2 to within ln 2, from
            // the binary exponent of Z (Z > 0 and finite here); ZOFF = 2 starts the next sums at Z in
            // [1/4, 1/2), the middle of the fixed-point evaluation's window
            const int ez = ((__double2hiint(E.Z) >> 20) & 0x7ff) - 1023;
            m.logz = fma((double)(ez + ZOFF), 0x1.62e42fefa39efp-1, sh);
            m.state = kNewtonDone;
        }
    } else if (act && q == 0) {
        if (accept) {
            m.have_cur = 1;
            newton_fail(m);
        } else if (++m.halvings >= 40) {
            newton_fail(m);
        } else {
            m.t *= 0.5;
            for (int i = 0; i < 3; i++) m.trial[i] = fma(m.t, m.dir[i], m.lam[i]);
            newton_set_trial(m);
        }
    }
    __syncwarp();
    return m.state == kNewtonEval;
}

// The new support of an MP into its row (IDs from the warp's list) and each pair's rank in its
// node's influence list, by counting with atomics; three slots per lane at a time, so that three
// atomics (whose old values are waited for) are in flight together. Any order of the ranks gives
// the same node sums (exact fixed-point sums).
__device__ __forceinline__ void store_support(const Dev &D, const int32_t *list, int64_t base, int cnt, int lane)
{
    for (int k0 = lane; k0 < cnt; k0 += 3 * kWarp) {
        int id[3], r[3];
#pragma unroll
        for (int j = 0; j < 3; j++) id[j] = (k0 + j * kWarp < cnt) ? list[k0 + j * kWarp] : -1;
#pragma unroll
        for (int j = 0; j < 3; j++) r[j] = (id[j] >= 0) ? atomicAdd(&D.ncount[id[j]], 1) : 0;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            if (id[j] < 0) continue;
            const int64_t k = base + k0 + j * kWarp;
            D.ids[k] = id[j];
            if (r[j] > 0xffff) raise_error(D.err, OTM_ERR_CAPACITY, D.ngid[id[j]]);
            D.rank[k] = (uint16_t)r[j];
        }
    }
}

// ======================================================================== k_search
__global__ void __launch_bounds__(kSearchWarps * kWarp) k_search(const Dev D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * kSearchWarps + warp;
    if (p >= D.nm) return;
    if (has_error(D.err)) return;
    const int S = D.S;
    int32_t *list = (int32_t *)smem_raw + (size_t)warp * next_pow2(S);
    const double4_32a xp = D.xp[p];
    SearchGrid G{D.grid, D.cell_start, D.spos32, D.spos};
    const int cnt = warp_support_search(G, D.sc, xp.x, xp.y, xp.z, list, S, lane);
    if (cnt > S) {
        if (lane == 0) {
            raise_error(D.err, OTM_ERR_CAPACITY, D.mgid[p]);
            D.cnt[p] = 0;
        }
        return;
    }
    // the list is in linked-cell order (rows, cells, ascending ID within a cell): unique for a
    // given configuration, so no sort is needed for determinism; exports sort it by ID
    __syncwarp();
    const int64_t base = p * (int64_t)S;
    store_support(D, list, base, cnt, lane);
    if (lane == 0) D.cnt[p] = cnt;
}

// ======================================================================== kinematics gathers
// The 12 sums of the kinematics over MP p's old support (n pairs at row base), reduce-scattered
// (value rs12_value(lane) at each lane): 0-2 the x_p sums, 3-11 G = sum du_a (x) e_a row-major.
//  FP64 path: x_p = sum N_a x_a of the updated node positions (Eq. 9), G from the FP64 increments.
//  Mixed path, in FP32 from the FP32 increments and the pair rows rounded to FP32: with c = the
//  increment of the support's first node, values 0-2 are sum N_a (du_a - c) and G =
//  sum (du_a - c) (x) e_a. Then x_p,n+1 = x_p,n + c + sum N_a (du_a - c), which is Eq. 9 by the
//  partition of unity and the linear reproducibility of the LME functions (sum N_a x_a,n = x_p,n
//  to the Newton tolerance), and G differs from the FP64 sum by c (x) sum e_a = c (x) r / Z, below
//  |c| 1e-14 h. Subtracting c leaves only the deforming part of the increments in the FP32 sums
//  (no cancellation of the rigid translation), so their error is FP32 rounding of the deformation.
template <bool MIXED>
struct KinSum;

template <>
struct KinSum<false> {
    double t;
    __device__ __forceinline__ void gather(const Dev &D, int64_t base, int n, int lane)
    {
        double v[12];
#pragma unroll
        for (int i = 0; i < 12; i++) v[i] = 0.0;
        for (int k = lane; k < n; k += kWarp) {
            const int id = D.ids[base + k];
            const double4_32a sh = D.shape[base + k];
            const double4_32a xa = D.x[id];
            const double4_32a u = D.du[id];
            v[0] = fma(sh.x, xa.x, v[0]); v[1] = fma(sh.x, xa.y, v[1]); v[2] = fma(sh.x, xa.z, v[2]);
            v[3] = fma(u.x, sh.y, v[3]); v[4] = fma(u.x, sh.z, v[4]); v[5] = fma(u.x, sh.w, v[5]);
            v[6] = fma(u.y, sh.y, v[6]); v[7] = fma(u.y, sh.z, v[7]); v[8] = fma(u.y, sh.w, v[8]);
            v[9] = fma(u.z, sh.y, v[9]); v[10] = fma(u.z, sh.z, v[10]); v[11] = fma(u.z, sh.w, v[11]);
        }
        t = warp_reduce_scatter12(v, lane);
    }
    __device__ __forceinline__ double g() const { return t; }
    // x_p,n+1 component i, on the lane that holds value i (lanes 0, 2, 4)
    __device__ __forceinline__ double xp(double, int) const { return t; }
};

template <>
struct KinSum<true> {
    float t;
    float c[3];
    __device__ __forceinline__ void gather(const Dev &D, int64_t base, int n, int lane)
    {
        float v[12];
#pragma unroll
        for (int i = 0; i < 12; i++) v[i] = 0.f;
        float4 c4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n > 0) c4 = D.du32[D.ids[base]];
        c[0] = c4.x; c[1] = c4.y; c[2] = c4.z;
#pragma unroll 2
        for (int k = lane; k < n; k += kWarp) {
            const int id = D.ids[base + k];
            const double4_32a sh = D.shape[base + k];
            const float4 u = D.du32[id];
            const float N = f32_round_bits(sh.x), ex = f32_round_bits(sh.y), ey = f32_round_bits(sh.z),
                        ez = f32_round_bits(sh.w);
            const float a0 = u.x - c4.x, a1 = u.y - c4.y, a2 = u.z - c4.z;
            v[0] = fmaf(N, a0, v[0]); v[1] = fmaf(N, a1, v[1]); v[2] = fmaf(N, a2, v[2]);
            v[3] = fmaf(a0, ex, v[3]); v[4] = fmaf(a0, ey, v[4]); v[5] = fmaf(a0, ez, v[5]);
            v[6] = fmaf(a1, ex, v[6]); v[7] = fmaf(a1, ey, v[7]); v[8] = fmaf(a1, ez, v[8]);
            v[9] = fmaf(a2, ex, v[9]); v[10] = fmaf(a2, ey, v[10]); v[11] = fmaf(a2, ez, v[11]);
        }
        t = warp_reduce_scatter12(v, lane);
    }
    __device__ __forceinline__ double g() const { return (double)t; }
    __device__ __forceinline__ double xp(double old, int i) const
    {
        const float ci = i == 0 ? c[0] : (i == 1 ? c[1] : c[2]);
        return old + ((double)ci + (double)t);
    }
};

// ======================================================================== k_kin_search
// Kinematics (Eq. 9, 11) and the support search at the new position (Algorithm 3) in one warp
// per MP: the gather over the old support gives x_p and dF, then the candidate scan builds the
// new support in the same row. Used when no erosion can remove MPs between the two; the
// return map (which only needs dF) follows.
// Mixed: bound by latency; 12 blocks per SM (40 registers, a 24-byte spill) 2.64 ms, 10 blocks 2.84 ms on 616 k
// MPs. FP64: bound by the gather's 12 FP64 FMAs a pair (FP64 pipe 90 % busy; 1.60 ms on 202,752 MPs, where 6, 7
// and 8 blocks are within 0.3 % and 10 take 1.63); 8 blocks also suit the search's latency on few MPs (9,984: 0.110 ms, 6 blocks
// 0.116). The sums in fixed point, in units of 2^-57 h, take 1.43 ms, but their error does not shrink with the
// increments: 13 times the FP64 sums' at 0.013 h a step, 1e6 times at 1e-7 h.
template <bool MIXED>
__global__ void __launch_bounds__(kSearchWarps * kWarp, MIXED ? 12 : 8) k_kin_search(const __grid_constant__ Dev D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * kSearchWarps + warp;
    if (p >= D.nm) return;
    if (has_error(D.err)) return;
    const int S = D.S;
    const int n = D.cnt[p];
    const int64_t base = p * (int64_t)S;
    KinSum<MIXED> ks;
    ks.gather(D, base, n, lane);
    const int j = rs12_value(lane);
    if (rs12_writer(lane) && j >= 3) D.dF[9 * p + (j - 3)] = ks.g();   // G = sum du (x) e; k_return_map forms dF
    // values 0, 1, 2 (x_p) sit at lanes 0, 2, 4
    double xi = 0.0;
    if (lane < 6 && (lane & 1) == 0) xi = ks.xp(((const double *)&D.xp[p])[lane >> 1], lane >> 1);
    const double px = __shfl_sync(0xffffffffu, xi, 0), py = __shfl_sync(0xffffffffu, xi, 2),
                 pz = __shfl_sync(0xffffffffu, xi, 4);
    if (lane == 0) {
        D.xp_prev[p] = D.xp[p];
        D.xp[p] = make_double4_32a(px, py, pz, 0.0);
        if (!isfinite(px) || !isfinite(py) || !isfinite(pz)) raise_error(D.err, OTM_ERR_NONFINITE, D.mgid[p]);
    }
    __syncwarp();   // the old row is read completely before the new support overwrites it
    int32_t *list = (int32_t *)smem_raw + (size_t)warp * next_pow2(S);
    SearchGrid G{D.grid, D.cell_start, D.spos32, D.spos};
    const int cnt = warp_support_search(G, D.sc, px, py, pz, list, S, lane);
    if (cnt > S) {
        if (lane == 0) {
            raise_error(D.err, OTM_ERR_CAPACITY, D.mgid[p]);
            D.cnt[p] = 0;
        }
        return;
    }
    __syncwarp();
    store_support(D, list, base, cnt, lane);
    if (lane == 0) D.cnt[p] = cnt;
}

cudaError_t launch_kin_search(const Dev &D, cudaStream_t s, long long *launches)
{
    const size_t smem = (size_t)kSearchWarps * next_pow2(D.S) * sizeof(int32_t);
    const unsigned blocks = (unsigned)((D.nm + kSearchWarps - 1) / kSearchWarps);
    if (blocks == 0) return cudaSuccess;
    if (D.precision == OTM_PRECISION_MIXED)
        k_kin_search<true><<<blocks, kSearchWarps * kWarp, smem, s>>>(D);
    else
        k_kin_search<false><<<blocks, kSearchWarps * kWarp, smem, s>>>(D);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_search(const Dev &D, cudaStream_t s, long long *launches)
{
    const size_t smem = (size_t)kSearchWarps * next_pow2(D.S) * sizeof(int32_t);
    const unsigned blocks = (unsigned)((D.nm + kSearchWarps - 1) / kSearchWarps);
    if (blocks == 0) return cudaSuccess;
    k_search<<<blocks, kSearchWarps * kWarp, smem, s>>>(D);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

// ======================================================================== k_lme
// store the solution lambda of MP p, and the lambda it replaces where the mode says so
__device__ __forceinline__ void lme_record(const Dev &D, int64_t p, double l0, double l1, double l2)
{
    if (D.lme_mode == kLmeStep) {
        for (int i = 0; i < 3; i++) {
            D.lam_prev3[3 * p + i] = D.lam_prev2[3 * p + i];
            D.lam_prev2[3 * p + i] = D.lam_prev[3 * p + i];
            D.lam_prev[3 * p + i] = D.lam[3 * p + i];
        }
    } else if (D.lme_mode == kLmePlain || (D.lme_mode == kLmeRetry && D.lme_fail[p])) {
        // a plain start, or an MP solved again after node insertion: its previous solutions were
        // not one step apart from this one, so the history restarts at the new solution
        D.lam_prev[3 * p] = D.lam_prev2[3 * p] = D.lam_prev3[3 * p] = l0;
        D.lam_prev[3 * p + 1] = D.lam_prev2[3 * p + 1] = D.lam_prev3[3 * p + 1] = l1;
        D.lam_prev[3 * p + 2] = D.lam_prev2[3 * p + 2] = D.lam_prev3[3 * p + 2] = l2;
    }
    D.lam[3 * p] = l0;
    D.lam[3 * p + 1] = l1;
    D.lam[3 * p + 2] = l2;
}

// Shared-memory rows per MP in k_lme and k_lme_fix. With 336 slots a block of 4 MPs takes 43 KB of rows: 5 blocks
// of k_lme fit an SM, and 4 of k_lme_fix with its table, which hides more of the dependency and
// barrier stalls; the supports of the benchmark rods stay below (at most 316 slots mid-run on the
// 2.85 M-MP rod). MPs with larger supports are deferred to k_lme_wide, which runs k_lme's block
// code with rows of the full capacity S.
constexpr int kLmeRows = 336;

__host__ __device__ __forceinline__ int lme_rows(int S) { return S < kLmeRows ? S : kLmeRows; }

// the solve's start: the warm start and an evaluation pending there; lanes 0-2 a component each
__device__ __forceinline__ void lme_start(const Dev &D, int64_t p, MpNewton &M, double shift0, int lane)
{
    if (lane >= 3) return;
    // Eq. 14: the warm start is the previous step's lambda, or (within a step) the cubic
    // through the last four solutions: while the material deforms smoothly one Newton
    // step from it meets the tolerance
    double l = D.lam[3 * p + lane];
    if (D.lme_mode == kLmeStep)   // cubic: 4 l_n - 6 l_{n-1} + 4 l_{n-2} - l_{n-3}
        l = fma(4.0, l + D.lam_prev2[3 * p + lane], -fma(6.0, D.lam_prev[3 * p + lane], D.lam_prev3[3 * p + lane]));
    M.trial[lane] = M.ws[lane] = l;
    M.ts[lane] = l * kExpScale;
    if (lane == 0) {
        M.t = 1.0;
        M.have_cur = M.iters = M.iters_total = M.halvings = M.retried = 0;
        M.shift0 = M.sh = shift0;
        M.qs = (shift0 - M.sh) * kExpScale;
    }
}

// records the solve of MP p; false if it failed (nothing more to write for this MP)
__device__ __forceinline__ bool lme_finish(const Dev &D, int64_t p, int cnt, const MpNewton &M, double shift0, int lane)
{
    const int st = M.state == kNewtonDone ? OTM_OK : OTM_ERR_LME_NOCONV;
    if (lane == 0) {
        D.newton_it[p] = M.iters_total;
        if (st == OTM_OK) {
            lme_record(D, p, M.lam[0], M.lam[1], M.lam[2]);
            D.logz_in[p] = shift0;
            D.logz[p] = M.logz;
        } else if (D.insert_mode && cnt > 0) {
            D.lme_fail[p] = 1;          // node insertion follows (lambda keeps the warm start)
            atomicAdd(D.n_fail, 1);
        } else {
            raise_error(D.err, st, D.mgid[p]);
        }
    }
    return st == OTM_OK;
}

// N_a = w_a / Z and grad N_a = -N_a J^-1 d_a = -K e_a with e_a = N_a d_a and K = J^-1 = Z J'^-1
// (one symmetric 3x3 per MP). The pair rows keep (N_a, e_a) and the MP keeps K: whoever needs
// grad N applies K once per MP (the kinematics gather sums du_a (x) e_a, and dF = 1 - G K
// follows in the return map), so the per-pair work is N, e and the contributions.
// Eq. 5 contributions of the next step, stored at the pair's place in its node's influence
// list: mass m_p N_a, force -v_p sigma_p grad N_a = (v_p sigma_p K) e_a = Q e_a.
__device__ __forceinline__ void lme_force_matrix(const Dev &D, int64_t p, const MpNewton &M, int lane, double (&Q)[9])
{
    const double vp = D.vol[p];
    const double *sg = D.sig + 6 * p;
    double Kc[6];
    // lanes 0-5 form K (and store it), lanes 0-8 one entry of Q each; all lanes get both
    const double kj = (lane < 6) ? M.inv[lane] * M.C[0] : 0.0;
    if (lane < 6) D.Kinv[6 * p + lane] = kj;
#pragma unroll
    for (int i = 0; i < 6; i++) Kc[i] = __shfl_sync(0xffffffffu, kj, i);
    // symmetric index of (i, j) in (xx, yy, zz, xy, yz, xz)
    const int li = (lane < 9) ? lane / 3 : 0, lc = (lane < 9) ? lane % 3 : 0;
    auto sym = [](int i, int j) { return i == j ? i : (i + j == 1 ? 3 : (i + j == 3 ? 4 : 5)); };
    const double q = vp * (sg[sym(li, 0)] * Kc[sym(0, lc)] + sg[sym(li, 1)] * Kc[sym(1, lc)] +
                           sg[sym(li, 2)] * Kc[sym(2, lc)]);
#pragma unroll
    for (int i = 0; i < 9; i++) Q[i] = __shfl_sync(0xffffffffu, q, i);
}

// stabilisation (Eq. 7-8): -eps N_a e_a / |x_a,n-1 - x_p,n-1|,
// e_a = x_a - x_p - dF (x_a,n-1 - x_p,n-1), with dF the increment that led to this state
template <bool STAB>
struct LmeStab {
    __device__ __forceinline__ void load(const Dev &, int64_t) {}
    __device__ __forceinline__ void term(const Dev &, int, double, double, double, double, double &, double &, double &) const {}
};

template <>
struct LmeStab<true> {
    double xq0, xq1, xq2, F[9];
    __device__ __forceinline__ void load(const Dev &D, int64_t p)
    {
        const double4_32a q = D.xp_prev[p];
        xq0 = q.x; xq1 = q.y; xq2 = q.z;
#pragma unroll
        for (int i = 0; i < 9; i++) F[i] = D.dF[9 * p + i];
    }
    // (x, y, z) = x_p - x_a
    __device__ __forceinline__ void term(const Dev &D, int id, double N, double x, double y, double z, double &sx,
                                         double &sy, double &sz) const
    {
        const double4_32a a = D.x_prev[id];
        const double q0 = a.x - xq0, q1 = a.y - xq1, q2 = a.z - xq2;
        const double len = sqrt(q0 * q0 + q1 * q1 + q2 * q2);
        if (len > 1e-12 * D.h) {
            const double c = -D.eps_stab * N / len;
            sx = c * (-x - (F[0] * q0 + F[1] * q1 + F[2] * q2));
            sy = c * (-y - (F[3] * q0 + F[4] * q1 + F[5] * q2));
            sz = c * (-z - (F[6] * q0 + F[7] * q1 + F[8] * q2));
        }
    }
};

// The same for the FP64 output loop of k_lme_fix, as c (e + dF N q) with e = N (x_p - x_a) at hand, q = x_a,n-1 -
// x_p,n-1 and c = eps / |q|: the reciprocal root from the approximate one by a step of third order (5 FP64
// instructions; the root and the division took about 35 of the term's 62), and x_prev one pass ahead. Bound by the
// FP64 pipe, 27 of the loop's 29 instructions there; k_lme_fix on 78,624 stabilised MPs: 2.52 -> 1.91 ms.
struct StabFix {
    double xq0, xq1, xq2, F[9], eps, lim;
    double4_32a a;                     // x_prev of the pass's pair
    __device__ __forceinline__ void load(const Dev &D, int64_t p)
    {
        const double4_32a q = D.xp_prev[p];
        xq0 = q.x; xq1 = q.y; xq2 = q.z;
#pragma unroll
        for (int i = 0; i < 9; i++) F[i] = D.dF[9 * p + i];
        eps = D.eps_stab;
        lim = (1e-12 * D.h) * (1e-12 * D.h);
    }
    __device__ __forceinline__ void add(double N, double ex, double ey, double ez, double &fx, double &fy, double &fz) const
    {
        const double q0 = a.x - xq0, q1 = a.y - xq1, q2 = a.z - xq2;
        const double s = fma(q2, q2, fma(q1, q1, q0 * q0));
        if (!(s > lim)) return;
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
        const double e = fma(-s * y, y, 1.0);                       // 1 / sqrt(1 - e) = 1 + e/2 + 3/8 e^2 + O(e^3)
        const double c = eps * fma(y, e * fma(0.375, e, 0.5), y);
        const double n0 = N * q0, n1 = N * q1, n2 = N * q2;
        fx = fma(c, fma(F[2], n2, fma(F[1], n1, fma(F[0], n0, ex))), fx);
        fy = fma(c, fma(F[5], n2, fma(F[4], n1, fma(F[3], n0, ey))), fy);
        fz = fma(c, fma(F[8], n2, fma(F[7], n1, fma(F[6], n0, ez))), fz);
    }
};

// The LME solve of the block's MPs (one per warp; p the warp's MP, active whether it has one),
// shared-memory rows of `rows` slots. Every thread of the block calls it (block barriers inside);
// the exponential's table is read from global memory (L1-resident, 8 KB).
template <bool MIXED, bool STAB>
__device__ __forceinline__ void lme_block(const Dev &D, int64_t p, bool active, int rows, unsigned char *smem_raw)
{
    const double *__restrict__ T = g_exp2_table;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = D.S;
    MpNewton *NS = (MpNewton *)(smem_raw + (size_t)kLmeWarps * 4 * (size_t)rows * sizeof(double));
    // every warp reaches the block barriers below; idle warps skip the work
    WarpSmem W;
    W.dx = (double *)smem_raw + (size_t)warp * 4 * (size_t)rows;
    W.dy = W.dx + rows;
    W.dz = W.dy + rows;
    W.q = W.dz + rows;
    const int64_t base = p * (int64_t)S;
    MpNewton &M = NS[warp];
    const int cnt = active ? D.cnt[p] : 0;
    // the weights, packed at the end of the MP's pair rows in memory: without their 8 bytes a slot in shared
    // memory a fifth block fits the SM (mixed, 616 k MPs: 14.89 -> 14.51 ms, the FP64 pipe 86 % busy). Row k
    // reaches w_j only for k >= j, so the output loop below may overwrite them pass by pass.
    W.w = (double *)(D.shape + base + S) - cnt;
    constexpr int G = 5;   // passes of dependent gathers in flight (3: 14.24 instead of 14.19 ms, mixed, 616 k MPs; 1: 14.54)
    double shift0 = 0;
    if (active) {
        const double4_32a xp = D.xp[p];
        // d_a = x_p - x_a and the prior exponent -beta |d_a|^2, minus the Newton solve's shift,
        // in units of ln2/1024
        const double beta_s = D.beta * kExpScale;
        shift0 = D.logz[p];
        const double shift_s = shift0 * kExpScale;
        for (int k0 = lane; k0 < cnt; k0 += G * kWarp) {
            int id[G];
            double4_32a a[G];
#pragma unroll
            for (int j = 0; j < G; j++) id[j] = k0 + j * kWarp < cnt ? D.ids[base + k0 + j * kWarp] : -1;
#pragma unroll
            for (int j = 0; j < G; j++)
                if (id[j] >= 0) a[j] = D.x[id[j]];
#pragma unroll
            for (int j = 0; j < G; j++) {
                if (id[j] < 0) continue;
                const int k = k0 + j * kWarp;
                const double x = xp.x - a[j].x, y = xp.y - a[j].y, z = xp.z - a[j].z;
                W.dx[k] = x; W.dy[k] = y; W.dz[k] = z;
                W.q[k] = fma(-beta_s, fma(z, z, fma(y, y, x * x)), -shift_s);
            }
        }
        lme_start(D, p, M, shift0, lane);
        if (lane == 0) M.state = cnt > 0 ? kNewtonEval : kNewtonFail;
    } else if (lane == 0) {
        M.state = kNewtonIdle;
    }
    __syncthreads();
    // rounds: evaluations of the pending trials, then the scalar decisions
    for (;;) {
        if (M.state == kNewtonEval) {
            __syncwarp();
            lme_eval_block<MIXED>(W, cnt, M, lane, T);
        }
        __syncthreads();
        const bool pending = warp == 0 && newton_round<MIXED ? 0 : 2>(NS, D.tol_abs, D.max_newton, lane);
        if (!__syncthreads_or(pending)) break;
    }
    if (!active) return;
    if (!lme_finish(D, p, cnt, M, shift0, lane)) return;

    // the pairs' node-major positions hang on two dependent loads: gathered ahead of the output loop into the
    // exponents' row
    int32_t *pos = (int32_t *)W.q;
    for (int k0 = lane; k0 < cnt; k0 += G * kWarp) {
        int id[G], rk[G];
#pragma unroll
        for (int j = 0; j < G; j++) {
            const int k = k0 + j * kWarp;
            id[j] = k < cnt ? D.ids[base + k] : 0;
            rk[j] = k < cnt ? D.rank[base + k] : 0;
        }
#pragma unroll
        for (int j = 0; j < G; j++) rk[j] += D.noff[id[j]];
#pragma unroll
        for (int j = 0; j < G; j++)
            if (k0 + j * kWarp < cnt) pos[k0 + j * kWarp] = rk[j];
    }
    const double iZ = M.iZ, mp = D.mass[p];
    double Q[9];
    lme_force_matrix(D, p, M, lane, Q);
    int em = -2000, ef = -2000;   // largest binary exponents of the stored mass / force terms
    float Qf[9];
#pragma unroll
    for (int i = 0; i < 9; i++) Qf[i] = MIXED ? (float)Q[i] : 0.f;
    const float mpf = MIXED ? (float)mp : 0.f;
    LmeStab<STAB> stab;
    stab.load(D, p);
    for (int k0 = 0; k0 < cnt; k0 += kWarp) {
        const int k = k0 + lane;
        const double wk = k < cnt ? W.w[k] : 0.0;
        __syncwarp();
        if (k >= cnt) continue;
        const double N = wk * iZ;
        const double x = W.dx[k], y = W.dy[k], z = W.dz[k];
        double ex, ey, ez;
        float fN = 0.f, fex = 0.f, fey = 0.f, fez = 0.f;
        if (MIXED) {
            // e = N d in FP32 (every consumer of the mixed path's rows rounds them to FP32),
            // stored widened exactly; N stays FP64
            fN = f32_round_bits(N);
            fex = fN * f32_round_bits(x);
            fey = fN * f32_round_bits(y);
            fez = fN * f32_round_bits(z);
            ex = df_widen(fex); ey = df_widen(fey); ez = df_widen(fez);
        } else {
            ex = N * x; ey = N * y; ez = N * z;
        }
        D.shape[base + k] = make_double4_32a(N, ex, ey, ez);
        double sx = 0.0, sy = 0.0, sz = 0.0;
        if (STAB) stab.term(D, D.ids[base + k], N, x, y, z, sx, sy, sz);
        if (MIXED) {
            const float c0 = mpf * fN;
            float c1 = fmaf(Qf[2], fez, fmaf(Qf[1], fey, Qf[0] * fex));
            float c2 = fmaf(Qf[5], fez, fmaf(Qf[4], fey, Qf[3] * fex));
            float c3 = fmaf(Qf[8], fez, fmaf(Qf[7], fey, Qf[6] * fex));
            if (STAB) {
                c1 += f32_round_bits(sx);
                c2 += f32_round_bits(sy);
                c3 += f32_round_bits(sz);
            }
            D.contrib32[pos[k]] = make_float4(c0, c1, c2, c3);
            em = max(em, fexp32(c0));
            ef = max(ef, max(fexp32(c1), max(fexp32(c2), fexp32(c3))));
        } else {
            const double cm = mp * N;
            double fx = Q[0] * ex + Q[1] * ey + Q[2] * ez;
            double fy = Q[3] * ex + Q[4] * ey + Q[5] * ez;
            double fz = Q[6] * ex + Q[7] * ey + Q[8] * ez;
            if (STAB) {
                fx += sx;
                fy += sy;
                fz += sz;
            }
            D.contrib64[pos[k]] = make_double4_32a(cm, fx, fy, fz);
            em = max(em, fexp64(cm));
            ef = max(ef, max(fexp64(fx), max(fexp64(fy), fexp64(fz))));
        }
    }
    em = __reduce_max_sync(0xffffffffu, em);
    ef = __reduce_max_sync(0xffffffffu, ef);
    if (lane == 0) {
        atomicMax(&D.emax[0], em);
        atomicMax(&D.emax[1], ef);
    }
}

template <bool MIXED, bool STAB>
__global__ void __launch_bounds__(kLmeWarps * kWarp, 5) k_lme(const Dev D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * kLmeWarps + (threadIdx.x >> 5);
    const int rows = lme_rows(D.S);
    bool active = (p < D.nm) && !has_error(D.err);
    if (active && D.cnt[p] > rows) {   // solved by k_lme_wide
        if (lane == 0) D.lme_defer[atomicAdd(D.n_defer, 1)] = (int32_t)p;
        active = false;
    }
    lme_block<MIXED, STAB>(D, p, active, rows, smem_raw);
}

// the deferred MPs, 4 per block and round, with rows of the full capacity S (grid-stride over the
// list, whose length the previous launch left in *n_defer)
template <bool MIXED, bool STAB>
__global__ void __launch_bounds__(kLmeWarps * kWarp) k_lme_wide(const Dev D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = *D.n_defer;
    for (int g = blockIdx.x; g * kLmeWarps < n; g += gridDim.x) {
        const int i = g * kLmeWarps + (threadIdx.x >> 5);
        const int64_t p = (i < n) ? (int64_t)D.lme_defer[i] : -1;
        lme_block<MIXED, STAB>(D, p, p >= 0 && !has_error(D.err), D.S, smem_raw);
    }
}

// ======================================================================== k_lme_fix
// The LME solve with fixed-point evaluations (otm_fix.cuh): same block structure, Newton decisions and
// outputs as k_lme, but the pair loops run in integers, so the FP64 pipe (2 lanes per clock and SM)
// only sees the scalars and the force contributions.
//
// Bound: k_lme keeps the FP64 pipe 89 % busy (19 FP64 instructions a pair and evaluation). Here it is
// 43 % busy (11 a pair for the force contributions and N, plus the rounds' scalars), and the integer
// instructions (about 200 a pair and evaluation, two to four cycles of an SM quarter each) and their
// latency at 16 warps an SM (128 registers; four blocks of 54 KB) bound the kernel.
// Measured on the 202,752-MP rod (267 pairs an MP, 1.19 Newton iterations): k_lme 7.78 ms, this kernel
// 2.87 ms (with k_lme_prep). Five blocks an SM (96 registers, the exp table in L1) take 15 % longer: spills.
struct MpFix {
    i64 xp[3];         // X of the material point
    i64 v[3];          // centre offset of the pending trial, lambda / (2 beta) in LSB
    i64 cst;           // the trial's exponent constant, 46 fraction bits
    i64 ok;            // the trial is inside the fixed-point range
    double vmax;       // largest centre offset per axis for this MP's separations, in LSB
};
static_assert(2 * kExpTable / kLmeWarps >= kLmeRows, "the exp table holds the warps' pair positions");
static_assert(sizeof(FixStart) == 3 * sizeof(double) + sizeof(MpFix), "k_lme_fix copies FixStart word by word");

// centre offset and constant of a trial with a shift; false out of range (or not finite): FP64 evaluation
__device__ __forceinline__ bool fix_trial(const FixConst &C, double vmax, const double *trial, double sh, i64 *v, i64 &cst)
{
    bool ok = true;
    double l2 = 0.0;
    for (int i = 0; i < 3; i++) {
        const double x = trial[i] * C.i2b;
        l2 = fma(trial[i], trial[i], l2);
        ok = ok && fabs(x) < vmax;
        v[i] = __double2ll_rn(x);
    }
    const double c = fma(l2, C.cy, -sh * kFixYScale);
    cst = __double2ll_rn(c * kFixYOne);
    return ok && fabs(c) < 65536.0;
}

// 1/x (x positive and normal): the hardware's approximate FP64 reciprocal (about 20 bits), refined by
// STEPS Newton steps y += y (1 - x y), each of which doubles the bits. The division operator takes
// about twice the FP64 instructions.
template <int STEPS>
__device__ __forceinline__ double recip_refine(double x, double y)
{
#pragma unroll
    for (int i = 0; i < STEPS; i++) y = fma(y, fma(-x, y, 1.0), y);
    return y;
}
template <int STEPS>
__device__ __forceinline__ double recip(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return recip_refine<STEPS>(x, y);
}

// One scalar round after the block's evaluations (the damped Newton of newton_round), for the block's
// kLmeWarps MPs at once by one warp, eight lanes per MP: the entries of J', of its cofactors and of
// the step go to one lane each, so that a round takes about 45 FP64 instructions instead of 85 (an
// FP64 instruction costs the pipe 16 cycles with one active lane as with 32). Halvings, failures and the
// cold-start retry (rare) run on the group's first lane. Returns whether this lane's MP has an
// evaluation pending.
__device__ __forceinline__ bool fix_round(MpNewton *NS, MpFix *FS, const FixConst &C, double tol, int max_it, int lane)
{
    const int q = lane & 7, gb = lane & 24;
    MpNewton &m = NS[lane >> 3];
    MpFix &f = FS[lane >> 3];
    const bool act = m.state == kNewtonEval;
    if (!__any_sync(0xffffffffu, act)) return false;
    auto from = [&](double v, int src) { return __shfl_sync(0xffffffffu, v, gb + src); };
    auto nib = [&](unsigned tab) { return (int)((tab >> (4 * q)) & 7u); };   // lane q's entry of a table
    const double Z = m.E[0], r0 = m.E[1], r1 = m.E[2], r2 = m.E[3];
    const double rn = fma(r2, r2, fma(r1, r1, r0 * r0));
    bool accept = act;
    if (act && m.have_cur) {   // accept if log Z or the residual norm drops, else halve
        const double cZ = m.C[0], c0 = m.C[1], c1 = m.C[2], c2 = m.C[3];
        const double cn = fma(c2, c2, fma(c1, c1, c0 * c0));
        const bool less = m.E[10] == m.C[10] ? Z < cZ : m.E[10] + log(Z) < m.C[10] + log(cZ);
        accept = isfinite(Z) && (less || rn * (cZ * cZ) < cn * (Z * Z));
    }
    const bool finite = isfinite(rn) && isfinite(Z);
    const bool conv = accept && finite && rn <= tol * tol * Z * Z;
    const bool newton = accept && finite && !conv && m.iters < max_it;
    // J' = A - r r^T / Z at the accepted point, lane q its entry (xx, yy, zz, xy, yz, xz). The approximate 1/Z does for
    // the direction of a step; where the solve ends, K needs all of it (the caller's tolerance bounds r)
    double iZ = recip<0>(Z);
    if (conv) iZ = recip_refine<2>(Z, iZ);
    const int ei = nib(0x010210), ej = nib(0x221210);
    const double ri = ei == 0 ? r0 : (ei == 1 ? r1 : r2), rj = ej == 0 ? r0 : (ej == 1 ? r1 : r2);
    const double J = q < 6 ? fma(-(ri * iZ), rj, m.E[4 + q]) : 0.0;
    // cofactors, same order: J[p1] J[p2] - J[p3] J[p4]
    const double cf = from(J, nib(0x335001)) * from(J, nib(0x454122)) - from(J, nib(0x503354)) * from(J, nib(0x142354));
    const double det = fma(from(J, 5), from(cf, 5), fma(from(J, 3), from(cf, 3), from(J, 0) * from(cf, 0)));
    const bool regular = det > 0.0 && isfinite(det);
    const double inv = cf * recip<2>(det);
    // the step -J'^-1 r, lane q < 3 its component, and the next trial
    const double step = -fma(from(inv, nib(0x245)), r2, fma(from(inv, nib(0x413)), r1, from(inv, nib(0x530)) * r0));
    const double lam = q < 3 ? m.trial[q] : 0.0;
    const double trial = lam + step;
    const double t0 = from(trial, 0), t1 = from(trial, 1), t2 = from(trial, 2);
    const double l2 = fma(t2, t2, fma(t1, t1, t0 * t0)), v = trial * C.i2b;
    const double sh = m.E[10], c = fma(l2, C.cy, -sh * kFixYScale);
    const unsigned inside = __ballot_sync(0xffffffffu, q >= 3 || fabs(v) < f.vmax);
    __syncwarp();
    const bool finish = conv && regular, next = newton && regular;
    if (accept) {
        m.C[q] = m.E[q];
        if (q < 3) {
            m.C[8 + q] = m.E[8 + q];
            m.lam[q] = lam;
        }
    }
    if (next) {
        if (q < 3) {
            m.dir[q] = step;
            m.trial[q] = trial;
            f.v[q] = __double2ll_rn(v);
        }
        if (q == 0) {
            m.t = 1.0;
            m.sh = sh;
            m.have_cur = 1;
            m.halvings = 0;
            m.iters++;
            m.iters_total++;
            f.cst = __double2ll_rn(c * kFixYOne);
            f.ok = ((inside >> gb) & 0xffu) == 0xffu && fabs(c) < 65536.0;
        }
    } else if (finish) {
        if (q < 6) m.inv[q] = inv;
        if (q == 0) {
            m.have_cur = 1;
            m.iZ = iZ;
            // the next solve's shift: its Z then starts in [1/4, 1/2) (see newton_round)
            const int ez = ((__double2hiint(Z) >> 20) & 0x7ff) - 1023;
            m.logz = fma((double)(ez + 2), 0x1.62e42fefa39efp-1, sh);
            m.state = kNewtonDone;
        }
    } else if (act && q == 0) {
        if (accept) {
            m.have_cur = 1;
            newton_fail(m);
        } else if (++m.halvings >= 40) {
            newton_fail(m);
        } else {
            m.t *= 0.5;
            for (int i = 0; i < 3; i++) m.trial[i] = fma(m.t, m.dir[i], m.lam[i]);
            newton_set_trial(m);
        }
        if (m.state == kNewtonEval) f.ok = fix_trial(C, f.vmax, m.trial, m.sh, f.v, f.cst) ? 1 : 0;
    }
    __syncwarp();
    return m.state == kNewtonEval;
}

// shared-memory rows of one warp: the support nodes' X and the weights of the last evaluation (FP64 bits)
struct FixSmem {
    i64 x0[kLmeRows], x1[kLmeRows], x2[kLmeRows];
    double w[kLmeRows];
};

// One evaluation in fixed point at the pending trial: weights into F.w, the sums into m.E. False if the
// weights leave the window (a weight of 1 or more, Z outside [2^-11, 1), A too large): the caller then
// evaluates in FP64. A function of the trial and the shift alone, so a restored state repeats it bit
// for bit. Warp-uniform.
template <bool LOLO>
__device__ __forceinline__ bool lme_eval_fix(const FixConst &C, FixSmem &F, int n, MpNewton &m, const MpFix &f,
                                             int lane, const u64 *T)
{
    FixSums s;
    fix_sums_zero(s);
    {
        const i64 c0 = f.xp[0] - f.v[0], c1 = f.xp[1] - f.v[1], c2 = f.xp[2] - f.v[2], cst = f.cst;
        const u64 bq = C.bq;
#pragma unroll 1
        for (int k = lane; k < n; k += kWarp)
            F.w[k] = fix_pair<LOLO>(F.x0[k], F.x1[k], F.x2[k], c0, c1, c2, cst, bq, T, s);
    }
    const uint32_t tr = fix_trace(s);
    if (__any_sync(0xffffffffu, s.top >= 0 || s.zc >= (1u << 26) || tr >= (1u << 30))) return false;
    const uint32_t zs = __reduce_add_sync(0xffffffffu, s.zc), ts = __reduce_add_sync(0xffffffffu, tr >> 5);
    if (zs < (1u << 15) || zs >= (1u << 26) - 1024u || ts >= (kFixTraceMax >> 5) - 64u) return false;
    i64 v[10];
    fix_combine(s, v);
    i64 t = warp_reduce_scatter10(v, lane);
    const i64 Z = __shfl_sync(0xffffffffu, t, 0);
    const i64 r0 = __shfl_sync(0xffffffffu, t, 2), r1 = __shfl_sync(0xffffffffu, t, 4), r2 = __shfl_sync(0xffffffffu, t, 8);
    // sums 1-3 are r, 4-9 A (00, 11, 22, 01, 12, 02): moved from the centre to the material point
    const int j = rs10_value(lane);
    const int a = j < 4 ? 0 : (j < 7 ? j - 4 : (j == 8 ? 1 : 0));
    const int b = j < 4 ? (j > 0 ? j - 1 : 0) : (j < 7 ? j - 4 : (j == 7 ? 1 : 2));
    const i64 ra = a == 0 ? r0 : (a == 1 ? r1 : r2), vb = f.v[b];
    const i64 rd = fix_r_about(Z, b == 0 ? r0 : (b == 1 ? r1 : r2), vb);
    if (j >= 4) t = fix_a_about(t, ra, rd, f.v[a], vb);
    else if (j >= 1) t = rd;
    const double d = (double)t * (j == 0 ? 0x1p-63 : (j < 4 ? C.r_unit : C.a_unit));
    if (rs10_writer(lane)) m.E[j] = d;
    if (lane == 0) m.E[10] = m.sh;
    return true;
}

// node positions as the step keeps them and as the stand-alone entry gets them
struct NodeX4 {
    const double4_32a *x;
    __device__ __forceinline__ void get(int id, double &a, double &b, double &c) const
    {
        const double4_32a v = x[id];
        a = v.x; b = v.y; c = v.z;
    }
};
struct NodeX3 {
    const double *x;
    __device__ __forceinline__ void get(int64_t id, double &a, double &b, double &c) const
    {
        a = x[3 * id]; b = x[3 * id + 1]; c = x[3 * id + 2];
    }
};

// the same evaluation in FP64, for trials outside the fixed-point range: coordinates from global memory, the
// weights to w (if given); shift handling as lme_eval_block
// exponent scale units of one pair's weight at lambda s / kExpScale with shift sh_s / kExpScale; d = x_p - x_a
template <typename X>
__device__ __forceinline__ double lme_weight64(X x, int id, double px, double py, double pz, double beta_s, double s0, double s1,
                                               double s2, double sh_s, double &dx, double &dy, double &dz)
{
    double ax, ay, az;
    x.get(id, ax, ay, az);
    dx = px - ax; dy = py - ay; dz = pz - az;
    const double q = fma(-beta_s, fma(dz, dz, fma(dy, dy, dx * dx)), -sh_s);
    return exp_scaled(fma(s2, dz, fma(s1, dy, fma(s0, dx, q))), g_exp2_table);
}

template <typename X>
__device__ __noinline__ void lme_eval64(X x, const int32_t *ids, double px, double py, double pz, double beta_s, double *w,
                                        int n, MpNewton &m, int lane)
{
    const double s0 = m.trial[0] * kExpScale, s1 = m.trial[1] * kExpScale, s2 = m.trial[2] * kExpScale;
    double sh = m.sh, v[10], t = 0.0;
    for (int pass = 0; pass < 2; pass++) {
        const double sh_s = sh * kExpScale;
#pragma unroll
        for (int i = 0; i < 10; i++) v[i] = 0.0;
        for (int k = lane; k < n; k += kWarp) {
            double dx, dy, dz;
            const double wk = lme_weight64(x, ids[k], px, py, pz, beta_s, s0, s1, s2, sh_s, dx, dy, dz);
            if (w) w[k] = wk;
            const double wx = wk * dx, wy = wk * dy, wz = wk * dz;
            v[0] += wk;
            v[1] += wx; v[2] += wy; v[3] += wz;
            v[4] = fma(wx, dx, v[4]); v[5] = fma(wy, dy, v[5]); v[6] = fma(wz, dz, v[6]);
            v[7] = fma(wx, dy, v[7]); v[8] = fma(wy, dz, v[8]); v[9] = fma(wx, dz, v[9]);
        }
        t = warp_reduce_scatter10(v, lane);
        const double Z = __shfl_sync(0xffffffffu, t, 0);
        if (pass == 1 || (Z > 1e-200 && Z < 1e200)) break;
        double mx = -INFINITY;   // over- or underflow: once more with the largest exponent as the shift
        for (int k = lane; k < n; k += kWarp) {
            double ax, ay, az;
            x.get(ids[k], ax, ay, az);
            const double dx = px - ax, dy = py - ay, dz = pz - az;
            mx = fmax(mx, fma(s2, dz, fma(s1, dy, s0 * dx)) - beta_s * fma(dz, dz, fma(dy, dy, dx * dx)));
        }
        sh = warp_max(mx) * (1.0 / kExpScale);
    }
    if (rs10_writer(lane)) m.E[rs10_value(lane)] = t;
    if (lane == 0) m.E[10] = sh;
}

// shared memory of one block: the exp table, the warps' rows (a compile-time stride, so that a slot's four
// words share one address register) and the solves' states
struct FixBlock {
    u64 table[kExpTable];
    FixSmem rows[kLmeWarps];
    MpNewton newton[kLmeWarps];
    MpFix fix[kLmeWarps];
};

template <bool MIXED, bool STAB>
__global__ void __launch_bounds__(kLmeWarps * kWarp, 4) k_lme_fix(const __grid_constant__ Dev D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * kLmeWarps + warp;
    const int rows = lme_rows(D.S), S = D.S;
    const FixConst &C = D.fix;
    FixBlock &B = *(FixBlock *)smem_raw;
    u64 *T = B.table;
    for (int j = threadIdx.x; j < kExpTable; j += kLmeWarps * kWarp) T[j] = g_exp2_mant[j];
    FixSmem &F = B.rows[warp];
    MpNewton &M = B.newton[warp];
    MpFix &X = B.fix[warp];
    bool active = (p < D.nm) && !has_error(D.err);
    if (active && (D.cnt[p] > rows || (D.lme_far && D.fstart[p].vmax < 0.0))) {   // solved by k_lme_wide
        if (lane == 0) D.lme_defer[atomicAdd(D.n_defer, 1)] = (int32_t)p;
        active = false;
    }
    const int64_t base = p * (int64_t)S;
    constexpr int G = 6;   // passes of dependent gathers in flight (4: 2.97 instead of 2.86 ms on 202,752 MPs)
    int cnt = 0;
    double shift0 = 0;
    if (active) {
        cnt = D.cnt[p];
        shift0 = D.logz[p];
        for (int k0 = lane; k0 < cnt; k0 += G * kWarp) {
            int id[G];
            longlong4_32a a[G];
#pragma unroll
            for (int j = 0; j < G; j++) id[j] = k0 + j * kWarp < cnt ? D.ids[base + k0 + j * kWarp] : -1;
#pragma unroll
            for (int j = 0; j < G; j++)
                if (id[j] >= 0) a[j] = D.xfix[id[j]];
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int k = k0 + j * kWarp;
                if (id[j] >= 0) { F.x0[k] = a[j].x; F.x1[k] = a[j].y; F.x2[k] = a[j].z; }
            }
        }
        if (lane < 12) {   // the start formed by k_lme_prep
            const i64 v = ((const i64 *)&D.fstart[p])[lane];
            if (lane < 3) M.trial[lane] = M.ws[lane] = fx_bits_d((u64)v);
            else ((i64 *)&X)[lane - 3] = v;
        }
        if (lane == 0) {
            M.t = 1.0;
            M.have_cur = M.iters = M.iters_total = M.halvings = M.retried = 0;
            M.shift0 = M.sh = shift0;
            M.state = cnt > 0 ? kNewtonEval : kNewtonFail;
        }
    } else if (lane == 0) {
        M.state = kNewtonIdle;
    }
    __syncthreads();
    for (;;) {
        if (M.state == kNewtonEval) {
            __syncwarp();
            if (!(X.ok && lme_eval_fix<!MIXED>(C, F, cnt, M, X, lane, T)))
                lme_eval64(NodeX4{D.x}, D.ids + base, D.xp[p].x, D.xp[p].y, D.xp[p].z, D.beta * kExpScale, F.w, cnt, M,
                           lane);
        }
        __syncthreads();
        const bool pending = warp == 0 && fix_round(B.newton, B.fix, C, D.tol_abs, D.max_newton, lane);
        if (!__syncthreads_or(pending)) break;
    }
    if (!active) return;
    if (!lme_finish(D, p, cnt, M, shift0, lane)) return;
    // the pairs' node-major positions hang on two dependent loads: gathered ahead of the output loop, G
    // passes in flight, into this warp's share of the exp table (every warp of the block is past its
    // last evaluation)
    int32_t *pos = (int32_t *)B.table + warp * (2 * kExpTable / kLmeWarps);
    for (int k0 = lane; k0 < cnt; k0 += G * kWarp) {
        int id[G], r[G];
#pragma unroll
        for (int j = 0; j < G; j++) {
            const int k = k0 + j * kWarp;
            id[j] = k < cnt ? D.ids[base + k] : 0;
            r[j] = k < cnt ? D.rank[base + k] : 0;
        }
#pragma unroll
        for (int j = 0; j < G; j++) r[j] += D.noff[id[j]];
#pragma unroll
        for (int j = 0; j < G; j++)
            if (k0 + j * kWarp < cnt) pos[k0 + j * kWarp] = r[j];
    }
    const double iZ = M.iZ, mp = D.mass[p];
    double Q[9];
    lme_force_matrix(D, p, M, lane, Q);
    const i64 xp0 = X.xp[0], xp1 = X.xp[1], xp2 = X.xp[2];
    const int fb = C.fb;
    // With the penalty term the FP64 pipe bounds the output loop: the products with Q then run in integers (1.89 ->
    // 1.76 ms on 78,624 stabilised MPs; without the term 2.87 -> 3.18 ms on 202,752). Q itself, for the
    // rare pair out of range, moves to shared memory (C is not needed any more).
    FixRows QR = {};
    if (STAB && !MIXED) {
        fix_rows(Q, fb, QR);
        __syncwarp();
        double q = 0.0;
#pragma unroll
        for (int i = 0; i < 9; i++) q = lane == i ? Q[i] : q;
        if (lane < 9) M.C[lane] = q;
        __syncwarp();
    }
    LmeStab<STAB && MIXED> st;
    st.load(D, p);
    StabFix sf;
    int id1 = 0;                       // the next pass's node
    if (STAB && !MIXED) {
        sf.load(D, p);
        if (lane < cnt) sf.a = D.x_prev[D.ids[base + lane]];
        if (lane + kWarp < cnt) id1 = D.ids[base + lane + kWarp];
    }
    // largest magnitudes of the stored mass / force terms by their high words (exponents at the end)
    unsigned hm = 0, hf = 0;
#pragma unroll 1
    for (int k = lane; k < cnt; k += kWarp) {
        const double N = F.w[k] * iZ;
        const i64 d0 = xp0 - F.x0[k], d1 = xp1 - F.x1[k], d2 = xp2 - F.x2[k];
        double sx = 0.0, sy = 0.0, sz = 0.0;
        if (STAB && MIXED) {
            const int id = D.ids[base + k];
            const double4_32a a = D.x[id], xp = D.xp[p];
            st.term(D, id, N, xp.x - a.x, xp.y - a.y, xp.z - a.z, sx, sy, sz);
        }
        double4_32a a1 = sf.a;
        if (STAB && !MIXED) {
            if (k + kWarp < cnt) a1 = D.x_prev[id1];
            if (k + 2 * kWarp < cnt) id1 = D.ids[base + k + 2 * kWarp];
        }
        if (MIXED) {
            // e = N d in FP32 (every consumer of the mixed path's rows rounds them to FP32),
            // stored widened exactly; N stays FP64
            const float fN = f32_round_bits(N);
            const float ex = fN * fix_to_float(d0, fb), ey = fN * fix_to_float(d1, fb), ez = fN * fix_to_float(d2, fb);
            D.shape[base + k] = make_double4_32a(N, df_widen(ex), df_widen(ey), df_widen(ez));
            const float c0 = (float)mp * fN;
            float c1 = fmaf((float)Q[2], ez, fmaf((float)Q[1], ey, (float)Q[0] * ex));
            float c2 = fmaf((float)Q[5], ez, fmaf((float)Q[4], ey, (float)Q[3] * ex));
            float c3 = fmaf((float)Q[8], ez, fmaf((float)Q[7], ey, (float)Q[6] * ex));
            if (STAB) {
                c1 += f32_round_bits(sx);
                c2 += f32_round_bits(sy);
                c3 += f32_round_bits(sz);
            }
            D.contrib32[pos[k]] = make_float4(c0, c1, c2, c3);
            hm = max(hm, __float_as_uint(c0) & 0x7fffffffu);
            hf = max(max(hf, __float_as_uint(c1) & 0x7fffffffu),
                     max(__float_as_uint(c2) & 0x7fffffffu, __float_as_uint(c3) & 0x7fffffffu));
        } else {
            double ex, ey, ez;
            fix_nd(N, d0, d1, d2, fb, C.r_unit, ex, ey, ez);
            D.shape[base + k] = make_double4_32a(N, ex, ey, ez);
            const double cm = mp * N;
            double fx, fy, fz;
            if (!(STAB && force_fix(QR, N, d0, d1, d2, fx, fy, fz))) {
                const double *q = STAB ? M.C : Q;
                fx = q[0] * ex + q[1] * ey + q[2] * ez;
                fy = q[3] * ex + q[4] * ey + q[5] * ez;
                fz = q[6] * ex + q[7] * ey + q[8] * ez;
            }
            if (STAB) {
                sf.add(N, ex, ey, ez, fx, fy, fz);
                sf.a = a1;
            }
            D.contrib64[pos[k]] = make_double4_32a(cm, fx, fy, fz);
            hm = max(hm, (unsigned)__double2hiint(cm) & 0x7fffffffu);
            hf = max(max(hf, (unsigned)__double2hiint(fx) & 0x7fffffffu),
                     max((unsigned)__double2hiint(fy) & 0x7fffffffu, (unsigned)__double2hiint(fz) & 0x7fffffffu));
        }
    }
    hm = __reduce_max_sync(0xffffffffu, hm);
    hf = __reduce_max_sync(0xffffffffu, hf);
    if (lane == 0) {
        // binary exponents; zero and subnormal terms count as -2000
        const int sft = MIXED ? 23 : 20, bias = MIXED ? 127 : 1023;
        atomicMax(&D.emax[0], (hm >> sft) ? (int)(hm >> sft) - bias : -2000);
        atomicMax(&D.emax[1], (hf >> sft) ? (int)(hf >> sft) - bias : -2000);
    }
}

// Before k_lme_fix: the nodes' fixed-point coordinates, the empty list of deferred MPs and, one thread
// per MP, the start of each solve (warm start, its centre and constant): about 30 FP64 instructions
// that would cost 16 cycles each in the MP's own warp and cost half a cycle a lane here.
__global__ void __launch_bounds__(256) k_lme_prep(const __grid_constant__ Dev D)
{
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    const FixConst &C = D.fix;
    if (t0 == 0) *D.n_defer = 0;
    for (int64_t i = t0; i < D.nn; i += nt) {
        const double4_32a a = D.x[i];
        longlong4_32a f;
        f.x = fix_from_double(a.x, C.fb);
        f.y = fix_from_double(a.y, C.fb);
        f.z = fix_from_double(a.z, C.fb);
        f.w = 0;
        D.xfix[i] = f;
    }
    for (int64_t p = t0; p < D.nm; p += nt) {
        // Eq. 14: the warm start is the previous step's lambda, or (within a step) the cubic through the
        // last four solutions, 4 l_n - 6 l_{n-1} + 4 l_{n-2} - l_{n-3}
        FixStart s;
        for (int i = 0; i < 3; i++) {
            double l = D.lam[3 * p + i];
            if (D.lme_mode == kLmeStep)
                l = fma(4.0, l + D.lam_prev2[3 * p + i], -fma(6.0, D.lam_prev[3 * p + i], D.lam_prev3[3 * p + i]));
            s.trial[i] = l;
        }
        const double4_32a x = D.xp[p];
        s.xp[0] = fix_from_double(x.x, C.fb);
        s.xp[1] = fix_from_double(x.y, C.fb);
        s.xp[2] = fix_from_double(x.z, C.fb);
        s.vmax = C.vmax;
        s.ok = fix_trial(C, s.vmax, s.trial, D.logz[p], s.v, s.cst) ? 1 : 0;
        D.fstart[p] = s;
    }
}

// Between k_lme_prep and k_lme_fix when the supports were not searched at the current positions (given or frozen
// supports, or positions set by the caller): separations may then exceed r_s by any factor, and k_lme_fix keeps
// coordinates modulo 2^64 (4.4 to 8.8 r_s). Warp per MP: the largest separation of any axis leaves the solve the
// rest of the range for its centre; from 2^62 units on (1.1 to 2.2 r_s, what the force products take) the MP is
// left to lme_block (k_lme_wide). Bound by the FP64 pipe (three subtractions a pair; the comparisons
// go by high words): 0.43 ms beside the solve's 2.48 on 202,752 MPs.
__global__ void __launch_bounds__(128) k_lme_far(const __grid_constant__ Dev D)
{
    const int lane = threadIdx.x & 31;
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= D.nm) return;
    const FixConst &C = D.fix;
    const int n = D.cnt[p];
    if (n > lme_rows(D.S)) return;   // goes to lme_block as it is
    const int64_t base = p * (int64_t)D.S;
    const double4_32a xp = D.xp[p];
    // magnitudes by their high words (non-finite ones are the largest)
    unsigned top = 0;
    for (int k = lane; k < n; k += kWarp) {
        const double4_32a a = D.x[D.ids[base + k]];
        const unsigned dx = (unsigned)__double2hiint(xp.x - a.x) & 0x7fffffffu, dy = (unsigned)__double2hiint(xp.y - a.y) & 0x7fffffffu,
                       dz = (unsigned)__double2hiint(xp.z - a.z) & 0x7fffffffu;
        top = max(max(top, dx), max(dy, dz));
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane != 0) return;
    FixStart &s = D.fstart[p];
    // within r_s (to 2^-20): as after a search, so that supports recorded from a run replay its solves bit for bit
    if (top <= C.near) return;
    const double far = __hiloint2double((int)(min(top, 0x7fefffffu) + 1u), 0) / C.r_unit;   // rounded up, in LSB
    s.vmax = far <= 0x1p62 ? fmin(C.vmax, kFixT - far) : -1.0;
    s.ok = fix_trial(C, s.vmax, s.trial, D.logz[p], s.v, s.cst) ? 1 : 0;
}

// The fixed-point evaluation's constants: fb so that the support radius lies between 2^63/4.4 and
// 2^63/2.2 LSB (a trial's centre may then move by 0.45 support radii or more per axis before it leaves
// the range). Off where the exponent scale does not fit 64 bits (support tolerances below about
// 2e-10) or for length scales outside the exponent arithmetic's range.
FixConst make_fix_const(double beta, double rs2)
{
    FixConst c = {};
    const double rs = std::sqrt(rs2);
    int ex = 0;
    std::frexp(2.2 * rs, &ex);                      // 2^63 LSB = 2^ex >= 2.2 rs
    c.fb = 63 - ex;
    const double a = std::ldexp(1.0, 32 - c.fb);
    const long double bq = std::ldexp((long double)beta * 256.0L / std::log(2.0L) * a * a, 46 + 63);
    c.on = std::isfinite((double)bq) && bq < 0x1p64L && bq >= 0x1p32L && c.fb > -60 && c.fb < 120;
    if (!c.on) return c;
    c.bq = (u64)bq;
    c.i2b = std::ldexp(1.0, c.fb) / (2.0 * beta);
    c.cy = 64.0 / (beta * std::log(2.0));
    c.vmax = kFixT - std::ldexp(rs, c.fb) * (1.0 + 1e-9);
    c.near = (uint32_t)(fx_d_bits(rs * (1.0 + 1e-9)) >> 32);
    c.r_unit = std::ldexp(1.0, -c.fb);
    c.a_unit = a * a / 16.0;
    return c;
}

static size_t lme_block_smem(int rows)
{
    return (size_t)kLmeWarps * 4 * (size_t)rows * sizeof(double) + (size_t)kLmeWarps * sizeof(MpNewton);
}

// Which kernel (D.lme_fix, set by the host step): the fixed-point one for the FP64 path's solves where
// its exponent range covers the problem (fix.on), and for regenerating the shape functions of a state
// that such a solve left, in either path. The mixed path's own solves keep k_lme: its FP32 increments
// turn a last-bit change of N into an FP32 ulp of a node's increment (1e-7 of the stress it leads to),
// so that recorded mixed runs would not be reproduced.
template <bool MIXED, bool STAB>
static cudaError_t launch_lme_t(const Dev &D, cudaStream_t s, unsigned blocks, long long *launches)
{
    cudaError_t e;
    if (D.lme_fix) {
        const size_t smem = sizeof(FixBlock);
        e = cudaFuncSetAttribute(k_lme_fix<MIXED, STAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int64_t pb = ((D.nn > D.nm ? D.nn : D.nm) + 255) / 256;
        if (pb > 152 * 8) pb = 152 * 8;
        k_lme_prep<<<(unsigned)pb, 256, 0, s>>>(D);
        if (D.lme_far) {
            k_lme_far<<<(unsigned)((D.nm * kWarp + 127) / 128), 128, 0, s>>>(D);
            if (launches) *launches += 1;
        }
        k_lme_fix<MIXED, STAB><<<blocks, kLmeWarps * kWarp, smem, s>>>(D);
        if (launches) *launches += 2;
    } else {
        const size_t smem = lme_block_smem(lme_rows(D.S));
        e = cudaFuncSetAttribute(k_lme<MIXED, STAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaMemsetAsync(D.n_defer, 0, sizeof(int32_t), s);
        if (e != cudaSuccess) return e;
        k_lme<MIXED, STAB><<<blocks, kLmeWarps * kWarp, smem, s>>>(D);
        if (launches) *launches += 1;
    }
    if (D.S > kLmeRows || (D.lme_fix && D.lme_far)) {
        // one persistent round of blocks over the deferred MPs (none on most steps: the launch then
        // returns at once)
        const size_t smem = lme_block_smem(D.S);
        e = cudaFuncSetAttribute(k_lme_wide<MIXED, STAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_lme_wide<MIXED, STAB><<<152 * 3, kLmeWarps * kWarp, smem, s>>>(D);
        if (launches) *launches += 1;
    }
    return cudaGetLastError();
}

cudaError_t launch_lme(const Dev &D, cudaStream_t s, long long *launches)
{
    const unsigned blocks = (unsigned)((D.nm + kLmeWarps - 1) / kLmeWarps);
    if (blocks == 0) return cudaSuccess;
    const bool mixed = D.precision == OTM_PRECISION_MIXED, stab = D.eps_stab > 0.0;
    return mixed ? (stab ? launch_lme_t<true, true>(D, s, blocks, launches) : launch_lme_t<true, false>(D, s, blocks, launches))
                 : (stab ? launch_lme_t<false, true>(D, s, blocks, launches)
                         : launch_lme_t<false, false>(D, s, blocks, launches));
}

// (N, grad N) of every slot of a padded row set, for state export: already stored in shape[]
// ======================================================================== k_kinematics
// warp per MP: the 12 sums x_p,i = sum N x_a,i and G_ij = sum du_a,i e_a,j (e_a = N_a d_a, the
// stored pair row) over the old support; lanes 2j write sum j. Eq. 11 is then
// dF = 1 + sum du_a (x) grad N_a = 1 - G K with K = J^-1 of the old support's LME solve, formed
// once per MP in the thread-per-MP return-map kernel with the products with F, det(dF) and the
// volume update.
template <bool MIXED>
__global__ void __launch_bounds__(128) k_kinematics(const __grid_constant__ Dev D)
{
    const int lane = threadIdx.x & 31;
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= D.nm) return;
    if (has_error(D.err)) return;
    const int n = D.cnt[p];
    const int64_t base = p * (int64_t)D.S;
    KinSum<MIXED> ks;
    ks.gather(D, base, n, lane);
    const int j = rs12_value(lane);
    if (rs12_writer(lane)) {
        if (j < 3) {
            const double old = ((const double *)&D.xp[p])[j];
            const double x = ks.xp(old, j);
            ((double *)&D.xp_prev[p])[j] = old;
            ((double *)&D.xp[p])[j] = x;
            if (!isfinite(x)) raise_error(D.err, OTM_ERR_NONFINITE, D.mgid[p]);
        } else {
            D.dF[9 * p + (j - 3)] = ks.g();   // row-major G = sum du (x) e; k_return_map forms dF
        }
    }
}

cudaError_t launch_kinematics(const Dev &D, cudaStream_t s, long long *launches)
{
    const unsigned blocks = (unsigned)((D.nm * 32 + 127) / 128);
    if (blocks == 0) return cudaSuccess;
    if (D.precision == OTM_PRECISION_MIXED)
        k_kinematics<true><<<blocks, 128, 0, s>>>(D);
    else
        k_kinematics<false><<<blocks, 128, 0, s>>>(D);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

// ======================================================================== return map without eigenvectors
// Logarithm after P. T. P. Tang ("Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16(4), 1990), for positive normal arguments: x = 2^e m with m in
// [0.7, 1.4), r ~ 1/m from a 1024-entry table, t = m r - 1 (one rounding, |t| < 2^-9.9), and log x = e ln 2 -
// log r + (t - t^2/2 + t^3/3 - t^4/4 + t^5/5). The table holds (r, -log r); absolute error below
// 1e-16 max(1, |log x|). About 11 FP64 instructions; the library's log takes the pipe time of 33.

__device__ __forceinline__ double log_pos(double x)
{
    const int hi = __double2hiint(x);
    int e = (hi >> 20) - 1023;
    const int j = (hi >> 10) & 1023;
    const bool up = j >= 424;          // m >= 1.414: m / 2 and e + 1, so that arguments about 1 have e = 0
    e += up;
    const double m = __hiloint2double((hi & 0xfffff) | (up ? 0x3fe00000 : 0x3ff00000), __double2loint(x));
    const double2 c = g_log_table[j];
    const double t = fma(m, c.x, -1.0);
    const double t2 = t * t;
    const double q = fma(t, fma(t, fma(t, 0.2, -0.25), 0x1.5555555555555p-2), -0.5);
    // the integer e as a double by its bits (a conversion costs an FP64 instruction as well; this one
    // is a subtraction of two exactly known values)
    const double ed = __hiloint2double(0x43300000, 0x40000000 + e) - 0x1.0000040000000p52;
    return fma(ed, 0x1.62e42fefa39efp-1, fma(ed, 0x1.abc9e3b39803fp-56, c.y + fma(t2, q, t)));
}

__device__ __forceinline__ double exp_of(double v) { return exp_scaled(v * kExpScale, g_exp2_table); }

// x^n for x > 0 by exp(n log x): relative error about (1 + |n log x|) 2e-16
__device__ __forceinline__ double pow_pos(double x, double n) { return exp_of(n * log_pos(x)); }

// Johnson-Cook flow stress at E = ebar_n + x (x > 0) and its derivative in x, as jc_sigma_y
__device__ __forceinline__ void jc_flow(const otm_material &M, double E, double x, double inv_dte, double therm, double &sy,
                                        double &dsy)
{
    const double ixE = recip<2>(x * E), ix = E * ixE, iE = x * ixE;
    const double rstar = x * inv_dte;
    double rate = 1.0, drate = 0.0;
    if (rstar > 1.0) {
        rate = fma(M.C, log_pos(rstar), 1.0);
        drate = M.C * ix;
    }
    const double bp = M.B * pow_pos(E, M.n), hard = M.A + bp;
    sy = hard * rate * therm;
    dsy = fma(M.n * bp * iE, rate, hard * drate) * therm;
}

// The consistency condition's root in FP32 (Newton inside the bracket [0, hi]): within about 1e-5 of
// the FP64 root, where two FP64 evaluations finish. All stresses divided by 3 mu.
__device__ __forceinline__ float jc_root32(const otm_material &M, float s3, float ebar, float inv_dte, float therm, float hi,
                                           float x)
{
    const float A = (float)M.A * s3 * therm, B = (float)M.B * s3 * therm, n = (float)M.n, C = (float)M.C;
    float lo = 0.f, up = hi;
    for (int it = 0; it < 6; it++) {
        const float E = ebar + x, p = B * exp2f(n * __log2f(E)), hard = A + p, rs = x * inv_dte;
        const bool on = rs > 1.f;
        const float rate = on ? fmaf(C, __logf(rs), 1.f) : 1.f;
        const float g = hi - x - hard * rate;
        const float d = 1.f + __fdividef(n * p, E) * rate + (on ? __fdividef(hard * C, x) : 0.f);
        if (g > 0.f) lo = x; else up = x;
        const float xn = x + __fdividef(g, d);
        const float y = (xn > lo && xn < up) ? xn : 0.5f * (lo + up);
        if (fabsf(y - x) <= 1e-6f * y) { x = y; break; }
        x = y;
    }
    return x;
}

// The constitutive update (return_map_point) for points whose deviatoric elastic strain is small,
// without the eigen decomposition: with b_tr = (1 + p)(I + Y), Y traceless and |Y| <= 1/32,
//   log b_tr = log(1 + p) I + log(I + Y),   b^e = (1 + p) exp(w) exp(2 rho dev e)
// by their power series reduced with Cayley-Hamilton (Y^3 = -I2 Y + I3 I: two FMAs a term); the radial
// return scales the deviator by rho, so neither needs principal axes. b_tr - I is formed from dF - I
// and b^e - I, free of the rounding about 1. Metals stay below the bound: it is a shear strain of
// about 1 %, ten times a copper's yield strain; anything else (and non-finite input) returns false
// and takes return_map_point.
//
// FP64 pipe bound. Measured (two thirds of the points plastic, Johnson-Cook): 1,000,003 stand-alone points
// 3.02 -> 0.78 ms a call; k_return_map on the 202,752-MP rod 1.40 -> 0.45 ms.
__device__ __forceinline__ bool return_map_small(const otm_material &M, const RmConst &R, const RmIn &in, RmOut &out, int &status)
{
    double y[6], H[9];   // b_tr - I as (xx, yy, zz, xy, yz, xz)
    {
        const double g[9] = {in.dF[0] - 1.0, in.dF[1], in.dF[2], in.dF[3], in.dF[4] - 1.0, in.dF[5],
                             in.dF[6], in.dF[7], in.dF[8] - 1.0};
        const double b[6] = {in.be[0] - 1.0, in.be[1] - 1.0, in.be[2] - 1.0, in.be[3], in.be[4], in.be[5]};
        // H = g (I + b), y = b + H + H^T + H g^T
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const double gx = g[3 * i], gy = g[3 * i + 1], gz = g[3 * i + 2];
            H[3 * i] = gx + fma(gx, b[0], fma(gy, b[3], gz * b[5]));
            H[3 * i + 1] = gy + fma(gx, b[3], fma(gy, b[1], gz * b[4]));
            H[3 * i + 2] = gz + fma(gx, b[5], fma(gy, b[4], gz * b[2]));
        }
        const int I[6] = {0, 1, 2, 0, 1, 0}, J[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const int i = I[c], j = J[c];
            y[c] = b[c] + (H[3 * i + j] + H[3 * j + i]) +
                   fma(H[3 * i], g[3 * j], fma(H[3 * i + 1], g[3 * j + 1], H[3 * i + 2] * g[3 * j + 2]));
        }
    }
    const double p = (y[0] + y[1] + y[2]) * (1.0 / 3.0);
    if (!(fabs(p) < 0.5)) return false;
    const double ip = recip<2>(1.0 + p);
    double Y[6];
#pragma unroll
    for (int c = 0; c < 6; c++) Y[c] = (c < 3 ? y[c] - p : y[c]) * ip;
    // Y^2, I2 = -tr(Y^2)/2, I3 = det Y
    double Y2[6];
    Y2[0] = fma(Y[0], Y[0], fma(Y[3], Y[3], Y[5] * Y[5]));
    Y2[1] = fma(Y[1], Y[1], fma(Y[3], Y[3], Y[4] * Y[4]));
    Y2[2] = fma(Y[2], Y[2], fma(Y[4], Y[4], Y[5] * Y[5]));
    Y2[3] = fma(Y[0], Y[3], fma(Y[3], Y[1], Y[5] * Y[4]));
    Y2[4] = fma(Y[3], Y[5], fma(Y[1], Y[4], Y[4] * Y[2]));
    Y2[5] = fma(Y[0], Y[5], fma(Y[3], Y[4], Y[5] * Y[2]));
    const double t2 = Y2[0] + Y2[1] + Y2[2];
    if (!(t2 <= 1.0 / 1024.0)) return false;
    const double h2 = 0.5 * t2;    // -I2
    const double I3 = fma(Y[0], fma(Y[1], Y[2], -Y[4] * Y[4]), fma(Y[3], fma(Y[4], Y[5], -Y[3] * Y[2]),
                                                                   Y[5] * fma(Y[3], Y[4], -Y[1] * Y[5])));
    // log(I + Y) = c0 I + c1 Y + c2 Y^2, Horner from the 11th term (|eigenvalue| < 0.0256: rest below 1e-20)
    double c0 = 1.0 / 11.0, c1 = 0.0, c2 = 0.0;
#pragma unroll
    for (int k = 10; k >= 0; k--) {   // (c0 + c1 Y + c2 Y^2) Y + a_k, a_k = -(-1)^k / k, a_0 = 0
        const double a = k == 0 ? 0.0 : ((k & 1) ? 1.0 : -1.0) / (k == 0 ? 1 : k);
        const double n0 = fma(c2, I3, a), n1 = fma(c2, h2, c0);
        c2 = c1;
        c1 = n1;
        c0 = n0;
    }
    const double w = fma(c2, t2, 3.0 * c0) * (1.0 / 3.0);   // tr log(I + Y) / 3
    const double q1 = 1.0 + p;
    const double tr = 1.5 * (log_pos(q1) + (p - (q1 - 1.0)) * ip + w);    // tr e
    double e[6];   // dev e
#pragma unroll
    for (int c = 0; c < 6; c++) e[c] = 0.5 * fma(c2, c < 3 ? Y2[c] - t2 * (1.0 / 3.0) : Y2[c], c1 * Y[c]);
    const double mu = R.mu;
    const double en2 = fma(2.0, fma(e[3], e[3], fma(e[4], e[4], e[5] * e[5])), fma(e[0], e[0], fma(e[1], e[1], e[2] * e[2])));
    const double sn = 2.0 * mu * sqrt(en2);
    const double q_tr = 1.2247448713915890491 * sn;   // sqrt(3/2) |s|
    double dep = 0.0;
    if (M.model == 0) {
        const double f_tr = sn - 0.81649658092772603273 * (M.sigma_y0 + M.H * in.ebar);
        if (f_tr > 0.0) dep = 0.81649658092772603273 * f_tr * R.ih;
    } else {
        const double tstar = fmin(fmax((in.T - M.T_room) * R.ispan, 0.0), 1.0);
        const double therm = tstar > 1e-300 ? 1.0 - pow_pos(tstar, M.m) : 1.0 - pow(tstar, M.m);
        const double pe = in.ebar > 1e-300 ? pow_pos(in.ebar, M.n) : pow(in.ebar, M.n);
        if (q_tr - (M.A + M.B * pe) * therm > 0.0) {
            // g(x) = q_tr - 3 mu x - sigma_y(x) on [0, q_tr / (3 mu)]: Newton safeguarded by bisection from the
            // FP32 root
            double lo = 0.0, hi = q_tr * R.i3mu;
            double x = (in.guess > 0.0 && in.guess < hi) ? in.guess : 0.5 * hi;
            const float x32 = jc_root32(M, (float)R.i3mu, (float)in.ebar, (float)R.idte, (float)therm, (float)hi, (float)x);
            if (x32 > 0.f && (double)x32 < hi) x = (double)x32;
            const double tol = 1e-12 * q_tr;
            bool ok = false;
            for (int it = 0; it < 300; it++) {
                double sy, dsy;
                jc_flow(M, in.ebar + x, x, R.idte, therm, sy, dsy);
                const double g = q_tr - 3.0 * mu * x - sy;
                const double xn = fma(g, recip<2>(fma(3.0, mu, dsy)), x);
                if (fabs(g) <= tol) {   // one more Newton step fixes the accepted iterate to rounding
                    if (xn > lo && xn < hi) x = xn;
                    ok = true;
                    break;
                }
                if (g > 0.0) lo = x; else hi = x;
                if (hi - lo <= 4e-16 * hi) { ok = true; break; }
                x = (xn > lo && xn < hi) ? xn : 0.5 * (lo + hi);
            }
            if (!ok) {
                status = OTM_ERR_RETURNMAP_NOCONV;
                return true;
            }
            dep = x;
        }
    }
    const double qn = q_tr - 3.0 * mu * dep;
    const double rho = dep > 0.0 ? 1.0 - 2.0 * mu * (1.2247448713915890491 * dep) / sn : 1.0;
    const double iJ = 1.0 / in.J, kt = R.K * tr, m2 = 2.0 * mu * rho;
#pragma unroll
    for (int c = 0; c < 6; c++) out.sig[c] = (c < 3 ? fma(m2, e[c], kt) : m2 * e[c]) * iJ;
    if (dep > 0.0) {
        // b^e = (1 + p) exp(w) exp(D), D = 2 rho dev e traceless: both by their Taylor series (D to the 9th
        // term, below 1e-19)
        double D[6], D2[6];
#pragma unroll
        for (int c = 0; c < 6; c++) D[c] = 2.0 * rho * e[c];
        D2[0] = fma(D[0], D[0], fma(D[3], D[3], D[5] * D[5]));
        D2[1] = fma(D[1], D[1], fma(D[3], D[3], D[4] * D[4]));
        D2[2] = fma(D[2], D[2], fma(D[4], D[4], D[5] * D[5]));
        D2[3] = fma(D[0], D[3], fma(D[3], D[1], D[5] * D[4]));
        D2[4] = fma(D[3], D[5], fma(D[1], D[4], D[4] * D[2]));
        D2[5] = fma(D[0], D[5], fma(D[3], D[4], D[5] * D[2]));
        const double d2 = 0.5 * (D2[0] + D2[1] + D2[2]);
        const double d3 = fma(D[0], fma(D[1], D[2], -D[4] * D[4]), fma(D[3], fma(D[4], D[5], -D[3] * D[2]),
                                                                       D[5] * fma(D[3], D[4], -D[1] * D[5])));
        constexpr double kInvFact[10] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040,
                                         1.0 / 40320, 1.0 / 362880};
        double a0 = kInvFact[9], a1 = 0.0, a2 = 0.0;
#pragma unroll
        for (int k = 8; k >= 0; k--) {
            const double n0 = fma(a2, d3, k == 0 ? 0.0 : kInvFact[k]), n1 = fma(a2, d2, a0);
            a2 = a1;
            a1 = n1;
            a0 = n0;
        }
        // exp(D) - I = a0 I + a1 D + a2 D^2; (1 + p) exp(w) - 1 = p + (1 + p)(exp(w) - 1), |w| < 5e-4
        const double ew = w * fma(w, fma(w, fma(w, fma(w, 1.0 / 120, 1.0 / 24), 1.0 / 6), 0.5), 1.0);
        const double v = fma(q1, ew, p), sc = 1.0 + v;
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const double x = fma(a2, D2[c], a1 * D[c]);
            out.be[c] = c < 3 ? 1.0 + (v + sc * (x + a0)) : sc * x;
        }
    } else {
#pragma unroll
        for (int c = 0; c < 6; c++) out.be[c] = c < 3 ? 1.0 + y[c] : y[c];
    }
    out.ebar = in.ebar + dep;
    out.rate = dep * R.idt;
    out.T = in.T;
    if (M.model == 1 && M.chi > 0.0 && dep > 0.0) out.T = fma(R.heat * qn, dep, in.T);
    out.failed = jc_fractured(M, kt * iJ, qn, iJ, out);
    status = OTM_OK;
    for (int c = 0; c < 6; c++)
        if (!isfinite(out.sig[c])) status = OTM_ERR_NONFINITE;
    return true;
}

RmConst make_rm_const(const otm_material &M, double dt)
{
    RmConst r;
    r.K = M.E / (3.0 * (1.0 - 2.0 * M.nu));
    r.mu = M.E / (2.0 * (1.0 + M.nu));
    r.i3mu = 1.0 / (3.0 * r.mu);
    r.ih = 1.0 / (2.0 * r.mu + 2.0 * M.H / 3.0);
    r.idt = 1.0 / dt;
    r.idte = 1.0 / (dt * M.eps_dot0);
    r.ispan = 1.0 / (M.T_melt - M.T_room);
    r.heat = M.chi / (M.rho0 * M.cp);
    return r;
}

// SMALL: the FP64 path; the mixed path keeps return_map_point (see launch_lme_t on its FP32 increments)
template <bool SMALL>
__global__ void __launch_bounds__(128) k_return_map(const __grid_constant__ Dev D)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= D.nm) return;
    if (has_error(D.err)) return;
    RmIn in;
    {   // Eq. 11: dF = 1 + sum du_a (x) grad N_a = 1 - G K (G from the kinematics gather, K = J^-1
        // of the LME solve the gather's shape functions came from)
        double G[9];
        for (int i = 0; i < 9; i++) G[i] = D.dF[9 * p + i];
        const double *k = D.Kinv + 6 * p;
        const double K[9] = {k[0], k[3], k[5], k[3], k[1], k[4], k[5], k[4], k[2]};
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                const double gk = G[3 * i] * K[j] + G[3 * i + 1] * K[3 + j] + G[3 * i + 2] * K[6 + j];
                in.dF[3 * i + j] = (i == j ? 1.0 : 0.0) - gk;
            }
        for (int i = 0; i < 9; i++) D.dF[9 * p + i] = in.dF[i];
    }
    const double *d = in.dF;
    // Eq. 10-12: F_{n+1} = dF F_n, v_{n+1} = det(dF) v_n
    const double det = d[0] * (d[4] * d[8] - d[5] * d[7]) - d[1] * (d[3] * d[8] - d[5] * d[6]) +
                       d[2] * (d[3] * d[7] - d[4] * d[6]);
    if (!(det > 0.0)) {
        raise_error(D.err, OTM_ERR_JACOBIAN, D.mgid[p]);
        return;
    }
    double *F = D.F + 9 * p;
    double Fo[9], Fn[9];
    for (int i = 0; i < 9; i++) Fo[i] = F[i];
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++)
            Fn[3 * i + j] = d[3 * i] * Fo[j] + d[3 * i + 1] * Fo[3 + j] + d[3 * i + 2] * Fo[6 + j];
    for (int i = 0; i < 9; i++) F[i] = Fn[i];
    D.vol[p] *= det;
    in.J = Fn[0] * (Fn[4] * Fn[8] - Fn[5] * Fn[7]) - Fn[1] * (Fn[3] * Fn[8] - Fn[5] * Fn[6]) +
           Fn[2] * (Fn[3] * Fn[7] - Fn[4] * Fn[6]);
    for (int i = 0; i < 6; i++) in.be[i] = D.be[6 * p + i];
    in.ebar = D.ebar[p];
    in.T = D.T[p];
    in.guess = D.rate[p] * D.dt;   // the previous step's plastic increment
    RmOut o;
    int st = OTM_OK;
    if (!SMALL || !return_map_small(D.mat[D.mat_id[p]], D.rmc[D.mat_id[p]], in, o, st)) {
        double Q0[9];
        for (int i = 0; i < 9; i++) Q0[i] = D.Qe[9 * p + i];
        in.Q0 = Q0;
        st = return_map_point(D.mat[D.mat_id[p]], D.dt, in, o);
        if (st == OTM_OK)
            for (int i = 0; i < 9; i++) D.Qe[9 * p + i] = o.Q[i];
    }
    if (st != OTM_OK) {
        raise_error(D.err, st, D.mgid[p]);
        return;
    }
    for (int i = 0; i < 6; i++) {
        D.be[6 * p + i] = o.be[i];
        D.sig[6 * p + i] = o.sig[i];
    }
    D.ebar[p] = o.ebar;
    D.T[p] = o.T;
    D.rate[p] = o.rate;
    D.failed[p] = (uint8_t)(o.failed && D.allow_erode);
}

cudaError_t launch_return_map(const Dev &D, cudaStream_t s, long long *launches)
{
    const unsigned blocks = (unsigned)((D.nm + 127) / 128);
    if (blocks == 0) return cudaSuccess;
    if (D.precision == OTM_PRECISION_MIXED)
        k_return_map<false><<<blocks, 128, 0, s>>>(D);
    else
        k_return_map<true><<<blocks, 128, 0, s>>>(D);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

// ======================================================================== stand-alone kernels
// Ascending bitonic sort of 32 R integers by one warp in registers (in shared memory it took 7,200 of a
// point's 9,200 instructions at 250 nodes a support; 600,007 points: 5.80 -> 2.19 ms), lane l holding the sorted elements
// [l R, (l + 1) R) afterwards (in any order before). Steps over fewer than R elements stay in the lane as plain
// minima and maxima, the others exchange with a lane of the same direction; lanes of a descending
// subsequence hold the complements instead.
template <int R>
__device__ __forceinline__ void warp_sort(int (&v)[R], int lane)
{
    int dir = 0;   // -1: complements
#pragma unroll
    for (int k = 2; k <= kWarp * R; k *= 2) {
        if (k >= R) {
            const int d = (lane * R & k) ? -1 : 0, f = d ^ dir;
#pragma unroll
            for (int r = 0; r < R; r++) v[r] ^= f;
            dir = d;
        }
#pragma unroll
        for (int j = k / 2; j > 0; j /= 2) {
            if (j >= R) {
                const bool lower = !(lane & (j / R));
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const int o = __shfl_xor_sync(0xffffffffu, v[r], j / R);
                    v[r] = lower ? min(v[r], o) : max(v[r], o);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r++)
                    if (!(r & j)) {
                        const int a = v[r], b = v[r + j];
                        const bool up = k >= R || !(r & k);
                        v[r] = up ? min(a, b) : max(a, b);
                        v[r + j] = up ? max(a, b) : min(a, b);
                    }
            }
        }
    }
}

// list[0..n) (n <= 32 R, room for 33 R) in ascending order
template <int R>
__device__ void warp_sort_list(int32_t *list, int n, int lane)
{
    int v[R];
#pragma unroll
    for (int r = 0; r < R; r++) v[r] = lane + kWarp * r < n ? list[lane + kWarp * r] : 0x7fffffff;
    __syncwarp();
    warp_sort<R>(v, lane);
#pragma unroll
    for (int r = 0; r < R; r++) {   // through a row of 33 words a warp's worth: no bank conflicts
        const int k = lane * R + r;
        list[k + k / kWarp] = v[r];
    }
    __syncwarp();
}

// shared-memory words of a warp's list of up to S IDs
__host__ __device__ __forceinline__ int search_list_words(int S)
{
    const int P2 = next_pow2(S < kWarp ? kWarp : S);
    return P2 + P2 / kWarp;
}

__global__ void __launch_bounds__(kSearchWarps * kWarp, 8)   // 64 registers; 48 the same, 40 (spills) 19 % slower
    k_search_only(const GridDev *g, const int32_t *cell_start, const float4 *spos32, const double4_32a *spos,
                  const SearchConst C, const double *mp_x, int64_t nm, int S, int32_t *ids, int32_t *counts,
                  int32_t *status, const unsigned long long *grid_err)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * kSearchWarps + warp;
    if (p >= nm) return;
    int32_t *list = (int32_t *)smem_raw + (size_t)warp * search_list_words(S);
    if (*grid_err != ~0ULL) {
        if (lane == 0) {
            atomicCAS(status, 0, (int)(-(int)(*grid_err & 0xff)));
            counts[p] = 0;
        }
        return;
    }
    const double px = mp_x[3 * p], py = mp_x[3 * p + 1], pz = mp_x[3 * p + 2];
    SearchGrid G{g, cell_start, spos32, spos};
    const int cnt = warp_support_search(G, C, px, py, pz, list, S, lane);
    const int n = min(cnt, S);
    __syncwarp();
    if (n <= kWarp) warp_sort_list<1>(list, n, lane);
    else if (n <= 2 * kWarp) warp_sort_list<2>(list, n, lane);
    else if (n <= 4 * kWarp) warp_sort_list<4>(list, n, lane);
    else if (n <= 8 * kWarp) warp_sort_list<8>(list, n, lane);
    else if (n <= 16 * kWarp) warp_sort_list<16>(list, n, lane);
    else warp_sort_list<kMaxS / kWarp>(list, n, lane);
    for (int k = lane; k < n; k += kWarp) ids[p * (int64_t)S + k] = list[k + k / kWarp];
    if (lane == 0) {
        counts[p] = cnt;
        if (cnt > S) atomicCAS(status, 0, OTM_ERR_CAPACITY);
    }
}

cudaError_t launch_search_only(const double *node_x, int64_t nn, const double *mp_x, int64_t nm, double rs2,
                               double cell, int S, int32_t *ids, int32_t *counts, void *scratch,
                               size_t scratch_bytes, double *grid_out, int32_t *status, cudaStream_t s)
{
    SearchScratch V;
    if (!carve_search_scratch(scratch, scratch_bytes, nn, &V)) return cudaErrorInvalidValue;
    cudaError_t e = build_search_grid(node_x, nn, cell, &V, grid_out, s);
    if (e != cudaSuccess) return e;
    const size_t smem = (size_t)kSearchWarps * search_list_words(S) * sizeof(int32_t);
    const unsigned blocks = (unsigned)((nm + kSearchWarps - 1) / kSearchWarps);
    if (blocks == 0) return cudaSuccess;
    k_search_only<<<blocks, kSearchWarps * kWarp, smem, s>>>(V.g, V.cell_start, V.spos32, V.spos,
                                                             make_search_const(cell, rs2), mp_x, nm, S, ids, counts,
                                                             status, V.err);
    return cudaGetLastError();
}

// Stand-alone LME with fixed-point evaluations: the block solve of k_lme_fix over caller arrays. The support
// radius is not an argument here, so the units are those of the default support tolerance (1e-6), every
// separation is checked against the range, and points outside it, or with more than kLmeRows nodes, or
// all of them where the length scale is outside the exponent arithmetic's (C.on = 0), are evaluated in FP64. The
// weights of more than kLmeRows nodes have no place in shared memory and are formed again for the output. The
// exponent shift is estimated in FP32 from the start. Measured (151,392 points of a rod, five evaluations
// each): 9.7 ms with all in FP64, 3.3 ms so.
__global__ void __launch_bounds__(kLmeWarps * kWarp, 4)
    k_lme_only_fix(const double *node_x, const double *mp_x, int64_t nm, const int32_t *ids, const int32_t *counts, int S,
                   double beta, const __grid_constant__ FixConst C, double tol, int max_newton, double *lam, double *shape,
                   int32_t *iters_out, int32_t *status)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * kLmeWarps + warp;
    FixBlock &B = *(FixBlock *)smem_raw;
    for (int j = threadIdx.x; j < kExpTable; j += kLmeWarps * kWarp) B.table[j] = g_exp2_mant[j];
    FixSmem &F = B.rows[warp];
    MpNewton &M = B.newton[warp];
    MpFix &X = B.fix[warp];
    bool active = p < nm;
    const int n = active ? counts[p] : 0;
    if (active && (n > S || n <= 0)) {
        if (lane == 0) atomicCAS(status, 0, n > S ? OTM_ERR_CAPACITY : OTM_ERR_LME_NOCONV);
        active = false;
    }
    const int64_t base = p * (int64_t)S;
    const NodeX3 nx{node_x};
    double px = 0, py = 0, pz = 0;
    bool fixed = false;             // every separation is inside the fixed-point range
    if (active) {
        px = mp_x[3 * p]; py = mp_x[3 * p + 1]; pz = mp_x[3 * p + 2];
        i64 P[3], Ph[3];
        bool ok = C.on && n <= kLmeRows;
        ok = fix_from_double_wide(px, C.fb, P[0], Ph[0]) && ok;
        ok = fix_from_double_wide(py, C.fb, P[1], Ph[1]) && ok;
        ok = fix_from_double_wide(pz, C.fb, P[2], Ph[2]) && ok;
        const double l0 = lam[3 * p], l1 = lam[3 * p + 1], l2 = lam[3 * p + 2];
        const float bf = (float)beta, lf0 = (float)l0, lf1 = (float)l1, lf2 = (float)l2, u32 = (float)(C.r_unit * 0x1p32);
        i64 far = 0;                // largest |D| of any component (less one unit for negative ones)
        float mx = -INFINITY, sum = 0.f;   // running log-sum of the exponents at the start
        constexpr int G = 4;        // passes of dependent gathers in flight (150 k points: 1 3.56, 2 3.47, 4 3.45 ms)
        for (int k0 = lane; k0 < n; k0 += G * kWarp) {
            int id[G];
            double ag[G][3];
#pragma unroll
            for (int j = 0; j < G; j++) id[j] = k0 + j * kWarp < n ? ids[base + k0 + j * kWarp] : -1;
#pragma unroll
            for (int j = 0; j < G; j++)
                if (k0 + j * kWarp < n) nx.get(id[j], ag[j][0], ag[j][1], ag[j][2]);
#pragma unroll
            for (int j = 0; j < G; j++) {
            const int k = k0 + j * kWarp;
            if (k >= n) continue;
            const double (&a)[3] = ag[j];
            float d[3];
#pragma unroll
            for (int i = 0; i < 3; i++) {
                i64 lo, hi;
                ok = fix_from_double_wide(a[i], C.fb, lo, hi) && ok;
                const i64 D = (i64)((u64)P[i] - (u64)lo);
                ok = ok && (Ph[i] - hi - ((u64)P[i] < (u64)lo ? 1 : 0)) == (D >> 63);
                far = max(far, D ^ (D >> 63));
                d[i] = (float)(int)(D >> 32) * u32;
                if (k < kLmeRows) (i == 0 ? F.x0 : (i == 1 ? F.x1 : F.x2))[k] = lo;
            }
            const float f = fmaf(lf0, d[0], fmaf(lf1, d[1], lf2 * d[2])) - bf * fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2]));
            const float m2 = fmaxf(mx, f);
            sum = sum * __expf(mx - m2) + __expf(f - m2);
            mx = m2;
            }
        }
        const float wm = warp_max_f(mx);
        const float ws = warp_sumf(sum > 0.f ? sum * __expf(mx - wm) : 0.f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) far = max(far, (i64)__shfl_xor_sync(0xffffffffu, far, o));
        fixed = __all_sync(0xffffffffu, ok) && (double)far < kFixT;
        // what the farthest node leaves of the range bounds every trial of this point (caller's supports may reach
        // well past the default radius that C.vmax is for)
        const double vmax = kFixT - (double)far;
        // log Z at the start, plus ln 2.8: Z begins near 0.35 (in FP64 evaluations any shift near log Z does)
        const float sh0 = wm + __logf(ws) + 1.04f;
        const double shift0 = isfinite(sh0) ? (double)sh0 : 0.0;
        if (lane < 3) X.xp[lane] = P[lane];
        if (lane == 0) {
            M.trial[0] = M.ws[0] = M.lam[0] = l0;
            M.trial[1] = M.ws[1] = M.lam[1] = l1;
            M.trial[2] = M.ws[2] = M.lam[2] = l2;
            M.t = 1.0;
            M.have_cur = M.iters = M.iters_total = M.halvings = 0;
            M.retried = 1;          // no second start here
            M.shift0 = M.sh = shift0;
            M.state = kNewtonEval;
            X.vmax = vmax;
            X.ok = fix_trial(C, vmax, M.trial, shift0, X.v, X.cst) ? 1 : 0;
        }
    } else if (lane == 0) {
        M.state = kNewtonIdle;
    }
    double *w = n <= kLmeRows ? F.w : nullptr;
    __syncthreads();
    for (;;) {
        if (M.state == kNewtonEval) {
            __syncwarp();
            if (!(fixed && X.ok && lme_eval_fix<true>(C, F, n, M, X, lane, B.table)))
                lme_eval64(nx, ids + base, px, py, pz, beta * kExpScale, w, n, M, lane);
        }
        __syncthreads();
        const bool pending = warp == 0 && fix_round(B.newton, B.fix, C, tol, max_newton, lane);
        if (!__syncthreads_or(pending)) break;
    }
    if (!active) return;
    const bool done = M.state == kNewtonDone;
    if (lane == 0) {
        if (iters_out) iters_out[p] = M.iters;
        if (!done) atomicCAS(status, 0, OTM_ERR_LME_NOCONV);
    }
    if (lane < 3) lam[3 * p + lane] = M.lam[lane];
    if (!done) return;
    // N = w / Z, grad N = -K N d, K = J^-1 = Z J'^-1
    const double iZ = M.iZ, Z = M.C[0];
    double K[6];
#pragma unroll
    for (int i = 0; i < 6; i++) K[i] = -M.inv[i] * Z;
    const bool wide = ((uintptr_t)shape & 31) == 0;
    const double s0 = M.lam[0] * kExpScale, s1 = M.lam[1] * kExpScale, s2 = M.lam[2] * kExpScale, sh_s = M.C[10] * kExpScale;
#pragma unroll 1
    for (int k = lane; k < n; k += kWarp) {
        double N, ex, ey, ez;
        if (!w) {
            double dx, dy, dz;
            N = lme_weight64(nx, ids[base + k], px, py, pz, beta * kExpScale, s0, s1, s2, sh_s, dx, dy, dz) * iZ;
            ex = N * dx; ey = N * dy; ez = N * dz;
        } else if (fixed) {
            N = w[k] * iZ;
            fix_nd(N, X.xp[0] - F.x0[k], X.xp[1] - F.x1[k], X.xp[2] - F.x2[k], C.fb, C.r_unit, ex, ey, ez);
        } else {
            double ax, ay, az;
            N = w[k] * iZ;
            nx.get(ids[base + k], ax, ay, az);
            ex = N * (px - ax); ey = N * (py - ay); ez = N * (pz - az);
        }
        double *o = shape + 4 * (base + k);
        const double4_32a row = make_double4_32a(N, fma(K[0], ex, fma(K[3], ey, K[5] * ez)), fma(K[3], ex, fma(K[1], ey, K[4] * ez)),
                                                 fma(K[5], ex, fma(K[4], ey, K[2] * ez)));
        if (wide) {
            *(double4_32a *)o = row;
        } else {
            o[0] = row.x; o[1] = row.y; o[2] = row.z; o[3] = row.w;
        }
    }
}

cudaError_t launch_lme_only(const double *node_x, const double *mp_x, int64_t nm, const int32_t *ids,
                            const int32_t *counts, int S, double beta, double tol_abs, int max_newton, double *lam,
                            double *shape, int32_t *iters, int32_t *status, cudaStream_t s)
{
    const unsigned blocks = (unsigned)((nm + kLmeWarps - 1) / kLmeWarps);
    if (blocks == 0) return cudaSuccess;
    const size_t smem = sizeof(FixBlock);
    const cudaError_t e = cudaFuncSetAttribute(k_lme_only_fix, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_lme_only_fix<<<blocks, kLmeWarps * kWarp, smem, s>>>(node_x, mp_x, nm, ids, counts, S, beta,
                                                          make_fix_const(beta, 13.815510557964274 / beta), tol_abs, max_newton,
                                                          lam, shape, iters, status);
    return cudaGetLastError();
}

// self-test of the table-driven exponential: mine = exp_scaled(y); ref = CUDA's exp of the same
// argument f = y ln2/1024 carried as a + b (a = fl(y c1), b its rounding error plus y times the
// low part of ln2/1024), ref = exp(a) (1 + b)
__global__ void k_exp_selftest(const double *y, int64_t n, double *mine, double *ref)
{
    __shared__ double T[kExpTable];
    exp_table_load(T);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = y[i];
        mine[i] = exp_scaled(v, T);
        const double a = v * kExpC1;
        const double b = fma(v, kExpC1, -a) + v * kExpC1lo;
        const double e = exp(a);
        ref[i] = fma(e, b, e);
    }
}

cudaError_t launch_exp_selftest(const double *x, int64_t n, double *mine, double *ref, cudaStream_t s)
{
    k_exp_selftest<<<152 * 4, 256, 0, s>>>(x, n, mine, ref);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(128)
    k_return_map_only(const __grid_constant__ otm_material M, const __grid_constant__ RmConst R, double dt, int64_t nm, const double *dF, const double *F_new, double *be,
                      double *ebar, double *T, double *sigma, double *rate, uint8_t *failed, int32_t *status)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nm) return;
    RmIn in;
    for (int i = 0; i < 9; i++) in.dF[i] = dF[9 * p + i];
    for (int i = 0; i < 6; i++) in.be[i] = be[6 * p + i];
    in.ebar = ebar[p];
    in.T = T[p];
    in.guess = 0.0;
    in.Q0 = nullptr;
    const double *Fn = F_new + 9 * p;
    in.J = Fn[0] * (Fn[4] * Fn[8] - Fn[5] * Fn[7]) - Fn[1] * (Fn[3] * Fn[8] - Fn[5] * Fn[6]) +
           Fn[2] * (Fn[3] * Fn[7] - Fn[4] * Fn[6]);
    RmOut o;
    int st = OTM_OK;
    if (!return_map_small(M, R, in, o, st)) st = return_map_point(M, dt, in, o);
    if (st != OTM_OK) {
        atomicCAS(status, 0, st);
        return;
    }
    for (int i = 0; i < 6; i++) {
        be[6 * p + i] = o.be[i];
        sigma[6 * p + i] = o.sig[i];
    }
    ebar[p] = o.ebar;
    T[p] = o.T;
    if (rate) rate[p] = o.rate;
    if (failed) failed[p] = (uint8_t)o.failed;
}

cudaError_t launch_return_map_only(const otm_material *mat, double dt, int64_t nm, const double *dF,
                                   const double *F_new, double *be, double *ebar, double *T, double *sigma,
                                   double *rate, uint8_t *failed, int32_t *status, cudaStream_t s)
{
    const unsigned blocks = (unsigned)((nm + 127) / 128);
    if (blocks == 0) return cudaSuccess;
    k_return_map_only<<<blocks, 128, 0, s>>>(*mat, make_rm_const(*mat, dt), dt, nm, dF, F_new, be, ebar, T, sigma, rate, failed, status);
    return cudaGetLastError();
}

}  // namespace otm
