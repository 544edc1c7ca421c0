// otm_node.cu -- the node kernel (sm_103a): lumped mass and internal force as a segmented
// reduction over each node's influence list (Eq. 5), the central-difference update (Eq. 4),
// rigid contact (Sec. 4.1 wall, Sec. 4.2 tool) and the position update (Eq. 6).
//
// Determinism without float atomics and without sorting: every pair contribution is converted
// to a fixed-point integer whose least significant bit is 2^(Emax - 110) (FP64 path, 128-bit
// accumulators) or 2^(Emax - 46) (mixed path, 64-bit accumulators), Emax being the largest
// binary exponent of that field over all pairs of the step. Integer addition is associative,
// so the sum is exact and independent of the order in which the influence list was filled.
// Terms below the least significant bit (2^-110, resp. 2^-46, of the largest term) are truncated.
//
// Headroom: a term is below 2^(Emax + 1), i.e. below 2^111 (FP64) or 2^47 (mixed) units, and a
// node has at most 65,536 influences (the search raises OTM_ERR_CAPACITY beyond), so a node sum
// stays below 2^127 resp. 2^63 and fits the signed accumulator whatever the signs.
#include "otm_dev.cuh"

#include <type_traits>

namespace otm {

__device__ __forceinline__ u64 shfl_xor_any(u64 v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ u128 shfl_xor_any(u128 v, int o)
{
    return ((u128)shfl_xor_any((u64)(v >> 64), o) << 64) | shfl_xor_any((u64)v, o);
}

// the warp's sum in every lane
template <typename U>
__device__ __forceinline__ U warp_total(const FixedSum<U> &a)
{
    U v = a.v + (U)(u64)a.neg;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += shfl_xor_any(v, o);
    return v;
}

__device__ __forceinline__ double sum_value(u128 a, int emax)
{
    // (hi * 2^64 + lo) * 2^(emax - 110)
    const double v = (double)(long long)(u64)(a >> 64) * 18446744073709551616.0 + (double)(u64)a;
    return ldexp(v, emax - 110);
}
__device__ __forceinline__ double sum_value(u64 a, int emax) { return ldexp((double)(long long)a, emax - 46); }

// ---------------------------------------------------------------------------- contact
// rigid frictionless wall: project a penetrating node onto the plane
__device__ __forceinline__ void wall_project(const Dev &D, double &x, double &y, double &z)
{
    const double g = (x - D.wall_p[0]) * D.wall_n[0] + (y - D.wall_p[1]) * D.wall_n[1] +
                     (z - D.wall_p[2]) * D.wall_n[2];
    if (g < 0.0) {
        x -= g * D.wall_n[0];
        y -= g * D.wall_n[1];
        z -= g * D.wall_n[2];
    }
}

// rigid tool (wedge between rake and flank faces, moving along -x): normal projection onto the
// nearer face, Coulomb stick/slip of the increment relative to the tool at the penalty limit
__device__ __forceinline__ void tool_project(const Dev &D, double t_next, double ux, double uy, double uz,
                                             double &x, double &y, double &z)
{
    const double xt = D.tool_x0 - D.tool_v * t_next, yt = D.tool_tip_y;
    const double nrx = -cos(D.tool_rake), nry = sin(D.tool_rake);
    const double nfx = sin(D.tool_clear), nfy = -cos(D.tool_clear);
    const double rx = x - xt, ry = y - yt;
    const double gr = rx * nrx + ry * nry, gf = rx * nfx + ry * nfy;
    if (!(gr < 0.0 && gf < 0.0)) return;
    const bool rake = (gr >= gf);
    const double nx = rake ? nrx : nfx, ny = rake ? nry : nfy;
    const double pen = -(rake ? gr : gf);
    x += pen * nx;
    y += pen * ny;
    const double wx = ux + D.tool_v * D.dt, wy = uy, wz = uz;
    const double wn = wx * nx + wy * ny;
    const double tx = wx - wn * nx, ty = wy - wn * ny, tz = wz;
    const double tn = sqrt(tx * tx + ty * ty + tz * tz);
    const double lim = D.friction * pen;
    const double sc = (tn <= lim) ? 1.0 : lim / tn;
    x -= sc * tx;
    y -= sc * ty;
    z -= sc * tz;
}

// ---------------------------------------------------------------------------- node kernel
// W warps a node. Bound by the integer pipes (about 30 instructions a term; the FP64 sums of 38 k nodes with
// 1,420 terms each, 1.7 GB: 0.50 ms with three-way branches on the shift, 0.35 ms without).
template <bool MIXED, int W>
__global__ void __launch_bounds__(kNodeWarps * kWarp) k_node_update(const __grid_constant__ Dev D, double t_next)
{
    using U = typename std::conditional<MIXED, u64, u128>::type;
    __shared__ U part[W > 1 ? kNodeWarps : 1][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * (kNodeWarps / W) + warp / W;
    if (W == 1 && (i >= D.nn || has_error(D.err))) return;
    if (W > 1 && __syncthreads_or(has_error(D.err))) return;   // one node a block
    const int b = D.noff[i], L = D.noff[i + 1] - b;
    const int em = D.emax[0], ef = D.emax[1];
    FixedSum<U> t[4];
#pragma unroll
    for (int j = 0; j < 4; j++) t[j].v = 0, t[j].neg = 0;
    // a lane's terms W warps apart, the next one loading while this one is added
    using T = typename std::conditional<MIXED, float4, double4_32a>::type;
    const T *src = (MIXED ? (const T *)D.contrib32 : (const T *)D.contrib64) + b;
    constexpr int step = W * kWarp;
    int k = (warp % W) * kWarp + lane;
    T c;
    if (k < L) c = src[k];
    for (; k < L; k += step) {
        T n = c;
        if (k + step < L) n = src[k + step];
        add_fixed(t[0], c.x, em);
        add_fixed(t[1], c.y, ef);
        add_fixed(t[2], c.z, ef);
        add_fixed(t[3], c.w, ef);
        c = n;
    }
    U v[4];
#pragma unroll
    for (int j = 0; j < 4; j++) v[j] = warp_total(t[j]);
    if (W > 1) {
        if (lane == 0) {
#pragma unroll
            for (int j = 0; j < 4; j++) part[warp][j] = v[j];
        }
        __syncthreads();
        if (warp != 0) return;
#pragma unroll
        for (int w = 1; w < W; w++)
#pragma unroll
            for (int j = 0; j < 4; j++) v[j] += part[w][j];
    }
    const double m = sum_value(v[0], em), rx = sum_value(v[1], ef), ry = sum_value(v[2], ef), rz = sum_value(v[3], ef);
    if (lane != 0) return;
    D.mr[i] = make_double4_32a(m, rx, ry, rz);
    const double4_32a xo = D.x[i];
    double ux, uy, uz;
    const bool fixed = (D.nflags[i] & OTM_FLAG_FIXED) != 0;
    const double dt2 = D.dt * D.dt;
    if (MIXED) {
        float4 u = D.du32[i];
        if (fixed) {
            u = make_float4(0.f, 0.f, 0.f, 0.f);
        } else if (m > 0.0) {
            const float s = (float)(dt2 / m);
            u.x += s * (float)rx;
            u.y += s * (float)ry;
            u.z += s * (float)rz;
        }
        ux = u.x; uy = u.y; uz = u.z;
    } else {
        double4_32a u = D.du[i];
        if (fixed) {
            u = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        } else if (m > 0.0) {
            u.x += dt2 * rx / m;
            u.y += dt2 * ry / m;
            u.z += dt2 * rz / m;
        }
        ux = u.x; uy = u.y; uz = u.z;
    }
    double x = xo.x + ux, y = xo.y + uy, z = xo.z + uz;
    if (!fixed) {
        if (D.wall) wall_project(D, x, y, z);
        if (D.tool) tool_project(D, t_next, ux, uy, uz, x, y, z);
    }
    ux = x - xo.x; uy = y - xo.y; uz = z - xo.z;
    if (MIXED)
        D.du32[i] = make_float4((float)ux, (float)uy, (float)uz, 0.f);
    D.du[i] = make_double4_32a(ux, uy, uz, 0.0);
    D.x_prev[i] = xo;
    D.x[i] = make_double4_32a(x, y, z, 0.0);
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) raise_error(D.err, OTM_ERR_NONFINITE, D.ngid[i]);
}

// A block per node (its list split over the warps) up to kNodeSplitMax nodes, a warp per node beyond: with a
// warp each, a few thousand nodes leave most of the chip's warps idle. FP64, warp / block per node: 45 / 30 us
// at 1.6 k nodes, 99 / 86 at 6 k, 157 / 155 at 13 k, 350 / 375 at 38 k.
constexpr int64_t kNodeSplitMax = 8192;

cudaError_t launch_node_update(const Dev &D, double t_next, cudaStream_t s, long long *launches)
{
    if (D.nn <= 0) return cudaSuccess;
    const bool split = D.nn <= kNodeSplitMax;
    const unsigned blocks = (unsigned)(split ? D.nn : (D.nn + kNodeWarps - 1) / kNodeWarps);
    const bool mixed = D.precision == OTM_PRECISION_MIXED;
    auto *k = mixed ? (split ? k_node_update<true, kNodeWarps> : k_node_update<true, 1>)
                    : (split ? k_node_update<false, kNodeWarps> : k_node_update<false, 1>);
    k<<<blocks, kNodeWarps * kWarp, 0, s>>>(D, t_next);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

}  // namespace otm
