// otm_grid.cu -- linked-cell grid as a device counting sort (Algorithm 3, step 1), the
// node-major (influence-domain) permutation of the support pairs, and integer scans.
//
// Grid: origin = componentwise minimum of the node positions (exact, ordered-integer atomics),
// dims = floor((max - min) / cell) + 1 per axis, cell id = (iz * ny + iy) * nx + ix.
// Nodes are counted into cells with integer atomics, the counts are scanned, the nodes are
// scattered, and each node's place in its cell's short list is the number of smaller IDs there, so
// the final (cell, ID) order is unique whatever order the atomics ran in. Up to kGridClusterNodes
// nodes one cluster does all of it in one launch.
#include "otm_dev.cuh"

#include <cooperative_groups.h>

namespace otm {

namespace cg = cooperative_groups;

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

// Exclusive scan of in[0..n) into out[0..n) by one block of kScanThreads, starting at `carry`; returns the
// total plus `carry`. Each tile's values are loaded while the tile before it is summed.
__device__ __forceinline__ int block_scan(const int32_t *in, int32_t *out, int64_t n, int carry)
{
    __shared__ int32_t wsum[2][kWarp];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int v[kScanItems];
    const int64_t t0 = (int64_t)threadIdx.x * kScanItems;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) v[k] = t0 + k < n ? in[t0 + k] : 0;
    int buf = 0;
    for (int64_t base = 0; base < n; base += kScanTile, buf ^= 1) {
        const int64_t i0 = base + t0, i1 = i0 + kScanTile;
        int nv[kScanItems], tsum = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            nv[k] = i1 + k < n ? in[i1 + k] : 0;
            tsum += v[k];
        }
        int incl = tsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[buf][warp] = incl;
        __syncthreads();
        // every warp scans the warp sums (two buffers: the next tile writes the other one)
        const int ws = wsum[buf][lane];
        int wi = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        int run = carry + __shfl_sync(0xffffffffu, wi - ws, warp) + incl - tsum;
        carry += __shfl_sync(0xffffffffu, wi, 31);
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            if (i0 + k < n) out[i0 + k] = run;
            run += v[k];
            v[k] = nv[k];
        }
    }
    return carry;
}

// ------------------------------------------------------------------------ bounding box
__global__ void k_bbox_init(GridDev *g)
{
    if (threadIdx.x < 3) {
        g->key_lo[threadIdx.x] = ~0ULL;
        g->key_hi[threadIdx.x] = 0ULL;
    }
}

// the bounding keys of the nodes first, first + stride, ... over the calling warp
__device__ __forceinline__ void warp_bbox(const double4_32a *__restrict__ x, int64_t n, int64_t first, int64_t stride,
                                          unsigned long long (&lo)[3], unsigned long long (&hi)[3])
{
    for (int d = 0; d < 3; d++) { lo[d] = ~0ULL; hi[d] = 0ULL; }
    for (int64_t i = first; i < n; i += stride) {
        double4_32a p = x[i];
        unsigned long long k0 = dkey(p.x), k1 = dkey(p.y), k2 = dkey(p.z);
        lo[0] = min(lo[0], k0); hi[0] = max(hi[0], k0);
        lo[1] = min(lo[1], k1); hi[1] = max(hi[1], k1);
        lo[2] = min(lo[2], k2); hi[2] = max(hi[2], k2);
    }
#pragma unroll
    for (int d = 0; d < 3; d++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    }
}

__global__ void k_bbox(const double4_32a *__restrict__ x, int64_t n, GridDev *g)
{
    unsigned long long lo[3], hi[3];
    warp_bbox(x, n, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, lo, hi);
    if ((threadIdx.x & 31) == 0) {
        for (int d = 0; d < 3; d++) {
            atomicMin(&g->key_lo[d], lo[d]);
            atomicMax(&g->key_hi[d], hi[d]);
        }
    }
}

// origin, dims and cell count from the bounding keys; *err (if given) takes what is wrong with them
__device__ __forceinline__ void grid_setup(const unsigned long long *key_lo, const unsigned long long *key_hi, double cell,
                                           int max_cells, double *origin, int *dims, int *n_cells, unsigned long long *err)
{
    double nd[3];
    bool ok = true;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const double lo = dkey_inv(key_lo[d]), hi = dkey_inv(key_hi[d]);
        origin[d] = lo;
        nd[d] = isfinite(lo) && isfinite(hi) ? floor(__ddiv_rn(__dsub_rn(hi, lo), cell)) + 1.0 : -1.0;
    }
    // the cell count is formed in FP64: each axis is at most max_cells (< 2^31), so the product
    // is below 2^93 and cannot wrap, and any product above max_cells is reported as capacity
    double total = 1.0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (nd[d] == -1.0 && err) raise_error(err, OTM_ERR_NONFINITE, 0);
        const bool in = nd[d] >= 0.0 && nd[d] <= (double)max_cells;
        ok = ok && in;
        dims[d] = in ? (int)nd[d] : 0;
        total *= nd[d];
    }
    if (ok && !(total <= (double)max_cells)) ok = false;
    if (!ok && err) raise_error(err, OTM_ERR_CAPACITY, 0);
    *n_cells = ok ? (int)total : 0;
}

__global__ void k_grid_setup(GridDev *g, double cell, int max_cells, unsigned long long *err)
{
    if (threadIdx.x != 0) return;
    grid_setup(g->key_lo, g->key_hi, cell, max_cells, g->origin, g->dims, &g->n_cells, err);
}

// ------------------------------------------------------------------------ counting sort
__global__ void k_cell_zero(int32_t *cell_count, const GridDev *g)
{
    int n = g->n_cells;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        cell_count[i] = 0;
}

// cell_coord(x, o, c, n, true) for x >= o: the FP64 quotient's floor from an FP32 quotient (error below 2^-22 of
// itself) unless that lies too close to a whole number (or q is not a number). One FP64 subtraction instead of a division, whose
// FP64 instructions (2 lanes a clock) took most of a small build: 14 us of a cluster's 1,024 nodes a block.
__device__ __forceinline__ int cell_coord_fast(double x, double o, double c, float ic, int n)
{
    const float q = f32_round_bits(__dsub_rn(x, o)) * ic;
    const float f = floorf(q), m = q * 0x1p-21f;
    if (!(q < 0.5f) && !(q - f > m && q - f < 1.f - m)) return cell_coord(x, o, c, n, true);
    return min((int)f, n - 1);
}

__device__ __forceinline__ int cell_of(const double4_32a &p, const double (&o)[3], const int (&n)[3], double cell)
{
    const float ic = cell > 1e-28 && cell < 1e28 ? 1.f / (float)cell : INFINITY;   // FP32's range, or the division
    const int ix = cell_coord_fast(p.x, o[0], cell, ic, n[0]);
    const int iy = cell_coord_fast(p.y, o[1], cell, ic, n[1]);
    const int iz = cell_coord_fast(p.z, o[2], cell, ic, n[2]);
    return (iz * n[1] + iy) * n[0] + ix;
}

__global__ void k_cell_count(const double4_32a *__restrict__ x, int64_t n, const GridDev *g, double cell,
                             int32_t *cell_count, int32_t *node_cell, int32_t *node_rank)
{
    if (g->n_cells == 0) return;
    const double o[3] = {g->origin[0], g->origin[1], g->origin[2]};
    const int nd[3] = {g->dims[0], g->dims[1], g->dims[2]};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = cell_of(x[i], o, nd, cell);
        node_cell[i] = c;
        node_rank[i] = atomicAdd(&cell_count[c], 1);
    }
}

// single-block exclusive scan of cell_count[0..n_cells) into cell_start[0..n_cells]
__global__ void __launch_bounds__(kScanThreads) k_scan_cells(const int32_t *count, int32_t *start,
                                                             const GridDev *g)
{
    const int n = g->n_cells;
    const int total = block_scan(count, start, n, 0);
    if (threadIdx.x == 0) start[n] = total;
}

__global__ void k_cell_fill(int64_t n, const int32_t *node_cell, const int32_t *node_rank,
                            const int32_t *cell_start, int32_t *list, const GridDev *g)
{
    if (g->n_cells == 0) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        list[cell_start[node_cell[i]] + node_rank[i]] = (int32_t)i;
}

// node i to its slot: its cell's first plus the number of smaller IDs in the cell (list: the cells' nodes
// in any order)
__device__ __forceinline__ void place_node(int64_t i, const double4_32a *__restrict__ x, const int32_t *node_cell,
                                           const int32_t *cell_start, const int32_t *list, const double (&o)[3],
                                           int32_t *sorted, double4_32a *spos, float4 *spos32)
{
    const int c = node_cell[i];
    double4_32a p = x[i];
    const int b = cell_start[c], e = cell_start[c + 1];
    int s = b;
    for (int j = b; j < e; j++) s += list[j] < (int)i;
    sorted[s] = (int)i;
    p.w = __longlong_as_double((long long)i);
    spos[s] = p;
    spos32[s] = make_float4((float)(p.x - o[0]), (float)(p.y - o[1]), (float)(p.z - o[2]), __int_as_float((int)i));
}

__global__ void k_spos(int64_t n, const int32_t *node_cell, const int32_t *cell_start, const int32_t *list,
                       const double4_32a *__restrict__ x, int32_t *sorted, double4_32a *spos, float4 *spos32,
                       const GridDev *g)
{
    if (g->n_cells == 0) return;
    const double o[3] = {g->origin[0], g->origin[1], g->origin[2]};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        place_node(i, x, node_cell, cell_start, list, o, sorted, spos, spos32);
}

// The whole build by one cluster: the passes above, a cluster barrier after each in the place of a launch
// (nine launches before). Bound by those launches for a few thousand nodes, then by the cluster's own 8 SMs.
struct GridArgs {
    const double4_32a *x;
    int64_t n;
    double cell;
    int max_cells;
    GridDev *g;
    int32_t *cell_count, *cell_start, *node_cell, *node_rank, *sorted;
    double4_32a *spos;
    float4 *spos32;
    unsigned long long *err;
};

__global__ void __launch_bounds__(kScanThreads) k_grid_cluster(const __grid_constant__ GridArgs A)
{
    __shared__ unsigned long long wlo[3][kWarp], whi[3][kWarp], box_lo[3], box_hi[3];
    __shared__ double origin[3];
    __shared__ int dims[3], n_cells, wtot[kWarp], btot;
    cg::cluster_group cl = cg::this_cluster();
    const int nb = (int)cl.num_blocks(), rb = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)rb * kScanThreads + threadIdx.x, T = (int64_t)nb * kScanThreads;
    unsigned long long lo[3], hi[3];
    warp_bbox(A.x, A.n, t0, T, lo, hi);
    if (lane == 0)
        for (int d = 0; d < 3; d++) { wlo[d][warp] = lo[d]; whi[d][warp] = hi[d]; }
    __syncthreads();
    if (warp < 3) {
        unsigned long long l = wlo[warp][lane], h = whi[warp][lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            l = min(l, __shfl_xor_sync(0xffffffffu, l, o));
            h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
        }
        if (lane == 0) { box_lo[warp] = l; box_hi[warp] = h; }
    }
    cl.sync();
    if (warp == 0) {
        for (int d = 0; d < 3; d++) {
            lo[d] = *cl.map_shared_rank(&box_lo[d], lane % nb);
            hi[d] = *cl.map_shared_rank(&box_hi[d], lane % nb);
        }
        for (int d = 0; d < 3; d++)
            for (int o = 16; o > 0; o >>= 1) {
                lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
                hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
            }
    }
    if (threadIdx.x == 0) {
        grid_setup(lo, hi, A.cell, A.max_cells, origin, dims, &n_cells, rb == 0 ? A.err : nullptr);
        if (rb == 0) {
            for (int d = 0; d < 3; d++) {
                A.g->key_lo[d] = lo[d];
                A.g->key_hi[d] = hi[d];
                A.g->origin[d] = origin[d];
                A.g->dims[d] = dims[d];
            }
            A.g->n_cells = n_cells;
        }
    }
    __syncthreads();
    const int nc = n_cells;
    for (int64_t c = t0; c < nc; c += T) A.cell_count[c] = 0;
    cl.sync();
    if (nc == 0) {
        if (rb == 0 && threadIdx.x == 0) A.cell_start[0] = 0;
        return;
    }
    const double o[3] = {origin[0], origin[1], origin[2]};
    const int nd[3] = {dims[0], dims[1], dims[2]};
    for (int64_t i = t0; i < A.n; i += T) {
        const int c = cell_of(A.x[i], o, nd, A.cell);
        A.node_cell[i] = c;
        A.node_rank[i] = atomicAdd(&A.cell_count[c], 1);
    }
    cl.sync();
    // a contiguous share of the cells a block: its total, the totals before it, then its scan
    const int per = (nc + nb - 1) / nb, c0 = min(rb * per, nc), c1 = min(c0 + per, nc);
    int sum = 0;
    for (int c = c0 + (int)threadIdx.x; c < c1; c += kScanThreads) sum += A.cell_count[c];
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) wtot[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        const int t = __reduce_add_sync(0xffffffffu, wtot[lane]);
        if (lane == 0) btot = t;
    }
    cl.sync();
    int off = 0;
    for (int r = 0; r < rb; r++) off += *cl.map_shared_rank(&btot, r);
    block_scan(A.cell_count + c0, A.cell_start + c0, c1 - c0, off);
    if (rb == 0 && threadIdx.x == 0) A.cell_start[nc] = (int)A.n;
    cl.sync();
    int32_t *list = A.cell_count;   // the counts are done with
    for (int64_t i = t0; i < A.n; i += T) list[A.cell_start[A.node_cell[i]] + A.node_rank[i]] = (int32_t)i;
    cl.sync();
    for (int64_t i = t0; i < A.n; i += T)
        place_node(i, A.x, A.node_cell, A.cell_start, list, o, A.sorted, A.spos, A.spos32);
}

static int grid_blocks(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 16) b = 152 * 16;
    if (b < 1) b = 1;
    return (int)b;
}

// One block up to kGridBlockNodes nodes (no cluster barriers across SMs: 1.5 us less at 300 nodes, the same at
// 1,000), a cluster of 8 up to kGridClusterNodes, eight launches over the chip beyond. In a step, eight
// launches against the cluster: 34 / 23 us at 1.6 k nodes, 37 / 23 at 6 k, 37 / 27 at 13 k, 43 / 39 at 38 k;
// replayed from a graph, where a launch costs less, 26 / 29 us at 2 k, 29 / 38 at 16 k, 33 / 51 at 32 k.
constexpr int64_t kGridBlockNodes = 512, kGridClusterNodes = 16384;

static cudaError_t grid_build_impl(const double4_32a *x, int64_t nn, double cell, int max_cells, GridDev *g,
                                   int32_t *cell_count, int32_t *cell_start, int32_t *node_cell,
                                   int32_t *node_rank, int32_t *sorted, double4_32a *spos, float4 *spos32,
                                   unsigned long long *err, cudaStream_t s, long long *launches)
{
    if (nn <= kGridClusterNodes) {
        const GridArgs A = {x, nn, cell, max_cells, g, cell_count, cell_start, node_cell, node_rank, sorted, spos, spos32, err};
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = nn <= kGridBlockNodes ? 1 : 8;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(at[0].val.clusterDim.x);
        cfg.blockDim = dim3(kScanThreads);
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_grid_cluster, A);
        if (launches) *launches += 1;
        return e;
    }
    int32_t *list = cell_count;   // after the scan the counts are done with
    k_bbox_init<<<1, 32, 0, s>>>(g);
    k_bbox<<<grid_blocks(nn, 256), 256, 0, s>>>(x, nn, g);
    k_grid_setup<<<1, 32, 0, s>>>(g, cell, max_cells, err);
    k_cell_zero<<<grid_blocks(max_cells, 256), 256, 0, s>>>(cell_count, g);
    k_cell_count<<<grid_blocks(nn, 256), 256, 0, s>>>(x, nn, g, cell, cell_count, node_cell, node_rank);
    k_scan_cells<<<1, kScanThreads, 0, s>>>(cell_count, cell_start, g);
    k_cell_fill<<<grid_blocks(nn, 256), 256, 0, s>>>(nn, node_cell, node_rank, cell_start, list, g);
    k_spos<<<grid_blocks(nn, 256), 256, 0, s>>>(nn, node_cell, cell_start, list, x, sorted, spos, spos32, g);
    if (launches) *launches += 8;
    return cudaGetLastError();
}

cudaError_t launch_grid_build(const Dev &D, cudaStream_t s, long long *launches)
{
    return grid_build_impl(D.x, D.nn, D.cell, D.max_cells, D.grid, D.cell_count, D.cell_start,
                           D.node_cell, D.node_rank, D.sorted, D.spos, D.spos32, D.err, s, launches);
}

// ------------------------------------------------------------------------ generic scan
// Exclusive scan of n int32 values into out[0..n] (out[n] = total). Three phases: tile sums,
// a single-block scan of the tile sums, and a rescan of every tile with its offset.
__global__ void __launch_bounds__(kScanThreads) k_tile_sums(const int32_t *in, int64_t n, int32_t *tile_sum)
{
    __shared__ int32_t wsum[kWarp];
    int64_t i0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    int t = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) t += (i0 + k < n) ? in[i0 + k] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        int v = wsum[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) tile_sum[blockIdx.x] = v;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tile_sums(int32_t *tile_sum, int64_t ntiles)
{
    __shared__ int32_t wsum[kWarp];
    __shared__ int32_t carry_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int64_t base = 0; base < ntiles; base += kScanThreads) {
        int64_t i = base + threadIdx.x;
        int v = (i < ntiles) ? tile_sum[i] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int ws = wsum[lane], wi = ws;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int t = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += t;
            }
            wsum[lane] = wi - ws;
        }
        __syncthreads();
        int excl = carry_s + wsum[warp] + incl - v;
        if (i < ntiles) tile_sum[i] = excl;
        __syncthreads();
        if (threadIdx.x == kScanThreads - 1) carry_s = excl + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) tile_sum[ntiles] = carry_s;
}

__global__ void __launch_bounds__(kScanThreads) k_tile_rescan(const int32_t *in, int64_t n,
                                                              const int32_t *tile_off, int32_t *out,
                                                              int64_t ntiles)
{
    __shared__ int32_t wsum[kWarp];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t i0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    int v[kScanItems];
    int tsum = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        v[k] = (i0 + k < n) ? in[i0 + k] : 0;
        tsum += v[k];
    }
    int incl = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int ws = wsum[lane], wi = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        wsum[lane] = wi - ws;
    }
    __syncthreads();
    int run = tile_off[blockIdx.x] + wsum[warp] + incl - tsum;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        if (i0 + k < n) out[i0 + k] = run;
        run += v[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = tile_off[ntiles];
}

// One block scans it all: 6 us at 1.6 k values, 8 at 6 k, 10 at 13 k, against 15 for the three launches; 16.4
// against 15 at 38 k.
__global__ void __launch_bounds__(kScanThreads) k_scan_block(const int32_t *in, int32_t *out, int64_t n)
{
    const int total = block_scan(in, out, n, 0);
    if (threadIdx.x == 0) out[n] = total;
}
constexpr int64_t kScanBlockMax = 24576;

// tile scratch: ntiles + 1 ints directly after out[n] is not available, so it lives in
// a static-size region of the caller's buffer `tmp`
cudaError_t launch_exclusive_scan_tmp(const int32_t *in, int32_t *out, int64_t n, int32_t *tmp,
                                      cudaStream_t s, long long *launches)
{
    if (n <= kScanBlockMax) {
        k_scan_block<<<1, kScanThreads, 0, s>>>(in, out, n);
        if (launches) *launches += 1;
        return cudaGetLastError();
    }
    const int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    k_tile_sums<<<(unsigned)ntiles, kScanThreads, 0, s>>>(in, n, tmp);
    k_scan_tile_sums<<<1, kScanThreads, 0, s>>>(tmp, ntiles);
    k_tile_rescan<<<(unsigned)ntiles, kScanThreads, 0, s>>>(in, n, tmp, out, ntiles);
    if (launches) *launches += 3;
    return cudaGetLastError();
}

size_t scan_tmp_ints(int64_t n) { return (size_t)((n + kScanTile - 1) / kScanTile + 2); }

// ------------------------------------------------------------------------ node-major offsets
// noff = exclusive scan of the influence counts; the LME kernel then writes each pair's
// contribution at noff[node] + rank, so every node's influence list is contiguous.
cudaError_t launch_node_offsets(const Dev &D, int32_t *tmp, cudaStream_t s, long long *launches)
{
    return launch_exclusive_scan_tmp(D.ncount, D.noff, D.nn, tmp, s, launches);
}

// ------------------------------------------------------------------------ stand-alone search scratch
static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

static int search_max_cells(int64_t nn) { return (int)(16 * nn + 65536); }

size_t search_scratch_bytes(int64_t nn)
{
    int mc = search_max_cells(nn);
    size_t b = 0;
    b += align256(sizeof(GridDev));
    b += 2 * align256((size_t)nn * sizeof(double4_32a));
    b += align256((size_t)nn * sizeof(float4));
    b += 2 * align256(((size_t)mc + 1) * sizeof(int32_t));
    b += 3 * align256((size_t)nn * sizeof(int32_t));
    b += align256(sizeof(unsigned long long));
    return b;
}

bool carve_search_scratch(void *base, size_t bytes, int64_t nn, SearchScratch *S)
{
    if (search_scratch_bytes(nn) > bytes) return false;
    char *p = (char *)base;
    int mc = search_max_cells(nn);
    S->g = (GridDev *)p; p += align256(sizeof(GridDev));
    S->x4 = (double4_32a *)p; p += align256((size_t)nn * sizeof(double4_32a));
    S->spos = (double4_32a *)p; p += align256((size_t)nn * sizeof(double4_32a));
    S->spos32 = (float4 *)p; p += align256((size_t)nn * sizeof(float4));
    S->cell_count = (int32_t *)p; p += align256(((size_t)mc + 1) * sizeof(int32_t));
    S->cell_start = (int32_t *)p; p += align256(((size_t)mc + 1) * sizeof(int32_t));
    S->node_cell = (int32_t *)p; p += align256((size_t)nn * sizeof(int32_t));
    S->node_rank = (int32_t *)p; p += align256((size_t)nn * sizeof(int32_t));
    S->sorted = (int32_t *)p; p += align256((size_t)nn * sizeof(int32_t));
    S->err = (unsigned long long *)p;
    S->max_cells = mc;
    return true;
}

__global__ void k_pack3to4(const double *__restrict__ x3, int64_t n, double4_32a *x4)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        x4[i] = make_double4_32a(x3[3 * i], x3[3 * i + 1], x3[3 * i + 2], 0.0);
}

// rows of `width` bytes (a multiple of 8) between a pitched layout and a dense one, 8 bytes per
// thread: a state transfer then moves one contiguous block instead of many short rows
__global__ void k_rows_to_dense(const char *__restrict__ src, size_t pitch, size_t width, int64_t rows,
                                double *__restrict__ dst)
{
    const int64_t words = (int64_t)(width / 8), total = rows * words;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / words, w = t - r * words;
        dst[t] = *(const double *)(src + (size_t)r * pitch + (size_t)w * 8);
    }
}

__global__ void k_rows_from_dense(const double *__restrict__ src, size_t pitch, size_t width, int64_t rows,
                                  char *__restrict__ dst)
{
    const int64_t words = (int64_t)(width / 8), total = rows * words;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / words, w = t - r * words;
        *(double *)(dst + (size_t)r * pitch + (size_t)w * 8) = src[t];
    }
}

cudaError_t launch_rows_to_dense(const void *src, size_t pitch, size_t width, int64_t rows, void *dst, cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    k_rows_to_dense<<<grid_blocks(rows * (int64_t)(width / 8), 256), 256, 0, s>>>((const char *)src, pitch, width,
                                                                                  rows, (double *)dst);
    return cudaGetLastError();
}

cudaError_t launch_rows_from_dense(const void *src, size_t pitch, size_t width, int64_t rows, void *dst,
                                   cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    k_rows_from_dense<<<grid_blocks(rows * (int64_t)(width / 8), 256), 256, 0, s>>>((const double *)src, pitch,
                                                                                    width, rows, (char *)dst);
    return cudaGetLastError();
}

cudaError_t launch_pack3to4(const double *x3, int64_t n, double4_32a *x4, cudaStream_t s, long long *launches)
{
    if (n <= 0) return cudaSuccess;
    k_pack3to4<<<grid_blocks(n, 256), 256, 0, s>>>(x3, n, x4);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

// initial state (Algorithm 1, REQUIRE): F = dF = b^e = 1, sigma = 0, ebar = 0, T = T0,
// lambda = 0, original IDs, x_prev = x, du32 = du
__global__ void k_init_state(const Dev D, double T0)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < D.nm;
         p += (int64_t)gridDim.x * blockDim.x) {
        for (int i = 0; i < 9; i++) D.F[9 * p + i] = D.dF[9 * p + i] = (i % 4 == 0) ? 1.0 : 0.0;
        for (int i = 0; i < 6; i++) {
            D.be[6 * p + i] = (i < 3) ? 1.0 : 0.0;
            D.sig[6 * p + i] = 0.0;
        }
        D.ebar[p] = 0.0;
        D.T[p] = T0;
        D.xp_prev[p] = D.xp[p];
        D.rate[p] = 0.0;
        D.lam[3 * p] = D.lam[3 * p + 1] = D.lam[3 * p + 2] = 0.0;
        D.lam_prev[3 * p] = D.lam_prev[3 * p + 1] = D.lam_prev[3 * p + 2] = 0.0;
        D.lam_prev2[3 * p] = D.lam_prev2[3 * p + 1] = D.lam_prev2[3 * p + 2] = 0.0;
        D.lam_prev3[3 * p] = D.lam_prev3[3 * p + 1] = D.lam_prev3[3 * p + 2] = 0.0;
        for (int i = 0; i < 9; i++) D.Qe[9 * p + i] = (i % 4 == 0) ? 1.0 : 0.0;
        D.logz[p] = D.logz0;
        D.logz_in[p] = D.logz0;
        D.failed[p] = 0;
        D.cnt[p] = 0;
        D.newton_it[p] = 0;
        D.mgid[p] = p;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < D.nn;
         i += (int64_t)gridDim.x * blockDim.x) {
        D.ngid[i] = i;
        D.x_prev[i] = D.x[i];
        const double4_32a u = D.du[i];
        D.du32[i] = make_float4((float)u.x, (float)u.y, (float)u.z, 0.f);
        D.mr[i] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    }
}

__global__ void k_du_to_f32(const Dev D)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < D.nn;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double4_32a u = D.du[i];
        D.du32[i] = make_float4((float)u.x, (float)u.y, (float)u.z, 0.f);
    }
}

cudaError_t launch_du_to_f32(const Dev &D, cudaStream_t s, long long *launches)
{
    k_du_to_f32<<<grid_blocks(D.nn, 256), 256, 0, s>>>(D);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_init_state(const Dev &D, double T0, cudaStream_t s, long long *launches)
{
    int64_t n = D.nm > D.nn ? D.nm : D.nn;
    k_init_state<<<grid_blocks(n, 256), 256, 0, s>>>(D, T0);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

__global__ void k_grid_out(const GridDev *g, double *out)
{
    if (threadIdx.x < 3) {
        out[threadIdx.x] = g->origin[threadIdx.x];
        out[3 + threadIdx.x] = (double)g->dims[threadIdx.x];
    }
}

cudaError_t build_search_grid(const double *node_x, int64_t nn, double cell, SearchScratch *S,
                              double *grid_out, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(S->err, 0xff, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    k_pack3to4<<<grid_blocks(nn, 256), 256, 0, s>>>(node_x, nn, S->x4);
    e = grid_build_impl(S->x4, nn, cell, S->max_cells, S->g, S->cell_count, S->cell_start, S->node_cell,
                        S->node_rank, S->sorted, S->spos, S->spos32, S->err, s, nullptr);
    if (e != cudaSuccess) return e;
    if (grid_out) k_grid_out<<<1, 32, 0, s>>>(S->g, grid_out);
    return cudaGetLastError();
}

}  // namespace otm
