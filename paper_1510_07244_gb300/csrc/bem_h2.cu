// H2-matrix-vector product and conjugate gradients on the device (Sections
// 2.4 and 4).
//
// The matrix is G ~ sum over near blocks N_ts + sum over admissible blocks
// V_t S_ts V_s^T with nested cluster bases: V_t of a leaf is its
// interpolation matrix, V_t of a cluster with sons is diag(V_t1, V_t2) V^_t
// (transfer matrix V^_t, rows = the sons' pivots).  y = G x runs as
//   near     p_b = N_ts x|s for every near block b            one warp per block
//   forward  x^_s = V_s^T x|s (all leaves), then V^_s^T (x^_s1; x^_s2), deepest level first
//   coupling p_b = S_ts x^_s for every admissible block b     one warp per block
//   backward y^_t = sum_b p_b + the father's part, (parts of y^_t1; y^_t2) = V^_t y^_t,
//            top level first; then y|t = sum_b p_b (near) + V_t y^_t (all leaves)
// Every sum has a fixed order (no atomics), so products are bitwise reproducible.
// The near field runs beside the levels and the coupling, which have a stream of
// their own.
// Clusters above the first admissible block take part in neither transformation.
// All arithmetic is FP64.  The matrix is memory- and latency-bound: per product it
// reads every near-field and coupling entry once (8 bytes each) and does 2 flops
// per entry; the levels are a chain of small launches.
//   - A warp per block, all its column loads in flight at once, keeps the two
//     block passes at the memory system's rate whatever the blocks per cluster
//     (one CTA per cluster with a warp per eighth block: 2.6 TB/s, 2 waves).
//   - The level launches overlap (programmatic dependent launch): each reads its
//     own matrices into registers before it waits for the level before it.
// 32768-triangle sphere, 14.2 M near and 30.7 M coupling entries, 13 levels:
// 336 us per product with a CTA per cluster everywhere and plain launches, 215 us
// so: near field 17 us beside the rest, coupling about 108 us (its multiplications
// alone keep the FP64 pipe busy for 63 us, its entries take 36 us of bandwidth), the
// chain of 19 level launches and the leaves 83 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "bem_internal.h"
#include "bem_pdl.cuh"

namespace bem {

struct alignas(16) H2Node {
    int64_t v_off;             // its matrix in vals / valsT
    int64_t src_off;           // its row sources in src
    int64_t near_off, far_off; // its blocks' products in near_part / far_part
    int32_t rows, rank;        // R_c, K_c
    int32_t hat;               // x^_c, y^_c in the hat vectors
    int32_t n_near, n_far;     // its near / admissible blocks
    int32_t idx;               // its index set in cl_idx
    int32_t leaf;
    int32_t up;                // 1: the father's part of y^_c is in yhat; bit 1: y^_c is needed at all
};

struct alignas(16) H2Block {
    int64_t val;               // first entry of the block's values
    int64_t out;               // its product in near_part / far_part
    int32_t nr, nc;            // rows, columns
    int32_t src, pad;          // near: column indices in cl_idx; far: x^ of the column cluster
};

}  // namespace bem

struct bem_h2 {
    int64_t n = 0;
    int32_t nc = 0, max_rank = 0;
    std::vector<void *> allocs;
    bem::H2Node *nodes = nullptr;  // per cluster (device)
    int32_t *src = nullptr;        // row sources: vector index (leaf) or hat index (else)
    double *vals = nullptr;        // basis matrices (rows x K_c row-major)
    double *valsT = nullptr;       // the same, each transposed (K_c x rows row-major)
    // near and admissible blocks, ordered by row cluster
    bem::H2Block *near_blk = nullptr, *far_blk = nullptr;
    int64_t n_near = 0, n_far = 0;
    const double *near_vals = nullptr, *far_vals = nullptr;
    double *near_part = nullptr, *far_part = nullptr;   // the blocks' products
    int32_t *cl_idx = nullptr;     // cluster index sets
    // device cluster lists: forward passes (all leaves, then by level, deepest
    // first), backward passes (by level from the top, then all leaves)
    std::vector<int32_t *> fwd, bwd;
    std::vector<int32_t> fwd_n, bwd_n;
    double *xhat = nullptr, *yhat = nullptr;
    int64_t n_hat = 0;
    double *diag = nullptr;        // added to the diagonal (null: none)
    // conjugate gradients: vectors and scalars
    double *r = nullptr, *p = nullptr, *q = nullptr, *part = nullptr, *scal = nullptr;
    // the levels and the coupling run on a stream of their own beside the near field
    cudaStream_t side = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};

namespace bem {

namespace {

constexpr int kDotBlocks = 512;

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr int kH2Warps = 8;

// Product of one block by one warp: lane i = row i (rows in passes of 32), all
// 32 column loads of a pass in flight; x: the column values, gathered through idx
// if GATHER.
template <bool GATHER>
__global__ void __launch_bounds__(256) k_h2_blocks(const H2Block *__restrict__ blk, int64_t n,
                                                   const double *__restrict__ vals,
                                                   const int32_t *__restrict__ idx,
                                                   const double *x, double *part)
{
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    H2Block B = {};
    if (b < n) B = blk[b];
    // entries of the first pass before the wait
    double a[32];
    const double *v = vals + B.val;
    auto load = [&](int i0, int c0) {
        const double *w = v + min(i0 + lane, B.nr - 1) + (int64_t)c0 * B.nr;
#pragma unroll
        for (int j = 0; j < 32; ++j) a[j] = c0 + j < B.nc ? __ldg(w + (int64_t)j * B.nr) : 0.0;
    };
    if (B.nr > 0) load(0, 0);
    if (!GATHER) {
        pdl_wait();
        pdl_launch();
    }
    for (int i0 = 0; i0 < B.nr; i0 += 32) {
        double acc = 0.0;
        for (int c0 = 0; c0 < B.nc; c0 += 32) {
            if (i0 + c0 > 0) load(i0, c0);
            const int nc = min(32, B.nc - c0);
            double xc = 0.0;
            if (lane < nc) xc = x[GATHER ? __ldg(idx + B.src + c0 + lane) : B.src + c0 + lane];
            double odd = 0.0;
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
                if (j >= nc) break;                    // uniform across the warp
                acc = fma(a[j], __shfl_sync(0xffffffffu, xc, j), acc);
                odd = fma(a[j + 1], __shfl_sync(0xffffffffu, xc, j + 1), odd);
            }
            acc += odd;
        }
        if (i0 + lane < B.nr) part[B.out + i0 + lane] = acc;
    }
}

// Forward transformation of a list of clusters: x^_c = V_c^T v, v = x at the
// leaf's indices or the sons' x^ entries.  One CTA per cluster: lane k = column k
// (K_c <= 32), the 8 warps take every 8th row, and their partial sums are added in
// warp order.  Up to 64 rows (every cluster with sons) the matrix and the row
// sources are in registers before the wait.
__global__ void __launch_bounds__(256) k_h2_forward(const H2Node *__restrict__ nodes,
                                                    const int32_t *__restrict__ list,
                                                    const double *__restrict__ vals,
                                                    const int32_t *__restrict__ sources,
                                                    const double *x, double *xhat)
{
    __shared__ double part[kH2Warps][32];
    const H2Node N = nodes[list[blockIdx.x]];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = N.rows, K = N.rank;
    const double *V = vals + N.v_off;
    const int32_t *src = sources + N.src_off;
    const double *v = N.leaf ? x : xhat;
    double acc = 0.0;
    if (R <= 8 * kH2Warps) {
        double a[8];
        int32_t at[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = warp + kH2Warps * u;
            at[u] = i < R ? __ldg(src + i) : 0;
            a[u] = i < R && lane < K ? __ldg(V + (int64_t)i * K + lane) : 0.0;
        }
        pdl_wait();
        pdl_launch();
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (warp + kH2Warps * u < R) acc = fma(a[u], v[at[u]], acc);
    } else {
        pdl_wait();
        pdl_launch();
        if (lane < K) {
#pragma unroll 4
            for (int i = warp; i < R; i += kH2Warps)
                acc = fma(V[(int64_t)i * K + lane], v[__ldg(src + i)], acc);
        }
    }
    part[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && lane < K) {
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < kH2Warps; ++k) sum += part[k][lane];
        xhat[N.hat + lane] = sum;
    }
}

// Backward transformation of a list of clusters: y^_c = the father's part + the
// sum of its blocks' products; every row i of V_c then gives (V_c y^_c)_i, the
// father's part of a son's y^ entry, or for a leaf (LEAF), added to its near
// blocks' products and diag x, the result at the leaf's index.  One CTA per
// cluster; four threads per row (columns k = part mod 4, combined by two fixed
// shuffles; the transposed basis makes consecutive rows consecutive words).
template <bool LEAF>
__global__ void __launch_bounds__(256) k_h2_backward(const H2Node *__restrict__ nodes,
                                                     const int32_t *__restrict__ list,
                                                     const double *__restrict__ valsT,
                                                     const int32_t *__restrict__ sources,
                                                     const double *far_part,
                                                     const double *__restrict__ near_part,
                                                     const double *__restrict__ diag,
                                                     const double *__restrict__ x, double *yhat,
                                                     double *y)
{
    __shared__ double part[kH2Warps][32];
    __shared__ double yc[32];
    const H2Node N = nodes[list[blockIdx.x]];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = N.rows, K = (N.up & 2) ? N.rank : 0;
    const double *VT = valsT + N.v_off;
    const int32_t *src = sources + N.src_off;
    const int row = threadIdx.x >> 2, quarter = threadIdx.x & 3;
    // first 64 rows: matrix (eight columns per thread) and target before the wait
    double a[8];
    int32_t to = 0;
    if (row < R) {
        to = __ldg(src + row);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = quarter + 4 * u;
            a[u] = k < K ? __ldg(VT + (int64_t)k * R + row) : 0.0;
        }
    }
    pdl_wait();
    pdl_launch();
    // the father's part, which may be much larger than the blocks' products, comes last
    double acc = 0.0, father = 0.0;
    if (lane < K) {
        if (warp == 0 && (N.up & 1)) father = yhat[N.hat + lane];
#pragma unroll 4
        for (int b = warp; b < N.n_far; b += kH2Warps) acc += far_part[N.far_off + (int64_t)b * K + lane];
    }
    part[warp][lane] = acc;
    __syncthreads();
    if (warp == 0) {
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < kH2Warps; ++k) sum += part[k][lane];
        yc[lane] = lane < K ? sum + father : 0.0;
    }
    __syncthreads();
    for (int i0 = 0; i0 < R; i0 += 64) {
        const int i = i0 + row;
        // near field and V y^ apart: a product added to the larger near field would be
        // rounded to its unit K_c times
        double s = 0.0, near = 0.0;
        if (i < R) {
            if (LEAF) {
#pragma unroll 4
                for (int b = quarter; b < N.n_near; b += 4) near += near_part[N.near_off + (int64_t)b * R + i];
            }
            if (i0 == 0) {
#pragma unroll
                for (int u = 0; u < 8; ++u) s = fma(a[u], yc[quarter + 4 * u], s);
            } else {
                to = __ldg(src + i);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = quarter + 4 * u;
                    if (k < K) s = fma(__ldg(VT + (int64_t)k * R + i), yc[k], s);
                }
            }
        }
        // the four parts of a row sit in four consecutive lanes
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (LEAF) {
            near += __shfl_xor_sync(0xffffffffu, near, 1);
            near += __shfl_xor_sync(0xffffffffu, near, 2);
        }
        if (i < R && quarter == 0) {
            if (LEAF) y[to] = (diag ? fma(diag[to], x[to], near) : near) + s;
            else yhat[to] = s;
        }
    }
}

// deterministic dot product: fixed grid, per-block partial sums, then one
// block adds the partials in order
__global__ void __launch_bounds__(256) k_dot_part(const double *__restrict__ a,
                                                  const double *__restrict__ b, int64_t n,
                                                  double *part)
{
    __shared__ double sh[8];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        acc = fma(a[i], b[i], acc);
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += sh[k];
        part[blockIdx.x] = s;
    }
}

__global__ void k_dot_final(const double *part, int np, double *out)
{
    __shared__ double sh[32];
    double acc = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) acc += part[i];
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += sh[k];
        *out = s;
    }
}

// scal: [0] r.r, [1] p.q, [2] new r.r
__global__ void __launch_bounds__(256) k_cg_step(int64_t n, const double *scal, double *x,
                                                 double *r, const double *p, const double *q)
{
    const double alpha = scal[0] / scal[1];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        x[i] = fma(alpha, p[i], x[i]);
        r[i] = fma(-alpha, q[i], r[i]);
    }
}

__global__ void __launch_bounds__(256) k_cg_dir(int64_t n, double *scal, const double *r, double *p)
{
    const double beta = scal[2] / scal[0];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = fma(beta, p[i], r[i]);
}

__global__ void k_cg_roll(double *scal) { scal[0] = scal[2]; }

cudaError_t matvec(const bem_h2 *h, const double *x, double *y, cudaStream_t st)
{
    const double *no = nullptr;
    const int32_t *noi = nullptr;
    auto warps = [](int64_t n) { return (unsigned)((n + kH2Warps - 1) / kH2Warps); };
    // fork: the chain of levels on the side stream of highest priority, the near
    // field on the caller's stream beside it (its CTAs fill the SMs that the chain's
    // small launches leave idle), joined before the leaves' pass
    cudaError_t e = cudaEventRecord(h->fork, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(h->side, h->fork, 0);
    bool pdl = false;   // the first launch of the chain waits for all earlier work
    for (size_t k = 0; k < h->fwd.size() && e == cudaSuccess; ++k)
        if (h->fwd_n[k] > 0) {
            e = launch_chain(pdl, (unsigned)h->fwd_n[k], 256, h->side, k_h2_forward, h->nodes, h->fwd[k], h->vals,
                          h->src, x, h->xhat);
            pdl = true;
        }
    if (e == cudaSuccess && h->n_near > 0)
        e = launch_chain(false, warps(h->n_near), 256, st, k_h2_blocks<true>, h->near_blk, h->n_near,
                      h->near_vals, h->cl_idx, x, h->near_part);
    if (e == cudaSuccess && h->n_far > 0) {
        e = launch_chain(pdl, warps(h->n_far), 256, h->side, k_h2_blocks<false>, h->far_blk, h->n_far, h->far_vals,
                      noi, h->xhat, h->far_part);
        pdl = true;
    }
    for (size_t k = 0; k + 1 < h->bwd.size() && e == cudaSuccess; ++k)
        if (h->bwd_n[k] > 0) {
            e = launch_chain(pdl, (unsigned)h->bwd_n[k], 256, h->side, k_h2_backward<false>, h->nodes, h->bwd[k],
                          h->valsT, h->src, h->far_part, no, no, no, h->yhat, y);
            pdl = true;
        }
    if (e == cudaSuccess) e = cudaEventRecord(h->join, h->side);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, h->join, 0);
    if (e == cudaSuccess && h->bwd_n.back() > 0)
        e = launch_chain(false, (unsigned)h->bwd_n.back(), 256, st, k_h2_backward<true>, h->nodes, h->bwd.back(),
                      h->valsT, h->src, h->far_part, h->near_part, h->diag, x, h->yhat, y);
    return e;
}

cudaError_t dot(const bem_h2 *h, const double *a, const double *b, double *out, cudaStream_t st)
{
    k_dot_part<<<kDotBlocks, 256, 0, st>>>(a, b, h->n, h->part);
    k_dot_final<<<1, 1024, 0, st>>>(h->part, kDotBlocks, out);
    return cudaGetLastError();
}

template <class T>
cudaError_t h2_upload(bem_h2 *h, T **d, const std::vector<T> &v)
{
    cudaError_t e = cudaMalloc((void **)d, std::max<size_t>(1, v.size()) * sizeof(T));
    if (e != cudaSuccess) return e;
    h->allocs.push_back(*d);
    if (!v.empty()) e = cudaMemcpy(*d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
    return e;
}

template <class T>
cudaError_t h2_alloc(bem_h2 *h, T **d, size_t n)
{
    cudaError_t e = cudaMalloc((void **)d, std::max<size_t>(1, n) * sizeof(T));
    if (e == cudaSuccess) h->allocs.push_back(*d);
    return e;
}

void h2_free(bem_h2 *h)
{
    for (void *a : h->allocs) cudaFree(a);
    if (h->fork) cudaEventDestroy(h->fork);
    if (h->join) cudaEventDestroy(h->join);
    if (h->side) cudaStreamDestroy(h->side);
    delete h;
}

}  // namespace

}  // namespace bem

extern "C" {

int bem_h2_create(bem_ctx *ctx, int64_t n, int32_t n_clusters, const int32_t *cl_ptr,
                  const int32_t *cl_idx, const int32_t *cl_son, const int32_t *piv_ptr,
                  const int32_t *piv_idx, const int64_t *v_off, const double *V, int64_t n_near,
                  const int32_t *near_row, const int32_t *near_col, const int64_t *near_off,
                  const double *near_vals, int64_t n_far, const int32_t *far_row,
                  const int32_t *far_col, const int64_t *far_off, const double *far_vals,
                  const double *diag, bem_h2 **out)
{
    using namespace bem;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!out || n < 1 || n_clusters < 1 || !cl_ptr || !cl_idx || !cl_son || !piv_ptr ||
        !piv_idx || !v_off || !V || n_near < 0 || n_far < 0 ||
        (n_near > 0 && (!near_row || !near_col || !near_off || !near_vals)) ||
        (n_far > 0 && (!far_row || !far_col || !far_off || !far_vals)))
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: bad arguments");
    *out = nullptr;
    const int nc = n_clusters;
    // host checks of the tree, the index sets and the bases' shapes
    if (cl_ptr[0] != 0 || piv_ptr[0] != 0 || v_off[0] != 0)
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: CSR arrays must start at 0");
    std::vector<int> parent(nc, -1), depth(nc, 0);
    for (int c = 0; c < nc; ++c) {
        if (cl_ptr[c + 1] < cl_ptr[c] || piv_ptr[c + 1] < piv_ptr[c] || v_off[c + 1] < v_off[c])
            return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: decreasing CSR pointers");
        if (piv_ptr[c + 1] - piv_ptr[c] > 32)
            return api_fail(ctx, BEM_ERR_UNSUPPORTED, "bem_h2_create: more than 32 pivots in a cluster");
        for (int s = 0; s < 2; ++s) {
            const int x = cl_son[2 * c + s];
            if (x < -1 || x >= nc || x == c || (x >= 0 && parent[x] >= 0))
                return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: bad son");
            if (x >= 0) parent[x] = c;
        }
    }
    for (int64_t k = 0; k < cl_ptr[nc]; ++k)
        if (cl_idx[k] < 0 || cl_idx[k] >= n)
            return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: index out of range");
    int max_depth = 0;
    for (int c = 0; c < nc; ++c) {
        int d = 0, x = c;
        while (parent[x] >= 0) {
            x = parent[x];
            if (++d > nc) return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: cycle");
        }
        depth[c] = d;
        max_depth = std::max(max_depth, d);
    }
    bem_h2 *h = new bem_h2();
    h->n = n;
    h->nc = nc;
    std::vector<int32_t> rows(nc), rank(nc), leaf(nc), src;
    std::vector<int64_t> voff(nc), soff(nc), hoff(nc);
    int64_t hat = 0;
    for (int c = 0; c < nc; ++c) {
        rank[c] = piv_ptr[c + 1] - piv_ptr[c];
        hoff[c] = hat;
        hat += rank[c];
    }
    for (int c = 0; c < nc; ++c) {
        const int s0 = cl_son[2 * c], s1 = cl_son[2 * c + 1];
        leaf[c] = (s0 < 0 && s1 < 0) ? 1 : 0;
        soff[c] = (int64_t)src.size();
        if (leaf[c]) {
            for (int32_t k = cl_ptr[c]; k < cl_ptr[c + 1]; ++k) src.push_back(cl_idx[k]);
        } else {
            for (int s : {s0, s1})
                if (s >= 0)
                    for (int k = 0; k < rank[s]; ++k) src.push_back((int32_t)(hoff[s] + k));
        }
        rows[c] = (int32_t)((int64_t)src.size() - soff[c]);
        voff[c] = v_off[c];
        if (v_off[c + 1] - v_off[c] != (int64_t)rows[c] * rank[c]) {
            h2_free(h);
            return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: basis matrix of the wrong size");
        }
        if (leaf[c] && rows[c] > 32 * 64) {
            h2_free(h);
            return api_fail(ctx, BEM_ERR_UNSUPPORTED, "bem_h2_create: leaf of more than 2048 indices");
        }
    }
    // blocks by row cluster
    auto by_row = [&](int64_t nb, const int32_t *br, const int32_t *bc, const int64_t *bo,
                      std::vector<int32_t> &ptr, std::vector<int32_t> &col,
                      std::vector<int64_t> &off) -> bool {
        ptr.assign(nc + 1, 0);
        for (int64_t b = 0; b < nb; ++b) {
            if (br[b] < 0 || br[b] >= nc || bc[b] < 0 || bc[b] >= nc || bo[b] < 0) return false;
            ptr[br[b] + 1]++;
        }
        for (int c = 0; c < nc; ++c) ptr[c + 1] += ptr[c];
        col.assign(nb, 0);
        off.assign(nb, 0);
        std::vector<int32_t> fill(ptr.begin(), ptr.end() - 1);
        for (int64_t b = 0; b < nb; ++b) {   // block order kept within a row cluster
            col[fill[br[b]]] = bc[b];
            off[fill[br[b]]++] = bo[b];
        }
        return true;
    };
    std::vector<int32_t> nptr, ncol, fptr, fcol;
    std::vector<int64_t> noff, foff;
    if (!by_row(n_near, near_row, near_col, near_off, nptr, ncol, noff) ||
        !by_row(n_far, far_row, far_col, far_off, fptr, fcol, foff)) {
        h2_free(h);
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: bad block list");
    }
    for (int c = 0; c < nc; ++c)
        if (!leaf[c] && nptr[c + 1] > nptr[c]) {
            h2_free(h);
            return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_create: near block on a non-leaf row cluster");
        }
    // clusters that take part: x^_c is used by an admissible block of c's column or of
    // an ancestor's, y^_c gets one of c's row or of an ancestor's
    std::vector<char> has_col(nc, 0), need_f(nc, 0), need_b(nc, 0);
    for (int32_t s : fcol) has_col[s] = 1;
    std::vector<int32_t> order(nc);
    for (int c = 0; c < nc; ++c) order[c] = c;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return depth[a] < depth[b]; });
    for (int c : order) {
        need_f[c] = has_col[c] || (parent[c] >= 0 && need_f[parent[c]]);
        need_b[c] = fptr[c + 1] > fptr[c] || (parent[c] >= 0 && need_b[parent[c]]);
    }
    std::vector<std::vector<int32_t>> fl(max_depth + 2), bl(max_depth + 2);
    std::vector<H2Node> nodes(nc);
    std::vector<H2Block> nblk(n_near), fblk(n_far);
    int64_t np = 0, fp = 0;
    for (int c = 0; c < nc; ++c) {
        H2Node &N = nodes[c];
        N.v_off = voff[c];
        N.src_off = soff[c];
        N.near_off = np;
        N.far_off = fp;
        N.rows = rows[c];
        N.rank = rank[c];
        N.hat = (int32_t)hoff[c];
        N.n_near = nptr[c + 1] - nptr[c];
        N.n_far = fptr[c + 1] - fptr[c];
        N.idx = cl_ptr[c];
        N.leaf = leaf[c];
        N.up = (parent[c] >= 0 && need_b[parent[c]] && rank[parent[c]] > 0 ? 1 : 0) | (need_b[c] ? 2 : 0);
        const int nr = cl_ptr[c + 1] - cl_ptr[c];
        for (int32_t b = nptr[c]; b < nptr[c + 1]; ++b, np += nr)
            nblk[b] = H2Block{noff[b], np, nr, cl_ptr[ncol[b] + 1] - cl_ptr[ncol[b]], cl_ptr[ncol[b]], 0};
        for (int32_t b = fptr[c]; b < fptr[c + 1]; ++b, fp += rank[c])
            fblk[b] = H2Block{foff[b], fp, rank[c], rank[fcol[b]], (int32_t)hoff[fcol[b]], 0};
        if (need_f[c] && rank[c] > 0) fl[leaf[c] ? 0 : 1 + max_depth - depth[c]].push_back(c);
        if (leaf[c]) bl[max_depth + 1].push_back(c);
        else if (need_b[c] && rank[c] > 0) bl[depth[c]].push_back(c);
    }
    cudaSetDevice(ctx->device);
    cudaError_t e = cudaSuccess;
    std::vector<int32_t> ci(cl_idx, cl_idx + cl_ptr[nc]);
    std::vector<double> vals(V, V + v_off[nc]), valsT(vals.size());
    for (int c = 0; c < nc; ++c)
        for (int i = 0; i < rows[c]; ++i)
            for (int k = 0; k < rank[c]; ++k)
                valsT[voff[c] + (int64_t)k * rows[c] + i] = vals[voff[c] + (int64_t)i * rank[c] + k];
    int low = 0, high = 0;
    if ((e = h2_upload(h, &h->nodes, nodes)) || (e = h2_upload(h, &h->src, src)) ||
        (e = h2_upload(h, &h->vals, vals)) || (e = h2_upload(h, &h->valsT, valsT)) ||
        (e = cudaDeviceGetStreamPriorityRange(&low, &high)) ||
        (e = cudaStreamCreateWithPriority(&h->side, cudaStreamNonBlocking, high)) ||
        (e = cudaEventCreateWithFlags(&h->fork, cudaEventDisableTiming)) ||
        (e = cudaEventCreateWithFlags(&h->join, cudaEventDisableTiming)) ||
        (e = h2_upload(h, &h->near_blk, nblk)) || (e = h2_upload(h, &h->far_blk, fblk)) ||
        (e = h2_upload(h, &h->cl_idx, ci)) || (e = h2_alloc(h, &h->near_part, np)) ||
        (e = h2_alloc(h, &h->far_part, fp)) || (e = h2_alloc(h, &h->xhat, hat)) ||
        (e = h2_alloc(h, &h->yhat, hat)) || (e = h2_alloc(h, &h->r, n)) ||
        (e = h2_alloc(h, &h->p, n)) || (e = h2_alloc(h, &h->q, n)) ||
        (e = h2_alloc(h, &h->part, kDotBlocks)) || (e = h2_alloc(h, &h->scal, 4))) {
        h2_free(h);
        return api_cuda_fail(ctx, e, "bem_h2_create");
    }
    if (diag) {
        std::vector<double> dg(diag, diag + n);
        if ((e = h2_upload(h, &h->diag, dg)) != cudaSuccess) {
            h2_free(h);
            return api_cuda_fail(ctx, e, "bem_h2_create");
        }
    }
    for (int pass = 0; pass < 2; ++pass)
        for (auto &l : pass ? bl : fl) {
            int32_t *d = nullptr;
            if ((e = h2_upload(h, &d, l)) != cudaSuccess) {
                h2_free(h);
                return api_cuda_fail(ctx, e, "bem_h2_create");
            }
            (pass ? h->bwd : h->fwd).push_back(d);
            (pass ? h->bwd_n : h->fwd_n).push_back((int32_t)l.size());
        }
    h->n_near = n_near;
    h->n_far = n_far;
    h->n_hat = hat;
    h->near_vals = near_vals;
    h->far_vals = far_vals;
    *out = h;
    return BEM_OK;
}

int bem_h2_matvec(bem_ctx *ctx, bem_h2 *h, const double *x, double *y)
{
    using namespace bem;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!h || !x || !y || x == y) return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_matvec: bad arguments");
    cudaError_t e = matvec(h, x, y, ctx->stream);
    if (e != cudaSuccess) return api_cuda_fail(ctx, e, "bem_h2_matvec");
    return BEM_OK;
}

int bem_h2_cg(bem_ctx *ctx, bem_h2 *h, const double *b, double *x, double tol, int32_t maxit,
              int32_t *iters, double *rel_res)
{
    using namespace bem;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!h || !b || !x || b == x || !(tol > 0.0) || maxit < 0 || !iters || !rel_res)
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_h2_cg: bad arguments");
    cudaStream_t st = ctx->stream;
    const size_t bytes = (size_t)h->n * sizeof(double);
    // x0 = 0, r = p = b, r.r and b.b
    cudaError_t e = cudaMemsetAsync(x, 0, bytes, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h->r, b, bytes, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h->p, b, bytes, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = dot(h, h->r, h->r, h->scal + 0, st);
    double rr = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&rr, h->scal + 0, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return api_cuda_fail(ctx, e, "bem_h2_cg");
    const double bb = rr;
    const unsigned grid = (unsigned)std::min<int64_t>((h->n + 255) / 256, 4 * 1024);
    int it = 0;
    while (it < maxit && rr > tol * tol * bb && bb > 0.0) {
        e = matvec(h, h->p, h->q, st);                          // q = A p
        if (e == cudaSuccess) e = dot(h, h->p, h->q, h->scal + 1, st);
        if (e == cudaSuccess) {
            k_cg_step<<<grid, 256, 0, st>>>(h->n, h->scal, x, h->r, h->p, h->q);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = dot(h, h->r, h->r, h->scal + 2, st);
        if (e == cudaSuccess) {
            k_cg_dir<<<grid, 256, 0, st>>>(h->n, h->scal, h->r, h->p);
            k_cg_roll<<<1, 1, 0, st>>>(h->scal);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&rr, h->scal + 0, sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return api_cuda_fail(ctx, e, "bem_h2_cg");
        if (!std::isfinite(rr)) return api_fail(ctx, BEM_ERR_DEGENERATE, "bem_h2_cg: breakdown");
        ++it;
    }
    *iters = it;
    *rel_res = bb > 0.0 ? std::sqrt(rr / bb) : 0.0;
    return BEM_OK;
}

int bem_h2_destroy(bem_ctx *ctx, bem_h2 *h)
{
    if (!ctx || !h) return BEM_ERR_INVALID_ARG;
    cudaStreamSynchronize(ctx->stream);
    bem::h2_free(h);
    return BEM_OK;
}

}  // extern "C"
