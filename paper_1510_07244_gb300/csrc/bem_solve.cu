// Potentials and a dense complex GMRES solve: the exterior Helmholtz problem
// of Section 4 (Brakhage-Werner formulation) end to end on the device.
//
//   bem_potentials     u(z_k) = sum_j w_j int_{T_j} k(z_k, y) dy for points z_k
//                      off the surface (piecewise-constant density w), with the
//                      library's kernels; one thread per (point, triangle) in the
//                      FP64 form's fixed-point arithmetic, a Duffy q x q rule per
//                      triangle, a cluster of CTAs per point, their sums added in order.
//   bem_dense_gmres    restarted GMRES (Saad and Schultz) for a dense complex
//                      system (A + diag(d)) x = b: Arnoldi with classical
//                      Gram-Schmidt applied twice, Givens rotations on the host.
//                      The matrix-vector product (column-major A, 32-row tiles
//                      times column ranges) and both projections run in a chain of
//                      overlapping launches; each Arnoldi step reads its projection
//                      coefficients and the new vector's norm back once (a few
//                      hundred bytes), beside the next step's product.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "bem_device.cuh"

namespace bem {

namespace {

// FP64 arithmetic for a triangle too close to the point for the fixed-point range
template <int KIND>
__device__ __noinline__ void potential_double(const double *z, const Tri &B, const Rule2D &R,
                                              double kappa, double eta, double &sr, double &si)
{
    sr = si = 0.0;
#pragma unroll 1
    for (int k = 0; k < R.np; ++k) {
        double d[3], kr, ki;
#pragma unroll
        for (int c = 0; c < 3; ++c)
            d[c] = z[c] - (B.v[0][c] + R.s[k] * (B.v[1][c] - B.v[0][c]) + R.t[k] * (B.v[2][c] - B.v[1][c]));
        kval<KIND>(d[0], d[1], d[2], B.n, kappa, kr, ki, eta);
        sr += R.w[k] * kr;
        si += R.w[k] * ki;
    }
}

// int_T k(z, y) dy without sqrt(g) / (4 pi): the trial side of a regular pair
// (bem_fixed_pair.cuh) for one test point
template <int KIND>
__device__ __forceinline__ bool potential_fixed(const double *z, const Tri &B, const Rule2D &R,
                                                double kappa, double eta, double &sr, double &si)
{
    // the vertices relative to z, whose roundings are independent (a common one of z
    // relative to a vertex would not average out over the points)
    double y[3][3], h = 0.0;
    int top = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            y[k][c] = B.v[k][c] - z[c];
            top = max(top, fx_mag(y[k][c]));
        }
        h = fma(-y[0][c], B.n[c], h);
    }
    const int e = top >> 20;
    if (e < 823 || e > 1223) return false;
    FxPair P;
    P.E = e - 1022;
    const double sc = fx_pow2(61 - P.E);
    s64 Y0[3];
    float d2 = 0.0f, rb = 0.0f, cb[3], yf[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        Y0[c] = __double2ll_rn(y[0][c] * sc);
        const s64 y1 = __double2ll_rn(y[1][c] * sc), y2 = __double2ll_rn(y[2][c] * sc);
        P.b1[c] = fx_split(y1 - Y0[c]);
        P.b2[c] = fx_split(y2 - y1);
        yf[0][c] = fx_hi(Y0[c]);   // S = 2^29
        yf[1][c] = fx_hi(y1);
        yf[2][c] = fx_hi(y2);
        cb[c] = (yf[0][c] + yf[1][c] + yf[2][c]) * (1.0f / 3.0f);
        d2 = fmaf(cb[c], cb[c], d2);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float v = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) v = fmaf(yf[k][c] - cb[c], yf[k][c] - cb[c], v);
        rb = fmaxf(rb, v);
    }
    P.kb = KIND == BEM_LAPLACE_SLP ? 4 : fx_kb((sqrtf(d2) - sqrtf(rb)) * 0.99999f - 8.0f);
    if (kind_has_height(KIND) && P.kb >= 3) {
        // from the rule's points (fx_near_kb): the bound of a point beside a triangle has
        // no digits left (8000 points, Brakhage-Werner kernel, root mean square error over
        // the sum of the terms' magnitudes 1.9e-15, so 3.2e-16; FP64 arithmetic 2.9e-16)
        float lo = 3.0e38f;
#pragma unroll 1
        for (int k = 0; k < R.np; ++k) {
            d2 = 0.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float d = fmaf(R.sf[k], yf[1][c] - yf[0][c], fmaf(R.tf[k], yf[2][c] - yf[1][c], yf[0][c]));
                d2 = fmaf(d, d, d2);
            }
            lo = fminf(lo, d2);
        }
        P.kb = fx_kb(sqrtf(lo) * 0.9999f - 32.0f);
    }
    FxUnits U;
    if (!fx_units<KIND>(P, P.kb, kappa, eta, U)) return false;
    // the sums (half of the weighted ones, whose weights add to a half) stay below 2^57;
    // four of their fraction's bits count here, where no outer sum averages the rounding
    constexpr int UP = 4;
    FxInner<KIND, 1> I;
    I.template clear<0, 0, UP>();
    int flag = 0;
#pragma unroll 1
    for (int k = 0; k < R.np; ++k) {
        s64 d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = (Y0[c] << 1) + fx_point(0, P.b1[c], P.b2[c], R.sx[k], R.tx[k]);
        const int32_t *w[1] = {R.wx[3][k]};
        I.point(d[0], d[1], d[2], P.kb, U.kn, U.shl, w, flag);
    }
    fx_combine<KIND, 1, UP>(I, 0, U, h * fx_pow2(-P.E), sr, si);
    const double f = fx_final<KIND>(U) * fx_pow2(-UP);
    sr *= f;
    si *= f;
    return (flag >> (16 + P.kb)) == 0;
}

// Cluster p: point p0 + p; its CTA s takes the triangles [s per, (s + 1) per), and
// the first CTA adds the sums in order through distributed shared memory: no scratch,
// so the call stays asynchronous and a captured one holds no pointer of the library's.
// A point's triangles spread over several CTAs where the points alone would not fill
// the GPU (256 points, 2048 triangles, Duffy q = 4, Brakhage-Werner kernel: one warp
// per point in FP64 arithmetic took 9.4 ms; 0.21 ms so, 0.09 for 64 points).
constexpr int kPotThreads = 256, kPotCluster = 16;   // at most; beyond 8 CTAs by opt-in

template <int KIND>
__global__ void __launch_bounds__(kPotThreads) k_potentials(MeshView m, const double *__restrict__ z,
                                                            int64_t p0, int64_t per,
                                                            const double2 *__restrict__ w,
                                                            const __grid_constant__ Rule2D R,
                                                            double kappa, double eta, double2 *out)
{
    __shared__ double2 ws[kPotThreads / 32], sum;
    const int64_t p = p0 + blockIdx.y;
    const int64_t j0 = (int64_t)blockIdx.x * per, j1 = min(m.nt, j0 + per);
    const double zp[3] = {z[3 * p], z[3 * p + 1], z[3 * p + 2]};
    double ar = 0.0, ai = 0.0;
    for (int64_t j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
        Tri B;
        load_tri(m.geom, j, B);
        double sr, si;
        if (!potential_fixed<KIND>(zp, B, R, kappa, eta, sr, si))
            potential_double<KIND>(zp, B, R, kappa, eta, sr, si);
        const double2 wj = w[j];
        const double sc = B.sg * kInv4Pi;
        sr *= sc;
        si *= sc;
        ar += wj.x * sr - wj.y * si;
        ai += wj.x * si + wj.y * sr;
    }
    ar = warp_sum(ar);
    ai = warp_sum(ai);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = make_double2(ar, ai);
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 s = ws[0];
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            s.x += ws[k].x;
            s.y += ws[k].y;
        }
        sum = s;
    }
    auto cluster = cooperative_groups::this_cluster();
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double2 s = sum;
        for (unsigned k = 1; k < cluster.num_blocks(); ++k) {
            const double2 v = *cluster.map_shared_rank(&sum, k);
            s.x += v.x;
            s.y += v.y;
        }
        out[p] = s;
    }
    cluster.sync();   // the CTAs' sums stay until the first has read them
}

// The kernels of one Arnoldi step run as a chain of dependent launches
// (bem_pdl.cuh); with the kernels below 111 -> 57 us per step (n = 2048, 36 steps).

// Partial products of y = A x, A column-major n x n complex: CTA (r, s) takes the
// 32 rows of tile r and the columns [s per, (s + 1) per), one row per lane, every
// 8th column per warp; the warps' sums are added in order into part[s n + row].
// FP64-bound (four FMAs per 16-byte entry, 2 lanes per SM and cycle: 29 us for
// n = 2048).  About eight CTAs per SM, so that the last ones leave little idle (two
// per SM: 44 us, eight: 37).
__global__ void __launch_bounds__(256) k_zgemv_part(int64_t n, int64_t per, unsigned tiles,
                                                    const double2 *__restrict__ A,
                                                    const double2 *x, double2 *part)
{
    __shared__ double2 ws[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r = blockIdx.x % tiles, s = blockIdx.x / tiles, i = r * 32 + lane;
    const int64_t j0 = s * per, j1 = min(n, j0 + per);
    pdl_wait();
    pdl_launch();
    double ar = 0.0, ai = 0.0;
    if (i < n) {
#pragma unroll 8
        for (int64_t j = j0 + warp; j < j1; j += 8) {
            const double2 a = __ldg(A + i + j * n), v = x[j];
            ar = fma(a.x, v.x, fma(-a.y, v.y, ar));
            ai = fma(a.x, v.y, fma(a.y, v.x, ai));
        }
    }
    ws[warp][lane] = make_double2(ar, ai);
    __syncthreads();
    if (warp == 0 && i < n) {
        double2 s2 = ws[0][lane];
#pragma unroll
        for (int k = 1; k < 8; ++k) {
            s2.x += ws[k][lane].x;
            s2.y += ws[k][lane].y;
        }
        part[s * n + i] = s2;
    }
}

// Sum over 8 warps of the lanes' values, in warp order (warp 0 has the result)
__device__ __forceinline__ double2 sum_warps(double2 v, double2 (*ws)[32])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ws[warp][lane] = v;
    __syncthreads();
    double2 s = ws[0][lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) {
        s.x += ws[k][lane].x;
        s.y += ws[k][lane].y;
    }
    return s;
}

// y = sum of the ns partial products + diag(d) x: 32 rows per CTA, every 8th
// partial product per warp
__global__ void __launch_bounds__(256) k_zgemv_sum(int64_t n, int ns, const double2 *part,
                                                   const double2 *__restrict__ d, const double2 *x,
                                                   double2 *y)
{
    __shared__ double2 ws[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    pdl_wait();
    pdl_launch();
    double2 v = make_double2(0.0, 0.0);
    if (i < n) {
#pragma unroll 4
        for (int s = warp; s < ns; s += 8) {
            const double2 a = part[(int64_t)s * n + i];
            v.x += a.x;
            v.y += a.y;
        }
    }
    v = sum_warps(v, ws);
    if (warp > 0 || i >= n) return;
    if (d) {
        const double2 a = d[i], u = x[i];
        v.x += a.x * u.x - a.y * u.y;
        v.y += a.x * u.y + a.y * u.x;
    }
    y[i] = v;
}

// h_k = <V_k, w> = sum_i conj(V[i, k]) w_i for k < kk (V column-major n x ld):
// one block per k, fixed reduction order (lanes, then warps)
__global__ void __launch_bounds__(256) k_project(int64_t n, const double2 *V, const double2 *w, double2 *h)
{
    __shared__ double2 ws[8];
    const int k = blockIdx.x;
    const double2 *v = V + (int64_t)k * n;
    pdl_wait();
    pdl_launch();
    double ar = 0.0, ai = 0.0;
#pragma unroll 8
    for (int64_t i = threadIdx.x; i < n; i += 256) {
        const double2 a = v[i], b = w[i];
        ar = fma(a.x, b.x, fma(a.y, b.y, ar));
        ai = fma(a.x, b.y, fma(-a.y, b.x, ai));
    }
    ar = warp_sum(ar);
    ai = warp_sum(ai);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = make_double2(ar, ai);
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 s = ws[0];
#pragma unroll
        for (int u = 1; u < 8; ++u) {
            s.x += ws[u].x;
            s.y += ws[u].y;
        }
        h[k] = s;
    }
}

// w -= V h (the first kk columns): 32 rows per CTA, every 8th column per warp (one
// thread per row ran a chain of kk loads and products: 18 us at kk = 36, n = 2048).
// sq: also the CTA's part of |w|^2.
__global__ void __launch_bounds__(256) k_subtract(int64_t n, int kk, const double2 *V, const double2 *h,
                                                  double2 *w, double *sq)
{
    __shared__ double2 ws[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    pdl_wait();
    pdl_launch();
    double2 v = make_double2(0.0, 0.0);
    if (i < n) {
#pragma unroll 4
        for (int k = warp; k < kk; k += 8) {
            const double2 a = V[i + (int64_t)k * n], b = h[k];
            v.x = fma(a.x, b.x, fma(-a.y, b.y, v.x));
            v.y = fma(a.x, b.y, fma(a.y, b.x, v.y));
        }
    }
    v = sum_warps(v, ws);
    if (warp > 0) return;
    double q = 0.0;
    if (i < n) {
        const double2 a = w[i];
        v = make_double2(a.x - v.x, a.y - v.y);
        w[i] = v;
        q = v.x * v.x + v.y * v.y;
    }
    if (sq) {
        q = warp_sum(q);
        if (lane == 0) sq[blockIdx.x] = q;
    }
}

// w = b - w
__global__ void __launch_bounds__(256) k_residual(int64_t n, const double2 *__restrict__ b, double2 *w)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    w[i] = make_double2(b[i].x - w[i].x, b[i].y - w[i].y);
}

// v = s w (complex scale)
__global__ void __launch_bounds__(256) k_scale(int64_t n, double sr, double si,
                                               const double2 *__restrict__ w, double2 *v)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 a = w[i];
    v[i] = make_double2(sr * a.x - si * a.y, sr * a.y + si * a.x);
}

// v = w / |w|, |w|^2 = the sum of the np parts in sq, also left in norm2 (real
// part); nothing for a zero vector
__global__ void __launch_bounds__(256) k_normalise(int64_t n, int np, const double *sq, double2 *norm2,
                                                   const double2 *w, double2 *v)
{
    __shared__ double ws[8];
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    pdl_wait();
    pdl_launch();
    double q = 0.0;
#pragma unroll 4
    for (int k = threadIdx.x; k < np; k += 256) q += sq[k];
    const double2 a = i < n ? w[i] : make_double2(0.0, 0.0);
    q = warp_sum(q);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = q;
    __syncthreads();
    q = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) q += ws[k];
    if (i == 0) *norm2 = make_double2(q, 0.0);
    const double s = sqrt(fmax(q, 0.0));
    if (i >= n || !(s > 0.0)) return;
    const double f = 1.0 / s;
    v[i] = make_double2(f * a.x, f * a.y);
}

// x += V y (the first kk columns)
__global__ void __launch_bounds__(256) k_update(int64_t n, int kk, const double2 *__restrict__ V,
                                                const double2 *__restrict__ y, double2 *x)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double ar = x[i].x, ai = x[i].y;
    for (int k = 0; k < kk; ++k) {
        const double2 a = V[i + (int64_t)k * n], b = y[k];
        ar += a.x * b.x - a.y * b.y;
        ai += a.x * b.y + a.y * b.x;
    }
    x[i] = make_double2(ar, ai);
}

// Scratch kept from one solve for the next: 100 vectors of 40000 unknowns.  A larger one's
// allocation (about 1 ms) is little beside its products.
constexpr size_t kSolveKeep = (size_t)64 << 20;

unsigned grid_of(int64_t n) { return (unsigned)((n + 255) / 256); }

}  // namespace

}  // namespace bem

extern "C" {

int bem_potentials(bem_ctx *ctx, int32_t mesh_id, const bem_kernel_desc *kernel, int32_t q,
                   const double *points, int64_t n_points, const double *density, double *out)
{
    using namespace bem;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    auto it = ctx->meshes.find(mesh_id);
    if (it == ctx->meshes.end()) return api_fail(ctx, BEM_ERR_INVALID_ARG, "unknown mesh id");
    const MeshView &m = it->second->v;
    if (m.basis != BEM_P0)
        return api_fail(ctx, BEM_ERR_UNSUPPORTED, "bem_potentials: piecewise-constant densities");
    if (!kernel || kernel->kind < BEM_LAPLACE_SLP || kernel->kind > BEM_HELMHOLTZ_BW ||
        !std::isfinite(kernel->kappa) || !std::isfinite(kernel->eta) || q < 1 || q > 5 ||
        n_points < 0)
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_potentials: bad arguments");
    if (n_points == 0) return BEM_OK;
    if (!points || !density || !out ||
        (reinterpret_cast<uintptr_t>(density) & 15) || (reinterpret_cast<uintptr_t>(out) & 15))
        return api_fail(ctx, BEM_ERR_INVALID_ARG,
                        "bem_potentials: null or misaligned pointer (complex arrays: 16 bytes)");
    Rule2D r2;
    if (!make_rule2d(BEM_RULE_DUFFY, q, r2)) return api_fail(ctx, BEM_ERR_INVALID_ARG, "bad order");
    const double2 *w = reinterpret_cast<const double2 *>(density);
    double2 *o = reinterpret_cast<double2 *>(out);
    const double ka = kernel->kappa, et = kernel->eta;
    cudaStream_t st = ctx->stream;
    // CTAs per point: a power of two that gives about 32 warps per SM in all, with 128
    // triangles or more each; CTAs of twice the warps where 16 of 4 warps a point leave
    // half of that empty and have the triangles
    const int64_t need = 32 * (int64_t)ctx->num_sms;
    const int threads = n_points * kPotCluster * 8 < need && m.nt > kPotCluster * 128 ? kPotThreads : 128;
    int ns = 1;
    while (ns < kPotCluster && ns * 128 < m.nt && n_points * ns * (threads / 32) < need) ns *= 2;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ns;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.blockDim = dim3((unsigned)threads);
    c.stream = st;
    c.attrs = at;
    c.numAttrs = 1;
    if (ns > 8) {
        // eight CTAs run everywhere, more where the device (or the part of it that is
        // this process') has room for such a cluster
        if (ctx->pot_cluster == 0) {
            auto k = k_potentials<BEM_HELMHOLTZ_BW>;
            cudaLaunchConfig_t q = c;
            q.gridDim = dim3((unsigned)ns);
            q.blockDim = dim3(kPotThreads);
            int room = 0;
            if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&room, k, &q) != cudaSuccess)
                cudaGetLastError();
            ctx->pot_cluster = room > 0 ? kPotCluster : 8;
        }
        ns = std::min(ns, ctx->pot_cluster);
        at[0].val.clusterDim.x = (unsigned)ns;
    }
    const int64_t per = (m.nt + ns - 1) / ns;
    cudaError_t e = cudaSuccess;
    constexpr int64_t kRows = 65535;   // grid limit
    for (int64_t p0 = 0; p0 < n_points && e == cudaSuccess; p0 += kRows) {
        c.gridDim = dim3((unsigned)ns, (unsigned)std::min(kRows, n_points - p0));
        auto run = [&](auto k) {
            cudaError_t ee = ns > 8 ? cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)
                                    : cudaSuccess;
            return ee == cudaSuccess ? cudaLaunchKernelEx(&c, k, m, points, p0, per, w, r2, ka, et, o) : ee;
        };
        switch (kernel->kind) {
        case BEM_LAPLACE_SLP: e = run(k_potentials<BEM_LAPLACE_SLP>); break;
        case BEM_LAPLACE_DLP: e = run(k_potentials<BEM_LAPLACE_DLP>); break;
        case BEM_HELMHOLTZ_SLP: e = run(k_potentials<BEM_HELMHOLTZ_SLP>); break;
        case BEM_HELMHOLTZ_DLP: e = run(k_potentials<BEM_HELMHOLTZ_DLP>); break;
        default: e = run(k_potentials<BEM_HELMHOLTZ_BW>); break;
        }
    }
    if (e != cudaSuccess) return api_cuda_fail(ctx, e, "bem_potentials");
    return BEM_OK;
}

int bem_dense_gmres(bem_ctx *ctx, int64_t n, const double *A, const double *diag,
                    const double *b, double *x, double tol, int32_t restart, int32_t maxit,
                    int32_t *iters, double *rel_res)
{
    using namespace bem;
    using cplx = std::complex<double>;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (n < 1 || !A || !b || !x || b == x || !(tol > 0.0) || restart < 1 || restart > 500 ||
        maxit < 0 || !iters || !rel_res)
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_dense_gmres: bad arguments");
    for (const double *p : {A, diag, b, (const double *)x})
        if (p && (reinterpret_cast<uintptr_t>(p) & 15))
            return api_fail(ctx, BEM_ERR_INVALID_ARG, "bem_dense_gmres: complex arrays must be 16-byte aligned");
    cudaStream_t st = ctx->stream;
    const double2 *dA = reinterpret_cast<const double2 *>(A);
    const double2 *dd = reinterpret_cast<const double2 *>(diag);
    const double2 *db = reinterpret_cast<const double2 *>(b);
    double2 *dx = reinterpret_cast<double2 *>(x);
    const int m = restart;
    // column ranges of the product: about eight CTAs per SM, at least 64 columns each
    const unsigned tiles = (unsigned)((n + 31) / 32);
    int64_t ns = std::max<int64_t>(1, std::min<int64_t>((8 * ctx->num_sms + tiles / 2) / tiles, n / 64));
    const int64_t per = (n + ns - 1) / ns;
    ns = (n + per - 1) / per;
    // scratch: V (restart + 1 vectors), w, the partial products, the projection
    // coefficients of one step (both passes, then the squared norm), parts of the norm
    const size_t nh = 2 * (size_t)(m + 1) + 1;
    int rc = api_ensure_scratch(ctx, sizeof(double2) * ((size_t)n * (m + 2 + ns) + nh + tiles));
    if (rc) return rc;
    if (!ctx->solve_host &&
        (cudaMallocHost((void **)&ctx->solve_host, sizeof(double2) * (2 * 501 + 1)) != cudaSuccess ||
         cudaEventCreateWithFlags(&ctx->solve_read, cudaEventDisableTiming) != cudaSuccess)) {
        cudaFreeHost(ctx->solve_host);
        ctx->solve_host = nullptr;
        return api_cuda_fail(ctx, cudaGetLastError(), "bem_dense_gmres");
    }
    const double2 *hh = reinterpret_cast<const double2 *>(ctx->solve_host);
    double2 *V = reinterpret_cast<double2 *>(ctx->scratch), *w = V + (size_t)n * (m + 1);
    double2 *part = w + n, *h = part + (size_t)n * ns;
    double *sq = reinterpret_cast<double *>(h + nh);
    cudaError_t e = cudaSuccess;
    auto done = [&](int code) {
        cudaStreamSynchronize(st);
        if (ctx->scratch_cap > kSolveKeep) {
            cudaFree(ctx->scratch);
            ctx->scratch = nullptr;
            ctx->scratch_cap = 0;
        }
        return code;
    };
    const unsigned g = grid_of(n);
    auto product = [&](const double2 *v, double2 *y) -> cudaError_t {
        cudaError_t ee = launch_chain(false, (unsigned)(tiles * ns), 256, st, k_zgemv_part, n, per, tiles,
                                      dA, v, part);
        if (ee != cudaSuccess) return ee;
        return launch_chain(true, tiles, 256, st, k_zgemv_sum, n, (int)ns, (const double2 *)part, dd, v, y);
    };
    // |b|
    auto norm = [&](const double2 *v, double &out) -> cudaError_t {
        k_project<<<1, 256, 0, st>>>(n, v, v, h);
        double2 r;
        cudaError_t ee = cudaMemcpyAsync(&r, h, sizeof(r), cudaMemcpyDeviceToHost, st);
        if (ee == cudaSuccess) ee = cudaStreamSynchronize(st);
        out = std::sqrt(std::max(r.x, 0.0));
        return ee;
    };
    double bn = 0.0;
    e = cudaMemsetAsync(dx, 0, sizeof(double2) * (size_t)n, st);
    if (e == cudaSuccess) e = norm(db, bn);
    if (e != cudaSuccess) return done(api_cuda_fail(ctx, e, "bem_dense_gmres"));
    int it = 0;
    double res = bn > 0.0 ? 1.0 : 0.0;
    std::vector<cplx> H((size_t)(m + 1) * m), cs(m), sn(m), gvec(m + 1), hk(m + 2);
    while (it < maxit && res > tol && bn > 0.0) {
        // r = b - (A + D) x (into w), beta = |r|, V_0 = r / beta
        e = product(dx, w);
        if (e != cudaSuccess) return done(api_cuda_fail(ctx, e, "bem_dense_gmres"));
        k_residual<<<g, 256, 0, st>>>(n, db, w);
        double beta = 0.0;
        e = norm(w, beta);
        if (e != cudaSuccess) return done(api_cuda_fail(ctx, e, "bem_dense_gmres"));
        res = beta / bn;
        if (res <= tol) break;
        k_scale<<<g, 256, 0, st>>>(n, 1.0 / beta, 0.0, w, V);
        std::fill(gvec.begin(), gvec.end(), cplx(0.0));
        gvec[0] = beta;
        int k = 0;
        e = product(V, w);
        for (; k < m && it < maxit; ++k, ++it) {
            // classical Gram-Schmidt, twice, the norm of what is left and the next
            // vector; the coefficients and the norm come back in one copy
            const int kk = k + 1;
            for (int pass = 0; pass < 2 && e == cudaSuccess; ++pass) {
                double2 *hp = h + pass * kk;
                e = launch_chain(true, (unsigned)kk, 256, st, k_project, n, (const double2 *)V,
                                 (const double2 *)w, hp);
                if (e == cudaSuccess)
                    e = launch_chain(true, tiles, 256, st, k_subtract, n, kk, (const double2 *)V,
                                     (const double2 *)hp, w, pass ? sq : (double *)nullptr);
            }
            if (e == cudaSuccess)
                e = launch_chain(true, g, 256, st, k_normalise, n, (int)tiles, (const double *)sq, h + 2 * kk,
                                 (const double2 *)w, V + (size_t)kk * n);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(ctx->solve_host, h, sizeof(double2) * (size_t)(2 * kk + 1),
                                    cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaEventRecord(ctx->solve_read, st);
            // the next step's product runs while the host reads this step's
            // coefficients (after the last step it is not used)
            if (e == cudaSuccess && kk < m && it + 1 < maxit) e = product(V + (size_t)kk * n, w);
            if (e == cudaSuccess) e = cudaEventSynchronize(ctx->solve_read);
            if (e != cudaSuccess) return done(api_cuda_fail(ctx, e, "bem_dense_gmres"));
            for (int i = 0; i <= k; ++i) {
                hk[i] = cplx(hh[i].x, hh[i].y);
                hk[i] += cplx(hh[k + 1 + i].x, hh[k + 1 + i].y);
            }
            const double hn = std::sqrt(std::max(hh[2 * (k + 1)].x, 0.0));
            hk[k + 1] = hn;
            // apply the previous rotations, then a new one that zeroes hk[k + 1]
            for (int i = 0; i < k; ++i) {
                const cplx t = std::conj(cs[i]) * hk[i] + std::conj(sn[i]) * hk[i + 1];
                hk[i + 1] = -sn[i] * hk[i] + cs[i] * hk[i + 1];
                hk[i] = t;
            }
            const double a = std::abs(hk[k]), bb = std::abs(hk[k + 1]);
            const double r = std::hypot(a, bb);
            if (r == 0.0) {
                cs[k] = 1.0;
                sn[k] = 0.0;
            } else {
                cs[k] = hk[k] / r;
                sn[k] = hk[k + 1] / r;
            }
            hk[k] = r;
            hk[k + 1] = 0.0;
            gvec[k + 1] = -sn[k] * gvec[k];
            gvec[k] = std::conj(cs[k]) * gvec[k];
            for (int i = 0; i <= k; ++i) H[(size_t)i * m + k] = hk[i];
            res = std::abs(gvec[k + 1]) / bn;
            if (res <= tol || hn == 0.0) {
                ++k;
                ++it;
                break;
            }
        }
        // y = H^-1 g (upper triangular k x k), x += V y
        std::vector<cplx> y(k);
        for (int i = k - 1; i >= 0; --i) {
            cplx s = gvec[i];
            for (int j = i + 1; j < k; ++j) s -= H[(size_t)i * m + j] * y[j];
            y[i] = s / H[(size_t)i * m + i];
        }
        std::vector<double2> yd(k);
        for (int i = 0; i < k; ++i) yd[i] = make_double2(y[i].real(), y[i].imag());
        e = cudaMemcpyAsync(h, yd.data(), sizeof(double2) * (size_t)k, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) {
            k_update<<<g, 256, 0, st>>>(n, k, V, h, dx);
            e = cudaStreamSynchronize(st);   // h is reused by the next cycle
        }
        if (e != cudaSuccess) return done(api_cuda_fail(ctx, e, "bem_dense_gmres"));
    }
    *iters = it;
    *rel_res = res;
    return done(BEM_OK);
}

}  // extern "C"
