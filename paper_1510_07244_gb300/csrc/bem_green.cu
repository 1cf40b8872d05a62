// Green quadrature matrices of the GCA (Section 2.3) on the device.
//
// For a cluster t, Green's representation formula on an auxiliary domain
// omega_t that encloses the supports of the cluster's basis functions,
// discretised by a quadrature rule (z_nu, w_nu) on the boundary of omega_t,
// turns the far field of every basis function phi_i of t into the rows of
//   A_t+[i, nu] = sp_nu int phi_i(x) g(x, z_nu) dx
//   A_t-[i, nu] = sm_nu int phi_i(x) d/dn(z_nu) g(x, z_nu) dx
// (the GCA takes sp = sqrt(w_nu) and sm = sqrt(w_nu) delta_t).  Cross
// approximation on these matrices picks the pivots of the H^2 coupling
// blocks.  The paper assembles them on the CPU, where they cost about as much
// as its whole GPU phase; here they are one launch for a list of clusters.
//
// g(x, z) = exp(i kappa r) / (4 pi r), r = |x - z| (kappa = 0 for the Laplace
// kernels), and the normal derivative is taken in z along the unit normal n:
//   n . grad_z g = (x - z).n (1 - i kappa r) exp(i kappa r) / (4 pi r^3).
// Every support triangle is integrated by a 2D rule on the reference triangle
// D = {0 <= t <= s <= 1} with the affine map Phi(s,t) = v0 + s (v1 - v0) +
// t (v2 - v1) and Gram factor sqrt(g) (Section 2.2), in FP64.
//
// Work split: a few CTAs per cluster; their warps take units of one row (basis
// function) and 32 of the cluster's points, one per lane.  The lanes of a warp
// walk the same support triangles and rule points, so the support loop of the
// piecewise-linear basis does not diverge and a triangle's rule points are
// computed by the lanes together; the lanes differ only in z_nu.  The plus and
// minus entries share the distance and its reciprocal square root.
//
// Arithmetic: the fixed point of bem_fixed.cuh in one frame per cluster (origin
// at the middle of its rows' and points' box, S = 2^E above every coordinate
// difference).  In FP64 a point took 25 operations on a pipe of 2 lanes per SM and
// cycle (62% of its peak); triangles nearer than S / 16 to a point still do.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "bem_device.cuh"

namespace bem {
namespace {

constexpr int kGreenThreads = 128;

struct GreenArgs {
    const int32_t *row_ptr, *row_idx, *pt_ptr;
    const double *z, *nz, *sp, *sm;
    const int64_t *out_off;
    void *out;
    int64_t n_row_idx, n_points, out_len;
    double kappa;
};

// Sums over one support triangle T of the rule points' contributions for the
// point z with normal n (Section 2.3), without sqrt(g) and 1/(4 pi), FP64:
//   plus  += w_q phi(s_q, t_q) exp(i kappa r) / r
//   minus += w_q phi(s_q, t_q) (x - z).n (1 - i kappa r) exp(i kappa r) / r^3
// with x = Phi_T(s_q, t_q), r = |x - z|.  loc < 0: constant basis; otherwise
// the local vertex (original order) whose hat function phi is.
template <bool HELM>
__device__ __noinline__ void green_double(const Tri &T, int loc, const double *z, const double *n,
                                          const Rule2D &R, double kappa, double out[4])
{
    double pr = 0.0, pi = 0.0, mr = 0.0, mi = 0.0;
#pragma unroll 1
    for (int q = 0; q < R.np; ++q) {
        const double s = R.s[q], t = R.t[q];
        const double phi = loc < 0 ? 1.0 : (loc == 0 ? 1.0 - s : (loc == 1 ? s - t : t));
        const double wq = R.w[q] * phi;
        double d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
            d[c] = (T.v[0][c] - z[c]) + s * (T.v[1][c] - T.v[0][c]) + t * (T.v[2][c] - T.v[1][c]);
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        const double ri = rsqrt(r2);
        const double dn = d[0] * n[0] + d[1] * n[1] + d[2] * n[2];
        const double h = wq * dn * (ri * ri * ri);
        if (!HELM) {
            pr += wq * ri;
            mr += h;
        } else {
            const double kr = kappa * (r2 * ri);
            double sn, cs;
            sincos(kr, &sn, &cs);
            pr += wq * cs * ri;
            pi += wq * sn * ri;
            mr += h * (cs + kr * sn);
            mi += h * (sn - kr * cs);
        }
    }
    out[0] = pr;
    out[1] = pi;
    out[2] = mr;
    out[3] = mi;
}

// The cluster's frame: origin, S = 2^E, and for the Helmholtz kernel the phase
// factor (fx_wave).
//
// Coordinates are taken to integers relative to the middle c0, exactly: differences of
// doubles where |c0| is above S (their last bits are above those kept), integers less
// the integer C0 below (a difference of doubles would round to 2^-53 S where the
// coordinates themselves are finer).
struct GreenFrame {
    double c0[3];       // 0 where C0 holds it
    s64 C0[3];          // 2^61 / S
    int E, ok, kexp;
    Fx2 kn;
    // x relative to the middle, 2^61 / S
    __device__ __forceinline__ s64 at(double x, int c, double sc) const
    {
        return __double2ll_rn((x - c0[c]) * sc) - C0[c];
    }
};

// Scale of the frame: the box of the points and of the rows' support triangles
// relative to the first point, in float (min, max: [x/z][min/max][3]).  Called by
// every thread of the CTA.
__device__ __forceinline__ void green_frame(const MeshView &m, const GreenArgs &a, int rb, int nr, int pb,
                                            int mp, int64_t lim, bool helm, float (*box)[12],
                                            GreenFrame &F)
{
    float lo[2][3], hi[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            lo[k][c] = 3.0e38f;
            hi[k][c] = -3.0e38f;
        }
    double ref[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) ref[c] = __ldg(a.z + 3 * (int64_t)pb + c);
    for (int k = threadIdx.x; k < mp; k += blockDim.x)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float d = (float)(__ldg(a.z + 3 * (int64_t)(pb + k) + c) - ref[c]);
            lo[1][c] = fminf(lo[1][c], d);
            hi[1][c] = fmaxf(hi[1][c], d);
        }
    for (int k = threadIdx.x; k < nr; k += blockDim.x) {
        const int i = __ldg(a.row_idx + rb + k);
        if (i < 0 || i >= lim) continue;
        const int klo = m.basis == BEM_P0 ? 0 : __ldg(m.vt_ptr + i);
        const int khi = m.basis == BEM_P0 ? 1 : __ldg(m.vt_ptr + i + 1);
        for (int t = klo; t < khi; ++t) {
            const double *g = m.geom + (int64_t)(m.basis == BEM_P0 ? i : __ldg(m.vt_tri + t)) * kGeomStride;
#pragma unroll
            for (int v = 0; v < 9; ++v) {
                const float d = (float)(__ldg(g + v) - ref[v % 3]);
                lo[0][v % 3] = fminf(lo[0][v % 3], d);
                hi[0][v % 3] = fmaxf(hi[0][v % 3], d);
            }
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo[k][c] = fminf(lo[k][c], __shfl_xor_sync(0xffffffffu, lo[k][c], o));
                hi[k][c] = fmaxf(hi[k][c], __shfl_xor_sync(0xffffffffu, hi[k][c], o));
            }
            if (lane == 0) {
                box[warp][6 * k + c] = lo[k][c];
                box[warp][6 * k + 3 + c] = hi[k][c];
            }
        }
    __syncthreads();
    if (threadIdx.x == 0) {
        float top = 0.0f, mids[3];
        for (int c = 0; c < 3; ++c) {
            float b[4] = {3.0e38f, -3.0e38f, 3.0e38f, -3.0e38f};
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
                for (int k = 0; k < 2; ++k) {
                    b[2 * k] = fminf(b[2 * k], box[w][6 * k + c]);
                    b[2 * k + 1] = fmaxf(b[2 * k + 1], box[w][6 * k + 3 + c]);
                }
            const float mid = 0.5f * (fminf(b[0], b[2]) + fmaxf(b[1], b[3]));
            mids[c] = mid;
            const float x = fmaxf(b[1] - mid, mid - b[0]), z = fmaxf(b[3] - mid, mid - b[2]);
            top = fmaxf(top, x + z);
        }
        top *= 1.0001f;
        const int ex = __float_as_int(top) >> 23;
        F.ok = ex > 27 && ex < 227;          // also false for boxes without rows or beyond float
        F.E = ex - 126;
        for (int c = 0; c < 3 && F.ok; ++c) {
            // a multiple of 2^-16 S
            const double c0 = rint((ref[c] + (double)mids[c]) * fx_pow2(16 - F.E)) * fx_pow2(F.E - 16);
            const bool whole = fabs(c0) <= fx_pow2(F.E);
            F.c0[c] = whole ? 0.0 : c0;
            F.C0[c] = whole ? __double2ll_rn(c0 * fx_pow2(61 - F.E)) : 0;
        }
        if (F.ok && helm) F.ok = fx_wave(a.kappa, F.E, -4, kFxLeastWave, F.kn, F.kexp);   // the phase's shift stays >= 0
    }
    __syncthreads();
}

// green_double's sums in fixed point; Z and N: the lane's point (2^62 / S) and normal
// (2^61).  The lanes compute the triangle's rule points together (lane 3 q + c:
// component c of point q, eight points at a time): every lane of the warp calls
// this with the same triangle.
template <bool HELM, int NP>
__device__ __forceinline__ bool green_fixed(const GreenFrame &F, const Tri &T, int loc, const s64 *Z,
                                            const Fx2 *N, const Rule2D &R, double kappa, int lane,
                                            double out[4])
{
    const double sc = fx_pow2(61 - F.E);
    // this lane's rule point components, 2^62 / S
    constexpr int NR = (NP + 7) / 8;
    s64 mine[NR];
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        const int q = 8 * u + lane / 3, c = lane % 3;
        mine[u] = 0;
        if (lane < 24 && q < NP) {
            const double v0 = c == 0 ? T.v[0][0] : (c == 1 ? T.v[0][1] : T.v[0][2]);
            const double v1 = c == 0 ? T.v[1][0] : (c == 1 ? T.v[1][1] : T.v[1][2]);
            const double v2 = c == 0 ? T.v[2][0] : (c == 1 ? T.v[2][1] : T.v[2][2]);
            const double x = (v0 - F.c0[c]) + R.s[q] * (v1 - v0) + R.t[q] * (v2 - v1);
            mine[u] = (__double2ll_rn(x * sc) - F.C0[c]) << 1;
        }
    }
    auto component = [&](int q, int c) {
        s64 part = mine[0];
#pragma unroll
        for (int u = 1; u < NR; ++u)
            if (q >= 8 * u) part = mine[u];
        return __shfl_sync(0xffffffffu, part, 3 * (q & 7) + c);
    };
    // kb from the smallest distance of the rule's points, in float
    float lo = 3.0e38f;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        float d2 = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float d = __shfl_sync(0xffffffffu, fx_hi(mine[q / 8]), 3 * (q & 7) + c) - fx_hi(Z[c]);
            d2 = fmaf(d, d, d2);
        }
        lo = fminf(lo, d2);
    }
    const int kb = fx_kb(sqrtf(lo) * 0.49995f - 64.0f);   // S = 2^30 here
    // sums of values up to 2^59 stay below 2^57; four bits of their fractions count, where no
    // outer sum averages the rounding
    constexpr int UP = 4;
    FxSum pr, pi, m3r, m3i, m2r, m2i;
    pr.clear<UP>();
    pi.clear<UP>();
    m3r.clear<UP>();
    m3i.clear<UP>();
    m2r.clear<UP>();
    m2i.clear<UP>();
    int flag = 0;
    const int wl = loc < 0 ? 3 : loc;
#pragma unroll 1
    for (int q = 0; q < NP; ++q) {
        s64 d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = component(q, c) - Z[c];
        const s64 r2 = fx_norm2(d[0], d[1], d[2]);
        const s64 y = fx_rinv(r2, kb, flag);                     // 2^(62 - kb) S / r
        const Fx2 t1 = fx_split(y);
        const Fx2 t2 = fx_split(fx_mul_up<2>(t1, t1));           // 2^(62 - 2 kb) (S / r)^2
        const Fx2 t3 = fx_split(fx_mul_up<2>(t2, t1));           // 2^(62 - 3 kb) (S / r)^3
        // (x - z).n at 2^60 / S (at most sqrt(3)), times (S / r)^3
        const Fx2 a = fx_split(d[0]), b = fx_split(d[1]), e = fx_split(d[2]);
        const s64 mid = fx_mad(a.h, N[0].l, fx_mad(a.l, N[0].h, fx_mad(b.h, N[1].l, fx_mad(b.l, N[1].h, 0)))) +
                        fx_mad(e.h, N[2].l, fx_mad(e.l, N[2].h, 0));
        const Fx2 dn = fx_split((fx_mad(a.h, N[0].h, fx_mad(b.h, N[1].h, fx_mad(e.h, N[2].h, fx_high(mid))))) << 1);
        // dn is at most r, so its products with the powers are at most the next lower ones:
        // kb + 1 bits that points of a small triangle in a large cluster need
        const Fx2 h3 = fx_split(fx_mul_up(t3, dn, kb + 1));      // 2^(59 - 2 kb) (S / r)^3 dn / S
        const int32_t *w = R.wx[wl][q];
        if (!HELM) {
            pr.add(w, fx_split(y >> 3));                         // 2^(59 - kb)
            m3r.add(w, h3);
            continue;
        }
        const Fx2 h2 = fx_split(fx_mul_up(t2, dn, kb + 1));      // 2^(59 - kb) (S / r)^2 dn / S
        const Fx2 rho = fx_split(fx_mul_up<4>(fx_split(r2), t1));   // 2^(62 - kb) r / S
        s64 cs, sn;
        fx_sincos((u64)fx_mul(rho, F.kn) << (4 + kb + F.kexp), cs, sn);
        const Fx2 c = fx_split(cs), s = fx_split(sn);
        pr.add(w, fx_split(fx_mul(c, t1)));                      // 2^(59 - kb)
        pi.add(w, fx_split(fx_mul(s, t1)));
        // (c + kappa r s) / r^3 and (s - kappa r c) / r^3, the two powers apart
        m3r.add(w, fx_split(fx_mul_up<3>(c, h3)));               // 2^(59 - 2 kb)
        m3i.add(w, fx_split(fx_mul_up<3>(s, h3)));
        m2r.add(w, fx_split(fx_mul_up<3>(s, h2)));               // 2^(59 - kb)
        m2i.add(w, fx_split(fx_mul_up<3>(c, h2)));
    }
    // the sums hold half of their values
    const double fp = fx_pow2(1 - UP - (59 - kb) - F.E), f3 = fx_pow2(1 - UP - (59 - 2 * kb) - 2 * F.E);
    out[0] = pr.value<UP>() * fp;
    if (!HELM) {
        out[2] = m3r.value<UP>() * f3;
    } else {
        const double f2 = kappa * fx_pow2(1 - UP - (59 - kb) - F.E);
        out[1] = pi.value<UP>() * fp;
        out[2] = fma(f3, m3r.value<UP>(), f2 * m2r.value<UP>());
        out[3] = fma(f3, m3i.value<UP>(), -f2 * m2i.value<UP>());
    }
    return (flag >> (16 + kb)) == 0;
}

template <bool HELM, int NP>
__global__ void __launch_bounds__(kGreenThreads) k_green(MeshView m, GreenArgs a,
                                                         const __grid_constant__ Rule2D R, int *status)
{
    __shared__ int s_ok;
    __shared__ int s_rb, s_nr, s_pb, s_mp;
    __shared__ long long s_off;
    __shared__ float box[kGreenThreads / 32][12];
    __shared__ GreenFrame F;
    const int c = blockIdx.x;
    if (threadIdx.x == 0) {
        const int32_t rb = a.row_ptr[c], re = a.row_ptr[c + 1];
        const int32_t pb = a.pt_ptr[c], pe = a.pt_ptr[c + 1];
        const int64_t off = a.out_off[c];
        // the row and point loops step in int: a cluster holds fewer than 2^30 of each
        bool ok = rb >= 0 && re >= rb && re <= a.n_row_idx && pb >= 0 && pe >= pb &&
                  pe <= a.n_points && re - rb < (1 << 30) && pe - pb < (1 << 30);
        if (ok && re > rb && pe > pb) {
            // both factors are below 2^31, so the block size fits in int64
            const int64_t need = 2 * (int64_t)(re - rb) * (int64_t)(pe - pb);
            ok = off >= 0 && off <= a.out_len - need;
        }
        if (!ok) set_status(status, BEM_ERR_INVALID_ARG);
        s_ok = ok && re > rb && pe > pb;
        s_rb = rb;
        s_nr = re - rb;
        s_pb = pb;
        s_mp = pe - pb;
        s_off = off;
    }
    __syncthreads();
    if (!s_ok) return;
    const int rb = s_rb, nr = s_nr, pb = s_pb, mp = s_mp;
    const int64_t off = s_off;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int64_t lim = m.basis == BEM_P0 ? m.nt : m.nv;
    green_frame(m, a, rb, nr, pb, mp, lim, HELM, box, F);
    const int chunks = (mp + 31) / 32;
    const int64_t units = (int64_t)nr * chunks;
    for (int64_t u = (int64_t)blockIdx.y * nwarps + warp; u < units; u += (int64_t)gridDim.y * nwarps) {
        const int r = (int)(u / chunks), base = (int)(u - (int64_t)r * chunks) * 32;
        const int i = __ldg(a.row_idx + rb + r);
        if (i < 0 || i >= lim) {
            if (lane == 0) set_status(status, BEM_ERR_INVALID_ARG);
            continue;
        }
        const int klo = m.basis == BEM_P0 ? 0 : __ldg(m.vt_ptr + i);
        const int khi = m.basis == BEM_P0 ? 1 : __ldg(m.vt_ptr + i + 1);
        const int nu = base + lane;
        const bool act = nu < mp;
        // idle lanes of the last chunk repeat the cluster's last point and write nothing
        const int64_t p = pb + (act ? nu : mp - 1);
        double z[3], n[3];
        s64 Z[3];
        Fx2 N[3];
        // normals are unit vectors: longer ones leave the fixed-point range (the middle sum
        // of (x - z).n fills 0.97 of 64 bits at length 1), shorter ones lose digits in it.
        // Infinite and NaN points or normals fail the tests too (converted to the largest
        // or the lowest integer); the box that the frame is made of drops a NaN.
        s64 nn = 0;
        bool inside = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            z[d] = __ldg(a.z + 3 * p + d);
            n[d] = __ldg(a.nz + 3 * p + d);
            const s64 zi = F.ok ? F.at(z[d], d, fx_pow2(61 - F.E)) : 0;
            inside = inside && abs(fx_high(zi) >> 1) <= 1 << 28;
            Z[d] = zi << 1;
            N[d] = fx_split(__double2ll_rn(n[d] * 2305843009213693952.0));
            nn = fx_mad(N[d].h >> 1, N[d].h >> 1, nn);      // 2^56
        }
        inside = inside && abs(fx_high(nn) - (1 << 24)) <= 1 << 14;
        const bool fixed = F.ok && __all_sync(0xffffffffu, inside);
        double pr = 0.0, pi = 0.0, mr = 0.0, mi = 0.0;
        for (int k = klo; k < khi; ++k) {
            const int tr = m.basis == BEM_P0 ? i : __ldg(m.vt_tri + k);
            Tri T;
            load_tri(m.geom, tr, T);
            int loc = -1;
            if (m.basis == BEM_P1) {
                const int4 tv = __ldg(m.tvid + tr);
                loc = tv.x == i ? 0 : (tv.y == i ? 1 : 2);
            }
            double v[4];
            if (!fixed || !green_fixed<HELM, NP>(F, T, loc, Z, N, R, a.kappa, lane, v))
                green_double<HELM>(T, loc, z, n, R, a.kappa, v);
            pr += T.sg * v[0];
            mr += T.sg * v[2];
            if (HELM) {
                pi += T.sg * v[1];
                mi += T.sg * v[3];
            }
        }
        if (act) {
            const double fp = (a.sp ? __ldg(a.sp + p) : 1.0) * kInv4Pi;
            const double fm = (a.sm ? __ldg(a.sm + p) : 1.0) * kInv4Pi;
            const int64_t ep = off + r + (int64_t)nu * nr;          // A+ column nu
            const int64_t em = off + r + (int64_t)(mp + nu) * nr;   // A- column nu
            if (HELM) {
                double2 *o = reinterpret_cast<double2 *>(a.out);
                o[ep] = make_double2(fp * pr, fp * pi);
                o[em] = make_double2(fm * mr, fm * mi);
            } else {
                double *o = reinterpret_cast<double *>(a.out);
                o[ep] = fp * pr;
                o[em] = fm * mr;
            }
        }
    }
}

// CTAs (cluster, part): the parts of a cluster share its units, so that a tree of a
// few hundred clusters of about 30 rows still fills the GPU several times over
// (four CTAs per SM are resident; one CTA of eight warps per cluster left the
// last of 3 waves nearly empty).  More than eight parts would repeat the frame's
// set-up for less than two units a warp.
template <bool HELM>
cudaError_t launch_green(const MeshView &m, const GreenArgs &a, int n_clusters, const Rule2D &R,
                         int *status, int num_sms, cudaStream_t st)
{
    const int parts = std::min(8, (24 * num_sms + n_clusters - 1) / n_clusters);
    const dim3 grid((unsigned)n_clusters, (unsigned)parts);
#define BEM_GREEN(NP) k_green<HELM, NP><<<grid, kGreenThreads, 0, st>>>(m, a, R, status)
    switch (R.np) {
    case 1: BEM_GREEN(1); break;
    case 4: BEM_GREEN(4); break;
    case 7: BEM_GREEN(7); break;
    case 9: BEM_GREEN(9); break;
    case 16: BEM_GREEN(16); break;
    case 25: BEM_GREEN(25); break;
    default: return cudaErrorInvalidValue;
    }
#undef BEM_GREEN
    return cudaGetLastError();
}

}  // namespace
}  // namespace bem

extern "C" int bem_green_matrices(bem_ctx *ctx, const bem_green_job *job)
{
    using namespace bem;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!job) return api_fail(ctx, BEM_ERR_INVALID_ARG, "null job");
    const bem_green_job &J = *job;
    auto it = ctx->meshes.find(J.mesh_id);
    if (it == ctx->meshes.end()) return api_fail(ctx, BEM_ERR_INVALID_ARG, "unknown mesh id");
    const Mesh *mesh = it->second;
    if (J.kernel.kind < BEM_LAPLACE_SLP || J.kernel.kind > BEM_HELMHOLTZ_SLP ||
        !std::isfinite(J.kernel.kappa))
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "bad kernel descriptor");
    Rule2D R;
    std::memset(&R, 0, sizeof R);
    if (!(J.rule == BEM_RULE_TRI7 || (J.rule == BEM_RULE_DUFFY && J.q >= 1 && J.q <= 5)) ||
        !make_rule2d(J.rule, J.q, R))
        return api_fail(ctx, BEM_ERR_INVALID_ARG,
                        "bem_green_matrices: rule must be TRI7 or DUFFY with q in [1, 5]");
    if (J.n_clusters < 0 || J.n_row_idx < 0 || J.n_points < 0 || J.out_len < 0)
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "negative count");
    if (J.n_clusters == 0) return BEM_OK;
    if (!J.row_ptr || !J.pt_ptr || !J.out_off || (J.n_row_idx > 0 && !J.row_idx) ||
        (J.n_points > 0 && (!J.z || !J.nz)) || (J.out_len > 0 && !J.out))
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "null pointer");
    const bool helm = J.kernel.kind == BEM_HELMHOLTZ_SLP;
    if (helm && (reinterpret_cast<uintptr_t>(J.out) & 15))
        return api_fail(ctx, BEM_ERR_INVALID_ARG, "complex output must be 16-byte aligned");
    GreenArgs a;
    a.row_ptr = J.row_ptr;
    a.row_idx = J.row_idx;
    a.pt_ptr = J.pt_ptr;
    a.z = J.z;
    a.nz = J.nz;
    a.sp = J.sp;
    a.sm = J.sm;
    a.out_off = J.out_off;
    a.out = J.out;
    a.n_row_idx = J.n_row_idx;
    a.n_points = J.n_points;
    a.out_len = J.out_len;
    a.kappa = helm ? J.kernel.kappa : 0.0;
    cudaError_t e;
    {
        ProfScope ps(ctx, "green");
        e = helm ? launch_green<true>(mesh->v, a, J.n_clusters, R, ctx->status, ctx->num_sms, ctx->stream)
                 : launch_green<false>(mesh->v, a, J.n_clusters, R, ctx->status, ctx->num_sms, ctx->stream);
    }
    if (e != cudaSuccess) return api_cuda_fail(ctx, e, "green kernel");
    return BEM_OK;
}

extern "C" int bem_gca_pivots_device(bem_ctx *ctx, int32_t mesh_id, const double *verts,
                                     int64_t nv, const int32_t *tris, int64_t nt, int32_t basis,
                                     double kappa, const int32_t *cl_ptr, const int32_t *cl_idx,
                                     const int32_t *cl_son, int32_t n_clusters,
                                     int32_t gauss_per_face, double eps, int32_t max_rank,
                                     int32_t n_threads, int32_t *piv_ptr, int32_t *piv_idx,
                                     int64_t cap)
{
    using namespace bem;
    if (!ctx) return BEM_ERR_INVALID_ARG;
    auto it = ctx->meshes.find(mesh_id);
    if (it == ctx->meshes.end()) return api_fail(ctx, BEM_ERR_INVALID_ARG, "unknown mesh id");
    const Mesh *mesh = it->second;
    if (mesh->v.nv != nv || mesh->v.nt != nt || mesh->v.basis != basis || !verts || !tris ||
        mesh_hash(verts, nv, tris, nt) != mesh->host_hash)
        return api_fail(ctx, BEM_ERR_INVALID_ARG,
                        "bem_gca_pivots_device: the host mesh is not the uploaded one "
                        "(coordinates, connectivity or basis)");
    Rule2D R;
    std::memset(&R, 0, sizeof R);
    make_rule2d(BEM_RULE_TRI7, 0, R);
    // one device buffer for a level's inputs and blocks, grown for the largest level
    struct Scratch {
        char *p = nullptr;
        size_t bytes = 0;
        ~Scratch()
        {
            if (p) cudaFree(p);
        }
    } S;
    auto produce = [&](const GreenLevel &L, bool cplx_out, std::vector<double> &out) -> int {
        auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
        const size_t n_cl = L.off.size();
        const size_t parts[9] = {L.row_ptr.size() * 4, L.pt_ptr.size() * 4, L.rows.size() * 4,
                                 L.z.size() * 8,       L.nz.size() * 8,     L.sp.size() * 8,
                                 L.sm.size() * 8,      n_cl * 8,            out.size() * 8};
        const void *src[8] = {L.row_ptr.data(), L.pt_ptr.data(), L.rows.data(), L.z.data(),
                              L.nz.data(),      L.sp.data(),     L.sm.data(),   L.off.data()};
        size_t at[9], need = 0;
        for (int k = 0; k < 9; ++k) {
            at[k] = need;
            need += al(std::max<size_t>(parts[k], 1));
        }
        cudaError_t e = cudaSuccess;
        if (need > S.bytes) {
            if (S.p) cudaFree(S.p);
            S.p = nullptr;
            S.bytes = 0;
            e = cudaMalloc((void **)&S.p, need);
            if (e != cudaSuccess) return api_cuda_fail(ctx, e, "cudaMalloc(GCA level)");
            S.bytes = need;
        }
        for (int k = 0; k < 8 && e == cudaSuccess; ++k)
            if (parts[k] > 0)
                e = cudaMemcpyAsync(S.p + at[k], src[k], parts[k], cudaMemcpyHostToDevice,
                                    ctx->stream);
        if (e != cudaSuccess) return api_cuda_fail(ctx, e, "GCA level upload");
        GreenArgs a;
        a.row_ptr = reinterpret_cast<const int32_t *>(S.p + at[0]);
        a.pt_ptr = reinterpret_cast<const int32_t *>(S.p + at[1]);
        a.row_idx = reinterpret_cast<const int32_t *>(S.p + at[2]);
        a.z = reinterpret_cast<const double *>(S.p + at[3]);
        a.nz = reinterpret_cast<const double *>(S.p + at[4]);
        a.sp = reinterpret_cast<const double *>(S.p + at[5]);
        a.sm = reinterpret_cast<const double *>(S.p + at[6]);
        a.out_off = reinterpret_cast<const int64_t *>(S.p + at[7]);
        a.out = S.p + at[8];
        a.n_row_idx = (int64_t)L.rows.size();
        a.n_points = (int64_t)L.sp.size();
        a.out_len = L.total;
        a.kappa = cplx_out ? kappa : 0.0;
        {
            ProfScope ps(ctx, "green");
            e = cplx_out ? launch_green<true>(mesh->v, a, (int)n_cl, R, ctx->status, ctx->num_sms, ctx->stream)
                         : launch_green<false>(mesh->v, a, (int)n_cl, R, ctx->status, ctx->num_sms, ctx->stream);
        }
        if (e != cudaSuccess) return api_cuda_fail(ctx, e, "green kernel");
        e = cudaMemcpyAsync(out.data(), S.p + at[8], parts[8], cudaMemcpyDeviceToHost, ctx->stream);
        if (e != cudaSuccess) return api_cuda_fail(ctx, e, "GCA level download");
        return bem_sync(ctx);
    };
    return gca_pivots_levels(verts, nv, tris, nt, basis, kappa, cl_ptr, cl_idx, cl_son, n_clusters,
                             gauss_per_face, eps, max_rank, n_threads, produce, piv_ptr, piv_idx,
                             cap);
}
