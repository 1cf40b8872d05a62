// Touching pairs of the FP64 form in the fixed-point arithmetic of bem_fixed.cuh:
// the Sauter-Schwab rules with xi integrated out (q^3 points per subdomain at
// xi = 1; for the complex kinds the sum over xi at each point in node pairs), one
// warp per pair.
//
// At xi = 1 every coordinate and difference of a common-edge or identical rule
// is e1 = eta_1 times a function of (eta_2, eta_3), so the table holds the
// columns divided by g = e1 (g = 1 for a common vertex): the direction v = (x - y)
// / g keeps a length of the order of the edges, within the fixed-point range,
// and r = g |v|.  The factors of g go into the weights.  A pair with a direction
// shorter than S / 16 (slivers) returns false and is evaluated in FP64.
//
// Values lie far below the largest that the shortest direction and the largest height
// allow, so products of a common vertex take their room from the points themselves, and
// lanes add their sums with fractions.  Double layers of the common vertices of a
// 96-triangle torus, root mean square error over the sum of the terms' magnitudes: Laplace
// 2.3e-16, Helmholtz 2.5e-16; without either 4.1e-16 and 7.2e-16; FP64 2.7e-16 and 2.8e-16.
#pragma once

#include "bem_device.cuh"

namespace bem {

// Sums over xi at one direction point: G_n = sum_k w_k xi_k^n exp(i theta xi_k), n = 1, 2.
// G_n = exp(i theta / 2) (A + i B)
__device__ __forceinline__ void fx_xi_sum(const XiFixed &X, int n, const s64 *c, const s64 *s, Fx2 c0,
                                          Fx2 s0, Fx2 &gr, Fx2 &gi)
{
    FxSum a, b;
    a.clear<2>();
    b.clear<2>();
#pragma unroll
    for (int j = 0; j < kMaxXiFixedPairs; ++j) {
        if (j >= X.npair) break;
        a.add(X.cp[j][n], fx_split(c[j]));
        b.add(X.cm[j][n], fx_split(s[j]));
    }
    // A, B and the rotation's result at 2^61
    const Fx2 A = fx_split(a.sum<2>() + (X.cmid[n] << 2)), B = fx_split(b.sum<2>());
    gr = fx_split(fx_mul_up<3>(A, c0) - fx_mul_up<3>(B, s0));
    gi = fx_split(fx_mul_up<3>(A, s0) + fx_mul_up<3>(B, c0));
}

template <int KIND, int BASIS, int CAS>
__device__ __forceinline__ bool touch_fixed(const MeshView &m, int idx, const int2 *__restrict__ fx,
                                            int np, double kappa, double eta, int lane,
                                            const XiFixed &X)
{
    constexpr bool HELM = kind_complex(KIND);
    static_assert(!HELM || BASIS == BEM_P0, "complex kinds: piecewise constant");
    constexpr bool HEIGHT = kind_has_height(KIND) && CAS != kIdentical;
    constexpr bool ONE = KIND == BEM_LAPLACE_SLP || KIND == BEM_HELMHOLTZ_SLP || KIND == BEM_HELMHOLTZ_BW;
    // sums: [ONE: re, im] [heights: 1/r^3 re, im, 1/r^2 re, im]; Laplace: one, or nine moments
    constexpr int NS = BASIS == BEM_P1 ? 9 : !HELM ? 1 : (ONE ? 2 : 0) + (HEIGHT ? 4 : 0);
    // weights of the heights' sums: a common edge's heights are x2 times one number, which
    // the weights hold; a common vertex' multiply every point's value (sums per coefficient
    // cancel where the heights do)
    constexpr int WB = CAS == kVertex ? kFxA : kFxB, WC = CAS == kVertex ? kFxA : kFxC;
    constexpr bool ZERO = NS == 0 || (KIND == BEM_LAPLACE_DLP && CAS == kIdentical);
    const int a = __ldg(m.nb_src + idx), b = __ldg(m.nb_tri + idx);
    const int pc = __ldg(m.nb_perm + idx);
    const int *pa = c_perm[pc / 6], *pb = c_perm[pc % 6];
    const double *ga = m.geom + (int64_t)a * kGeomStride, *gb = m.geom + (int64_t)b * kGeomStride;
    s64 tot[NS > 0 ? NS : 1];
#pragma unroll
    for (int k = 0; k < (NS > 0 ? NS : 1); ++k) tot[k] = 0;
    double height = 0.0;   // a common edge's h21, the unit of a common vertex' heights
    int E = 0, flag = 0, kbs = 0, up = 0, k3 = 3, k2 = 3;
    if (!ZERO) {
        // lane 3 e + c: component c of edge e (a: v1 - v0, v2 - v1; b: the same)
        double val = 0.0, far = 0.0;
        if (lane < 12) {
            const int e = lane / 3, c = lane - 3 * e, hi = (e & 1) + 1;
            const double *g = e < 2 ? ga : gb;
            const int *p = e < 2 ? pa : pb;
            const double v = __ldg(g + 3 * p[hi] + c);
            val = v - __ldg(g + 3 * p[hi - 1] + c);
            far = CAS == kVertex ? v - __ldg(g + 3 * p[0] + c) : val;
        }
        // S = 2^E above every component of a direction: at most a corner of a minus one of b
        // for a common vertex, else the sum of the edges that occur.  No larger than needed:
        // the squared length is held to 2^-60 S^2
        const float f = __double2float_ru(fabs(far));
        const float f1 = __shfl_sync(0xffffffffu, f, (lane + 3) & 31), f2 = __shfl_sync(0xffffffffu, f, (lane + 6) & 31),
                    f3 = __shfl_sync(0xffffffffu, f, (lane + 9) & 31);
        float sum = CAS == kVertex ? fmaxf(f, f1) + fmaxf(f2, f3) : (CAS == kEdge ? f + f1 + f3 : f + f1);
        sum = fmaxf(fmaxf(__shfl_sync(0xffffffffu, sum, 0), __shfl_sync(0xffffffffu, sum, 1)),
                    __shfl_sync(0xffffffffu, sum, 2)) * 1.000001f;
        const int ex = __float_as_int(sum) >> 23;
        if (ex < 7 || ex > 246) return false;   // uniform across the warp
        E = ex - 126;
        const Fx2 mine = fx_split(__double2ll_rn(val * fx_pow2(61 - E)));
        Fx2 ed[4][3];
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                ed[e][c].h = __shfl_sync(0xffffffffu, mine.h, 3 * e + c);
                ed[e][c].l = __shfl_sync(0xffffffffu, mine.l, 3 * e + c);
            }
        // heights of a's vertices 1, 2 above b's plane (vertex 0 lies in it): x1 h1 + x2 h21,
        // for a common edge h1 = 0.  Sums of products exact to 2^-60 of the largest: a
        // rounding of a height would be one of every point's value
        Fx2 n1 = {0, 0}, n2 = {0, 0};
        int eh = 0;
        if (HEIGHT) {
            double t = 0.0, e = 0.0;
            if (lane < 6) {
                const int k = lane / 3, c = lane - 3 * k;
                const double x = __ldg(ga + 3 * pa[k + 1] + c) - __ldg(gb + 3 * pb[0] + c), nc = __ldg(gb + 9 + c);
                t = x * nc;
                e = fma(x, nc, -t);
            }
            eh = max((__reduce_max_sync(0xffffffffu, fx_mag(t)) >> 20) - 1022, -900);
            s64 i = __double2ll_rn(t * fx_pow2(60 - eh)) + __double2ll_rn(e * fx_pow2(60 - eh));
            i += __shfl_sync(0xffffffffu, i, (lane + 1) & 31) + __shfl_sync(0xffffffffu, i, (lane + 2) & 31);
            const s64 d1 = __shfl_sync(0xffffffffu, i, 0), d2 = __shfl_sync(0xffffffffu, i, 3);
            if (CAS == kVertex) {
                // both below 2^59, their unit 2^59
                const s64 d = d2 - d1;
                const int hup = __clzll((d1 ^ (d1 >> 63)) | (d ^ (d >> 63))) - 5;
                n1 = fx_split(hup >= 0 ? d1 << hup : d1 >> -hup);
                n2 = fx_split(hup >= 0 ? d << hup : d >> -hup);
                height = fx_pow2(eh - 1 - hup);
            } else {
                height = (double)d2 * fx_pow2(eh - 60);
            }
        }
        Fx2 kn = {0, 0};
        int kexp = 0;
        if (HELM && !fx_wave(kappa, E, kFxLeastWave, kFxLeastWave, kn, kexp)) return false;   // uniform across the warp
        auto shifted = [](s64 v, int n) { return n >= 0 ? (u64)v << n : (u64)(v >> -n); };
        auto col = [&](int c, int p) {
            const int2 v = __ldg(fx + (int64_t)c * np + p);
            Fx2 r;
            r.h = v.x;
            r.l = v.y;
            return r;
        };
        // kb: S / |v| <= 2^kb, from the shortest direction of all points in float (a
        // tenth of a point's work; the powers of 1/r gain up to 3 bits per unit)
        // A common vertex: also the largest height times 1/|v|^3 and 1/|v|^2, for which the
        // products leave room (not for the largest height at the shortest direction)
        constexpr bool UP = HEIGHT && CAS == kVertex;
        float lo = 3.0e38f, m3 = 0.0f, m2 = 0.0f;
#pragma unroll 2
        for (int p = lane; p < np; p += 32) {
            const float w0 = (float)__ldg(&fx[p].x), w1 = (float)__ldg(&fx[np + p].x);
            const float w2 = CAS != kIdentical ? (float)__ldg(&fx[2 * np + p].x) : 0.0f;
            const float w3 = CAS == kVertex ? (float)__ldg(&fx[3 * np + p].x) : 0.0f;
            float d2 = 0.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float d = fmaf(w0, (float)ed[0][c].h, w1 * (float)ed[1][c].h);
                if (CAS == kVertex) d = fmaf(-w2, (float)ed[2][c].h, fmaf(-w3, (float)ed[3][c].h, d));
                if (CAS == kEdge) d = fmaf(-w2, (float)ed[3][c].h, d);
                d2 = fmaf(d, d, d2);
            }
            lo = fminf(lo, d2);
            if (UP) {
                const float ri = rsqrt_fast(d2) * 288230376151711744.0f;   // S / |v|
                const float hi = fabsf(fmaf(w0, (float)n1.h, w1 * (float)n2.h)) * (ri * ri);   // height at 2^56
                m2 = fmaxf(m2, hi);
                m3 = fmaxf(m3, hi * ri);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        const int kb = fx_kb(sqrtf(lo) * (float)(0.9999 / 536870912.0) - 64.0f);   // 2^58 -> 2^29
        // bits of the products with t3 and t2 that keep them below 2^61 (1.02: float roundings
        // of heights that cancel)
        if (UP) {
            const int e3 = (int)(__reduce_max_sync(0xffffffffu, __float_as_uint(m3 * 1.02f)) >> 23) - 126;
            const int e2 = (int)(__reduce_max_sync(0xffffffffu, __float_as_uint(m2 * 1.02f)) >> 23) - 126;
            k3 = max(min(59 + 3 * kb - e3, 30), 0);
            k2 = max(min(59 + 2 * kb - e2, 30), 0);
        }
        // a lane's points in runs of 4: values up to 2^61 keep the sums' middle parts
        // within 64 bits
        constexpr int RUN = 32 * 4;
        FxSum acc[NS > 0 ? NS : 1];
#pragma unroll
        for (int k = 0; k < NS; ++k) acc[k].hi = acc[k].mid = 0;
        for (int p0 = lane; p0 < np; p0 += RUN) {
#pragma unroll 1
            for (int p = p0; p < min(np, p0 + RUN); p += 32) {
                // direction at 2^62 / S
                s64 v[3];
                const Fx2 u0 = col(kFxX, p), u1 = col(kFxX + 1, p);
                Fx2 u2 = {0, 0}, u3 = {0, 0};
                if (CAS != kIdentical) u2 = col(kFxX + 2, p);
                if (CAS == kVertex) u3 = col(kFxX + 3, p);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    // identical: d1 e1 + d2 e2; edge: d1 e1 + x2 e2 - y2 e2b;
                    // vertex: x1 e1 + x2 e2 - y1 e1b - y2 e2b
                    const Fx2 e1 = ed[0][c], e2 = ed[1][c];
                    s64 mid = fx_mad(e1.h, u0.l, fx_mad(e1.l, u0.h, fx_mad(e2.h, u1.l, fx_mad(e2.l, u1.h, 0))));
                    s64 hi = fx_mad(e1.h, u0.h, fx_mad(e2.h, u1.h, 0));
                    if (CAS != kIdentical) {
                        const Fx2 e3 = CAS == kEdge ? ed[3][c] : ed[2][c];
                        mid -= fx_mad(e3.h, u2.l, fx_mad(e3.l, u2.h, 0));
                        hi -= fx_mad(e3.h, u2.h, 0);
                    }
                    if (CAS == kVertex) {
                        const Fx2 e4 = ed[3][c];
                        mid -= fx_mad(e4.h, u3.l, fx_mad(e4.l, u3.h, 0));
                        hi -= fx_mad(e4.h, u3.h, 0);
                    }
                    v[c] = fx_shl(hi + fx_high(mid), 4);
                }
                const s64 r2 = fx_norm2(v[0], v[1], v[2]);
                auto add = [&](int k, int c, Fx2 value) {
                    const Fx2 w = col(c, p);
                    const int32_t ww[2] = {w.h, w.l};
                    acc[k].add(ww, value);
                };
                if (!HELM && ONE) {
                    const Fx2 T = fx_split(fx_rinv(r2, kb + 1, flag));        // 2^(61 - kb) S / |v|
                    if (BASIS == BEM_P0) {
                        add(0, kFxA, T);
                    } else {
#pragma unroll
                        for (int k = 0; k < 9; ++k) add(k, kFxMS + k, T);
                    }
                    continue;
                }
                const Fx2 T = fx_split(fx_rinv(r2, kb, flag));                // 2^(62 - kb) S / |v|
                Fx2 t2, t3;
                if (HEIGHT) {
                    // (S/|v|)^2 at 2^(62 - 2 kb), (S/|v|)^3 at 2^(62 - 3 kb) (2^61 where it is summed)
                    t2 = fx_split(fx_mul_up<2>(T, T));
                    constexpr int K3 = !HELM && CAS == kEdge ? 1 : 2;
                    t3 = fx_split(fx_mul_up<K3>(t2, T));
                }
                if (HEIGHT && CAS == kVertex) {
                    // height at 2^60 in its unit, into the powers
                    const s64 mid = fx_mad(n1.h, u0.l, fx_mad(n1.l, u0.h, fx_mad(n2.h, u1.l, fx_mad(n2.l, u1.h, 0))));
                    const Fx2 dn = fx_split((fx_mad(n1.h, u0.h, fx_mad(n2.h, u1.h, fx_high(mid)))) << 4);
                    // 2^(58 + k3 - 3 kb) (S/|v|)^3 dn, 2^(58 + k2 - 2 kb) (S/|v|)^2 dn; complex: twice that
                    t3 = fx_split(fx_mul_up(t3, dn, HELM ? k3 + 1 : k3));
                    if (HELM) t2 = fx_split(fx_mul_up(t2, dn, k2 + 1));
                }
                if (!HELM) {
                    if (BASIS == BEM_P0) {
                        add(0, WB, t3);
                    } else {
#pragma unroll
                        for (int k = 0; k < 9; ++k) add(k, kFxMD + k, t3);
                    }
                    continue;
                }
                // theta = kappa g |v|: |v| at 2^58 / S, times g, times kappa S / (2 pi)
                const s64 rho = fx_mul_up<4>(fx_split(r2), T) >> (4 - kb);
                const s64 rg = CAS == kVertex ? rho : fx_mul(fx_split(rho << 2), col(kFxG, p));   // g at 2^62
                const s64 turns = fx_mul_up<4>(fx_split(rg), kn);                  // theta / (2 pi) 2^(60 - kexp)
                const Fx2 th = fx_split(turns);
                s64 cs[kMaxXiFixedPairs], sn[kMaxXiFixedPairs];
#pragma unroll
                for (int j = 0; j < kMaxXiFixedPairs; ++j) {
                    if (j >= X.npair) break;
                    Fx2 tj;
                    tj.h = X.t[j][0];
                    tj.l = X.t[j][1];
                    fx_sincos(shifted(fx_mul_up<4>(th, tj), kexp + 2), cs[j], sn[j]);   // t_j at 2^62
                }
                s64 c0, s0;
                fx_sincos(shifted(turns, kexp + 3), c0, s0);                  // half of theta
                const Fx2 C0 = fx_split(c0), S0 = fx_split(s0);
                Fx2 g2r, g2i;
                fx_xi_sum(X, 1, cs, sn, C0, S0, g2r, g2i);
                if (ONE) {
                    add(0, kFxA, fx_split(fx_mul_up<2>(g2r, T)));             // 2^(61 - kb) S / |v|
                    add(1, kFxA, fx_split(fx_mul_up<2>(g2i, T)));
                }
                if (HEIGHT) {
                    Fx2 g1r, g1i;
                    fx_xi_sum(X, 0, cs, sn, C0, S0, g1r, g1i);
                    const Fx2 xr = fx_split(fx_mul_up<2>(g1r, t3)), xi = fx_split(fx_mul_up<2>(g1i, t3));   // 2^(61 - 3 kb) (S/|v|)^3
                    const Fx2 yr = fx_split(fx_mul_up<2>(g2r, t2)), yi = fx_split(fx_mul_up<2>(g2i, t2));   // 2^(61 - 2 kb) (S/|v|)^2
                    constexpr int o = ONE ? 2 : 0;
                    add(o, WB, xr);
                    add(o + 1, WB, xi);
                    add(o + 2, WC, yr);
                    add(o + 3, WC, yi);
                }
            }
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                acc[k].hi += fx_high(acc[k].mid);
                acc[k].mid = fx_low(acc[k].mid);
            }
        }
        flag = __reduce_or_sync(0xffffffffu, (unsigned)flag);
        if (flag >> (16 + kb)) return false;
        kbs = kb;
        // the lanes' sums with as many bits of their fractions as the 32 leave room for
        unsigned top = 0;
#pragma unroll
        for (int k = 0; k < NS; ++k) top |= (unsigned)fx_high(acc[k].hi ^ (acc[k].hi >> 63));
        up = min(max(__clz(__reduce_or_sync(0xffffffffu, top)) - 7, 0), 24);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const s64 f = acc[k].mid + ((s64)1 << (31 - up)), t = acc[k].hi + fx_high(f);
            tot[k] = fx_join(fx_funnel_l(fx_low(f), fx_low(t), up), (int)fx_funnel_l(fx_low(t), (unsigned)fx_high(t), up));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], o);
        }
    }
    if (lane == 0) {
        const double scale = __ldg(ga + 12) * __ldg(gb + 12) * kInv4Pi * fx_pow2(-up);
        if (BASIS == BEM_P0) {
            double re = 0.0, im = 0.0;
            if (!ZERO && !HELM) {
                // weights at 2^63: sums / 2
                if (ONE) re = (double)tot[0] * fx_pow2(1 - 61 + kbs - E);
                else re = height * (double)tot[0] * fx_pow2(1 - 58 - k3 + 3 * kbs - 3 * E);
                re *= xi_moment(KIND, 0, 0);
            } else if (!ZERO) {
                if (ONE) {
                    const double f1 = fx_pow2(1 - 61 + kbs - E), zr = (double)tot[0] * f1, zi = (double)tot[1] * f1;
                    re = KIND == BEM_HELMHOLTZ_BW ? eta * zi : zr;
                    im = KIND == BEM_HELMHOLTZ_BW ? -eta * zr : zi;
                }
                if (HEIGHT) {
                    const double f3 = fx_pow2(1 - 58 - k3 + 3 * kbs - 3 * E), f2 = kappa * fx_pow2(1 - 58 - k2 + 2 * kbs - 2 * E);
                    constexpr int o = ONE ? 2 : 0;
                    re += height * fma(f3, (double)tot[o], f2 * (double)tot[o + 3]);
                    im += height * fma(f3, (double)tot[o + 1], -f2 * (double)tot[o + 2]);
                }
            }
            m.table[idx] = make_double2(re * scale, im * scale);
        } else {
            double M[9], hr[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                M[k] = 0.0;
                if (!ZERO) {
                    M[k] = (double)tot[k] * xi_moment(KIND, k / 3, k % 3);
                    if (KIND == BEM_LAPLACE_SLP) M[k] *= fx_pow2(1 - 61 + kbs - E);
                    else M[k] *= height * fx_pow2(1 - 58 - k3 + 3 * kbs - 3 * E);
                }
            }
            moments_to_hats(M, hr);
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    m.table[(int64_t)idx * 9 + pa[i] * 3 + pb[j]] = make_double2(hr[i * 3 + j] * scale, 0.0);
        }
    }
    return true;
}

}  // namespace bem
