// Regular (disjoint) pairs of the FP64 form in the fixed-point arithmetic of
// bem_fixed.cuh: the product of a 2D rule with itself, one thread per pair.
// Included by bem_device.cuh (needs Tri, Rule2D and the FP64 pair integrals,
// which take over pairs outside the fixed-point range).
#pragma once

#include "bem_fixed.cuh"

namespace bem {

__device__ __forceinline__ double fx_pow2(int n) { return __hiloint2double((1023 + n) << 20, 0); }

// a 2^n by its exponent (an integer operation); a and a 2^n zero or normal
__device__ __forceinline__ double fx_scale(double a, int n)
{
    const int h = __double2hiint(a);
    return __hiloint2double(h != 0 ? h + (n << 20) : 0, __double2loint(a));
}

// Upper bound of |a|: the high word of a double, its lowest bit raised
__device__ __forceinline__ int fx_mag(double a) { return (__double2hiint(a) & 0x7fffffff) + 1; }

// kappa S / (2 pi) = kn 2^(kexp - 62), S = 2^E, |kn| <= 2^62: the factor that takes a
// length in units of S to a phase in turns.  1 / (2 pi) and the product as sums of two
// doubles: a relative error of kn is one of every phase of the pair.  kexp >= low.
// false below 2^(least - 1) turns (and above 2^20): the imaginary parts, sines of phases that
// small, are held to about 2^-57 of the magnitudes and would lose digits of their own, which
// FP64 arithmetic keeps (sphere of 80 triangles, root mean square error of the imaginary
// parts relative to themselves 2e-11 at kappa 1e-6, 1e-15 at 0.01, where the line lies).
constexpr int kFxLeastWave = -6;
__device__ __forceinline__ bool fx_small_wave(double kappa, int E)
{
    return kappa != 0.0 && ((__double2hiint(kappa * 0.15915494309189535) >> 20) & 2047) - 1022 + E < kFxLeastWave;
}
__device__ __forceinline__ bool fx_wave(double kappa, int E, int low, int least, Fx2 &kn, int &kexp)
{
    const double hi = kappa * 0.15915494309189535;
    const double lo = fma(kappa, 0.15915494309189535, -hi) + kappa * -9.839338337591243e-18;
    kexp = ((__double2hiint(hi) >> 20) & 2047) - 1022 + E;
    if (kexp > 20 || (kexp < least && kappa != 0.0)) return false;   // shifts of 4 + kb + kexp stay below 32
    kexp = max(kexp, low);
    const double up = fx_pow2(62 + E - kexp);
    kn = fx_split(__double2ll_rn(hi * up) + __double2ll_rn(lo * up));
    return true;
}

// Weighted sum of 64-bit values T with weights w = 2^63 times a rule's:
// value() = sum w T / 2 (the products of the low words dropped).  |T| <= 2^59
// keeps the middle sum within 64 bits for every rule (at most 25 points).
struct FxSum {
    s64 hi, mid;
    template <int K = 0>
    __device__ __forceinline__ void clear()
    {
        hi = 0;
        mid = (s64)1 << (31 - K);   // rounds sum<K>()
    }
    __device__ __forceinline__ void add(const int32_t *w, Fx2 T)
    {
        hi = fx_mad(w[0], T.h, hi);
        mid = fx_mad(w[0], T.l, fx_mad(w[1], T.h, mid));
    }
    // sum w T / 2, times 2^K
    template <int K = 0>
    __device__ __forceinline__ s64 sum() const
    {
        const s64 p = hi + fx_high(mid);
        if (K == 0) return p;
        return fx_join(fx_funnel_l(fx_low(mid), fx_low(p), K), (int)fx_funnel_l(fx_low(p), (unsigned)fx_high(p), K));
    }
    template <int K = 0>
    __device__ __forceinline__ double value() const { return (double)sum<K>(); }
};

// Vertices of a pair relative to the trial triangle's vertex 0, scaled to
// 2^61 / S with S = 2^E above every coordinate difference of the two triangles.
struct FxPair {
    s64 x0[3];                 // test triangle's vertex 0 / 4
    Fx2 a1[3], a2[3];          // test triangle's edges v1 - v0, v2 - v1
    Fx2 b1[3], b2[3];          // trial triangle's
    int E;
    int kb;                    // S / r <= 2^kb for every point of the pair (4: no bound known)
};

// kb of a lower bound r of the distances (S = 2^29)
__device__ __forceinline__ int fx_kb(float r)
{
    return r >= 33554432.0f ? max(0, 29 - ((__float_as_int(r) >> 23) - 127)) : 4;
}

__device__ __forceinline__ float fx_hi(s64 v) { return (float)(int)(v >> 32); }

// kb of a pair from a lower bound of its distances, the centroids' minus both
// circumradii about them; 8 covers the truncations (X, Y: vertices at 2^61 / S)
__device__ __forceinline__ int fx_centroid_kb(const s64 X[3][3], const s64 Y[3][3])
{
    float xf[3][3], yf[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xf[k][c] = fx_hi(X[k][c]);   // S = 2^29
            yf[k][c] = fx_hi(Y[k][c]);
        }
    float d2 = 0.0f, ra = 0.0f, rb = 0.0f, ca[3], cb[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        ca[c] = (xf[0][c] + xf[1][c] + xf[2][c]) * (1.0f / 3.0f);
        cb[c] = (yf[0][c] + yf[1][c] + yf[2][c]) * (1.0f / 3.0f);
        d2 = fmaf(ca[c] - cb[c], ca[c] - cb[c], d2);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float u = 0.0f, v = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            u = fmaf(xf[k][c] - ca[c], xf[k][c] - ca[c], u);
            v = fmaf(yf[k][c] - cb[c], yf[k][c] - cb[c], v);
        }
        ra = fmaxf(ra, u);
        rb = fmaxf(rb, v);
    }
    return fx_kb((sqrtf(d2) - sqrtf(ra) - sqrtf(rb)) * 0.99999f - 8.0f);
}

// Heights of the test triangle above the trial plane, h(s, t) = h[0] + s h[1] + t h[2]
// in units of S / 2^(the result), below 2^59 each (a height, a sum of up to three, stays
// below 2^61).  x: the test vertices relative to the trial triangle's vertex 0.  Each
// component of x and of the normal is scaled by itself: with one scale for all, heights
// were held to 2^-58 S, which loses digits of a pair of planes parallel to a coordinate
// plane (nine points, gap 1e-3 of the size: 2.8e-15 of the terms' magnitudes, FP64
// arithmetic 3.5e-16, so 3.1e-16; 1% of a double-layer matrix's time).
__device__ __forceinline__ int fx_heights(const double x[3][3], const Tri &B, int E, s64 h[3])
{
    int ex[3], en[3], top = -100000;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int m = max(max(fx_mag(x[0][c]), fx_mag(x[1][c])), fx_mag(x[2][c]));
        ex[c] = max((m >> 20) - 1022, E - 300);
        en[c] = max((fx_mag(B.n[c]) >> 20) - 1022, -100);
        top = max(top, ex[c] + en[c]);
    }
    h[0] = h[1] = h[2] = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const Fx2 n = fx_split(__double2ll_rn(B.n[c] * fx_pow2(61 - en[c])));
        const double sc = fx_pow2(61 - ex[c]);
        const int down = min(top - ex[c] - en[c], 63);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            h[k] += fx_mul_up<2>(fx_split(__double2ll_rn(x[k][c] * sc)), n) >> down;   // 2^60 / 2^top
    }
    h[2] -= h[1];
    h[1] -= h[0];
    const s64 m = (h[0] ^ (h[0] >> 63)) | (h[1] ^ (h[1] >> 63)) | (h[2] ^ (h[2] >> 63));
    const int up = __clzll(m) - 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) h[k] = up >= 0 ? h[k] << up : h[k] >> -up;
    return 60 + up - top + E;
}

// false: out of range (the caller takes the FP64 path).  BOUND: also kb (the
// single layer's sums of 1/r do without: 2^-55 of the largest possible term).  HEIGHT:
// also the heights and their unit (fx_heights).
template <bool BOUND, bool HEIGHT, bool WAVE>
__device__ __forceinline__ bool fx_pair(const Tri &A, const Tri &B, double kappa, FxPair &P, s64 h[3], int &hb)
{
    double x[3][3], y[3][3];
    int top = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int mx = 0, my = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k][c] = A.v[k][c] - B.v[0][c];
            y[k][c] = B.v[k][c] - B.v[0][c];
            mx = max(mx, fx_mag(x[k][c]));
            my = max(my, fx_mag(y[k][c]));
        }
        top = max(top, fx_mag(__hiloint2double(mx, 0) + __hiloint2double(my, 0)));
    }
    const int e = top >> 20;               // the sum is below 2^(e - 1022)
    if (e < 823 || e > 1223) return false;
    P.E = e - 1022;
    if (WAVE && fx_small_wave(kappa, P.E)) return false;
    if (HEIGHT) hb = fx_heights(x, B, P.E, h);
    const double sc = fx_pow2(61 - P.E);
    s64 X[3][3], Y[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            X[k][c] = __double2ll_rn(x[k][c] * sc);
            Y[k][c] = k == 0 ? 0 : __double2ll_rn(y[k][c] * sc);
        }
    P.kb = 4;
    if (BOUND) P.kb = fx_centroid_kb(X, Y);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        P.x0[c] = X[0][c] >> 2;
        P.a1[c] = fx_split(X[1][c] - X[0][c]);
        P.a2[c] = fx_split(X[2][c] - X[1][c]);
        P.b1[c] = fx_split(Y[1][c]);
        P.b2[c] = fx_split(Y[2][c] - Y[1][c]);
    }
    return true;
}

// v0 + s e1 + t e2 at scale 2^62 / S (v0 comes divided by 4; s, t scaled by
// 2^62): a few units of 2^-59 S
__device__ __forceinline__ s64 fx_point(s64 v0, Fx2 e1, Fx2 e2, const int32_t *s, const int32_t *t)
{
    const s64 mid = fx_mad(e1.h, s[1], fx_mad(e1.l, s[0], fx_mad(e2.h, t[1], fx_mad(e2.l, t[0], 0))));
    return fx_mad(e1.h, s[0], fx_mad(e2.h, t[0], v0 + fx_high(mid))) << 3;
}

// kb of every test point (four bits each, point 0 lowest): the powers of 1/r of the
// double layers lose 2 or 3 bits per unit of an overestimated kb.  The centroid bound is
// within a factor 2 for pairs apart; for the others (kb >= 3) the smallest distance of
// the test point to the rule's trial points in float, 7 FP32 operations per point.  One
// kb for the pair would let near test points, whose heights may vanish, cost the others
// their bits (1500 pairs with S / r from 8 to 16, root mean square error over the sum of
// the terms' magnitudes: Helmholtz double layer 4.6e-16, piecewise linear 1.6e-15; so
// 1.8e-16 and 2.6e-16; FP64 arithmetic 2.6e-16 and 3.0e-16).
template <int NP>
__device__ __forceinline__ u64 fx_near_kb(const FxPair &P, const Rule2D &R)
{
    static_assert(NP <= 16, "four bits per test point");
    float a0[3], a1[3], a2[3], b1[3], b2[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        a0[c] = 4.0f * fx_hi(P.x0[c]);
        a1[c] = (float)P.a1[c].h;
        a2[c] = (float)P.a2[c].h;
        b1[c] = (float)P.b1[c].h;
        b2[c] = (float)P.b2[c].h;
    }
    u64 kbs = 0;
#pragma unroll 1
    for (int i = 0; i < NP; ++i) {
        float x[3], lo = 3.0e38f;
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c] = fmaf(R.sf[i], a1[c], fmaf(R.tf[i], a2[c], a0[c]));
#pragma unroll 3
        for (int j = 0; j < NP; ++j) {
            float d2 = 0.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float d = fmaf(-R.sf[j], b1[c], fmaf(-R.tf[j], b2[c], x[c]));
                d2 = fmaf(d, d, d2);
            }
            lo = fminf(lo, d2);
        }
        // roundings: a few units of 2^-24 S
        kbs |= (u64)fx_kb(sqrtf(lo) * 0.9999f - 32.0f) << (4 * i);
    }
    return kbs;
}

// The same for every test point
__device__ __forceinline__ u64 fx_one_kb(int kb) { return 0x1111111111111111ull * (unsigned)kb; }
__device__ __forceinline__ int fx_kb_of(u64 kbs, int i) { return (int)(kbs >> (4 * i)) & 15; }

// T = 2^(59 - kb) S / r -> 2^(59 - 3 kb) (S / r)^3
__device__ __forceinline__ Fx2 fx_inverse_cube(Fx2 T)
{
    const Fx2 t2 = fx_split(fx_mul_up<7>(T, T));           // 2^(61 - 2 kb) (S / r)^2
    return fx_split(fx_mul_up<3>(t2, T));
}

// Trial-side sums of one test point: NM weights per trial point (the rule's
// weights, or those times the three hat functions), kernel KIND.  The sums'
// units: power 1 of 1/r 2^-(59 - kb), power 2 2^-(59 - 2 kb) and power 3
// 2^-(57 - 3 kb) (complex kinds; 2^-(59 - 3 kb) for the Laplace double layer).
template <int KIND, int NM>
struct FxInner {
    static constexpr bool HELM = kind_complex(KIND);
    static constexpr bool P1 = KIND == BEM_LAPLACE_SLP || KIND == BEM_HELMHOLTZ_SLP ||
                               KIND == BEM_HELMHOLTZ_BW;
    static constexpr bool P3 = KIND == BEM_LAPLACE_DLP || KIND == BEM_HELMHOLTZ_DLP ||
                               KIND == BEM_HELMHOLTZ_BW;
    FxSum c1[NM], s1[NM], c2[NM], s2[NM], c3[NM], s3[NM];
    template <int K1 = 0, int K3 = 0, int K = 0>
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int q = 0; q < NM; ++q) {
            c1[q].template clear<K + K1>(); s1[q].template clear<K>(); c2[q].template clear<K>();
            s2[q].template clear<K>(); c3[q].template clear<K + K3>(); s3[q].template clear<K>();
        }
    }
    __device__ __forceinline__ void point(s64 dx, s64 dy, s64 dz, int kb, Fx2 kn, int shl,
                                          const int32_t *const *w, int &flag)
    {
        const s64 r2 = fx_norm2(dx, dy, dz);
        if (KIND == BEM_LAPLACE_SLP) {
            const Fx2 T = fx_split(fx_rinv(r2, 7, flag));      // 2^55 S / r
#pragma unroll
            for (int q = 0; q < NM; ++q) c1[q].add(w[q], T);
            return;
        }
        if (!HELM) {
            const Fx2 t3 = fx_inverse_cube(fx_split(fx_rinv(r2, kb + 3, flag)));
#pragma unroll
            for (int q = 0; q < NM; ++q) c3[q].add(w[q], t3);
            return;
        }
        const Fx2 T = fx_split(fx_rinv(r2, kb, flag));     // 2^(62 - kb) S / r
        Fx2 t2, t3;
        if (P3) {
            t2 = fx_split(fx_mul_up<2>(T, T));             // 2^(62 - 2 kb) (S / r)^2
            t3 = fx_split(fx_mul(t2, T));                  // 2^(60 - 3 kb) (S / r)^3
        }
        // kappa r / (2 pi) modulo 1
        const s64 rho = fx_mul_up<4>(fx_split(r2), T);          // 2^(62 - kb) r / S
        const u64 turn = (u64)fx_shl(fx_mul(fx_split(rho), kn), shl);   // shl < 32
        s64 cs, sn;
        fx_sincos(turn, cs, sn);
        const Fx2 c = fx_split(cs), s = fx_split(sn);
        if (P1) {
            const Fx2 vc = fx_split(fx_mul(c, T)), vs = fx_split(fx_mul(s, T));
#pragma unroll
            for (int q = 0; q < NM; ++q) {
                c1[q].add(w[q], vc);
                s1[q].add(w[q], vs);
            }
        }
        if (P3) {
            const Fx2 vc2 = fx_split(fx_mul(c, t2)), vs2 = fx_split(fx_mul(s, t2));
            const Fx2 vc3 = fx_split(fx_mul(c, t3)), vs3 = fx_split(fx_mul(s, t3));
#pragma unroll
            for (int q = 0; q < NM; ++q) {
                c2[q].add(w[q], vc2);
                s2[q].add(w[q], vs2);
                c3[q].add(w[q], vc3);
                s3[q].add(w[q], vs3);
            }
        }
    }
};

// The factors that take FxInner's sums at kb to the kernel's value (without 1/(4 pi))
struct FxUnits {
    double f1, f2, f3;      // 1/r, kappa / r^2, 1/r^3 (with S for the height's unit)
    Fx2 kn;                 // kappa S / (2 pi) = kn 2^(kexp - 62)
    int shl;
    // the same at kb + n
    __device__ __forceinline__ FxUnits at(int n) const
    {
        return FxUnits{fx_scale(f1, n), fx_scale(f2, 2 * n), fx_scale(f3, 3 * n), kn, shl + n};
    }
};

template <int KIND>
__device__ __forceinline__ bool fx_units(const FxPair &P, int kb, double kappa, double eta, FxUnits &U)
{
    U.f1 = fx_pow2(1 - (59 - kb) - P.E);
    if (KIND == BEM_HELMHOLTZ_BW) U.f1 *= eta;
    U.f2 = U.f3 = 0.0;
    U.kn = Fx2{0, 0};
    U.shl = 0;
    if (KIND == BEM_LAPLACE_DLP) U.f3 = fx_pow2(1 - (59 - 3 * kb) - 2 * P.E);
    if (kind_complex(KIND)) {
        int kexp;
        if (!fx_wave(kappa, P.E, -4 - kb, kFxLeastWave, U.kn, kexp)) return false;   // shl >= 0
        U.shl = 4 + kb + kexp;
        U.f2 = kappa * fx_pow2(1 - (59 - 2 * kb) - P.E);
        U.f3 = fx_pow2(1 - (57 - 3 * kb) - 2 * P.E);
    }
    return true;
}

// FxInner's sums q -> kernel sums (re, im), times 2^K; h: height / S
template <int KIND, int NM, int K = 0>
__device__ __forceinline__ void fx_combine(const FxInner<KIND, NM> &I, int q, const FxUnits &U, double h,
                                           double &re, double &im)
{
    im = 0.0;
    if (KIND == BEM_LAPLACE_SLP) {
        re = I.c1[q].template value<K>();          // factor f1 at the end
    } else if (KIND == BEM_LAPLACE_DLP) {
        re = h * I.c3[q].template value<K>();      // factor f3 at the end
    } else if (KIND == BEM_HELMHOLTZ_SLP) {
        re = I.c1[q].template value<K>();
        im = I.s1[q].template value<K>();
    } else {
        re = h * fma(U.f3, I.c3[q].template value<K>(), U.f2 * I.s2[q].template value<K>());
        im = h * fma(U.f3, I.s3[q].template value<K>(), -U.f2 * I.c2[q].template value<K>());
        if (KIND == BEM_HELMHOLTZ_BW) {
            re = fma(U.f1, I.s1[q].template value<K>(), re);
            im = fma(-U.f1, I.c1[q].template value<K>(), im);
        }
    }
}

template <int KIND>
__device__ __forceinline__ double fx_final(const FxUnits &U)
{
    return KIND == BEM_LAPLACE_SLP || KIND == BEM_HELMHOLTZ_SLP ? U.f1
                                                                : (KIND == BEM_LAPLACE_DLP ? U.f3 : 1.0);
}

// Trial points at a time: three overlap their dependent chains with 80 registers
// and 24 warps per SM (2048-triangle dense matrix, Duffy q = 3: single layer 1.30
// ms, Brakhage-Werner 6.09; all nine points unrolled 1.39 ms, one at a time 6.24
// for the latter).  The trial points are indexed in local memory (L1).
constexpr int kFxUnroll = 3;

// Regular pair, piecewise constant: regular_p0's integral.
template <int KIND, int NP>
__device__ __forceinline__ bool fixed_p0(const Tri &A, const Tri &B, const Rule2D &R, double kappa,
                                         double &out_re, double &out_im, double eta)
{
    FxPair P;
    FxUnits U;
    s64 hs[3];
    int hb;
    if (!fx_pair<KIND != BEM_LAPLACE_SLP, kind_has_height(KIND), kind_complex(KIND)>(A, B, kappa, P, hs, hb)) return false;
    constexpr bool HEIGHT = kind_has_height(KIND);
    u64 kbs = 0;
    if (HEIGHT) kbs = P.kb >= 3 ? fx_near_kb<NP>(P, R) : fx_one_kb(P.kb);
    if (!fx_units<KIND>(P, HEIGHT ? 0 : P.kb, kappa, eta, U)) return false;
    double h[3] = {0.0, 0.0, 0.0};
    if (HEIGHT) {
#pragma unroll
        for (int k = 0; k < 3; ++k) h[k] = (double)hs[k] * fx_pow2(-hb);
    }
    s64 yx[NP], yy[NP], yz[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        yx[j] = fx_point(0, P.b1[0], P.b2[0], R.sx[j], R.tx[j]);
        yy[j] = fx_point(0, P.b1[1], P.b2[1], R.sx[j], R.tx[j]);
        yz[j] = fx_point(0, P.b1[2], P.b2[2], R.sx[j], R.tx[j]);
    }
    int bad = 0;
    double sr = 0.0, si = 0.0;
#pragma unroll 1
    for (int i = 0; i < NP; ++i) {
        const s64 xx = fx_point(P.x0[0], P.a1[0], P.a2[0], R.sx[i], R.tx[i]);
        const s64 xy = fx_point(P.x0[1], P.a1[1], P.a2[1], R.sx[i], R.tx[i]);
        const s64 xz = fx_point(P.x0[2], P.a1[2], P.a2[2], R.sx[i], R.tx[i]);
        const int kb = HEIGHT ? fx_kb_of(kbs, i) : P.kb;
        const FxUnits Ui = HEIGHT ? U.at(kb) : U;
        int flag = 0;
        FxInner<KIND, 1> I;
        I.clear();
#pragma unroll kFxUnroll
        for (int j = 0; j < NP; ++j) {
            const int32_t *w[1] = {R.wx[3][j]};
            I.point(xx - yx[j], xy - yy[j], xz - yz[j], kb, Ui.kn, Ui.shl, w, flag);
        }
        double re, im;
        fx_combine<KIND, 1>(I, 0, Ui, fma(R.t[i], h[2], fma(R.s[i], h[1], h[0])), re, im);
        bad |= flag >> (16 + kb);
        if (bad) break;
        sr = fma(KIND == BEM_LAPLACE_DLP ? fx_scale(R.w[i], 3 * kb) : R.w[i], re, sr);
        if (kind_complex(KIND)) si = fma(R.w[i], im, si);
    }
    const double scale = A.sg * B.sg * kInv4Pi * fx_final<KIND>(U);
    out_re = sr * scale;
    out_im = si * scale;
    return bad == 0;
}

// Bits that the Laplace kernels' inner sums keep below their values' unit: a sum is at
// most a twelfth of the largest value, 2^59 for both layers, and stays below 2^62.
constexpr int kFxUpS = 6, kFxUpD = 5;

// The double layer's inner sum at one test point times its height: v in [-2^61, 2^61] times
// h / 2^62, h scaled up to its own digits by 2^lz
struct FxHeight {
    Fx2 h;
    int lz;
    __device__ __forceinline__ FxHeight(s64 hi)
    {
        lz = __clzll(hi ^ (hi >> 63)) - 3;
        h = fx_split(hi << lz);
    }
    __device__ __forceinline__ double times(s64 v) const { return (double)fx_mul_up<2>(fx_split(v), h); }
};

// Regular pair, piecewise linear (3 x 3 local matrix): regular_p1's integrals.
// The outer sums of the single layer stay in fixed point (27 widening multiply-adds per
// test point).  The double layer's are FP64, three conversions and nine products per test
// point beside the integer pipe: fixed-point ones have to leave room for the largest term
// that S / r and the heights allow, which cost entries up to seven bits (1500 pairs with
// S / r from 8 to 16, root mean square error over the sum of the terms' magnitudes
// 3.1e-14, FP64 arithmetic 3.6e-16; from 2 to 4 1.8e-15, now 2.2e-16 against 2.8e-16.
// Double layer of the 2592-triangle sphere 11.3 -> 12.1 ms).
template <int KIND, int NP>
__device__ __forceinline__ bool fixed_p1(const Tri &A, const Tri &B, const Rule2D &R, double kappa,
                                         double *accr, double *acci, double eta)
{
    constexpr bool HELM = kind_complex(KIND), HEIGHT = kind_has_height(KIND);
    FxPair P;
    FxUnits U;
    double h[3] = {0.0, 0.0, 0.0};
    s64 hs[3];
    int hb;
    if (!fx_pair<KIND != BEM_LAPLACE_SLP, kind_has_height(KIND), kind_complex(KIND)>(A, B, kappa, P, hs, hb)) return false;
    u64 kbs = 0;
    if (HEIGHT) kbs = P.kb >= 3 ? fx_near_kb<NP>(P, R) : fx_one_kb(P.kb);
    if (!fx_units<KIND>(P, HEIGHT ? 0 : P.kb, kappa, eta, U)) return false;
    if (HELM && HEIGHT) {
#pragma unroll
        for (int k = 0; k < 3; ++k) h[k] = (double)hs[k] * fx_pow2(-hb);
    }
    const Fx2 h1 = fx_split(HEIGHT ? hs[1] : 0), h2 = fx_split(HEIGHT ? hs[2] : 0);
    s64 yx[NP], yy[NP], yz[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        yx[j] = fx_point(0, P.b1[0], P.b2[0], R.sx[j], R.tx[j]);
        yy[j] = fx_point(0, P.b1[1], P.b2[1], R.sx[j], R.tx[j]);
        yz[j] = fx_point(0, P.b1[2], P.b2[2], R.sx[j], R.tx[j]);
    }
    int bad = 0;
    s64 acc[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        accr[k] = acci[k] = 0.0;
        acc[k] = 0;
    }
#pragma unroll 1
    for (int i = 0; i < NP; ++i) {
        const s64 xx = fx_point(P.x0[0], P.a1[0], P.a2[0], R.sx[i], R.tx[i]);
        const s64 xy = fx_point(P.x0[1], P.a1[1], P.a2[1], R.sx[i], R.tx[i]);
        const s64 xz = fx_point(P.x0[2], P.a1[2], P.a2[2], R.sx[i], R.tx[i]);
        const int kb = HEIGHT ? fx_kb_of(kbs, i) : P.kb;
        const FxUnits Ui = HEIGHT ? U.at(kb) : U;
        int flag = 0;
        FxInner<KIND, 3> I;
        I.template clear<HELM ? 0 : kFxUpS, HELM ? 0 : kFxUpD>();
        constexpr int UN = HELM ? 1 : kFxUnroll;   // the complex sums want the registers
#pragma unroll UN
        for (int j = 0; j < NP; ++j) {
            const int32_t *w[3] = {R.wx[0][j], R.wx[1][j], R.wx[2][j]};
            I.point(xx - yx[j], xy - yy[j], xz - yz[j], kb, Ui.kn, Ui.shl, w, flag);
        }
        bad |= flag >> (16 + kb);
        if (bad) break;
        if (KIND == BEM_LAPLACE_SLP) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const Fx2 V = fx_split(I.c1[q].template sum<kFxUpS>());
#pragma unroll
                for (int p = 0; p < 3; ++p) acc[p * 3 + q] += fx_mul(Fx2{R.wx[p][i][0], R.wx[p][i][1]}, V);
            }
        } else if (KIND == BEM_LAPLACE_DLP) {
            const FxHeight H(fx_point(hs[0] >> 2, h1, h2, R.sx[i], R.tx[i]) >> 1);   // S / 2^hb
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const double v = H.times(I.c3[q].template sum<kFxUpD>());
#pragma unroll
                for (int p = 0; p < 3; ++p) accr[p * 3 + q] = fma(fx_scale(R.wd[p][i], 3 * kb - H.lz), v, accr[p * 3 + q]);
            }
        } else {
            const double hi = fma(R.t[i], h[2], fma(R.s[i], h[1], h[0]));
            double re[3], im[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) fx_combine<KIND, 3>(I, q, Ui, hi, re[q], im[q]);
#pragma unroll
            for (int p = 0; p < 3; ++p)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    accr[p * 3 + q] = fma(R.wd[p][i], re[q], accr[p * 3 + q]);
                    acci[p * 3 + q] = fma(R.wd[p][i], im[q], acci[p * 3 + q]);
                }
        }
    }
    double scale = A.sg * B.sg * kInv4Pi * fx_final<KIND>(U);
    // the single layer's outer sums: half, kFxUpS bits up; the double layer's: the product's
    // 2^62, the heights' 2^hb and kFxUpD
    if (KIND == BEM_LAPLACE_SLP) scale *= fx_pow2(1 - kFxUpS);
    if (KIND == BEM_LAPLACE_DLP) scale *= fx_pow2(62 - kFxUpD - hb);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        accr[k] = KIND == BEM_LAPLACE_SLP ? (double)acc[k] * scale : accr[k] * scale;
        if (HELM) acci[k] *= scale;
    }
    return bad == 0;
}

// Both Laplace layers of a regular pair, piecewise linear (two 3 x 3 local
// matrices): fixed_p1's integrals, sharing points, distances and reciprocal square
// roots, which are 70 of the 110 instructions of a point of either.  Every layer
// gets the bits of fixed_p1 (a single call and a plan give the same matrix).  Plan of
// the 1352-triangle sphere, nine points: 4.77 ms for the layers apart, 3.8 fused.
template <int NP>
__device__ __forceinline__ bool fixed_p1_fused(const Tri &A, const Tri &B, const Rule2D &R, double *accs,
                                               double *accd)
{
    FxPair P;
    s64 hs[3];
    int hb;
    if (!fx_pair<true, true, false>(A, B, 0.0, P, hs, hb)) return false;
    const u64 kbs = P.kb >= 3 ? fx_near_kb<NP>(P, R) : fx_one_kb(P.kb);
    const s64 h0 = hs[0] >> 2;
    const Fx2 h1 = fx_split(hs[1]), h2 = fx_split(hs[2]);
    s64 yx[NP], yy[NP], yz[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        yx[j] = fx_point(0, P.b1[0], P.b2[0], R.sx[j], R.tx[j]);
        yy[j] = fx_point(0, P.b1[1], P.b2[1], R.sx[j], R.tx[j]);
        yz[j] = fx_point(0, P.b1[2], P.b2[2], R.sx[j], R.tx[j]);
    }
    int bad = 0;
    s64 as[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        as[k] = 0;
        accd[k] = 0.0;
    }
#pragma unroll 1
    for (int i = 0; i < NP; ++i) {
        const s64 xx = fx_point(P.x0[0], P.a1[0], P.a2[0], R.sx[i], R.tx[i]);
        const s64 xy = fx_point(P.x0[1], P.a1[1], P.a2[1], R.sx[i], R.tx[i]);
        const s64 xz = fx_point(P.x0[2], P.a1[2], P.a2[2], R.sx[i], R.tx[i]);
        const int kb = fx_kb_of(kbs, i);
        int flag = 0;
        FxSum cs[3], cd[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            cs[q].template clear<kFxUpS>();
            cd[q].template clear<kFxUpD>();
        }
#pragma unroll kFxUnroll
        for (int j = 0; j < NP; ++j) {
            const s64 r2 = fx_norm2(xx - yx[j], xy - yy[j], xz - yz[j]);
            const s64 inv = fx_rinv(r2, kb + 3, flag);                   // 2^(59 - kb) S / r
            const Fx2 T = fx_split(fx_sar(inv, 4 - kb));                 // 2^55 S / r
            const Fx2 t3 = fx_inverse_cube(fx_split(inv));
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                cs[q].add(R.wx[q][j], T);
                cd[q].add(R.wx[q][j], t3);
            }
        }
        bad |= flag >> (16 + kb);
        const FxHeight H(fx_point(h0, h1, h2, R.sx[i], R.tx[i]) >> 1);   // S / 2^hb
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const Fx2 vs = fx_split(cs[q].template sum<kFxUpS>());
            const double vd = H.times(cd[q].template sum<kFxUpD>());
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                as[p * 3 + q] += fx_mul(Fx2{R.wx[p][i][0], R.wx[p][i][1]}, vs);
                accd[p * 3 + q] = fma(fx_scale(R.wd[p][i], 3 * kb - H.lz), vd, accd[p * 3 + q]);
            }
        }
    }
    // a rule's weights come at 2^63: factor 2 per sum
    const double sc = A.sg * B.sg * kInv4Pi;
    const double fs = sc * fx_pow2(1 - 55 - P.E) * fx_pow2(1 - kFxUpS);
    const double fd = sc * fx_pow2(1 - 59 - 2 * P.E) * fx_pow2(62 - kFxUpD - hb);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        accs[k] = (double)as[k] * fs;
        accd[k] *= fd;
    }
    return bad == 0;
}

}  // namespace bem
