// 64-bit fixed-point arithmetic for the FP64 form's quadrature points.
//
// The FP64 pipe of sm_103a retires 2 lanes per SM and cycle (measured: 1.6
// DFMA), the integer pipe 64 widening 32 x 32 + 64 multiply-adds (60 measured)
// and 128 additions, so one FP64 operation costs as much as 30 to 70 integer
// ones.  A quadrature point needs a difference of points, a squared distance,
// a reciprocal square root and a weighted sum: 13 FP64 operations for the single
// layer, about 60 with a sine and cosine.  Here the points of a pair are
// integers scaled to the pair (62 bits), and a single layer's point takes 90
// instructions (34 of them multiply-adds) instead of 13 on the FP64 pipe, each
// worth 64.  Bound by instruction issue: 0.6 of the issue slots, the ALU pipe half
// busy, the multiplier 0.45 (2048 triangles, nine points: 8.82 ms on the FP64 pipe, 1.30 so).
//
// Precision: a coordinate carries an absolute error of a few 2^-59 S, S = the
// power of two above the largest coordinate difference of the pair; FP64
// arithmetic on the same differences carries 2^-53 S.  The squared distance is
// held to 2^-60 S^2, the reciprocal distance to 2^-54 of itself.  The
// distances of a pair must stay above S / 16 (fx_rinv flags smaller ones, and
// the caller evaluates that pair in FP64); disjoint pairs of shape-regular
// meshes keep S / r below 8 or so.
//
// Host compilable (tests of the arithmetic on the CPU).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <cmath>

namespace bem {

#define BEM_HD __host__ __device__ __forceinline__

typedef long long s64;
typedef unsigned long long u64;

// h 2^32 + l with l signed: products of two such numbers need signed 32 x 32
// multiplications only.
struct Fx2 {
    int h, l;
};

// 64-bit words from and to their halves, and the steps below, spelled out: from the
// plain 64-bit expressions the compiler makes full 64-bit products wherever an
// operand is part of a word, and shifts of both halves (a Helmholtz point of the
// Brakhage-Werner operator took 1.4 times the instructions).
BEM_HD int fx_high(s64 a)
{
#ifdef __CUDA_ARCH__
    int l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(a));
    return h;
#else
    return (int)(a >> 32);
#endif
}

BEM_HD unsigned fx_low(s64 a) { return (unsigned)(u64)a; }

BEM_HD s64 fx_join(unsigned l, int h)
{
#ifdef __CUDA_ARCH__
    s64 a;
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "r"(l), "r"(h));
    return a;
#else
    return (s64)(((u64)(unsigned)h << 32) | l);
#endif
}

// upper word of (h : l) << n, lower word of (h : l) >> n, 0 <= n < 32
BEM_HD unsigned fx_funnel_l(unsigned l, unsigned h, int n)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_l(l, h, n);
#else
    return (unsigned)((((u64)h << 32 | l) << n) >> 32);
#endif
}

BEM_HD unsigned fx_funnel_r(unsigned l, unsigned h, int n)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_r(l, h, n);
#else
    return (unsigned)(((u64)h << 32 | l) >> n);
#endif
}

// a 2^n modulo 2^64, 0 <= n < 32
BEM_HD s64 fx_shl(s64 a, int n)
{
    return fx_join(fx_low(a) << n, (int)fx_funnel_l(fx_low(a), (unsigned)fx_high(a), n));
}

// a / 2^n rounded down, 0 <= n < 32
BEM_HD s64 fx_sar(s64 a, int n)
{
    return fx_join(fx_funnel_r(fx_low(a), (unsigned)fx_high(a), n), fx_high(a) >> n);
}

BEM_HD Fx2 fx_split(s64 a)
{
    Fx2 r;
    r.l = (int)fx_low(a);
    r.h = fx_high(a) + (int)(fx_low(a) >> 31);
    return r;
}

// a b + c in one widening multiply-add
BEM_HD s64 fx_mad(int a, int b, s64 c)
{
#ifdef __CUDA_ARCH__
    s64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (s64)a * (s64)b + c;
#endif
}

BEM_HD u64 fx_madu(unsigned a, unsigned b, u64 c)
{
#ifdef __CUDA_ARCH__
    u64 d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (u64)a * (u64)b + c;
#endif
}

// a b / 2^64 rounded, the product of the low words dropped (at most a quarter
// unit); |a.h|, |b.h| <= 2^30 keep the middle sum within 64 bits
BEM_HD s64 fx_mul(Fx2 a, Fx2 b)
{
    const s64 mid = fx_mad(a.h, b.l, fx_mad(a.l, b.h, (s64)1 << 31));
    return fx_mad(a.h, b.h, fx_high(mid));
}

// a b / 2^(64 - K): K more bits of the same product (which must fit)
template <int K>
BEM_HD s64 fx_mul_up(Fx2 a, Fx2 b)
{
    const s64 mid = fx_mad(a.h, b.l, fx_mad(a.l, b.h, (s64)1 << (31 - K)));
    const s64 p = fx_mad(a.h, b.h, fx_high(mid));
    return fx_join(fx_funnel_l(fx_low(mid), fx_low(p), K),
                   (int)fx_funnel_l(fx_low(p), (unsigned)fx_high(p), K));
}

// the same, 0 <= n < 32 bits
BEM_HD s64 fx_mul_up(Fx2 a, Fx2 b, int n)
{
    const s64 mid = fx_mad(a.h, b.l, fx_mad(a.l, b.h, (s64)(1u << (31 - n))));
    const s64 p = fx_mad(a.h, b.h, fx_high(mid));
    return fx_join(fx_funnel_l(fx_low(mid), fx_low(p), n),
                   (int)fx_funnel_l(fx_low(p), (unsigned)fx_high(p), n));
}

BEM_HD int fx_float_bits(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_int(f);
#else
    int i;
    memcpy(&i, &f, 4);
    return i;
#endif
}

BEM_HD float fx_rsqrt_estimate(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / sqrtf(x);
#endif
}

BEM_HD int fx_round(float x)
{
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return (int)lrintf(x);
#endif
}

// Squared length of (x, y, z), |x|, |y|, |z| <= 2^62: the sum of squares / 2^64
// (the squares of the low words dropped: below one unit), at most 3 2^60.
BEM_HD s64 fx_norm2(s64 x, s64 y, s64 z)
{
    const Fx2 a = fx_split(x), b = fx_split(y), c = fx_split(z);
    const s64 hl = fx_mad(a.h, a.l, fx_mad(b.h, b.l, fx_mad(c.h, c.l, (s64)1 << 30)));
    const int h = fx_high(hl);
    const s64 two = fx_join(fx_funnel_l(fx_low(hl), (unsigned)h, 1), h >> 31);   // hl / 2^31
    return fx_mad(a.h, a.h, fx_mad(b.h, b.h, fx_mad(c.h, c.h, two)));
}

// Reciprocal square root: r2 = 2^60 (r / S)^2 -> 2^(62 - kb) S / r, given
// S / r <= 2^kb, 0 <= kb <= 4.  A 20-bit estimate m of 2^16 S / r (hardware
// reciprocal square root, rounded by adding 12, whose ulp is 2^-20) has the
// residual E = 1 - r2 m^2 / 2^92 with |E| < 2^-15, formed exactly to 2^-60;
// (1 - E)^(-1/2) = 1 + E/2 + 3/8 E^2 + 5/16 E^3 + ... corrects it, the second
// and third terms in float (they are below 2^-31, so 24 bits leave 2^-56).
// flag collects the estimates: any bit from 2^20 on means a distance below
// S / 16 (or a zero one), where the result is meaningless.
BEM_HD s64 fx_rinv(s64 r2, int kb, int &flag)
{
    const unsigned rl = fx_low(r2), rh = (unsigned)fx_high(r2);
    const float y = fx_rsqrt_estimate((float)(int)rh);
    const float g = y * 1024.0f + 12.0f;
    const unsigned m = (unsigned)(fx_float_bits(g) - 0x41400000);
    flag |= (int)m;
    const u64 q = fx_madu(m, m, 0);
    const unsigned ql = (unsigned)q, qh = (unsigned)(q >> 32);
    // r2 q / 2^32 modulo 2^64 (it is 2^60 (1 - E))
    u64 b = fx_madu(rh, ql, (unsigned)fx_high((s64)fx_madu(rl, ql, 0)));
    b = fx_madu(rl, qh, b);
    b = (u64)fx_join(fx_low((s64)b), fx_high((s64)b) + (int)(rh * qh));
    const s64 E = (s64)(((u64)1 << 60) - b);
    const float e = (float)(int)fx_funnel_r(fx_low(E), (unsigned)fx_high(E), 15);   // E 2^45
    // 2 c = E + 3/4 E^2 + 5/8 E^3 in units of 2^-60
    const float k2 = e * (float)(0.625 / 1073741824.0 / 35184372088832.0) + (float)(0.75 / 1073741824.0);
    const s64 C = fx_mad(fx_round((e * e) * k2), 1, E);
    // m (1 + c) 2^(46 - kb)
    const s64 mc = (s64)fx_madu(m, fx_low(C), (u64)fx_join(0, (int)(m * (unsigned)fx_high(C))));
    return fx_join(fx_funnel_r(fx_low(mc), (unsigned)fx_high(mc), 15 + kb),
                   (fx_high(mc) >> (15 + kb)) + (int)(m << (14 - kb)));
}

// Cosine and sine of `turn` (2^64 = one turn), scaled by 2^61: the table's multiple
// of 1/128 turn next to it, rotated by the remainder, at most beta = pi / 128, whose
// series are short: with u = remainder / beta and z = u^2
//   sin / u = beta - z (beta^3 / 6 - z (beta^5 / 120 - z beta^7 / 5040))
//   1 - cos = z (beta^2 / 2 - z (beta^4 / 24 - z (beta^6 / 720 - z beta^8 / 40320)))
// truncated below 2^-59, the inner steps in 32 bits.  76 instructions; Taylor
// polynomials to the 17th power on an eighth of a turn took 112 (Helmholtz single
// layer of 2048 triangles: 4.42 ms, now 4.07; absolute error 2.8e-17, now 7.7e-18).
constexpr s64 kFxCos[33] = {   // cos(2 pi k / 128) 2^61
    2305843009213693952ll, 2303065520325098980ll, 2294739744873325982ll,
    2280885740380690081ll, 2261536882357481515ll, 2236739783897437994ll,
    2206554183382719070ll, 2171052800568911040ll, 2130321161396766249ll,
    2084457391952720625ll, 2033571982074556626ll, 1977787519171706257ll,
    1917238392901444355ll, 1852070471412433076ll, 1782440749935575221ll,
    1708516972568751838ll, 1630477228166597777ll, 1548509521308852131ll,
    1462811319380858392ll, 1373589076857337057ll, 1281057737935472749ll,
    1185440218715516311ll, 1086966870176374159ll, 985874923239923734ll,
    882407917260943721ll, 776815113319476863ll, 669350893729055444ll,
    560274149207426732ll, 449847655186137774ll, 338337438761504393ll,
    226012137812034940ll, 113142353826251070ll, 0ll,
};
constexpr s64 kFxB1 = 452751216129820178ll, kFxB3 = 2840980145336ll;             // beta 2^64, beta^3 / 6 2^60
constexpr int kFxB5 = 342277223, kFxB7 = 19637;                         // beta^5 / 120 2^62, beta^7 / 5040 2^64
constexpr s64 kFxD2 = 5556093337880030ll;                             // beta^2 / 2 2^64
constexpr unsigned kFxD4 = 2179004481u;                              // beta^4 / 24 2^57
constexpr int kFxD6 = 1400124, kFxD8 = 60;                             // beta^6 / 720 2^62, beta^8 / 40320 2^64

struct FxTurns {
    s64 cs[128][2];   // cosine, sine of k / 128 turn
};

constexpr FxTurns fx_turns()
{
    FxTurns t = {};
    for (int k = 0; k < 128; ++k)
        for (int q = 0; q < 2; ++q) {
            const int j = (k + (q ? 96 : 0)) % 128;      // sin x = cos(x - 1/4 turn)
            const int m = j > 64 ? 128 - j : j;
            t.cs[k][q] = m <= 32 ? kFxCos[m] : -kFxCos[64 - m];
        }
    return t;
}
#ifdef __CUDACC__
__device__ constexpr FxTurns kFxTurnsDev = fx_turns();
#endif
static constexpr FxTurns kFxTurnsHost = fx_turns();

BEM_HD unsigned fx_mulhi(unsigned a, unsigned b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (unsigned)(((u64)a * b) >> 32);
#endif
}

// (a x + b y) / 2^64 rounded
BEM_HD s64 fx_mul2(Fx2 a, Fx2 x, Fx2 b, Fx2 y)
{
    const s64 mid = fx_mad(a.h, x.l, fx_mad(a.l, x.h, fx_mad(b.h, y.l, fx_mad(b.l, y.h, (s64)1 << 31))));
    return fx_mad(a.h, x.h, fx_mad(b.h, y.h, fx_high(mid)));
}

BEM_HD void fx_sincos(u64 turn, s64 &c, s64 &s)
{
    const unsigned tl = fx_low((s64)turn), th = (unsigned)fx_high((s64)turn);
    const unsigned k = (th + (1u << 24)) >> 25;
    const unsigned dh = th - (k << 25);
    // remainder, 2^62 = beta
    const Fx2 xs = fx_split(fx_join(tl << 6, (int)fx_funnel_l(tl, dh, 6)));
#ifdef __CUDA_ARCH__
    const longlong2 e = __ldg(reinterpret_cast<const longlong2 *>(kFxTurnsDev.cs[k & 127]));
    const s64 C = e.x, S = e.y;
#else
    const s64 C = kFxTurnsHost.cs[k & 127][0], S = kFxTurnsHost.cs[k & 127][1];
#endif
    const s64 z = fx_mul_up<2>(xs, xs);                                // u^2 2^62
    const Fx2 zs = fx_split(z);
    const unsigned z30 = (unsigned)fx_high(z), z31 = fx_funnel_l(fx_low(z), z30, 1);
    // sine 2^64
    const unsigned q5 = (unsigned)kFxB5 - fx_mulhi((unsigned)kFxB7, z30);
    const Fx2 w = fx_split(kFxB3 - (s64)fx_mulhi(q5, z30));           // 2^60
    const Fx2 sb = fx_split(kFxB1 - fx_mul_up<6>(w, zs));
    const s64 sv = fx_mul_up<2>(sb, xs);
    const Fx2 sa = fx_split(sv), sn = fx_split(-sv);
    // 1 - cosine 2^64
    const unsigned q6 = (unsigned)kFxD6 - fx_mulhi((unsigned)kFxD8, z30);
    const unsigned r = kFxD4 - (fx_mulhi(q6, z30) >> 3);               // 2^57
    const u64 rz = fx_madu(r, z31, 0);                                 // 2^88
    const s64 d = kFxD2 - fx_join(fx_funnel_r((unsigned)rz, (unsigned)(rz >> 32), 24), (int)((unsigned)(rz >> 32) >> 24));
    const Fx2 cm = fx_split(fx_mul_up<2>(fx_split(d), zs));
    const Fx2 Cs = fx_split(C), Ss = fx_split(S);
    c = C - fx_mul2(Cs, cm, Ss, sa);
    s = S - fx_mul2(Ss, cm, Cs, sn);
}

}  // namespace bem
