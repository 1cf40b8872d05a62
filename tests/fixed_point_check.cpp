// The fixed-point arithmetic of bem_fixed.cuh on the host, against long double:
// prints the largest errors of the squared length (units), the reciprocal
// square root (relative, for every bound 2^kb of S / r), and the sine and cosine.
#include <cmath>
#include <cstdio>
#include <random>

#include "bem_fixed.cuh"

using namespace bem;

int main()
{
    std::mt19937_64 g(7);
    auto uni = [&]() { return (long double)(g() >> 11) / 9007199254740992.0L; };
    long double norm = 0.0L;
    for (int i = 0; i < 400000; ++i) {
        const int sh = (int)(g() % 6);
        const s64 x = (s64)g() >> (1 + sh), y = (s64)g() >> (1 + sh), z = (s64)g() >> (1 + sh);
        const long double e = fx_norm2(x, y, z) -
                              ((long double)x * x + (long double)y * y + (long double)z * z) / 18446744073709551616.0L;
        norm = std::max(norm, std::fabs(e));
    }
    std::printf("norm2 %.3Lg\n", norm);
    for (int kb = 0; kb <= 4; ++kb) {
        long double worst = 0.0L;
        int flagged = 0;
        for (int i = 0; i < 400000; ++i) {
            // r / S from the bound's edge to sqrt(3)
            const long double r = std::exp2(-(long double)kb + uni() * (kb + 0.79L));
            const s64 r2 = (s64)(r * r * 1152921504606846976.0L);
            int flag = 0;
            const s64 t = fx_rinv(r2, kb, flag);
            if (flag >> (16 + kb)) {
                ++flagged;
                continue;
            }
            const long double ref = std::exp2(62.0L - kb) / std::sqrt((long double)r2 / 1152921504606846976.0L);
            worst = std::max(worst, std::fabs((t - ref) / ref));
        }
        std::printf("rinv%d %.3Lg %d\n", kb, worst, flagged);
    }
    int flag = 0, seen = 0;
    for (s64 r2 : {(s64)0, (s64)1, (s64)1 << 40, ((s64)1 << 52) - ((s64)1 << 34)}) {
        flag = 0;
        fx_rinv(r2, 4, flag);
        seen += (flag >> 20) != 0;
    }
    std::printf("flags %d\n", seen);
    long double cs = 0.0L;
    for (int i = 0; i < 400000; ++i) {
        // every other one near a multiple of an eighth of a turn
        u64 t = g();
        if (i & 1) t = (u64)(g() % 8) * ((u64)1 << 61) + (u64)((s64)(g() % 2001) - 1000);
        s64 c, s;
        fx_sincos(t, c, s);
        const long double a = 6.283185307179586476925286766559005768L * ((long double)t / 18446744073709551616.0L);
        cs = std::max(cs, std::max(std::fabs(c / 2305843009213693952.0L - std::cos(a)),
                                   std::fabs(s / 2305843009213693952.0L - std::sin(a))));
    }
    std::printf("sincos %.3Lg\n", cs);
}
