// Host build of the fixed-point transform arithmetic (csrc/fix_fft.h): the largest error of each
// piece in units of its last place against long double, over seeded random operands.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <random>

#include "fix_fft.h"

using namespace rsdft::fix;
typedef long double ld;
typedef std::complex<ld> C;

static std::mt19937_64 g(1);
static i64 draw(int bits) { return (i64)(g() >> (64 - bits)) - ((i64)1 << (bits - 1)); }
static const ld PI = 3.14159265358979323846264338327950288L;

template <int R, bool INV> static double dft_error() {
    double worst = 0;
    for (int it = 0; it < 2000; ++it) {
        I2 v[R];
        C x[R];
        for (int i = 0; i < R; ++i) {
            v[i] = I2{draw(59), draw(59)};   // the largest that a radix-8 stage takes
            x[i] = C(v[i].x, v[i].y);
        }
        dft<R, INV>(v);
        for (int p = 0; p < R; ++p) {
            C s = 0;
            for (int q = 0; q < R; ++q) s += x[q] * std::polar((ld)1, (INV ? 1 : -1) * 2 * PI * ((p * q) % R) / R);
            worst = std::max(worst, (double)std::abs(s - C(v[p].x, v[p].y)));
        }
    }
    return worst;
}

int main() {
    std::printf("dft2 %g\ndft3 %g\ndft4 %g\ndft5 %g\ndft8 %g\n", dft_error<2, false>(), dft_error<3, false>(),
                dft_error<4, true>(), dft_error<5, true>(), dft_error<8, false>());
    double mul = 0, conj = 0, con = 0, from = 0, to = 0, shift = 0, bias = 0;
    for (int it = 0; it < 100000; ++it) {
        const ld t = 2 * PI * (g() % 997) / 997;
        const i64 c = llroundl(cosl(t) * 0x1p62L), s = llroundl(sinl(t) * 0x1p62L);
        const W4 w{hi_of(c), lo_of(c), hi_of(s), lo_of(s)};
        const I2 v{draw(62), draw(62)};
        const C z(v.x, v.y), u((ld)c * 0x1p-62L, (ld)s * 0x1p-62L);
        const I2 a = mul_w<false>(v, w), b = mul_w<true>(v, w);
        mul = std::max(mul, (double)std::abs(z * u / (ld)4 - C(a.x, a.y)));
        conj = std::max(conj, (double)std::abs(z * std::conj(u) / (ld)4 - C(b.x, b.y)));
        con = std::max(con, (double)fabsl((ld)v.x * SQRT1_2 - mul_c(v.x, FIX_C(SQRT1_2))));
        const double d = std::ldexp((double)draw(53), (int)(g() % 9) - 30);
        long long bits;
        std::memcpy(&bits, &d, 8);
        const i64 f = from_double((int)(bits >> 32), (unsigned)bits, 30);
        from = std::max(from, (double)fabsl((ld)f - ldexpl((ld)d, 30)));
        bool odd = false;
        const u64 o = to_double_bits(v.x, -77, &odd);
        double back;
        std::memcpy(&back, &o, 8);
        to = std::max(to, std::fabs(back - std::ldexp((double)v.x, -77)));
        to_double_bits(v.x, -1200, &odd);
        if (!odd) to = 1e300;
        const i64 q = v.x >> 50;
        const int sh = 1 + (int)(g() % 4);
        shift = std::max(shift, std::fabs((double)rshift(q, sh) - std::ldexp((double)q, -sh)));
        bias += (double)rshift(q, 1) - 0.5 * (double)q;
    }
    std::printf("mul %g\nconj %g\nconst %g\nfrom %g\nto %g\nshift %g\nbias %g\n", mul, conj, con, from, to, shift,
                std::fabs(bias) / 100000);
    return 0;
}
