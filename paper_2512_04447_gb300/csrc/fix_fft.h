// Fixed-point arithmetic of the FP64 transforms (fft_fix.cu): complex values as pairs of 64-bit
// integers with one exponent per block.
//
// GB300 issues a warp's FP64 instruction in 64 cycles of its sub-partition and integer
// instructions in 2 to 4, so a 64-bit integer addition (2 instructions) costs a fifteenth of an
// FP64 one and a complex product with a twiddle factor (12 multiply-adds of 32 x 32 -> 64 bits)
// a third.  Values are kept below 2^62.5 in magnitude.  Before every stage the block is shifted to
// the largest scale at which the stage's sums cannot overflow, by the bits that its values
// really have, so that a rounding error is one unit of some 2^-58 of the block's largest value at
// each stage, where the FP64 transform rounds to 2^-53 of each value at each addition.
// Host and device, so that it can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define FIX_HD __host__ __device__ __forceinline__
#else
#define FIX_HD inline
#endif

namespace rsdft {
namespace fix {

typedef long long i64;
typedef unsigned long long u64;

struct I2 {
    i64 x, y;
};
struct W4 {          // a factor w of magnitude <= 1: round(w 2^62) = h 2^32 + l with signed l
    int rh, rl, ih, il;
};

constexpr int TOP = 62;   // components are at most 2^TOP before the sums of a stage are formed, 2^62.5 after

FIX_HD I2 add(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
FIX_HD I2 sub(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
template <bool INV> FIX_HD I2 rot(I2 a) { return INV ? I2{-a.y, a.x} : I2{a.y, -a.x}; }   // times -+i

FIX_HD int lo_of(i64 v) { return (int)(unsigned)v; }
FIX_HD int hi_of(i64 v) { return (int)((v + 0x80000000ll) >> 32); }   // v = hi 2^32 + (signed) lo
FIX_HD i64 mw(int a, int b, i64 c) { return (i64)a * b + c; }         // 32 x 32 + 64 -> 64

// v >> s to nearest, ties to even (0 <= s < 63): rounding ties one way would add up coherently over a
// block and come out of the inverse transform in a few points
FIX_HD i64 rshift(i64 v, int s) { return s > 0 ? (v + ((v >> s) & 1) + (((i64)1 << (s - 1)) - 1)) >> s : v; }
FIX_HD I2 rshift(I2 v, int s) { return I2{rshift(v.x, s), rshift(v.y, s)}; }

// v w / 4 (CONJ: v conj(w) / 4) for |v| < 2^62.5; the product of the low words is left out.  The sums of
// the mixed products stay below 2^62.8: |xl rh| + |yl ih| <= 2^31 sqrt(2) 2^30 and
// |xh rl| + |yh il| <= sqrt(2) 2^30.5 2^31.
template <bool CONJ> FIX_HD I2 mul_w(I2 v, W4 w) {
    const int xl = lo_of(v.x), xh = hi_of(v.x), yl = lo_of(v.y), yh = hi_of(v.y);
    const i64 half = 0x80000000ll;
    const i64 a = mw(xl, w.rh, mw(xh, w.rl, half)), b = mw(yl, w.ih, mw(yh, w.il, 0));
    const i64 c = mw(xl, w.ih, mw(xh, w.il, CONJ ? 0 : half)), d = mw(yl, w.rh, mw(yh, w.rl, CONJ ? half : 0));
    if (CONJ) return I2{mw(xh, w.rh, mw(yh, w.ih, (a + b) >> 32)), mw(yh, w.rh, 0) - mw(xh, w.ih, 0) + ((d - c) >> 32)};
    return I2{mw(xh, w.rh, 0) - mw(yh, w.ih, 0) + ((a - b) >> 32), mw(xh, w.ih, mw(yh, w.rh, (c + d) >> 32))};
}

// v c for a constant 0 < c < 1 given as round(c 2^63) = ch 2^32 + cl, signed cl; |v| < 2^62.5
FIX_HD i64 mul_c(i64 v, int ch, int cl) {
    const int l = lo_of(v), h = hi_of(v);
    return (mw(h, ch, 0) << 1) + (mw(l, ch, mw(h, cl, 0x40000000ll)) >> 31);
}
FIX_HD I2 mul_c(I2 v, int ch, int cl) { return I2{mul_c(v.x, ch, cl), mul_c(v.y, ch, cl)}; }
constexpr i64 split_c(long double c) { return (i64)(c * 9223372036854775808.0L + 0.5L); }
constexpr int const_h(long double c) { return (int)((split_c(c) + 0x80000000ll) >> 32); }
constexpr int const_l(long double c) { return (int)(unsigned)split_c(c); }
#define FIX_C(c) const_h(c), const_l(c)

constexpr long double SQRT3_2 = 0.866025403784438646763723170753L, SQRT1_2 = 0.707106781186547524400844362105L,
                      C1_5 = 0.309016994374947424102293417183L, C2_5 = 0.809016994374947424102293417183L,
                      S1_5 = 0.951056516295153572116439333379L, S2_5 = 0.587785252292473129168705954639L;

// sums grow by at most R: bits provided for
FIX_HD constexpr int growth(int r) { return r <= 2 ? 1 : (r <= 4 ? 2 : 3); }

template <int R, bool INV> FIX_HD void dft(I2 *v) {
    if constexpr (R == 2) {
        const I2 a = v[0], b = v[1];
        v[0] = add(a, b);
        v[1] = sub(a, b);
    } else if constexpr (R == 3) {
        const I2 t1 = add(v[1], v[2]);
        const I2 t2 = sub(v[0], rshift(t1, 1));
        const I2 r = rot<INV>(mul_c(sub(v[1], v[2]), FIX_C(SQRT3_2)));
        v[0] = add(v[0], t1);
        v[1] = add(t2, r);
        v[2] = sub(t2, r);
    } else if constexpr (R == 4) {
        const I2 a0 = add(v[0], v[2]), a1 = sub(v[0], v[2]);
        const I2 a2 = add(v[1], v[3]), a3 = rot<INV>(sub(v[1], v[3]));
        v[0] = add(a0, a2);
        v[2] = sub(a0, a2);
        v[1] = add(a1, a3);
        v[3] = sub(a1, a3);
    } else if constexpr (R == 5) {
        const I2 a1 = add(v[1], v[4]), b1 = sub(v[1], v[4]), a2 = add(v[2], v[3]), b2 = sub(v[2], v[3]), x0 = v[0];
        v[0] = add(x0, add(a1, a2));
        const I2 r1 = add(x0, sub(mul_c(a1, FIX_C(C1_5)), mul_c(a2, FIX_C(C2_5))));
        const I2 r2 = add(x0, sub(mul_c(a2, FIX_C(C1_5)), mul_c(a1, FIX_C(C2_5))));
        const I2 i1 = rot<INV>(add(mul_c(b1, FIX_C(S1_5)), mul_c(b2, FIX_C(S2_5))));
        const I2 i2 = rot<INV>(sub(mul_c(b1, FIX_C(S2_5)), mul_c(b2, FIX_C(S1_5))));
        v[1] = add(r1, i1);
        v[4] = sub(r1, i1);
        v[2] = add(r2, i2);
        v[3] = sub(r2, i2);
    } else {
        I2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft<4, INV>(e);
        dft<4, INV>(o);
        const I2 o1 = o[1], o3 = o[3];
        o[1] = mul_c(add(o1, rot<INV>(o1)), FIX_C(SQRT1_2));
        o[2] = rot<INV>(o[2]);
        o[3] = mul_c(sub(rot<INV>(o3), o3), FIX_C(SQRT1_2));
        for (int p = 0; p < 4; ++p) {
            v[p] = add(e[p], o[p]);
            v[p + 4] = sub(e[p], o[p]);
        }
    }
}

// bits of |v|
FIX_HD int bits_of(u64 v) {
#ifdef __CUDA_ARCH__
    return 64 - __clzll((long long)v);
#else
    return v ? 64 - __builtin_clzll(v) : 0;
#endif
}

// The double with these words as an integer of units 2^-s (|x| 2^s <= 2^62), rounded
FIX_HD i64 from_double(int hi, unsigned lo, int s) {
    const int e = (hi >> 20) & 0x7ff;
    u64 m = ((u64)(unsigned)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 42) | ((u64)lo << 10);   // 2^62 <= m < 2^63
    int r = 1085 - e - s;   // x 2^s = m 2^-r
    if (e == 0) {           // subnormal: the same with its leading bit brought there
        const int k = m ? 63 - bits_of(m) : 0;
        m <<= k;
        r += k - 1;
    }
    r = r < 1 ? 1 : (r > 63 ? 63 : r);
    const i64 v = (i64)((m + (1ull << (r - 1))) >> r);
    return hi < 0 ? -v : v;
}

// The high and low words of v 2^e as a double, to nearest even; exponents beyond the normal range
// are told by *odd (the caller scales v by other means)
FIX_HD u64 to_double_bits(i64 v, int e, bool *odd) {
    *odd = false;
    if (v == 0) return 0;
    const u64 a = v < 0 ? (u64)-v : (u64)v;
    const int lz = 64 - bits_of(a);
    const u64 t = a << lz, rest = t & 0x7ff;
    u64 r = t >> 11;                                   // 2^52 <= r < 2^53
    r += rest > 0x400 || (rest == 0x400 && (r & 1));
    const int field = 1023 + 63 - lz + e;
    if (field < 1 || field > 2045) *odd = true;
    return (((u64)(unsigned)(field - 1) << 52) + r) | (v < 0 ? 0x8000000000000000ull : 0ull);
}

}  // namespace fix
}  // namespace rsdft
