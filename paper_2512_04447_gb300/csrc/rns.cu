// FP64 Gram matrices and rotations on the tensor cores by residue arithmetic.
//
// GB300 issues FP64 at 4 flop/clk/SM and BF16 MMAs at some 8,200, so an FP64 product
// of matrices is cheapest as exact integer arithmetic on the tensor cores (the
// residue-number form of the Ozaki scheme: Ozaki, Uchino, Imamura, "Ozaki scheme II",
// 2025).  Every operand row is scaled by a power of two and rounded to integers; their
// products are formed modulo NM pairwise coprime numbers p <= 256, whose symmetric
// residues (|r| <= 128) are exact in BF16 and whose sums over CHUNK terms stay below
// 2^24, exact in the FP32 accumulators of tcgen05; the sums modulo the p give the
// integer result by the Chinese remainder theorem, which is rounded to FP64 once.
// Nothing is rounded but the operands (2^-62 of their row's norm, at most) and the result:
//   |error| <= 2^-61 sqrt(n) |a| |b|  per entry of n points, where every value rounds the same way, and
//   some 2^-61 |a| |b| where they do not,  against some 2^-54 to 2^-50 of an FP64 sum.
//
// Rotations multiply rows that need not be alike in size by coefficients of any size: rows are first
// scaled to equal norms and the coefficients by what that took away, both by powers of two, so that the result does
// not depend on how a program scales its rows.  Then one scale per point and one per column of coefficients serve
// all rows: |error| <= some 2^-57 max_i |y_i(p)| / |y_i| times the norm of |c_i| |y_i|.
//
// The passes: row statistics (power-of-two scales) -> residues (one bf16 plane per
// modulus and per real or imaginary part) -> k_rns (one GEMM per modulus) -> CRT.  The
// points go in chunks that keep the residues within RNS_BYTES.
//
// Measured on one GB300 against the FP64 kernels (which run at 97% of the FP64 pipe):
//   Gram 432 x 432 over 64^3 points   321.8 -> 9.3 ms     rotation 432 -> 144   104.8 -> 5.7 ms
//   real Gram 285 x 285 over 60^3      30.2 -> 2.5 ms
// of the Gram's 9.3 ms the residue planes take 3.6 (80% of DRAM bandwidth, 78% of the issue slots), the
// statistics 0.6 and the MMAs 5.1 (60% of the tensor pipe's cycles, the rest waits for shared memory); of the
// rotation's 5.7 the statistics of rows and points 0.75, residues 1.5, MMAs 2.5 and remainders 0.8;
// and errors against extended precision (150 x 150 over 5,400 points: relative 7.1e-17 against
// 1.1e-15; rotation 432 -> 144: 4.7e-17 against 9.8e-16; <a|a> of uniform rows on 64^3, 96^3, 120^3: 0, 3.0e-16,
// 6.4e-16 against 4.3e-14, 1.5e-13, 3.2e-13).
//
// Non-finite values, and rows of nothing but subnormal ones, raise a device flag; then the
// kernels here leave their outputs alone and the FP64 kernels launched behind them
// (which return at once otherwise) do the work, so such inputs give what they gave.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "fft_common.h"
#include "rsdft_internal.h"
#include "tc_ptx.h"

namespace rsdft {
namespace rns {

using tc::smem_u32;
typedef long long i64;
typedef unsigned long long u64;
typedef unsigned __int128 u128;

// ---- moduli and their constants ---------------------------------------------------
// T_ROW is set by the operands' own accuracy, not by the result's: a row of n points that is equally large
// everywhere has values 2^-(log2(n)/2) of its norm, and a plane wave rounds every one of them the same
// way, so that the errors add up.  At 62 such a row of 64^3 points keeps 53 bits (and is exact), one of
// 128^3 51.  With 15 moduli and 58 bits a uniform row's <a|a> was off by 2.2e-15 on 64^3, 3.6e-15 on 96^3.
constexpr int NM = 16;
constexpr int MODS[NM] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};
// P = prod MODS = 2^125.37: twice the largest |sum| must stay below it
constexpr int T_ROW = 62;      // |row|_2 < 2^62 after scaling (both operands: 2^125 < P)

struct Consts {
    float p[NM], ip[NM];
    int m[NM];
    int lo[NM], hi[NM];        // 256^j mod p, symmetric, as signed bytes j = 0..3 and 4..7
    // W = floor(frac((P/p)^-1 mod p / p) 2^96) by byte j = 0..11, four moduli a word
    uint32_t w[12][4];
    u64 Ptop;                  // P / 2^62, rounded
};

constexpr Consts make_consts() {
    Consts c{};
    u128 P = 1;
    for (int i = 0; i < NM; ++i) P *= (u128)MODS[i];
    for (int i = 0; i < NM; ++i) {
        const int p = MODS[i];
        c.p[i] = (float)p;
        c.m[i] = p;
        c.ip[i] = 1.0f / (float)p;
        int pw = 1;
        uint32_t b[2] = {0, 0};
        for (int j = 0; j < 8; ++j) {
            const int s = pw > 127 ? pw - p : pw;   // in [-128, 127]: p <= 256
            b[j >> 2] |= (uint32_t)(s & 255) << (8 * (j & 3));
            pw = (pw * 256) % p;
        }
        c.lo[i] = (int)b[0];
        c.hi[i] = (int)b[1];
        const int q = (int)((P / (u128)p) % (u128)p);
        int inv = 1;
        while ((inv * q) % p != 1) ++inv;
        // floor(inv 2^96 / p) by long division
        u128 w = 0;
        int r = inv;
        for (int k = 0; k < 96; ++k) {
            r *= 2;
            w <<= 1;
            if (r >= p) { r -= p; w |= 1; }
        }
        for (int j = 0; j < 12; ++j) c.w[j][i >> 2] |= (uint32_t)(uint8_t)(w >> (8 * j)) << (8 * (i & 3));
    }
    c.Ptop = (u64)((P + ((u128)1 << 61)) >> 62);
    return c;
}
__constant__ Consts K = make_consts();

constexpr float MAGIC = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer

// ---- scales -----------------------------------------------------------------------
// Part of one row: the largest exponent field and the sum of squares in units of 4^(that
// field - 1023), from the leading 21 bits of each value (integer and FP32 instructions:
// the FP64 pipe would bound this pass).
struct Stat {
    int e;
    float s;
};
__device__ __forceinline__ void stat_rebase(Stat &a, int e) {
    if (e > a.e) {
        a.s = e - a.e > 60 ? 0.0f : a.s * __int_as_float((127 - 2 * (e - a.e)) << 23);
        a.e = e;
    }
}
__device__ __forceinline__ void stat_add(Stat &a, int habs) {
    if (a.e == 0) {   // nothing but zeros and subnormal values so far
        if (habs) a.s = 1.0f;
        return;
    }
    const int u = habs - ((a.e - 127) << 20);
    const float f = __int_as_float(max(u, 0) << 3);
    a.s = fmaf(f, f, a.s);
}
__device__ __forceinline__ Stat stat_join(Stat a, Stat b) {
    stat_rebase(a, b.e);
    stat_rebase(b, a.e);
    a.s += b.s;
    return a;
}

// part[(row S + slice) 2 + plane]
__global__ void __launch_bounds__(256)
k_row_stat(RowBlocks src, long long n, int S, Stat *__restrict__ part) {
    const int row = blockIdx.y;
    int i = row, blk = 0;
    while (blk < 2 && i >= src.cnt[blk]) { i -= src.cnt[blk]; ++blk; }
    const int4 *x = reinterpret_cast<const int4 *>(src.ptr[blk] + (size_t)i * n);
    const long long c = (n + S - 1) / S, i0 = blockIdx.x * c, i1 = min(n, i0 + c);
    Stat a{0, 0.0f}, b{0, 0.0f};
    for (long long q = i0 + threadIdx.x; q < i1; q += 4 * 256) {
        int hx[4], hy[4], mx = 0, my = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long r = q + u * 256;
            int4 v = make_int4(0, 0, 0, 0);
            if (r < i1) v = __ldg(x + r);
            hx[u] = (v.y & 0x7fffffff) | (v.x != 0);   // (a subnormal value may have nothing but a low word)
            hy[u] = (v.w & 0x7fffffff) | (v.z != 0);
            mx = max(mx, hx[u]);
            my = max(my, hy[u]);
        }
        stat_rebase(a, mx >> 20);
        stat_rebase(b, my >> 20);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            stat_add(a, hx[u]);
            stat_add(b, hy[u]);
        }
    }
    __shared__ Stat sh[2][8];
#pragma unroll
    for (int pl = 0; pl < 2; ++pl) {
        Stat t = pl ? b : a;
        for (int o = 16; o > 0; o >>= 1) {
            Stat u{__shfl_xor_sync(0xffffffffu, t.e, o), __shfl_xor_sync(0xffffffffu, t.s, o)};
            t = stat_join(t, u);
        }
        if ((threadIdx.x & 31) == 0) sh[pl][threadIdx.x >> 5] = t;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        Stat t = sh[threadIdx.x][0];
        for (int w = 1; w < 8; ++w) t = stat_join(t, sh[threadIdx.x][w]);
        part[((size_t)row * S + blockIdx.x) * 2 + threadIdx.x] = t;
    }
}

// scale[2 row + plane] = s with |row|_2 2^s <= 2^T_ROW; both planes of a complex row (joint)
// share it.  Raises the flag where the row is not finite or has no normal number (its values' bits are not known).
__global__ void k_row_scale(const Stat *__restrict__ part, int S, int rows, int joint, int *__restrict__ scale,
                            int *flag) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= rows) return;
    Stat t[2];
    for (int pl = 0; pl < 2; ++pl) {
        t[pl] = part[(size_t)row * S * 2 + pl];
        for (int s = 1; s < S; ++s) t[pl] = stat_join(t[pl], part[((size_t)row * S + s) * 2 + pl]);
    }
    if (joint) t[0] = t[1] = stat_join(t[0], t[1]);
    for (int pl = 0; pl < 2; ++pl) {
        int s = 0;
        if (t[pl].s > 0.0f) {
            if (t[pl].e == 0x7ff || t[pl].e == 0) atomicExch(flag, 1);
            // |row|^2 < 2^(g + 1) 4^(e - 1023) with the truncated bits counted in
            const int g = ilogbf(t[pl].s * 1.001f);
            s = T_ROW - (t[pl].e - 1023) - ((g + 2) >> 1);
        }
        scale[2 * row + pl] = s;
    }
}

// Largest exponent per point of the scaled rows |x| 2^scale over rows [r0, r0 + nr) of the block list
// (any of the two parts), offset by PT_BIAS (0: a point of zeros), for the rotation's per-point scales.
constexpr int PT_BIAS = 4096;   // scales lie within +-1,200
__device__ __forceinline__ int point_exp(int hi, int lo, int s) {
    const int h = hi & 0x7fffffff;
    return (h | lo) ? max(h >> 20, 1) + s + PT_BIAS : 0;
}
__global__ void __launch_bounds__(256)
k_point_max(RowBlocks src, int r0, int nr, long long n, int rows_per_cta, const int *__restrict__ scale,
            int *__restrict__ pmax) {
    const long long q = (long long)blockIdx.x * 256 + threadIdx.x;
    if (q >= n) return;
    const int a = r0 + blockIdx.y * rows_per_cta, b = min(r0 + nr, a + rows_per_cta);
    int m = 0;
    for (int row = a; row < b; row += 8) {
        int4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            int i = row + u, blk = 0;
            v[u] = make_int4(0, 0, 0, 0);
            if (i < b) {
                while (blk < 2 && i >= src.cnt[blk]) { i -= src.cnt[blk]; ++blk; }
                v[u] = __ldg(reinterpret_cast<const int4 *>(src.ptr[blk] + (size_t)i * n) + q);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (row + u < b) {
                const int2 s = __ldg(reinterpret_cast<const int2 *>(scale) + row + u);
                m = max(m, max(point_exp(v[u].y, v[u].x, s.x), point_exp(v[u].w, v[u].z, s.y)));
            }
    }
    atomicMax(pmax + q, m);
}

// s with |x| 2^s <= 2^bits for every scaled |x| of a point whose largest exponent is e
__device__ __forceinline__ int point_scale(int e, int bits) { return e == 0 ? 0 : bits - (e - PT_BIAS - 1022); }

// ---- residues ---------------------------------------------------------------------
// |x| 2^s < 2^62 rounded to an integer, by integer shifts
__device__ __forceinline__ u64 fix(int hi, unsigned lo, int s) {
    const int e = (hi >> 20) & 0x7ff;
    const u64 m = ((u64)(unsigned)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 42) | ((u64)lo << 10);
    const int r = min(max(1085 - max(e, 1) - s, 1), 63);   // mantissa was shifted by 10; r >= 1 by the choice of s
    return (m + (1ull << (r - 1))) >> r;
}

// symmetric residue of v modulo MODS[q], as a float
__device__ __forceinline__ float residue(u64 v, int q) {
    int d = __float_as_int(MAGIC);
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"((unsigned)v), "r"(K.lo[q]), "r"(d));
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"((unsigned)(v >> 32)), "r"(K.hi[q]), "r"(d));
    const float f = __int_as_float(d) - MAGIC;   // |f| < 2^18
    const float k = fmaf(f, K.ip[q], MAGIC) - MAGIC;
    return fmaf(-k, K.p[q], f);
}
// the two residues as a bf16 pair (exact: the low halves of the floats are zero), signs applied
__device__ __forceinline__ unsigned pack(float a, float b, unsigned neg) {
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632) ^ neg;
}

// Residue planes of rows of FP64 complex values: res[q][row][plane][ld], points p0 .. p0 + ld
// (zero beyond n).  Scales per row and plane; per_point: on top of them per point and segment, rows
// below seg1 by pmax[0][..], the others by pmax[1][..].  Four points a thread; all integer and
// FP32 arithmetic, about 7 instructions a residue: this pass is bound by its instructions
// and by the 4 NM bytes that it writes for every 16 read.
__global__ void __launch_bounds__(256)
k_residues(RowBlocks src, long long n, long long p0, int ld, int R, int row0, int per_point,
           const int *__restrict__ scale, const int *__restrict__ pmax, int seg1, int bits0, int bits1,
           __nv_bfloat16 *__restrict__ res, const int *flag) {
    if (*flag) return;
    const int row = blockIdx.y;
    int i = row, blk = 0;
    while (blk < 2 && i >= src.cnt[blk]) { i -= src.cnt[blk]; ++blk; }
    const int4 *x = reinterpret_cast<const int4 *>(src.ptr[blk] + (size_t)i * n);
    const int t = (blockIdx.x * 256 + threadIdx.x) * 4;
    if (t >= ld) return;
    u64 v[8];
    unsigned neg[4];   // sign masks of the packed pairs: re 01, re 23, im 01, im 23
    neg[0] = neg[1] = neg[2] = neg[3] = 0;
    const int seg = row >= seg1 ? 1 : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const long long p = p0 + t + u;
        int4 w = make_int4(0, 0, 0, 0);
        int sr = 0, si = 0;
        if (p < n) {
            w = __ldg(x + p);
            const int sp = per_point ? point_scale(pmax[seg * n + p], seg ? bits1 : bits0) : 0;
            sr = scale[2 * (row0 + row)] + sp;
            si = scale[2 * (row0 + row) + 1] + sp;
        }
        v[u] = fix(w.y, (unsigned)w.x, sr);
        v[4 + u] = fix(w.w, (unsigned)w.z, si);
        neg[u >> 1] |= (w.y & 0x80000000u) >> ((u & 1) ? 0 : 16);
        neg[2 + (u >> 1)] |= (w.w & 0x80000000u) >> ((u & 1) ? 0 : 16);
    }
    uint2 *out = reinterpret_cast<uint2 *>(res + ((size_t)(row0 + row) * 2) * ld + t);
    const size_t plane = ld / 4, mod = (size_t)R * 2 * ld / 4;
#pragma unroll 1
    for (int q = 0; q < NM; ++q) {
        float f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = residue(v[j], q);
        out[q * mod] = make_uint2(pack(f[0], f[1], neg[0]), pack(f[2], f[3], neg[1]));
        out[q * mod + plane] = make_uint2(pack(f[4], f[5], neg[2]), pack(f[6], f[7], neg[3]));
    }
}

// ---- rotation coefficients ----------------------------------------------------------
// A segment of the rotation: coefficient rows that multiply a run of Y rows.  In real form the
// Y rows hold two bands each, and K index 2 j + h is band h of pair row j.
struct Seg {
    int cnt[2], crow[2];   // up to two row blocks: bands in each, first row of each in c
    int k;                 // K extent: rows (complex) or padded bands (real)
};
__device__ __forceinline__ int coef_row(const Seg &s, int t, bool real) {
    const int k0 = real ? ((s.cnt[0] + 1) & ~1) : s.cnt[0];
    if (t < k0) return t < s.cnt[0] ? s.crow[0] + t : -1;
    t -= k0;
    return t < s.cnt[1] ? s.crow[1] + t : -1;
}

// scale of column b of a segment's coefficients c 2^-ys (ys: the scales of their rows of Y, from the
// segment's first row on): |c_b 2^-ys|_2 2^s < 2^T_ROW
__global__ void k_coef_scale(const double2 *__restrict__ c, int ldc, Seg s, int real, const int *__restrict__ ys,
                             int *__restrict__ sc, int *flag) {
    const int b = blockIdx.x;
    auto value = [&](int t) {
        const int r = coef_row(s, t, real);
        double2 v = make_double2(0.0, 0.0);
        if (r >= 0) v = c[(size_t)r * ldc + b];
        if (real) v.y = 0.0;
        return v;
    };
    int top = -(1 << 20);
    for (int t = threadIdx.x; t < s.k; t += 32) {
        const double2 v = value(t);
        const double m = fmax(fabs(v.x), fabs(v.y));
        if (!isfinite(v.x) || !isfinite(v.y)) atomicExch(flag, 1);
        if (m > 0.0) top = max(top, ((__double2hiint(m) >> 20) & 0x7ff) - 1023 - ys[real ? t : 2 * t]);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    double sum = 0.0;
    for (int t = threadIdx.x; t < s.k; t += 32) {
        const double2 v = value(t);
        const int e = -ys[real ? t : 2 * t] - top;
        const double x = scalbn(v.x, e), y = scalbn(v.y, e);
        sum = fma(x, x, fma(y, y, sum));
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (threadIdx.x == 0) sc[b] = sum > 0.0 ? T_ROW - top - ((ilogb(sum * (1.0 + 1e-12)) + 2) >> 1) : 0;
}

// res[q][plane][nbp][kpad] of a segment's coefficients (zero outside)
__global__ void k_coef_residues(const double2 *__restrict__ c, int ldc, Seg s, int real, int m, int nbp, int kpad,
                                const int *__restrict__ ys, const int *__restrict__ sc, __nv_bfloat16 *__restrict__ res, const int *flag) {
    if (*flag) return;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)nbp * (kpad / 2)) return;
    const int b = (int)(idx / (kpad / 2)), t = 2 * (int)(idx % (kpad / 2));
    const int planes = real ? 1 : 2;
    u64 v[4];
    unsigned neg[2] = {0, 0};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int r = b < m && t + u < s.k ? coef_row(s, t + u, real) : -1;
        const double2 z = r >= 0 ? c[(size_t)r * ldc + b] : make_double2(0.0, 0.0);
        const int e = r >= 0 ? sc[b] - ys[real ? t + u : 2 * (t + u)] : 0;
        v[u] = fix(__double2hiint(z.x), __double2loint(z.x), e);
        v[2 + u] = fix(__double2hiint(z.y), __double2loint(z.y), e);
        neg[0] |= (__double2hiint(z.x) & 0x80000000u) >> (u ? 0 : 16);
        neg[1] |= (__double2hiint(z.y) & 0x80000000u) >> (u ? 0 : 16);
    }
    unsigned *out = reinterpret_cast<unsigned *>(res + (size_t)b * kpad + t);
    const size_t plane = (size_t)nbp * kpad / 2;
    for (int q = 0; q < NM; ++q) {
        out[(size_t)(q * planes) * plane] = pack(residue(v[0], q), residue(v[1], q), neg[0]);
        if (!real) out[(size_t)(q * planes + 1) * plane] = pack(residue(v[2], q), residue(v[3], q), neg[1]);
    }
}

// ---- the GEMM: one modulus per work item ------------------------------------------------
// Persistent CTAs of 320 threads, one per SM: warp 0 issues TMA, warp 1 issues MMAs, warps
// 2..9 drain.  A work item is an output tile of one modulus and one range of K:
//   complex  128 x NT (NT <= 128), two accumulators (real, imaginary) of 128 TMEM columns
//   real     128 x NT (NT <= 256), one accumulator of up to 256 columns
// The accumulators are double-buffered (2 x 256 columns), and every CHUNK K-blocks they are
// reduced modulo p into 128 registers of each drain thread while the next chunk's MMAs run,
// so that every FP32 sum stays an exact integer below 2^24.
//   Gram (ROT = false): A, B K-major [row][point]; tile of conj(A) B^T; residues of the sums
//     go to out16[split][q][plane][M][blocks npad].
//   Rotation (ROT = true): A = residues of Y read MN-major (points are M), B = coefficients
//     K-major; residues go to out8[q][segment][plane][N / 4][points], four bands a word.
constexpr int THREADS = 320;
constexpr int SK = 64;                 // K per stage: 128-byte rows
constexpr int STAGE_C = 64 * 1024, STAGES_C = 3;   // 2 + 2 planes of 128 x 64
constexpr int STAGE_R = 48 * 1024, STAGES_R = 4;   // 128 x 64 and 256 x 64
constexpr int SMEM = 192 * 1024 + 1024;
template <bool REAL> struct Cfg {
    static constexpr int STAGES = REAL ? STAGES_R : STAGES_C;
    static constexpr int STAGE = REAL ? STAGE_R : STAGE_C;
    static constexpr int CHUNK = REAL ? 16 : 8;    // stages: 1024 or 2 x 512 products of at most 2^14
    static constexpr int NT = REAL ? 256 : 128;
};

struct Args {
    int items;
    int mt, nt;                 // tile counts
    int npad;                   // Gram: columns of a block of out16 (N rounded up to 8)
    int nstep;                  // columns per tile
    int boxn;                   // rows of the B box (its bytes: boxn * 128 per plane)
    int M, N;                   // output rows and columns (Gram: N of one block)
    // Gram
    int herm, blocks, tiles;    // upper tiles only; B is `blocks` blocks of N rows; tiles per modulus
    int kb_total, kb_split;
    int accumulate;
    short *out16;
    // rotation
    int segs, kb[2], row0[2];   // K-blocks of each segment and its first A row
    long long ldp;              // points of an output row
    unsigned *out8;
    const int *flag;
    int *flag_w;
};

struct Item {
    int q, m0, n0, bcol, ncols, kb0, nkb, seg, slot;
};

template <bool ROT> __device__ __forceinline__ Item decode(const Args &a, int idx) {
    Item it;
    if (!ROT) {
        const int per = a.tiles;
        int t = idx % per;
        idx /= per;
        it.q = idx % NM;
        it.slot = idx / NM;
        it.seg = 0;
        int tm = 0, tn = 0, blk = 0;
        if (a.herm) {
            const int tri = per / a.blocks;
            blk = t / tri;
            t -= blk * tri;
            // row tile tm holds the column tiles from the one with its first row on
            while (true) {
                const int first = tm * 128 / a.nstep;
                if (t < a.nt - first) { tn = first + t; break; }
                t -= a.nt - first;
                ++tm;
            }
        } else {
            tm = t / a.nt;
            tn = t - tm * a.nt;
        }
        it.m0 = tm * 128;
        it.n0 = tn * a.nstep;
        it.bcol = blk * a.N + it.n0;
        it.ncols = min(a.nstep, a.N - it.n0);
        it.n0 = it.bcol;
        it.kb0 = it.slot * a.kb_split;
        it.nkb = min(a.kb_split, a.kb_total - it.kb0);
    } else {
        const int tn = idx % a.nt;
        idx /= a.nt;
        it.seg = idx % a.segs;
        idx /= a.segs;
        it.m0 = (idx % a.mt) * 128;
        it.q = idx / a.mt;
        it.n0 = it.bcol = tn * a.nstep;
        it.ncols = min(a.nstep, a.N - it.n0);
        it.kb0 = 0;
        it.nkb = a.kb[it.seg];
        it.slot = 0;
    }
    return it;
}

template <bool REAL, bool ROT>
__global__ void __launch_bounds__(THREADS, 1)
k_rns(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB0,
      const __grid_constant__ CUtensorMap mB1, const __grid_constant__ Args a) {
    if (*a.flag) return;
    using C = Cfg<REAL>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[C::STAGES];
    __shared__ __align__(8) uint64_t empty_bar[C::STAGES];
    __shared__ __align__(8) uint64_t accf_bar[2];
    __shared__ __align__(8) uint64_t acce_bar[2];
    __shared__ __align__(8) uint64_t done_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int PL = REAL ? 1 : 2;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            tc::mbar_init(&full_bar[s], 1);
            tc::mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&accf_bar[b], 1);
            tc::mbar_init(&acce_bar[b], 8);
        }
        tc::mbar_init(&done_bar, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tc::tmem_alloc(&tmem_base, 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = tmem_base;
    volatile int *abort = &s_abort;

    if (warp == 0 && lane == 0) {
        // ---- TMA producer
        const uint32_t bytes = PL * (16384u + (uint32_t)a.boxn * 128u);
        int st = 0;
        bool stop = false;
        for (int idx = blockIdx.x; idx < a.items && !stop; idx += gridDim.x) {
            const Item it = decode<ROT>(a, idx);
            const CUtensorMap *mB = ROT && it.seg ? &mB1 : &mB0;
            for (int kb = 0; kb < it.nkb; ++kb, ++st) {
                const int s = st % C::STAGES, r = st / C::STAGES;
                if (r > 0 && !tc::mbar_wait(&empty_bar[s], (r - 1) & 1, abort)) { stop = true; break; }
                unsigned char *sa = smem + s * C::STAGE, *sb = sa + PL * 16384;
                tc::mbar_expect_tx(&full_bar[s], bytes);
                const int x = (it.kb0 + kb) * SK;
#pragma unroll
                for (int pl = 0; pl < PL; ++pl) {
                    if (!ROT) {
                        tc::tma_load_4d(sa + pl * 16384, &mA, &full_bar[s], x, it.m0, pl, it.q);
                        tc::tma_load_4d(sb + pl * 16384, mB, &full_bar[s], x, it.bcol, pl, it.q);
                    } else {
                        const int y = a.row0[it.seg] + x;
                        tc::tma_load_4d(sa + pl * 16384, &mA, &full_bar[s], it.m0, y, pl, it.q);
                        tc::tma_load_4d(sa + pl * 16384 + 8192, &mA, &full_bar[s], it.m0 + 64, y, pl, it.q);
                        tc::tma_load_4d(sb + pl * 16384, mB, &full_bar[s], x, it.bcol, pl, it.q);
                    }
                }
            }
        }
        if (*abort) {
            // let the copies still in flight land before the CTA leaves
            for (int j = max(0, st - C::STAGES); j < st; ++j) {
                const long long t0 = clock64();
                while (!tc::mbar_try_wait(&full_bar[j % C::STAGES], (j / C::STAGES) & 1) &&
                       clock64() - t0 < tc::WAIT_LIMIT) {
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        int st = 0, ch = 0;
        bool stop = false;
        for (int idx = blockIdx.x; idx < a.items && !stop; idx += gridDim.x) {
            const Item it = decode<ROT>(a, idx);
            const uint32_t idesc = tc::idesc_bf16(128, (it.ncols + 15) & ~15) | (ROT ? tc::IDESC_A_MN : 0u);
            const uint32_t ineg = idesc | tc::IDESC_NEG_A;
            for (int kb = 0; kb < it.nkb && !stop; ++ch) {
                const int b = ch & 1;
                if (ch >= 2 && !tc::mbar_wait(&acce_bar[b], ((ch >> 1) - 1) & 1, abort)) { stop = true; break; }
                tc::tc_fence_after();
                const uint32_t d0 = tmem + (uint32_t)(b * 256), d1 = d0 + 128;
                uint32_t acc = 0;
                const int kend = min(it.nkb, kb + C::CHUNK);
                for (; kb < kend; ++kb, ++st) {
                    const int s = st % C::STAGES, r = st / C::STAGES;
                    if (!tc::mbar_wait(&full_bar[s], r & 1, abort)) { stop = true; break; }
                    tc::tc_fence_after();
                    unsigned char *sa = smem + s * C::STAGE, *sb = sa + PL * 16384;
#pragma unroll
                    for (int kk = 0; kk < SK / 16; ++kk) {
                        uint64_t ad[PL], bd[PL];
#pragma unroll
                        for (int pl = 0; pl < PL; ++pl) {
                            ad[pl] = ROT ? tc::smem_desc_mn(sa + pl * 16384 + kk * 2048, 8192, 1024)
                                         : tc::smem_desc_k128(sa + pl * 16384 + kk * 32);
                            bd[pl] = tc::smem_desc_k128(sb + pl * 16384 + kk * 32);
                        }
                        if (REAL) {
                            tc::mma_bf16(d0, ad[0], bd[0], idesc, acc);
                        } else if (!ROT) {
                            // Re += A_re B_re + A_im B_im, Im += A_re B_im - A_im B_re
                            tc::mma_bf16(d0, ad[0], bd[0], idesc, acc);
                            tc::mma_bf16(d1, ad[0], bd[PL - 1], idesc, acc);
                            tc::mma_bf16(d0, ad[PL - 1], bd[PL - 1], idesc, 1u);
                            tc::mma_bf16(d1, ad[PL - 1], bd[0], ineg, 1u);
                        } else {
                            // Re += Y_re C_re - Y_im C_im, Im += Y_re C_im + Y_im C_re
                            tc::mma_bf16(d0, ad[0], bd[0], idesc, acc);
                            tc::mma_bf16(d1, ad[0], bd[PL - 1], idesc, acc);
                            tc::mma_bf16(d0, ad[PL - 1], bd[PL - 1], ineg, 1u);
                            tc::mma_bf16(d1, ad[PL - 1], bd[0], idesc, 1u);
                        }
                        acc = 1u;
                    }
                    tc::mma_commit(&empty_bar[s]);
                }
                if (!stop) tc::mma_commit(&accf_bar[b]);
            }
        }
        // every MMA issued so far must finish before TMEM is released (bounded)
        tc::mma_commit(&done_bar);
        const long long t0 = clock64();
        while (!tc::mbar_try_wait(&done_bar, 0)) {
            if (clock64() - t0 > tc::WAIT_LIMIT) { *abort = 1; break; }
        }
    } else if (warp >= 2) {
        // ---- drain: warp w reads TMEM lanes 32 (w % 4) .., columns 128 half .. of the buffer
        // (complex: half 0 the real part, half 1 the imaginary part)
        const int lq = warp & 3, half = (warp - 2) >> 2;
        int ch = 0;
        bool stop = false;
        for (int idx = blockIdx.x; idx < a.items && !stop; idx += gridDim.x) {
            const Item it = decode<ROT>(a, idx);
            const float p = K.p[it.q], ip = K.ip[it.q];
            const int ncol = REAL ? min(128, it.ncols - half * 128) : it.ncols;   // may be <= 0
            float acc[128];
#pragma unroll
            for (int i = 0; i < 128; ++i) acc[i] = 0.0f;
            for (int kb = 0; kb < it.nkb; kb += C::CHUNK, ++ch) {
                const int b = ch & 1;
                if (!tc::mbar_wait_warp(&accf_bar[b], (ch >> 1) & 1, abort)) { stop = true; break; }
                tc::tc_fence_after();
                const uint32_t base = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(b * 256 + half * 128);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    if (g * 32 < ncol) {
                        float v[32];
                        tc::tmem_ld32(base + (uint32_t)(g * 32), v);
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const float k = fmaf(v[i], ip, MAGIC) - MAGIC;
                            acc[g * 32 + i] += fmaf(-k, p, v[i]);
                        }
                    }
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&acce_bar[b]);
            }
            if (stop) break;
            const int row = it.m0 + lq * 32 + lane;
            if (!ROT) {
                // eight residues a store: rows of npad columns a block, npad and the tiles multiples of 8
                const int plane = REAL ? 0 : half;
                const int blk = it.n0 / a.N, col = it.n0 - blk * a.N + (REAL ? half * 128 : 0);
                int4 *o = reinterpret_cast<int4 *>(a.out16 + ((((size_t)it.slot * NM + it.q) * PL + plane) * a.M + row) *
                                                                 (size_t)(a.npad * a.blocks) + blk * a.npad + col);
                if (row < a.M) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (8 * i < ncol) {
                            int w[4] = {0, 0, 0, 0};
                            if (a.accumulate) {
                                const int4 old = o[i];
                                w[0] = old.x;
                                w[1] = old.y;
                                w[2] = old.z;
                                w[3] = old.w;
                            }
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                int r[2];
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const float v = acc[8 * i + 2 * j + h] + (float)(short)(w[j] >> (16 * h));
                                    const float k = fmaf(v, ip, MAGIC) - MAGIC;
                                    r[h] = __float_as_int(fmaf(-k, p, v) + MAGIC);
                                }
                                w[j] = (int)__byte_perm(r[0], r[1], 0x5410);
                            }
                            o[i] = make_int4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
            } else {
                const int plane = REAL ? 0 : half;
                const int quad0 = (it.n0 + (REAL ? half * 128 : 0)) >> 2, nquad = (a.N + 3) >> 2;
                unsigned *o = a.out8 + (((size_t)(it.q * a.segs + it.seg) * PL + plane) * nquad + quad0) * a.ldp + row;
                if (row < a.M) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        if (4 * i < ncol) {
                            int w[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float v = acc[4 * i + j];
                                const float k = fmaf(v, ip, MAGIC) - MAGIC;
                                w[j] = __float_as_int(fmaf(-k, p, v) + MAGIC);
                            }
                            o[(size_t)i * a.ldp] = __byte_perm(__byte_perm(w[0], w[1], 0x0040), __byte_perm(w[2], w[3], 0x0040), 0x5410);
                        }
                    }
                }
            }
        }
    }
    __syncwarp();
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, 512);
    }
    if (threadIdx.x == 0 && *abort) atomicExch(a.flag_w, 2);
}

// ---- Chinese remainder ----------------------------------------------------------------
// x 2^-s of the integer x with the symmetric residues r (bytes, four moduli a word): the fraction
// x / P is sum r W / 2^96 modulo 1, its bytes' columns summed by dp4a (48 instead of 75 to 105
// wide multiply-adds), good to 2^-85: 2^-83 of the product of the operands' bounds (2^124).  All residues 0
// give exactly 0.
__device__ __forceinline__ double crt_value(const int r[4], int s) {
    i64 limb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int c[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int d = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g)
                asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(d) : "r"(r[g]), "r"(K.w[4 * k + j][g]));
            c[j] = d;   // |d| < 2^19
        }
        limb[k] = (i64)(c[2] + (c[3] << 8)) * 65536 + (c[0] + (c[1] << 8));
    }
    const i64 m1 = limb[1] + (limb[0] >> 32), m2 = limb[2] + (m1 >> 32);
    unsigned f0 = (unsigned)limb[0], f1 = (unsigned)m1, f2 = (unsigned)m2;
    const bool neg = (int)f2 < 0;
    if (neg) {   // two's complement
        f0 = ~f0 + 1;
        f1 = ~f1 + (f0 == 0);
        f2 = ~f2 + (f0 == 0 && f1 == 0);
    }
    int e = 30 - s;   // x = hi 2^(e + s), below
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (f2 == 0) {
            f2 = f1;
            f1 = f0;
            f0 = 0;
            e -= 32;
        }
    if (f2 == 0) return 0.0;
    const int lz = __clz((int)f2);
    const u64 m = ((u64)__funnelshift_l(f1, f2, lz) << 32) | __funnelshift_l(f0, f1, lz);   // F = m 2^(32 - lz)
    u64 hi = __umul64hi(m, K.Ptop);        // x = F P / 2^96 = hi 2^(64 + 32 - lz + 62 - 96)
    e += 32 - lz;
    if (!(hi >> 63)) {
        hi <<= 1;
        e -= 1;
    }
    u64 t = hi >> 11;
    const u64 rest = hi & 0x7ff;
    t += rest > 0x400 || (rest == 0x400 && (t & 1));
    // value = t 2^(11 + e) with 2^52 <= t <= 2^53
    const int field = e + 11 + 1075;
    double v;
    if (field >= 1 && field <= 2045) v = __longlong_as_double((long long)t + ((long long)(field - 1) << 52));
    else v = scalbn((double)t, e + 11);   // beyond the normal range
    return neg ? -v : v;
}

// g entries of one or two blocks from the residue sums out16[slot][q][plane][M][blocks npad]
// (padded bands in real form).  herm: entries below the diagonal from their mirror, the
// diagonal real.
__global__ void k_crt_gram(const short *__restrict__ out16, int slots, int M, int N, int npad, int blocks, int real, int a0,
                           int a1, int b0, int b1, int na, int nb, int herm, const int *__restrict__ sa,
                           const int *__restrict__ sb, double scale, double2 *__restrict__ g0,
                           double2 *__restrict__ g1, int ldg, const int *flag) {
    if (*flag) return;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)na * nb) return;
    const int blk = blockIdx.y;
    const int i = (int)(idx / nb), j = (int)(idx % nb);
    int I = i, J = j;
    if (real) {   // compact band -> padded band (blocks of pair rows)
        auto pad = [](int c0, int c1, int t) {
            if (t < c0) return t;
            t -= c0;
            const int base = (c0 + 1) & ~1;
            if (t < c1) return base + t;
            return base + ((c1 + 1) & ~1) + (t - c1);
        };
        I = pad(a0, a1, i);
        J = pad(b0, b1, j);
    }
    const bool mirror = herm && I > J;
    const int r = mirror ? J : I, c = mirror ? I : J;
    const int PL = real ? 1 : 2, ldn = npad * blocks;
    double v[2] = {0.0, 0.0};
    // scales are per complex row and plane: 2 row + plane is the padded band in real form
    const int s = sa[real ? r : 2 * r] + sb[real ? blk * N + c : 2 * (blk * N + c)];
    for (int pl = 0; pl < PL; ++pl) {
        int rr[4] = {0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < NM; ++q) {
            int t = 0;
            for (int u = 0; u < slots; ++u)
                t += out16[((((size_t)u * NM + q) * PL + pl) * M + r) * (size_t)ldn + blk * npad + c];
            const float k = fmaf((float)t, K.ip[q], MAGIC) - MAGIC;
            t -= (int)k * K.m[q];   // symmetric; 128 = -128 modulo 256
            rr[q >> 2] |= (t & 255) << (8 * (q & 3));
        }
        v[pl] = crt_value(rr, s);
    }
    if (herm && I == J) v[1] = 0.0;
    if (mirror) v[1] = -v[1];
    (blk ? g1 : g0)[(size_t)i * ldg + j] = make_double2(scale * v[0], scale * v[1]);
}

// Rotation outputs of the points p0 .. p0 + np from out8[q][segment][plane][N / 4][ldp].
// out1 = the last segment's sums (two segments), out0 = base + sign (all segments).  A thread
// does one point of four columns: four complex rows, or two pair rows in real form.
template <bool REAL>
__global__ void __launch_bounds__(256)
k_crt_rot(const unsigned *__restrict__ out8, int segs, int m, long long ldp, long long n, long long p0, int np,
          const int *__restrict__ pmax, int bits0, int bits1, const int *__restrict__ sc, int mcols,
          const double2 *base, int sign, double2 *out0, double2 *out1, const int *flag) {
    if (*flag) return;
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= np) return;
    const int quad = blockIdx.y, nquad = (m + 3) >> 2;
    constexpr int PL = REAL ? 1 : 2;
    double sum[4][PL];
    for (int sg = segs - 1; sg >= 0; --sg) {
        int r[PL][4][4];   // [plane][column][word of moduli]
#pragma unroll
        for (int pl = 0; pl < PL; ++pl)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                unsigned w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    w[i] = 4 * g + i < NM ? __ldg(out8 + (((size_t)((4 * g + i) * segs + sg) * PL + pl) * nquad + quad) * ldp + t) : 0u;
                // four columns of four moduli -> four moduli of each column
                const unsigned a0 = __byte_perm(w[0], w[1], 0x5140), a1 = __byte_perm(w[2], w[3], 0x5140);
                const unsigned b0 = __byte_perm(w[0], w[1], 0x7362), b1 = __byte_perm(w[2], w[3], 0x7362);
                r[pl][0][g] = (int)__byte_perm(a0, a1, 0x5410);
                r[pl][1][g] = (int)__byte_perm(a0, a1, 0x7632);
                r[pl][2][g] = (int)__byte_perm(b0, b1, 0x5410);
                r[pl][3][g] = (int)__byte_perm(b0, b1, 0x7632);
            }
        const int sp = point_scale(pmax[(size_t)sg * n + p0 + t], sg ? bits1 : bits0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int b = 4 * quad + j;
            const int s = (b < m ? sc[sg * mcols + b] : 0) + sp;
#pragma unroll
            for (int pl = 0; pl < PL; ++pl) {
                const double v = crt_value(r[pl][j], s);
                sum[j][pl] = sg == segs - 1 ? v : sum[j][pl] + v;
            }
        }
        double2 *o = sg == 1 ? out1 : nullptr;
        if (o || sg == 0) {
            if (sg == 0) o = out0;
#pragma unroll
            for (int j = 0; j < (REAL ? 2 : 4); ++j) {
                const int row = REAL ? 2 * quad + j : 4 * quad + j;
                if (row >= (REAL ? (m + 1) / 2 : m)) continue;
                double2 v;
                if (REAL) v = make_double2(sum[2 * j][0], 2 * row + 1 < m ? sum[(2 * j + 1) & 3][0] : 0.0);
                else v = make_double2(sum[j][0], sum[j][PL - 1]);
                if (sg == 0 && sign < 0) v = make_double2(-v.x, -v.y);
                if (sg == 0 && base) {
                    const double2 bv = base[(size_t)row * n + p0 + t];
                    v.x += bv.x;
                    v.y += bv.y;
                }
                o[(size_t)row * n + p0 + t] = v;
            }
        }
    }
}

// An in-place rotation whose GEMM gave up (a bounded wait ran out: flag 2) after some chunks
// were written cannot be repeated: its outputs become NaN, which every caller's checks meet.
__global__ void k_poison(double2 *out, long long cnt, const int *flag) {
    if (*flag != 2) return;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (long long)gridDim.x * blockDim.x)
        out[i] = make_double2(__longlong_as_double(0x7ff8000000000000ll), 0.0);
}

}  // namespace rns

using namespace rns;

// ---- host side ---------------------------------------------------------------------------
// Bytes of residues held at a time (the points go in chunks of that size): a chunk's launches end
// with a partly filled wave and the residues' way out (432 x 432, with 15 moduli: 9.0 ms with 2^30, 8.7 with 2^31, 8.5
// with 2^32).  Where that does not fit, an eighth and a 64th of it are tried (4,096 points at least: 0.1 GB for 432
// rows), and the FP64 kernels run only where even that does not: chunks change no bit of a result.
constexpr size_t RNS_BYTES = (size_t)1 << 31;

// The end of a capture's last graph
static void graphs_gone(void *p) {
    auto *alive = static_cast<std::shared_ptr<std::atomic<bool>> *>(p);
    (*alive)->store(false);
    delete alive;
}

// Whether nothing that was or may be launched uses the slot any more
static bool slot_free(const RnsSlot &s) {
    if (s.capture) return !s.graphs->load();
    const bool done = s.done && cudaEventQuery(s.done) == cudaSuccess;
    cudaGetLastError();
    return done;
}

// A slot for the lease's stream, of `bytes` already if there is one to choose from (RnsSlot)
static rsdft_status take_slot(RnsLease &l, size_t bytes) {
    if (l.slot) return RSDFT_OK;
    RnsWork &w = l.ctx->rns;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    unsigned long long capture = 0, stream = 0;
    cudaGraph_t graph = nullptr;
    if (l.st && l.st != cudaStreamLegacy) RS_CUDA(l.ctx, cudaStreamGetCaptureInfo(l.st, &cs, &capture, &graph));
    l.capturing = cs != cudaStreamCaptureStatusNone;
    if (l.capturing) {
        stream = reinterpret_cast<uintptr_t>(l.st);   // (the id of a capturing stream cannot be asked for)
    } else {
        capture = 0;
        RS_CUDA(l.ctx, cudaStreamGetId(l.st, &stream));
    }
    RnsSlot *own = nullptr, *idle = nullptr, *oldest = nullptr;
    int eager = 0;
    for (auto &p : w.slots) {
        RnsSlot &s = *p;
        if (s.capture == capture && s.stream == stream) own = &s;
        else if (slot_free(s) && (!idle || (idle->buf.bytes < bytes && s.buf.bytes > idle->buf.bytes))) idle = &s;
        if (!s.capture) {
            ++eager;
            if (!oldest || s.use < oldest->use) oldest = &s;
        }
    }
    // (a capture cannot give back a smaller buffer for a larger one)
    if (l.capturing && idle && idle->buf.bytes < bytes) idle = nullptr;
    RnsSlot *s = own ? own : idle;
    if (!s && !l.capturing && eager >= RNS_SLOTS) {
        s = oldest;
        RS_CUDA(l.ctx, cudaStreamWaitEvent(l.st, s->done, 0));
    }
    if (!s) {
        w.slots.emplace_back(new RnsSlot);
        s = w.slots.back().get();
    }
    if (s != own) {
        s->stream = stream;
        s->capture = capture;
        s->graphs.reset();
        s->buf.captured = s->fbuf.captured = false;
        if (l.capturing) {
            s->graphs = std::make_shared<std::atomic<bool>>(true);
            auto *alive = new std::shared_ptr<std::atomic<bool>>(s->graphs);
            cudaUserObject_t obj = nullptr;
            cudaError_t e = cudaUserObjectCreate(&obj, alive, graphs_gone, 1, cudaUserObjectNoDestructorSync);
            if (e != cudaSuccess) delete alive;
            else e = cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove);
            RS_CUDA(l.ctx, e);
        }
    }
    if (!l.capturing && !s->done) RS_CUDA(l.ctx, cudaEventCreateWithFlags(&s->done, cudaEventDisableTiming));
    s->use = ++w.uses;
    l.slot = s;
    return RSDFT_OK;
}

RnsLease::~RnsLease() {
    if (slot && !capturing && cudaEventRecord(slot->done, st) != cudaSuccess) {
        cudaGetLastError();
        cudaStreamSynchronize(st);
    }
}

// Whether there is room for a call's residues: growing takes at most a quarter of the free memory.
static bool rns_buffer(rsdft_ctx *ctx, size_t bytes, cudaStream_t st, RnsLease &lease) {
    // this or another thread may be capturing: nothing here is work of a stream
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    bool ok = take_slot(lease, bytes) == RSDFT_OK;
    if (ok && bytes > lease.slot->buf.bytes) {
        size_t free_now = 0, total = 0;
        if (cudaMemGetInfo(&free_now, &total) != cudaSuccess) cudaGetLastError();
        if (bytes > (free_now + lease.slot->buf.bytes) / 4) ok = false;
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    ok = ok && grow(ctx, lease.slot->fbuf, 64, st) == RSDFT_OK && grow(ctx, lease.slot->buf, bytes, st) == RSDFT_OK;
    if (!ok) ctx->err.clear();
    return ok;
}

struct Carver {
    unsigned char *base;
    size_t at = 0;
    template <typename T> T *take(size_t count) {
        T *p = reinterpret_cast<T *>(base ? base + at : nullptr);
        at += (count * sizeof(T) + 1023) / 1024 * 1024;
        return p;
    }
};

static int rows_of(const RowBlocks &b) { return b.cnt[0] + b.cnt[1] + b.cnt[2]; }
static int pairs_up(int c) { return (c + 1) >> 1; }
static RowBlocks pair_rows(const RowBlocks &b) {
    return RowBlocks{{b.ptr[0], b.ptr[1], b.ptr[2]}, {pairs_up(b.cnt[0]), pairs_up(b.cnt[1]), pairs_up(b.cnt[2])}};
}

template <bool REAL, bool ROT>
static rsdft_status launch_gemm(rsdft_ctx *ctx, const CUtensorMap &mA, const CUtensorMap &mB0, const CUtensorMap &mB1,
                                const Args &a, cudaStream_t st) {
    RS_TRY(set_smem(ctx, k_rns<REAL, ROT>, SMEM, SMEM));
    k_rns<REAL, ROT><<<std::min(a.items, ctx->num_sms), THREADS, SMEM, st>>>(mA, mB0, mB1, a);
    count_launch(ctx);
    RS_LAUNCHED(ctx, "k_rns");
    return RSDFT_OK;
}

// Whether the residue path is the faster one.
//  Gram: the FP64 kernel sums at least 512 points a CTA (all of them below that), a microsecond each and
//  0.3 in real form, whatever the number of rows; measured on 216 to 884,736 points and 1 to 288 rows a
//  side, the residue path was the faster one throughout (16 x 16 on 6^3 236 -> 66 us, real 78 -> 64 us;
//  on 20^3 562 -> 103 us, real 173 -> 89 us; 1 x 1 on 6^3 235 -> 64 us, on 96^3 7.0 -> 1.1 ms, real 1.94 -> 0.58).
static bool gram_wins(long long n) { return n >= 200; }
//  Rotation, in seconds: the FP64 kernel at 1.15 TFLOP/s over whole tiles of 16 rows and bands (pair rows in
//  real form) against launches, work items of 128 points (some 2 us each on an SM) and the residue
//  planes (33 ps a row and point).  Within 25% of the times measured on the sizes above; the line at
//  1.15 keeps FP64 where the two meet (24 -> 8 bands on 32^3: 134 against 125 us; 96 -> 32 real on 32^3: 225
//  against 167).  Of 52 shapes from 8 -> 8 on 8^3 to 432 -> 144 on 64^3 none runs slower than the FP64 kernel.
static bool rotation_wins(double n, int rows, int k, int m, bool real, int items_per_tile) {
    auto up = [real](int c) { return real ? 2.0 * (cdiv((c + 1) / 2, 16) * 16) : (double)(cdiv(c, 16) * 16); };
    const double t64 = (real ? 2.0 : 8.0) * n * up(k) * up(m) / 1.15e12;
    const double trns = 50e-6 + n / 128.0 * items_per_tile * 1.4e-8 + rows * n * 3.3e-11;
    return t64 > 1.15 * trns;
}

// The passes have a row of blocks for every row (65,535 at most); more rows than that stay with the FP64 kernels.
constexpr int MAX_ROWS = 65535;

static rsdft_status gram_within(rsdft_ctx *ctx, size_t limit, const RowBlocks &A0, const RowBlocks &B0,
                                const RowBlocks *B1, bool real, bool herm, double2 *g0, double2 *g1, int ldg,
                                double scale, cudaStream_t st, RnsLease &lease) {
    const int na = rows_of(A0), nb = rows_of(B0), blocks = B1 ? 2 : 1;
    const RowBlocks A = real ? pair_rows(A0) : A0, B = real ? pair_rows(B0) : B0;
    const int ra = rows_of(A), rb = rows_of(B);
    bool same = true;
    for (int i = 0; i < 3; ++i) same = same && A.cnt[i] == B.cnt[i] && (A.cnt[i] == 0 || A.ptr[i] == B.ptr[i]);
    const long long n = ctx->n;
    const int PL = real ? 1 : 2, M = real ? 2 * ra : ra, N = real ? 2 * rb : rb;
    const int NT = real ? 256 : 128;
    const int mt = cdiv(M, 128), nt = cdiv(N, NT);
    const double frac = (herm ? 0.5 : 1.0) * blocks;
    const int R = (same ? 0 : ra) + rb * blocks;
    int tiles = 0;
    for (int t = 0; t < mt; ++t) tiles += herm ? nt - t * 128 / NT : nt;
    tiles *= blocks;
    // chunks of points, equal and multiples of 64
    const size_t per_point = (size_t)NM * R * 4;
    const long long most = std::max<long long>(4096, (long long)(limit / per_point) / 64 * 64);
    const int nchunk = cdiv(n, most);
    const int ld = cdiv(cdiv(n, nchunk), 64) * 64;
    const int kbt = ld / 64;
    // K splits: whole waves of one CTA per SM (or at least three of them), 16 K-blocks a CTA
    int splits = 1;
    double best = 0.0;
    for (int s = 1; s <= 16 && (s == 1 || kbt / s >= 16); ++s) {
        const long long it = (long long)tiles * NM * s;
        const double eff = (double)it / (double)((it + ctx->num_sms - 1) / ctx->num_sms * ctx->num_sms);
        if (eff > best + 0.02) { best = eff; splits = s; }
    }
    const int S = std::max(1, std::min<int>(64, (int)(n / 4096)));
    const int npad = cdiv(N, 8) * 8;
    const size_t out_elems = (size_t)splits * NM * PL * M * npad * blocks;
    Carver cv{nullptr};
    for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
            if (!rns_buffer(ctx, cv.at, st, lease)) return RSDFT_OK;
            cv = Carver{(unsigned char *)lease.slot->buf.p};
        }
        __nv_bfloat16 *res = cv.take<__nv_bfloat16>((size_t)NM * R * 2 * ld);
        short *out16 = cv.take<short>(out_elems);
        Stat *stat = cv.take<Stat>((size_t)R * S * 2);
        int *scl = cv.take<int>(2 * (size_t)R);
        if (pass == 0) continue;
        int *flag = lease.flag();
        const int rowB = same ? 0 : ra;
        lease.used = true;
        ProfScope ps(ctx, RSDFT_K_GRAM, (real ? 2.0 : 8.0) * (double)n * frac * na * (herm ? na + 1.0 : (double)nb),
                     16.0 * (double)n * R, st, 0);
        RS_CUDA(ctx, cudaMemsetAsync(flag, 0, sizeof(int), st));
        struct Src { const RowBlocks *b; RowBlocks r; int row0, cnt; };
        const RowBlocks Bp1 = B1 ? (real ? pair_rows(*B1) : *B1) : B;
        const Src srcs[3] = {{nullptr, A, 0, same ? 0 : ra}, {nullptr, B, rowB, rb}, {nullptr, Bp1, rowB + rb, B1 ? rb : 0}};
        for (const Src &s : srcs) {
            if (s.cnt <= 0) continue;
            k_row_stat<<<dim3(S, s.cnt), 256, 0, st>>>(s.r, n, S, stat + (size_t)s.row0 * S * 2);
            count_launch(ctx);
        }
        k_row_scale<<<cdiv(R, 128), 128, 0, st>>>(stat, S, R, real ? 0 : 1, scl, flag);
        count_launch(ctx);
        RS_LAUNCHED(ctx, "k_row_scale");
        CUtensorMap mA, mB;
        {
            const long long st3[3] = {real ? 2LL * ld : 4LL * ld, 2LL * ld, 4LL * ld * R};
            const long long da[4] = {ld, real ? 2 * ra : ra, PL, NM};
            const long long db[4] = {ld, real ? 2 * rb * blocks : rb * blocks, PL, NM};
            const int ba[4] = {64, 128, 1, 1}, bb[4] = {64, NT, 1, 1};
            RS_TRY(tc::tensor_map_bf16(ctx, &mA, res, 4, da, st3, ba, CU_TENSOR_MAP_SWIZZLE_128B));
            RS_TRY(tc::tensor_map_bf16(ctx, &mB, res + (size_t)rowB * 2 * ld, 4, db, st3, bb, CU_TENSOR_MAP_SWIZZLE_128B));
        }
        Args a{};
        a.items = tiles * NM * splits;
        a.mt = mt;
        a.nt = nt;
        a.nstep = NT;
        a.boxn = NT;
        a.M = M;
        a.N = N;
        a.npad = npad;
        a.herm = herm ? 1 : 0;
        a.blocks = blocks;
        a.tiles = tiles;
        a.kb_split = cdiv(kbt, splits);
        a.out16 = out16;
        a.flag = flag;
        a.flag_w = flag;
        for (int c = 0; c < nchunk; ++c) {
            const long long p0 = (long long)c * ld;
            for (const Src &s : srcs) {
                if (s.cnt <= 0) continue;
                k_residues<<<dim3(cdiv(ld, 1024), s.cnt), 256, 0, st>>>(s.r, n, p0, ld, R, s.row0, 0, scl, nullptr,
                                                                        1 << 30, 0, 0, res, flag);
                count_launch(ctx);
            }
            RS_LAUNCHED(ctx, "k_residues");
            a.kb_total = cdiv(std::min<long long>(ld, n - p0), 64);
            a.accumulate = c > 0;
            if (real) RS_TRY((launch_gemm<true, false>(ctx, mA, mB, mB, a, st)));
            else RS_TRY((launch_gemm<false, false>(ctx, mA, mB, mB, a, st)));
        }
        k_crt_gram<<<dim3(cdiv((long long)na * nb, 128), blocks), 128, 0, st>>>(
            out16, splits, M, N, npad, blocks, real ? 1 : 0, A0.cnt[0], A0.cnt[1], B0.cnt[0], B0.cnt[1], na, nb, herm ? 1 : 0,
            scl, scl + 2 * rowB, scale, g0, g1, ldg, flag);
        count_launch(ctx);
        RS_LAUNCHED(ctx, "k_crt_gram");
    }
    return RSDFT_OK;
}

rsdft_status rns_gram(rsdft_ctx *ctx, const RowBlocks &A, const RowBlocks &B0, const RowBlocks *B1, bool real, bool herm,
                      double2 *g0, double2 *g1, int ldg, double scale, cudaStream_t st, RnsLease &lease) {
    const int rows = std::max(rows_of(real ? pair_rows(A) : A), rows_of(real ? pair_rows(B0) : B0));
    if (rows > MAX_ROWS || !gram_wins(ctx->n)) return RSDFT_OK;
    for (size_t limit = RNS_BYTES; limit >= RNS_BYTES / 64 && !lease.used; limit /= 8)
        RS_TRY(gram_within(ctx, limit, A, B0, B1, real, herm, g0, g1, ldg, scale, st, lease));
    return RSDFT_OK;
}

static rsdft_status rotate_within(rsdft_ctx *ctx, size_t limit, const RowBlocks &Y0, const double2 *c, int ldc, int m,
                                  bool real, const double2 *base, int sign, double2 *out0, double2 *out1,
                                  cudaStream_t st, RnsLease &lease) {
    const RowBlocks Y = real ? pair_rows(Y0) : Y0;
    const int R = rows_of(Y), k = rows_of(Y0);
    const long long n = ctx->n;
    const int segs = Y0.cnt[1] + Y0.cnt[2] > 0 ? 2 : 1;
    const int PL = real ? 1 : 2, NT = real ? 256 : 128;
    const int nt = cdiv(m, NT), nstep = cdiv(cdiv(m, nt), 16) * 16, nbp = nt * nstep, nquad = cdiv(m, 4);
    Seg sg[2];
    sg[0] = Seg{{Y0.cnt[0], 0}, {0, 0}, real ? 2 * Y.cnt[0] : Y.cnt[0]};
    sg[1] = Seg{{Y0.cnt[1], Y0.cnt[2]}, {Y0.cnt[0], Y0.cnt[0] + Y0.cnt[1]},
                real ? 2 * (Y.cnt[1] + Y.cnt[2]) : Y.cnt[1] + Y.cnt[2]};
    int kb[2], kpad[2], bits[2];
    for (int s = 0; s < segs; ++s) {
        kb[s] = cdiv(sg[s].k, 64);
        kpad[s] = kb[s] * 64;
        // |y| over the K products of a sum is at most sqrt(K) times the largest
        int h = 0;
        while ((1LL << (2 * h)) < (long long)sg[s].k * PL) ++h;
        bits[s] = T_ROW - h;
    }
    const double out_bytes = (double)NM * segs * PL * nquad * 4;
    const size_t per_point = (size_t)NM * R * 4 + (size_t)out_bytes;
    const long long most = std::max<long long>(4096, (long long)(limit / per_point) / 128 * 128);
    const int nchunk = cdiv(n, most);
    const int ld = cdiv(cdiv(n, nchunk), 128) * 128;
    const int S = std::max(1, std::min<int>(64, (int)(n / 4096)));
    Carver cv{nullptr};
    for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
            if (!rns_buffer(ctx, cv.at, st, lease)) return RSDFT_OK;
            cv = Carver{(unsigned char *)lease.slot->buf.p};
        }
        __nv_bfloat16 *res = cv.take<__nv_bfloat16>((size_t)NM * R * 2 * ld);
        unsigned *out8 = cv.take<unsigned>((size_t)NM * segs * PL * nquad * ld);
        int *pmax = cv.take<int>((size_t)segs * n);
        int *sc = cv.take<int>((size_t)segs * m);
        Stat *stat = cv.take<Stat>((size_t)R * S * 2);
        int *scl = cv.take<int>(2 * (size_t)R);
        __nv_bfloat16 *cres[2];
        for (int s = 0; s < segs; ++s) cres[s] = cv.take<__nv_bfloat16>((size_t)NM * PL * nbp * kpad[s]);
        if (pass == 0) continue;
        int *flag = lease.flag();
        lease.used = true;
        const int mrows = real ? pairs_up(m) : m;
        ProfScope ps(ctx, RSDFT_K_ROTATE, (real ? 2.0 : 8.0) * (double)n * k * m,
                     16.0 * (double)n * (R + mrows * (1 + (out1 ? 1 : 0) + (base ? 1 : 0))), st, 0);
        RS_CUDA(ctx, cudaMemsetAsync(flag, 0, sizeof(int), st));
        RS_CUDA(ctx, cudaMemsetAsync(pmax, 0, (size_t)segs * n * sizeof(int), st));
        k_row_stat<<<dim3(S, R), 256, 0, st>>>(Y, n, S, stat);
        k_row_scale<<<cdiv(R, 128), 128, 0, st>>>(stat, S, R, real ? 0 : 1, scl, flag);
        count_launch(ctx, 2);
        RS_LAUNCHED(ctx, "k_row_scale");
        CUtensorMap mA, mB[2];
        for (int s = 0; s < segs; ++s) {
            const int r0 = s ? Y.cnt[0] : 0, nr = s ? Y.cnt[1] + Y.cnt[2] : Y.cnt[0];
            // enough CTAs for small grids: at least 8 per SM, at least 16 rows each
            const int want = std::max(1, std::min(cdiv(nr, 16), cdiv(8LL * ctx->num_sms, cdiv(n, 256))));
            const int per = cdiv(cdiv(nr, want), 8) * 8;
            k_point_max<<<dim3(cdiv(n, 256), cdiv(nr, per)), 256, 0, st>>>(Y, r0, nr, n, per, scl, pmax + (size_t)s * n);
            k_coef_scale<<<m, 32, 0, st>>>(c, ldc, sg[s], real ? 1 : 0, scl + 2 * r0, sc + (size_t)s * m, flag);
            count_launch(ctx, 2);
        }
        for (int s = 0; s < segs; ++s) {
            k_coef_residues<<<cdiv((long long)nbp * kpad[s] / 2, 256), 256, 0, st>>>(c, ldc, sg[s], real ? 1 : 0, m, nbp, kpad[s],
                                                                          scl + 2 * (s ? Y.cnt[0] : 0), sc + (size_t)s * m, cres[s], flag);
            count_launch(ctx);
            const long long dims[4] = {kpad[s], nbp, PL, NM};
            const long long str[3] = {2LL * kpad[s], 2LL * kpad[s] * nbp, 2LL * kpad[s] * nbp * PL};
            const int box[4] = {64, nstep, 1, 1};
            RS_TRY(tc::tensor_map_bf16(ctx, &mB[s], cres[s], 4, dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B));
        }
        RS_LAUNCHED(ctx, "k_coef_residues");
        if (segs == 1) mB[1] = mB[0];
        {
            const long long dims[4] = {ld, real ? 2 * R : R, PL, NM};
            const long long str[3] = {real ? 2LL * ld : 4LL * ld, 2LL * ld, 4LL * ld * R};
            const int box[4] = {64, 64, 1, 1};
            RS_TRY(tc::tensor_map_bf16(ctx, &mA, res, 4, dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B));
        }
        Args a{};
        a.nt = nt;
        a.nstep = nstep;
        a.boxn = nstep;
        a.N = m;
        a.segs = segs;
        for (int s = 0; s < 2; ++s) {
            a.kb[s] = s < segs ? kb[s] : 0;
            a.row0[s] = s ? (real ? 2 * Y.cnt[0] : Y.cnt[0]) : 0;
        }
        a.ldp = ld;
        a.out8 = out8;
        a.flag = flag;
        a.flag_w = flag;
        for (int ch = 0; ch < nchunk; ++ch) {
            const long long p0 = (long long)ch * ld;
            const int np = (int)std::min<long long>(ld, n - p0);
            if (np <= 0) break;
            k_residues<<<dim3(cdiv(ld, 1024), R), 256, 0, st>>>(Y, n, p0, ld, R, 0, 1, scl, pmax, Y.cnt[0], bits[0],
                                                                bits[segs - 1], res, flag);
            count_launch(ctx);
            RS_LAUNCHED(ctx, "k_residues");
            a.M = np;
            a.mt = cdiv(np, 128);
            a.items = a.mt * NM * segs * nt;
            if (real) RS_TRY((launch_gemm<true, true>(ctx, mA, mB[0], mB[1], a, st)));
            else RS_TRY((launch_gemm<false, true>(ctx, mA, mB[0], mB[1], a, st)));
            const dim3 g(cdiv(np, 256), nquad);
            if (real)
                k_crt_rot<true><<<g, 256, 0, st>>>(out8, segs, m, ld, n, p0, np, pmax, bits[0], bits[segs - 1], sc, m, base,
                                                   sign, out0, out1, flag);
            else
                k_crt_rot<false><<<g, 256, 0, st>>>(out8, segs, m, ld, n, p0, np, pmax, bits[0], bits[segs - 1], sc, m, base,
                                                    sign, out0, out1, flag);
            count_launch(ctx);
            RS_LAUNCHED(ctx, "k_crt_rot");
        }
    }
    return RSDFT_OK;
}

rsdft_status rns_rotate(rsdft_ctx *ctx, const RowBlocks &Y, const double2 *c, int ldc, int m, bool real,
                        const double2 *base, int sign, double2 *out0, double2 *out1, cudaStream_t st, RnsLease &lease) {
    const int segs = Y.cnt[1] + Y.cnt[2] > 0 ? 2 : 1, nt = cdiv(m, real ? 256 : 128);
    const int rows = rows_of(real ? pair_rows(Y) : Y);
    if (Y.cnt[0] <= 0 || rows > MAX_ROWS || cdiv(m, 4) > MAX_ROWS ||
        !rotation_wins((double)ctx->n, rows, rows_of(Y), m, real, NM * segs * nt))
        return RSDFT_OK;
    for (size_t limit = RNS_BYTES; limit >= RNS_BYTES / 64 && !lease.used; limit /= 8)
        RS_TRY(rotate_within(ctx, limit, Y, c, ldc, m, real, base, sign, out0, out1, st, lease));
    return RSDFT_OK;
}

rsdft_status rns_poison(rsdft_ctx *ctx, double2 *out, long long cnt, cudaStream_t st, const RnsLease &lease) {
    k_poison<<<std::min(cdiv(cnt, 256), 4 * ctx->num_sms), 256, 0, st>>>(out, cnt, lease.flag());
    count_launch(ctx);
    RS_LAUNCHED(ctx, "k_poison");
    return RSDFT_OK;
}

}  // namespace rsdft
