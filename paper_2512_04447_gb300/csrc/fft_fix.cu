// FP64 3D FFT passes of H psi, TPA and the field solvers in 64-bit fixed point (fix_fft.h).
//
// The passes are those of fft.cu (xy planes, z slabs with the per-G factor, xy planes with the
// epilogue; digit-reversed spectrum in between), FP64 in and out.  A block (an xy plane, or the
// slab of one y) is scaled to integers by its largest value; between the passes the buffer
// holds integers, and (exponent, bits) of every block says what they are worth, so that the
// next pass brings its rows to one exponent.  The per-G factor keeps its relative precision (53
// bits, the kinetic one 61): products are formed with a normalised factor and its exponent and shifted to the
// largest one of the slab.
//
// What bounds it: the FP64 passes ran at some 80% of the FP64 pipe; the integer instructions on
// 64-bit values bound these.  144 bands on 64^3, one GB300: forward 3.23 -> 0.68 ms (1.49 with
// the projector gather, then 1.77 on its own), z 3.66 -> 0.87 ms, inverse 5.9 -> 2.2 ms with the
// projector scatter; TPA of 53
// bands on 45^3 1.94 -> 0.54 ms.  Errors against 64-bit FFTs are those of the reference itself:
// relative 4.4e-16 (FP64 passes 4.8e-16) for TPA, 7.1e-16 (8.4e-16) for H psi.
//
// Non-finite values make a block's exponent BAD, which every following pass hands on, and the
// outputs of that band NaN.
#include <algorithm>
#include <cmath>

#include "fft_common.h"
#include "fix_fft.h"
#include "proj.h"
#include "rsdft_internal.h"

namespace rsdft {

using fix::I2;
using fix::i64;
using fix::u64;
using fix::W4;

namespace {

constexpr int BAD = 0x40000000;        // exponent of a block with non-finite values
constexpr int EMPTY = -0x10000000;     // exponent of a block of zeros
constexpr int MAX_THREADS = 768;       // 85 registers: three CTAs of 256 threads on a 64 x 64 plane
constexpr int HEAD = 32;               // reduction words ahead of the plane
constexpr int SHIFTS = MAX_N * 4;      // row shifts behind it (xy planes with padded rows keep them in the padding)

struct FixTabs {
    AxisPlan ax[3];
    const W4 *tw[3];
    const longlong2 *kin[3];           // G_a^2 / (2 n) in units of 2^-kexp, by position: whole part, 2^32 times the rest
    int kexp;
    const double *g2[3], *g1[3];       // by position
    const double *g2abs[3];            // G_a^2 by |frequency index|
    const unsigned char *fabs[3];      // |frequency index| by position
    double inv_n;
};

struct Meta { int e, bits; };          // block values are integers below 2^bits times 2^e

__device__ __forceinline__ unsigned mag_hi(I2 v) {
    const int hx = (int)(v.x >> 32), hy = (int)(v.y >> 32);
    return (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
}
__device__ __forceinline__ int bits_hi(unsigned m) { return 64 - __clz((int)m); }   // 32 for m = 0
__device__ __forceinline__ int bits_of(I2 v) { return fix::bits_of((u64)(v.x ^ (v.x >> 63)) | (u64)(v.y ^ (v.y >> 63))); }

// Every thread's word joined over the block (or / max); red: a zeroed word of shared memory
__device__ __forceinline__ unsigned block_or(unsigned v, unsigned *red) {
    v = __reduce_or_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicOr(red, v);
    __syncthreads();
    return *red;
}
__device__ __forceinline__ int block_max(int v, int *red) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(red, v);
    __syncthreads();
    return *red;
}

// State of one transform: every component is below 2^bits, in units of 2^e; stage counter.
struct Scale { int bits, e, n; };

// sh: right shift of the inputs (left where negative)
template <int R, bool INV, bool RAW>
__device__ __forceinline__ unsigned bfly(I2 *s, int base, int step, int j, int twstep, const W4 *tw, int sh, int s0,
                                         bool twiddle) {
    I2 v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        v[q] = s[base + q * step];
        if (RAW) {
            v[q].x = fix::from_double((int)(v[q].x >> 32), (unsigned)v[q].x, s0);
            v[q].y = fix::from_double((int)(v[q].y >> 32), (unsigned)v[q].y, s0);
        }
    }
    if (!RAW) {
        if (sh > 0) {
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = fix::rshift(v[q], sh);
        } else if (sh < 0) {
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = I2{v[q].x << -sh, v[q].y << -sh};
        }
    }
    // times w^(j p) / 4; j = 0 (a whole warp's lines share j) is a shift
    auto turn = [&] {
        v[0] = fix::rshift(v[0], 2);
        if (j == 0) {
#pragma unroll
            for (int p = 1; p < R; ++p) v[p] = fix::rshift(v[p], 2);
            return;
        }
#pragma unroll
        for (int p = 1; p < R; ++p) {
            const int4 w = __ldg(reinterpret_cast<const int4 *>(tw + j * p * twstep));
            v[p] = fix::mul_w<INV>(v[p], W4{w.x, w.y, w.z, w.w});
        }
    };
    if (INV && twiddle) turn();
    fix::dft<R, INV>(v);
    if (!INV && twiddle) turn();
    unsigned m = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        s[base + q * step] = v[q];
        m |= mag_hi(v[q]);
    }
    return m;
}

template <int R, bool INV, bool RAW>
__device__ __forceinline__ unsigned stage(I2 *s, const AxisPlan &ax, int st, const W4 *tw, int nlines, unsigned nlmag,
                                          int lstride, int es, int sh, int s0) {
    const int N = ax.N, len = ax.len[st], sub = ax.sub[st];
    const unsigned smag = ax.submag[st];
    const int total = N / R * nlines, twstep = N / len, step = sub * es;
    unsigned m = 0;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int bf = qdiv(idx, nlmag), line = idx - bf * nlines;   // consecutive threads: consecutive lines
        const int b = qdiv(bf, smag), j = bf - b * sub;
        m |= bfly<R, INV, RAW>(s, line * lstride + (b * len + j) * es, step, j, twstep, tw, sh, s0, sub > 1);
    }
    return m;
}

// bits that the first stage of a transform provides for
__device__ __forceinline__ int first_growth(const AxisPlan &ax, bool inv) {
    return fix::growth(ax.radix[inv ? ax.nstage - 1 : 0]);
}

// All stages of nlines transforms in shared memory (fft.cu's fft_lines).  Each stage brings its
// inputs to the largest scale at which its sums cannot overflow, from the bits that the stage
// before left (slot: three words in turn, so that one can be cleared while the others are in use).
// RAW: the first stage reads doubles, scaled by 2^s0 to sc.bits as it reads them.
template <bool INV, bool RAW>
__device__ void lines(I2 *s, const AxisPlan &ax, const W4 *tw, int nlines, unsigned nlmag, int lstride, int es, Scale &sc,
                      int s0, unsigned *slot) {
    for (int t = 0; t < ax.nstage; ++t) {
        const int st = INV ? ax.nstage - 1 - t : t;
        const int r = ax.radix[st];
        const bool twiddle = ax.sub[st] > 1;
        // (an inverse stage turns before it sums, at 2^62 at most)
        const int room = fix::TOP - fix::growth(r), sh = sc.bits - (INV && twiddle ? min(room + 2, 62) : room);
        sc.e += sh + (twiddle ? 2 : 0);
        const int now = sc.n % 3;
        if (threadIdx.x == 0) slot[(now + 1) % 3] = 0;
        unsigned m;
        if (RAW && t == 0) {
            switch (r) {
                case 2: m = stage<2, INV, RAW>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                case 3: m = stage<3, INV, RAW>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                case 4: m = stage<4, INV, RAW>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                case 5: m = stage<5, INV, RAW>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                default: m = stage<8, INV, RAW>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
            }
        } else {
            switch (r) {
                case 2: m = stage<2, INV, false>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                case 3: m = stage<3, INV, false>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                case 4: m = stage<4, INV, false>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                case 5: m = stage<5, INV, false>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
                default: m = stage<8, INV, false>(s, ax, st, tw, nlines, nlmag, lstride, es, sh, s0); break;
            }
        }
        sc.bits = bits_hi(block_or(m, slot + now));
        ++sc.n;
    }
}

// shifts that bring rows of the given blocks to one exponent, the largest value just below
// 2^bits: row r is read as rshift(v, shift[r]) (left for negative shifts) in units of 2^(return value);
// BAD if a block is.
__device__ __forceinline__ int row_shifts(const Meta *meta, int rows, int bits, int *shift, int stride, int *red) {
    int top = EMPTY, bad = 0;
    Meta m{EMPTY, 0};
    if ((int)threadIdx.x < rows) {
        m = meta[threadIdx.x];
        bad = m.e == BAD;
        top = bad ? EMPTY : m.e + m.bits;
    }
    const int any = __syncthreads_or(bad);
    if ((int)threadIdx.x == 0) *red = EMPTY;
    __syncthreads();
    const int e = block_max(top, red) - bits;
    if ((int)threadIdx.x < rows) shift[threadIdx.x * stride] = min(max(e - m.e, -62), 63);
    __syncthreads();
    return any ? BAD : (e < EMPTY / 2 ? 0 : e);
}
__device__ __forceinline__ i64 shifted(i64 v, int s) {
    if (s < 0) return v << -s;
    return s > 62 ? 0 : fix::rshift(v, s);
}

__device__ __forceinline__ double value(i64 v, int e) {
    bool odd;
    const u64 b = fix::to_double_bits(v, e, &odd);
    return odd ? scalbn((double)v, e) : __longlong_as_double((long long)b);
}

// v w 2^-64 for w given as (h, l) with |w| < 2^62 (half: rounds)
__device__ __forceinline__ i64 mul_hl(i64 v, int h, int l) {
    const int vl = fix::lo_of(v), vh = fix::hi_of(v);
    return fix::mw(vh, h, fix::mw(vl, h, fix::mw(vh, l, 0x80000000ll)) >> 32);
}
// (v w + u z) 2^-64
__device__ __forceinline__ i64 mul2_hl(i64 v, int wh, int wl, i64 u, int zh, int zl) {
    const int vl = fix::lo_of(v), vh = fix::hi_of(v), ul = fix::lo_of(u), uh = fix::hi_of(u);
    const i64 mid = fix::mw(vl, wh, fix::mw(vh, wl, 0x80000000ll)) + fix::mw(ul, zh, fix::mw(uh, zl, 0));
    return fix::mw(vh, wh, fix::mw(uh, zh, mid >> 32));
}

// fft.cu's gather on an integer plane in units of 2^e, with the factors in units of 2^-62: the values
// leave room for the sum over the widest disc
__device__ __forceinline__ void gather_plane_fix(const I2 *plane, int RS, const Discs &t, int z, int Nx, int e,
                                                 double2 *__restrict__ part) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int d1 = t.plane_start[z + 1];
    for (int d = t.plane_start[z] + (threadIdx.x >> 5); d < d1; d += nw) {
        const int2 m = __ldg(reinterpret_cast<const int2 *>(t.meta + d));
        const int rows = disc_rows(m.y), w = disc_width(m.y);
        const int4 *gx = t.gxfix + (size_t)d * t.wmax;
        i64 s[6] = {0, 0, 0, 0, 0, 0};
        for (int r0 = 0; r0 < rows; r0 += 32) {
            int4 q = make_int4(0, 0, 0, 0);
            int hl = 0;
            if (r0 + lane < rows) {
                const DiscRowFix *rp = t.rowfix + m.x + r0 + lane;
                q = __ldg(reinterpret_cast<const int4 *>(rp));
                hl = __ldg(&rp->hl);
            }
            const I2 *row = plane + (q.x & 255) * RS;
            int x = disc_x0(m.y);
            I2 U{0, 0}, V{0, 0};   // sums of gx v, hx v along the row
#pragma unroll 2
            for (int j = 0; j < w; ++j) {
                const int4 k = __ldg(gx + j);
                I2 v = row[x];
                if (!in_row(q.x, j)) v = I2{0, 0};
                U.x += mul_hl(v.x, k.x, k.y);
                U.y += mul_hl(v.y, k.x, k.y);
                V.x += mul_hl(v.x, k.z, k.w);
                V.y += mul_hl(v.y, k.z, k.w);
                x = x + 1 == Nx ? 0 : x + 1;
            }
            U = fix::rshift(U, 5);   // room for the 128 rows' sum
            V = fix::rshift(V, 5);
            s[0] += mul_hl(U.x, q.y, q.z);
            s[1] += mul_hl(U.y, q.y, q.z);
            s[2] += mul_hl(V.x, q.y, q.z);
            s[3] += mul_hl(V.y, q.y, q.z);
            s[4] += mul_hl(U.x, q.w, hl);
            s[5] += mul_hl(U.y, q.w, hl);
        }
#pragma unroll
        for (int k = 0; k < 6; ++k)
            for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        if (lane < 3) {
            const i64 re = lane == 0 ? s[0] : (lane == 1 ? s[2] : s[4]), im = lane == 0 ? s[1] : (lane == 1 ? s[3] : s[5]);
            part[(size_t)d * 3 + lane] = make_double2(value(re, e + 9), value(im, e + 9));
        }
    }
}

// fft.cu's scatter into an integer plane of sc: the coefficients go to the plane's unit, or the plane
// to the coefficients' where those are larger.  Returns false where a coefficient is not finite.
__device__ __forceinline__ bool scatter_plane_fix(I2 *plane, int RS, const Discs &t, int z, int Nx, int Ny,
                                                  const double2 *__restrict__ ab, I2 *uw, int room, Scale &sc, int *red) {
    const int lane = threadIdx.x & 31;
    const int d0 = t.plane_start[z], nd = t.plane_start[z + 1] - d0;
    if (nd == 0) return true;
    const double *a = reinterpret_cast<const double *>(ab + 3 * (size_t)d0);
    int hmax = 0;
    for (int i = threadIdx.x; i < 6 * nd; i += blockDim.x) hmax = max(hmax, __double2hiint(a[i]) & 0x7fffffff);
    const int top = block_max(hmax, red) >> 20;
    if (top == 0x7ff) return false;
    // a point gets at most nd times 3 of the largest coefficient: below 2^59 units of 2^e
    const int e = max(sc.e, top - 1022 + 3 + (32 - __clz(nd)) - 60);
    if (e > sc.e) {
        const int sh = min(e - sc.e, 63);
        for (int i = threadIdx.x; i < Ny * RS; i += blockDim.x) {
            const I2 v = plane[i];
            plane[i] = I2{shifted(v.x, sh), shifted(v.y, sh)};
        }
        sc.e = e;
    }
    auto in = [&](double v) { return fix::from_double(__double2hiint(v), (unsigned)__double2loint(v), 4 - e); };
    // U and W of disc d at x offset l
    auto make_uw = [&](int d, int l, I2 &U, I2 &W) {
        const int4 g = __ldg(t.gxfix + (size_t)d * t.wmax + l);
        const double2 A = __ldg(ab + 3 * (size_t)d), Bx = __ldg(ab + 3 * (size_t)d + 1), By = __ldg(ab + 3 * (size_t)d + 2);
        U = I2{mul2_hl(in(A.x), g.x, g.y, in(Bx.x), g.z, g.w), mul2_hl(in(A.y), g.x, g.y, in(Bx.y), g.z, g.w)};
        W = I2{mul_hl(in(By.x), g.x, g.y), mul_hl(in(By.y), g.x, g.y)};
    };
    int base = d0;
    for_discs(t, z, room ? room : nd, [&](int c0, int n) {
        base = d0 + c0;
        if (room == 0) return;   // no room beside the plane: U and W where they are used
        for (int i = threadIdx.x; i < n * t.wmax; i += blockDim.x) {
            const int d = i / t.wmax;
            make_uw(base + d, i - d * t.wmax, uw[2 * i], uw[2 * i + 1]);
        }
    }, [&](int d, int ja, int jb) {
        const int2 m = __ldg(reinterpret_cast<const int2 *>(t.meta + d));
        const int rows = disc_rows(m.y);
        const I2 *ue = uw + 2 * (size_t)(d - base) * t.wmax;
        for (int r0 = 0; r0 < rows; r0 += 32) {
            int4 q = make_int4(0, 0, 0, 0);
            int hl = 0;
            if (r0 + lane < rows) {
                const DiscRowFix *rp = t.rowfix + m.x + r0 + lane;
                q = __ldg(reinterpret_cast<const int4 *>(rp));
                hl = __ldg(&rp->hl);
            }
            I2 *row = plane + (q.x & 255) * RS;
            int x = disc_x0(m.y) + ja;
            if (x >= Nx) x -= Nx;
            for (int j = ja; j < jb; ++j) {
                I2 U, W;
                if (room) {
                    U = ue[2 * j];
                    W = ue[2 * j + 1];
                } else {
                    make_uw(d, j, U, W);
                }
                if (in_row(q.x, j)) {
                    I2 o = row[x];
                    o.x += mul2_hl(U.x, q.y, q.z, W.x, q.w, hl);
                    o.y += mul2_hl(U.y, q.y, q.z, W.y, q.w, hl);
                    row[x] = o;
                }
                x = x + 1 == Nx ? 0 : x + 1;
            }
        }
    });
    return true;
}

}  // namespace

// ---- xy forward pass ------------------------------------------------------------
template <Src SRC>
__global__ void __launch_bounds__(MAX_THREADS)
k_xy_forward_fix(FixTabs tb, const double2 *__restrict__ src, const double2 *__restrict__ src2,
                 const double *__restrict__ theta, const int *__restrict__ act, const double *__restrict__ rsrc, int RS,
                 I2 *__restrict__ dst, Meta *__restrict__ meta, Discs discs, int disc_bits, double2 *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *red = reinterpret_cast<int *>(smem_raw);
    I2 *s_plane = reinterpret_cast<I2 *>(smem_raw + HEAD);
    const int Nx = tb.ax[0].N, Ny = tb.ax[1].N, Nz = tb.ax[2].N;
    const int z = blockIdx.x, band = blockIdx.y;
    const int plane = Nx * Ny;
    const size_t n = (size_t)plane * Nz, off = (size_t)z * plane;
    const unsigned nxm = tb.ax[0].nmag;
    unsigned *slot = reinterpret_cast<unsigned *>(red + 4);
    if (threadIdx.x < 8) red[threadIdx.x] = 0;
    int hmax = 0;
    auto put = [&](int i, double2 v) {
        // (subnormal values may have nothing but a low word)
        const int hx = (__double2hiint(v.x) & 0x7fffffff) | (__double2loint(v.x) != 0);
        const int hy = (__double2hiint(v.y) & 0x7fffffff) | (__double2loint(v.y) != 0);
        hmax = max(hmax, max(hx, hy));
        s_plane[pidx(i, Nx, RS, nxm)] = I2{__double_as_longlong(v.x), __double_as_longlong(v.y)};
    };
    const bool gather = SRC == Src::Plain && part;
    if (SRC == Src::Plain) {
        const double2 *in = src + band * n + off;
        stage_in<double2>(plane, [&](int i) { return in[i]; }, put);
    } else if (SRC == Src::Residual) {
        const int b = act[band];
        const double th = theta[b];
        const double2 *hx = src + b * n + off, *x = src2 + b * n + off;
        stage_in<double2>(plane, [&](int i) {
            const double2 h = hx[i], v = x[i];
            return make_double2(h.x - th * v.x, h.y - th * v.y);
        }, put);
    } else {
        const double *in = rsrc + off;
        stage_in<double2>(plane, [&](int i) { return make_double2(in[i], 0.0); }, put);
    }
    __syncthreads();
    const int big = block_max(hmax, red), top = big >> 20;
    Meta *m = meta + (size_t)band * Nz + z;
    if (top == 0x7ff) {
        if (threadIdx.x == 0) *m = Meta{BAD, 0};
        if (gather) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            for (int i = 3 * discs.plane_start[z] + threadIdx.x; i < 3 * discs.plane_start[z + 1]; i += blockDim.x)
                part[(size_t)band * discs.ndisc * 3 + i] = make_double2(nan, nan);
        }
        return;
    }
    int bits0 = fix::TOP - first_growth(tb.ax[0], false);
    if (gather) bits0 = min(bits0, disc_bits);
    const int s0 = bits0 - (top ? top - 1022 : 32 - __clz(big) - 1042);   // subnormal: by its high word's bits
    Scale sc{bits0, -s0, 0};
    if (gather) {
        for (int i = threadIdx.x; i < Ny * RS; i += blockDim.x) {
            const I2 v = s_plane[i];
            s_plane[i] = I2{fix::from_double((int)(v.x >> 32), (unsigned)v.x, s0),
                            fix::from_double((int)(v.y >> 32), (unsigned)v.y, s0)};
        }
        __syncthreads();
        gather_plane_fix(s_plane, RS, discs, z, Nx, -s0, part + (size_t)band * discs.ndisc * 3);
        __syncthreads();
        lines<false, false>(s_plane, tb.ax[0], tb.tw[0], Ny, tb.ax[1].nmag, RS, 1, sc, 0, slot);
    } else {
        lines<false, true>(s_plane, tb.ax[0], tb.tw[0], Ny, tb.ax[1].nmag, RS, 1, sc, s0, slot);
    }
    lines<false, false>(s_plane, tb.ax[1], tb.tw[1], Nx, tb.ax[0].nmag, 1, RS, sc, 0, slot);
    I2 *out = dst + band * n + off;
    for (int i = threadIdx.x; i < plane; i += blockDim.x) out[i] = s_plane[pidx(i, Nx, RS, nxm)];
    if (threadIdx.x == 0) *m = Meta{big == 0 ? EMPTY : sc.e, sc.bits};
}

// ---- z pass with the per-G factor ------------------------------------------------
template <Mid MID> __device__ __forceinline__ double factor(const FixTabs &tb, int x, int y, int z) {
    if constexpr (MID == Mid::GradX) return tb.g1[0][x] * tb.inv_n;
    if constexpr (MID == Mid::GradY) return tb.g1[1][y] * tb.inv_n;
    if constexpr (MID == Mid::GradZ) return tb.g1[2][z] * tb.inv_n;
    const double g2 = tb.g2[0][x] + tb.g2[1][y] + tb.g2[2][z];   // Hartree
    return g2 > 0.0 ? 4.0 * M_PI / g2 * tb.inv_n : 0.0;
}
__device__ __forceinline__ double tpa_factor(double x, double c) {
    const double num = 27.0 + x * (18.0 + x * (12.0 + 8.0 * x));
    return c * num / (num + 16.0 * x * x * x * x);
}
struct Fac { i64 w; int nf; };   // a factor w 2^-nf, 2^61 <= w < 2^62 (0 for factors of zero)
__device__ __forceinline__ Fac fac_of(double f) {   // |f|
    const int hi = __double2hiint(f), e = (hi >> 20) & 0x7ff;
    if (e == 0) return Fac{0, 0};
    return Fac{((i64)((hi & 0xfffff) | 0x100000) << 41) | ((i64)(unsigned)__double2loint(f) << 9), 1084 - e};
}
__device__ __forceinline__ Fac fac_of(longlong2 a, longlong2 b, longlong2 c) {   // their sum, below 2^60
    const u64 rest = (u64)(a.y + b.y + c.y);
    u64 h = (u64)(a.x + b.x + c.x) + (rest >> 32);
    unsigned l = (unsigned)rest;
    int nf = 0;
    if (h == 0) {
        if (l == 0) return Fac{0, 0};
        h = l;
        l = 0;
        nf = 32;
    }
    const int k = __clzll((i64)h) - 2;
    return Fac{(i64)((h << k) | (k < 32 ? (u64)(l >> (32 - k)) : (u64)l << (k - 32))), nf + k};
}

// tab: TPA's factor depends on |k| of each axis only, so a slab evaluates it once per (|kz|, |kx|),
// into shared memory after the slab (table != 0), a quarter of the FP64 divisions; slabs too large
// for that evaluate it per point.
template <Mid MID>
__global__ void __launch_bounds__(MAX_THREADS)
k_z_mid_fix(FixTabs tb, I2 *__restrict__ buf, const double *__restrict__ tkin, const Meta *__restrict__ min,
            Meta *__restrict__ mout, int table) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *red = reinterpret_cast<int *>(smem_raw);
    I2 *s_slab = reinterpret_cast<I2 *>(smem_raw + HEAD);
    const int Nx = tb.ax[0].N, Ny = tb.ax[1].N, Nz = tb.ax[2].N;
    const int y = blockIdx.x, band = blockIdx.y;
    const size_t zstride = (size_t)Nx * Ny;
    I2 *base = buf + band * zstride * Nz + (size_t)y * Nx;
    const int tot = Nx * Nz;
    const unsigned nxm = tb.ax[0].nmag;
    int *shift = reinterpret_cast<int *>(s_slab + tot);
    double *tab = reinterpret_cast<double *>(shift + SHIFTS / 4);
    const int hx = Nx / 2 + 1, hz = Nz / 2 + 1;
    double tk = 1.0;
    if (MID == Mid::Tpa) {
        const double t = tkin[band];
        if (t >= 1e-12) tk = t;
    }
    unsigned *slot = reinterpret_cast<unsigned *>(red + 4);
    if (threadIdx.x > 0 && threadIdx.x < 8) red[threadIdx.x] = threadIdx.x == 1 ? EMPTY : 0;
    const int bits0 = fix::TOP - first_growth(tb.ax[2], false);
    Meta *m = mout + (size_t)band * Ny + y;
    const int e0 = row_shifts(min + (size_t)band * Nz, Nz, bits0, shift, 1, red);
    if (e0 == BAD) {
        if (threadIdx.x == 0) *m = Meta{BAD, 0};
        return;
    }
    stage_in<I2>(tot, [&](int i) {
        const int z = qdiv(i, nxm), x = i - z * Nx;
        return base[z * zstride + x];
    }, [&](int i, I2 v) {
        const int s = shift[qdiv(i, nxm)];
        s_slab[i] = I2{shifted(v.x, s), shifted(v.y, s)};
    });
    if (MID == Mid::Tpa && table) {
        const double gy = tb.g2[1][y];
        for (int i = threadIdx.x; i < hx * hz; i += blockDim.x) {
            const int z = i / hx, x = i - z * hx;
            const double g2 = tb.g2abs[0][x] + gy + tb.g2abs[2][z];
            tab[i] = tpa_factor(0.5 * g2 / tk, tb.inv_n);
        }
    }
    __syncthreads();
    Scale sc{bits0, e0, 0};
    lines<false, false>(s_slab, tb.ax[2], tb.tw[2], Nx, nxm, 1, Nx, sc, 0, slot);
    const longlong2 ky = MID == Mid::Kinetic ? tb.kin[1][y] : make_longlong2(0, 0);
    auto f_of = [&](int i, bool &neg) -> Fac {
        const int z = qdiv(i, nxm), x = i - z * Nx;
        if constexpr (MID == Mid::Kinetic) {
            return fac_of(tb.kin[0][x], ky, tb.kin[2][z]);
        } else if constexpr (MID == Mid::Tpa) {
            if (table) return fac_of(tab[(int)tb.fabs[2][z] * hx + tb.fabs[0][x]]);
            const double g2 = tb.g2[0][x] + tb.g2[1][y] + tb.g2[2][z];
            return fac_of(tpa_factor(0.5 * g2 / tk, tb.inv_n));
        } else {
            const double f = factor<MID>(tb, x, y, z);
            neg = f < 0.0;
            return fac_of(f);
        }
    };
    // bits of the largest product, then the products shifted to it (all bits count: a value that rounds to nothing may
    // meet the largest factor)
    int big = EMPTY;
    bool neg = false;
    for (int i = threadIdx.x; i < tot; i += blockDim.x) {
        const Fac f = f_of(i, neg);
        if (f.w) big = max(big, bits_of(s_slab[i]) - f.nf - 2);
    }
    big = block_max(big, red + 1);
    const int g = big <= EMPTY / 2 ? 0 : fix::TOP - big;   // v w 2^-64 has two bits less than v
    constexpr bool GRAD = MID == Mid::GradX || MID == Mid::GradY || MID == Mid::GradZ;
    for (int i = threadIdx.x; i < tot; i += blockDim.x) {
        bool ng = false;
        const Fac f = f_of(i, ng);
        I2 v{0, 0};
        if (f.w) {
            v = fix::mul_w<false>(s_slab[i], W4{fix::hi_of(f.w), fix::lo_of(f.w), 0, 0});   // v w 2^-64
            const int d = ::min(g - f.nf, 63);
            v = I2{shifted(v.x, -d), shifted(v.y, -d)};
            if (GRAD) v = ng ? fix::rot<false>(v) : fix::rot<true>(v);   // i f v
        }
        s_slab[i] = v;
    }
    __syncthreads();
    sc.bits = fix::TOP;
    sc.e += 64 - (MID == Mid::Kinetic ? tb.kexp : 0) - g;
    lines<true, false>(s_slab, tb.ax[2], tb.tw[2], Nx, nxm, 1, Nx, sc, 0, slot);
    for (int i = threadIdx.x; i < tot; i += blockDim.x) {
        const int z = qdiv(i, nxm), x = i - z * Nx;
        base[z * zstride + x] = s_slab[i];
    }
    if (threadIdx.x == 0) *m = Meta{big <= EMPTY / 2 ? EMPTY : sc.e, sc.bits};
}

// ---- xy inverse pass + epilogue ------------------------------------------------------
enum class FixEpi { Plain, Hpsi, Real };

template <FixEpi EPI>
__global__ void __launch_bounds__(MAX_THREADS)
k_xy_inverse_fix(FixTabs tb, const I2 *__restrict__ buf, const Meta *__restrict__ meta, const double2 *__restrict__ psi,
                 const double *__restrict__ vloc, Discs discs, const double2 *__restrict__ ab, int room, int RS,
                 double2 *__restrict__ out, double *__restrict__ rout) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *red = reinterpret_cast<int *>(smem_raw);
    I2 *s_plane = reinterpret_cast<I2 *>(smem_raw + HEAD);
    const int Nx = tb.ax[0].N, Ny = tb.ax[1].N, Nz = tb.ax[2].N;
    int *shift = reinterpret_cast<int *>(RS > Nx ? s_plane + Nx : s_plane + (size_t)Ny * RS);
    const int sst = RS > Nx ? 4 * RS : 1;
    const int z = blockIdx.x, band = blockIdx.y;
    const int plane = Nx * Ny;
    const size_t n = (size_t)plane * Nz, off = (size_t)z * plane;
    const I2 *in = buf + band * n + off;
    const unsigned nxm = tb.ax[0].nmag;
    unsigned *slot = reinterpret_cast<unsigned *>(red + 4);
    if (threadIdx.x > 0 && threadIdx.x < 8) red[threadIdx.x] = 0;
    const int bits0 = fix::TOP - first_growth(tb.ax[1], true);   // the last radix's stage has no twiddles
    const int e0 = row_shifts(meta + (size_t)band * Ny, Ny, bits0, shift, sst, red);
    Scale sc{bits0, e0, 0};
    if (e0 != BAD) {
        stage_in<I2>(plane, [&](int i) { return in[i]; }, [&](int i, I2 v) {
            const int s = shift[qdiv(i, nxm) * sst];
            s_plane[pidx(i, Nx, RS, nxm)] = I2{shifted(v.x, s), shifted(v.y, s)};
        });
        __syncthreads();
        lines<true, false>(s_plane, tb.ax[1], tb.tw[1], Nx, nxm, 1, RS, sc, 0, slot);
        lines<true, false>(s_plane, tb.ax[0], tb.tw[0], Ny, tb.ax[1].nmag, RS, 1, sc, 0, slot);
    }
    bool good = e0 != BAD;
    if (EPI == FixEpi::Hpsi && good && ab)
        good = scatter_plane_fix(s_plane, RS, discs, z, Nx, Ny, ab + (size_t)band * discs.ndisc * 3,
                                 s_plane + (size_t)Ny * RS + (RS > Nx ? 0 : SHIFTS / 16), room, sc, red + 1);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    auto at = [&](int i) {
        if (!good) return make_double2(nan, nan);
        const I2 v = s_plane[pidx(i, Nx, RS, nxm)];
        return make_double2(value(v.x, sc.e), value(v.y, sc.e));
    };
    if (EPI == FixEpi::Plain) {
        double2 *o = out + band * n + off;
        for (int i = threadIdx.x; i < plane; i += blockDim.x) o[i] = at(i);
    } else if (EPI == FixEpi::Real) {
        double *o = rout + off;
        for (int i = threadIdx.x; i < plane; i += blockDim.x) o[i] = at(i).x;
    } else {
        const double2 *ps = psi + band * n + off;
        const double *vv = vloc + off;
        double2 *o = out + band * n + off;
        for (int i = threadIdx.x; i < plane; i += blockDim.x) {
            const double2 t = at(i), y = ps[i];
            const double vi = vv[i];
            o[i] = make_double2(t.x + vi * y.x, t.y + vi * y.y);
        }
    }
}

// ---- host side -------------------------------------------------------------------------
namespace {

// An xy plane: rows padded to an odd stride, or as they are with the shifts behind them
int plane_stride(const rsdft_ctx *ctx) { return ctx->N[0] | 1; }
size_t plane_smem(const rsdft_ctx *ctx) {
    return HEAD + (size_t)(ctx->N[0] | 1) * ctx->N[1] * sizeof(I2) + (ctx->N[0] & 1 ? SHIFTS : 0);
}

// what the passes take: planes and slabs of at most 227 KB with an odd stride
rsdft_status check_plane(rsdft_ctx *ctx) {
    const size_t odd = (size_t)(ctx->N[0] | 1) * ctx->N[1] * sizeof(I2), slab = (size_t)ctx->N[0] * ctx->N[2] * sizeof(I2);
    if (std::max(odd, slab) > MAX_DYN_SMEM)
        return fail(ctx, RSDFT_E_INVALID, "plane needs %zu B of shared memory", std::max(odd, slab));
    return RSDFT_OK;
}

// (at least one thread a row)
int threads_for(const rsdft_ctx *ctx, size_t smem, int points, const dim3 &grid) {
    return pass_threads(smem, points, (long long)grid.x * grid.y, ctx->num_sms, 128);
}

// buf: the buffer between the passes, which says whose exponents
rsdft_status ensure_meta(rsdft_ctx *ctx, const double2 *buf, int nb, Meta **planes, Meta **slabs, cudaStream_t st) {
    Scratch &m = buf == ctx->scf.cbuf ? ctx->fix.field_meta : ctx->fix.meta;
    RS_TRY(grow(ctx, m, (size_t)nb * (ctx->N[1] + ctx->N[2]) * sizeof(Meta), st));
    *planes = static_cast<Meta *>(m.p);
    *slabs = *planes + (size_t)nb * ctx->N[2];
    return RSDFT_OK;
}

FixTabs tabs_of(const rsdft_ctx *ctx) {
    FixTabs t;
    for (int a = 0; a < 3; ++a) {
        t.ax[a] = ctx->fft.ax[a];
        t.tw[a] = static_cast<const W4 *>(ctx->fix.tw[a]);
        t.kin[a] = ctx->fix.kin[a];
        t.g2[a] = ctx->fft.g2pos[a];
        t.g1[a] = ctx->fft.gpos[a];
        t.g2abs[a] = ctx->fix.g2abs[a];
        t.fabs[a] = ctx->fix.fabs[a];
    }
    t.kexp = ctx->fix.kexp;
    t.inv_n = 1.0 / (double)ctx->n;
    return t;
}

}  // namespace

rsdft_status fft_xy_forward(rsdft_ctx *ctx, Src kind, const double2 *src, const double2 *src2, const double *theta,
                            const int *act, const double *rsrc, double2 *dst, int nb, cudaStream_t st, double2 *part) {
    if (nb <= 0) return RSDFT_OK;
    RS_TRY(check_plane(ctx));
    Meta *mp, *ms;
    RS_TRY(ensure_meta(ctx, dst, nb, &mp, &ms, st));
    const int RS = plane_stride(ctx);
    const size_t sm = HEAD + (size_t)RS * ctx->N[1] * sizeof(I2);
    const dim3 grid(ctx->N[2], nb);
    const int th = threads_for(ctx, sm, ctx->N[0] * ctx->N[1], grid);
    const double nxy = (double)ctx->N[0] * ctx->N[1];
    const double bpp = kind == Src::Plain ? 32.0 : (kind == Src::Residual ? 48.0 : 24.0);
    ProfScope ps(ctx, RSDFT_K_FFT_XY_FWD, 5.0 * nxy * std::log2(nxy) * ctx->N[2] * nb, bpp * (double)ctx->n * nb, st);
    const FixTabs tb = tabs_of(ctx);
    I2 *o = reinterpret_cast<I2 *>(dst);
    int db = 63;   // bits at which the sum over a disc's row cannot overflow
    while ((1 << (63 - db)) < ctx->discs.wmax) --db;
    switch (kind) {
        case Src::Plain:
            RS_TRY(set_smem(ctx, k_xy_forward_fix<Src::Plain>, sm));
            k_xy_forward_fix<Src::Plain><<<grid, th, sm, st>>>(tb, src, src2, theta, act, rsrc, RS, o, mp, ctx->discs,
                                                                db, part);
            break;
        case Src::Residual:
            RS_TRY(set_smem(ctx, k_xy_forward_fix<Src::Residual>, sm));
            k_xy_forward_fix<Src::Residual><<<grid, th, sm, st>>>(tb, src, src2, theta, act, rsrc, RS, o, mp, ctx->discs,
                                                                db, part);
            break;
        case Src::RealField:
            RS_TRY(set_smem(ctx, k_xy_forward_fix<Src::RealField>, sm));
            k_xy_forward_fix<Src::RealField><<<grid, th, sm, st>>>(tb, src, src2, theta, act, rsrc, RS, o, mp, ctx->discs,
                                                                db, part);
            break;
    }
    RS_LAUNCHED(ctx, "k_xy_forward_fix");
    return RSDFT_OK;
}

rsdft_status fft_z_mid(rsdft_ctx *ctx, Mid mid, double2 *buf, const double *tkin, int nb, cudaStream_t st) {
    if (nb <= 0) return RSDFT_OK;
    RS_TRY(check_plane(ctx));
    Meta *mp, *ms;
    RS_TRY(ensure_meta(ctx, buf, nb, &mp, &ms, st));
    size_t sm = HEAD + (size_t)ctx->N[0] * ctx->N[2] * sizeof(I2) + SHIFTS;
    const size_t tabb = (size_t)(ctx->N[0] / 2 + 1) * (ctx->N[2] / 2 + 1) * sizeof(double);
    int table = 0;
    if (mid == Mid::Tpa && sm + tabb <= MAX_DYN_SMEM) {
        table = 1;
        sm += tabb;
    }
    const dim3 grid(ctx->N[1], nb);
    const int th = threads_for(ctx, sm, ctx->N[0] * ctx->N[2], grid);
    ProfScope ps(ctx, RSDFT_K_FFT_Z, 10.0 * (double)ctx->n * std::log2((double)ctx->N[2]) * nb, 32.0 * (double)ctx->n * nb, st);
    const FixTabs tb = tabs_of(ctx);
    I2 *b = reinterpret_cast<I2 *>(buf);
#define RS_Z(M)                                                              \
    case M:                                                                  \
        RS_TRY(set_smem(ctx, k_z_mid_fix<M>, sm));                           \
        k_z_mid_fix<M><<<grid, th, sm, st>>>(tb, b, tkin, mp, ms, table);    \
        break;
    switch (mid) {
        RS_Z(Mid::Kinetic)
        RS_Z(Mid::Tpa)
        RS_Z(Mid::Hartree)
        RS_Z(Mid::GradX)
        RS_Z(Mid::GradY)
        RS_Z(Mid::GradZ)
    }
#undef RS_Z
    RS_LAUNCHED(ctx, "k_z_mid_fix");
    return RSDFT_OK;
}

rsdft_status fft_xy_inverse(rsdft_ctx *ctx, const double2 *buf, const double2 *psi, const double2 *ab, double2 *out,
                            double *rout, int nb, cudaStream_t st) {
    if (nb <= 0) return RSDFT_OK;
    RS_TRY(check_plane(ctx));
    Meta *mp, *ms;
    RS_TRY(ensure_meta(ctx, buf, nb, &mp, &ms, st));
    const int RS = plane_stride(ctx);
    size_t sm = plane_smem(ctx);
    int room = 0;
    if (psi && ab) {   // the scatter table beside the plane
        const size_t per = 2 * (size_t)ctx->discs.wmax * sizeof(I2);
        room = disc_room(sm, per, ctx->discs.maxdiscs, MAX_DYN_SMEM);
        sm += room * per;
    }
    const dim3 grid(ctx->N[2], nb);
    const int th = threads_for(ctx, sm, ctx->N[0] * ctx->N[1], grid);
    const double nxy = (double)ctx->N[0] * ctx->N[1];
    const double bpp = rout ? 24.0 : (psi ? 48.0 : 32.0);
    ProfScope ps(ctx, RSDFT_K_FFT_XY_INV, 5.0 * nxy * std::log2(nxy) * ctx->N[2] * nb,
                 bpp * (double)ctx->n * nb + (psi ? 8.0 * (double)ctx->n : 0.0), st);
    const FixTabs tb = tabs_of(ctx);
    const I2 *b = reinterpret_cast<const I2 *>(buf);
    if (rout) {
        RS_TRY(set_smem(ctx, k_xy_inverse_fix<FixEpi::Real>, sm));
        k_xy_inverse_fix<FixEpi::Real><<<grid, th, sm, st>>>(tb, b, ms, psi, ctx->v, ctx->discs, ab, room, RS, out,
                                                               rout);
    } else if (psi) {
        RS_TRY(set_smem(ctx, k_xy_inverse_fix<FixEpi::Hpsi>, sm));
        k_xy_inverse_fix<FixEpi::Hpsi><<<grid, th, sm, st>>>(tb, b, ms, psi, ctx->v, ctx->discs, ab, room, RS, out,
                                                               rout);
    } else {
        RS_TRY(set_smem(ctx, k_xy_inverse_fix<FixEpi::Plain>, sm));
        k_xy_inverse_fix<FixEpi::Plain><<<grid, th, sm, st>>>(tb, b, ms, psi, ctx->v, ctx->discs, ab, room, RS, out,
                                                               rout);
    }
    RS_LAUNCHED(ctx, "k_xy_inverse_fix");
    return RSDFT_OK;
}

}  // namespace rsdft
