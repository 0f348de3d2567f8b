// Batched 3D FFT kernels of the FP32 data path, the projector gather and H psi (SCF tasks (1)
// and (4)).  The FP64 passes, of the same shape, are in fft_fix.cu.
//
// What bounds the passes is their instructions (72% of the issue slots), most of them around the
// butterflies: addresses, shared-memory accesses, twiddle loads.  So a thread holds up to 16 points
// and an axis has two stages where its length allows (96 = 12 x 8 instead of 8 x 4 x 3): the
// z pass of 160 bands on 96^3 went from 1.04 to 0.78 ms, its instructions from 0.96 to 0.60 billion.
//
// Layout: orbital block [band][z][y][x] complex, x fastest.  A 3D transform is
// three shared-memory passes over HBM:
//   xy-forward  (one CTA per (band, z) plane: x lines then y lines, DIF)
//   z-mid       (one CTA per (band, y) slab: z DIF, multiply by a function of
//                |G|^2 at the digit-reversed position, z DIT)
//   xy-inverse  (one CTA per (band, z) plane: y and x DIT, then the epilogue:
//                + V psi and the projector scatter by discs for H psi)
// Forward stages leave the spectrum in mixed-radix digit-reversed order and
// the inverse stages take it back to natural order, so the per-G factor is
// applied through position-indexed |G|^2 tables and no permutation pass exists.
#include <algorithm>
#include <cmath>

#include <mutex>
#include <vector>

#include "fft_common.h"
#include "proj.h"
#include "rsdft_internal.h"

namespace rsdft {

// ---- complex helpers ---------------------------------------
template <typename V> __device__ __forceinline__ V mk(typename Sc<V>::T x, typename Sc<V>::T y) {
    V r; r.x = x; r.y = y; return r;
}
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { return mk<V>(a.x - b.x, a.y - b.y); }
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
    return mk<V>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename V> __device__ __forceinline__ V cmulconj(V a, V b) {  // a * conj(b)
    return mk<V>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename V> __device__ __forceinline__ V cscale(V a, typename Sc<V>::T s) { return mk<V>(a.x * s, a.y * s); }
// multiply by -i (forward sign) or +i (inverse sign)
template <typename V, bool INV> __device__ __forceinline__ V rot(V a) {
    return INV ? mk<V>(-a.y, a.x) : mk<V>(a.y, -a.x);
}

// ---- small DFTs: y_p = sum_q x_q exp(-+2 pi i p q / R) ----------------------
// Constants are cos/sin of 2 pi k / R written out to 30 digits.
#define RS_SQRT3_2 0.866025403784438646763723170753
#define RS_SQRT1_2 0.707106781186547524400844362105
#define RS_C1_5 0.309016994374947424102293417183
#define RS_C2_5 (-0.809016994374947424102293417183)
#define RS_S1_5 0.951056516295153572116439333379
#define RS_S2_5 0.587785252292473129168705954639

template <typename V, bool INV> __device__ __forceinline__ void dft2(V *v) {
    V a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
}
template <typename V, bool INV> __device__ __forceinline__ void dft3(V *v) {
    using T = typename Sc<V>::T;
    V t1 = cadd(v[1], v[2]);
    V t2 = csub(v[0], cscale(t1, (T)0.5));
    V t3 = cscale(csub(v[1], v[2]), (T)RS_SQRT3_2);
    v[0] = cadd(v[0], t1);
    V r = rot<V, INV>(t3);  // -i t3 (forward)
    v[1] = cadd(t2, r);
    v[2] = csub(t2, r);
}
template <typename V, bool INV> __device__ __forceinline__ void dft4(V *v) {
    V a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
    V a2 = cadd(v[1], v[3]), a3 = rot<V, INV>(csub(v[1], v[3]));
    v[0] = cadd(a0, a2);
    v[2] = csub(a0, a2);
    v[1] = cadd(a1, a3);
    v[3] = csub(a1, a3);
}
template <typename V, bool INV> __device__ __forceinline__ void dft5(V *v) {
    using T = typename Sc<V>::T;
    V a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
    V a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    V x0 = v[0];
    v[0] = cadd(x0, cadd(a1, a2));
    V r1 = cadd(x0, cadd(cscale(a1, (T)RS_C1_5), cscale(a2, (T)RS_C2_5)));
    V i1 = rot<V, INV>(cadd(cscale(b1, (T)RS_S1_5), cscale(b2, (T)RS_S2_5)));
    V r2 = cadd(x0, cadd(cscale(a1, (T)RS_C2_5), cscale(a2, (T)RS_C1_5)));
    V i2 = rot<V, INV>(csub(cscale(b1, (T)RS_S2_5), cscale(b2, (T)RS_S1_5)));
    v[1] = cadd(r1, i1);
    v[4] = csub(r1, i1);
    v[2] = cadd(r2, i2);
    v[3] = csub(r2, i2);
}
template <typename V, bool INV> __device__ __forceinline__ void dft8(V *v) {
    using T = typename Sc<V>::T;
    V e[4] = {v[0], v[2], v[4], v[6]};
    V o[4] = {v[1], v[3], v[5], v[7]};
    dft4<V, INV>(e);
    dft4<V, INV>(o);
    // o_p *= w8^p, w8 = exp(-+ i pi / 4)
    const T h = (T)RS_SQRT1_2;
    V o1 = o[1], o3 = o[3];
    // (1 -+ i) h * o1
    o[1] = cscale(cadd(o1, rot<V, INV>(o1)), h);
    o[2] = rot<V, INV>(o[2]);
    // (-1 -+ i) h * o3
    o[3] = cscale(csub(rot<V, INV>(o3), o3), h);
    for (int p = 0; p < 4; ++p) {
        v[p] = cadd(e[p], o[p]);
        v[p + 4] = csub(e[p], o[p]);
    }
}

// Composite radices: R = A B as A transforms over B.  Coprime factors need no twiddles (Good and
// Thomas: input q = (B q1 + A q2) mod R, output p with p mod A = p1 and p mod B = p2 and the inner
// exponents as in a two-dimensional transform of A x B points); 9 and 16 have theirs.
template <typename V, int R, bool INV> __device__ __forceinline__ void dftR(V *v);
template <typename V, int A, int B, bool INV> __device__ __forceinline__ void dft_coprime(V *v) {
    constexpr int R = A * B;
    V t[B][A];
#pragma unroll
    for (int q2 = 0; q2 < B; ++q2) {
#pragma unroll
        for (int q1 = 0; q1 < A; ++q1) t[q2][q1] = v[(B * q1 + A * q2) % R];
        dftR<V, A, INV>(t[q2]);
    }
#pragma unroll
    for (int p1 = 0; p1 < A; ++p1) {
        V c[B];
#pragma unroll
        for (int q2 = 0; q2 < B; ++q2) c[q2] = t[q2][p1];
        dftR<V, B, INV>(c);
        // exp(2 pi i (B q1 + A q2) p / R) = exp(2 pi i q1 p / A) exp(2 pi i q2 p / B): p = (p1, p2)
#pragma unroll
        for (int p = 0; p < R; ++p)
            if (p % A == p1) v[p] = c[p % B];
    }
}
// exp(-2 pi i k / R) of the inner twiddles of R = 9 and 16
template <int R> __device__ __forceinline__ constexpr double inner_cos(int k) {
    constexpr double c9[5] = {1.0, 0.766044443118978035202392650555, 0.173648177666930348851716626769, -0.5,
                              -0.939692620785908384054109277325};
    constexpr double c16[10] = {1.0, 0.923879532511286756128183189397, 0.707106781186547524400844362105,
                                0.382683432365089771728459984030, 0.0, -0.382683432365089771728459984030,
                                -0.707106781186547524400844362105, -0.923879532511286756128183189397, -1.0,
                                -0.923879532511286756128183189397};
    return R == 9 ? c9[k] : c16[k];
}
template <int R> __device__ __forceinline__ constexpr double inner_sin(int k) {
    constexpr double s9[5] = {0.0, 0.642787609686539326322643409907, 0.984807753012208059366743024590,
                              0.866025403784438646763723170753, 0.342020143325668733044099614682};
    constexpr double s16[10] = {0.0, 0.382683432365089771728459984030, 0.707106781186547524400844362105,
                                0.923879532511286756128183189397, 1.0, 0.923879532511286756128183189397,
                                0.707106781186547524400844362105, 0.382683432365089771728459984030, 0.0,
                                -0.382683432365089771728459984030};
    return R == 9 ? s9[k] : s16[k];
}
template <typename V, int A, bool INV> __device__ __forceinline__ void dft_square(V *v) {   // R = A A
    using T = typename Sc<V>::T;
    constexpr int R = A * A;
    V t[A][A];
#pragma unroll
    for (int q2 = 0; q2 < A; ++q2) {
#pragma unroll
        for (int q1 = 0; q1 < A; ++q1) t[q2][q1] = v[A * q1 + q2];
        dftR<V, A, INV>(t[q2]);
    }
#pragma unroll
    for (int p1 = 0; p1 < A; ++p1) {
        V c[A];
#pragma unroll
        for (int q2 = 0; q2 < A; ++q2) {
            const V w = mk<V>((T)inner_cos<R>(p1 * q2), (T)(-inner_sin<R>(p1 * q2)));
            c[q2] = p1 * q2 == 0 ? t[q2][p1] : (INV ? cmulconj(t[q2][p1], w) : cmul(t[q2][p1], w));
        }
        dftR<V, A, INV>(c);
#pragma unroll
        for (int p2 = 0; p2 < A; ++p2) v[p1 + A * p2] = c[p2];
    }
}

template <typename V, int R, bool INV> __device__ __forceinline__ void dftR(V *v) {
    if constexpr (R == 2) dft2<V, INV>(v);
    else if constexpr (R == 3) dft3<V, INV>(v);
    else if constexpr (R == 4) dft4<V, INV>(v);
    else if constexpr (R == 5) dft5<V, INV>(v);
    else if constexpr (R == 6) dft_coprime<V, 2, 3, INV>(v);
    else if constexpr (R == 8) dft8<V, INV>(v);
    else if constexpr (R == 9) dft_square<V, 3, INV>(v);
    else if constexpr (R == 10) dft_coprime<V, 2, 5, INV>(v);
    else if constexpr (R == 12) dft_coprime<V, 3, 4, INV>(v);
    else dft_square<V, 4, INV>(v);
}

template <typename V> __device__ __forceinline__ V ldtw(const V *tw, int k) { return __ldg(tw + k); }

// One radix-R butterfly of a stage, in place in shared memory (j = 0: unit twiddles).
template <typename V, int R, bool INV>
__device__ __forceinline__ void bfly(V *s, int step, int j, int twstep, const V *tw) {
    V v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = s[q * step];
    if (INV && j) {
#pragma unroll
        for (int p = 1; p < R; ++p) v[p] = cmulconj(v[p], ldtw(tw, j * p * twstep));
    }
    dftR<V, R, INV>(v);
    if (!INV && j) {
#pragma unroll
        for (int p = 1; p < R; ++p) v[p] = cmul(v[p], ldtw(tw, j * p * twstep));
    }
#pragma unroll
    for (int q = 0; q < R; ++q) s[q * step] = v[q];
}

template <typename V, int R, bool INV>
__device__ __forceinline__ void stage(V *s, const AxisPlan &ax, int st, const V *tw, int nlines, unsigned nlmag,
                                      int lstride, int es) {
    const int N = ax.N, len = ax.len[st], sub = ax.sub[st];
    const unsigned smag = ax.submag[st];
    const int total = N / R * nlines, twstep = N / len, step = sub * es;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int bf = qdiv(idx, nlmag), line = idx - bf * nlines;   // consecutive threads: consecutive lines
        const int b = qdiv(bf, smag), j = bf - b * sub;
        bfly<V, R, INV>(s + line * lstride + (b * len + j) * es, step, j, twstep, tw);
    }
}

// All stages of nlines 1D transforms of length ax.N in shared memory: element e of line l at
// s[l * lstride + e * es] (nlmag: multiply-high divisor of nlines, total < 2^16).
template <typename V, bool INV>
__device__ void fft_lines(V *s, const AxisPlan &ax, const V *tw, int nlines, unsigned nlmag, int lstride, int es) {
    for (int t = 0; t < ax.nstage; ++t) {
        const int st = INV ? ax.nstage - 1 - t : t;
        switch (ax.radix[st]) {
            case 2: stage<V, 2, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 3: stage<V, 3, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 4: stage<V, 4, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 5: stage<V, 5, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 6: stage<V, 6, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 8: stage<V, 8, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 9: stage<V, 9, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 10: stage<V, 10, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            case 12: stage<V, 12, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
            default: stage<V, 16, INV>(s, ax, st, tw, nlines, nlmag, lstride, es); break;
        }
        __syncthreads();
    }
}

// 80 registers: a radix-16 butterfly without spills
constexpr int FFT_THREADS = 768;   // at most (fft_threads)

// Tables of one precision: twiddles exp(-2 pi i k/N) and G_a^2 at each
// digit-reversed position.
template <typename V> struct FftTabs {
    AxisPlan ax[3];
    const V *tw[3];
    const typename Sc<V>::T *g2[3];
    double inv_n;   // 1 / (Nx Ny Nz), formed on the host
};

static FftTabs<float2> tabs_of(const rsdft_ctx *ctx, float2 *) {
    FftTabs<float2> t;
    for (int a = 0; a < 3; ++a) {
        t.ax[a] = ctx->fft.ax32[a];
        t.tw[a] = ctx->fft.tw32[a];
        t.g2[a] = ctx->fft.g2pos32[a];
    }
    t.inv_n = 1.0 / (double)ctx->n;
    return t;
}
static const float *v_of(const rsdft_ctx *ctx, float2 *) { return ctx->v32; }

// part[disc][3] = sums of gx gy v, hx gy v, gx hy v over each disc of plane z (row stride RS)
__device__ __forceinline__ void gather_plane(const float2 *plane, int RS, const Discs &t, int z, int Nx,
                                             float2 *__restrict__ part) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int d1 = t.plane_start[z + 1];
    for (int d = t.plane_start[z] + (threadIdx.x >> 5); d < d1; d += nw) {
        const int2 m = __ldg(reinterpret_cast<const int2 *>(t.meta + d));
        const int rows = disc_rows(m.y), w = disc_width(m.y);
        const float2 *gx = t.gx + (size_t)d * t.wmax;
        float s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int r0 = 0; r0 < rows; r0 += 32) {
            int4 q = make_int4(0, 0, 0, 0);
            if (r0 + lane < rows) q = __ldg(reinterpret_cast<const int4 *>(t.row + m.x + r0 + lane));
            const float2 *row = plane + (q.x & 255) * RS;
            int x = disc_x0(m.y);
            float ux = 0.f, uy = 0.f, vx = 0.f, vy = 0.f;   // sums of gx v, hx v along the row
#pragma unroll 4
            for (int j = 0; j < w; ++j) {
                const float2 k = __ldg(gx + j);
                const float2 v = row[x];
                const bool in = in_row(q.x, j);   // a select, not a branch
                const float g = in ? k.x : 0.f, h = in ? k.y : 0.f;
                ux = fmaf(g, v.x, ux);
                uy = fmaf(g, v.y, uy);
                vx = fmaf(h, v.x, vx);
                vy = fmaf(h, v.y, vy);
                x = x + 1 == Nx ? 0 : x + 1;
            }
            const float g = __int_as_float(q.y), h = __int_as_float(q.z);
            s[0] += g * ux;
            s[1] += g * uy;
            s[2] += g * vx;
            s[3] += g * vy;
            s[4] += h * ux;
            s[5] += h * uy;
        }
#pragma unroll
        for (int k = 0; k < 6; ++k)
            for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        if (lane < 3)
            part[(size_t)d * 3 + lane] = make_float2(lane == 0 ? s[0] : (lane == 1 ? s[2] : s[4]),
                                                     lane == 0 ? s[1] : (lane == 1 ? s[3] : s[5]));
    }
}

// ---- xy forward pass ------------------------------------------------------------
template <typename V, Src SRC>
__global__ void __launch_bounds__(FFT_THREADS)
k_xy_forward(FftTabs<V> tb, const V *__restrict__ src, const V *__restrict__ src2,
             const double *__restrict__ theta, const int *__restrict__ act, V *__restrict__ dst,
             Discs discs, V *__restrict__ part) {
    using T = typename Sc<V>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *s_plane = reinterpret_cast<V *>(smem_raw);
    const int Nx = tb.ax[0].N, Ny = tb.ax[1].N, Nz = tb.ax[2].N;
    const int z = blockIdx.x, band = blockIdx.y;
    const size_t n = (size_t)Nx * Ny * Nz;
    const size_t plane = (size_t)Nx * Ny;
    const size_t off = (size_t)z * plane;
    const int RS = plane_rs(Nx);
    const unsigned nxm = tb.ax[0].nmag;
    auto put = [&](int i, V v) { s_plane[pidx(i, Nx, RS, nxm)] = v; };
    if (SRC == Src::Plain) {
        const V *in = src + band * n + off;
        stage_in<V>((int)plane, [&](int i) { return in[i]; }, put);
    } else if (SRC == Src::Residual) {
        const int b = act[band];
        const T th = (T)theta[b];
        const V *hx = src + b * n + off;
        const V *x = src2 + b * n + off;
        stage_in<V>((int)plane, [&](int i) {
            const V h = hx[i], v = x[i];
            return mk<V>(h.x - th * v.x, h.y - th * v.y);
        }, put);
    }
    __syncthreads();
    if (SRC == Src::Plain && part) {
        gather_plane(s_plane, RS, discs, z, Nx, part + (size_t)band * discs.ndisc * 3);
        __syncthreads();
    }
    fft_lines<V, false>(s_plane, tb.ax[0], tb.tw[0], Ny, tb.ax[1].nmag, RS, 1);
    fft_lines<V, false>(s_plane, tb.ax[1], tb.tw[1], Nx, tb.ax[0].nmag, 1, RS);
    V *out = dst + band * n + off;
    for (int i = threadIdx.x; i < (int)plane; i += blockDim.x) out[i] = s_plane[pidx(i, Nx, RS, nxm)];
}

// ---- z pass with the per-G factor ------------------------------------------------
template <typename T> __device__ __forceinline__ T tpa_k(T x) {
    T num = (T)27 + x * ((T)18 + x * ((T)12 + (T)8 * x));
    return num / (num + (T)16 * x * x * x * x);
}

template <typename V, Mid MID>
__global__ void __launch_bounds__(FFT_THREADS)
k_z_mid(FftTabs<V> tb, V *__restrict__ buf, const double *__restrict__ tkin) {
    using T = typename Sc<V>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *s_slab = reinterpret_cast<V *>(smem_raw);
    const int Nx = tb.ax[0].N, Ny = tb.ax[1].N, Nz = tb.ax[2].N;
    const int y = blockIdx.x, band = blockIdx.y;
    const size_t n = (size_t)Nx * Ny * Nz;
    const size_t zstride = (size_t)Nx * Ny;
    V *base = buf + band * n + (size_t)y * Nx;
    const int tot = Nx * Nz;
    stage_in<V>(tot, [&](int i) {
        const int z = qdiv(i, tb.ax[0].nmag), x = i - z * Nx;
        return base[z * zstride + x];
    }, [&](int i, V v) { s_slab[i] = v; });
    __syncthreads();
    fft_lines<V, false>(s_slab, tb.ax[2], tb.tw[2], Nx, tb.ax[0].nmag, 1, Nx);
    const T inv_n = (T)tb.inv_n;
    const T gy2 = tb.g2[1][y];
    T tk = (T)1;
    if (MID == Mid::Tpa) {
        double t = tkin[band];
        if (!(t >= 1e-12)) t = 1.0;
        tk = (T)t;
    }
    for (int i = threadIdx.x; i < tot; i += blockDim.x) {
        const int z = qdiv(i, tb.ax[0].nmag), x = i - z * Nx;
        T g2 = tb.g2[0][x] + gy2 + tb.g2[2][z];
        T f;
        if (MID == Mid::Kinetic) f = (T)0.5 * g2 * inv_n;
        else f = tpa_k<T>((T)0.5 * g2 / tk) * inv_n;
        s_slab[i] = mk<V>(s_slab[i].x * f, s_slab[i].y * f);
    }
    __syncthreads();
    fft_lines<V, true>(s_slab, tb.ax[2], tb.tw[2], Nx, tb.ax[0].nmag, 1, Nx);
    for (int i = threadIdx.x; i < tot; i += blockDim.x) {
        const int z = qdiv(i, tb.ax[0].nmag), x = i - z * Nx;
        base[z * zstride + x] = s_slab[i];
    }
}

// plane += sum over its discs of gx (gy A + hy By) + hx gy Bx, ab[disc] = (A, Bx, By); uw: room discs
__device__ __forceinline__ void scatter_plane(float2 *s_plane, int RS, const Discs &t, int z, int Nx,
                                              const float2 *__restrict__ ab, float4 *uw, int room) {
    const int lane = threadIdx.x & 31, d0 = t.plane_start[z];
    int base = 0;
    for_discs(t, z, room, [&](int c0, int n) {
        base = d0 + c0;
        for (int i = threadIdx.x; i < n * t.wmax; i += blockDim.x) {
            const int d = base + i / t.wmax;
            const float2 k = __ldg(t.gx + (size_t)base * t.wmax + i);
            const float2 A = __ldg(ab + 3 * (size_t)d), Bx = __ldg(ab + 3 * (size_t)d + 1), By = __ldg(ab + 3 * (size_t)d + 2);
            uw[i] = make_float4(k.x * A.x + k.y * Bx.x, k.x * A.y + k.y * Bx.y, k.x * By.x, k.x * By.y);
        }
    }, [&](int d, int ja, int jb) {
        const int2 m = __ldg(reinterpret_cast<const int2 *>(t.meta + d));
        const int rows = disc_rows(m.y);
        const float4 *ue = uw + (d - base) * t.wmax;
        for (int r0 = 0; r0 < rows; r0 += 32) {
            int4 q = make_int4(0, 0, 0, 0);
            if (r0 + lane < rows) q = __ldg(reinterpret_cast<const int4 *>(t.row + m.x + r0 + lane));
            const float g = __int_as_float(q.y), h = __int_as_float(q.z);
            float2 *row = s_plane + (q.x & 255) * RS;
            int x = disc_x0(m.y) + ja;
            if (x >= Nx) x -= Nx;
#pragma unroll 4
            for (int j = ja; j < jb; ++j) {
                const float4 k = ue[j];
                if (in_row(q.x, j)) {
                    float2 o = row[x];
                    o.x += g * k.x + h * k.z;
                    o.y += g * k.y + h * k.w;
                    row[x] = o;
                }
                x = x + 1 == Nx ? 0 : x + 1;
            }
        }
    });
}

// ---- xy inverse pass + epilogue ------------------------------------------------------
enum class Epi { Plain, Hpsi };

template <typename V, Epi EPI>
__global__ void __launch_bounds__(FFT_THREADS)
k_xy_inverse(FftTabs<V> tb, const V *__restrict__ buf, const V *__restrict__ psi,
             const typename Sc<V>::T *__restrict__ v, Discs discs, int room,
             const V *__restrict__ ab, V *__restrict__ out) {
    using T = typename Sc<V>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *s_plane = reinterpret_cast<V *>(smem_raw);
    const int Nx = tb.ax[0].N, Ny = tb.ax[1].N, Nz = tb.ax[2].N;
    const int z = blockIdx.x, band = blockIdx.y;
    const size_t n = (size_t)Nx * Ny * Nz;
    const size_t plane = (size_t)Nx * Ny;
    const size_t off = (size_t)z * plane;
    const V *in = buf + band * n + off;
    const int RS = plane_rs(Nx);
    const unsigned nxm = tb.ax[0].nmag;
    const bool scatter = EPI == Epi::Hpsi && ab;
    const V *abb = ab + (size_t)band * discs.ndisc * 3;
    float4 *uw = reinterpret_cast<float4 *>(s_plane + (((size_t)Ny * RS + 1) & ~(size_t)1));
    stage_in<V>((int)plane, [&](int i) { return in[i]; }, [&](int i, V v) { s_plane[pidx(i, Nx, RS, nxm)] = v; });
    __syncthreads();
    fft_lines<V, true>(s_plane, tb.ax[1], tb.tw[1], Nx, tb.ax[0].nmag, 1, RS);
    fft_lines<V, true>(s_plane, tb.ax[0], tb.tw[0], Ny, tb.ax[1].nmag, RS, 1);
    if (EPI == Epi::Plain) {
        V *o = out + band * n + off;
        for (int i = threadIdx.x; i < (int)plane; i += blockDim.x) o[i] = s_plane[pidx(i, Nx, RS, nxm)];
    } else {
        const V *ps = psi + band * n + off;
        const T *vv = v + off;
        if (scatter) {
            scatter_plane(s_plane, RS, discs, z, Nx, abb, uw, room);
        }
        V *o = out + band * n + off;
        for (int i = threadIdx.x; i < (int)plane; i += blockDim.x) {
            const V t = s_plane[pidx(i, Nx, RS, nxm)];
            const V y = ps[i];
            const T vi = vv[i];
            o[i] = mk<V>(t.x + vi * y.x, t.y + vi * y.y);
        }
    }
}

// ---- projectors --------------------------------------------------------------------------
constexpr int PROJ_THREADS = 256;

// p[band][atom nproj + j] = <beta_j|psi> in FP64: a block per (band, atom), a warp per disc of the atom, joined
// in the block, so that the call needs no memory but the caller's.  lane = x; discs of at most 16 or 8
// points across take two or four rows at a time.  A point costs four multiply-adds (a warp's 64 cycles each, which
// bounds the kernel) and the factors of a row are loaded.  One GB300, against partial sums per
// plane in scratch with the factors converted from fixed point: 144 bands on 64^3, 64 atoms 5,033 -> 1,443 us (a table
// of every point's values 1,734), one band 127 -> 40 (51), 64 bands on 24^3, 8 atoms 106 -> 31 (31).
__global__ void __launch_bounds__(PROJ_THREADS)
k_project(Discs t, ProjTables pt, const double2 *__restrict__ psi, int Nx, int Ny, long long n, double dV,
          double2 *__restrict__ p) {
    const int band = blockIdx.x / t.natom, a = blockIdx.x - band * t.natom;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i1 = t.atom_start[a + 1];
    double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i = t.atom_start[a] + warp; i < i1; i += PROJ_THREADS / 32) {
        const int d = t.atom_disc[i];
        const int2 m = __ldg(reinterpret_cast<const int2 *>(t.meta + d));
        const int rows = disc_rows(m.y), w = disc_width(m.y);
        const double2 *plane = psi + (size_t)band * n + (size_t)pt.plane[d] * Nx * Ny;
        double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // sums of gx gy, hx gy and gx hy times psi
        const int W = w <= 8 ? 8 : (w <= 16 ? 16 : 32);   // lanes a row
        for (int c = 0; c < w; c += W) {
            const int l = c + (lane & (W - 1));
            int x = disc_x0(m.y) + l;
            if (x >= Nx) x -= Nx;
            double ax = 0.0, ay = 0.0, bx = 0.0, by = 0.0;
#pragma unroll 4
            for (int r = lane / W; r < rows; r += 32 / W) {
                const int k = __ldg(&t.row[m.x + r].packed);
                if (in_row(k, l)) {
                    const double2 u = plane[(k & 255) * Nx + x], f = __ldg(pt.row + m.x + r);
                    ax += f.x * u.x;
                    ay += f.x * u.y;
                    bx += f.y * u.x;
                    by += f.y * u.y;
                }
            }
            if (l < w) {
                const double2 f = __ldg(pt.gx + (size_t)d * t.wmax + l);
                v[0] += f.x * ax;
                v[1] += f.x * ay;
                v[2] += f.y * ax;
                v[3] += f.y * ay;
                v[4] += f.x * bx;
                v[5] += f.x * by;
            }
        }
        const double2 gd = t.gz[d];
#pragma unroll
        for (int k = 0; k < 6; ++k) s[k] += gd.x * v[k];
        s[6] += gd.y * v[0];
        s[7] += gd.y * v[1];
    }
    // the eight sums over the warp, half of them going to each half of the lanes at every step: 9 additions instead of 40
#pragma unroll
    for (int o = 16, m = 4; m > 0; o >>= 1, m >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < m; ++k) {
            const double give = up ? s[k] : s[k + m];
            s[k] = (up ? s[k + m] : s[k]) + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
    __shared__ double red[PROJ_THREADS / 32][8];
    if ((lane & 3) == 0) red[warp][lane >> 2] = s[0];   // bits 4, 3, 2 of the lane: those of the sum's number
    __syncthreads();
    const int j = threadIdx.x >> 1, part = threadIdx.x & 1;
    if (j < t.nproj) {
        double q = 0.0;
        for (int k = 0; k < PROJ_THREADS / 32; ++k) q += red[k][threadIdx.x];
        double *o = reinterpret_cast<double *>(p + (size_t)blockIdx.x * t.nproj + j);
        o[part] = t.cnorm[4 * a + j] * dV * q;
    }
}

// The gather alone on FP32 planes in global memory (lane = x), for the solvers: a CTA's discs are those of one
// plane, whose rows it reads from L1 again (144 bands on 64^3 0.30 ms; a block per atom, as above, 0.51).
__global__ void __launch_bounds__(PROJ_THREADS)
k_gather(Discs t, const float2 *__restrict__ psi, int Nx, int Ny, long long n, float2 *__restrict__ part) {
    const int z = blockIdx.x, band = blockIdx.y;
    const float2 *plane = psi + (size_t)band * n + (size_t)z * Nx * Ny;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int d1 = t.plane_start[z + 1];
    for (int d = t.plane_start[z] + (threadIdx.x >> 5); d < d1; d += nw) {
        const DiscMeta m = t.meta[d];
        const int rows = disc_rows(m.packed), w = disc_width(m.packed);
        float s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int c = 0; c < w; c += 32) {
            const int l = c + lane;
            int x = disc_x0(m.packed) + l;
            if (x >= Nx) x -= Nx;
            float ax = 0.f, ay = 0.f, bx = 0.f, by = 0.f;
#pragma unroll 4
            for (int r = 0; r < rows; ++r) {
                const int4 k = __ldg(reinterpret_cast<const int4 *>(t.row + m.row0 + r));
                const float g = __int_as_float(k.y), h = __int_as_float(k.z);
                if (in_row(k.x, l)) {
                    const float2 v = plane[(k.x & 255) * Nx + x];
                    ax += g * v.x;
                    ay += g * v.y;
                    bx += h * v.x;
                    by += h * v.y;
                }
            }
            const float2 k = l < w ? __ldg(t.gx + (size_t)d * t.wmax + l) : make_float2(0.f, 0.f);
            s[0] += k.x * ax;
            s[1] += k.x * ay;
            s[2] += k.y * ax;
            s[3] += k.y * ay;
            s[4] += k.x * bx;
            s[5] += k.x * by;
        }
#pragma unroll
        for (int k = 0; k < 6; ++k)
            for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        if (lane < 3)
            part[((size_t)band * t.ndisc + d) * 3 + lane] = make_float2(lane == 0 ? s[0] : (lane == 1 ? s[2] : s[4]),
                                                                       lane == 0 ? s[1] : (lane == 1 ? s[3] : s[5]));
    }
}

// One warp per (band, atom): the disc sums joined with their z factors, p[band][atom nproj + j] =
// <beta_j|psi> (p may be null) and the scatter coefficients of every disc, ab[band][disc] =
// (gz q_s + hz q_z, gz q_x, gz q_y) with q_j = c_j E_j <beta_j|psi> (ab may be null).
template <typename V>
__global__ void __launch_bounds__(PROJ_THREADS)
k_disc_fin(Discs t, const V *__restrict__ part, int nb, typename Sc<V>::T dV, V *__restrict__ p,
           V *__restrict__ ab) {
    using T = typename Sc<V>::T;
    const int w = (blockIdx.x * PROJ_THREADS + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int band = w / t.natom, a = w - band * t.natom;
    if (band >= nb) return;
    const int i0 = t.atom_start[a], i1 = t.atom_start[a + 1];
    T s[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] = (T)0;
    const V *pb = part + (size_t)band * t.ndisc * 3;
    for (int i = i0 + lane; i < i1; i += 32) {
        const int d = t.atom_disc[i];
        const double2 gd = t.gz[d];
        const V g = mk<V>((T)gd.x, (T)gd.y), v0 = pb[3 * (size_t)d], v1 = pb[3 * (size_t)d + 1], v2 = pb[3 * (size_t)d + 2];
        s[0] += g.x * v0.x;
        s[1] += g.x * v0.y;
        s[2] += g.x * v1.x;
        s[3] += g.x * v1.y;
        s[4] += g.x * v2.x;
        s[5] += g.x * v2.y;
        s[6] += g.y * v0.x;
        s[7] += g.y * v0.y;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    V q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const T c = (T)t.cnorm[4 * a + j];   // 0 for projectors that are not there
        q[j] = mk<V>(c * dV * s[2 * j], c * dV * s[2 * j + 1]);
        if (p && lane == 0 && j < t.nproj) p[(size_t)band * t.natom * t.nproj + a * t.nproj + j] = q[j];
        const T e = j < t.nproj ? c * (T)t.e_kb[a * t.nproj + j] : (T)0;
        q[j] = mk<V>(e * q[j].x, e * q[j].y);
    }
    if (!ab) return;
    V *ob = ab + (size_t)band * t.ndisc * 3;
    for (int i = i0 + lane; i < i1; i += 32) {
        const int d = t.atom_disc[i];
        const double2 gd = t.gz[d];
        const V g = mk<V>((T)gd.x, (T)gd.y);
        ob[3 * (size_t)d] = mk<V>(g.x * q[0].x + g.y * q[3].x, g.x * q[0].y + g.y * q[3].y);
        ob[3 * (size_t)d + 1] = mk<V>(g.x * q[1].x, g.x * q[1].y);
        ob[3 * (size_t)d + 2] = mk<V>(g.x * q[2].x, g.x * q[2].y);
    }
}

__global__ void k_to_float(const double *__restrict__ in, long long n, float *__restrict__ out) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

// ---- launchers -------------------------------------------------------------------------
template <typename V> static size_t plane_bytes(const rsdft_ctx *ctx) {
    return (size_t)(ctx->N[0] | 1) * ctx->N[1] * sizeof(V);   // odd row stride
}
static int fft_threads(const rsdft_ctx *ctx, size_t smem, int points, const dim3 &grid) {
    return pass_threads(smem, points, (long long)grid.x * grid.y, ctx->num_sms, 64);
}
template <typename V> static size_t slab_bytes(const rsdft_ctx *ctx) {
    return (size_t)ctx->N[0] * ctx->N[2] * sizeof(V);
}

// shared memory of a plane with the scatter table of its discs beside it
static rsdft_status disc_smem(rsdft_ctx *ctx, size_t *sm, int *room) {
    const size_t base = (*sm + 15) / 16 * 16, per = (size_t)ctx->discs.wmax * sizeof(float4);
    *room = disc_room(base, per, ctx->discs.maxdiscs, MAX_DYN_SMEM);
    if (*room < 1) return fail(ctx, RSDFT_E_INVALID, "no shared memory for the projectors beside a plane");
    *sm = base + *room * per;
    return RSDFT_OK;
}

template <typename V>
rsdft_status fft_xy_forward_t(rsdft_ctx *ctx, Src kind, const V *src, const V *src2,
                              const double *theta, const int *act, V *dst,
                              int nb, cudaStream_t st, V *part) {
    if (nb <= 0) return RSDFT_OK;
    const size_t sm = plane_bytes<V>(ctx);
    dim3 grid(ctx->N[2], nb);
    const int pts = ctx->N[0] * ctx->N[1];
    const double nxy = (double)ctx->N[0] * ctx->N[1];
    const double e = (double)sizeof(V);
    const double bpp = kind == Src::Plain ? 2 * e : 3 * e;
    ProfScope ps(ctx, RSDFT_K_FFT_XY_FWD, 5.0 * nxy * std::log2(nxy) * ctx->N[2] * nb,
                 bpp * (double)ctx->n * nb, st);
    const FftTabs<V> tb = tabs_of(ctx, (V *)nullptr);
    const Discs &discs = ctx->discs;
    if (kind == Src::Plain) {
        RS_TRY(set_smem(ctx, k_xy_forward<V, Src::Plain>, sm));
        k_xy_forward<V, Src::Plain><<<grid, fft_threads(ctx, sm, pts, grid), sm, st>>>(tb, src, src2, theta, act, dst, discs, part);
    } else {
        RS_TRY(set_smem(ctx, k_xy_forward<V, Src::Residual>, sm));
        k_xy_forward<V, Src::Residual><<<grid, fft_threads(ctx, sm, pts, grid), sm, st>>>(tb, src, src2, theta, act, dst, discs, part);
    }
    RS_LAUNCHED(ctx, "k_xy_forward");
    return RSDFT_OK;
}

template <typename V>
rsdft_status fft_z_mid_t(rsdft_ctx *ctx, Mid mid, V *buf, const double *tkin, int nb,
                         cudaStream_t st) {
    if (nb <= 0) return RSDFT_OK;
    const size_t sm = slab_bytes<V>(ctx);
    dim3 grid(ctx->N[1], nb);
    const int pts = ctx->N[0] * ctx->N[2];
    ProfScope ps(ctx, RSDFT_K_FFT_Z, 10.0 * (double)ctx->n * std::log2((double)ctx->N[2]) * nb,
                 2.0 * sizeof(V) * (double)ctx->n * nb, st);
    const FftTabs<V> tb = tabs_of(ctx, (V *)nullptr);
    if (mid == Mid::Kinetic) {
        RS_TRY(set_smem(ctx, k_z_mid<V, Mid::Kinetic>, sm));
        k_z_mid<V, Mid::Kinetic><<<grid, fft_threads(ctx, sm, pts, grid), sm, st>>>(tb, buf, tkin);
    } else {
        RS_TRY(set_smem(ctx, k_z_mid<V, Mid::Tpa>, sm));
        k_z_mid<V, Mid::Tpa><<<grid, fft_threads(ctx, sm, pts, grid), sm, st>>>(tb, buf, tkin);
    }
    RS_LAUNCHED(ctx, "k_z_mid");
    return RSDFT_OK;
}

template <typename V>
rsdft_status fft_xy_inverse_t(rsdft_ctx *ctx, const V *buf, const V *psi, const V *ab, V *out, int nb,
                              cudaStream_t st) {
    if (nb <= 0) return RSDFT_OK;
    size_t sm = plane_bytes<V>(ctx);
    int room = 0;
    if (ab) RS_TRY(disc_smem(ctx, &sm, &room));
    dim3 grid(ctx->N[2], nb);
    const int pts = ctx->N[0] * ctx->N[1];
    const double nxy = (double)ctx->N[0] * ctx->N[1];
    const double e = (double)sizeof(V);
    const double bpp = psi ? 3 * e : 2 * e;
    ProfScope ps(ctx, RSDFT_K_FFT_XY_INV, 5.0 * nxy * std::log2(nxy) * ctx->N[2] * nb,
                 bpp * (double)ctx->n * nb + (psi ? 0.5 * e * (double)ctx->n : 0.0), st);
    const FftTabs<V> tb = tabs_of(ctx, (V *)nullptr);
    const Discs &discs = ctx->discs;
    const auto *v = v_of(ctx, (V *)nullptr);
    if (psi) {
        RS_TRY(set_smem(ctx, k_xy_inverse<V, Epi::Hpsi>, sm));
        k_xy_inverse<V, Epi::Hpsi><<<grid, fft_threads(ctx, sm, pts, grid), sm, st>>>(tb, buf, psi, v, discs, room, ab, out);
    } else {
        RS_TRY(set_smem(ctx, k_xy_inverse<V, Epi::Plain>, sm));
        k_xy_inverse<V, Epi::Plain><<<grid, fft_threads(ctx, sm, pts, grid), sm, st>>>(tb, buf, psi, v, discs, room, ab, out);
    }
    RS_LAUNCHED(ctx, "k_xy_inverse");
    return RSDFT_OK;
}

// Partial-sum and coefficient buffers of nb bands (of the calls that work in the orbitals' workspace), and the sums
// joined per atom: p (or null) the projections, ab (or null) the scatter coefficients E <beta|psi> of every disc.
static rsdft_status disc_buffers(rsdft_ctx *ctx, int nb, double2 **part, double2 **ab, cudaStream_t st) {
    const size_t per = (size_t)ctx->discs.ndisc * 3;
    RS_TRY(grow(ctx, ctx->discbuf, std::max<size_t>(16, 2 * per * nb * sizeof(double2)), st));
    *part = static_cast<double2 *>(ctx->discbuf.p);
    *ab = *part + per * nb;
    return RSDFT_OK;
}

template <typename V>
static rsdft_status disc_finish(rsdft_ctx *ctx, const V *part, int nb, V *p, V *ab, cudaStream_t st) {
    using T = typename Sc<V>::T;
    k_disc_fin<V><<<cdiv((long long)nb * ctx->pt.natom * 32, PROJ_THREADS), PROJ_THREADS, 0, st>>>(
        ctx->discs, part, nb, (T)ctx->dV, p, ab);
    count_launch(ctx);
    RS_LAUNCHED(ctx, "k_disc_fin");
    return RSDFT_OK;
}

rsdft_status project(rsdft_ctx *ctx, const double2 *psi, double2 *p, int nb, cudaStream_t st) {
    if (nb <= 0 || ctx->pt.natom == 0) return RSDFT_OK;
    const double ne = (double)ctx->nent;
    ProfScope ps(ctx, RSDFT_K_PROJECT, 4.0 * ctx->pt.nproj * ne * nb, 16.0 * ne * nb, st);
    k_project<<<nb * ctx->pt.natom, PROJ_THREADS, 0, st>>>(ctx->discs, ctx->pt, psi, ctx->N[0], ctx->N[1], ctx->n, ctx->dV,
                                                            p);
    RS_LAUNCHED(ctx, "k_project");
    return RSDFT_OK;
}
rsdft_status project32(rsdft_ctx *ctx, const float2 *psi, float2 *p, int nb, cudaStream_t st) {
    if (nb <= 0 || ctx->pt.natom == 0) return RSDFT_OK;
    double2 *buf, *ab;
    RS_TRY(disc_buffers(ctx, nb, &buf, &ab, st));
    float2 *part = reinterpret_cast<float2 *>(buf);
    const double ne = (double)ctx->nent;
    {
        ProfScope ps(ctx, RSDFT_K_PROJECT, 4.0 * ctx->pt.nproj * ne * nb, 8.0 * ne * nb, st);
        k_gather<<<dim3(ctx->N[2], nb), PROJ_THREADS, 0, st>>>(ctx->discs, psi, ctx->N[0], ctx->N[1], ctx->n, part);
    }
    RS_LAUNCHED(ctx, "k_gather");
    return disc_finish<float2>(ctx, part, nb, p, nullptr, st);
}

rsdft_status fft_xy_forward32(rsdft_ctx *ctx, Src kind, const float2 *src, const float2 *src2,
                              const double *theta, const int *act, float2 *dst, int nb,
                              cudaStream_t st, float2 *part) {
    return fft_xy_forward_t<float2>(ctx, kind, src, src2, theta, act, dst, nb, st, part);
}
rsdft_status fft_z_mid32(rsdft_ctx *ctx, Mid mid, float2 *buf, const double *tkin, int nb,
                         cudaStream_t st) {
    return fft_z_mid_t<float2>(ctx, mid, buf, tkin, nb, st);
}
rsdft_status fft_xy_inverse32(rsdft_ctx *ctx, const float2 *buf, const float2 *psi,
                              const float2 *ab, float2 *out, int nb, cudaStream_t st) {
    return fft_xy_inverse_t<float2>(ctx, buf, psi, ab, out, nb, st);
}
rsdft_status refresh_v32(rsdft_ctx *ctx, cudaStream_t st) {
    k_to_float<<<std::max(1, std::min(cdiv(ctx->n, 256), 608)), 256, 0, st>>>(ctx->v, ctx->n, ctx->v32);
    count_launch(ctx);
    RS_LAUNCHED(ctx, "k_to_float");
    return RSDFT_OK;
}

// H psi: the forward pass gathers the projections of its planes, the inverse pass scatters them.
rsdft_status apply_h64(rsdft_ctx *ctx, const double2 *psi, double2 *hpsi, int nb, cudaStream_t st) {
    if (nb <= 0) return RSDFT_OK;
    RS_TRY(ensure_workspace(ctx, nb));
    double2 *part = nullptr, *ab = nullptr;
    const bool nl = ctx->discs.ndisc > 0;
    if (nl) RS_TRY(disc_buffers(ctx, nb, &part, &ab, st));
    RS_TRY(fft_xy_forward(ctx, Src::Plain, psi, nullptr, nullptr, nullptr, nullptr, ctx->ws.T1, nb, st, part));
    if (nl) RS_TRY(disc_finish<double2>(ctx, part, nb, nullptr, ab, st));
    RS_TRY(fft_z_mid(ctx, Mid::Kinetic, ctx->ws.T1, nullptr, nb, st));
    RS_TRY(fft_xy_inverse(ctx, ctx->ws.T1, psi, ab, hpsi, nullptr, nb, st));
    return RSDFT_OK;
}

// FP32 H psi; the FP32 copy of V must be current (refresh_v32).
rsdft_status apply_h32(rsdft_ctx *ctx, const float2 *psi, float2 *hpsi, int nb, cudaStream_t st) {
    if (nb <= 0) return RSDFT_OK;
    RS_TRY(ensure_workspace(ctx, nb));
    double2 *part = nullptr, *ab = nullptr;
    const bool nl = ctx->discs.ndisc > 0;
    if (nl) RS_TRY(disc_buffers(ctx, nb, &part, &ab, st));
    float2 *part32 = reinterpret_cast<float2 *>(part), *ab32 = reinterpret_cast<float2 *>(ab);
    float2 *t1 = reinterpret_cast<float2 *>(ctx->ws.T1);
    RS_TRY(fft_xy_forward32(ctx, Src::Plain, psi, nullptr, nullptr, nullptr, t1, nb, st, part32));
    if (nl) RS_TRY(disc_finish<float2>(ctx, part32, nb, nullptr, ab32, st));
    RS_TRY(fft_z_mid32(ctx, Mid::Kinetic, t1, nullptr, nb, st));
    RS_TRY(fft_xy_inverse32(ctx, t1, psi, ab32, hpsi, nb, st));
    return RSDFT_OK;
}

}  // namespace rsdft

using namespace rsdft;

extern "C" {

rsdft_status rsdft_apply_h(rsdft_ctx *ctx, const void *psi_dev, void *hpsi_dev, int nband,
                           rsdft_precision prec, void *stream) {
    if (!ctx) return fail(nullptr, RSDFT_E_INVALID, "ctx is NULL");
    if (nband < 0 || (nband > 0 && (!psi_dev || !hpsi_dev)))
        return fail(ctx, RSDFT_E_INVALID, "bad psi/hpsi/nband");
    if (psi_dev == hpsi_dev && nband > 0) return fail(ctx, RSDFT_E_INVALID, "psi and hpsi must not overlap");
    if (prec == RSDFT_MIXED) {
        RS_TRY(refresh_v32(ctx, as_stream(stream)));
        return apply_h32(ctx, (const float2 *)psi_dev, (float2 *)hpsi_dev, nband, as_stream(stream));
    }
    if (prec != RSDFT_FP64) return fail(ctx, RSDFT_E_INVALID, "unknown precision");
    return apply_h64(ctx, (const double2 *)psi_dev, (double2 *)hpsi_dev, nband, as_stream(stream));
}

rsdft_status rsdft_project(rsdft_ctx *ctx, const void *psi_dev, void *p_dev, int nband, void *stream) {
    if (!ctx) return fail(nullptr, RSDFT_E_INVALID, "ctx is NULL");
    if (nband < 0 || (nband > 0 && (!psi_dev || !p_dev))) return fail(ctx, RSDFT_E_INVALID, "bad arguments");
    return project(ctx, (const double2 *)psi_dev, (double2 *)p_dev, nband, as_stream(stream));
}

rsdft_status rsdft_precondition_tpa(rsdft_ctx *ctx, const void *r_dev, void *w_dev,
                                    const double *tkin_dev, int nband, void *stream) {
    if (!ctx) return fail(nullptr, RSDFT_E_INVALID, "ctx is NULL");
    if (nband < 0 || (nband > 0 && (!r_dev || !w_dev || !tkin_dev)))
        return fail(ctx, RSDFT_E_INVALID, "bad arguments");
    if (nband == 0) return RSDFT_OK;
    cudaStream_t st = as_stream(stream);
    RS_TRY(ensure_workspace(ctx, nband));
    RS_TRY(fft_xy_forward(ctx, Src::Plain, (const double2 *)r_dev, nullptr, nullptr, nullptr, nullptr,
                          ctx->ws.T1, nband, st));
    RS_TRY(fft_z_mid(ctx, Mid::Tpa, ctx->ws.T1, tkin_dev, nband, st));
    RS_TRY(fft_xy_inverse(ctx, ctx->ws.T1, nullptr, nullptr, (double2 *)w_dev, nullptr, nband, st));
    return RSDFT_OK;
}

}  // extern "C"
