// Householder tridiagonalisation of a Hermitian k x k matrix (k <= 448) by one
// thread-block cluster of 16 CTAs, the matrix resident in their shared memory
// and all arithmetic in double-float (dfloat.h).
//
// The reduction is the unblocked one of the cooperative FP64 kernel in dense.cu
// (LAPACK zhetd2 order, lower form), step i = 0 .. k-2 with L = k-1-i:
//   x = A[i+1:, i] -> reflector v_i (v_i[0] = 1), tau_i, beta_i = e_i; d_i = A[i][i]
//   y = A[i+1:, i+1:] v_i,  w = tau_i y,  w' = w - 1/2 tau_i (w^H v_i) v_i
//   A[i+1:, i+1:] -= v_i w'^H + w' v_i^H.
// On GB300 that kernel is bound by the latency of its per-step FP64 chains
// (a warp FP64 instruction takes 64 cycles of its sub-partition) and by a grid
// barrier per step.  Here:
//   - the matrix lives in distributed shared memory: row r in CTA r mod 16,
//     full rows of complex double-floats (16 B), so k <= 448 fits in 227 KB;
//   - one exchange per step: after a cluster barrier every CTA holds y = A v_{i-1} of all rows and the
//     next pivot row (their owners stored them into every CTA's shared memory), and forms w', the updated
//     pivot row and its reflector by itself, an element a thread.  A second barrier says that y
//     and the pivot row have been read; its wait comes long after and costs nothing;
//   - the reflector's scalars (norm, root, reciprocals: a chain) are one warp's work, beside the rank-2
//     update by the other 15;
//   - warps whose columns are all reduced already leave the per-element work;
//   - double-float keeps about 48 significant bits, so the reduction's backward
//     error is a small multiple of 2^-46 |A| instead of 2^-53 |A|.
// Bound: the FP32 lanes for the first half of the columns (115 operations an element in the update, 55 in
// A v; packed pairs have the same rate), the chain of a step for the rest.  SM cycles a column by quarters, k = 432:
//   28.2k, 19.3k, 11.1k, 7.4k; before (the owner of the pivot row formed the reflector, a second exchange
//   gave it out): 31.0k, 21.7k, 14.2k, 10.0k.
// Measured, the whole eigensolve (a third of the vectors): k = 144 1.28 -> 1.10 ms, 288 2.89 -> 2.52 ms, 432 5.39 -> 4.90 ms.
// Over all SMs, with polled values in global memory instead of cluster barriers, a column took 14k cycles
// throughout (7k of them until the last value was seen): 3.5 ms at k = 432 and slower below 360.
// Outputs as the FP64 kernel: d, e (real), tau, and v_i in vh row i (columns
// i+1 .. k-1), for the compact-WY back-transformation.
#include <cooperative_groups.h>

#include <algorithm>

#include "dfloat.h"
#include "rsdft_internal.h"

namespace rsdft {

namespace cg = cooperative_groups;
using namespace dfl;

constexpr int TC_C = 16;     // CTAs in the cluster
constexpr int TC_T = 512;    // threads per CTA
constexpr int TC_W = TC_T / 32;
constexpr int TC_WORK = TC_W - 1;      // warps of the rank-2 update; the last one does the scalars meanwhile
constexpr int TC_KMAX = 448;           // largest k whose rows fit the cluster's shared memory
constexpr int TC_ROWS = TC_KMAX / TC_C;
constexpr int TC_SPLIT = 8;            // pieces of a row, at most
constexpr int TC_PARTS = 64;           // pieces of all rows, at most

__device__ __forceinline__ cdf ld4(const float4 &v) { return cdf{df{v.x, v.y}, df{v.z, v.w}}; }
__device__ __forceinline__ float4 st4(const cdf &c) { return make_float4(c.re.h, c.re.l, c.im.h, c.im.l); }

__device__ __forceinline__ void cl_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// s + sum of one product's exact pieces: the running sum keeps its hi part by
// TwoSum and collects every rounding error in lo (one renormalisation at the end)
struct Acc {
    float h, l;
};
__device__ __forceinline__ void acc_prod(Acc &s, float ah, float al, float bh, float bl) {
    const df p = two_prod(ah, bh);
    const df t = two_sum(s.h, p.h);
    s.h = t.h;
    s.l = fadd(s.l, fadd(t.l, ffma(ah, bl, ffma(al, bh, p.l))));
}
__device__ __forceinline__ void acc_df(Acc &s, df x) {
    const df t = two_sum(s.h, x.h);
    s.h = t.h;
    s.l = fadd(s.l, fadd(t.l, x.l));
}
__device__ __forceinline__ df acc_get(const Acc &s) { return fast_two_sum(s.h, s.l); }

// 1 / x and sqrt(x), x > 0 well inside FP32's range, with one division or root: the correction term
// (2^-24 of the value) takes the FP32 reciprocal, an error of some 2^-47
__device__ __forceinline__ df rcp_df(df x) {
    const float r = fdiv(1.0f, x.h);
    return fast_two_sum(r, fmul(r, ffma(-r, x.l, ffma(-r, x.h, 1.0f))));
}
__device__ __forceinline__ df sqrt_df(df x, float half_rsq) {   // half_rsq = 0.5 / sqrt(x) to FP32's accuracy
    const float s = fsqrt(x.h);
    return fast_two_sum(s, fmul(fadd(ffma(-s, s, x.h), x.l), half_rsq));
}

// a - v_r conj(w_c) - w_r conj(v_c), all complex double-float
__device__ __forceinline__ cdf rank2(const cdf &a, const cdf &vr, const cdf &wr, const cdf &vc, const cdf &wc) {
    // re: a.re - (vr.re wc.re + vr.im wc.im + wr.re vc.re + wr.im vc.im)
    Acc re{a.re.h, a.re.l}, im{a.im.h, a.im.l};
    acc_prod(re, -vr.re.h, -vr.re.l, wc.re.h, wc.re.l);
    acc_prod(re, -vr.im.h, -vr.im.l, wc.im.h, wc.im.l);
    acc_prod(re, -wr.re.h, -wr.re.l, vc.re.h, vc.re.l);
    acc_prod(re, -wr.im.h, -wr.im.l, vc.im.h, vc.im.l);
    // im: a.im - (vr.im wc.re - vr.re wc.im + wr.im vc.re - wr.re vc.im)
    acc_prod(im, -vr.im.h, -vr.im.l, wc.re.h, wc.re.l);
    acc_prod(im, vr.re.h, vr.re.l, wc.im.h, wc.im.l);
    acc_prod(im, -wr.im.h, -wr.im.l, vc.re.h, vc.re.l);
    acc_prod(im, wr.re.h, wr.re.l, vc.im.h, vc.im.l);
    return cdf{acc_get(re), acc_get(im)};
}

__device__ __forceinline__ df shfl_df(df x, int o) {
    return df{__shfl_xor_sync(0xffffffffu, x.h, o), __shfl_xor_sync(0xffffffffu, x.l, o)};
}

// the same over one xor step of a warp
__device__ __forceinline__ void acc_xor(Acc &s, int o) {
    const df t = two_sum(s.h, __shfl_xor_sync(0xffffffffu, s.h, o));
    s.l = fadd(fadd(s.l, __shfl_xor_sync(0xffffffffu, s.l, o)), t.l);
    s.h = t.h;
}

// re and im over a warp: the sum of re in lanes 0-15, of im in lanes 16-31
__device__ __forceinline__ Acc warp_sum2(const Acc &re, const Acc &im, bool up) {
    Acc s{up ? im.h : re.h, up ? im.l : re.l};
    const float oh = __shfl_xor_sync(0xffffffffu, up ? re.h : im.h, 16);
    const float ol = __shfl_xor_sync(0xffffffffu, up ? re.l : im.l, 16);
    const df t = two_sum(s.h, oh);
    s = Acc{t.h, fadd(fadd(s.l, ol), t.l)};
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) acc_xor(s, o);
    return s;
}

__global__ void __launch_bounds__(TC_T, 1)
k_tridiag_cluster(const double2 *__restrict__ a, int k, int ld, double2 *__restrict__ vh, int ldv,
                  double2 *__restrict__ tau, double *__restrict__ d, double *__restrict__ e) {
    cg::cluster_group cl = cg::this_cluster();
    const int me = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = (k + TC_C - 1) / TC_C;   // row slots per CTA
    extern __shared__ float4 sm[];
    float4 *A = sm;                        // [R][k]: row me + 16 j in slot j
    float4 *V = A + (size_t)R * k;         // v of the last reflector, by column
    float4 *W = V + k;                     // its w'
    float4 *Y = W + k;                     // y = A v, stored here by the owners of its rows
    float4 *P = Y + k;                     // the next pivot row, stored here by its owner
    __shared__ float4 s_alpha, s_pub[3];
    __shared__ float2 s_sum[2][TC_W], s_norm[TC_W], s_part[2][TC_PARTS];
    __shared__ unsigned char s_split[TC_ROWS + 1];
    const int c = tid;                     // this thread's column (k < TC_T)
    const bool up = lane >= 16;
    const cdf zero{df{0.f, 0.f}, df{0.f, 0.f}};
    const cdf one{df{1.f, 0.f}, df{0.f, 0.f}};

    for (int idx = tid; idx < R * k; idx += TC_T) {
        const int j = idx / k, q = idx - j * k, r = me + TC_C * j;
        cdf v = zero;
        if (r < k) {
            const double2 x = a[(size_t)r * ld + q];
            v = cdf{from_double(x.x), from_double(x.y)};
        }
        A[idx] = st4(v);
    }
    // pieces a row of the matrix-vector product is cut into when nr own rows (of about 16 nr columns)
    // are left: the fewest turns, of 55 instructions a column and 100 for the sum of a piece
    if (tid <= TC_ROWS) {
        int best = 1, cost = 1 << 30;
        for (int S = 1; S <= TC_SPLIT && S * tid <= TC_PARTS; ++S) {
            const int t = ((tid * S + TC_W - 1) / TC_W) * (((16 * tid + 32 * S - 1) / (32 * S)) * 55 + 100);
            if (t < cost) {
                cost = t;
                best = S;
            }
        }
        s_split[tid] = (unsigned char)best;
    }
    cdf t = zero, v = zero, x = zero;      // tau_i, v_i[c], conj of the pivot row at c
    df half{0.f, 0.f};                     // -|tau_i|^2 / 2
    cl_arrive();
    for (int i = -1;; ++i) {
        const int n = i + 1;               // the reflector this pass forms, over columns n + 1 .. k - 1
        cl_wait();                         // Y and P are complete
        if (i < 0) {
            if (c < k) {
                const double2 p = a[c];
                x = cdf{from_double(p.x), neg(from_double(p.y))};
                if (me == 1 && c == 0) d[0] = p.x;
            }
            cl_arrive();
        } else {
            const bool live = warp * 32 + 31 >= n && warp * 32 < k;   // this warp has columns left
            const bool in = c >= n && c < k;
            const cdf y = in ? ld4(Y[c]) : zero, p = in ? ld4(P[c]) : zero;
            cl_arrive();                   // Y and P have been read: the owners may store the next ones
            Acc wr{0.f, 0.f}, wi{0.f, 0.f};
            cdf w = zero;
            if (live) {
                // y^H v
                Acc sr{0.f, 0.f}, si{0.f, 0.f};
                acc_prod(sr, y.re.h, y.re.l, v.re.h, v.re.l);
                acc_prod(si, y.re.h, y.re.l, v.im.h, v.im.l);
                acc_prod(sr, y.im.h, y.im.l, v.im.h, v.im.l);
                acc_prod(si, -y.im.h, -y.im.l, v.re.h, v.re.l);
                const Acc q = warp_sum2(sr, si, up);
                if ((lane & 15) == 0) s_sum[up][warp] = make_float2(q.h, q.l);
                // tau y, which does not wait for that sum
                acc_prod(wr, t.re.h, t.re.l, y.re.h, y.re.l);
                acc_prod(wi, t.re.h, t.re.l, y.im.h, y.im.l);
                acc_prod(wr, -t.im.h, -t.im.l, y.im.h, y.im.l);
                acc_prod(wi, t.im.h, t.im.l, y.re.h, y.re.l);
            } else if ((lane & 15) == 0) {
                s_sum[up][warp] = make_float2(0.f, 0.f);
            }
            __syncthreads();
            if (live) {
                const float2 q = s_sum[up][lane & (TC_W - 1)];
                Acc s{q.x, q.y};
#pragma unroll
                for (int o = TC_W / 2; o > 0; o >>= 1) acc_xor(s, o);
                // w' = tau y - |tau|^2 / 2 (y^H v) v
                const df al = mul(half, acc_get(s));
                const df ar{__shfl_sync(0xffffffffu, al.h, 0), __shfl_sync(0xffffffffu, al.l, 0)};
                const df ai{__shfl_sync(0xffffffffu, al.h, 16), __shfl_sync(0xffffffffu, al.l, 16)};
                acc_prod(wr, ar.h, ar.l, v.re.h, v.re.l);
                acc_prod(wi, ar.h, ar.l, v.im.h, v.im.l);
                acc_prod(wr, -ai.h, -ai.l, v.im.h, v.im.l);
                acc_prod(wi, ai.h, ai.l, v.re.h, v.re.l);
                w = cdf{acc_get(wr), acc_get(wi)};
                if (in) W[c] = st4(w);
            }
            __syncthreads();
            // the pivot row n with the update (v_n = 1)
            if (live) {
                const cdf wn = ld4(W[n]);
                Acc xr{p.re.h, p.re.l}, xi{p.im.h, p.im.l};
                acc_df(xr, neg(w.re));
                acc_df(xi, w.im);
                acc_prod(xr, -wn.re.h, -wn.re.l, v.re.h, v.re.l);
                acc_prod(xi, -wn.im.h, -wn.im.l, v.re.h, v.re.l);
                acc_prod(xr, -wn.im.h, -wn.im.l, v.im.h, v.im.l);
                acc_prod(xi, wn.re.h, wn.re.l, v.im.h, v.im.l);
                x = cdf{acc_get(xr), neg(acc_get(xi))};
                if (me == 1 && c == n) d[n] = to_double(x.re);
            }
            if (n == k - 1) break;
        }
        const int L = k - 1 - n;
        {
            Acc s{0.f, 0.f};
            if (warp * 32 + 31 > n + 1 && warp * 32 < k) {
                if (c > n + 1 && c < k) {
                    acc_prod(s, x.re.h, x.re.l, x.re.h, x.re.l);
                    acc_prod(s, x.im.h, x.im.l, x.im.h, x.im.l);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc_xor(s, o);
            }
            if (lane == 0) s_norm[warp] = make_float2(s.h, s.l);
            if (c == n + 1) s_alpha = st4(x);
        }
        __syncthreads();
        cl_wait();                         // every CTA has read Y and P
        // own rows > n: slots j0 .. j0 + nr - 1
        const int j0 = (n + 1 - me + TC_C - 1) / TC_C;   // n + 1 - me > -TC_C
        const int nr = max(0, (k - me + TC_C - 1) / TC_C - j0);
        if (warp == TC_WORK) {
            // ---- the reflector's scalars
            const float2 q = s_norm[lane & (TC_W - 1)];
            Acc s{q.x, q.y};
#pragma unroll
            for (int o = TC_W / 2; o > 0; o >>= 1) acc_xor(s, o);
            const df xnorm2 = acc_get(s);
            const cdf x0 = ld4(s_alpha);
            cdf tn = zero, scal = zero;
            df beta;
            // a column below 1e-18 (squares near FP32's underflow) is taken as
            // reduced already: H = I, beta = Re alpha (an absolute change below
            // 1e-18, far under the rounding of an Ha-scale matrix)
            const df nb2 = add(cabs2(x0), xnorm2);
            if ((xnorm2.h == 0.f && x0.im.h == 0.f) || !(nb2.h > 1e-36f)) {
                beta = x0.re;
            } else {
                // beta = -sign(Re alpha) |(alpha, x)|, tau = (beta - alpha) / beta,
                // scal = 1 / (alpha - beta) = conj(alpha - beta) / |alpha - beta|^2
                const df nb = sqrt_df(nb2, 0.5f * rsqrtf(nb2.h));
                beta = x0.re.h >= 0.f ? neg(nb) : nb;
                const cdf den{sub(x0.re, beta), x0.im};
                const df rb = rcp_df(beta), rd = rcp_df(cabs2(den));
                tn = cdf{mul(sub(beta, x0.re), rb), neg(mul(x0.im, rb))};
                scal = cdf{mul(den.re, rd), neg(mul(den.im, rd))};
            }
            if (lane == 0) {
                const df h = mul_f(cabs2(tn), -0.5f);
                s_pub[0] = st4(tn);
                s_pub[1] = st4(scal);
                s_pub[2] = make_float4(h.h, h.l, 0.f, 0.f);
                if (me == 1) {
                    e[n] = to_double(beta);
                    tau[n] = make_double2(to_double(tn.re), to_double(tn.im));
                }
            }
        } else {
            // ---- the rank-2 update of the own rows: units of a row and 64 columns, ordered by columns
            // (v and w' of a column stay in registers), a share for each warp; row n + 1, the next
            // pivot row, goes to every CTA
            const int total = nr * ((L + 63) >> 6);
            const int u1 = (warp + 1) * total / TC_WORK;
            int u = warp * total / TC_WORK;
            while (u < u1) {
                const int blk = u / nr;
                int j = u - blk * nr;
                const int je = min(nr, j + u1 - u);
                u += je - j;
                const int ca = n + 1 + blk * 64 + lane, cb = ca + 32;
                const bool ina = ca < k, inb = cb < k;
                cdf va = zero, wa = zero, vb = zero, wb = zero;
                if (i >= 0 && ina) {
                    va = ld4(V[ca]);
                    wa = ld4(W[ca]);
                }
                if (i >= 0 && inb) {
                    vb = ld4(V[cb]);
                    wb = ld4(W[cb]);
                }
                for (; j < je; ++j) {
                    const int r = me + TC_C * (j0 + j);
                    float4 *row = A + (size_t)(j0 + j) * k;
                    float4 za = make_float4(0.f, 0.f, 0.f, 0.f), zb = za;
                    if (ina) za = row[ca];
                    if (inb) zb = row[cb];
                    if (i >= 0) {
                        const cdf vr = ld4(V[r]), wr = ld4(W[r]);
                        za = st4(rank2(ld4(za), vr, wr, va, wa));
                        zb = st4(rank2(ld4(zb), vr, wr, vb, wb));
                        if (ina) row[ca] = za;
                        if (inb) row[cb] = zb;
                    }
                    if (r == n + 1)
                        for (int b = 0; b < TC_C; ++b) {
                            float4 *dst = cl.map_shared_rank(P, b);
                            if (ina) dst[ca] = za;
                            if (inb) dst[cb] = zb;
                        }
                }
            }
        }
        __syncthreads();
        t = ld4(s_pub[0]);
        half = df{s_pub[2].x, s_pub[2].y};
        v = zero;
        if (c > n && c < k) {
            v = c == n + 1 ? one : cmul(x, ld4(s_pub[1]));
            V[c] = st4(v);
            // the FP64 copy for the back-transformation: one warp's range per CTA
            if (warp == me) vh[(size_t)n * ldv + c] = make_double2(to_double(v.re), to_double(v.im));
        }
        __syncthreads();
        // ---- y = A v over the own rows
        const int S = s_split[nr], seg = (L + S - 1) / S;
        for (int u = warp; u < nr * S; u += TC_W) {
            const int j = u / S, c0 = n + 1 + (u - j * S) * seg, c1 = min(k, c0 + seg);
            const float4 *row = A + (size_t)(j0 + j) * k;
            Acc yr{0.f, 0.f}, yi{0.f, 0.f};
            for (int cc = c0 + lane; cc < c1; cc += 32) {
                const cdf z = ld4(row[cc]), s = ld4(V[cc]);
                acc_prod(yr, z.re.h, z.re.l, s.re.h, s.re.l);
                acc_prod(yi, z.re.h, z.re.l, s.im.h, s.im.l);
                acc_prod(yr, -z.im.h, -z.im.l, s.im.h, s.im.l);
                acc_prod(yi, z.im.h, z.im.l, s.re.h, s.re.l);
            }
            const Acc q = warp_sum2(yr, yi, up);
            if ((lane & 15) == 0) s_part[up][u] = make_float2(q.h, q.l);
        }
        __syncthreads();
        // every row's sum into every CTA (one remote store a thread)
        if (tid < nr * TC_C) {
            const int j = tid / TC_C;
            Acc yr{0.f, 0.f}, yi{0.f, 0.f};
            for (int s = 0; s < S; ++s) {
                const float2 q = s_part[0][j * S + s], z = s_part[1][j * S + s];
                acc_df(yr, df{q.x, q.y});
                acc_df(yi, df{z.x, z.y});
            }
            cl.map_shared_rank(Y, tid & (TC_C - 1))[me + TC_C * (j0 + j)] = st4(cdf{acc_get(yr), acc_get(yi)});
        }
        cl_arrive();
    }
    cl_wait();   // no CTA leaves while another may still read its shared memory
}

// Each reflector made unitary in FP64.  H = I - tau v v^H is unitary exactly when
// 2 Re(tau) = |tau|^2 |v|^2; the double-float reduction leaves that true to about
// 2^-46, and the back-transformed eigenvectors would be orthonormal only to
// ~k 2^-46.  Re(tau) is reset to the root of nu a^2 - 2 a + nu b^2 = 0 (b = Im tau,
// nu = |v|^2 summed in FP64) nearest its value: a change of ~2^-46 relative, within
// the reduction's own backward error.  One warp per reflector.
__global__ void __launch_bounds__(256)
k_unitarize(int k, const double2 *__restrict__ vh, int ldv, double2 *__restrict__ tau) {
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= k - 1) return;
    const double2 *v = vh + (size_t)i * ldv;
    double s = 0.0;
    for (int c = i + 1 + lane; c < k; c += 32) s = fma(v[c].x, v[c].x, fma(v[c].y, v[c].y, s));
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane != 0 || !(s > 0.0)) return;
    const double2 t = tau[i];
    const double disc = 1.0 - s * s * t.y * t.y;
    if (!(disc >= 0.0)) return;
    const double r = ::sqrt(disc);
    const double a_lo = s * t.y * t.y / (1.0 + r);   // (1 - r) / nu without cancellation
    const double a_hi = (1.0 + r) / s;
    tau[i].x = fabs(t.x - a_lo) <= fabs(t.x - a_hi) ? a_lo : a_hi;
}

size_t tridiag_cluster_smem(int k) {
    const size_t R = (size_t)(k + TC_C - 1) / TC_C;
    return (R * k + 4 * (size_t)k) * sizeof(float4);
}

bool tridiag_cluster_fits(int k) { return k >= 2 && k <= TC_KMAX; }

rsdft_status tridiag_cluster(rsdft_ctx *ctx, const double2 *a, int k, int ld, double2 *vh, int ldv, double2 *tau,
                             double *d, double *e, cudaStream_t st, bool *done) {
    *done = false;
    if (!tridiag_cluster_fits(k)) return RSDFT_OK;
    const size_t smem = tridiag_cluster_smem(k);
    // the attributes once per process (largest size), then a residency check
    static const bool ok = [] {
        bool good = cudaFuncSetAttribute(k_tridiag_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                        cudaSuccess &&
                    cudaFuncSetAttribute(k_tridiag_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)tridiag_cluster_smem(TC_KMAX)) == cudaSuccess;
        if (good) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = TC_C;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(TC_C);
            cfg.blockDim = dim3(TC_T);
            cfg.dynamicSmemBytes = tridiag_cluster_smem(TC_KMAX);
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int ncl = 0;
            good = cudaOccupancyMaxActiveClusters(&ncl, k_tridiag_cluster, &cfg) == cudaSuccess && ncl >= 1;
        }
        cudaGetLastError();
        return good;
    }();
    if (!ok) return RSDFT_OK;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = TC_C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(TC_C);
    cfg.blockDim = dim3(TC_T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, k_tridiag_cluster, a, k, ld, vh, ldv, tau, d, e);
    if (err != cudaSuccess) {
        cudaGetLastError();
        return RSDFT_OK;   // the caller falls back to the cooperative FP64 kernel
    }
    count_launch(ctx);
    RS_LAUNCHED(ctx, "k_tridiag_cluster");
    k_unitarize<<<cdiv(k - 1, 8), 256, 0, st>>>(k, vh, ldv, tau);
    count_launch(ctx);
    RS_LAUNCHED(ctx, "k_unitarize");
    *done = true;
    return RSDFT_OK;
}

}  // namespace rsdft
