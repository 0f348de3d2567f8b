// Kleinman-Bylander projectors as discs: the sphere of an atom cut by the xy planes of the grid.
//
// The projectors are products of Gaussians, beta = c (1, dx/rc, dy/rc, dz/rc) gx gy gz, cut at
// |d| < rcut: a plane holds a disc of an atom, a disc rows of consecutive x.  With the factors of a
// row held by its lane, a point costs four multiply-adds instead of eight and no table entry of its own
// (the entries of all points, 20 to 36 bytes read again by every band, bounded both directions).
//   gather   a warp a disc, lane = row, a loop over x whose factors are the same for all lanes: three
//            sums per disc, joined over the discs of an atom by k_disc_fin
//   scatter  the same loop, with U = gx A + hx Bx and W = gx By of the plane's discs in shared memory;
//            colour after colour, so that no two warps write a point at a time and the order
//            of the sums is fixed
// What bounds both is the number of instructions.  One GB300, before and after: H psi of 144 bands on
// 64^3 (64 atoms, FP64, after the fixed-point transforms) 6.73 -> 4.58 ms, its gather 1.77 -> 0.8
// and scatter 2.8 -> 1.3 ms; of 160 bands on 96^3 (216 atoms, FP32) gather 1.16 -> 0.6 ms, scatter 1.9 ->
// 1.6 ms.
#pragma once

#include "rsdft_internal.h"

namespace rsdft {

template <typename V> struct Sc;
template <> struct Sc<double2> { using T = double; };
template <> struct Sc<float2> { using T = float; };

// DiscMeta::packed and DiscRow::packed (rsdft_internal.h)
__device__ __forceinline__ int disc_rows(unsigned p) { return p & 255; }
__device__ __forceinline__ int disc_width(unsigned p) { return (p >> 8) & 255; }
__device__ __forceinline__ int disc_x0(unsigned p) { return p >> 16; }
__device__ __forceinline__ bool in_row(int packed, int l) {
    return (unsigned)(l - ((packed >> 8) & 255)) < (unsigned)(packed >> 16);
}

// Discs whose scatter table (per bytes each) is held beside a plane of `base` bytes: what the largest
// number of CTAs on an SM that leaves room for all of them allows, else what there is.
inline int disc_room(size_t base, size_t per, int most, size_t limit) {
    for (int n = 4; n >= 2; --n) {
        const size_t have = (size_t)227 * 1024 / n - 1024;
        if (have >= base + (size_t)most * per) return most;
    }
    return base < limit ? (int)std::min<size_t>(most, (limit - base) / per) : 0;
}

// Runs f(disc, first, last column) for every disc of plane z, the warps of the block sharing the discs
// of one colour at a time (several warps a disc where there are fewer discs than warps); table(c0, n)
// makes what f needs of the plane's discs c0 .. c0 + n, `room` of them at a time.
template <typename Table, typename F>
__device__ __forceinline__ void for_discs(const Discs &t, int z, int room, Table table, F f) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int d0 = t.plane_start[z], d1 = t.plane_start[z + 1], q0 = t.color_ptr[z], q1 = t.color_ptr[z + 1];
    for (int c0 = d0; c0 < d1; c0 += room) {
        const int c1 = min(d1, c0 + room);
        __syncthreads();
        table(c0 - d0, c1 - c0);
        __syncthreads();
        for (int q = q0; q < q1; ++q) {
            const int a = max(__ldg(t.color_start + q), c0), b = min(__ldg(t.color_start + q + 1), c1), n = b - a;
            if (n <= 0) continue;
            const int each = n < nw ? nw / n : 1, part = warp % each;   // warps a disc
            for (int k = warp / each; k < n; k += nw / each) {
                if (warp / each >= nw / each) break;
                const int w = disc_width(__ldg(&t.meta[a + k].packed)), s = (w + each - 1) / each;
                f(a + k, part * s, min(w, part * s + s));
            }
            __syncthreads();
        }
    }
}

}  // namespace rsdft
