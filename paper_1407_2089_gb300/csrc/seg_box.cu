// seg_box.cu -- the background of the denoise front end (Background Noise
// Removal, Eq. 1): three rounded box passes of radius r along x, then y, then
// z, each pass with replicate edges.
//
// One thread follows one line (or a chunk of one) and runs all three passes at
// once: position p of the input feeds the first running sum, whose value at
// p - r feeds the second, whose value at p - 2r feeds the third, which gives
// the output at p - 3r.  The 2r + 1 values in each window stay in registers as
// three rings indexed at compile time (the loop is unrolled by the window, one
// instance per radius), so a voxel costs one load, three additions, three
// multiply-highs and one store, and no pass goes through memory.
//
// Ends of a line: the passes' values before position 0 repeat the value at 0
// and those past the end the last one.  A line's first chunk therefore works
// out the first two passes' values at 0 beforehand and starts with rings full
// of them; a chunk inside a line starts 3r positions early with empty rings,
// which fill by the time its first output is due.
//
// Bound by instruction issue.  4 volumes of 512 x 512 x 64, r = 8: x 238 -> 223,
// y 154 -> 101, z 214 -> 148 us against three passes through shared memory with a
// barrier each.  Chunks of 256 positions along x (two blocks fewer resident) take
// 330 us there.
#include <algorithm>
#include <cstdint>

#include "seg_internal.h"

namespace seg {
namespace {

constexpr int BX_THREADS = 128;

// (n + r) / w for n + r < 2^24 and w = 2r + 1 <= 65, as a multiply-high by
// mul = ceil(2^32 / w) (division by an invariant integer, Granlund and
// Montgomery 1994): the product's error n * (mul * w - 2^32) / (w 2^32) stays
// below 2^-8 < 1/w, so the floor is exact.
__device__ __forceinline__ uint32_t box_div(uint32_t n, uint32_t mul) { return __umulhi(n, mul); }

// Outputs [c0, c1) of one line of n voxels, `st` elements apart, from src to
// dst (src itself allowed: an output is written after its position was read).
// start: position 0 is the line's first, and c0 <= 3 R (else src lies 3 R or more positions
// inside the line and c0 >= 3 R).  Positions from c1 + 3 R on are not read.
// start, c0, c1 and n are the same in every thread of the block.
template <int R>
__device__ __forceinline__ void box_line(const uint16_t *src, uint16_t *dst, size_t st, int n, int c0, int c1,
                                         bool start, uint32_t mul) {
    constexpr int W = 2 * R + 1;
    const int e = min(n, c1 + 3 * R);
    auto at = [&](int q) -> uint32_t { return src[(size_t)min(q, e - 1) * st]; };
    uint32_t g1[W], g2[W], g3[W];  // windows of the input and of the first two passes
    uint32_t x[W];                    // the next W inputs
    int p = max(c0 - 3 * R, 0);
    auto load = [&]() {
        if (p + W <= e) {
            const uint16_t *a = src + (size_t)p * st;
#pragma unroll
            for (int s = 0; s < W; ++s) x[s] = a[(size_t)s * st];
        } else {
#pragma unroll
            for (int s = 0; s < W; ++s) x[s] = at(p + s);
        }
    };
    load();
    uint32_t x0 = 0, f1 = 0, f2 = 0;  // values at positions before 0
    if (start) {  // (p = 0)
        x0 = x[0];
        // the sums hold the window sum plus the rounding term R
        uint32_t t = (uint32_t)R + (uint32_t)(R + 1) * x0;
#pragma unroll
        for (int i = 1; i <= R; ++i) t += x[i];
        uint32_t b = box_div(t, mul);
        f1 = b;
        uint32_t u = (uint32_t)R + (uint32_t)(R + 1) * b;
#pragma unroll
        for (int q = 1; q <= R; ++q) {
            if (q < n) {
                t += x[q + R] - x0;  // (position q - R - 1 < 0 leaves the window)
                b = box_div(t, mul);
            }
            u += b;
        }
        f2 = box_div(u, mul);
    }
#pragma unroll
    for (int s = 0; s < W; ++s) {
        g1[s] = x0;
        g2[s] = f1;
        g3[s] = f2;
    }
    uint32_t s1 = (uint32_t)R + W * x0, s2 = (uint32_t)R + W * f1, s3 = (uint32_t)R + W * f2;
    uint32_t l1 = 0, l2 = 0;  // the passes' latest values
    for (;;) {
        if (p >= 2 * R && p - 3 * R >= c0 && p + W - 3 * R <= c1 && p + W - R <= n) {
            // every pass inside the line, every output wanted
            uint16_t *o = dst + (size_t)(p - 3 * R) * st;
#pragma unroll
            for (int s = 0; s < W; ++s) {
                s1 += x[s] - g1[s];
                g1[s] = x[s];
                l1 = box_div(s1, mul);
                s2 += l1 - g2[s];
                g2[s] = l1;
                l2 = box_div(s2, mul);
                s3 += l2 - g3[s];
                g3[s] = l2;
                o[(size_t)s * st] = (uint16_t)box_div(s3, mul);
            }
        } else {
#pragma unroll
            for (int s = 0; s < W; ++s) {
                const int q1 = p + s - R, q2 = q1 - R, q3 = q2 - R;
                s1 += x[s] - g1[s];
                g1[s] = x[s];
                const uint32_t b1 = box_div(s1, mul);
                l1 = q1 < 0 ? f1 : (q1 < n ? b1 : l1);
                s2 += l1 - g2[s];
                g2[s] = l1;
                const uint32_t b2 = box_div(s2, mul);
                l2 = q2 < 0 ? f2 : (q2 < n ? b2 : l2);
                s3 += l2 - g3[s];
                g3[s] = l2;
                if (q3 >= c0 && q3 < c1) dst[(size_t)q3 * st] = (uint16_t)box_div(s3, mul);
            }
        }
        p += W;
        if (p >= c1 + 3 * R) break;
        load();
    }
}

// box_line for a radius of class CLS (1..4, 5..8, 9..16: a kernel per class,
// so that small radii are not held to the registers of the largest).
template <int CLS>
__device__ __forceinline__ void box_line_r(int r, const uint16_t *src, uint16_t *dst, size_t st, int n, int c0, int c1,
                                           uint32_t mul, bool start) {
#define SEG_BOX_R(K) \
    case K: box_line<K>(src, dst, st, n, c0, c1, start, mul); break;
    if (CLS == 0) {
        switch (r) { SEG_BOX_R(1) SEG_BOX_R(2) SEG_BOX_R(3) SEG_BOX_R(4) }
    } else if (CLS == 1) {
        switch (r) { SEG_BOX_R(5) SEG_BOX_R(6) SEG_BOX_R(7) SEG_BOX_R(8) }
    } else {
        switch (r) {
            SEG_BOX_R(9) SEG_BOX_R(10) SEG_BOX_R(11) SEG_BOX_R(12) SEG_BOX_R(13) SEG_BOX_R(14) SEG_BOX_R(15)
            SEG_BOX_R(16)
        }
    }
#undef SEG_BOX_R
}

__device__ __forceinline__ int box_class(uint32_t r) { return r <= 4 ? 0 : (r <= 8 ? 1 : 2); }

template <int AXIS>
__device__ __forceinline__ uint32_t box_base(const VolDev &V) {
    return AXIS == 0 ? V.dn_base0 : (AXIS == 1 ? V.dn_base1 : V.dn_base2);
}

// The volume of flat box item `it` (volumes without the front end hold none).
template <int AXIS>
__device__ __forceinline__ uint32_t box_volume(const BatchHdr *__restrict__ h, uint32_t it) {
    uint32_t lo = 0, hi = h->nvol;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (box_base<AXIS>(h->vol[mid]) <= it) lo = mid; else hi = mid;
    }
    return lo;
}

// Along y (AXIS 1: dn_a -> dn_b) or z (AXIS 2: dn_b -> dn_a): an item is
// BX_THREADS consecutive lines (x fastest, whatever X is) and a chunk of at
// most DN_CHUNK positions.
template <int AXIS, int CLS>
__global__ void __launch_bounds__(BX_THREADS) k_box_lines(const BatchHdr *__restrict__ h) {
    for (uint32_t it = blockIdx.x; it < h->dn_items[AXIS]; it += gridDim.x) {
        const VolDev &V = h->vol[box_volume<AXIS>(h, it)];
        if (box_class(V.dn_r) != CLS) continue;
        const uint32_t li = it - box_base<AXIS>(V);
        const uint32_t len = AXIS == 1 ? V.Y : V.Z, nchunk = box_chunks(len, DN_CHUNK);
        const BoxChunk c = box_chunk(len, DN_CHUNK, li % nchunk, V.dn_r);
        const uint64_t line = (uint64_t)(li / nchunk) * BX_THREADS + threadIdx.x;
        if (line >= (uint64_t)V.X * (AXIS == 1 ? V.Z : V.Y) || c.c0 >= c.c1) continue;
        const size_t plane = (size_t)V.X * V.Y, st = AXIS == 1 ? (size_t)V.X : plane;
        const size_t o = (AXIS == 1 ? line / V.X * plane + line % V.X : (size_t)line) + c.first * st;
        const uint16_t *src = AXIS == 1 ? V.dn_a : V.dn_b;
        uint16_t *dst = AXIS == 1 ? V.dn_b : V.dn_a;
        box_line_r<CLS>((int)V.dn_r, src + o, dst + o, st, c.n, c.c0, c.c1, V.dn_mul, c.start);
    }
}

// Along x (dn_src -> dn_a): an item is BX_THREADS rows and a chunk of at most
// DN_CHUNK_X positions, which pass through shared memory [position][row], read
// and written with lanes along x; the lines run in place there.
constexpr int BX_PITCH = BX_THREADS + 2;  // an odd number of words
size_t box_x_smem(int r) { return 2ull * (DN_CHUNK_X + 6 * r) * BX_PITCH; }

template <int CLS>
__global__ void __launch_bounds__(BX_THREADS) k_box_x(const BatchHdr *__restrict__ h) {
    extern __shared__ __align__(16) uint16_t bsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int WARPS = BX_THREADS / 32, RB = 8;
    for (uint32_t it = blockIdx.x; it < h->dn_items[0]; it += gridDim.x) {
        const VolDev &V = h->vol[box_volume<0>(h, it)];
        if (box_class(V.dn_r) != CLS) continue;
        const uint32_t li = it - V.dn_base0;
        const int n = (int)V.X, r = (int)V.dn_r, nchunk = (n + DN_CHUNK_X - 1) / DN_CHUNK_X;
        const int per = (n + nchunk - 1) / nchunk;
        const uint32_t row0 = li / (uint32_t)nchunk * BX_THREADS;
        const int c0 = (int)(li % (uint32_t)nchunk) * per, c1 = min(c0 + per, n);
        const int nrow = (int)min((uint32_t)BX_THREADS, V.rows - row0);
        const int lo = max(c0 - 3 * r, 0), hi = min(c1 + 3 * r, n);  // positions read
        __syncthreads();  // the previous item is done with the buffer
        if (c0 < c1) {
            // RB rows' loads in flight per warp
            for (int w0 = warp; w0 < nrow; w0 += WARPS * RB) {
                for (int q = lo + lane; q < hi; q += 32) {
                    uint16_t v[RB];
#pragma unroll
                    for (int k = 0; k < RB; ++k) {
                        const int w = w0 + k * WARPS;
                        v[k] = w < nrow ? V.dn_src[(size_t)(row0 + w) * n + q] : (uint16_t)0;
                    }
#pragma unroll
                    for (int k = 0; k < RB; ++k) {
                        const int w = w0 + k * WARPS;
                        if (w < nrow) bsm[(q - lo) * BX_PITCH + w] = v[k];
                    }
                }
            }
        }
        __syncthreads();
        if (c0 < c1 && (int)threadIdx.x < nrow) {
            // the line from position lo on: lo is 0 or 3r before the chunk
            uint16_t *line = bsm + threadIdx.x;
            box_line_r<CLS>(r, line, line, BX_PITCH, n - lo, c0 - lo, c1 - lo, V.dn_mul, lo == 0);
        }
        __syncthreads();
        if (c0 < c1) {
            for (int w = warp; w < nrow; w += WARPS) {
                uint16_t *row = V.dn_a + (size_t)(row0 + w) * n;
                for (int q = c0 + lane; q < c1; q += 32) row[q] = bsm[(q - lo) * BX_PITCH + w];
            }
        }
    }
}

template <int CLS>
void launch_class(const BatchHdr *d, const LaunchPlan &p, cudaStream_t s) {
    k_box_x<CLS><<<p.grid_box, BX_THREADS, box_x_smem(CLS == 0 ? 4 : (CLS == 1 ? 8 : 16)), s>>>(d);
    k_box_lines<1, CLS><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    k_box_lines<2, CLS><<<p.grid_box, BX_THREADS, 0, s>>>(d);
}

}  // namespace

uint32_t box_lines_items(uint64_t lines, uint32_t n, uint32_t chunk) {
    return (uint32_t)((lines + BX_THREADS - 1) / BX_THREADS * box_chunks(n, chunk));
}

cudaError_t configure_box() {
    const void *fn[3] = {(const void *)k_box_x<0>, (const void *)k_box_x<1>, (const void *)k_box_x<2>};
    const int r[3] = {4, 8, 16};
    for (int k = 0; k < 3; ++k) {
        const cudaError_t e =
            cudaFuncSetAttribute(fn[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)box_x_smem(r[k]));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void launch_box_passes(const BatchHdr *d, const LaunchPlan &p, cudaStream_t s) {
    if (p.denoise & 1u) launch_class<0>(d, p, s);
    if (p.denoise & 2u) launch_class<1>(d, p, s);
    if (p.denoise & 4u) launch_class<2>(d, p, s);
}

}  // namespace seg
