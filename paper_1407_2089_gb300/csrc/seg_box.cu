// seg_box.cu -- the background of the denoise front end (Background Noise
// Removal, Eq. 1): three rounded box passes of radius r along x, then y, then
// z, each pass with replicate edges.
//
// Two forms, chosen per axis (box_rings()).  In register rings one thread
// follows one line (or a chunk of one) and runs all three passes at
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
// Bound by the latency of its loads along x and y (IPC 1.8 and 1.9 of 4,
// long scoreboard first), between that and instruction issue along z (2.3).  4 volumes
// of 512 x 512 x 64, r = 8: x 238 -> 223, y 153 -> 101, z 214 -> 147 us against the
// other form, three passes through shared memory with a barrier each (k_box3),
// which is the faster one for small batches and large radii.  Chunks of 256
// positions along x (two blocks fewer resident) take 330 us there.
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
        if (box_class(V.dn_r) != CLS || !(V.dn_ring >> AXIS & 1u)) continue;
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
        if (box_class(V.dn_r) != CLS || !(V.dn_ring & 1u)) continue;
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

// The same passes through shared memory, for small batches and large radii
// (box_rings()): an item is 64 lines x a chunk of at most BOX_CHUNK positions,
// loaded with a halo of 3r positions on each side; pass k runs over the
// positions the next one needs, four threads per line, each reading its input at
// positions clamped to the line, which is the replicate edge of every pass.
// Four times the threads per voxel of the register rings, and registers that do
// not grow with r.  Shared layout [position][lane], lanes padded to 66 so that
// both the lane-major passes and the position-major copies of axis x avoid bank
// conflicts.
constexpr int BOX_THREADS = 256, BOX_CHUNK = 128;
constexpr int BOX_LANES = 64, BOX_PITCH = BOX_LANES + 2;
constexpr int BOX_POS = BOX_CHUNK + 6 * DN_MAX_R;
constexpr size_t BOX_SMEM = 2ull * BOX_POS * BOX_PITCH * sizeof(uint16_t);

template <int AXIS>
__global__ void __launch_bounds__(BOX_THREADS) k_box3(const BatchHdr *__restrict__ h) {
    extern __shared__ __align__(16) uint16_t bsm[];
    uint16_t *bufA = bsm, *bufB = bsm + BOX_POS * BOX_PITCH;
    const int t = threadIdx.x;
    for (uint32_t it = blockIdx.x; it < h->dn_items[AXIS]; it += gridDim.x) {
        const VolDev &V = h->vol[box_volume<AXIS>(h, it)];
        if (V.dn_ring >> AXIS & 1u) continue;
        const uint32_t li = it - box_base<AXIS>(V), X = V.X;
        const uint32_t len = AXIS == 0 ? X : (AXIS == 1 ? V.Y : V.Z), nchunk = box_chunks(len, BOX_CHUNK);
        const uint32_t group = li / nchunk;
        const int r = (int)V.dn_r;
        const uint32_t mul = V.dn_mul;
        const BoxChunk c = box_chunk(len, BOX_CHUNK, li % nchunk, V.dn_r);
        const int n = c.n, c0 = c.c0, c1 = c.c1;
        if (c0 >= c1) continue;  // (the same in every thread)
        const int base = c0 - 3 * r, lo = 0, hi = min(c1 + 3 * r, n);  // loaded: [lo, hi)
        // lane l of this group: its line's position 0 and the step along it
        int nl;            // lanes of this group that exist
        size_t gstart;     // element of lane 0 at position 0
        size_t lstride, pstride;
        if (AXIS == 0) {
            nl = (int)min((uint32_t)BOX_LANES, V.rows - group * BOX_LANES);
            gstart = (size_t)group * BOX_LANES * X;
            lstride = X;
            pstride = 1;
        } else {
            const uint32_t nxg = (X + BOX_LANES - 1) / BOX_LANES, gx = group % nxg, other = group / nxg;
            nl = (int)min((uint32_t)BOX_LANES, X - gx * BOX_LANES);
            lstride = 1;
            if (AXIS == 1) {
                gstart = (size_t)gx * BOX_LANES + (size_t)X * V.Y * other;
                pstride = X;
            } else {
                gstart = (size_t)gx * BOX_LANES + (size_t)X * other;
                pstride = (size_t)X * V.Y;
            }
        }
        gstart += c.first * pstride;
        const uint16_t *src = AXIS == 0 ? V.dn_src : (AXIS == 1 ? V.dn_a : V.dn_b);
        uint16_t *dst = AXIS == 1 ? V.dn_b : V.dn_a;
        const int np = hi - lo;
        __syncthreads();  // the previous item is done with the buffers
        // load: consecutive threads on consecutive elements in memory, eight
        // independent loads in flight per thread before the shared stores
        constexpr int NB = 8;
        if (AXIS == 0) {
            // one warp per line (a row segment), lanes along it
            const int lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
            for (int l = warp; l < nl; l += nw) {
                const uint16_t *row = src + gstart + (size_t)l * lstride;
                for (int q0 = lo + lane; q0 < hi; q0 += 32 * NB) {
                    uint16_t v[NB];
#pragma unroll
                    for (int j = 0; j < NB; ++j)
                        if (q0 + 32 * j < hi) v[j] = row[q0 + 32 * j];
#pragma unroll
                    for (int j = 0; j < NB; ++j)
                        if (q0 + 32 * j < hi) bufA[(q0 + 32 * j - base) * BOX_PITCH + l] = v[j];
                }
            }
        } else if ((X & 7u) == 0u) {
            // rows of 8-voxel octets (X % 8 == 0, scratch buffers 16-byte
            // aligned): thread t moves lanes 8 (t % 8) .. + 7 of positions
            // t / 8 + 32 i as one 16-byte load and four 4-byte shared stores
            // (pitch 66: the 32 threads of a warp hit 32 different banks)
            const int oct = t & 7, pr = t >> 3;
            constexpr int NV = 4;
            if (8 * oct < nl) {
                const uint16_t *col = src + gstart + 8 * oct;
                for (int q0 = lo + pr; q0 < hi; q0 += 32 * NV) {
                    uint4 v[NV];
#pragma unroll
                    for (int j = 0; j < NV; ++j)
                        if (q0 + 32 * j < hi)
                            v[j] = *reinterpret_cast<const uint4 *>(col + (size_t)(q0 + 32 * j) * pstride);
#pragma unroll
                    for (int j = 0; j < NV; ++j)
                        if (q0 + 32 * j < hi) {
                            uint32_t *w = reinterpret_cast<uint32_t *>(bufA + (q0 + 32 * j - base) * BOX_PITCH + 8 * oct);
                            w[0] = v[j].x; w[1] = v[j].y; w[2] = v[j].z; w[3] = v[j].w;
                        }
                }
            }
        } else {
            const int total = np * BOX_LANES, nt = blockDim.x;
            for (int i0 = t; i0 < total; i0 += nt * NB) {
                uint16_t v[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const int i = i0 + j * nt, l = i % BOX_LANES, q = lo + i / BOX_LANES;
                    if (i < total && l < nl) v[j] = src[gstart + (size_t)l * lstride + (size_t)q * pstride];
                }
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const int i = i0 + j * nt, l = i % BOX_LANES, q = lo + i / BOX_LANES;
                    if (i < total && l < nl) bufA[(q - base) * BOX_PITCH + l] = v[j];
                }
            }
        }
        __syncthreads();
        // three passes: A -> B over [c0-2r, c1+2r), B -> A over [c0-r, c1+r), A -> B over [c0, c1)
        const int l = t % BOX_LANES, seg = t / BOX_LANES;
        for (int k = 0; k < 3; ++k) {
            const uint16_t *in = (k == 1) ? bufB : bufA;
            uint16_t *out = (k == 1) ? bufA : bufB;
            const int p0 = max(c0 - (2 - k) * r, 0), p1 = min(c1 + (2 - k) * r, n);
            const int per = (p1 - p0 + 3) / 4;
            const int q0 = p0 + seg * per, q1 = min(q0 + per, p1);
            if (l < nl && q0 < q1) {
                // every read lies in [q0 - r, q1 - 1 + r] clamped to the line,
                // inside the positions the previous pass (or the load) covered
                auto at = [&](int q) { return (uint32_t)in[(min(max(q, 0), n - 1) - base) * BOX_PITCH + l]; };
                // sum holds the window sum plus the rounding term r
                uint32_t sum = (uint32_t)r;
                if (q0 - r >= 0 && q0 + r < n) {
                    const uint16_t *pw = in + (q0 - r - base) * BOX_PITCH + l;
                    for (int i = 0; i <= 2 * r; ++i) sum += pw[i * BOX_PITCH];
                } else {
                    for (int q = q0 - r; q <= q0 + r; ++q) sum += at(q);
                }
                out[(q0 - base) * BOX_PITCH + l] = (uint16_t)box_div(sum, mul);
                // positions q whose window [q - r - 1, q + r] needs no
                // clamping run through three moving pointers
                const int qa = min(max(q0 + 1, r + 1), q1), qb = max(min(q1, n - r), qa);
                int q = q0 + 1;
                for (; q < qa; ++q) {
                    sum += at(q + r) - at(q - r - 1);
                    out[(q - base) * BOX_PITCH + l] = (uint16_t)box_div(sum, mul);
                }
                const uint16_t *pin = in + (q + r - base) * BOX_PITCH + l;
                const uint16_t *pout = in + (q - r - 1 - base) * BOX_PITCH + l;
                uint16_t *po = out + (q - base) * BOX_PITCH + l;
#pragma unroll 4
                for (; q < qb; ++q) {
                    sum += (uint32_t)*pin - (uint32_t)*pout;
                    *po = (uint16_t)box_div(sum, mul);
                    pin += BOX_PITCH;
                    pout += BOX_PITCH;
                    po += BOX_PITCH;
                }
                for (; q < q1; ++q) {
                    sum += at(q + r) - at(q - r - 1);
                    out[(q - base) * BOX_PITCH + l] = (uint16_t)box_div(sum, mul);
                }
            }
            __syncthreads();
        }
        // store the chunk from B
        const int nc = c1 - c0;
        if (AXIS == 0) {
            const int lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
            for (int ll = warp; ll < nl; ll += nw) {
                uint16_t *row = dst + gstart + (size_t)ll * lstride;
                for (int q = c0 + lane; q < c1; q += 32) row[q] = bufB[(q - base) * BOX_PITCH + ll];
            }
        } else if ((X & 7u) == 0u) {
            const int oct = t & 7, pr = t >> 3;
            if (8 * oct < nl) {
                uint16_t *col = dst + gstart + 8 * oct;
                for (int q = c0 + pr; q < c1; q += 32) {
                    const uint32_t *w = reinterpret_cast<const uint32_t *>(bufB + (q - base) * BOX_PITCH + 8 * oct);
                    *reinterpret_cast<uint4 *>(col + (size_t)q * pstride) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        } else {
            for (int i = t; i < nc * BOX_LANES; i += blockDim.x) {
                const int ll = i % BOX_LANES, q = c0 + i / BOX_LANES;
                if (ll < nl) dst[gstart + (size_t)ll * lstride + (size_t)q * pstride] = bufB[(q - base) * BOX_PITCH + ll];
            }
        }
    }
}

}  // namespace

uint64_t box_items(int axis, bool ring, uint32_t X, uint32_t Y, uint32_t Z) {
    const uint32_t n = axis == 0 ? X : (axis == 1 ? Y : Z);
    if (ring) {
        const uint64_t lines = axis == 0 ? (uint64_t)Y * Z : (uint64_t)X * (axis == 1 ? Z : Y);
        return (lines + BX_THREADS - 1) / BX_THREADS * box_chunks(n, axis == 0 ? DN_CHUNK_X : DN_CHUNK);
    }
    const uint64_t groups = axis == 0 ? ((uint64_t)Y * Z + BOX_LANES - 1) / BOX_LANES
                                      : (uint64_t)((X + BOX_LANES - 1) / BOX_LANES) * (axis == 1 ? Z : Y);
    return groups * box_chunks(n, BOX_CHUNK);
}

// Where the rings are the faster ones, from both timed per axis for radii 1..16
// on 40 batches (64 x 64 x 12 to 2000 x 2000 x 16).  They need enough lines (a
// thread each; 128 x 128 x 32 at r = 8: 17.2 us along x and 8.1 along y, 10.2 and
// 6.7 through shared memory), registers for the windows (above r = 8 two or three
// blocks are resident: 512 x 512 x 64 at r = 12, x 130 against 68 us) and are
// worth most where the shared copies of lines across rows are narrow (X % 8 != 0)
// or the halo is long against the line (small Z):
//   x: up to r = 8, for rows of one chunk (64 x 64 x 2000: 36 against 47 us) and
//      large batches of whole chunks or small radii (four 512 x 512 x 64 volumes,
//      r = 8: 223 against 238; not 700 x 700 x 80 at r = 8: 178 against 152);
//   y: whole octets from r = 3 (few loads in flight below: r = 1 takes 1.3 times
//      the time) to 8 (four 512 x 512 x 64 volumes: 101 against 153); ragged rows
//      at any radius (511 x 511 x 64, r = 12: 39 against 70);
//   z: up to r = 8 (147 against 214), above it for ragged rows and few planes
//      (512 x 512 x 12, r = 10: 26 against 38; not 512 x 512 x 64 at r = 16: 81
//      against 63).
uint32_t box_rings(uint32_t X, uint32_t Z, uint32_t r, const uint64_t *items, int sms) {
    const double S = (double)sms, x = (double)items[0] / S, y = (double)items[1] / S, z = (double)items[2] / S;
    const bool octets = X % 8u == 0u;
    uint32_t m = 0;
    if (r <= 8u && (X <= 64u ? x >= 3.0 : (r <= 4u || X % 128u == 0u) && x >= 16.0)) m |= 1u;
    if (octets ? r >= 2u && r <= 8u && y >= (r == 2u ? 3.0 : 2.5) : y >= (r == 1u ? 2.5 : (r == 2u ? 1.25 : 0.75))) m |= 2u;
    if (z >= 2.0 && (r <= 8u || !octets || (r <= 12u && Z <= 32u))) m |= 4u;
    return m;
}

cudaError_t configure_box(LaunchPlan &plan) {
    const void *fn[5] = {(const void *)k_box_x<0>, (const void *)k_box_x<1>, (const void *)k_box3<0>,
                         (const void *)k_box3<1>, (const void *)k_box3<2>};
    const size_t smem[5] = {box_x_smem(4), box_x_smem(8), BOX_SMEM, BOX_SMEM, BOX_SMEM};
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 5 && e == cudaSuccess; ++k)
        e = cudaFuncSetAttribute(fn[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem[k]);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_box3<1>, BOX_THREADS, BOX_SMEM)) != cudaSuccess)
        return e;
    plan.grid_box3 = plan.sms * (per_sm > 0 ? per_sm : 1);
    plan.grid_box = 16 * plan.sms;  // every ring kernel's resident blocks, at most
    return cudaSuccess;
}

void launch_box_passes(const BatchHdr *d, const LaunchPlan &p, cudaStream_t s) {
    auto on = [&](int axis, int route) { return (p.denoise >> box_route_bit(axis, route) & 1u) != 0u; };
    if (on(0, 0)) k_box_x<0><<<p.grid_box, BX_THREADS, box_x_smem(4), s>>>(d);
    if (on(0, 1)) k_box_x<1><<<p.grid_box, BX_THREADS, box_x_smem(8), s>>>(d);
    if (on(0, 3)) k_box3<0><<<p.grid_box3, BOX_THREADS, BOX_SMEM, s>>>(d);
    if (on(1, 0)) k_box_lines<1, 0><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    if (on(1, 1)) k_box_lines<1, 1><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    if (on(1, 2)) k_box_lines<1, 2><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    if (on(1, 3)) k_box3<1><<<p.grid_box3, BOX_THREADS, BOX_SMEM, s>>>(d);
    if (on(2, 0)) k_box_lines<2, 0><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    if (on(2, 1)) k_box_lines<2, 1><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    if (on(2, 2)) k_box_lines<2, 2><<<p.grid_box, BX_THREADS, 0, s>>>(d);
    if (on(2, 3)) k_box3<2><<<p.grid_box3, BOX_THREADS, BOX_SMEM, s>>>(d);
}

}  // namespace seg
