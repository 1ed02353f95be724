// seg_montage.cu -- montage registration (Registration section, Eq. 4):
// overlapping tiles are scored at every shift of a search window by the
// normalized covariance of their shared voxels, each overlapping pair keeps
// its best shift, and a maximum spanning tree of the pairs gives every tile
// its correction relative to an anchored one.
//
// Per pair and shift s the score needs six exact integer sums over the
// shared box: N, Sa, Sb, Saa, Sbb and Sab.  The GPU computes
//   * Sab for all shifts at once (k_reg_corr): a block stages a sub-box of
//     tile a and the matching region of tile b widened by the window (b
//     zero outside its box, so no bounds test per product), and each thread
//     takes shifts, summing the products over the sub-box from shared
//     memory;
//   * Sa, Saa (tile a) and Sb, Sbb (tile b) from the sums of every plane over
//     each shift's x- and y-range (k_reg_plane), because the shared box varies
//     only at its faces, then per shift a sum over the planes of its box
//     (k_reg_box).
// Every kernel takes all pairs of a group in one launch.
// The host then forms the Pearson correlation in 128-bit integers and
// binary64, picks the first best shift in z, y, x order, builds the maximum
// spanning tree (Kruskal) and sums the shifts from the root.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <numeric>
#include <utility>
#include <vector>

#include "seg.h"

namespace {

constexpr int RC_TX = 32, RC_TY = 16, RC_TZ = 16;  // tile-a sub-box of a k_reg_corr block
constexpr int RC_THREADS = 256;
static_assert(RC_TY >= RC_THREADS / 32 && RC_TX == 32, "staging by row per warp");
// row pitch of the staged tile-b region: an odd number of 32-bit words, so that
// lanes on consecutive rows read distinct banks
__host__ __device__ constexpr int rc_pitch(int rx) { return 2 * (((RC_TX + 2 * rx + 1) / 2) | 1); }

// Half-open range [lo, hi) of one axis.
struct Range {
    int lo, hi;
};

// Shared range along one axis for tile b's origin at d in tile a's frame:
// in a's coordinates (side 0) or in b's (side 1).  d + D and D - d are only
// formed where they are at most D, so that no tile extent overflows them.
__host__ __device__ inline Range shared_range(int d, int D, int side) {
    if (side == 0) return Range{d > 0 ? d : 0, d < 0 ? d + D : D};
    return Range{d < 0 ? -d : 0, d > 0 ? D - d : D};
}

// One overlapping pair on the device: tile b's origin in tile a's frame, the
// search region of each side (0: a, 1: b) in that tile's frame.
struct RegPair {
    const uint16_t *tile[2];
    int3 d0;
    int3 u0[2], u1[2];
};

// Sab for every shift: block (x, y) = sub-box x (RC_TX x RC_TY x RC_TZ) of the
// search region U of tile a of pair y (in a's coordinates).  Shift index
// si = ((sz + rz) SY + (sy + ry)) SX + (sx + rx).  Thread (g, c) takes the
// (y, z)-shift g = (sy, sz) for every x-shift (KX = 2 RX + 1 of them) over
// the sub-box rows c, c + C, ...: along a row the x-shifts need b values
// x + 2 RX - k, so a register window of KX b values slides with x and every
// product costs one multiply-add.  Products are added in 32 bits over as many
// rows as the sub-box's largest values allow (32 rows at 2000 x 2000), then
// moved to 64-bit sums; only where one row could overflow are the sums 64-bit
// throughout (three instructions per product instead of one).  Bound by
// instruction issue (one multiply-add per product, a third more for staging
// and unpacking): 1.83 ms for the 20.5 G products of 3 x 3 tiles of 1024 x 1024
// x 64 with a tenth of overlap and radius 4, 4, 1, where 64-bit sums over 8 x 8
// rows took 3.2 ms; 8 x 16 rows take 2.1 ms.  Wider windows stage more per block
// (75 KB at radius 6, 6, 2, 211 KB at 12, 12, 6) and gain less: whole calls of 2 x
// 2 tiles of 1024 x 1024 x 64 at 6, 6, 2 take 2.81 ms against 3.48, of two tiles of
// 1024 x 1024 x 32 at 12, 12, 6 3.31 against 3.85.  The threads' sums meet in
// shared memory and go out with one atomic per (block, shift).
template <int RX>
__global__ void __launch_bounds__(RC_THREADS) k_reg_corr(const RegPair *__restrict__ pairs, int X, int Y, int Z, int ry,
                                                         int rz, unsigned long long *__restrict__ sums, size_t per) {
    constexpr int KX = 2 * RX + 1;
    constexpr int BX = RC_TX + 2 * RX, BP = rc_pitch(RX);
    extern __shared__ __align__(16) unsigned long long rsm64[];
    __shared__ uint32_t smax[2];
    const RegPair &P = pairs[blockIdx.y];
    const uint16_t *__restrict__ A = P.tile[0], *__restrict__ B = P.tile[1];
    const int3 u0 = P.u0[0], u1 = P.u1[0], d0 = P.d0;
    unsigned long long *sab = sums + per * blockIdx.y;
    const int BY = RC_TY + 2 * ry, SY = 2 * ry + 1, G = SY * (2 * rz + 1);
    unsigned long long *red = rsm64;                                      // [G][KX]
    uint16_t *As = reinterpret_cast<uint16_t *>(rsm64 + ((size_t)G * KX + 1) / 2 * 2);  // [RC_TZ][RC_TY][RC_TX]
    uint16_t *Bs = As + RC_TX * RC_TY * RC_TZ;                            // [BZ][BY][BP]
    if (u1.x <= u0.x || u1.y <= u0.y || u1.z <= u0.z) return;
    const int nbx = (u1.x - u0.x + RC_TX - 1) / RC_TX, nby = (u1.y - u0.y + RC_TY - 1) / RC_TY;
    const int nbz = (u1.z - u0.z + RC_TZ - 1) / RC_TZ;
    const int bi = (int)blockIdx.x;
    if ((long long)bi >= (long long)nbx * nby * nbz) return;
    const int ax0 = u0.x + (bi % nbx) * RC_TX, ay0 = u0.y + ((bi / nbx) % nby) * RC_TY;
    const int az0 = u0.z + (bi / (nbx * nby)) * RC_TZ;
    // a sub-box at the region's end (all of them, for flat tiles) has fewer
    // planes (3 x 3 tiles of 1024 x 1024 x 4: 0.64 ms for the call, 0.99 with the
    // missing ones multiplied as zeros)
    const int TZ = min(RC_TZ, u1.z - az0), ROWS = RC_TY * TZ, BZ = TZ + 2 * rz;
    if (threadIdx.x < 2) smax[threadIdx.x] = 0u;
    for (int i = threadIdx.x; i < G * KX; i += RC_THREADS) red[i] = 0ull;
    __syncthreads();
    // a row per warp, four rows' loads in flight
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int WARPS = RC_THREADS / 32, RB = 4;
    uint32_t ma = 0, mb = 0;
    for (int r0 = warp; r0 < ROWS; r0 += WARPS * RB) {
        uint32_t v[RB];
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int row = r0 + k * WARPS, x = ax0 + lane, y = ay0 + row % RC_TY, z = az0 + row / RC_TY;
            v[k] = row < ROWS && x < u1.x && y < u1.y && z < u1.z ? A[((size_t)z * Y + y) * X + x] : 0u;
        }
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int row = r0 + k * WARPS;
            if (row < ROWS) As[row * RC_TX + lane] = (uint16_t)v[k];
            ma = max(ma, v[k]);
        }
    }
    // b coordinates of a's sub-box under every shift: a - d0 - s
    const int bx0 = ax0 - d0.x - RX, by0 = ay0 - d0.y - ry, bz0 = az0 - d0.z - rz;
    const int xa = bx0 + lane, xb = xa + 32;  // (BX <= 56)
    const bool ina = xa >= 0 && xa < X, inb = xb >= 0 && xb < X && lane + 32 < BX;
    // row = warp, warp + WARPS, ... as (ty, tz), stepped without divisions (BY >= WARPS)
    int ty = warp, tz = 0;
    for (int r0 = warp; r0 < BY * BZ; r0 += WARPS * RB) {
        uint32_t v[RB], w[RB];
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int y = by0 + ty, z = bz0 + tz;
            const bool in = tz < BZ && y >= 0 && y < Y && z >= 0 && z < Z;
            const uint16_t *b = B + (in ? ((size_t)z * Y + y) * X : 0);
            v[k] = in && ina ? b[xa] : 0u;
            w[k] = in && inb ? b[xb] : 0u;
            ty += WARPS;
            if (ty >= BY) {
                ty -= BY;
                ++tz;
            }
        }
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int row = r0 + k * WARPS;
            if (row < BY * BZ) {
                Bs[row * BP + lane] = (uint16_t)v[k];
                if (lane + 32 < BX) Bs[row * BP + lane + 32] = (uint16_t)w[k];
            }
            mb = max(mb, max(v[k], w[k]));
        }
    }
    ma = __reduce_max_sync(0xFFFFFFFFu, ma);
    mb = __reduce_max_sync(0xFFFFFFFFu, mb);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&smax[0], ma);
        atomicMax(&smax[1], mb);
    }
    __syncthreads();
    const int C = G >= RC_THREADS ? 1 : min(ROWS, RC_THREADS / G);  // row chunks per shift group
    // rows whose products sum to less than 2^32: each of the RC_TX products
    // is at most smax[0] smax[1] (< 2^32)
    const uint32_t most = smax[0] * smax[1];
    const int fit = most ? (int)min(0xFFFFFFFFu / most / RC_TX, (uint32_t)ROWS) : ROWS;
    // one row: acc[k] += a(x) b(x + 2 RX - k) over x
    auto add_row = [&](int row, int sy, int sz, auto &acc) {
        const int y = row % RC_TY, z = row / RC_TY;
        const uint4 *ar = reinterpret_cast<const uint4 *>(As + row * RC_TX);
        const uint32_t *br = reinterpret_cast<const uint32_t *>(Bs + ((z - sz + rz) * BY + (y - sy + ry)) * BP);
        uint32_t win[KX + 1];  // b at x .. x + 2 RX (+ 1): win[(x + j) % (KX + 1)] holds b(x + j)
#pragma unroll
        for (int j = 0; j < RX; ++j) {
            const uint32_t w = br[j];
            win[2 * j] = w & 0xFFFFu;
            win[2 * j + 1] = w >> 16;
        }
#pragma unroll
        for (int x0 = 0; x0 < RC_TX; x0 += 8) {
            const uint4 a4 = ar[x0 / 8];
            const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int x = x0 + 2 * h;
                const uint32_t w = br[RX + x / 2];  // b at x + 2 RX, x + 2 RX + 1
                win[(x + 2 * RX) % (KX + 1)] = w & 0xFFFFu;
                win[(x + 2 * RX + 1) % (KX + 1)] = w >> 16;
                const uint32_t al = aw[h] & 0xFFFFu, ah = aw[h] >> 16;
#pragma unroll
                for (int k = 0; k < KX; ++k) acc[k] += al * win[(x + 2 * RX - k) % (KX + 1)];
#pragma unroll
                for (int k = 0; k < KX; ++k) acc[k] += ah * win[(x + 1 + 2 * RX - k) % (KX + 1)];
            }
        }
    };
    for (int w = threadIdx.x; w < G * C; w += RC_THREADS) {
        const int g = w % G, c = w / G;
        const int sy = g % SY - ry, sz = g / SY - rz;
        unsigned long long acc[KX];
#pragma unroll
        for (int k = 0; k < KX; ++k) acc[k] = 0ull;
        if (fit > 0) {
            for (int row = c; row < ROWS;) {
                uint32_t part[KX];
#pragma unroll
                for (int k = 0; k < KX; ++k) part[k] = 0u;
                for (int n = 0; n < fit && row < ROWS; ++n, row += C) add_row(row, sy, sz, part);
#pragma unroll
                for (int k = 0; k < KX; ++k) acc[k] += part[k];
            }
        } else {
            for (int row = c; row < ROWS; row += C) add_row(row, sy, sz, acc);
        }
#pragma unroll
        for (int k = 0; k < KX; ++k)
            if (acc[k]) atomicAdd(red + g * KX + k, acc[k]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G * KX; i += RC_THREADS)
        if (red[i]) atomicAdd(sab + i, red[i]);
}

// Shared memory of k_reg_corr<RX>.
size_t reg_corr_smem(int rx, int ry, int rz) {
    const size_t G = (size_t)(2 * ry + 1) * (2 * rz + 1), KX = 2 * rx + 1;
    return 16 * ((G * KX + 1) / 2) + 2 * ((size_t)RC_TX * RC_TY * RC_TZ +
                             (size_t)rc_pitch(rx) * (RC_TY + 2 * ry) * (RC_TZ + 2 * rz));
}

using RegCorrFn = void (*)(const RegPair *, int, int, int, int, int, unsigned long long *, size_t);
template <int... R>
RegCorrFn reg_corr_fn(int rx, std::integer_sequence<int, R...>) {
    RegCorrFn f = nullptr;
    ((rx == R ? (f = k_reg_corr<R>, 0) : 0), ...);
    return f;
}

// Sums of v and v^2 over one slab of rows of one plane of a side's region U for
// every x-range (one per x-shift) and y-range (one per y-shift): p1, p2[(slab SY
// + syi) SX + sxi] of the side's `per` slabs.  Block (slab, 2 pair + side); a
// plane is `ns` consecutive slabs, one unless the planes are too few to fill the
// GPU (two tiles of 4096 x 4096 x 1 with a tenth of overlap: the call takes 186
// us, 715 with a block per plane), and planes start at z0.  Ranges move monotonically with the shift:
// all of them share a core [clo, chi) in x and in y, and outside it lie at most
// 2 rx columns on either side.  The rows of the y-core add up in registers, the
// x-core per lane and the outer columns one per lane, and are reduced once per
// plane; only the at most 4 ry rows outside the y-core are reduced row by row
// and added to the y-ranges that hold them.  Where the ranges share no core in
// x the region is at most 2 rx columns wide (the overlap or the tile is
// narrower than the window), and all of them count as left outer ones.  Bound
// by reading the plane.
constexpr int RP_THREADS = 256, RP_SY = 2 * SEG_REG_MAX_RXY + 1;
constexpr int RP_COLS = 64;  // outer columns: 32 left, 32 right (2 rx <= 24 used)

__global__ void __launch_bounds__(RP_THREADS) k_reg_plane(const RegPair *__restrict__ pairs, int X, int Y, int3 r,
                                                          int z0, int ns, size_t per,
                                                          unsigned long long *__restrict__ p1,
                                                          unsigned long long *__restrict__ p2) {
    // sums of v and v^2: entry SY holds the y-core, entry syi the other rows
    // of y-range syi; the x-core, and each outer column
    __shared__ unsigned long long xc[2][RP_SY + 1], col[2][RP_SY + 1][RP_COLS];
    const RegPair &P = pairs[blockIdx.y >> 1];
    const int side = blockIdx.y & 1;
    const int3 u0 = P.u0[side], u1 = P.u1[side], d0 = P.d0;
    const int z = u0.z + z0 + (int)blockIdx.x / ns;
    if (u1.x <= u0.x || u1.y <= u0.y || z >= u1.z) return;
    const int uy = u1.y - u0.y, sh = (uy + ns - 1) / ns;  // this block's rows: [ya, yb)
    const int ya = u0.y + min((int)blockIdx.x % ns * sh, uy), yb = min(ya + sh, u1.y);
    const int SX = 2 * r.x + 1, SY = 2 * r.y + 1;
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 2 * (RP_SY + 1); i += RP_THREADS) (&xc[0][0])[i] = 0ull;
    for (int i = threadIdx.x; i < 2 * (RP_SY + 1) * RP_COLS; i += RP_THREADS) (&col[0][0][0])[i] = 0ull;
    const Range xf = shared_range(d0.x - r.x, X, side), xl = shared_range(d0.x + r.x, X, side);
    const Range yf = shared_range(d0.y - r.y, Y, side), yl = shared_range(d0.y + r.y, Y, side);
    int clo = max(xf.lo, xl.lo), chi = min(xf.hi, xl.hi);
    const int ylo = max(yf.lo, yl.lo), yhi = min(yf.hi, yl.hi);
    if (clo >= chi) clo = chi = u1.x;  // no core: at most 2 rx columns, all left ones
    // this lane's outer columns: u0.x + lane before clo, and chi + lane
    const int xa = u0.x + lane, xr = chi + lane;
    __syncthreads();
    const uint16_t *plane = P.tile[side] + (size_t)z * X * Y;
    unsigned long long a1 = 0, a2 = 0, l1 = 0, l2 = 0, h1 = 0, h2 = 0;  // y-core
    constexpr int WARPS = RP_THREADS / 32, RB = 4;
    const int warp = threadIdx.x >> 5;
    // the y-core, RB rows' loads in flight
    const int ye = min(yhi, yb);
    for (int y0 = max(ylo, ya) + warp; y0 < ye; y0 += WARPS * RB) {
        const uint16_t *t[RB];
        bool on[RB];
        uint32_t va[RB], vr[RB];
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int y = y0 + k * WARPS;
            on[k] = y < ye;
            t[k] = plane + (size_t)(on[k] ? y : y0) * X;
            va[k] = on[k] && xa < clo ? t[k][xa] : 0u;
            vr[k] = on[k] && xr < u1.x ? t[k][xr] : 0u;
        }
        for (int x = clo + lane; x < chi; x += 32) {
            uint32_t v[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) v[k] = on[k] ? t[k][x] : 0u;
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                a1 += v[k];
                a2 += v[k] * v[k];
            }
        }
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            l1 += va[k];
            l2 += va[k] * va[k];
            h1 += vr[k];
            h2 += vr[k] * vr[k];
        }
    }
    // the rows outside it
    const int before = max(min(ylo, yb) - ya, 0), start = max(yhi, ya + before);
    for (int i = warp; i < before + max(yb - start, 0); i += WARPS) {
        const int y = i < before ? ya + i : start + (i - before);
        const uint16_t *t = plane + (size_t)y * X;
        const uint32_t va = xa < clo ? t[xa] : 0u, vr = xr < u1.x ? t[xr] : 0u;
        unsigned long long s1 = 0, s2 = 0;
        for (int x = clo + lane; x < chi; x += 32) {
            const uint32_t v = t[x];
            s1 += v;
            s2 += v * v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
            s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
        }
        for (int sy = 0; sy < SY; ++sy) {
            const Range w = shared_range(d0.y + sy - r.y, Y, side);
            if (y < w.lo || y >= w.hi) continue;
            if (lane == 0) {
                atomicAdd(&xc[0][sy], s1);
                atomicAdd(&xc[1][sy], s2);
            }
            if (xa < clo) {
                atomicAdd(&col[0][sy][lane], (unsigned long long)va);
                atomicAdd(&col[1][sy][lane], (unsigned long long)(va * va));
            }
            if (xr < u1.x) {
                atomicAdd(&col[0][sy][32 + lane], (unsigned long long)vr);
                atomicAdd(&col[1][sy][32 + lane], (unsigned long long)(vr * vr));
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a1 += __shfl_xor_sync(0xFFFFFFFFu, a1, o);
        a2 += __shfl_xor_sync(0xFFFFFFFFu, a2, o);
    }
    if (lane == 0) {
        atomicAdd(&xc[0][SY], a1);
        atomicAdd(&xc[1][SY], a2);
    }
    atomicAdd(&col[0][SY][lane], l1);
    atomicAdd(&col[1][SY][lane], l2);
    atomicAdd(&col[0][SY][32 + lane], h1);
    atomicAdd(&col[1][SY][32 + lane], h2);
    __syncthreads();
    const size_t o = per * blockIdx.y + (size_t)blockIdx.x * SY * SX;
    for (int i = threadIdx.x; i < SY * SX; i += RP_THREADS) {
        const int sy = i / SX;
        const Range wx = shared_range(d0.x + i % SX - r.x, X, side), wy = shared_range(d0.y + sy - r.y, Y, side);
        unsigned long long s[2] = {0ull, 0ull};
        if (wx.lo < wx.hi && wy.lo < wy.hi) {
            for (int k = 0; k < 2; ++k) {
                s[k] = xc[k][sy] + xc[k][SY];
                for (int x = wx.lo; x < min(clo, wx.hi); ++x) s[k] += col[k][sy][x - u0.x] + col[k][SY][x - u0.x];
                for (int x = chi; x < wx.hi; ++x) s[k] += col[k][sy][32 + x - chi] + col[k][SY][32 + x - chi];
            }
        }
        p1[o + i] = s[0];
        p2[o + i] = s[1];
    }
}

// Per shift: the sums of v and v^2 over a side's shared box, one thread per
// shift adding the slabs of BOX_SLABS / ns planes from z0 on; block (shifts,
// 2 pair + side, planes).  With all planes in one thread deep tiles waited for
// it (two tiles of 16 x 16 x 20000: 5.7 ms for the call, now 0.92).
constexpr int BOX_SLABS = 64;

__global__ void k_reg_box(const RegPair *__restrict__ pairs, const unsigned long long *__restrict__ p1,
                          const unsigned long long *__restrict__ p2, int X, int Y, int Z, int3 r, int z0, int z1,
                          int ns, size_t pper, unsigned long long *__restrict__ sums, size_t per) {
    const RegPair &P = pairs[blockIdx.y >> 1];
    const int side = blockIdx.y & 1;
    const int3 u0 = P.u0[side], u1 = P.u1[side], d0 = P.d0;
    const int SX = 2 * r.x + 1, SY = 2 * r.y + 1, S = SX * SY * (2 * r.z + 1);
    const int si = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (si >= S || u1.x <= u0.x || u1.y <= u0.y) return;
    const Range zr = shared_range(d0.z + si / (SX * SY) - r.z, Z, side);
    const int nz = max(BOX_SLABS / ns, 1), za = z0 + (int)blockIdx.z * nz;  // planes from u0.z on
    const int lo = max(zr.lo - u0.z, za), hi = min(zr.hi - u0.z, min(za + nz, z1));
    if (lo >= hi) return;
    unsigned long long a = 0, b = 0;
    const size_t at = pper * blockIdx.y + si % (SX * SY);
    for (int q = (lo - z0) * ns; q < (hi - z0) * ns; ++q) {
        const size_t i = at + (size_t)q * SY * SX;
        a += p1[i];
        b += p2[i];
    }
    unsigned long long *o = sums + per * (blockIdx.y >> 1) + (size_t)(1 + 2 * side) * S;
    if (a) atomicAdd(o + si, a);
    if (b) atomicAdd(o + S + si, b);
}

int fail(cudaError_t e) {
    if (e == cudaSuccess) return SEG_OK;
    cudaGetLastError();
    return SEG_ECUDA;
}

#define RK(call)                                 \
    do {                                         \
        const cudaError_t e__ = (call);          \
        if (e__ != cudaSuccess) return fail(e__); \
    } while (0)

// Device scratch of one call, from the stream-ordered pool on its stream s,
// freed on every return path.
struct Scratch {
    std::vector<void *> ptrs;
    cudaStream_t s = nullptr;
    ~Scratch() {
        for (void *p : ptrs) cudaFreeAsync(p, s);
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
    }
    cudaError_t init() { return cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking); }
    template <class T>
    cudaError_t alloc(T **p, size_t n) {
        void *q = nullptr;
        const cudaError_t e = cudaMallocAsync(&q, n ? n * sizeof(T) : 1, s);
        if (e == cudaSuccess) ptrs.push_back(q);
        *p = static_cast<T *>(q);
        return e;
    }
};

// Search region of one side (0: tile a, 1: tile b) in that tile's frame:
// the union over the window of the shared boxes.
void side_region(const int *d0, const int *r, const int *D, int side, int3 &u0, int3 &u1) {
    int lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
        const Range a = shared_range(d0[k] - r[k], D[k], side), b = shared_range(d0[k] + r[k], D[k], side);
        lo[k] = std::min(a.lo, b.lo);
        hi[k] = std::max(a.hi, b.hi);
        if (lo[k] > hi[k]) hi[k] = lo[k];
    }
    u0 = make_int3(lo[0], lo[1], lo[2]);
    u1 = make_int3(hi[0], hi[1], hi[2]);
}

uint32_t uf_root(std::vector<uint32_t> &p, uint32_t i) {
    while (p[i] != i) {
        p[i] = p[p[i]];
        i = p[i];
    }
    return i;
}

}  // namespace

extern "C" int seg_register_montage(int device, const uint16_t *const *tiles, int on_device, uint32_t n_tiles,
                                    seg_dims dims, const seg_offset *stage, seg_offset radius, uint32_t root,
                                    seg_offset *delta, seg_montage_edge *edges, uint32_t edges_cap,
                                    uint32_t *n_edges) {
    if (!tiles || !stage || !delta || !n_edges || n_tiles == 0 || root >= n_tiles || dims.x == 0 || dims.y == 0 ||
        dims.z == 0)
        return SEG_EINVAL;
    if (radius.x < 0 || radius.y < 0 || radius.z < 0 || radius.x > SEG_REG_MAX_RXY || radius.y > SEG_REG_MAX_RXY ||
        radius.z > SEG_REG_MAX_RZ)
        return SEG_EINVAL;
    for (uint32_t i = 0; i < n_tiles; ++i)
        if (!tiles[i]) return SEG_EINVAL;
    const uint64_t n = (uint64_t)dims.x * dims.y * dims.z;
    // the kernels step up to 63 positions past a tile's end in signed integers
    if (n >= (1ull << 32) || dims.x > SEG_MAX_YZ || dims.y > SEG_MAX_YZ || dims.z > SEG_MAX_YZ) return SEG_ETOOBIG;
    const int D[3] = {(int)dims.x, (int)dims.y, (int)dims.z};
    const int r[3] = {radius.x, radius.y, radius.z};
    // pairs whose stage boxes overlap, in (a, b) order
    std::vector<seg_montage_edge> E;
    for (uint32_t a = 0; a < n_tiles; ++a)
        for (uint32_t b = a + 1; b < n_tiles; ++b) {
            const int64_t o[3] = {(int64_t)stage[b].x - stage[a].x, (int64_t)stage[b].y - stage[a].y,
                                  (int64_t)stage[b].z - stage[a].z};
            bool ov = true;
            for (int k = 0; k < 3; ++k) ov = ov && o[k] < D[k] && -o[k] < D[k];
            if (!ov) continue;
            seg_montage_edge e;
            std::memset(&e, 0, sizeof(e));
            e.a = a;
            e.b = b;
            e.score = -2.0;
            E.push_back(e);
        }
    *n_edges = (uint32_t)E.size();
    if (E.size() > edges_cap || (!edges && !E.empty())) return SEG_ESMALL;

    RK(cudaSetDevice(device));
    {
        // keep freed scratch in the pool between calls
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, device) == cudaSuccess) {
            uint64_t thr = UINT64_MAX;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
        }
        cudaGetLastError();
    }
    Scratch sc;
    RK(sc.init());
    // the tiles on the device
    std::vector<const uint16_t *> dt(n_tiles);
    if (on_device) {
        for (uint32_t i = 0; i < n_tiles; ++i) dt[i] = tiles[i];
    } else {
        for (uint32_t i = 0; i < n_tiles; ++i) {
            uint16_t *p;
            RK(sc.alloc(&p, n));
            RK(cudaMemcpyAsync(p, tiles[i], 2 * n, cudaMemcpyHostToDevice, sc.s));
            dt[i] = p;
        }
    }
    const int SX = 2 * r[0] + 1, SY = 2 * r[1] + 1, S = SX * SY * (2 * r[2] + 1);
    // Pairs go in groups of up to REG_GROUP: every pair of a group gets its
    // own slice of sums (Sab, Sa, Saa, Sb, Sbb of every shift), each kernel
    // takes the whole group in one launch, and one copy and one
    // synchronisation bring its sums to the host.
    constexpr size_t REG_GROUP = 64;
    const size_t per = 5 * (size_t)S;
    const size_t gmax = std::max<size_t>(1, std::min(E.size(), REG_GROUP));
    unsigned long long *dsum, *dp1, *dp2;
    RegPair *dpair;
    std::vector<RegPair> pairs(E.size());
    int most_y = 0, most_z = 0;  // rows and planes of the largest search regions, voxels of a plane
    size_t most_xy = 0;
    for (size_t ei = 0; ei < E.size(); ++ei) {
        const seg_montage_edge &e = E[ei];
        RegPair &P = pairs[ei];
        const int d0[3] = {stage[e.b].x - stage[e.a].x, stage[e.b].y - stage[e.a].y, stage[e.b].z - stage[e.a].z};
        P.tile[0] = dt[e.a];
        P.tile[1] = dt[e.b];
        P.d0 = make_int3(d0[0], d0[1], d0[2]);
        for (int side = 0; side < 2; ++side) {
            side_region(d0, r, D, side, P.u0[side], P.u1[side]);
            const int uy = P.u1[side].y - P.u0[side].y;
            most_xy = std::max(most_xy, (size_t)uy * (P.u1[side].x - P.u0[side].x));
            most_y = std::max(most_y, uy);
            most_z = std::max(most_z, P.u1[side].z - P.u0[side].z);
        }
    }
    // Planes are cut into slabs while a group has fewer than PLANE_BLOCKS of
    // them per multiprocessor, down to SLAB_ROWS rows and SLAB_VOXELS voxels
    // (slabs of 40 rows of 20 voxels cost 10 % of a call that takes 132 us with
    // whole planes), and taken PZ at a time so that their sums stay within
    // PLANE_BYTES (a single plane of every pair: at most 82 MB, for 64 pairs, 64
    // slabs and 25 x 25 shifts).
    constexpr int SLAB_ROWS = 32, PLANE_BLOCKS = 4, MAX_SLABS = 64;
    constexpr size_t SLAB_VOXELS = 16384, PLANE_BYTES = 256u << 20;
    int sms = 0;
    RK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    int ns = 1;
    while (ns < MAX_SLABS && 2 * ns * SLAB_ROWS <= most_y && 2 * ns * SLAB_VOXELS <= most_xy &&
           2 * gmax * most_z * ns < (size_t)PLANE_BLOCKS * sms)
        ns *= 2;
    const size_t plane = (size_t)SX * SY * ns;  // sums of one plane of one side
    const int PZ = (int)std::max<size_t>(
        1, std::min<size_t>(std::min<size_t>((size_t)most_z, 65535),  // (the last grid dimension of k_reg_box)
                            PLANE_BYTES / (2 * sizeof(unsigned long long) * 2 * gmax * plane)));
    const size_t pper = plane * PZ;
    RK(sc.alloc(&dsum, per * gmax));
    RK(sc.alloc(&dp1, 2 * gmax * pper));
    RK(sc.alloc(&dp2, 2 * gmax * pper));
    RK(sc.alloc(&dpair, gmax));
    std::vector<unsigned long long> hs(per * gmax);
    const size_t smem = reg_corr_smem(r[0], r[1], r[2]);
    const RegCorrFn corr = reg_corr_fn(r[0], std::make_integer_sequence<int, SEG_REG_MAX_RXY + 1>{});
    if (!corr) return SEG_EINVAL;
    RK(cudaFuncSetAttribute(corr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int3 r3 = make_int3(r[0], r[1], r[2]);
    for (size_t g0 = 0; g0 < E.size(); g0 += REG_GROUP) {
        const size_t g1 = std::min(E.size(), g0 + REG_GROUP);
        const unsigned ng = (unsigned)(g1 - g0);
        // a pair's blocks: sub-boxes of side 0, planes of either side
        size_t nb = 0;
        int nz = 0;
        for (size_t ei = g0; ei < g1; ++ei) {
            const int3 u0 = pairs[ei].u0[0], u1 = pairs[ei].u1[0];
            nb = std::max(nb, (size_t)((u1.x - u0.x + RC_TX - 1) / RC_TX) * ((u1.y - u0.y + RC_TY - 1) / RC_TY) *
                                  ((u1.z - u0.z + RC_TZ - 1) / RC_TZ));
            for (int side = 0; side < 2; ++side) nz = std::max(nz, pairs[ei].u1[side].z - pairs[ei].u0[side].z);
        }
        RK(cudaMemcpyAsync(dpair, pairs.data() + g0, ng * sizeof(RegPair), cudaMemcpyHostToDevice, sc.s));
        RK(cudaMemsetAsync(dsum, 0, per * ng * sizeof(unsigned long long), sc.s));
        for (int z0 = 0; z0 < nz; z0 += PZ) {
            const int n = std::min(PZ, nz - z0), bz = std::max(BOX_SLABS / ns, 1);
            k_reg_plane<<<dim3((unsigned)(n * ns), 2 * ng), RP_THREADS, 0, sc.s>>>(dpair, D[0], D[1], r3, z0, ns, pper,
                                                                                   dp1, dp2);
            k_reg_box<<<dim3((unsigned)((S + 63) / 64), 2 * ng, (unsigned)((n + bz - 1) / bz)), 64, 0, sc.s>>>(
                dpair, dp1, dp2, D[0], D[1], D[2], r3, z0, z0 + n, ns, pper, dsum, per);
        }
        if (nb > 0)
            corr<<<dim3((unsigned)nb, ng), RC_THREADS, smem, sc.s>>>(dpair, D[0], D[1], D[2], r[1], r[2], dsum, per);
        RK(cudaGetLastError());
        RK(cudaMemcpyAsync(hs.data(), dsum, per * ng * sizeof(unsigned long long), cudaMemcpyDeviceToHost, sc.s));
        RK(cudaStreamSynchronize(sc.s));
        for (size_t ei = g0; ei < g1; ++ei) {
            seg_montage_edge &e = E[ei];
            const unsigned long long *h = hs.data() + per * (ei - g0);
            const int d0[3] = {stage[e.b].x - stage[e.a].x, stage[e.b].y - stage[e.a].y,
                               stage[e.b].z - stage[e.a].z};
            // the first best shift in z, y, x order
            for (int si = 0; si < S; ++si) {
                const int s[3] = {si % SX - r[0], (si / SX) % SY - r[1], si / (SX * SY) - r[2]};
                uint64_t cnt = 1;
                for (int k = 0; k < 3; ++k) {
                    const Range q = shared_range(d0[k] + s[k], D[k], 0);
                    cnt *= (uint64_t)(q.hi > q.lo ? q.hi - q.lo : 0);
                }
                if (cnt == 0) continue;
                const unsigned long long sab = h[si], sa = h[S + si], saa = h[2 * (size_t)S + si];
                const unsigned long long sb = h[3 * (size_t)S + si], sbb = h[4 * (size_t)S + si];
                const __int128 N = (__int128)cnt;
                const __int128 num = N * (__int128)sab - (__int128)sa * (__int128)sb;
                const __int128 va = N * (__int128)saa - (__int128)sa * (__int128)sa;
                const __int128 vb = N * (__int128)sbb - (__int128)sb * (__int128)sb;
                if (va == 0 || vb == 0) continue;
                const double rho = (double)num / std::sqrt((double)va * (double)vb);
                if (rho > e.score) {
                    e.score = rho;
                    e.shift.x = s[0];
                    e.shift.y = s[1];
                    e.shift.z = s[2];
                }
            }
        }
    }
    // maximum spanning tree: scores highest first, ties by (a, b)
    std::vector<uint32_t> order(E.size());
    std::iota(order.begin(), order.end(), 0u);
    std::stable_sort(order.begin(), order.end(), [&](uint32_t i, uint32_t j) { return E[i].score > E[j].score; });
    std::vector<uint32_t> par(n_tiles);
    std::iota(par.begin(), par.end(), 0u);
    std::vector<std::vector<uint32_t>> adj(n_tiles);
    for (uint32_t i : order) {
        seg_montage_edge &e = E[i];
        if (e.score < -1.5) continue;  // no defined score
        const uint32_t ra = uf_root(par, e.a), rb = uf_root(par, e.b);
        if (ra == rb) continue;
        par[ra] = rb;
        e.in_tree = 1;
        adj[e.a].push_back(i);
        adj[e.b].push_back(i);
    }
    // corrections from the root along the tree
    for (uint32_t i = 0; i < n_tiles; ++i) delta[i] = seg_offset{0, 0, 0};
    std::vector<uint8_t> seen(n_tiles, 0);
    std::vector<uint32_t> todo{root};
    seen[root] = 1;
    while (!todo.empty()) {
        const uint32_t t = todo.back();
        todo.pop_back();
        for (uint32_t i : adj[t]) {
            const seg_montage_edge &e = E[i];
            const uint32_t o = e.a == t ? e.b : e.a;
            if (seen[o]) continue;
            const int sg = e.a == t ? 1 : -1;  // delta(b) = delta(a) + shift
            delta[o] = seg_offset{delta[t].x + sg * e.shift.x, delta[t].y + sg * e.shift.y,
                                  delta[t].z + sg * e.shift.z};
            seen[o] = 1;
            todo.push_back(o);
        }
    }
    if (!E.empty()) std::memcpy(edges, E.data(), E.size() * sizeof(seg_montage_edge));
    return SEG_OK;
}
