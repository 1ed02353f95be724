// seg_internal.h -- device-side batch descriptors shared by the runtime and
// the kernels of libseg (not part of the public ABI).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "seg.h"

namespace seg {

// Per-volume status words (VolDev::stat).
enum StatWord : uint32_t {
    ST_THRESH = 0,     // Otsu level t* (foreground = s > t*)
    ST_RUNS = 1,       // number of foreground runs R
    ST_CELLS = 2,      // number of surviving cells K
    ST_LABEL_RUNS = 3, // number of runs of surviving cells
    ST_ERROR = 4,      // error bits (ERR_*)
    ST_MRF_STEPS = 5,  // MRF denoise: steps kept
    ST_MRF_SEL = 6,    // MRF denoise: result buffer (0 input, 1 mrf_buf[0], 2 mrf_buf[1])
    ST_MRF_DONE = 7,   // MRF denoise: stopped
    ST_MRF_DELTA = 8,  // MRF denoise: step size (0: fewer than two levels)
    ST_MRF_CNT = 9,    // MRF denoise: tiles done in the current launch
    ST_MRF_CHG = 10,   // MRF denoise: some voxel changed in the current step
    ST_MRF_E = 12,     // MRF denoise: uint64 at words 12-13, Laplacian sum S, then sum d^2
    ST_MRF_LIMIT = 14, // MRF denoise: binary64 bound N sigma^2 at words 14-15
    ST_WORDS = 16,
};

enum ErrBits : uint32_t {
    ERR_UNION = 1u << 0,   // union retry limit reached
    ERR_KCAP = 1u << 1,    // more cells than the feature buffer holds
    ERR_RCAP = 1u << 2,    // more runs than the run buffer holds
    ERR_OTSU = 1u << 3,    // histogram total differs from the voxel count
    ERR_TIMEOUT = 1u << 4, // a bounded wait on an asynchronous copy gave up
};

constexpr int TILE_X = 64;        // smoothing tile width (outputs along x)
constexpr uint32_t UNION_LIMIT = 1u << 24;  // union-find retries before ERR_UNION
constexpr int ROW_TILE = 256;     // rows per row tile (run kernels; their block size)
constexpr int ROW_TILE_MIN = 32;  // smallest row tile (batches with few rows)
// Label tile: LABEL_WORDS label words (256 KB) in whole rows, at most ROW_TILE
// rows; halved for batches with few tiles, down to LABEL_WORDS >> LABEL_SHRINK.
constexpr uint32_t LABEL_WORDS = 65536;
constexpr uint32_t LABEL_SHRINK = 4;
constexpr int HIST_BINS = 65536;
// Union-find bricks: bk_y x bk_z rows (at most BRICK_ROWS, the block size),
// whose runs are united in shared memory when there are at most BRICK_CAP of
// them.
constexpr int BRICK_ROWS = 256;
constexpr int BRICK_CAP = 3072;

// One volume-channel inside a batch.  All pointers are device addresses.
struct VolDev {
    const uint16_t *raw;      // [Z][Y][X]
    uint32_t *labels;         // [Z][Y][X] output
    seg_cell_features *feat;  // k_cap cells output
    uint32_t *stat;           // ST_WORDS words
    uint32_t *hist;           // 65536 uint32 bins
    uint16_t *smooth;         // [Z][Y][sm_pitch] smoothed voxels (pass 1 -> threshold pass)
    uint16_t *wmax;           // rows x W: largest smoothed value of each mask word (k_smooth_rows
                              // volumes with X % 32 == 0 or X > 512; else null)
    uint32_t *mask;           // rows x W words, bit b of word w is x = 32w + b
    uint32_t *rowoff;         // rows + 1: run count per row, then run offsets
    uint32_t *rowk;           // rows: kept-root count per row, then label base
    uint32_t *tsum;           // row tiles: run totals, then offsets
    uint32_t *tkeep;          // row tiles: kept-root totals, then offsets
    uint32_t *run_x;          // r_cap: x0 | x1 << 16 (inclusive run ends)
    uint32_t *run_par;        // r_cap: union-find parent (run index)
    uint32_t *run_aux;        // r_cap: voxel count at roots, then label
    uint64_t k_cap;
    uint64_t r_cap;
    uint32_t X, Y, Z, W;      // W = words per mask row
    uint32_t sm_pitch;        // voxels per row of smooth: X, or X rounded up to 8 (voxels past X are 0)
    uint32_t rows;            // Y * Z
    uint32_t min_volume;
    uint32_t union_limit;     // retries before a union gives up (ERR_UNION)
    uint32_t ntx, nty, ntz;   // smoothing tiles per axis (k_smooth_hist; 0 for row-aligned volumes)
    uint32_t nrt;             // row tiles (of BatchHdr::row_tile rows)
    uint32_t tile_base;       // first flat smoothing-tile index
    // k_smooth_rows (X % 8 == 0 with a 16-byte aligned input, or X even and
    // at least 10 with a 4-byte aligned input); fs_ntx = 0 for the other volumes
    uint32_t fs_rt;           // octets per tile row (min(ceil(X / 8), 64))
    uint32_t fs_ty;           // rows per tile (FS_NT / fs_rt)
    uint32_t fs_hx;           // 1: x-tiled (X > 512), staged rows carry a halo chunk on each side
    uint32_t fs_rag;          // 1: X % 8 != 0 (X even): 4-byte copies and stores, a partial last octet
    uint32_t fs_tz;           // planes per tile
    uint32_t fs_ntx, fs_nty, fs_ntz;  // tiles per axis
    uint32_t fs_base;         // first flat k_smooth_rows tile index
    uint32_t rt_base;         // first flat row-tile index
    uint32_t lb_rows;         // rows per label tile (at most ROW_TILE)
    uint32_t nlb;             // label tiles
    uint32_t lb_base;         // first flat label-tile index
    uint32_t bk_y, bk_z;      // rows of a union-find brick along y and z (powers of two)
    uint32_t nby;             // union-find bricks along y
    uint32_t nbk;             // union-find bricks
    uint32_t bk_base;         // first flat brick index
    uint32_t nbt;             // row pairs that cross a brick face (k_union tasks)
    uint32_t bt_base;         // first flat k_union thread index
    uint32_t bt_lanes;        // log2 of the threads per row pair
    // denoise front end (dn_r > 0); raw then points at dn_out
    const uint16_t *dn_src;   // observed image [Z][Y][X]
    uint16_t *dn_a, *dn_b;    // box-pass ping-pong buffers (the background ends in dn_a)
    uint16_t *dn_out;         // denoised image (the smoothing's input)
    uint32_t dn_r;            // box radius, 0 = no denoise
    uint32_t dn_mul;          // ceil(2^32 / (2 dn_r + 1)): division by the box width
    uint32_t dn_ring;         // bit a: axis a by register rings (box_rings())
    uint32_t dn_n[3];         // box-pass items per axis (groups of lines x chunks)
    uint32_t dn_base0, dn_base1, dn_base2;  // first flat box item per axis
    uint32_t dn_tiles;        // median tiles
    uint32_t dn_tbase;        // first flat median tile
    // closing of the foreground (cl_r > 0)
    uint32_t *cl_ext;         // dilated mask on rows y in [-r, Y+r), z in [-r, Z+r), W + 2 words each
    uint32_t cl_r;            // ball radius, 0 = no closing
    uint32_t cl_n;            // dilation items (words of the extended mask)
    uint32_t cl_base;         // first flat dilation item
    uint32_t cl_pad;
    // distance map of the final foreground (dt_w[0] > 0)
    uint32_t *dt_out;         // [Z][Y][X] weighted squared distances (output)
    uint32_t *dt_h;           // [Z][Y][X] distances of the x and y passes
    uint32_t *dt_g;           // [Z][Y][X] x-pass distances (long-line path only)
    uint16_t *dt_sp;          // [Z][Y][X] stack positions (long-line path only)
    uint32_t dt_w[3];         // weights of dx^2, dy^2, dz^2; 0 = no distance map
    uint32_t dt_base[6];      // first flat item of this volume in each DtKernel
    uint32_t dt_zlt;          // lines of a k_dist_z tile (32, 64, 96 or 128)
    uint32_t dt_pad;
    // MRF vessel denoise (mrf_max > 0); raw is rewritten on the device to the
    // kept image before the smoothing reads it
    const uint16_t *mrf_in;   // the input I^0 [Z][Y][X]
    uint16_t *mrf_buf[2];     // steps: it 0 reads mrf_in, it > 0 mrf_buf[it & 1]; writes mrf_buf[(it + 1) & 1]
    uint32_t *mrf_bits;       // 2048 words: levels present in the input
    uint32_t mrf_max;         // step limit, 0 = off
    uint32_t mrf_tiles;       // k_mrf_stats tiles of MRF_TILE octets (8 x-consecutive voxels)
    uint32_t mrf_tbase;       // first flat k_mrf_stats tile
    uint32_t mrf_ctiles;      // k_mrf_step tiles of a plane (MRF_TILE octets of it)
    uint32_t mrf_align;       // alignment of every octet of input and buffers: 16 (X % 8 == 0), 4 (X even) or 2 bytes
    uint64_t mrf_ubase;       // first flat k_mrf_step unit (plane of a tile, z fastest)
};

// The distance-map kernels and their work items.  A volume takes the fused
// x+y kernel when its lines along y fit one block (Y <= 1024, X < 65536), the
// shared-memory z kernel when its lines along z do (Z <= 256); otherwise the
// long-line kernels, which keep their stacks in global memory.
enum DtKernel : int {
    DT_XY16 = 0,  // k_dist_xy<16>: (mask word, z) tiles, Y <= 512
    DT_XY32 = 1,  // k_dist_xy<32>: (mask word, z) tiles, 512 < Y <= 1024
    DT_X = 2,     // k_dist_x: mask rows (long y lines)
    DT_Y = 3,     // k_dist_line<1>: y lines (long y lines)
    DT_Z = 4,     // k_dist_z: (mask word, y group) tiles, Z <= 256
    DT_ZL = 5,    // k_dist_line<2>: z lines (Z > 256)
    DT_NK = 6,
};
constexpr int DZ_ELEMS = 8192;   // k_dist_z shared stack entries per block
constexpr int MRF_TILE = 256;    // octets per k_mrf_stats and k_mrf_step tile (one per thread)
constexpr uint32_t MRF_MAX_ITER = 1000;

// Batch header, followed in memory by VolDev[nvol].
struct BatchHdr {
    uint32_t nvol;
    uint32_t ntiles;     // smoothing tiles over the batch
    uint32_t nrowtiles;  // row tiles over the batch
    uint32_t tile_z;     // z-chunk of a smoothing tile
    uint32_t tile_y;     // rows of a smoothing tile
    uint32_t fs_tiles;   // k_smooth_rows tiles over the batch
    uint32_t nbricks;    // union-find bricks over the batch
    uint32_t nbtasks;    // k_union threads over the batch
    uint32_t dn_items[3];// denoise box-pass items per axis over the batch
    uint32_t dn_tiles;   // denoise median tiles over the batch
    uint32_t cl_items;   // closing dilation items over the batch
    uint32_t dt_items[DT_NK]; // distance-map items per DtKernel over the batch
    uint32_t mrf_tiles;       // k_mrf_stats tiles over the batch
    uint64_t mrf_units;       // k_mrf_step units over the batch
    uint32_t row_tile;        // rows per row tile: ROW_TILE, or down to ROW_TILE_MIN
                              // so that a batch with few rows still fills the GPU
    uint32_t nlabtiles;       // label tiles over the batch
    VolDev vol[1];       // nvol entries
};

inline size_t batch_bytes(uint32_t nvol) {
    return offsetof(BatchHdr, vol) + sizeof(VolDev) * (nvol ? nvol : 1);
}

// Host-side description of the kernels launched for one batch.
constexpr int NUM_KERNELS = 25;
extern const char *const kKernelNames[NUM_KERNELS];

struct LaunchPlan {
    int sms;             // multiprocessors on the device
    int tile_y;          // 8, 16 or 32
    int grid_hist;       // persistent grid of the histogram kernel
    int grid_vols;       // per-volume kernels
    // persistent grids of the row-tile, brick and run kernels: the blocks
    // that are resident at once (occupancy x SMs), so no block waits for a
    // slot while others already loop over their second item
    int grid_thr;        // k_threshold_runs
    int grid_rows;       // k_row_runs, k_keep_count, k_rank
    int grid_ul;         // k_union_local
    int grid_task;       // k_union, k_flatten
    int grid_lab;        // k_label_features
    int grid_box;        // k_box_x, k_box_lines
    int grid_box3;       // k_box3
    int grid_med;        // k_median27
    bool rows;           // some volume of the batch takes k_smooth_rows
    bool tiles;          // some volume of the batch takes k_smooth_hist
    uint32_t denoise;    // denoise front end: box_route_bit()s of its volumes (0: none)
    bool closing;        // some volume of the batch closes its foreground
    bool distance;       // some volume of the batch has a distance map
    int grid_dist;       // k_dist_x, k_dist_line
    int grid_dxy16;      // k_dist_xy<16>
    int grid_dxy32;      // k_dist_xy<32>
    int grid_dz;         // k_dist_z
    int grid_mrf;        // k_mrf_stats
    int grid_mrfs;       // k_mrf_step
    uint32_t mrf_iters;  // k_mrf_step launches: the largest step limit in the batch (0: none)
};

// Enqueues the whole pipeline for a batch whose header lives at d_hdr (device)
// on `stream`.  ev, when non-null, holds NUM_KERNELS + 1 events recorded
// around the launches (external records, so they survive graph capture).
// stat_out receives nvol * ST_WORDS status words (volume-major).
cudaError_t launch_pipeline(const BatchHdr *d_hdr, const LaunchPlan &plan, cudaStream_t stream,
                            cudaEvent_t *ev, uint32_t *stat_out);

// Only the tile-dependent part (init + smoothing/histogram), for tile tuning.
cudaError_t launch_tile_probe(const BatchHdr *d_hdr, const LaunchPlan &plan, cudaStream_t stream);

// Denoise front end of the volumes with dn_r > 0 (none: the kernels exit).
constexpr int DN_CHUNK = 256;    // box-pass positions per chunk of a line along y or z ...
constexpr int DN_CHUNK_X = 128;  // ... and along x
constexpr int MED_TILE_X = 64, MED_TILE_Y = 8, MED_TILE_Z = 8;  // k_median27 tile (voxels)
constexpr int DN_MAX_R = 16;
constexpr int CL_MAX_R = 8;      // closing ball radius limit
cudaError_t launch_denoise(const BatchHdr *d_hdr, const LaunchPlan &plan, cudaStream_t stream);
// A line's chunk in the box passes: its outputs [c0, c1), in positions from
// `first` on (the first position read; 3 r before the chunk, or the line's
// start).  Relative positions keep the kernels' 32-bit arithmetic exact for
// lines of up to SEG_MAX_YZ positions, whose ends leave no room for a chunk's
// halo below 2^31.
struct BoxChunk {
    uint32_t first;
    int n;           // positions of the line from `first` on
    int c0, c1;      // none when c0 >= c1
    bool start;      // `first` is the line's own start
};
__host__ __device__ inline uint32_t box_chunks(uint32_t n, uint32_t chunk) {
    return n / chunk + (n % chunk != 0u ? 1u : 0u);
}
// Chunk k of a line of n positions in box_chunks(n, chunk) equal chunks.
__host__ __device__ inline BoxChunk box_chunk(uint32_t n, uint32_t chunk, uint32_t k, uint32_t r) {
    const uint32_t per = box_chunks(n, box_chunks(n, chunk)), at = k * per;
    if (at >= n) return BoxChunk{0u, 0, 0, 0, false};
    const uint32_t lead = at < 3u * r ? at : 3u * r, len = n - at < per ? n - at : per;
    return BoxChunk{at - lead, (int)(n - (at - lead)), (int)lead, (int)(lead + len), at == lead};
}
// Box passes (seg_box.cu).  Route of a volume along an axis: 0, 1 or 2, the
// register rings of its radius class (1..4, 5..8, 9..16), or 3, the passes
// through shared memory; LaunchPlan::denoise has a bit per axis and route.
__host__ __device__ inline int box_class(uint32_t r) { return r <= 4u ? 0 : (r <= 8u ? 1 : 2); }
inline int box_route_bit(int axis, int route) { return 4 * axis + route; }
// Work items of one axis of one volume, by either route.
uint64_t box_items(int axis, bool ring, uint32_t X, uint32_t Y, uint32_t Z);
// The axes (bit 0: x, 1: y, 2: z) along which a volume takes the rings; items:
// the batch's items per axis, were all its volumes to take them.
uint32_t box_rings(uint32_t X, uint32_t Z, uint32_t r, const uint64_t *items, int sms);
// Kernel attributes and the grids of `plan`, and the launches.
cudaError_t configure_box(LaunchPlan &plan);
void launch_box_passes(const BatchHdr *d, const LaunchPlan &plan, cudaStream_t s);

// Cell-to-vessel distance: out[k - 1] = min of map over the voxels labelled k.
cudaError_t launch_cell_distance(const uint32_t *labels, const uint32_t *map, uint64_t n, uint32_t *out, uint64_t k,
                                 int sms, cudaStream_t s);
// Where k_label_features leaves a volume's run records: at the end of its
// cell table (k_cap cells of 64 bytes, of which the first K are used), when
// they fit there behind the K cells.  words: R records of three words (the
// fields of a seg_label_run, label 0 for a dropped run); tiles: per
// label tile its first run and its number of labelled runs.  Null: no room.
struct RunRecords {
    uint32_t *words;
    uint2 *tiles;
    __host__ __device__ RunRecords(seg_cell_features *feat, uint64_t k_cap, uint32_t cells, uint32_t runs,
                                   uint32_t ntiles) {
        const uint64_t room = sizeof(seg_cell_features) * k_cap, used = sizeof(seg_cell_features) * (uint64_t)cells;
        const uint64_t table = 8ull * ntiles, need = table + 12ull * runs;
        words = nullptr;
        tiles = nullptr;
        if (used + need > room) return;
        char *at = reinterpret_cast<char *>(feat) + ((room - need) & ~15ull);
        if (at < reinterpret_cast<char *>(feat) + used) return;
        tiles = reinterpret_cast<uint2 *>(at);
        words = reinterpret_cast<uint32_t *>(at + table);
    }
};

// The labelled runs of the records, in order, as three words each into out
// (device memory or mapped host memory).
cudaError_t launch_runs_compact(const RunRecords &rec, uint32_t ntiles, uint32_t runs, uint32_t *out, int sms,
                                cudaStream_t s);

// Label runs of one label image (rows = Y*Z rows of X voxels): the count
// pass (per-row counts into rowcnt, per-block offsets into tiles, the total
// into *total) and the write pass (records into out, nothing when *total >
// cap; then, with mapped != null, the records copied on to that
// device-visible host memory).
uint32_t label_runs_tiles(uint32_t rows);
cudaError_t launch_label_runs_count(const uint32_t *labels, uint32_t X, uint32_t rows, uint32_t *rowcnt,
                                    uint32_t *tiles, uint32_t *total, int sms, cudaStream_t s);
cudaError_t launch_label_runs_write(const uint32_t *labels, uint32_t X, uint32_t rows, const uint32_t *rowcnt,
                                    const uint32_t *tiles, const uint32_t *total, uint64_t cap, seg_label_run *out,
                                    seg_label_run *mapped, int sms, cudaStream_t s);

// Tile height and z-chunk of seg_otsu_threshold_noalloc for one volume on
// `blocks` blocks that take equal shares of the tiles: the pair whose fullest
// block takes the least time, the four halo planes of each tile counted.  A
// 64-row plane costs 1.4 times a 32-row one (1.6 and 1.15 us), so 64 rows are
// better for whole tiles (701 x 512 x 64: 77 us against 95; 141 with 32 rows and
// 64 planes whatever the volume: 176 tiles are two rounds of 152 blocks, the
// second nearly empty), and 32 where most of a tile's rows would lie past the
// volume (4096 x 32 x 256: 160 us for the call, 220 with 64 rows).  Fewer columns
// than blocks are tried in the most chunks that fit 1 to 64 rounds of the blocks,
// so that a lone column is cut as often as there are blocks (64 x 64 x 20000:
// 253 us, 530 in at most 64 chunks, 394 in chunks of 64 planes); others in 1 to
// 64 chunks.
struct HistSplit {
    uint32_t ty, tz;
};
inline HistSplit hist_split(uint32_t X, uint32_t Y, uint32_t Z, uint32_t blocks) {
    HistSplit best{64u, Z};
    uint64_t cost = UINT64_MAX;
    for (uint32_t ty = 64u; ty >= 32u; ty /= 2u) {
        const uint64_t columns = ((uint64_t)X + TILE_X - 1) / TILE_X * (((uint64_t)Y + ty - 1) / ty);
        for (uint32_t k = 1; k <= 64u; ++k) {
            const uint64_t most = columns < blocks ? (uint64_t)k * blocks / columns : k;
            const uint32_t n = most < Z ? (uint32_t)most : Z, tz = (Z - 1) / n + 1;
            const uint64_t tiles = columns * ((Z - 1) / tz + 1);
            const uint64_t c = (tiles + blocks - 1) / blocks * (tz + 4ull) * (ty == 64u ? 7u : 5u);
            if (c < cost) {
                cost = c;
                best = HistSplit{ty, tz};
            }
            if (n == Z) break;
        }
    }
    return best;
}

// Histogram-kernel shared memory per block for a tile height.
size_t hist_smem_bytes(int tile_y);
// k_smooth_rows: threads per block, octets per tile row at most, and the
// tile shape of a row-aligned volume of width X.
constexpr int FS_NT = 512;
constexpr int FS_RT = 64;
inline uint32_t fs_rows_rt(uint32_t X) { return X >= 8u * FS_RT ? (uint32_t)FS_RT : (X + 7u) / 8u; }
// Sets kernel attributes on `device` and fills the persistent grid sizes of
// `plan` (plan.sms must be set).
cudaError_t configure_kernels(int device, LaunchPlan &plan);

}  // namespace seg
