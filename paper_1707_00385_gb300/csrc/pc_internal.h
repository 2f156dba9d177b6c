// pc_internal.h -- what the host runtime (pc_api.cu) and the kernels
// (pc_fit_*.cu) share.  Not part of the public C ABI.
#pragma once
#include <cuda_runtime.h>

#ifdef __CUDACC__
#define PC_HD __host__ __device__
#else
#define PC_HD
#endif

namespace pcurv {

// Pinhole intrinsics (pixels) and their reciprocals.
struct Camera {
    float fx, fy, cx, cy;
    float ifx, ify;
};

// Method parameters as the kernels read them.
struct FitConfig {
    int r;             // window radius
    int rn;            // initial-normal radius
    int T;             // re-weighted iterations
    int stride;        // window sampling stride
    float invk;        // 1/k of W(eps) = k/(k+eps^2) = 1/(1 + eps^2/k)
    int reject;        // rejection filter on/off
    float reject_ratio;
    float det_tol;
    float pivot_tol;
    int min_window;
    int kahan;         // compensated moment sums
    float fp64_pivot;  // refactorise in FP64 below this scaled pivot (0 = never)
    int sms;           // SMs of the device launches go to (0: not known yet)
};

// Output tile of one CTA: TILE_W x th pixels, in five variants
//   0: 32 x 8 pixels, one thread each (256 threads)
//   1: 32 x 4 pixels, one thread each (128 threads; frames with few tiles)
//   2: 32 x 4 pixels, 2 lanes each; 3: 32 x 2, 4 lanes; 4: 32 x 1, 8 lanes
//      (256 threads; the lanes of a pixel share its window rows)
// Variants 0 and 1 give the same bits; the lane groups add the moment sums in
// another order, which changes single-precision rounding only.
constexpr int TILE_W = 32;
constexpr int NUM_TILE_VARIANTS = 5;
inline int tile_h_of(int variant) {
    constexpr int h[NUM_TILE_VARIANTS] = {8, 4, 4, 2, 1};
    return h[variant];
}
inline int lanes_of(int variant) {
    constexpr int g[NUM_TILE_VARIANTS] = {1, 1, 2, 4, 8};
    return g[variant];
}
// The variant of a lane-group size (2, 4, 8), else -1.
inline int variant_of_lanes(int lanes) { return lanes == 2 ? 2 : lanes == 4 ? 3 : lanes == 8 ? 4 : -1; }
// storage tiles of the 16-bit range format (pc_pack_depth): 32 x 8
constexpr int PACK_TILE_H = 8;

// The initial-normal patch radius compiled with unrolled loops: 3, the 7 x 7
// patch of Sec. 3.2.1 (other radii run the same code with run-time loops).
constexpr int NORMAL_RADIUS_UNROLLED = 3;

inline int halo_of(const FitConfig& c) { return c.r > c.rn ? c.r : c.rn; }

// Sums of J^T W J whose running totals the one-lane FP32 kernels keep in
// shared memory, as one pair of floats per thread (fit_tile, fold_rows).
constexpr int FOLD_SUMS = 20;

// Tiles of a band of `rows` pixel rows of a frame W pixels wide, for CTAs of
// 32 x th threads.  Lane groups (strips = false) cover the width with 32-pixel
// columns.  One thread per pixel: the columns that fill 32 pixels, then the
// rest of the width, in a last column or, where that takes fewer tiles, in
// strips 16 and 8 pixels wide whose tiles are 2 and 4 times as tall, so that a
// ragged width leaves the threads of at most 7 pixel columns idle instead of
// 31.  The kernels' time goes with the warps that run, whether or not their
// threads have a pixel.  GB300, with the rule that chooses the tile height:
// one 323 x 241 frame (r = 5, T = 5) 127.0 -> 110.8 us, one 682 x 579 frame
// (r = 2, rejection) 246 -> 166 us, 27 frames of 122 x 64, 792 x 709 and
// 64 x 52 in one batch (r = 9) 18.84 -> 18.63 ms; widths that are a multiple of
// 32 have no strips.  Queue order: columns (row by row of tiles), 16-wide
// strip, 8-wide strip.
struct Tiling {
    int cols;          // 32-pixel columns
    int full, n16, n8; // tiles in the columns and in the two strips
};
struct TilePos {
    int ub, vb;        // first pixel (vb from the band's first row)
    int lg;            // log2 of the width: 5, 4 or 3; the height is (32 th) >> lg
};
PC_HD inline Tiling tiling_of(int rows, int W, int th, bool strips) {
    Tiling t;
    const int rem = W % TILE_W, rows_t = (rows + th - 1) / th;
    t.cols = W / TILE_W;
    t.n16 = rem > 8 ? (rows + 2 * th - 1) / (2 * th) : 0;
    t.n8 = (rem > 0 && rem <= 8) || rem > 16 ? (rows + 4 * th - 1) / (4 * th) : 0;
    if (rem > 0 && (!strips || rem > 24 || t.n16 + t.n8 >= rows_t)) {
        t.cols++;
        t.n16 = t.n8 = 0;
    }
    t.full = t.cols * rows_t;
    return t;
}
PC_HD inline TilePos tile_pos(const Tiling& t, int i, int th) {
    if (i < t.full) {
        const int row = i / t.cols;
        return TilePos{(i - row * t.cols) * TILE_W, row * th, 5};
    }
    i -= t.full;
    if (i < t.n16) return TilePos{t.cols * TILE_W, i * 2 * th, 4};
    return TilePos{t.cols * TILE_W + (t.n16 > 0 ? 16 : 0), (i - t.n16) * 4 * th, 3};
}
inline Tiling tiling_of_variant(int rows, int W, int variant) {
    return tiling_of(rows, W, tile_h_of(variant), lanes_of(variant) == 1);
}
inline long long tiles_of(int rows, int W, int variant) {
    const Tiling t = tiling_of_variant(rows, W, variant);
    return (long long)t.full + t.n16 + t.n8;
}
inline bool has_strips(const Tiling& t) { return t.n16 + t.n8 > 0; }

// First row of the frame that a band ending at row vend does not read.  A strip
// tile is taller than a tile row and may overhang the band; the band's windows
// end `halo` rows past it, and the rows after those may not have been copied to
// the device yet (pc_compute_host).  The staging stops here, and a band waits
// for the copy of the rows up to here.
PC_HD inline int staged_end(int vend, int halo, int H) { return H - vend > halo ? vend + halo : H; }

// Row pitch of the staged planes of a tile tw pixels wide.  A warp of a strip
// tile spans 2 rows of 16 or 4 rows of 8 pixels: the pitch is padded so that
// those rows fall into different shared-memory banks.
PC_HD inline int tile_pitch(int tw, int halo) {
    const int sw = tw + 2 * halo;
    return tw == 16 ? sw + (48 - sw % 32) % 32 : tw == 8 ? sw + (24 - sw % 16) % 16 : sw;
}

// Z and c planes of the tile + halo, per-row valid counts (of a 32-pixel tile
// or, with strips, the largest of the three shapes) and, for fold_threads > 0,
// the folded totals of that many threads (8-byte aligned).  A launch without a
// strip asks for what 32-pixel tiles need: what a strip needs more is taken from
// the L1 cache, which holds the registers a window loop spills (GB300, the 37 x
// 37 patch with rejection, 64 x 48: 65.7 us, with the strips' request 70.8).
inline size_t fit_smem_bytes(const FitConfig& c, int th, bool strips, int fold_threads = 0) {
    const int h = halo_of(c);
    size_t planes = 0;
    for (int tw = TILE_W; tw >= (strips ? 8 : TILE_W); tw /= 2) {
        const int rows = TILE_W * th / tw + 2 * h;
        const size_t b = (size_t)tile_pitch(tw, h) * rows * 2 * sizeof(float) + (size_t)rows * tw * sizeof(int);
        planes = b > planes ? b : planes;
    }
    return (planes + 7) / 8 * 8 + (size_t)fold_threads * FOLD_SUMS * 8;
}

// One frame: caller-owned device buffers, size and intrinsics.
struct FrameArgs {
    const float* depth;
    int H, W;
    Camera cam;
    float* k1;
    float* k2;
    float* normal;  // may be nullptr
    // centred 16-bit storage instead of depth (the kernels reading it): per
    // pixel an offset (format 1 FP16, 2 BF16), per 32x8 tile an FP32 base
    const unsigned short* packed;
    const float* tile_base;
    int format;
};

// A frame of a batch and its place in the flattened tile queue.
struct BatchFrame {
    FrameArgs f;
    int tile_begin;  // first queue index of this frame
    int pad;
};

// Forms of the persistent kernel over a table of tiles: with strips among them,
// with 32-pixel columns only, and with columns only in a queue so short that its
// end counts (k_fit_batch).
enum BatchForm { BATCH_STRIPS, BATCH_COLUMNS, BATCH_FEW, NUM_BATCH_FORMS };
// Tiles per CTA of the persistent grid up to which a queue is short.  The state
// formed a pair ahead and the registers of the strips pay in a queue of many
// tiles; where the last tiles of the SMs decide, or a warp is alone on its
// scheduler, they cost more than they give.  GB300, T = 5, without / with a kernel
// for short queues: one 640 x 480 frame r = 9 1035 / 940 us, r = 10 1220 / 1137,
// two of r = 7 1239 / 1189, three of r = 7 level (12 tiles a CTA); one 64 x 48
// frame r = 12 150 / 141, the 37 x 37 patch 56.8 / 52.7, with rejection 512 x 424
// 574 / 510.
constexpr int FEW_TILES = 8;
inline BatchForm batch_form(bool strips, int tiles, int grid) {
    return strips ? BATCH_STRIPS : tiles / FEW_TILES < grid ? BATCH_FEW : BATCH_COLUMNS;
}

// Device-resident batch table: header followed by nframes descriptors.
struct BatchTable {
    int nframes;
    int total_tiles;
    int pad[2];
    BatchFrame frames[1];  // nframes entries
};

inline size_t batch_table_bytes(int nframes) {
    return sizeof(BatchTable) + (size_t)(nframes > 1 ? nframes - 1 : 0) * sizeof(BatchFrame);
}

// Kernel entry points of one instantiation (window radius, dense or run-time),
// per tile variant (nullptr where a variant is not compiled).
struct KernelOps {
    // tile rows [ty0, ty1) of one frame (the variant's tile height)
    cudaError_t (*fit[NUM_TILE_VARIANTS])(const FrameArgs&, const FitConfig&, cudaStream_t, int ty0, int ty1);
    cudaError_t (*batch[NUM_TILE_VARIANTS])(const BatchTable*, unsigned*, int grid, const FitConfig&, BatchForm,
                                            cudaStream_t);
    cudaError_t (*occupancy[NUM_TILE_VARIANTS])(const FitConfig&, int*);
};

// Instantiation groups (one translation unit each, compiled in parallel);
// each returns its table for radius r, or nullptr.  ops_r* and ops_generic
// hold the one-lane variants, ops_lanes the lane-group variants (run-time
// radius and stride, serving every window).
const KernelOps* ops_r1_4(int r);
const KernelOps* ops_r5_8(int r);
const KernelOps* ops_r9_12(int r);
const KernelOps* ops_generic();
const KernelOps* ops_lanes();
// The sparsely sampled 37 x 37 patch of Sec. 4.2.1 (radius 18, read as every
// third pixel), unrolled like the dense radii; nullptr for other windows.
constexpr int SPARSE_RADIUS = 18, SPARSE_STRIDE = 3;
const KernelOps* ops_sparse(int r, int stride);

// Kernels of compensated sums (run-time radius and stride), for float32 ranges
// or 16-bit storage.
const KernelOps* ops_kahan(bool packed);
// Plain sums on 16-bit range storage, 32 x 8 tiles: dense windows of radius 1
// to 6 and 7 to 12 with unrolled columns (nullptr outside), and run-time radius
// and stride (r = 0).
const KernelOps* ops_packed_r0_6(int r);
const KernelOps* ops_packed_r7_12(int r);
// The kernels reading 16-bit storage (either format) under cfg.
const KernelOps* select_packed_ops(const FitConfig& cfg);

// The instantiation serving cfg (dense radii 1..12 unrolled, anything else
// run-time; compensated sums on the precision kernels), all five variants.
const KernelOps* select_ops(const FitConfig& cfg);

// Packs float32 ranges into per-tile-centred 16-bit storage (format 1 FP16, 2 BF16).
cudaError_t launch_pack(const float* depth, int H, int W, int format, unsigned short* packed,
                        float* tile_base, cudaStream_t stream);

// Organised outputs (pc_outputs.cu): point cloud and initial-normal field.
cudaError_t launch_backproject(const float* depth, int H, int W, const Camera& cam, float* xyz, int sms,
                               cudaStream_t stream);
cudaError_t launch_initial_normals(const float* depth, int H, int W, const Camera& cam, int rn, float det_tol,
                                   float* normal, int sms, cudaStream_t stream);

}  // namespace pcurv

struct pc_ctx;

namespace pcurv {

// Read access to a context's kernel parameters, and a way to leave a message
// for pc_last_error(), for entry points defined outside pc_api.cu.
const FitConfig& ctx_config(const pc_ctx* ctx);
void ctx_set_error(pc_ctx* ctx, const char* msg);
// The tile variant the context's parameters force (a lane group of
// lanes_per_pixel, or a one-lane tile height), else -1.
int ctx_forced_variant(const pc_ctx* ctx);

}  // namespace pcurv
