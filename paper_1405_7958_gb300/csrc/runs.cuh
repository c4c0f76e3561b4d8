// Hole filling and component labeling on runs of bit rows (FillHoles,
// BWLabel and AreaThreshold), for a batch of images in one launch per stage.
#pragma once

#include "common.cuh"

namespace rtk {

constexpr int kRunSide = 64;          // tiles of 64 rows x one 64-bit word
// Component slots per tile: components that touch the tile's rim, whose 252
// pixels hold at most 126 of them.
constexpr int kRunSlots = 128;
constexpr int kRunSides = 4 * kRunSide;
constexpr int kRunWords = kRunSide * kRunSide / 2;   // runs of a tile at most
constexpr int kRunMaxImgs = 32;

// One image. Tiles are numbered row by row from tile_base.
struct RunImage {
    int H, W, nx, ny, tile_base;
    const uint8_t *in;     // byte image to pack (nonzero = foreground) or to threshold, stride ld_in; NULL: bits are given
    int64_t ld_in;
    uint8_t *filled;       // nullable: F as bytes 0/1, stride ld_filled
    int64_t ld_filled;
    int32_t *labels;       // stride ld_lab
    int64_t ld_lab;
    int32_t *n_kept;       // nullable: number of components kept (zeroed by the local stage)
};

// Up to kRunMaxImgs images and the batch's workspace, passed by value.
struct RunBatch {
    int n, ntiles;
    int32_t amin, amax;              // area range kept, inclusive
    unsigned long long *bits;        // per tile: 64 rows, bit = column; foreground
    unsigned long long *seeds;       // the same layout, launch_run_reach: pixels the marker reaches by itself
    int lo, hi;                      // launch_run_reach: threshold, and threshold + marker offset (>= 0)
    unsigned long long *kept;        // nullable: the kept pixels, in the same layout
    uint8_t *sides;                  // per tile: slot (255: none) of the top, bottom, left, right pixels
    uint8_t *cnt;                    // per tile: slots of the fill's background components
    uint32_t *outside;               // forest over 1 + tile * kRunSlots + slot; 0 = outside
    uint32_t *U, *A, *M;             // the same nodes for the labels: forest, area, first pixel
    uint8_t *lcnt;                   // per tile: slots of the labels
    uint32_t *words;                 // per tile: its runs' words after the local stage (runs.cu)
    RunImage img[kRunMaxImgs];
};

size_t run_tiles(int H, int W);
// Appends an image (its tile counts and base are set here).
RunImage &run_add(RunBatch &b, int H, int W);
// byte images -> bits
cudaError_t launch_run_pack(const RunBatch &b, cudaStream_t s);
// bits = (R < lo) for the reconstruction R by dilation of the chain's marker
// under the images, 8-connected, but for the last step, which launch_run_fill
// takes with again = true: the part of bits that its fill adds first
cudaError_t launch_run_reach(const RunBatch &b, cudaStream_t s);
// Holes filled in bits (and filled written); conn 4 or 8 is the background's
// connectivity. With label_conn 8 (0: none, another: cudaErrorInvalidValue)
// the last launch also makes the local components that launch_run_label needs.
cudaError_t launch_run_fill(const RunBatch &b, int conn, int label_conn, cudaStream_t s, bool again = false);
// local components of bits, where launch_run_fill has not made them
cudaError_t launch_run_local(const RunBatch &b, int conn, cudaStream_t s);
// labels with the area filter, counts and kept bits
cudaError_t launch_run_label(const RunBatch &b, int conn, cudaStream_t s);

}  // namespace rtk
