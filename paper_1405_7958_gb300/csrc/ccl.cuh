// Union-find connected components on the GPU (BWLabel + AreaThreshold), for
// a batch of images in one launch per stage.
#pragma once

#include "common.cuh"

namespace rtk {

constexpr int kUfBlock = 32;                   // block side
constexpr int kUfEdge = 4 * kUfBlock;
constexpr int kUfMaxRoots = kUfBlock * kUfBlock / 2;   // local components of a block (4-conn checkerboard)
constexpr int kUfMaxImgs = 32;
// Images of at most this many 64 x 64 tiles are labeled here: its four short
// launches beat the five of the union-find over runs, whose stages are bound
// by their slowest tile (whole calls of rt_label_area, which pack bytes to
// bits for the runs; nuclei images, 180 nuclei per megapixel:
// 24 against 34 us at 700 x 700, 26 against 36 at 1024 x 1024, 35 against 41
// at 2048 x 2048, equal at 2400 x 2400, 58 against 54 at 3000 x 3000, 94
// against 63 at 4096 x 4096; with 380 nuclei the lines cross at 2048 x 2048,
// with 60 at 3000 x 3000).
constexpr int kUfMaxTiles = 1444;

// One image of a labeling batch: the binary input, the workspace arrays
// (carved by the caller, uf_workspace_bytes long in total) and the outputs.
struct UfImage {
    const uint8_t *in;   // binary input (nonzero = foreground), H x W, stride ld_in
    int64_t ld_in;
    int H, W;
    int nbx, nby;        // 32 x 32 blocks per row / column
    int64_t blk_base;    // first block of this image in the batch's block numbering
    int32_t *U;          // forest over block-local roots, indexed by pixel index r*W + c (sparse use)
    int32_t *A;          // per local root: its area, then the component's (sparse use)
    int32_t *edge;       // per block, kUfEdge entries: local root of the top row, bottom row,
                         // left column, right column pixels (-1 = not in a component)
    int32_t *list;       // per block, kUfMaxRoots slots: the block's local roots
    uint16_t *cnt;       // per block: number of local roots
    uint16_t *lroot;     // per pixel (stride W): its local root inside its block (lr * 32 + lc), 0xFFFF = none;
                         // not written for blocks without foreground
    uint8_t *bempty;     // per block: 1 = no foreground
    int32_t *labels;     // output, H x W, stride ld_lab
    int64_t ld_lab;
    int32_t *n_kept;     // nullable: number of components kept (zeroed by the first stage)
};

struct UfBatch {
    int n;
    int64_t nblk;        // blocks over all images
    int32_t amin, amax;  // area range kept, inclusive
    UfImage img[kUfMaxImgs];
};

// Workspace bytes of one H x W image (every array above, 256-byte aligned pieces).
size_t uf_workspace_bytes(int H, int W);
// Carves the workspace arrays of `d` from base (uf_workspace_bytes(H, W) bytes, 256-byte aligned) and sets
// the block counts; in, labels and n_kept are left to the caller.
void uf_carve(UfImage &d, char *base, int H, int W);
// Appends image `d` to the batch (sets its blk_base).
void uf_add(UfBatch &b, const UfImage &d);
// Labels with the area filter for every image of the batch: block-local
// components, merges across block edges, final roots with their areas, and
// the output pass (four launches).
cudaError_t launch_label_batch(const UfBatch &b, int conn, cudaStream_t s);

}  // namespace rtk
