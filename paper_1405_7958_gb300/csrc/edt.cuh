// Exact squared Euclidean distance transform on the GPU.
#pragma once

#include "common.cuh"

namespace rtk {

// One image for the kernels of rt_edt_noalloc, byte input (fg = byte != 0).
struct EdtArgs {
    const uint8_t *fg8;
    int64_t ld_in;
    int H, W;
    int32_t *d2;            // output
    int64_t ld_d2;
    uint16_t *g;            // workspace: vertical distance, H x W (stride W)
    int32_t *seg;           // workspace: 2 x nseg x W, first / last background row of each segment
    uint32_t *any_bg;       // workspace word
};

cudaError_t launch_edt(const EdtArgs &a, cudaStream_t s);

// A batch of images given as bits of their foreground, per 64 x 64 tile 64
// rows (bit = column; tiles row by row, image after image).
constexpr int kEdtMaxImgs = 32;
constexpr int kEdtSide = 64;
struct EdtBitsImage {
    int H, W, nx, ny;       // tiles per row, per column
    int tile_base;          // first tile of the image in the batch
    int band_base;          // first of its ny bands of 64 rows
    int32_t *d2;            // output
    int64_t ld_d2;
    uint32_t *cmask;        // workspace: per segment s and column c, bit i set where row 32 s + i is
                            // background (nseg x W)
    int32_t *seg;           // workspace: 2 x nseg x W, the last background row above and the first
                            // below each segment (-1: none)
};
struct EdtBitsBatch {
    int n, ntiles, nbands, maxW;
    const unsigned long long *bits;
    // control words, zeroed before the launches: a pixel is farther than the
    // near stage sees, a grid barrier's words, and which rows of each band
    uint32_t *far_any, *has_bg, *bar;
    unsigned long long *far_rows;
    int32_t *err;           // device status word
    EdtBitsImage img[kEdtMaxImgs];
};
// Workspace bytes of one H x W image (cmask and seg, 256-byte aligned pieces).
size_t edt_bits_workspace_bytes(int H, int W);
// Carves cmask and seg from base and appends the image.
void edt_bits_add(EdtBitsBatch &b, int H, int W, int32_t *d2, int64_t ld_d2, char *base);
cudaError_t launch_edt_bits_batch(const EdtBitsBatch &b, int num_sms, uint64_t timeout_ns, cudaStream_t s);

}  // namespace rtk
