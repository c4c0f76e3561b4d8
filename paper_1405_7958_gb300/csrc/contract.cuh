// Reconstruction by dilation by contraction (contract.cu): data structures
// shared with the host entry points (api.cu).
#pragma once

#include "common.cuh"

namespace rtk {

constexpr int kCtSide = 64;                    // tiles of 64 x 64 pixels
constexpr int kCtPx = kCtSide * kCtSide;
// Node slots per tile. A node is a cluster that holds a pixel on the tile's
// rim, which has 252 pixels; slot 255 of a pixel's entry means "no node".
constexpr int kCtNodes = 256;
constexpr uint32_t kCtNoNode = 255u;
// Edge slots per tile: at most 251 edges of the forest between its nodes,
// and at most 257 across its right and lower seams (per seam one diagonal
// for each of its 2 x 2 windows and one straight pair per pixel).
constexpr int kCtEdges = 512;
constexpr int kCtMaxImgs = 32;
constexpr int64_t kCtMaxTiles = int64_t(1) << 23;   // edge slots are numbered in 32 bits

struct CtImage {
    const uint8_t *marker;   // NULL: derived from the mask with h_offset
    int64_t ld_marker;
    const uint8_t *mask;
    int64_t ld_mask;
    int H, W;
    int nx, ny;              // tiles per row, per column
    int tile_base;           // first tile of the image in the batch (row by row)
    int h_offset;
    uint8_t *out;            // nullable: R, H x W, stride ld_out
    int64_t ld_out;
    uint8_t *bin;            // nullable: B = (R < threshold), H x W, stride ld_bin
    int64_t ld_bin;
};

// Up to kCtMaxImgs images and the workspace of the batch, passed by value.
struct CtBatch {
    int n, ntiles;
    uint16_t *plane;         // per pixel (tile by tile): node of the tile << 8 | bound
    uint32_t *cnt;           // per tile: nodes | forest edges << 16
    uint32_t *S;             // per node: best marker value that reaches it; bit 31: final
    unsigned long long *link;   // per node: weight << 32 | parent (itself: a root)
    unsigned long long *best;   // per node: its best edge of the round
    uint32_t *act;           // per node slot: the warps' lists of roots still open
    uint32_t *ea, *eb;       // per edge slot: its nodes
    uint8_t *ew;             //                its weight
    uint32_t *ctl;           // kCtCtlWords control words, zeroed before the launches
    int32_t *err;            // device status word
    CtImage img[kCtMaxImgs];
};

constexpr int kCtCtlBar = 0;      // grid barrier: arrivals, generation
constexpr int kCtCtlOpen = 2;     // three counters of open roots, used in turn
constexpr int kCtCtlWords = 8;

void ct_plan_image(CtBatch &b, const uint8_t *marker, int64_t ld_marker, const uint8_t *mask, int64_t ld_mask, int H,
                   int W, int h_offset);
// local contraction of every tile, then the global contraction (cooperative)
cudaError_t launch_contract(const CtBatch &b, int num_sms, uint64_t timeout_ns, cudaStream_t s);
// R and B = (R < threshold) into every image's out / bin (either may be NULL)
cudaError_t launch_contract_out(const CtBatch &b, int threshold, cudaStream_t s);

}  // namespace rtk
