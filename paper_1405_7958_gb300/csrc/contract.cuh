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
// The global stage's units: a quarter of a tile's nodes (at most 63) and of
// the forest between them (at most 63 edges), and half of its right or lower
// seam (at most 32 diagonals, one per 2 x 2 window, and 32 straight pairs).
constexpr int kCtUnits = 4;
constexpr int kCtUnitNodes = kCtNodes / kCtUnits;
constexpr int kCtUnitEdges = 128;
constexpr int kCtMaxImgs = 32;
constexpr int64_t kCtMaxTiles = int64_t(1) << 20;   // an edge names its nodes in 28 bits each

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
};

// Up to kCtMaxImgs images and the workspace of the batch, passed by value.
struct CtBatch {
    int n, ntiles;
    uint16_t *plane;         // per pixel (tile by tile): node of the tile << 8 | bound
    uint32_t *cnt;           // per tile: nodes | forest edges << 16
    unsigned long long *link;   // per node: its parent and link weight, or a root's state (contract.cu)
    unsigned long long *best;   // per node: its best edge of the round
    uint32_t *S;             // per node that joined another: its sources' best value
    uint32_t *act;           // per node slot: the warps' lists of roots still open
    unsigned long long *edge;   // per edge slot: weight and nodes
    uint8_t *ecnt;           // per unit: its edges
    uint16_t *rim;           // per tile: its upper row, lower row, left and right column: node << 8 | I
    unsigned long long *bits;   // nullable: B = (R < threshold), per tile 64 rows, bit = column
    uint32_t *ctl;           // kCtCtlWords control words, zeroed before the launches
    int32_t *err;            // device status word
    CtImage img[kCtMaxImgs];
};

constexpr int kCtCtlBar = 0;      // grid barrier: arrivals, open roots handed in (64 bits)
constexpr int kCtCtlWords = 8;

void ct_plan_image(CtBatch &b, const uint8_t *marker, int64_t ld_marker, const uint8_t *mask, int64_t ld_mask, int H,
                   int W, int h_offset);
// local contraction of every tile, then the global contraction (cooperative)
cudaError_t launch_contract(const CtBatch &b, int num_sms, uint64_t timeout_ns, cudaStream_t s);
// R into every image's out and B = (R < threshold) into bits (either may be NULL)
cudaError_t launch_contract_out(const CtBatch &b, int threshold, cudaStream_t s);

}  // namespace rtk
