// Exact squared Euclidean distance transform (input of the Pre-Watershed
// step, Section 5.1):
//     d2(p) = min over background q of (r_p - r_q)^2 + (c_p - c_q)^2.
// Separable form (the same decomposition as Meijster et al. 2000):
//     g(r, c)  = distance from (r, c) to the nearest background pixel of
//                column c (vertical pass),
//     d2(r, c) = min over c' of (c - c')^2 + g(r, c')^2 (horizontal pass).
// Vertical pass: columns are cut into 32-row segments; a first kernel
// records each segment's first and last background row, a second one walks
// every segment with the carries from the segments above and below.
// Horizontal pass: a CTA per row stages g in shared memory. For pixel c the
// candidate c' = c gives g(r,c)^2, and any c' with |c - c'| >= sqrt(best)
// cannot win, so the search runs outward from c and stops as soon as
// (c - c')^2 reaches the best value found. The result is exact for any
// input; the work per pixel grows with its distance, which is small on
// nuclei masks. rt_edt_noalloc runs these kernels.
//
// rt_edt and the chain work on bit planes in 64 x 64 tiles, where two facts
// save most of that work: most tiles of a nuclei mask have no foreground at
// all, and a distance below 32 needs only the 64 columns and 64 rows around
// the pixel. edt_near_kernel takes a CTA per tile: an empty tile is zeros;
// otherwise the foreground pixels are listed, and a thread per pixel looks at
// rows r - d and r + d for growing d: the windows of 64 background bits
// around the column are combined by OR, and the nearest column on either side
// is one count of leading or trailing zeros. It ends once d^2 reaches the best
// value. A pixel that finds nothing nearer than 32 (or lies in a tile
// that large objects fill) is written as 1024, no other distance of this stage, and flags its row, and edt_far_kernel (which
// returns at once if no row is flagged) searches for those pixels as above,
// with g from column masks of 32-row segments and never stored. Such images
// pay for both stages: discs of radius 300 take 95 -> 185 us at 1024 x 1024
// and 1.36 -> 1.81 ms at 4096 x 4096 against the kernels above, nuclei 76 -> 36
// at 4096 x 4096.
#include "edt.cuh"

namespace rtk {

constexpr int kSeg = 32;
constexpr uint16_t kInf = 0xFFFFu;

__device__ __forceinline__ bool edt_is_bg(const EdtArgs &a, int r, int c)
{
    return a.fg8[(int64_t)r * a.ld_in + c] == 0;
}

// thread per (column, segment): first / last background row in the segment
__global__ void edt_seg_kernel(EdtArgs a)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int s = blockIdx.y;
    if (c >= a.W) return;
    const int nseg = (int)ceil_div(a.H, kSeg);
    const int rb = s * kSeg, re = min(a.H, rb + kSeg);
    int first = -1, last = -1;
    for (int r = rb; r < re; ++r) {
        if (edt_is_bg(a, r, c)) {
            if (first < 0) first = r;
            last = r;
        }
    }
    a.seg[(int64_t)s * a.W + c] = first;
    a.seg[(int64_t)(nseg + s) * a.W + c] = last;
    if (first >= 0 && *a.any_bg == 0) atomicOr(a.any_bg, 1u);
}

// thread per (column, segment): g for the rows of the segment
__global__ void edt_col_kernel(EdtArgs a)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int s = blockIdx.y;
    if (c >= a.W) return;
    const int nseg = (int)ceil_div(a.H, kSeg);
    const int rb = s * kSeg, re = min(a.H, rb + kSeg);
    int above = -1;                      // last background row < rb
    for (int t = s - 1; t >= 0; --t) {
        const int v = a.seg[(int64_t)(nseg + t) * a.W + c];
        if (v >= 0) { above = v; break; }
    }
    int below = -1;                      // first background row >= re
    for (int t = s + 1; t < nseg; ++t) {
        const int v = a.seg[(int64_t)t * a.W + c];
        if (v >= 0) { below = v; break; }
    }
    int up[kSeg];
    int last = above;
    for (int r = rb; r < re; ++r) {
        if (edt_is_bg(a, r, c)) last = r;
        up[r - rb] = last;
    }
    int next = below;
    for (int r = re - 1; r >= rb; --r) {
        if (up[r - rb] == r) next = r;
        int d = 0x7fffffff;
        if (up[r - rb] >= 0) d = r - up[r - rb];
        if (next >= 0 && next - r < d) d = next - r;
        a.g[(int64_t)r * a.W + c] = d == 0x7fffffff ? kInf : (uint16_t)d;
    }
}

// d2 of one row from its g values in shared memory: for pixel c the search
// runs outward from c and stops once (c - c')^2 reaches the best value. A
// pixel that finds no background in any column gets -1 (the image has no
// background: a column with background gives every row a finite g there).
__device__ __forceinline__ void edt_row_search(const uint16_t *sg, int W, bool any, int32_t *out)
{
    for (int c = threadIdx.x; c < W; c += blockDim.x) {
        if (!any) {
            out[c] = -1;
            continue;
        }
        const int gc = sg[c];
        constexpr long long kNone = 0x7fffffffffffLL;
        long long best = gc == kInf ? kNone : (long long)gc * gc;
        for (int d = 1; (long long)d * d < best; ++d) {
            const int cl = c - d, cr = c + d;
            if (cl < 0 && cr >= W) break;
            if (cl >= 0) {
                const int g = sg[cl];
                if (g != kInf) {
                    const long long v = (long long)d * d + (long long)g * g;
                    if (v < best) best = v;
                }
            }
            if (cr < W) {
                const int g = sg[cr];
                if (g != kInf) {
                    const long long v = (long long)d * d + (long long)g * g;
                    if (v < best) best = v;
                }
            }
        }
        out[c] = best == kNone ? -1 : (int32_t)best;
    }
}

// CTA per row: exact minimum over columns with early termination
__global__ void edt_row_kernel(EdtArgs a)
{
    extern __shared__ uint16_t sg[];
    const int r = blockIdx.x;
    const uint16_t *grow = a.g + (int64_t)r * a.W;
    if ((a.W & 7) == 0) {   // rows 16-byte aligned: 8 values per load
        const uint4 *src = reinterpret_cast<const uint4 *>(grow);
        uint4 *dst = reinterpret_cast<uint4 *>(sg);
        for (int k = threadIdx.x; k < a.W / 8; k += blockDim.x) dst[k] = __ldcs(src + k);
    } else {
        for (int c = threadIdx.x; c < a.W; c += blockDim.x) sg[c] = grow[c];
    }
    __syncthreads();
    edt_row_search(sg, a.W, *a.any_bg != 0, a.d2 + (int64_t)r * a.ld_d2);
}

cudaError_t launch_edt(const EdtArgs &a, cudaStream_t s)
{
    const int nseg = (int)ceil_div(a.H, kSeg);
    cudaError_t e = cudaMemsetAsync(a.any_bg, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const size_t smem = (size_t)a.W * sizeof(uint16_t);
    if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(edt_row_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const dim3 g1((unsigned)ceil_div(a.W, 128), (unsigned)nseg);
    edt_seg_kernel<<<g1, 128, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    edt_col_kernel<<<g1, 128, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    edt_row_kernel<<<(unsigned)a.H, 256, smem, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------- bit-plane batch
namespace {

size_t piece(size_t bytes) { return (size_t)round_up((int64_t)bytes, 256); }

typedef unsigned long long u64;

// Threads per tile of the near stage: 256 up to kFewTiles tiles, where a
// tile's latency counts (900 x 900, dense nuclei: a call takes 20 us, with 128
// threads 23; equal at 4096 x 4096), 128 above (eight of these: 116 us, with
// 256 129).
constexpr int kFewTiles = 4096;
constexpr int kReach = 32;                       // rows and columns a tile looks beyond itself
constexpr uint32_t kNearMax = kReach * kReach;   // distances below are exact
constexpr int kFarThreads = 256;
constexpr int kRowWords = 4;                     // 32-bit words of a row: 32 + 64 + 32 columns
constexpr int kRowsIn = kEdtSide + 2 * kReach;

}  // namespace

size_t edt_bits_workspace_bytes(int H, int W)
{
    const size_t nseg = (size_t)ceil_div(H, kSeg);
    return piece(nseg * W * sizeof(uint32_t)) + piece(2 * nseg * W * sizeof(int32_t));
}

void edt_bits_add(EdtBitsBatch &b, int H, int W, int32_t *d2, int64_t ld_d2, char *base)
{
    EdtBitsImage &d = b.img[b.n++];
    const int64_t nseg = ceil_div(H, kSeg);
    d.H = H;
    d.W = W;
    d.nx = (int)ceil_div(W, kEdtSide);
    d.ny = (int)ceil_div(H, kEdtSide);
    d.d2 = d2;
    d.ld_d2 = ld_d2;
    d.cmask = reinterpret_cast<uint32_t *>(base);
    d.seg = reinterpret_cast<int32_t *>(base + piece((size_t)nseg * W * sizeof(uint32_t)));
    d.tile_base = b.ntiles;
    d.band_base = b.nbands;
    b.ntiles += d.nx * d.ny;
    b.nbands += d.ny;
    b.maxW = W > b.maxW ? W : b.maxW;
}

// ------------------------------------------------------------------- near
template <int NT>
__global__ void __launch_bounds__(NT) edt_near_kernel(const __grid_constant__ EdtBitsBatch b)
{
    start_early();
    __shared__ uint32_t bg[kRowsIn][kRowWords + 1];   // background bits of rows and columns -32 .. 95
    __shared__ uint16_t list[kEdtSide * kEdtSide];
    __shared__ __align__(16) uint16_t dist[kEdtSide * kEdtSide];
    __shared__ int s_n;
    __shared__ uint32_t s_far[2];   // rows with far pixels
    const int tile = blockIdx.x, t = threadIdx.x, lane = t & 31;
    int k = 0;
    while (k + 1 < b.n && tile >= b.img[k + 1].tile_base) ++k;
    const EdtBitsImage &d = b.img[k];
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const int r0 = ty * kEdtSide, c0 = tx * kEdtSide;
    const int nr = min(kEdtSide, d.H - r0), nc = min(kEdtSide, d.W - c0);
    const bool wide = nc == kEdtSide && (((uintptr_t)d.d2 | (uintptr_t)d.ld_d2 * 4u) & 15u) == 0;
    // own bits: thread = half a row
    uint32_t own = t < 2 * kEdtSide ? reinterpret_cast<const uint32_t *>(b.bits + (int64_t)tile * kEdtSide)[t] : 0u;
    if (!__syncthreads_or(own != 0u)) {
        if (wide) {
            for (int i = t >> 4; i < nr; i += NT / 16)
                reinterpret_cast<int4 *>(d.d2 + (int64_t)(r0 + i) * d.ld_d2 + c0)[t & 15] = make_int4(0, 0, 0, 0);
        } else if (nc == kEdtSide) {
            for (int i = t >> 4; i < nr; i += NT / 16)
                store_row64(d.d2 + (int64_t)(r0 + i) * d.ld_d2 + c0, t & 15, [](int) { return 0; });
        } else {
            for (int i = t >> 6; i < nr; i += NT / 64)
                if ((t & 63) < nc) d.d2[(int64_t)(r0 + i) * d.ld_d2 + c0 + (t & 63)] = 0;
        }
        return;
    }
    if (t == 0) s_n = 0, s_far[0] = s_far[1] = 0u;
    uint32_t any = 0;
    // background of the neighbourhood: word w of a row = columns c0 - 32 + 32 w; only pixels inside the image count
    for (int i = t; i < kRowsIn * kRowWords; i += NT) {
        const int y = i / kRowWords, w = i - y * kRowWords;
        const int r = r0 - kReach + y, c = c0 - kReach + 32 * w;
        uint32_t v = 0;
        if (r >= 0 && r < d.H && c >= 0 && c < d.W) {
            const int64_t nt = (int64_t)d.tile_base + (int64_t)(r / kEdtSide) * d.nx + c / kEdtSide;
            v = ~reinterpret_cast<const uint32_t *>(b.bits + nt * kEdtSide + r % kEdtSide)[c / 32 & 1];
            if (d.W - c < 32) v &= (1u << (d.W - c)) - 1u;
        }
        bg[y][w] = v;
        any |= v;
    }
    for (int i = t; i < kEdtSide * kEdtSide / 8; i += NT)
        reinterpret_cast<uint4 *>(dist)[i] = make_uint4(0u, 0u, 0u, 0u);
    const int some = __syncthreads_count(any != 0u);   // threads whose words hold background
    {
        const int n = __popc(own);
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        int at = 0;
        if (lane == 31) at = atomicAdd(&s_n, inc);
        at = __shfl_sync(0xffffffffu, at, 31) + inc - n;
        const int base = (t >> 1) * kEdtSide + (t & 1) * 32;
        while (own) {
            list[at++] = (uint16_t)(base + __ffs(own) - 1);
            own &= own - 1;
        }
    }
    __syncthreads();
    const int n = s_n;
    // A tile inside large objects, with background in a few words only, is
    // left to the far stage, whose step costs half as much where distances are
    // long (2048 x 2048, one pixel in a thousand background: 178 us in this
    // stage against 24). Nuclei never fill three quarters of a tile.
    const uint32_t reach = n > 3 * kEdtSide * kEdtSide / 4 && some < NT / 4 ? 0u : kNearMax;
    for (int i = t; i < n; i += NT) {
        const int p = list[i], r = p / kEdtSide, c = p % kEdtSide;
        // window: columns c - 32 .. c + 31 of the row = bits c .. c + 63
        const int w = c >> 5, sh = c & 31;
        uint32_t best = kNearMax;
        for (uint32_t dy = 0; dy * dy < min(best, reach); ++dy) {   // dy < 32
            const uint32_t *u = &bg[r + kReach - (int)dy][w], *v = &bg[r + kReach + (int)dy][w];
            const uint32_t a0 = u[0] | v[0], a1 = u[1] | v[1], a2 = u[2] | v[2];
            const uint32_t lo = __funnelshift_r(a0, a1, sh), hi = __funnelshift_r(a1, a2, sh);
            // nearest background left of the column (1 .. 32) and from it on (0 .. 31)
            const uint32_t dx = min((uint32_t)__clz((int)lo) + 1u, (uint32_t)__clz((int)__brev(hi)));
            best = min(best, dy * dy + dx * dx);
        }
        dist[p] = (uint16_t)best;
        if (best >= kNearMax && !((reinterpret_cast<volatile uint32_t *>(s_far)[r >> 5] >> (r & 31)) & 1u))
            atomicOr(&s_far[r >> 5], 1u << (r & 31));
    }
    __syncthreads();
    if (t == 0 && (s_far[0] | s_far[1])) {
        atomicOr(b.far_rows + d.band_base + ty, (u64)s_far[1] << 32 | s_far[0]);
        *b.far_any = 1u;
    }
    if (wide) {
        for (int i = t >> 4; i < nr; i += NT / 16) {
            const uint2 v = *reinterpret_cast<const uint2 *>(dist + i * kEdtSide + 4 * (t & 15));
            reinterpret_cast<int4 *>(d.d2 + (int64_t)(r0 + i) * d.ld_d2 + c0)[t & 15] =
                make_int4((int)(v.x & 0xffffu), (int)(v.x >> 16), (int)(v.y & 0xffffu), (int)(v.y >> 16));
        }
    } else if (nc == kEdtSide) {
        for (int i = t >> 4; i < nr; i += NT / 16)
            store_row64(d.d2 + (int64_t)(r0 + i) * d.ld_d2 + c0, t & 15,
                        [&](int c) { return (int)dist[i * kEdtSide + c]; });
    } else {
        for (int i = t >> 6; i < nr; i += NT / 64)
            if ((t & 63) < nc) d.d2[(int64_t)(r0 + i) * d.ld_d2 + c0 + (t & 63)] = dist[i * kEdtSide + (t & 63)];
    }
}

// -------------------------------------------------------------------- far
// Lane i loads the plane word (32 columns starting at 32 * wc) of row
// rb + i; 32 ballots turn the rows' words into the columns' masks, lane j
// getting column 32 * wc + j with bit i set where row rb + i is background.
// Rows past the end count as foreground.
__device__ __forceinline__ uint32_t seg_bg_mask(const EdtBitsBatch &b, const EdtBitsImage &a, int wc, int rb, int lane)
{
    const int r = rb + lane;
    const int64_t tile = (int64_t)a.tile_base + (int64_t)(r / kEdtSide) * a.nx + wc / 2;
    const uint32_t w = r < a.H ? __ldg(reinterpret_cast<const uint32_t *>(b.bits + tile * kEdtSide + r % kEdtSide) + (wc & 1))
                               : 0xffffffffu;
    uint32_t m = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t v = __ballot_sync(0xffffffffu, !((w >> j) & 1u));
        m = lane == j ? v : m;
    }
    return m;
}

// The rows that hold a pixel with no background nearer than 32, for the
// whole batch (cooperative; returns at once when there is none): column masks
// of every 32-row segment, the nearest background row above and below every
// segment, then a CTA per flagged row. An image without background is -1.
__global__ void __launch_bounds__(kFarThreads) edt_far_kernel(const __grid_constant__ EdtBitsBatch b, uint64_t timeout_ns)
{
    extern __shared__ uint16_t sg[];
    __shared__ int s_n;
    uint16_t *list = sg + b.maxW;
    if (*b.far_any == 0u) return;   // written by the launch before: the same for every CTA
    const int lane = threadIdx.x & 31;
    const int64_t gt = (int64_t)blockIdx.x * kFarThreads + threadIdx.x, nt = (int64_t)gridDim.x * kFarThreads;
    uint32_t any = 0;   // images with a background pixel
    for (int k = 0; k < b.n; ++k) {
        const EdtBitsImage &a = b.img[k];
        const int nseg = (int)ceil_div(a.H, kSeg), wpr = (a.W + 31) / 32;   // at most 32 images: a bit each in has_bg
        for (int64_t i = gt / 32; i < (int64_t)nseg * wpr; i += nt / 32) {
            const int s = (int)(i / wpr), wc = (int)(i - (int64_t)s * wpr), c = wc * 32 + lane;
            const uint32_t m = seg_bg_mask(b, a, wc, s * kSeg, lane);   // whole warp
            if (c < a.W) {
                a.cmask[(int64_t)s * a.W + c] = m;
                if (m) any |= 1u << k;
            }
        }
    }
    any = __reduce_or_sync(0xffffffffu, any);
    if (lane == 0 && (any & ~ld_acquire(b.has_bg))) atomicOr(b.has_bg, any);
    if (!grid_barrier(b.bar, gridDim.x, b.err, timeout_ns)) return;
    any = ld_acquire(b.has_bg);
    for (int k = 0; k < b.n; ++k) {
        if (!((any >> k) & 1u)) continue;
        const EdtBitsImage &a = b.img[k];
        const int nseg = (int)ceil_div(a.H, kSeg);
        for (int64_t i = gt; i < (int64_t)nseg * a.W; i += nt) {
            const int s = (int)(i / a.W), c = (int)(i - (int64_t)s * a.W);
            int above = -1;
            for (int q = s - 1; q >= 0; --q) {
                const uint32_t m = __ldcg(a.cmask + (int64_t)q * a.W + c);
                if (m) { above = q * kSeg + 31 - __clz((int)m); break; }
            }
            int under = -1;
            for (int q = s + 1; q < nseg; ++q) {
                const uint32_t m = __ldcg(a.cmask + (int64_t)q * a.W + c);
                if (m) { under = q * kSeg + __ffs((int)m) - 1; break; }
            }
            a.seg[(int64_t)s * a.W + c] = above;
            a.seg[(int64_t)(nseg + s) * a.W + c] = under;
        }
    }
    if (!grid_barrier(b.bar, gridDim.x, b.err, timeout_ns)) return;
    for (int k = 0; k < b.n; ++k) {
        const EdtBitsImage &a = b.img[k];
        const int nseg = (int)ceil_div(a.H, kSeg);
        for (int r = blockIdx.x; r < a.H; r += gridDim.x) {
            if (!((b.far_rows[a.band_base + r / kEdtSide] >> (r % kEdtSide)) & 1ull)) continue;   // whole CTA
            if (!((any >> k) & 1u)) {
                for (int c = threadIdx.x; c < a.W; c += kFarThreads) a.d2[(int64_t)r * a.ld_d2 + c] = -1;
                continue;
            }
            const int s = r / kSeg, i = r % kSeg, rb = s * kSeg;
            int32_t *out = a.d2 + (int64_t)r * a.ld_d2;
            if (threadIdx.x == 0) s_n = 0;
            __syncthreads();
            // g of the row, and the columns to search
#pragma unroll 4
            for (int c = threadIdx.x; c < a.W; c += kFarThreads) {
                const uint32_t m = __ldcg(a.cmask + (int64_t)s * a.W + c);
                uint16_t g = 0;
                if (!((m >> i) & 1u)) {
                    const uint32_t upto = m & (0xffffffffu >> (31 - i));   // rows rb .. r
                    const uint32_t from = m & (0xffffffffu << i);          // rows r .. rb + 31
                    const int up = upto ? rb + 31 - __clz((int)upto) : __ldcg(a.seg + (int64_t)s * a.W + c);
                    const int dn = from ? rb + __ffs((int)from) - 1 : __ldcg(a.seg + (int64_t)(nseg + s) * a.W + c);
                    int v = 0x7fffffff;
                    if (up >= 0) v = r - up;
                    if (dn >= 0 && dn - r < v) v = dn - r;
                    g = v == 0x7fffffff ? kInf : (uint16_t)v;
                    if (out[c] == (int32_t)kNearMax) list[atomicAdd(&s_n, 1)] = (uint16_t)c;
                }
                sg[c] = g;
            }
            __syncthreads();
            // sides are at most 32768: d^2 + g^2 < 2^31 is exact in 32 bits
            for (int q = threadIdx.x; q < s_n; q += kFarThreads) {
                const int c = list[q];
                const uint32_t gc = sg[c];
                uint32_t best = gc == kInf ? 0xffffffffu : gc * gc;
                for (uint32_t e = 1; e * e < best; ++e) {
                    const int cl = c - (int)e, cr = c + (int)e;
                    if (cl < 0 && cr >= a.W) break;
                    if (cl >= 0) {
                        const uint32_t g = sg[cl];
                        if (g != kInf) best = min(best, e * e + g * g);
                    }
                    if (cr < a.W) {
                        const uint32_t g = sg[cr];
                        if (g != kInf) best = min(best, e * e + g * g);
                    }
                }
                out[c] = (int32_t)best;
            }
            __syncthreads();
        }
    }
}

cudaError_t launch_edt_bits_batch(const EdtBitsBatch &b, int num_sms, uint64_t timeout_ns, cudaStream_t s)
{
    if (b.n < 1 || b.n > kEdtMaxImgs) return cudaErrorInvalidValue;
    if (b.ntiles <= kFewTiles) launch_early(edt_near_kernel<256>, (unsigned)b.ntiles, 256, 0, s, b);
    else launch_early(edt_near_kernel<128>, (unsigned)b.ntiles, 128, 0, s, b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = 2 * (size_t)b.maxW * sizeof(uint16_t);
    if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(edt_far_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, edt_far_kernel, kFarThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t rows = (int64_t)b.nbands * kEdtSide;
    int grid = per_sm * num_sms;
    if (grid > rows) grid = (int)rows;
    EdtBitsBatch bb = b;
    void *args[] = {&bb, &timeout_ns};
    return cudaLaunchCooperativeKernel((const void *)edt_far_kernel, dim3((unsigned)grid), dim3(kFarThreads), args, smem, s);
}

}  // namespace rtk
