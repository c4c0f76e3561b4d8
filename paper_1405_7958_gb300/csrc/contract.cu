// ReconToNuclei (Section 5.1 of the Region Templates paper): grayscale
// morphological reconstruction by dilation, 8-connected, by contraction.
//
// R(p) is the best value that reaches p: the maximum over all pixels q and
// all paths from q to p of min(J(q), the smallest I on the path). That is a
// widest-path problem: take the pixels as nodes, an edge of weight
// min(I(p), I(q)) between neighbours, and a source S(p) = min(J(p), I(p)) at
// every pixel. Widest paths survive contraction along maximum spanning
// forest edges (Boruvka's algorithm): let C be a cluster with root r whose
// best edge to another cluster C' (root r') weighs w.
//   * If S(C) = max of the members' sources is >= w, nothing better can
//     enter: R(r) = S(C) is final.
//   * Otherwise R(r) = min(w, R(r')) exactly, and C joins C' below r' with
//     link weight w; S(C') becomes max(S(C'), S(C)).
// Every pixel p keeps its cluster's root and the smallest weight b on its
// way there, and in the end R(p) = min(b, R(root)). Instead of carrying
// values pixel by pixel across the image, each round at least halves the
// open clusters, so the chain of dependent steps is logarithmic.
//
// Three facts make the first steps cheap:
//   * a pixel with a neighbour q of I(q) >= I(p) satisfies R(p) =
//     min(I(p), R(q)) for any such q, so the first contraction is one
//     3 x 3 maximum: every pixel points at its largest neighbour (ties by
//     raster order) and only the local maxima remain as clusters (one in
//     nine pixels of a noisy image);
//   * an edge that is the smallest of a triangle is in no maximum spanning
//     forest. In a 2 x 2 window all four pixels are neighbours, so of its
//     six edges only the three at its largest pixel can matter; and of two
//     edges from one pixel into one cluster only the larger can.
//
// Launches: ct_local_kernel contracts every 64 x 64 tile in shared memory
// until each open cluster's best edge leaves the tile; what is left of a
// tile are its nodes (clusters that touch its rim, about 50 of 4096 pixels
// on nuclei tiles), the forest between them, and 2 bytes per pixel (node,
// bound). ct_global_kernel adds the edges across the seams and contracts
// the nodes of the whole batch (one persistent cooperative launch).
// ct_out_kernel writes R.
//
// Measured on one GB300 against the directional sweeps (rt_segment_batch or
// rt_reconstruct, whole call): 512 x 512 reconstruction 155 us against 341;
// one 4096 x 4096 tile 0.81 ms against 1.40; eight of them 4.84 ms against
// 5.69; a 16384 x 16384 slide 9.4 ms against 10.3. So the contraction runs
// wherever the call leaves the schedule to the library.
#include "contract.cuh"

namespace rtk {

namespace {

constexpr int kT = 256;                    // threads of the local kernel
constexpr int kWarps = kT / 32;
constexpr int kStride = 68;                // words per row of the pixel array
// Pixel (r, c) of the tile, -1 <= r, c <= 64 (one pixel of halo), is word
// (r + 1) * kStride + c + 4; column 64 falls on the unused first word of the
// next row. Indices grow in raster order.
constexpr int kPixWords = (kCtSide + 2) * kStride + 4;
// Roots of the first contraction: local maxima in the tile, no two adjacent.
constexpr int kRoots = 1024;
// Edges between clusters after the triangle rule: one diagonal in each of
// the 65 x 65 windows that meet the tile, at most 32 straight pairs per row
// or column of windows (2 x 32 x 65), less the tree edges of the first
// contraction that are among them (at least 3072 - 252).
constexpr int kList = 5632;
constexpr size_t kLocalSmem = sizeof(uint32_t) * (kPixWords + kList + 2 * kRoots);

// A pixel's word: I << 24 | index << 11 | low. Words order pixels by (I,
// raster index). A pixel outside the image is 0, below every pixel. low of a
// pixel of the tile: first the step to its parent + 128, then kIn | cluster;
// low of a halo pixel: its row and column parity (no two of a 2 x 2 window
// alike).
constexpr uint32_t kLow = 0x7ffu, kIn = 0x400u, kIdx = 0x3ffu;

// An edge's key: I << 24 | index << 11 of its smaller pixel, I of the larger
// one << 3, direction from the smaller to the larger (0..7 in raster order:
// NW N NE W E SW S SE). Keys order the edges totally, by (smaller, larger)
// pixel, in the same way in every tile that sees them. 0: none.
__device__ __forceinline__ int step_of(uint32_t key)
{
    // bytes -69 -68 -67 -1 | 1 67 68 69
    return (int)(int8_t)__byte_perm(0xffbdbcbbu, 0x45444301u, key & 7u);
}
__device__ __forceinline__ uint32_t edge_key(uint32_t lo, uint32_t hi, uint32_t dir)
{
    return (lo & ~kLow) | ((hi >> 24) << 3) | dir;
}

// A cluster's link word: root: kRootBit | S; else weight << 16 | parent.
constexpr uint32_t kRootBit = 0x80000000u;
__device__ __forceinline__ uint32_t root_of(const volatile uint32_t *nlink, uint32_t k)
{
    const uint32_t v = nlink[k];   // links point at the root between rounds
    return (v & kRootBit) ? k : (v & 0xffffu);
}

__device__ __forceinline__ const CtImage &ct_image(const CtBatch &b, int t)
{
    int k = 0;
    while (k + 1 < b.n && t >= b.img[k + 1].tile_base) ++k;
    return b.img[k];
}

__device__ __forceinline__ uint32_t max3(uint32_t a, uint32_t b, uint32_t c) { return max(a, max(b, c)); }

}  // namespace

// ------------------------------------------------------------------ local
template <bool MARKER>
__global__ void __launch_bounds__(kT, 4) ct_local_kernel(const __grid_constant__ CtBatch b)
{
    extern __shared__ __align__(16) uint32_t ct_smem[];
    uint32_t *W = ct_smem;                      // pixel words
    uint32_t *list = W + kPixWords;             // edge keys
    volatile uint32_t *best = list + kList;     // per cluster: its best edge
    volatile uint32_t *nlink = best + kRoots;   // per cluster: link word
    volatile uint32_t *VW = W;
    __shared__ int s_roots, s_edges, s_nodes, s_forest;

    const int tile = blockIdx.x;
    const CtImage &d = ct_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const int r0 = ty * kCtSide, c0 = tx * kCtSide;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t below = (1u << lane) - 1u;

    if (t == 0) s_roots = s_edges = s_nodes = s_forest = 0;

    // ---- load the tile and its halo
    {
        const bool wide = (((uintptr_t)d.mask | (uintptr_t)d.ld_mask) & 3u) == 0;
        const int q = t & 15;
        const int c = c0 + 4 * q;
        for (int rr = t >> 4; rr < kCtSide + 2; rr += kT / 16) {
            const int r = r0 + rr - 1;
            const int n = (r >= 0 && r < d.H) ? min(4, d.W - c) : 0;   // may be negative: none
            uint32_t v = 0;
            const uint8_t *p = d.mask + (int64_t)r * d.ld_mask + c;
            if (n == 4 && wide) {
                v = __ldg(reinterpret_cast<const uint32_t *>(p));
            } else {
                for (int k = 0; k < n; ++k) v |= (uint32_t)__ldg(p + k) << (8 * k);
            }
            const int idx = rr * kStride + 4 * q + 4;
            const bool halo = rr == 0 || rr == kCtSide + 1;
            uint32_t o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t low = halo ? (uint32_t)((rr & 1) << 1 | (k & 1)) : 0u;
                o[k] = k < n ? ((v >> (8 * k)) & 0xffu) << 24 | (uint32_t)(idx + k) << 11 | low : 0u;
            }
            *reinterpret_cast<uint4 *>(W + idx) = make_uint4(o[0], o[1], o[2], o[3]);
        }
        if (t < 2 * (kCtSide + 2)) {
            const int rr = t >> 1, right = t & 1;
            const int r = r0 + rr - 1, ch = right ? c0 + kCtSide : c0 - 1;
            const int idx = rr * kStride + (right ? kCtSide + 4 : 3);
            uint32_t w = 0;
            if (r >= 0 && r < d.H && ch >= 0 && ch < d.W)
                w = (uint32_t)__ldg(d.mask + (int64_t)r * d.ld_mask + ch) << 24 | (uint32_t)idx << 11 |
                    (uint32_t)((rr & 1) << 1 | (right ? 0 : 1));
            W[idx] = w;
        }
    }
    __syncthreads();

    // ---- first contraction: every pixel points at the largest pixel of its
    // 3 x 3 neighbourhood in the tile. Thread = column, 16 rows of one strip.
    // Only the low bits of words change here, which no comparison sees.
    const int c = t & (kCtSide - 1), rs = (t >> 6) * 16;
    uint32_t rootmask = 0;
    {
        auto row3 = [&](int r, uint32_t &ctr) -> uint32_t {
            if (r < 0 || r >= kCtSide) {
                ctr = 0u;
                return 0u;
            }
            const volatile uint32_t *x = VW + (r + 1) * kStride + c + 4;
            ctr = x[0];
            const uint32_t l = c > 0 ? x[-1] : 0u, rt = c < kCtSide - 1 ? x[1] : 0u;
            return max3(l, ctr, rt);
        };
        uint32_t ca, cb, cc;
        uint32_t ha = row3(rs - 1, ca), hb = row3(rs, cb);
#pragma unroll 4
        for (int j = 0; j < 16; ++j) {
            const uint32_t hc = row3(rs + j + 1, cc);
            const uint32_t m = max3(ha, hb, hc);
            if (cb) {
                if (m == cb) {
                    rootmask |= 1u << j;
                } else {
                    const int idx = (rs + j + 1) * kStride + c + 4;
                    const int st = (int)((m >> 11) & 0x1fffu) - idx;
                    VW[idx] = (cb & ~kLow) | (uint32_t)(st + 128);
                }
            }
            ha = hb;
            hb = hc;
            cb = cc;
        }
    }
    {
        const int n = __popc(rootmask);
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        int base = 0;
        if (lane == 31) base = atomicAdd(&s_roots, inc);
        uint32_t k = (uint32_t)(__shfl_sync(0xffffffffu, base, 31) + inc - n);
        while (rootmask) {
            const int j = __ffs(rootmask) - 1;
            rootmask &= rootmask - 1;
            const int idx = (rs + j + 1) * kStride + c + 4;
            const uint32_t w = VW[idx];
            // the derived marker's largest value in the cluster is at its maximum
            const uint32_t I = w >> 24;
            const uint32_t S = MARKER ? 0u : (I > (uint32_t)d.h_offset ? I - (uint32_t)d.h_offset : 0u);
            VW[idx] = (w & ~kLow) | kIn | k;
            nlink[k] = kRootBit | S;
            best[k] = 0u;
            ++k;
        }
    }
    __syncthreads();
    const int nr = s_roots;

    // ---- every pixel's cluster: follow the steps uphill. A finished pixel's
    // word ends the walk of those that come through it.
    {
        bool bad = false;
#pragma unroll 4
        for (int j = 0; j < 16; ++j) {
            const int r = rs + j, idx = (r + 1) * kStride + c + 4;
            uint32_t w = VW[idx];
            if (!w) continue;
            if (!(w & kIn)) {
                int x = idx;
                uint32_t v = w;
                for (int n = 0; n < kCtPx && !(v & kIn); ++n) {
                    x += (int)(v & 0xffu) - 128;
                    v = VW[x];
                }
                w = (w & ~kLow) | (v & kLow);
                VW[idx] = w;
            }
            const uint32_t k = w & kIdx, I = w >> 24;
            const int gr = r0 + r, gc = c0 + c;
            uint32_t *sk = const_cast<uint32_t *>(nlink + k);
            if (MARKER) {
                const uint32_t J = __ldg(d.marker + (int64_t)gr * d.ld_marker + gc);
                bad |= J > I;
                const uint32_t v = kRootBit | min(J, I);
                if (nlink[k] < v) atomicMax(sk, v);
            } else if (gr == 0 || gr == d.H - 1 || gc == 0 || gc == d.W - 1) {
                atomicMax(sk, kRootBit | I);
            }
        }
        if (MARKER && bad) raise_status(b.err, RT_EMARKER);
    }
    __syncthreads();

    // ---- edges between clusters that pass the triangle rule. The owner of
    // an edge is the window whose upper left pixel is (r, c).
    {
        // larger pixel hi, smaller lo; x: a common neighbour. The edge can go
        // if x is above both, or above lo and in lo's cluster.
        auto drops = [&](uint32_t x, uint32_t lo, uint32_t hi) {
            return x > (((x ^ lo) & kLow) == 0u ? lo : hi);
        };
        auto joins = [&](uint32_t lo, uint32_t hi) {   // both exist, one in the tile, not one cluster
            return lo && ((lo | hi) & kIn) && ((lo ^ hi) & kLow);
        };
        auto diagonal = [&](uint32_t m, uint32_t mr, uint32_t dn, uint32_t dr) -> uint32_t {
            const bool main = max(m, dr) > max(mr, dn);
            const uint32_t p = main ? m : mr, q = main ? dr : dn;   // p in the upper row
            const uint32_t x = main ? mr : m, y = main ? dn : dr;
            const uint32_t lo = min(p, q), hi = max(p, q);
            if (!joins(lo, hi) || drops(x, lo, hi) || drops(y, lo, hi)) return 0u;
            const uint32_t dir = lo == p ? (main ? 7u : 5u) : (main ? 0u : 2u);
            return edge_key(lo, hi, dir);
        };
        auto straight = [&](uint32_t p, uint32_t q, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                            uint32_t dp, uint32_t dq) -> uint32_t {
            const uint32_t lo = min(p, q), hi = max(p, q);
            if (!joins(lo, hi) || drops(x0, lo, hi) || drops(x1, lo, hi) || drops(x2, lo, hi) || drops(x3, lo, hi))
                return 0u;
            return edge_key(lo, hi, lo == p ? dp : dq);
        };
        auto append = [&](uint32_t e0, uint32_t e1, uint32_t e2) {   // whole warp
            const int n = (e0 != 0u) + (e1 != 0u) + (e2 != 0u);
            const uint32_t b0 = __ballot_sync(0xffffffffu, n & 1), b1 = __ballot_sync(0xffffffffu, n & 2);
            const int total = __popc(b0) + 2 * __popc(b1);
            if (total == 0) return;
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_edges, total);
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(b0 & below) + 2 * __popc(b1 & below);
            if (at + n > kList) return;   // cannot happen (see kList)
            if (e0) list[at++] = e0;
            if (e1) list[at++] = e1;
            if (e2) list[at] = e2;
        };
        const int first = rs == 0 ? -1 : rs;
        const uint32_t *x = W + (first + 1) * kStride + c + 4;
        uint32_t u = 0, ur = 0;                       // row above (only rows >= 0 use it)
        if (first > 0) u = x[-kStride], ur = x[1 - kStride];
        uint32_t ml = x[-1], m = x[0], mr = x[1];
        for (int r = first; r < rs + 16; ++r) {
            x += kStride;
            const uint32_t dl = x[-1], dn = x[0], dr = x[1];
            const uint32_t e0 = diagonal(m, mr, dn, dr);
            const uint32_t e1 = straight(m, mr, u, ur, dn, dr, 4u, 3u);
            const uint32_t e2 = straight(m, dn, ml, mr, dl, dr, 6u, 1u);
            append(e0, e1, e2);
            u = m, ur = mr;
            ml = dl, m = dn, mr = dr;
        }
        // the windows left of the tile (c = -1)
        if (warp < 3) {
            const int r = t - 1;
            uint32_t e0 = 0, e1 = 0;
            if (r < kCtSide) {
                const uint32_t *y = W + (r + 1) * kStride + 3;
                e0 = diagonal(y[0], y[1], y[kStride], y[kStride + 1]);
                if (r >= 0) e1 = straight(y[0], y[1], y[-kStride], y[1 - kStride], y[kStride], y[kStride + 1], 4u, 3u);
            }
            append(e0, e1, 0u);
        }
    }
    __syncthreads();

    // ---- contraction rounds. Each warp keeps a range of the list and
    // compacts it in place: edges inside one cluster leave.
    int start, cnt;
    {
        const int n = min(s_edges, kList);
        const int per = (((n + kWarps - 1) / kWarps) + 31) & ~31;
        start = min(warp * per, n);
        cnt = min(per, n - start);
    }
    auto edge_pass = [&]() {
        int kept = 0;
        for (int i = 0; i < cnt; i += 32) {
            const bool have = i + lane < cnt;
            const uint32_t key = have ? list[start + i + lane] : 0u;
            uint32_t ra = ~0u, rb = ~0u;
            if (have) {
                const int lo = (int)((key >> 11) & 0x1fffu);
                const uint32_t wl = W[lo], wh = W[lo + step_of(key)];
                if (wl & kIn) ra = root_of(nlink, wl & kIdx);
                if (wh & kIn) rb = root_of(nlink, wh & kIdx);
            }
            const bool keep = ra != rb;
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                list[start + kept + __popc(m & below)] = key;
                if (ra != ~0u && best[ra] < key) atomicMax(const_cast<uint32_t *>(best + ra), key);
                if (rb != ~0u && best[rb] < key) atomicMax(const_cast<uint32_t *>(best + rb), key);
            }
            kept += __popc(m);
            __syncwarp();
        }
        cnt = kept;
    };
    edge_pass();
    __syncthreads();
    for (;;) {
        // decide: S << 24 | weight << 16 | parent, parent 0xffff: stays
        uint32_t dec[kRoots / kT];
        int any = 0;
#pragma unroll
        for (int q = 0; q < kRoots / kT; ++q) {
            const uint32_t k = t + q * kT;
            dec[q] = 0xffffu;
            if (k >= (uint32_t)nr) continue;
            const uint32_t v = nlink[k], key = best[k];
            if (!(v & kRootBit) || !key) continue;
            const uint32_t w = key >> 24, S = v & 0xffu;
            if (S >= w) continue;                                  // final
            const int lo = (int)((key >> 11) & 0x1fffu);
            const uint32_t wl = W[lo], wh = W[lo + step_of(key)];
            if (!(wl & wh & kIn)) continue;                        // its best edge leaves the tile
            const uint32_t ra = root_of(nlink, wl & kIdx);
            const uint32_t o = ra == k ? root_of(nlink, wh & kIdx) : ra;
            if (k < o && best[o] == key && (nlink[o] & 0xffu) < w) continue;   // o joins this one
            dec[q] = S << 24 | w << 16 | o;
            any = 1;
        }
        if (!__syncthreads_or(any)) break;
#pragma unroll
        for (int q = 0; q < kRoots / kT; ++q)
            if ((dec[q] & 0xffffu) != 0xffffu) nlink[t + q * kT] = dec[q] & 0xffffffu;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kRoots / kT; ++q) {
            const uint32_t k = t + q * kT;
            if (k >= (uint32_t)nr) continue;
            uint32_t v = nlink[k];
            if (v & kRootBit) {
                best[k] = 0u;
                continue;
            }
            uint32_t w = v >> 16, x = v & 0xffffu;
            for (int n = 0; n < kRoots; ++n) {
                v = nlink[x];
                if (v & kRootBit) break;
                w = min(w, v >> 16);
                x = v & 0xffffu;
            }
            nlink[k] = w << 16 | x;
            if ((dec[q] & 0xffffu) != 0xffffu) atomicMax(const_cast<uint32_t *>(nlink + x), kRootBit | dec[q] >> 24);
        }
        __syncthreads();
        edge_pass();
        __syncthreads();
    }

    // ---- nodes: the clusters with a pixel on a side that has a neighbour
    // tile. best[k] becomes 1 + the node of root k, 0 for the others (which
    // are final: no edge of theirs leaves the tile).
    for (int k = t; k < nr; k += kT) best[k] = 0u;
    __syncthreads();
    {
        const int side = t >> 6, i = t & 63;
        const bool open = side == 0 ? ty > 0 : side == 1 ? ty + 1 < d.ny : side == 2 ? tx > 0 : tx + 1 < d.nx;
        const int r = side == 0 ? 0 : side == 1 ? kCtSide - 1 : i, cc = side < 2 ? i : side == 2 ? 0 : kCtSide - 1;
        const uint32_t w = W[(r + 1) * kStride + cc + 4];
        if (open && w) best[root_of(nlink, w & kIdx)] = 1u;
    }
    __syncthreads();
    for (int k0 = warp * 32; k0 < nr; k0 += kT) {
        const int k = k0 + lane;
        const bool f = k < nr && best[k] != 0u;
        const uint32_t m = __ballot_sync(0xffffffffu, f);
        if (!m) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(&s_nodes, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (f) best[k] = 1u + base + __popc(m & below);
    }
    __syncthreads();
    const int nn = s_nodes;
    // the edges between nodes stay (as node | node << 8 | weight << 16); an
    // edge from a node to a final cluster f gives the node min(weight, R(f))
    // as a source of its own
    {
        int kept = 0;
        for (int i = 0; i < cnt; i += 32) {
            uint32_t e = 0;
            bool keep = false;
            if (i + lane < cnt) {
                const uint32_t key = list[start + i + lane];
                const int lo = (int)((key >> 11) & 0x1fffu);
                const uint32_t wl = W[lo], wh = W[lo + step_of(key)];
                if (wl & wh & kIn) {
                    const uint32_t ra = root_of(nlink, wl & kIdx), rb = root_of(nlink, wh & kIdx);
                    const uint32_t na = best[ra], nb = best[rb], w = key >> 24;
                    keep = na && nb;
                    e = (na - 1u) | (nb - 1u) << 8 | w << 16;
                    if (na && !nb) atomicMax(const_cast<uint32_t *>(nlink + ra), kRootBit | min(w, nlink[rb] & 0xffu));
                    if (nb && !na) atomicMax(const_cast<uint32_t *>(nlink + rb), kRootBit | min(w, nlink[ra] & 0xffu));
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) list[start + kept + __popc(m & below)] = e;
            kept += __popc(m);
            __syncwarp();
        }
        cnt = kept;
    }
    __syncthreads();
    // per cluster: node << 8 | bound (kCtNoNode: the value itself)
    {
        uint32_t tab[kRoots / kT];
#pragma unroll
        for (int q = 0; q < kRoots / kT; ++q) {
            const uint32_t k = t + q * kT;
            tab[q] = 0u;
            if (k >= (uint32_t)nr) continue;
            uint32_t v = nlink[k], w = 255u, x = k;
            if (!(v & kRootBit)) {
                w = v >> 16;
                x = v & 0xffffu;
                v = nlink[x];
            }
            const uint32_t n = best[x];
            tab[q] = n ? (n - 1u) << 8 | w : kCtNoNode << 8 | min(w, v & 0xffu);
            if (n && x == k) {
                const uint32_t g = (uint32_t)tile * kCtNodes + n - 1u;
                b.S[g] = v & 0xffu;
                b.link[g] = 255ull << 32 | g;
                b.best[g] = 0ull;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kRoots / kT; ++q) {
            const uint32_t k = t + q * kT;
            if (k < (uint32_t)nr) nlink[k] = tab[q];
        }
        // the forest rounds below use best as two arrays of 256 words
        if (t < nn) best[t] = t;
        best[kT + t] = 0u;
    }
    __syncthreads();
    {
        uint16_t *o = b.plane + (int64_t)tile * kCtPx + rs * kCtSide + c;
#pragma unroll 4
        for (int j = 0; j < 16; ++j) {
            const uint32_t w = W[(rs + j + 1) * kStride + c + 4];
            const uint32_t e = nlink[w & kIdx];
            if (w) o[j * kCtSide] = (uint16_t)((e & 0xff00u) | min(e & 0xffu, w >> 24));
        }
    }

    // ---- maximum spanning forest of the nodes (only these edges can matter)
    volatile uint32_t *comp = best, *fb = best + kT;
    for (;;) {
        int kept = 0;
        for (int i = 0; i < cnt; i += 32) {
            const bool have = i + lane < cnt;
            const uint32_t e = have ? list[start + i + lane] : 0u;
            uint32_t ca = 0, cb = 0;
            if (have) ca = comp[e & 0xffu], cb = comp[(e >> 8) & 0xffu];
            const bool keep = ca != cb;
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const uint32_t pos = start + kept + __popc(m & below);
                list[pos] = e;
                const uint32_t key = ((e >> 16) << 13 | pos) + 1u;
                if (fb[ca] < key) atomicMax(const_cast<uint32_t *>(fb + ca), key);
                if (fb[cb] < key) atomicMax(const_cast<uint32_t *>(fb + cb), key);
            }
            kept += __popc(m);
            __syncwarp();
        }
        cnt = kept;
        __syncthreads();
        uint32_t join = ~0u;
        if (t < nn && comp[t] == (uint32_t)t && fb[t]) {
            const uint32_t key = fb[t], e = list[(key - 1u) & 0x1fffu];
            const uint32_t ca = comp[e & 0xffu], o = ca == (uint32_t)t ? comp[(e >> 8) & 0xffu] : ca;
            if (!((uint32_t)t < o && fb[o] == key)) {
                join = o;
                const int64_t g = (int64_t)tile * kCtEdges + atomicAdd(&s_forest, 1);
                b.ea[g] = (uint32_t)tile * kCtNodes + (e & 0xffu);
                b.eb[g] = (uint32_t)tile * kCtNodes + ((e >> 8) & 0xffu);
                b.ew[g] = (uint8_t)(e >> 16);
            }
        }
        if (!__syncthreads_or(join != ~0u)) break;
        if (join != ~0u) comp[t] = join;
        __syncthreads();
        if (t < nn) {
            uint32_t x = comp[t];
            for (int n = 0; n < kCtNodes && comp[x] != x; ++n) x = comp[x];
            comp[t] = x;
            fb[t] = 0u;
        }
        __syncthreads();
    }
    if (t == 0) b.cnt[tile] = (uint32_t)nn | (uint32_t)s_forest << 16;
}

// ----------------------------------------------------------------- global
namespace {

constexpr int kGT = 256;
constexpr uint32_t kMix = 2654435761u, kUnmix = 244002641u;   // inverses mod 2^32: ties in no geometric order
constexpr uint32_t kDone = 0x80000000u;
constexpr int kMaxRounds = 64;
static_assert(kMix * kUnmix == 1u, "inverse");

__device__ __forceinline__ uint32_t ct_node(const CtBatch &b, const CtImage &d, int r, int c)
{
    const int t = d.tile_base + (r / kCtSide) * d.nx + c / kCtSide;
    const uint32_t e = __ldcg(b.plane + (int64_t)t * kCtPx + (r % kCtSide) * kCtSide + c % kCtSide);
    return (uint32_t)t * kCtNodes + (e >> 8);
}

__device__ __forceinline__ uint32_t ct_root(const CtBatch &b, uint32_t x)
{
    for (int n = 0; n < (1 << 20); ++n) {
        const uint32_t p = (uint32_t)__ldcg(b.link + x);
        if (p == x) break;
        x = p;
    }
    return x;
}

}  // namespace

// Contraction of the nodes of the batch. Every warp owns the tiles [t0, t1),
// with their nodes and the edges of their slots, which it keeps compacted at
// the start of its range; so no list is shared. A round: (1) the edges find
// their clusters and raise the clusters' best edges; (2) every open root
// takes its decision. A grid barrier follows each. Roots that joined are
// pointed at their new root, with the smallest weight on the way, at the
// start of the next round's (1); readers that come first walk on.
__global__ void __launch_bounds__(kGT, 4) ct_global_kernel(const __grid_constant__ CtBatch b, uint64_t timeout_ns)
{
    const int lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)blockIdx.x * (kGT / 32) + (threadIdx.x >> 5), nw = (int64_t)gridDim.x * (kGT / 32);
    const int t0 = (int)(gw * b.ntiles / nw), t1 = (int)((gw + 1) * b.ntiles / nw);
    const uint32_t below = (1u << lane) - 1u;
    const int64_t ebase = (int64_t)t0 * kCtEdges;
    uint32_t *act = b.act + (int64_t)t0 * kCtNodes;
    int ne = 0, na = 0;
    __shared__ uint32_t s_open;

    auto emit = [&](bool valid, uint32_t a, uint32_t c, uint32_t w) {   // whole warp: one edge per node pair
        valid = valid && (a & 0xffu) != kCtNoNode && (c & 0xffu) != kCtNoNode;   // always: rim pixels are in nodes
        const unsigned long long pair = valid ? (unsigned long long)a << 32 | c : ~0ull;
        const uint32_t peers = __match_any_sync(0xffffffffu, pair);
        const uint32_t wm = __reduce_max_sync(peers, w);
        const bool lead = valid && lane == __ffs(peers) - 1;
        const uint32_t m = __ballot_sync(0xffffffffu, lead);
        if (lead) {
            const int64_t g = ebase + ne + __popc(m & below);
            b.ea[g] = a;
            b.eb[g] = c;
            b.ew[g] = (uint8_t)wm;
        }
        ne += __popc(m);
    };
    for (int t = t0; t < t1; ++t) {
        const CtImage &d = ct_image(b, t);
        const int lt = t - d.tile_base;
        const int ty = lt / d.nx, tx = lt - ty * d.nx;
        const uint32_t cn = __ldcg(b.cnt + t);
        const int nn = (int)(cn & 0xffffu), nf = (int)(cn >> 16);
        for (int i = lane; i < nn; i += 32) act[na + i] = (uint32_t)t * kCtNodes + i;
        na += nn;
        // the tile's forest moves up (never past its own slots)
        for (int i = 0; i < nf; i += 32) {
            const int64_t from = (int64_t)t * kCtEdges + i + lane, to = ebase + ne + i + lane;
            uint32_t a = 0, c = 0;
            uint8_t w = 0;
            if (i + lane < nf) a = b.ea[from], c = b.eb[from], w = b.ew[from];
            __syncwarp();
            if (i + lane < nf) b.ea[to] = a, b.eb[to] = c, b.ew[to] = w;
            __syncwarp();
        }
        ne += nf;
        // seams: keys order the pixels of a window by (I, raster order), 0 = outside
        auto key = [&](int r, int c, uint32_t at) -> uint32_t {
            if (r < 0 || r >= d.H || c < 0 || c >= d.W) return 0u;
            return ((uint32_t)__ldg(d.mask + (int64_t)r * d.ld_mask + c) + 1u) << 4 | at;
        };
        auto weight = [&](uint32_t k1, uint32_t k2) { return (min(k1, k2) >> 4) - 1u; };
        if (tx + 1 < d.nx) {
            const int c = tx * kCtSide + kCtSide - 1;
            for (int h = 0; h < kCtSide; h += 32) {
                const int r = ty * kCtSide + h + lane;
                const uint32_t u0 = key(r - 1, c, 0), u1 = key(r - 1, c + 1, 1), m0 = key(r, c, 2),
                               m1 = key(r, c + 1, 3), d0 = key(r + 1, c, 4), d1 = key(r + 1, c + 1, 5);
                const bool in = m0 && m1;
                const bool s = in && max(m0, m1) > max(max(u0, u1), max(d0, d1));
                emit(s, s ? ct_node(b, d, r, c) : 0u, s ? ct_node(b, d, r, c + 1) : 0u, s ? weight(m0, m1) : 0u);
                const bool q = in && d0 && d1, main = max(m0, d1) > max(m1, d0);
                emit(q, q ? ct_node(b, d, main ? r : r + 1, c) : 0u, q ? ct_node(b, d, main ? r + 1 : r, c + 1) : 0u,
                     q ? (main ? weight(m0, d1) : weight(m1, d0)) : 0u);
            }
        }
        if (ty + 1 < d.ny) {
            const int r = ty * kCtSide + kCtSide - 1;
            for (int h = 0; h < kCtSide; h += 32) {
                const int c = tx * kCtSide + h + lane;
                const uint32_t l0 = key(r, c - 1, 0), m0 = key(r, c, 1), r0 = key(r, c + 1, 2),
                               l1 = key(r + 1, c - 1, 3), m1 = key(r + 1, c, 4), r1 = key(r + 1, c + 1, 5);
                const bool in = m0 && m1;
                const bool s = in && max(m0, m1) > max(max(l0, l1), max(r0, r1));
                emit(s, s ? ct_node(b, d, r, c) : 0u, s ? ct_node(b, d, r + 1, c) : 0u, s ? weight(m0, m1) : 0u);
                // the window at the tile's corner belongs to the right seam
                const bool q = in && r0 && r1 && h + lane < kCtSide - 1, main = max(m0, r1) > max(m1, r0);
                emit(q, q ? ct_node(b, d, r, main ? c : c + 1) : 0u, q ? ct_node(b, d, r + 1, main ? c + 1 : c) : 0u,
                     q ? (main ? weight(m0, r1) : weight(m1, r0)) : 0u);
            }
        }
        __syncwarp();
    }

    for (int round = 0; round < kMaxRounds; ++round) {
        // (0) roots that joined: final links of the last round; the others stay open
        if (round > 0) {
            int kept = 0;
            for (int i = 0; i < na; i += 32) {
                bool open = false;
                uint32_t r = 0;
                if (i + lane < na) {
                    r = act[i + lane];
                    const unsigned long long l = __ldcg(b.link + r);
                    uint32_t x = (uint32_t)l;
                    open = x == r;
                    if (!open) {
                        uint32_t w = (uint32_t)(l >> 32);
                        for (int n = 0; n < (1 << 20); ++n) {
                            const unsigned long long lx = __ldcg(b.link + x);
                            if ((uint32_t)lx == x) break;
                            w = min(w, (uint32_t)(lx >> 32));
                            x = (uint32_t)lx;
                        }
                        __stcg(b.link + r, (unsigned long long)w << 32 | x);
                        atomicMax(b.S + x, __ldcg(b.S + r) & 0xffu);
                    }
                }
                const uint32_t m = __ballot_sync(0xffffffffu, open);
                if (open) act[kept + __popc(m & below)] = r;
                kept += __popc(m);
                __syncwarp();
            }
            na = kept;
        }
        // (1) edges; a key holds the round, so the last round's bests count as none
        int kept = 0;
        for (int i = 0; i < ne; i += 32) {
            uint32_t a = 0, c = 0, w = 0;
            bool keep = false, oa = false, oc = false;
            if (i + lane < ne) {
                const int64_t g = ebase + i + lane;
                a = b.ea[g];
                c = b.eb[g];
                w = b.ew[g];
                if (round > 0) {
                    a = ct_root(b, a);
                    c = ct_root(b, c);
                    oa = !(__ldcg(b.S + a) & kDone);
                    oc = !(__ldcg(b.S + c) & kDone);
                } else {
                    oa = oc = true;
                }
                keep = a != c && (oa || oc);
            }
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int64_t g = ebase + kept + __popc(m & below);
                b.ea[g] = a;
                b.eb[g] = c;
                b.ew[g] = (uint8_t)w;
                const unsigned long long k =
                    (unsigned long long)(round + 1) << 48 | (unsigned long long)(w + 1u) << 32 | (uint32_t)g * kMix;
                if (oa && __ldcg(b.best + a) < k) atomicMax(b.best + a, k);
                if (oc && __ldcg(b.best + c) < k) atomicMax(b.best + c, k);
            }
            kept += __popc(m);
            __syncwarp();
        }
        ne = kept;
        // open roots of the batch: the round's counter (the next one's is cleared)
        uint32_t *open_cnt = b.ctl + kCtCtlOpen + round % 3;
        if (lane == 0 && na) atomicAdd(open_cnt, (uint32_t)na);
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(b.ctl + kCtCtlOpen + (round + 1) % 3, 0u);
        if (!grid_barrier(b.ctl + kCtCtlBar, gridDim.x, b.err, timeout_ns)) return;
        if (threadIdx.x == 0) s_open = ld_acquire(open_cnt);
        __syncthreads();
        if (s_open == 0u) return;
        // (2) decisions
        kept = 0;
        for (int i = 0; i < na; i += 32) {
            bool open = false;
            uint32_t r = 0;
            if (i + lane < na) {
                r = act[i + lane];
                const unsigned long long k = __ldcg(b.best + r);
                const uint32_t S = __ldcg(b.S + r) & 0xffu;
                const bool some = (uint32_t)(k >> 48) == (uint32_t)(round + 1);
                const uint32_t w = ((uint32_t)(k >> 32) & 0xffffu) - 1u;
                if (!some || S >= w) {
                    atomicOr(b.S + r, kDone);
                } else {
                    open = true;
                    const uint32_t g = (uint32_t)k * kUnmix;
                    const uint32_t a = __ldcg(b.ea + g), c = __ldcg(b.eb + g), o = a == r ? c : a;
                    const bool mutual = __ldcg(b.best + o) == k && (__ldcg(b.S + o) & 0xffu) < w;
                    if (!(mutual && r < o)) __stcg(b.link + r, (unsigned long long)w << 32 | o);
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, open);
            if (open) act[kept + __popc(m & below)] = r;
            kept += __popc(m);
            __syncwarp();
        }
        na = kept;
        if (!grid_barrier(b.ctl + kCtCtlBar, gridDim.x, b.err, timeout_ns)) return;
    }
    raise_status(b.err, RT_ETIMEOUT);   // not reached: every round at least halves the open roots of a component
}

// ----------------------------------------------------------------- output
__global__ void __launch_bounds__(256) ct_out_kernel(const __grid_constant__ CtBatch b, int threshold)
{
    __shared__ uint32_t val[kCtNodes];
    const int tile = blockIdx.x, t = threadIdx.x;
    const CtImage &d = ct_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const int nn = (int)(b.cnt[tile] & 0xffffu);
    uint32_t v = 255u;
    if (t < nn) {
        uint32_t x = (uint32_t)tile * kCtNodes + t;
        for (int n = 0; n < (1 << 20); ++n) {
            const unsigned long long l = b.link[x];
            if ((uint32_t)l == x) break;
            v = min(v, (uint32_t)(l >> 32));
            x = (uint32_t)l;
        }
        v = min(v, b.S[x] & 0xffu);
    }
    val[t] = v;
    __syncthreads();
    const int r = ty * kCtSide + (t >> 2), c = tx * kCtSide + (t & 3) * 16;
    const int n = min(16, d.W - c);
    if (r >= d.H || n <= 0) return;
    const uint4 *src = reinterpret_cast<const uint4 *>(b.plane + (int64_t)tile * kCtPx + (t >> 2) * kCtSide + (t & 3) * 16);
    const uint4 s0 = __ldcs(src), s1 = __ldcs(src + 1);
    const uint32_t e[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
    uint32_t R[4] = {0, 0, 0, 0}, B[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k >= n) break;   // entries past the image are not written
        const uint32_t x = (e[k >> 1] >> (16 * (k & 1))) & 0xffffu;
        const uint32_t p = min(x & 0xffu, val[x >> 8]);
        R[k >> 2] |= p << (8 * (k & 3));
        B[k >> 2] |= (uint32_t)((int)p < threshold) << (8 * (k & 3));
    }
    auto store = [&](uint8_t *o, const uint32_t *w) {
        if (n == 16 && ((uintptr_t)o & 15u) == 0) {
            *reinterpret_cast<uint4 *>(o) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (k < n) o[k] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
        }
    };
    if (d.out) store(d.out + (int64_t)r * d.ld_out + c, R);
    if (d.bin) store(d.bin + (int64_t)r * d.ld_bin + c, B);
}

void ct_plan_image(CtBatch &b, const uint8_t *marker, int64_t ld_marker, const uint8_t *mask, int64_t ld_mask, int H,
                   int W, int h_offset)
{
    CtImage &d = b.img[b.n++];
    d.marker = marker;
    d.ld_marker = ld_marker;
    d.mask = mask;
    d.ld_mask = ld_mask;
    d.H = H;
    d.W = W;
    d.nx = (int)ceil_div(W, kCtSide);
    d.ny = (int)ceil_div(H, kCtSide);
    d.tile_base = b.ntiles;
    d.h_offset = h_offset;
    d.out = d.bin = nullptr;
    d.ld_out = d.ld_bin = 0;
    b.ntiles += d.nx * d.ny;
}

cudaError_t launch_contract(const CtBatch &b, int num_sms, uint64_t timeout_ns, cudaStream_t s)
{
    const bool given = b.img[0].marker != nullptr;   // all images of a batch, or none
    const void *fn = given ? (const void *)ct_local_kernel<true> : (const void *)ct_local_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLocalSmem);
    if (e != cudaSuccess) return e;
    if (given) ct_local_kernel<true><<<(unsigned)b.ntiles, kT, kLocalSmem, s>>>(b);
    else ct_local_kernel<false><<<(unsigned)b.ntiles, kT, kLocalSmem, s>>>(b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ct_global_kernel, kGT, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int grid = per_sm * num_sms;
    const int need = (int)ceil_div(b.ntiles, kGT / 32);
    if (grid > need) grid = need;
    CtBatch bb = b;
    void *args[] = {&bb, &timeout_ns};
    return cudaLaunchCooperativeKernel((const void *)ct_global_kernel, dim3((unsigned)grid), dim3(kGT), args, 0, s);
}

cudaError_t launch_contract_out(const CtBatch &b, int threshold, cudaStream_t s)
{
    ct_out_kernel<<<(unsigned)b.ntiles, 256, 0, s>>>(b, threshold);
    return cudaGetLastError();
}

}  // namespace rtk
