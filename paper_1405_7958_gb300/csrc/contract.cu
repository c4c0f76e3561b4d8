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
// Two facts make the first steps cheap:
//   * a pixel with a neighbour q of I(q) >= I(p) satisfies R(p) =
//     min(I(p), R(q)) for any such q, so the first contraction is one
//     3 x 3 maximum: every pixel points at its largest neighbour (ties by
//     raster order) and only the local maxima remain as clusters (one in
//     nine pixels of a noisy image);
//   * an edge that is the smallest of a cycle is in no maximum spanning
//     forest. A pixel p needs one edge of weight I(p) into each connected
//     group of its larger neighbours (inside a group they reach each other by
//     larger edges), and the group of its largest neighbour is the one p
//     already points into. So only the pixels whose larger neighbours fall
//     into several groups (one in four) have edges between clusters to give.
//
// Launches: ct_local_kernel contracts every 64 x 64 tile in shared memory
// until each open cluster's best edge leaves the tile; what is left of a
// tile are its nodes (clusters that touch its rim, about 50 of 4096 pixels
// on nuclei tiles), the forest between them, and 2 bytes per pixel (node,
// bound). ct_seam_kernel adds the edges across the seams; ct_global_kernel
// contracts the nodes of the whole batch (one persistent cooperative launch).
// ct_out_kernel writes R.
//
// Measured on one GB300 against the directional sweeps (rt_segment_batch or
// rt_reconstruct, whole call; the chain's other stages are the same):
// 512 x 512 reconstruction 67 us against 357; one 4096 x 4096 tile 0.43 ms
// against 1.13; eight of them 2.42 ms against 4.6. So the contraction runs wherever the call leaves the
// schedule to the library. Smooth images, with few local maxima and long
// walks to them, are where the sweeps win: a reconstruction of 4096 x 4096
// pixels interpolated between random values 40 pixels apart takes 418 us
// against 222, of zeros 203 against 92.
#include "contract.cuh"

namespace rtk {

namespace {

// Roots of the first contraction: local maxima in the tile, no two adjacent.
constexpr int kRoots = 1024;
// Edges that the pixels give: the groups of larger neighbours beyond the
// first, summed over the tile, are roots + minima - 1 (Euler characteristic;
// a minimum: all four edge neighbours larger, so no two of them adjacent and
// none on the rim): at most 1024 + 62 * 62 / 2.
constexpr int kList = 2976;
// A neighbour's code: (row + 1) * 3 + column + 1 of its step; 4: the pixel itself.
constexpr int kCodes = 9;
// Shared memory: pixel words, edges, link words, the parents (whose memory
// then holds the best edges and two lists of roots), the groups' table. It
// is cut to let five CTAs share an SM.
constexpr size_t kLocalSmem = sizeof(uint32_t) * (kCtPx + kList + kRoots) + sizeof(uint16_t) * (kCtPx + kCodes * 256);
static_assert(sizeof(uint16_t) * kCtPx == sizeof(uint32_t) * kRoots + 2 * sizeof(uint16_t) * kRoots, "reused memory");

// For every set of larger neighbours (bit j: kNear[j]) and code of the
// largest: one neighbour of each group that does not hold the largest, as up
// to three nibbles code + 1, and their number in the fourth.
struct alignas(16) GroupTable {
    uint16_t v[kCodes * 256];
};
constexpr int kNear[8] = {0, 1, 2, 3, 5, 6, 7, 8};
constexpr GroupTable group_table()
{
    GroupTable g{};
    for (int c = 0; c < kCodes; ++c)
        for (int m = 0; m < 256; ++m) {
            int left = m, out = 0, shift = 0;
            bool valid = false;
            for (int j = 0; j < 8; ++j) valid = valid || (kNear[j] == c && ((m >> j) & 1));
            while (valid && left) {
                int grp = left & -left, rep = 0;
                while (!((left >> rep) & 1)) ++rep;
                for (bool more = true; more;) {
                    more = false;
                    for (int a = 0; a < 8; ++a)
                        for (int b = 0; b < 8; ++b) {
                            const int dr = kNear[a] / 3 - kNear[b] / 3, dc = kNear[a] % 3 - kNear[b] % 3;
                            const bool next = dr >= -1 && dr <= 1 && dc >= -1 && dc <= 1;
                            if (((grp >> a) & 1) && ((m >> b) & 1) && !((grp >> b) & 1) && next) grp |= 1 << b, more = true;
                        }
                }
                left &= ~grp;
                bool own = false;
                for (int j = 0; j < 8; ++j) own = own || (((grp >> j) & 1) && kNear[j] == c);
                if (!own) out += 0x1000 | (kNear[rep] + 1) << shift, shift += 4;
            }
            g.v[c * 256 + m] = (uint16_t)out;
        }
    return g;
}
__device__ constexpr GroupTable kGroupTable = group_table();

// A pixel's word: I << 24 | index in the tile << 12 | kPix, later | kIn |
// cluster. Words order the tile's pixels by (I, raster index); a pixel
// outside the image is 0, below every pixel.
constexpr uint32_t kPix = 0x800u, kIn = 0x400u, kIdx = 0x3ffu, kLabel = 0x7ffu;

// A node's link word: root: kNodeRoot | kNodeDone (final) | S << 40 | itself;
// else weight << 32 | parent. An edge of nodes: weight << 56 | node << 28 | node.
constexpr unsigned long long kNodeRoot = 1ull << 63, kNodeDone = 1ull << 62;
constexpr uint32_t kNodeId = (1u << 28) - 1u;
__device__ __forceinline__ unsigned long long node_edge(uint32_t a, uint32_t b, uint32_t w)
{
    return (unsigned long long)w << 56 | (unsigned long long)a << 28 | b;
}
__device__ __forceinline__ uint32_t node_S(unsigned long long root) { return (uint32_t)(root >> 40) & 0xffu; }

// A cluster's link word: root: kRootBit | X << 8 | S, X = 1 + the weight of its
// best edge that leaves the tile (0: none); else weight << 16 | parent.
constexpr uint32_t kRootBit = 0x80000000u;
__device__ __forceinline__ uint32_t root_of(const volatile uint32_t *nlink, uint32_t k)
{
    const uint32_t v = nlink[k];   // k was a root in the last round, or links are compressed
    return (v & kRootBit) ? k : (v & 0xffffu);
}
// In the rounds an edge is weight << 24 | cluster << 12 | cluster.
__device__ __forceinline__ const CtImage &ct_image(const CtBatch &b, int t)
{
    int k = 0;
    while (k + 1 < b.n && t >= b.img[k + 1].tile_base) ++k;
    return b.img[k];
}

__device__ __forceinline__ uint32_t max3(uint32_t a, uint32_t b, uint32_t c) { return max(a, max(b, c)); }
}  // namespace

// ------------------------------------------------------------------ local
// NT threads; a warp takes 64 / warps rows, a lane two adjacent columns.
// Bound by instruction issue (74 % active, 45 k warp instructions a tile,
// 205 us per 4096 x 4096 image, DRAM idle). What it measured on that image:
// edges from 2 x 2 windows with flags 377 us; cluster ids in the edges, lists
// of open roots, parents apart from the pixel words 290; edges from groups of
// larger neighbours by table 240; loops kept rolled (43 KB of code instead of
// 88, which missed the instruction cache) and five CTAs an SM instead of four
// 220; edges counted first and written at one position per warp, not per row,
// 215; no tests of the image's border in inner tiles and none of roots that
// no warp has 205. The first full version took 373 us.
template <bool MARKER, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 5 : 1) ct_local_kernel(const __grid_constant__ CtBatch b)
{
    start_early();
    constexpr int kWarps = NT / 32, kRows = kCtSide / kWarps, kPer = kRoots / NT;
    extern __shared__ __align__(16) uint32_t ct_smem[];
    uint32_t *W = ct_smem;                      // pixel words
    uint32_t *list = W + kCtPx;                 // edges
    volatile uint32_t *nlink = list + kList;    // per cluster: link word
    volatile uint16_t *P = reinterpret_cast<volatile uint16_t *>(nlink + kRoots);   // per pixel: code << 12 | parent
    volatile uint32_t *best = nlink + kRoots;   // then, per cluster: weight << 13 | position of its best edge, + 1
    volatile uint16_t *live = P + 2 * kRoots;   // and two lists of open roots
    uint16_t *table = const_cast<uint16_t *>(P) + kCtPx;                            // kGroupTable
    volatile uint32_t *VW = W;
    __shared__ int s_roots, s_edges, s_nodes, s_forest, s_live[2];

    const int tile = blockIdx.x;
    const CtImage &d = ct_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const int r0 = ty * kCtSide, c0 = tx * kCtSide;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t below = (1u << lane) - 1u;
    const int rs = warp * kRows, cl = 2 * lane;

    if (t == 0) s_roots = s_edges = s_nodes = s_forest = s_live[0] = s_live[1] = 0;

    // ---- load the tile; the rim threads (four sides of 64) also the largest
    // halo pixel next to their pixel, + 1 (0: none)
    uint32_t halo = 0;
    const int side = t >> 6, si = t & 63;
    const int rim = side == 0 ? si : side == 1 ? (kCtSide - 1) * kCtSide + si : side == 2 ? si * kCtSide : si * kCtSide + kCtSide - 1;
    if (t < 256) {
        const bool open = side == 0 ? ty > 0 : side == 1 ? ty + 1 < d.ny : side == 2 ? tx > 0 : tx + 1 < d.nx;
        if (open) {
#pragma unroll
            for (int k = -1; k <= 1; ++k) {
                const int r = side == 0 ? r0 - 1 : side == 1 ? r0 + kCtSide : r0 + si + k;
                const int c = side == 2 ? c0 - 1 : side == 3 ? c0 + kCtSide : c0 + si + k;
                if (r >= 0 && r < d.H && c >= 0 && c < d.W)
                    halo = max(halo, (uint32_t)d.mask[(int64_t)r * d.ld_mask + c] + 1u);
            }
        }
    }
#pragma unroll 1
    for (int i = t; i < kCodes * 256 / 8; i += NT)
        reinterpret_cast<uint4 *>(table)[i] = __ldg(reinterpret_cast<const uint4 *>(kGroupTable.v) + i);
    {
        const int c = c0 + 4 * (t & 15);
#pragma unroll
        for (int rr = t >> 4; rr < kCtSide; rr += NT / 16) {
            const int r = r0 + rr, n = r < d.H ? min(4, d.W - c) : 0;   // may be negative: none
            uint32_t v = 0;
            const uint8_t *p = d.mask + (int64_t)r * d.ld_mask + c;
            const uint32_t off = (uint32_t)(uintptr_t)p & 3u;
            if (n == 4 && (off == 0 || (c >= 4 && c + 8 <= d.W))) {   // the aligned words around them, in the row
                const uint32_t *q = reinterpret_cast<const uint32_t *>(p - off);
                v = q[0];
                if (off) v = __funnelshift_r(v, q[1], 8u * off);
            } else {
#pragma unroll 1
                for (int k = 0; k < n; ++k) v |= (uint32_t)p[k] << (8 * k);
            }
            const uint32_t idx = (uint32_t)(rr * kCtSide + 4 * (t & 15));
            uint32_t o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = k < n ? __byte_perm(v, 0u, k << 12 | 0x0444u) | (idx + k) << 12 | kPix : 0u;
            *reinterpret_cast<uint4 *>(W + idx) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
    __syncthreads();

    // ---- first contraction: every pixel points at the largest pixel of its
    // 3 x 3 neighbourhood in the tile. (At the row's ends the shuffles return
    // the lane's own word, which is in the neighbourhood anyway.)
    auto row_of = [&](int r) -> uint2 {
        if (r < 0 || r >= kCtSide) return make_uint2(0u, 0u);   // whole warp
        return *reinterpret_cast<const uint2 *>(W + r * kCtSide + cl);
    };
    uint32_t rootmask = 0;   // bit 2 j + k: pixel (rs + j, cl + k) is a root
    {
        auto across = [&](uint2 v) -> uint2 {
            const uint32_t l = __shfl_up_sync(0xffffffffu, v.y, 1), r = __shfl_down_sync(0xffffffffu, v.x, 1);
            const uint32_t m = max(v.x, v.y);
            return make_uint2(max(lane ? l : 0u, m), max(lane < 31 ? r : 0u, m));
        };
        uint2 vb = row_of(rs), ha = across(row_of(rs - 1)), hb = across(vb);
#pragma unroll 2
        for (int j = 0; j < kRows; ++j) {
            const uint2 vc = row_of(rs + j + 1), hc = across(vc);
            const uint32_t m0 = max3(ha.x, hb.x, hc.x) >> 12, m1 = max3(ha.y, hb.y, hc.y) >> 12;
            if (vb.x && m0 == vb.x >> 12) rootmask |= 1u << (2 * j);
            if (vb.y && m1 == vb.y >> 12) rootmask |= 2u << (2 * j);
            const uint32_t at = (uint32_t)((rs + j) * kCtSide + cl);
            auto pack = [](uint32_t own, uint32_t to, uint32_t here) -> uint32_t {
                if (!own) to = here;
                const uint32_t step = to - here + 65u;   // 64 (row + 1) + column + 1
                return to | ((step >> 6) * 3u + (step & 3u)) << 12;
            };
            reinterpret_cast<volatile uint32_t *>(P)[at / 2] = pack(vb.x, m0 & 0xfffu, at) | pack(vb.y, m1 & 0xfffu, at + 1) << 16;
            ha = hb;
            hb = hc;
            vb = vc;
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
#pragma unroll 1
        while (rootmask) {
            const int j = __ffs(rootmask) - 1;
            rootmask &= rootmask - 1;
            const int idx = (rs + (j >> 1)) * kCtSide + cl + (j & 1);
            const uint32_t w = VW[idx];
            // the derived marker's largest value in the cluster is at its maximum
            const uint32_t I = w >> 24;
            const uint32_t S = MARKER ? 0u : (I > (uint32_t)d.h_offset ? I - (uint32_t)d.h_offset : 0u);
            VW[idx] = w | kIn | k;
            nlink[k] = kRootBit | S;
            ++k;
        }
    }
    __syncthreads();
    const int nr = s_roots;

    // ---- every pixel's cluster: four steps uphill without a test (nearly
    // always enough), then until a root or a pixel that has found its own.
    // Parents are replaced by what was found, which shortens the long walks
    // of flat images; the rows are taken from below, as ties lead down (from
    // above every row walked to the tile's last one: a constant 4096 x 4096
    // image 581 us a call, now 238; nuclei 312 and 311).
    {
        bool bad = false;
        const bool rim_tile = ty == 0 || tx == 0 || ty == d.ny - 1 || tx == d.nx - 1;   // holds pixels of the image's border
#pragma unroll 2
        for (int j = kRows - 1; j >= 0; --j) {
            const int at = (rs + j) * kCtSide + cl;
            const uint2 ow = *reinterpret_cast<const uint2 *>(W + at);
            const uint32_t pp = reinterpret_cast<volatile uint32_t *>(P)[at / 2];
            uint32_t x[2] = {pp & 0xfffu, (pp >> 16) & 0xfffu}, v[2], own[2] = {ow.x, ow.y};
#pragma unroll
            for (int n = 0; n < 3; ++n) x[0] = P[x[0]] & 0xfffu, x[1] = P[x[1]] & 0xfffu;
            v[0] = VW[x[0]], v[1] = VW[x[1]];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll 1
                for (int n = 0; n < kCtPx && own[q] && !(v[q] & kIn); ++n) {
                    x[q] = P[x[q]] & 0xfffu;
                    v[q] = VW[x[q]];
                }
            reinterpret_cast<volatile uint32_t *>(P)[at / 2] = (pp & 0xf000f000u) | x[0] | x[1] << 16;
            uint2 nw = ow;
            if (ow.x) nw.x = ow.x | (v[0] & kLabel);
            if (ow.y) nw.y = ow.y | (v[1] & kLabel);
            *reinterpret_cast<uint2 *>(W + at) = nw;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int r = rs + j, c = cl + q;
                if (!own[q]) continue;
                const uint32_t k = v[q] & kIdx, I = own[q] >> 24;
                const int gr = r0 + r, gc = c0 + c;
                uint32_t *sk = const_cast<uint32_t *>(nlink + k);
                if (MARKER) {
                    const uint32_t J = d.marker[(int64_t)gr * d.ld_marker + gc];
                    bad |= J > I;
                    const uint32_t s = kRootBit | min(J, I);
                    if (nlink[k] < s) atomicMax(sk, s);
                } else if (rim_tile && (gr == 0 || gr == d.H - 1 || gc == 0 || gc == d.W - 1)) {
                    atomicMax(sk, kRootBit | I);
                }
            }
        }
        if (MARKER && bad) raise_status(b.err, RT_EMARKER);
    }
    __syncthreads();

    // ---- the pixels' edges, as index | (code + 1) << 12, and the best edge of
    // every rim cluster that leaves the tile
    if (halo) {
        const uint32_t w = W[rim];
        if (w) {
            const uint32_t k = w & kIdx, old = nlink[k], v = kRootBit | min((w >> 24) + 1u, halo) << 8 | (old & 0xffu);
            if (old < v) atomicMax(const_cast<uint32_t *>(nlink + k), v);
        }
    }
    {
        // rows of words >> 4 (only their order counts), with the columns beside the lane's two
        auto load = [&](int r, uint32_t (&o)[4]) {
            const uint2 v = row_of(r);
            o[1] = v.x >> 4;
            o[2] = v.y >> 4;
            o[0] = __shfl_up_sync(0xffffffffu, o[2], 1);
            o[3] = __shfl_down_sync(0xffffffffu, o[1], 1);
            if (lane == 0) o[0] = 0u;
            if (lane == 31) o[3] = 0u;
        };
        uint32_t u[4], m[4], n[4];
        load(rs - 1, u);
        load(rs, m);
        // the pixels' groups take the place of their parents and are counted; then every lane writes its own
        int cnt = 0;
#pragma unroll 1   // the loops over rows stay rolled: the kernel's time is lost to instruction fetch otherwise
        for (int j = 0; j < kRows; ++j) {
            const int r = rs + j;
            load(r + 1, n);
            const uint32_t pp = reinterpret_cast<volatile uint32_t *>(P)[(r * kCtSide + cl) / 2];
            uint32_t g[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                // bit j of the set: kNear[j] is larger (the sign of a difference, shifted in)
                const uint32_t near[8] = {u[q], u[q + 1], u[q + 2], m[q], m[q + 2], n[q], n[q + 1], n[q + 2]};
                uint32_t set = 0;
#pragma unroll
                for (int j = 7; j >= 0; --j) set = __funnelshift_l(m[q + 1] - near[j], set, 1);
                // (code << 8 | set; code 4, a root or outside the image, has no groups)
                g[q] = table[((q ? pp >> 20 : pp >> 4) & 0xf00u) | set];
                cnt += (int)(g[q] >> 12);
            }
            reinterpret_cast<volatile uint32_t *>(P)[(r * kCtSide + cl) / 2] = g[0] | g[1] << 16;
#pragma unroll
            for (int q = 0; q < 4; ++q) u[q] = m[q], m[q] = n[q];
        }
        int pos = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += v;
        }
        int base = 0;
        if (lane == 31) base = atomicAdd(&s_edges, pos);
        pos += __shfl_sync(0xffffffffu, base, 31) - cnt;
#pragma unroll 1
        for (int j = 0; j < kRows && cnt; ++j) {
            const uint32_t at0 = (uint32_t)((rs + j) * kCtSide + cl);
            const uint32_t gg = reinterpret_cast<volatile uint32_t *>(P)[at0 / 2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t f = (q ? gg >> 16 : gg) & 0xfffu;
                if (!f) continue;
                if (pos < kList) list[pos] = (at0 + q) | (f & 0xfu) << 12;   // pos < kList: always (see kList)
                ++pos;
#pragma unroll 1
                while (f >>= 4) {
                    if (pos < kList) list[pos] = (at0 + q) | (f & 0xfu) << 12;
                    ++pos;
                }
            }
        }
    }
    __syncthreads();

#pragma unroll 1
    for (int k = t; k < nr; k += NT) best[k] = 0u;   // in the parents' memory
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
    auto edge_pass = [&](bool first) {
        int kept = 0;
#pragma unroll 1
        for (int i = lane; i < cnt + lane; i += 32) {
            uint32_t e = 0, ra = 0, rb = 0;
            if (i < cnt) {
                e = list[start + i];
                if (first) {
                    const uint32_t p = e & 0xfffu, code = (e >> 12) - 1u;
                    const uint32_t wp = W[p], wq = W[p + code + 61u * (code * 11u >> 5) - 65u];   // 64 row + column
                    e = wp;
                    ra = wp & kIdx;
                    rb = wq & kIdx;
                } else {
                    ra = root_of(nlink, e & kIdx);
                    rb = root_of(nlink, (e >> 12) & kIdx);
                }
            }
            const bool keep = ra != rb;
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const uint32_t pos = start + kept + __popc(m & below);
                list[pos] = (e & 0xff000000u) | rb << 12 | ra;
                const uint32_t key = ((e >> 24) << 13) + pos + 1u;
                atomicMax(const_cast<uint32_t *>(best + ra), key);
                atomicMax(const_cast<uint32_t *>(best + rb), key);
            }
            kept += __popc(m);
            __syncwarp();
        }
        cnt = kept;
    };
    edge_pass(true);
    __syncthreads();
    // Only open roots are visited (round 0: all; then the list that the round
    // before left). A root that is final, or whose best edge leaves the tile,
    // stays: another may still join it.
    int nl = nr;
#pragma unroll 1
    for (int round = 0;; ++round) {
        const volatile uint16_t *from = live + (round & 1) * kRoots;
        volatile uint16_t *to = live + (~round & 1) * kRoots;
        // decide: S << 24 | weight << 16 | parent, parent 0xffff: stays
        uint32_t dec[kPer], id[kPer];
        int any = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (q * NT >= nl) break;   // (q > 0: round 0 only, as a rule)
            dec[q] = 0xffffu;
            id[q] = 0u;
            if (t + q * NT >= nl) continue;
            const uint32_t k = round ? from[t + q * NT] : (uint32_t)(t + q * NT);
            id[q] = k;
            const uint32_t key = best[k];
            if (!key) continue;
            const uint32_t w = (key - 1u) >> 13, v = nlink[k], S = v & 0xffu;
            if (S >= w || ((v >> 8) & 0x1ffu) > w + 1u) continue;
            const uint32_t e = list[(key - 1u) & 0x1fffu];
            const uint32_t ra = e & kIdx, o = ra == k ? (e >> 12) & kIdx : ra;
            const uint32_t vo = nlink[o];
            if (k < o && best[o] == key && (vo & 0xffu) < w && ((vo >> 8) & 0x1ffu) <= w + 1u) continue;   // o joins this one
            dec[q] = S << 24 | w << 16 | o;
            id[q] = k | (v & 0x1ff00u) << 8;
            any = 1;
        }
        if (t == 0) s_live[~round & 1] = 0;
        if (!__syncthreads_or(any)) break;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (q * NT >= nl) break;
            if ((dec[q] & 0xffffu) != 0xffffu) nlink[id[q] & 0xffffu] = dec[q] & 0xffffffu;
        }
        __syncthreads();
        // joined: find the new root, with the smallest weight on the way, and
        // hand it the sources; the others make the next list
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (warp * 32 + q * NT >= nl) break;   // whole warp
            const bool in = t + q * NT < nl, joined = (dec[q] & 0xffffu) != 0xffffu;
            const uint32_t k = id[q] & 0xffffu;
            if (joined) {
                uint32_t w = (dec[q] >> 16) & 0xffu, x = dec[q] & 0xffffu;
#pragma unroll 1
                for (int n = 0; n < kRoots; ++n) {
                    const uint32_t v = nlink[x];
                    if (v & kRootBit) break;
                    w = min(w, v >> 16);
                    x = v & 0xffffu;
                }
                nlink[k] = w << 16 | x;
#pragma unroll 1
                for (uint32_t v = nlink[x];;) {   // both maxima at once; ends when nobody else raised them between
                    const uint32_t m = kRootBit | max(v & 0x1ff00u, id[q] >> 8 & 0x1ff00u) | max(v & 0xffu, dec[q] >> 24);
                    if (m == v) break;
                    const uint32_t old = atomicCAS(const_cast<uint32_t *>(nlink + x), v, m);
                    if (old == v) break;
                    v = old;
                }
            } else if (in) {
                best[k] = 0u;
            }
            const bool stays = in && !joined;
            const uint32_t m = __ballot_sync(0xffffffffu, stays);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&s_live[~round & 1], __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (stays) to[base + __popc(m & below)] = (uint16_t)k;
        }
        __syncthreads();
        nl = s_live[~round & 1];
        edge_pass(false);
        __syncthreads();
    }

    // ---- nodes: the clusters with a pixel on a side that has a neighbour
    // tile. best[k] becomes 1 + the node of root k, 0 for the others (which
    // are final: no edge of theirs leaves the tile).
#pragma unroll 1
    for (int k = t; k < nr; k += NT) {
        best[k] = 0u;
        uint32_t v = nlink[k];
        if (v & kRootBit) {
            nlink[k] = v & (kRootBit | 0xffu);
            continue;
        }
        uint32_t w = v >> 16, x = v & 0xffffu;   // links of earlier rounds: one step per round
#pragma unroll 1
        for (int n = 0; n < kRoots; ++n) {
            v = nlink[x];
            if (v & kRootBit) break;
            w = min(w, v >> 16);
            x = v & 0xffffu;
        }
        nlink[k] = w << 16 | x;
    }
    __syncthreads();
    if (halo) {
        const uint32_t w = W[rim];
        if (w) best[root_of(nlink, w & kIdx)] = 1u;
    }
    __syncthreads();
#pragma unroll 1
    for (int k0 = warp * 32; k0 < nr; k0 += NT) {
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
#pragma unroll 1
        for (int i = 0; i < cnt; i += 32) {
            uint32_t e = 0;
            bool keep = false;
            if (i + lane < cnt) {
                const uint32_t f = list[start + i + lane];
                const uint32_t ra = f & kIdx, rb = (f >> 12) & kIdx, w = f >> 24;
                const uint32_t na = best[ra], nb = best[rb];
                keep = na && nb;
                e = (na - 1u) | (nb - 1u) << 8 | w << 16;
                if (na && !nb) atomicMax(const_cast<uint32_t *>(nlink + ra), kRootBit | min(w, nlink[rb] & 0xffu));
                if (nb && !na) atomicMax(const_cast<uint32_t *>(nlink + rb), kRootBit | min(w, nlink[ra] & 0xffu));
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
        uint32_t tab[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const uint32_t k = t + q * NT;
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
                b.link[g] = kNodeRoot | (unsigned long long)(v & 0xffu) << 40 | g;
                b.best[g] = 0ull;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const uint32_t k = t + q * NT;
            if (k < (uint32_t)nr) nlink[k] = tab[q];
        }
        // the forest rounds below use best and what follows as arrays per node
        if (t < nn) best[t] = t;
        if (t < kCtNodes) best[kRoots + t] = 0u;
    }
    __syncthreads();
    if (t < 4 * kCtSide) {
        const uint32_t w = W[rim];
        b.rim[(int64_t)tile * 4 * kCtSide + t] = (uint16_t)(w ? (nlink[w & kIdx] & 0xff00u) | w >> 24 : kCtNoNode << 8);
    }
    {
        uint16_t *o = b.plane + (int64_t)tile * kCtPx + rs * kCtSide + cl;
#pragma unroll 2
        for (int j = 0; j < kRows; ++j) {
            const uint2 v = row_of(rs + j);
            const uint32_t e0 = nlink[v.x & kIdx], e1 = nlink[v.y & kIdx];
            *reinterpret_cast<uint32_t *>(o + j * kCtSide) = (e0 & 0xff00u) | min(e0 & 0xffu, v.x >> 24) |
                                                             (e1 & 0xff00u) << 16 | min(e1 & 0xffu, v.y >> 24) << 16;
        }
    }

    // ---- maximum spanning forest of the nodes (only these edges can matter)
    volatile uint32_t *comp = best, *fb = best + kRoots;
#pragma unroll 1
    for (;;) {
        int kept = 0;
#pragma unroll 1
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
                const int i = atomicAdd(&s_forest, 1);   // dealt to the tile's units in turn
                b.edge[((int64_t)tile * kCtUnits + i % kCtUnits) * kCtUnitEdges + i / kCtUnits] =
                    node_edge((uint32_t)tile * kCtNodes + (e & 0xffu), (uint32_t)tile * kCtNodes + ((e >> 8) & 0xffu),
                              e >> 16);
            }
        }
        if (!__syncthreads_or(join != ~0u)) break;
        if (join != ~0u) comp[t] = join;
        __syncthreads();
        if (t < nn) {
            uint32_t x = comp[t];
#pragma unroll 1
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

constexpr int kGT = 1024;
constexpr int kGCluster = 8;
constexpr int64_t kGClusterUnits = 512;
constexpr int kFewTiles = 304;
constexpr uint32_t kMix = 2654435761u, kUnmix = 244002641u;   // inverses mod 2^32: ties in no geometric order
constexpr int kMaxRounds = 64;
static_assert(kMix * kUnmix == 1u, "inverse");

// A barrier of the cooperative grid that also adds up a number per CTA: word
// counts arrivals in its low half and the numbers in its high half (zero
// before the launch), `target` is all arrivals up to this barrier. An
// arrival is one release without an answer and the wait one polled word, 1.5
// us; counting down, a generation and separate fences took 3.7. The wait is
// bounded: RT_ETIMEOUT and false.
__device__ __forceinline__ bool sum_barrier(unsigned long long *word, uint32_t target, uint32_t add, uint32_t &sum,
                                            int32_t *err, uint64_t timeout_ns)
{
    __shared__ uint32_t s_sum;
    __shared__ int s_ok;
    if (threadIdx.x == 0) {   // the caller has synchronised the CTA
        const unsigned long long one = 1ull | (unsigned long long)add << 32;
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(one) : "memory");
        unsigned long long v;
        int ok = 1;
        uint64_t t0 = 0;
        for (uint32_t spins = 1;; ++spins) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(word) : "memory");
            if ((int32_t)((uint32_t)v - target) >= 0) break;
            if ((spins & 255u) != 0) continue;
            __nanosleep(64);
            const uint64_t now = globaltimer_ns();
            if (!t0) t0 = now;
            if (now - t0 > timeout_ns) {
                raise_status(err, RT_ETIMEOUT);
                ok = 0;
                break;
            }
        }
        s_sum = (uint32_t)(v >> 32);
        s_ok = ok;
    }
    __syncthreads();
    sum = s_sum;
    return s_ok != 0;
}

// The roots above the ends of two edges and their link words, the walks side
// by side.
__device__ __forceinline__ void ct_roots(const CtBatch &b, uint32_t (&x)[4], unsigned long long (&l)[4],
                                         const bool (&have)[2])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) l[k] = have[k / 2] ? __ldcg(b.link + x[k]) : kNodeRoot;
#pragma unroll 1
    for (int n = 0; n < (1 << 20); ++n) {
        bool more = false;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (!(l[k] & kNodeRoot)) {
                x[k] = (uint32_t)l[k];
                l[k] = __ldcg(b.link + x[k]);
                more = true;
            }
        if (!more) break;
    }
}

// An edge's key in round `round`: later rounds first, then heavier ones, then
// by the edge's slot g, mixed.
__device__ __forceinline__ unsigned long long edge_key(int round, uint32_t w, uint32_t g)
{
    return (unsigned long long)(round + 1) << 48 | (unsigned long long)(w + 1u) << 32 | g * kMix;
}

}  // namespace

// ------------------------------------------------------------------- seams
// The edges across the seams and round 0's best edge of every node, a CTA
// per tile. A tile has four units, each a quarter of its nodes and forest and
// half a seam (parts 0, 1: the right one, 2, 3: the lower one); warp w writes
// the edges of part w behind the part's forest edges. The pixels come from
// the tiles' rims, a few words a lane. The best edges are first found in
// shared memory, for the nodes of the tile and of its right and its lower
// neighbour: by weight, then among equals by the mixed slot, which is what
// edge_key orders by; then one global maximum a node. (The global kernel's
// warps built the seams and raced for the bests one unit after the other:
// 240 us of 505 for eight 4096 x 4096 images; this kernel takes 15 us for each
// of these images, 4096 CTAs.)
__global__ void __launch_bounds__(kCtUnits * 32) ct_seam_kernel(const __grid_constant__ CtBatch b)
{
    start_early();
    __shared__ __align__(16) uint32_t bw[3 * kCtNodes], bg[3 * kCtNodes];
    const int tile = blockIdx.x, t = threadIdx.x, lane = t & 31, part = t >> 5;
    const uint32_t all = 0xffffffffu, below = (1u << lane) - 1u;
    const CtImage &d = ct_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const bool down = part >= 2;
    const int u = tile * kCtUnits + part;
    // this lane's edges: up to two of the forest, two of the seam
    uint32_t ea[4], ec[4], ew[4], eg[4];
    bool have[4] = {false, false, false, false};
    const int nf = ((int)(__ldcg(b.cnt + tile) >> 16) - part + kCtUnits - 1) / kCtUnits;
    unsigned long long *edge = b.edge + (int64_t)u * kCtUnitEdges;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        have[k] = lane + 32 * k < nf;
        const unsigned long long e = have[k] ? __ldcg(edge + lane + 32 * k) : 0ull;
        ea[k] = (uint32_t)(e >> 28) & kNodeId;
        ec[k] = (uint32_t)e & kNodeId;
        ew[k] = (uint32_t)(e >> 56);
        eg[k] = (uint32_t)u * kCtUnitEdges + lane + 32 * k;
    }
    for (int i = t; i < 3 * kCtNodes / 4; i += kCtUnits * 32) {
        reinterpret_cast<uint4 *>(bw)[i] = make_uint4(0u, 0u, 0u, 0u);
        reinterpret_cast<uint4 *>(bg)[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // half a seam: a lane takes the pixel m0 on this side, the one across m1,
    // and the window of both and their next neighbours n0, n1; p0, p1 are
    // their previous neighbours. Rim words: node << 8 | I, node kCtNoNode
    // outside the image. Keys order the pixels by (I, raster order), 0 =
    // outside.
    int ne = nf;
    if (down ? ty + 1 < d.ny : tx + 1 < d.nx) {   // whole warp
        const int i = (part & 1) * 32 + lane;
        const int t1 = down ? tile + d.nx : tile + 1;           // the tile across
        const int step = down ? 1 : d.nx;                       // to the next tile along the seam
        const int s0 = down ? 1 : 3, s1 = down ? 0 : 2;         // the sides that meet
        auto rim = [&](int ut, int side, int at) { return (uint32_t)b.rim[((int64_t)ut * 4 + side) * kCtSide + at]; };
        const uint32_t none = kCtNoNode << 8;
        const uint32_t m0 = rim(tile, s0, i), m1 = rim(t1, s1, i);
        // the ends' neighbours along the seam may be the next tiles'
        const bool end = lane == 0 || lane == 31;
        const int ni = lane == 0 ? i - 1 : i + 1;
        const int hop = ni < 0 ? -step : ni >= kCtSide ? step : 0;
        const bool there = hop == 0 || (hop < 0 ? (down ? tx > 0 : ty > 0) : (down ? tx + 1 < d.nx : ty + 1 < d.ny));
        uint32_t x0 = none, x1 = none;
        if (end && there) {
            x0 = rim(tile + hop, s0, ni & (kCtSide - 1));
            x1 = rim(t1 + hop, s1, ni & (kCtSide - 1));
        }
        uint32_t p0 = __shfl_up_sync(all, m0, 1), p1 = __shfl_up_sync(all, m1, 1), n0 = __shfl_down_sync(all, m0, 1),
                 n1 = __shfl_down_sync(all, m1, 1);
        if (lane == 0) p0 = x0, p1 = x1;
        if (lane == 31) n0 = x0, n1 = x1;
        auto key = [&](uint32_t w, uint32_t along, uint32_t across) {
            return w >= none ? 0u : ((w & 0xffu) + 1u) << 4 | (down ? across * 3u + along : along * 2u + across);
        };
        const uint32_t k0 = key(m0, 1, 0), k1 = key(m1, 1, 1), l0 = key(n0, 2, 0), l1 = key(n1, 2, 1);
        const bool in = k0 && k1;
        have[2] = in && max(k0, k1) > max(max(key(p0, 0, 0), key(p1, 0, 1)), max(l0, l1));
        // the window at the tile's corner belongs to the right seam
        have[3] = in && l0 && l1 && !(down && i == kCtSide - 1);
        const bool main = max(k0, l1) > max(k1, l0);
        const int nt = lane == 31 ? hop : 0;   // the next neighbours' tiles
        const uint32_t a0 = (uint32_t)tile * kCtNodes + (m0 >> 8), a1 = (uint32_t)t1 * kCtNodes + (m1 >> 8),
                       c0 = (uint32_t)(tile + nt) * kCtNodes + (n0 >> 8), c1 = (uint32_t)(t1 + nt) * kCtNodes + (n1 >> 8);
        ea[2] = a0, ec[2] = a1, ew[2] = (min(k0, k1) >> 4) - 1u;
        ea[3] = main ? a0 : c0, ec[3] = main ? c1 : a1, ew[3] = (main ? min(k0, l1) : min(k1, l0)) / 16u - 1u;
#pragma unroll
        for (int k = 2; k < 4; ++k) {
            // of neighbouring lanes' edges between the same nodes the heaviest (the first of equals): a vote on all
            // equal pairs of the warp takes longer than the few edges more
            const uint32_t w = have[k] ? ew[k] + 1u : 0u;
            const uint32_t pa = __shfl_up_sync(all, ea[k], 1), pc = __shfl_up_sync(all, ec[k], 1),
                           pw = __shfl_up_sync(all, w, 1), na = __shfl_down_sync(all, ea[k], 1),
                           nc = __shfl_down_sync(all, ec[k], 1), nw = __shfl_down_sync(all, w, 1);
            if (lane > 0 && pa == ea[k] && pc == ec[k] && pw >= w) have[k] = false;
            if (lane < 31 && na == ea[k] && nc == ec[k] && nw > w) have[k] = false;
            const uint32_t m = __ballot_sync(all, have[k]);
            const int at = ne + __popc(m & below);
            eg[k] = (uint32_t)u * kCtUnitEdges + at;
            if (have[k]) edge[at] = node_edge(ea[k], ec[k], ew[k]);
            ne += __popc(m);
        }
    }
    if (lane == 0) b.ecnt[u] = (uint8_t)ne;
    // a node's place in bw and bg; elsewhere (over the corner): -1
    auto place = [&](uint32_t x) {
        const int ut = (int)(x >> 8);
        return ut == tile ? (int)(x & 0xffu) : ut == tile + 1 ? kCtNodes + (int)(x & 0xffu)
               : ut == tile + d.nx ? 2 * kCtNodes + (int)(x & 0xffu) : -1;
    };
    int pl[8];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        pl[k] = -1;
        if (!have[k / 2]) continue;
        const uint32_t x = k & 1 ? ec[k / 2] : ea[k / 2], w = ew[k / 2] + 1u;
        pl[k] = place(x);
        if (pl[k] < 0) atomicMax(b.best + x, edge_key(0, ew[k / 2], eg[k / 2]));
        else if (bw[pl[k]] < w) atomicMax(bw + pl[k], w);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (pl[k] >= 0 && bw[pl[k]] == ew[k / 2] + 1u) atomicMax(bg + pl[k], eg[k / 2] * kMix);
    __syncthreads();
#pragma unroll
    for (int i = t; i < 3 * kCtNodes; i += kCtUnits * 32) {
        const uint32_t w = bw[i];
        const int ut = i < kCtNodes ? tile : i < 2 * kCtNodes ? tile + 1 : tile + d.nx;
        if (w) atomicMax(b.best + (uint32_t)ut * kCtNodes + (i & (kCtNodes - 1)),
                         1ull << 48 | (unsigned long long)w << 32 | bg[i]);
    }
}

// ------------------------------------------------------- few nodes: one CTA
// The nodes and edges of up to kSmallTiles tiles, if they fit, are contracted
// by one CTA in shared memory: the rounds of the global kernel below are L2
// round trips and barriers, 5 to 6 us each however little they do. Bound by
// the issue rate of the one SM, so larger batches stay with the L2: a 256 x
// 256 reconstruction takes 44 us against 60, a 512 x 512 one (2600 nodes,
// 8400 edges) 65 against 69.
namespace {
constexpr int kSmallTiles = 128, kSmallNodes = 4096, kSmallEdges = 16384;
constexpr size_t kSmallSmem = sizeof(uint32_t) * (kSmallEdges + 2 * kSmallNodes) + 2 * sizeof(uint16_t) * kSmallNodes;
// An edge is weight << 24 | node << 12 | node, a link word as in the local stage: kRootBit | kSmallDone | S, else
// weight << 16 | parent. A best edge is weight << 14 | mixed position, + 1: ties in no geometric order.
constexpr uint32_t kSmallDone = 0x40000000u, kMixPos = 0x19e5u, kUnmixPos = 0x3bedu;
constexpr uint32_t kPosMask = kSmallEdges - 1;
static_assert(((kMixPos * kUnmixPos) & kPosMask) == 1u, "inverse");

struct SmallSums {
    int node[kSmallTiles + 1], edge[kSmallTiles * kCtUnits + 1];   // exclusive prefix sums over tiles, over units
};

// Sums the batch's nodes and edges; whole CTA. True if they fit.
__device__ __forceinline__ bool small_sums(const CtBatch &b, SmallSums &p)
{
    const int t = threadIdx.x;
    if (b.ntiles > kSmallTiles) return false;   // all threads
    if (t < 32) {
        int nodes = 0, edges = 0;
#pragma unroll
        for (int k = 0; k < kSmallTiles; k += 32) {
            const int i = k + t;
            const int n = i < b.ntiles ? (int)(__ldcg(b.cnt + i) & 0xffffu) : 0;
            const uint32_t e4 = i < b.ntiles ? __ldcg(reinterpret_cast<const uint32_t *>(b.ecnt) + i) : 0u;
            int e[kCtUnits], sum = 0;
#pragma unroll
            for (int q = 0; q < kCtUnits; ++q) sum += e[q] = (int)((e4 >> (8 * q)) & 0xffu);
            int ni = n, ei = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, ni, o), y = __shfl_up_sync(0xffffffffu, ei, o);
                if (t >= o) ni += x, ei += y;
            }
            p.node[i] = nodes + ni - n;
            int at = edges + ei - sum;
#pragma unroll
            for (int q = 0; q < kCtUnits; ++q) {
                p.edge[i * kCtUnits + q] = at;
                at += e[q];
            }
            nodes += __shfl_sync(0xffffffffu, ni, 31);
            edges += __shfl_sync(0xffffffffu, ei, 31);
        }
        if (t == 0) p.node[kSmallTiles] = nodes, p.edge[kSmallTiles * kCtUnits] = edges;
    }
    __syncthreads();
    return p.node[kSmallTiles] <= kSmallNodes && p.edge[kSmallTiles * kCtUnits] <= kSmallEdges;
}

__device__ __forceinline__ void small_contract(const CtBatch &b, const SmallSums &p)
{
    extern __shared__ __align__(16) uint32_t small_smem[];
    uint32_t *E = small_smem;
    volatile uint32_t *link = E + kSmallEdges, *best = link + kSmallNodes;
    volatile uint16_t *act = reinterpret_cast<volatile uint16_t *>(best + kSmallNodes);   // two lists
    __shared__ int s_open[2];
    constexpr int kWarps = kGT / 32, kPer = kSmallNodes / kGT;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t below = (1u << lane) - 1u;
    const int nn = p.node[kSmallTiles], nedge = p.edge[kSmallTiles * kCtUnits];
    if (t < 2) s_open[t] = 0;
    auto key_of = [](uint32_t w, uint32_t pos) { return (w << 14 | ((pos * kMixPos) & kPosMask)) + 1u; };
    // a warp takes whole tiles: their nodes, with round 0's best edges, and their units' edges
#pragma unroll 1
    for (int tile = warp; tile < b.ntiles; tile += kWarps) {
        const int n0 = p.node[tile], n = p.node[tile + 1] - n0;
        for (int i = lane; i < n; i += 32) {
            const unsigned long long l = __ldcg(b.link + tile * kCtNodes + i), k = __ldcg(b.best + tile * kCtNodes + i);
            const uint32_t g = (uint32_t)k * kUnmix;   // the edge's slot
            link[n0 + i] = kRootBit | node_S(l);
            best[n0 + i] = k ? key_of(((uint32_t)(k >> 32) & 0xffffu) - 1u,
                                      (uint32_t)p.edge[g / kCtUnitEdges] + g % kCtUnitEdges) : 0u;
            act[n0 + i] = (uint16_t)(n0 + i);
        }
#pragma unroll
        for (int q = 0; q < kCtUnits; ++q) {
            const int u = tile * kCtUnits + q, e0 = p.edge[u], ne = p.edge[u + 1] - e0;
#pragma unroll 2
            for (int i = lane; i < ne; i += 32) {
                const unsigned long long e = __ldcg(b.edge + (int64_t)u * kCtUnitEdges + i);
                const uint32_t a = (uint32_t)(e >> 28) & kNodeId, c = (uint32_t)e & kNodeId;
                E[e0 + i] = (uint32_t)(e >> 56) << 24 | ((uint32_t)p.node[a >> 8] + (a & 0xffu)) << 12 |
                            ((uint32_t)p.node[c >> 8] + (c & 0xffu));
            }
        }
    }
    __syncthreads();
    // each warp keeps a range of the edges and compacts it in place
    const int per = (((nedge + kWarps - 1) / kWarps) + 31) & ~31;
    const int start = min(warp * per, nedge);
    int cnt = min(per, nedge - start), nl = nn;
#pragma unroll 1
    for (int round = 0;; ++round) {
        int kept = round ? 0 : cnt;
#pragma unroll 1
        for (int i = lane; round && i < cnt + lane; i += 32) {
            bool keep = false, oa = false, oc = false;
            uint32_t a = 0, c = 0, w = 0;
            if (i < cnt) {
                const uint32_t e = E[start + i];
                w = e >> 24;
                a = (e >> 12) & 0xfffu;
                c = e & 0xfffu;
                uint32_t la = link[a], lc = link[c];
                if (!(la & kRootBit)) la = link[a = la & 0xffffu];   // links of the last round are compressed
                if (!(lc & kRootBit)) lc = link[c = lc & 0xffffu];
                oa = !(la & kSmallDone);
                oc = !(lc & kSmallDone);
                keep = a != c && (oa || oc);
            }
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const uint32_t pos = (uint32_t)(start + kept + __popc(m & below));
                E[pos] = w << 24 | a << 12 | c;
                const uint32_t key = key_of(w, pos);
                if (oa && best[a] < key) atomicMax(const_cast<uint32_t *>(best + a), key);
                if (oc && best[c] < key) atomicMax(const_cast<uint32_t *>(best + c), key);
            }
            kept += __popc(m);
            __syncwarp();
        }
        cnt = kept;
        __syncthreads();
        // decisions: w << 16 | parent, or none
        const volatile uint16_t *from = act + (round & 1) * kSmallNodes;
        volatile uint16_t *to = act + (~round & 1) * kSmallNodes;
        constexpr uint32_t kNo = ~0u, kStay = ~0u - 1u;
        uint32_t dec[kPer], id[kPer];
        uint32_t S[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            dec[q] = kNo;
            id[q] = S[q] = 0u;
            if (t + q * kGT >= nl) continue;
            const uint32_t k = from[t + q * kGT], key = best[k], w = (key - 1u) >> 14;
            id[q] = k;
            S[q] = link[k] & 0xffu;
            if (!key || S[q] >= w) {
                dec[q] = kNo;   // final
                continue;
            }
            const uint32_t e = E[((key - 1u) * kUnmixPos) & kPosMask], a = (e >> 12) & 0xfffu, c = e & 0xfffu,
                           o = a == k ? c : a;
            // o joins k by the same edge: the smaller of the two stays
            const bool mutual = k < o && best[o] == key && (link[o] & 0xffu) < w;
            dec[q] = mutual ? kStay : w << 16 | o;
        }
        if (t == 0) s_open[~round & 1] = 0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (t + q * kGT >= nl) continue;
            if (dec[q] == kNo) link[id[q]] = link[id[q]] | kSmallDone;
            else if (dec[q] != kStay) link[id[q]] = dec[q];
            else best[id[q]] = 0u;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (warp * 32 + q * kGT >= nl) continue;   // whole warp
            const bool in = t + q * kGT < nl;
            if (in && dec[q] < kStay) {
                uint32_t w = dec[q] >> 16, x = dec[q] & 0xffffu, v = link[x];
#pragma unroll 1
                for (int n = 0; n < kSmallNodes && !(v & kRootBit); ++n) {
                    w = min(w, v >> 16);
                    x = v & 0xffffu;
                    v = link[x];
                }
                link[id[q]] = w << 16 | x;
                if ((v & 0xffu) < S[q]) atomicMax(const_cast<uint32_t *>(link + x), kRootBit | S[q]);
            }
            const bool stays = in && dec[q] == kStay;
            const uint32_t m = __ballot_sync(0xffffffffu, stays);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&s_open[~round & 1], __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (stays) to[base + __popc(m & below)] = (uint16_t)id[q];
        }
        __syncthreads();
        nl = s_open[~round & 1];
        if (nl == 0) break;
    }
    // every node's value, as a root
#pragma unroll 1
    for (int tile = warp; tile < b.ntiles; tile += kWarps) {
        const int n0 = p.node[tile], n = p.node[tile + 1] - n0;
        for (int i = lane; i < n; i += 32) {
            uint32_t v = 255u, l = link[n0 + i];
#pragma unroll 1
            for (int k = 0; k < kSmallNodes && !(l & kRootBit); ++k) {
                v = min(v, l >> 16);
                l = link[l & 0xffffu];
            }
            const uint32_t g = (uint32_t)(tile * kCtNodes + i);
            b.link[g] = kNodeRoot | (unsigned long long)min(v, l & 0xffu) << 40 | g;
        }
    }
}
}  // namespace

// Contraction of the nodes of the batch. The work is cut into units, four a
// tile; every warp owns the units [u0, u1) and keeps their nodes and, from
// round 1 on, edges compacted at the start of their slots, so no list is
// shared. A round: (1) the edges find their clusters and raise the clusters'
// best edges (round 0: by ct_seam_kernel); (2) every open root takes its
// decision. A grid barrier follows each. Roots that joined are pointed at
// their new root, with the smallest weight on the way, at the start of the
// next round's (1); readers that come first walk on. Bound by the latency of
// dependent reads in L2, so a lane has two edges or roots in flight, and by
// the barriers (8 rounds); one CTA an SM: a barrier's cost is its arrivals at
// one address. CLUSTER: the grid is one cluster, and the barrier the
// hardware's. 1024 x 1024: 50 us (79 with the seams, one in flight and the
// slower barrier), 4096 x 4096: 80 (138), eight of them: 190 (505).
template <bool CLUSTER>
__global__ void __launch_bounds__(kGT, 1) ct_global_kernel(const __grid_constant__ CtBatch b, uint64_t timeout_ns)
{
    const int lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)blockIdx.x * (kGT / 32) + (threadIdx.x >> 5), nw = (int64_t)gridDim.x * (kGT / 32);
    const int64_t units = (int64_t)b.ntiles * kCtUnits;
    const int u0 = (int)(gw * units / nw), u1 = (int)((gw + 1) * units / nw);
    const uint32_t all = 0xffffffffu, below = (1u << lane) - 1u;
    unsigned long long *edge = b.edge + (int64_t)u0 * kCtUnitEdges;
    uint32_t *act = b.act + (int64_t)u0 * kCtUnitNodes;
    unsigned long long *word = reinterpret_cast<unsigned long long *>(b.ctl + kCtCtlBar);
    int ne = 0, na = 0;
    uint32_t target = 0, seen = 0;   // arrivals at the barriers so far, open roots handed in
    // open roots: of the CTA, or (CLUSTER) of the cluster, in turn
    __shared__ uint32_t s_open[3];
    if (threadIdx.x < 3) s_open[threadIdx.x] = 0u;
    __syncthreads();
    if (CLUSTER) {
        __shared__ SmallSums sums;
        if (small_sums(b, sums)) {   // the same answer in every CTA
            if (blockIdx.x == 0) small_contract(b, sums);
            return;
        }
    }
    if (CLUSTER)   // no CTA adds to another's before it is zero
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");

    // this warp's nodes, 32 units at a time
#pragma unroll 1
    for (int ub = u0; ub < u1; ub += 32) {
        const int u = ub + lane;
        const int cn = u < u1 ? (int)(__ldcg(b.cnt + u / kCtUnits) & 0xffffu) : 0;
        const int mine = max(0, (cn - u % kCtUnits + kCtUnits - 1) / kCtUnits);
#pragma unroll 1
        for (int j = 0; j < 32 && ub + j < u1; ++j) {
            const int n = __shfl_sync(all, mine, j);
            const uint32_t first = (uint32_t)((ub + j) / kCtUnits * kCtNodes + (ub + j) % kCtUnits);
#pragma unroll 1
            for (int i = lane; i < n; i += 32) act[na + i] = first + (uint32_t)(i * kCtUnits);
            na += n;
        }
    }
    __syncwarp();

    // (1) on two edges a lane; they move to the front of the warp's slots
    int kept = 0;
    auto edges = [&](int round, const unsigned long long (&e)[2], const bool (&have)[2]) {   // whole warp
        uint32_t x[4];
        unsigned long long l[4];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            x[2 * k] = (uint32_t)(e[k] >> 28) & kNodeId;
            x[2 * k + 1] = (uint32_t)e[k] & kNodeId;
        }
        ct_roots(b, x, l, have);
        bool keep[2], oa[2], oc[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            oa[k] = !(l[2 * k] & kNodeDone);
            oc[k] = !(l[2 * k + 1] & kNodeDone);
            keep[k] = have[k] && x[2 * k] != x[2 * k + 1] && (oa[k] || oc[k]);
        }
        __syncwarp();
        unsigned long long old[4], key[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t m = __ballot_sync(all, keep[k]);
            const int at = kept + __popc(m & below);
            const uint32_t w = (uint32_t)(e[k] >> 56);
            key[k] = edge_key(round, w, (uint32_t)u0 * kCtUnitEdges + at);
            if (keep[k]) edge[at] = node_edge(x[2 * k], x[2 * k + 1], w);
            kept += __popc(m);
            old[2 * k] = keep[k] && oa[k] ? __ldcg(b.best + x[2 * k]) : ~0ull;
            old[2 * k + 1] = keep[k] && oc[k] ? __ldcg(b.best + x[2 * k + 1]) : ~0ull;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (old[k] < key[k / 2]) atomicMax(b.best + x[k], key[k / 2]);
    };

#pragma unroll 1
    for (int round = 0; round < kMaxRounds; ++round) {
        if (round > 0) {
            // (0) roots that joined: final links of the last round; the others stay open
            kept = 0;
#pragma unroll 1
            for (int i = 0; i < na; i += 32) {
                bool open = false;
                uint32_t r = 0;
                if (i + lane < na) {
                    r = act[i + lane];
                    unsigned long long l = __ldcg(b.link + r);
                    open = (l & kNodeRoot) != 0ull;
                    if (!open) {
                        const uint32_t S = b.S[r];   // stored by this warp when it joined
                        uint32_t w = (uint32_t)(l >> 32), x = (uint32_t)l;
#pragma unroll 1
                        for (int n = 0; n < (1 << 20); ++n) {
                            l = __ldcg(b.link + x);
                            if (l & kNodeRoot) break;
                            w = min(w, (uint32_t)(l >> 32));
                            x = (uint32_t)l;
                        }
                        __stcg(b.link + r, (unsigned long long)w << 32 | x);
                        if (node_S(l) < S) atomicMax(b.link + x, kNodeRoot | (unsigned long long)S << 40 | x);
                    }
                }
                const uint32_t m = __ballot_sync(all, open);
                if (open) act[kept + __popc(m & below)] = r;
                kept += __popc(m);
                __syncwarp();
            }
            na = kept;
            // (1) edges; a key holds the round, so the last round's bests count as none
            kept = 0;
            if (round == 1) {
                // out of the units' own slots: their edges in a row, a lane finds its by the units' prefix sums
#pragma unroll 1
                for (int ub = u0; ub < u1; ub += 32) {
                    const int n = ub + lane < u1 ? (int)__ldcg(b.ecnt + ub + lane) : 0;
                    int end = n;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(all, end, o);
                        if (lane >= o) end += v;
                    }
                    const int total = __shfl_sync(all, end, 31);
#pragma unroll 1
                    for (int i = 0; i < total; i += 64) {
                        unsigned long long e[2];
                        bool have[2];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const int f = i + 32 * k + lane;
                            int j = 0;   // units that end at or before f
#pragma unroll
                            for (int o = 16; o > 0; o >>= 1)
                                if (__shfl_sync(all, end, j + o - 1) <= f) j += o;
                            const int first = __shfl_sync(all, end - n, j & 31);
                            have[k] = f < total;
                            e[k] = have[k] ? __ldcg(b.edge + (int64_t)(ub + j) * kCtUnitEdges + (f - first)) : 0ull;
                        }
                        edges(round, e, have);
                        __syncwarp();
                    }
                }
            } else {
#pragma unroll 1
                for (int i = 0; i < ne; i += 64) {
                    unsigned long long e[2];
                    bool have[2];
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        have[k] = i + 32 * k + lane < ne;
                        e[k] = have[k] ? edge[i + 32 * k + lane] : 0ull;
                    }
                    edges(round, e, have);
                    __syncwarp();
                }
            }
            ne = kept;
            // open roots of the batch: all of them hand in theirs with the barrier
            const int slot = round % 3;
            uint32_t open;
            if (CLUSTER) {
                if (na && lane < kGCluster) {
                    uint32_t at = (uint32_t)__cvta_generic_to_shared(s_open + slot);
                    asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(at) : "r"(lane));
                    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(at), "r"(na) : "memory");
                }
                if (threadIdx.x == 0) s_open[(round + 1) % 3] = 0u;   // last read two rounds ago
                __syncwarp();
                asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
                open = *(volatile uint32_t *)(s_open + slot);
            } else {
                if (na && lane == 0) atomicAdd(s_open + slot, (uint32_t)na);
                __syncthreads();
                uint32_t sum;
                if (!sum_barrier(word, target += gridDim.x, s_open[slot], sum, b.err, timeout_ns)) return;
                if (threadIdx.x == 0) s_open[slot] = 0u;
                open = sum - seen;
                seen = sum;
            }
            if (open == 0u) return;
        }
        // (2) decisions, two a lane
        kept = 0;
#pragma unroll 1
        for (int i = 0; i < na; i += 64) {
            bool in[2], open[2];
            uint32_t r[2], w[2], S[2];
            unsigned long long key[2], e[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                in[k] = i + 32 * k + lane < na;
                r[k] = in[k] ? act[i + 32 * k + lane] : 0u;
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                key[k] = in[k] ? __ldcg(b.best + r[k]) : 0ull;
                S[k] = in[k] ? node_S(__ldcg(b.link + r[k])) : 0u;
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool some = (uint32_t)(key[k] >> 48) == (uint32_t)(round + 1);
                w[k] = ((uint32_t)(key[k] >> 32) & 0xffffu) - 1u;
                open[k] = in[k] && some && S[k] < w[k];
                e[k] = open[k] ? __ldcg(b.edge + (uint32_t)key[k] * kUnmix) : 0ull;
                if (in[k] && !open[k]) atomicOr(b.link + r[k], kNodeDone);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (open[k]) {
                    const uint32_t a = (uint32_t)(e[k] >> 28) & kNodeId, c = (uint32_t)e[k] & kNodeId,
                                   o = a == r[k] ? c : a;
                    // o joins r by the same edge: the smaller of the two stays
                    // (o may have joined already; its link word is no root's then)
                    bool mutual = false;
                    if (r[k] < o && __ldcg(b.best + o) == key[k]) {
                        const unsigned long long lo = __ldcg(b.link + o);
                        mutual = !(lo & kNodeRoot) || node_S(lo) < w[k];
                    }
                    if (!mutual) {
                        b.S[r[k]] = S[k];
                        __stcg(b.link + r[k], (unsigned long long)w[k] << 32 | o);
                    }
                }
                const uint32_t m = __ballot_sync(all, open[k]);
                if (open[k]) act[kept + __popc(m & below)] = r[k];
                kept += __popc(m);
                __syncwarp();
            }
        }
        na = kept;
        if (CLUSTER) {
            asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else {
            __syncthreads();
            uint32_t sum;
            if (!sum_barrier(word, target += gridDim.x, 0u, sum, b.err, timeout_ns)) return;
        }
    }
    raise_status(b.err, RT_ETIMEOUT);   // not reached: every round at least halves the open roots of a component
}

// ----------------------------------------------------------------- output
// CTA of 128 threads per tile, 32 pixels of a row each. Bound by the latency
// of the walks from the tile's nodes to their roots, so as many tiles as
// possible share an SM and the pixels' words are on their way meanwhile (256
// threads and loads after the walk: 125 us for eight 4096 x 4096 tiles; now
// 96).
constexpr int kOutThreads = 128;
__global__ void __launch_bounds__(kOutThreads) ct_out_kernel(const __grid_constant__ CtBatch b, int threshold)
{
    start_early();
    __shared__ uint8_t val[kCtNodes];
    const int tile = blockIdx.x, t = threadIdx.x;
    const uint4 *src = reinterpret_cast<const uint4 *>(b.plane + (int64_t)tile * kCtPx + t * 32);
    const uint4 s0 = __ldcs(src), s1 = __ldcs(src + 1), s2 = __ldcs(src + 2), s3 = __ldcs(src + 3);
    const int nn = (int)(b.cnt[tile] & 0xffffu);
    const CtImage &d = ct_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
#pragma unroll
    for (int k = t; k < kCtNodes; k += kOutThreads) {
        uint32_t v = 255u;
        if (k < nn) {
            unsigned long long l = b.link[(uint32_t)tile * kCtNodes + k];
#pragma unroll 1
            for (int n = 0; n < (1 << 20) && !(l & kNodeRoot); ++n) {
                v = min(v, (uint32_t)(l >> 32));
                l = b.link[(uint32_t)l];
            }
            v = min(v, node_S(l));
        }
        val[k] = (uint8_t)v;
    }
    __syncthreads();
    const int r = ty * kCtSide + (t >> 1), c = tx * kCtSide + (t & 1) * 32;
    const int n = r < d.H ? min(32, d.W - c) : 0;   // may be negative: none
    const uint32_t e[16] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w,
                            s2.x, s2.y, s2.z, s2.w, s3.x, s3.y, s3.z, s3.w};
    uint32_t R[8] = {0, 0, 0, 0, 0, 0, 0, 0}, B = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const uint32_t x = (e[k >> 1] >> (16 * (k & 1))) & 0xffffu;
        const uint32_t p = min(x & 0xffu, (uint32_t)val[x >> 8]);
        R[k >> 2] |= p << (8 * (k & 3));
        B |= (uint32_t)((int)p < threshold) << k;
    }
    // nothing past the image
    if (b.bits) reinterpret_cast<uint32_t *>(b.bits + (int64_t)tile * kCtSide)[t] = n >= 32 ? B : n > 0 ? B & ((1u << n) - 1u) : 0u;
    if (!d.out) return;
    const uint32_t next = __shfl_down_sync(0xffffffffu, R[0], 1);   // half a row further
    if (n <= 0) return;
    uint8_t *o = d.out + (int64_t)r * d.ld_out + c;
    const int head = (int)(-(uintptr_t)o & 3u);
    if (head && d.W - tx * kCtSide >= kCtSide) {   // the row's aligned words, shifted together; its ends by bytes
        const bool first = (t & 1) == 0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < 7 || first)
                *reinterpret_cast<uint32_t *>(o + head + 4 * k) = __funnelshift_r(R[k], k < 7 ? R[k + 1 < 8 ? k + 1 : 7] : next, 8u * head);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (first && k < head) o[k] = (uint8_t)(R[0] >> (8 * k));
            if (!first && k >= head) o[28 + k] = (uint8_t)(R[7] >> (8 * k));
        }
    } else {
        store_bytes(o, n, R);
    }
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
    d.out = nullptr;
    d.ld_out = 0;
    b.ntiles += d.nx * d.ny;
}

cudaError_t launch_contract(const CtBatch &b, int num_sms, uint64_t timeout_ns, cudaStream_t s)
{
    const bool given = b.img[0].marker != nullptr;   // all images of a batch, or none
    // With two tiles per SM or fewer little hides a tile's latency: then 512
    // threads share it (512 x 512: 66 us against 75 for all stages, 1024 x
    // 1024: 85 against 90; equal at 1280 x 1280, and above that the barriers
    // of larger CTAs cost more: 108 against 102 at 1536 x 1536).
    const bool few = b.ntiles <= kFewTiles;
    auto *fn = few ? (given ? ct_local_kernel<true, 512> : ct_local_kernel<false, 512>)
                   : (given ? ct_local_kernel<true, 256> : ct_local_kernel<false, 256>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLocalSmem);
    if (e != cudaSuccess) return e;
    launch_early(fn, (unsigned)b.ntiles, few ? 512 : 256, kLocalSmem, s, b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_early(ct_seam_kernel, (unsigned)b.ntiles, kCtUnits * 32, 0, s, b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t units = (int64_t)b.ntiles * kCtUnits;
    const int need = (int)ceil_div(units, kGT / 32);
    // One cluster of eight CTAs while its 256 warps hold two units each at
    // most (640 x 640: 71 us against 73 for all stages; 768 x 768: equal; 1024
    // x 1024: 88 against 85); a smaller one may fit a single CTA.
    if (units <= kGClusterUnits) {
        auto *gfn = ct_global_kernel<true>;
        e = cudaFuncSetAttribute(gfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kGCluster);
        cfg.blockDim = dim3(kGT);
        cfg.dynamicSmemBytes = kSmallSmem;
        cfg.stream = s;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kGCluster;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, gfn, b, timeout_ns);
    }
    CtBatch bb = b;
    void *args[] = {&bb, &timeout_ns};
    return cudaLaunchCooperativeKernel((const void *)ct_global_kernel<false>, dim3((unsigned)(need < num_sms ? need : num_sms)),
                                       dim3(kGT), args, 0, s);
}

cudaError_t launch_contract_out(const CtBatch &b, int threshold, cudaStream_t s)
{
    launch_early(ct_out_kernel, (unsigned)b.ntiles, kOutThreads, 0, s, b, threshold);
    return cudaGetLastError();
}

}  // namespace rtk
