// FillHoles (Sections 3.2.1 and 5.1) and BWLabel + AreaThreshold (Sections
// 5.1 and 3.2.1) by union-find over the runs of bit rows.
//
// An image is a bit plane cut into tiles of 64 rows x 64 columns, one 64-bit
// word per row; a warp takes a tile, a lane two rows. A maximal run of set
// bits is one node from the start (a row of a nuclei tile has one or two),
// and two runs of adjacent rows are joined once, where they first touch:
// bit operations on the two words list those places. So the work follows
// the number of runs, not of pixels. The forest's roots are always the
// smaller run, so a component's root is its first run in raster order and
// the root's first pixel the canonical label.
//
// Components that touch a side with a neighbour tile get a slot of the tile;
// a warp per tile joins the slots across its right and lower seams in
// global memory. Everything else is decided inside its tile.
//   * fill: the components are those of the background. One inside a tile
//     is a hole at once; the slots of components on the image border start
//     below node 0, the outside, and after the seams a slot whose root is
//     not 0 is a hole.
//   * labels: the components of the foreground, with their areas and first
//     pixels summed over the slots of a tree. The output stage reads the
//     tile's run words back and writes labels, the kept bits and the count.
//
// Measured on one GB300 as stages of the chain, where the bits are there
// already and the fill's last launch also makes the labels' local components,
// nuclei tiles: the fill of eight 4096 x 4096 tiles takes 222 us (281 as
// bit-plane floods swept to a fixed point), their labels 137 (661 as a
// union-find over pixels); one tile 55 (109) and 40 (101); a 1024 x 1024 tile
// 43 (79) and 25 (35). (rt_label_area, a call of its own, packs bytes to bits
// first and makes its local components itself; with these two launches more
// the pixels win on small images: kUfMaxTiles in ccl.cuh.) The local stages
// are bound by the latency of the tiles with the most runs, the label stage by
// its stores (4 bytes a pixel). Speckle, whose runs are about as many as its
// pixels, is where floods were faster: rt_fill_holes on 4096 x 4096 pixels of
// which 60 % are set at random 80 -> 284 us.
#include "runs.cuh"

namespace rtk {

namespace {

typedef unsigned long long u64;

constexpr int kFewTiles = 2048;
constexpr int kWarps = 4;                 // tiles per CTA; 1 while they fit in one wave (kFewTiles)
// Shared memory: a warp's share holds a tile of up to kLightRuns runs (most
// nuclei tiles) and lists the pairs of touching runs to join kLightPairs at a
// time. A tile with more (up to kMaxRuns) waits until the other warps are done
// and takes the whole block's. With room for the worst tile at every warp an
// SM held 22 tiles; now it holds 32 or more, and 16 to 22 of an image of
// nothing but heavy tiles. Eight 4096 x 4096 tiles: the local stages 80 and
// 137 -> 63 and 114 us; one: 19 and 33 -> 17 and 27. Few tiles (kFewTiles)
// fit all the same, and a heavy one would only wait, so there a block has one
// warp (ALONE): 1024 x 1024 20 us against 22.
constexpr int kMaxRuns = kRunWords;
constexpr int kLightRuns = 384, kLightPairs = 256, kWarpWords = kLightRuns + kLightPairs;
constexpr int kHeavyPairs = kWarps * kWarpWords - kMaxRuns;
constexpr size_t kRunSmem = sizeof(uint32_t) * kWarpWords * kWarps;
template <bool ALONE>
struct Mem {
    bool heavy;
    __device__ __forceinline__ volatile uint32_t *runs() const   // a word per run
    {
        extern __shared__ uint32_t run_smem[];
        return run_smem + (ALONE || heavy ? 0 : (threadIdx.x >> 5) * kWarpWords);
    }
    __device__ __forceinline__ volatile uint32_t *pairs() const { return runs() + (ALONE || heavy ? kMaxRuns : kLightRuns); }
    __device__ __forceinline__ int cap() const { return ALONE || heavy ? kHeavyPairs : kLightPairs; }
};
// Calls f(memory of the tile) for every warp of the block with its number of
// runs; all threads of the block call it. ALONE: a block of one warp.
template <bool ALONE, class F>
__device__ __forceinline__ void with_memory(int runs, F &&f)
{
    if (ALONE) {
        f(Mem<ALONE>{false});
        return;
    }
    const bool heavy = runs > kLightRuns;
    if (!heavy) f(Mem<ALONE>{false});
    if (!__syncthreads_or(heavy)) return;
#pragma unroll 1
    for (int turn = 0; turn < kWarps; ++turn) {
        if (heavy && turn == (int)(threadIdx.x >> 5)) f(Mem<ALONE>{true});
        __syncthreads();
    }
}
constexpr uint32_t kRim = 1u << 31, kBorder = 1u << 30, kParent = 0xffffu;
constexpr int kSlotShift = 16;
constexpr uint32_t kSlotMask = kRunSlots - 1;

__device__ __forceinline__ const RunImage &run_image(const RunBatch &b, int t)
{
    int k = 0;
    while (k + 1 < b.n && t >= b.img[k + 1].tile_base) ++k;
    return b.img[k];
}

__device__ __forceinline__ u64 shfl64(u64 v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

// ------------------------------------------------------------ global forest
// U[x] holds the parent of node x as a mixed number, mix(x) = x * kMix; the
// smaller mixed number is the root. Neighbouring tiles' nodes are ordered at
// random that way: linked by their own numbers the background of a large
// image grows chains as long as the tile grid (an empty image's seams took
// 100 us at 1024 x 1024). Node 0, the outside, stays the smallest. Hooking
// and halving are both atomicMin, so every parent only moves down in the same
// growing tree while unions run concurrently.
constexpr uint32_t kMix = 2654435761u, kUnmix = 244002641u;   // inverses mod 2^32
static_assert(kMix * kUnmix == 1u, "inverse");
__device__ __forceinline__ uint32_t mix(uint32_t x) { return x * kMix; }
__device__ __forceinline__ uint32_t parent(const uint32_t *U, uint32_t v) { return __ldcg(U + v * kUnmix); }

__device__ __forceinline__ uint32_t node_find(uint32_t *U, uint32_t v)
{
    uint32_t p = parent(U, v);
    while (p != v) {
        if (p == 0u) return 0u;   // the outside: no need to read its word, which all would read
        const uint32_t gp = parent(U, p);
        if (gp != p) atomicMin(U + v * kUnmix, gp);
        v = gp;
        p = parent(U, v);
    }
    return v;
}
__device__ __forceinline__ void node_union(uint32_t *U, uint32_t a, uint32_t b)
{
    a = mix(a);
    b = mix(b);
    for (;;) {
        a = node_find(U, a);
        b = node_find(U, b);
        if (a == b) return;
        if (a < b) {
            const uint32_t t = a;
            a = b;
            b = t;
        }
        const uint32_t old = atomicMin(U + a * kUnmix, b);
        if (old == a) return;
        a = old;
    }
}

// --------------------------------------------------------------------- runs
// The runs of a warp's tile: two rows per lane. Run ids count the runs in
// raster order.
struct Runs {
    u64 m[2], st[2];     // rows 2 lane, 2 lane + 1: bits, first bits of runs
    int n[2], base[2];   // runs of the row, id of its first
    int total;           // runs of the tile

    __device__ __forceinline__ int id(int j, int pos) const { return base[j] + __popcll(st[j] & (~0ull >> (63 - pos))) - 1; }
};

// Points every run at its root: a word is written by its own lane only, and
// moves to its grandparent until nothing moves. Whole warp.
__device__ __forceinline__ void flatten(volatile uint32_t *P, int total, int lane)
{
    for (;;) {
        bool more = false;
        for (int i = lane; i < total; i += 32) {
            const uint32_t q = P[i], g = P[q];
            if (g != q) {
                P[i] = g;
                more = true;
            }
        }
        __syncwarp();
        if (!__any_sync(0xffffffffu, more)) return;
    }
}

__device__ __forceinline__ int count_runs(u64 m0, u64 m1)
{
    return (int)__reduce_add_sync(0xffffffffu, (uint32_t)(__popcll(m0 & ~(m0 << 1)) + __popcll(m1 & ~(m1 << 1))));
}

// The runs of (m0, m1).
__device__ __forceinline__ Runs runs_of(u64 m0, u64 m1, int lane)
{
    Runs r;
    r.m[0] = m0;
    r.m[1] = m1;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        r.st[j] = r.m[j] & ~(r.m[j] << 1);
        r.n[j] = __popcll(r.st[j]);
    }
    int inc = r.n[0] + r.n[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    r.base[0] = inc - r.n[0] - r.n[1];
    r.base[1] = r.base[0] + r.n[0];
    r.total = __shfl_sync(0xffffffffu, inc, 31);
    return r;
}

// Components of the runs of (m0, m1): afterwards P[run] is its root run
// (upper bits 0). Whole warp.
// The lanes list the places where two runs of adjacent rows first touch (the
// first column of a stretch they share, or, for 8-connectivity, a corner),
// then all lanes share the list: every pair whose roots differ hooks the
// larger root under the smaller (lost to another pair's hook, it stays for
// the next round), the trees are flattened, and at least half of the
// components that can still join are gone. Unions by the rows' own lanes, one
// after the other, kept a speckled nucleus's few lanes busy for 25 us a tile.
template <int CONN, bool ALONE>
__device__ __forceinline__ Runs components(u64 m0, u64 m1, const Mem<ALONE> &mem, int lane)
{
    volatile uint32_t *P = mem.runs(), *pairs = mem.pairs();
    const int cap = mem.cap();
    const Runs r = runs_of(m0, m1, lane);
    const uint32_t below = (1u << lane) - 1u;
    for (int i = lane; i < r.total; i += 32) P[i] = (uint32_t)i;
    // the next lane's first row
    u64 dm = __shfl_down_sync(0xffffffffu, r.m[0], 1);
    const u64 dst = __shfl_down_sync(0xffffffffu, r.st[0], 1);
    const int dbase = __shfl_down_sync(0xffffffffu, r.base[0], 1);
    if (lane == 31) dm = 0ull;
    auto touch = [](u64 a, u64 b) {
        const u64 e = a & b;
        return e & ~(e << 1);
    };
    // right: a's run and b's run one column further; left: one column back
    auto right_of = [](u64 a, u64 b) { return CONN == 8 ? a & (b >> 1) & ~(a >> 1) & ~b : 0ull; };
    auto left_of = [](u64 a, u64 b) { return CONN == 8 ? a & (b << 1) & ~(a << 1) & ~b : 0ull; };
    u64 e[6] = {touch(r.m[0], r.m[1]), right_of(r.m[0], r.m[1]), left_of(r.m[0], r.m[1]),
                touch(r.m[1], dm),     right_of(r.m[1], dm),     left_of(r.m[1], dm)};
    for (;;) {
        int n = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            if (CONN == 4 && k % 3) continue;
            const u64 sa = k < 3 ? r.st[0] : r.st[1], sb = k < 3 ? r.st[1] : dst;
            const int ba = k < 3 ? r.base[0] : r.base[1], bb = k < 3 ? r.base[1] : dbase;
            constexpr int kStep[3] = {0, 1, -1};
#pragma unroll 1
            while (n + 32 <= cap && __any_sync(0xffffffffu, e[k] != 0ull)) {
                const bool some = e[k] != 0ull;
                const uint32_t m = __ballot_sync(0xffffffffu, some);
                if (some) {
                    const int pos = __ffsll((long long)e[k]) - 1;
                    e[k] &= e[k] - 1;
                    const uint32_t a = (uint32_t)(ba + __popcll(sa & (~0ull >> (63 - pos))) - 1),
                                   c = (uint32_t)(bb + __popcll(sb & (~0ull >> (63 - pos - kStep[k % 3]))) - 1);
                    pairs[n + __popc(m & below)] = a | c << 16;
                }
                n += __popc(m);
            }
        }
        __syncwarp();
        if (n == 0) return r;
        while (n) {
            int kept = 0;
            for (int i = 0; i < n; i += 32) {
                bool open = false;
                uint32_t v = 0;
                if (i + lane < n) {
                    v = pairs[i + lane];
                    const uint32_t a = P[v & 0xffffu], c = P[v >> 16];
                    open = a != c;
                    if (open) {
                        atomicMin(const_cast<uint32_t *>(P + max(a, c)), min(a, c));
                        v = a | c << 16;
                    }
                }
                const uint32_t m = __ballot_sync(0xffffffffu, open);
                if (open) pairs[kept + __popc(m & below)] = v;
                kept += __popc(m);
                __syncwarp();
            }
            n = kept;
            if (n) flatten(P, r.total, lane);
        }
    }
}

// Where a tile lies.
struct Place {
    int tile, ty, tx, r0, c0;
    bool open[4];   // top, bottom, left, right: there is a neighbour tile
};
__device__ __forceinline__ Place place_of(const RunImage &d, int tile)
{
    Place p;
    const int lt = tile - d.tile_base;
    p.tile = tile;
    p.ty = lt / d.nx;
    p.tx = lt - p.ty * d.nx;
    p.r0 = p.ty * kRunSide;
    p.c0 = p.tx * kRunSide;
    p.open[0] = p.ty > 0;
    p.open[1] = p.ty + 1 < d.ny;
    p.open[2] = p.tx > 0;
    p.open[3] = p.tx + 1 < d.nx;
    return p;
}
// The bits of row r0 + i of the tile that lie inside the image.
__device__ __forceinline__ u64 exists(const RunImage &d, const Place &p, int i)
{
    if (p.r0 + i >= d.H) return 0ull;
    const int n = d.W - p.c0;   // >= 1
    return n >= kRunSide ? ~0ull : (1ull << n) - 1ull;
}

// Flags the roots of the runs [first, first + n).
__device__ __forceinline__ void flag_runs(volatile uint32_t *P, int first, int n, uint32_t flag, int lane)
{
    for (int i = lane; i < n; i += 32) atomicOr(const_cast<uint32_t *>(P + (P[first + i] & kParent)), flag);
}

// Marks the roots of components on the open sides (kRim).
__device__ __forceinline__ void flag_rim(const Runs &r, const Place &p, volatile uint32_t *P, int lane)
{
    if (p.open[0]) flag_runs(P, 0, __shfl_sync(0xffffffffu, r.n[0], 0), kRim, lane);
    if (p.open[1]) {
        const int n = __shfl_sync(0xffffffffu, r.n[1], 31);
        flag_runs(P, r.total - n, n, kRim, lane);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        if (p.open[2] && (r.m[j] & 1ull)) atomicOr(const_cast<uint32_t *>(P + (P[r.base[j]] & kParent)), kRim);
        if (p.open[3] && (r.m[j] >> 63)) atomicOr(const_cast<uint32_t *>(P + (P[r.base[j] + r.n[j] - 1] & kParent)), kRim);
    }
    __syncwarp();
}

// Numbers the marked roots in order: their slots. f(run, slot) per slot.
template <class F>
__device__ __forceinline__ int number_slots(const Runs &r, volatile uint32_t *P, int lane, F &&f)
{
    int cnt = 0;
    for (int i0 = 0; i0 < r.total; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t v = i < r.total ? P[i] : 0u;
        const bool slot = (v & kRim) && (v & kParent) == (uint32_t)i;
        const uint32_t m = __ballot_sync(0xffffffffu, slot);
        if (slot) {
            const int k = cnt + __popc(m & ((1u << lane) - 1u));
            P[i] = v | (uint32_t)k << kSlotShift;
            f(i, k);
        }
        cnt += __popc(m);
    }
    __syncwarp();
    return cnt;
}

// Writes the slots of the pixels on the open sides.
__device__ __forceinline__ void write_sides(const RunBatch &b, const Runs &r, const Place &p, const volatile uint32_t *P,
                                            int lane)
{
    uint8_t *s = b.sides + (int64_t)p.tile * kRunSides;
    auto slot = [&](int run) { return (P[P[run] & kParent] >> kSlotShift) & kSlotMask; };
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (!p.open[k]) continue;
        const u64 m = shfl64(r.m[k], k ? 31 : 0), st = shfl64(r.st[k], k ? 31 : 0);
        const int base = __shfl_sync(0xffffffffu, r.base[k], k ? 31 : 0);
        uint32_t v = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int c = 2 * lane + q;
            const uint32_t x = (m >> c) & 1ull ? slot(base + __popcll(st & (~0ull >> (63 - c))) - 1) : 255u;
            v |= x << (8 * q);
        }
        reinterpret_cast<uint16_t *>(s + k * kRunSide)[lane] = (uint16_t)v;
    }
    if (p.open[2]) {
        const uint32_t a = r.m[0] & 1ull ? slot(r.base[0]) : 255u, c = r.m[1] & 1ull ? slot(r.base[1]) : 255u;
        reinterpret_cast<uint16_t *>(s + 2 * kRunSide)[lane] = (uint16_t)(a | c << 8);
    }
    if (p.open[3]) {
        const uint32_t a = r.m[0] >> 63 ? slot(r.base[0] + r.n[0] - 1) : 255u,
                       c = r.m[1] >> 63 ? slot(r.base[1] + r.n[1] - 1) : 255u;
        reinterpret_cast<uint16_t *>(s + 3 * kRunSide)[lane] = (uint16_t)(a | c << 8);
    }
}

// The bits of the run that starts at pos (a first bit of m).
__device__ __forceinline__ u64 run_bits(u64 m, int pos) { return m & ~(m + (1ull << pos)); }

// Background components of a tile (foreground f), marked kRim and kBorder
// (on the image border, or SEEDS: with a pixel of seed), the rim ones
// numbered.
template <int CONN, bool SEEDS, bool ALONE, class F>
__device__ __forceinline__ Runs background(const RunImage &d, const Place &p, ulonglong2 f, ulonglong2 seed,
                                           const Mem<ALONE> &mem, int lane, int &cnt, F &&fn)
{
    volatile uint32_t *P = mem.runs();
    const Runs r = components<CONN>(exists(d, p, 2 * lane) & ~f.x, exists(d, p, 2 * lane + 1) & ~f.y, mem, lane);
    if (SEEDS) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            u64 s = r.st[j];
            for (int k = 0; s; ++k, s &= s - 1)
                if (run_bits(r.m[j], __ffsll((long long)s) - 1) & (j ? seed.y : seed.x))
                    atomicOr(const_cast<uint32_t *>(P + (P[r.base[j] + k] & kParent)), kBorder);
        }
    } else {
        if (p.ty == 0) flag_runs(P, 0, __shfl_sync(0xffffffffu, r.n[0], 0), kBorder, lane);
        const int last = d.H - 1 - p.r0;
        if (last < kRunSide) {   // whole warp
            const int first = __shfl_sync(0xffffffffu, last & 1 ? r.base[1] : r.base[0], last >> 1);
            const int n = __shfl_sync(0xffffffffu, last & 1 ? r.n[1] : r.n[0], last >> 1);
            flag_runs(P, first, n, kBorder, lane);
        }
        const int right = d.W - 1 - p.c0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (p.tx == 0 && (r.m[j] & 1ull)) atomicOr(const_cast<uint32_t *>(P + (P[r.base[j]] & kParent)), kBorder);
            if (right < kRunSide && ((r.m[j] >> right) & 1ull))
                atomicOr(const_cast<uint32_t *>(P + (P[r.id(j, right)] & kParent)), kBorder);
        }
    }
    flag_rim(r, p, P, lane);
    cnt = number_slots(r, P, lane, fn);
    return r;
}

// The local stage of a fill in forest U: holes inside the tile are known
// afterwards (words), the other background components become slots.
template <int CONN, bool SEEDS, bool ALONE>
__device__ __forceinline__ void fill_tile(const RunBatch &b, uint32_t *U, const RunImage &d, const Place &p, ulonglong2 f,
                                          ulonglong2 seed, const Mem<ALONE> &mem, int lane)
{
    const uint32_t node = 1u + (uint32_t)p.tile * kRunSlots;
    if (p.tile == 0 && lane == 0) U[0] = 0u;
    if (!__any_sync(0xffffffffu, (f.x | f.y) != 0ull)) {   // nothing but background (no words): one component
        const bool border = SEEDS ? __any_sync(0xffffffffu, (seed.x | seed.y) != 0ull)
                                  : p.ty == 0 || p.tx == 0 || p.r0 + kRunSide >= d.H || p.c0 + kRunSide >= d.W;
        const bool rim = p.open[0] || p.open[1] || p.open[2] || p.open[3];
        uint16_t *s = reinterpret_cast<uint16_t *>(b.sides + (int64_t)p.tile * kRunSides) + lane;
        const int nr = min(kRunSide, d.H - p.r0), nc = min(kRunSide, d.W - p.c0);
        auto pair = [&](int n) { return (uint16_t)((2 * lane < n ? 0u : 255u) | (2 * lane + 1 < n ? 0u : 255u) << 8); };
        if (p.open[0]) s[0] = pair(nc);
        if (p.open[1]) s[kRunSide / 2] = pair(nc);
        if (p.open[2]) s[2 * kRunSide / 2] = pair(nr);
        if (p.open[3]) s[3 * kRunSide / 2] = pair(nr);
        if (lane == 0) {
            b.cnt[p.tile] = rim ? 1u : 0u;   // no neighbour: the whole image, whose border is outside
            if (rim) U[node] = border ? 0u : mix(node);
        }
        return;
    }
    volatile uint32_t *P = mem.runs();
    int cnt = 0;
    const Runs r = background<CONN, SEEDS>(d, p, f, seed, mem, lane, cnt, [&](int i, int k) {
        U[node + k] = P[i] & kBorder ? 0u : mix(node + k);
    });
    uint32_t *words = b.words + (int64_t)p.tile * kRunWords;
    for (int i = lane; i < r.total; i += 32) words[i] = P[i];
    write_sides(b, r, p, P, lane);
    if (lane == 0) b.cnt[p.tile] = (uint8_t)cnt;
}

// The holes of the fill in U: components that neither are outside in the tile
// nor reach it through their slot. From fill_tile's words.
template <bool ALONE>
__device__ __forceinline__ ulonglong2 holes_of(const RunBatch &b, uint32_t *U, const RunImage &d, const Place &p,
                                               ulonglong2 f, const Mem<ALONE> &mem, int lane)
{
    const uint32_t node = 1u + (uint32_t)p.tile * kRunSlots;
    u64 add[2] = {0ull, 0ull};
    if (!__any_sync(0xffffffffu, (f.x | f.y) != 0ull)) {
        if (b.cnt[p.tile] && node_find(U, mix(node)) != 0u) {
            add[0] = exists(d, p, 2 * lane);
            add[1] = exists(d, p, 2 * lane + 1);
        }
    } else {
        volatile uint32_t *P = mem.runs();
        const Runs r = runs_of(exists(d, p, 2 * lane) & ~f.x, exists(d, p, 2 * lane + 1) & ~f.y, lane);
        const uint32_t *words = b.words + (int64_t)p.tile * kRunWords;
        for (int i = lane; i < r.total; i += 32) {
            uint32_t v = words[i];
            if ((v & kParent) == (uint32_t)i) {   // roots: kBorder if outside
                if ((v & kRim) && node_find(U, mix(node + ((v >> kSlotShift) & kSlotMask))) == 0u) v |= kBorder;
                v = (v & kBorder) | (uint32_t)i;
            }
            P[i] = v;
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            u64 s = r.st[j];
            for (int k = 0; s; ++k, s &= s - 1)
                if (!(P[P[r.base[j] + k] & kParent] & kBorder))
                    add[j] |= run_bits(r.m[j], __ffsll((long long)s) - 1);
        }
        __syncwarp();
    }
    return make_ulonglong2(add[0], add[1]);
}

}  // namespace

// --------------------------------------------------------------------- pack
// CTA per tile: thread = 16 columns of a row.
__global__ void __launch_bounds__(256) run_pack_kernel(const __grid_constant__ RunBatch b)
{
    start_early();
    const int tile = blockIdx.x, t = threadIdx.x;
    const RunImage &d = run_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const int r = ty * kRunSide + (t >> 2), c = tx * kRunSide + (t & 3) * 16;
    const int n = r < d.H ? min(16, d.W - c) : 0;   // may be negative: none
    uint32_t w[4], m = 0;
    load_row16(d.in + (int64_t)r * d.ld_in, c, n, d.W, w);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) m |= (uint32_t)(((w[q] >> (8 * k)) & 0xffu) != 0u) << (4 * q + k);
    reinterpret_cast<uint16_t *>(b.bits + (int64_t)tile * kRunSide)[t] = (uint16_t)m;
}

// Bit 8 k + 7: byte k of v is at least t (0 <= t <= 255).
__device__ __forceinline__ uint32_t at_least(uint32_t v, uint32_t t)
{
    const uint32_t low = ((v & 0x7f7f7f7fu) | 0x80808080u) - (t & 0x7fu) * 0x01010101u;
    return (t < 128u ? v | low : v & low) & 0x80808080u;
}

// CTA per tile, thread = 16 columns of a row: bits = (I < lo) and seeds = (J
// >= lo), J the chain's marker: I >= hi, or I >= lo on the image border.
__global__ void __launch_bounds__(256) run_threshold_kernel(const __grid_constant__ RunBatch b)
{
    start_early();
    const int tile = blockIdx.x, t = threadIdx.x;
    const RunImage &d = run_image(b, tile);
    const int lt = tile - d.tile_base;
    const int ty = lt / d.nx, tx = lt - ty * d.nx;
    const int r = ty * kRunSide + (t >> 2), c = tx * kRunSide + (t & 3) * 16;
    const int n = r < d.H ? min(16, d.W - c) : 0;   // may be negative: none
    uint32_t w[4];
    load_row16(d.in + (int64_t)r * d.ld_in, c, n, d.W, w);
    uint32_t m = 0, sd = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // four flags of a word to a nibble: no two products of the multiplication meet
        m |= ((at_least(w[q], (uint32_t)min(b.lo, 255)) >> 7) * 0x10204080u >> 28) << (4 * q);
        sd |= ((at_least(w[q], (uint32_t)min(b.hi, 255)) >> 7) * 0x10204080u >> 28) << (4 * q);
    }
    const uint32_t in = n >= 16 ? 0xffffu : n > 0 ? (1u << n) - 1u : 0u;
    m = b.lo > 255 ? 0u : m & in;
    sd = b.hi > 255 ? 0u : sd & in;
    uint32_t border = r == 0 || r == d.H - 1 ? 0xffffu : 0u;
    if (c == 0) border |= 1u;
    if (d.W - 1 - c < 16 && d.W - 1 >= c) border |= 1u << (d.W - 1 - c);
    sd |= border & m;
    reinterpret_cast<uint16_t *>(b.bits + (int64_t)tile * kRunSide)[t] = (uint16_t)(in & ~m);
    reinterpret_cast<uint16_t *>(b.seeds + (int64_t)tile * kRunSide)[t] = (uint16_t)sd;
}

// --------------------------------------------------------------------- fill
// Warp per tile: the local stage of a fill. AGAIN: after the fill of the
// unreached parts (b.U), whose holes join the foreground first.
template <int CONN, bool SEEDS, bool AGAIN, bool ALONE>
__global__ void __launch_bounds__(ALONE ? 32 : kWarps * 32) run_fill_local_kernel(const __grid_constant__ RunBatch b)
{
    start_early();
    const int lane = threadIdx.x & 31, at = blockIdx.x * (ALONE ? 1 : kWarps) + (threadIdx.x >> 5);
    const bool mine = at < b.ntiles;
    const int tile = mine ? at : 0;
    const RunImage &d = run_image(b, tile);
    const Place p = place_of(d, tile);
    ulonglong2 *row = reinterpret_cast<ulonglong2 *>(b.bits + (int64_t)tile * kRunSide) + lane;
    const ulonglong2 f = *row;
    ulonglong2 seed = make_ulonglong2(0ull, 0ull);
    if (SEEDS) seed = *(reinterpret_cast<const ulonglong2 *>(b.seeds + (int64_t)tile * kRunSide) + lane);
    // (AGAIN: what stays of the background is some of its runs)
    with_memory<ALONE>(count_runs(exists(d, p, 2 * lane) & ~f.x, exists(d, p, 2 * lane + 1) & ~f.y),
                       [&](const Mem<ALONE> &mem) {
        if (!mine) return;
        ulonglong2 g = f;
        if (AGAIN) {
            const ulonglong2 add = holes_of(b, b.U, d, p, f, mem, lane);
            g = make_ulonglong2(f.x | add.x, f.y | add.y);
            if (__any_sync(0xffffffffu, (add.x | add.y) != 0ull)) *row = g;
        }
        fill_tile<CONN, SEEDS>(b, SEEDS ? b.U : b.outside, d, p, g, seed, mem, lane);
    });
}

// Warp per tile: joins the slots across its right and lower seams (and, for
// 8-connectivity, at its lower right corner).
template <int CONN>
__global__ void __launch_bounds__(kWarps * 32) run_seam_kernel(const __grid_constant__ RunBatch b, uint32_t *U)
{
    start_early();
    __shared__ uint32_t s_pairs[kWarps][2 * kRunSide * 3];
    const int lane = threadIdx.x & 31;
    const int tile = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (tile >= b.ntiles) return;
    const RunImage &d = run_image(b, tile);
    const Place p = place_of(d, tile);
    // pairs of slots to join; then the lanes join them side by side
    volatile uint32_t *pairs = s_pairs[threadIdx.x >> 5];
    int n = 0;
    auto join = [&](int which, uint32_t a, uint32_t c) {   // whole warp; which: 0 right, 1 lower neighbour
        // (once per stretch of the side: the same pair further on costs less than a vote on all equal ones)
        const bool valid = a != 255u && c != 255u;
        const uint32_t v = valid ? a << 8 | c : ~0u, before = __shfl_up_sync(0xffffffffu, v, 1);
        const bool lead = valid && (lane == 0 || before != v);
        const uint32_t m = __ballot_sync(0xffffffffu, lead);
        if (lead) pairs[n + __popc(m & ((1u << lane) - 1u))] = (uint32_t)which << 16 | a << 8 | c;
        n += __popc(m);
    };
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {   // right, lower
        if (!p.open[k ? 1 : 3]) continue;
        const int other = k ? tile + d.nx : tile + 1;
        const uint8_t *mine = b.sides + (int64_t)tile * kRunSides + (k ? 1 : 3) * kRunSide;
        const uint8_t *its = b.sides + (int64_t)other * kRunSides + (k ? 0 : 2) * kRunSide;
#pragma unroll 1
        for (int h = 0; h < kRunSide; h += 32) {
            const int i = h + lane;
            const uint32_t a = mine[i], c = its[i];
            if (!__any_sync(0xffffffffu, a != 255u) && CONN == 4) continue;
            join(k, a, c);
            if (CONN == 8) {
                const bool in = i + 1 < kRunSide;
                const uint32_t an = in ? mine[i + 1] : 255u, cn = in ? its[i + 1] : 255u;
                // needed only where neither of the two straight pairs joins them
                join(k, an == 255u && c == 255u ? a : 255u, cn);
                join(k, a == 255u && cn == 255u ? an : 255u, c);
            }
        }
    }
    auto node = [&](int t, uint32_t slot) { return 1u + (uint32_t)t * kRunSlots + slot; };
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
        const uint32_t v = pairs[i];
        node_union(U, node(tile, (v >> 8) & 0xffu), node(v >> 16 ? tile + d.nx : tile + 1, v & 0xffu));
    }
    if (CONN == 8 && p.open[1] && p.open[3]) {
        auto side = [&](int t, int s, int i) -> uint32_t { return b.sides[(int64_t)t * kRunSides + s * kRunSide + i]; };
        if (lane == 0) {
            const uint32_t a = side(tile, 3, kRunSide - 1), c = side(tile + d.nx + 1, 2, 0);
            if (a != 255u && c != 255u) node_union(U, node(tile, a), node(tile + d.nx + 1, c));
        }
        if (lane == 1) {
            const uint32_t a = side(tile + 1, 2, kRunSide - 1), c = side(tile + d.nx, 3, 0);
            if (a != 255u && c != 255u) node_union(U, node(tile + 1, a), node(tile + d.nx, c));
        }
    }
}

// Warp per tile. FILL: slots that did not reach the outside are filled, F is
// written. LABEL: then the foreground's components become slots.
template <bool FILL, int LABEL, bool ALONE>
__global__ void __launch_bounds__(ALONE ? 32 : kWarps * 32) run_local_kernel(const __grid_constant__ RunBatch b)
{
    start_early();
    const int lane = threadIdx.x & 31, at = blockIdx.x * (ALONE ? 1 : kWarps) + (threadIdx.x >> 5);
    const bool mine = at < b.ntiles;
    const int tile = mine ? at : 0;
    const RunImage &d = run_image(b, tile);
    const Place p = place_of(d, tile);
    ulonglong2 *row = reinterpret_cast<ulonglong2 *>(b.bits + (int64_t)tile * kRunSide) + lane;
    ulonglong2 f = *row;
    // the background's runs and the foreground's after filling: a row's filled runs join what they touch, or are the
    // row's only one
    auto starts = [](u64 m) { return __popcll(m & ~(m << 1)); };
    int runs = starts(f.x) + starts(f.y);
    if (FILL)
        runs = max(starts(f.x), starts(exists(d, p, 2 * lane) & ~f.x)) +
               max(starts(f.y), starts(exists(d, p, 2 * lane + 1) & ~f.y));
    with_memory<ALONE>((int)__reduce_add_sync(0xffffffffu, (uint32_t)runs), [&](const Mem<ALONE> &mem) {
        if (!mine) return;
        volatile uint32_t *P = mem.runs();
        if (FILL) {
            const ulonglong2 add = holes_of(b, b.outside, d, p, f, mem, lane);
            if (__any_sync(0xffffffffu, (add.x | add.y) != 0ull)) {
                f = make_ulonglong2(f.x | add.x, f.y | add.y);
                *row = f;
            }
            if (d.filled) {
                // lane: 16 columns (lane & 3) of row 8 q + lane / 4
#pragma unroll 2
                for (int q = 0; q < 8; ++q) {
                    const int i = 8 * q + (lane >> 2), r = p.r0 + i, c = p.c0 + (lane & 3) * 16;
                    const u64 w0 = shfl64(f.x, i >> 1), w1 = shfl64(f.y, i >> 1), bits = i & 1 ? w1 : w0;
                    const uint32_t m = (uint32_t)(bits >> ((lane & 3) * 16)) & 0xffffu;
                    const int n = r < d.H ? min(16, d.W - c) : 0;
                    if (n <= 0) continue;
                    auto spread = [](uint32_t x) { return ((x & 0xfu) * 0x00204081u) & 0x01010101u; };
                    uint8_t *o = d.filled + (int64_t)r * d.ld_filled + p.c0;
                    const int head = (int)(-(uintptr_t)o & 3u);
                    if (head && d.W - p.c0 >= kRunSide) {   // the row's aligned words, from its bits; its ends by bytes
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int at = head + 16 * (lane & 3) + 4 * k;
                            if (at + 4 <= kRunSide) *reinterpret_cast<uint32_t *>(o + at) = spread((uint32_t)(bits >> at));
                        }
                        if ((lane & 3) < head) o[lane & 3] = (uint8_t)((bits >> (lane & 3)) & 1ull);
                        else o[kRunSide - 4 + (lane & 3)] = (uint8_t)((bits >> (kRunSide - 4 + (lane & 3))) & 1ull);
                    } else {
                        uint32_t w[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) w[k] = spread(m >> (4 * k));
                        store_bytes(o + (lane & 3) * 16, n, w);
                    }
                }
            }
        }
        if (LABEL) {
            if (tile == d.tile_base && lane == 0 && d.n_kept) *d.n_kept = 0;
            const uint32_t node = 1u + (uint32_t)tile * kRunSlots;
            if (!__any_sync(0xffffffffu, (f.x | f.y) != 0ull)) {
                uint16_t *s = reinterpret_cast<uint16_t *>(b.sides + (int64_t)tile * kRunSides) + lane;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (p.open[k]) s[k * kRunSide / 2] = 0xffffu;
                if (lane == 0) b.lcnt[tile] = 0u;
                return;
            }
            const Runs r = components<LABEL ? LABEL : 8>(f.x, f.y, mem, lane);
            flag_rim(r, p, P, lane);
            const int cnt = number_slots(r, P, lane, [&](int, int k) {
                b.U[node + k] = mix(node + k);
                b.A[node + k] = 0u;
            });
            write_sides(b, r, p, P, lane);
            __syncwarp();
            // areas: a slot's to its node, with its first pixel (a root run is its
            // component's first), another component's to its root's upper bits
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                u64 s = r.st[j];
                for (int k = 0; s; ++k, s &= s - 1) {
                    const int run = r.base[j] + k, pos = __ffsll((long long)s) - 1;
                    const uint32_t root = P[run] & kParent, v = P[root], area = (uint32_t)__popcll(run_bits(r.m[j], pos));
                    if (v & kRim) {
                        const uint32_t slot = node + ((v >> kSlotShift) & kSlotMask);
                        atomicAdd(b.A + slot, area);
                        if (root == (uint32_t)run) b.M[slot] = (uint32_t)((int64_t)(p.r0 + 2 * lane + j) * d.W + p.c0 + pos);
                    } else {
                        atomicAdd(const_cast<uint32_t *>(P + root), area << kSlotShift);
                    }
                }
            }
            __syncwarp();
            uint32_t *words = b.words + (int64_t)tile * kRunWords;
            for (int i = lane; i < r.total; i += 32) words[i] = P[i];
            if (lane == 0) b.lcnt[tile] = (uint8_t)cnt;
        }
    });
}

// ------------------------------------------------------------------- labels
// Thread per slot: areas and first pixels of a tree meet at its root.
__global__ void __launch_bounds__(256) run_roots_kernel(const __grid_constant__ RunBatch b)
{
    start_early();
    const int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int tile = (int)(g / 32), lane = (int)(g % 32);   // a warp per tile
    if (tile >= b.ntiles) return;
    for (int k = lane; k < (int)b.lcnt[tile]; k += 32) {
        const uint32_t x = 1u + (uint32_t)tile * kRunSlots + k, v = node_find(b.U, mix(x)), root = v * kUnmix;
        if (root == x) continue;
        b.U[x] = v;   // plain store: no concurrent value can be smaller
        atomicAdd(b.A + root, b.A[x]);
        atomicMin(b.M + root, b.M[x]);
    }
}

// Warp per tile: labels with the area filter, kept bits and count, from the
// run words of the local stage, in shared memory or, where they do not fit in
// a warp's share (!ALONE), in place: a block then never waits for one of its
// warps (waiting for the block's memory as above: 122 us for eight 4096 x 4096
// tiles instead of 102).
template <bool ALONE>
__global__ void __launch_bounds__(ALONE ? 32 : kWarps * 32) run_label_kernel(const __grid_constant__ RunBatch b)
{
    start_early();
    const int lane = threadIdx.x & 31, at = blockIdx.x * (ALONE ? 1 : kWarps) + (threadIdx.x >> 5);
    const int tile = at;
    if (tile >= b.ntiles) return;
    const RunImage &d = run_image(b, tile);
    const Place p = place_of(d, tile);
    const ulonglong2 f = *(reinterpret_cast<const ulonglong2 *>(b.bits + (int64_t)tile * kRunSide) + lane);
    auto label = [&](volatile uint32_t *P, bool in_place) {
        // rows [i0, nr) of the tile: its share when several warps take a tile (one alone works in place)
        const int share = in_place ? kRunSide : kRunSide / (int)gridDim.y, i0 = (int)blockIdx.y * share;
        if (i0 >= kRunSide) return;
        const int nr = min(i0 + share, d.H - p.r0), c = p.c0 + 2 * lane;
        int32_t *out = d.labels + (int64_t)p.r0 * d.ld_lab + c;
        const bool both = c + 1 < d.W, one = c < d.W;
        const bool wide = both && (((uintptr_t)d.labels | (uintptr_t)d.ld_lab * 4u) & 7u) == 0;
        auto store = [&](int i, int32_t x, int32_t y) {
            int32_t *o = out + (int64_t)i * d.ld_lab;
            if (wide) {
                *reinterpret_cast<int2 *>(o) = make_int2(x, y);
            } else {
                if (one) o[0] = x;
                if (both) o[1] = y;
            }
        };
        u64 keep[2] = {0ull, 0ull};
        const uint32_t rows = __ballot_sync(0xffffffffu, f.x != 0ull), rows1 = __ballot_sync(0xffffffffu, f.y != 0ull);
        if (!(rows | rows1)) {
#pragma unroll 4
            for (int i = i0; i < nr; ++i) store(i, -1, -1);
        } else {
            const Runs r = runs_of(f.x, f.y, lane);
            const uint32_t *words = b.words + (int64_t)tile * kRunWords;
            for (int i = lane; i < r.total && !in_place; i += 32) P[i] = words[i];
            __syncwarp();
            // roots' labels (in their lane's order), then every run's
            int kept = 0;
            const uint32_t node = 1u + (uint32_t)tile * kRunSlots;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                u64 s = r.st[j];
                for (int k = 0; s; ++k, s &= s - 1) {
                    const int run = r.base[j] + k;
                    const uint32_t v = P[run];
                    if ((v & kParent) != (uint32_t)run) continue;
                    int32_t area, label;
                    bool first = true;
                    if (v & kRim) {
                        const uint32_t x = node + ((v >> kSlotShift) & kSlotMask), root = b.U[x] * kUnmix;
                        area = (int32_t)b.A[root];
                        label = (int32_t)b.M[root];
                        first = root == x;
                    } else {
                        area = (int32_t)(v >> kSlotShift);
                        label = (int32_t)((int64_t)(p.r0 + 2 * lane + j) * d.W + p.c0 + __ffsll((long long)s) - 1);
                    }
                    const bool in = area >= b.amin && area <= b.amax;
                    kept += in && first;
                    P[run] = in ? (uint32_t)label | kRim : kBorder;   // a root's final word: kRim | label, or kBorder: dropped
                }
            }
            __syncwarp();
            // every run takes its root's word; a root keeps its own (bit 31 or 30
            // set marks final words, which others read through their parent)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                u64 s = r.st[j];
                for (int k = 0; s; ++k, s &= s - 1) {
                    const int run = r.base[j] + k;
                    const uint32_t v = P[run];
                    const uint32_t w = v & (kRim | kBorder) ? v : P[v];
                    if (w & kRim) keep[j] |= run_bits(r.m[j], __ffsll((long long)s) - 1);
                }
            }
            __syncwarp();
            kept = __reduce_add_sync(0xffffffffu, kept);
            if (lane == 0 && kept && d.n_kept && i0 == 0) atomicAdd(d.n_kept, kept);
#pragma unroll 2
            for (int i = i0; i < nr; ++i) {
                int32_t v[2] = {-1, -1};
                if (((i & 1 ? rows1 : rows) >> (i >> 1)) & 1u) {   // whole warp
                    const u64 m = shfl64(i & 1 ? f.y : f.x, i >> 1), st = m & ~(m << 1);
                    const int base = __shfl_sync(0xffffffffu, i & 1 ? r.base[1] : r.base[0], i >> 1);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int x = 2 * lane + q;
                        if ((m >> x) & 1ull) {
                            uint32_t w = P[base + __popcll(st & (~0ull >> (63 - x))) - 1];
                            if (!(w & (kRim | kBorder))) w = P[w];
                            if (w & kRim) v[q] = (int32_t)(w & ~kRim);
                        }
                    }
                }
                store(i, v[0], v[1]);
            }
        }
        if (b.kept && i0 == 0)
            *(reinterpret_cast<ulonglong2 *>(b.kept + (int64_t)tile * kRunSide) + lane) = make_ulonglong2(keep[0], keep[1]);
    };
    extern __shared__ uint32_t run_smem[];
    if (ALONE || count_runs(f.x, f.y) <= kWarpWords) label(run_smem + (ALONE ? 0 : (threadIdx.x >> 5) * kWarpWords), false);
    else label(b.words + (int64_t)tile * kRunWords, true);
}

// --------------------------------------------------------------------- host
namespace {

// `alone` while there are few tiles, else `four`; y: CTAs that share a tile.
using RunKernel = void (*)(RunBatch);
cudaError_t warp_per_tile(RunKernel alone, RunKernel four, const RunBatch &b, cudaStream_t s, int y = 1)
{
    const bool few = b.ntiles <= kFewTiles;
    const int w = few ? 1 : kWarps;
    launch_early((few ? alone : four), dim3((unsigned)ceil_div(b.ntiles, w), y), w * 32, kRunSmem, s, b);
    return cudaGetLastError();
}

cudaError_t launch_seam(const RunBatch &b, int conn, uint32_t *U, cudaStream_t s)
{
    const unsigned grid = (unsigned)ceil_div(b.ntiles, kWarps);
    if (conn == 8) launch_early(run_seam_kernel<8>, grid, kWarps * 32, 0, s, b, U);
    else launch_early(run_seam_kernel<4>, grid, kWarps * 32, 0, s, b, U);
    return cudaGetLastError();
}

}  // namespace

size_t run_tiles(int H, int W) { return (size_t)(ceil_div(H, kRunSide) * ceil_div(W, kRunSide)); }

RunImage &run_add(RunBatch &b, int H, int W)
{
    RunImage &d = b.img[b.n++];
    d = RunImage{};
    d.H = H;
    d.W = W;
    d.nx = (int)ceil_div(W, kRunSide);
    d.ny = (int)ceil_div(H, kRunSide);
    d.tile_base = b.ntiles;
    b.ntiles += d.nx * d.ny;
    return d;
}

cudaError_t launch_run_pack(const RunBatch &b, cudaStream_t s)
{
    launch_early(run_pack_kernel, (unsigned)b.ntiles, 256, 0, s, b);
    return cudaGetLastError();
}

cudaError_t launch_run_reach(const RunBatch &b, cudaStream_t s)
{
    launch_early(run_threshold_kernel, (unsigned)b.ntiles, 256, 0, s, b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = warp_per_tile(run_fill_local_kernel<8, true, false, true>, run_fill_local_kernel<8, true, false, false>, b, s);
    return e != cudaSuccess ? e : launch_seam(b, 8, b.U, s);
}

cudaError_t launch_run_fill(const RunBatch &b, int conn, int label_conn, cudaStream_t s, bool again)
{
    if ((conn != 4 && conn != 8) || (label_conn != 0 && label_conn != 8)) return cudaErrorInvalidValue;
    cudaError_t e;
    if (conn == 8)
        e = again ? warp_per_tile(run_fill_local_kernel<8, false, true, true>, run_fill_local_kernel<8, false, true, false>, b, s)
                  : warp_per_tile(run_fill_local_kernel<8, false, false, true>, run_fill_local_kernel<8, false, false, false>, b, s);
    else
        e = again ? warp_per_tile(run_fill_local_kernel<4, false, true, true>, run_fill_local_kernel<4, false, true, false>, b, s)
                  : warp_per_tile(run_fill_local_kernel<4, false, false, true>, run_fill_local_kernel<4, false, false, false>, b, s);
    if (e != cudaSuccess) return e;
    if ((e = launch_seam(b, conn, b.outside, s)) != cudaSuccess) return e;
    return label_conn ? warp_per_tile(run_local_kernel<true, 8, true>, run_local_kernel<true, 8, false>, b, s)
                      : warp_per_tile(run_local_kernel<true, 0, true>, run_local_kernel<true, 0, false>, b, s);
}

cudaError_t launch_run_local(const RunBatch &b, int conn, cudaStream_t s)
{
    if (conn != 4 && conn != 8) return cudaErrorInvalidValue;
    return conn == 8 ? warp_per_tile(run_local_kernel<false, 8, true>, run_local_kernel<false, 8, false>, b, s)
                     : warp_per_tile(run_local_kernel<false, 4, true>, run_local_kernel<false, 4, false>, b, s);
}

cudaError_t launch_run_label(const RunBatch &b, int conn, cudaStream_t s)
{
    if (conn != 4 && conn != 8) return cudaErrorInvalidValue;
    cudaError_t e = launch_seam(b, conn, b.U, s);
    if (e != cudaSuccess) return e;
    launch_early(run_roots_kernel, (unsigned)ceil_div(b.ntiles, 8), 256, 0, s, b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // few tiles: four warps write a tile's labels (a warp's 64 rows are 10 us of latency)
    return warp_per_tile(run_label_kernel<true>, run_label_kernel<false>, b, s, b.ntiles <= kFewTiles ? 4 : 1);
}

}  // namespace rtk
