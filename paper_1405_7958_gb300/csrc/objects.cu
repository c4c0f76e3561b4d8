// The per-object steps that follow the labels in the paper's pipeline
// (Section 5.1, "Example Application"):
//   * the feature computation stage, restructured as the paper describes:
//     the objects are cut out by their minimum bounding boxes, one group of
//     threads per box computes the intermediate results (histograms,
//     co-occurrence matrix, moments), then one thread per object turns them
//     into the features;
//   * the Watershed after the Pre-Watershed step, which splits touching
//     nuclei: marker-controlled flooding of the distance map inside every
//     object, in shared memory when the box is small enough.
// In both a warp takes an object with a small box and a block one with a
// large box. Both start from the same enumeration of the objects of a label
// image whose labels are the linear index of each object's first pixel (as
// rt_label_area writes them): one pass over the labels finds those first
// pixels and the ends of the runs of equal labels, a second one over the
// runs alone lists the objects by label and grows their bounding boxes.
#include "objects.cuh"

namespace rtk {

namespace {

size_t piece(size_t bytes) { return (size_t)round_up((int64_t)bytes, 256); }

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned long long kUnl = ~0ull;   // watershed state of a pixel without a basin yet

}  // namespace

size_t obj_workspace_bytes(int H, int W, bool features, bool watershed, int cap)
{
    const size_t N = (size_t)H * W;
    const size_t nch = (size_t)ceil_div((int64_t)N, kObjChunk);
    size_t b = 2 * piece(nch * 4) + piece(64) + piece(N * 8) + piece(N * 4) + piece(N * 16);
    if (features) b += piece((size_t)(cap > 0 ? cap : 1) * sizeof(ObjInter));
    if (watershed) b += piece(N * 4) + piece(N * 8) + piece(N);
    return b;
}

void obj_carve(ObjArgs &a, char *base, bool features, bool watershed)
{
    const size_t N = (size_t)a.H * a.W;
    const size_t nch = (size_t)ceil_div((int64_t)N, kObjChunk);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base + off;
        off += piece(bytes);
        return p;
    };
    a.chunk_cnt = reinterpret_cast<uint32_t *>(take(nch * 4));
    a.block_cnt = reinterpret_cast<uint32_t *>(take(nch * 4));
    a.ctl = reinterpret_cast<uint32_t *>(take(64));
    a.rec = reinterpret_cast<uint2 *>(take(N * 8));
    a.big = reinterpret_cast<int32_t *>(a.rec);   // written when the records have been read
    a.olabel = reinterpret_cast<int32_t *>(take(N * 4));
    a.box = reinterpret_cast<int32_t *>(take(N * 16));
    a.inter = features ? reinterpret_cast<ObjInter *>(take((size_t)(a.cap > 0 ? a.cap : 1) * sizeof(ObjInter)))
                       : nullptr;
    if (watershed) {
        a.R = reinterpret_cast<int32_t *>(take(N * 4));
        a.st = reinterpret_cast<unsigned long long *>(take(N * 8));
        a.nm = reinterpret_cast<uint8_t *>(take(N));
    } else {
        a.R = nullptr;
        a.st = nullptr;
        a.nm = nullptr;
    }
}

// ------------------------------------------------------------ enumeration
// Warp per chunk of kObjChunk pixels (raster order), four pixels a lane and
// 128 a step, all of the chunk's loads in flight at once. A lane cuts its
// four pixels into stretches of one label and keeps those at which a run of
// the row starts or ends: the stretches inside a run add nothing to a box.
// The kept ones go to the chunk's records in raster order (label; offset and
// length), so the pass that grows the boxes never reads the labels of the
// other pixels again. An object's first pixel (L(p) == p) sets up its box,
// which is kept under the label itself, so no index is needed to find it.
// With a basin image, -1 goes everywhere; the objects' pixels are written
// by the flooding. VEC: rows of 16-byte aligned quads of pixels. Half bound
// by issue, half by memory: 21 us for the 67 MB of a 4096 x 4096 label image
// with 2180 nuclei, 9 for the boxes (count, prefix sum, emit and a pass over
// all pixels for the boxes: 45 + 20 + 46 + 56).
template <bool VEC>
__global__ void __launch_bounds__(kThreads) obj_scan_kernel(ObjArgs a)
{
    start_early();
    constexpr int kSteps = kObjChunk / 128;
    __shared__ uint32_t roots_of[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ch = (int64_t)blockIdx.x * kWarps + warp;
    const int64_t N = (int64_t)a.H * a.W;
    if (blockIdx.x == 0 && threadIdx.x < 8) {
        a.ctl[threadIdx.x] = 0u;
        if (threadIdx.x == 0 && a.n_basins) *a.n_basins = 0;
    }
    uint32_t nrec = 0, nroot = 0;
    if (ch * kObjChunk < N) {   // whole warp
        const uint32_t W = (uint32_t)a.W, n32 = (uint32_t)N, p0 = (uint32_t)ch * kObjChunk;   // N <= 2^30
        uint32_t p = p0 + 4 * lane, r = p / W, c = p - r * W;
        const uint32_t c0 = c;
        int32_t l[kSteps][4];
#pragma unroll
        for (int k = 0; k < kSteps; ++k, p += 128) {
            if (k) {
                c += 128;
                while (c >= W) {
                    c -= W;
                    ++r;
                }
            }
            l[k][0] = l[k][1] = l[k][2] = l[k][3] = -1;
            if (VEC) {
                if (p < n32) {
                    const int4 v = *reinterpret_cast<const int4 *>(a.L + (int64_t)r * a.ld_L + c);
                    l[k][0] = v.x;
                    l[k][1] = v.y;
                    l[k][2] = v.z;
                    l[k][3] = v.w;
                    if (a.basins)
                        *reinterpret_cast<int4 *>(a.basins + (int64_t)r * a.ld_B + c) = make_int4(-1, -1, -1, -1);
                }
            } else {
                uint32_t rj = r, cj = c;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (p + j < n32) {
                        l[k][j] = a.L[(int64_t)rj * a.ld_L + cj];
                        if (a.basins) a.basins[(int64_t)rj * a.ld_B + cj] = -1;
                    }
                    if (++cj == W) {
                        cj = 0;
                        ++rj;
                    }
                }
            }
        }
        // the pixels before and after the chunk (the same row's: others do not count)
        int32_t before = -1, after = -1;
        if (lane == 0 && c0 > 0) before = a.L[(int64_t)(p0 / W) * a.ld_L + c0 - 1];
        if (lane == 31 && p0 + kObjChunk < n32) {
            const uint32_t pa = p0 + kObjChunk, ra = pa / W;
            after = a.L[(int64_t)ra * a.ld_L + (pa - ra * W)];
        }
        uint2 *rec = a.rec + (int64_t)p0;
        p = p0 + 4 * lane;
        c = c0;
#pragma unroll
        for (int k = 0; k < kSteps; ++k, p += 128) {
            if (k) {
                c += 128;
                while (c >= W) c -= W;
            }
            const int32_t *q = l[k];
            if (!__any_sync(0xffffffffu, (q[0] & q[1] & q[2] & q[3]) >= 0)) continue;
            const int32_t wl = k ? __shfl_sync(0xffffffffu, l[k ? k - 1 : 0][3], 31) : before;
            const int32_t wr = k + 1 < kSteps ? __shfl_sync(0xffffffffu, l[k + 1 < kSteps ? k + 1 : k][0], 0) : after;
            int32_t lf = __shfl_up_sync(0xffffffffu, q[3], 1), rt = __shfl_down_sync(0xffffffffu, q[0], 1);
            if (lane == 0) lf = wl;
            if (lane == 31) rt = wr;
            uint32_t first = 0;   // bit j: pixel j is the first of its row (4: the pixel after the quad)
            if (VEC) {
                first = (c == 0 ? 1u : 0u) | (c + 4 == W ? 16u : 0u);
            } else {
                uint32_t cj = c;
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    first |= cj == 0 ? 1u << j : 0u;
                    if (++cj == W) cj = 0;
                }
            }
            const uint32_t obj = (q[0] >= 0 ? 1u : 0u) | (q[1] >= 0 ? 2u : 0u) | (q[2] >= 0 ? 4u : 0u) |
                                 (q[3] >= 0 ? 8u : 0u);
            // bit j: pixel j differs from the one before it in its row (bit 4: the pixel after the quad)
            const uint32_t cut = first | (lf != q[0] ? 1u : 0u) | (q[0] != q[1] ? 2u : 0u) | (q[1] != q[2] ? 4u : 0u) |
                                 (q[2] != q[3] ? 8u : 0u) | (q[3] != rt ? 16u : 0u);
            // the stretches to keep, by their first pixels: all that start a run, and the one going on from the
            // quad before if it ends a run
            const uint32_t tails = obj & ((cut >> 1) | 8u);
            uint32_t emit = obj & cut;
            if ((obj & ~cut & 1u) && ((cut >> __ffs(tails)) & 1u)) emit |= 1u;
            const uint32_t any = __ballot_sync(0xffffffffu, emit != 0);
            if (!any) continue;
            const uint32_t cnt = __popc(emit), lt = (1u << lane) - 1u;
            const uint32_t m0 = __ballot_sync(0xffffffffu, cnt & 1u), m1 = __ballot_sync(0xffffffffu, cnt & 2u),
                           m2 = __ballot_sync(0xffffffffu, cnt & 4u);
            uint32_t at = nrec + __popc(m0 & lt) + 2u * __popc(m1 & lt) + 4u * __popc(m2 & lt);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if ((emit >> j) & 1u) {
                    const int e = j + __ffs(tails >> j) - 1;   // its last pixel in the quad
                    rec[at++] = make_uint2((uint32_t)q[j], (p - p0 + j) | ((uint32_t)(e - j) << 16));
                    if ((uint32_t)q[j] == p + j) {
                        const int rr = (int)((p + j) / W), cc = (int)(p + j - rr * W);
                        reinterpret_cast<int4 *>(a.box)[p + j] = make_int4(rr, cc, rr, cc);
                        ++nroot;
                    }
                }
            nrec += __popc(m0) + 2u * __popc(m1) + 4u * __popc(m2);
        }
        nroot = __reduce_add_sync(0xffffffffu, nroot);
        if (lane == 0) a.chunk_cnt[ch] = nrec | (nroot << 16);
    }
    if (lane == 0) roots_of[warp] = nroot;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += roots_of[w];
        a.block_cnt[blockIdx.x] = s;
    }
}

// Each block takes a span of the scan's blocks, a warp one of their chunks:
// the objects of the blocks before the span give the rank of its first one
// (a few loads per thread instead of a kernel of its own for the prefix
// sum). A record grows its object's box; one at an object's first pixel
// also writes the label at its rank. A label that is not the linear index
// of an earlier-or-equal pixel carrying that same label is not canonical:
// RT_EINVAL in the status.
__global__ void __launch_bounds__(kThreads) obj_grow_kernel(ObjArgs a, int nblk, int span)
{
    start_early();
    __shared__ uint32_t part[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t N = (int64_t)a.H * a.W, nch = ceil_div(N, kObjChunk);
    const uint32_t W = (uint32_t)a.W;
    const int b0 = blockIdx.x * span, b1 = min(nblk, b0 + span);
    uint32_t s = 0;
    for (int i = threadIdx.x; i < b0; i += kThreads) s += a.block_cnt[i];
    s = __reduce_add_sync(0xffffffffu, s);
    if (lane == 0) part[warp] = s;
    __syncthreads();
    uint32_t base = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) base += part[w];
    for (int blk = b0; blk < b1; ++blk) {
        const int64_t ch0 = (int64_t)blk * kWarps, ch = ch0 + warp;
        const uint32_t word = lane < kWarps && ch0 + lane < nch ? a.chunk_cnt[ch0 + lane] : 0u;
        const uint32_t mine = __shfl_sync(0xffffffffu, word, warp);
        uint32_t rank = base + __reduce_add_sync(0xffffffffu, lane < warp ? word >> 16 : 0u);
        base += __reduce_add_sync(0xffffffffu, word >> 16);
        const uint32_t n = mine & 0xffffu;
        const uint2 *rec = a.rec + ch * kObjChunk;
        for (uint32_t i0 = 0; i0 < n; i0 += 32) {
            bool root = false;
            uint32_t l = 0;
            if (i0 + lane < n) {
                const uint2 q = rec[i0 + lane];
                const uint32_t p = (uint32_t)ch * kObjChunk + (q.y & 0xffffu);
                l = q.x;
                root = l == p;
                const uint32_t rl = l / W, cl = l - rl * W;
                if (l > p || a.L[(int64_t)rl * a.ld_L + cl] != (int32_t)l) {
                    raise_status(a.err, RT_EINVAL);
                } else {
                    const int r = (int)(p / W), c = (int)(p - r * W), e = c + (int)(q.y >> 16);
                    int32_t *bx = a.box + 4 * (int64_t)l;
                    const int4 b = __ldcg(reinterpret_cast<const int4 *>(bx));
                    if (b.z < r) atomicMax(bx + 2, r);
                    if (b.y > c) atomicMin(bx + 1, c);
                    if (b.w < e) atomicMax(bx + 3, e);
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, root);
            if (root) a.olabel[rank + __popc(m & ((1u << lane) - 1u))] = (int32_t)l;
            rank += __popc(m);
        }
    }
    if (b1 == nblk && b0 < nblk && threadIdx.x == 0) {
        a.ctl[0] = base;
        if (a.n_obj) *a.n_obj = (int32_t)base;
    }
}

cudaError_t launch_enumeration(const ObjArgs &a, int num_sms, cudaStream_t s, int *launches)
{
    const int64_t nch = ceil_div((int64_t)a.H * a.W, kObjChunk);
    const int nblk = (int)ceil_div(nch, kWarps);
    auto quads = [](const void *p, int64_t ld) { return ((uintptr_t)p & 15u) == 0 && ld % 4 == 0; };
    if (a.W % 4 == 0 && quads(a.L, a.ld_L) && (!a.basins || quads(a.basins, a.ld_B)))
        launch_early(obj_scan_kernel<true>, nblk, kThreads, 0, s, a);
    else
        launch_early(obj_scan_kernel<false>, nblk, kThreads, 0, s, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int span = (int)ceil_div(nblk, num_sms * 8);
    launch_early(obj_grow_kernel, (unsigned)ceil_div(nblk, span), kThreads, 0, s, a, nblk, span);
    *launches += 2;
    return cudaGetLastError();
}

// Next entry of the list of large objects for this block (dynamic: boxes
// differ in size); -1 when done.
__device__ __forceinline__ int next_big(const ObjArgs &a, int *slot)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t q = atomicAdd(a.ctl + 1, 1u);
        *slot = q < a.ctl[3] ? a.big[q] : -1;
    }
    __syncthreads();
    return *slot;
}

// --------------------------------------------------------------- features
__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;   // lane 0
}

__device__ __forceinline__ int64_t warp_sum_l(int64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;   // lane 0
}

// One warp: what the features need of the histogram (which it overwrites)
// and of the co-occurrence matrix of an object of n pixels, into o (lane 0
// writes). A lane owns 8 bins and 2 cells. This is the part that is bound by
// the double-precision rate (2 operations an SM and cycle), so the entropy's
// terms, a division and a logarithm each, are taken once for every count
// that occurs, times the number of bins that have it: a nucleus fills about
// 80 bins with 10 different counts, one step of the warp. The co-occurrence
// sums are integers, the homogeneity's over the common denominator 840 of
// 1 + |a - b|.
__device__ void obj_hist_stats(uint32_t *hist, const uint32_t *glcm, int64_t n, ObjInter &o)
{
    const int lane = threadIdx.x & 31;
    const double da = (double)n;
    uint32_t hb[8];
    uint32_t tot = 0;
    int lo = -1, hi = -1;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        hb[q] = hist[8 * lane + q];
        tot += hb[q];
        if (!hb[q]) continue;
        if (lo < 0) lo = 8 * lane + q;
        hi = 8 * lane + q;
    }
    const uint32_t has = __ballot_sync(0xffffffffu, tot != 0);
    const int vmin = __shfl_sync(0xffffffffu, lo, __ffs(has) - 1);
    const int vmax = __shfl_sync(0xffffffffu, hi, 31 - __clz(has));
    // median: the smallest v with 2 cum(v) >= n (exclusive prefix over lanes)
    uint32_t pre = tot;
#pragma unroll
    for (int o2 = 1; o2 < 32; o2 <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, pre, o2);
        if (lane >= o2) pre += t;
    }
    int64_t cum = (int64_t)pre - tot;
    int med = -1;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        cum += hb[q];
        if (med < 0 && hb[q] && 2 * cum >= n) med = 8 * lane + q;
        hist[8 * lane + q] = 0u;   // now: bins by their count, below 256
    }
    const uint32_t mh = __ballot_sync(0xffffffffu, med >= 0);
    med = __shfl_sync(0xffffffffu, med, __ffs(mh) - 1);
    __syncwarp();
    double ent = 0.0;
    auto term = [&](uint32_t h, uint32_t times) {
        const double p = __ddiv_rn((double)h, da);
        ent = __dsub_rn(ent, __dmul_rn((double)times, __dmul_rn(p, log2(p))));
    };
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
        uint32_t h = hb[0];
#pragma unroll
        for (int z = 1; z < 8; ++z) h = q == z ? hb[z] : h;
        if (h >= 256) term(h, 1u);
        else if (h) atomicAdd(hist + h, 1u);
    }
    __syncwarp();
    // the counts in use, packed to the front: count | bins << 16
    uint32_t used = 0, at = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        hb[q] = hist[8 * lane + q];
        used += hb[q] != 0;
    }
    at = used;
#pragma unroll
    for (int o2 = 1; o2 < 32; o2 <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, at, o2);
        if (lane >= o2) at += t;
    }
    const int nz = __shfl_sync(0xffffffffu, (int)at, 31);
    at -= used;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (hb[q]) hist[at++] = (uint32_t)(8 * lane + q) | (hb[q] << 16);   // every bin has been read
    __syncwarp();
    for (int i = lane; i < nz; i += 32) term(hist[i] & 0xffffu, hist[i] >> 16);
    ent = warp_sum_d(ent);
    int64_t n2 = 0, con = 0, en = 0, hom = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int c = 2 * lane + q;
        const int64_t g = glcm[c];
        const int d = (c >> 3) - (c & 7), ad = d < 0 ? -d : d;
        n2 += g;
        con += (int64_t)(d * d) * g;
        en += g * g;
        hom += (int64_t)(840 / (1 + ad)) * g;
    }
    n2 = warp_sum_l(n2);
    con = warp_sum_l(con);
    en = warp_sum_l(en);
    hom = warp_sum_l(hom);
    if (lane == 0) {
        o.n2 = n2;
        o.con = con;
        o.en = en;
        o.hom = hom;
        o.ent = ent;
        o.vmin = vmin;
        o.vmax = vmax;
        o.med = med;
    }
}

// The moment features of one object from the exact integer sums, by four
// neighbouring lanes (`q`: which; all lanes of the warp call it, `on`: with
// an object): the divisions and square roots, a thousand cycles each, run
// side by side in six steps instead of one lane's seventeen. Every
// floating-point step is an explicitly rounded operation (no contraction
// into fused multiply-adds).
__device__ void obj_finish(const ObjArgs &a, int64_t k, int q, bool on)
{
    const uint32_t all = 0xffffffffu;
    const ObjInter &o = a.inter[k];
    const int64_t n = o.area;
    const double da = (double)n, a2 = __dmul_rn(da, da);
    auto pick = [&](auto w, auto x, auto y, auto z) { return q == 0 ? w : q == 1 ? x : q == 2 ? y : z; };
    // variances of the rows and the columns, their covariance, variance of the intensities
    const __int128 num = (__int128)n * pick(o.srr, o.scc, o.src, o.sii) -
                         (__int128)pick(o.sr, o.sc, o.sr, o.si) * pick(o.sr, o.sc, o.sc, o.si);
    const double var = __ddiv_rn((double)num, a2);
    const double vrr = __shfl_sync(all, var, 0, 4), vcc = __shfl_sync(all, var, 1, 4), vrc = __shfl_sync(all, var, 2, 4);
    const double half = __dmul_rn(__dadd_rn(vrr, vcc), 0.5), dh = __dmul_rn(__dsub_rn(vrr, vcc), 0.5);
    const double root = __dsqrt_rn(q == 3 ? var : __dadd_rn(__dmul_rn(dh, dh), __dmul_rn(vrc, vrc)));
    const double disc = __shfl_sync(all, root, 0, 4);
    const double l1 = __dadd_rn(half, disc);
    double l2 = __dsub_rn(half, disc);
    if (l2 < 0.0) l2 = 0.0;
    const double axis = __dmul_rn(4.0, __dsqrt_rn(q == 0 ? l1 : l2));
    // centroid, l2 / l1, mean intensity
    const bool flat = !(l1 > 0.0);
    const double quot = __ddiv_rn(pick((double)o.sr, (double)o.sc, l2, (double)o.si), q == 2 ? (flat ? 1.0 : l1) : da);
    const double ecc = __dsqrt_rn(q == 2 ? __dsub_rn(1.0, quot) : 1.0);
    // compactness, contrast, energy, homogeneity
    const double P = (double)o.per, dn2 = (double)(o.n2 > 0 ? o.n2 : 1);
    const double f4 = __ddiv_rn(pick(__dmul_rn(__dmul_rn(4.0, 3.14159265358979323846), da), (double)o.con, (double)o.en,
                                     (double)o.hom),
                                pick(__dmul_rn(P, P), dn2, __dmul_rn(dn2, dn2), (double)(840 * (o.n2 > 0 ? o.n2 : 1))));
    if (!on) return;
    const int32_t l = a.olabel[k];
    const int4 b = reinterpret_cast<const int4 *>(a.box)[l];
    double *f = a.feat + k * kObjFeat;
    if (q == 0) {
        a.out_labels[k] = l;
        f[0] = da;
        f[2] = (double)(b.z - b.x + 1);
        f[4] = __dadd_rn((double)b.x, quot);
        f[6] = axis;
        f[9] = f4;
        f[12] = o.vmin;
    } else if (q == 1) {
        f[1] = P;
        f[3] = (double)(b.w - b.y + 1);
        f[5] = __dadd_rn((double)b.y, quot);
        f[7] = axis;
        f[13] = o.vmax;
        f[17] = o.n2 > 0 ? f4 : 0.0;
    } else if (q == 2) {
        f[8] = flat ? 0.0 : ecc;
        f[14] = o.med;
        f[15] = o.ent;
        f[18] = o.n2 > 0 ? f4 : 0.0;
    } else {
        f[10] = quot;
        f[11] = root;
        f[16] = (double)o.n2;
        f[19] = o.n2 > 0 ? f4 : 0.0;
    }
}

// A warp takes the boxes up to these limits. Within them every sum of the
// warp fits 32 bits: the largest, of the squared rows, is at most
// kWarpBoxPx * kWarpBoxSide^2 / 3 + a lower term < 2^32.
constexpr int kWarpBoxPx = 8192, kWarpBoxSide = 1024;

__device__ __forceinline__ bool warp_box(int bh, int bw)
{
    return bh <= kWarpBoxSide && bw <= kWarpBoxSide && bh * bw <= kWarpBoxPx;
}

// Warp per object with a small box: intermediate results over its bounding
// box, 31 columns at a time (lane 31 is only the right neighbour of lane
// 30), row after row, so the neighbours come from a vote and the last row
// instead of memory. An inner pair of adjacent pixels hides two pixel
// edges: perimeter = 4 area - 2 pairs. Objects with a large box are listed
// for the blocks of the next kernel. With the histogram's part 24 us for the
// 2180 nuclei of a 4096 x 4096 tile, bound by the latency of a box's rows and
// the double-precision part (a block per object, with its barriers, 29, and
// 87 for the features by a warp each from 1.3 KB per object in memory; now
// 10).
__global__ void __launch_bounds__(kThreads) obj_inter_kernel(ObjArgs a)
{
    start_early();
    __shared__ __align__(16) uint32_t hist_of[kWarps][256];
    __shared__ __align__(16) uint32_t glcm_of[kWarps][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int limit = min((int)a.ctl[0], a.cap);
    uint32_t *hist = hist_of[warp], *glcm = glcm_of[warp];
    // warp 0 of every block first: fewer objects than warps spread over all SMs
    for (int64_t k = (int64_t)warp * gridDim.x + blockIdx.x; k < limit; k += (int64_t)gridDim.x * kWarps) {
        const int32_t l = a.olabel[k];
        const int4 b = reinterpret_cast<const int4 *>(a.box)[l];
        const int bh = b.z - b.x + 1, bw = b.w - b.y + 1;
        if (!warp_box(bh, bw)) {
            if (lane == 0) a.big[atomicAdd(a.ctl + 3, 1u)] = (int32_t)k;
            continue;
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2; ++q) reinterpret_cast<uint4 *>(hist)[lane + 32 * q] = make_uint4(0u, 0u, 0u, 0u);
        reinterpret_cast<uint2 *>(glcm)[lane] = make_uint2(0u, 0u);
        __syncwarp();
        uint32_t area = 0, vp = 0, hp = 0, sr = 0, sc = 0, srr = 0, scc = 0, src = 0, si = 0, sii = 0;
        for (int x0 = 0; x0 < bw; x0 += 31) {
            const int x = x0 + lane;
            const bool col = x < bw;
            const int32_t *Lp = a.L + (int64_t)b.x * a.ld_L + b.y + x;
            const uint8_t *Ip = a.I + (int64_t)b.x * a.ld_I + b.y + x;
            uint32_t n = 0, sy = 0, syy = 0;
            bool prev = false;
            for (int y0 = 0; y0 < bh; y0 += 8) {
                int32_t lv[8];
                int iv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const bool in = col && y0 + u < bh;
                    lv[u] = in ? Lp[(int64_t)(y0 + u) * a.ld_L] : -1;
                    iv[u] = in ? Ip[(int64_t)(y0 + u) * a.ld_I] : 0;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const bool in = lv[u] == l;
                    const uint32_t m = __ballot_sync(0xffffffffu, in);
                    const int vr = __shfl_down_sync(0xffffffffu, iv[u], 1);
                    if (in && lane < 31) {
                        const uint32_t y = (uint32_t)(y0 + u), v = (uint32_t)iv[u];
                        ++n;
                        sy += y;
                        syy += y * y;
                        si += v;
                        sii += v * v;
                        vp += prev;
                        atomicAdd(hist + v, 1u);
                        if ((m >> (lane + 1)) & 1u) {
                            ++hp;
                            atomicAdd(glcm + (v >> 5) * 8 + (vr >> 5), 1u);
                        }
                    }
                    prev = in;
                }
            }
            area += n;
            sr += sy;
            srr += syy;
            sc += n * x;
            scc += n * x * x;
            src += sy * x;
        }
        const uint32_t all = 0xffffffffu;
        area = __reduce_add_sync(all, area);
        const uint32_t pairs = __reduce_add_sync(all, vp + hp);
        sr = __reduce_add_sync(all, sr);
        sc = __reduce_add_sync(all, sc);
        srr = __reduce_add_sync(all, srr);
        scc = __reduce_add_sync(all, scc);
        src = __reduce_add_sync(all, src);
        si = __reduce_add_sync(all, si);
        sii = __reduce_add_sync(all, sii);
        ObjInter &o = a.inter[k];
        if (lane == 0) {
            o.area = area;
            o.per = 4 * (int64_t)area - 2 * (int64_t)pairs;
            o.sr = sr;
            o.sc = sc;
            o.srr = srr;
            o.scc = scc;
            o.src = src;
            o.si = si;
            o.sii = sii;
        }
        __syncwarp();
        obj_hist_stats(hist, glcm, area, o);
    }
}

// First the listed objects with a large box, a block each, from their
// intermediate results to the features; then four lanes per other object.
__global__ void __launch_bounds__(kThreads) obj_feature_kernel(ObjArgs a)
{
    start_early();
    __shared__ uint32_t hist[256], glcm[64];
    __shared__ unsigned long long sums[9];
    __shared__ int slot;
    if (a.ctl[3]) {
        for (;;) {
            const int k = next_big(a, &slot);
            if (k < 0) break;
            for (int i = threadIdx.x; i < 256; i += kThreads) hist[i] = 0u;
            if (threadIdx.x < 64) glcm[threadIdx.x] = 0u;
            if (threadIdx.x < 9) sums[threadIdx.x] = 0ull;
            __syncthreads();
            const int32_t l = a.olabel[k];
            const int4 b = reinterpret_cast<const int4 *>(a.box)[l];
            const int bh = b.z - b.x + 1, bw = b.w - b.y + 1;
            const int m = bh * bw;   // H * W <= 2^30
            int64_t area = 0, per = 0, sr = 0, sc = 0, srr = 0, scc = 0, src = 0, si = 0, sii = 0;
            for (int i = threadIdx.x; i < m; i += kThreads) {
                const int y = i / bw, x = i - y * bw;
                const int r = b.x + y, c = b.y + x;
                const int32_t *Lr = a.L + (int64_t)r * a.ld_L;
                if (Lr[c] != l) continue;
                const int v = a.I[(int64_t)r * a.ld_I + c];
                ++area;
                per += (r == 0 || Lr[c - a.ld_L] != l) + (r + 1 == a.H || Lr[c + a.ld_L] != l) +
                       (c == 0 || Lr[c - 1] != l);
                const bool right_in = c + 1 < a.W && Lr[c + 1] == l;
                per += !right_in;
                sr += y;
                sc += x;
                srr += (int64_t)y * y;
                scc += (int64_t)x * x;
                src += (int64_t)y * x;
                si += v;
                sii += (int64_t)v * v;
                atomicAdd(hist + v, 1u);
                if (right_in) atomicAdd(glcm + (v >> 5) * 8 + (a.I[(int64_t)r * a.ld_I + c + 1] >> 5), 1u);
            }
            const int64_t vals[9] = {area, per, sr, sc, srr, scc, src, si, sii};
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const int64_t v = warp_sum_l(vals[q]);
                if ((threadIdx.x & 31) == 0 && v) atomicAdd(sums + q, (unsigned long long)v);
            }
            __syncthreads();
            ObjInter &o = a.inter[k];
            if (threadIdx.x < 32) {
                if (threadIdx.x < 9) {
                    int64_t *dst = &o.area;
                    dst[threadIdx.x] = (int64_t)sums[threadIdx.x];
                }
                obj_hist_stats(hist, glcm, (int64_t)sums[0], o);
                __syncwarp();
                obj_finish(a, k, threadIdx.x & 3, threadIdx.x < 4);
            }
        }
    }
    const int limit = min((int)a.ctl[0], a.cap);
    const int64_t group = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;   // spread over the SMs
    for (int64_t k0 = group * 8; k0 < limit; k0 += (int64_t)gridDim.x * (kThreads / 4)) {
        int64_t k = k0 + ((threadIdx.x & 31) >> 2);
        bool on = k < limit;
        if (!on) k = k0;
        const int4 b = reinterpret_cast<const int4 *>(a.box)[a.olabel[k]];
        on &= warp_box(b.z - b.x + 1, b.w - b.y + 1);
        obj_finish(a, k, threadIdx.x & 3, on);
    }
}

int persistent_grid(const void *fn, size_t smem, int num_sms, int threads = kThreads)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        per_sm = 1;
    }
    return (per_sm > 0 ? per_sm : 1) * num_sms;
}

cudaError_t launch_object_features(const ObjArgs &a, int num_sms, cudaStream_t s, int *launches)
{
    *launches = 0;
    cudaError_t e = launch_enumeration(a, num_sms, s, launches);
    if (e != cudaSuccess) return e;
    if (a.cap < 1) return cudaSuccess;
    launch_early(obj_inter_kernel, (unsigned)persistent_grid((const void *)obj_inter_kernel, 0, num_sms), kThreads, 0, s, a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_early(obj_feature_kernel, (unsigned)(2 * num_sms), kThreads, 0, s, a);
    *launches += 2;
    return cudaGetLastError();
}

// -------------------------------------------------------------- watershed
// Views of one object's box for the watershed block: i = y * bw + x indexes
// the box. The shared-memory view holds D, R, the state and the flags of
// the box; the global view reads L and D in place and keeps R, the state
// and the flags in image-sized arrays (only the object's pixels are
// touched, so objects never share a word).
struct SmemView {
    int32_t *d, *r;
    unsigned long long *st;
    uint8_t *fl;   // bit 0: in the object, bit 1: not a maximum
    __device__ __forceinline__ bool in(int i) const { return fl[i] & 1u; }
    __device__ __forceinline__ int32_t D(int i) const { return d[i]; }
    __device__ __forceinline__ int32_t &R(int i) const { return r[i]; }
    __device__ __forceinline__ unsigned long long &S(int i) const { return st[i]; }
    __device__ __forceinline__ bool nm(int i) const { return fl[i] & 2u; }
    __device__ __forceinline__ void set_nm(int i) const { fl[i] |= 2u; }
};

struct GlobalView {
    const ObjArgs *a;
    int32_t label;
    int r0, c0, bw;
    __device__ __forceinline__ int64_t pix(int i) const
    {
        const int y = i / bw, x = i - y * bw;
        return (int64_t)(r0 + y) * a->W + (c0 + x);
    }
    __device__ __forceinline__ bool in(int i) const
    {
        const int y = i / bw, x = i - y * bw;
        return a->L[(int64_t)(r0 + y) * a->ld_L + c0 + x] == label;
    }
    __device__ __forceinline__ int32_t D(int i) const
    {
        const int y = i / bw, x = i - y * bw;
        return a->D[(int64_t)(r0 + y) * a->ld_D + c0 + x];
    }
    __device__ __forceinline__ int32_t &R(int i) const { return a->R[pix(i)]; }
    __device__ __forceinline__ unsigned long long &S(int i) const { return a->st[pix(i)]; }
    __device__ __forceinline__ bool nm(int i) const { return *reinterpret_cast<volatile uint8_t *>(a->nm + pix(i)) != 0; }
    __device__ __forceinline__ void set_nm(int i) const { a->nm[pix(i)] = 1u; }
};

// The threads that work on one object: a whole block (large boxes) or one
// warp (small boxes, eight objects per block in flight).
template <int NT>
struct BlockGroup {
    static constexpr int size = NT;
    int *red;   // shared reduction word
    __device__ __forceinline__ int rank() const { return threadIdx.x; }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    __device__ __forceinline__ bool any(bool p) const { return __syncthreads_or(p) != 0; }
    __device__ __forceinline__ int32_t max(int32_t v) const
    {
        v = __reduce_max_sync(0xffffffffu, v);
        __syncthreads();
        if (threadIdx.x == 0) *red = -1;
        __syncthreads();
        if ((threadIdx.x & 31) == 0) atomicMax(red, v);
        __syncthreads();
        return *red;
    }
};


// Largest D below `below` over the object's pixels that have no basin yet
// (-1: none). The levels strictly descend, so the flooding ends; a pixel
// left unlabelled at one level (not yet connected to a basin) is taken at a
// lower one, when its level set joins a basin.
template <class V, class G>
__device__ __forceinline__ int32_t max_unlabelled(const V &v, const G &g, int m, int32_t below)
{
    int32_t mx = -1;
    for (int i = g.rank(); i < m; i += G::size)
        if (v.in(i) && v.S(i) == kUnl && v.D(i) < below) mx = max(mx, v.D(i));
    return g.max(mx);
}

template <class V, class G>
__device__ void watershed_object(const V &v, const G &g, const ObjArgs &a, int r0, int c0, int bh, int bw)
{
    const int m = bh * bw;   // H * W <= 2^30
    auto for_nbrs = [&](int i, auto &&fn) {
        const int y = i / bw, x = i - y * bw;
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                if (dy == 0 && dx == 0) continue;
                const int yy = y + dy, xx = x + dx;
                if (yy < 0 || yy >= bh || xx < 0 || xx >= bw) continue;
                const int j = yy * bw + xx;
                if (v.in(j)) fn(j);
            }
    };
    // 1. h-maxima transform: R = reconstruction of max(D - h, 0) under D
    for (int i = g.rank(); i < m; i += G::size)
        if (v.in(i)) v.R(i) = max(v.D(i) - a.h, 0);
    g.sync();
    for (;;) {
        int ch = 0;
        for (int i = g.rank(); i < m; i += G::size) {
            if (!v.in(i)) continue;
            volatile int32_t &Ri = v.R(i);
            int32_t mx = Ri;
            for_nbrs(i, [&](int j) { mx = max(mx, *(volatile int32_t *)&v.R(j)); });
            mx = min(mx, v.D(i));
            if (mx > Ri) {
                Ri = mx;
                ch = 1;
            }
        }
        if (!g.any(ch)) break;
    }
    // 2. not a maximum: a higher neighbour, or an equal one that is not
    for (int i = g.rank(); i < m; i += G::size) {
        if (!v.in(i)) continue;
        bool hi = false;
        const int32_t ri = v.R(i);
        for_nbrs(i, [&](int j) { hi |= v.R(j) > ri; });
        if (hi) v.set_nm(i);
    }
    g.sync();
    for (;;) {
        int ch = 0;
        for (int i = g.rank(); i < m; i += G::size) {
            if (!v.in(i) || v.nm(i)) continue;
            bool f = false;
            const int32_t ri = v.R(i);
            for_nbrs(i, [&](int j) { f |= v.R(j) == ri && v.nm(j); });
            if (f) {
                v.set_nm(i);
                ch = 1;
            }
        }
        if (!g.any(ch)) break;
    }
    // 3. markers: each plateau of maxima takes its smallest linear index
    for (int i = g.rank(); i < m; i += G::size) {
        if (!v.in(i)) continue;
        const int y = i / bw, x = i - y * bw;
        v.S(i) = v.nm(i) ? kUnl : (unsigned long long)(uint32_t)((r0 + y) * a.W + (c0 + x));
    }
    g.sync();
    for (;;) {
        int ch = 0;
        for (int i = g.rank(); i < m; i += G::size) {
            if (!v.in(i) || v.nm(i)) continue;
            volatile unsigned long long &Si = v.S(i);
            unsigned long long mn = Si;
            for_nbrs(i, [&](int j) {
                if (!v.nm(j)) {
                    const unsigned long long sj = *(volatile unsigned long long *)&v.S(j);
                    mn = sj < mn ? sj : mn;
                }
            });
            if (mn < Si) {
                Si = mn;
                ch = 1;
            }
        }
        if (!g.any(ch)) break;
    }
    int nb = 0;
    for (int i = g.rank(); i < m; i += G::size) {
        if (!v.in(i) || v.nm(i)) continue;
        const int y = i / bw, x = i - y * bw;
        nb += v.S(i) == (unsigned long long)(uint32_t)((r0 + y) * a.W + (c0 + x));
    }
    nb = __reduce_add_sync(0xffffffffu, nb);
    if ((g.rank() & 31) == 0 && nb && a.n_basins) atomicAdd(a.n_basins, nb);
    // 4. flooding by levels of D, highest first, in breadth-first layers. A
    // level ends after the first layer whose new pixels have no unlabelled
    // neighbour with D >= t (the next layer could only take such pixels);
    // the next level, the largest D below t among unlabelled pixels, is
    // found during the level's first layer (those pixels do not change
    // within the level).
    uint32_t layer = 1;
    int32_t t = max_unlabelled(v, g, m, INT32_MAX);
    while (t >= 0) {
        int32_t next = -1;
        for (bool first = true;; first = false) {
            int more = 0;
            for (int i = g.rank(); i < m; i += G::size) {
                if (!v.in(i) || v.S(i) != kUnl) continue;
                const int32_t di = v.D(i);
                if (di < t) {
                    if (first) next = max(next, di);
                    continue;
                }
                uint32_t mn = 0xffffffffu;
                for_nbrs(i, [&](int j) {
                    const unsigned long long sj = *(volatile unsigned long long *)&v.S(j);
                    if (sj != kUnl && (uint32_t)(sj >> 32) < layer) mn = min(mn, (uint32_t)sj);
                });
                if (mn != 0xffffffffu) {
                    *(volatile unsigned long long *)&v.S(i) = ((unsigned long long)layer << 32) | mn;
                    for_nbrs(i, [&](int j) {
                        more |= *(volatile unsigned long long *)&v.S(j) == kUnl && v.D(j) >= t;
                    });
                }
            }
            ++layer;
            if (first) next = g.max(next);
            if (!g.any(more)) break;
        }
        t = next;
    }
    // 5. basins out
    for (int i = g.rank(); i < m; i += G::size) {
        if (!v.in(i)) continue;
        const int y = i / bw, x = i - y * bw;
        a.basins[(int64_t)(r0 + y) * a.ld_B + (c0 + x)] = (int32_t)(uint32_t)v.S(i);
    }
}

constexpr int kWsThreads = 256;
constexpr size_t kWsSmemBytes = (size_t)kWsSmemPx * (4 + 4 + 8 + 1) + 64;

// Carves a shared-memory view of `px` pixels at base (8-byte aligned).
__device__ __forceinline__ SmemView smem_view(unsigned char *base, int px)
{
    SmemView sv;
    sv.st = reinterpret_cast<unsigned long long *>(base);
    sv.d = reinterpret_cast<int32_t *>(sv.st + px);
    sv.r = sv.d + px;
    sv.fl = reinterpret_cast<uint8_t *>(sv.r + px);
    return sv;
}

// ---- small boxes: one warp per object, four for the medium ones, a block for a few
// Box cells (the object's box with a border of one cell) of the slots of a
// block: its first four warps share one for medium boxes, each of the
// others has one for small boxes. Four such blocks share an SM.
constexpr int kWsSmallPx = 640, kWsMediumPx = 2944, kWsMediumWarps = 4;
constexpr int kWsCellBytes = 10;
constexpr size_t kWsWarpSmem = (size_t)kWsCellBytes * (kWsMediumPx + (kWarps - kWsMediumWarps) * kWsSmallPx);
constexpr int kWsScan = 1;   // objects the warps of the medium boxes look at in one turn

// The NW warps that work on one object: votes and lists over all of them.
// The first NW warps of the block if NW > 1; sh: their words in shared
// memory (0: length of the list, 1: cells, 2: largest, 3: smallest).
template <int NW>
struct WarpsOf {
    static constexpr int size = 32 * NW;
    int *sh;
    __device__ __forceinline__ int rank() const { return NW == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x; }
    __device__ __forceinline__ void sync() const
    {
        if (NW == 1) __syncwarp();
        else asm volatile("barrier.cta.sync 1, %0;" ::"n"(size) : "memory");
    }
    // syncs
    __device__ __forceinline__ bool any(bool p) const
    {
        if (NW == 1) {
            __syncwarp();
            return __any_sync(0xffffffffu, p);
        }
        uint32_t r;
        asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, %2, p;\n"
                     " selp.u32 %0, 1, 0, q;\n}" : "=r"(r) : "r"((uint32_t)p), "n"(size) : "memory");
        return r != 0;
    }
    // Place of this thread's entry in a list of n so far (all threads call it; n is kept here if NW = 1,
    // else in sh[0])
    __device__ __forceinline__ int place(bool p, int &n) const
    {
        const uint32_t t = __ballot_sync(0xffffffffu, p);
        const int before = __popc(t & ((1u << (threadIdx.x & 31)) - 1u));
        int at = n;
        if (NW == 1) {
            n += __popc(t);
        } else {
            if ((threadIdx.x & 31) == 0 && t) at = atomicAdd(sh, __popc(t));
            at = __shfl_sync(0xffffffffu, at, 0);
        }
        return at + before;
    }
    // Largest and smallest of v and w; syncs
    __device__ __forceinline__ void range(int &v, int &w) const
    {
        v = __reduce_max_sync(0xffffffffu, v);
        w = __reduce_min_sync(0xffffffffu, w);
        if (NW > 1 && (threadIdx.x & 31) == 0) {
            atomicMax(sh + 2, v);
            atomicMin(sh + 3, w);
        }
        sync();
        if (NW == 1) return;
        v = *(volatile int *)(sh + 2);
        w = *(volatile int *)(sh + 3);
    }
};

// lab: the cell that names the basin, or no basin yet, or outside the object (as D there)
constexpr uint32_t kNone = 0xfffeu, kOut = 0xffffu;

// Smallest basin beside a cell (from kNone on: none)
__device__ __forceinline__ uint32_t least_beside(const volatile uint16_t *lab, int i, int pw)
{
    const volatile uint16_t *u = lab + i - pw, *d = lab + i + pw;
    const uint32_t u0 = u[-1], u1 = u[0], u2 = u[1], l = lab[i - 1], r = lab[i + 1], d0 = d[-1], d1 = d[0], d2 = d[1];
    return min(min(min(u0, u1), min(u2, l)), min(min(r, d0), min(d1, d2)));
}

__device__ __forceinline__ uint32_t most_beside(const volatile uint16_t *R, int i, int pw)
{
    const volatile uint16_t *u = R + i - pw, *d = R + i + pw;
    const uint32_t a = max(max((uint32_t)u[-1], (uint32_t)u[0]), (uint32_t)u[1]);
    const uint32_t b = max((uint32_t)R[i - 1], (uint32_t)R[i + 1]);
    const uint32_t c = max(max((uint32_t)d[-1], (uint32_t)d[0]), (uint32_t)d[1]);
    return max(max(a, b), c);
}

// Flooding by levels, highest first, in breadth-first layers, by one warp:
// the cells at this level or above it without a basin that see one take the
// smallest, all of a layer at once. A window of 32 cells of the list is
// kept in registers, so an ordinary level, a few cells in one layer, costs
// one look at the neighbours; cells that see no basin yet wait in act. A
// level of more than a window, or with cells waiting (one in 200), goes
// through act, with R for a layer's answers. (Four warps on one object
// spent three times as long here, in barriers.)
__device__ __forceinline__ void flood_levels(int n, const uint16_t *D, const uint16_t *list, volatile uint16_t *lab,
                             volatile uint16_t *R, uint16_t *act, int pw)
{
    const int lane = threadIdx.x & 31;
    const uint32_t all = 0xffffffffu, lt = (1u << lane) - 1u;
    int na = 0, at = -32;   // waiting; place of the window
    int i = 0;
    uint32_t d = 0, starts = 0, need = 0;   // of the window's cells: first of a level, no basin yet
    const volatile uint16_t *up = lab, *dn = lab;
    auto window = [&](int pos) {
        at = pos;
        const bool have = pos + lane < n;
        i = have ? list[pos + lane] : pw + 1;
        d = have ? D[i] : 0x10000u;
        up = lab + i - pw;
        dn = lab + i + pw;
        const uint32_t before = __shfl_up_sync(all, d, 1);
        starts = __ballot_sync(all, lane == 0 || d != before);
        need = __ballot_sync(all, have && lab[i] == kNone);
    };
    for (int pos = 0; pos < n;) {
        if (at < 0 || pos - at >= 32) window(pos);
        uint32_t later = starts & ~((2u << (pos - at)) - 1u);   // 2 << 31 is 0: none
        if (!later && pos > at && at + 32 < n) {   // the level may go on
            window(pos);
            later = starts & ~1u;
        }
        if ((later || at + 32 >= n) && na == 0) {
            const int o = pos - at, e = later ? __ffs(later) - 1 : 32;
            pos = min(at + e, n);
            uint32_t m = need & (~0u << o) & (e < 32 ? (1u << e) - 1u : ~0u);
            while (m) {
                const uint32_t u0 = up[-1], u1 = up[0], u2 = up[1], l = up[pw - 1], r = up[pw + 1], d0 = dn[-1],
                               d1 = dn[0], d2 = dn[1];
                const uint32_t v = min(min(min(u0, u1), min(u2, l)), min(min(r, d0), min(d1, d2)));
                const bool one = (m >> lane) & 1u, got = one && v < kNone;
                const uint32_t rest = __ballot_sync(all, one && !got);   // after all have looked
                if (got) lab[i] = (uint16_t)v;
                __syncwarp();
                if (rest == m) break;
                m = rest;
            }
            if (m) {
                if ((m >> lane) & 1u) act[__popc(m & lt)] = (uint16_t)i;
                na = __popc(m);
                __syncwarp();
            }
            continue;
        }
        const uint32_t t = D[list[pos]];
        for (;;) {
            const bool have = pos + lane < n;
            const int j = have ? list[pos + lane] : 0;
            const uint32_t eq = __ballot_sync(all, have && D[j] == t);
            const bool take = ((eq >> lane) & 1u) && lab[j] == kNone;
            const uint32_t tk = __ballot_sync(all, take);
            if (take) act[na + __popc(tk & lt)] = (uint16_t)j;
            na += __popc(tk);
            pos += __popc(eq);
            if (eq != all) break;
        }
        at = -32;   // the window's cells may have got theirs
        __syncwarp();
        while (na > 0) {
            for (int q = lane; q < na; q += 32) R[q] = (uint16_t)least_beside(lab, act[q], pw);
            __syncwarp();
            int kept = 0;
            for (int q0 = 0; q0 < na; q0 += 32) {
                const bool have = q0 + lane < na;
                const int j = have ? act[q0 + lane] : 0;
                const uint32_t v = have ? R[q0 + lane] : kNone;
                const bool got = v < kNone;
                const uint32_t rest = __ballot_sync(all, have && !got);
                if (got) lab[j] = (uint16_t)v;
                else if (have) act[kept + __popc(rest & lt)] = (uint16_t)j;
                kept += __popc(rest);
            }
            __syncwarp();
            const bool none = kept == na;
            na = kept;
            if (none) break;
        }
    }
}

// The watershed of one object, all of it in shared memory, 16 bits a value:
// local cell indices and distances below the number of cells (larger or
// negative distances, which no distance map of the object itself has:
// false, nothing done). The object's cells are listed by descending
// distance (counting sort): a level of the flooding is then a stretch of
// the list, so a layer costs a step for the cells that can change, where a
// sweep over the box costs one for all of them (100 sweeps an object); and
// the h-maxima's reconstruction, swept in that order, carries a peak's value
// to the foot of its hill in a few sweeps. What is left is the latency of a
// chain of dependent steps, 13 us for a nucleus on average and 40 for the
// longest: 4096 x 4096 with 2180 nuclei 471 -> 56 us (a block per object,
// with its barriers and 96 thousand instructions).
template <int NW>
__device__ __forceinline__ bool watershed_small(const ObjArgs &a, int4 b, int32_t l, uint16_t *mem, int cells, int *sh)
{
    const WarpsOf<NW> g{sh};
    constexpr int kN = WarpsOf<NW>::size;
    constexpr int kLoad = NW == 1 ? 8 : 4;   // loads of each kind in flight
    const int lane = threadIdx.x & 31, rank = g.rank();
    const uint32_t all = 0xffffffffu;
    const int bh = b.z - b.x + 1, bw = b.w - b.y + 1, pw = bw + 2, m = (bh + 2) * pw;
    uint16_t *D = mem, *list = D + cells;
    volatile uint16_t *lab = list + cells, *R = lab + cells;
    uint16_t *act = const_cast<uint16_t *>(R) + cells;   // 4-byte aligned (cells is even)
    uint32_t *hist = reinterpret_cast<uint32_t *>(act);  // 16-bit counters, two a word, before act's use
    const int sy = kN / pw, sx = kN - sy * pw;
    auto step = [&](int &y, int &x) {
        y += sy;
        x += sx;
        if (x >= pw) {
            x -= pw;
            ++y;
        }
    };
    g.sync();   // the object before has read its words
    if (NW > 1 && rank < 4) sh[rank] = 0;
    for (int i = rank; 2 * i < m; i += kN) hist[i] = 0u;
    g.sync();
    int mx = 0, mn = 0;
    {
        int y = rank / pw, x = rank - y * pw;
        for (int i0 = rank; i0 < m; i0 += kLoad * kN) {
            int32_t lv[kLoad], dv[kLoad];
#pragma unroll
            for (int u = 0; u < kLoad; ++u, step(y, x)) {
                lv[u] = ~l;
                dv[u] = 0;
                if (y >= 1 && y <= bh && x >= 1 && x <= bw) {
                    const int64_t r = b.x + y - 1, c = b.y + x - 1;
                    lv[u] = a.L[r * a.ld_L + c];
                    dv[u] = a.D[r * a.ld_D + c];
                }
            }
#pragma unroll
            for (int u = 0; u < kLoad; ++u) {
                const int i = i0 + kN * u;
                if (i >= m) break;
                const bool in = lv[u] == l;
                const int32_t d = in ? dv[u] : 0;
                mx = max(mx, d);
                mn = min(mn, d);
                D[i] = in ? (uint16_t)d : (uint16_t)kOut;
                lab[i] = (uint16_t)(in ? kNone : kOut);
                R[i] = (uint16_t)max(d - a.h, 0);   // 0, which raises nothing, outside
                if (in && d >= 0 && d < m) atomicAdd(hist + (d >> 1), 1u << (16 * (d & 1)));
            }
        }
    }
    g.range(mx, mn);
    if (mx >= m || mn < 0) return false;
    // counting sort, largest distance first
    int n = 0;
    if (rank < 32) {
        volatile uint16_t *h16 = act;
        for (int j = mx; j >= 0; j -= 32) {
            const int bin = j - lane;
            const uint32_t v = bin >= 0 ? h16[bin] : 0u;
            uint32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(all, inc, o);
                if (lane >= o) inc += t;
            }
            if (bin >= 0) h16[bin] = (uint16_t)(n + inc - v);
            n += __shfl_sync(all, inc, 31);
        }
        if (NW > 1 && lane == 0) sh[1] = n;
    }
    g.sync();
    if (NW > 1) n = *(volatile int *)(sh + 1);
    for (int i0 = rank; i0 < m; i0 += 4 * kN) {
        uint32_t d[4], at[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) d[u] = i0 + kN * u < m ? D[i0 + kN * u] : kOut;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (d[u] != kOut) at[u] = atomicAdd(hist + (d[u] >> 1), 1u << (16 * (d[u] & 1)));
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (d[u] != kOut) list[(at[u] >> (16 * (d[u] & 1))) & 0xffffu] = (uint16_t)(i0 + kN * u);
    }
    g.sync();
    // 1. h-maxima transform: R = reconstruction of max(D - h, 0) under D. Two cells a lane are taken until
    // they rest before the next ones (a value crosses a flat stretch of the list without a sweep for every
    // step). The last sweep, which changes nothing, leaves the cell in lab where no neighbour is higher
    for (;;) {
        bool ch = false;
        for (int q0 = 0; q0 < n; q0 += 2 * kN) {
            const int q = q0 + rank;
            if (q0 + (rank & ~31) >= n) break;   // whole warp
            const bool one = q < n, two = q + kN < n;
            const int i = one ? list[q] : pw + 1, j = two ? list[q + kN] : i;
            const uint32_t di = one ? D[i] : 0u, dj = two ? D[j] : di;
            for (;;) {
                const uint32_t ri = R[i], rj = R[j];
                const uint32_t ni = most_beside(R, i, pw), nj = most_beside(R, j, pw);
                const uint32_t vi = min(ni, di), vj = min(nj, dj);
                const bool f = vi > ri || vj > rj;
                if (vi > ri) R[i] = (uint16_t)vi;
                if (vj > rj) R[j] = (uint16_t)vj;
                ch |= f;
                if (__any_sync(all, f)) continue;
                if (one) lab[i] = (uint16_t)(ni <= ri ? i : kNone);
                if (two) lab[j] = (uint16_t)(nj <= rj ? j : kNone);
                break;
            }
        }
        if (!g.any(ch)) break;
    }
    // 2. of these the ones not on a plateau that has a higher neighbour elsewhere
    int na = 0;
    for (int q0 = 0; q0 < n; q0 += kN) {
        const int i = q0 + rank < n ? list[q0 + rank] : 0;
        const bool top = q0 + rank < n && lab[i] != kNone;
        const int at = g.place(top, na);
        if (top) act[at] = (uint16_t)i;
    }
    g.sync();
    if (NW > 1) na = *(volatile int *)sh;
    // and 3. markers: each plateau of maxima takes its smallest index. Up to 32 cells (nearly always): a warp
    // notes which are neighbours of the same height and goes from cell to cell by votes. More: every cell of a
    // plateau takes the smallest name around, and its name's name, until all have one; a name is marked in R
    // if a cell of its plateau has a neighbour of the same height that is no candidate (it has a higher one)
    int nb = 0;
    auto nbr = [&](int i, int z) { return i + (z / 3 - 1) * pw + z % 3 - 1; };   // z = 0 .. 8, 4: i itself
    if (na <= 32) {
        if (rank < 32) {
            const bool top = lane < na;
            const int i = top ? act[lane] : pw + 1;
            if (top) lab[i] = (uint16_t)lane;
            __syncwarp();
            const uint32_t r = R[i];
            uint32_t beside = 0;
            bool f = !top;
#pragma unroll
            for (int z = 0; z < 9; ++z) {
                if (z == 4) continue;
                const uint32_t v = lab[nbr(i, z)], rv = R[nbr(i, z)];
                if (rv == r && v < kNone) beside |= 1u << v;
                f |= rv == r && v == kNone;
            }
            if (!top) beside = 0;
            uint32_t fallen = __ballot_sync(all, f);
            for (;;) {
                const uint32_t more = fallen | __ballot_sync(all, (beside & fallen) != 0);
                if (more == fallen) break;
                fallen = more;
            }
            uint32_t left = ~fallen;
            const bool stays = (left >> lane) & 1u;
            uint32_t name = kNone;
            while (left) {
                uint32_t flat = left & -left;   // the plateau of the first cell left
                for (;;) {
                    const uint32_t more = flat | __ballot_sync(all, (beside & flat) != 0);
                    if (more == flat) break;
                    flat = more;
                }
                const bool here = (flat >> lane) & 1u;
                const uint32_t least = __reduce_min_sync(all, here ? (uint32_t)i : kNone);
                if (here) name = least;
                left &= ~flat;
            }
            if (top) lab[i] = (uint16_t)name;
            nb = stays && name == (uint32_t)i;
            if (nb) act[cells - 1] = (uint16_t)i;   // no list reaches there
        }
    } else {
        for (;;) {
            bool ch = false;
            for (int q = rank; q < na; q += kN) {
                const int i = act[q];
                const uint32_t own = lab[i], r = R[i];
                uint32_t v = own;
#pragma unroll
                for (int z = 0; z < 9; ++z) {
                    const uint32_t u = z != 4 ? (uint32_t)lab[nbr(i, z)] : kNone;
                    if (u < v && R[nbr(i, z)] == r) v = u;
                }
                v = lab[v];   // names are cells of the plateau, and fall along these links
                if (v < own) {
                    lab[i] = (uint16_t)v;
                    if (v < lab[own]) lab[own] = (uint16_t)v;
                    ch = true;
                }
            }
            if (!g.any(ch)) break;
        }
        constexpr uint32_t kFalls = 0x8000u;   // above all cells
        for (int q = rank; q < na; q += kN) {
            const int i = act[q];
            const uint32_t r = R[i];
            bool f = false;
#pragma unroll
            for (int z = 0; z < 9; ++z)
                if (z != 4) f |= lab[nbr(i, z)] == kNone && R[nbr(i, z)] == r;
            if (f) act[q] = (uint16_t)(i | kFalls);
        }
        g.sync();   // all heights have been read
        for (int q = rank; q < na; q += kN)
            if (act[q] & kFalls) R[lab[act[q] & ~kFalls]] = (uint16_t)kFalls;
        g.sync();
        for (int q = rank; q < na; q += kN) {
            const int i = act[q] & ~kFalls;
            const uint32_t own = lab[i];
            const bool marker = R[own] != kFalls;
            if (!marker) lab[i] = (uint16_t)kNone;
            if (marker && own == (uint32_t)i) {
                ++nb;
                act[cells - 1] = (uint16_t)i;
            }
        }
    }
    nb = __reduce_add_sync(all, nb);
    if (lane == 0 && nb) {
        if (a.n_basins) atomicAdd(a.n_basins, nb);
        if (NW > 1) atomicAdd(sh + 3, nb);   // 0 here: the smallest distance, and nothing below 0
    }
    g.sync();
    if (NW > 1) nb = *(volatile int *)(sh + 3);
    // 4. flooding; with one marker every cell ends in its basin: each 8-connected part of the object has one
    const uint32_t only = nb == 1 ? act[cells - 1] : kNone;
    if (nb != 1) {
        if (rank < 32) flood_levels(n, D, list, lab, R, act, pw);
        g.sync();
    }
    // 5. basins out. A cell index over pw by a reciprocal: both below 2^13, so the half keeps it exact
    const float inv = 1.0f / (float)pw;
    {
        const uint16_t *done = const_cast<const uint16_t *>(lab);
        int y = rank / pw, x = rank - y * pw;
        for (int i0 = rank; i0 < m; i0 += 4 * kN) {
            uint32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = i0 + kN * u < m ? done[i0 + kN * u] : kOut;
#pragma unroll
            for (int u = 0; u < 4; ++u, step(y, x)) {
                if (v[u] == kOut) continue;
                if (nb == 1) v[u] = only;
                const int by = (int)(((float)v[u] + 0.5f) * inv), bx = (int)v[u] - by * pw;
                a.basins[(int64_t)(b.x + y - 1) * a.ld_B + b.y + x - 1] =
                    v[u] == kNone ? -1 : (b.x + by - 1) * a.W + b.y + bx - 1;
            }
        }
    }
    return true;
}

// The first warps of a block take the objects with a medium box and list
// those with a larger one, the others take the objects with a small box;
// each kind goes over the whole list of objects, so no pass sorts them by
// size first.
__global__ void __launch_bounds__(kThreads, 4) obj_watershed_small_kernel(ObjArgs a)
{
    start_early();
    extern __shared__ __align__(16) uint16_t slots[];
    __shared__ int sh[5];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_obj = (int)a.ctl[0];
    if (warp < kWsMediumWarps) {
        const WarpsOf<kWsMediumWarps> g{sh};
        for (;;) {
            g.sync();
            if (threadIdx.x == 0) sh[4] = (int)atomicAdd(a.ctl + 4, (uint32_t)kWsScan);
            g.sync();
            const int k0 = *(volatile int *)(sh + 4);
            if (k0 >= n_obj) return;
            // the boxes of the turn side by side; every warp comes to the same answer
            int4 b = make_int4(0, 0, 0, 0);
            int32_t l = 0;
            int64_t m = 0;
            if (lane < kWsScan && k0 + lane < n_obj) {
                l = a.olabel[k0 + lane];
                b = reinterpret_cast<const int4 *>(a.box)[l];
                m = (int64_t)(b.z - b.x + 3) * (b.w - b.y + 3);
            }
            uint32_t todo = __ballot_sync(0xffffffffu, m > kWsSmallPx);
            for (; todo; todo &= todo - 1) {
                const int j = __ffs(todo) - 1;
                const int4 bj = make_int4(__shfl_sync(0xffffffffu, b.x, j), __shfl_sync(0xffffffffu, b.y, j),
                                          __shfl_sync(0xffffffffu, b.z, j), __shfl_sync(0xffffffffu, b.w, j));
                const int32_t lj = __shfl_sync(0xffffffffu, l, j);
                if (__shfl_sync(0xffffffffu, m, j) > kWsMediumPx ||
                    !watershed_small<kWsMediumWarps>(a, bj, lj, slots, kWsMediumPx, sh)) {
                    if (threadIdx.x == 0) a.big[atomicAdd(a.ctl + 3, 1u)] = k0 + j;
                }
            }
        }
    }
    uint16_t *mem = slots + (size_t)(kWsCellBytes / 2) * (kWsMediumPx + (warp - kWsMediumWarps) * kWsSmallPx);
    for (;;) {
        int k = 0;
        if (lane == 0) k = (int)atomicAdd(a.ctl + 5, 1u);
        k = __shfl_sync(0xffffffffu, k, 0);
        if (k >= n_obj) return;
        const int32_t l = a.olabel[k];
        const int4 b = reinterpret_cast<const int4 *>(a.box)[l];
        if ((int64_t)(b.z - b.x + 3) * (b.w - b.y + 3) > kWsSmallPx) continue;
        if (!watershed_small<1>(a, b, l, mem, kWsSmallPx, nullptr) && lane == 0)
            a.big[atomicAdd(a.ctl + 3, 1u)] = k;
    }
}

// A block per listed object. Boxes of up to kWsBlockCells cells as above;
// the others, and objects whose distances do not fit there, by sweeps over
// the box: in shared memory up to kWsSmemPx pixels, else in the image-sized
// global arrays.
constexpr int kWsBlockCells = (int)(kWsSmemBytes / kWsCellBytes) & ~1;

__global__ void __launch_bounds__(kWsThreads) obj_watershed_kernel(ObjArgs a)
{
    start_early();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int slot, red, sh[4];
    const SmemView sv = smem_view(smem, kWsSmemPx);
    const BlockGroup<kWsThreads> g{&red};
    if (a.ctl[3] == 0) return;
    for (;;) {
        const int k = next_big(a, &slot);
        if (k < 0) return;
        const int32_t l = a.olabel[k];
        const int4 b = reinterpret_cast<const int4 *>(a.box)[l];
        const int bh = b.z - b.x + 1, bw = b.w - b.y + 1;
        const int m = bh * bw;   // H * W <= 2^30
        const int64_t cells = (int64_t)(bh + 2) * (bw + 2);
        if (cells > kWsMediumPx && cells <= kWsBlockCells &&
            watershed_small<kWsThreads / 32>(a, b, l, reinterpret_cast<uint16_t *>(smem), kWsBlockCells, sh))
            continue;
        if (m <= kWsSmemPx) {
            for (int i = threadIdx.x; i < m; i += kWsThreads) {
                const int y = i / bw, x = i - y * bw;
                const int r = b.x + y, c = b.y + x;
                const bool in = a.L[(int64_t)r * a.ld_L + c] == l;
                sv.fl[i] = in ? 1u : 0u;
                sv.d[i] = in ? a.D[(int64_t)r * a.ld_D + c] : 0;
            }
            __syncthreads();
            watershed_object(sv, g, a, b.x, b.y, bh, bw);
        } else {
            GlobalView gv{&a, l, b.x, b.y, bw};
            for (int i = threadIdx.x; i < m; i += kWsThreads)
                if (gv.in(i)) a.nm[gv.pix(i)] = 0u;
            __syncthreads();
            watershed_object(gv, g, a, b.x, b.y, bh, bw);
        }
    }
}

cudaError_t launch_watershed(const ObjArgs &a, int num_sms, cudaStream_t s, int *launches)
{
    *launches = 0;
    cudaError_t e = launch_enumeration(a, num_sms, s, launches);
    if (e != cudaSuccess) return e;
    const cudaFuncAttribute dyn = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if ((e = cudaFuncSetAttribute(obj_watershed_small_kernel, dyn, (int)kWsWarpSmem)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(obj_watershed_kernel, dyn, (int)kWsSmemBytes)) != cudaSuccess) return e;
    launch_early(obj_watershed_small_kernel, (unsigned)persistent_grid((const void *)obj_watershed_small_kernel, kWsWarpSmem, num_sms), kThreads, kWsWarpSmem, s, a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_early(obj_watershed_kernel, (unsigned)persistent_grid((const void *)obj_watershed_kernel, kWsSmemBytes, num_sms, kWsThreads), kWsThreads, kWsSmemBytes, s, a);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace rtk
