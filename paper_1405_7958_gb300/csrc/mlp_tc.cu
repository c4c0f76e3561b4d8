// The picker network's forward pass on the 5th-generation tensor cores
// (tcgen05), for training batches.
//
// One CTA of 256 threads takes 128 samples: the M = 128 rows of three
// products whose accumulators live in tensor memory,
//   H1 = Xn W1^T (K = 24, padded to 32),  H2 = relu(H1 + b1) W2^T (K = 64),
//   Z  = relu(H2 + b2) W3^T (N = 3, padded to 16),
// with bf16 operands (the parameters are bf16 already; the normalised input
// and the two hidden layers are rounded to bf16 to enter a product) and fp32
// accumulation. Threads t and t + 128 own sample t: each writes one half of
// the columns of row t of an A operand and reads that half of row t
// (tensor-memory lane t) of an accumulator. One thread issues the products;
// their completion arrives on an mbarrier. The products are a few hundred
// cycles: what counts is the latency of the chain and the number of memory
// instructions around them, so global and shared memory are accessed 16
// bytes at a time (VEC: the pointers are 16-byte aligned; else 2 or 4 bytes),
// the input by all threads in order, and the samples' columns are halved
// between two threads. Batch of 256: forward 9 us, backward 10 (a thread
// per sample, 2- and 4-byte accesses a row apart: 30 and 34).
//
// Operands sit in shared memory in the no-swizzle K-major layout of 8-row x
// 16-byte core matrices: element (r, k) of a K-wide operand is at
//   (r / 8) * (K / 8) * 128 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2
// bytes, so core matrices are 128 bytes apart along K (leading byte offset)
// and K * 16 bytes apart along M or N (stride byte offset).
#include <cuda_bf16.h>

#include "mlp.cuh"

namespace rtk {
namespace {

constexpr int kTcM = 128;       // samples per CTA = tensor-memory lanes
constexpr int kTcThreads = 2 * kTcM;
constexpr int kK1 = 32;         // layer 1 K: 24 inputs, zero-padded
constexpr int kN3 = 16;         // layer 3 N: 3 outputs, zero-padded
constexpr int kTmemCols = 256;  // H1 at columns 0..63, H2 at 64..127, Z at 128..143

// shared memory (bytes): the three A operands share one buffer in turn
constexpr int kOffA = 0;                          // 128 x 64 bf16 (layer 1 uses 128 x 32)
constexpr int kOffB1 = kOffA + kTcM * kMlpH * 2;  // 64 x 32
constexpr int kOffB2 = kOffB1 + kMlpH * kK1 * 2;  // 64 x 64
constexpr int kOffB3 = kOffB2 + kMlpH * kMlpH * 2;   // 16 x 64
constexpr int kOffEnd = kOffB3 + kN3 * kMlpH * 2;
constexpr int kTcSmem = kOffEnd;

__device__ __forceinline__ uint32_t core_off(int r, int k, int K)
{
    return (uint32_t)((r >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading byte offset (128:
// next core matrix along K), stride byte offset (K * 16: next 8 rows), the
// descriptor version bit of this architecture, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, int K)
{
    const uint64_t lbo = 128, sbo = (uint64_t)K * 16;
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((lbo >> 4) << 16) | ((sbo >> 4) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, N and M
__host__ __device__ constexpr uint32_t instr_desc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :
        : "r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

// waits for the mbarrier phase `parity` to complete; false after the bound
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    for (uint32_t k = 0; k < (1u << 22); ++k) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        if (k > 64) __nanosleep(32);
    }
    return false;
}

// 16 consecutive fp32 accumulator columns of this thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ uint16_t to_bf16(float f) { return __bfloat16_as_ushort(__float2bfloat16_rn(f)); }

__device__ __forceinline__ uint32_t two_bf16(float a, float b)
{
    return (uint32_t)to_bf16(a) | ((uint32_t)to_bf16(b) << 16);
}

__device__ __forceinline__ float of_bf16(uint16_t u) { return __uint_as_float((uint32_t)u << 16); }

template <bool VEC>
__device__ __forceinline__ void load4(const float *p, float *v)
{
    if (VEC) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = p[i];
    }
}

template <bool VEC>
__device__ __forceinline__ void store4(float *p, const float *v)
{
    if (VEC) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = v[i];
    }
}

// 8 consecutive bf16 parameters, one row of a core matrix
template <bool VEC>
__device__ __forceinline__ uint4 load_w8(const uint16_t *p)
{
    if (VEC) return *reinterpret_cast<const uint4 *>(p);
    uint32_t u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = (uint32_t)p[2 * i] | ((uint32_t)p[2 * i + 1] << 16);
    return make_uint4(u[0], u[1], u[2], u[3]);
}

// ReLU(acc + bias) of the 32 accumulator columns from `col` of this thread's
// lane, the columns j0 .. j0 + 31 of the hidden layer: saved in fp32 (act)
// and written to row `row` of the next A operand
template <bool VEC>
__device__ __forceinline__ void hidden_row(uint32_t tbase, int col, const float *bias, uint8_t *A, int row, int j0,
                                           float *act_row)
{
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        float v[16];
        tmem_ld16(tbase + (uint32_t)(col + j0 + 16 * q), v);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i] + bias[j0 + 16 * q + i], 0.f);
#pragma unroll
        for (int i = 0; i < 16; i += 8)
            *reinterpret_cast<uint4 *>(A + core_off(row, j0 + 16 * q + i, kMlpH)) =
                make_uint4(two_bf16(v[i], v[i + 1]), two_bf16(v[i + 2], v[i + 3]), two_bf16(v[i + 4], v[i + 5]),
                           two_bf16(v[i + 6], v[i + 7]));
        if (act_row) {
#pragma unroll
            for (int i = 0; i < 16; i += 4) store4<VEC>(act_row + j0 + 16 * q + i, v + i);
        }
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kTcThreads) mlp_forward_tc_kernel(const uint16_t *wb, const float *norm, const float *x,
                                                              int B, float *logits, float *act, int32_t *pick,
                                                              float min_prob, int fallback, int32_t *err)
{
    start_early();
    __shared__ __align__(1024) uint8_t sm[kTcSmem];
    __shared__ __align__(8) uint64_t mbar_store;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float bias[2 * kMlpH + kMlpOut];
    const int t = threadIdx.x, warp = t >> 5, row = t & (kTcM - 1), j0 = (t / kTcM) * (kMlpH / 2);
    const int b = blockIdx.x * kTcM + row;
    const bool live = b < B;
    uint8_t *A = sm + kOffA;
    const uint32_t mbar = smem_u32(&mbar_store);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // B operands (the parameters, zero-padded), the biases, and the layer-1 A
    // operand (the normalised input, zero-padded)
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = t; i < kMlpH * kK1 / 8; i += kTcThreads) {
        const int n = i / (kK1 / 8), k = 8 * (i % (kK1 / 8));
        *reinterpret_cast<uint4 *>(sm + kOffB1 + core_off(n, k, kK1)) =
            k < kMlpIn ? load_w8<VEC>(wb + kW1 + n * kMlpIn + k) : zero;
    }
#pragma unroll
    for (int i = t; i < kMlpH * kMlpH / 8; i += kTcThreads) {
        const int n = i / (kMlpH / 8), k = 8 * (i % (kMlpH / 8));
        *reinterpret_cast<uint4 *>(sm + kOffB2 + core_off(n, k, kMlpH)) = load_w8<VEC>(wb + kW2 + n * kMlpH + k);
    }
    if (t < kN3 * kMlpH / 8) {
        const int n = t / (kMlpH / 8), k = 8 * (t % (kMlpH / 8));
        *reinterpret_cast<uint4 *>(sm + kOffB3 + core_off(n, k, kMlpH)) =
            n < kMlpOut ? load_w8<VEC>(wb + kW3 + n * kMlpH + k) : zero;
    }
    if (t < 2 * kMlpH + kMlpOut)
        bias[t] = of_bf16(wb[t < kMlpH ? kB1 + t : t < 2 * kMlpH ? kB2 + t - kMlpH : kB3 + t - 2 * kMlpH]);
#pragma unroll
    for (int u = 0; u < kTcM * kMlpIn / 4 / kTcThreads; ++u) {
        const int i = t + kTcThreads * u, r = i / (kMlpIn / 4), k = 4 * (i % (kMlpIn / 4));
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (blockIdx.x * kTcM + r < B) {
            load4<VEC>(x + (int64_t)blockIdx.x * kTcM * kMlpIn + 4 * i, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = (v[e] - norm[k + e]) / norm[kMlpIn + k + e];
        }
        *reinterpret_cast<uint2 *>(A + core_off(r, k, kK1)) = make_uint2(two_bf16(v[0], v[1]), two_bf16(v[2], v[3]));
    }
    if (t < kTcM) *reinterpret_cast<uint4 *>(A + core_off(t, kMlpIn, kK1)) = zero;
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tmem = tmem_base;
    const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16);   // this warp's 32 lanes
    const uint32_t aaddr = smem_u32(A);
    bool ok = true;

    // layer 1: H1 = Xn W1^T, two K = 16 steps
    if (t == 0) {
        for (int s = 0; s < kK1 / 16; ++s)
            mma_bf16(tmem, smem_desc(aaddr + 256 * s, kK1), smem_desc(smem_u32(sm + kOffB1) + 256 * s, kK1),
                     instr_desc(kTcM, kMlpH), s > 0);
        mma_commit(mbar);
    }
    ok = mbar_wait(mbar, 0) && ok;
    tc_after_sync();
    hidden_row<VEC>(tlane, 0, bias, A, row, j0, live && act ? act + (int64_t)b * kMlpAct : nullptr);
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();

    // layer 2: H2 = relu(H1 + b1) W2^T, four K = 16 steps
    if (t == 0 && ok) {
        for (int s = 0; s < kMlpH / 16; ++s)
            mma_bf16(tmem + kMlpH, smem_desc(aaddr + 256 * s, kMlpH), smem_desc(smem_u32(sm + kOffB2) + 256 * s, kMlpH),
                     instr_desc(kTcM, kMlpH), s > 0);
        mma_commit(mbar);
    }
    ok = ok && mbar_wait(mbar, 1);
    tc_after_sync();
    hidden_row<VEC>(tlane, kMlpH, bias + kMlpH, A, row, j0, live && act ? act + (int64_t)b * kMlpAct + kMlpH : nullptr);
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();

    // layer 3: Z = relu(H2 + b2) W3^T, N padded to 16
    if (t == 0 && ok) {
        for (int s = 0; s < kMlpH / 16; ++s)
            mma_bf16(tmem + 2 * kMlpH, smem_desc(aaddr + 256 * s, kMlpH),
                     smem_desc(smem_u32(sm + kOffB3) + 256 * s, kMlpH), instr_desc(kTcM, kN3), s > 0);
        mma_commit(mbar);
    }
    ok = ok && mbar_wait(mbar, 0);
    tc_after_sync();
    float zv[16];
    tmem_ld16(tlane + 2 * kMlpH, zv);
    tc_before_sync();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    if (!ok) {
        if (t == 0) raise_status(err, RT_ETIMEOUT);
        return;
    }
    if (!live || j0) return;
    float z[kMlpOut];
    int best = 0;
#pragma unroll
    for (int k = 0; k < kMlpOut; ++k) {
        z[k] = zv[k] + bias[2 * kMlpH + k];
        if (logits) logits[(int64_t)b * kMlpOut + k] = z[k];
        if (z[k] > z[best]) best = k;
    }
    if (min_prob > 0.f) {
        float se = 0.f;
#pragma unroll
        for (int k = 0; k < kMlpOut; ++k) se += expf(z[k] - z[best]);
        if (1.f / se < min_prob) best = fallback;
    }
    if (pick) pick[b] = best;
}

// Backward on the tensor cores, 128 samples per CTA (threads t and t + 128:
// sample t).
//   dz  = (softmax(z) - onehot(label)) / B               (fp32, per thread)
//   dh2 = (dz W3) * [h2 > 0]                              (fp32, per thread: K = 3)
//   dh1 = (dh2 W2) * [h1 > 0]                             (product 1: 128 x 64, K = 64)
//   [dW2 db2; dW1 db1] from [dh2 | dh1]^T [h1 | xn | 1]   (product 2: M = 128
//                                                          features, N = 96, K = 128 samples)
// Product 2 stacks both weight gradients in one M = 128 accumulator: rows
// 0..63 are dh2's features against h1 (dW2) and a column of ones (db2), rows
// 64..127 dh1's features against xn (dW1) and the ones (db1); the two mixed
// blocks are not read. Each CTA writes its partial sums of W1, b1, W2, b2
// and its samples' dz and loss; a second kernel adds the partials of the
// CTAs in a fixed order and forms W3 and b3 from dz and h2 (fp32), so the
// result is deterministic.
constexpr int kBwN2 = 96;                           // product 2 N: h1 (64) | xn (24) | ones | pad
constexpr int kBwOne = kMlpH + kMlpIn;              // the ones column (88)
constexpr int kBwA1 = 0;                            // 128 x 64: dh2 (product 1 A)
constexpr int kBwB1 = kBwA1 + kTcM * kMlpH * 2;     // 64 x 64: W2^T
constexpr int kBwA2 = kBwB1 + kMlpH * kMlpH * 2;    // 128 x 128: [dh2 | dh1]^T
constexpr int kBwB2 = kBwA2 + kTcM * kTcM * 2;      // 96 x 128: [h1 | xn | 1]^T
constexpr int kBwSmem = kBwB2 + kBwN2 * kTcM * 2;   // 73728 bytes (dynamic)
constexpr int kBwPart = kW3;                        // partial sums per CTA: W1 b1 W2 b2
constexpr int kBwEarly = 4;                         // CTAs up to which the second kernel is placed early

// Column t (even and odd lanes side by side) of a K = 128 operand, rows
// n .. n + 15: lanes exchange one value of each pair of rows, so every store
// is two samples of one row.
__device__ __forceinline__ void store_column16(uint8_t *op, int n, int t, const float *v)
{
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const uint32_t mine = two_bf16(v[i], v[i + 1]), other = __shfl_xor_sync(0xffffffffu, mine, 1);
        const uint32_t both = (t & 1) ? __byte_perm(other, mine, 0x7632) : __byte_perm(mine, other, 0x5410);
        *reinterpret_cast<uint32_t *>(op + core_off(n + i + (t & 1), t & ~1, kTcM)) = both;
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kTcThreads) mlp_backward_tc_kernel(const uint16_t *wb, const float *norm,
                                                                     const float *x, const float *act,
                                                                     const float *logits, const int32_t *label, int B,
                                                                     float *part, float *dz_out, float *loss_out,
                                                                     int32_t *err)
{
    start_early();
    extern __shared__ __align__(1024) uint8_t smb[];
    __shared__ __align__(8) uint64_t mbar_store;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float w3[kMlpOut * kMlpH];
    constexpr int kHalf = kMlpH / 2;
    const int t = threadIdx.x, warp = t >> 5, row = t & (kTcM - 1), half = t / kTcM, j0 = half * kHalf;
    const int b = blockIdx.x * kTcM + row;
    const bool live = b < B;
    const uint32_t mbar = smem_u32(&mbar_store);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // W2^T as product 1's B: B[n][k] = W2[k][n], 8 columns of rows k and k + 1 per thread
    {
        static_assert(kMlpH / 2 * (kMlpH / 8) == kTcThreads, "one pair of 16-byte pieces per thread");
        const int k = 2 * (t / (kMlpH / 8)), n = 8 * (t % (kMlpH / 8));
        const uint4 p = load_w8<VEC>(wb + kW2 + k * kMlpH + n), q = load_w8<VEC>(wb + kW2 + (k + 1) * kMlpH + n);
        const uint32_t a[4] = {p.x, p.y, p.z, p.w}, c[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 8; ++e)
            *reinterpret_cast<uint32_t *>(smb + kBwB1 + core_off(n + e, k, kMlpH)) =
                __byte_perm(a[e / 2], c[e / 2], (e & 1) ? 0x7632 : 0x5410);
    }
    if (t < kMlpOut * kMlpH) w3[t] = of_bf16(wb[kW3 + t]);
    // this sample's deltas of the output (both of its threads) and of half the second hidden layer (fp32)
    float h2[kHalf], h1[kHalf], xn[16], dz[kMlpOut];
#pragma unroll
    for (int k = 0; k < kMlpOut; ++k) dz[k] = 0.f;
#pragma unroll
    for (int j = 0; j < kHalf; ++j) h1[j] = h2[j] = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) xn[k] = 0.f;
    if (live) {
        const float *ar = act + (int64_t)b * kMlpAct + j0;
#pragma unroll
        for (int j = 0; j < kHalf; j += 4) load4<VEC>(ar + kMlpH + j, h2 + j);
#pragma unroll
        for (int j = 0; j < kHalf; j += 4) load4<VEC>(ar + j, h1 + j);
        // the input columns 0 .. 15, or 16 .. 23 and the one
#pragma unroll
        for (int k = 0; k < 16; k += 4)
            if (half == 0 || k < kMlpIn - 16) load4<VEC>(x + (int64_t)b * kMlpIn + 16 * half + k, xn + k);
        const float *z = logits + (int64_t)b * kMlpOut;
        float m = z[0];
#pragma unroll
        for (int k = 1; k < kMlpOut; ++k) m = fmaxf(m, z[k]);
        float se = 0.f;
#pragma unroll
        for (int k = 0; k < kMlpOut; ++k) se += expf(z[k] - m);
        const int y = label[b];
#pragma unroll
        for (int k = 0; k < kMlpOut; ++k) {
            dz[k] = (expf(z[k] - m) / se - (k == y ? 1.f : 0.f)) / (float)B;
            if (half == 0) dz_out[(int64_t)b * kMlpOut + k] = dz[k];
        }
        if (half == 0) loss_out[b] = logf(se) + m - z[y];
    }
    __syncthreads();   // w3
#pragma unroll
    for (int j = 0; j < kHalf; ++j) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < kMlpOut; ++k) s = fmaf(w3[k * kMlpH + j0 + j], dz[k], s);
        h2[j] = h2[j] > 0.f ? s : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kHalf; j += 8)   // row of product 1's A
        *reinterpret_cast<uint4 *>(smb + kBwA1 + core_off(row, j0 + j, kMlpH)) =
            make_uint4(two_bf16(h2[j], h2[j + 1]), two_bf16(h2[j + 2], h2[j + 3]), two_bf16(h2[j + 4], h2[j + 5]),
                       two_bf16(h2[j + 6], h2[j + 7]));
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tmem = tmem_base;
    const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    bool ok = true;
    if (t == 0) {
        for (int s = 0; s < kMlpH / 16; ++s)
            mma_bf16(tmem, smem_desc(smem_u32(smb + kBwA1) + 256 * s, kMlpH),
                     smem_desc(smem_u32(smb + kBwB1) + 256 * s, kMlpH), instr_desc(kTcM, kMlpH), s > 0);
        mma_commit(mbar);
    }
    // meanwhile: column `row` of product 2's A (dh2) and B (h1, xn, a one and the padding), as bf16
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        store_column16(smb + kBwA2, j0 + 16 * q, row, h2 + 16 * q);
        store_column16(smb + kBwB2, j0 + 16 * q, row, h1 + 16 * q);
    }
    if (live) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int c = 16 * half + k;
            if (c < kMlpIn) xn[k] = (xn[k] - norm[c]) / norm[kMlpIn + c];
            if (c == kMlpIn) xn[k] = 1.f;
        }
    }
    store_column16(smb + kBwB2, kMlpH + 16 * half, row, xn);
    ok = mbar_wait(mbar, 0) && ok;
    tc_after_sync();
    // dh1 = (dh2 W2) * [h1 > 0]: column `row` of product 2's A, rows 64..127
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        float v[16];
        tmem_ld16(tlane + (uint32_t)(j0 + 16 * q), v);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = h1[16 * q + i] > 0.f ? v[i] : 0.f;   // 0 if not live
        store_column16(smb + kBwA2, kMlpH + j0 + 16 * q, row, v);
    }
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    if (t == 0 && ok) {
        for (int s = 0; s < kTcM / 16; ++s)
            mma_bf16(tmem + kMlpH, smem_desc(smem_u32(smb + kBwA2) + 256 * s, kTcM),
                     smem_desc(smem_u32(smb + kBwB2) + 256 * s, kTcM), instr_desc(kTcM, kBwN2), s > 0);
        mma_commit(mbar);
    }
    ok = ok && mbar_wait(mbar, 1);
    tc_after_sync();
    // row `row` of product 2: feature `row` of dh2 (< 64) or of dh1; the workspace is aligned
    float *pc = part + (int64_t)blockIdx.x * kBwPart;
    if ((warp & 3) < 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float v[16];
            tmem_ld16(tlane + kMlpH + (uint32_t)(j0 + 16 * q), v);
#pragma unroll
            for (int i = 0; i < 16; i += 4) store4<true>(pc + kW2 + row * kMlpH + j0 + 16 * q + i, v + i);
        }
        if (half) {
            float v[16];
            tmem_ld16(tlane + kMlpH + 80, v);
            pc[kB2 + row] = v[kBwOne - 80];
        }
    } else {
        const int i1 = row - kMlpH;
        float v[16];
        tmem_ld16(tlane + kMlpH + 64 + 16 * (uint32_t)half, v);
#pragma unroll
        for (int i = 0; i < 16; i += 4)
            if (half == 0 || i < kMlpIn - 16) store4<true>(pc + kW1 + i1 * kMlpIn + 16 * half + i, v + i);
        if (half) pc[kB1 + i1] = v[kBwOne - 80];
    }
    tc_before_sync();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    if (!ok && t == 0) raise_status(err, RT_ETIMEOUT);
}

// the gradient, one warp per parameter: W1, b1, W2, b2 as the sum of the
// CTAs' partials, W3 and b3 over the samples from dz and h2 (fp32); the last
// warp sums the loss. Lane l adds the terms l, l + 32, ... in order, then a
// fixed butterfly adds the lanes, so the result does not depend on
// scheduling.
__global__ void mlp_grad_tc_kernel(const float *part, int nblk, const float *dz, const float *act, const float *lossb,
                                   int B, float *grad, float *loss)
{
    start_early();
    const int p = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (p > kMlpParams) return;
    float s = 0.f;
    if (p == kMlpParams) {
        for (int b = lane; b < B; b += 32) s += lossb[b];
    } else if (p < kW3) {
        for (int k = lane; k < nblk; k += 32) s += part[(int64_t)k * kBwPart + p];
    } else if (p < kB3) {
        const int k = (p - kW3) / kMlpH, j = (p - kW3) % kMlpH;
        for (int b = lane; b < B; b += 32)
            s = fmaf(dz[(int64_t)b * kMlpOut + k], act[(int64_t)b * kMlpAct + kMlpH + j], s);
    } else {
        for (int b = lane; b < B; b += 32) s += dz[(int64_t)b * kMlpOut + (p - kB3)];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane != 0) return;
    if (p == kMlpParams) {
        if (loss) *loss = s / (float)B;
    } else {
        grad[p] = s;
    }
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

size_t mlp_backward_tc_workspace_bytes(int B)
{
    const int64_t nblk = ceil_div(B, kTcM);
    return sizeof(float) * (size_t)(nblk * kBwPart + (int64_t)B * (kMlpOut + 1));
}

cudaError_t launch_mlp_backward_tc(const uint16_t *wb, const float *norm, const float *x, const float *act,
                                   const float *logits, const int32_t *label, int B, float *grad, float *loss,
                                   float *ws, int32_t *err, cudaStream_t s)
{
    if (B <= 0) return cudaErrorInvalidValue;
    const int nblk = (int)ceil_div(B, kTcM);
    float *part = ws;
    float *dz = part + (int64_t)nblk * kBwPart;
    float *lossb = dz + (int64_t)B * kMlpOut;
    const auto kernel = aligned16(wb) && aligned16(x) && aligned16(act) ? mlp_backward_tc_kernel<true>
                                                                        : mlp_backward_tc_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwSmem);
    if (e != cudaSuccess) return e;
    launch_early(kernel, nblk, kTcThreads, kBwSmem, s, wb, norm, x, act, logits, label, B, part, dz, lossb, err);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // The sums live on their sectors staying in L1 (eight parameters share
    // one). Blocks placed early sit beside the products' 72 KB of shared
    // memory, which L1 is cut by, so they are only placed early for a batch
    // of few CTAs: whole backward with and without, 16.1 and 16.6 us for 512
    // samples, 19.7 and 18.7 for 1024, 40 and 33 for 4096, 253 and 107 for
    // 20000.
    const unsigned grid = (unsigned)ceil_div((int64_t)(kMlpParams + 1) * 32, 256);
    if (nblk <= kBwEarly) launch_early(mlp_grad_tc_kernel, grid, 256, 0, s, part, nblk, dz, act, lossb, B, grad, loss);
    else mlp_grad_tc_kernel<<<grid, 256, 0, s>>>(part, nblk, dz, act, lossb, B, grad, loss);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward_tc(const uint16_t *wb, const float *norm, const float *x, int B, float *logits,
                                  float *act, int32_t *pick, float min_prob, int fallback, int32_t *err,
                                  cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    const auto kernel = aligned16(wb) && aligned16(x) && aligned16(act) ? mlp_forward_tc_kernel<true>
                                                                        : mlp_forward_tc_kernel<false>;
    launch_early(kernel, (unsigned)ceil_div(B, kTcM), kTcThreads, 0, s, wb, norm, x, B, logits, act, pick, min_prob, fallback, err);
    return cudaGetLastError();
}

}  // namespace rtk
