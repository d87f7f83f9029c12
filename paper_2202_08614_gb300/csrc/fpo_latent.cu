// Latent decoder on the 5th-generation tensor cores (tcgen05, TMEM).
//
// Each leaf stores a 32-dim FP16 latent; a shared MLP 32 -> 64 -> 64 -> 166
// (ReLU) decodes the leaf's n1 + 27 n2 Fourier coefficients.  Eq. 7 and 9 are
// linear in the coefficients, so the frame's IDFT is folded into the last
// layer: W3'(t) = B(t) W3, b3'(t) = B(t) b3 with B(t) the 28 x 166 map to
// (sigma_raw, z_{c,k}), and the kernel writes the same per-frame table as the
// coefficient IDFT pass: [max(0, sigma), 27 z, 0 x 4] per leaf.
//
// Per CTA the weights are staged once in shared memory in the no-swizzle
// K-major core-matrix layout (8 rows x 16 B blocks) and W3'(t) is computed
// in the prologue.  Eight warpgroups (1024 threads, all 512 TMEM columns)
// then run independent tile pipelines
// (own A buffers, own 64 TMEM columns, own mbarrier and named barrier): for
// each tile of 128 leaves the threads lay the latents out as the A operand,
// one elected thread issues tcgen05.mma (M = 128, K = 16 per instruction,
// FP16 x FP16 -> FP32 in TMEM) and commits to the mbarrier, and the warps
// read the accumulator rows back with tcgen05.ld (one row per thread, a
// warp's TMEM lane quarter), apply ReLU while rounding to FP16 and write the
// next layer's A operand.  The 64 columns hold every layer's accumulator in
// turn.  The output tile goes out by one TMA tensor store per tile.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <cstdint>

#include "fpo_internal.h"
#include "fpo_ptx.cuh"

namespace fpo {
namespace {

// Independent warpgroup pipelines per CTA (one CTA per SM): 8 (1024 threads,
// all 512 TMEM columns) when the decoder has the SM to itself, 2 (256
// threads, 128 columns) beside the traversal in the frame pipeline.
constexpr int LT_GROUPS_FULL = 8, LT_GROUPS_PIPE = 2;
constexpr int LT_M = 128;          // leaves per tile = MMA M
// 64 accumulator columns per warpgroup
template <int G>
__host__ __device__ constexpr uint32_t lt_tmem_cols() { return 64u * G; }
static_assert(lt_tmem_cols<LT_GROUPS_FULL>() <= 512 && lt_tmem_cols<LT_GROUPS_PIPE>() >= 32, "TMEM allocation");
constexpr uint64_t LT_WAIT_NS = 2000000000ull;

// Biases ride in the MMAs: every A operand carries two constant-one columns
// after its data and every B operand the bias split into two FP16 halves
// (hi = fp16(b), lo = fp16(b - hi), so hi + lo carries b to about 22 bits)
// in the same two columns; the accumulator then already holds W x + b.  K
// is padded to a multiple of 16 with zeros: 32 + 16 for layer 1, 64 + 16 for
// layers 2 and 3.
constexpr int K1 = 48, K2 = 80;

// Shared-memory layout (bytes), all operands no-swizzle K-major.
constexpr int OFF_W1 = 0;          // 64 x 48  f16:  6 KB
constexpr int OFF_W2 = 6144;       // 64 x 80  f16: 10 KB
constexpr int OFF_W3 = 16384;      // 32 x 80  f16:  5 KB
// A1 (layer-1 input) and A2 share one region per group: MMA 1 has finished
// reading A1 before the layer-1 epilogue writes A2, and the next tile's A1 is
// written only after the tensor store has read the previous output from A2.
constexpr int OFF_A1 = 22528;      // per group: 128 x 48 f16: 12 KB
constexpr int OFF_A2 = 22528;      // per group: 128 x 80 f16: 20 KB (1024-byte aligned: output staging)
constexpr int GROUP_BYTES = 20480; // one warpgroup's region
template <int G>
__host__ __device__ constexpr int lt_smem() { return OFF_A1 + G * GROUP_BYTES + 1024; }  // + alignment slack

// Byte offset of element (row, k) in a K-major core-matrix layout whose rows
// hold K elements: core matrix (row / 8, k / 8) at ((row/8) * K/8 + k/8) * 128,
// inside it row % 8 at 16 B per row.
__device__ __forceinline__ uint32_t core_off(int row, int k, int K)
{
    return (uint32_t)((((row >> 3) * (K >> 3) + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// kind::f16 instruction descriptor: A, B f16, D f32, both K-major, M x N.
__device__ __forceinline__ uint32_t idesc_f16(int M, int N)
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     ptx::smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 32 consecutive FP32 columns of this thread's TMEM lane; waits for them.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Tensor store of a 128-row tile of the table (box 32 floats x 128 rows,
// 128-byte swizzle) from shared memory, committed as its own bulk group.
__device__ __forceinline__ void tensor_store_rows(const CUtensorMap *map, const void *src, uint32_t row0)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];\n\t"
                 "cp.async.bulk.commit_group;" ::"l"(reinterpret_cast<uint64_t>(map)),
                 "r"(0), "r"(row0), "r"(ptx::smem_u32(src))
                 : "memory");
}
// Waits until every committed bulk store has finished reading shared memory.
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Waits until every committed bulk store has completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Rounds 8 consecutive values to FP16 with ReLU (max(x, 0) after rounding
// equals rounding after max) and writes them as K-chunk j of row `row` of a
// core layout.  `hmax` keeps the packed running maximum of what was written:
// a value beyond the FP16 range rounds to +inf, which the maximum keeps.
__device__ __forceinline__ void put8_relu(unsigned char *base, int row, int j, int K, const float *v, __half2 &hmax)
{
    uint32_t h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {  // the first operand goes to the upper half
        asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(h[e]) : "f"(v[2 * e + 1]), "f"(v[2 * e]));
        hmax = __hmax2(hmax, *reinterpret_cast<const __half2 *>(&h[e]));
    }
    *reinterpret_cast<uint4 *>(base + core_off(row, 8 * j, K)) = make_uint4(h[0], h[1], h[2], h[3]);
}

constexpr float F16_MAX = 65504.0f;  // the largest finite FP16 value

// Writes 8 consecutive values of row `row` (K-chunk j) into a core layout.
__device__ __forceinline__ void put8(unsigned char *base, int row, int j, int K, const float *v)
{
    __half2 h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = __floats2half2_rn(v[2 * e], v[2 * e + 1]);
    *reinterpret_cast<uint4 *>(base + core_off(row, 8 * j, K)) = *reinterpret_cast<const uint4 *>(h);
}

// K-chunk j of row `row` = {hi(b), lo(b), 0 x 6}: the bias columns of a B
// operand; with `ones`, {1, 1, 0 x 6}: the constant columns of an A operand.
__device__ __forceinline__ void put_bias_chunk(unsigned char *base, int row, int j, int K, float b, bool ones)
{
    const __half hi = ones ? __float2half_rn(1.0f) : __float2half_rn(b);
    const __half lo = ones ? __float2half_rn(1.0f) : __float2half_rn(b - __half2float(hi));
    const __half2 h0 = __halves2half2(hi, lo), z = __float2half2_rn(0.0f);
    uint4 u;
    u.x = *reinterpret_cast<const uint32_t *>(&h0);
    u.y = u.z = u.w = *reinterpret_cast<const uint32_t *>(&z);
    *reinterpret_cast<uint4 *>(base + core_off(row, 8 * j, K)) = u;
}

__device__ __forceinline__ void put_zero_chunk(unsigned char *base, int row, int j, int K)
{
    *reinterpret_cast<uint4 *>(base + core_off(row, 8 * j, K)) = make_uint4(0, 0, 0, 0);
}

// Issues the K / 16 MMAs of D[128 x N] = A[128 x K] B[N x K]^T.
__device__ __forceinline__ void gemm(uint32_t d_tmem, uint32_t a_saddr, uint32_t b_saddr, int K, int N)
{
    const uint32_t idesc = idesc_f16(LT_M, N);
    const uint32_t sbo = (uint32_t)(K / 8) * 128u;
#pragma unroll 1
    for (int s = 0; s < K / 16; ++s) {
        const uint64_t a = smem_desc(a_saddr + 256u * s, 128u, sbo);
        const uint64_t b = smem_desc(b_saddr + 256u * s, 128u, sbo);
        mma_f16(d_tmem, a, b, idesc, s > 0 ? 1u : 0u);
    }
}

}  // namespace

__device__ __forceinline__ void group_sync(int group)
{
    asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory");
}

template <int G>
__global__ void __launch_bounds__(128 * G, 8 / G) latent_table_kernel(const __grid_constant__ LatentParams p)
{
    constexpr int LT_GROUPS = G, LT_THREADS = 128 * G;
    constexpr uint32_t LT_TMEM_COLS = lt_tmem_cols<G>();
    extern __shared__ __align__(1024) unsigned char lt_smem_raw[];
    // the 128-byte-swizzled output staging needs 1024-byte aligned buffers
    unsigned char *lt_smem = lt_smem_raw + ((1024u - (ptx::smem_u32(lt_smem_raw) & 1023u)) & 1023u);
    __shared__ float s_basis[32];
    __shared__ uint64_t s_bar[LT_GROUPS];
    __shared__ uint64_t s_never;  // FPO_FLAG_TEST_DEVICE_TIMEOUT: a barrier nothing signals
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail[LT_GROUPS];
    __shared__ int s_range;  // a weight or bias beyond the FP16 range
    const int tid = threadIdx.x, warp = tid >> 5;
    const int group = tid >> 7, gt = tid & 127;  // warpgroup and thread within it

    // --- prologue: basis, weights (bf16 -> f16, core layout), folded layer 3
    if (tid < 32) s_basis[tid] = p.b[tid];
    if (tid == 0) s_range = 0;
    if (tid < LT_GROUPS) {
        s_fail[tid] = 0;
        ptx::mbar_init(&s_bar[tid], 1);
        if (tid == 0) ptx::mbar_init(&s_never, 1);
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(&s_tmem)),
                     "r"(LT_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // 8 consecutive BF16 weights as FP32, in one 16-byte load where the arrays allow it
    const bool a16 = ((reinterpret_cast<uintptr_t>(p.w1) | reinterpret_cast<uintptr_t>(p.w2) | reinterpret_cast<uintptr_t>(p.w3)) & 15u) == 0;
    auto load8 = [&](const uint16_t *src, float v[8]) {
        uint32_t u[4];
        if (a16) {
            const uint4 w = __ldg(reinterpret_cast<const uint4 *>(src));
            u[0] = w.x, u[1] = w.y, u[2] = w.z, u[3] = w.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) u[e] = (uint32_t)__ldg(src + 2 * e) | ((uint32_t)__ldg(src + 2 * e + 1) << 16);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[2 * e] = __uint_as_float(u[e] << 16);
            v[2 * e + 1] = __uint_as_float(u[e] & 0xffff0000u);
        }
    };
    auto in_range = [&](const float v[8]) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (!(fabsf(v[e]) <= F16_MAX)) s_range = 1;
    };
#pragma unroll 2
    for (int q = tid; q < 64 * (K1 / 8); q += LT_THREADS) {  // W1 | b1: 64 rows x 6 chunks
        const int n = q / (K1 / 8), j = q % (K1 / 8);
        if (j < 4) {
            float v[8];
            load8(p.w1 + n * 32 + 8 * j, v);
            in_range(v);
            put8(lt_smem + OFF_W1, n, j, K1, v);
        } else if (j == 4) {
            if (!(fabsf(p.b1[n]) <= F16_MAX)) s_range = 1;
            put_bias_chunk(lt_smem + OFF_W1, n, j, K1, p.b1[n], false);
        } else {
            put_zero_chunk(lt_smem + OFF_W1, n, j, K1);
        }
    }
#pragma unroll 3
    for (int q = tid; q < 64 * (K2 / 8); q += LT_THREADS) {  // W2 | b2: 64 rows x 10 chunks
        const int n = q / (K2 / 8), j = q % (K2 / 8);
        if (j < 8) {
            float v[8];
            load8(p.w2 + n * 64 + 8 * j, v);
            in_range(v);
            put8(lt_smem + OFF_W2, n, j, K2, v);
        } else if (j == 8) {
            if (!(fabsf(p.b2[n]) <= F16_MAX)) s_range = 1;
            put_bias_chunk(lt_smem + OFF_W2, n, j, K2, p.b2[n], false);
        } else {
            put_zero_chunk(lt_smem + OFF_W2, n, j, K2);
        }
    }
    __syncthreads();  // s_basis ready
    // W3'(t): row 0 = sum_i b_i W3[i], row 1 + q = sum_i b_i W3[n1 + q n2 + i],
    // rows 28..31 = 0.  Eight output elements per thread: 16-byte loads,
    // independent of each other, so the fold costs a few memory latencies
    // (element by element it took most of the prologue).
    for (int q = tid; q < 32 * 8; q += LT_THREADS) {
        const int r = q >> 3, c = q & 7;
        const int row0 = r == 0 ? 0 : p.n1 + (r - 1) * p.n2, terms = r == 0 ? p.n1 : (r <= 27 ? p.n2 : 0);
        float acc[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 5
        for (int i = 0; i < terms; ++i) {
            float v[8];
            load8(p.w3 + (row0 + i) * 64 + 8 * c, v);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = fmaf(s_basis[i], v[e], acc[e]);
        }
        in_range(acc);
        put8(lt_smem + OFF_W3, r, c, K2, acc);
    }
    if (tid < 32) {
        const int row0 = tid == 0 ? 0 : p.n1 + (tid - 1) * p.n2, terms = tid == 0 ? p.n1 : (tid <= 27 ? p.n2 : 0);
        float acc = 0.0f;
#pragma unroll 8
        for (int i = 0; i < terms; ++i) acc = fmaf(s_basis[i], p.b3[row0 + i], acc);
        if (!(fabsf(acc) <= F16_MAX)) s_range = 1;
        put_bias_chunk(lt_smem + OFF_W3, tid, 8, K2, acc, false);  // rows 28..31: b = 0
        put_zero_chunk(lt_smem + OFF_W3, tid, 9, K2);
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    // this warpgroup's accumulator columns; this warp's lane quarter
    const uint32_t tmem = s_tmem + 64u * (uint32_t)group;
    const uint32_t my_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    unsigned char *ga1 = lt_smem + OFF_A1 + group * GROUP_BYTES;
    unsigned char *ga2 = lt_smem + OFF_A2 + group * GROUP_BYTES;
    const uint32_t sa_w1 = ptx::smem_u32(lt_smem + OFF_W1), sa_w2 = ptx::smem_u32(lt_smem + OFF_W2),
                   sa_w3 = ptx::smem_u32(lt_smem + OFF_W3), sa_a1 = ptx::smem_u32(ga1), sa_a2 = ptx::smem_u32(ga2);
    uint32_t phase = 0;
    __half2 hmax = __float2half2_rn(0.0f);  // packed maximum of the FP16 activations written
    const uint32_t n_tiles = (p.n_leaves + LT_M - 1) / LT_M;
    const uint32_t first = blockIdx.x * LT_GROUPS + group, step = gridDim.x * LT_GROUPS;
    const int m = gt;  // this thread's accumulator row (TMEM lane) and leaf in the tile


    // One layer: the group's elected thread issues the MMAs and commits;
    // the group waits on its mbarrier (bounded).  The outcome is made
    // group-uniform so that the collective TMEM loads never diverge.  On a
    // time-out `phase` stays at the pending commit, which the drain after
    // the loop waits for before TMEM is freed.  The failure-path test makes
    // the group's first wait (on a barrier nothing signals) run out.
    bool first_wait = p.test_timeout != 0;
    auto run_layer = [&](uint32_t a_addr, uint32_t b_addr, int K, int N) -> bool {
        if (gt == 0) {
            fence_after();
            gemm(tmem, a_addr, b_addr, K, N);
            mma_commit(&s_bar[group]);
        }
        const bool ok = first_wait ? ptx::mbar_wait_bounded(&s_never, 0, TEST_WAIT_LIMIT_NS)
                                   : ptx::mbar_wait_bounded(&s_bar[group], phase, LT_WAIT_NS);
        first_wait = false;
        if (!ok) s_fail[group] = 1;
        group_sync(group);
        fence_after();
        if (s_fail[group]) return false;
        phase ^= 1u;
        return true;
    };
    auto hand_off = [&]() {  // generic smem writes and TMEM reads before the next MMA
        fence_async_smem();
        fence_before();
        group_sync(group);
    };
    // The tile's latents (128 rows x 64 B, contiguous) in coalesced 16-byte
    // pieces: thread gt takes pieces gt + 128 i, i.e. row (gt + 128 i) / 4,
    // K-chunk (gt + 128 i) % 4; rows past the end read as zeros.
    auto load_tile = [&](uint32_t tile, uint4 q[4]) {
        const uint4 *src = reinterpret_cast<const uint4 *>(p.latents) + (size_t)tile * LT_M * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int piece = gt + 128 * i;
            q[i] = make_uint4(0, 0, 0, 0);
            if (tile < n_tiles && tile * LT_M + (uint32_t)(piece >> 2) < p.n_leaves) q[i] = __ldg(src + piece);
        }
    };
    uint4 nextq[4];
    load_tile(first, nextq);
    for (uint32_t tile = first; tile < n_tiles; tile += step) {
        if (gt == 0) bulk_wait_read();  // the previous tile's table store has left A2
        group_sync(group);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int piece = gt + 128 * i;
            *reinterpret_cast<uint4 *>(ga1 + core_off(piece >> 2, 8 * (piece & 3), K1)) = nextq[i];
        }
        // the constant-one columns of this thread's row (A2 writes reuse the region)
        put_bias_chunk(ga1, m, 4, K1, 0.0f, true);
        put_zero_chunk(ga1, m, 5, K1);
        hand_off();
        if (!run_layer(sa_a1, sa_w1, K1, 64)) break;
        // layer 1 epilogue: bias + ReLU -> layer-2 A operand (MMA 1 is done with A1)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[32];
            tmem_ld32(my_lane + 32 * h, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) put8_relu(ga2, m, 4 * h + c, K2, v + 8 * c, hmax);
        }
        put_bias_chunk(ga2, m, 8, K2, 0.0f, true);
        put_zero_chunk(ga2, m, 9, K2);
        hand_off();
        if (!run_layer(sa_a2, sa_w2, K2, 64)) break;
        // layer 2 epilogue -> layer-3 A operand, in place (MMA 2 has finished
        // reading A2, and each thread rewrites only its own row)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[32];
            tmem_ld32(my_lane + 32 * h, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) put8_relu(ga2, m, 4 * h + c, K2, v + 8 * c, hmax);
        }
        hand_off();
        load_tile(tile + step, nextq);  // in flight while layer 3 runs
        if (!run_layer(sa_a2, sa_w3, K2, 32)) break;
        {
            // output rows [max(0, sigma), 27 z, 0 x 4] into A2 (free since MMA 3
            // finished), then one bulk copy of the tile's contiguous rows
            float o[32];
            tmem_ld32(my_lane, o);
            // the accumulator holds W3'x + b3': sigma gets its clamp, columns
            // 28..31 are exactly zero
            float *w = o;
            w[0] = fmaxf(w[0], 0.0f);
            // 128-byte swizzle (chunk q of row m at chunk q ^ (m % 8)): the 8
            // lanes of a store phase hit 8 different bank groups, and the
            // tensor store un-swizzles on the way out
            if (p.half_table) {
                // FP16 rows of 64 B with the 64-byte swizzle (chunk q of row m
                // at chunk q ^ ((m / 2) % 4)): again no bank conflicts
                uint4 *row = reinterpret_cast<uint4 *>(ga2 + m * (TABLE_STRIDE * 2));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t h[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const __half2 hh = __floats2half2_rn(w[8 * q + 2 * e], w[8 * q + 2 * e + 1]);
                        h[e] = *reinterpret_cast<const uint32_t *>(&hh);
                    }
                    row[q ^ ((m >> 1) & 3)] = make_uint4(h[0], h[1], h[2], h[3]);
                }
            } else {
                float4 *row = reinterpret_cast<float4 *>(ga2 + m * (TABLE_STRIDE * 4));
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    row[q ^ (m & 7)] = make_float4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
            }
        }
        fence_async_smem();
        fence_before();
        group_sync(group);  // the rows are in A2; the accumulator is free for the next tile
        if (gt == 0) tensor_store_rows(&p.table_map, ga2, tile * LT_M);  // rows past the end are clipped
    }
    if (gt == 0) bulk_wait_all();  // every table store has completed
    // FP16 operands: a hidden activation, weight or bias beyond the FP16
    // range (it became +inf) makes the table wrong; report it
    if (p.status && (!(__low2float(hmax) <= F16_MAX) || !(__high2float(hmax) <= F16_MAX) || (tid == 0 && s_range)))
        atomicOr(p.status, STATUS_FP16_RANGE);
    if (s_fail[group] && gt == 0) {
        // the commit whose wait gave up: wait for it once more (bounded)
        // before TMEM is freed
        ptx::mbar_wait_bounded(&s_bar[group], phase, LT_WAIT_NS);
        if (p.status) atomicOr(p.status, STATUS_DEVICE_TIMEOUT);
    }
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(LT_TMEM_COLS) : "memory");
}

// ---------------------------------------------------------------------------
// Tensor-core training step of the decoder: the forward pass, the weighted L2
// loss against target coefficients (plus an optional extra dL/dy), and the
// back-propagation to every weight, bias and latent, with BF16 operands (A
// and B of each MMA both BF16; FP32's exponent range, so no loss scaling)
// and FP32 accumulation in TMEM.  One CTA per SM (all 512 TMEM columns): four
// warpgroups for the epilogues (thread t of each owns row t of a 128-leaf tile,
// TMEM lane t, and a quarter of each layer's columns) and one warp that
// issues the MMAs.  Per tile, nine GEMMs (M = 128):
//   Z1 = X W1^T,  Z2 = H1 W2^T,  Y = H2 W3^T                       (forward)
//   dH2 = dY W3,  dH1 = d2 W2,  dX = d1 W1                        (data)
//   G3 += [H2 1]^T dY,  G2 += [H1 1]^T d2,  G1 += [X 1]^T d1       (weights)
// H = relu(Z + b) in BF16 (the biases are added in FP32), d2 = dH2 [Z2 > 0],
// d1 = dH1 [Z1 > 0], dY = 2 cw (Y - target) + extra.  The weight gradients
// accumulate in TMEM over all of the CTA's tiles, transposed (lane = input
// feature, column = output feature); the ones column after each activation's
// features makes lane 64 (32 for layer 1) the bias gradient.
//
// Every matrix is in shared memory once, row-major in 8 x 16-byte core
// matrices: the GEMMs that sum over features read it K-major, those that sum
// over the tile's rows (the weight gradients) or over output features (the
// data gradients' weights) read the same core matrices MN-major through the
// descriptor's transpose bits.  (Writing transposed copies from the
// epilogues, 2 bytes at a time, took most of a tile's time, and left no
// room for what follows.)  The target rows, gathered by leaf, arrive by
// asynchronous copies, a row by contiguous 8-byte pieces, while the tile
// before is back-propagated.  The M = 128 A operands of the weight GEMMs hold
// 40 or 72 meaningful features; the rest of each descriptor's extent reads
// whatever lies after them in shared memory, which lands only in TMEM lanes
// that are never read.
// What bounds it: the chain of six dependent MMA rounds with their epilogues,
// about 1,500 cycles each (cycle counters; with two warpgroups, the MMAs
// issued by one of their threads and the weights staged 4 bytes at a time, the
// dY epilogue alone took 7,500 of a tile's 24,000 cycles and the prologue
// 15,000).  65,536 leaves: 177 us in the first form, 76 with two warpgroups,
// 49 now.
namespace {

constexpr int TG_EPI = 512, TG_THREADS = TG_EPI + 32, TG_NC = 176;  // epilogue threads; with the MMA warp
constexpr int TG_KX = 40, TG_KH = 72;              // features and the ones column, in 8-wide chunks
constexpr int TGO_W1 = 0;                          // [64][32]   W1
constexpr int TGO_W2 = TGO_W1 + 64 * 32 * 2;       // [64][64]   W2
constexpr int TGO_W3 = TGO_W2 + 64 * 64 * 2;       // [176][64]  W3
constexpr int TGO_X = TGO_W3 + TG_NC * 64 * 2;     // [128][40]  [X 1]
constexpr int TGO_H1 = TGO_X + 128 * TG_KX * 2;    // [128][72]  [H1 1]
constexpr int TGO_H2 = TGO_H1 + 128 * TG_KH * 2;   // [128][72]  [H2 1]
constexpr int TGO_DY = TGO_H2 + 128 * TG_KH * 2;   // [128][176] dY, then [128][64] d2, then d1
constexpr int TGO_T = TGO_DY + 128 * TG_NC * 2;    // [128][stride] FP32 target rows
constexpr int TG_TSTRIDE = TG_NC + 2;              // floats; target_stride(nc) at most
constexpr int TGO_B = TGO_T + 128 * TG_TSTRIDE * 4;  // b1[64] b2[64] b3[176] cw[176]
constexpr int TG_SMEM = TGO_B + (64 + 64 + 2 * TG_NC) * 4;
static_assert(TG_SMEM <= 227 * 1024 - 1024, "one CTA per SM");
// TMEM columns: per-tile scratch (Z1, Z2, Y, dH2, dH1, dX) and the weight gradients
constexpr uint32_t TC_SCR = 0, TC_G3 = 192, TC_G2 = 384, TC_G1 = 448, TC_COLS = 512;

// Row stride of the target tile: even (8-byte copies) and 2 mod 4, so that the
// 8-byte reads of 16 consecutive rows hit 16 different bank pairs.
__host__ __device__ constexpr int target_stride(int nc) { return nc + (6 - nc % 4) % 4; }

struct DecoderGradTcParams {
    fpo_mlp w, g;
    const uint32_t *rows;
    uint32_t batch;
    const float *latents, *targets, *coef_weight, *extra_dy;
    float *dlatents;
    double *loss;
    uint32_t *status;
    int nc;
    int test_timeout;
};

__device__ __forceinline__ uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// An operand as the MMAs of one GEMM read it: start address, byte strides
// between 8-element groups along K (per 16-wide MMA step: two groups) and
// along M or N, and whether M or N is the contiguous direction.
struct Operand {
    uint32_t addr, k8, mn8;
    bool mn_major;
};
// A row-major matrix in core matrices with `cols` columns: summed over its
// columns (K-major), or over its rows (MN-major).
__device__ __forceinline__ Operand over_cols(uint32_t addr, int cols) { return {addr, 128u, (uint32_t)cols * 16u, false}; }
__device__ __forceinline__ Operand over_rows(uint32_t addr, int cols) { return {addr, (uint32_t)cols * 16u, 128u, true}; }

// D[128 x N] (+)= A B^T over K, BF16; acc0: accumulate from the first K slice on.
// No-swizzle descriptors: K-major, LBO = K group stride, SBO = row group stride;
// MN-major, LBO = K group stride, SBO = M/N group stride.
template <int K, int N>
__device__ __forceinline__ void gemm_bf16(uint32_t d_tmem, Operand a, Operand b, uint32_t acc0)
{
    const uint32_t idesc = idesc_bf16(128, N) | (a.mn_major ? 1u << 15 : 0u) | (b.mn_major ? 1u << 16 : 0u);
    const uint64_t da = smem_desc(a.addr, a.k8, a.mn8), db = smem_desc(b.addr, b.k8, b.mn8);
#pragma unroll
    for (int s = 0; s < K / 16; ++s)  // (the address field counts 16 bytes and does not overflow)
        mma_f16(d_tmem, da + (uint64_t)(s * (a.k8 >> 3)), db + (uint64_t)(s * (b.k8 >> 3)), idesc, s > 0 ? 1u : acc0);
}

// 16 consecutive FP32 columns of this thread's TMEM lane; waits for them.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void cp_async(void *dst, const void *src, bool pair)
{
    if (pair) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 8 consecutive values of row `row` (K-chunk j) as BF16.
__device__ __forceinline__ void put8_bf(unsigned char *base, int row, int j, int K, const float *v)
{
    uint32_t h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
        h[e] = *reinterpret_cast<const uint32_t *>(&b);
    }
    *reinterpret_cast<uint4 *>(base + core_off(row, 8 * j, K)) = make_uint4(h[0], h[1], h[2], h[3]);
}

// K-chunk j of row `row` = {c, 0 x 7} in BF16: the ones column of an activation.
__device__ __forceinline__ void put_one_bf(unsigned char *base, int row, int j, int K, float c)
{
    const __nv_bfloat162 p = __floats2bfloat162_rn(c, 0.0f);
    *reinterpret_cast<uint4 *>(base + core_off(row, 8 * j, K)) =
        make_uint4(*reinterpret_cast<const uint32_t *>(&p), 0u, 0u, 0u);
}
}  // namespace

__global__ void __launch_bounds__(TG_THREADS, 1) decoder_grad_tc_kernel(const __grid_constant__ DecoderGradTcParams p)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ uint64_t s_bar, s_never;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_fail[2];
    __shared__ double s_loss;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const bool epi = t < TG_EPI;           // (the other warp issues the MMAs)
    const int m = t & 127, part = t >> 7;  // row of the tile, and which quarter of the columns
    const int nc = p.nc, ts = target_stride(nc);
    const bool pair = (nc & 1) == 0 && (reinterpret_cast<uintptr_t>(p.targets) & 7u) == 0;
    float *s_t = reinterpret_cast<float *>(sm + TGO_T);
    float *s_b1 = reinterpret_cast<float *>(sm + TGO_B), *s_b2 = s_b1 + 64, *s_b3 = s_b2 + 64, *s_cw = s_b3 + TG_NC;
    const uint32_t n_tiles = (p.batch + 127) / 128;
    constexpr int WR = 128 / (TG_EPI / 32);  // rows of a tile that a warp moves

    // Epilogue warp w moves rows WR w .. WR w + WR - 1 of a tile: the target
    // rows by asynchronous copies, the latents into registers (lane = feature).
    // Rows past the end are zeros (next_ids: their leaf numbers, fetched ahead).
    float xr[WR];
    auto tile_ids = [&](uint32_t tile) -> uint32_t {
        const uint32_t r = tile * 128 + (uint32_t)(warp * WR + lane);
        return lane < WR && tile < n_tiles && r < p.batch ? p.rows[r] : 0u;
    };
    auto load_rows = [&](uint32_t tile, uint32_t ids) {
        const uint32_t r0 = tile * 128 + (uint32_t)(warp * WR);
#pragma unroll
        for (int i = 0; i < WR; ++i) {
            const size_t row = __shfl_sync(0xffffffffu, ids, i);
            const float *src = p.targets + row * nc;
            float *dst = s_t + (warp * WR + i) * ts;
            const bool there = tile < n_tiles && r0 + i < p.batch;
            xr[i] = there ? p.latents[row * 32 + lane] : 0.0f;
            if (there && pair) {
                for (int c = 2 * lane; c < nc; c += 64) cp_async(dst + c, src + c, true);
            } else if (there) {
                for (int c = lane; c < nc; c += 32) cp_async(dst + c, src + c, false);
            } else {
                for (int c = lane; c < nc; c += 32) dst[c] = 0.0f;
            }
        }
    };
    uint32_t next_ids = 0;
    if (epi) load_rows(blockIdx.x, tile_ids(blockIdx.x));
    if (t == 0) {
        s_fail[0] = s_fail[1] = 0;
        s_loss = 0.0;
        ptx::mbar_init(&s_bar, 1);
        ptx::mbar_init(&s_never, 1);
        ptx::fence_barrier_init();
    }
    if (warp == TG_EPI / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(&s_tmem)),
                     "r"(TC_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // --- weights as BF16 operands (all of a thread's loads in flight together)
    // and FP32 biases, once per CTA
    if (epi) {
        constexpr int C1 = 64 * 4, C2 = 64 * 8, CH = C1 + C2 + TG_NC * 8, PER = (CH + TG_EPI - 1) / TG_EPI;
        const bool a16 = ((reinterpret_cast<uintptr_t>(p.w.w1) | reinterpret_cast<uintptr_t>(p.w.w2) |
                           reinterpret_cast<uintptr_t>(p.w.w3)) & 15u) == 0;
        float v[PER][8];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int q = t + TG_EPI * i;
            const float *src = q < C1 ? p.w.w1 + q * 8 : (q < C1 + C2 ? p.w.w2 + (q - C1) * 8 : p.w.w3 + (q - C1 - C2) * 8);
            const bool there = q < C1 + C2 + nc * 8;
            if (there && a16) {
                const float4 lo = __ldg(reinterpret_cast<const float4 *>(src)), hi = __ldg(reinterpret_cast<const float4 *>(src) + 1);
                v[i][0] = lo.x, v[i][1] = lo.y, v[i][2] = lo.z, v[i][3] = lo.w;
                v[i][4] = hi.x, v[i][5] = hi.y, v[i][6] = hi.z, v[i][7] = hi.w;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[i][e] = there ? __ldg(src + e) : 0.0f;
            }
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int q = t + TG_EPI * i;
            if (q < C1) put8_bf(sm + TGO_W1, q >> 2, q & 3, 32, v[i]);
            else if (q < C1 + C2) put8_bf(sm + TGO_W2, (q - C1) >> 3, (q - C1) & 7, 64, v[i]);
            else if (q < CH) put8_bf(sm + TGO_W3, (q - C1 - C2) >> 3, (q - C1 - C2) & 7, 64, v[i]);
        }
        if (t < 64) {
            s_b1[t] = p.w.b1[t];
            s_b2[t] = p.w.b2[t];
        }
        if (t < TG_NC) {
            s_b3[t] = t < nc ? p.w.b3[t] : 0.0f;
            s_cw[t] = t < nc ? p.coef_weight[t] : 0.0f;
        }
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();

    const uint32_t tm = s_tmem;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;  // this warp's lane quarter
    const uint32_t sa = ptx::smem_u32(sm);
    float lsum = 0.0f;
    uint32_t commits = 0;  // MMA warp: rounds issued
    // End of an epilogue (generic smem writes and TMEM reads before the next
    // MMAs), and the MMA warp's signal to issue them.  False once a wait has
    // run out anywhere in the CTA: every thread leaves the loop here.  Hand-offs
    // take the two words of s_fail by turns (six a tile, so each has its own):
    // the waits before this one report in s_fail[turn], those after it in the
    // other, and a slow thread still reads here what the fast ones read.
    auto hand_off = [&](const int turn) -> bool {
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        return s_fail[turn] == 0;
    };
    if (epi) {
        uint32_t phase = 0;
        bool first_wait = p.test_timeout != 0;
        // (bounded; a warp whose wait runs out goes on to the next hand_off)
        auto wait_mmas = [&](const int turn) -> bool {  // turn: of the hand-off after it
            bool done = first_wait ? ptx::mbar_wait_bounded(&s_never, 0, TEST_WAIT_LIMIT_NS)
                                   : ptx::mbar_wait_bounded(&s_bar, phase, LT_WAIT_NS);
            done = __all_sync(0xffffffffu, done);
            first_wait = false;
            if (!done) s_fail[turn] = 1;
            fence_after();
            phase ^= 1u;
            return done;
        };
        // H = relu(Z + b) of this thread's 16 columns into `dst`; returns the mask of Z + b > 0
        auto relu_part = [&](unsigned char *dst, const float *b) -> uint32_t {
            float v[16];
            tmem_ld16(tm + lane_off + TC_SCR + 16 * part, v);
            uint32_t mask = 0;
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 bv = *reinterpret_cast<const float4 *>(b + 16 * part + e);
                const float bq[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float z = v[e + k] + bq[k];
                    if (z > 0.0f) mask |= 1u << (e + k);
                    v[e + k] = fmaxf(z, 0.0f);
                }
            }
            put8_bf(dst, m, 2 * part, TG_KH, v);
            put8_bf(dst, m, 2 * part + 1, TG_KH, v + 8);
            return mask;
        };
        // d = dH [mask] of this thread's 16 columns (over dY, or over the layer's before)
        auto masked_part = [&](uint32_t mask) {
            float v[16];
            tmem_ld16(tm + lane_off + TC_SCR + 16 * part, v);
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = (mask >> e) & 1u ? v[e] : 0.0f;
            put8_bf(sm + TGO_DY, m, 2 * part, 64, v);
            put8_bf(sm + TGO_DY, m, 2 * part + 1, 64, v + 8);
        };
        for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            const uint32_t r0 = tile * 128;
            const bool valid = r0 + (uint32_t)m < p.batch;
            const float one = valid ? 1.0f : 0.0f;
            next_ids = tile_ids(tile + gridDim.x);
            // (the previous tile's last MMAs, which read X, H1 and d1, are done)
#pragma unroll
            for (int i = 0; i < WR; ++i)
                *reinterpret_cast<__nv_bfloat16 *>(sm + TGO_X + core_off(warp * WR + i, lane, TG_KX)) = __float2bfloat16_rn(xr[i]);
            if (part == 0) put_one_bf(sm + TGO_X, m, 4, TG_KX, one);
            else if (part == 1) put_one_bf(sm + TGO_H1, m, 8, TG_KH, one);
            else if (part == 2) put_one_bf(sm + TGO_H2, m, 8, TG_KH, one);
            if (!hand_off(0)) break;
            wait_mmas(1);
            const uint32_t m1 = relu_part(sm + TGO_H1, s_b1);
            if (!hand_off(1)) break;
            wait_mmas(0);
            const uint32_t m2 = relu_part(sm + TGO_H2, s_b2);
            cp_async_wait();  // this thread's copies of the tile's targets (all threads': the barrier)
            if (!hand_off(0)) break;
            wait_mmas(1);
            // dY = 2 cw (Y + b3 - target) + extra of this thread's 48 (the last quarter's 32) columns
            const float *trow = s_t + m * ts;
            const float *xrow = p.extra_dy && valid ? p.extra_dy + (size_t)p.rows[r0 + m] * nc : nullptr;
#pragma unroll 1
            for (int c = 3 * part; c < min(3 * part + 3, TG_NC / 16); ++c) {
                float v[16];
                tmem_ld16(tm + lane_off + TC_SCR + 16 * c, v);
                if (16 * c + 16 <= nc) {
#pragma unroll
                    for (int e = 0; e < 16; e += 2) {
                        const float2 tv = *reinterpret_cast<const float2 *>(trow + 16 * c + e);
                        const float2 bv = *reinterpret_cast<const float2 *>(s_b3 + 16 * c + e);
                        const float2 cw = *reinterpret_cast<const float2 *>(s_cw + 16 * c + e);
                        const float e0 = one * (v[e] + bv.x - tv.x), e1 = one * (v[e + 1] + bv.y - tv.y);
                        const float d0 = cw.x * e0, d1 = cw.y * e1;
                        lsum = fmaf(d0, e0, lsum);
                        lsum = fmaf(d1, e1, lsum);
                        v[e] = 2.0f * d0;
                        v[e + 1] = 2.0f * d1;
                    }
                } else {  // the chunk that nc ends in, and any past it
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int j = 16 * c + e;
                        float d = 0.0f;
                        if (j < nc) {
                            const float err = one * (v[e] + s_b3[j] - trow[j]);
                            d = s_cw[j] * err;
                            lsum = fmaf(d, err, lsum);
                        }
                        v[e] = 2.0f * d;
                    }
                }
                if (xrow) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (16 * c + e < nc) v[e] += xrow[16 * c + e];
                }
                put8_bf(sm + TGO_DY, m, 2 * c, TG_NC, v);
                put8_bf(sm + TGO_DY, m, 2 * c + 1, TG_NC, v + 8);
            }
            if (!hand_off(1)) break;
            load_rows(tile + gridDim.x, next_ids);  // the target tile is free: in flight from here on
            wait_mmas(0);
            masked_part(m2);
            if (!hand_off(0)) break;
            wait_mmas(1);
            masked_part(m1);
            if (!hand_off(1)) break;
            // dL/d(latent) of the tile's rows
            if (wait_mmas(0) && part < 2) {
                float v[16];
                tmem_ld16(tm + lane_off + TC_SCR + 16 * part, v);
                if (valid) {
                    float *dst = p.dlatents + (size_t)(r0 + m) * 32 + 16 * part;
                    if ((reinterpret_cast<uintptr_t>(p.dlatents) & 15u) == 0) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            reinterpret_cast<float4 *>(dst)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                    } else {  // (the caller's array needs only float alignment)
#pragma unroll
                        for (int k = 0; k < 16; ++k) dst[k] = v[k];
                    }
                }
            }
        }
        cp_async_wait();
    } else {
        uint32_t acc_w = 0;  // the weight gradients accumulate from the CTA's second tile on
        auto commit = [&]() {
            mma_commit(&s_bar);
            ++commits;
        };
        const Operand xf = over_cols(sa + TGO_X, TG_KX), h1f = over_cols(sa + TGO_H1, TG_KH), h2f = over_cols(sa + TGO_H2, TG_KH),
                      xg = over_rows(sa + TGO_X, TG_KX), h1g = over_rows(sa + TGO_H1, TG_KH), h2g = over_rows(sa + TGO_H2, TG_KH),
                      dyf = over_cols(sa + TGO_DY, TG_NC), dyg = over_rows(sa + TGO_DY, TG_NC), df = over_cols(sa + TGO_DY, 64),
                      dg = over_rows(sa + TGO_DY, 64);
        for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            if (!hand_off(0)) break;
            if (lane == 0) {
                gemm_bf16<32, 64>(tm + TC_SCR, xf, over_cols(sa + TGO_W1, 32), 0);
                commit();
            }
            if (!hand_off(1)) break;
            if (lane == 0) {
                gemm_bf16<64, 64>(tm + TC_SCR, h1f, over_cols(sa + TGO_W2, 64), 0);
                commit();
            }
            if (!hand_off(0)) break;
            if (lane == 0) {
                gemm_bf16<64, TG_NC>(tm + TC_SCR, h2f, over_cols(sa + TGO_W3, 64), 0);
                commit();
            }
            if (!hand_off(1)) break;
            if (lane == 0) {
                gemm_bf16<TG_NC, 64>(tm + TC_SCR, dyf, over_rows(sa + TGO_W3, 64), 0);
                gemm_bf16<128, TG_NC>(tm + TC_G3, h2g, dyg, acc_w);
                commit();
            }
            if (!hand_off(0)) break;
            if (lane == 0) {
                gemm_bf16<64, 64>(tm + TC_SCR, df, over_rows(sa + TGO_W2, 64), 0);
                gemm_bf16<128, 64>(tm + TC_G2, h1g, dg, acc_w);
                commit();
            }
            if (!hand_off(1)) break;
            if (lane == 0) {
                gemm_bf16<64, 32>(tm + TC_SCR, df, over_rows(sa + TGO_W1, 32), 0);
                gemm_bf16<128, 64>(tm + TC_G1, xg, dg, acc_w);
                commit();
            }
            acc_w = 1;
        }
    }
    hand_off(0);  // every wait of the last tile is over
    const bool ok = (s_fail[0] | s_fail[1]) == 0;
    if (ok && epi) {
        // the weight gradients: lane k of G3 / G2 / G1 is input feature k, lane
        // 64 (32 for G1) the bias; column j / o the output feature
#pragma unroll 1
        for (int c = 3 * part; c < min(3 * part + 3, TG_NC / 16); ++c) {
            float v[16];
            tmem_ld16(tm + lane_off + TC_G3 + 16 * c, v);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int j = 16 * c + e;
                if (j >= nc) continue;
                if (m < 64) atomicAdd(p.g.w3 + j * 64 + m, v[e]);
                else if (m == 64) atomicAdd(p.g.b3 + j, v[e]);
            }
        }
        float v[16];
        tmem_ld16(tm + lane_off + TC_G2 + 16 * part, v);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int o = 16 * part + e;
            if (m < 64) atomicAdd(p.g.w2 + o * 64 + m, v[e]);
            else if (m == 64) atomicAdd(p.g.b2 + o, v[e]);
        }
        tmem_ld16(tm + lane_off + TC_G1 + 16 * part, v);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int o = 16 * part + e;
            if (m < 32) atomicAdd(p.g.w1 + o * 32 + m, v[e]);
            else if (m == 32) atomicAdd(p.g.b1 + o, v[e]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0) atomicAdd(&s_loss, (double)lsum);
    } else if (!ok && t == TG_EPI) {
        // the last round committed, whose wait gave up: wait for it once more
        // (bounded) before TMEM is freed
        if (commits) ptx::mbar_wait_bounded(&s_bar, (commits - 1) & 1u, LT_WAIT_NS);
        if (p.status) atomicOr(p.status, STATUS_DEVICE_TIMEOUT);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (t == 0 && p.loss && ok) atomicAdd(p.loss, s_loss);
    if (warp == TG_EPI / 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(TC_COLS) : "memory");
}

// ---------------------------------------------------------------------------
// Decode of every leaf into a render context's FP32 records on the tensor
// cores, with the numerics of the inference decoder (FP16 latents, weights
// rounded to BF16 and then FP16, FP16 hidden activations, biases as FP16
// hi/lo pairs, FP32 accumulation) but the last layer unfolded (all
// n1 + 27 n2 coefficients): what the pixel loss of the decoder's training
// renders.  Eight independent warpgroup pipelines per CTA, one CTA per SM,
// each with 64 TMEM columns (Z1, then Z2, then the last layer in three windows
// of 64 columns that overlap by 8) and one shared-memory region for its
// tile's A operands.  Tile rows are records: thread i gathers latent
// perm[i] and writes record i, 32 bytes of it at a time straight from its
// TMEM lane (a piece of 8 SH values never crosses a window, and 8 values
// start on 32 bytes where the record's stride allows it).  Turning the rows
// through shared memory to write them coalesced took most of the time, and
// the memory of four more pipelines: 438k leaves 266 -> 103 us.
namespace {
constexpr int DR_GROUPS = 8, DR_NC = 176, DR_COLS = 64, DR_WINDOWS = 3, DR_STEP = 56;
static_assert((DR_WINDOWS - 1) * DR_STEP + DR_COLS == DR_NC, "the windows cover the last layer");
constexpr int DRO_W1 = 0;                        // [64][48]  W1 | b1
constexpr int DRO_W2 = DRO_W1 + 64 * K1 * 2;     // [64][80]  W2 | b2
constexpr int DRO_W3 = DRO_W2 + 64 * K2 * 2;     // [176][80] W3 | b3
constexpr int DRO_A = DRO_W3 + DR_NC * K2 * 2;   // per group: [128][80] (X, then H1, then H2)
constexpr int DR_GROUP_BYTES = 128 * K2 * 2;
constexpr int DR_SMEM = DRO_A + DR_GROUPS * DR_GROUP_BYTES;

// Four pieces of 8 consecutive columns of this thread's TMEM lane; waits for them.
__device__ __forceinline__ void tmem_ld8x4(const uint32_t a[4], float v[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3])
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float tmem_ld1(uint32_t a)
{
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=r"(r) : "r"(a) : "memory");
    return __uint_as_float(r);
}

// 8 floats to a 32-byte aligned global address.
__device__ __forceinline__ void stg256(float *p, const float *v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                 "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

struct DecodeTcParams {
    fpo_mlp w;                  // FP32 master weights
    const float *latents;       // [n][32] FP32, upload order
    const uint32_t *perm;       // record -> latent row
    float *sig, *zc;            // FP32 records
    uint32_t n;
    int n1, nc, ss, zs;
    uint32_t *status;
    int test_timeout;
};
}  // namespace

__global__ void __launch_bounds__(128 * DR_GROUPS, 1) decode_records_tc_kernel(const __grid_constant__ DecodeTcParams p)
{
    extern __shared__ __align__(1024) unsigned char dr_smem_raw[];
    unsigned char *sm = dr_smem_raw + ((1024u - (ptx::smem_u32(dr_smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t s_bar[DR_GROUPS];
    __shared__ uint64_t s_never;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail[DR_GROUPS];
    __shared__ int s_range;
    const int tid = threadIdx.x, warp = tid >> 5, group = tid >> 7, m = tid & 127;
    const int nc = p.nc;
    if (tid == 0) {
        s_range = 0;
        for (int g = 0; g < DR_GROUPS; ++g) {
            s_fail[g] = 0;
            ptx::mbar_init(&s_bar[g], 1);
        }
        ptx::mbar_init(&s_never, 1);
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(&s_tmem)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // weights as FP16 B operands, through BF16 as the inference decoder holds
    // them (values beyond the FP16 range are reported)
    auto wv = [&](float x) {
        x = __bfloat162float(__float2bfloat16_rn(x));
        if (!(fabsf(x) <= F16_MAX)) s_range = 1;
        return x;
    };
    auto bv = [&](float x) {  // biases stay FP32 (an FP16 hi/lo pair in the operand)
        if (!(fabsf(x) <= F16_MAX)) s_range = 1;
        return x;
    };
    for (int q = tid; q < 64 * (K1 / 8); q += 128 * DR_GROUPS) {
        const int n = q / (K1 / 8), j = q % (K1 / 8);
        if (j < 4) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = wv(p.w.w1[n * 32 + 8 * j + e]);
            put8(sm + DRO_W1, n, j, K1, v);
        } else if (j == 4) put_bias_chunk(sm + DRO_W1, n, j, K1, bv(p.w.b1[n]), false);
        else put_zero_chunk(sm + DRO_W1, n, j, K1);
    }
    for (int q = tid; q < 64 * (K2 / 8); q += 128 * DR_GROUPS) {
        const int n = q / (K2 / 8), j = q % (K2 / 8);
        if (j < 8) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = wv(p.w.w2[n * 64 + 8 * j + e]);
            put8(sm + DRO_W2, n, j, K2, v);
        } else if (j == 8) put_bias_chunk(sm + DRO_W2, n, j, K2, bv(p.w.b2[n]), false);
        else put_zero_chunk(sm + DRO_W2, n, j, K2);
    }
    for (int q = tid; q < DR_NC * (K2 / 8); q += 128 * DR_GROUPS) {
        const int n = q / (K2 / 8), j = q % (K2 / 8);
        if (n >= nc || j == 9) put_zero_chunk(sm + DRO_W3, n, j, K2);
        else if (j < 8) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = wv(p.w.w3[n * 64 + 8 * j + e]);
            put8(sm + DRO_W3, n, j, K2, v);
        } else put_bias_chunk(sm + DRO_W3, n, j, K2, bv(p.w.b3[n]), false);
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem + (uint32_t)DR_COLS * (uint32_t)group;
    const uint32_t my_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    unsigned char *ga = sm + DRO_A + group * DR_GROUP_BYTES;
    const uint32_t sa_a = ptx::smem_u32(ga), sa_w1 = ptx::smem_u32(sm + DRO_W1), sa_w2 = ptx::smem_u32(sm + DRO_W2),
                   sa_w3 = ptx::smem_u32(sm + DRO_W3);
    uint32_t phase = 0;
    __half2 hmax = __float2half2_rn(0.0f);
    bool first_wait = p.test_timeout != 0;
    auto issue_layer = [&](uint32_t b_addr, int K, int N) {
        if (m == 0) {
            fence_after();
            gemm(tmem, sa_a, b_addr, K, N);
            mma_commit(&s_bar[group]);
        }
    };
    auto wait_layer = [&]() -> bool {
        const bool ok = first_wait ? ptx::mbar_wait_bounded(&s_never, 0, TEST_WAIT_LIMIT_NS)
                                   : ptx::mbar_wait_bounded(&s_bar[group], phase, LT_WAIT_NS);
        first_wait = false;
        if (!ok) s_fail[group] = 1;
        group_sync(group);
        fence_after();
        if (s_fail[group]) return false;
        phase ^= 1u;
        return true;
    };
    auto run_layer = [&](uint32_t b_addr, int K, int N) -> bool {
        issue_layer(b_addr, K, N);
        return wait_layer();
    };
    auto hand_off = [&]() {
        fence_async_smem();
        fence_before();
        group_sync(group);
    };
    const uint32_t n_tiles = (p.n + 127) / 128;
    const uint32_t first = blockIdx.x * DR_GROUPS + group, step = gridDim.x * DR_GROUPS;
    const bool lat16 = (reinterpret_cast<uintptr_t>(p.latents) & 15u) == 0;
    const int zpieces = (p.zs + 7) / 8, nz = nc - p.n1;
    const int whole = min(zpieces, (DR_NC - p.n1) / 8);  // pieces that end inside the layer
    for (uint32_t tile = first; tile < n_tiles; tile += step) {
        const uint32_t rec = tile * 128 + (uint32_t)m;
        const bool valid = rec < p.n;
        {
            // this thread's row: the gathered FP32 latent (all zero past the end)
            const float *src = p.latents + (valid ? (size_t)p.perm[rec] : 0) * 32;
            __half2 hx = __float2half2_rn(0.0f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // FP16 latents, as the inference decoder holds them
                float x[8];
                if (valid && lat16) {
                    const float4 lo = __ldg(reinterpret_cast<const float4 *>(src) + 2 * j), hi = __ldg(reinterpret_cast<const float4 *>(src) + 2 * j + 1);
                    x[0] = lo.x, x[1] = lo.y, x[2] = lo.z, x[3] = lo.w, x[4] = hi.x, x[5] = hi.y, x[6] = hi.z, x[7] = hi.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = valid ? __ldg(src + 8 * j + e) : 0.0f;
                }
                put8(ga, m, j, K1, x);
#pragma unroll
                for (int e = 0; e < 8; ++e) hx = __hmax2(hx, __float2half2_rn(fabsf(x[e])));
            }
            hmax = __hmax2(hmax, hx);
            put_bias_chunk(ga, m, 4, K1, 0.0f, true);
            put_zero_chunk(ga, m, 5, K1);
        }
        hand_off();
        if (!run_layer(sa_w1, K1, 64)) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[32];
            tmem_ld32(my_lane + 32 * h, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) put8_relu(ga, m, 4 * h + c, K2, v + 8 * c, hmax);
        }
        put_bias_chunk(ga, m, 8, K2, 0.0f, true);
        put_zero_chunk(ga, m, 9, K2);
        hand_off();
        if (!run_layer(sa_w2, K2, 64)) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[32];
            tmem_ld32(my_lane + 32 * h, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) put8_relu(ga, m, 4 * h + c, K2, v + 8 * c, hmax);
        }
        hand_off();
        // Y -> record `rec`, window by window: the density record from the
        // first, and the pieces of 8 SH values that each window holds whole
        bool ok = true;
        int k = 0;
#pragma unroll 1
        for (int win = 0; win < DR_WINDOWS; ++win) {
            const int col0 = DR_STEP * win;
            issue_layer(sa_w3 + (uint32_t)core_off(col0, 0, K2), K2, DR_COLS);
            if (!(ok = wait_layer())) break;
            if (win == 0) {
                float v[32];
                tmem_ld32(my_lane, v);
                if (valid) {
                    float *dst = p.sig + (size_t)rec * p.ss;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (4 * q < p.ss)
                            *reinterpret_cast<float4 *>(dst + 4 * q) =
                                make_float4(4 * q < p.n1 ? v[4 * q] : 0.0f, 4 * q + 1 < p.n1 ? v[4 * q + 1] : 0.0f,
                                            4 * q + 2 < p.n1 ? v[4 * q + 2] : 0.0f, 4 * q + 3 < p.n1 ? v[4 * q + 3] : 0.0f);
                }
            }
            // 8 values of SH piece q (elements past 27 n2 are padding: zero)
            auto put_piece = [&](int q, float *v) {
                if (!valid) return;
                float *dst = p.zc + (size_t)rec * p.zs + 8 * q;
                if (8 * q + 8 > nz) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = 8 * q + e < nz ? v[e] : 0.0f;
                }
                if ((p.zs & 7) == 0) {
                    stg256(dst, v);
                } else {
                    *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
                    if (8 * q + 4 < p.zs) *reinterpret_cast<float4 *>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
                }
            };
            const int k_end = win == DR_WINDOWS - 1 ? whole : min(whole, (col0 + DR_COLS - 8 - p.n1) / 8 + 1);
#pragma unroll 1
            for (; k < k_end; k += 4) {
                float v[32];
                uint32_t a[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = my_lane + (uint32_t)(p.n1 + 8 * (k + q < k_end ? k + q : k) - col0);
                tmem_ld8x4(a, v);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (k + q < k_end) put_piece(k + q, v + 8 * q);
            }
            if (win == DR_WINDOWS - 1 && whole < zpieces) {
                // the last piece ends past the layer: only the columns there are
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int c = p.n1 + 8 * whole + e;
                    v[e] = c < nc ? tmem_ld1(my_lane + (uint32_t)(c - col0)) : 0.0f;
                }
                put_piece(whole, v);
            }
            k = k_end;
            fence_before();  // TMEM reads done before the group's next MMAs
            group_sync(group);
        }
        if (!ok) break;
    }
    if (p.status && (!(__low2float(hmax) <= F16_MAX) || !(__high2float(hmax) <= F16_MAX) || (tid == 0 && s_range)))
        atomicOr(p.status, STATUS_FP16_RANGE);
    if (s_fail[group] && m == 0) {
        ptx::mbar_wait_bounded(&s_bar[group], phase, LT_WAIT_NS);
        if (p.status) atomicOr(p.status, STATUS_DEVICE_TIMEOUT);
    }
    __syncthreads();
    fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(512u) : "memory");
}

// cuTensorMapEncodeTiled from the driver, looked up once.
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }();
    return fn;
}

int launch_latent_table(const LatentParams &pin, int sm_count, void *stream)
{
    if (pin.n_leaves == 0) return (int)cudaSuccess;
    LatentParams p = pin;
    // the table as a 2-D tensor [n_leaves][32] of FP32 (128-byte rows) or FP16
    // (64-byte rows), stored in boxes of 128 rows from swizzled shared memory
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return (int)cudaErrorNotSupported;
    const cuuint64_t dims[2] = {TABLE_STRIDE, p.n_leaves};
    const cuuint64_t strides[1] = {TABLE_STRIDE * (p.half_table ? 2u : 4u)};
    const cuuint32_t box[2] = {TABLE_STRIDE, LT_M};
    const cuuint32_t estr[2] = {1, 1};
    if (enc(&p.table_map, p.half_table ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
            p.table, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            p.half_table ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return (int)cudaErrorInvalidValue;
    auto launch = [&](auto kern, int G, int smem, int ctas_per_sm) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     p.carveout > 0 ? p.carveout : (int)cudaSharedmemCarveoutDefault);
        if (e != cudaSuccess) return e;
        int per_sm = ctas_per_sm;
        if (per_sm <= 0) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128 * G, smem);
            if (e != cudaSuccess) return e;
            if (per_sm < 1) per_sm = 1;
        }
        if (per_sm * 64 * G > 512) per_sm = 512 / (64 * G);  // TMEM has 512 columns
        const uint32_t n_tiles = (p.n_leaves + LT_M - 1) / LT_M;
        uint64_t blocks = (uint64_t)sm_count * per_sm;
        const uint64_t need = (n_tiles + G - 1) / G;
        if (blocks > need) blocks = need;
        kern<<<(unsigned)blocks, 128 * G, smem, (cudaStream_t)stream>>>(p);
        return cudaGetLastError();
    };
    if (p.pipeline)
        return (int)launch(latent_table_kernel<LT_GROUPS_PIPE>, LT_GROUPS_PIPE, lt_smem<LT_GROUPS_PIPE>(), 1);
    return (int)launch(latent_table_kernel<LT_GROUPS_FULL>, LT_GROUPS_FULL, lt_smem<LT_GROUPS_FULL>(), 0);
}

int latent_pipeline_smem_bytes() { return lt_smem<LT_GROUPS_PIPE>(); }

int launch_decode_records_tc(const fpo_mlp &w, int n1, int n2, uint32_t n, const float *latents, const uint32_t *perm,
                             float *sig, float *zc, uint32_t *status, bool test_timeout, int sm_count, void *stream)
{
    if (n == 0) return (int)cudaSuccess;
    DecodeTcParams p{};
    p.w = w;
    p.latents = latents;
    p.perm = perm;
    p.sig = sig;
    p.zc = zc;
    p.n = n;
    p.n1 = n1;
    p.nc = n1 + 27 * n2;
    p.ss = sig_stride(n1);
    p.zs = z_stride(n2);
    p.status = status;
    p.test_timeout = test_timeout;
    const int smem = DR_SMEM + 1024;
    cudaError_t e = cudaFuncSetAttribute(decode_records_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return (int)e;
    const uint32_t n_tiles = (n + 127) / 128;
    const uint32_t need = (n_tiles + DR_GROUPS - 1) / DR_GROUPS;
    const uint32_t blocks = need < (uint32_t)sm_count ? need : (uint32_t)sm_count;
    decode_records_tc_kernel<<<blocks, 128 * DR_GROUPS, smem, (cudaStream_t)stream>>>(p);
    return (int)cudaGetLastError();
}

}  // namespace fpo

extern "C" int fpo_decoder_grad_tc(const fpo_mlp *w, int32_t n1, int32_t n2, uint32_t batch, const uint32_t *rows,
                                   const float *latents, const float *targets, const float *coef_weight,
                                   const float *extra_dy, const fpo_mlp *grad, float *dlatents, double *loss,
                                   uint32_t *status, uint32_t flags, void *cuda_stream)
{
    using namespace fpo;
    if (!w || !grad || !w->w1 || !w->b1 || !w->w2 || !w->b2 || !w->w3 || !w->b3 || !grad->w1 || !grad->b1 ||
        !grad->w2 || !grad->b2 || !grad->w3 || !grad->b3)
        return set_last_error(FPO_ERR_INVALID_ARG, "NULL weights");
    if (n1 < 1 || n2 < 1 || n1 + 27 * n2 > TG_NC) return set_last_error(FPO_ERR_INVALID_ARG, "n1 + 27 n2 must be in [28, 176]");
    if (flags & ~(uint32_t)FPO_FLAG_TEST_DEVICE_TIMEOUT) return set_last_error(FPO_ERR_INVALID_ARG, "unknown flags");
    if (batch == 0) return FPO_OK;
    if (!rows || !latents || !targets || !coef_weight || !dlatents) return set_last_error(FPO_ERR_INVALID_ARG, "NULL array");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    DecoderGradTcParams p{};
    p.w = *w;
    p.g = *grad;
    p.rows = rows;
    p.batch = batch;
    p.latents = latents;
    p.targets = targets;
    p.coef_weight = coef_weight;
    p.extra_dy = extra_dy;
    p.dlatents = dlatents;
    p.loss = loss;
    p.status = status;
    p.nc = n1 + 27 * n2;
    p.test_timeout = (flags & FPO_FLAG_TEST_DEVICE_TIMEOUT) != 0;
    const int smem = TG_SMEM;
    e = cudaFuncSetAttribute(decoder_grad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    const uint32_t n_tiles = (batch + 127) / 128;
    const uint32_t blocks = n_tiles < (uint32_t)sms ? n_tiles : (uint32_t)sms;
    decoder_grad_tc_kernel<<<blocks, TG_THREADS, smem, (cudaStream_t)cuda_stream>>>(p);
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    return FPO_OK;
}

using namespace fpo;

extern "C" int fpo_latent_table(const fpo_decoder *dec, int32_t n1, int32_t n2, double t, double period_T,
                                uint32_t n_leaves, const uint16_t *latents, float *table, uint32_t *status,
                                void *cuda_stream)
{
    if (!dec) return set_last_error(FPO_ERR_INVALID_ARG, "dec is NULL");
    if (n1 < 1 || n1 > 32 || n2 < 1 || n2 > 16) return set_last_error(FPO_ERR_INVALID_ARG, "n1 in [1, 32], n2 in [1, 16]");
    if (!(period_T > 0.0)) return set_last_error(FPO_ERR_INVALID_ARG, "period_T must be > 0");
    if (n_leaves == 0) return FPO_OK;
    if (!latents || !table || !dec->w1 || !dec->b1 || !dec->w2 || !dec->b2 || !dec->w3 || !dec->b3)
        return set_last_error(FPO_ERR_INVALID_ARG, "NULL array");
    if (reinterpret_cast<uintptr_t>(latents) % 16 != 0 || reinterpret_cast<uintptr_t>(table) % 16 != 0)
        return set_last_error(FPO_ERR_INVALID_ARG, "latents and table must be 16-byte aligned");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    LatentParams p{};
    p.latents = latents;
    p.w1 = dec->w1;
    p.b1 = dec->b1;
    p.w2 = dec->w2;
    p.b2 = dec->b2;
    p.w3 = dec->w3;
    p.b3 = dec->b3;
    p.n1 = n1;
    p.n2 = n2;
    time_basis(t, period_T, n1 > n2 ? n1 : n2, p.b);
    p.n_leaves = n_leaves;
    p.table = table;
    p.status = status;
    const int ce = launch_latent_table(p, sms, cuda_stream);
    if (ce != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString((cudaError_t)ce));
    return FPO_OK;
}
