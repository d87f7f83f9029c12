// Training kernels of the latent decoder (FP32 masters, SIMT):
//
//  decoder_grad_kernel  for a batch of leaves, the MLP forward
//                       (32 -> 64 -> 64 -> n1 + 27 n2, ReLU), the weighted L2
//                       loss against target coefficients (plus an optional
//                       extra dL/dy, e.g. from the render adjoint), and the
//                       back-propagation to the latents and to every weight.
//                       Each CTA keeps all weights in shared memory, walks
//                       tiles of 64 leaves with register-tiled products, sums
//                       its weight gradients in registers, and adds them to
//                       the global gradients once at the end.
//  ray_batch_kernel     training rays from drawn (camera, pixel, frame) indices.
//  adam_parts_kernel    Adam (Kingma & Ba) on dense arrays and on the rows of
//                       a batch (distinct rows), several arrays in one launch.
//  leaf_adam_kernel     Adam on the marked leaves' coefficient rows, written
//                       back into the renderer's FP32 records.
#include <cuda_runtime.h>

#include <cstdint>

#include "fpo_internal.h"

namespace fpo {
namespace {

// Tiles of TG_ROWS leaves; thread (tr, tc) = (tid >> 4, tid & 15) owns rows
// 4 tr .. 4 tr + 3 in the products over a tile: with the outputs tc + 16 j of
// each layer going forward, with the features 4 tc .. 4 tc + 3 going back; and
// the weight-gradient entries (output 4 tc + 64 q + e, feature 4 tr + i) of
// each layer, summed in registers over all of its CTA's tiles.  Weights are
// kept as [out][in] rows and activations as [row][feature] rows, both padded
// to 4 mod 32 floats: every operand is then read 16 bytes at a time (4 reads
// for 44 to 64 FMAs, where single words took 15 for 44) in the fewest
// wavefronts, whichever index a warp varies.  8,191 leaves: 65 -> 52 us.
constexpr int TG_THREADS = 256;
constexpr int TG_ROWS = 64;   // leaves per tile
constexpr int TG_MAXC = 176;  // n1 + 27 n2 <= 176 (31 + 135 = 166)
constexpr int TG_J = TG_MAXC / 16;
constexpr int S1 = 36, S2 = 68, SY = TG_MAXC + 4;  // padded row strides

struct alignas(16) GradSmem {
    float w1[64 * S1], w2[64 * S2], w3[TG_MAXC * S2], b1[64], b2[64], b3[TG_MAXC];
    float x[TG_ROWS * S1], h1[TG_ROWS * S2], h2[TG_ROWS * S2], dy[TG_ROWS * SY];
    float d2[TG_ROWS * S2], d1[TG_ROWS * S2];
    uint32_t row[TG_ROWS];
    double loss;
};

__device__ __forceinline__ void lds4(const float *p, float v[4])
{
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}

// a[i][j] += sum_k x[4 tr + i][k] w[tc + 16 j][k], k < K in order.
template <int K, int J, int S>
__device__ __forceinline__ void product_forward(float a[4][J], const float *x, const float *w, int tr, int tc)
{
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float xv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) lds4(x + (4 * tr + i) * S + k, xv[i]);
#pragma unroll
        for (int j = 0; j < J; ++j) {
            float wv[4];
            lds4(w + (tc + 16 * j) * S + k, wv);
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i][j] = fmaf(xv[i][e], wv[e], a[i][j]);
        }
    }
}

// a[i][f] += sum_c d[4 tr + i][c] w[c][4 tc + f], c < C (a multiple of 4) in order.
template <int SD, int SW>
__device__ __forceinline__ void product_back(float a[4][4], const float *d, const float *w, int C, int tr, int tc)
{
#pragma unroll 2
    for (int c = 0; c < C; c += 4) {
        float dv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) lds4(d + (4 * tr + i) * SD + c, dv[i]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float wv[4];
            lds4(w + (c + e) * SW + 4 * tc, wv);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int f = 0; f < 4; ++f) a[i][f] = fmaf(dv[i][e], wv[f], a[i][f]);
        }
    }
}

}  // namespace

__global__ void __launch_bounds__(TG_THREADS, 1) decoder_grad_kernel(const __grid_constant__ DecoderGradParams p)
{
    extern __shared__ __align__(16) unsigned char tg_raw[];
    GradSmem &S = *reinterpret_cast<GradSmem *>(tg_raw);
    const int tid = threadIdx.x, nc = p.nc;
    const int tr = tid >> 4, tc = tid & 15;
    for (int i = tid; i < 64 * 32; i += TG_THREADS) S.w1[(i >> 5) * S1 + (i & 31)] = p.w.w1[i];
    for (int i = tid; i < 64 * 64; i += TG_THREADS) S.w2[(i >> 6) * S2 + (i & 63)] = p.w.w2[i];
    for (int i = tid; i < TG_MAXC * 64; i += TG_THREADS) {
        const int j = i >> 6;
        S.w3[j * S2 + (i & 63)] = j < nc ? p.w.w3[i] : 0.0f;
    }
    for (int i = tid; i < 64; i += TG_THREADS) { S.b1[i] = p.w.b1[i]; S.b2[i] = p.w.b2[i]; }
    for (int i = tid; i < TG_MAXC; i += TG_THREADS) S.b3[i] = i < nc ? p.w.b3[i] : 0.0f;
    if (tid == 0) S.loss = 0.0;

    float g3[12][4], g2[4][4], g1[4][2], gb = 0.0f, gb2 = 0.0f, gb1 = 0.0f, lsum = 0.0f;
#pragma unroll
    for (int j = 0; j < 12; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) g3[j][i] = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) g2[j][i] = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) g1[j][0] = g1[j][1] = 0.0f;

    const uint32_t n_tiles = (p.batch + TG_ROWS - 1) / TG_ROWS;
    for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const uint32_t r0 = tile * TG_ROWS;
        const int nr = (int)min((uint32_t)TG_ROWS, p.batch - r0);
        __syncthreads();  // weights staged; the previous tile is done with every buffer
        if (tid < TG_ROWS) S.row[tid] = tid < nr ? p.rows[r0 + tid] : 0u;
        __syncthreads();
        for (int i = tid; i < TG_ROWS * 32; i += TG_THREADS) {
            const int r = i >> 5;
            S.x[r * S1 + (i & 31)] = r < nr ? p.latents[(size_t)S.row[r] * 32 + (i & 31)] : 0.0f;
        }
        __syncthreads();
        // h1 = relu(W1 x + b1)
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = S.b1[tc + 16 * j];
            product_forward<32, 4, S1>(a, S.x, S.w1, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) S.h1[(4 * tr + i) * S2 + tc + 16 * j] = fmaxf(a[i][j], 0.0f);
        }
        __syncthreads();
        // h2 = relu(W2 h1 + b2)
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = S.b2[tc + 16 * j];
            product_forward<64, 4, S2>(a, S.h1, S.w2, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) S.h2[(4 * tr + i) * S2 + tc + 16 * j] = fmaxf(a[i][j], 0.0f);
        }
        __syncthreads();
        // y = W3 h2 + b3; dy = 2 cw (y - target) + extra (0 on padding rows and columns)
        {
            float a[4][TG_J];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < TG_J; ++j) a[i][j] = S.b3[tc + 16 * j];
            product_forward<64, TG_J, S2>(a, S.h2, S.w3, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 4 * tr + i;
                const size_t row = S.row[r];
#pragma unroll
                for (int j = 0; j < TG_J; ++j) {
                    const int c = tc + 16 * j;
                    float d = 0.0f;
                    if (r < nr && c < nc) {
                        const float e = a[i][j] - p.targets[row * nc + c];
                        const float cw = p.coef_weight[c];
                        lsum = fmaf(cw * e, e, lsum);
                        d = 2.0f * cw * e;
                        if (p.extra_dy) d += p.extra_dy[row * nc + c];
                    }
                    S.dy[r * SY + c] = d;
                }
            }
        }
        __syncthreads();
        // d2 = (W3^T dy) * [h2 > 0];  g3 += dy h2^T;  gb3 += dy
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = 0.0f;
            // (the columns from nc to TG_MAXC of dy and the rows of W3 there are zero)
            product_back<SY, S2>(a, S.dy, S.w3, (nc + 3) & ~3, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int o = (4 * tr + i) * S2 + 4 * tc;
                float h[4];
                lds4(S.h2 + o, h);
                *reinterpret_cast<float4 *>(S.d2 + o) = make_float4(h[0] > 0.0f ? a[i][0] : 0.0f, h[1] > 0.0f ? a[i][1] : 0.0f,
                                                                    h[2] > 0.0f ? a[i][2] : 0.0f, h[3] > 0.0f ? a[i][3] : 0.0f);
            }
#pragma unroll 2
            for (int r = 0; r < nr; ++r) {
                float hv[4];
                lds4(S.h2 + r * S2 + 4 * tr, hv);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    float dv[4];
                    lds4(S.dy + r * SY + (q < 2 || tc < 12 ? 4 * tc + 64 * q : 0), dv);  // (176 = 2 x 64 + 4 x 12 outputs)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int i = 0; i < 4; ++i) g3[4 * q + e][i] = fmaf(dv[e], hv[i], g3[4 * q + e][i]);
                }
            }
            if (tid < nc)
                for (int r = 0; r < nr; ++r) gb += S.dy[r * SY + tid];
        }
        __syncthreads();
        // d1 = (W2^T d2) * [h1 > 0];  g2 += d2 h1^T;  gb2 += d2
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = 0.0f;
            product_back<S2, S2>(a, S.d2, S.w2, 64, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int o = (4 * tr + i) * S2 + 4 * tc;
                float h[4];
                lds4(S.h1 + o, h);
                *reinterpret_cast<float4 *>(S.d1 + o) = make_float4(h[0] > 0.0f ? a[i][0] : 0.0f, h[1] > 0.0f ? a[i][1] : 0.0f,
                                                                    h[2] > 0.0f ? a[i][2] : 0.0f, h[3] > 0.0f ? a[i][3] : 0.0f);
            }
#pragma unroll 4
            for (int r = 0; r < nr; ++r) {
                float dv[4], hv[4];
                lds4(S.d2 + r * S2 + 4 * tc, dv);
                lds4(S.h1 + r * S2 + 4 * tr, hv);
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int i = 0; i < 4; ++i) g2[e][i] = fmaf(dv[e], hv[i], g2[e][i]);
            }
            if (tid < 64)
                for (int r = 0; r < nr; ++r) gb2 += S.d2[r * S2 + tid];
        }
        __syncthreads();
        // dx = W1^T d1 (the latents' gradient);  g1 += d1 x^T;  gb1 += d1
        {
            float a[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i][0] = a[i][1] = 0.0f;
#pragma unroll 2
            for (int o = 0; o < 64; o += 4) {  // features 2 tc, 2 tc + 1
                float dv[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) lds4(S.d1 + (4 * tr + i) * S2 + o, dv[i]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 wv = *reinterpret_cast<const float2 *>(S.w1 + (o + e) * S1 + 2 * tc);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        a[i][0] = fmaf(dv[i][e], wv.x, a[i][0]);
                        a[i][1] = fmaf(dv[i][e], wv.y, a[i][1]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 4 * tr + i;
                if (r < nr) {
                    p.dlatents[(size_t)(r0 + r) * 32 + 2 * tc] = a[i][0];
                    p.dlatents[(size_t)(r0 + r) * 32 + 2 * tc + 1] = a[i][1];
                }
            }
#pragma unroll 4
            for (int r = 0; r < nr; ++r) {
                float dv[4];
                lds4(S.d1 + r * S2 + 4 * tc, dv);
                const float2 xv = *reinterpret_cast<const float2 *>(S.x + r * S1 + 2 * tr);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    g1[e][0] = fmaf(dv[e], xv.x, g1[e][0]);
                    g1[e][1] = fmaf(dv[e], xv.y, g1[e][1]);
                }
            }
            if (tid < 64)
                for (int r = 0; r < nr; ++r) gb1 += S.d1[r * S2 + tid];
        }
    }
    // this CTA's sums into the global gradients
    const bool a16 = ((reinterpret_cast<uintptr_t>(p.g.w3) | reinterpret_cast<uintptr_t>(p.g.w2)) & 15u) == 0;
    auto add4 = [&](float *dst, const float *v) {
        if (a16) {
            atomicAdd(reinterpret_cast<float4 *>(dst), make_float4(v[0], v[1], v[2], v[3]));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) atomicAdd(dst + i, v[i]);
        }
    };
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if ((q < 2 || tc < 12) && 4 * tc + 64 * q + e < nc) add4(p.g.w3 + (4 * tc + 64 * q + e) * 64 + 4 * tr, g3[4 * q + e]);
#pragma unroll
    for (int e = 0; e < 4; ++e) add4(p.g.w2 + (4 * tc + e) * 64 + 4 * tr, g2[e]);
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int i = 0; i < 2; ++i) atomicAdd(p.g.w1 + (4 * tc + e) * 32 + 2 * tr + i, g1[e][i]);
    if (tid < nc) atomicAdd(p.g.b3 + tid, gb);
    if (tid < 64) {
        atomicAdd(p.g.b2 + tid, gb2);
        atomicAdd(p.g.b1 + tid, gb1);
    }
    // loss: warp sums, then one shared double per CTA
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    __syncthreads();
    if ((tid & 31) == 0) atomicAdd(&S.loss, (double)lsum);
    __syncthreads();
    if (tid == 0 && p.loss) atomicAdd(p.loss, S.loss);
}

int launch_decoder_grad(const DecoderGradParams &p, int sm_count, void *stream)
{
    if (p.batch == 0) return (int)cudaSuccess;
    const int smem = (int)sizeof(GradSmem);
    cudaError_t e = cudaFuncSetAttribute(decoder_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return (int)e;
    const uint32_t n_tiles = (p.batch + TG_ROWS - 1) / TG_ROWS;
    uint32_t blocks = (uint32_t)sm_count;
    if (blocks > n_tiles) blocks = n_tiles;
    decoder_grad_kernel<<<blocks, TG_THREADS, smem, (cudaStream_t)stream>>>(p);
    return (int)cudaGetLastError();
}

int decoder_grad_max_coeffs() { return TG_MAXC; }

// FP32 decode of every leaf: y = W3 relu(W2 relu(W1 x + b1) + b2) + b3.  A CTA
// keeps the transposed weights in shared memory and walks tiles of 64 leaves;
// each thread owns 4 rows x the output columns 4 tc + 64 g + e (e = 0..3; g = 0
// for the 64-wide hidden layers, g = 0..2 for the last layer), so per input
// feature it reads its weights with one 16-byte load per group (16 threads
// read 256 consecutive bytes) and its 4 activations as broadcasts.  In the
// last layer, columns 176..191 of group 2 read into the next weight row (or the
// biases after it) and are discarded.
// Record mode (perm != nullptr): output row i is the context's FP32 record
// i, decoded from latent row perm[i], its first n1 values going to the
// density records (stride ss) and the rest to the SH records (stride zs).
constexpr int DF_ROWS = 64, DF_THREADS = 256, DF_MAXC = 176;

struct DecodeSmem {
    float w1t[32 * 64], w2t[64 * 64], w3t[64 * DF_MAXC], b1[64], b2[64], b3[DF_MAXC + 16];
    float x[DF_ROWS * 33], h1[DF_ROWS * 65], h2[DF_ROWS * 65];
    uint32_t src[DF_ROWS];
};

struct DecodeOut {
    float *coeffs;          // [n][nc], or nullptr in record mode
    const uint32_t *perm;   // record -> latent row (record mode)
    float *sig, *zc;        // FP32 records (record mode)
    int n1, ss, zs;
};

// a[i][4 g + e] += sum_k in[(4 tr + i) * ld_in + k] * wt[k * ldw + 4 tc + 64 g + e]
template <int G>
__device__ __forceinline__ void decode_layer(const float *in, int ld_in, int K, const float *wt, int ldw,
                                             float (&a)[4][4 * G], int tr, int tc)
{
#pragma unroll 2
    for (int k = 0; k < K; ++k) {
        float xv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) xv[i] = in[(4 * tr + i) * ld_in + k];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float4 w = *reinterpret_cast<const float4 *>(wt + k * ldw + 4 * tc + 64 * g);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i][4 * g] = fmaf(xv[i], w.x, a[i][4 * g]);
                a[i][4 * g + 1] = fmaf(xv[i], w.y, a[i][4 * g + 1]);
                a[i][4 * g + 2] = fmaf(xv[i], w.z, a[i][4 * g + 2]);
                a[i][4 * g + 3] = fmaf(xv[i], w.w, a[i][4 * g + 3]);
            }
        }
    }
}

__global__ void __launch_bounds__(DF_THREADS, 2) decoder_forward_kernel(const fpo_mlp w, int nc, uint32_t n,
                                                                         const float *__restrict__ latents,
                                                                         const DecodeOut o)
{
    extern __shared__ __align__(16) unsigned char df_raw[];
    DecodeSmem &S = *reinterpret_cast<DecodeSmem *>(df_raw);
    const int tid = threadIdx.x;
    for (int i = tid; i < 64 * 32; i += DF_THREADS) S.w1t[(i & 31) * 64 + (i >> 5)] = w.w1[i];
    for (int i = tid; i < 64 * 64; i += DF_THREADS) S.w2t[(i & 63) * 64 + (i >> 6)] = w.w2[i];
    for (int i = tid; i < DF_MAXC * 64; i += DF_THREADS) {
        const int c = i >> 6, k = i & 63;
        S.w3t[k * DF_MAXC + c] = c < nc ? w.w3[c * 64 + k] : 0.0f;
    }
    for (int i = tid; i < 64; i += DF_THREADS) { S.b1[i] = w.b1[i]; S.b2[i] = w.b2[i]; }
    for (int i = tid; i < DF_MAXC + 16; i += DF_THREADS) S.b3[i] = i < nc ? w.b3[i] : 0.0f;
    const int tr = tid >> 4, tc = tid & 15;  // rows 4 tr .. 4 tr + 3; columns 4 tc + 64 g + e
    const uint32_t n_tiles = (n + DF_ROWS - 1) / DF_ROWS;
    for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const uint32_t r0 = tile * DF_ROWS;
        const int nr = (int)min((uint32_t)DF_ROWS, n - r0);
        __syncthreads();  // weights staged; the previous tile is done with x, h1, h2, src
        if (tid < DF_ROWS) S.src[tid] = tid < nr ? (o.perm ? o.perm[r0 + tid] : r0 + tid) : 0u;
        __syncthreads();
        for (int i = tid; i < DF_ROWS * 32; i += DF_THREADS) {
            const int r = i >> 5;
            S.x[r * 33 + (i & 31)] = r < nr ? latents[(size_t)S.src[r] * 32 + (i & 31)] : 0.0f;
        }
        __syncthreads();
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) a[i][e] = S.b1[4 * tc + e];
            decode_layer<1>(S.x, 33, 32, S.w1t, 64, a, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) S.h1[(4 * tr + i) * 65 + 4 * tc + e] = fmaxf(a[i][e], 0.0f);
        }
        __syncthreads();
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) a[i][e] = S.b2[4 * tc + e];
            decode_layer<1>(S.h1, 65, 64, S.w2t, 64, a, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) S.h2[(4 * tr + i) * 65 + 4 * tc + e] = fmaxf(a[i][e], 0.0f);
        }
        __syncthreads();
        {
            float a[4][12];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 12; ++j) a[i][j] = S.b3[4 * tc + 64 * (j >> 2) + (j & 3)];
            decode_layer<3>(S.h2, 65, 64, S.w3t, DF_MAXC, a, tr, tc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 4 * tr + i;
                if (r < nr) {
                    const size_t row = r0 + r;
#pragma unroll
                    for (int j = 0; j < 12; ++j) {
                        const int c = 4 * tc + 64 * (j >> 2) + (j & 3);
                        if (c >= nc) continue;
                        if (!o.perm) o.coeffs[row * nc + c] = a[i][j];
                        else if (c < o.n1) o.sig[row * o.ss + c] = a[i][j];
                        else o.zc[row * o.zs + (c - o.n1)] = a[i][j];
                    }
                }
            }
        }
    }
}

static int launch_decode(const fpo_mlp &w, int nc, uint32_t n, const float *latents, const DecodeOut &o,
                         int sm_count, void *stream)
{
    if (n == 0) return (int)cudaSuccess;
    const int smem = (int)sizeof(DecodeSmem);
    cudaError_t e = cudaFuncSetAttribute(decoder_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return (int)e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, decoder_forward_kernel, DF_THREADS, smem);
    if (e != cudaSuccess) return (int)e;
    if (per_sm < 1) per_sm = 1;
    const uint32_t n_tiles = (n + DF_ROWS - 1) / DF_ROWS;
    uint64_t blocks = (uint64_t)sm_count * per_sm;
    if (blocks > n_tiles) blocks = n_tiles;
    decoder_forward_kernel<<<(unsigned)blocks, DF_THREADS, smem, (cudaStream_t)stream>>>(w, nc, n, latents, o);
    return (int)cudaGetLastError();
}

int launch_decoder_forward(const fpo_mlp &w, int nc, uint32_t n, const float *latents, float *out, int sm_count,
                           void *stream)
{
    DecodeOut o{};
    o.coeffs = out;
    return launch_decode(w, nc, n, latents, o, sm_count, stream);
}

int launch_decode_records(const fpo_mlp &w, int n1, int n2, uint32_t n, const float *latents, const uint32_t *perm,
                          float *sig, float *zc, int sm_count, void *stream)
{
    DecodeOut o{};
    o.perm = perm;
    o.sig = sig;
    o.zc = zc;
    o.n1 = n1;
    o.ss = sig_stride(n1);
    o.zs = z_stride(n2);
    return launch_decode(w, n1 + 27 * n2, n, latents, o, sm_count, stream);
}

// Training rays from drawn (camera, pixel, frame) indices.  One launch in place
// of some twenty elementwise ones, which took 0.4 ms of host time for the 8,192
// rays of a pixel-loss step; the _rn operations keep those launches' rounding
// (a scalar division is a product with the rounded reciprocal, and the norm
// sums x^2 + z^2 first).
__global__ void __launch_bounds__(256) ray_batch_kernel(const float *__restrict__ basis, const int64_t *__restrict__ cam,
                                                        const int64_t *__restrict__ pixel, const int64_t *__restrict__ frame,
                                                        uint32_t n, int64_t W, float fw, float iw, float ih, float th,
                                                        float *__restrict__ o, float *__restrict__ d, float *__restrict__ t)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float *b = basis + 12 * cam[i];
        const int64_t p = pixel[i];
        const float cx = __fmul_rn(2.0f, __fadd_rn((float)(p % W), 0.5f)), cy = __fmul_rn(2.0f, __fadd_rn((float)(p / W), 0.5f));
        const float sx = __fmul_rn(__fmul_rn(__fmul_rn(__fadd_rn(__fmul_rn(cx, iw), -1.0f), th), fw), ih);
        const float sy = __fmul_rn(__fadd_rn(1.0f, -__fmul_rn(cy, ih)), th);
        float v[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            o[3 * (size_t)i + k] = b[k];
            v[k] = __fadd_rn(__fadd_rn(b[3 + k], __fmul_rn(sx, b[6 + k])), __fmul_rn(sy, b[9 + k]));
        }
        const float len = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(v[0], v[0]), __fmul_rn(v[2], v[2])), __fmul_rn(v[1], v[1])));
#pragma unroll
        for (int k = 0; k < 3; ++k) d[3 * (size_t)i + k] = __fdiv_rn(v[k], len);
        t[i] = (float)frame[i];
    }
}

// Adam: g *= scale, m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2,
// p -= lr (m / (1 - b1^step)) / (sqrt(v / (1 - b2^step)) + eps), for several
// arrays in one launch: the decoder's six weight arrays hold 17k values
// between them, and a training step was bound by the launches that zeroed,
// scaled and updated them one by one (22 launches, 270 us for 77 us of
// gradient kernel).  Blocks are divided among the parts; arrays whose
// bases and lengths allow it move 16 bytes a thread.
struct AdamPart {
    float *p, *g, *m, *v;
    const uint32_t *rows;   // p, m, v are indexed by rows[i / dim], or nullptr: by i
    uint32_t dim;
    uint32_t first_block;
    uint64_t n;
    float lr, scale;        // (scale 1: g is only read)
    bool vec;
};
constexpr uint32_t ADAM_MAX_PARTS = 8;
struct AdamParts {
    AdamPart part[ADAM_MAX_PARTS];
    uint32_t n_parts;
    float b1, b2, eps, bc1, bc2;
};

__global__ void __launch_bounds__(256) adam_parts_kernel(const __grid_constant__ AdamParts A)
{
    uint32_t k = 0;
    while (k + 1 < A.n_parts && blockIdx.x >= A.part[k + 1].first_block) ++k;
    const AdamPart &q = A.part[k];
    const uint32_t end_block = k + 1 < A.n_parts ? A.part[k + 1].first_block : gridDim.x;
    const uint64_t step = (uint64_t)(end_block - q.first_block) * blockDim.x;
    auto update = [&](float g, float &p, float &m, float &v) {
        m = A.b1 * m + (1.0f - A.b1) * g;
        v = A.b2 * v + (1.0f - A.b2) * g * g;
        p -= q.lr * (m / A.bc1) / (sqrtf(v / A.bc2) + A.eps);
    };
    const uint64_t first = (uint64_t)(blockIdx.x - q.first_block) * blockDim.x + threadIdx.x;
    if (q.vec) {
        for (uint64_t u = first; u < q.n / 4; u += step) {
            const uint64_t i = 4 * u;
            const size_t at = q.rows ? (size_t)q.rows[i / q.dim] * q.dim + i % q.dim : (size_t)i;
            float4 g = *reinterpret_cast<const float4 *>(q.g + i);
            float4 p = *reinterpret_cast<const float4 *>(q.p + at), m = *reinterpret_cast<const float4 *>(q.m + at),
                   v = *reinterpret_cast<const float4 *>(q.v + at);
            if (q.scale != 1.0f) {
                g = make_float4(g.x * q.scale, g.y * q.scale, g.z * q.scale, g.w * q.scale);
                *reinterpret_cast<float4 *>(q.g + i) = g;
            }
            update(g.x, p.x, m.x, v.x);
            update(g.y, p.y, m.y, v.y);
            update(g.z, p.z, m.z, v.z);
            update(g.w, p.w, m.w, v.w);
            *reinterpret_cast<float4 *>(q.p + at) = p;
            *reinterpret_cast<float4 *>(q.m + at) = m;
            *reinterpret_cast<float4 *>(q.v + at) = v;
        }
        return;
    }
    for (uint64_t i = first; i < q.n; i += step) {
        const size_t at = q.rows ? (size_t)q.rows[i / q.dim] * q.dim + i % q.dim : (size_t)i;
        float g = q.g[i];
        if (q.scale != 1.0f) {
            g *= q.scale;
            q.g[i] = g;
        }
        float p = q.p[at], m = q.m[at], v = q.v[at];
        update(g, p, m, v);
        q.p[at] = p;
        q.m[at] = m;
        q.v[at] = v;
    }
}

int launch_adam(const fpo_adam_part *parts, uint32_t n_parts, float b1, float b2, float eps, uint32_t step, int sm_count,
                void *stream)
{
    AdamParts A{};
    uint64_t blocks = 0;
    for (uint32_t k = 0; k < n_parts; ++k) {
        const fpo_adam_part &s = parts[k];
        if (s.n == 0) continue;
        AdamPart &q = A.part[A.n_parts++];
        q.p = s.param;
        q.g = s.grad;
        q.m = s.m;
        q.v = s.v;
        q.rows = s.rows;
        q.dim = s.rows ? s.dim : 1;
        q.n = s.n;
        q.lr = s.lr;
        q.scale = s.grad_scale;
        const uintptr_t bases = reinterpret_cast<uintptr_t>(s.param) | reinterpret_cast<uintptr_t>(s.grad) |
                                reinterpret_cast<uintptr_t>(s.m) | reinterpret_cast<uintptr_t>(s.v);
        q.vec = (bases & 15u) == 0 && s.n % 4 == 0 && (!s.rows || s.dim % 4 == 0);
        q.first_block = (uint32_t)blocks;
        uint64_t b = ((q.vec ? s.n / 4 : s.n) + 255) / 256;
        if (b > (uint64_t)sm_count * 16) b = (uint64_t)sm_count * 16;
        blocks += b;
    }
    if (A.n_parts == 0) return (int)cudaSuccess;
    A.b1 = b1;
    A.b2 = b2;
    A.eps = eps;
    A.bc1 = (float)(1.0 - pow((double)b1, (double)step));
    A.bc2 = (float)(1.0 - pow((double)b2, (double)step));
    adam_parts_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(A);
    return (int)cudaGetLastError();
}

// Row-sparse Adam (Kingma & Ba) for the fine-tuning of Sec. 4.3: only the
// leaves whose mark is set (those the batch visited) are updated, as in a
// sparse-gradient Adam.  A warp takes 32 internal leaves at a time: one
// coalesced read of perm and one gather of the marks decide, by ballot, which
// of them it updates.  Marked rows go LEAF_ADAM_ROWS at a time (all their
// loads in flight together), lanes across each row's elements; every row gets
// the Adam step, goes back into the FP32 records at its internal slot, and
// has its gradient row and mark cleared for the next batch.

constexpr int LEAF_ADAM_CHUNK = 96;   // row elements per unrolled pass
constexpr int LEAF_ADAM_ROWS = 2;     // marked rows processed together

__global__ void __launch_bounds__(256, 4) leaf_adam_kernel(const __grid_constant__ LeafAdamParams p)
{
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
    const int nc = p.n1 + 27 * p.n2;
    constexpr int PER = LEAF_ADAM_CHUNK / 32;
    for (uint32_t base = warp * 32; base < p.n_leaves; base += n_warps * 32) {
        const uint32_t i = base + lane;
        uint32_t id = 0;
        bool marked = false;
        if (i < p.n_leaves) {
            id = __ldg(p.perm + i);
            marked = p.leaf_mark[id] != 0;
        }
        uint32_t todo = __ballot_sync(0xffffffffu, marked);
        while (todo) {
            uint32_t leaf[LEAF_ADAM_ROWS];
            size_t at[LEAF_ADAM_ROWS];
            bool have[LEAF_ADAM_ROWS];
#pragma unroll
            for (int r = 0; r < LEAF_ADAM_ROWS; ++r) {
                have[r] = todo != 0;
                const int src = have[r] ? __ffs(todo) - 1 : 0;
                todo &= todo - 1;
                leaf[r] = base + src;
                at[r] = (size_t)__shfl_sync(0xffffffffu, id, src) * nc;
            }
            for (int j0 = 0; j0 < nc; j0 += LEAF_ADAM_CHUNK) {
                float g[LEAF_ADAM_ROWS][PER], m[LEAF_ADAM_ROWS][PER], v[LEAF_ADAM_ROWS][PER],
                    w[LEAF_ADAM_ROWS][PER];
#pragma unroll
                for (int r = 0; r < LEAF_ADAM_ROWS; ++r)
#pragma unroll
                    for (int jj = 0; jj < PER; ++jj) {
                        const int j = j0 + lane + 32 * jj;
                        if (have[r] && j < nc) {
                            g[r][jj] = p.grad[at[r] + j];
                            m[r][jj] = p.m[at[r] + j];
                            v[r][jj] = p.v[at[r] + j];
                            w[r][jj] = p.param[at[r] + j];
                        }
                    }
#pragma unroll
                for (int r = 0; r < LEAF_ADAM_ROWS; ++r)
#pragma unroll
                    for (int jj = 0; jj < PER; ++jj) {
                        const int j = j0 + lane + 32 * jj;
                        if (have[r] && j < nc) {
                            const float mm = p.beta1 * m[r][jj] + (1.0f - p.beta1) * g[r][jj];
                            const float vv = p.beta2 * v[r][jj] + (1.0f - p.beta2) * g[r][jj] * g[r][jj];
                            const float ww = w[r][jj] - p.lr * (mm / p.bc1) / (sqrtf(vv / p.bc2) + p.eps);
                            p.m[at[r] + j] = mm;
                            p.v[at[r] + j] = vv;
                            p.param[at[r] + j] = ww;
                            p.grad[at[r] + j] = 0.0f;
                            if (j < p.n1) p.sig[(size_t)leaf[r] * p.sig_stride + j] = ww;
                            else p.zc[(size_t)leaf[r] * p.z_stride + (j - p.n1)] = ww;
                        }
                    }
            }
        }
        if (marked) p.leaf_mark[id] = 0;
    }
}

// The same step with the batch's gradient as a list of visits (and, for the
// leaves with a mark, the rows of grad too): a row's gradient is summed over
// its leaf's first VL_SLOTS visits in registers, so for most leaves no gradient
// row is written, read or cleared: 7 row transfers per updated leaf instead of
// 9, and none in the adjoint.  The visits past those are in the rows of grad
// before this kernel runs (grad_scatter_kernel).  Compile-time sizes: those of the adjoint.  A warp has one whole
// row in flight, and four CTAs share an SM: 0.97 ms for 0.86M rows of the
// 3.5M-leaf body (4.1 TB/s of randomly placed rows, what a plain random
// read-add-write reaches); two rows of 96 elements at three CTAs 1.25 ms.
template <int N1, int N2>
__global__ void __launch_bounds__(256, 4) leaf_adam_visits_kernel(const __grid_constant__ LeafAdamParams p)
{
    constexpr int NZ = 9 * N2, NC = N1 + 27 * N2, PER = (NC + 31) / 32;
    constexpr uint32_t NONE = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
    const VisitList &L = p.list;
    for (uint32_t base = warp * 32; base < p.n_leaves; base += n_warps * 32) {
        const uint32_t i = base + lane;
        uint32_t id = 0, visits = 0;
        bool marked = false;
        if (i < p.n_leaves) {
            id = __ldg(p.perm + i);
            visits = min(L.visits[id], VL_SLOTS);
            marked = p.leaf_mark[id] != 0;
        }
        // every lane fetches its own leaf's first visit: one latency for the warp
        uint4 slot = make_uint4(NONE, NONE, NONE, NONE);
        if (visits) slot = L.slot[id];
        uint32_t ray = 0;
        float4 val = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (slot.x != NONE) {
            ray = L.id[slot.x].y;
            val = L.val[slot.x];
        }
        for (uint32_t todo = __ballot_sync(0xffffffffu, marked || visits); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const uint32_t leaf = base + src;
            const size_t at = (size_t)__shfl_sync(0xffffffffu, id, src) * NC;
            const bool listed = __shfl_sync(0xffffffffu, slot.x, src) != NONE, dense = __shfl_sync(0xffffffffu, marked, src);
            const uint32_t n = __shfl_sync(0xffffffffu, visits, src);
            const float *w0 = L.w + (size_t)__shfl_sync(0xffffffffu, ray, src) * (N1 + NZ);
            const float4 c = make_float4(__shfl_sync(0xffffffffu, val.x, src), __shfl_sync(0xffffffffu, val.y, src),
                                         __shfl_sync(0xffffffffu, val.z, src), __shfl_sync(0xffffffffu, val.w, src));
            auto pick = [](const float4 &x, int jz) { return jz < 0 ? x.x : (jz < NZ ? x.y : (jz < 2 * NZ ? x.z : x.w)); };
            float g[PER], m[PER], v[PER], w[PER];
            // every load of the row first, the weights of its first visit among them
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int j = 32 * r + lane, jz = j - N1;
                g[r] = 0.0f;
                if (j < NC) {
                    m[r] = p.m[at + j];
                    v[r] = p.v[at + j];
                    w[r] = p.param[at + j];
                    if (listed) g[r] = __ldg(w0 + (jz < 0 ? j : N1 + jz % NZ));
                }
            }
#pragma unroll
            for (int r = 0; r < PER; ++r) g[r] *= pick(c, 32 * r + lane - N1);
            for (uint32_t k = 1; k < n; ++k) {  // the leaf's other visits
                const uint32_t e = __shfl_sync(0xffffffffu, k == 1 ? slot.y : (k == 2 ? slot.z : slot.w), src);
                if (e == NONE) continue;
                const float *wr = L.w + (size_t)L.id[e].y * (N1 + NZ);
                const float4 x = L.val[e];
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const int j = 32 * r + lane, jz = j - N1;
                    if (j < NC) g[r] = fmaf(pick(x, jz), __ldg(wr + (jz < 0 ? j : N1 + jz % NZ)), g[r]);
                }
            }
            if (dense) {
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const int j = 32 * r + lane;
                    if (j < NC) {
                        g[r] += p.grad[at + j];
                        p.grad[at + j] = 0.0f;
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int j = 32 * r + lane;
                if (j < NC) {
                    const float mm = p.beta1 * m[r] + (1.0f - p.beta1) * g[r];
                    const float vv = p.beta2 * v[r] + (1.0f - p.beta2) * g[r] * g[r];
                    const float ww = w[r] - p.lr * (mm / p.bc1) / (sqrtf(vv / p.bc2) + p.eps);
                    p.m[at + j] = mm;
                    p.v[at + j] = vv;
                    p.param[at + j] = ww;
                    if (j < N1) p.sig[(size_t)leaf * p.sig_stride + j] = ww;
                    else p.zc[(size_t)leaf * p.z_stride + (j - N1)] = ww;
                }
            }
        }
        if (marked) p.leaf_mark[id] = 0;
        if (visits) L.visits[id] = 0u;
    }
    // the last warp empties the list
    if (lane == 0) {
        __threadfence();
        if (atomicAdd(L.count + 1, 1u) == n_warps - 1) {
            atomicExch(L.count, 0u);
            atomicExch(L.count + 1, 0u);
            atomicExch(L.count + 2, 0u);
        }
    }
}

int launch_leaf_adam(const LeafAdamParams &p, int sm_count, void *stream)
{
    if (p.n_leaves == 0) return (int)cudaSuccess;
    uint64_t blocks = ((uint64_t)p.n_leaves + 255) / 256;
    if (blocks > (uint64_t)sm_count * 8) blocks = (uint64_t)sm_count * 8;
    if (p.list.cap) {
        const int ce = launch_grad_scatter_over(p.list, p.n1, p.n2, p.grad, p.leaf_mark, sm_count, stream);
        if (ce != cudaSuccess) return ce;
        auto go = [&](auto kern) {
            kern<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(p);
            return (int)cudaGetLastError();
        };
        if (p.n1 == 31 && p.n2 == 5) return go(leaf_adam_visits_kernel<31, 5>);
        if (p.n1 == 11 && p.n2 == 5) return go(leaf_adam_visits_kernel<11, 5>);
        if (p.n1 == 21 && p.n2 == 5) return go(leaf_adam_visits_kernel<21, 5>);
        if (p.n1 == 31 && p.n2 == 11) return go(leaf_adam_visits_kernel<31, 11>);
        return (int)cudaErrorInvalidValue;  // (the adjoint makes no list for other sizes)
    }
    leaf_adam_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(p);
    return (int)cudaGetLastError();
}


}  // namespace fpo

using namespace fpo;

extern "C" int fpo_decoder_grad(const fpo_mlp *w, int32_t n1, int32_t n2, uint32_t batch, const uint32_t *rows,
                                const float *latents, const float *targets, const float *coef_weight,
                                const float *extra_dy, const fpo_mlp *grad, float *dlatents, double *loss,
                                void *cuda_stream)
{
    if (!w || !grad) return set_last_error(FPO_ERR_INVALID_ARG, "NULL weights");
    if (n1 < 1 || n2 < 1 || n1 + 27 * n2 > decoder_grad_max_coeffs())
        return set_last_error(FPO_ERR_INVALID_ARG, "n1 + 27 n2 must be in [28, 176]");
    if (batch == 0) return FPO_OK;
    if (!rows || !latents || !targets || !coef_weight || !dlatents)
        return set_last_error(FPO_ERR_INVALID_ARG, "NULL array");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    DecoderGradParams p{};
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
    p.nc = n1 + 27 * n2;
    const int ce = launch_decoder_grad(p, sms, cuda_stream);
    if (ce != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString((cudaError_t)ce));
    return FPO_OK;
}

extern "C" int fpo_decoder_forward(const fpo_mlp *w, int32_t n1, int32_t n2, uint32_t n, const float *latents,
                                   float *coeffs, void *cuda_stream)
{
    if (!w || !w->w1 || !w->b1 || !w->w2 || !w->b2 || !w->w3 || !w->b3)
        return set_last_error(FPO_ERR_INVALID_ARG, "NULL weights");
    if (n1 < 1 || n2 < 1 || n1 + 27 * n2 > DF_MAXC) return set_last_error(FPO_ERR_INVALID_ARG, "n1 + 27 n2 must be in [28, 176]");
    if (n == 0) return FPO_OK;
    if (!latents || !coeffs) return set_last_error(FPO_ERR_INVALID_ARG, "NULL array");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    const int ce = launch_decoder_forward(*w, n1 + 27 * n2, n, latents, coeffs, sms, cuda_stream);
    if (ce != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString((cudaError_t)ce));
    return FPO_OK;
}

extern "C" int fpo_camera_ray_batch(const float *basis, const int64_t *cam, const int64_t *pixel, const int64_t *frame,
                                    uint32_t n, uint32_t width, uint32_t height, double fov_y_deg, float *o, float *d,
                                    float *t, void *cuda_stream)
{
    if (n == 0) return FPO_OK;
    if (!basis || !cam || !pixel || !frame || !o || !d || !t) return set_last_error(FPO_ERR_INVALID_ARG, "NULL array");
    if (width == 0 || height == 0) return set_last_error(FPO_ERR_INVALID_ARG, "width and height must be > 0");
    const float th = (float)tan(fov_y_deg * (3.14159265358979323846 / 180.0) / 2.0);
    ray_batch_kernel<<<(n + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(basis, cam, pixel, frame, n, (int64_t)width,
                                                                              (float)width, 1.0f / (float)width,
                                                                              1.0f / (float)height, th, o, d, t);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    return FPO_OK;
}

extern "C" int fpo_adam_parts(const fpo_adam_part *parts, uint32_t n_parts, float beta1, float beta2, float eps,
                              uint32_t step, void *cuda_stream)
{
    if (n_parts > ADAM_MAX_PARTS) return set_last_error(FPO_ERR_INVALID_ARG, "at most 8 arrays");
    if (n_parts && !parts) return set_last_error(FPO_ERR_INVALID_ARG, "parts is NULL");
    uint64_t n = 0;
    for (uint32_t k = 0; k < n_parts; ++k) {
        const fpo_adam_part &q = parts[k];
        if (q.n == 0) continue;
        n += q.n;
        if (!q.param || !q.grad || !q.m || !q.v) return set_last_error(FPO_ERR_INVALID_ARG, "NULL array");
        if (q.rows && q.dim == 0) return set_last_error(FPO_ERR_INVALID_ARG, "dim must be > 0 with rows");
    }
    if (n == 0) return FPO_OK;
    if (step < 1) return set_last_error(FPO_ERR_INVALID_ARG, "step counts from 1");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString(e));
    const int ce = launch_adam(parts, n_parts, beta1, beta2, eps, step, sms, cuda_stream);
    if (ce != cudaSuccess) return set_last_error(FPO_ERR_CUDA, cudaGetErrorString((cudaError_t)ce));
    return FPO_OK;
}

extern "C" int fpo_adam(float *param, const float *grad, float *m, float *v, uint64_t n, const uint32_t *rows,
                        uint32_t dim, float lr, float beta1, float beta2, float eps, uint32_t step, void *cuda_stream)
{
    const fpo_adam_part q = {param, const_cast<float *>(grad), m, v, n, rows, dim, lr, 1.0f};  // (scale 1: grad is read only)
    return fpo_adam_parts(&q, 1, beta1, beta2, eps, step, cuda_stream);
}
