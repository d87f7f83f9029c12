// Internal declarations shared by the host packer, the ABI layer and the
// CUDA kernels of the FPO renderer.  Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include <cuda.h>  // CUtensorMap (a header type; nothing links the driver library)
#include <vector_types.h>

#include "fpo.h"

namespace fpo {

// ---------------------------------------------------------------------------
// Node array (breadth-first).  One node = 8 child slots of 32 bits = 32 bytes,
// one L2 sector.  Slot values: 0 = empty space, LEAF_BIT | i = leaf with
// internal index i, otherwise the index (>= 1) of an internal child node.
// The root is node 0 and is never referenced from a slot; its own kind is
// passed separately (ROOT_*).  Child c of a node covers the octant with
// bit 0 = x, bit 1 = y, bit 2 = z of the next level's coordinates.
constexpr uint32_t LEAF_BIT = 0x80000000u;
constexpr uint32_t ROOT_EMPTY = 0, ROOT_LEAF = 1, ROOT_NODE = 2;
constexpr int MAX_DEPTH = 12;

// Brick index, for trees whose leaves are all finest cells (every union octree
// of fully divided frames), 4 <= depth <= 11: the finest grid as 4x4x4 bricks,
// grouped 4x4x4 again into 16^3-cell blocks.  Bit x + 4y + 16z of a 64-bit mask
// stands for child (x, y, z).  Both records are 16 bytes:
//   top[block], a dense grid of blocks, x fastest: {mask of its non-empty
//     bricks (low, high), index of the first of them, side of the octree's
//     largest empty cube around it if the mask is 0};
//   bricks[i], in the order of the mask bits: {mask of its leaves (low, high),
//     first leaf, 0}.
// A brick's leaves are numbered in the order of its mask bits.  The cubes found
// in it (leaf, empty 1, 2, 4, 8, 16, ...) are the octree's.  The 3.5M-leaf body
// takes 0.5 + 1 MB, its node array 17 MB.
constexpr int BRICK_MIN_DEPTH = 4, BRICK_MAX_DEPTH = 11;
// The top grid is dense, 16 bytes a block: a tree gets the index when that is at
// most 256 bytes a leaf (the coefficient records take 672 at n1 = 31, n2 = 5), or
// 64 KB; sparser trees of depth 9 to 11 keep the octree walk.  Blocks a leaf, with
// n1 = n2 = 1, upload in ms without and with it and an 800x800 frame in us: depth
// 9, 6.0: 0.47 / 0.80, 126 / 92; 10, 6.0: 3.7 / 6.0, 223 / 156; 11, 6.0: 28 / 51,
// 507 / 323; 10, 48: 0.56 / 1.4, 125 / 88; 11, 48: 4.3 / 10.9, 212 / 143.  Ten
// leaves at depth 11 took 22 ms to pack and 33 MB.
constexpr bool brick_index_fits(uint64_t n_leaves, int depth)
{
    return (1ull << (3 * (depth - 4))) <= (n_leaves > 256 ? 16 * n_leaves : 4096);
}

// Leaf records.  FP32 storage: a density record of SIG_STRIDE(n1) floats
// (n1 rounded up to a multiple of 4, 128 bytes for n1 = 31) and an SH record
// of Z_STRIDE(n2) floats (27 n2 rounded up to a multiple of 4), both arrays
// indexed by internal leaf index (breadth-first order, siblings adjacent).
inline int sig_stride(int n1) { return (n1 + 3) & ~3; }
inline int z_stride(int n2) { return (27 * n2 + 3) & ~3; }

// Stored record layout for any storage precision: element counts padded so
// that each record is a multiple of 16 bytes (bulk-copy granularity).  FP32
// gives sig_stride / z_stride above.  FP8 adds one FP32 scale per leaf in a
// separate array (codes are coefficient / scale).
struct RecordLayout {
    int sig_elems, z_elems, elem_bytes;
    bool scaled;
    int sig_bytes() const { return sig_elems * elem_bytes; }
    int z_bytes() const { return z_elems * elem_bytes; }
};
inline RecordLayout record_layout(int storage, int n1, int n2)
{
    const int eb = storage == FPO_STORAGE_F32 ? 4 : (storage == FPO_STORAGE_FP8_E4M3 ? 1 : 2);
    const int per16 = 16 / eb;
    RecordLayout L;
    L.elem_bytes = eb;
    L.sig_elems = (n1 + per16 - 1) / per16 * per16;
    L.z_elems = (27 * n2 + per16 - 1) / per16 * per16;
    L.scaled = storage == FPO_STORAGE_FP8_E4M3;
    return L;
}

// Host encoders (round to nearest even) from the format definitions:
// bfloat16 (1-8-7), IEEE binary16 (1-5-10, overflow to infinity) and
// FP8 E4M3 (1-4-3, bias 7, no infinities, saturating at +-448).
uint16_t encode_bf16(float x);
uint16_t encode_f16(float x);
uint8_t encode_e4m3(float x);

// Per-frame IDFT table: one 128-byte record per leaf,
// [sigma(t) clamped at 0, z_{c,k}(t) for c = 0..2, k = 0..8 (27 values), 4 zeros].
constexpr int TABLE_STRIDE = 32;

// Camera rays are scheduled in warp tiles of TILE_W x TILE_H pixels.
#ifndef FPO_TILE_W
#define FPO_TILE_W 4
#endif
constexpr int TILE_W = FPO_TILE_W, TILE_H = 32 / FPO_TILE_W;
static_assert(TILE_W * TILE_H == 32, "a tile is one warp of rays");

// Device status word bits.
constexpr uint32_t STATUS_TRAVERSAL_LIMIT = 1u, STATUS_VISIT_OVERFLOW = 2u, STATUS_DEVICE_TIMEOUT = 4u,
                   STATUS_FP16_RANGE = 8u;
// Limit of the waits that FPO_FLAG_TEST_DEVICE_TIMEOUT makes run out: 1 ms.
constexpr uint64_t TEST_WAIT_LIMIT_NS = 1000000ull;

struct PackedTree {
    uint32_t root_kind = ROOT_EMPTY;
    int depth = 0;                 // grid depth D: finest cell = 1 / 2^D of the cube
    std::vector<uint32_t> nodes;   // [n_nodes * 8]
    std::vector<uint32_t> perm;    // internal leaf index -> upload index
    std::vector<uint32_t> top, bricks;  // brick index, 4 words per entry (empty: none)
};

// Validates a tree description (and packs it when `out` is non-null).
// Returns FPO_OK, FPO_ERR_INVALID_ARG or FPO_ERR_BAD_TREE (message in *err).
int validate_and_pack(const fpo_tree_desc *tree, int n1, int n2, PackedTree *out,
                      std::string *err,
                      bool any_density = true);

// ---------------------------------------------------------------------------
// Kernel parameters.

struct FrameParams {
    int mode;                 // FPO_RAYS_*
    uint32_t width, height, n_rays;
    uint32_t y0, rows;        // camera: the rows of this launch, y0 .. y0 + rows - 1 (its rays are numbered from 0)
    double eye[3], target[3], up[3];
    double fov_y_deg;
    double t, period_T;
    const float *ro, *rd, *rt; // explicit rays (device)
};

// What every CTA of a frame's kernels would otherwise derive in FP64 for
// itself: Eq. 8 at the frame time and the camera frame, computed once per call
// on the host in FP64 and rounded to FP32 (the GPU's FP64 rate made the
// kernels' own prologue some microseconds long).
struct FrameConsts {
    float b[32];                     // IDFT_i(t), i < max(n1, n2); 0 beyond
    float f[3], r[3], u[3], eye[3];  // camera: forward, right, up, eye
    float sx_scale, sy_scale;        // tan(fov / 2) times the aspect ratio, and plain
};
// cos(pi x), or sin(pi x) with `sine`, on the host.
double cospi_h(double x, bool sine);
// Eq. 8 at time t for i < n into b (32 values, zero from n on).
void time_basis(double t, double period_T, int n, float b[32]);

struct TraverseParams {
    FrameParams fr;
    FrameConsts fc;
    // tree
    const uint32_t *nodes;
    const uint4 *top, *bricks; // brick index (nullptr: leaves at several depths, or a very shallow or deep tree)
    int top_bits;              // log2 of the top grid's cells a side
    uint32_t root_kind;
    int depth;
    float grid_scale;         // 2^D / aabb_size
    float amin[3];
    double grid_scale64, amin64[3];  // the same in FP64 (gradient-check replay)
    // leaf data
    const float4 *table;      // per-frame IDFT table (materialised mode)
    int half_table;           // the table holds FP16 (64-byte lines) instead of FP32 (128-byte lines)
    const float4 *sig;        // density coefficient records (fused mode)
    const float *zc;          // SH coefficient records (fused mode)
    int n1, n2, sig_stride4, z_stride;
    // options and outputs
    float bg[3];
    float stop_T;
    uint32_t flags;
    float *out_rgb;
    float *out_T;
    uint32_t *visit_log;
    uint32_t visit_cap;
    uint32_t *visit_count;
    uint8_t *leaf_mark;
    const uint32_t *perm;
    // scheduling
    uint32_t *status;         // status bits (atomicOr)
    uint32_t *tiles;          // [0] tile counter, [1] finished warps (reset by the last warp)
    uint32_t n_tiles, tiles_x;
    uint32_t max_steps;
    uint32_t refill_min;      // warp refills its idle lanes once this many are idle (32: whole tiles)
    uint32_t inner_steps;     // steps a lane takes between two refill checks
    int block_threads;        // 128 or 256
    int few_tiles_split;      // 1: smaller CTAs when there are few tiles (block_threads is not the user's choice)
    int form;                 // fused mode: ray_form
    const uint32_t *coherent; // LANES_IF_COHERENT: coherence_kernel's answer for this call, else nullptr
    int rays_per_warp, list_cap; // fused mode: rays of one warp and length of its visit list (set by the launcher)
    int max_ctas_per_sm;      // 0: as many as fit
    int carveout;             // preferred shared-memory carveout in percent (0: the driver's default)
    unsigned long long *stats; // FPO_FLAG_STATS: [steps, leaf visits, rays entering the tree]
};

// Ray k (0..31) of a tile: a camera pixel of a TILE_W x TILE_H block, or an
// explicit ray.
__host__ __device__ __forceinline__ bool tile_ray(const TraverseParams &p, uint32_t tile, uint32_t k, uint32_t &ray,
                                                  int &px, int &py)
{
    if (p.fr.mode == FPO_RAYS_CAMERA) {
        // row-major tiles: the tiles in flight form one band of rows, whose
        // table lines stay in L2
        const uint32_t tx = tile % p.tiles_x, ty = tile / p.tiles_x;
        const uint32_t row = ty * TILE_H + k / TILE_W;
        px = (int)(tx * TILE_W + k % TILE_W);
        py = (int)(p.fr.y0 + row);
        ray = row * p.fr.width + (uint32_t)px;
        return px < (int)p.fr.width && row < p.fr.rows;
    }
    ray = tile * 32 + k;
    return ray < p.fr.n_rays;
}

// The queue of the fused mode holds single rays, counted in 32 bits: slot
// 32 tile + k is ray k of a tile.  Of a camera frame a few pixels wide or high
// the tiles are mostly empty slots, up to 32 a pixel; when they would pass
// 2^31 the frame is taken pixel by pixel instead (tiles_x = 0), so that the
// slots, and what the warps count past them, always fit.
inline void fused_queue(TraverseParams &p)
{
    if (p.fr.mode != FPO_RAYS_CAMERA || p.n_tiles < (1u << 26)) return;
    p.tiles_x = 0;
    p.n_tiles = (p.fr.n_rays + 31) / 32;
}
__host__ __device__ __forceinline__ bool slot_ray(const TraverseParams &p, uint32_t slot, uint32_t &ray, int &px, int &py)
{
    if (p.fr.mode != FPO_RAYS_CAMERA || p.tiles_x) return tile_ray(p, slot >> 5, slot & 31u, ray, px, py);
    ray = slot;
    px = (int)(slot % p.fr.width);
    py = (int)(p.fr.y0 + slot / p.fr.width);
    return slot < p.fr.n_rays;
}

struct MaterialiseParams {
    const void *sig;          // [n_leaves] records of sig_stride elements
    const void *zc;           // [n_leaves] records of z_stride elements
    const float *scale;       // [n_leaves] (FP8 storage) or nullptr
    float *table;             // [n_leaves][32] FP32, or [n_leaves][32] FP16 when half_table
    int half_table;
    uint32_t n_leaves;
    int storage;              // FPO_STORAGE_*
    int n1, n2, sig_stride, z_stride;  // strides in elements
    int stages;               // shared-memory pipeline depth (materialise_stages)
    int pipeline;             // 1: the frame-pipeline shape (materialise_pipeline_shape)
    int max_ctas_per_sm;      // 0: as many as fit
    int carveout;             // preferred shared-memory carveout in percent (0: the driver's default)
    float b[32];              // Eq. 8 at the frame time (time_basis)
    uint32_t *status;
    int test_timeout;         // 1: the first wait of each CTA gives up (failure-path test)
};

// Read-only view of a context's uploaded tree and launch settings.
struct CtxView {
    int device, sm_count;
    int n1, n2;
    double period_T;
    int traverse_threads, refill_min, inner_steps, max_steps;
    uint32_t *d_status;
    bool half_table;
    bool has_tree;
    uint32_t n_leaves, n_nodes, root_kind;
    int depth;
    double aabb_min[3], aabb_size;
    const uint32_t *d_nodes, *d_perm;
    int storage;
    const void *d_sig, *d_z;
    const float *d_scale;
};
CtxView ctx_view(const fpo_ctx *ctx);
// Records `msg` as the calling thread's last error; returns `code`.
int set_last_error(int code, const char *msg);

// Argument checks shared by the render entry points (FPO_OK or the status
// they recorded): the rays (camera validity, finite t, ray count), and the
// options and output of one render.
int check_rays(const fpo_rays *r, uint64_t *n_rays);
int check_render_opts(const fpo_ctx *ctx, const fpo_frame_opts *opts, uint64_t n_rays, const float *out_rgb);
// Kernel parameters of one render (or adjoint) call; p.table is the context's
// own per-frame table, which a caller may point elsewhere.
TraverseParams traverse_params(const fpo_ctx *ctx, const fpo_rays *rays, const fpo_frame_opts *opts,
                               float *out_rgb, uint64_t n_rays, uint32_t y0 = 0);
// The per-frame table for time t into `table` on `stream`: the tensor-core
// decoder for LATENT storage, else the IDFT pass over the stored coefficients
// (at most max_ctas_per_sm CTAs per SM when > 0; with pipe_stages > 0 the
// frame-pipeline shape with that many stages and the given carveout).
// Returns a cudaError_t.
// test_timeout: the failure-path test of FPO_FLAG_TEST_DEVICE_TIMEOUT.
int launch_table_pass(const fpo_ctx *ctx, double t, float *table, int max_ctas_per_sm, void *stream,
                      int pipe_stages, int carveout, bool test_timeout);

// Latent decoder (per-leaf FP16 latents, MLP 32 -> 64 -> 64 -> n1 + 27 n2,
// ReLU).  Weights are BF16 bit patterns, row-major [out][in]; biases FP32.
struct LatentParams {
    const uint16_t *latents;  // FP16 [n_leaves][32]
    const uint16_t *w1;       // [64][32]
    const float *b1;          // [64]
    const uint16_t *w2;       // [64][64]
    const float *b2;          // [64]
    const uint16_t *w3;       // [n1 + 27 n2][64]
    const float *b3;          // [n1 + 27 n2]
    int n1, n2;
    float b[32];              // Eq. 8 at the frame time (time_basis)
    uint32_t n_leaves;
    float *table;             // [n_leaves][TABLE_STRIDE] FP32, or FP16 when half_table
    int half_table;
    uint32_t *status;
    int test_timeout;         // 1: each warpgroup's first wait gives up (failure-path test)
    int pipeline;             // 1: the frame-pipeline shape (one 256-thread CTA per SM)
    int carveout;             // preferred shared-memory carveout in percent (0: the driver's default)
    CUtensorMap table_map;    // set by launch_latent_table: the table as a [n_leaves][32] tensor
};

int launch_latent_table(const LatentParams &p, int sm_count, void *stream);
int latent_pipeline_smem_bytes();  // dynamic shared memory of the pipeline-shape decoder CTA

struct DecoderGradParams {
    fpo_mlp w, g;             // FP32 weights; gradients (accumulated)
    const uint32_t *rows;     // [batch] leaf rows (distinct)
    uint32_t batch;
    const float *latents;     // [N][32]
    const float *targets;     // [N][nc]
    const float *coef_weight; // [nc]
    const float *extra_dy;    // [N][nc] or nullptr
    float *dlatents;          // [batch][32]
    double *loss;             // accumulated, or nullptr
    int nc;
};
int launch_decoder_grad(const DecoderGradParams &p, int sm_count, void *stream);
int launch_gather_rows(const void *src, void *dst, const uint32_t *perm, uint32_t n, uint32_t bytes,
                       int sm_count, void *stream);
int decoder_grad_max_coeffs();
int launch_decoder_forward(const fpo_mlp &w, int nc, uint32_t n, const float *latents, float *out, int sm_count,
                           void *stream);
int launch_decode_records(const fpo_mlp &w, int n1, int n2, uint32_t n, const float *latents, const uint32_t *perm,
                          float *sig, float *zc, int sm_count, void *stream);
// The same on the tensor cores with the inference decoder's FP16 numerics
// (fpo_latent.cu); FP16-range and time-out reports go to *status.
int launch_decode_records_tc(const fpo_mlp &w, int n1, int n2, uint32_t n, const float *latents, const uint32_t *perm,
                             float *sig, float *zc, uint32_t *status, bool test_timeout, int sm_count, void *stream);
int launch_adam(const fpo_adam_part *parts, uint32_t n_parts, float b1, float b2, float eps, uint32_t step, int sm_count,
                void *stream);

// Deferred visits that a leaf Adam step sums for one leaf, one after another.
// A leaf's later ones are added to its gradient row first, evenly divided: a
// coarse leaf in front of the cameras can have thousands (65,536 rays on 0.3M
// leaves, one of them 64 cells wide: 6.0 ms a step with the visits of every
// leaf in one chain, 0.88 now).  Three slots beside the count in one 16-byte
// word send so many more visits of the 3.5M-leaf body the other way that its
// step takes 1.93 instead of 1.81 ms.
constexpr uint32_t VL_SLOTS = 4;

// Visits of an adjoint call, kept for a second pass (a workspace of the
// context): what a visit adds to the gradient row of its leaf is the outer
// product of 4 numbers (dL/dsigma_raw and dL/du_c) and its ray's weights.
struct VisitList {
    uint32_t cap;             // entries; 0: no list
    uint32_t *count;          // [0] entries appended (may exceed cap), [1] finished warps of the pass over them, [2] in `over`
    uint2 *id;                // upload leaf id, ray (ray_base + index in the call)
    float4 *val;
    uint32_t *visits;         // deferred gradients: per leaf, its visits so far
    uint4 *slot;              // ... the entries of the first VL_SLOTS of them (~0: not in the list); else nullptr
    uint32_t *over;           // ... and the entries of all later ones, any leaf's
    float *w;                 // [rays][n1 + 9 n2]: IDFT_i(t), then Y_k(d) IDFT_i(t)
    uint32_t ray_base;
};

struct BackwardParams {
    VisitList list;
    TraverseParams tp;          // rays, tree and options as for the fused forward
    const float *out_rgb;       // forward colour [rays][3]
    const float *dL_drgb;       // [rays][3]
    float *dL_dcoeffs;          // [n_leaves][n1 + 27 n2], canonical, upload order (accumulated)
    double *dL_dcoeffs64;       // the same in FP64 (gradient-check replay), else nullptr
    uint8_t *leaf_mark;         // optional [n_leaves] (upload order): set to 1 for every visited leaf
};

// Row-sparse Adam over the coefficients of the leaves a batch visited, fused
// with the write-back into the FP32 records and the reset of their gradient
// rows and marks.
struct LeafAdamParams {
    float *param, *grad, *m, *v;  // [n_leaves][nc], canonical, upload order
    uint8_t *leaf_mark;           // [n_leaves], upload order
    const uint32_t *perm;         // internal leaf -> upload id
    float *sig, *zc;              // FP32 records (internal order)
    uint32_t n_leaves;
    int n1, n2, sig_stride, z_stride;
    float lr, beta1, beta2, eps, bc1, bc2;  // bc = 1 - beta^step
    VisitList list;               // the deferred gradient (cap 0: none)
};

// Launchers (return cudaError_t as int).
int launch_materialise(const MaterialiseParams &p, int sm_count, void *stream);
int materialise_stages(int storage, int n1, int n2);
// Shape of the IDFT pass when it shares each SM with the traversal (frame
// pipeline): CTAs per SM and stages such that the CTAs of one SM hold at most
// smem_budget bytes of records; smem_per_cta is the dynamic shared memory.
struct MatShape {
    int ctas_per_sm, stages, smem_per_cta;
};
MatShape materialise_pipeline_shape(int storage, int n1, int n2, int smem_budget);
int materialise_smem_bytes(const MaterialiseParams &p);  // dynamic shared memory of one CTA
// (form LANES_IF_COHERENT: asks, and launches the lanes' kernel only; the parts by
// warps, with the same `coherent`, are the caller's)
int launch_backward(const BackwardParams &q, int sm_count, void *stream);
// Adds the list's visits to q.dL_dcoeffs and empties it.
int launch_grad_scatter(const BackwardParams &q, int sm_count, void *stream);
// Adds the visits in list.over to grad and sets their leaves' marks.
int launch_grad_scatter_over(const VisitList &list, int n1, int n2, float *grad, uint8_t *leaf_mark, int sm_count, void *stream);
int launch_dft(const float *values, float *coeffs, uint32_t n_leaves, int n1, int n2, int T, uint32_t *status,
               bool test_timeout, int sm_count, void *stream);
int launch_set_coeffs(const float *src, const uint32_t *perm, float *sig, float *zc, uint32_t n_leaves,
                      int n1, int n2, int sm_count, void *stream);
int launch_leaf_adam(const LeafAdamParams &p, int sm_count, void *stream);
int launch_traverse(const TraverseParams &p, bool materialised, bool debug, int sm_count,
                    void *stream);
int traverse_smem_bytes(bool brick, int threads);
// Whether the traversal walks the brick index; the compaction schedule
// (refill_min < 32, a tuning option) walks the octree of every tree.
constexpr bool brick_walk(bool has_index, uint32_t refill_min) { return has_index && refill_min >= 32; }
bool fused_supported(int n1, int n2);
// How the fused mode takes a call: by warps that evaluate their visits
// together, or with one lane a ray, each reading its visits' records by itself.
// The lanes are the faster way for many rays on a small tree and for whole
// images, where neighbours read the same records.  Camera frames are images;
// of explicit rays only their data tell (an image's rays in pixel order, or a
// random batch), so that large calls look at some of them on the device first
// (LANES_IF_COHERENT: coherence_kernel, and both forms launched, of which one
// returns at once: 5 us).  Forward, us, warps / lanes:
//   leaves       camera 640x400  800x800     1920x1080    image 800x800  random 400k  random 1M
//   2,252        106 /   70      265 /   97   545 /  150   293 /  130     281 /  254   660 /  574
//   5,430        111 /   78      267 /   97   545 /  148   294 /  130     271 /  291   636 /  654
//   41,929       181 /  201      394 /  221   722 /  304   433 /  271     381 /  461   878 / 1036
//   348,592      341 /  491      599 /  470  1064 /  561   640 /  557     565 / 1114  1278 / 2541
//   3,506,408    765 / 1216     1347 / 1381  2199 / 1726  1408 / 1473    1068 / 2432  2414 / 5540
// (an image of 400x400 explicit rays: 102 / 84, 104 / 94, 172 / 202 on the first
// three; 512x512: 141 / 91, 139 / 99, 225 / 210, 378 / 529.)
enum RayForm { BY_WARPS, BY_LANES, LANES_IF_COHERENT };
constexpr RayForm ray_form(bool camera, uint64_t rays, uint32_t n_leaves)
{
    if (n_leaves < 4096) return rays >= (1u << 17) ? BY_LANES : BY_WARPS;
    if (camera) {
        const uint64_t least = n_leaves < (1u << 15) ? 1u << 17 : (n_leaves < (1u << 17) ? 1u << 18 : 1u << 19);
        return rays >= least ? BY_LANES : BY_WARPS;
    }
    return rays >= (n_leaves < (1u << 17) ? 3u << 16 : 1u << 20) ? LANES_IF_COHERENT : BY_WARPS;
}

}  // namespace fpo
