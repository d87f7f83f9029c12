// The C ABI of the FPO renderer (include/fpo.h): context, tree upload,
// render dispatch and device status.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <limits>
#include <new>
#include <string>

#include "fpo_internal.h"

using namespace fpo;

namespace {

thread_local std::string g_err;

int fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    std::vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int cuda_fail(cudaError_t e, const char *what)
{
    return fail(e == cudaErrorMemoryAllocation ? FPO_ERR_OOM : FPO_ERR_CUDA, "%s: %s", what,
                cudaGetErrorString(e));
}

// Restores the caller's current device on scope exit.
struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        ok = cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

template <class T>
void dfree(T *&p)
{
    if (p) cudaFree((void *)p);
    p = nullptr;
}

// Launch shapes of the frame pipeline (fpo_render_frames).  The traversal of
// frame k and the IDFT pass of frame k + 1 share every SM: 768 traversal
// threads (64 registers each) leave a quarter of the register file to the
// IDFT pass (materialise_pipeline_shape: one 128-thread CTA of the
// thread-per-leaf form, or two 256-thread CTAs of the warp-cooperative form),
// whose stage rings are capped so that all CTAs' shared memory fits one
// carveout.  With the FP16 table the passes are short, and what counts is how
// soon the next traversal's warps take the places of the last ones: CTAs of
// two warps, and six tables in flight (BF16 frames 407 -> 381 us, latent
// 790 -> 766, FP8 views 231 -> 200; 128 threads 384 / 773 / 201, depth 8 the
// same).  The FP32-table frames, 4.72 ms for eight, gain from neither (4.87
// with CTAs of 64, 4.72 at depth 6).
#ifndef FPO_PIPE_TRAV_THREADS_F16
#define FPO_PIPE_TRAV_THREADS_F16 64
#endif
#ifndef FPO_PIPE_TRAV_CTAS_F16
#define FPO_PIPE_TRAV_CTAS_F16 12
#endif
#ifndef FPO_PIPE_DEPTH_F16
#define FPO_PIPE_DEPTH_F16 6
#endif
#ifndef FPO_PIPE_TRAV_THREADS
#define FPO_PIPE_TRAV_THREADS 384
#endif
#ifndef FPO_PIPE_TRAV_CTAS
#define FPO_PIPE_TRAV_CTAS 2
#endif
#ifndef FPO_PIPE_MAT_CTAS
#define FPO_PIPE_MAT_CTAS 0  // IDFT-pass CTAs per SM in the pipeline (0: materialise_pipeline_shape's choice)
#endif
#ifndef FPO_PIPE_DEPTH
// Tables (and traversal streams) in flight in fpo_render_frames, FP32 table.
#define FPO_PIPE_DEPTH 4
#endif
constexpr int PIPE_MAX = 8;
static_assert(FPO_PIPE_DEPTH >= 2 && FPO_PIPE_DEPTH <= PIPE_MAX && FPO_PIPE_DEPTH_F16 >= 2 && FPO_PIPE_DEPTH_F16 <= PIPE_MAX,
              "pipeline depth");
static_assert(1 + 2 * PIPE_MAX <= 24, "tile counters stay below the visit list's status words");
#ifndef FPO_PIPE_SLOT_STREAMS
#define FPO_PIPE_SLOT_STREAMS 1  // each pipeline slot's traversals on its own stream (0: all on the caller's)
#endif
#ifndef FPO_PIPE_MAT_SMEM_KB
#define FPO_PIPE_MAT_SMEM_KB 88
#endif
constexpr int PIPE_TRAV_THREADS = FPO_PIPE_TRAV_THREADS;
constexpr int PIPE_TRAV_CTAS = FPO_PIPE_TRAV_CTAS;
constexpr int PIPE_MAT_SMEM_BUDGET = FPO_PIPE_MAT_SMEM_KB * 1024;  // bytes of coefficient records in flight per SM
constexpr int PIPE_STATIC_SMEM = 512;            // allowance for each kernel's static shared memory
constexpr int SMEM_CONFIGS_KB[] = {0, 8, 16, 32, 64, 100, 132, 164, 196, 228};  // per SM, sm_100 family
constexpr int DEFAULT_TRAVERSE_THREADS = 256;
constexpr uint32_t DEFAULT_REFILL_MIN = 32;
constexpr uint32_t DEFAULT_INNER_STEPS = 0xffffffffu;  // a lane runs its ray to the end

// Visit list of an adjoint call: batches of up to VL_MAX_RAYS rays, room for
// VL_PER_RAY visits a ray (the 3.5M-leaf body: 15 on average), counter words.
constexpr uint32_t VL_MAX_RAYS = 1u << 18, VL_PER_RAY = 32;
// The first VL_BASE_RAYS rays' list shares the allocation of the SH records: an
// allocation of its own took 130 to 220 us of a context's first adjoint, which
// for batches of this size and trees of some ten thousand leaves was more than
// the list had gained.
constexpr uint32_t VL_BASE_RAYS = 4096;
constexpr int VL_COUNT = 24, VL_COUNTS = 3;
constexpr int COHERENT_WORD = 28;  // coherence_kernel's answer

}  // namespace

struct fpo_ctx {
    fpo_config cfg{};
    int sm_count = 0;
    // [0] status bits; [1], [2] tile counter and finished warps of a traversal;
    // [1 + 2b], [2 + 2b] the same for slot b of fpo_render_frames, whose
    // traversals run on streams of their own; [24..26] the visit list's counters;
    // [28] whether a fused call's rays are coherent
    uint32_t *d_status = nullptr;
    // tree
    bool has_tree = false;
    uint32_t n_leaves = 0, n_nodes = 0, root_kind = ROOT_EMPTY;
    int depth = 0;
    uint32_t max_depth = 0;
    double aabb_min[3] = {0, 0, 0}, aabb_size = 1.0;
    uint32_t *d_nodes = nullptr;
    uint32_t *d_top = nullptr, *d_bricks = nullptr;  // brick index, or NULL
    uint32_t *d_perm = nullptr;
    void *d_sig = nullptr;    // density records (storage precision)
    void *d_z = nullptr;      // SH records (storage precision)
    float *d_scale = nullptr; // FP8: per-leaf scale, padded to a multiple of 4 leaves
    uint16_t *d_latents = nullptr;  // LATENT: FP16 [n_leaves][32], internal leaf order
    uint16_t *d_dec_w = nullptr;    // LATENT: w1 | w2 | w3 (BF16 bits)
    float *d_dec_b = nullptr;       // LATENT: b1 | b2 | b3
    bool has_latents = false;
    float *d_table = nullptr;
    size_t table_leaves = 0;
    // frame pipeline (fpo_render_frames): second table, aux stream, events
    bool half_table = false;  // the per-frame table holds FP16 (64 B per leaf)
    bool table_ok = false;    // d_table holds the IDFT pass of table_t for the current coefficients
    double table_t = 0.0;
    // slot b of the pipeline: frames b, b + depth, ... (slot 0: d_table, the caller's stream)
    float *d_ptables = nullptr;           // the tables of slots 1 .. ptable_slots, one after another
    int ptable_slots = 0;
    int pipe_cap = PIPE_MAX;              // slots that this tree's tables were found to leave memory for
    cudaStream_t aux = nullptr;           // IDFT passes / decodes
    cudaStream_t trav[PIPE_MAX] = {};     // slots 1.. : their traversal streams
    // visits of an adjoint call (VisitList), grown by visit_list
    unsigned char *vl_base = nullptr;   // room for VL_BASE_RAYS behind the SH records
    unsigned char *d_vl_block = nullptr;  // an allocation for more rays
    uint2 *d_vl_id = nullptr;
    float4 *d_vl_val = nullptr;
    uint32_t *d_vl_over = nullptr;
    uint4 *d_vl_slot = nullptr;         // per leaf: its deferred visits' entries, then in the same allocation
    uint32_t *d_vl_visits = nullptr;    // their number
    float *d_vl_w = nullptr;
    uint32_t vl_cap = 0, vl_rays = 0;   // entries; rays with room for weights
    uint32_t vl_used = 0;               // rays whose visits await fpo_adam_leaves
    cudaEvent_t ev_entry = nullptr, ev_mat[PIPE_MAX] = {}, ev_trav[PIPE_MAX] = {};

    // Bytes of a visit list for `rays` rays, and its arrays in a block of that size.
    size_t vl_bytes(uint32_t rays) const
    {
        return (size_t)rays * (VL_PER_RAY * (sizeof(float4) + sizeof(uint2) + sizeof(uint32_t)) +
                               ((size_t)cfg.n1 + 9 * (size_t)cfg.n2) * sizeof(float));
    }
    void set_visit_list(unsigned char *block, uint32_t rays)
    {
        const size_t e = block ? (size_t)rays * VL_PER_RAY : 0;
        d_vl_val = reinterpret_cast<float4 *>(block);
        d_vl_id = reinterpret_cast<uint2 *>(d_vl_val + e);
        d_vl_over = reinterpret_cast<uint32_t *>(d_vl_id + e);
        d_vl_w = reinterpret_cast<float *>(d_vl_over + e);
        vl_cap = (uint32_t)e;
        vl_rays = block ? rays : 0;
    }

    void free_tree()
    {
        dfree(d_vl_block);
        vl_base = nullptr;
        set_visit_list(nullptr, 0);
        dfree(d_vl_slot);
        d_vl_visits = nullptr;
        vl_used = 0;
        if (d_status) cudaMemset(d_status + VL_COUNT, 0, VL_COUNTS * sizeof(uint32_t));
        dfree(d_nodes);
        dfree(d_top);
        dfree(d_bricks);
        dfree(d_perm);
        dfree(d_sig);
        dfree(d_z);
        dfree(d_scale);
        dfree(d_latents);
        dfree(d_dec_w);
        dfree(d_dec_b);
        has_latents = false;
        dfree(d_table);
        table_leaves = 0;
        table_ok = false;
        dfree(d_ptables);
        ptable_slots = 0;
        pipe_cap = PIPE_MAX;
        has_tree = false;
    }
};

namespace fpo {

// Bytes of one leaf's row of the per-frame table.
static size_t table_row_bytes(const fpo_ctx *c) { return c->half_table ? TABLE_STRIDE * 2 : TABLE_STRIDE * 4; }
// Bytes of a per-frame table: rows rounded up to a multiple of 8 leaves, so
// that a prefetch of the aligned 512-byte group of rows holding any leaf
// stays inside the allocation.
static size_t table_alloc_bytes(const fpo_ctx *c) { return (((size_t)c->n_leaves + 7) & ~(size_t)7) * table_row_bytes(c); }

CtxView ctx_view(const fpo_ctx *c)
{
    CtxView v{};
    v.device = c->cfg.device;
    v.sm_count = c->sm_count;
    v.n1 = c->cfg.n1;
    v.n2 = c->cfg.n2;
    v.period_T = c->cfg.period_T;
    v.traverse_threads = c->cfg.traverse_threads;
    v.refill_min = c->cfg.refill_min;
    v.inner_steps = c->cfg.inner_steps;
    v.max_steps = c->cfg.max_steps;
    v.d_status = c->d_status;
    v.half_table = c->half_table;
    v.has_tree = c->has_tree;
    v.n_leaves = c->n_leaves;
    v.n_nodes = c->n_nodes;
    v.root_kind = c->root_kind;
    v.depth = c->depth;
    for (int k = 0; k < 3; ++k) v.aabb_min[k] = c->aabb_min[k];
    v.aabb_size = c->aabb_size;
    v.d_nodes = c->d_nodes;
    v.d_perm = c->d_perm;
    v.storage = c->cfg.storage;
    v.d_sig = c->d_sig;
    v.d_z = c->d_z;
    v.d_scale = c->d_scale;
    return v;
}

int set_last_error(int code, const char *msg) { return fail(code, "%s", msg); }

}  // namespace fpo

extern "C" {

const char *fpo_last_error(void) { return g_err.c_str(); }

int fpo_version(void) { return 102; }

int fpo_create(fpo_ctx **out, const fpo_config *cfg)
{
    if (!out) return fail(FPO_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!cfg) return fail(FPO_ERR_INVALID_ARG, "cfg is NULL");
    if (cfg->n1 < 1 || cfg->n1 > 32) return fail(FPO_ERR_INVALID_ARG, "n1 must be in [1, 32]");
    if (cfg->n2 < 1 || cfg->n2 > 16) return fail(FPO_ERR_INVALID_ARG, "n2 must be in [1, 16]");
    if (cfg->sh_degree != 2) return fail(FPO_ERR_UNSUPPORTED, "only sh_degree 2 is supported");
    if (!(cfg->period_T > 0.0) || !std::isfinite(cfg->period_T))
        return fail(FPO_ERR_INVALID_ARG, "period_T must be finite and > 0");
    if (cfg->storage < FPO_STORAGE_F32 || cfg->storage > FPO_STORAGE_LATENT)
        return fail(FPO_ERR_INVALID_ARG, "unknown storage %d", cfg->storage);
    if (cfg->idft_mode < FPO_IDFT_AUTO || cfg->idft_mode > FPO_IDFT_MATERIALISE)
        return fail(FPO_ERR_INVALID_ARG, "unknown idft_mode %d", cfg->idft_mode);
    if (cfg->traverse_threads != 0 && cfg->traverse_threads != 128 && cfg->traverse_threads != 256)
        return fail(FPO_ERR_INVALID_ARG, "traverse_threads must be 0, 128 or 256");
    if (cfg->refill_min < 0 || cfg->refill_min > 32)
        return fail(FPO_ERR_INVALID_ARG, "refill_min must be in [0, 32]");
    if (cfg->inner_steps < 0) return fail(FPO_ERR_INVALID_ARG, "inner_steps must be >= 0");
    if (cfg->max_steps < 0) return fail(FPO_ERR_INVALID_ARG, "max_steps must be >= 0");
    if (cfg->table_precision < FPO_TABLE_AUTO || cfg->table_precision > FPO_TABLE_F16)
        return fail(FPO_ERR_INVALID_ARG, "table_precision must be FPO_TABLE_AUTO, _F32 or _F16");
    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceCount");
    if (cfg->device < 0 || cfg->device >= ndev)
        return fail(FPO_ERR_INVALID_ARG, "device %d out of range (%d devices)", cfg->device, ndev);
    DeviceGuard g(cfg->device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice(%d) failed", cfg->device);
    fpo_ctx *c = new (std::nothrow) fpo_ctx;
    if (!c) return fail(FPO_ERR_OOM, "host allocation failed");
    c->cfg = *cfg;
    c->half_table = cfg->table_precision == FPO_TABLE_F16 ||
                    (cfg->table_precision == FPO_TABLE_AUTO && cfg->storage != FPO_STORAGE_F32);
    e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, cfg->device);
    if (e != cudaSuccess) { delete c; return cuda_fail(e, "cudaDeviceGetAttribute"); }
    e = cudaMalloc((void **)&c->d_status, 32 * sizeof(uint32_t));
    if (e != cudaSuccess) { delete c; return cuda_fail(e, "cudaMalloc(status)"); }
    e = cudaMemset(c->d_status, 0, 32 * sizeof(uint32_t));
    if (e != cudaSuccess) { cudaFree(c->d_status); delete c; return cuda_fail(e, "cudaMemset"); }
    *out = c;
    g_err.clear();
    return FPO_OK;
}

int fpo_validate_tree(const fpo_tree_desc *tree, const fpo_config *cfg)
{
    if (!cfg) return fail(FPO_ERR_INVALID_ARG, "cfg is NULL");
    std::string err;
    int st = validate_and_pack(tree, cfg->n1, cfg->n2, nullptr, &err);
    if (st != FPO_OK) return fail(st, "%s", err.c_str());
    return FPO_OK;
}

int fpo_upload_tree(fpo_ctx *ctx, const fpo_tree_desc *tree)
{
    if (!ctx) return fail(FPO_ERR_INVALID_ARG, "ctx is NULL");
    PackedTree pk;
    std::string err;
    const bool latent = ctx->cfg.storage == FPO_STORAGE_LATENT;
    int st = validate_and_pack(tree, latent ? 0 : ctx->cfg.n1, ctx->cfg.n2, &pk, &err, false);
    if (st != FPO_OK) return fail(st, "%s", err.c_str());
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    ctx->free_tree();

    const int n1 = ctx->cfg.n1, n2 = ctx->cfg.n2, nc = n1 + 27 * n2;
    const int storage = ctx->cfg.storage;
    const RecordLayout L = record_layout(latent ? FPO_STORAGE_F32 : storage, n1, n2);
    const size_t n = latent ? 0 : tree->n_leaves;  // latent storage keeps no coefficient records
    // Reorder the coefficients into breadth-first leaf order, split into the
    // density and the SH record arrays (zero padded), encoded in the storage
    // precision; FP8 codes hold coefficient / scale with a per-leaf scale
    // max|k| / 448 (448 = the largest E4M3 value).
    std::vector<uint8_t> sig(n * L.sig_bytes(), 0), zc(n * L.z_bytes(), 0);
    std::vector<float> scale(L.scaled ? (n + 3) / 4 * 4 : 0, 0.0f);
    auto put = [&](uint8_t *rec, int j, float v) {
        switch (storage) {
        case FPO_STORAGE_BF16: { const uint16_t c = encode_bf16(v); std::memcpy(rec + 2 * j, &c, 2); break; }
        case FPO_STORAGE_F16: { const uint16_t c = encode_f16(v); std::memcpy(rec + 2 * j, &c, 2); break; }
        case FPO_STORAGE_FP8_E4M3: rec[j] = encode_e4m3(v); break;
        default: std::memcpy(rec + 4 * j, &v, 4);
        }
    };
    for (size_t i = 0; i < n; ++i) {
        const float *src = tree->coeffs + (size_t)pk.perm[i] * nc;
        float sc = 1.0f;
        if (L.scaled) {
            float mx = 0.0f;
            for (int j = 0; j < nc; ++j) mx = std::fmax(mx, std::fabs(src[j]));
            sc = mx > 0.0f ? mx / 448.0f : 1.0f;
            scale[i] = sc;
        }
        uint8_t *rs = &sig[i * L.sig_bytes()];
        uint8_t *rz = &zc[i * L.z_bytes()];
        for (int j = 0; j < n1; ++j) put(rs, j, L.scaled ? src[j] / sc : src[j]);
        for (int j = 0; j < 27 * n2; ++j) put(rz, j, L.scaled ? src[n1 + j] / sc : src[n1 + j]);
    }
    const size_t n_nodes = pk.nodes.size() / 8;
    cudaError_t e = cudaSuccess;
    auto up = [&](void **dst, const void *src, size_t bytes, const char *what, size_t room = 0) -> int {
        if (bytes == 0) return FPO_OK;
        e = cudaMalloc(dst, bytes + room);
        if (e != cudaSuccess) return cuda_fail(e, what);
        e = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(e, what);
        return FPO_OK;
    };
    // (where an adjoint will want it, and the records already take a block of
    // their own: it made a tree of 2,252 leaves, whose arrays share small
    // blocks, 0.5 instead of 0.34 ms to upload again into the same context)
    const size_t vl_room = storage == FPO_STORAGE_F32 && fused_supported(n1, n2) && zc.size() >= (2u << 20) ? ctx->vl_bytes(VL_BASE_RAYS) : 0;
    const size_t vl_at = (zc.size() + 255) / 256 * 256;
    if ((st = up((void **)&ctx->d_nodes, pk.nodes.data(), pk.nodes.size() * 4, "nodes")) ||
        (st = up((void **)&ctx->d_top, pk.top.data(), pk.top.size() * 4, "top blocks")) ||
        (st = up((void **)&ctx->d_bricks, pk.bricks.data(), pk.bricks.size() * 4, "bricks")) ||
        (st = up((void **)&ctx->d_perm, pk.perm.data(), pk.perm.size() * 4, "perm")) ||
        (st = up((void **)&ctx->d_sig, sig.data(), sig.size(), "sigma records")) ||
        (st = up((void **)&ctx->d_z, zc.data(), zc.size(), "SH records", vl_at - zc.size() + vl_room)) ||
        (st = up((void **)&ctx->d_scale, scale.data(), scale.size() * 4, "FP8 scales"))) {
        ctx->free_tree();
        return st;
    }
    if (vl_room && ctx->d_z) {
        ctx->vl_base = static_cast<unsigned char *>(ctx->d_z) + vl_at;
        ctx->set_visit_list(ctx->vl_base, VL_BASE_RAYS);
    }
    ctx->n_leaves = tree->n_leaves;
    ctx->n_nodes = (uint32_t)n_nodes;
    ctx->root_kind = pk.root_kind;
    ctx->depth = pk.depth;
    ctx->max_depth = tree->max_depth;
    for (int k = 0; k < 3; ++k) ctx->aabb_min[k] = tree->aabb_min[k];
    ctx->aabb_size = tree->aabb_size;
    ctx->has_tree = true;
    g_err.clear();
    return FPO_OK;
}

int fpo_tree_info_get(const fpo_ctx *ctx, fpo_tree_info *out)
{
    if (!ctx || !out) return fail(FPO_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "no tree uploaded");
    out->n_leaves = ctx->n_leaves;
    out->n_nodes = ctx->n_nodes;
    out->max_depth = ctx->max_depth;
    out->n_smem_nodes = 0;  // every node slot is read from global memory
    out->node_bytes = (uint64_t)ctx->n_nodes * 32;
    if (ctx->cfg.storage == FPO_STORAGE_LATENT) {
        out->leaf_record_bytes = 64;  // one FP16 latent of 32 values (the decoder is shared)
    } else {
        const RecordLayout L = record_layout(ctx->cfg.storage, ctx->cfg.n1, ctx->cfg.n2);
        out->leaf_record_bytes = (uint64_t)(L.sig_bytes() + L.z_bytes() + (L.scaled ? 4 : 0));
    }
    out->leaf_bytes = out->leaf_record_bytes * ctx->n_leaves;
    out->table_bytes = (uint64_t)ctx->table_leaves * table_row_bytes(ctx);
    return FPO_OK;
}

}  // extern "C"

namespace fpo {

int check_rays(const fpo_rays *r, uint64_t *n_rays)
{
    if (r->mode == FPO_RAYS_CAMERA) {
        const double fov = r->fov_y_deg;
        if (!(fov > 0.0 && fov < 180.0)) return fail(FPO_ERR_INVALID_ARG, "fov_y_deg must be in (0, 180)");
        double f[3], c[3];
        for (int k = 0; k < 3; ++k) f[k] = r->target[k] - r->eye[k];
        c[0] = f[1] * r->up[2] - f[2] * r->up[1];
        c[1] = f[2] * r->up[0] - f[0] * r->up[2];
        c[2] = f[0] * r->up[1] - f[1] * r->up[0];
        const double fl = f[0] * f[0] + f[1] * f[1] + f[2] * f[2];
        const double cl = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
        if (!(fl > 0.0) || !(cl > 0.0) || !std::isfinite(fl) || !std::isfinite(cl))
            return fail(FPO_ERR_INVALID_ARG, "degenerate camera (eye == target or up parallel to the view)");
        if (!std::isfinite(r->t)) return fail(FPO_ERR_INVALID_ARG, "t must be finite");
        *n_rays = (uint64_t)r->width * r->height;
    } else if (r->mode == FPO_RAYS_EXPLICIT) {
        if (r->n > 0 && (!r->o || !r->d)) return fail(FPO_ERR_INVALID_ARG, "o and d must be non-NULL");
        if (!r->t_per_ray && !std::isfinite(r->t)) return fail(FPO_ERR_INVALID_ARG, "t must be finite");
        *n_rays = r->n;
    } else {
        return fail(FPO_ERR_INVALID_ARG, "unknown ray mode %d", r->mode);
    }
    if (*n_rays >= (1ull << 31)) return fail(FPO_ERR_INVALID_ARG, "too many rays");
    return FPO_OK;
}

int check_render_opts(const fpo_ctx *ctx, const fpo_frame_opts *opts, uint64_t n_rays, const float *out_rgb)
{
    if (n_rays > 0 && !out_rgb) return fail(FPO_ERR_INVALID_ARG, "out_rgb is NULL");
    const uint32_t fl = opts->flags;
    if ((fl & FPO_FLAG_RECORD_VISITS) && (!opts->visit_count || (opts->visit_cap && !opts->visit_log)))
        return fail(FPO_ERR_INVALID_ARG, "RECORD_VISITS needs visit_count (and visit_log if visit_cap > 0)");
    if ((fl & FPO_FLAG_OUT_T) && !opts->out_T) return fail(FPO_ERR_INVALID_ARG, "OUT_T needs out_T");
    if ((fl & FPO_FLAG_STATS) && !opts->stats) return fail(FPO_ERR_INVALID_ARG, "STATS needs stats");
    if ((fl & FPO_FLAG_MARK_LEAVES) && !opts->leaf_mark && ctx->n_leaves)
        return fail(FPO_ERR_INVALID_ARG, "MARK_LEAVES needs leaf_mark");
    if (!(opts->stop_T >= 0.0f)) return fail(FPO_ERR_INVALID_ARG, "stop_T must be >= 0");
    return FPO_OK;
}

// cos(pi x) and sin(pi x), exact at multiples of 1/2: x is reduced exactly to
// [-1, 1] and then to a quarter period.
double cospi_h(double x, bool sine)
{
    x = std::remainder(x, 2.0);
    const double q = std::nearbyint(2.0 * x);
    const double a = (x - 0.5 * q) * 3.14159265358979323846;
    switch (((int)q + (sine ? 3 : 0)) & 3) {  // sin(y) = cos(y - pi / 2)
    case 0: return std::cos(a);
    case 1: return -std::sin(a);
    case 2: return -std::cos(a);
    default: return std::sin(a);
    }
}

void time_basis(double t, double period_T, int n, float b[32])
{
    const double u = t / period_T;
    for (int i = 0; i < 32; ++i) {
        if (i >= n) b[i] = 0.0f;
        else if (!std::isfinite(u)) b[i] = std::numeric_limits<float>::quiet_NaN();
        else b[i] = (float)((i & 1) ? cospi_h((double)(i + 1) * u, true) : cospi_h((double)i * u, false));
    }
}

// The frame's constants: the time basis and, for camera rays, the camera frame.
static void frame_consts(const FrameParams &fr, int nb, FrameConsts &c)
{
    time_basis(fr.t, fr.period_T, nb, c.b);
    if (fr.mode != FPO_RAYS_CAMERA) return;
    double f[3], r[3], u[3];
    for (int k = 0; k < 3; ++k) f[k] = fr.target[k] - fr.eye[k];
    const double fl = std::sqrt(f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
    for (int k = 0; k < 3; ++k) f[k] /= fl;
    r[0] = f[1] * fr.up[2] - f[2] * fr.up[1];
    r[1] = f[2] * fr.up[0] - f[0] * fr.up[2];
    r[2] = f[0] * fr.up[1] - f[1] * fr.up[0];
    const double rl = std::sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    for (int k = 0; k < 3; ++k) r[k] /= rl;
    u[0] = r[1] * f[2] - r[2] * f[1];
    u[1] = r[2] * f[0] - r[0] * f[2];
    u[2] = r[0] * f[1] - r[1] * f[0];
    const double th = std::tan(0.5 * fr.fov_y_deg * 3.14159265358979323846 / 180.0);
    for (int k = 0; k < 3; ++k) {
        c.f[k] = (float)f[k];
        c.r[k] = (float)r[k];
        c.u[k] = (float)u[k];
        c.eye[k] = (float)fr.eye[k];
    }
    c.sx_scale = (float)(th * (double)fr.width / (double)fr.height);
    c.sy_scale = (float)th;
}

// Kernel parameters of one render (or adjoint) call from the context, rays
// and options; of a camera frame, n_rays rays from row y0 on.
TraverseParams traverse_params(const fpo_ctx *ctx, const fpo_rays *rays, const fpo_frame_opts *opts,
                               float *out_rgb, uint64_t n_rays, uint32_t y0)
{
    const uint32_t fl = opts->flags;
    TraverseParams p{};
    p.fr.mode = rays->mode;
    p.fr.width = rays->width;
    p.fr.height = rays->height;
    p.fr.y0 = y0;
    p.fr.rows = rays->mode == FPO_RAYS_CAMERA && rays->width ? (uint32_t)(n_rays / rays->width) : 0;
    p.fr.n_rays = (uint32_t)n_rays;
    for (int k = 0; k < 3; ++k) {
        p.fr.eye[k] = rays->eye[k];
        p.fr.target[k] = rays->target[k];
        p.fr.up[k] = rays->up[k];
    }
    p.fr.fov_y_deg = rays->fov_y_deg;
    p.fr.t = rays->t;
    p.fr.period_T = ctx->cfg.period_T;
    p.fr.ro = rays->o;
    p.fr.rd = rays->d;
    p.fr.rt = rays->t_per_ray;
    frame_consts(p.fr, ctx->cfg.n1 > ctx->cfg.n2 ? ctx->cfg.n1 : ctx->cfg.n2, p.fc);
    p.nodes = ctx->d_nodes;
    p.top = reinterpret_cast<const uint4 *>(ctx->d_top);
    p.bricks = reinterpret_cast<const uint4 *>(ctx->d_bricks);
    p.top_bits = ctx->depth - 4;
    p.root_kind = ctx->root_kind;
    p.depth = ctx->depth;
    p.grid_scale64 = (double)(1u << ctx->depth) / ctx->aabb_size;
    p.grid_scale = (float)p.grid_scale64;
    for (int k = 0; k < 3; ++k) {
        p.amin64[k] = ctx->aabb_min[k];
        p.amin[k] = (float)ctx->aabb_min[k];
    }
    p.table = reinterpret_cast<const float4 *>(ctx->d_table);
    p.sig = reinterpret_cast<const float4 *>(ctx->d_sig);
    p.zc = static_cast<const float *>(ctx->d_z);
    p.n1 = ctx->cfg.n1;
    p.n2 = ctx->cfg.n2;
    p.sig_stride4 = sig_stride(ctx->cfg.n1) / 4;
    p.z_stride = z_stride(ctx->cfg.n2);
    for (int k = 0; k < 3; ++k) p.bg[k] = opts->bg[k];
    p.stop_T = opts->stop_T;
    p.flags = fl;
    p.out_rgb = out_rgb;
    p.out_T = opts->out_T;
    p.visit_log = opts->visit_log;
    p.visit_cap = opts->visit_cap;
    p.visit_count = opts->visit_count;
    p.leaf_mark = opts->leaf_mark;
    p.perm = ctx->d_perm;
    p.status = ctx->d_status;
    p.tiles = ctx->d_status + 1;
    p.half_table = ctx->half_table;
    if (rays->mode == FPO_RAYS_CAMERA) {
        p.tiles_x = (rays->width + TILE_W - 1) / TILE_W;
        const uint32_t tiles_y = (p.fr.rows + TILE_H - 1) / TILE_H;
        p.n_tiles = p.tiles_x * tiles_y;
    } else {
        p.tiles_x = 0;
        p.n_tiles = (uint32_t)((n_rays + 31) / 32);
    }
    p.form = ray_form(rays->mode == FPO_RAYS_CAMERA, n_rays, ctx->n_leaves);
    p.coherent = p.form == LANES_IF_COHERENT ? ctx->d_status + COHERENT_WORD : nullptr;
    p.max_steps = ctx->cfg.max_steps > 0 ? (uint32_t)ctx->cfg.max_steps : 3u * (1u << ctx->depth) + 16u;
    p.block_threads = ctx->cfg.traverse_threads ? ctx->cfg.traverse_threads : DEFAULT_TRAVERSE_THREADS;
    p.few_tiles_split = ctx->cfg.traverse_threads == 0;
    p.refill_min = ctx->cfg.refill_min ? (uint32_t)ctx->cfg.refill_min : DEFAULT_REFILL_MIN;
    p.inner_steps = ctx->cfg.inner_steps ? (uint32_t)ctx->cfg.inner_steps : DEFAULT_INNER_STEPS;
    p.stats = reinterpret_cast<unsigned long long *>(opts->stats);
    return p;
}

// The per-frame table for time t into `table` on stream s: the tensor-core
// decoder for LATENT storage, else the bulk-copy IDFT pass over the stored
// coefficients (at most max_ctas_per_sm CTAs per SM when > 0).
// With pipe_stages > 0 the pass takes the frame-pipeline shape with that many
// stages (materialise_pipeline_shape), co-scheduled with the traversal.
int launch_table_pass(const fpo_ctx *ctx, double t, float *table, int max_ctas_per_sm, void *stream,
                      int pipe_stages, int carveout, bool test_timeout)
{
    const cudaStream_t s = (cudaStream_t)stream;
    if (ctx->cfg.storage == FPO_STORAGE_LATENT) {
        LatentParams lp{};
        lp.latents = ctx->d_latents;
        lp.w1 = ctx->d_dec_w;
        lp.w2 = ctx->d_dec_w + 64 * 32;
        lp.w3 = ctx->d_dec_w + 64 * 32 + 64 * 64;
        lp.b1 = ctx->d_dec_b;
        lp.b2 = ctx->d_dec_b + 64;
        lp.b3 = ctx->d_dec_b + 128;
        lp.n1 = ctx->cfg.n1;
        lp.n2 = ctx->cfg.n2;
        time_basis(t, ctx->cfg.period_T, ctx->cfg.n1 > ctx->cfg.n2 ? ctx->cfg.n1 : ctx->cfg.n2, lp.b);
        lp.n_leaves = ctx->n_leaves;
        lp.table = table;
        lp.half_table = ctx->half_table;
        lp.status = ctx->d_status;
        lp.test_timeout = test_timeout;
        lp.pipeline = pipe_stages > 0;
        lp.carveout = carveout;
        return launch_latent_table(lp, ctx->sm_count, s);
    }
    MaterialiseParams mp{};
    const RecordLayout L = record_layout(ctx->cfg.storage, ctx->cfg.n1, ctx->cfg.n2);
    mp.sig = ctx->d_sig;
    mp.zc = ctx->d_z;
    mp.scale = ctx->d_scale;
    mp.table = table;
    mp.n_leaves = ctx->n_leaves;
    mp.storage = ctx->cfg.storage;
    mp.n1 = ctx->cfg.n1;
    mp.n2 = ctx->cfg.n2;
    mp.sig_stride = L.sig_elems;
    mp.z_stride = L.z_elems;
    mp.stages = pipe_stages > 0 ? pipe_stages : materialise_stages(ctx->cfg.storage, ctx->cfg.n1, ctx->cfg.n2);
    mp.pipeline = pipe_stages > 0;
    mp.max_ctas_per_sm = max_ctas_per_sm;
    mp.carveout = carveout;
    mp.half_table = ctx->half_table;
    time_basis(t, ctx->cfg.period_T, ctx->cfg.n1 > ctx->cfg.n2 ? ctx->cfg.n1 : ctx->cfg.n2, mp.b);
    mp.status = ctx->d_status;
    mp.test_timeout = test_timeout;
    return launch_materialise(mp, ctx->sm_count, s);
}

}  // namespace fpo

extern "C" {

int fpo_render(fpo_ctx *ctx, const fpo_rays *rays, const fpo_frame_opts *opts, float *out_rgb,
               void *cuda_stream)
{
    if (!ctx || !rays || !opts) return fail(FPO_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "render before fpo_upload_tree");
    uint64_t n_rays = 0;
    int st = check_rays(rays, &n_rays);
    if (st != FPO_OK) return st;
    if ((st = check_render_opts(ctx, opts, n_rays, out_rgb)) != FPO_OK) return st;
    const uint32_t fl = opts->flags;
    const bool per_ray_t = rays->mode == FPO_RAYS_EXPLICIT && rays->t_per_ray;
    int mode = ctx->cfg.idft_mode;
    if (mode == FPO_IDFT_AUTO) mode = per_ray_t ? FPO_IDFT_FUSED : FPO_IDFT_MATERIALISE;
    if (mode == FPO_IDFT_MATERIALISE && per_ray_t)
        return fail(FPO_ERR_INVALID_ARG, "per-ray times need the FUSED IDFT mode");
    const bool mat = mode == FPO_IDFT_MATERIALISE && ctx->n_leaves > 0;
    if (!mat && ctx->n_leaves > 0 && ctx->cfg.storage != FPO_STORAGE_F32)
        return fail(FPO_ERR_UNSUPPORTED, "the fused IDFT reads FP32 records only; use the table mode");
    if (mat && ctx->cfg.storage == FPO_STORAGE_LATENT && !ctx->has_latents)
        return fail(FPO_ERR_INVALID_ARG, "LATENT storage: call fpo_set_latents before rendering");
    if (!mat && !fused_supported(ctx->cfg.n1, ctx->cfg.n2))
        return fail(FPO_ERR_UNSUPPORTED, "the fused IDFT supports (n1, n2) in {(31,5), (11,5), (21,5), (31,11)}");

    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    cudaError_t e;
    if (mat && ctx->table_leaves < ctx->n_leaves) {
        dfree(ctx->d_table);
        e = cudaMalloc((void **)&ctx->d_table, table_alloc_bytes(ctx));
        if (e != cudaSuccess) { ctx->table_leaves = 0; return cuda_fail(e, "cudaMalloc(table)"); }
        ctx->table_leaves = ctx->n_leaves;
    }
    auto rec = [&](int i) -> cudaError_t {
        return opts->events[i] ? cudaEventRecord((cudaEvent_t)opts->events[i], s) : cudaSuccess;
    };
    if ((e = rec(0)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    if (n_rays == 0) {
        if ((e = rec(1)) != cudaSuccess || (e = rec(2)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
        return FPO_OK;
    }
    if (mat && !((fl & FPO_FLAG_REUSE_TABLE) && ctx->table_ok && ctx->table_t == rays->t)) {
        ctx->table_ok = false;
        const int ce = launch_table_pass(ctx, rays->t, ctx->d_table, 0, s, 0, 0,
                                         (fl & FPO_FLAG_TEST_DEVICE_TIMEOUT) != 0);
        if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "IDFT table launch");
        ctx->table_ok = (fl & FPO_FLAG_TEST_DEVICE_TIMEOUT) == 0;
        ctx->table_t = rays->t;
    }
    if ((e = rec(1)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");

    TraverseParams p = traverse_params(ctx, rays, opts, out_rgb, n_rays);
    const bool dbg = (fl & (FPO_FLAG_RECORD_VISITS | FPO_FLAG_OUT_T | FPO_FLAG_MARK_LEAVES |
                            FPO_FLAG_STATS)) != 0;
    int ce = launch_traverse(p, mat, dbg, ctx->sm_count, s);
    if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "traverse launch");
    if ((e = rec(2)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    return FPO_OK;
}

int fpo_render_frames(fpo_ctx *ctx, const fpo_rays *frames, uint32_t n_frames, const fpo_frame_opts *opts,
                      float *out_rgb, void *const *frame_done, void *cuda_stream)
{
    if (!ctx || !opts || (n_frames && !frames)) return fail(FPO_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "render before fpo_upload_tree");
    if (opts->flags) return fail(FPO_ERR_INVALID_ARG, "fpo_render_frames takes no debug outputs (flags must be 0)");
    uint64_t R = 0;
    for (uint32_t k = 0; k < n_frames; ++k) {
        uint64_t nr = 0;
        const int st = check_rays(&frames[k], &nr);
        if (st != FPO_OK) return st;
        if (frames[k].mode == FPO_RAYS_EXPLICIT && frames[k].t_per_ray)
            return fail(FPO_ERR_INVALID_ARG, "per-ray times need fpo_render (fused IDFT)");
        if (k == 0) R = nr;
        else if (nr != R) return fail(FPO_ERR_INVALID_ARG, "every frame must have the same number of rays");
    }
    if (n_frames == 0 || R == 0) return FPO_OK;
    if (!out_rgb) return fail(FPO_ERR_INVALID_ARG, "out_rgb is NULL");
    if (!(opts->stop_T >= 0.0f)) return fail(FPO_ERR_INVALID_ARG, "stop_T must be >= 0");
    fpo_frame_opts o1 = *opts;
    for (int i = 0; i < 3; ++i) o1.events[i] = nullptr;
    const bool mat = ctx->cfg.idft_mode != FPO_IDFT_FUSED && ctx->n_leaves > 0;
    if (!mat || n_frames == 1) {
        for (uint32_t k = 0; k < n_frames; ++k) {
            const int st = fpo_render(ctx, &frames[k], &o1, out_rgb + (size_t)k * R * 3, cuda_stream);
            if (st != FPO_OK) return st;
            if (frame_done && frame_done[k]) {
                const cudaError_t e = cudaEventRecord((cudaEvent_t)frame_done[k], (cudaStream_t)cuda_stream);
                if (e != cudaSuccess) return cuda_fail(e, "cudaEventRecord(frame_done)");
            }
        }
        return FPO_OK;
    }
    if (ctx->cfg.storage == FPO_STORAGE_LATENT && !ctx->has_latents)
        return fail(FPO_ERR_INVALID_ARG, "LATENT storage: call fpo_set_latents before rendering");
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    cudaError_t e = cudaSuccess;
    // Views of one frame time (every t bit-equal): one table pass, and every
    // traversal of the call reads that table (nothing rewrites it before the
    // call's end, after which the caller's stream has waited for them all).
    bool one_t = n_frames > 1;
    for (uint32_t k = 1; k < n_frames && one_t; ++k)
        one_t = memcmp(&frames[k].t, &frames[0].t, sizeof(double)) == 0;
    int depth = ctx->half_table ? FPO_PIPE_DEPTH_F16 : FPO_PIPE_DEPTH;
    if (depth > ctx->pipe_cap) depth = ctx->pipe_cap;
    int slots = n_frames < (uint32_t)depth ? (int)n_frames : depth;  // in use by this call
    const int trav_threads = ctx->half_table ? FPO_PIPE_TRAV_THREADS_F16 : PIPE_TRAV_THREADS;
    const int trav_ctas = ctx->half_table ? FPO_PIPE_TRAV_CTAS_F16 : PIPE_TRAV_CTAS;
    // Tables, streams and events as this call needs them, the further slots'
    // tables in one allocation: what a context's first call of a few small
    // frames spends most of its time on.
    if (ctx->table_leaves < ctx->n_leaves) {
        dfree(ctx->d_table);
        e = cudaMalloc((void **)&ctx->d_table, table_alloc_bytes(ctx));
        if (e != cudaSuccess) { ctx->table_leaves = 0; return cuda_fail(e, "cudaMalloc(table)"); }
        ctx->table_leaves = ctx->n_leaves;
    }
    while (!one_t && ctx->ptable_slots < slots - 1) {
        dfree(ctx->d_ptables);
        ctx->ptable_slots = 0;
        e = cudaMalloc((void **)&ctx->d_ptables, (size_t)(slots - 1) * table_alloc_bytes(ctx));
        if (e == cudaSuccess) {
            ctx->ptable_slots = slots - 1;
        } else {
            ctx->d_ptables = nullptr;
            if (e != cudaErrorMemoryAllocation || slots <= FPO_PIPE_DEPTH) return cuda_fail(e, "cudaMalloc(table)");
            cudaGetLastError();  // a tree so large that six tables do not fit: four
            slots = depth = ctx->pipe_cap = FPO_PIPE_DEPTH;
        }
    }
    if (!ctx->aux || !ctx->trav[slots - 1] || !ctx->ev_trav[slots - 1]) {
        // created once; a failed attempt is retried whole
        if (!ctx->aux) e = cudaStreamCreateWithFlags(&ctx->aux, cudaStreamNonBlocking);
        if (e == cudaSuccess && !ctx->ev_entry) e = cudaEventCreateWithFlags(&ctx->ev_entry, cudaEventDisableTiming);
        for (int b = 0; b < slots && e == cudaSuccess; ++b) {
            if (b && !ctx->trav[b]) e = cudaStreamCreateWithFlags(&ctx->trav[b], cudaStreamNonBlocking);
            if (e == cudaSuccess && !ctx->ev_mat[b]) e = cudaEventCreateWithFlags(&ctx->ev_mat[b], cudaEventDisableTiming);
            if (e == cudaSuccess && !ctx->ev_trav[b]) e = cudaEventCreateWithFlags(&ctx->ev_trav[b], cudaEventDisableTiming);
        }
        if (e != cudaSuccess) return cuda_fail(e, "stream/event creation");
    }
    // Shapes that let both kernels be resident on an SM at once: the IDFT
    // pass in materialise_pipeline_shape, or for LATENT storage one 256-thread
    // decoder CTA (two warpgroup pipelines, 128 TMEM columns) per SM.
    bool overlap = true;
    MatShape mshape{};
    int carveout = 0;
    if (overlap) {
        int max_smem = 0, reserved = 0;
        if ((e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, ctx->cfg.device)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, ctx->cfg.device)) != cudaSuccess)
            return cuda_fail(e, "cudaDeviceGetAttribute");
        if (ctx->cfg.storage == FPO_STORAGE_LATENT) {
            mshape.ctas_per_sm = 1;
            mshape.stages = 1;  // (a positive value selects the pipeline shape)
            mshape.smem_per_cta = latent_pipeline_smem_bytes();
        } else {
            mshape = materialise_pipeline_shape(ctx->cfg.storage, ctx->cfg.n1, ctx->cfg.n2, PIPE_MAT_SMEM_BUDGET);
            if (FPO_PIPE_MAT_CTAS > 0) mshape.ctas_per_sm = FPO_PIPE_MAT_CTAS;
        }
        const bool brick = brick_walk(ctx->d_top != nullptr, ctx->cfg.refill_min ? (uint32_t)ctx->cfg.refill_min : DEFAULT_REFILL_MIN);
        const long need = (long)trav_ctas * (traverse_smem_bytes(brick, trav_threads) + PIPE_STATIC_SMEM + reserved) +
                          (long)mshape.ctas_per_sm * (mshape.smem_per_cta + PIPE_STATIC_SMEM + reserved);
        // The driver rounds a carveout request up to one of the SM's shared-
        // memory configurations: ask for the smallest one that holds `need`.
        long config = -1;
        for (const int kb : SMEM_CONFIGS_KB)
            if ((long)kb * 1024 >= need) { config = (long)kb * 1024; break; }
        if (config < 0 || config > max_smem) overlap = false;
        else carveout = (int)(config * 100 / max_smem);
    }
    ctx->table_ok = false;  // the pipeline writes every slot's table
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // Frame k takes slot b = k mod depth: the slot's table and traversal
    // stream (slot 0: d_table and the caller's stream) and tile counter.  The
    // table passes run in order on the auxiliary stream, ahead of the
    // traversals; the traversals of consecutive frames run on different
    // streams, so that the next ones fill the SMs that the last warps of the
    // earlier ones leave idle.  Table b is rewritten only after the
    // traversal that read it (event ev_trav[b]), and the caller's stream
    // waits for every slot's last traversal at the end.
    if ((e = cudaEventRecord(ctx->ev_entry, s)) != cudaSuccess || (e = cudaStreamWaitEvent(ctx->aux, ctx->ev_entry, 0)) != cudaSuccess)
        return cuda_fail(e, "stream ordering");
    for (int b = 1; b < slots; ++b)
        if ((e = cudaStreamWaitEvent(ctx->trav[b], ctx->ev_entry, 0)) != cudaSuccess) return cuda_fail(e, "stream ordering");
    for (uint32_t k = 0; k < n_frames; ++k) {
        const int b = (int)(k % (uint32_t)depth);
        float *tbl = one_t || b == 0 ? ctx->d_table
                                     : ctx->d_ptables + (size_t)(b - 1) * (table_alloc_bytes(ctx) / sizeof(float));
        cudaStream_t ts = FPO_PIPE_SLOT_STREAMS && b ? ctx->trav[b] : s;
        int ce = cudaSuccess;
        if (!one_t || k == 0) {
            if (k >= (uint32_t)depth && (e = cudaStreamWaitEvent(ctx->aux, ctx->ev_trav[b], 0)) != cudaSuccess)
                return cuda_fail(e, "wait");
            ce = overlap ? launch_table_pass(ctx, frames[k].t, tbl, mshape.ctas_per_sm, ctx->aux, mshape.stages, carveout, false)
                         : launch_table_pass(ctx, frames[k].t, tbl, 0, ctx->aux, 0, 0, false);
            if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "IDFT table launch");
            if ((e = cudaEventRecord(ctx->ev_mat[b], ctx->aux)) != cudaSuccess)
                return cuda_fail(e, "stream ordering");
        }
        if ((e = cudaStreamWaitEvent(ts, ctx->ev_mat[one_t ? 0 : b], 0)) != cudaSuccess)
            return cuda_fail(e, "stream ordering");
        TraverseParams p = traverse_params(ctx, &frames[k], &o1, out_rgb + (size_t)k * R * 3, R);
        p.table = reinterpret_cast<const float4 *>(tbl);
        p.tiles = ctx->d_status + 1 + (FPO_PIPE_SLOT_STREAMS ? 2 * b : 0);  // this slot's tile counter and finished warps
        if (overlap) {
            p.block_threads = trav_threads;
            p.max_ctas_per_sm = trav_ctas;
            p.carveout = carveout;
        }
        ce = launch_traverse(p, true, false, ctx->sm_count, ts);
        if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "traverse launch");
        if ((e = cudaEventRecord(ctx->ev_trav[b], ts)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
        if (frame_done && frame_done[k] && (e = cudaEventRecord((cudaEvent_t)frame_done[k], ts)) != cudaSuccess)
            return cuda_fail(e, "cudaEventRecord(frame_done)");
    }
    // everything above is ordered before the caller's later work
    for (int b = 1; b < slots; ++b)
        if ((e = cudaStreamWaitEvent(s, ctx->ev_trav[b], 0)) != cudaSuccess) return cuda_fail(e, "stream ordering");
    return FPO_OK;
}

}  // extern "C"

namespace {

// Rays from which an adjoint without a list (capture, no memory, other visits
// waiting) takes one lane a ray: the lanes' adds follow one another where a
// warp's wait for its longest ray (us, warps / lanes: camera 160x120 308 / 744,
// 320x240 956 / 781, 480x360 1786 / 938 on 348,592 leaves, 4730 / 2247 on 3.5M;
// 65,536 explicit rays 490 / 465 and 1155 / 1057, 131,072 946 / 736 and 2313 /
// 1756).  (A transmittance within rounding of stop_T may then stop a visit apart
// from a forward by warps.)
constexpr uint64_t NO_LIST_LANES = 1u << 16;

// Whether work on s goes into a graph (a stream that cannot be asked counts as such).
bool capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return true;
}

// Lets this thread allocate while some other stream is being captured.
struct CaptureElsewhere {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    CaptureElsewhere() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~CaptureElsewhere() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The context's visit list for an adjoint call over n_rays rays.  `defer` holds
// for batches of up to n_leaves rays: with more, a leaf has so many visits that
// adding them all to the gradient rows now, evenly divided, is the faster way
// (fine-tuning step, deferred against added now, us: 43,575 leaves, 4,096 rays
// 206 and 208, 16,384 280 and 284, 65,536 471 and 400; 5,430 leaves, 4,096 rays
// 190 and 200, 16,384 262 and 210, 65,536 347 and 277; 348,592 leaves, 65,536
// rays 763 and 849).  The list stays
// empty (cap 0: the replay adds its rows itself) for large batches, when the
// workspace would have to grow while it holds deferred visits, when there is
// no memory for it, and during a stream capture: a graph that held the list
// would write to freed memory once the list has grown, and its replays would
// mix their visits with those that wait here.
VisitList visit_list(fpo_ctx *c, uint64_t n_rays, bool defer, cudaStream_t s)
{
    VisitList L{};
    defer = defer && n_rays <= c->n_leaves;
    if (n_rays > VL_MAX_RAYS || (c->vl_used && !defer) || capturing(s)) return L;
    const uint32_t n = (uint32_t)n_rays;
    if (c->vl_used + n > c->vl_rays) {
        if (c->vl_used) return L;
        const CaptureElsewhere relaxed;
        dfree(c->d_vl_block);
        c->set_visit_list(c->vl_base, VL_BASE_RAYS);  // (none on a small tree)
        uint32_t room = VL_BASE_RAYS;  // rays, in powers of two
        while (room < n) room *= 2;
        if (cudaMalloc((void **)&c->d_vl_block, c->vl_bytes(room)) != cudaSuccess) {
            cudaGetLastError();
            c->d_vl_block = nullptr;
            return L;
        }
        c->set_visit_list(c->d_vl_block, room);
    }
    if (defer && !c->d_vl_slot) {
        const CaptureElsewhere relaxed;
        const size_t nl = c->n_leaves;
        if (cudaMalloc((void **)&c->d_vl_slot, nl * (sizeof(uint4) + sizeof(uint32_t))) != cudaSuccess) {
            cudaGetLastError();
            c->d_vl_slot = nullptr;
            return L;
        }
        c->d_vl_visits = reinterpret_cast<uint32_t *>(c->d_vl_slot + nl);
        if (cudaMemsetAsync(c->d_vl_visits, 0, nl * sizeof(uint32_t), s) != cudaSuccess) {
            cudaGetLastError();
            dfree(c->d_vl_slot);
            return L;
        }
    }
    L.cap = c->vl_cap;
    L.count = c->d_status + VL_COUNT;
    L.id = c->d_vl_id;
    L.val = c->d_vl_val;
    L.over = c->d_vl_over;
    L.visits = c->d_vl_visits;
    L.slot = defer ? c->d_vl_slot : nullptr;
    L.w = c->d_vl_w;
    L.ray_base = c->vl_used;
    return L;
}

// The call that takes or drops deferred visits has to run now, not in a graph.
constexpr char VISITS_WAIT[] = "deferred visits wait for fpo_adam_leaves: not during a stream capture";

// Deferred visits that no fpo_adam_leaves has taken are forgotten.
cudaError_t drop_visits(fpo_ctx *c, cudaStream_t s)
{
    if (!c->vl_used) return cudaSuccess;
    c->vl_used = 0;
    cudaError_t e = cudaMemsetAsync(c->d_vl_visits, 0, (size_t)c->n_leaves * sizeof(uint32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->d_status + VL_COUNT, 0, VL_COUNTS * sizeof(uint32_t), s);
    return e;
}

}  // namespace

extern "C" {

int fpo_render_backward(fpo_ctx *ctx, const fpo_rays *rays, const fpo_frame_opts *opts,
                        const float *out_rgb, const float *dL_drgb, float *dL_dcoeffs,
                        void *cuda_stream)
{
    if (!ctx || !rays || !opts) return fail(FPO_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "backward before fpo_upload_tree");
    uint64_t n_rays = 0;
    int st = check_rays(rays, &n_rays);
    if (st != FPO_OK) return st;
    if (ctx->cfg.storage != FPO_STORAGE_F32)
        return fail(FPO_ERR_UNSUPPORTED, "gradients are taken with respect to FP32 records only");
    if (!fused_supported(ctx->cfg.n1, ctx->cfg.n2))
        return fail(FPO_ERR_UNSUPPORTED, "the adjoint supports (n1, n2) in {(31,5), (11,5), (21,5), (31,11)}");
    if (n_rays > 0 && (!out_rgb || !dL_drgb)) return fail(FPO_ERR_INVALID_ARG, "out_rgb and dL_drgb must be non-NULL");
    if (ctx->n_leaves > 0 && !dL_dcoeffs) return fail(FPO_ERR_INVALID_ARG, "dL_dcoeffs is NULL");
    const bool fp64 = (opts->flags & FPO_FLAG_FP64_GRADCHECK) != 0;
    if (reinterpret_cast<uintptr_t>(dL_dcoeffs) % (fp64 ? 8 : 16) != 0)
        return fail(FPO_ERR_INVALID_ARG, fp64 ? "dL_dcoeffs must be 8-byte aligned" : "dL_dcoeffs must be 16-byte aligned");
    if (!(opts->stop_T >= 0.0f)) return fail(FPO_ERR_INVALID_ARG, "stop_T must be >= 0");
    if (n_rays == 0 || ctx->n_leaves == 0) return FPO_OK;
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    const bool mark = (opts->flags & FPO_FLAG_MARK_LEAVES) != 0;
    if (mark && !opts->leaf_mark) return fail(FPO_ERR_INVALID_ARG, "FPO_FLAG_MARK_LEAVES needs leaf_mark");
    const bool defer = (opts->flags & FPO_FLAG_DEFER_GRADIENT) != 0;
    if (defer && (fp64 || !mark))
        return fail(FPO_ERR_INVALID_ARG, "FPO_FLAG_DEFER_GRADIENT needs FPO_FLAG_MARK_LEAVES and the FP32 adjoint");
    fpo_frame_opts o = *opts;
    o.flags = 0;  // the other debug outputs belong to the forward
    BackwardParams q{};
    q.tp = traverse_params(ctx, rays, &o, nullptr, n_rays);
    q.out_rgb = out_rgb;
    q.dL_drgb = dL_drgb;
    q.dL_dcoeffs = fp64 ? nullptr : dL_dcoeffs;
    q.dL_dcoeffs64 = fp64 ? reinterpret_cast<double *>(dL_dcoeffs) : nullptr;
    q.leaf_mark = mark ? opts->leaf_mark : nullptr;
    // A batch larger than the list holds goes in equal parts, each with its
    // pass over the list (whole 32-ray groups, or whole rows of tiles).
    const bool camera = rays->mode == FPO_RAYS_CAMERA;
    const uint64_t parts = (n_rays + VL_MAX_RAYS - 1) / VL_MAX_RAYS;
    const uint64_t unit = camera ? (uint64_t)TILE_H * rays->width : 32;  // rays
    uint64_t step = ((n_rays + parts - 1) / parts + unit - 1) / unit * unit;
    if (parts > 1 && step > VL_MAX_RAYS) step = VL_MAX_RAYS / unit * unit;
    if (!fp64 && q.tp.form != BY_LANES && step) q.list = visit_list(ctx, step < n_rays ? step : n_rays, defer && parts == 1, (cudaStream_t)cuda_stream);
    const uint32_t *coherent = nullptr;
    if (!q.list.cap) {
        step = n_rays;
        if (n_rays >= NO_LIST_LANES) q.tp.form = BY_LANES;
    } else if (q.tp.form == LANES_IF_COHERENT && parts > 1) {
        coherent = q.tp.coherent;
        const int ce = launch_backward(q, ctx->sm_count, cuda_stream);
        if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "backward launch");
    }
    if (q.tp.form == LANES_IF_COHERENT) q.tp.form = BY_WARPS;
    q.tp.coherent = coherent;
    for (uint64_t at = 0; at < n_rays; at += step) {
        const uint64_t n = n_rays - at < step ? n_rays - at : step;
        if (n < n_rays) {
            fpo_rays part = *rays;
            if (!camera) {
                part.n = (uint32_t)n;
                part.o = rays->o + 3 * at;
                part.d = rays->d + 3 * at;
                part.t_per_ray = rays->t_per_ray ? rays->t_per_ray + at : nullptr;
            }
            q.tp = traverse_params(ctx, &part, &o, nullptr, n, (uint32_t)(camera ? at / rays->width : 0));
            q.tp.form = BY_WARPS;
            q.tp.coherent = coherent;
            q.out_rgb = out_rgb + 3 * at;
            q.dL_drgb = dL_drgb + 3 * at;
        }
        int ce = launch_backward(q, ctx->sm_count, cuda_stream);
        if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "backward launch");
        if (q.list.slot) {
            ctx->vl_used += (uint32_t)n_rays;
        } else if (q.list.cap) {
            ce = launch_grad_scatter(q, ctx->sm_count, cuda_stream);
            if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "gradient scatter launch");
        }
    }
    return FPO_OK;
}

int fpo_set_latents(fpo_ctx *ctx, const uint16_t *latents, const fpo_decoder *dec, void *cuda_stream)
{
    if (!ctx || !dec) return fail(FPO_ERR_INVALID_ARG, "NULL argument");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "set_latents before fpo_upload_tree");
    if (ctx->cfg.storage != FPO_STORAGE_LATENT) return fail(FPO_ERR_UNSUPPORTED, "context storage is not LATENT");
    if (!dec->w1 || !dec->b1 || !dec->w2 || !dec->b2 || !dec->w3 || !dec->b3 || (ctx->n_leaves && !latents))
        return fail(FPO_ERR_INVALID_ARG, "NULL array");
    ctx->table_ok = false;  // the coefficients change
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    const int nc = ctx->cfg.n1 + 27 * ctx->cfg.n2;
    const size_t nw = 64 * 32 + 64 * 64 + (size_t)nc * 64, nb = 64 + 64 + (size_t)nc;
    cudaError_t e = cudaSuccess;
    if (!ctx->d_dec_w) e = cudaMalloc((void **)&ctx->d_dec_w, nw * 2);
    if (e == cudaSuccess && !ctx->d_dec_b) e = cudaMalloc((void **)&ctx->d_dec_b, nb * 4);
    if (e == cudaSuccess && !ctx->d_latents && ctx->n_leaves)
        e = cudaMalloc((void **)&ctx->d_latents, (size_t)ctx->n_leaves * 64);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(latents)");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    struct { void *dst; const void *src; size_t bytes; } cp[6] = {
        {ctx->d_dec_w, dec->w1, 64 * 32 * 2}, {ctx->d_dec_w + 64 * 32, dec->w2, 64 * 64 * 2},
        {ctx->d_dec_w + 64 * 32 + 64 * 64, dec->w3, (size_t)nc * 64 * 2}, {ctx->d_dec_b, dec->b1, 64 * 4},
        {ctx->d_dec_b + 64, dec->b2, 64 * 4}, {ctx->d_dec_b + 128, dec->b3, (size_t)nc * 4}};
    for (auto &c : cp) {
        e = cudaMemcpyAsync(c.dst, c.src, c.bytes, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return cuda_fail(e, "decoder copy");
    }
    const int ce = launch_gather_rows(latents, ctx->d_latents, ctx->d_perm, ctx->n_leaves, 64, ctx->sm_count, s);
    if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "latent gather");
    ctx->has_latents = true;
    return FPO_OK;
}

int fpo_set_coeffs(fpo_ctx *ctx, const float *coeffs, void *cuda_stream)
{
    if (!ctx) return fail(FPO_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "set_coeffs before fpo_upload_tree");
    if (ctx->cfg.storage != FPO_STORAGE_F32)
        return fail(FPO_ERR_UNSUPPORTED, "in-place coefficient updates need FP32 storage");
    if (ctx->n_leaves == 0) return FPO_OK;
    if (!coeffs) return fail(FPO_ERR_INVALID_ARG, "coeffs is NULL");
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    if (ctx->vl_used && capturing((cudaStream_t)cuda_stream)) return fail(FPO_ERR_INVALID_ARG, "%s", VISITS_WAIT);
    ctx->table_ok = false;  // the coefficients change
    const cudaError_t de = drop_visits(ctx, (cudaStream_t)cuda_stream);
    if (de != cudaSuccess) return cuda_fail(de, "visit list reset");
    const int ce = launch_set_coeffs(coeffs, ctx->d_perm, static_cast<float *>(ctx->d_sig),
                                     static_cast<float *>(ctx->d_z), ctx->n_leaves, ctx->cfg.n1,
                                     ctx->cfg.n2, ctx->sm_count, cuda_stream);
    if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "set_coeffs launch");
    return FPO_OK;
}

int fpo_set_coeffs_from_decoder(fpo_ctx *ctx, const fpo_mlp *w, const float *latents, uint32_t flags, void *cuda_stream)
{
    if (!ctx) return fail(FPO_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "set_coeffs_from_decoder before fpo_upload_tree");
    if (ctx->cfg.storage != FPO_STORAGE_F32)
        return fail(FPO_ERR_UNSUPPORTED, "in-place coefficient updates need FP32 storage");
    if (!w || !w->w1 || !w->b1 || !w->w2 || !w->b2 || !w->w3 || !w->b3) return fail(FPO_ERR_INVALID_ARG, "NULL weights");
    if (ctx->cfg.n1 + 27 * ctx->cfg.n2 > decoder_grad_max_coeffs())
        return fail(FPO_ERR_UNSUPPORTED, "n1 + 27 n2 above the decoder's 176 outputs");
    if (ctx->n_leaves == 0) return FPO_OK;
    if (!latents) return fail(FPO_ERR_INVALID_ARG, "latents is NULL");
    if (flags & ~(uint32_t)(FPO_FLAG_TENSOR_CORES | FPO_FLAG_TEST_DEVICE_TIMEOUT))
        return fail(FPO_ERR_INVALID_ARG, "unknown flags");
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    if (ctx->vl_used && capturing((cudaStream_t)cuda_stream)) return fail(FPO_ERR_INVALID_ARG, "%s", VISITS_WAIT);
    ctx->table_ok = false;  // the coefficients change
    const cudaError_t de = drop_visits(ctx, (cudaStream_t)cuda_stream);
    if (de != cudaSuccess) return cuda_fail(de, "visit list reset");
    const int ce = (flags & FPO_FLAG_TENSOR_CORES)
                       ? launch_decode_records_tc(*w, ctx->cfg.n1, ctx->cfg.n2, ctx->n_leaves, latents, ctx->d_perm,
                                                  static_cast<float *>(ctx->d_sig), static_cast<float *>(ctx->d_z),
                                                  ctx->d_status, (flags & FPO_FLAG_TEST_DEVICE_TIMEOUT) != 0,
                                                  ctx->sm_count, cuda_stream)
                       : launch_decode_records(*w, ctx->cfg.n1, ctx->cfg.n2, ctx->n_leaves, latents, ctx->d_perm,
                                               static_cast<float *>(ctx->d_sig), static_cast<float *>(ctx->d_z),
                                               ctx->sm_count, cuda_stream);
    if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "decode launch");
    return FPO_OK;
}

int fpo_adam_leaves(fpo_ctx *ctx, float *param, float *grad, float *m, float *v, uint8_t *leaf_mark, float lr,
                    float beta1, float beta2, float eps, uint32_t step, void *cuda_stream)
{
    if (!ctx) return fail(FPO_ERR_INVALID_ARG, "ctx is NULL");
    if (!ctx->has_tree) return fail(FPO_ERR_NO_TREE, "adam_leaves before fpo_upload_tree");
    if (ctx->cfg.storage != FPO_STORAGE_F32)
        return fail(FPO_ERR_UNSUPPORTED, "in-place coefficient updates need FP32 storage");
    if (ctx->n_leaves == 0) return FPO_OK;
    if (!param || !grad || !m || !v || !leaf_mark) return fail(FPO_ERR_INVALID_ARG, "NULL array");
    if (step < 1) return fail(FPO_ERR_INVALID_ARG, "step counts from 1");
    if (!(lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return fail(FPO_ERR_INVALID_ARG, "lr >= 0, beta in [0, 1), eps > 0");
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    if (ctx->vl_used && capturing((cudaStream_t)cuda_stream)) return fail(FPO_ERR_INVALID_ARG, "%s", VISITS_WAIT);
    ctx->table_ok = false;  // the coefficients change
    LeafAdamParams p{};
    p.param = param;
    p.grad = grad;
    p.m = m;
    p.v = v;
    p.leaf_mark = leaf_mark;
    p.perm = ctx->d_perm;
    p.sig = static_cast<float *>(ctx->d_sig);
    p.zc = static_cast<float *>(ctx->d_z);
    p.n_leaves = ctx->n_leaves;
    p.n1 = ctx->cfg.n1;
    p.n2 = ctx->cfg.n2;
    p.sig_stride = sig_stride(ctx->cfg.n1);
    p.z_stride = z_stride(ctx->cfg.n2);
    p.lr = lr;
    p.beta1 = beta1;
    p.beta2 = beta2;
    p.eps = eps;
    p.bc1 = (float)(1.0 - std::pow((double)beta1, (double)step));
    p.bc2 = (float)(1.0 - std::pow((double)beta2, (double)step));
    if (ctx->vl_used) {
        p.list.cap = ctx->vl_cap;
        p.list.count = ctx->d_status + VL_COUNT;
        p.list.id = ctx->d_vl_id;
        p.list.val = ctx->d_vl_val;
        p.list.over = ctx->d_vl_over;
        p.list.visits = ctx->d_vl_visits;
        p.list.slot = ctx->d_vl_slot;
        p.list.w = ctx->d_vl_w;
    }
    const int ce = launch_leaf_adam(p, ctx->sm_count, cuda_stream);
    if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "adam_leaves launch");
    ctx->vl_used = 0;
    return FPO_OK;
}

int fpo_dft_leaves(int32_t n1, int32_t n2, uint32_t n_frames, uint32_t n_leaves, const float *values,
                   float *coeffs, uint32_t *status, uint32_t flags, void *cuda_stream)
{
    if (n1 < 1 || n1 > 32 || n2 < 1 || n2 > 16) return fail(FPO_ERR_INVALID_ARG, "n1 in [1, 32], n2 in [1, 16]");
    if (flags & ~(uint32_t)FPO_FLAG_TEST_DEVICE_TIMEOUT) return fail(FPO_ERR_INVALID_ARG, "unknown flags");
    if (n_frames < 1 || n_frames > 256) return fail(FPO_ERR_INVALID_ARG, "n_frames must be in [1, 256]");
    if (n_leaves == 0) return FPO_OK;
    if (!values || !coeffs) return fail(FPO_ERR_INVALID_ARG, "NULL array");
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e, "device query");
    const int ce = launch_dft(values, coeffs, n_leaves, n1, n2, (int)n_frames, status,
                              (flags & FPO_FLAG_TEST_DEVICE_TIMEOUT) != 0, sms, cuda_stream);
    if (ce != cudaSuccess) return cuda_fail((cudaError_t)ce, "dft launch");
    return FPO_OK;
}

int fpo_status_sync(fpo_ctx *ctx, void *cuda_stream)
{
    if (!ctx) return fail(FPO_ERR_INVALID_ARG, "ctx is NULL");
    DeviceGuard g(ctx->cfg.device);
    if (!g.ok) return fail(FPO_ERR_CUDA, "cudaSetDevice failed");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    uint32_t st = 0;
    cudaError_t e = cudaMemcpyAsync(&st, ctx->d_status, sizeof st, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "status read");
    if (st) {
        e = cudaMemsetAsync(ctx->d_status, 0, sizeof st, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "status clear");
    }
    if (st & STATUS_TRAVERSAL_LIMIT) return fail(FPO_ERR_TRAVERSAL_LIMIT, "a ray exceeded its step cap");
    if (st & STATUS_VISIT_OVERFLOW) return fail(FPO_ERR_VISIT_OVERFLOW, "a ray had more visits than visit_cap");
    if (st & STATUS_DEVICE_TIMEOUT) return fail(FPO_ERR_DEVICE_TIMEOUT, "a device-side wait gave up after its time limit");
    if (st & STATUS_FP16_RANGE)
        return fail(FPO_ERR_RANGE, "a latent decoder weight, bias or hidden activation exceeded the FP16 range (65504)");
    return FPO_OK;
}

void fpo_destroy(fpo_ctx *ctx)
{
    if (!ctx) return;
    {
        DeviceGuard g(ctx->cfg.device);
        ctx->free_tree();
        dfree(ctx->d_status);
        if (ctx->aux) cudaStreamDestroy(ctx->aux);
        if (ctx->ev_entry) cudaEventDestroy(ctx->ev_entry);
        for (int b = 0; b < PIPE_MAX; ++b) {
            if (ctx->trav[b]) cudaStreamDestroy(ctx->trav[b]);
            if (ctx->ev_mat[b]) cudaEventDestroy(ctx->ev_mat[b]);
            if (ctx->ev_trav[b]) cudaEventDestroy(ctx->ev_trav[b]);
        }
    }
    delete ctx;
}

}  // extern "C"
