// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "grf.h"

#define GRF_CUDA_TRY(expr)                                  \
    do {                                                    \
        cudaError_t _e = (expr);                            \
        if (_e != cudaSuccess) return GRF_ERR_CUDA;         \
    } while (0)

#define GRF_TRY(expr)                                       \
    do {                                                    \
        int _rc = (expr);                                   \
        if (_rc != GRF_OK) return _rc;                      \
    } while (0)

// A device buffer that only ever grows; owned by a context or a feature object.
struct grf_buf {
    void* ptr = nullptr;
    size_t bytes = 0;
    int device = -1;                // of the block at ptr
};

struct grf_ctx {
    int device = 0;
    uint64_t id = 0;                // of this context alone, from 1
    cudaStream_t stream = nullptr;
    int sm_count = 0;
    int64_t launches = 0;
    // sampler scratch
    grf_buf stage_col, stage_val;   // merged rows at a fixed stride, before compaction
    grf_buf edge_records;           // the graph's edges as the walks read them
    grf_buf counts;                 // nonzeros per row of both matrices, then per column of Psi: three arrays of 16-byte aligned length
    grf_buf scan_blocks;            // block totals of the two-level scan
    // sampler scratch when the walks' deposits are kept (grf_ctx_keep_walks)
    bool keep_walks = false;
    grf_buf stage_dep_start, stage_dep_t, stage_dep_load, dep_counts, dep_rowptr2;
    // transpose scratch
    grf_buf t_cursor;               // per column: count, then scatter cursor; number of long buckets; their list
    grf_buf t_tmp;                  // unordered buckets of (row, value)
    // denominators of whole states when the caller wants none (grf_den_scratch); what graphs still name beside the present block,
    // every one at most half as large as the next
    grf_buf den_scratch, den_kept[40];
    int den_kept_count = 0;
    bool den_in_graphs = false;     // a captured call names the present block
    grf_buf pair_scratch;           // records of (row, node) pairs that the caller's workspace has no room for
    // host-buffer path
    grf_buf h_rowptr, h_col, h_w, h_q, h_k, h_v, h_out, h_ws;
    grf_features* h_feat = nullptr;
    // host-buffer path: phi(Q), phi(K), V are uploaded on one stream and the outputs downloaded on another, in
    // parts of a few problems each, beside the sampler and the attention of the other parts
    static constexpr int HOST_PARTS = 4;     // most parts grf_step_host splits a batch into
    cudaStream_t copy_stream = nullptr, down_stream = nullptr;
    cudaEvent_t up_done[HOST_PARTS] = {}, part_done[HOST_PARTS] = {}, down_done = nullptr;
    // small pinned host block for read-backs; [PINNED_EDGES]: edges of a graph whose records found no room, written by its sample
    static constexpr int PINNED_EDGES = 10;
    int32_t* pinned = nullptr;
    int* error_word = nullptr;      // device word set by a kernel that gave up a bounded wait
    bool use_tensor_cores = true;
    bool states_only = false;       // grf_masked_linear_attn never takes the mask (grf_ctx_use_tensor_cores(ctx, 2))
    bool tiles_only = false;        // state build and gather run on the tensor cores wherever the shape allows it (3)
    bool prefer_mask_route = false; // grf_step_host evaluates the attention over the materialised mask where it can
    bool check_graphs = false;      // grf_sample validates the device-resident CSR first (debugging aid)
    // optional per-launch timing
    bool timing = false;
    struct timed_launch { int cls; cudaEvent_t beg, end; };
    std::vector<timed_launch> timed;
    std::vector<cudaEvent_t> free_events;
};

// Brackets one kernel launch (or a short run of launches of one class) with events when timing is on.
struct grf_launch_scope {
    grf_ctx* ctx;
    int cls;
    int n;
    cudaEvent_t beg = nullptr, end = nullptr;
    grf_launch_scope(grf_ctx* c, int cls_, int n_launches = 1);
    ~grf_launch_scope();
};

struct grf_csr_dev {
    int32_t rows = 0, cols = 0;
    int64_t nnz = 0;
    grf_buf rowptr, col, val;
};

#define GRF_PLAN_BLOCK 128   // queries per block of the tensor-core gather kernel

// The deposits behind every entry of Phi (index 0) and Psi (index 1), kept when the sampler was asked to: entry p
// of the matrix owns deposits dep_ptr[p] .. dep_ptr[p+1]-1, each a (step t, load of the prefix) pair, in the
// order in which the sampler adds them.
struct grf_kept_walks {
    bool valid = false;
    int32_t n_walks = 0, max_len = 0;
    int64_t deposits[2] = {0, 0};
    grf_buf dep_ptr[2], dep_t[2], dep_load[2];
    bool perm_valid = false;        // psit_perm[x] = the entry of Psi that entry x of Psi^T copies (built by the first re-modulation)
    grf_buf psit_perm;
};

// The mask estimate Mhat = Phi Psi^T held as dense blocks: for every block of GRF_PLAN_BLOCK consecutive rows the
// sorted list of the keys j that any of its rows reaches (padded to a multiple of GRF_MASK_TILE with the last key
// and zero values; see GRF_MASK_SMALL) and the block's values in bf16, laid out [group of 16 keys][row of the block][16 keys].
#define GRF_MASK_TILE 64
// Up to this many keys a block's list is made of whole aligned tiles, all of them between its first and last key
// (attn_mhat_small.cu): at most eight.  Places of keys that no row of the block reaches are padding too: they hold another key.
#define GRF_MASK_SMALL 512
struct grf_mask_dev {
    bool ready = false;             // the blocks hold the mask of the present features
    bool requested = false;         // the caller asked for it (grf_features_materialise); else it is grf_masked_linear_attn's own
    bool refused = false;           // its blocks would be too large for the present structure: not tried again
    bool no_room = false;           // its memory could not be had for grf_masked_linear_attn, which then keeps to the states
    bool lists_ready = false;       // key sets, counts and sizes match the features' structure (what deciding the route needs)
    int64_t positions = 0;          // (node, key) pairs over all blocks, -1 when they passed 2^31
    int32_t longest = 0;            // longest key list of a block
    bool structure_ready = false;   // key lists (and positions) match the features' structure; values may be stale
    bool by_position = false;       // which of the two value kernels the structure serves
    int32_t blocks = 0;
    int64_t entries = 0;            // padded key entries over all blocks
    grf_buf off, cnt, key;          // cnt holds [blocks] padded counts, then [blocks] the blocks by decreasing count
    grf_buf bits;                   // per block one bit per key and the ranks, where positions are looked up row by row
    // build scratch: where each node's key positions start within its block, the positions, and per non-zero of Phi the
    // start of its node's positions
    grf_buf node_off, pos16, phi_pos;
    grf_buf totals;                 // sizes as the structure kernel adds them up
    grf_buf val;
};

// Where the kernels of a sample leave its sizes: non-zeros of Phi and Psi, deposits of both.  It belongs to the feature
// object, not to the context that samples, so whichever context and thread has the object can read them.
struct grf_size_slot {
    int32_t* host = nullptr;        // pinned
    cudaEvent_t ready = nullptr;    // behind the kernels that write them
    cudaEvent_t built = nullptr;    // behind what an attention call has built inside the object (grf_built_by)
};

struct grf_features {
    int device = 0;
    grf_csr_dev phi, psi, psit;
    grf_size_slot sizes;
    bool sizes_pending = false;     // nnz of the matrices is still to be read from `sizes` (grf_features_sizes)
    double expected_entries = 0.0;  // non-zeros per matrix that the walks leave at most on average (0: not sampled)
    uint64_t built_by = 0;          // context on whose stream sizes.built was recorded last
    bool sampled = false;           // holds, or has held, a sample
    grf_kept_walks kept;
    grf_mask_dev mask;
    // block plan of Phi: per block of GRF_PLAN_BLOCK rows, the sorted distinct columns
    grf_buf plan_off, plan_cnt, plan_col, plan_total;
    grf_buf plan_coef;              // dense bf16 coefficients [quad of union entries][row of the block][4]
    int32_t plan_blocks = 0;
    int64_t plan_entries = 0;       // node-list entries over all blocks (padded to multiples of 4)
    bool plan_ready = false;
    bool plan_coef_ready = false;   // the gather kernel's coefficient table exists for the present plan
    bool plan_stale = true;         // Phi changed since the plan was built: the gather kernel's launcher rebuilds it
    bool plan_settled = false;      // Phi has not changed at all since then, and the device had finished with it
};

int grf_buf_reserve(grf_buf* b, size_t bytes);          // grows (contents not preserved)
void grf_buf_release(grf_buf* b);
int grf_csr_reserve(grf_csr_dev* m, int32_t rows, int32_t cols, int64_t nnz_cap);
int grf_features_new(grf_features** out, int device);   // empty; `device` is current
void grf_features_clear(grf_features* feat);
bool grf_capturing(cudaStream_t stream);
// For as long as it lives this thread may allocate while a stream is captured.
struct grf_relaxed_capture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    grf_relaxed_capture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~grf_relaxed_capture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};
int grf_den_scratch(grf_ctx* ctx, int64_t count, float** den);
int grf_settle_sizes(grf_features* feat);
// before nnz of a matrix is read: waits for the sample's sizes if they have not been read yet
static inline int grf_features_sizes(const grf_features* feat)
{
    return feat->sizes_pending ? grf_settle_sizes(const_cast<grf_features*>(feat)) : GRF_OK;
}

// What a call builds inside an object (mask values, the gather's coefficients) is queued on that call's stream, and callers
// that see a const object cannot order other streams behind it.  grf_built_by: after such a build.  grf_wait_built: before a
// call uses or builds any of it; lets the stream wait if another context built last (whose stream then waited for the one
// before it).  A stream under capture neither records nor waits: who replays a graph orders it.
void grf_built_by(grf_ctx* ctx, grf_features* feat);
int grf_wait_for_build(grf_ctx* ctx, const grf_features* feat);
static inline int grf_wait_built(grf_ctx* ctx, const grf_features* feat)
{
    return feat->built_by == 0 || feat->built_by == ctx->id ? GRF_OK : grf_wait_for_build(ctx, feat);
}

// sample.cu
struct grf_walk_params {
    int32_t N, n_walks, max_len;
    uint32_t key0, key1, halt_threshold;
    float inv_keep, inv_n;
    int32_t cap;        // n_walks * (max_len + 1)
    int32_t seq_bits;   // ceil(log2(cap)), at least 1
    int32_t last_step[2];   // last step with a non-zero coefficient, per ensemble: no walk goes further
    float f[2][GRF_MAX_WALK_LEN + 1];
};
int grf_walk_params_init(grf_walk_params* p, int32_t N, uint64_t seed, int32_t n_walks, float p_halt,
                         int32_t max_len, const float* f_phi, const float* f_psi);

// scan.cu: exclusive scan of `segments` independent int32 arrays of length n each (in[s*n + i]) into
// out[s*(n+1) + i], with out[s*(n+1) + n] = total.
int grf_exclusive_scan(grf_ctx* ctx, const int32_t* in, int32_t* out, int32_t n, int32_t segments);

int grf_exclusive_scan_scratch(cudaStream_t stream, const int32_t* in, int32_t* out, int32_t n, int32_t segments,
                               int32_t* totals);

// The same for up to three arrays of one length n <= GRF_SCAN_DIRECT_MAX in one launch (in: 16-byte aligned): out[n] is the
// total, which also goes to host_total (pinned host memory); copy, if any, receives out[0 .. n-1] once more.
#define GRF_SCAN_DIRECT_MAX (1 << 18)
struct grf_scan_job { const int32_t* in; int32_t* out; int32_t* copy; int32_t* host_total; };
struct grf_scan_jobs { grf_scan_job job[3]; };
int grf_scan_jobs_launch(grf_ctx* ctx, cudaStream_t stream, const grf_scan_jobs& jobs, int count, int32_t n);

// transpose.cu
// Last step of a regrouping by column: every bucket of (row, value) pairs is ordered by row into t_col, t_val.  long_count
// (zero before) and long_list: scratch for the buckets too long to rank; rows bounds a bucket's length.
int grf_order_buckets(cudaStream_t stream, int32_t rows, int32_t cols, const int32_t* t_rowptr, int2* tmp, int32_t* long_count,
                      int32_t* long_list, int32_t* t_col, float* t_val);
int grf_reserve_buckets(grf_ctx* ctx, int64_t nnz);
int grf_transpose_launch(grf_ctx* ctx, int32_t rows, int32_t cols, int64_t nnz,
                         const int32_t* rowptr, const int32_t* col, const float* val,
                         int32_t* t_rowptr, int32_t* t_col, float* t_val);

// attn_state.cu / attn_gather.cu
// by_column: the states in the ALU gather's layout (below) instead of the tensor-core gather's records
int grf_build_states(grf_ctx* ctx, const grf_csr_dev& psit, int32_t G, int32_t N, int32_t m, int32_t d, int dtype,
                     const void* phiK, const void* V, void* states, bool by_column);
int grf_build_states_tc(grf_ctx* ctx, const grf_csr_dev& psit, int32_t G, int32_t N, int32_t m, int32_t d,
                        const void* phiK, const void* V, void* states, bool by_column);
int grf_gather_contract_alu(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d,
                            int dtype, const void* phiQ, const void* states, void* out, float* den_out);
// attn_pairs.cu
bool grf_pairs_shape(const grf_ctx* ctx, int32_t m, int32_t d);
double grf_pairs_ns(double nnz, int32_t G, int32_t m, int32_t d, int dtype, size_t workspace_per_problem);
double grf_states_by_rows_ns(double nnz, int32_t nodes, int32_t G, int32_t m, int32_t d, int dtype);
bool grf_pairs_fit(int64_t nnz, int dtype);
int grf_pairs_attn(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t G_all, int32_t N, int32_t m, int32_t d, int dtype, const void* phiQ,
                   const void* phiK, const void* V, void* out, float* den_out, void* workspace, size_t workspace_bytes);
// attn_mhat.cu
void grf_mask_invalidate(grf_features* feat);
void grf_mask_values_stale(grf_features* feat);
// Whether grf_masked_linear_attn evaluates this batch over the materialised mask; forms the mask when it does.
int grf_linear_by_mask(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d, int dtype,
                       bool* by_mask);
int grf_mhat_launch(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d, const void* phiQ,
                    const void* phiK, const void* V, void* out, float* den_out);
void grf_mask_release(grf_features* feat);
// attn_mhat_small.cu: the same for N <= GRF_MASK_SMALL; 1 (nothing launched) where no tensor map can be made of the operands
int grf_mhat_small_launch(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d, const void* phiQ,
                          const void* phiK, const void* V, void* out, float* den_out);
// attn_gather_tc.cu
int grf_build_block_plan(grf_ctx* ctx, grf_features* feat, bool with_coef = true);
int grf_ensure_block_plan(grf_ctx* ctx, const grf_features* feat, bool with_coef = true);   // builds it if Phi changed since the last build
// Estimated times in nanoseconds of the two gathers for a batch of G problems; the first needs the block plan's sizes.
double grf_gather_tiles_ns(const grf_features* feat, int32_t G, int32_t m);
double grf_gather_rows_ns(const grf_features* feat, int32_t G, int32_t m, int32_t d);
// Batches whose plain-ALU gather takes less than this gain nothing from a block plan, which alone takes half of it.
constexpr double GRF_PLAN_WORTH_NS = 30000.0;
// Which gather serves this object and shape (prepares the block plan it needs).
int grf_gather_by_tensor_cores(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t m, int32_t d, int dtype, bool* yes);
int grf_gather_contract_tc(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d,
                           const void* phiQ, const void* records, void* out, float* den_out);

// Where the states of one problem lie inside the workspace; R nodes, E = bytes of an element of T.
//
// For the tensor-core gather: one record per node, the state tile S_l (m x d), then z_l (m fp32 values), then z_l once more
// in bf16 (the denominators kernel reads that copy: half the bytes per (query, node) pair).  The tile is made of 16-byte
// chunks that hold 8 consecutive feature rows a of one column b, ordered [a / 8][b][a % 8]: the K-major, unswizzled
// shared-memory operand layout (8-row core matrices of 128 contiguous bytes), so a tile is brought in with one contiguous
// bulk copy.
//
// For the ALU gather (by column): all tiles first, each [b][a] so that any range of columns is contiguous, then all z_l in
// fp32; tiles and z_l start on whole cache lines.
//
// Both fit the R * (m d E + 4 m (+ 2 m with bf16)) bytes that a problem's workspace has.
template <typename T> __host__ __device__ constexpr int grf_tile_chunk() { return 16 / (int)sizeof(T); }
template <typename T> __host__ __device__ constexpr size_t grf_record_bytes(int M, int D)
{
    return (size_t)M * D * sizeof(T) + (size_t)M * sizeof(float) + (sizeof(T) == 2 ? (size_t)M * 2 : 0);
}
// bytes from one problem's states to the next one's
template <typename T> __host__ __device__ constexpr size_t grf_states_stride(size_t R, int M, int D)
{
    return (R * grf_record_bytes<T>(M, D) + 255) & ~(size_t)255;
}
// tile chunk holding feature rows a .. a + 7 (fp32: a + 3) of column b, and z_l, of node l
template <typename T> __host__ __device__ constexpr size_t grf_chunk_at(bool by_column, size_t l, int a, int b, int M, int D)
{
    constexpr int CH = grf_tile_chunk<T>();
    return by_column ? l * ((size_t)M * D * sizeof(T)) + ((size_t)b * M + a) * sizeof(T)
                     : l * grf_record_bytes<T>(M, D) + ((size_t)(a / CH) * D + b) * 16;
}
template <typename T> __host__ __device__ constexpr size_t grf_z_at(bool by_column, size_t l, size_t R, int M, int D)
{
    return by_column ? R * ((size_t)M * D * sizeof(T)) + l * ((size_t)M * sizeof(float))
                     : l * grf_record_bytes<T>(M, D) + (size_t)M * D * sizeof(T);
}

static inline int grf_ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }
