// C-ABI entry points that are not kernels themselves: contexts, buffers, feature objects, the
// attention driver (Alg. 1 step 5 in chunks of problems) and the host-buffer path.
#include <atomic>
#include <cstring>
#include <map>
#include <mutex>
#include <new>

#include <nvtx3/nvToolsExt.h>

#include "grf_internal.cuh"

// Device blocks that were given back, for the next object of about that size: making a feature object costs a dozen
// cudaMalloc calls otherwise (3 .. 300 ms on a busy host, against 1.5 ms for sampling and attention at N = 32768), and
// replacing one as many cudaFree calls.  At most POOL_BYTES per device; emptied when the last context goes and when
// an allocation fails.  A block is given back only after the device has finished with it, as with cudaFree.
namespace {

struct block_pool {
    static constexpr size_t POOL_BYTES = (size_t)1 << 30;
    static constexpr int DEVICES = 64;
    std::mutex lock;
    std::multimap<size_t, void*> blocks[DEVICES];
    size_t held[DEVICES] = {};
    // the same for the size slots of feature objects (pinning host memory waits for the device as well)
    static constexpr int SLOTS = 64;
    grf_size_slot slots[DEVICES][SLOTS];
    int slots_held[DEVICES] = {};
    int contexts = 0;

    void* take(int dev, size_t bytes, size_t* got)
    {
        std::lock_guard<std::mutex> g(lock);
        auto it = blocks[dev].lower_bound(bytes);
        if (it == blocks[dev].end() || it->first > bytes + bytes / 2 + 4096) return nullptr;
        void* p = it->second;
        *got = it->first;
        held[dev] -= it->first;
        blocks[dev].erase(it);
        return p;
    }
    bool put(int dev, void* p, size_t bytes)
    {
        std::lock_guard<std::mutex> g(lock);
        if (contexts == 0 || held[dev] + bytes > POOL_BYTES) return false;
        try { blocks[dev].emplace(bytes, p); }
        catch (const std::bad_alloc&) { return false; }
        held[dev] += bytes;
        return true;
    }
    void empty(int dev)
    {
        std::lock_guard<std::mutex> g(lock);
        for (auto& b : blocks[dev]) cudaFree(b.second);
        blocks[dev].clear();
        held[dev] = 0;
    }
    bool take_slot(int dev, grf_size_slot* s)
    {
        std::lock_guard<std::mutex> g(lock);
        if (slots_held[dev] == 0) return false;
        *s = slots[dev][--slots_held[dev]];
        return true;
    }
    bool put_slot(int dev, const grf_size_slot& s)
    {
        std::lock_guard<std::mutex> g(lock);
        if (contexts == 0 || slots_held[dev] == SLOTS) return false;
        slots[dev][slots_held[dev]++] = s;
        return true;
    }
};

void slot_destroy(grf_size_slot* s)
{
    if (s->ready) cudaEventDestroy(s->ready);
    if (s->built) cudaEventDestroy(s->built);
    if (s->host) cudaFreeHost(s->host);
    *s = grf_size_slot();
}

block_pool& pool() { static block_pool* p = new block_pool; return *p; }   // never destroyed: objects may outlive main()

int current_device()
{
    int dev = 0;
    return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < block_pool::DEVICES ? dev : -1;
}

// Makes a block's device current for as long as something is done with the block.
struct device_scope {
    int before;
    explicit device_scope(int dev) : before(current_device()) { if (dev >= 0 && dev != before) cudaSetDevice(dev); else before = -1; }
    ~device_scope() { if (before >= 0) cudaSetDevice(before); }
};

}  // namespace

// A buffer that already has a block grows on that block's device, whichever is current; an empty one takes the current.
int grf_buf_reserve(grf_buf* b, size_t bytes)
{
    if (bytes == 0) bytes = 1;
    if (b->bytes >= bytes) return GRF_OK;
    const device_scope scope(b->ptr ? b->device : -1);
    if (b->ptr) {
        cudaDeviceSynchronize();
        grf_buf_release(b);
    }
    // rounded up to an eighth of its power of two, so that blocks of nearly equal objects serve one another
    size_t step = 512;
    while (step * 16 < bytes) step *= 2;
    bytes = (bytes + step - 1) / step * step;
    const int dev = current_device();
    void* p = dev >= 0 ? pool().take(dev, bytes, &bytes) : nullptr;
    if (!p && cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
        if (dev >= 0) pool().empty(dev);
        if (cudaMalloc(&p, bytes) != cudaSuccess) { cudaGetLastError(); return GRF_ERR_NOMEM; }
    }
    b->ptr = p; b->bytes = bytes; b->device = dev;
    return GRF_OK;
}

// The device must have finished with the block: callers that cannot know it wait first.
void grf_buf_release(grf_buf* b)
{
    if (b->ptr && (b->device < 0 || !pool().put(b->device, b->ptr, b->bytes))) cudaFree(b->ptr);
    b->ptr = nullptr; b->bytes = 0;
}

int grf_features_new(grf_features** out, int device)
{
    grf_features* f = new (std::nothrow) grf_features();
    if (!f) return GRF_ERR_NOMEM;
    f->device = device;
    if (device >= block_pool::DEVICES || !pool().take_slot(device, &f->sizes)) {
        int rc = GRF_OK;
        if (cudaMallocHost((void**)&f->sizes.host, 64) != cudaSuccess) rc = GRF_ERR_NOMEM;
        else if (cudaEventCreateWithFlags(&f->sizes.ready, cudaEventDisableTiming) != cudaSuccess ||
                 cudaEventCreateWithFlags(&f->sizes.built, cudaEventDisableTiming) != cudaSuccess) rc = GRF_ERR_CUDA;
        if (rc != GRF_OK) {
            cudaGetLastError();
            slot_destroy(&f->sizes);
            delete f;
            return rc;
        }
    }
    *out = f;
    return GRF_OK;
}

// Empties an object (its buffers stay for the next sample): no call finds a matrix in it.
void grf_features_clear(grf_features* feat)
{
    for (grf_csr_dev* m : {&feat->phi, &feat->psi, &feat->psit}) { m->rows = m->cols = 0; m->nnz = 0; }
    feat->sizes_pending = false;
    feat->kept.valid = feat->kept.perm_valid = false;
    feat->plan_stale = true;
    feat->plan_ready = feat->plan_coef_ready = false;
    grf_mask_invalidate(feat);
}

int grf_settle_sizes(grf_features* feat)
{
    GRF_CUDA_TRY(cudaEventSynchronize(feat->sizes.ready));
    feat->phi.nnz = feat->sizes.host[0];
    feat->psi.nnz = feat->psit.nnz = feat->sizes.host[1];
    feat->sizes_pending = false;
    return GRF_OK;
}

bool grf_capturing(cudaStream_t stream)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
    cudaGetLastError();                                 // the default stream, while another one is captured
    return true;
}

// Room for denominators that nobody asked for.  A graph goes on naming the block that it was captured with: such a block stays until
// the context goes, and a larger call takes another one, at least twice as large (so that there are few).  A captured call may
// be the first that needs one: eager calls of its shape may have taken another route.
int grf_den_scratch(grf_ctx* ctx, int64_t count, float** den)
{
    const size_t bytes = sizeof(float) * (size_t)count;
    const bool captured = grf_capturing(ctx->stream);
    grf_buf& b = ctx->den_scratch;
    if (b.bytes < bytes && (captured || ctx->den_in_graphs)) {
        constexpr int KEPT = sizeof(ctx->den_kept) / sizeof(ctx->den_kept[0]);
        if (ctx->den_kept_count == KEPT) return GRF_ERR_NOMEM;
        const grf_relaxed_capture relaxed;
        grf_buf larger;
        GRF_TRY(grf_buf_reserve(&larger, bytes > 2 * b.bytes ? bytes : 2 * b.bytes));
        if (b.ptr) ctx->den_kept[ctx->den_kept_count++] = b;
        b = larger;
        ctx->den_in_graphs = false;
    }
    GRF_TRY(grf_buf_reserve(&b, bytes));
    if (captured) ctx->den_in_graphs = true;
    *den = (float*)b.ptr;
    return GRF_OK;
}

void grf_built_by(grf_ctx* ctx, grf_features* feat)
{
    if (grf_capturing(ctx->stream)) return;
    if (cudaEventRecord(feat->sizes.built, ctx->stream) == cudaSuccess) feat->built_by = ctx->id;
}

int grf_wait_for_build(grf_ctx* ctx, const grf_features* feat)
{
    if (!grf_capturing(ctx->stream)) GRF_CUDA_TRY(cudaStreamWaitEvent(ctx->stream, feat->sizes.built, 0));
    return GRF_OK;
}

int grf_csr_reserve(grf_csr_dev* m, int32_t rows, int32_t cols, int64_t nnz_cap)
{
    m->rows = rows; m->cols = cols;
    GRF_TRY(grf_buf_reserve(&m->rowptr, sizeof(int32_t) * ((size_t)rows + 1)));
    GRF_TRY(grf_buf_reserve(&m->col, sizeof(int32_t) * (size_t)(nnz_cap > 0 ? nnz_cap : 1)));
    GRF_TRY(grf_buf_reserve(&m->val, sizeof(float) * (size_t)(nnz_cap > 0 ? nnz_cap : 1)));
    return GRF_OK;
}

extern "C" int grf_ctx_create(grf_ctx** out, int device, void* cuda_stream)
{
    if (!out || device < 0) return GRF_ERR_INVALID;
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || device >= count) { cudaGetLastError(); return GRF_ERR_CUDA; }
    GRF_CUDA_TRY(cudaSetDevice(device));
    grf_ctx* c = new (std::nothrow) grf_ctx();
    if (!c) return GRF_ERR_NOMEM;
    static std::atomic<uint64_t> contexts_made{0};
    c->id = ++contexts_made;
    c->device = device;
    c->stream = (cudaStream_t)cuda_stream;
    if (cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaMallocHost((void**)&c->pinned, 64) != cudaSuccess ||
        cudaMalloc((void**)&c->error_word, 2 * sizeof(int)) != cudaSuccess ||
        cudaMemset(c->error_word, 0, 2 * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return GRF_ERR_CUDA;
    }
    memset(c->pinned, 0, 64);
    {
        std::lock_guard<std::mutex> g(pool().lock);
        ++pool().contexts;
    }
    *out = c;
    return GRF_OK;
}

extern "C" int grf_ctx_destroy(grf_ctx* ctx)
{
    if (!ctx) return GRF_ERR_INVALID;
    cudaSetDevice(ctx->device);
    cudaDeviceSynchronize();
    grf_buf* bufs[] = {&ctx->edge_records, &ctx->stage_col, &ctx->stage_val, &ctx->counts, &ctx->scan_blocks,
                       &ctx->stage_dep_start, &ctx->stage_dep_t, &ctx->stage_dep_load, &ctx->dep_counts, &ctx->dep_rowptr2,
                       &ctx->t_cursor, &ctx->t_tmp, &ctx->den_scratch, &ctx->pair_scratch, &ctx->h_rowptr, &ctx->h_col, &ctx->h_w,
                       &ctx->h_q, &ctx->h_k, &ctx->h_v, &ctx->h_out, &ctx->h_ws};
    for (grf_buf* b : bufs) grf_buf_release(b);
    for (grf_buf& b : ctx->den_kept) grf_buf_release(&b);
    if (ctx->h_feat) grf_features_free(ctx->h_feat);
    if (ctx->pinned) cudaFreeHost(ctx->pinned);
    if (ctx->error_word) cudaFree(ctx->error_word);
    if (ctx->copy_stream) {
        cudaStreamSynchronize(ctx->copy_stream); cudaStreamSynchronize(ctx->down_stream);
        cudaStreamDestroy(ctx->copy_stream); cudaStreamDestroy(ctx->down_stream);
        for (int p = 0; p < grf_ctx::HOST_PARTS; ++p) { cudaEventDestroy(ctx->up_done[p]); cudaEventDestroy(ctx->part_done[p]); }
        cudaEventDestroy(ctx->down_done);
    }
    for (auto& t : ctx->timed) { cudaEventDestroy(t.beg); cudaEventDestroy(t.end); }
    for (cudaEvent_t e : ctx->free_events) cudaEventDestroy(e);
    delete ctx;
    bool last = false, holds[block_pool::DEVICES];
    {
        std::lock_guard<std::mutex> g(pool().lock);
        last = --pool().contexts == 0;
        for (int dev = 0; dev < block_pool::DEVICES; ++dev) holds[dev] = pool().held[dev] > 0 || pool().slots_held[dev] > 0;
    }
    if (last) {
        int before = 0;
        cudaGetDevice(&before);
        for (int dev = 0; dev < block_pool::DEVICES; ++dev)
            if (holds[dev] && cudaSetDevice(dev) == cudaSuccess) {
                pool().empty(dev);
                for (grf_size_slot s; pool().take_slot(dev, &s);) slot_destroy(&s);
            }
        cudaSetDevice(before);
    }
    return GRF_OK;
}

static cudaEvent_t take_event(grf_ctx* c)
{
    if (!c->free_events.empty()) { cudaEvent_t e = c->free_events.back(); c->free_events.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return e;
}

// names of the kernel classes, as ranges in a profiler's timeline
static const char* const kernel_class_names[GRF_KERNEL_CLASSES] = {
    "grf:walk_merge", "grf:scan", "grf:compact", "grf:regroup", "grf:build_states", "grf:gather_contract",
    "grf:row_denominators", "grf:block_plan", "grf:mask_build", "grf:mhat_attention"};

grf_launch_scope::grf_launch_scope(grf_ctx* c, int cls_, int n_launches) : ctx(c), cls(cls_), n(n_launches)
{
    nvtxRangePushA(kernel_class_names[cls]);     // costs nothing unless a tool is attached
    if (!ctx->timing) return;
    beg = take_event(ctx); end = take_event(ctx);
    if (beg && end) cudaEventRecord(beg, ctx->stream);
}

grf_launch_scope::~grf_launch_scope()
{
    nvtxRangePop();
    ctx->launches += n;
    if (!ctx->timing || !beg || !end) return;
    cudaEventRecord(end, ctx->stream);
    try { ctx->timed.push_back({cls, beg, end}); }
    catch (const std::bad_alloc&) { cudaEventDestroy(beg); cudaEventDestroy(end); }     // this launch goes untimed
}

extern "C" int grf_ctx_use_tensor_cores(grf_ctx* ctx, int enable)
{
    if (!ctx) return GRF_ERR_INVALID;
    ctx->use_tensor_cores = enable != 0;
    ctx->states_only = enable == 2 || enable == 3;
    ctx->tiles_only = enable == 3;
    return GRF_OK;
}

extern "C" int grf_ctx_prefer_mask_route(grf_ctx* ctx, int enable)
{
    if (!ctx) return GRF_ERR_INVALID;
    ctx->prefer_mask_route = enable != 0;
    return GRF_OK;
}

extern "C" int grf_ctx_check_graphs(grf_ctx* ctx, int enable)
{
    if (!ctx) return GRF_ERR_INVALID;
    ctx->check_graphs = enable != 0;
    return GRF_OK;
}

extern "C" int grf_ctx_check(grf_ctx* ctx)
{
    if (!ctx) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_CUDA_TRY(cudaMemcpyAsync(ctx->pinned + 8, ctx->error_word, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    GRF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    if (ctx->pinned[8] != 0) {
        cudaMemsetAsync(ctx->error_word, 0, sizeof(int), ctx->stream);
        return GRF_ERR_TIMEOUT;
    }
    return GRF_OK;
}

extern "C" int grf_ctx_enable_timing(grf_ctx* ctx, int enable)
{
    if (!ctx) return GRF_ERR_INVALID;
    ctx->timing = enable != 0;
    return GRF_OK;
}

extern "C" int grf_ctx_kernel_times(grf_ctx* ctx, float* ms, int64_t* launches)
{
    if (!ctx || !ms || !launches) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    for (int k = 0; k < GRF_KERNEL_CLASSES; ++k) { ms[k] = 0.0f; launches[k] = 0; }
    for (auto& t : ctx->timed) {
        float x = 0.0f;
        if (cudaEventElapsedTime(&x, t.beg, t.end) == cudaSuccess) { ms[t.cls] += x; launches[t.cls] += 1; }
        for (cudaEvent_t e : {t.beg, t.end}) {
            try { ctx->free_events.push_back(e); }
            catch (const std::bad_alloc&) { cudaEventDestroy(e); }
        }
    }
    ctx->timed.clear();
    cudaGetLastError();
    return GRF_OK;
}

extern "C" int64_t grf_ctx_launch_count(const grf_ctx* ctx) { return ctx ? ctx->launches : -1; }

extern "C" int grf_deconvolve(const double* alpha, int32_t len, double* f_out)
{
    if (!alpha || !f_out || len < 1 || !(alpha[0] > 0.0)) return GRF_ERR_INVALID;
    // sum_{p=0..k} f_p f_{k-p} = alpha_k  =>  f_0 = sqrt(alpha_0), then solve for f_k (Remark 3.1)
    f_out[0] = sqrt(alpha[0]);
    for (int32_t k = 1; k < len; ++k) {
        double cross = 0.0;
        for (int32_t p = 1; p < k; ++p) cross += f_out[p] * f_out[k - p];
        f_out[k] = (alpha[k] - cross) / (2.0 * f_out[0]);
    }
    return GRF_OK;
}

extern "C" int grf_attn_flops(const grf_features* feat, int32_t m, int32_t d, int64_t* masked,
                              int64_t* unmasked_linear, int64_t* softmax)
{
    if (!feat || m <= 0 || d <= 0) return GRF_ERR_INVALID;
    GRF_TRY(grf_features_sizes(feat));
    const int64_t N = feat->phi.rows;
    const int64_t per_nonzero = (int64_t)m + 2 * (int64_t)m * (d + 1);     // scale phi(.), then multiply-add into [S_l | z_l]
    if (masked) *masked = (feat->phi.nnz + feat->psit.nnz) * per_nonzero + N * d;
    if (unmasked_linear) *unmasked_linear = 4 * N * m * (d + 1) + N * d;
    if (softmax) *softmax = N * N * (2 * (int64_t)m + 2 + 2 * (int64_t)d) + N * d;
    return GRF_OK;
}

static void csr_release(grf_csr_dev* m)
{
    grf_buf_release(&m->rowptr); grf_buf_release(&m->col); grf_buf_release(&m->val);
}

extern "C" int grf_features_free(grf_features* feat)
{
    if (!feat) return GRF_ERR_INVALID;
    cudaSetDevice(feat->device);
    cudaDeviceSynchronize();                        // its buffers may serve another object next
    csr_release(&feat->phi); csr_release(&feat->psi); csr_release(&feat->psit);
    grf_buf_release(&feat->plan_off); grf_buf_release(&feat->plan_cnt);
    grf_buf_release(&feat->plan_col); grf_buf_release(&feat->plan_total); grf_buf_release(&feat->plan_coef);
    grf_mask_release(feat);
    for (int e = 0; e < 2; ++e) {
        grf_buf_release(&feat->kept.dep_ptr[e]); grf_buf_release(&feat->kept.dep_t[e]); grf_buf_release(&feat->kept.dep_load[e]);
    }
    grf_buf_release(&feat->kept.psit_perm);
    if (feat->device >= block_pool::DEVICES || !pool().put_slot(feat->device, feat->sizes)) slot_destroy(&feat->sizes);
    delete feat;
    return GRF_OK;
}

extern "C" int grf_features_view(const grf_features* feat, int which, int32_t* rows, int32_t* cols, int64_t* nnz,
                                 const int32_t** rowptr, const int32_t** col, const float** val)
{
    if (!feat || which < 0 || which > 2) return GRF_ERR_INVALID;
    GRF_TRY(grf_features_sizes(feat));
    const grf_csr_dev& m = which == 0 ? feat->phi : (which == 1 ? feat->psi : feat->psit);
    if (rows) *rows = m.rows;
    if (cols) *cols = m.cols;
    if (nnz) *nnz = m.nnz;
    if (rowptr) *rowptr = (const int32_t*)m.rowptr.ptr;
    if (col) *col = (const int32_t*)m.col.ptr;
    if (val) *val = (const float*)m.val.ptr;
    return GRF_OK;
}

extern "C" int grf_features_copy(grf_ctx* ctx, const grf_features* feat, int which, int32_t* rowptr, int32_t* col,
                                 float* val)
{
    if (!ctx || !feat || which < 0 || which > 2 || !rowptr) return GRF_ERR_INVALID;
    GRF_TRY(grf_features_sizes(feat));
    const grf_csr_dev& m = which == 0 ? feat->phi : (which == 1 ? feat->psi : feat->psit);
    if (m.rows == 0 || (m.nnz > 0 && (!col || !val))) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_CUDA_TRY(cudaMemcpyAsync(rowptr, m.rowptr.ptr, sizeof(int32_t) * ((size_t)m.rows + 1), cudaMemcpyDeviceToDevice,
                                 ctx->stream));
    if (m.nnz > 0) {
        GRF_CUDA_TRY(cudaMemcpyAsync(col, m.col.ptr, sizeof(int32_t) * (size_t)m.nnz, cudaMemcpyDeviceToDevice, ctx->stream));
        GRF_CUDA_TRY(cudaMemcpyAsync(val, m.val.ptr, sizeof(float) * (size_t)m.nnz, cudaMemcpyDeviceToDevice, ctx->stream));
    }
    return GRF_OK;
}

extern "C" int grf_features_from_csr(grf_ctx* ctx, int32_t N, int32_t R,
                                     const int32_t* phi_rowptr, const int32_t* phi_col, const float* phi_val,
                                     const int32_t* psi_rowptr, const int32_t* psi_col, const float* psi_val,
                                     grf_features** out)
{
    if (!ctx || !out || N <= 0 || R <= 0 || !phi_rowptr || !psi_rowptr) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_CUDA_TRY(cudaMemcpyAsync(ctx->pinned + 0, phi_rowptr + N, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    GRF_CUDA_TRY(cudaMemcpyAsync(ctx->pinned + 1, psi_rowptr + N, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    GRF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    const int64_t nnz_phi = ctx->pinned[0], nnz_psi = ctx->pinned[1];
    if (nnz_phi < 0 || nnz_psi < 0) return GRF_ERR_INVALID;
    if ((nnz_phi > 0 && (!phi_col || !phi_val)) || (nnz_psi > 0 && (!psi_col || !psi_val))) return GRF_ERR_INVALID;
    grf_features* f = nullptr;
    GRF_TRY(grf_features_new(&f, ctx->device));
    int rc = grf_csr_reserve(&f->phi, N, R, nnz_phi);
    if (rc == GRF_OK) rc = grf_csr_reserve(&f->psi, N, R, nnz_psi);
    if (rc == GRF_OK) rc = grf_csr_reserve(&f->psit, R, N, nnz_psi);
    if (rc != GRF_OK) { grf_features_free(f); return rc; }
    f->phi.nnz = nnz_phi; f->psi.nnz = nnz_psi; f->psit.nnz = nnz_psi;
    auto copy = [&](grf_csr_dev& m, const int32_t* rp, const int32_t* c, const float* v, int64_t nnz) {
        cudaMemcpyAsync(m.rowptr.ptr, rp, sizeof(int32_t) * ((size_t)N + 1), cudaMemcpyDeviceToDevice, ctx->stream);
        if (nnz > 0) {
            cudaMemcpyAsync(m.col.ptr, c, sizeof(int32_t) * (size_t)nnz, cudaMemcpyDeviceToDevice, ctx->stream);
            cudaMemcpyAsync(m.val.ptr, v, sizeof(float) * (size_t)nnz, cudaMemcpyDeviceToDevice, ctx->stream);
        }
    };
    copy(f->phi, phi_rowptr, phi_col, phi_val, nnz_phi);
    copy(f->psi, psi_rowptr, psi_col, psi_val, nnz_psi);
    rc = grf_transpose_launch(ctx, N, R, nnz_psi, (const int32_t*)f->psi.rowptr.ptr, (const int32_t*)f->psi.col.ptr,
                              (const float*)f->psi.val.ptr, (int32_t*)f->psit.rowptr.ptr,
                              (int32_t*)f->psit.col.ptr, (float*)f->psit.val.ptr);
    if (rc == GRF_OK) { f->plan_stale = true; f->plan_ready = false; }   // built at the first attention that needs it
    if (rc == GRF_OK && cudaGetLastError() != cudaSuccess) rc = GRF_ERR_CUDA;
    if (rc != GRF_OK) { grf_features_free(f); return rc; }
    *out = f;
    return GRF_OK;
}

static bool dim_ok(int32_t x) { return x == 8 || x == 16 || x == 32 || x == 64 || x == 128; }
static size_t elem_size(int dtype) { return dtype == GRF_DTYPE_F32 ? 4 : 2; }
static bool aligned16(const void* a, const void* b, const void* c, const void* d)
{
    return (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 15u) == 0;
}
static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// per-problem workspace, 256-byte aligned
static size_t ws_per_problem(int32_t R, int32_t m, int32_t d, int dtype)
{
    // per node: the state tile, z (fp32) and, with bf16 storage, room for z once more in bf16
    return align256((size_t)R * ((size_t)m * d * elem_size(dtype) + (size_t)m * sizeof(float) +
                                 (dtype == GRF_DTYPE_BF16 ? (size_t)m * 2 : 0)));
}

extern "C" size_t grf_attn_workspace_bytes(int32_t G, int32_t R, int32_t m, int32_t d, int dtype)
{
    if (G <= 0 || R <= 0 || !dim_ok(m) || !dim_ok(d) || (dtype != GRF_DTYPE_F32 && dtype != GRF_DTYPE_BF16)) return 0;
    return ws_per_problem(R, m, d, dtype) * (size_t)G;
}

// The tensor-core build takes 35 us at least (a bucket's chain of segments); the plain one 8 us and 0.27 ns per non-zero
// and problem at m = 32, d = 64.  us measured, plain / tensor cores: lattice of 400 nodes, 4 problems 10 / 36, grid of
// 196, 8 problems 29 / 44, expander of 1024, 2 problems, m = 16 29 / 44, 4 problems, m = 32 69 / 47.
static double plain_build_ns(const grf_features* feat, int32_t G, int32_t m, int32_t d)
{
    return 0.27 * ((double)m * d + 512.0) / 2560.0 * (double)G * (double)feat->psit.nnz;
}
constexpr double PLAIN_BUILD_WORTH_NS = 25000.0;

// Whether the states of a batch are used where they are made (attn_pairs.cu) instead of being stored and gathered.  Decided by
// the features' sizes, the shape and the whole batch's G_all, so that parts of a batch give the bits of the whole.  The sizes
// of a sample whose kernels may still be running are waited for only where its walks' expectation leaves the choice open.  A
// call under stream capture keeps to whole states, which need the caller's memory and denominators (grf_den_scratch): the pairs lie in
// buffers of the context that a later call may replace while the graph still names them, and their places and launches follow the number of non-zeros,
// which a graph would keep while the kernels of whole states read the row pointers of whatever sample the object then holds.
static int states_by_pairs(grf_ctx* ctx, const grf_features* feat, int32_t G_all, int32_t m, int32_t d, int dtype, const void* phiQ,
                           const void* phiK, const void* V, const void* out, bool* yes)
{
    *yes = false;
    if (!grf_pairs_shape(ctx, m, d) || !aligned16(phiQ, phiK, V, out)) return GRF_OK;
    const size_t per = ws_per_problem(feat->phi.cols, m, d, dtype);
    auto cheaper = [&](double nnz) {
        return grf_pairs_ns(nnz, G_all, m, d, dtype, per) < grf_states_by_rows_ns(nnz, feat->phi.cols, G_all, m, d, dtype);
    };
    if (feat->sizes_pending && !cheaper(feat->expected_entries)) return GRF_OK;
    if (grf_capturing(ctx->stream)) return GRF_OK;
    GRF_TRY(grf_features_sizes(feat));
    const double nnz = 0.5 * ((double)feat->phi.nnz + (double)feat->psit.nnz);
    if (!cheaper(nnz) || !grf_pairs_fit(feat->phi.nnz, dtype)) return GRF_OK;
    if (dtype == GRF_DTYPE_BF16) {
        // (the plain build of small batches does not round Psi phi(k) to bf16: outputs 2.0e-3 off fp64 against 2.05e-3)
        if (plain_build_ns(feat, G_all, m, d) <= PLAIN_BUILD_WORTH_NS) return GRF_OK;
        // whole states by tiles, where rows of a block share their nodes
        GRF_TRY(grf_ensure_block_plan(ctx, feat, false));
        if (feat->plan_ready && grf_gather_tiles_ns(feat, G_all, m) + 45000.0 + G_all * nnz * (0.03 + 0.001 * m) <
                                    grf_pairs_ns(nnz, G_all, m, d, dtype, per)) return GRF_OK;
    }
    *yes = true;
    return GRF_OK;
}

// The attention of G problems once the route is known: over the mask in one launch, or through the per-node states in
// chunks of as many problems as the workspace holds.  G_all is the size of the whole batch that they belong to: it picks
// the kernels, so that parts of a batch give the bits of the whole.
static int linear_attn(grf_ctx* ctx, const grf_features* feat, bool by_mask, int32_t G_all, int32_t G, int32_t N, int32_t m, int32_t d,
                       int dtype, const void* phiQ, const void* phiK, const void* V, void* out, float* den_out,
                       void* workspace, size_t workspace_bytes)
{
    if (by_mask) return grf_mhat_launch(ctx, feat, G, N, m, d, phiQ, phiK, V, out, den_out);
    bool by_pairs = false;
    GRF_TRY(states_by_pairs(ctx, feat, G_all, m, d, dtype, phiQ, phiK, V, out, &by_pairs));
    if (by_pairs) {
        const int rc = grf_pairs_attn(ctx, feat, G, G_all, N, m, d, dtype, phiQ, phiK, V, out, den_out, workspace, workspace_bytes);
        if (rc != GRF_ERR_NOMEM) return rc;                     // its scratch could not be had: whole states need none
    }
    const size_t per = ws_per_problem(feat->phi.cols, m, d, dtype);
    int64_t chunk = (int64_t)(workspace_bytes / per);
    if (chunk > G) chunk = G;
    if (chunk > 65535) chunk = 65535;
    const size_t es = elem_size(dtype);
    // the plan's build waits for the stream once: do it before the attention kernels are queued, not between them
    bool tc_gather = false;
    const bool tensor_cores = dtype == GRF_DTYPE_BF16 && ctx->use_tensor_cores;
    if (tensor_cores) GRF_TRY(grf_features_sizes(feat));        // the choices below read them
    const bool tc_states = tensor_cores && (plain_build_ns(feat, G_all, m, d) > PLAIN_BUILD_WORTH_NS || ctx->tiles_only);
    GRF_TRY(grf_gather_by_tensor_cores(ctx, feat, G_all, m, d, dtype, &tc_gather));
    for (int64_t g0 = 0; g0 < G; g0 += chunk) {
        const int32_t gc = (int32_t)((G - g0) < chunk ? (G - g0) : chunk);
        const char* k_ptr = (const char*)phiK + (size_t)g0 * N * m * es;
        const char* v_ptr = (const char*)V + (size_t)g0 * N * d * es;
        const char* q_ptr = (const char*)phiQ + (size_t)g0 * N * m * es;
        char* o_ptr = (char*)out + (size_t)g0 * N * d * es;
        float* den_ptr = den_out ? den_out + (size_t)g0 * N : nullptr;
        int rs = 1;
        if (tc_states)
            rs = grf_build_states_tc(ctx, feat->psit, gc, N, m, d, k_ptr, v_ptr, workspace, !tc_gather);
        if (rs > 0) rs = grf_build_states(ctx, feat->psit, gc, N, m, d, dtype, k_ptr, v_ptr, workspace, !tc_gather);
        GRF_TRY(rs);
        if (tc_gather) GRF_TRY(grf_gather_contract_tc(ctx, feat, gc, N, m, d, q_ptr, workspace, o_ptr, den_ptr));
        else GRF_TRY(grf_gather_contract_alu(ctx, feat, gc, N, m, d, dtype, q_ptr, workspace, o_ptr, den_ptr));
    }
    return GRF_OK;
}

extern "C" int grf_masked_linear_attn(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m,
                                      int32_t d, int dtype, const void* phiQ, const void* phiK, const void* V,
                                      void* out, float* den_out, void* workspace, size_t workspace_bytes)
{
    if (!ctx || !feat || !phiQ || !phiK || !V || !out || !workspace) return GRF_ERR_INVALID;
    if (G <= 0 || N <= 0 || !dim_ok(m) || !dim_ok(d)) return GRF_ERR_INVALID;
    if (dtype != GRF_DTYPE_F32 && dtype != GRF_DTYPE_BF16) return GRF_ERR_INVALID;
    if (feat->phi.rows != N || feat->psit.cols != N || feat->phi.cols != feat->psit.rows) return GRF_ERR_INVALID;
    if (((uintptr_t)workspace & 255) != 0) return GRF_ERR_INVALID;
    const int32_t R = feat->phi.cols;
    const size_t per = ws_per_problem(R, m, d, dtype);
    if (workspace_bytes < per) return GRF_ERR_WORKSPACE;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_TRY(grf_wait_built(ctx, feat));
    bool by_mask = false;
    if (aligned16(phiQ, phiK, V, out)) GRF_TRY(grf_linear_by_mask(ctx, feat, G, N, m, d, dtype, &by_mask));
    return linear_attn(ctx, feat, by_mask, G, G, N, m, d, dtype, phiQ, phiK, V, out, den_out, workspace, workspace_bytes);
}

static int check_graph_host(int32_t N, const int32_t* rowptr, const int32_t* col)
{
    if (rowptr[0] != 0) return GRF_ERR_BADGRAPH;
    for (int32_t i = 0; i < N; ++i)
        if (rowptr[i + 1] < rowptr[i]) return GRF_ERR_BADGRAPH;
    const int64_t E = rowptr[N];
    for (int64_t p = 0; p < E; ++p)
        if (col[p] < 0 || col[p] >= N) return GRF_ERR_BADGRAPH;
    return GRF_OK;
}

static int step_host(grf_ctx* ctx, int32_t N, const int32_t* rowptr, const int32_t* col, const float* w, uint64_t seed,
                     int32_t n_walks, float p_halt, int32_t max_len, const float* f_phi, const float* f_psi, int32_t G, int32_t m,
                     int32_t d, int dtype, const void* phiQ, const void* phiK, const void* V, void* out)
{
    if (!ctx || !rowptr || !col || !w || !phiQ || !phiK || !V || !out || N <= 0 || G <= 0) return GRF_ERR_INVALID;
    if (!dim_ok(m) || !dim_ok(d) || (dtype != GRF_DTYPE_F32 && dtype != GRF_DTYPE_BF16)) return GRF_ERR_INVALID;
    GRF_TRY(check_graph_host(N, rowptr, col));
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    const size_t E = (size_t)rowptr[N], es = elem_size(dtype);
    const size_t qk_bytes = (size_t)G * N * m * es, v_bytes = (size_t)G * N * d * es;
    GRF_TRY(grf_buf_reserve(&ctx->h_rowptr, ((size_t)N + 1) * 4));
    GRF_TRY(grf_buf_reserve(&ctx->h_col, E * 4));
    GRF_TRY(grf_buf_reserve(&ctx->h_w, E * 4));
    GRF_TRY(grf_buf_reserve(&ctx->h_q, qk_bytes));
    GRF_TRY(grf_buf_reserve(&ctx->h_k, qk_bytes));
    GRF_TRY(grf_buf_reserve(&ctx->h_v, v_bytes));
    GRF_TRY(grf_buf_reserve(&ctx->h_out, v_bytes));
    cudaStream_t s = ctx->stream;
    GRF_CUDA_TRY(cudaMemcpyAsync(ctx->h_rowptr.ptr, rowptr, ((size_t)N + 1) * 4, cudaMemcpyHostToDevice, s));
    if (E > 0) {
        GRF_CUDA_TRY(cudaMemcpyAsync(ctx->h_col.ptr, col, E * 4, cudaMemcpyHostToDevice, s));
        GRF_CUDA_TRY(cudaMemcpyAsync(ctx->h_w.ptr, w, E * 4, cudaMemcpyHostToDevice, s));
    }
    // The problems are handled in parts: the inputs of part p travel on a second stream while the features are
    // sampled and the earlier parts are computed; its outputs leave on a third stream while the next part runs.
    if (!ctx->copy_stream) {
        GRF_CUDA_TRY(cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
        GRF_CUDA_TRY(cudaStreamCreateWithFlags(&ctx->down_stream, cudaStreamNonBlocking));
        for (int p = 0; p < grf_ctx::HOST_PARTS; ++p) {
            GRF_CUDA_TRY(cudaEventCreateWithFlags(&ctx->up_done[p], cudaEventDisableTiming));
            GRF_CUDA_TRY(cudaEventCreateWithFlags(&ctx->part_done[p], cudaEventDisableTiming));
        }
        GRF_CUDA_TRY(cudaEventCreateWithFlags(&ctx->down_done, cudaEventDisableTiming));
    }
    const int want_parts = grf_ctx::HOST_PARTS;
    const int parts = G >= 2 * want_parts ? want_parts : (G >= 2 ? 2 : 1);
    const int32_t gp = (G + parts - 1) / parts;           // problems per part
    for (int p = 0; p < parts; ++p) {
        const int32_t g0 = p * gp, gc = g0 + gp <= G ? gp : G - g0;
        if (gc <= 0) break;
        const size_t qo = (size_t)g0 * N * m * es, vo = (size_t)g0 * N * d * es;
        const size_t qb = (size_t)gc * N * m * es, vb = (size_t)gc * N * d * es;
        GRF_CUDA_TRY(cudaMemcpyAsync((char*)ctx->h_q.ptr + qo, (const char*)phiQ + qo, qb, cudaMemcpyHostToDevice, ctx->copy_stream));
        GRF_CUDA_TRY(cudaMemcpyAsync((char*)ctx->h_k.ptr + qo, (const char*)phiK + qo, qb, cudaMemcpyHostToDevice, ctx->copy_stream));
        GRF_CUDA_TRY(cudaMemcpyAsync((char*)ctx->h_v.ptr + vo, (const char*)V + vo, vb, cudaMemcpyHostToDevice, ctx->copy_stream));
        GRF_CUDA_TRY(cudaEventRecord(ctx->up_done[p], ctx->copy_stream));
    }
    GRF_TRY(grf_sample(ctx, N, (const int32_t*)ctx->h_rowptr.ptr, (const int32_t*)ctx->h_col.ptr,
                       (const float*)ctx->h_w.ptr, seed, n_walks, p_halt, max_len, f_phi, f_psi, &ctx->h_feat));
    // route: over the materialised mask when the caller prefers it and the shape and the graph allow it, or when the
    // whole batch is cheaper that way (the parts below follow one decision, so the split does not change the bits)
    bool by_mask = false;
    if (ctx->prefer_mask_route && dtype == GRF_DTYPE_BF16 && d == 64 && (m == 16 || m == 32 || m == 64)) {
        const int rc = grf_features_materialise(ctx, ctx->h_feat);
        if (rc == GRF_OK) by_mask = true;
        else if (rc == GRF_ERR_NOMEM) { cudaDeviceSynchronize(); grf_mask_release(ctx->h_feat); }     // the states need less
        else if (rc != GRF_ERR_TOO_LARGE) return rc;          // too large = no locality: the S/z route serves it
    } else {
        GRF_TRY(grf_linear_by_mask(ctx, ctx->h_feat, G, N, m, d, dtype, &by_mask));
    }
    // Inputs always travel in the parts above.  The attention follows part by part over the mask (it is short, so most of
    // the outputs leave while later parts are computed), and in two steps through the per-node states, whose kernels lose
    // more on small batches than the finer overlap returns.
    const int per_step = by_mask ? 1 : (parts + 1) / 2;        // upload parts per attention step
    const int32_t gs = gp * per_step;
    // workspace: one part's records if that is modest, else chunks of about 1 GiB
    const size_t per = by_mask ? 256 : ws_per_problem(N, m, d, dtype);
    size_t want = per * (size_t)(gs < G ? gs : G);
    const size_t cap = (size_t)1 << 31;
    if (want > cap) want = per * (cap / per > 0 ? cap / per : 1);
    GRF_TRY(grf_buf_reserve(&ctx->h_ws, want));
    for (int p = 0; p * per_step < parts; ++p) {
        const int32_t g0 = p * gs, gc = g0 + gs <= G ? gs : G - g0;
        if (gc <= 0) break;
        const size_t qo = (size_t)g0 * N * m * es, vo = (size_t)g0 * N * d * es;
        for (int u = p * per_step; u < (p + 1) * per_step && u < parts; ++u)
            if (u * gp < G) GRF_CUDA_TRY(cudaStreamWaitEvent(s, ctx->up_done[u], 0));
        GRF_TRY(linear_attn(ctx, ctx->h_feat, by_mask, G, gc, N, m, d, dtype, (const char*)ctx->h_q.ptr + qo,
                            (const char*)ctx->h_k.ptr + qo, (const char*)ctx->h_v.ptr + vo, (char*)ctx->h_out.ptr + vo,
                            nullptr, ctx->h_ws.ptr, ctx->h_ws.bytes));
        GRF_CUDA_TRY(cudaEventRecord(ctx->part_done[p], s));
        GRF_CUDA_TRY(cudaStreamWaitEvent(ctx->down_stream, ctx->part_done[p], 0));
        GRF_CUDA_TRY(cudaMemcpyAsync((char*)out + vo, (const char*)ctx->h_out.ptr + vo, (size_t)gc * N * d * es,
                                     cudaMemcpyDeviceToHost, ctx->down_stream));
    }
    GRF_CUDA_TRY(cudaEventRecord(ctx->down_done, ctx->down_stream));
    GRF_CUDA_TRY(cudaStreamWaitEvent(s, ctx->down_done, 0));
    return grf_ctx_check(ctx);
}

extern "C" int grf_step_host(grf_ctx* ctx, int32_t N, const int32_t* rowptr, const int32_t* col, const float* w,
                             uint64_t seed, int32_t n_walks, float p_halt, int32_t max_len,
                             const float* f_phi, const float* f_psi,
                             int32_t G, int32_t m, int32_t d, int dtype,
                             const void* phiQ, const void* phiK, const void* V, void* out)
{
    const int rc = step_host(ctx, N, rowptr, col, w, seed, n_walks, p_halt, max_len, f_phi, f_psi, G, m, d, dtype, phiQ, phiK, V,
                             out);
    if (rc != GRF_OK && ctx) {                      // copies from and to the caller's buffers may be on their way
        cudaStreamSynchronize(ctx->stream);
        if (ctx->copy_stream) cudaStreamSynchronize(ctx->copy_stream);
        if (ctx->down_stream) cudaStreamSynchronize(ctx->down_stream);
    }
    return rc;
}

extern "C" const char* grf_strerror(int code)
{
    switch (code) {
        case GRF_OK: return "ok";
        case GRF_ERR_INVALID: return "invalid argument";
        case GRF_ERR_TOO_LARGE: return "size exceeds a documented limit";
        case GRF_ERR_WORKSPACE: return "workspace too small";
        case GRF_ERR_CUDA: return "CUDA runtime error";
        case GRF_ERR_NOMEM: return "out of memory";
        case GRF_ERR_BADGRAPH: return "inconsistent graph CSR";
        case GRF_ERR_TIMEOUT: return "a kernel gave up a bounded wait";
        default: return "unknown error";
    }
}
