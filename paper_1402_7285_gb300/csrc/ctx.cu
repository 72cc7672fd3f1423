// Context, status strings and host/device staging.
#include <algorithm>
#include <cstdarg>

#include "common.cuh"

namespace tbgf {

int set_error(tb_ctx *ctx, int code, const char *fmt, ...) {
    if (ctx) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        ctx->last_error = buf;
    }
    return code;
}

int ws_get(tb_ctx *ctx, int slot, size_t bytes, void **out) {
    if (slot < 0 || slot >= WS_COUNT) return set_error(ctx, TB_ERR_ARG, "bad workspace slot %d", slot);
    if ((int)ctx->ws_ptr.size() < WS_COUNT) {
        ctx->ws_ptr.resize(WS_COUNT, nullptr);
        ctx->ws_size.resize(WS_COUNT, 0);
    }
    bytes = align_up(bytes < 256 ? 256 : bytes, 256);
    if (ctx->ws_size[slot] < bytes) {
        ws_free(ctx, slot);
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return set_error(ctx, TB_ERR_ALLOC, "cudaMalloc(%zu) for workspace slot %d: %s", bytes, slot,
                             cudaGetErrorString(e));
        }
        ctx->ws_ptr[slot] = p;
        ctx->ws_size[slot] = bytes;
    }
    *out = ctx->ws_ptr[slot];
    return TB_OK;
}

void ws_free(tb_ctx *ctx, int slot) {
    if (slot >= (int)ctx->ws_ptr.size() || !ctx->ws_ptr[slot]) return;
    cudaDeviceSynchronize(); // earlier work may still read the buffer
    cudaFree(ctx->ws_ptr[slot]);
    ctx->ws_ptr[slot] = nullptr;
    ctx->ws_size[slot] = 0;
}

static bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) { // the legacy stream during a capture elsewhere
        cudaGetLastError();
        return true;
    }
    return st != cudaStreamCaptureStatusNone;
}

StageOrder::StageOrder(tb_ctx *ctx, cudaStream_t s) : ctx_(ctx), stream_(s) {
    if (capturing(s)) return;
    cudaError_t e = cudaSuccess;
    if (!ctx->stage_ev) e = cudaEventCreateWithFlags(&ctx->stage_ev, cudaEventDisableTiming);
    if (e == cudaSuccess && ctx->stage_used) e = cudaStreamWaitEvent(s, ctx->stage_ev, 0);
    if (e != cudaSuccess)
        rc = set_error(ctx, TB_ERR_CUDA, "order of the workspace's calls: %s", cudaGetErrorString(e));
    else
        on_ = true;
}

StageOrder::~StageOrder() {
    if (on_ && cudaEventRecord(ctx_->stage_ev, stream_) == cudaSuccess) ctx_->stage_used = true;
}

bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

void Stager::add(const void *p, size_t bytes, bool is_input, bool is_output, void **dev_out) {
    if (!p || bytes == 0 || is_device_ptr(p)) {
        *dev_out = const_cast<void *>(p);
        return;
    }
    any_host_ = true;
    Item it{p, bytes, total_, is_input, is_output, dev_out};
    total_ = align_up(total_ + bytes, 256);
    items_.push_back(it);
}

int Stager::commit() {
    if (items_.empty()) return TB_OK;
    void *base = nullptr;
    int rc = ws_get(ctx_, slot_, total_, &base);
    if (rc != TB_OK) return rc;
    base_ = (char *)base;
    for (auto &it : items_) {
        *it.dev_out = base_ + it.offset;
        if (it.in)
            TB_CUDA_TRY(ctx_, cudaMemcpyAsync(base_ + it.offset, it.host, it.bytes, cudaMemcpyHostToDevice,
                                              stream_));
    }
    return TB_OK;
}

int Stager::finish() {
    bool any_out = false;
    for (auto &it : items_) {
        if (!it.out) continue;
        any_out = true;
        TB_CUDA_TRY(ctx_, cudaMemcpyAsync(const_cast<void *>(it.host), base_ + it.offset, it.bytes,
                                          cudaMemcpyDeviceToHost, stream_));
    }
    if (any_host_) TB_CUDA_TRY(ctx_, cudaStreamSynchronize(stream_));
    (void)any_out;
    return TB_OK;
}

__global__ void k_validate_bsr(const int64_t *rp, const int32_t *ci, int64_t n_brows, int64_t nnzb, int *bad) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < n_brows; a += stride)
        if (const int f = bsr_row_fault(rp, ci, n_brows, nnzb, a)) atomicOr(bad, f);
}

static __global__ void k_check_bsr(const int64_t *rp, const int32_t *ci, int64_t n_brows, int64_t nnzb, int *words,
                                   int *host) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < n_brows; a += stride)
        if (const int f = bsr_row_fault(rp, ci, n_brows, nnzb, a)) atomicOr(words, f);
    publish_check(words, host);
}

int check_words(tb_ctx *ctx, int **words, int **host) {
    if (!ctx->chk_dev) {
        int *d = nullptr;
        TB_CUDA_TRY(ctx, cudaMalloc((void **)&d, 4 * sizeof(int)));
        cudaError_t e = cudaMemset(d, 0, 4 * sizeof(int));
        if (e == cudaSuccess) e = cudaHostAlloc((void **)&ctx->chk_host, 512, cudaHostAllocPortable);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->chk_ev, cudaEventDisableTiming);
        // the memset ran on the legacy stream, which a caller's non-blocking stream does not wait for
        if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
        if (e != cudaSuccess) {
            cudaFree(d);
            if (ctx->chk_host) cudaFreeHost((void *)ctx->chk_host);
            if (ctx->chk_ev) cudaEventDestroy(ctx->chk_ev);
            ctx->chk_host = nullptr;
            ctx->chk_ev = nullptr;
            return set_error(ctx, TB_ERR_CUDA, "structure check words: %s", cudaGetErrorString(e));
        }
        ctx->chk_dev = d;
    }
    *words = ctx->chk_dev;
    *host = (int *)ctx->chk_host;
    return TB_OK;
}

int check_wait(tb_ctx *ctx, cudaStream_t s, int *result) {
    TB_CUDA_TRY(ctx, cudaGetLastError());
    TB_CUDA_TRY(ctx, cudaEventRecord(ctx->chk_ev, s));
    TB_CUDA_TRY(ctx, cudaEventSynchronize(ctx->chk_ev));
    *result = *ctx->chk_host;
    return TB_OK;
}

int validate_bsr(tb_ctx *ctx, const int64_t *row_ptr, const int32_t *col_idx, const void *val, int64_t n_brows,
                 int64_t nnzb, cudaStream_t s, const char *name) {
    if (((uintptr_t)val & 15u) != 0)
        return set_error(ctx, TB_ERR_ARG, "%s values must be 16-byte aligned", name);
    if (n_brows <= 0 || nnzb < 0) return set_error(ctx, TB_ERR_STRUCTURE, "%s: bad sizes", name);
    int *words = nullptr, *host = nullptr, h = 0;
    int rc = check_words(ctx, &words, &host);
    if (rc) return rc;
    const int g = (int)std::min<int64_t>((n_brows + 255) / 256, 152 * 8);
    k_check_bsr<<<g < 1 ? 1 : g, 256, 0, s>>>(row_ptr, col_idx, n_brows, nnzb, words, host);
    rc = check_wait(ctx, s, &h);
    if (rc) return rc;
    if (h) return set_error(ctx, TB_ERR_STRUCTURE, "%s: malformed BSR structure (code %d)", name, h);
    return TB_OK;
}

} // namespace tbgf

extern "C" {

int tb_ctx_create(tb_ctx **out) {
    if (!out) return TB_ERR_ARG;
    *out = nullptr;
    tb_ctx *c = new (std::nothrow) tb_ctx();
    if (!c) return TB_ERR_ALLOC;
    if (cudaGetDevice(&c->device) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return TB_ERR_CUDA;
    }
    c->ws_ptr.assign(tbgf::WS_COUNT, nullptr);
    c->ws_size.assign(tbgf::WS_COUNT, 0);
    *out = c;
    return TB_OK;
}

int tb_ctx_destroy(tb_ctx *ctx) {
    if (!ctx) return TB_OK;
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != ctx->device) cudaSetDevice(ctx->device);
    cudaDeviceSynchronize();
    for (void *p : ctx->ws_ptr)
        if (p) cudaFree(p);
    if (ctx->chk_dev) {
        cudaFree(ctx->chk_dev);
        cudaFreeHost((void *)ctx->chk_host);
        cudaEventDestroy(ctx->chk_ev);
    }
    if (ctx->stage_ev) cudaEventDestroy(ctx->stage_ev);
    if (dev >= 0 && dev != ctx->device) cudaSetDevice(dev);
    delete ctx;
    return TB_OK;
}

const char *tb_status_string(int status) {
    switch (status) {
    case TB_OK: return "ok";
    case TB_ERR_ARG: return "invalid argument";
    case TB_ERR_CUDA: return "CUDA error";
    case TB_ERR_ALLOC: return "allocation failed";
    case TB_ERR_UNSUPPORTED: return "unsupported request";
    case TB_ERR_SIZE: return "size exceeds a limit";
    case TB_ERR_STRUCTURE: return "malformed matrix structure";
    default: break;
    }
    if (status > 0) return "some columns did not converge (see per-column status)";
    return "unknown status";
}

const char *tb_last_error(const tb_ctx *ctx) { return ctx ? ctx->last_error.c_str() : ""; }

int tb_version(void) { return 10100; }

void tb_solve_opts_default(tb_solve_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->tol = 1e-10;
    o->max_iter = 100000;
    o->precision = TB_PREC_FP64;
    o->panel_w = 0;
    o->seed_shift = -1;
    o->inner_tol = 0.0;
    o->inner_max = 0;
    o->stream = nullptr;
}

} // extern "C"
