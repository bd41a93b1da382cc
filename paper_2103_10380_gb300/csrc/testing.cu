// testing.cu -- test hooks (fnr_testing.h): failure injection and the choice
// of the cache-build kernel's form; and the device allocation helpers every
// library allocation goes through.
#include <atomic>

#include "fnr_internal.h"
#include "fnr_testing.h"

namespace fnr {

fnr_status fail(fnr_status st, const char *fmt, ...);
void clear_error();

namespace {
std::atomic<int> g_alloc_skip{0}, g_alloc_fail{0};
std::atomic<long long> g_mlp_wait_limit{0}, g_mlp_withhold{-1};
std::atomic<int> g_mlp_cta_pair{0};
}  // namespace

bool mlp_cta_pair() { return g_mlp_cta_pair.load() != 0; }

// Whether the next allocation is one of those made to fail.
static bool injected_failure() {
    if (g_alloc_fail.load() <= 0) return false;
    if (g_alloc_skip.load() > 0) {
        g_alloc_skip.fetch_sub(1);
        return false;
    }
    g_alloc_fail.fetch_sub(1);
    return true;
}

cudaError_t dev_malloc(void **p, size_t bytes) {
    *p = nullptr;
    return injected_failure() ? cudaErrorMemoryAllocation : cudaMalloc(p, bytes);
}

// A stream capture, in whichever thread, does not mind these calls of this thread: pools have no stream.
struct OutsideCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

cudaMemPool_t make_temp_pool(int device) {
    OutsideCapture relaxed;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    uint64_t keep = kPoolKeepBytes;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) cudaGetLastError();
    return pool;
}

void destroy_temp_pool(cudaMemPool_t pool) {
    OutsideCapture relaxed;
    if (pool) cudaMemPoolDestroy(pool);
}

cudaError_t TempBuf::alloc(const fnr_context *ctx, size_t bytes, cudaStream_t s) {
    release();
    if (injected_failure()) return cudaErrorMemoryAllocation;
    pooled = ctx->pool && bytes <= kPooledBytes;
    stream = s;
    const cudaError_t e = pooled ? cudaMallocFromPoolAsync(&p, bytes, ctx->pool, s) : cudaMalloc(&p, bytes);
    if (e != cudaSuccess) p = nullptr;
    return e;
}

void TempBuf::release() {
    if (!p) return;
    if (pooled) cudaFreeAsync(p, stream);
    else cudaFree(p);
    p = nullptr;
}

void take_mlp_fault(long long *wait_limit, long long *withhold) {
    const long long w = g_mlp_wait_limit.exchange(0);
    const long long h = g_mlp_withhold.exchange(-1);
    if (w > 0) {
        *wait_limit = w;
        *withhold = h;
    }
}

}  // namespace fnr

using namespace fnr;

extern "C" fnr_status fnr_testing_fail_allocations(int32_t skip, int32_t count) {
    clear_error();
    if (skip < 0 || count < 0) return fail(FNR_ERR_INVALID_ARG, "negative skip or count");
    g_alloc_fail.store(0);
    g_alloc_skip.store(skip);
    g_alloc_fail.store(count);
    return FNR_OK;
}

extern "C" fnr_status fnr_testing_mlp_fault(int64_t wait_limit, int64_t withhold_chunk) {
    clear_error();
    if (wait_limit < 1) return fail(FNR_ERR_INVALID_ARG, "wait_limit must be >= 1");
    g_mlp_withhold.store(withhold_chunk);
    g_mlp_wait_limit.store(wait_limit);
    return FNR_OK;
}

extern "C" fnr_status fnr_testing_mlp_cta_pair(int32_t on) {
    clear_error();
    g_mlp_cta_pair.store(on != 0 ? 1 : 0);
    return FNR_OK;
}
