// Device memory of plans, and the CUDA context's ID.
//
// cudaMalloc and cudaFree cost 60 us each, and a plan makes two of each: a third of
// the time of mapping and packing a 32K cache. So the memory of a released plan is kept
// for the next one while other plans of its context live: mapping and packing a 32-layer
// model at 32K takes 559 us if the new plan is made before the old one is released, 832
// if after (at 16K in place 299 and 578).
//
// At most kKeepBytes a context, so that memory that no plan uses stays small beside a
// cache: enough for a 32-layer plan at 32K (39 MB); a 128K one (73 MB) is freed and
// allocated anew. All of a context's kept memory is given back when its last plan is
// released while the context is current (from another one, the blocks stay until the
// context's next plan: it may be gone, and its addresses may be another's by then).
// Only a block that the device is known to have finished with is kept (a wait can fail,
// under stream capture for one), so a kept one serves any stream and thread at once; and
// only in its own context.
#include "dkv_pool.cuh"

#include <cuda.h>

#include <mutex>
#include <new>
#include <vector>

namespace dkv {
namespace {

constexpr size_t kKeepBytes = size_t(64) << 20;

struct Context {
    unsigned long long id;
    int live;                       // blocks in use
    size_t kept_bytes;
    std::vector<PlanMemory> kept;   // idle blocks
};

std::mutex g_mu;
std::vector<Context> g_contexts;

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

template <class F>
F driver_fn(const char* name)
{
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
        return nullptr;
    return reinterpret_cast<F>(p);
}

}  // namespace

// The runtime's primary context of the current device is made current first if none is.
cudaError_t current_context_id(unsigned long long* id)
{
    static const CtxGetCurrentFn get_current = driver_fn<CtxGetCurrentFn>("cuCtxGetCurrent");
    static const CtxGetIdFn get_id = driver_fn<CtxGetIdFn>("cuCtxGetId");
    if (!get_current || !get_id) return cudaErrorNotSupported;
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    if (!ctx) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaSetDevice(dev);  // initialises the device's primary context
        if (e != cudaSuccess) return e;
        if (get_current(&ctx) != CUDA_SUCCESS || !ctx) return cudaErrorDeviceUninitialized;
    }
    return get_id(ctx, id) == CUDA_SUCCESS ? cudaSuccess : cudaErrorDeviceUninitialized;
}

namespace {

// The entry of context `id`, null if the host has no memory for one; g_mu is held.
Context* context_of(unsigned long long id)
{
    for (Context& c : g_contexts)
        if (c.id == id) return &c;
    try {
        g_contexts.push_back(Context{id, 0, 0, {}});
    } catch (const std::bad_alloc&) {
        return nullptr;
    }
    return &g_contexts.back();
}

void give_back(Context& c)
{
    for (const PlanMemory& m : c.kept) cudaFree(m.ptr);
    c.kept.clear();
    c.kept_bytes = 0;
}

}  // namespace

cudaError_t plan_alloc(PlanMemory* m, size_t bytes)
{
    *m = PlanMemory{};
    unsigned long long id = 0;
    cudaError_t e = current_context_id(&id);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_mu);
    Context* entry = context_of(id);
    if (!entry) return cudaErrorMemoryAllocation;
    Context& c = *entry;
    // The smallest kept block that fits, unless it is more than twice as large.
    size_t best = c.kept.size();
    for (size_t i = 0; i < c.kept.size(); ++i)
        if (c.kept[i].bytes >= bytes && c.kept[i].bytes / 2 <= bytes &&
            (best == c.kept.size() || c.kept[i].bytes < c.kept[best].bytes))
            best = i;
    if (best < c.kept.size()) {
        *m = c.kept[best];
        c.kept.erase(c.kept.begin() + (std::ptrdiff_t)best);
        c.kept_bytes -= m->bytes;
        ++c.live;
        return cudaSuccess;
    }
    void* p = nullptr;
    e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation && !c.kept.empty()) {
        cudaGetLastError();
        give_back(c);
        e = cudaMalloc(&p, bytes);
    }
    if (e != cudaSuccess) return e;
    m->ptr = p;
    m->bytes = bytes;
    m->context = id;
    ++c.live;
    return cudaSuccess;
}

void plan_free(const PlanMemory& m, bool idle)
{
    if (!m.ptr) return;
    unsigned long long id = 0;
    const bool own = current_context_id(&id) == cudaSuccess && id == m.context;
    std::lock_guard<std::mutex> lock(g_mu);
    Context& c = *context_of(m.context);  // (there since plan_alloc)
    --c.live;
    bool keep = own && idle && c.live > 0 && c.kept_bytes + m.bytes <= kKeepBytes;
    if (keep) try {
            c.kept.push_back(m);
            c.kept_bytes += m.bytes;
        } catch (const std::bad_alloc&) {
            keep = false;
        }
    if (!keep) cudaFree(m.ptr);
    if (own && c.live == 0) give_back(c);
}

}  // namespace dkv
