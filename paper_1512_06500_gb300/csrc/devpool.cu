// Device memory, streams, events and pinned host pages kept from one handle to the next.
//
// A handle takes two to eight device blocks (up to 14 GB at d = 65536, n = 2000), a second stream for the independent
// halves of its build and a dozen small readbacks, and the driver's calls for them cost as much as the kernels of a small
// problem: cudaMalloc and cudaFree of one d = 65536 pipeline took 10 ms of its 74 ms, those of a batch of 32 problems on 16
// host threads (with their streams) 3 s of summed thread time in 0.4 s. So freed blocks are kept and handed out again, best
// fit first.
//
// What is kept belongs to one context (its identity, not the device number: a device reset takes the memory away) and is
// bounded: at most a sixteenth of the device's memory and kMaxBlocks blocks; a block that kMaxAge later frees have passed over is
// released, so what stays is the working set of the most recent handles; when an allocation fails everything kept is
// released and the allocation tried again; eda_release_cached gives it all back.
//
// A block enters the cache only when the GPU has finished with it: dev_free's callers have synchronised (see below), so any
// stream of any thread may take it next. The lists are guarded by one mutex, held for list operations only.
#include "eda_internal.cuh"

#include <algorithm>
#include <cstring>
#include <list>
#include <unordered_map>

namespace eda {

namespace {

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

constexpr size_t kCacheShare = 16;      // of the device's memory
constexpr size_t kMaxBlocks = 512;
constexpr uint64_t kMaxAge = 1024;      // frees
constexpr size_t kMaxKits = 128;

struct Block {
    void* p;
    size_t bytes;
    unsigned long long ctx;
    uint64_t stamp;
};
std::mutex g_mu;
std::list<Block> g_cache;                        // most recently freed first
std::unordered_map<void*, Block> g_live;         // blocks handed out
size_t g_cached_bytes = 0;
uint64_t g_frees = 0;
std::vector<HostKit*> g_kits;

// Bytes that may be kept on the current device (queried once per process: every handle of a process uses one GPU type).
size_t cache_cap() {
    static size_t cap = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) cap = tot / kCacheShare;
        cudaGetLastError();
    });
    return cap;
}

// Blocks of the given context out of the cache, by a predicate; they are freed outside the lock.
template <class Pred>
void evict(unsigned long long ctx, Pred drop) {
    std::vector<void*> gone;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        for (auto it = g_cache.begin(); it != g_cache.end();) {
            if (it->ctx == ctx && drop(*it)) {
                gone.push_back(it->p);
                g_cached_bytes -= it->bytes;
                it = g_cache.erase(it);
            } else {
                ++it;
            }
        }
    }
    for (void* p : gone) cudaFree(p);
}

}  // namespace

// Identity of the calling thread's current context (0 when there is none or the driver does not
// offer context identities, in which case nothing is cached).
unsigned long long current_ctx_id() {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<CtxGetCurrentFn>(p);
        p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(p);
        cudaGetLastError();
    });
    if (!get_current || !get_id) return 0;
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (get_current(&ctx) != CUDA_SUCCESS || ctx == nullptr) return 0;
    if (get_id(ctx, &id) != CUDA_SUCCESS) return 0;
    return id;
}

int dev_alloc(void** out, size_t bytes) {
    *out = nullptr;
    bytes = (std::max<size_t>(bytes, 1) + 511) / 512 * 512;
    unsigned long long ctx = current_ctx_id();
    if (ctx) {
        std::lock_guard<std::mutex> lk(g_mu);
        // the smallest kept block that holds the request, at most an eighth (and 1 MiB) larger than it
        auto best = g_cache.end();
        for (auto it = g_cache.begin(); it != g_cache.end(); ++it)
            if (it->ctx == ctx && it->bytes >= bytes && it->bytes <= bytes + bytes / 8 + (size_t(1) << 20) &&
                (best == g_cache.end() || it->bytes < best->bytes))
                best = it;
        if (best != g_cache.end()) {
            *out = best->p;
            g_live[best->p] = *best;
            g_cached_bytes -= best->bytes;
            g_cache.erase(best);
            return EDA_OK;
        }
    }
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        ctx = current_ctx_id();
        evict(ctx, [](const Block&) { return true; });
        e = cudaMalloc(&p, bytes);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        note_cuda_error(e, __FILE__, __LINE__);
        return e == cudaErrorMemoryAllocation ? EDA_ERR_OOM : EDA_ERR_CUDA;
    }
    ctx = current_ctx_id();   // the first call of a process makes the primary context current
    if (ctx) {
        std::lock_guard<std::mutex> lk(g_mu);
        g_live[p] = Block{p, bytes, ctx, 0};
    }
    *out = p;
    return EDA_OK;
}

void dev_free(void* p) {
    if (!p) return;
    const unsigned long long ctx = current_ctx_id();
    const size_t cap = cache_cap();
    bool keep = false, old = false;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        auto it = g_live.find(p);
        if (it != g_live.end()) {
            Block b = it->second;
            g_live.erase(it);
            b.stamp = ++g_frees;
            keep = ctx != 0 && b.ctx == ctx && b.bytes <= cap;
            if (keep) {
                g_cache.push_front(b);
                g_cached_bytes += b.bytes;
                old = g_cached_bytes > cap || g_cache.size() > kMaxBlocks || b.stamp - g_cache.back().stamp > kMaxAge;
            }
        }
    }
    if (!keep) {
        cudaFree(p);
        return;
    }
    if (old) {
        // from the oldest on until the bounds hold again
        size_t bytes = 0, count = 0;
        uint64_t from = 0;
        {
            std::lock_guard<std::mutex> lk(g_mu);
            for (const Block& b : g_cache) {
                bytes += b.bytes;
                ++count;
                if (bytes > cap || count > kMaxBlocks || g_frees - b.stamp > kMaxAge) {
                    from = b.stamp;
                    break;
                }
            }
        }
        if (from) evict(ctx, [from](const Block& b) { return b.stamp <= from; });
    }
}

int dev_free_idle(void* p) {
    if (!p) return EDA_OK;
    const cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(p);
        note_cuda_error(e, __FILE__, __LINE__);
        return EDA_ERR_CUDA;
    }
    dev_free(p);
    return EDA_OK;
}

int host_kit_take(HostKit** out) {
    *out = nullptr;
    const unsigned long long ctx = current_ctx_id();
    if (ctx) {
        std::lock_guard<std::mutex> lk(g_mu);
        for (size_t i = g_kits.size(); i-- > 0;)
            if (g_kits[i]->ctx == ctx) {
                *out = g_kits[i];
                g_kits.erase(g_kits.begin() + (ptrdiff_t)i);
                return EDA_OK;
            }
    }
    HostKit* k = new (std::nothrow) HostKit();
    if (!k) return EDA_ERR_OOM;
    cudaError_t e = cudaStreamCreateWithFlags(&k->s, cudaStreamNonBlocking);
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&k->order[i], cudaEventDisableTiming);
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaEventCreate(&k->timer[i]);
    if (e == cudaSuccess) e = cudaHostAlloc(&k->page, kHostPage, cudaHostAllocDefault);
    if (e != cudaSuccess) {
        note_cuda_error(e, __FILE__, __LINE__);
        cudaGetLastError();
        host_kit_destroy(k);
        return e == cudaErrorMemoryAllocation ? EDA_ERR_OOM : EDA_ERR_CUDA;
    }
    k->ctx = current_ctx_id();
    *out = k;
    return EDA_OK;
}

void host_kit_destroy(HostKit* k) {
    if (!k) return;
    if (k->s) cudaStreamDestroy(k->s);   // released once its queued work has finished
    for (cudaEvent_t e : k->order)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : k->timer)
        if (e) cudaEventDestroy(e);
    if (k->page) cudaFreeHost(k->page);
    delete k;
}

void host_kit_give(HostKit* k) {
    if (!k) return;
    if (k->ctx != 0 && k->ctx == current_ctx_id()) {
        std::lock_guard<std::mutex> lk(g_mu);
        if (g_kits.size() < kMaxKits) {
            g_kits.push_back(k);
            return;
        }
    }
    host_kit_destroy(k);
}

int Note::open(cudaStream_t stream) {
    s = stream;
    if (hold.open() != EDA_OK) {
        hold.kit = nullptr;
        cudaGetLastError();
        return EDA_OK;
    }
    std::memset(hold.kit->page, 0, 3 * sizeof(int));
    return EDA_OK;
}

Note::~Note() {
    if (pending) cudaStreamSynchronize(s);
}

NoteRef Note::next() {
    if (!hold.kit) return {};
    pending = true;
    return {static_cast<int*>(hold.kit->page), ++tag};
}

int Note::wait(int out[2], const int* dev) {
    if (!hold.kit) return read_back(out, dev, 2 * sizeof(int), s);
    const int* w = static_cast<const int*>(hold.kit->page);
    for (bool done = false;;) {
        for (int i = 0; i < 4096; ++i)
            if (__atomic_load_n(w + 2, __ATOMIC_ACQUIRE) == tag) {
                out[0] = w[0];
                out[1] = w[1];
                pending = false;
                return EDA_OK;
            }
        if (done) return EDA_ERR_CUDA;   // the stream ran dry without the note
        const cudaError_t q = cudaStreamQuery(s);
        if (q == cudaSuccess) done = true;
        else if (q != cudaErrorNotReady) EDA_CUDA_TRY(q);
    }
}

int read_back(void* host, const void* dev, size_t bytes, cudaStream_t s) {
    HostHold hold;
    if (bytes <= kHostPage && hold.open() == EDA_OK) {
        EDA_CUDA_TRY(cudaMemcpyAsync(hold.kit->page, dev, bytes, cudaMemcpyDeviceToHost, s));
        EDA_CUDA_TRY(cudaStreamSynchronize(s));
        std::memcpy(host, hold.kit->page, bytes);
        return EDA_OK;
    }
    EDA_CUDA_TRY(cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, s));
    EDA_CUDA_TRY(cudaStreamSynchronize(s));
    return EDA_OK;
}

}  // namespace eda

extern "C" int eda_release_cached(void) {
    using namespace eda;
    const unsigned long long ctx = current_ctx_id();
    if (!ctx) return EDA_OK;
    evict(ctx, [](const Block&) { return true; });
    std::vector<HostKit*> kits;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        for (size_t i = g_kits.size(); i-- > 0;)
            if (g_kits[i]->ctx == ctx) {
                kits.push_back(g_kits[i]);
                g_kits.erase(g_kits.begin() + (ptrdiff_t)i);
            }
    }
    for (HostKit* k : kits) host_kit_destroy(k);
    return EDA_OK;
}
