// The kept slabs behind Scratch (see scratch.h).
#include "scratch.h"

#include <cuda.h>

#include <algorithm>
#include <mutex>
#include <vector>

namespace nvisr {

namespace {

struct Slab {
    uint64_t ctx;  // the context's unique id: slabs of a context that is gone are never used again
    uint8_t *dev;
    size_t bytes;
    int *err, *err_dev;
};

struct Kept {
    std::mutex mu;
    std::vector<Slab> slabs;  // oldest first
};

// Never destroyed: at process exit the device memory goes with the context.
Kept &kept() {
    static Kept *k = new Kept();
    return *k;
}

// Unique id of the current context (0: unknown, nothing is kept).
uint64_t context_id() {
    typedef CUresult (*GetCurrent)(CUcontext *);
    typedef CUresult (*GetId)(CUcontext, unsigned long long *);
    struct Fns {
        GetCurrent cur = nullptr;
        GetId id = nullptr;
        Fns() {
            void *p = nullptr;
            cudaDriverEntryPointQueryResult q;
            if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                q == cudaDriverEntryPointSuccess)
                cur = (GetCurrent)p;
            p = nullptr;
            if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                q == cudaDriverEntryPointSuccess)
                id = (GetId)p;
        }
    };
    static const Fns f;
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (!f.cur || !f.id || f.cur(&c) != CUDA_SUCCESS || !c || f.id(c, &id) != CUDA_SUCCESS) return 0;
    return (uint64_t)id + 1;
}

void free_slab(const Slab &s) {
    if (s.dev) cudaFree(s.dev);
    if (s.err) cudaFreeHost(s.err);
}

}  // namespace

void scratch_trim() {
    std::vector<Slab> out;
    Kept &k = kept();
    {
        std::lock_guard<std::mutex> lock(k.mu);
        if (k.slabs.empty()) return;
    }
    (void)cudaFree(nullptr);  // binds the device's context to a thread new to it
    const uint64_t ctx = context_id();
    {
        std::lock_guard<std::mutex> lock(k.mu);
        for (size_t i = 0; i < k.slabs.size();)
            if (k.slabs[i].ctx == ctx) {
                out.push_back(k.slabs[i]);
                k.slabs.erase(k.slabs.begin() + (long)i);
            } else {
                ++i;
            }
    }
    for (const Slab &s : out) free_slab(s);
}

cudaError_t device_malloc(void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        scratch_trim();
        e = cudaMalloc(p, bytes);
    }
    return e;
}

cudaError_t Scratch::open() {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st_, &cap);
    if (e != cudaSuccess) return e;
    if (cap != cudaStreamCaptureStatusNone) return cudaErrorStreamCaptureUnsupported;
    ctx_ = context_id();
    const size_t want = std::max<size_t>(need_, 256);
    {
        Kept &k = kept();
        std::lock_guard<std::mutex> lock(k.mu);
        size_t best = k.slabs.size();
        for (size_t i = 0; i < k.slabs.size(); ++i)
            if (ctx_ && k.slabs[i].ctx == ctx_ && k.slabs[i].bytes >= want &&
                (best == k.slabs.size() || k.slabs[i].bytes < k.slabs[best].bytes))
                best = i;
        if (best < k.slabs.size()) {
            const Slab s = k.slabs[best];
            k.slabs.erase(k.slabs.begin() + (long)best);
            dev_ = s.dev;
            bytes_ = s.bytes;
            err_ = s.err;
            err_dev_ = s.err_dev;
        }
    }
    if (!dev_) {
        void *p = nullptr, *h = nullptr, *hd = nullptr;
        e = device_malloc(&p, want);
        if (e == cudaSuccess) e = cudaHostAlloc(&h, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable);
        if (e == cudaSuccess) e = cudaHostGetDevicePointer(&hd, h, 0);
        if (e != cudaSuccess) {
            if (h) cudaFreeHost(h);
            if (p) cudaFree(p);
            (void)cudaGetLastError();
            return e;
        }
        if (!ctx_) ctx_ = context_id();  // the first call may have created the context
        dev_ = static_cast<uint8_t *>(p);
        bytes_ = want;
        err_ = static_cast<int *>(h);
        err_dev_ = static_cast<int *>(hd);
    }
    *const_cast<volatile int *>(err_) = 0;
    return cudaSuccess;
}

cudaError_t Scratch::finish() {
    const cudaError_t e = cudaStreamSynchronize(st_);
    idle_ = e == cudaSuccess;
    return e;
}

Scratch::~Scratch() {
    if (!dev_) return;
    if (!idle_ && cudaStreamSynchronize(st_) != cudaSuccess) return;  // a broken context: nothing to hand back
    const Slab s = {ctx_, dev_, bytes_, err_, err_dev_};
    std::vector<Slab> out;
    if (!ctx_ || bytes_ > SCRATCH_KEEP) {
        out.push_back(s);
    } else {
        Kept &k = kept();
        std::lock_guard<std::mutex> lock(k.mu);
        k.slabs.push_back(s);
        size_t total = 0;
        for (const Slab &o : k.slabs)
            if (o.ctx == ctx_) total += o.bytes;
        for (size_t i = 0; i < k.slabs.size() && total > SCRATCH_KEEP;)
            if (k.slabs[i].ctx == ctx_) {
                total -= k.slabs[i].bytes;
                out.push_back(k.slabs[i]);
                k.slabs.erase(k.slabs.begin() + (long)i);
            } else {
                ++i;
            }
    }
    for (const Slab &o : out) free_slab(o);
}

}  // namespace nvisr
