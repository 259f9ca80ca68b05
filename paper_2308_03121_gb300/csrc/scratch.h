// Working memory of the per-call entry points (nvisr_conv2d, nvisr_resblock2d, nvisr_dcn2d): one
// device slab per call, kept for later calls instead of cudaMalloc / cudaFree of every buffer
// (which took 1.0-1.3 ms of a call and synchronised the whole device).
//
// A slab belongs to one call at a time, so calls on several threads and streams never share
// one: a call takes a kept slab that is large enough, or allocates its own, and hands it back
// after its stream has been synchronised.  At most SCRATCH_KEEP bytes stay kept per device
// context; larger slabs, and the oldest kept ones past that, are freed.  scratch_trim() gives the
// kept slabs back, which the library does itself when a device allocation fails.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace nvisr {

constexpr size_t SCRATCH_KEEP = (size_t)1 << 30;

// Frees the kept slabs of the current device's context.
void scratch_trim();

class Scratch {
public:
    explicit Scratch(cudaStream_t st) : st_(st) {}
    Scratch(const Scratch &) = delete;
    Scratch &operator=(const Scratch &) = delete;
    // Hands the slab back; waits for the stream first unless finish() did.
    ~Scratch();
    // Before open(): room for `bytes` (256-byte aligned); returns its offset in the slab.
    size_t plan(size_t bytes) {
        const size_t at = need_;
        need_ += (bytes + 255) / 256 * 256;
        return at;
    }
    // Takes the slab.  A capturing stream is refused: these calls read results back.
    cudaError_t open();
    template <typename T>
    T *at(size_t offset) const { return reinterpret_cast<T *>(dev_ + offset); }
    // The call's error word: pinned host memory that kernels may write (zero after open()), so
    // reading it back is no copy.
    int *err() const { return err_dev_; }
    int host_err() const { return *const_cast<volatile int *>(err_); }
    // Synchronises the stream.
    cudaError_t finish();

private:
    cudaStream_t st_;
    size_t need_ = 0, bytes_ = 0;
    uint8_t *dev_ = nullptr;
    int *err_ = nullptr, *err_dev_ = nullptr;
    uint64_t ctx_ = 0;
    bool idle_ = false;  // the stream has no work of this call in flight
};

}  // namespace nvisr
