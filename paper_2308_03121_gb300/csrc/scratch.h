// Working memory of the per-call entry points (nvisr_conv2d, nvisr_resblock2d, nvisr_dcn2d): one
// device slab per call, kept for later calls instead of cudaMalloc / cudaFree of every buffer
// (which took 1.0-1.3 ms of a call and synchronised the whole device).
//
// A slab belongs to one call at a time, so calls on several threads and streams never share
// one: a call takes the smallest kept slab that is large enough, or allocates its own, and hands it
// back after its stream has been synchronised.  At most SCRATCH_KEEP bytes stay kept per device
// context; larger slabs, and the oldest kept ones past that, are freed.  scratch_trim() gives the
// kept slabs back: a program's call (nvisr_release_scratch), the destruction of an engine and a
// device allocation of this library that would fail otherwise (device_malloc) do that.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace nvisr {

// What stays kept: enough for one call at the largest sizes that a layer has in the networks here (a
// 3840 x 2160 residual block takes 1012 MB, a 1920 x 1080 deformable layer 759 MB) and less than 0.4 %
// of the device.  An allocation and its release take about 1.0 ms: that block 1.23 ms a call with its
// slab kept and 2.24 without, that layer 1.51 and 2.41; a call past the limit pays it each time.
constexpr size_t SCRATCH_KEEP = (size_t)1 << 30;

// Frees the kept slabs of the current device's context.
void scratch_trim();

// cudaMalloc that gives the kept slabs back before it fails for want of memory.
cudaError_t device_malloc(void **p, size_t bytes);

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
