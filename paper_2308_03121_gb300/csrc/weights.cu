// Device-side layout of one layer's weights, for the entry points whose caller hands over plain
// OIHW float32 weights on the device (nvisr_conv2d and its kin).  One launch writes the whole
// image of the kernel that will run (padding included), the zero-padded bias and, for FP8, the
// scaled E4M3 values: the same bytes the host-side layouts (prepare_weights_*) give.  A layer
// has at most a few hundred thousand weights that sit in L2, so the launch costs its latency
// (about 3 us); copying them to the host, laying them out there and copying them back took
// two synchronisations and 100-200 us.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace nvisr {

namespace {

template <typename T>
__device__ __forceinline__ T to_elem(float v);
template <>
__device__ __forceinline__ float to_elem<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_elem<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ __half to_elem<__half>(float v) { return __float2half_rn(v); }
template <>
__device__ __forceinline__ __nv_fp8_e4m3 to_elem<__nv_fp8_e4m3>(float v) { return __nv_fp8_e4m3(v); }

// One thread per destination element; blockIdx.y selects one of a launch's layers.  The next kernel
// of a layer call changes the input's layout and needs nothing of this one: it may start at
// once, and itself ends only when this one has (with a residual block's two layers in one launch
// 357 -> 351 us at 1080p, 444 -> 441 for a 540p deformable layer, 127 -> 124 for a 853 x 479 layer).
// The layer's own kernel loads this one's results only after its wait (w_fresh, launch_dependent).
template <typename T>
__global__ void __launch_bounds__(256) weights_kernel(WeightArgs a0, WeightArgs a1, int64_t total) {
    griddep_launch_dependents();
    const WeightArgs &a = blockIdx.y ? a1 : a0;
    constexpr int UPC = 16 / (int)sizeof(T);  // elements of a 16-byte unit
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = t0; i < a.nbias; i += step) a.dst_bias[i] = a.bias && i < a.cout ? a.bias[i] : 0.f;
    const int kk = a.k * a.k;
    T *dst = static_cast<T *>(a.dst);
    for (int64_t i = t0; i < total; i += step) {
        int o, c, t;
        if (a.layout == WL_SIMT) {  // [cin_pad][k * k][cout_pad]
            o = (int)(i % a.cout_pad);
            const int64_t ct = i / a.cout_pad;
            t = (int)(ct % kk);
            c = (int)(ct / kk);
        } else if (a.layout == WL_ROWS) {  // [kx][2 - ky][64 out][64 in, 128-byte swizzled]
            const int n = (int)(i / 64 % 64), kyr = (int)(i / 4096 % 3), kx = (int)(i / 12288);
            o = n;
            c = (((int)(i % 64) / 8) ^ (n & 7)) * 8 + (int)(i % 8);
            t = (2 - kyr) * 3 + kx;
        } else {  // [slice of ns][tap][K chunk][n][chunk], swizzled when a chunk is 128 bytes
            const int cpc = a.layout == WL_TC128 ? 64 : UPC;
            const int chunks = a.cin_pad / cpc;
            int e = (int)(i % cpc);
            int64_t r = i / cpc;
            const int n = (int)(r % a.ns);
            r /= a.ns;
            const int kc = (int)(r % chunks);
            r /= chunks;
            t = (int)(r % kk);
            o = (int)(r / kk) * a.ns + n;
            if (a.layout == WL_TC128) e = ((e / UPC) ^ (n & 7)) * UPC + e % UPC;
            c = kc * cpc + e;
        }
        dst[i] = to_elem<T>(o < a.cout && c < a.cin ? a.w[((int64_t)o * a.cin + c) * kk + t] * a.scale : 0.f);
    }
}

// max |v| of n values into *out (its float bits; *out starts at zero).
__global__ void __launch_bounds__(256) absmax_kernel(const float *__restrict__ v, int64_t n, unsigned *out) {
    float m = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(__ldg(v + i)));
    const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) atomicMax(out, u);
}

int grid_for(int64_t n) {
    return (int)std::min<int64_t>(std::max<int64_t>((n + 255) / 256, 1), (int64_t)device_sm_count() * 8);
}

}  // namespace

cudaError_t launch_weights(const WeightArgs &a, cudaStream_t st, const WeightArgs *second) {
    const int64_t total = a.layout == WL_ROWS ? (int64_t)9 * 64 * 64 : (int64_t)a.k * a.k * a.cin_pad * a.cout_pad;
    const dim3 grid((unsigned)grid_for(std::max<int64_t>(total, a.nbias)), second ? 2 : 1);
    const WeightArgs &b = second ? *second : a;
    switch (a.dt) {
        case DT_F32: weights_kernel<float><<<grid, 256, 0, st>>>(a, b, total); break;
        case DT_BF16: weights_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(a, b, total); break;
        case DT_F16: weights_kernel<__half><<<grid, 256, 0, st>>>(a, b, total); break;
        default: weights_kernel<__nv_fp8_e4m3><<<grid, 256, 0, st>>>(a, b, total); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_absmax(const float *v, int64_t n, unsigned *out, cudaStream_t st) {
    absmax_kernel<<<grid_for((n + 3) / 4), 256, 0, st>>>(v, n, out);
    return cudaGetLastError();
}

}  // namespace nvisr
