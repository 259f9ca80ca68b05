// FP32 SIMT convolution and modulated deformable convolution (the "plain" path).
//
// The networks NNVISR hosts are stacks of 3x3 convolutions (Section 3.1) plus
// the DCN v2 operator the paper ships (Section 3.1, torchvision semantics).
// This file computes both on the FP32 CUDA-core lanes, as implicit GEMM:
//   M = output pixels (a 128-pixel row segment per block),
//   N = output channels (NB per block),
//   K = taps x input channels, walked in slices of 8 input channels.
// Per slice a block stages the input halo (conv: 8 ch x KS rows x 130 px) or
// the bilinear-sampled, mask-weighted im2col tile (DCN: 8 ch x 9 taps x 128
// px) in shared memory, plus the weights [8][KS*KS][NB]; each thread
// accumulates 8 pixels x 4 output channels in registers.  The epilogue fuses
// bias, LeakyReLU(0.1), the residual add, and -- for a network's last layer
// -- PixelShuffle(2) plus the skip (nearest / bilinear upsample of the input
// frame) into a planar float32 image.
//
// Tensors use the blocked layout [C/4][H][W][4] (16-byte channel chunks).
//
// 3x3 layers without a shuffle, nearly all of the path's work, run on conv3_f32_kernel
// (below), with the same sums in the same order.
#include "common.cuh"
#include "epilogue.cuh"
#include "sm100_ptx.cuh"

namespace nvisr {

namespace {

constexpr int TW = 128;  // output pixels per block (one row segment)

// Bilinear sample with zero contribution from out-of-image corners, 4 channels.
__device__ __forceinline__ float4 bilinear4(const float4 *plane, int H, int W, float sy, float sx) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const float fy = floorf(sy), fx = floorf(sx);
    const int y0 = (int)fy, x0 = (int)fx;
    const float ly = sy - fy, lx = sx - fx;
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
        const int yy = y0 + dy;
        if (yy < 0 || yy >= H) continue;
        const float wy = dy ? ly : 1.f - ly;
#pragma unroll
        for (int dx = 0; dx < 2; ++dx) {
            const int xx = x0 + dx;
            if (xx < 0 || xx >= W) continue;
            const float wgt = wy * (dx ? lx : 1.f - lx);
            const float4 t = plane[(int64_t)yy * W + xx];
            v.x += wgt * t.x; v.y += wgt * t.y; v.z += wgt * t.z; v.w += wgt * t.w;
        }
    }
    return v;
}

// MODE 0: convolution (halo staging); MODE 1: DCN (sampled im2col staging).
template <int NB, int KS, int MODE>
__global__ void __launch_bounds__(16 * NB / 4) conv_simt_kernel(ConvArgs a, DcnArgs d) {
    constexpr int NT = 16 * NB / 4;
    constexpr int KK = KS * KS;
    constexpr int PAD = (KS - 1) / 2;
    constexpr int APX = (MODE == 0) ? (KS == 3 ? 132 : 128) : 128;  // row pitch of the staged tile
    constexpr int AROWS = (MODE == 0) ? KS : KK;                   // halo rows or taps
    extern __shared__ __align__(16) float smem_f[];
    float(*As)[AROWS][APX] = reinterpret_cast<float(*)[AROWS][APX]>(smem_f);
    float(*Bs)[KK][NB] = reinterpret_cast<float(*)[KK][NB]>(smem_f + 8 * AROWS * APX);

    const int H = MODE == 0 ? a.H : d.H;
    const int W = MODE == 0 ? a.W : d.W;
    const int cin_pad = MODE == 0 ? a.cin_pad : d.cin_pad;
    const int cout_pad = MODE == 0 ? a.cout_pad : d.cout_pad;
    const float *wts = (const float *)(MODE == 0 ? a.w : d.w);
    const float4 *xin = (const float4 *)(MODE == 0 ? a.x : d.x);

    const int tiles_x = (W + TW - 1) / TW;
    const int tile = blockIdx.x;
    const int img = tile / (tiles_x * H);
    const int rem = tile - img * tiles_x * H;
    const int y = rem / tiles_x;
    const int x0 = (rem - y * tiles_x) * TW;
    const int ot = blockIdx.y;
    const int tid = threadIdx.x;
    const int pg = tid % 16, og = tid / 16;
    const int64_t HW = (int64_t)H * W;
    const float4 *ximg = xin + (int64_t)img * (cin_pad / 4) * HW;

    float acc[8][4];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[p][n] = 0.f;

    for (int s = 0; s < cin_pad / 8; ++s) {
        // ---- stage A
        if (MODE == 0) {
            constexpr int PXN = TW + KS - 1;
            for (int i = tid; i < 2 * KS * PXN; i += NT) {
                const int cl = i / (KS * PXN);
                const int r = (i / PXN) % KS;
                const int p = i % PXN;
                const int iy = y + r - PAD, ix = x0 + p - PAD;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (iy >= 0 && iy < H && ix >= 0 && ix < W)
                    v = ximg[(int64_t)(s * 2 + cl) * HW + (int64_t)iy * W + ix];
                As[cl * 4 + 0][r][p] = v.x;
                As[cl * 4 + 1][r][p] = v.y;
                As[cl * 4 + 2][r][p] = v.z;
                As[cl * 4 + 3][r][p] = v.w;
            }
        } else {
            const int cpg = d.cin_pad / d.groups;
            for (int i = tid; i < 2 * KK * TW; i += NT) {
                const int cl = i / (KK * TW);
                const int k = (i / TW) % KK;
                const int p = i % TW;
                const int xx = x0 + p;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (xx < W) {
                    const int c = (s * 2 + cl) * 4;
                    const int g = c / cpg;
                    const int64_t pix = (int64_t)y * W + xx;
                    auto omv = [&](int ch) { return d.om[((int64_t)(ch >> 2) * HW + pix) * 4 + (ch & 3)]; };
                    const int cd = dcn_off_channel(g, k, d.groups, d.om_tap_major != 0);
                    const bool planar = d.om_mask != nullptr;
                    const float dy = planar ? d.om[(int64_t)cd * HW + pix] : omv(cd);
                    const float dx = planar ? d.om[(int64_t)(cd + 1) * HW + pix] : omv(cd + 1);
                    float m = planar ? d.om_mask[(int64_t)(g * 9 + k) * HW + pix]
                                     : omv(dcn_mask_channel(g, k, d.groups, d.om_tap_major != 0));
                    if (d.mask_logits) m = 1.f / (1.f + expf(-m));
                    const float sy = (float)(y + k / 3 - 1) + dy;
                    const float sx = (float)(xx + k % 3 - 1) + dx;
                    v = bilinear4(ximg + (int64_t)(s * 2 + cl) * HW, H, W, sy, sx);
                    v.x *= m; v.y *= m; v.z *= m; v.w *= m;
                }
                As[cl * 4 + 0][k][p] = v.x;
                As[cl * 4 + 1][k][p] = v.y;
                As[cl * 4 + 2][k][p] = v.z;
                As[cl * 4 + 3][k][p] = v.w;
            }
        }
        // ---- stage B: weights [cin_pad][KK][cout_pad] -> Bs[8][KK][NB]
        for (int i = tid; i < 8 * KK * NB / 4; i += NT) {
            const int c = i / (KK * NB / 4);
            const int t = (i / (NB / 4)) % KK;
            const int n4 = i % (NB / 4);
            const float4 v = *reinterpret_cast<const float4 *>(
                wts + ((int64_t)(s * 8 + c) * KK + t) * cout_pad + ot * NB + n4 * 4);
            *reinterpret_cast<float4 *>(&Bs[c][t][n4 * 4]) = v;
        }
        __syncthreads();
        // ---- multiply
#pragma unroll 2
        for (int c = 0; c < 8; ++c) {
            if (MODE == 0) {
#pragma unroll
                for (int ky = 0; ky < KS; ++ky) {
                    float av[8 + KS - 1];
                    const float *ar = &As[c][ky][pg * 8];
                    const float4 a0 = *reinterpret_cast<const float4 *>(ar);
                    const float4 a1 = *reinterpret_cast<const float4 *>(ar + 4);
                    av[0] = a0.x; av[1] = a0.y; av[2] = a0.z; av[3] = a0.w;
                    av[4] = a1.x; av[5] = a1.y; av[6] = a1.z; av[7] = a1.w;
                    if (KS == 3) {
                        const float2 a2 = *reinterpret_cast<const float2 *>(ar + 8);
                        av[8 % (8 + KS - 1)] = a2.x;
                        av[9 % (8 + KS - 1)] = a2.y;
                    }
#pragma unroll
                    for (int kx = 0; kx < KS; ++kx) {
                        const float4 b = *reinterpret_cast<const float4 *>(&Bs[c][ky * KS + kx][og * 4]);
#pragma unroll
                        for (int p = 0; p < 8; ++p) {
                            const float v = av[p + kx];
                            acc[p][0] += v * b.x; acc[p][1] += v * b.y;
                            acc[p][2] += v * b.z; acc[p][3] += v * b.w;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < KK; ++k) {
                    const float *ar = &As[c][k][pg * 8];
                    const float4 a0 = *reinterpret_cast<const float4 *>(ar);
                    const float4 a1 = *reinterpret_cast<const float4 *>(ar + 4);
                    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                    const float4 b = *reinterpret_cast<const float4 *>(&Bs[c][k][og * 4]);
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        acc[p][0] += av[p] * b.x; acc[p][1] += av[p] * b.y;
                        acc[p][2] += av[p] * b.z; acc[p][3] += av[p] * b.w;
                    }
                }
            }
        }
        __syncthreads();
    }

    // ---- epilogue
    const int oc0 = ot * NB + og * 4;
    const float *bias = MODE == 0 ? a.bias : d.bias;
    const float accs = MODE == 0 ? a.acc_scale : d.acc_scale;
    const float4 bv = *reinterpret_cast<const float4 *>(bias + oc0);
    const int act = MODE == 0 ? a.act : 0;
    float4 *yout = (float4 *)(MODE == 0 ? a.y : d.y);
    for (int p = 0; p < 8; ++p) {
        const int xx = x0 + pg * 8 + p;
        if (xx >= W) break;
        float v[4] = {acc[p][0] * accs + bv.x, acc[p][1] * accs + bv.y,
                      acc[p][2] * accs + bv.z, acc[p][3] * accs + bv.w};
        if (act == 1) {
#pragma unroll
            for (int n = 0; n < 4; ++n) v[n] = lrelu(v[n]);
        }
        if (MODE == 0 && a.ps > 0) {
            // PixelShuffle(2): channels oc0..oc0+3 are output channel oc0/4 at
            // sub-positions (i, j) = (0,0), (0,1), (1,0), (1,1).
            const int c = oc0 / 4;
            if (oc0 + 3 >= a.cout) continue;
            if (a.ps_out) {
                for (int ij = 0; ij < 4; ++ij) {
                    const int Y = 2 * y + (ij >> 1), X = 2 * xx + (ij & 1);
                    float o = v[ij] + skip_value(a, c, Y, X, a.skip_scale, a.skip_h, a.skip_w);
                    a.ps_out[(int64_t)c * a.ps_pitch * (2 * H) + (int64_t)Y * a.ps_pitch + X] = o;
                }
            } else {
                float *yo = (float *)a.y + (int64_t)img * (a.cout / 4) * 4 * HW;
                for (int ij = 0; ij < 4; ++ij) {
                    const int Y = 2 * y + (ij >> 1), X = 2 * xx + (ij & 1);
                    float o = v[ij];
                    if (a.ps_act == 1) o = lrelu(o);
                    yo[(((int64_t)(c / 4) * (2 * H) + Y) * (2 * W) + X) * 4 + (c % 4)] = o;
                }
            }
            continue;
        }
        const int64_t off = (int64_t)img * (cout_pad / 4) * HW + (int64_t)(oc0 / 4) * HW +
                            (int64_t)y * W + xx;
        if (MODE == 0 && a.res) {
            const float4 r = reinterpret_cast<const float4 *>(a.res)[off];
            v[0] += r.x; v[1] += r.y; v[2] += r.z; v[3] += r.w;
        }
        yout[off] = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// ---------------------------------------------------------------- 3x3 layers

// A block computes 2 rows x 64 pixels x NB outputs; warp = (row, 32 pixels), lane = (pixel group
// lane / 8, output group lane % 8), a thread 8 pixels (2 runs of 4, 16 apart) x NB / 8 outputs, so
// 8 x 8 sums at NB = 64.  What bounds it is the FP32 FMA rate.  The 8 x 4 thread tile of
// conv_simt_kernel read 22 shared-memory words per 96 FMAs, with 2- to 4-way bank conflicts, and
// staged each slice of 8 input channels between two barriers with nothing else to do.  Here a
// (channel, ky) reads 36 words without conflicts per 192 FMAs, issued as 96 packed FMAs
// (fma.rn.f32x2, each half an IEEE FMA), and the next slice's rows and weights arrive by cp.async
// meanwhile.  Three blocks of four warps share an SM.  960 x 540, 64 -> 64: 763 us with 16 pixels a
// thread and 8 rows a block, which halves the weight reads but leaves two warps to a scheduler (FMA
// pipe 71 % busy); with 8 pixels 722, 709 and 688 us with 8, 4 and 2 rows a block (blocks of more
// rows wait for each other at the slice barriers and fill the last round worse: 64 x 64 takes 129,
// 82 and 60 us); 675 with the registers of three resident blocks (150 a thread) instead of four (126);
// 660 with the channel loop unrolled four times (two 660, eight 662; 64 x 64 57, 60 and 60).
// Products are summed in the same order (channel, ky, kx), so the values are the same.  960 x 540,
// 64 -> 64: the layer call 1162 -> 660 us (58 TFLOP/s; a chain of independent FMAs runs at 79).
// PLANAR: x, y and the residual are planar float32 [C][H][W] (the caller's tensors, no layout copy).
constexpr int C3_TX = 64;       // pixels of a block's row
constexpr int C3_R = 2;         // its rows
constexpr int C3_NT = 64 * C3_R;
constexpr int C3_PITCH = 68;    // floats of a staged row (66 used)

__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint64_t pair_f32(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void ffma2_64(uint64_t &acc, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

template <int NB>
constexpr size_t c3_smem() { return 2 * sizeof(float) * (8 * (C3_R + 2) * C3_PITCH + 8 * 9 * NB); }

template <int NB, bool PLANAR>
__global__ void __launch_bounds__(C3_NT, 3) conv3_f32_kernel(const __grid_constant__ ConvArgs a) {
    constexpr int R = C3_R;
    constexpr int N = NB / 8;          // outputs of a thread
    constexpr int ASZ = 8 * (R + 2) * C3_PITCH, BSZ = 8 * 9 * NB;
    extern __shared__ __align__(16) float smem_f[];
    float *As = smem_f, *Bs = smem_f + 2 * ASZ;
    const int H = a.H, W = a.W;
    const int64_t HW = (int64_t)H * W;
    const int tiles_x = (W + C3_TX - 1) / C3_TX, tiles_y = (H + R - 1) / R;
    const int tile = blockIdx.x;
    const int img = tile / (tiles_x * tiles_y);
    const int rem = tile - img * tiles_x * tiles_y;
    const int y0 = rem / tiles_x * R, x0 = rem % tiles_x * C3_TX;
    const int oc_base = blockIdx.y * NB;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int og = lane & 7, pg = lane >> 3;
    const int row = warp % R, half = warp / R;
    const float *x = static_cast<const float *>(a.x) + (PLANAR ? 0 : (int64_t)img * (a.cin_pad / 4) * HW * 4);
    const float *wts = static_cast<const float *>(a.w);

    auto stage = [&](int sl, int buf) {
        // input rows: a warp per (channel, row), pixels x0 - 1 .. x0 + 64, zero outside the image
        for (int i = warp; i < 8 * (R + 2); i += 2 * R) {
            const int c = i / (R + 2), r = i - c * (R + 2);
            const int ch = sl * 8 + c, iy = y0 + r - 1;
            const bool rok = iy >= 0 && iy < H && (!PLANAR || ch < a.cin);
            const uint32_t dst = smem_u32(As + buf * ASZ + i * C3_PITCH);
#pragma unroll
            for (int p = lane; p < C3_TX + 2; p += 32) {
                const int ix = x0 - 1 + p;
                const bool ok = rok && ix >= 0 && ix < W;
                const int64_t pix = (int64_t)iy * W + ix;
                const int64_t at = PLANAR ? (int64_t)ch * HW + pix : ((int64_t)(ch >> 2) * HW + pix) * 4 + (ch & 3);
                cp_async4(dst + 4u * (uint32_t)p, ok ? x + at : x, ok);
            }
        }
        for (int i = threadIdx.x; i < BSZ / 4; i += C3_NT) {
            const int ct = i / (NB / 4), n4 = i - ct * (NB / 4);
            cp_async16(smem_u32(Bs + buf * BSZ + i * 4), wts + ((int64_t)sl * 72 + ct) * a.cout_pad + oc_base + n4 * 4);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    uint64_t acc[8][N / 2];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int n = 0; n < N / 2; ++n) acc[p][n] = 0;

    const int nsl = a.cin_pad / 8;
    stage(0, 0);
    for (int sl = 0; sl < nsl; ++sl) {
        const int buf = sl & 1;
        if (sl + 1 < nsl) {
            stage(sl + 1, buf ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *ar0 = As + buf * ASZ + row * C3_PITCH + 32 * half + 4 * pg;
        const float *br0 = Bs + buf * BSZ;
#pragma unroll 4
        for (int c = 0; c < 8; ++c) {
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                float av[2][6];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float *ar = ar0 + (c * (R + 2) + ky) * C3_PITCH + 16 * j;
                    const float4 v0 = *reinterpret_cast<const float4 *>(ar);
                    const float2 v1 = *reinterpret_cast<const float2 *>(ar + 4);
                    av[j][0] = v0.x; av[j][1] = v0.y; av[j][2] = v0.z; av[j][3] = v0.w;
                    av[j][4] = v1.x; av[j][5] = v1.y;
                }
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const float *br = br0 + (c * 9 + ky * 3 + kx) * NB;
                    uint64_t b[N / 2];
                    if constexpr (N == 2) {
                        b[0] = *reinterpret_cast<const uint64_t *>(br + 2 * og);
                    } else {
#pragma unroll
                        for (int h = 0; h < N / 4; ++h) {
                            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(br + 32 * h + 4 * og);
                            b[2 * h] = t.x;
                            b[2 * h + 1] = t.y;
                        }
                    }
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const float v = av[p / 4][p % 4 + kx];
                        const uint64_t vv = pair_f32(v, v);
#pragma unroll
                        for (int n = 0; n < N / 2; ++n) ffma2_64(acc[p][n], vv, b[n]);
                    }
                }
            }
        }
        __syncthreads();
    }

    // ---- epilogue: outputs oc(n) = oc_base + 4 og + n (NB 64: the upper half 32 further; NB 16: 2 og + n)
    const int y = y0 + row;
    if (y >= H) return;
    auto oc_of = [&](int n) { return oc_base + (N == 2 ? 2 * og + n : 32 * (n / 4) + 4 * og + n % 4); };
    float v[N][4];  // a run of 4 pixels
    const bool vec = PLANAR && W % 4 == 0 && (reinterpret_cast<uintptr_t>(a.y) & 15) == 0;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int xx = x0 + 32 * half + 16 * j + 4 * pg;
        if (xx >= W) continue;
        const int64_t pix = (int64_t)y * W + xx;
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const float bv = a.bias[oc_of(n)];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint64_t w2 = acc[4 * j + i][n / 2];
                const float s = __uint_as_float((uint32_t)(n & 1 ? w2 >> 32 : w2));
                float o = fmaf(s, a.acc_scale, bv);
                v[n][i] = a.act == 1 ? lrelu(o) : o;
            }
        }
        if constexpr (PLANAR) {
            const float *res = static_cast<const float *>(a.res);
            float *yo = static_cast<float *>(a.y);
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const int oc = oc_of(n);
                if (oc >= a.cout) continue;
                const int64_t at = (int64_t)oc * HW + pix;
                if (res)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (xx + i < W) v[n][i] += __ldg(res + at + i);
                if (vec) {
                    *reinterpret_cast<float4 *>(yo + at) = make_float4(v[n][0], v[n][1], v[n][2], v[n][3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (xx + i < W) yo[at + i] = v[n][i];
                }
            }
        } else {
            constexpr int U = N < 4 ? N : 4;  // outputs of one 16-byte unit this thread holds
            const int64_t plane0 = (int64_t)img * (a.cout_pad / 4) * HW;
#pragma unroll
            for (int h = 0; h < N / U; ++h) {
                const int oc = oc_of(h * U);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (xx + i >= W) break;
                    const int64_t at = (plane0 + (int64_t)(oc / 4) * HW + pix + i) * 4 + oc % 4;
                    float o[U];
#pragma unroll
                    for (int n = 0; n < U; ++n) o[n] = v[h * U + n][i];
                    if (a.res)
#pragma unroll
                        for (int n = 0; n < U; ++n) o[n] += __ldg(static_cast<const float *>(a.res) + at + n);
                    float *d = static_cast<float *>(a.y) + at;
                    if constexpr (U == 4) *reinterpret_cast<float4 *>(d) = make_float4(o[0], o[1], o[2], o[3]);
                    else *reinterpret_cast<float2 *>(d) = make_float2(o[0], o[1]);
                }
            }
        }
    }
}

template <int NB, bool PLANAR>
cudaError_t launch_c3(const ConvArgs &a, cudaStream_t st) {
    constexpr size_t smem = c3_smem<NB>();
    const cudaError_t e = set_smem_limit<conv3_f32_kernel<NB, PLANAR>>((int)smem);
    if (e != cudaSuccess) return e;
    const int tiles = (a.W + C3_TX - 1) / C3_TX * ((a.H + C3_R - 1) / C3_R);
    const dim3 grid((unsigned)(tiles * a.nimg), (unsigned)(a.cout_pad / NB));
    conv3_f32_kernel<NB, PLANAR><<<grid, C3_NT, smem, st>>>(a);
    return cudaGetLastError();
}

template <int NB, int KS, int MODE>
cudaError_t launch_nb(const ConvArgs &a, const DcnArgs &d, int H, int W, int nimg, int cout_pad,
                      cudaStream_t st) {
    constexpr int KK = KS * KS;
    constexpr int APX = (MODE == 0) ? (KS == 3 ? 132 : 128) : 128;
    constexpr int AROWS = (MODE == 0) ? KS : KK;
    constexpr size_t smem = sizeof(float) * (8 * AROWS * APX + 8 * KK * NB);
    static bool configured = false;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(conv_simt_kernel<NB, KS, MODE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    dim3 grid(((W + TW - 1) / TW) * H * nimg, cout_pad / NB);
    conv_simt_kernel<NB, KS, MODE><<<grid, 16 * NB / 4, smem, st>>>(a, d);
    return cudaGetLastError();
}

}  // namespace

size_t simt_weight_bytes(int cin_pad, int cout_pad, int k) {
    return (size_t)cin_pad * k * k * cout_pad * sizeof(float);
}

void prepare_weights_simt(const float *w, int cout, int cin, int k, int cin_pad, int cout_pad, float *dst) {
    const int kk = k * k;
    for (size_t i = 0; i < (size_t)cin_pad * kk * cout_pad; ++i) dst[i] = 0.f;
    for (int o = 0; o < cout; ++o)
        for (int c = 0; c < cin; ++c)
            for (int t = 0; t < kk; ++t)
                dst[((size_t)c * kk + t) * cout_pad + o] = w[((size_t)o * cin + c) * kk + t];
}

cudaError_t launch_conv_simt(const ConvArgs &a, cudaStream_t st) {
    if (a.rq.on) return cudaErrorNotSupported;  // requantise is fused into tensor-core tails only
    DcnArgs d{};
    if (a.cin_pad % 8 || a.cout_pad % 16) return cudaErrorInvalidValue;
    const int nb = a.cout_pad % 64 == 0 ? 64 : (a.cout_pad % 32 == 0 ? 32 : 16);
    if (a.k == 3 && a.ps == 0) {
        if (nb == 64) return a.planar ? launch_c3<64, true>(a, st) : launch_c3<64, false>(a, st);
        if (nb == 32) return a.planar ? launch_c3<32, true>(a, st) : launch_c3<32, false>(a, st);
        return a.planar ? launch_c3<16, true>(a, st) : launch_c3<16, false>(a, st);
    }
    if (a.planar) return cudaErrorInvalidValue;
    if (a.k == 3) return launch_nb<16, 3, 0>(a, d, a.H, a.W, a.nimg, a.cout_pad, st);  // PixelShuffle: 4 channels a thread
    const int use_nb = a.ps > 0 ? 16 : nb;
    if (a.k == 1) {
        if (use_nb == 64) return launch_nb<64, 1, 0>(a, d, a.H, a.W, a.nimg, a.cout_pad, st);
        if (use_nb == 32) return launch_nb<32, 1, 0>(a, d, a.H, a.W, a.nimg, a.cout_pad, st);
        return launch_nb<16, 1, 0>(a, d, a.H, a.W, a.nimg, a.cout_pad, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_dcn_simt(const DcnArgs &d, cudaStream_t st) {
    ConvArgs a{};
    if (d.cin_pad % 8 || d.cout_pad % 16 || (d.cin_pad / d.groups) % 4) return cudaErrorInvalidValue;
    const int nb = d.cout_pad % 64 == 0 ? 64 : (d.cout_pad % 32 == 0 ? 32 : 16);
    if (nb == 64) return launch_nb<64, 3, 1>(a, d, d.H, d.W, 1, d.cout_pad, st);
    if (nb == 32) return launch_nb<32, 3, 1>(a, d, d.H, d.W, 1, d.cout_pad, st);
    return launch_nb<16, 3, 1>(a, d, d.H, d.W, 1, d.cout_pad, st);
}

}  // namespace nvisr
