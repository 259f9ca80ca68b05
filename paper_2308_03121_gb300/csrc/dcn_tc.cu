// Modulated deformable convolution (DCN v2) on the tensor cores, sm_103a.
//
// The paper ships a DCN v2 operator compatible with torchvision's
// deform_conv2d because video enhancement networks align neighbouring frames
// with it (Section 3.1).  For output pixel p, tap k and input channel c of
// offset group g:
//     y[o,p] = b[o] + sum_{c,k} w[o,c,k] * m[g,k](p) * bilinear(x_c, p + p_k + d[g,k](p))
// with out-of-image bilinear corners contributing zero.
//
// Kernel: one CTA per SM walks tiles of 32 x 4 pixels.  For each tile and tap, sixteen producer
// warps (a warp per 8-channel chunk and half tile, a lane per pixel) read the tap's offsets and
// mask, issue the bilinear corner loads of all their pixels before using any (so many gathers
// are in flight at once), blend them in FP32 with the mask folded into the row weights, and
// store 16-byte rows of the canonical no-swizzle K-major A tile in shared memory (the sampled
// im2col tile of that tap).  One warp issues the tap's tcgen05.mma's against the resident
// weights into a double-buffered TMEM accumulator; four epilogue warps add the bias and store
// the blocked output.  Every wait is bounded in time.
//
// What bounds it: the L1 data stage, one wavefront per distinct 128-byte line of a request, and
// instruction issue.  x comes in pixel pairs (launch_dcn_pairs): a 32-byte entry holds the
// 8 channels of pixels x and x + 1, so a lane fetches both corners of a sample row with one
// aligned 32-byte load and blends all 8 channels itself.  (From 16-byte entries a lane pair
// shared each pixel: 9 shuffles per 16 pixels for the records and the halves, and twice the
// blend's overhead: 311 M warp instructions at 960 x 540 and 8 groups.)  Where a filter's plan has
// no memory for the second half of the pairs (see launch_dcn_pairs) the same gather reads 16-byte
// entries, two loads a sample row.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace nvisr {

namespace {

constexpr int TM = 128;
// A tile's pixels: TY rows of TX.  The nine taps of neighbouring pixels read the same input, and a
// tile of several rows keeps that window small enough for L1: with random offsets (sigma 2) the
// 960 x 540 call takes 494, 460, 444, 446 and 463 us with rows of 128, 64, 32, 16 and 8 pixels,
// with zero offsets 393, 377, 378, 385 and 390, and the space-time filter's two layers 684, 650, 652,
// 668 and 685.  32 also leaves a warp's offset loads whole 128-byte lines.
constexpr int TX = 32, TY = TM / TX;
constexpr int NGATHER = 512;            // gather threads (a lane per pixel and chunk, two passes)
constexpr int MMA_WARP = NGATHER / 32;  // then 4 epilogue warps, the first also loads the weights and issues the MMAs
constexpr int NT = NGATHER + 128;       // 20 warps: 5 per SM sub-partition leaves 96 registers a thread
constexpr uint64_t WAIT_NS = 2000000000ull;
constexpr int SMEM_LIMIT = 232448;
// Stages of sampled taps.  Shared memory beyond 164 KB would shrink L1, which needs a line for every
// corner load in flight: at 960 x 540 with independent offsets of sigma 2 px a whole nvisr_dcn2d
// call takes 492 us with 5 stages (92 KB of L1) and 798 us with 8 (28 KB); the space-time filter's
// layer with its input copy 340 against 400 us (both with one-row tiles).
constexpr int MAX_STAGES = 5;

template <typename T>
struct Cv;
template <>
struct Cv<__nv_bfloat16> {
    static __device__ __forceinline__ float in(__nv_bfloat16 v) { return __bfloat162float(v); }
    static __device__ __forceinline__ __nv_bfloat16 out(float v) { return __float2bfloat16_rn(v); }
};
template <>
struct Cv<__half> {
    static __device__ __forceinline__ float in(__half v) { return __half2float(v); }
    static __device__ __forceinline__ __half out(float v) { return __float2half_rn(v); }
};

// Two 16-bit elements of a 32-bit word (element 0 in the low half) <-> two floats.
template <typename T>
__device__ __forceinline__ float2 unpack_pair(uint32_t w);
template <>
__device__ __forceinline__ float2 unpack_pair<__nv_bfloat16>(uint32_t w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
template <>
__device__ __forceinline__ float2 unpack_pair<__half>(uint32_t w) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&w));
}
template <typename T>
__device__ __forceinline__ uint32_t pack_pair(float lo, float hi);
template <>
__device__ __forceinline__ uint32_t pack_pair<__nv_bfloat16>(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}
template <>
__device__ __forceinline__ uint32_t pack_pair<__half>(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// acc += s * v on two lanes: one packed FP32 FMA (each lane an IEEE fma, as the scalar form).
__device__ __forceinline__ void ffma2(float2 &acc, float s, float2 v) {
    uint64_t d, x, w;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(acc.x), "f"(acc.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(v.x), "f"(v.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(w) : "f"(s));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(w), "l"(x));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc.x), "=f"(acc.y) : "l"(d));
}

__device__ __forceinline__ float2 fmul2(float s, float2 v) {
    uint64_t d, x, w;
    float2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(v.x), "f"(v.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(w) : "f"(s));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(w), "l"(x));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}

// T: 16-bit element type of x / y; NS: output channels (one slice); C: input channels; PLANAR:
// planar offsets and mask; PAIRS: x in pixel pairs (32-byte entries), else in 8-channel planes of
// 16-byte entries.
template <typename T, int NS, int C, bool PLANAR, bool PAIRS>
__global__ void __launch_bounds__(NT, 1) dcn_tc_kernel(const DcnArgs a, int stages) {
    constexpr int CPC = 8;                 // channels per 16-byte chunk
    constexpr int NCH = C / CPC;           // chunks per tap (= K / 8)
    constexpr uint32_t LBO = TM * 16;      // chunk stride inside a stage
    constexpr uint32_t STAGE = NCH * LBO;  // one tap's A tile
    constexpr int AFMT = std::is_same<T, __nv_bfloat16>::value ? 1 : 0;
    constexpr uint32_t IDESC = instr_desc(TM, NS, AFMT, AFMT);
    constexpr uint32_t NCOLS = 2 * NS <= 32 ? 32 : (2 * NS <= 64 ? 64 : (2 * NS <= 128 ? 128 : 256));
    static_assert(NCH % 2 == 0, "two chunks per MMA");

    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);
    uint64_t *empty = full + 8;
    uint64_t *tfull = empty + 8;
    uint64_t *tempty = tfull + 2;
    uint64_t *wbar = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(wbar + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const uint32_t wbytes = 9 * NCH * NS * 16;
    uint8_t *wsm = smem + 1024;
    uint8_t *stage0 = wsm + ((wbytes + 1023) & ~1023u);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int H = a.H, W = a.W;
    // blocked layouts [C/cpc][H][W][cpc]: byte address of the 8-channel unit starting at channel c
    const int ycpc = a.y_cpc;
    const int64_t HW = (int64_t)H * W;
    const int tiles_x = (W + TX - 1) / TX;
    const int ntiles = tiles_x * ((H + TY - 1) / TY);
    const int S = stages;

    if (a.w_fresh) griddep_wait();
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], NGATHER);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], 128);
        }
        mbar_init(wbar, 1);
        *abort = 0;
        fence_mbarrier_init();
        // the weights are not the previous kernel's: they load before the wait below (or after the
        // one above)
        mbar_arrive_expect_tx(wbar, wbytes);
        for (uint32_t off = 0; off < wbytes; off += 32768u)
            bulk_load(wsm + off, static_cast<const uint8_t *>(a.w) + off, min(32768u, wbytes - off), wbar);
    }
    if (warp == MMA_WARP) {
        tmem_alloc(tmem_slot, NCOLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // the next kernel may be scheduled once every CTA got here (after the TMEM allocation);
    // the features and offsets are read only after the previous kernels completed
    griddep_launch_dependents();
    griddep_wait();

    if (warp < NGATHER / 32) {
        // ------------------------------------------------ gather producers
        constexpr int NGW = NGATHER / 32;  // gather warps
        constexpr int WPC = NGW / NCH;     // warps per chunk
        constexpr int PPW = TM / WPC;      // pixels per warp
        constexpr int NPASS = PPW / 32;    // 32 pixels per pass
        static_assert(NGW % NCH == 0 && PPW % 32 == 0, "gather mapping");
        const int cc = warp % NCH;         // channel chunk of this warp
        const int pb = (warp / NCH) * PPW + lane;
        const int G = a.groups;
        const int g = (cc * CPC) / (a.cin_pad / G);
        const bool tapm = a.om_tap_major != 0;
        // this chunk's plane of pixel pairs, or of single pixels (below 4 GiB)
        constexpr uint32_t ENTRY = PAIRS ? 32 : 16;
        const uint8_t *plane = static_cast<const uint8_t *>(!PAIRS || cc < NCH / 2 ? a.x : a.x_hi) +
                               (int64_t)(PAIRS ? cc % (NCH / 2) : cc) * HW * ENTRY;
        const uint32_t rowb = (uint32_t)W * ENTRY;
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        // Corner values [pass][row]: words 0-3 the entry's first pixel, 4-7 the second.  A row is
        // loaded only when its weights are not all zero, which the bounds checks allow only
        // inside the image.  A skipped row keeps the values of an earlier load (or zero), which
        // its zero weights cancel (x is finite).
        uint32_t v[NPASS][2][8];
#pragma unroll
        for (int h = 0; h < NPASS; ++h)
#pragma unroll
            for (int e = 0; e < 8; ++e) v[h][0][e] = v[h][1][e] = 0u;
        // offsets and mask of this lane's pixels for tap k of tile t: loaded one tap ahead of
        // their use, so that their DRAM latency overlaps the previous tap
        auto load_om = [&](int t, int k, float2 (&d)[NPASS], float (&lg)[NPASS]) {
            const int ty = t / tiles_x;
            const int yt = ty * TY, xt = (t - ty * tiles_x) * TX;
            // float offsets in 32 bits (the tensors are < 2^31 floats)
            uint32_t od, oms;
            if (PLANAR) {
                od = (uint32_t)dcn_off_channel(g, k, G, false) * (uint32_t)HW;
                oms = (uint32_t)(g * 9 + k) * (uint32_t)HW;
            } else {
                const int cd = dcn_off_channel(g, k, G, tapm), cm = dcn_mask_channel(g, k, G, tapm);
                od = (uint32_t)(cd >> 2) * (uint32_t)HW * 4u + (cd & 3);
                oms = (uint32_t)(cm >> 2) * (uint32_t)HW * 4u + (cm & 3);
            }
#pragma unroll
            for (int h = 0; h < NPASS; ++h) {
                const uint32_t pix = (uint32_t)(min(yt + (pb + 32 * h) / TX, H - 1) * W + min(xt + (pb + 32 * h) % TX, W - 1));
                if (PLANAR) {
                    d[h] = make_float2(__ldg(a.om + od + pix), __ldg(a.om + od + (uint32_t)HW + pix));
                    lg[h] = __ldg(a.om_mask + oms + pix);
                } else {
                    d[h] = __ldg(reinterpret_cast<const float2 *>(a.om + od + pix * 4u));
                    lg[h] = __ldg(a.om + oms + pix * 4u);
                }
            }
        };
        float2 nd[NPASS];
        float nlg[NPASS];
        if (blockIdx.x < ntiles && !a.starve) load_om(blockIdx.x, 0, nd, nlg);
        for (int t = blockIdx.x; t < ntiles && ok && !a.starve; t += gridDim.x) {
            const int ty = t / tiles_x;
            const int yt = ty * TY, xt = (t - ty * tiles_x) * TX;
            for (int k = 0; k < 9; ++k) {
                float2 cd[NPASS];
                float clg[NPASS];
#pragma unroll
                for (int h = 0; h < NPASS; ++h) {
                    cd[h] = nd[h];
                    clg[h] = nlg[h];
                }
                if (k < 8) load_om(t, k + 1, nd, nlg);
                else if (t + (int)gridDim.x < ntiles) load_om(t + gridDim.x, 0, nd, nlg);
                // row weights (times the mask) and column weights, each zero outside the image,
                // then the corner loads (every load of the tap is issued before the first blend)
                float wy[NPASS][2], wxa[NPASS], wxb[NPASS];
#pragma unroll
                for (int h = 0; h < NPASS; ++h) {
                    const int px = xt + (pb + 32 * h) % TX, py = yt + (pb + 32 * h) / TX;
                    // mask = sigmoid(logit) with the fast exponential and division: a relative
                    // error near 1e-6, far below the 16-bit rounding of the sample it scales
                    // (0 and 1 at the extremes); the exact form cost 4 % of the launch
                    const float m = a.mask_logits ? __fdividef(1.f, 1.f + __expf(-clg[h])) : clg[h];
                    const float sy = (float)(py + k / 3 - 1) + cd[h].x;
                    const float sx = (float)(px + k % 3 - 1) + cd[h].y;
                    const float fy = floorf(sy), fx = floorf(sx);
                    const int y0 = (int)fy, x0 = (int)fx;
                    const float ly = sy - fy, lx = sx - fx;
                    const bool in = px < W && py < H;
                    wy[h][0] = in && (unsigned)y0 < (unsigned)H ? (1.f - ly) * m : 0.f;
                    wy[h][1] = in && (unsigned)(y0 + 1) < (unsigned)H ? ly * m : 0.f;
                    const float wx0 = (unsigned)x0 < (unsigned)W ? 1.f - lx : 0.f;
                    const float wx1 = (unsigned)(x0 + 1) < (unsigned)W ? lx : 0.f;
                    // left of the image (x0 = -1) column x0 + 1 is entry 0's first pixel
                    wxa[h] = x0 < 0 ? wx1 : wx0;
                    wxb[h] = x0 < 0 ? 0.f : wx1;
                    const bool need = wxa[h] != 0.f || wxb[h] != 0.f;
                    const uint32_t o0 = ((uint32_t)y0 * (uint32_t)W + (uint32_t)max(x0, 0)) * ENTRY;
                    // single pixels: the row's last one has no right neighbour (its weight is zero)
                    const uint32_t next = max(x0, 0) + 1 < W ? ENTRY : 0u;
                    auto load = [&](uint32_t o, uint32_t (&r)[8]) {
                        if constexpr (PAIRS) {
                            ld_global_nc_v8(plane + o, r);
                        } else {
                            const uint4 p0 = __ldg(reinterpret_cast<const uint4 *>(plane + o));
                            const uint4 p1 = __ldg(reinterpret_cast<const uint4 *>(plane + (o + next)));
                            r[0] = p0.x; r[1] = p0.y; r[2] = p0.z; r[3] = p0.w;
                            r[4] = p1.x; r[5] = p1.y; r[6] = p1.z; r[7] = p1.w;
                        }
                    };
                    if (need && wy[h][0] != 0.f) load(o0, v[h][0]);
                    if (need && wy[h][1] != 0.f) load(o0 + rowb, v[h][1]);
                }
                // the corner loads are in flight while the warp waits for a free stage
                const bool got = mbar_wait_bounded(&empty[s], ph ^ 1, abort, WAIT_NS);
                if (!__all_sync(0xffffffffu, got)) {
                    *abort = 1;
                    if (a.err) atomicExch(a.err, DEVERR_TIMEOUT);
                    ok = false;
                    break;
                }
                uint8_t *stg = stage0 + (size_t)s * STAGE + (size_t)cc * LBO;
#pragma unroll
                for (int h = 0; h < NPASS; ++h) {
                    // channels 0-3 add column x0 before x0 + 1, channels 4-7 the other way round
                    float2 acc[4];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float fa = wy[h][r] * wxa[h], fb = wy[h][r] * wxb[h];
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            const float2 pa = unpack_pair<T>(v[h][r][w]), pbv = unpack_pair<T>(v[h][r][4 + w]);
                            if (r == 0) acc[w] = fmul2(w < 2 ? fa : fb, w < 2 ? pa : pbv);
                            else ffma2(acc[w], w < 2 ? fa : fb, w < 2 ? pa : pbv);
                            ffma2(acc[w], w < 2 ? fb : fa, w < 2 ? pbv : pa);
                        }
                    }
                    *reinterpret_cast<uint4 *>(stg + (size_t)(pb + h * 32) * 16) =
                        make_uint4(pack_pair<T>(acc[0].x, acc[0].y), pack_pair<T>(acc[1].x, acc[1].y),
                                   pack_pair<T>(acc[2].x, acc[2].y), pack_pair<T>(acc[3].x, acc[3].y));
                }
                fence_proxy_async();  // generic smem writes -> visible to the tensor core
                mbar_arrive(&full[s]);
                if (++s == S) { s = 0; ph ^= 1; }
            }
        }
    } else {
        // ------------------------------------------------ epilogue (the last 4 warps, one per lane quadrant);
        // the first also issues every tile's MMAs (its elected lane), and stores its quadrant
        // of tile i - 1 after issuing tile i
        const bool issuer = warp == MMA_WARP;
        const int q = warp & 3;
        const int m = q * 32 + lane;
        uint8_t *yb = static_cast<uint8_t *>(a.y);
        const uint32_t wbase = smem_u32(wsm);
        bool run = true;     // this warp's epilogue still runs
        bool issue = true;   // the issuer still issues
        int s = 0, last_ab = -1;
        uint32_t ph = 0, last_par = 0;
        uint32_t el = 0;
        auto fail = [&]() {
            if (lane == 0) {
                *abort = 1;
                if (a.err) atomicExch(a.err, DEVERR_TIMEOUT);
            }
        };
        auto await = [&](uint64_t *bar, uint32_t parity) {
            return (bool)__all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, abort, WAIT_NS));
        };
        if (issuer) {
            el = elect_one();
            issue = await(wbar, 0);
            if (!issue) fail();
        }
        // issues the 9 taps of tile number it (buffer it & 1); false when a wait gave up
        auto issue_tile = [&](int it) -> bool {
            const int ab = it & 1;
            const uint32_t u = (uint32_t)(it >> 1);
            bool good = await(&tempty[ab], (u & 1) ^ 1);
            if (good) {
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(ab * NS);
                for (int k = 0; k < 9; ++k) {
                    good = await(&full[s], ph);
                    if (!good) {
                        if (k > 0) {  // the final wait then covers the taps already issued
                            umma_commit_warp(el, &tfull[ab]);
                            last_ab = ab;
                            last_par = u & 1;
                        }
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sb = smem_u32(stage0 + (size_t)s * STAGE);
#pragma unroll
                    for (int j = 0; j < NCH / 2; ++j) {
                        const uint64_t ad = smem_desc(sb + 2 * j * LBO, LBO, 128);
                        const uint64_t bd = smem_desc(wbase + (uint32_t)((k * NCH + 2 * j) * NS * 16), NS * 16, 128);
                        umma_warp<0>(el, d_tmem, ad, bd, IDESC, (k | j) != 0 ? 1u : 0u);
                    }
                    umma_commit_warp(el, &empty[s]);
                    if (++s == S) { s = 0; ph ^= 1; }
                }
                if (good) {
                    umma_commit_warp(el, &tfull[ab]);
                    last_ab = ab;
                    last_par = u & 1;
                }
            }
            if (!good) fail();
            return good;
        };
        // stores this warp's quadrant of tile t (number it); false when the wait gave up
        auto store_tile = [&](int t, int it) -> bool {
            const int ab = it & 1;
            const uint32_t u = (uint32_t)(it >> 1);
            if (!await(&tfull[ab], u & 1)) {
                fail();
                return false;
            }
            tc_fence_after();
            const int ty = t / tiles_x;
            const int yy = ty * TY + m / TX, xx = (t - ty * tiles_x) * TX + m % TX;
            const bool inside = yy < H && xx < W;
            const int64_t pix = (int64_t)yy * W + xx;
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * NS);
#pragma unroll
            for (int j = 0; j < NS / 16; ++j) {
                float v[16];
                tmem_ld16(taddr + (uint32_t)(j * 16), v);
                if (!inside) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    alignas(16) T o[CPC];
#pragma unroll
                    for (int e = 0; e < CPC; ++e) {
                        const int n = j * 16 + h * 8 + e;
                        o[e] = Cv<T>::out(v[h * 8 + e] * a.acc_scale + a.bias[n]);
                    }
                    const int n = j * 16 + h * 8;
                    *reinterpret_cast<uint4 *>(yb + ((int64_t)(n / ycpc) * HW + pix) * ycpc * 2 + (n % ycpc) * 2) =
                        *reinterpret_cast<const uint4 *>(o);
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty[ab]);
            return true;
        };
        int it = 0, prev_t = -1;
        for (int t = blockIdx.x; t < ntiles && run; t += gridDim.x, ++it) {
            if (issuer) {
                if (issue) issue = issue_tile(it);
                if (!issue) break;
                if (prev_t >= 0) run = store_tile(prev_t, it - 1);
                prev_t = t;
            } else {
                run = store_tile(t, it);
            }
        }
        if (issuer && issue && run && prev_t >= 0) store_tile(prev_t, it - 1);
        if (issuer && lane == 0) {
            // nothing of this CTA's may still be in flight when it leaves
            if (last_ab >= 0) mbar_wait_bounded(&tfull[last_ab], last_par, nullptr, WAIT_NS);
            mbar_wait_bounded(wbar, 0, nullptr, WAIT_NS);
        }
    }
    __syncthreads();
    if (warp == MMA_WARP) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, NCOLS);
    }
}

template <typename T, int NS, int C, bool PLANAR, bool PAIRS>
cudaError_t run(const DcnArgs &a, cudaStream_t st) {
    constexpr uint32_t STAGE = (C / 8) * TM * 16;
    constexpr uint32_t wbytes = 9 * (C / 8) * NS * 16;
    const uint32_t wround = (wbytes + 1023) & ~1023u;
    int stages = (SMEM_LIMIT - 2048 - (int)wround) / (int)STAGE;
    if (stages > MAX_STAGES) stages = MAX_STAGES;
    if (stages < 2) return cudaErrorInvalidConfiguration;
    int smem = 2048 + (int)wround + stages * (int)STAGE;
    if (smem < 118 * 1024) smem = 118 * 1024;
    auto kern = dcn_tc_kernel<T, NS, C, PLANAR, PAIRS>;
    cudaError_t e = set_smem_limit<dcn_tc_kernel<T, NS, C, PLANAR, PAIRS>>(smem);
    if (e != cudaSuccess) return e;
    const int tiles = ((a.W + TX - 1) / TX) * ((a.H + TY - 1) / TY);
    int grid = device_sm_count();
    if (grid > tiles) grid = tiles;
    return launch_dependent(kern, grid, NT, smem, st, a, stages);
}

// One thread per (pixel, 8-channel chunk), chunk fastest: a warp reads four pixels' 128-byte
// channel lines (and their right neighbours, which L1 holds) and writes four 32-byte entries of
// eight planes, 128 contiguous bytes each, with one 32-byte store a lane (two 16-byte stores wrote each
// sector in halves: 7 us more at 960 x 540).  PAIRS = false writes 16-byte entries, all eight planes
// to lo.
template <bool PAIRS>
__global__ void __launch_bounds__(256) dcn_pairs_kernel(const uint4 *__restrict__ x, int64_t HW, int W, int per,
                                                        uint4 *__restrict__ lo, uint4 *__restrict__ hi) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p = u >> 3;
    const int cc = (int)(u & 7);
    if (p >= HW) return;
    const uint4 *src = x + ((int64_t)(cc / per) * HW + p) * per + cc % per;  // per: chunks per pixel line
    const bool last = (int)(p % W) == W - 1;
    const uint4 v0 = __ldg(src);
    if (!PAIRS) {
        lo[(int64_t)cc * HW + p] = v0;
        return;
    }
    const uint4 v1 = last ? make_uint4(0u, 0u, 0u, 0u) : __ldg(src + per);
    st_global_v8((cc < 4 ? lo : hi) + ((int64_t)(cc & 3) * HW + p) * 2, v0, v1);
}

// The same from planar float32: one lane per pixel, blockIdx.y the chunk; a lane's right
// neighbour comes from lane + 1 (lane 31 reads it itself).
template <typename T>
__global__ void __launch_bounds__(256) dcn_pairs_planar_kernel(const float *__restrict__ x, int64_t HW, int W,
                                                               uint4 *__restrict__ lo, uint4 *__restrict__ hi) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int cc = blockIdx.y;
    const float *src = x + (int64_t)cc * 8 * HW;
    auto load = [&](int64_t q) {
        float f[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = q < HW ? __ldg(src + (int64_t)e * HW + q) : 0.f;
        return make_uint4(pack_pair<T>(f[0], f[1]), pack_pair<T>(f[2], f[3]), pack_pair<T>(f[4], f[5]),
                          pack_pair<T>(f[6], f[7]));
    };
    const uint4 v0 = load(p);
    uint4 v1;
    v1.x = __shfl_down_sync(0xffffffffu, v0.x, 1);
    v1.y = __shfl_down_sync(0xffffffffu, v0.y, 1);
    v1.z = __shfl_down_sync(0xffffffffu, v0.z, 1);
    v1.w = __shfl_down_sync(0xffffffffu, v0.w, 1);
    if ((threadIdx.x & 31) == 31) v1 = load(p + 1);
    if ((int)(p % W) == W - 1) v1 = make_uint4(0u, 0u, 0u, 0u);
    if (p < HW) st_global_v8((cc < 4 ? lo : hi) + ((int64_t)(cc & 3) * HW + p) * 2, v0, v1);
    griddep_wait();  // (launched beside the weights' layout)
}

}  // namespace

cudaError_t launch_dcn_pairs(const void *x, int H, int W, int x_cpc, void *lo, void *hi, cudaStream_t st) {
    if (x_cpc != 8 && x_cpc != 64) return cudaErrorInvalidValue;
    const int64_t HW = (int64_t)H * W;
    const unsigned grid = (unsigned)((HW * 8 + 255) / 256);
    const uint4 *xs = static_cast<const uint4 *>(x);
    uint4 *l = static_cast<uint4 *>(lo), *h = static_cast<uint4 *>(hi);
    if (h) dcn_pairs_kernel<true><<<grid, 256, 0, st>>>(xs, HW, W, x_cpc / 8, l, h);
    else dcn_pairs_kernel<false><<<grid, 256, 0, st>>>(xs, HW, W, x_cpc / 8, l, h);
    return cudaGetLastError();
}

cudaError_t launch_dcn_pairs_planar(const float *x, int H, int W, int dt, void *lo, void *hi, cudaStream_t st) {
    const int64_t HW = (int64_t)H * W;
    const dim3 grd((unsigned)((HW + 255) / 256), 8);
    uint4 *l = static_cast<uint4 *>(lo), *h = static_cast<uint4 *>(hi);
    if (dt == DT_BF16) return launch_dependent(dcn_pairs_planar_kernel<__nv_bfloat16>, grd, dim3(256), 0, st, x, HW, W, l, h);
    if (dt == DT_F16) return launch_dependent(dcn_pairs_planar_kernel<__half>, grd, dim3(256), 0, st, x, HW, W, l, h);
    return cudaErrorInvalidValue;
}

cudaError_t launch_dcn_tc(const DcnArgs &a0, cudaStream_t st) {
    DcnArgs a = a0;
    a.starve = test_starve();
    if (a.y_cpc == 0) a.y_cpc = 8;
    if (a.cin_pad != 64 || a.cout_pad != 64 || (a.cin_pad / a.groups) % 8) return cudaErrorNotSupported;
    const bool planar = a.om_mask != nullptr, pairs = a.x_hi != nullptr;
    if ((planar && !pairs) || (a.y_cpc != 8 && a.y_cpc != 64)) return cudaErrorNotSupported;
    if (a.om_tap_major && a.groups % 2) return cudaErrorNotSupported;
    // 32-bit gather offsets into a plane of x and into the offsets and mask
    if ((int64_t)a.H * a.W * 32 >= (int64_t(1) << 32) || (int64_t)a.H * a.W * a.om_cpad >= (int64_t(1) << 31))
        return cudaErrorNotSupported;
    auto go = [&](auto elem) {
        using T = decltype(elem);
        if (planar) return run<T, 64, 64, true, true>(a, st);
        return pairs ? run<T, 64, 64, false, true>(a, st) : run<T, 64, 64, false, false>(a, st);
    };
    if (a.in_dt == DT_BF16 && a.out_dt == DT_BF16) return go(__nv_bfloat16{});
    if (a.in_dt == DT_F16 && a.out_dt == DT_F16) return go(__half{});
    return cudaErrorNotSupported;
}

}  // namespace nvisr
