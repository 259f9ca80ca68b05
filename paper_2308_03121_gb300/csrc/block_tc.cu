// Residual block of the enhancement trunk, y = x + conv2(LeakyReLU(conv1(x) + b1)) + b2
// (Section 3.1: the networks NNVISR runs are stacks of such 3x3 blocks), both convs
// 64 -> 64 channels with zero padding, in one launch of 2-CTA clusters whose two SMs work
// as one M = 256 tensor-core pair (tcgen05 cta_group::2).
//
// Each CTA of the pair owns one column tile of the image and runs both convolutions on it;
// every MMA covers 128 pixels of both tiles.  What bounds the block is the SMs' shared-memory
// bandwidth: a 128-pixel x (3 stacked taps x 64 outputs) MMA takes 96 cycles and reads 4 KB of
// pixels and 6 KB of weights, 107 of the 128 bytes per clock that shared memory delivers, so
// that the epilogues' traffic stalls the tensor pipe.  In a pair each SM holds and reads half
// of the weight rows (3 KB per MMA), and the middle tensor h stays on the SM that computes it.
//
//  * Stacked taps: input row n feeds accumulator rows n - 1 (ky = 2), n (ky = 1) and n + 1
//    (ky = 0) with one N = 192 MMA per (kx, 16-channel K step), 12 per row.
//  * Accumulators: three rows, row i in slot i % 3 of a fixed 192-column TMEM window per conv,
//    so a row of the MMA's N never wraps.  The order of the taps along N rotates with n
//    instead: the weights of a kx lie in shared memory as the blocks ky = 2, 1, 0, 2, 1 and the
//    MMA starts at block 0, 1 or 2.  The epilogue zeroes a slot as it drains it, so every MMA
//    accumulates: no first-product case, and the rows before and after a strip are drained
//    and dropped.
//  * The pair splits N in halves, the lower one from CTA 0: CTA c holds output channels
//    [32c, 32c + 32) of every block, and a slot's channels 0-31 lie at window column 32 slot,
//    channels 32-63 at 96 + 32 slot, in both CTAs' TMEM.
//  * Roles per CTA: warp 0 TMA-loads rows of x; warps 2-9 turn each finished conv1 row into
//    h = LeakyReLU(acc + b1), rounded to the activation type and staged 128-byte swizzled
//    where conv2's MMAs read it; warps 10-17 add b2 and the residual x (a TMA load, an L2 hit)
//    to each finished conv2 row, in the tile the residual came in, which warp 18 stores by TMA.
//    Warp 1 of CTA 0 issues every MMA: conv1 of row n, then conv2 of the h row that conv1's
//    row n - 1 completed, so each conv's epilogue has the other conv's MMAs to run behind.
//    Warp 19 of CTA 1 reports its landed x rows to CTA 0.
//
// h never reaches device memory: the DRAM traffic is x read once plus y written once (at
// 1920 x 1080 531 MB instead of 1327 MB for two single-layer launches).
//
// Tiles: conv1 computes the 128 h pixels [x0 - 1, x0 + 127) of a row (the MMA's M), which
// give conv2 the 126 outputs [x0, x0 + 126): column tiles are 126 pixels wide (x0 = 126 c)
// and conv2's two last accumulator lanes are discarded.  h pixels or rows outside the
// image are written as zero (conv2's zero padding).  A pair takes column tiles 2k and 2k + 1
// over the same rows; the last tile of an odd count is cut into its upper and lower half, one
// per CTA.  The (image, tile pair, row) sequence is cut into equal contiguous ranges, one
// per cluster; a range is one or more strips of output rows [ra, rb) of one tile pair, for
// which conv1 produces h rows [ra - 1, rb] from x rows [ra - 2, rb + 1].
//
// Measured, BF16 (a filter's trunk, block after block): at 1920 x 1080 197 us per block, 231 us
// before with one conv per SM of the cluster and cta_group::1; at 960 x 540 55 us instead of 70.
// A row step takes 2430 cycles against 2304 of its 24 MMAs; at 1920 x 1080 the chip's power cap
// then holds the clock near 1.5 GHz (1.55 PFLOP/s, 0.93 of the sustained cuBLAS rate), so what
// is left is the arithmetic itself, with 5 % of it in the last, 30-pixel column tile.
//
// What the SMs hand each other are signals: h rows, x rows, weights and accumulators are written
// and read in one SM's memory, whichever CTA's thread issues the MMA (mbar_arrive_cluster).
//
// Every wait is bounded in time; a CTA that gives up raises the abort flags of both CTAs and
// the error word.  Both CTAs end with two cluster barriers: between them each waits for the
// last MMA commit onto its barriers, so neither leaves while the other may still write into
// its shared memory.
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tc_util.cuh"

namespace nvisr {

namespace {

constexpr int BT = 126;                   // output pixels of a column tile
constexpr int TMH = 128;                  // h pixels of a row tile (half of the pair's M)
constexpr int PXS = TMH + 2;              // x pixels of a row box
constexpr int BTHREADS = 640;             // warps: 0 x loads, 1 MMA, 2-9 conv1 epilogue, 10-17 conv2 epilogue,
                                          // 18 residual loads and y stores, 19 x rows' report
constexpr int XST = 3;                    // x rows in shared memory
constexpr int NTILE = 2;                  // residual / output tiles
constexpr int NRING = 4;                  // barriers per kind of per-row event
constexpr uint32_t AROW = PXS * 128;      // bytes of one 130-pixel row of 64 channels
constexpr uint32_t ROWB = 17408;          // its 1 KB-aligned slot
constexpr uint32_t TILEB = TMH * 128;     // one h row, one output / residual row tile
constexpr uint32_t WBLK = 32 * 128;       // weights of one (kx, ky): 32 outputs x 128 B
constexpr uint32_t WKX = 5 * WBLK;        // one kx: blocks ky = 2, 1, 0, 2, 1
constexpr uint32_t WB = 3 * WKX;          // one conv
constexpr uint32_t GKX = 3 * 64 * 128;    // one kx of the global image [kx][2 - ky][64 out][128 B]
constexpr uint32_t HDR = 1024;            // barriers, flags, biases
constexpr uint32_t WIN2 = 256;            // TMEM column of conv2's window (conv1's starts at 0)
// the MMAs read 256 bytes past the h row (they feed the two discarded lanes only): the tiles follow
constexpr int BLOCK_SMEM = 1024 + (int)(HDR + 2 * WB + XST * ROWB + TILEB + NTILE * TILEB);
constexpr uint64_t WAIT_NS = 2000000000ull;
static_assert(BLOCK_SMEM <= 232448, "227 KB per CTA");

struct BlockParams {
    int H, W, nimg;
    int ncols;                 // column tiles per image: ceil(W / 126)
    const uint8_t *w1, *w2;    // stacked weights of conv1 and conv2
    const float *b1, *b2;      // biases [64]
    int *err;
    int w_fresh;               // wait for the previous kernels before the weights and biases too
    int starve;                // test drill: no input is loaded, the pipeline waits run out
    float *yp;                 // PLANAR: the output [64][H][W] float32
};

// Units (pair rows) of an image: H for each two column tiles, half of them for a last single one.
__host__ __device__ inline int64_t block_units(int H, int ncols) {
    return (int64_t)(ncols / 2) * H + (ncols % 2 ? (H + 1) / 2 : 0);
}

// MULTI: the images of several streams (one BlockProblem each, any sizes) share the launch;
// otherwise nimg images of one size stacked along the maps' outer dimension.  PLANAR (one image):
// y goes to planar float32, rounded to the activation type, straight from the registers (128
// contiguous bytes per warp and channel) instead of through the tiles: the launch is bound by its
// MMAs, and the layout pass this saves read 265 MB and wrote 531 MB at 1080p (call 461 -> 356 us).
template <int DT, bool MULTI, bool PLANAR>
__global__ void __launch_bounds__(BTHREADS, 1)
    res_block_kernel(const __grid_constant__ CUtensorMap xmap,  // x: 130-pixel row boxes, OOB zero
                     const __grid_constant__ CUtensorMap rmap,  // x: 128-pixel row tiles (residual)
                     const __grid_constant__ CUtensorMap ymap,  // y: 126-pixel row tiles
                     const BlockParams p, const BlockProblem *__restrict__ probs, int nprob) {
    using TO = typename Elem<DT>::T;
    constexpr int AFMT = DT == DT_BF16 ? 1 : 0;
    extern __shared__ uint8_t smem_raw[];
    // same offset in both CTAs: the dynamic shared memory starts at the same address
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);  // own x row landed
    uint64_t *pfull = full + 4;                           // CTA 0: CTA 1's x row landed
    uint64_t *done1 = full + 8;                           // conv1's MMAs of an input row complete (both CTAs)
    uint64_t *done2 = full + 12;                          // conv2's
    uint64_t *free1 = full + 16;                          // CTA 0: conv1's finished row drained and zeroed by both
    uint64_t *free2 = full + 20;                          // CTA 0: conv2's
    uint64_t *hfull = full + 24;                          // CTA 0: h row written by both
    uint64_t *resfull = full + 25;                        // residual tile landed
    uint64_t *outfull = full + 27;                        // output tile written
    uint64_t *wbar = full + 29;
    uint64_t *drain = full + 30;                          // the issuer's last commit (both CTAs)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + 256);
    volatile int *abort = reinterpret_cast<volatile int *>(smem + 260);
    float *sbias = reinterpret_cast<float *>(smem + 512);  // b1, b2
    uint8_t *wsm = smem + HDR;
    uint8_t *xring = wsm + 2 * WB;
    uint8_t *hrow_sm = xring + XST * ROWB;
    uint8_t *tiles = hrow_sm + TILEB;  // residual in, output out

    const uint32_t rank = cluster_ctarank();
    const bool lead = rank == 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t npairs = cluster_count_x(), pair = cluster_id_x();
    const int64_t total = MULTI ? probs[nprob - 1].u0 + block_units(probs[nprob - 1].H, probs[nprob - 1].ncols)
                                : p.nimg * block_units(p.H, p.ncols);
    const int64_t u_begin = total * pair / npairs, u_end = total * (pair + 1) / npairs;
    // the strip at position u of this cluster's range: problem (MULTI), image, this CTA's column
    // tile, its output rows [ra, rb) (of a last single tile's lower half they may pass the image)
    struct Strip {
        int pi, img, col, ra, rb;
    };
    auto strip_at = [&](int64_t u) -> Strip {
        Strip s;
        s.pi = 0;
        int64_t local = u;
        int H = p.H, nc = p.ncols;
        if (MULTI) {
            while (s.pi + 1 < nprob && u >= probs[s.pi + 1].u0) ++s.pi;
            local = u - probs[s.pi].u0;
            H = probs[s.pi].H;
            nc = probs[s.pi].ncols;
        }
        const int64_t per = block_units(H, nc);
        s.img = MULTI ? 0 : (int)(local / per);
        local -= s.img * per;
        const int64_t fulls = (int64_t)(nc / 2) * H;
        const bool half = local >= fulls;
        if (half) local -= fulls;
        const int rows = half ? (H + 1) / 2 : H;
        const int k = (int)(local / rows);
        const int off = half ? (int)rank * rows : 0;
        s.col = half ? nc - 1 : 2 * k + (int)rank;
        s.ra = (int)(local - (int64_t)k * rows);
        s.rb = (int)min((int64_t)rows, s.ra + (u_end - u));
        s.ra += off;
        s.rb += off;
        return s;
    };
    auto xmap_of = [&](int pi) { return MULTI ? &probs[pi].xmap : &xmap; };
    auto rmap_of = [&](int pi) { return MULTI ? &probs[pi].rmap : &rmap; };
    auto ymap_of = [&](int pi) { return MULTI ? &probs[pi].ymap : &ymap; };
    auto height_of = [&](int pi) { return MULTI ? probs[pi].H : p.H; };
    auto width_of = [&](int pi) { return MULTI ? probs[pi].W : p.W; };
    const uint32_t peer_abort = mapa_shared(smem_u32(const_cast<int *>(abort)), rank ^ 1u);
    auto fail = [&]() {
        *abort = 1;
        st_cluster_u32(peer_abort, 1u);
        if (p.err) atomicExch(p.err, DEVERR_TIMEOUT);
    };
    // barrier `bar` of CTA 0, for arrivals from either CTA
    auto lead_bar = [&](uint64_t *bar) { return mapa_shared(smem_u32(bar), 0u); };

    if (p.w_fresh) griddep_wait();
    if (threadIdx.x == 0) {
        for (int k = 0; k < XST; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&pfull[k], 1);
        }
        for (int k = 0; k < NRING; ++k) {
            mbar_init(&done1[k], 1);
            mbar_init(&done2[k], 1);
            mbar_init(&free1[k], 16);  // the 8 draining warps of both CTAs
            mbar_init(&free2[k], 16);
        }
        mbar_init(hfull, 16);
        for (int k = 0; k < NTILE; ++k) {
            mbar_init(&resfull[k], 1);
            mbar_init(&outfull[k], 8);
        }
        mbar_init(wbar, 1);
        mbar_init(drain, 1);
        *abort = 0;
        fence_mbarrier_init();
        // a filter's weights are written once at its creation: loaded before the wait on the previous
        // kernel (a layer call's after the one above)
        mbar_arrive_expect_tx(wbar, 2 * WB);
        for (int c = 0; c < 2; ++c)
            for (int kx = 0; kx < 3; ++kx)
                for (int b = 0; b < 5; ++b)
                    bulk_load(wsm + c * WB + kx * WKX + b * WBLK,
                              (c ? p.w2 : p.w1) + kx * GKX + (b % 3) * (64 * 128) + rank * WBLK, WBLK, wbar);
    }
    if (threadIdx.x >= 64 && threadIdx.x < 192)
        sbias[threadIdx.x - 64] = (threadIdx.x < 128 ? p.b1 : p.b2)[(threadIdx.x - 64) & 63];
    if (warp == 1) {
        tmem_alloc2(tmem_slot, 512);
        tmem_relinquish2();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (warp >= 2 && warp < 10) {  // both windows start at zero
        const uint32_t t = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (warp < 6 ? 0u : WIN2);
        for (int k = 0; k < 6; ++k) tmem_zero32(t + (uint32_t)(32 * k));
        tmem_wait_st();
    }
    tc_fence_before();
    cluster_sync_all();  // both CTAs' barriers and accumulators are ready before either uses the other's
    tc_fence_after();
    griddep_launch_dependents();
    griddep_wait();

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- producer: x rows ra - 2 .. rb + 1 of each strip; row n takes the
            // stage of row n - 3, whose MMAs done1 reports
            int n = 0;
            bool ok = true;
            for (int64_t u = u_begin; u < u_end && ok && !p.starve;) {
                const Strip s = strip_at(u);
                u += s.rb - s.ra;
                const int xb = s.col * BT - 2;  // box pixel 0 = h pixel col * BT - 1 minus one
                for (int r = s.ra - 2; r <= s.rb + 1; ++r, ++n) {
                    const int k = n - XST;
                    if (k >= 0 && !mbar_wait_bounded(&done1[k % NRING], (uint32_t)((k / NRING) & 1), abort, WAIT_NS)) {
                        fail();
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&full[n % XST], AROW);
                    tma_load_4d(xring + (size_t)(n % XST) * ROWB, xmap_of(s.pi), &full[n % XST], 0, xb, r, s.img);
                }
            }
            // copies still in flight after an early exit land before the CTA ends
            for (int k = 0; k < XST && k < n; ++k) {
                const int i = n - 1 - k;
                mbar_wait_bounded(&full[i % XST], (uint32_t)((i / XST) & 1), nullptr, WAIT_NS);
            }
            mbar_wait_bounded(wbar, 0, nullptr, WAIT_NS);
        }
    } else if (warp == 1) {
        if (lead) {
            // ---------------- MMA issuer.  The whole warp runs the loop with uniform values and
            // one elected lane issues: 96 cycles per MMA back to back, where a lane-0 branch
            // spends 57 cycles or more on each issue whatever its N.
            const uint32_t el = elect_one();
            const uint32_t id = instr_desc(256, 192, AFMT, AFMT);
            bool ok = true;
            // both CTAs' weights: the peer's have landed before its first x row is reported
            auto await = [&](uint64_t *bar, int i, int ring) {
                ok = ok && __all_sync(0xffffffffu, mbar_wait_bounded(&bar[i % ring], (uint32_t)((i / ring) & 1), abort,
                                                                     WAIT_NS));
            };
            auto issue = [&](const uint8_t *row, const uint8_t *wts, uint32_t win, int n, uint64_t *done) {
                tc_fence_after();
                // taps of slots 0, 1, 2 for input row n: blocks start at 1, 0, 2 for n % 3 = 0, 1, 2
                const int rot = n % 3 == 2 ? 2 : 1 - n % 3;
                const uint64_t a0 = smem_desc_sw128(smem_u32(row), 0);
                const uint64_t b0 = smem_desc_sw128(smem_u32(wts) + (uint32_t)rot * WBLK, 0);
#pragma unroll
                for (int t = 0; t < 12; ++t)
                    umma2_warp(el, tmem_base + win, a0 + (uint64_t)(((t / 4) * 128 + (t % 4) * 32) >> 4),
                               b0 + (uint64_t)(((t / 4) * WKX + (t % 4) * 32) >> 4), id);
                umma2_commit_warp(el, &done[n % NRING]);
            };
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(wbar, 0, abort, WAIT_NS));
            int n = 0, m = 0, kept = 0;  // conv1 inputs, conv2 inputs issued; h rows of the conv1 inputs before n
            auto conv2 = [&]() {
                await(hfull, m, 1);
                if (m > 0) await(free2, m - 1, NRING);
                if (ok) issue(hrow_sm, wsm + WB, WIN2, m, done2);
                ++m;
            };
            for (int64_t u = u_begin; u < u_end && ok;) {
                const Strip s = strip_at(u);
                u += s.rb - s.ra;
                const int rows = s.rb - s.ra + 4;
                for (int t = 0; t < rows && ok; ++t, ++n) {
                    await(full, n, XST);
                    await(pfull, n, XST);
                    if (n > 0) await(free1, n - 1, NRING);
                    if (ok) issue(xring + (size_t)(n % XST) * ROWB, wsm, 0u, n, done1);
                    if (ok && m < kept) conv2();
                    if (t >= 2) ++kept;  // the strip's first two completed rows are dropped
                }
            }
            while (ok && m < kept) conv2();
            if (!ok && lane == 0) fail();
            umma2_commit_warp(el, drain);  // after everything issued, also by an early exit
        }
    } else if (warp == 19) {
        if (!lead && lane == 0) {
            // ---------------- CTA 1: reports its weights and landed x rows to the issuer
            bool ok = mbar_wait_bounded(wbar, 0, abort, WAIT_NS);
            int n = 0;
            for (int64_t u = u_begin; u < u_end && ok;) {
                const Strip s = strip_at(u);
                u += s.rb - s.ra;
                for (int t = 0; t < s.rb - s.ra + 4 && ok; ++t, ++n) {
                    ok = mbar_wait_bounded(&full[n % XST], (uint32_t)((n / XST) & 1), abort, WAIT_NS);
                    if (ok) mbar_arrive_cluster(lead_bar(&pfull[n % XST]));
                }
            }
            if (!ok) fail();
        }
    } else if (warp == 18) {
        if (lane == 0) {
            // ---------------- residual tiles in, output tiles out: kept row k uses tile k % 2, whose
            // residual is loaded once the store of row k - 2 has read it
            int64_t ru = u_begin;
            Strip rs = {0, 0, 0, 0, 0};
            int ro = 0, loads = 0;
            auto load_res = [&]() {
                if (ro >= rs.rb) {
                    if (ru >= u_end) return;
                    rs = strip_at(ru);
                    ru += rs.rb - rs.ra;
                    ro = rs.ra;
                }
                const int k = loads % NTILE;
                mbar_arrive_expect_tx(&resfull[k], TILEB);
                tma_load_4d(tiles + (size_t)k * TILEB, rmap_of(rs.pi), &resfull[k], 0, rs.col * BT, ro, rs.img);
                ++ro;
                ++loads;
            };
            for (int k = 0; k < NTILE; ++k) load_res();
            bool ok = true;
            int yrow = 0;
            for (int64_t u = u_begin; u < u_end && ok;) {
                const Strip s = strip_at(u);
                u += s.rb - s.ra;
                const int Hs = height_of(s.pi);
                for (int o = s.ra; o < s.rb; ++o, ++yrow) {
                    const int k = yrow % NTILE;
                    if (!mbar_wait_bounded(&outfull[k], (uint32_t)((yrow / NTILE) & 1), abort, WAIT_NS)) {
                        fail();
                        ok = false;
                        break;
                    }
                    if (!PLANAR && o < Hs) {
                        tma_store_4d(ymap_of(s.pi), tiles + (size_t)k * TILEB, 0, s.col * BT, o, s.img);
                        bulk_commit_group();
                        bulk_wait_group_read<0>();  // the store has read the tile
                    }
                    load_res();
                }
            }
            bulk_wait_group<0>();
            // residual loads still in flight after an early exit land before the CTA ends
            for (int k = max(0, loads - NTILE); k < loads; ++k)
                mbar_wait_bounded(&resfull[k % NTILE], (uint32_t)((k / NTILE) & 1), nullptr, WAIT_NS);
        }
    } else {
        // ---------------- epilogues: warp w reads TMEM lane quadrant w % 4 (pixel m) and one half of
        // the channels; group 0 (warps 2-9) drains conv1's rows into the h row, group 1 (warps
        // 10-17) conv2's into the output tiles.  (Four warps per group, each with all 64 columns,
        // took 4700 cycles per row step: 1600 to drain and zero, 1400 to compute, 1300 to hand over.)
        const int g = warp < 10 ? 0 : 1;
        const int half = ((warp - 2) >> 2) & 1;
        const int q = warp & 3;
        const int m = q * 32 + lane;
        const uint32_t lanes = tmem_base + ((uint32_t)(q * 32) << 16) + (g ? WIN2 : 0u) + 96u * (uint32_t)half;
        uint64_t *done = g ? done2 : done1;
        const uint32_t freed = lead_bar(g ? free2 : free1);
        const float *sb = sbias + 64 * g + 32 * half;
        bool w = true;
        float v[32];
        auto await = [&](uint64_t *bar, uint32_t parity) {
            w = __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, abort, WAIT_NS));
            if (!w && lane == 0) fail();
            return w;
        };
        // waits for input row i's MMAs, takes the accumulator row they completed (slot (i - 1) % 3)
        // into v, zeroes it and adds the bias, in packed f32x2 arithmetic (the single-layer kernel's)
        auto drain_row = [&](int i, bool keep) {
            if (!await(&done[i % NRING], (uint32_t)((i / NRING) & 1))) return false;
            tc_fence_after();
            const uint32_t t = lanes + 32u * (uint32_t)((i + 2) % 3);
            if (keep) {
                uint32_t r[32];
                tmem_ld32_nowait(t, r);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]);
            }
            tmem_zero32(t);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(freed + (uint32_t)(i % NRING) * 8u);
            if (keep) {
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    const float4 b = *reinterpret_cast<const float4 *>(sb + e);
                    add_f32x2(v[e], v[e + 1], b.x, b.y);
                    add_f32x2(v[e + 2], v[e + 3], b.z, b.w);
                }
            }
            return true;
        };
        // 16-byte unit uu of this half's 64 bytes of a 128-byte-swizzled line
        auto unit_at = [&](uint8_t *row, int uu) {
            return reinterpret_cast<uint4 *>(row + m * 128 + (((half * 4 + uu) ^ (m & 7)) * 16));
        };
        auto pack_unit = [&](int uu) {
            uint4 ov;
            ov.x = pack2<TO>(v[uu * 8 + 0], v[uu * 8 + 1]);
            ov.y = pack2<TO>(v[uu * 8 + 2], v[uu * 8 + 3]);
            ov.z = pack2<TO>(v[uu * 8 + 4], v[uu * 8 + 5]);
            ov.w = pack2<TO>(v[uu * 8 + 6], v[uu * 8 + 7]);
            return ov;
        };
        int i = 0;  // input rows of this group's conv
        if (g == 0) {
            const uint32_t hfull_lead = lead_bar(hfull);
            int hrow = 0;  // h rows written
            for (int64_t u = u_begin; u < u_end && w;) {
                const Strip s = strip_at(u);
                u += s.rb - s.ra;
                const int px = s.col * BT - 1 + m;
                const bool colok = px >= 0 && px < width_of(s.pi);
                const int Hs = height_of(s.pi);
                for (int t = 0; t < s.rb - s.ra + 4; ++t, ++i) {
                    const bool keep = t >= 2;
                    if (!drain_row(i, keep)) break;
                    if (!keep) continue;
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        float t0 = v[e], t1 = v[e + 1];
                        mul_f32x2(t0, t1, 0.1f, 0.1f);
                        v[e] = fmaxf(v[e], t0);
                        v[e + 1] = fmaxf(v[e + 1], t1);
                    }
                    const int o = s.ra - 1 + t - 2;
                    const bool inside = colok && o >= 0 && o < Hs;  // else conv2's zero padding
                    uint4 ov[4];
#pragma unroll
                    for (int uu = 0; uu < 4; ++uu) {
                        ov[uu] = pack_unit(uu);
                        if (!inside) ov[uu] = make_uint4(0u, 0u, 0u, 0u);
                    }
                    // the previous h row has been read by conv2's MMAs
                    const int k = hrow - 1;
                    if (k >= 0 && !await(&done2[k % NRING], (uint32_t)((k / NRING) & 1))) break;
#pragma unroll
                    for (int uu = 0; uu < 4; ++uu) *unit_at(hrow_sm, uu) = ov[uu];
                    fence_proxy_async();  // the row, before the MMAs read it
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(hfull_lead);
                    ++hrow;
                }
            }
        } else {
            int yrow = 0;  // y rows finished
            for (int64_t u = u_begin; u < u_end && w;) {
                const Strip s = strip_at(u);
                u += s.rb - s.ra;
                for (int t = 0; t < s.rb - s.ra + 2; ++t, ++i) {
                    const bool keep = t >= 2;
                    if (!drain_row(i, keep)) break;
                    if (!keep) continue;
                    const int k = yrow % NTILE;
                    if (!await(&resfull[k], (uint32_t)((yrow / NTILE) & 1))) break;
                    uint8_t *tile = tiles + (size_t)k * TILEB;
#pragma unroll
                    for (int uu = 0; uu < 4; ++uu) {
                        uint4 *at = unit_at(tile, uu);
                        const uint4 raw = *at;
                        const uint32_t wd[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            float r0, r1;
                            unpack2<TO>(wd[h], r0, r1);
                            add_f32x2(v[uu * 8 + 2 * h], v[uu * 8 + 2 * h + 1], r0, r1);
                        }
                        if (!PLANAR) *at = pack_unit(uu);
                    }
                    fence_proxy_async();  // the tile's accesses before the async proxy
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&outfull[k]);
                    ++yrow;
                    if constexpr (PLANAR) {
                        const int px = s.col * BT + m, o = s.ra + t - 2;
                        if (m < BT && px < p.W && o < p.H) {
                            const int64_t HW = (int64_t)p.H * p.W;
                            float *yo = p.yp + (int64_t)(32 * half) * HW + (int64_t)o * p.W + px;
#pragma unroll
                            for (int e = 0; e < 32; e += 2) {
                                round2<TO>(v[e], v[e + 1]);
                                yo[(int64_t)e * HW] = v[e];
                                yo[(int64_t)(e + 1) * HW] = v[e + 1];
                            }
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    cluster_sync_all();  // every arrival and MMA commit towards either CTA has been issued
    if (warp == 1 && lane == 0) mbar_wait_bounded(drain, 0, nullptr, WAIT_NS);
    __syncthreads();
    cluster_sync_all();  // neither CTA leaves while the other may still write into its shared memory
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc2(tmem_base, 512);
    }
}

// Clusters of this kernel that fit the device at once (one CTA per SM), looked up once per device.
template <int DT, bool MULTI, bool PLANAR>
int max_pairs() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    if (cached[dev] > 0) return cached[dev];
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(2 * std::max(1, device_sm_count() / 2));
    cfg.blockDim = dim3(BTHREADS);
    cfg.dynamicSmemBytes = BLOCK_SMEM;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, res_block_kernel<DT, MULTI, PLANAR>, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        return 0;
    }
    cached[dev] = n;
    return n;
}

// units: the launch's pair rows (each cluster gets an equal range)
template <int DT, bool MULTI, bool PLANAR>
cudaError_t run_block(const CUtensorMap &xmap, const CUtensorMap &rmap, const CUtensorMap &ymap,
                      const BlockParams &p, const BlockProblem *probs, int nprob, int64_t units, cudaStream_t st) {
    cudaError_t e = set_smem_limit<res_block_kernel<DT, MULTI, PLANAR>>(BLOCK_SMEM);
    if (e != cudaSuccess) return e;
    int npairs = max_pairs<DT, MULTI, PLANAR>();
    if (npairs < 1) return cudaErrorInvalidConfiguration;
    // a strip costs its cluster about five more row steps, but while clusters are idle a shorter
    // strip still ends sooner
    npairs = (int)std::max<int64_t>(1, std::min<int64_t>(npairs, units / 4));
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * npairs);
    cfg.blockDim = dim3(BTHREADS);
    cfg.dynamicSmemBytes = BLOCK_SMEM;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, res_block_kernel<DT, MULTI, PLANAR>, xmap, rmap, ymap, p, probs, nprob);
}

cudaError_t encode_block_map(CUtensorMap *map, const void *base, int W, int H, int nimg, int box_px) {
    auto enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    cuuint64_t dims[4] = {128, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)nimg};
    cuuint64_t strides[3] = {128, (cuuint64_t)W * 128, (cuuint64_t)W * H * 128};
    cuuint32_t box[4] = {128, (cuuint32_t)box_px, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t encode_block_maps(const ConvArgs &c1, const ConvArgs &c2, CUtensorMap *xmap, CUtensorMap *rmap,
                              CUtensorMap *ymap) {
    cudaError_t e = encode_block_map(xmap, c1.x, c1.W, c1.H, c1.nimg, PXS);
    if (e == cudaSuccess) e = encode_block_map(rmap, c1.x, c1.W, c1.H, c1.nimg, TMH);
    if (e == cudaSuccess) e = encode_block_map(ymap, c2.y, c1.W, c1.H, c1.nimg, BT);
    return e;
}

BlockParams block_params(const ConvArgs &c1, const ConvArgs &c2) {
    BlockParams p{};
    p.H = c1.H;
    p.W = c1.W;
    p.nimg = c1.nimg;
    p.ncols = (c1.W + BT - 1) / BT;
    p.w1 = static_cast<const uint8_t *>(c1.w_rows);
    p.w2 = static_cast<const uint8_t *>(c2.w_rows);
    p.b1 = c1.bias;
    p.b2 = c2.bias;
    p.err = c1.err ? c1.err : c2.err;
    p.w_fresh = c1.w_fresh | c2.w_fresh;
    p.starve = test_starve();
    p.yp = c2.y_planar;
    return p;
}

}  // namespace

bool res_block_fits(const ConvArgs &c1, const ConvArgs &c2) {
    if (!rows_kernel_fits(c1) || !rows_kernel_fits(c2)) return false;
    if (c2.in_dt != c1.in_dt || c1.nimg != c2.nimg || c1.H != c2.H || c1.W != c2.W || c1.nimg < 1) return false;
    if (c1.act != 1 || c1.res || c2.act != 0 || c2.res != c1.x || c2.x != c1.y) return false;
    if (c1.y2 || c2.y2 || c1.amax || c2.amax || c1.acc_scale != 1.f || c1.out_scale != 1.f || c2.acc_scale != 1.f ||
        c2.out_scale != 1.f)
        return false;
    // other clusters still read x (halo rows and columns) while y is written
    const size_t bytes = (size_t)c1.nimg * c1.H * c1.W * 128;
    const uint8_t *xb = static_cast<const uint8_t *>(c1.x), *yb = static_cast<const uint8_t *>(c2.y);
    return !(yb < xb + bytes && xb < yb + bytes);
}

cudaError_t launch_res_block(const ConvArgs &c1, const ConvArgs &c2, cudaStream_t st) {
    if (!res_block_fits(c1, c2)) return cudaErrorInvalidValue;
    CUtensorMap xmap, rmap, ymap;
    cudaError_t e = encode_block_maps(c1, c2, &xmap, &rmap, &ymap);
    if (e != cudaSuccess) return e;
    const BlockParams p = block_params(c1, c2);
    const int64_t units = p.nimg * block_units(p.H, p.ncols);
    if (p.yp) {
        if (p.nimg != 1) return cudaErrorInvalidValue;
        return c1.in_dt == DT_BF16 ? run_block<DT_BF16, false, true>(xmap, rmap, ymap, p, nullptr, 0, units, st)
                                   : run_block<DT_F16, false, true>(xmap, rmap, ymap, p, nullptr, 0, units, st);
    }
    return c1.in_dt == DT_BF16 ? run_block<DT_BF16, false, false>(xmap, rmap, ymap, p, nullptr, 0, units, st)
                               : run_block<DT_F16, false, false>(xmap, rmap, ymap, p, nullptr, 0, units, st);
}

cudaError_t launch_res_block_multi(const ConvArgs *c1, const ConvArgs *c2, int n, BlockProblem *host_tab,
                                   BlockProblem *dev_tab, cudaStream_t st, bool copy_table, bool launch) {
    if (n < 1) return cudaSuccess;
    for (int i = 0; i < n; ++i) {
        // one image each; the same weights, biases and dtype
        if (!res_block_fits(c1[i], c2[i]) || c1[i].nimg != 1 || c1[i].in_dt != c1[0].in_dt ||
            c1[i].w_rows != c1[0].w_rows || c2[i].y_planar || c2[i].w_rows != c2[0].w_rows || c1[i].bias != c1[0].bias ||
            c2[i].bias != c2[0].bias)
            return cudaErrorInvalidValue;
    }
    int64_t units = 0;
    for (int i = 0; i < n; ++i) {
        BlockProblem &q = host_tab[i];
        cudaError_t e = encode_block_maps(c1[i], c2[i], &q.xmap, &q.rmap, &q.ymap);
        if (e != cudaSuccess) return e;
        q.H = c1[i].H;
        q.W = c1[i].W;
        q.ncols = (c1[i].W + BT - 1) / BT;
        q.pad_ = 0;
        q.u0 = units;
        units += block_units(q.H, q.ncols);
    }
    if (copy_table) {
        cudaError_t e = cudaMemcpyAsync(dev_tab, host_tab, sizeof(BlockProblem) * n, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return e;
    }
    if (!launch) return cudaSuccess;
    const BlockParams p = block_params(c1[0], c2[0]);
    return c1[0].in_dt == DT_BF16
               ? run_block<DT_BF16, true, false>(host_tab[0].xmap, host_tab[0].rmap, host_tab[0].ymap, p, dev_tab, n, units, st)
               : run_block<DT_F16, true, false>(host_tab[0].xmap, host_tab[0].rmap, host_tab[0].ymap, p, dev_tab, n, units, st);
}

}  // namespace nvisr
