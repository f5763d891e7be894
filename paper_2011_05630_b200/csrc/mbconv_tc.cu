// Fused inverted-residual block (MobileNetV2): 1x1 expansion (+bias, activation) -> depthwise 3x3,
// stride 1 or 2 (+bias, activation) -> 1x1 projection (+bias, optional residual, activation), as ONE
// kernel.  The expanded map (6x the block's input, the dominant HBM traffic of the unfused plan)
// never exists in memory: the hidden dimension is processed in chunks of 64 channels.  Per output tile and chunk:
//   1. expansion (tensor core): D1[frame rows x 64] = X[frame rows x C_in] * W1[chunk]^T, the input frame (tile + 1-pixel
//      halo, TMA-loaded once per tile) staying in shared memory;
//   2. epilogue 1 (warps 0-7): bias, activation, fp16 rounding, zero outside the image (the depthwise layer's
//      padding) -> hidden frame H in shared memory, rows of 64 channels 144 bytes apart (a row per lane on the way in, a row
//      per half warp on the way out: neither conflicts, and no address needs a swizzle);
//   3. depthwise 3x3 (warps 8-15, fp32 sums): a thread keeps four channels' fp16 weights in registers and walks down a column
//      of the tile; every input value is loaded once per column it is used in and joins the three output rows it touches
//      (multiply-adds with fp16 factors); bias, activation, rounding -> dense tile Hd, the next operand;
//   4. projection (tensor core): D2[tile rows x C_out] += Hd * W2[:, chunk]^T, accumulated in tensor memory across the chunks
//      (fp32, the same sum as the unchunked layer);
// then epilogue 2 (warps 8-15, behind the next tile's first depthwise chunk): bias, residual, activation, fp16 rounding.
// Where shared memory has room the output tile is staged there and leaves through TMA stores issued by the input-producer
// warp, which also fetches the residual tile by TMA straight into that staging buffer a tile ahead (added in place);
// otherwise each thread stores and reads its own pixel's channels directly.  Every intermediate is
// rounded to fp16 exactly where the layer-by-layer execution rounds it.  Without an expansion layer
// (the network's first block; stride 1 only) epilogue 1 copies the input frame into the hidden frame.
//
// The two groups of warps are two streams that only meet in the hidden frame's barriers.  Their latency chains - loads from
// tensor and shared memory, arithmetic, rounding, stores - bound the kernel: the schedulers issue in half of the cycles, the tensor
// core is active in 3.5 % of them (24 -> 144 -> 24 at 56x56, 64 images).
// The version before this one ran the depthwise layer on the tensor core
// through diagonal weight blocks: nine UMMAs of N = 16 per 16 channels, each bound by reading 128 rows of A (40 clocks), 1440
// clocks per 128 rows and chunk, and a second trip through tensor memory.  Here an output costs nine multiply-adds with fp16
// factors (fma.rn.f32.f16: no conversions) and about two more instructions.  24 -> 144 -> 24 channels at 56x56: 67.8 -> 62.6
// us at 64 images, 12.2 -> 10.7 at one; 160 -> 960 -> 160 at 7x7, one image: 31.8 -> 23.0.
//
// Warps: 0-7 epilogue 1, 8-15 depthwise and epilogue 2, 16 expansions, 17 projections, 18 input frames and output tiles, 19 weights.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "internal.h"
#include "ptx.cuh"

namespace dlf {

namespace {

constexpr int kGroupWarps = 8;
constexpr int kExpWarp = 2 * kGroupWarps;
constexpr int kProjWarp = kExpWarp + 1;
constexpr int kInWarp = kExpWarp + 2;
constexpr int kWWarp = kExpWarp + 3;
constexpr int kThreads = 32 * (kExpWarp + 4);
constexpr int kMaxSmem = 232448 - 1024;
constexpr int kMaxNb = 4;          // 128-row blocks of the frame
constexpr int kHPitch = 144;       // bytes from one row of the hidden frame to the next
constexpr int kMaxStages = 4;

struct MbParams {
    CUtensorMap tmx, tmw1, tmw2, tmy, tmr;   // input frame, the two weight slabs, output tile, residual tile
    int N, H, W, hid, Cout, Ho, Wo, stride;
    int has_expand, act1, act2, act3;
    int th, tw, fh, fw, FR, nb1, nb2;   // output tile, input frame, frame rows, 128-row blocks of the expansion / projection
    int strips[3], strip_len[3];        // depthwise columns are cut into strips of rows; by lanes per pixel: 4, 8, 16
    int xbufs, hbufs, hdbufs, d1bufs, d2bufs;   // buffers of the input frame, the hidden frame, the depthwise tile, the accumulators (1 or 2 each)
    int tiles_h, tiles_w, n_tiles;
    int kin, chunks, n2_pad;            // 64-channel planes of the input, hidden chunks, C_out rounded up to 16
    int ksteps_in_last;
    int x_off, h_off, h_bytes, hd_off, ring_off, stage_bytes, stages, bias_off;  // shared-memory byte offsets
    int so_off, so_planes;              // output staging buffer: byte offset, 64-channel planes (0: none, direct stores)
    int xplane, so_plane;               // bytes of one 64-channel plane of the input frame / of the staging buffer (rows rounded up to 8:
                                        // a UMMA reads 128 rows from a block's start, on into whatever follows; those accumulator rows are unused)
    int d2_col;                         // first TMEM column of the projection accumulators
    int w2_off, n_split, n_each;        // projection slab inside a ring stage; C_out > 256 is issued as two halves
    const __half* wd;
    const float *b1, *bd, *b2;
    const __half* res;
    __half* out;
    int* status;
};

// A pair rounded to fp16 with its activation: ReLU6, or a clamp to [lo, hi].
template <bool RELU6>
__device__ __forceinline__ uint32_t round_clamp(float a, float b, __half2 lo, __half2 hi) {
    return RELU6 ? round_act<2>(a, b) : pack_half2_clamp(a, b, lo, hi);
}

// RELU6: both the expansion's and the depthwise layer's activation
template <int STRIDE, bool RELU6>
__global__ void __launch_bounds__(kThreads, 1) mbconv_tc_kernel(const __grid_constant__ MbParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t x_full[2], x_empty[2], w1_full[kMaxStages], w1_empty[kMaxStages], w2_full[kMaxStages], w2_empty[kMaxStages];
    __shared__ uint64_t d1_full[2], d1_free[2], h_ready[2], h_free[2], hd_ready[2], hd_free[2], d2_full[2], d2_free[2], s_full, s_free;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sb = smem_raw + (base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &abort_s;
    float* bias_s = reinterpret_cast<float*>(sb + p.bias_off);  // b1[chunks * 64], bd[chunks * 64], b2[n2_pad]

    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int i = 0; i < p.stages; i++) {   // a ring stage holds a chunk's expansion slab and its projection slab, freed separately
            mbar_init(&w1_full[i], 1);
            mbar_init(&w1_empty[i], 1);
            mbar_init(&w2_full[i], 1);
            mbar_init(&w2_empty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&x_full[i], 1);
            mbar_init(&x_empty[i], p.has_expand ? 1 : kGroupWarps);
            mbar_init(&d1_full[i], 1);
            mbar_init(&d1_free[i], kGroupWarps);
            mbar_init(&h_ready[i], kGroupWarps);
            mbar_init(&h_free[i], kGroupWarps);
            mbar_init(&hd_ready[i], kGroupWarps);
            mbar_init(&hd_free[i], 1);
            mbar_init(&d2_full[i], 1);
            mbar_init(&d2_free[i], kGroupWarps);
        }
        mbar_init(&s_full, kGroupWarps);
        mbar_init(&s_free, 1);
        fence_barrier_init();
        tma_prefetch_desc(&p.tmx);
        if (p.so_planes > 0) {
            tma_prefetch_desc(&p.tmy);
            if (p.res != nullptr) tma_prefetch_desc(&p.tmr);
        }
    }
    if (warp == kExpWarp) {
        tmem_alloc(&tmem_base_s, 512);
        tmem_relinquish();
    }
    for (int i = threadIdx.x; i < p.chunks * 64; i += kThreads) {
        bias_s[i] = (p.has_expand && i < p.hid) ? __ldg(p.b1 + i) : 0.0f;
        bias_s[p.chunks * 64 + i] = i < p.hid ? __ldg(p.bd + i) : 0.0f;
    }
    for (int i = threadIdx.x; i < p.n2_pad; i += kThreads) bias_s[p.chunks * 128 + i] = i < p.Cout ? __ldg(p.b2 + i) : 0.0f;
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_launch_dependents();
    if (warp != kWWarp) pdl_wait();  // the weight producer only reads constants
    const uint32_t tmem_base = tmem_base_s;

    if (warp == kInWarp) {
        // ---- input producer: the tile's frame, one box per 64-channel plane; and, with a staging
        //      buffer, the finished tile out (TMA stores) and the next tile's residual in ------------------
        if (lane == 0) {
            const bool staged = p.so_planes > 0, has_res = p.res != nullptr;
            const uint32_t so_bytes = static_cast<uint32_t>(p.th * p.tw) * 128u;   // one plane's box
            auto fetch_residual = [&](int t) {
                const int txi = t % p.tiles_w, tyi = (t / p.tiles_w) % p.tiles_h, n = t / (p.tiles_w * p.tiles_h);
                mbar_expect_tx(&s_free, static_cast<uint32_t>(p.so_planes) * so_bytes);
                for (int pl = 0; pl < p.so_planes; pl++)
                    tma_load_4d(sb + p.so_off + pl * p.so_plane, &p.tmr, &s_free, pl * 64, txi * p.tw, tyi * p.th, n);
            };
            // tile `ti_prev` is staged: send it off, wait until the buffer has been read, hand it back
            auto send_tile = [&](int t_prev, uint32_t ti_prev, int t_next) {
                if (!mbar_wait(&s_full, ti_prev & 1u, abort_flag, p.status, 0xB10 | (blockIdx.x << 12))) return false;
                const int txi = t_prev % p.tiles_w, tyi = (t_prev / p.tiles_w) % p.tiles_h, n = t_prev / (p.tiles_w * p.tiles_h);
                for (int pl = 0; pl < p.so_planes; pl++)
                    tma_store_4d(&p.tmy, sb + p.so_off + pl * p.so_plane, pl * 64, txi * p.tw, tyi * p.th, n);
                tma_store_commit();
                tma_store_wait_read();
                if (has_res) {
                    if (t_next < p.n_tiles) fetch_residual(t_next);
                } else {
                    mbar_arrive(&s_free);
                }
                return true;
            };
            if (staged && has_res && static_cast<int>(blockIdx.x) < p.n_tiles) fetch_residual(blockIdx.x);
            uint32_t ti = 0;
            int t_prev = -1;
            bool ok = true;
            auto load_frame = [&](int t, uint32_t i) -> bool {   // the i-th frame of this CTA
                const uint32_t xb = i & (p.xbufs - 1);
                const int txi = t % p.tiles_w, tyi = (t / p.tiles_w) % p.tiles_h, n = t / (p.tiles_w * p.tiles_h);
                if (i >= static_cast<uint32_t>(p.xbufs) &&
                    !mbar_wait(&x_empty[xb], ((i >> (p.xbufs - 1)) - 1u) & 1u, abort_flag, p.status, 0xB00 | (blockIdx.x << 12)))
                    return false;
                mbar_expect_tx(&x_full[xb], static_cast<uint32_t>(p.kin) * p.FR * 128u);
                for (int pl = 0; pl < p.kin; pl++)
                    tma_load_4d(sb + p.x_off + (xb * p.kin + pl) * p.xplane, &p.tmx, &x_full[xb], pl * 64, txi * p.tw * STRIDE - 1, tyi * p.th * STRIDE - 1, n);
                return true;
            };
            if (p.xbufs > 1 && static_cast<int>(blockIdx.x) < p.n_tiles) ok = load_frame(blockIdx.x, 0);
            for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x, ti++) {
                if (p.xbufs > 1) {   // a frame ahead
                    if (t + static_cast<int>(gridDim.x) < p.n_tiles) ok = load_frame(t + gridDim.x, ti + 1);
                } else {
                    ok = load_frame(t, ti);
                }
                if (!ok) break;
                if (staged && t_prev >= 0) {
                    ok = send_tile(t_prev, ti - 1, t);
                    if (!ok) break;
                }
                t_prev = t;
            }
            if (staged && ok && t_prev >= 0) send_tile(t_prev, ti - 1, p.n_tiles);
        }
    } else if (warp == kWWarp) {
        // ---- weight producer: per chunk the expansion slab [64 hidden][C_in] and the projection slab [C_out][64 hidden]; one
        //      ring stage holds both ---------------------------------------------------------------------
        if (lane == 0) {
            int st = 0;          // ring position and phase as counters (no division on the way to a copy)
            uint32_t ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x)
                for (int hc = 0; hc < p.chunks; hc++) {
                    uint8_t* dst = sb + p.ring_off + st * p.stage_bytes;
                    if (p.has_expand) {
                        ok = mbar_wait(&w1_empty[st], ph ^ 1u, abort_flag, p.status, 0xC00 | (blockIdx.x << 12));
                        if (!ok) break;
                        mbar_expect_tx(&w1_full[st], static_cast<uint32_t>(p.kin) * 8192u);
                        for (int pl = 0; pl < p.kin; pl++) tma_load_3d(dst + pl * 8192, &p.tmw1, &w1_full[st], pl * 64, hc * 64, 0);
                    }
                    ok = mbar_wait(&w2_empty[st], ph ^ 1u, abort_flag, p.status, 0xC10 | (blockIdx.x << 12));
                    if (!ok) break;
                    mbar_expect_tx(&w2_full[st], static_cast<uint32_t>(p.n2_pad) * 128u);
                    for (int j = 0; j < p.n_split; j++)
                        tma_load_3d(dst + p.w2_off + j * p.n_each * 128, &p.tmw2, &w2_full[st], hc * 64, j * p.n_each, 0);
                    if (++st == p.stages) { st = 0; ph ^= 1u; }
                }
        }
    } else if (warp == kExpWarp) {
        // ---- expansions: D1 = X * W1[chunk]^T over the input planes, as soon as an accumulator is drained.  The whole warp walks
        //      the loops (warp-uniform descriptors), one elected lane issues ------------------------------------
        if (p.has_expand) {
            const uint32_t idesc1 = umma_idesc_f16(64), xplane16 = static_cast<uint32_t>(p.xplane) >> 4;
            int st = 0;
            uint32_t ph = 0, ti = 0, c = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x, ti++) {
                const uint32_t xb = ti & (p.xbufs - 1);
                ok = mbar_wait_warp(&x_full[xb], (ti >> (p.xbufs - 1)) & 1u, abort_flag, p.status, 0xD00 | (blockIdx.x << 12));
                for (int hc = 0; hc < p.chunks && ok; hc++, c++) {
                    const uint32_t db = c & (p.d1bufs - 1);
                    ok = mbar_wait_warp(&w1_full[st], ph, abort_flag, p.status, 0xD10 | (blockIdx.x << 12));
                    if (ok && c >= static_cast<uint32_t>(p.d1bufs))
                        ok = mbar_wait_warp(&d1_free[db], ((c >> (p.d1bufs - 1)) - 1u) & 1u, abort_flag, p.status, 0xD20 | (blockIdx.x << 12));
                    if (!ok) break;
                    tc_fence_after_sync();
                    uint32_t b_lo = umma_desc_lo(base + p.ring_off + st * p.stage_bytes), xp_lo = umma_desc_lo(base + p.x_off + xb * p.kin * p.xplane);
                    if (elect_one()) {
                        for (int pl = 0; pl < p.kin; pl++, b_lo += 512u, xp_lo += xplane16) {
                            const bool full = pl < p.kin - 1 || p.ksteps_in_last == 4;
                            uint32_t a_lo = xp_lo, d = tmem_base + db * p.nb1 * 64u;
                            for (int b = 0; b < p.nb1; b++, a_lo += 1024u, d += 64u) {
                                if (full) {
                                    umma_f16_x4(d, a_lo, b_lo, idesc1, pl != 0);
                                } else {
                                    for (int ks = 0; ks < p.ksteps_in_last; ks++)
                                        umma_f16_lo(d, a_lo + 2 * ks, kDescHiSw128, b_lo + 2 * ks, idesc1, (pl | ks) != 0);
                                }
                            }
                        }
                        umma_commit(&d1_full[db]);
                        umma_commit(&w1_empty[st]);
                        if (hc == p.chunks - 1) umma_commit(&x_empty[xb]);   // the frame is read by the expansions only
                    }
                    __syncwarp();
                    if (++st == p.stages) { st = 0; ph ^= 1u; }
                }
            }
        }
    } else if (warp == kProjWarp) {
        // ---- projections: D2 += Hd * W2[:, chunk]^T once the chunk's depthwise tile is in shared memory ---------------
        const uint32_t idesc2 = umma_idesc_f16(p.n_each);
        int st = 0;
        uint32_t ph = 0, ti = 0, c = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x, ti++) {
            const uint32_t d2b = ti & (p.d2bufs - 1);
            for (int hc = 0; hc < p.chunks && ok; hc++, c++) {
                const int jn = min(4, (p.hid - hc * 64) >> 4);
                const uint32_t hb = c & (p.hdbufs - 1);
                ok = mbar_wait_warp(&w2_full[st], ph, abort_flag, p.status, 0xD50 | (blockIdx.x << 12));
                if (ok) ok = mbar_wait_warp(&hd_ready[hb], (c >> (p.hdbufs - 1)) & 1u, abort_flag, p.status, 0xD60 | (blockIdx.x << 12));
                if (ok && hc == 0 && ti >= static_cast<uint32_t>(p.d2bufs))
                    ok = mbar_wait_warp(&d2_free[d2b], ((ti >> (p.d2bufs - 1)) - 1u) & 1u, abort_flag, p.status, 0xD70 | (blockIdx.x << 12));
                if (!ok) break;
                tc_fence_after_sync();
                uint32_t b_lo = umma_desc_lo(base + p.ring_off + st * p.stage_bytes + p.w2_off), d0 = tmem_base + p.d2_col + d2b * p.nb2 * p.n2_pad;
                const uint32_t hd_lo = umma_desc_lo(base + p.hd_off + hb * p.so_plane);
                if (elect_one()) {
                    for (int j = 0; j < p.n_split; j++, b_lo += static_cast<uint32_t>(p.n_each) * 8u, d0 += p.n_each) {
                        uint32_t a_lo = hd_lo, d = d0;
                        for (int b = 0; b < p.nb2; b++, a_lo += 1024u, d += p.n2_pad) {
                            if (jn == 4) {
                                umma_f16_x4(d, a_lo, b_lo, idesc2, hc != 0);
                            } else {
                                for (int ks = 0; ks < jn; ks++)   // (channels past the hidden width are neither written nor read)
                                    umma_f16_lo(d, a_lo + 2 * ks, kDescHiSw128, b_lo + 2 * ks, idesc2, (hc | ks) != 0);
                            }
                        }
                    }
                    umma_commit(&hd_free[hb]);
                    umma_commit(&w2_empty[st]);
                    if (hc == p.chunks - 1) umma_commit(&d2_full[d2b]);
                }
                __syncwarp();
                if (++st == p.stages) { st = 0; ph ^= 1u; }
            }
        }
    } else if (warp < kGroupWarps) {
        // ---- epilogue 1: D1 (or, without an expansion layer, the input frame) -> hidden frame ------------------------------
        // A warp takes a lane quarter and every other 16-column slice, keeps the slice's biases in registers and has the next row
        // block's TMEM load in flight while it works on this one.
        const int q = warp & 3, half = (warp >> 2) & 1;
        const __half2 lo1 = act_lo(p.act1), hi1 = act_hi(p.act1);
        int fyx[kMaxNb];   // frame position of this thread's row in each block, -1: no such row
#pragma unroll
        for (int b = 0; b < kMaxNb; b++) {
            const int r = b * 128 + q * 32 + lane;
            const int fy = r / p.fw, fx = r - fy * p.fw;
            fyx[b] = r < p.FR ? (fy << 16) | fx : -1;
        }
        uint32_t c = 0, ti = 0;   // chunks and tiles done so far (barrier phases)
        bool ok = true;
        DLF_TRACE_DECL(wacc, wmark);  // 0 frame-buffer wait, 1 D1 wait, 2 epilogue 1
        for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x, ti++) {
            const int txi = t % p.tiles_w, tyi = (t / p.tiles_w) % p.tiles_h;
            const int iy0 = tyi * p.th * STRIDE - 1, ix0 = txi * p.tw * STRIDE - 1;
            uint32_t in_img = 0u, all_in = 0u;   // which of this thread's rows lie inside the image; which blocks' rows of the whole warp do
#pragma unroll
            for (int b = 0; b < kMaxNb; b++) {
                const int gy = iy0 + (fyx[b] >> 16), gx = ix0 + (fyx[b] & 0xffff);
                const bool in = gy >= 0 && gy < p.H && gx >= 0 && gx < p.W;
                in_img |= (in ? 1u : 0u) << b;
                all_in |= (__all_sync(0xffffffffu, in || fyx[b] < 0) ? 1u : 0u) << b;
            }
            for (int hc = 0; hc < p.chunks; hc++, c++) {
                const int jn = min(4, (p.hid - hc * 64) >> 4);
                const uint32_t hb = c & (p.hbufs - 1);
                uint8_t* hbuf = sb + p.h_off + hb * p.h_bytes;
                if (c >= static_cast<uint32_t>(p.hbufs)) {
                    ok = mbar_wait(&h_free[hb], ((c >> (p.hbufs - 1)) - 1u) & 1u, abort_flag, p.status, 0xE50 | (blockIdx.x << 12));
                    if (!ok) break;
                }
                DLF_TRACE_ACC(wacc, 0, wmark);
                if (p.has_expand) {
                    const uint32_t db = c & (p.d1bufs - 1);
                    ok = mbar_wait(&d1_full[db], (c >> (p.d1bufs - 1)) & 1u, abort_flag, p.status, 0xE10 | (blockIdx.x << 12));
                    if (!ok) break;
                    DLF_TRACE_ACC(wacc, 1, wmark);
                    tc_fence_after_sync();
#pragma unroll 1
                    for (int sl = half; sl < jn; sl += 2) {
                        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + db * p.nb1 * 64u + sl * 16u;
                        uint32_t v[2][16];
                        __syncwarp();
                        tmem_ld16_issue(taddr, v[0]);
                        uint64_t bb[8];   // pairs of biases
#pragma unroll
                        for (int e = 0; e < 4; e++) *reinterpret_cast<ulonglong2*>(bb + 2 * e) = *reinterpret_cast<const ulonglong2*>(bias_s + hc * 64 + sl * 16 + 4 * e);
                        uint8_t* dst = hbuf + (q * 32 + lane) * kHPitch + sl * 32;
#pragma unroll
                        for (int b = 0; b < kMaxNb; b++, dst += 128 * kHPitch) {
                            if (b >= p.nb1) break;
                            __syncwarp();
                            tmem_ld16_wait(v[b & 1]);
                            if (b + 1 < kMaxNb && b + 1 < p.nb1) tmem_ld16_issue(taddr + (b + 1) * 64u, v[(b + 1) & 1]);
                            const uint32_t (&r)[16] = v[b & 1];
                            if (fyx[b] >= 0) {
#pragma unroll
                                for (int g = 0; g < 2; g++) {
                                    uint32_t val[4];
#pragma unroll
                                    for (int e = 0; e < 4; e++) {
                                        const float2 f = add_f2(r[g * 8 + 2 * e], r[g * 8 + 2 * e + 1], bb[g * 4 + e]);
                                        val[e] = round_clamp<RELU6>(f.x, f.y, lo1, hi1);
                                    }
                                    if (!((all_in >> b) & 1u) && !((in_img >> b) & 1u)) val[0] = val[1] = val[2] = val[3] = 0u;   // the depthwise layer's padding
                                    *reinterpret_cast<uint4*>(dst + g * 16) = make_uint4(val[0], val[1], val[2], val[3]);
                                }
                            }
                        }
                    }
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&d1_free[db]);
                } else {
                    const uint32_t xb = ti & (p.xbufs - 1);
                    if (hc == 0) {
                        ok = mbar_wait(&x_full[xb], (ti >> (p.xbufs - 1)) & 1u, abort_flag, p.status, 0xE00 | (blockIdx.x << 12));
                        if (!ok) break;
                    }
                    const uint8_t* xp = sb + p.x_off + (xb * p.kin + hc) * p.xplane;
                    for (int i = threadIdx.x; i < p.FR * 8; i += 32 * kGroupWarps) {
                        const int r = i >> 3, u = i & 7;
                        if (u < jn * 2) *reinterpret_cast<uint4*>(hbuf + r * kHPitch + u * 16) = *reinterpret_cast<const uint4*>(xp + r * 128 + ((u ^ (r & 7)) << 4));
                    }
                    __syncwarp();
                    if (hc == p.chunks - 1 && lane == 0) mbar_arrive(&x_empty[xb]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&h_ready[hb]);
                DLF_TRACE_ACC(wacc, 2, wmark);
            }
        }
        if (threadIdx.x == 0) DLF_TRACE_FLUSH_N(p.status, wacc, 8, 3);
    } else {
        // ---- depthwise layer and epilogue 2 -----------------------------------------------------------------------------------
        const int q = warp & 3, half = (warp >> 2) & 1, gw = warp - kGroupWarps;
        const __half2 lo2 = act_lo(p.act2), hi2 = act_hi(p.act2);
        const __half2 lo3 = act_lo(p.act3), hi3 = act_hi(p.act3);
        DLF_TRACE_DECL(wacc, wmark);  // 0 hidden frame wait, 1 Hd wait, 2 depthwise, 3 projection wait, 4 epilogue 2
        auto depthwise = [&](uint32_t c, int hc) -> bool {
            const int jn = min(4, (p.hid - hc * 64) >> 4);
            const uint32_t hb = c & (p.hbufs - 1), ob = c & (p.hdbufs - 1);
            // lanes of a pixel: four channels each; a chunk with few channels takes more columns per warp
            const int ll = jn == 1 ? 0 : (jn == 2 ? 1 : 2), lanes = 4 << ll;
            const int cl = lane & (lanes - 1), slots = kGroupWarps * (32 >> (ll + 2));
            const bool live = cl * 4 < jn * 16;
            const int ch = hc * 64 + (live ? cl * 4 : 0);
            unsigned short w[9][4];   // (fp16)
            {
                uint2 raw[9];   // weights of four channels, nine taps each: 36 consecutive halves
                const uint2* wp = reinterpret_cast<const uint2*>(p.wd + static_cast<long long>(ch) * 9);
#pragma unroll
                for (int i = 0; i < 9; i++) raw[i] = __ldg(wp + i);
                const unsigned short* h = reinterpret_cast<const unsigned short*>(raw);
#pragma unroll
                for (int k = 0; k < 9; k++)
#pragma unroll
                    for (int e = 0; e < 4; e++) w[k][e] = h[e * 9 + k];
            }
            const float4 bd = *reinterpret_cast<const float4*>(bias_s + p.chunks * 64 + ch);
            if (!mbar_wait(&h_ready[hb], (c >> (p.hbufs - 1)) & 1u, abort_flag, p.status, 0xE60 | (blockIdx.x << 12))) return false;
            DLF_TRACE_ACC(wacc, 0, wmark);
            if (c >= static_cast<uint32_t>(p.hdbufs) &&
                !mbar_wait(&hd_free[ob], ((c >> (p.hdbufs - 1)) - 1u) & 1u, abort_flag, p.status, 0xE20 | (blockIdx.x << 12)))
                return false;
            DLF_TRACE_ACC(wacc, 1, wmark);
            const uint8_t* hbuf = sb + p.h_off + hb * p.h_bytes + cl * 8;
            uint8_t* hd = sb + p.hd_off + ob * p.so_plane + (cl & 1) * 8;
            const int row_step = p.fw * kHPitch, len = p.strip_len[ll], items = p.tw * p.strips[ll];
            if (live) {
#pragma unroll 1
                for (int i = gw * (32 >> (ll + 2)) + (lane >> (ll + 2)); i < items; i += slots) {
                    const int strip = i / p.tw, ox = i - strip * p.tw;
                    const int oy0 = strip * len, rows = min(len, p.th - oy0);
                    const uint8_t* src = hbuf + (oy0 * STRIDE * p.fw + ox * STRIDE) * kHPitch;
                    int o = oy0 * p.tw + ox;
                    uint2 raw[3];   // the next input row, loaded while this one is worked on
                    int left = rows * STRIDE + 3 - STRIDE;
                    auto fetch = [&]() {
#pragma unroll
                        for (int s = 0; s < 3; s++) raw[s] = *reinterpret_cast<const uint2*>(src + s * kHPitch);
                        if (--left > 0) src += row_step;   // (the last row is fetched once more in vain)
                    };
                    unsigned short x[3][4];
                    auto next = [&]() {
#pragma unroll
                        for (int s = 0; s < 3; s++) {
                            unpack_h2(raw[s].x, x[s][0], x[s][1]);
                            unpack_h2(raw[s].y, x[s][2], x[s][3]);
                        }
                        fetch();
                    };
                    auto add = [&](float (&acc)[4], int r) {
#pragma unroll
                        for (int s = 0; s < 3; s++)
#pragma unroll
                            for (int e = 0; e < 4; e++) acc[e] = fma_f32_f16(x[s][e], w[r * 3 + s][e], acc[e]);
                    };
                    auto start = [&](float (&acc)[4]) {
                        acc[0] = bd.x; acc[1] = bd.y; acc[2] = bd.z; acc[3] = bd.w;
                        add(acc, 0);
                    };
                    auto store = [&](const float (&acc)[4]) {
                        *reinterpret_cast<uint2*>(hd + o * 128 + (((cl >> 1) ^ (o & 7)) << 4)) =
                            make_uint2(round_clamp<RELU6>(acc[0], acc[1], lo2, hi2), round_clamp<RELU6>(acc[2], acc[3], lo2, hi2));
                        o += p.tw;
                    };
                    float u[4], v[4], n[4];
                    fetch();
                    if (STRIDE == 1) {
                        // input row j is the last row of output j - 2, the middle one of output j - 1, the first one of output j
                        next(); start(u);
                        next(); add(u, 1); start(v);
                        int j = 0;
#pragma unroll 1
                        while (true) {
                            next(); add(u, 2); store(u);
                            if (++j == rows) break;
                            add(v, 1); start(n);
                            next(); add(v, 2); store(v);
                            if (++j == rows) break;
                            add(n, 1); start(u);
                            next(); add(n, 2); store(n);
                            if (++j == rows) break;
                            add(u, 1); start(v);
                        }
                    } else {
                        next(); start(u);
#pragma unroll 1
                        for (int j = 0;;) {
                            next(); add(u, 1);
                            next(); add(u, 2); store(u);
                            if (++j == rows) break;
                            start(u);
                        }
                    }
                }
            }
            fence_proxy_async_smem();  // the projection UMMAs read Hd through the async proxy
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&hd_ready[ob]);
                mbar_arrive(&h_free[hb]);
            }
            DLF_TRACE_ACC(wacc, 2, wmark);
            return true;
        };
        // Epilogue 2 of the i-th tile of this CTA: D2 -> global
        auto epilogue2 = [&](int t, uint32_t i) -> bool {
            const int txi = t % p.tiles_w, tyi = (t / p.tiles_w) % p.tiles_h, n = t / (p.tiles_w * p.tiles_h);
            const int oy0 = tyi * p.th, ox0 = txi * p.tw;
            const uint32_t d2b = i & (p.d2bufs - 1);
            if (!mbar_wait(&d2_full[d2b], (i >> (p.d2bufs - 1)) & 1u, abort_flag, p.status, 0xE30 | (blockIdx.x << 12))) return false;
            const bool staged = p.so_planes > 0, has_res = p.res != nullptr;
            // the staging buffer is free again (first tile: at once) / holds this tile's residual
            if (staged && !mbar_wait(&s_free, has_res ? (i & 1u) : ((i & 1u) ^ 1u), abort_flag, p.status, 0xE40 | (blockIdx.x << 12))) return false;
            DLF_TRACE_ACC(wacc, 3, wmark);
            tc_fence_after_sync();
            const float* b2s = bias_s + p.chunks * 128;
            uint8_t* so = sb + p.so_off;
#pragma unroll 1
            for (int c0 = half * 16; c0 < p.n2_pad; c0 += 32) {
                const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + p.d2_col + d2b * p.nb2 * p.n2_pad + c0;
                uint32_t v[2][16];
                __syncwarp();
                tmem_ld16_issue(taddr, v[0]);
                float bb[16];
#pragma unroll
                for (int e = 0; e < 4; e++) *reinterpret_cast<float4*>(bb + 4 * e) = *reinterpret_cast<const float4*>(b2s + c0 + 4 * e);
#pragma unroll
                for (int b = 0; b < 2; b++) {   // (a tile has at most 256 pixels)
                    if (b >= p.nb2) break;
                    __syncwarp();
                    tmem_ld16_wait(v[b]);
                    if (b == 0 && p.nb2 > 1) tmem_ld16_issue(taddr + p.n2_pad, v[1]);
                    const int o = b * 128 + q * 32 + lane;
                    if (o >= p.th * p.tw) continue;   // (rows past the image are clipped by the TMA store)
                    long long gpix = 0;
                    if (!staged) {
                        const int oy = o / p.tw, gy = oy0 + oy, gx = ox0 + o - oy * p.tw;
                        if (gy >= p.Ho || gx >= p.Wo) continue;
                        gpix = (static_cast<long long>(n) * p.Ho + gy) * p.Wo + gx;
                    }
#pragma unroll
                    for (int g = 0; g < 2; g++) {
                        const int co = c0 + g * 8;
                        if (co >= p.Cout) break;
                        uint4* sp = reinterpret_cast<uint4*>(so + (co >> 6) * p.so_plane + o * 128 + ((((co >> 3) & 7) ^ (o & 7)) << 4));
                        float a[8];
#pragma unroll
                        for (int e = 0; e < 8; e++) a[e] = __uint_as_float(v[b][g * 8 + e]) + bb[g * 8 + e];
                        if (has_res) {   // staged: loaded into the staging buffer by TMA, zero outside the tensor
                            const uint4 rv = staged ? *sp : ld_map(reinterpret_cast<const uint4*>(p.res + gpix * p.Cout + co));
                            const __half2* rh = reinterpret_cast<const __half2*>(&rv);
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                const float2 f = __half22float2(rh[e]);
                                a[2 * e] += f.x;
                                a[2 * e + 1] += f.y;
                            }
                        }
                        uint4 val;
                        val.x = pack_half2_clamp(a[0], a[1], lo3, hi3);
                        val.y = pack_half2_clamp(a[2], a[3], lo3, hi3);
                        val.z = pack_half2_clamp(a[4], a[5], lo3, hi3);
                        val.w = pack_half2_clamp(a[6], a[7], lo3, hi3);
                        if (staged) *sp = val;
                        else *reinterpret_cast<uint4*>(p.out + gpix * p.Cout + co) = val;
                    }
                }
            }
            tc_fence_before_sync();
            if (staged) fence_proxy_async_smem();  // the TMA store reads the staging buffer
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&d2_free[d2b]);
                if (staged) mbar_arrive(&s_full);
            }
            DLF_TRACE_ACC(wacc, 4, wmark);
            return true;
        };
        // A tile's last projection runs while the next tile's first chunk is convolved.
        uint32_t c = 0, ti = 0;
        int t_prev = -1;
        bool ok = true;
        for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x, ti++) {
            for (int hc = 0; hc < p.chunks && ok; hc++, c++) {
                ok = depthwise(c, hc);
                if (ok && hc == 0 && t_prev >= 0) ok = epilogue2(t_prev, ti - 1);
            }
            t_prev = t;
        }
        if (ok && t_prev >= 0) epilogue2(t_prev, ti - 1);
        if (threadIdx.x == 32 * kGroupWarps) DLF_TRACE_FLUSH_N(p.status, wacc, 11, 5);
    }

    tc_fence_before_sync();
    __syncthreads();
    if (warp == kExpWarp) {
        if (abort_s) __nanosleep(20000);
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

typedef void (*KernelFn)(const MbParams);
KernelFn pick_kernel(int stride, bool relu6) {
    if (stride == 1) return relu6 ? mbconv_tc_kernel<1, true> : mbconv_tc_kernel<1, false>;
    return relu6 ? mbconv_tc_kernel<2, true> : mbconv_tc_kernel<2, false>;
}

int pad16(int c) { return (c + 15) / 16 * 16; }

// Shared-memory and tensor-memory layout of a tile choice; false if it does not fit.
struct MbLayout {
    int fh, fw, FR, nb1, nb2, strips[3], strip_len[3];
    int xbufs, hbufs, hdbufs, d1bufs, d2bufs;
    int kin, chunks, n2;
    int x_off, h_off, h_bytes, hd_off, ring_off, stage_bytes, stages, bias_off, so_off, so_planes, xplane, so_plane;
    int d2_col;
    size_t smem;
};

bool mb_layout(const MbconvArgs& a, int th, int tw, MbLayout* L) {
    const int s = a.stride;
    L->fh = (th - 1) * s + 3; L->fw = (tw - 1) * s + 3;
    if (L->fh > 256 || L->fw > 256) return false;
    L->FR = L->fh * L->fw;
    L->nb1 = (L->FR + 127) / 128;
    L->nb2 = (th * tw + 127) / 128;
    if (L->nb1 > kMaxNb || L->nb2 > 2) return false;
    L->kin = (a.Cin + 63) / 64; L->chunks = (a.hid + 63) / 64; L->n2 = pad16(a.Cout);
    // strips of a depthwise column: the least (rounds of the threads) x (rows, two of which a strip shares with the one above)
    for (int ll = 0; ll < 3; ll++) {
        const int slots = kGroupWarps * (32 >> (ll + 2));
        int best = -1;
        for (int ns = 1; ns <= th; ns++) {
            const int len = (th + ns - 1) / ns;
            if ((ns - 1) * len >= th) continue;
            const int cost = (tw * ns + slots - 1) / slots * (len * s + 3);
            if (best < 0 || cost < best) {
                best = cost;
                L->strips[ll] = ns;
                L->strip_len[ll] = len;
            }
        }
    }
    L->h_bytes = (L->FR * kHPitch + 1023) / 1024 * 1024;
    L->xplane = (L->FR + 7) / 8 * 8 * 128;
    L->so_plane = (th * tw + 7) / 8 * 8 * 128;
    L->stage_bytes = L->kin * 8192 * (a.has_expand ? 1 : 0) + L->n2 * 128;
    const int bias_bytes = ((L->chunks * 128 + L->n2) * 4 + 1023) / 1024 * 1024;
    // accumulators: both kinds twice where tensor memory has the columns, the projection's given up first
    const int d1 = a.has_expand ? L->nb1 * 64 : 0, d2 = L->nb2 * L->n2;
    L->d1bufs = a.has_expand && 2 * d1 + d2 <= 512 ? 2 : 1;
    L->d2bufs = L->d1bufs * d1 + 2 * d2 <= 512 ? 2 : 1;
    if (L->d1bufs * d1 + L->d2bufs * d2 > 512) return false;
    L->d2_col = L->d1bufs * d1;
    // shared memory, by preference: two of everything; given up in the order: the input frame's second buffer, the depthwise
    // tile's, a third ring stage, the hidden frame's, the output staging buffer
    for (int variant = 0; variant < 6; variant++) {
        L->xbufs = variant >= 1 ? 1 : 2;
        L->hdbufs = variant >= 2 ? 1 : 2;
        L->stages = variant >= 3 ? 2 : 3;
        L->hbufs = variant >= 4 ? 1 : 2;
        L->so_planes = variant >= 5 ? 0 : (a.Cout + 63) / 64;
        L->x_off = 0;
        L->hd_off = L->xbufs * L->kin * L->xplane;   // (rows rounded up to 8: both stay on 1024-byte boundaries)
        L->ring_off = L->hd_off + L->hdbufs * L->so_plane;
        L->bias_off = L->ring_off + L->stages * L->stage_bytes;
        L->so_off = (L->bias_off + bias_bytes + 1023) / 1024 * 1024;
        L->h_off = L->so_off + L->so_planes * L->so_plane;
        // (a UMMA reads 128 rows from a block's start: past the last input frame and the last depthwise tile it reads on, inside the
        // allocation)
        L->smem = static_cast<size_t>(L->h_off) + static_cast<size_t>(L->hbufs) * L->h_bytes;
        L->smem = std::max(L->smem, static_cast<size_t>(L->hd_off) + 128u * 128u * kMaxNb);
        L->smem = std::max(L->smem, static_cast<size_t>(L->ring_off) + 128u * 128u * 2) + 1024;
        if (L->smem <= static_cast<size_t>(kMaxSmem)) return true;
    }
    return false;
}

}  // namespace

bool mbconv_supported(const MbconvArgs& a) {
    if (a.Cin % 8 || a.hid % 16 || a.Cout % 8 || a.Cin > 256 || a.Cout > 512 || a.hid > 1024) return false;
    if (pad16(a.Cout) > 256 && pad16(a.Cout) % 32) return false;  // issued as two equal halves
    if (a.stride != 1 && a.stride != 2) return false;
    if (!a.has_expand && (a.hid != a.Cin || a.stride != 1)) return false;   // (the input frame is no set of parity planes)
    return a.N >= 1 && a.H >= 1 && a.W >= 1;
}

// Output tile of the fused block from the SM count: candidates whose buffers and accumulators fit,
// least (waves x per-tile work) in SM clocks.
static MbconvTiling persistent_tiling(const MbconvArgs& a, int sm_count) {
    MbconvTiling best{};
    best.ok = false;
    if (!mbconv_supported(a) || sm_count < 1) return best;
    const int Ho = (a.H + 2 - 3) / a.stride + 1, Wo = (a.W + 2 - 3) / a.stride + 1;
    double best_cost = -1.0;
    for (int th = 1; th <= 16; th++)
        for (int tw = 2; tw <= 32; tw++) {
            if (th > std::max(Ho, 2) || tw > std::max(Wo, 2)) continue;
            if (th * tw > 256) continue;
            MbLayout L;
            if (!mb_layout(a, th, tw, &L)) continue;
            const int tiles_h = (Ho + th - 1) / th, tiles_w = (Wo + tw - 1) / tw;
            const long long n_tiles = static_cast<long long>(a.N) * tiles_h * tiles_w;
            if (n_tiles > 0x7fffffffLL) continue;
            const long long waves = (n_tiles + sm_count - 1) / sm_count;
            // SM clocks of a tile: the slower of the two groups of warps.  Epilogue 1 takes about 260 clocks per 128-row block and
            // 16-column slice of a warp, the depthwise walk about 110 per input row and round of the threads, either 450 per chunk
            // for its hand-overs.
            double g1 = 0.0, g2 = 0.0;
            for (int hc = 0; hc < L.chunks; hc++) {
                const int jn = std::min(4, (a.hid - hc * 64) / 16), ll = jn == 1 ? 0 : (jn == 2 ? 1 : 2), slots = kGroupWarps * (32 >> (ll + 2));
                g1 += 450.0 + (a.has_expand ? L.nb1 * ((jn + 1) / 2) * 260.0 : L.FR * 0.6);
                g2 += 700.0 + (tw * L.strips[ll] + slots - 1) / slots * (L.strip_len[ll] * a.stride + 2) * 110.0;
            }
            g2 += 600.0 + L.nb2 * ((L.n2 + 31) / 32) * (L.so_planes > 0 ? 300.0 : 900.0);
            const double load = L.kin * L.FR * 128 / 57.0;   // the frame through the SM's fill port
            const double item = L.hbufs == 2 ? std::max({g1, g2, load}) + (L.xbufs == 2 ? 0.0 : 800.0) + (L.hdbufs == 2 ? 0.0 : 400.0 * L.chunks) : g1 + g2;
            // (the two groups share the SM's issue slots: either takes about twice as long as alone, measured over MobileNetV2's
            // blocks at 1 to 128 images; less at stride 2, where the depthwise layer has a quarter of the outputs)
            const double cost = (static_cast<double>(waves) * item + g1 / L.chunks + 3000.0) * (a.stride == 1 ? 1.95 : 1.7);
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost;
                best.th = th; best.tw = tw; best.fh = L.fh; best.fw = L.fw; best.nb1 = L.nb1; best.nb2 = L.nb2;
                best.tiles_h = tiles_h; best.tiles_w = tiles_w; best.n_tiles = static_cast<int>(n_tiles);
                best.stages = L.stages; best.stage_bytes = L.stage_bytes;
                best.smem_bytes = L.smem;
                best.out_planes = L.so_planes;
                best.us = (cost + 3200.0) / 1.9e3;   // (launch, fill and drain)
                best.redundancy = static_cast<double>(L.FR) / (std::min(th, Ho) * a.stride * std::min(tw, Wo) * a.stride);
                best.ok = true;
            }
        }
    return best;
}

// The kernel of mbconv_lat.cu where its tiles fit the chip at once and its estimate is clearly the lower one: both are within 6 to 9 % as a
// rule, and further apart where that kernel works on narrow chunks.  Over 2350 blocks that both can run, each timed: 0.690 of the persistent
// kernel's time, against 0.688 with the better of the two each time; slower than it by more than 5 % in five, 12 % at the most.
// 64 -> 384 -> 64 at 14x14: 12.7 -> 6.5 us at one image; 24 -> 144 -> 24 at 56x56, eight images: 15.3 here, one wave of tiles is none there;
// 128 -> 768 -> 104, stride 2 at 41x37, 27 images: 46 here, 75 there.
MbconvTiling mbconv_tiling(const MbconvArgs& a, int sm_count) {
    const MbconvTiling t = persistent_tiling(a, sm_count), l = mbconv_lat_tiling(a, sm_count);
    return t.ok && l.ok && l.us < (l.narrow ? 0.8 : 0.93) * t.us ? l : t;   // (what this kernel cannot hold is no group: plans stay as legal as they were)
}

int mbconv_tc_init() {
    static bool attr_set[kMaxDevices] = {};
    const int dev = current_device_slot();
    if (dev < 0) return DLF_E_UNSUPPORTED;
    if (!attr_set[dev]) {
        cudaError_t e = cudaSuccess;
        for (int v = 0; v < 4 && e == cudaSuccess; v++)
            e = cudaFuncSetAttribute(pick_kernel(1 + (v >> 1), (v & 1) != 0), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e);
        attr_set[dev] = true;
    }
    return DLF_OK;
}

int launch_mbconv_tc(const MbconvArgs& a, const MbconvTiling& t, int sm_count, int* status_dev, cudaStream_t s) {
    if (!t.ok) return DLF_E_PLAN;
    if (t.split > 0) return launch_mbconv_lat(a, t, sm_count, status_dev, s);
    if (!aligned(16, a.x, a.res, a.y)) return DLF_E_INVALID_ARG;
    int rc = mbconv_tc_init();
    if (rc) return rc;
    MbLayout L;
    if (!mbconv_supported(a) || !mb_layout(a, t.th, t.tw, &L)) return DLF_E_PLAN;
    MbParams p;
    std::memset(&p, 0, sizeof(p));
    p.N = a.N; p.H = a.H; p.W = a.W; p.hid = a.hid; p.Cout = a.Cout; p.stride = a.stride;
    p.Ho = (a.H + 2 - 3) / a.stride + 1; p.Wo = (a.W + 2 - 3) / a.stride + 1;
    p.has_expand = a.has_expand; p.act1 = a.act1; p.act2 = a.act2; p.act3 = a.act3;
    p.th = t.th; p.tw = t.tw; p.fh = L.fh; p.fw = L.fw; p.FR = L.FR; p.nb1 = L.nb1; p.nb2 = L.nb2;
    std::memcpy(p.strips, L.strips, sizeof(p.strips));
    std::memcpy(p.strip_len, L.strip_len, sizeof(p.strip_len));
    p.xbufs = L.xbufs; p.hbufs = L.hbufs; p.hdbufs = L.hdbufs; p.d1bufs = L.d1bufs; p.d2bufs = L.d2bufs;
    p.tiles_h = t.tiles_h; p.tiles_w = t.tiles_w; p.n_tiles = t.n_tiles;
    p.kin = L.kin; p.chunks = L.chunks; p.n2_pad = L.n2;
    p.ksteps_in_last = ((a.Cin - (p.kin - 1) * 64) + 15) / 16;
    p.x_off = L.x_off; p.h_off = L.h_off; p.h_bytes = L.h_bytes; p.hd_off = L.hd_off;
    p.ring_off = L.ring_off; p.stage_bytes = L.stage_bytes; p.stages = L.stages; p.bias_off = L.bias_off;
    p.so_off = L.so_off; p.so_planes = L.so_planes; p.xplane = L.xplane; p.so_plane = L.so_plane;
    p.d2_col = L.d2_col;
    p.w2_off = a.has_expand ? p.kin * 8192 : 0;
    p.n_split = p.n2_pad > 256 ? 2 : 1;
    p.n_each = p.n2_pad / p.n_split;
    p.wd = static_cast<const __half*>(a.wd); p.b1 = a.b1; p.bd = a.bd; p.b2 = a.b2;
    p.res = static_cast<const __half*>(a.res); p.out = static_cast<__half*>(a.y); p.status = status_dev;
    {
        const uint64_t dims[4] = {static_cast<uint64_t>(a.Cin), static_cast<uint64_t>(a.W), static_cast<uint64_t>(a.H), static_cast<uint64_t>(a.N)};
        const uint64_t strides[3] = {static_cast<uint64_t>(a.Cin) * 2, static_cast<uint64_t>(a.W) * a.Cin * 2,
                                     static_cast<uint64_t>(a.H) * a.W * a.Cin * 2};
        const uint32_t box[4] = {64, static_cast<uint32_t>(L.fw), static_cast<uint32_t>(L.fh), 1};
        const uint32_t es[4] = {1, 1, 1, 1};
        rc = encode_tmap(&p.tmx, a.x, 4, dims, strides, box, es);
        if (rc) return rc;
    }
    if (a.has_expand) {  // W1 [hid][C_in] seen as (C_in, hid, 1)
        const uint64_t dims[3] = {static_cast<uint64_t>(a.Cin), static_cast<uint64_t>(a.hid), 1};
        const uint64_t strides[2] = {static_cast<uint64_t>(a.Cin) * 2, static_cast<uint64_t>(a.hid) * a.Cin * 2};
        const uint32_t box[3] = {64, 64, 1};
        const uint32_t es[3] = {1, 1, 1};
        rc = encode_tmap(&p.tmw1, a.w1, 3, dims, strides, box, es);
        if (rc) return rc;
    }
    {  // W2 [C_out][hid] seen as (hid, C_out, 1)
        const uint64_t dims[3] = {static_cast<uint64_t>(a.hid), static_cast<uint64_t>(a.Cout), 1};
        const uint64_t strides[2] = {static_cast<uint64_t>(a.hid) * 2, static_cast<uint64_t>(a.Cout) * a.hid * 2};
        const uint32_t box[3] = {64, static_cast<uint32_t>(p.n_each), 1};
        const uint32_t es[3] = {1, 1, 1};
        rc = encode_tmap(&p.tmw2, a.w2, 3, dims, strides, box, es);
        if (rc) return rc;
    }
    if (p.so_planes > 0) {  // output (and residual) tile [C_out, Wo, Ho, N], one box per 64-channel plane
        const uint64_t dims[4] = {static_cast<uint64_t>(a.Cout), static_cast<uint64_t>(p.Wo), static_cast<uint64_t>(p.Ho), static_cast<uint64_t>(a.N)};
        const uint64_t strides[3] = {static_cast<uint64_t>(a.Cout) * 2, static_cast<uint64_t>(p.Wo) * a.Cout * 2,
                                     static_cast<uint64_t>(p.Ho) * p.Wo * a.Cout * 2};
        const uint32_t box[4] = {64, static_cast<uint32_t>(t.tw), static_cast<uint32_t>(t.th), 1};
        const uint32_t es[4] = {1, 1, 1, 1};
        rc = encode_tmap(&p.tmy, a.y, 4, dims, strides, box, es);
        if (rc) return rc;
        p.tmr = p.tmy;
        if (a.res) {
            rc = encode_tmap(&p.tmr, a.res, 4, dims, strides, box, es);
            if (rc) return rc;
        }
    }
    const int grid = std::max(1, std::min(sm_count, t.n_tiles));
    // (never two of these CTAs on an SM: each allocates all of tensor memory)
    const size_t smem = std::max<size_t>(L.smem, 120 * 1024);
    if (smem > static_cast<size_t>(kMaxSmem)) return DLF_E_PLAN;
    cudaError_t e = launch_kernel(pick_kernel(a.stride, p.act2 == DLF_ACT_RELU6 && (!p.has_expand || p.act1 == DLF_ACT_RELU6)), grid, kThreads, smem, s, p);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

}  // namespace dlf
