// Fused inverted-residual block (1x1 expansion -> depthwise 3x3 -> 1x1 projection, see mbconv_tc.cu) for maps whose tiles fit the chip
// at once: one tile per CTA, or per CLUSTER of 2, 4 or 8 CTAs that share the tile's hidden channels out, and nothing persistent.
// What bounds a block on few images is the chain of its hidden chunks, one after the other on each of few tiles, and every CTA's
// stream of all of its weights; a cluster divides both.
//
// The expansion is computed transposed, so that a hidden channel is a LANE of tensor memory and a thread, and the depthwise layer
// runs in registers: the hidden map is in no memory at all.  A unit is 8 x bh output pixels of one image, a tile up to eight units (at
// most 128 pixels).  Per chunk of (as a rule) 128 hidden channels:
//   1. expansion (tensor core): D1[128 channels x pixels of the units' input windows] = W1[chunk] * X^T, the windows (one pixel of
//      halo) TMA-loaded once;
//   2. a warp takes the 32 channels of its lane quarter for some rows of a unit: it walks down the window row by row - tensor-memory
//      load of a row (10 or 17 pixels), bias, activation, fp16 rounding, zero outside the image - and every input value joins the
//      output rows it touches (fma.rn.f32.f16, weights in registers); a finished row of eight outputs (bias, activation, rounding) is
//      one 16-byte store into Hd[channel][pixel];
//   3. projection (tensor core): D2[pixels x C_out] += Hd^T * W2[:, chunk]^T (operand A lies pixels-contiguous), fp32 in tensor memory.
// At the end every CTA of the cluster has a partial D2: each warp sends the rows it drains straight into the shared memory of the CTA
// that finishes them (st.async, counted by that CTA's barrier; conv_lat.cu), which adds them up in the order of the ranks, then bias,
// residual, activation, rounding.  Every intermediate is rounded to fp16 where the layer-by-layer execution rounds it.
//
// Against mbconv_tc.cu's kernel: 64 -> 384 -> 64 channels at 14x14 12.7 -> 6.5 us at one image (three kernels 10.4), 18.4 -> 12.8 at 64;
// 96 -> 576 -> 96 there at 64 24.7 -> 18.8; 160 -> 960 -> 160 at 7x7, one image 23.0 -> 7.1 (three kernels 11.1); 32 -> 192 -> 32 at 28x28,
// one image 10.1 -> 6.6, eight 10.8 -> 8.1; MobileNetV2 b1 166 -> 113 us, b64 554 -> 513.
// Measured bounds: a row of eight outputs takes a scheduler about 205 clocks (72 multiply-adds with fp16 factors, 2 clocks each; rounding,
// clamps and unpacking, half rate, on the other pipe); a control warp's step between two chunks 500-1000.
// With many tiles per CTA the kernel of mbconv_tc.cu is the faster one (24 -> 144 -> 24 at 56x56, 64 images 64.8 us against 68 of a
// persistent form of this one): here a task's fixed part - weights, addresses, waits, about 2000 clocks - is a few rows' time.
//
// Work is handed round in order: every depthwise warp passes every job (chunk, units of one accumulator) and every chunk, waits for
// those it does not work on as well and counts as a reader of them, so that no barrier phase can overtake a warp.
//
// Warps: 0-15 depthwise and epilogue, 16 expansions, 17 projections and their weights, 18 input windows, 19 expansion weights.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "internal.h"
#include "ptx.cuh"

namespace dlf {

namespace {

constexpr int kDwWarps = 16;
constexpr int kExpWarp = kDwWarps;
constexpr int kProjWarp = kExpWarp + 1;
constexpr int kInWarp = kExpWarp + 2;
constexpr int kW1Warp = kExpWarp + 3;
constexpr int kThreads = 32 * (kExpWarp + 4);
constexpr int kMaxSmem = 232448 - 2048;    // the 227 KB per-CTA limit minus the static barriers
constexpr int kUnitW = 8;                  // output columns of a unit: one 16-byte vector of Hd
constexpr int kMaxUnits = 8;               // units of a tile
constexpr int kMaxSlots = 8;               // D1 accumulators
constexpr int kMaxStages = 4;

struct LatBlockParams {
    CUtensorMap tmx, tmw1, tmw2;        // input window, the two weight slabs
    int H, W, hid, Cout, Ho, Wo;
    int act1, act2, act3;
    int bh, U, fpx, npx;                // rows of a unit, units of a tile, pixels of a unit's input window and the same rounded up to 16
    int UG, parts, part_rows;           // units of a job (one accumulator); a unit's rows are walked in parts, a warp each
    int units_x, units_y, n_units;
    int kin, ksteps_in_last;            // 64-channel planes of the input, UMMAs of the last one
    int chunks, cg;                     // hidden chunks, each of up to cg groups of 32 channels
    int n2_pad, n_split, n_each;        // C_out rounded up to 16; above 256 it is issued as two halves
    int hdbufs, w1_stages, w2_stages, slots;
    int xplane;                         // bytes of one 64-channel plane of a window (plane by plane, a plane's windows side by side)
    int hd_off, hd_bytes, w1_off, w1_bytes, w2_off, w2_bytes, bias_off;   // shared memory (the windows come first)
    int d2_col;                         // first TMEM column of the projection's accumulator
    int rows_per, red_off;              // clusters: pixels a CTA finishes, byte offset of the ranks' partial sums of them
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

// A row of a unit's window from tensor memory: 10 (stride 1) or 17 consecutive columns of the thread's lane.
template <int NX>
__device__ __forceinline__ void ld_row_issue(uint32_t taddr, uint32_t (&r)[NX]) {
    if (NX == 10) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[8]), "=r"(r[9]) : "r"(taddr + 8u) : "memory");
    } else {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8 % NX]), "=r"(r[9 % NX]),
              "=r"(r[10 % NX]), "=r"(r[11 % NX]), "=r"(r[12 % NX]), "=r"(r[13 % NX]), "=r"(r[14 % NX]), "=r"(r[15 % NX])
            : "r"(taddr) : "memory");
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[16 % NX]) : "r"(taddr + 16u) : "memory");
    }
}
template <int NX>
__device__ __forceinline__ void ld_row_wait(uint32_t (&r)[NX]) {
    if (NX == 10)
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]));
    else
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8 % NX]), "+r"(r[9 % NX]),
                       "+r"(r[10 % NX]), "+r"(r[11 % NX]), "+r"(r[12 % NX]), "+r"(r[13 % NX]), "+r"(r[14 % NX]), "+r"(r[15 % NX]), "+r"(r[16 % NX]));
}

// One warp's depthwise work: 32 channels of some rows of one unit.
struct DwTask {
    uint32_t src;       // tensor-memory address of the window's first pixel
    int y0, x0;         // image position of the window's first pixel
    int rows;           // output rows
    bool live;          // this lane's channel exists
    uint32_t dst;       // shared-memory address of this channel's pixels in Hd (first 64-pixel block)
    int v0;             // first 8-pixel vector of the unit in the tile
    uint32_t lbo;       // bytes from one 64-pixel block to the next: the chunk's 32-channel groups, 4096 each
    uint32_t k7;        // the channel's row within a swizzle atom
};
template <int STRIDE, bool RELU6>
__device__ __forceinline__ void depthwise_task(const LatBlockParams& p, const DwTask& t, const unsigned short (&w)[9], float b1, float bd) {
    constexpr int NX = 7 * STRIDE + 3, NP = (NX + 1) / 2;
    const __half2 lo1 = act_lo(p.act1), hi1 = act_hi(p.act1), lo2 = act_lo(p.act2), hi2 = act_hi(p.act2);
    const int in_rows = (t.rows - 1) * STRIDE + 3;
    uint32_t src = t.src;
    // windows that reach past the image: hidden values there are the depthwise layer's padding
    const bool edge = (t.y0 < 0 || t.x0 < 0 || t.y0 + in_rows > p.H || t.x0 + NX > p.W);
    uint32_t mask[NP] = {};
    if (edge) {
#pragma unroll
        for (int i = 0; i < NP; i++) {
            const bool a = static_cast<unsigned>(t.x0 + 2 * i) < static_cast<unsigned>(p.W), b = static_cast<unsigned>(t.x0 + 2 * i + 1) < static_cast<unsigned>(p.W);
            mask[i] = (a ? 0xffffu : 0u) | (b ? 0xffff0000u : 0u);
        }
    }
    uint64_t b1b1;
    asm("mov.b64 %0, {%1, %1};" : "=l"(b1b1) : "f"(b1));
    unsigned short x[NX];
    uint32_t raw[NX];
    int iy = t.y0, left = in_rows;
    // A row is used once it has landed (wait()); the one behind it is on its way while it is worked on, but over no branch and from no trip
    // of a loop to the next: until the wait its registers hold nothing that may be copied.
    auto wait = [&]() { ld_row_wait<NX>(raw); };
    ld_row_issue<NX>(src, raw);
    wait();
    auto next = [&]() {
        const uint32_t row_in = static_cast<unsigned>(iy) < static_cast<unsigned>(p.H) ? 0xffffffffu : 0u;
        uint32_t h[NP];
#pragma unroll
        for (int i = 0; i < NP; i++) {
            const float2 f = add_f2(raw[2 * i], 2 * i + 1 < NX ? raw[(2 * i + 1) % NX] : 0u, b1b1);
            h[i] = round_clamp<RELU6>(f.x, f.y, lo1, hi1);
        }
        if (edge) {
#pragma unroll
            for (int i = 0; i < NP; i++) h[i] &= mask[i] & row_in;
        }
#pragma unroll
        for (int i = 0; i < NP; i++) {
            unsigned short a, b;
            unpack_h2(h[i], a, b);
            x[2 * i] = a;
            if (2 * i + 1 < NX) x[(2 * i + 1) % NX] = b;
        }
        if (--left > 0) src += NX;   // (behind the last row that one once more: a load in one branch alone would have to be merged with what `raw` holds in the other)
        ld_row_issue<NX>(src, raw);
        iy++;
    };
    auto add = [&](float (&acc)[kUnitW], int r) {
#pragma unroll
        for (int s = 0; s < 3; s++)
#pragma unroll
            for (int o = 0; o < kUnitW; o++) acc[o] = fma_f32_f16(x[o * STRIDE + s], w[r * 3 + s], acc[o]);
    };
    auto start = [&](float (&acc)[kUnitW]) {
#pragma unroll
        for (int o = 0; o < kUnitW; o++) acc[o] = bd;
        add(acc, 0);
    };
    int v = t.v0;
    const uint32_t live = t.live;
    auto store = [&](const float (&acc)[kUnitW]) {
        uint4 o;
        o.x = round_clamp<RELU6>(acc[0], acc[1], lo2, hi2);
        o.y = round_clamp<RELU6>(acc[2], acc[3], lo2, hi2);
        o.z = round_clamp<RELU6>(acc[4], acc[5], lo2, hi2);
        o.w = round_clamp<RELU6>(acc[6], acc[7], lo2, hi2);
        const uint32_t at = t.dst + ((v & 8) ? t.lbo : 0u) + (((static_cast<uint32_t>(v) & 7u) ^ t.k7) << 4);
        asm volatile("{\n .reg .pred live;\n setp.ne.u32 live, %5, 0;\n @live st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n}"
                     ::"r"(at), "r"(o.x), "r"(o.y), "r"(o.z), "r"(o.w), "r"(live) : "memory");
        v++;
    };
    const int rows = t.rows;
    float a[kUnitW], b[kUnitW];
    if (STRIDE == 1) {
        // input row j is the last row of output j - 2, the middle one of output j - 1, the first one of output j
        float c[kUnitW];
        next(); start(a); wait();
        next(); add(a, 1); start(b); wait();
        int j = 0;
#pragma unroll 1
        while (true) {
            next(); add(a, 2); store(a); wait();
            if (++j == rows) break;
            add(b, 1); start(c);
            next(); add(b, 2); store(b); wait();
            if (++j == rows) break;
            add(c, 1); start(a);
            next(); add(c, 2); store(c); wait();
            if (++j == rows) break;
            add(a, 1); start(b);
        }
    } else {
        next(); start(a); wait();
#pragma unroll 1
        for (int j = 0;;) {
            next(); add(a, 1); wait();
            next(); add(a, 2); store(a); wait();
            if (++j == rows) break;
            start(a);
        }
    }
}

// SPLIT: CTAs of the cluster.  RELU6: both the expansion's and the depthwise layer's activation.
template <int STRIDE, bool RELU6, int SPLIT>
__global__ void __cluster_dims__(SPLIT, 1, 1) __launch_bounds__(kThreads, 1) mbconv_lat_kernel(const __grid_constant__ LatBlockParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t x_full[kMaxUnits], w1_full[kMaxStages], w1_empty[kMaxStages], w2_full[kMaxStages], w2_empty[kMaxStages];
    __shared__ uint64_t d1_full[kMaxSlots], d1_free[kMaxSlots], hd_ready[4], hd_free[4], d2_full, red_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, red_abort_s;

    const int rank = SPLIT > 1 ? static_cast<int>(cluster_rank()) : 0;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sb = smem_raw + (base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &abort_s;
    float* b2s = reinterpret_cast<float*>(sb + p.bias_off);
    const int code0 = blockIdx.x << 12, tile = static_cast<int>(blockIdx.x) / SPLIT;

    if (warp == kProjWarp) {   // barriers, one or two to a lane
        if (lane < kMaxUnits) {
            mbar_init(&x_full[lane], 1);
            mbar_init(&d1_full[lane], 1);
            mbar_init(&d1_free[lane], kDwWarps);
        } else if (lane < 12) {
            mbar_init(&w1_full[lane - 8], 1);
            mbar_init(&w1_empty[lane - 8], 1);
            mbar_init(&w2_full[lane - 8], 1);
            mbar_init(&w2_empty[lane - 8], 1);
        } else if (lane < 16) {
            mbar_init(&hd_ready[lane - 12], kDwWarps);
            mbar_init(&hd_free[lane - 12], 1);
        } else if (lane == 16) {
            mbar_init(&d2_full, 1);
        } else if (lane == 20) {
            mbar_init(&red_bar, 1);
            abort_s = 0;
            red_abort_s = 0;
        }
        fence_barrier_init();
        // the bytes that the cluster's CTAs will send here (before the cluster's barrier, which every sender waits for)
        if (SPLIT > 1 && lane == 20) mbar_expect_tx(&red_bar, static_cast<uint32_t>(SPLIT * max(0, min(p.rows_per, p.U * kUnitW * p.bh - rank * p.rows_per)) * p.n2_pad) * 4u);
    }
    if (warp == kInWarp && lane == 0) {
        tma_prefetch_desc(&p.tmx);
        tma_prefetch_desc(&p.tmw1);
        tma_prefetch_desc(&p.tmw2);
    }
    if (warp == kExpWarp) {
        tmem_alloc(&tmem_base_s, 512);
        tmem_relinquish();
    }
    for (int i = threadIdx.x; i < p.n2_pad; i += kThreads) b2s[i] = i < p.Cout ? __ldg(p.b2 + i) : 0.0f;
    tc_fence_before_sync();
    __syncthreads();
    if (SPLIT > 1) cluster_arrive();   // all CTAs of the cluster run (waited for before sums go to the others)
    tc_fence_after_sync();
    pdl_launch_dependents();
    const uint32_t tmem_base = tmem_base_s;
    // position of a unit
    struct Unit { int n, oy, ox; };
    auto unit_of = [&](int id) {
        Unit u;
        const int r = id / p.units_x;
        u.ox = (id - r * p.units_x) * kUnitW;
        u.n = r / p.units_y;
        u.oy = (r - u.n * p.units_y) * p.bh;
        return u;
    };

    if (warp < kDwWarps) {
        // ---- depthwise layer --------------------------------------------------------------------------------------------
        const int q = warp & 3, set = warp >> 2, px = kUnitW * p.bh, pixels = p.U * px;
        {
            int slot = 0, hb = 0;
            uint32_t slot_ph = 0, hb_ph = 1, cc = 0, turn = 0;   // ring positions and phases; chunks so far; this quarter's tasks so far
            bool ok = true;
            const Unit mine = unit_of(tile * p.U + min(lane, p.U - 1));   // lane u holds unit u's position
            for (int c = rank; c < p.chunks && ok; c += SPLIT, cc++) {
                const int ch0 = c * 32 * p.cg, groups = min(p.cg, (p.hid - ch0 + 31) >> 5);
                unsigned short w[9] = {};   // (a quarter works on one group of the chunk)
                float b1 = 0.0f, bd = 0.0f;
                if (q < groups) {
                    const int ch = min(ch0 + q * 32 + lane, p.hid - 1);
                    const unsigned short* wp = reinterpret_cast<const unsigned short*>(p.wd) + static_cast<long long>(ch) * 9;
#pragma unroll
                    for (int i = 0; i < 9; i++) w[i] = __ldg(wp + i);
                    b1 = __ldg(p.b1 + ch);
                    bd = __ldg(p.bd + ch);
                }
                if (cc >= static_cast<uint32_t>(p.hdbufs)) ok = mbar_wait_warp<true>(&hd_free[hb], hb_ph, abort_flag, p.status, 0xE20 | code0);
                for (int u0 = 0; u0 < p.U && ok; u0 += p.UG) {
                    ok = mbar_wait_warp<true>(&d1_full[slot], slot_ph, abort_flag, p.status, 0xE10 | code0);
                    if (!ok) break;
                    if (q < groups) {
                        tc_fence_after_sync();
                        for (int u = u0; u < u0 + p.UG; u++)
                            for (int part = 0; part < p.parts; part++) {
                                if ((turn++ & 3u) != static_cast<uint32_t>(set)) continue;
                                const int kc = q * 32 + lane, r0 = part * p.part_rows;
                                DwTask k;
                                k.rows = min(p.part_rows, p.bh - r0);
                                k.y0 = (__shfl_sync(0xffffffffu, mine.oy, u) + r0) * STRIDE - 1;
                                k.x0 = __shfl_sync(0xffffffffu, mine.ox, u) * STRIDE - 1;
                                k.v0 = u * p.bh + r0;
                                k.live = ch0 + kc < p.hid;
                                k.lbo = static_cast<uint32_t>(groups) * 4096u;
                                k.k7 = static_cast<uint32_t>(kc) & 7u;
                                k.dst = base + p.hd_off + hb * p.hd_bytes + kc * 128;
                                k.src = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + (slot * p.UG + u - u0) * p.npx + static_cast<uint32_t>(r0 * STRIDE * (7 * STRIDE + 3));
                                depthwise_task<STRIDE, RELU6>(p, k, w, b1, bd);
                            }
                        tc_fence_before_sync();
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&d1_free[slot]);
                    if (++slot == p.slots) { slot = 0; slot_ph ^= 1u; }
                }
                fence_proxy_async_smem();   // the projection's UMMAs read Hd through the async proxy
                __syncwarp();
                if (lane == 0 && ok) mbar_arrive(&hd_ready[hb]);
                if (++hb == p.hdbufs) { hb = 0; hb_ph ^= 1u; }
            }
        }
        // ---- epilogue: a warp drains its lane quarter's pixels, 16 columns at a time -----------------------------------------------
        const int m = q * 32 + lane;
        const __half2 lo3 = act_lo(p.act3), hi3 = act_hi(p.act3);
        // where a pixel of the tile goes; negative: nowhere
        auto pixel_at = [&](int mo) {
            const int mu = mo / px, mp = mo - mu * px, id = tile * p.U + mu;
            if (mo >= pixels || id >= p.n_units) return -1ll;
            const Unit u = unit_of(id);
            const int gy = u.oy + (mp >> 3), gx = u.ox + (mp & 7);
            if (gy >= p.Ho || gx >= p.Wo) return -1ll;
            return ((static_cast<long long>(u.n) * p.Ho + gy) * p.Wo + gx) * p.Cout;
        };
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + p.d2_col;
        pdl_wait();   // (the residual)
        if (SPLIT == 1) {
            const long long at = pixel_at(m);
            const bool ok = mbar_wait_warp<true>(&d2_full, 0u, abort_flag, p.status, 0xE30 | code0);
            tc_fence_after_sync();
#pragma unroll 1
            for (int c0 = set * 16; c0 < p.n2_pad; c0 += 64) {
                uint32_t v[16];
                tmem_ld16_issue(taddr + c0, v);
                tmem_ld16_wait(v);
#pragma unroll
                for (int g = 0; g < 2; g++) {
                    const int co = c0 + g * 8;
                    if (at < 0 || !ok || co >= p.Cout) break;
                    uint4 rv = make_uint4(0u, 0u, 0u, 0u);
                    if (p.res) rv = ld_map(reinterpret_cast<const uint4*>(p.res + at + co));
                    float a[8];
#pragma unroll
                    for (int e = 0; e < 8; e++) a[e] = __uint_as_float(v[g * 8 + e]);
                    *reinterpret_cast<uint4*>(p.out + at + co) = finish8(a, b2s + co, rv, lo3, hi3);
                }
                __syncwarp();   // (the next load is the whole warp's)
            }
        } else {
            const uint32_t swz = p.n2_pad % 32 == 0 ? 7u : 3u;   // (a row's 16-byte vectors in an order that depends on the row: other banks)
            bool ok = mbar_wait_warp<true>(&d2_full, 0u, abort_flag, p.status, 0xE30 | code0);
            tc_fence_after_sync();
            cluster_wait();   // every CTA of the cluster runs and its barrier expects these rows
            const int dest = min(m / p.rows_per, SPLIT - 1), row = m - dest * p.rows_per;
            const uint32_t slab = static_cast<uint32_t>(p.rows_per * p.n2_pad * 4);   // one rank's partial rows
            const uint32_t dst = mapa(base + p.red_off + rank * slab + row * p.n2_pad * 4, dest), dst_bar = mapa(smem_u32(&red_bar), dest);
#pragma unroll 1
            for (int c0 = set * 16; c0 < p.n2_pad; c0 += 64) {
                uint32_t v[16];
                tmem_ld16_issue(taddr + c0, v);
                tmem_ld16_wait(v);
                if (m < pixels) {   // (sent whatever happened: the other CTAs wait for the bytes)
#pragma unroll
                    for (int e = 0; e < 4; e++)
                        st_async_v4(dst + ((static_cast<uint32_t>((c0 >> 2) + e) ^ (static_cast<uint32_t>(row) & swz)) << 4), __uint_as_float(v[4 * e]),
                                    __uint_as_float(v[4 * e + 1]), __uint_as_float(v[4 * e + 2]), __uint_as_float(v[4 * e + 3]), dst_bar);
                }
                __syncwarp();
            }
            // All rows of this CTA are here.  It must not retire before that, whatever its own part came to, hence a limit above the senders'
            // and a flag of its own.
            ok = mbar_wait<true>(&red_bar, 0u, &red_abort_s, p.status, 0xE50 | code0, 4 * kWaitLimitNs) && ok;
            const int mine = max(0, min(p.rows_per, pixels - rank * p.rows_per)), bn8 = p.n2_pad >> 3;
            const uint8_t* red = sb + p.red_off;
            for (int i = threadIdx.x; i < mine * bn8 && ok; i += 32 * kDwWarps) {
                const int r = i / bn8, g = i - r * bn8, co = g * 8;
                const long long at = pixel_at(rank * p.rows_per + r);
                if (at < 0 || co >= p.Cout) continue;
                uint4 rv = make_uint4(0u, 0u, 0u, 0u);
                if (p.res) rv = ld_map(reinterpret_cast<const uint4*>(p.res + at + co));
                const uint32_t src = static_cast<uint32_t>(r * p.n2_pad * 4) + ((static_cast<uint32_t>(2 * g) ^ (static_cast<uint32_t>(r) & swz)) << 4);
                float4 a = *reinterpret_cast<const float4*>(red + src), b = *reinterpret_cast<const float4*>(red + (src ^ 16u));
#pragma unroll
                for (int sp = 1; sp < SPLIT; sp++) {
                    const float4 a2 = *reinterpret_cast<const float4*>(red + sp * slab + src), b2 = *reinterpret_cast<const float4*>(red + sp * slab + (src ^ 16u));
                    a.x += a2.x; a.y += a2.y; a.z += a2.z; a.w += a2.w;
                    b.x += b2.x; b.y += b2.y; b.z += b2.z; b.w += b2.w;
                }
                const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                *reinterpret_cast<uint4*>(p.out + at + co) = finish8(v, b2s + co, rv, lo3, hi3);
            }
        }
    } else if (warp == kInWarp) {
        // ---- input windows: lane u loads unit u's, one box per 64-channel plane -------------------------------------------
        pdl_wait();
        if (lane < p.U) {
            const int id = tile * p.U + lane;
            if (id < p.n_units) {
                const Unit u = unit_of(id);
                mbar_expect_tx(&x_full[lane], static_cast<uint32_t>(p.kin) * p.fpx * 128u);
                for (int pl = 0; pl < p.kin; pl++)
                    tma_load_4d(sb + (pl * p.U + lane) * p.xplane, &p.tmx, &x_full[lane], pl * 64, u.ox * STRIDE - 1, u.oy * STRIDE - 1, u.n);
            } else {
                mbar_arrive(&x_full[lane]);   // (past the last unit: whatever lies there is worked on and not stored)
            }
        }
        __syncwarp();
    } else if (warp == kW1Warp) {
        // ---- the expansion's weights: per chunk a slab of boxes of 32 hidden channels x 64 inputs, a lane per box.  Constants: no wait
        //      for the previous kernel -----------------------------------------------------------------------------------------
        int s1 = 0;
        uint32_t ph1 = 1;
        for (int c = rank; c < p.chunks; c += SPLIT) {
            const int ch0 = c * 32 * p.cg, groups = min(p.cg, (p.hid - ch0 + 31) >> 5);
            if (!mbar_wait_warp(&w1_empty[s1], ph1, abort_flag, p.status, 0xC00 | code0)) break;
            if (lane == 0) mbar_expect_tx(&w1_full[s1], static_cast<uint32_t>(p.kin * groups) * 4096u);
            __syncwarp();
            if (lane < p.kin * groups) {
                const int pl = lane / groups, g = lane - pl * groups;
                tma_load_3d(sb + p.w1_off + s1 * p.w1_bytes + pl * 16384 + g * 4096, &p.tmw1, &w1_full[s1], pl * 64, ch0 + g * 32, 0);
            }
            __syncwarp();
            if (++s1 == p.w1_stages) { s1 = 0; ph1 ^= 1u; }
        }
    } else if (warp == kExpWarp) {
        // ---- expansions: D1 = W1[chunk] * X^T, as soon as an accumulator is free.  The whole warp walks the loops (warp-uniform
        //      descriptors), one elected lane issues --------------------------------------------------------------------------
        const uint32_t idesc1 = umma_idesc_f16(p.UG * p.npx), xplane16 = static_cast<uint32_t>(p.U * p.xplane) >> 4;
        int s1 = 0, slot = 0;
        uint32_t ph1 = 0, slot_ph = 1;
        bool ok = true;
        for (int c = rank; c < p.chunks && ok; c += SPLIT) {
            ok = mbar_wait_warp<true>(&w1_full[s1], ph1, abort_flag, p.status, 0xD10 | code0);
            const uint32_t a0 = umma_desc_lo(base + p.w1_off + s1 * p.w1_bytes);
            for (int u = 0; u < p.U && ok; u += p.UG) {
                if (c == rank)
                    for (int v = u; v < u + p.UG && ok; v++) ok = mbar_wait_warp<true>(&x_full[v], 0u, abort_flag, p.status, 0xD00 | code0);
                if (ok) ok = mbar_wait_warp<true>(&d1_free[slot], slot_ph, abort_flag, p.status, 0xD20 | code0);
                if (!ok) break;
                tc_fence_after_sync();
                uint32_t a_lo = a0, b_lo = umma_desc_lo(base + u * p.xplane);
                const uint32_t d = tmem_base + slot * p.UG * p.npx;
                if (elect_one()) {
                    for (int pl = 0; pl < p.kin; pl++, a_lo += 1024u, b_lo += xplane16) {
                        const int ks = pl < p.kin - 1 ? 4 : p.ksteps_in_last;
                        if (ks == 4) umma_f16_steps<4>(d, a_lo, b_lo, idesc1, pl != 0);
                        else if (ks == 3) umma_f16_steps<3>(d, a_lo, b_lo, idesc1, pl != 0);
                        else if (ks == 2) umma_f16_steps<2>(d, a_lo, b_lo, idesc1, pl != 0);
                        else umma_f16_steps<1>(d, a_lo, b_lo, idesc1, pl != 0);
                    }
                    umma_commit(&d1_full[slot]);
                    if (u + p.UG >= p.U) umma_commit(&w1_empty[s1]);
                }
                __syncwarp();
                if (++slot == p.slots) { slot = 0; slot_ph ^= 1u; }
            }
            if (++s1 == p.w1_stages) { s1 = 0; ph1 ^= 1u; }
        }
    } else {
        // ---- projections: D2 += Hd^T * W2[:, chunk]^T once all of the chunk's pixels are in shared memory; and their weights, planes of
        //      64 hidden channels, loaded one chunk after their stage's last use was issued --------------------------------------------
        const uint32_t idesc2 = umma_idesc_f16(p.n_each) | kIdescAmn;
        int s2 = 0, hb = 0;
        uint32_t ph2 = 0, hb_ph = 0;
        bool ok = true;
        int wc = rank, ws = 0;   // chunk and stage of the next load
        uint32_t ws_ph = 1;
        auto load_w2 = [&]() {
            if (wc >= p.chunks) return true;
            const int ch0 = wc * 32 * p.cg, planes = (min(p.cg, (p.hid - ch0 + 31) >> 5) + 1) >> 1;
            if (!mbar_wait_warp(&w2_empty[ws], ws_ph, abort_flag, p.status, 0xC10 | code0)) return false;
            if (lane == 0) mbar_expect_tx(&w2_full[ws], static_cast<uint32_t>(planes * p.n2_pad) * 128u);
            __syncwarp();
            if (lane < planes * p.n_split) {
                const int pl = lane / p.n_split, j = lane - pl * p.n_split;
                tma_load_3d(sb + p.w2_off + ws * p.w2_bytes + (pl * p.n2_pad + j * p.n_each) * 128, &p.tmw2, &w2_full[ws], ch0 + pl * 64, j * p.n_each, 0);
            }
            __syncwarp();
            if (++ws == p.w2_stages) { ws = 0; ws_ph ^= 1u; }
            wc += SPLIT;
            return true;
        };
        for (int i = 0; i < p.w2_stages && ok; i++) ok = load_w2();
        for (int c = rank; c < p.chunks && ok; c += SPLIT) {
            const int ksteps = min(2 * p.cg, (p.hid - c * 32 * p.cg) >> 4);
            ok = mbar_wait_warp<true>(&w2_full[s2], ph2, abort_flag, p.status, 0xD50 | code0);
            if (ok) ok = mbar_wait_warp<true>(&hd_ready[hb], hb_ph, abort_flag, p.status, 0xD60 | code0);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t a0 = umma_desc_mn_lo(base + p.hd_off + hb * p.hd_bytes, ((ksteps + 1) >> 1) * 4096), b0 = umma_desc_lo(base + p.w2_off + s2 * p.w2_bytes);
            const uint32_t plane16 = static_cast<uint32_t>(p.n2_pad) * 8u;
            if (elect_one()) {
                for (int j = 0; j < p.n_split; j++) {
                    const uint32_t d = tmem_base + p.d2_col + j * p.n_each, bj = b0 + static_cast<uint32_t>(j * p.n_each) * 8u;
                    // 16 channels a step: two atoms of eight, 2048 bytes (channels past the hidden width are not read)
                    for (int k0 = 0; k0 < ksteps; k0 += 4) {
                        const uint32_t ak = a0 + k0 * 128u, bk = bj + (k0 >> 2) * plane16, acc = c != rank || k0 != 0;
                        const int n = min(4, ksteps - k0);
                        if (n == 4) umma_f16_mn_steps<4>(d, ak, bk, idesc2, acc);
                        else if (n == 3) umma_f16_mn_steps<3>(d, ak, bk, idesc2, acc);
                        else if (n == 2) umma_f16_mn_steps<2>(d, ak, bk, idesc2, acc);
                        else umma_f16_mn_steps<1>(d, ak, bk, idesc2, acc);
                    }
                }
                umma_commit(&hd_free[hb]);
                umma_commit(&w2_empty[s2]);
                if (c + SPLIT >= p.chunks) umma_commit(&d2_full);
            }
            __syncwarp();
            // (the stage of the chunk before this one, whose UMMAs have long run by the time this one's are issued; of a ring of one
            // stage, this one's)
            if (p.w2_stages == 1 || c != rank) ok = load_w2();
            if (++s2 == p.w2_stages) { s2 = 0; ph2 ^= 1u; }
            if (++hb == p.hdbufs) { hb = 0; hb_ph ^= 1u; }
        }
    }
    __syncwarp();
    if (SPLIT > 1 && warp >= kDwWarps) cluster_wait();

    tc_fence_before_sync();
    __syncthreads();
    if (warp == kExpWarp) {
        if (abort_s) __nanosleep(20000);
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

typedef void (*KernelFn)(const LatBlockParams);
template <int STRIDE, bool RELU6>
KernelFn pick_split(int split) {
    switch (split) {
        case 1: return mbconv_lat_kernel<STRIDE, RELU6, 1>;
        case 2: return mbconv_lat_kernel<STRIDE, RELU6, 2>;
        case 4: return mbconv_lat_kernel<STRIDE, RELU6, 4>;
        default: return mbconv_lat_kernel<STRIDE, RELU6, 8>;
    }
}
KernelFn pick_kernel(int stride, bool relu6, int split) {
    if (stride == 1) return relu6 ? pick_split<1, true>(split) : pick_split<1, false>(split);
    return relu6 ? pick_split<2, true>(split) : pick_split<2, false>(split);
}

int pad16(int c) { return (c + 15) / 16 * 16; }

// Shared-memory and tensor-memory layout of a choice of units; false if it does not fit.
struct LatLayout {
    int fh, fw, fpx, npx, part_rows, units_x, units_y, n_units, n_tiles;
    int kin, chunks, cg, n2, per_cta;
    int hdbufs, w1_stages, w2_stages, slots, d2_col;
    int xplane, hd_off, hd_bytes, w1_off, w1_bytes, w2_off, w2_bytes, bias_off, rows_per, red_off;
    size_t smem;
};

bool lat_layout(const MbconvArgs& a, int bh, int U, int UG, int parts, int split, int sm_count, LatLayout* L) {
    const int s = a.stride, Ho = (a.H + 2 - 3) / s + 1, Wo = (a.W + 2 - 3) / s + 1;
    L->fh = (bh - 1) * s + 3; L->fw = (kUnitW - 1) * s + 3;
    L->fpx = L->fh * L->fw;
    L->npx = pad16(L->fpx);
    const int pixels = U * bh * kUnitW, job_cols = UG * L->npx;
    if (job_cols > 256 || U > kMaxUnits || U % UG || pixels > 128) return false;
    L->part_rows = (bh + parts - 1) / parts;
    if ((bh + L->part_rows - 1) / L->part_rows != parts) return false;
    L->units_x = (Wo + kUnitW - 1) / kUnitW; L->units_y = (Ho + bh - 1) / bh;
    const long long n_units = static_cast<long long>(a.N) * L->units_x * L->units_y;
    if (n_units > 128ll * sm_count) return false;
    L->n_units = static_cast<int>(n_units); L->n_tiles = (L->n_units + U - 1) / U;
    // one wave; clusters of four find whole places on about 16 of a GPC's 18 SMs, of eight on 14 (7x7, 8 images: 16 clusters 17 us, 14
    // 11)
    if (L->n_tiles * split > (split > 2 ? sm_count / 18 * (split > 4 ? 14 : 16) : sm_count)) return false;
    L->kin = (a.Cin + 63) / 64; L->n2 = pad16(a.Cout);
    L->slots = std::min(kMaxSlots, (512 - L->n2) / job_cols);
    if (L->slots < 1) return false;
    L->d2_col = L->slots * job_cols;
    L->xplane = L->npx * 128;
    L->rows_per = (pixels + split - 1) / split;
    // by preference: three stages of weights, two, chunks of 64 channels instead of 128, one buffer of each
    struct Variant { int hdbufs, w1, w2, cg; };
    static const Variant kVariants[] = {{2, 3, 3, 4}, {2, 2, 2, 4}, {1, 2, 2, 4}, {1, 2, 1, 4}, {2, 2, 2, 2}, {1, 2, 2, 2}, {1, 1, 1, 2}};
    for (const Variant& v : kVariants) {
        L->cg = v.cg;
        L->chunks = (a.hid + 32 * v.cg - 1) / (32 * v.cg);
        while (L->chunks < split && L->cg > 1) {   // a chunk per CTA of the cluster at least
            L->cg--;
            L->chunks = (a.hid + 32 * L->cg - 1) / (32 * L->cg);
        }
        if (L->chunks < split) return false;
        L->per_cta = (L->chunks + split - 1) / split;
        L->hdbufs = std::min(v.hdbufs, L->per_cta);
        L->w1_stages = std::min(v.w1, L->per_cta);
        L->w2_stages = std::min(v.w2, L->per_cta);
        L->hd_bytes = L->cg * 8192;
        L->w1_bytes = L->kin * 16384;
        L->w2_bytes = L->n2 * 128 * ((L->cg + 1) / 2);
        L->hd_off = U * L->kin * L->xplane;
        L->w1_off = L->hd_off + L->hdbufs * L->hd_bytes;
        L->w2_off = L->w1_off + L->w1_stages * L->w1_bytes;
        L->red_off = L->w2_off + L->w2_stages * L->w2_bytes;
        L->bias_off = L->red_off + (split > 1 ? split * L->rows_per * L->n2 * 4 : 0);
        L->smem = static_cast<size_t>(L->bias_off) + L->n2 * 4 + 1024;
        if (L->smem <= static_cast<size_t>(kMaxSmem)) return true;
    }
    return false;
}

// What one choice of units and clusters takes against another one of the same block, in SM clocks: least squares over 6000 measured choices
// of nine MobileNetV2 blocks at 1 to 64 images (the choices made by it take 535 us in all over 46 cases, the best ones 526).  A round is
// what a lane quarter's four warps do side by side, a job what one accumulator takes to be issued and handed over; a cluster's exchange of
// sums takes 1.5 us, less the smaller a CTA's share of them.
double lat_rank(const MbconvArgs& a, const LatLayout& L, int bh, int U, int UG, int parts, int split, int sm_count) {
    const int tasks = U * parts, rounds = L.per_cta * ((tasks + 3) / 4), jobs = L.per_cta * (U / UG), side = std::min(4, tasks);
    const double in_rows = (L.part_rows - 1) * a.stride + 3;
    const double load = (0.4 * L.per_cta * L.cg * 32 * (L.n2 * 2 + L.kin * 128) + 3.7 * U * L.kin * L.xplane) / 57.0;
    return 3785.0 + rounds * (in_rows * (95.0 + 109.0 * side) - 51.0 * side * L.part_rows) + 383.0 * jobs + (2168.0 + 90.0 * std::max(0, tasks - 4)) * L.per_cta + load +
           80.0 * L.n2 * U * bh / 16.0 + (L.n_tiles * split > sm_count / 2 ? 1650.0 : 0.0) + (split > 1 ? 3465.0 - 598.0 * (split == 2 ? 1 : split == 4 ? 2 : 3) : 0.0);
}

// The time of the choice that was made, among other kernels and launch included: least squares over 12300 measured choices for 3900 blocks
// (8 to 256 channels in, to 320 out, 16 to 1024 hidden, maps of 4x4 to 130x112, 1 to 64 images, 16 to 148 SMs; 6.3 % rms, at most 26 % too low,
// where lat_rank is 10 % and 74).  What those nine blocks do not show: chunks that wait for each other because there is room for one
// accumulator or one Hd buffer only, and the expansion's own time, which goes with its columns and input planes.
double lat_us(const MbconvArgs& a, const LatLayout& L, int bh, int U, int UG, int parts, int split, int sm_count) {
    const int tasks = U * parts, rounds = L.per_cta * ((tasks + 3) / 4), jobs = L.per_cta * (U / UG), side = std::min(4, tasks);
    const double in_rows = (L.part_rows - 1) * a.stride + 3;
    const double load = (0.6 * L.per_cta * L.cg * 32 * (L.n2 * 2 + L.kin * 128) + 0.7 * U * L.kin * L.xplane) / 57.0;
    double clocks = 8730.0 + rounds * in_rows * (114.0 + 97.0 * side) + 448.0 * jobs + 73.0 * std::max(0, tasks - 4) * L.per_cta + load + 1.8 * L.per_cta * L.kin * U * L.npx +
                  41.0 * L.n2 * U * bh / 16.0 + (L.n_tiles * split > sm_count / 2 ? 1076.0 : 0.0) + (split > 1 ? 1266.0 + 197.0 * (split == 2 ? 1 : split == 4 ? 2 : 3) : 0.0);
    if (L.per_cta > 1) clocks += (L.hdbufs == 1 ? 962.0 * L.per_cta : 0.0) + (L.slots == 1 ? 593.0 * jobs : 0.0);
    return clocks / 1.9e3;
}

}  // namespace

// Units and clusters of the block, the least of lat_rank; not `ok` where the block is none of this kernel's: no expansion layer, more
// tiles than fit the chip at once, or fewer than 128 hidden channels at stride 1, where lane quarters would stand idle (at stride 2 the
// persistent kernel's walk over four times the outputs' inputs costs more than that: 16 -> 96 -> 24 at 112x112, one image 9.1 -> 7.1 us,
// three 10.2 -> 8.5).
MbconvTiling mbconv_lat_tiling(const MbconvArgs& a, int sm_count) {
    MbconvTiling best{};
    best.ok = false;
    double best_rank = 0.0;
    if (!a.has_expand || (a.hid < 128 && a.stride == 1) || !mbconv_supported(a) || sm_count < 1) return best;
    const int Ho = (a.H + 2 - 3) / a.stride + 1, Wo = (a.W + 2 - 3) / a.stride + 1;
    const long long unit_cols = static_cast<long long>(a.N) * ((Wo + kUnitW - 1) / kUnitW);
    for (int bh = 1, rows = 0; bh <= std::min(16, Ho); bh++) {
        if ((Ho + bh - 1) / bh == rows) continue;   // (as many units as with the height before: its rows would only be idle)
        rows = (Ho + bh - 1) / bh;
        for (int U : {1, 2, 3, 4, 6, 8}) {
            if (U * bh > 16 || (unit_cols * rows + U - 1) / U > sm_count) continue;
            for (int UG = 1; UG <= std::min(4, U); UG *= 2)
                for (int parts = 1; parts <= 4 / UG; parts *= 2)
                    for (int split = 1; split <= 8; split *= 2) {
                        LatLayout L;
                        if (!lat_layout(a, bh, U, UG, parts, split, sm_count, &L)) continue;
                        const double rank = lat_rank(a, L, bh, U, UG, parts, split, sm_count);
                        if (best.ok && rank >= best_rank) continue;
                        best_rank = rank;
                        best.bh = bh; best.units = U; best.job_units = UG; best.parts = parts; best.split = split; best.n_tiles = L.n_tiles;
                        best.smem_bytes = L.smem;
                        best.narrow = L.cg <= 2 && L.per_cta > 1;
                        best.us = lat_us(a, L, bh, U, UG, parts, split, sm_count);
                        best.redundancy = static_cast<double>(L.fpx) / (std::min(bh, Ho) * a.stride * std::min(kUnitW, Wo) * a.stride);
                        best.ok = true;
                    }
        }
    }
    return best;
}

int mbconv_lat_init() {
    static bool attr_set[kMaxDevices] = {};
    const int dev = current_device_slot();
    if (dev < 0) return DLF_E_UNSUPPORTED;
    if (!attr_set[dev]) {
        cudaError_t e = cudaSuccess;
        for (int v = 0; v < 4; v++)
            for (int split = 1; split <= 8 && e == cudaSuccess; split *= 2)
                e = cudaFuncSetAttribute(pick_kernel(1 + (v & 1), v >= 2, split), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e);
        attr_set[dev] = true;
    }
    return DLF_OK;
}

int launch_mbconv_lat(const MbconvArgs& a, const MbconvTiling& t, int sm_count, int* status_dev, cudaStream_t s) {
    if (!aligned(16, a.x, a.res, a.y)) return DLF_E_INVALID_ARG;
    int rc = mbconv_lat_init();
    if (rc) return rc;
    LatLayout L;
    if (!t.ok || !lat_layout(a, t.bh, t.units, t.job_units, t.parts, t.split, sm_count, &L)) return DLF_E_PLAN;
    LatBlockParams p;
    std::memset(&p, 0, sizeof(p));
    p.H = a.H; p.W = a.W; p.hid = a.hid; p.Cout = a.Cout;
    p.Ho = (a.H + 2 - 3) / a.stride + 1; p.Wo = (a.W + 2 - 3) / a.stride + 1;
    p.act1 = a.act1; p.act2 = a.act2; p.act3 = a.act3;
    p.bh = t.bh; p.U = t.units; p.UG = t.job_units; p.parts = t.parts; p.part_rows = L.part_rows; p.fpx = L.fpx; p.npx = L.npx;
    p.units_x = L.units_x; p.units_y = L.units_y; p.n_units = L.n_units;
    p.kin = L.kin; p.chunks = L.chunks; p.cg = L.cg; p.n2_pad = L.n2;
    p.ksteps_in_last = ((a.Cin - (p.kin - 1) * 64) + 15) / 16;
    p.n_split = p.n2_pad > 256 ? 2 : 1;
    p.n_each = p.n2_pad / p.n_split;
    p.hdbufs = L.hdbufs; p.w1_stages = L.w1_stages; p.w2_stages = L.w2_stages; p.slots = L.slots;
    p.xplane = L.xplane; p.hd_off = L.hd_off; p.hd_bytes = L.hd_bytes;
    p.w1_off = L.w1_off; p.w1_bytes = L.w1_bytes; p.w2_off = L.w2_off; p.w2_bytes = L.w2_bytes; p.bias_off = L.bias_off;
    p.d2_col = L.d2_col; p.rows_per = L.rows_per; p.red_off = L.red_off;
    p.wd = static_cast<const __half*>(a.wd); p.b1 = a.b1; p.bd = a.bd; p.b2 = a.b2;
    p.res = static_cast<const __half*>(a.res); p.out = static_cast<__half*>(a.y); p.status = status_dev;
    const uint32_t ones[4] = {1, 1, 1, 1};
    {
        const uint64_t dims[4] = {static_cast<uint64_t>(a.Cin), static_cast<uint64_t>(a.W), static_cast<uint64_t>(a.H), static_cast<uint64_t>(a.N)};
        const uint64_t strides[3] = {static_cast<uint64_t>(a.Cin) * 2, static_cast<uint64_t>(a.W) * a.Cin * 2, static_cast<uint64_t>(a.H) * a.W * a.Cin * 2};
        const uint32_t box[4] = {64, static_cast<uint32_t>(L.fw), static_cast<uint32_t>(L.fh), 1};
        rc = encode_tmap(&p.tmx, a.x, 4, dims, strides, box, ones);
    }
    if (rc == DLF_OK) {  // W1 [hid][C_in] seen as (C_in, hid, 1)
        const uint64_t dims[3] = {static_cast<uint64_t>(a.Cin), static_cast<uint64_t>(a.hid), 1};
        const uint64_t strides[2] = {static_cast<uint64_t>(a.Cin) * 2, static_cast<uint64_t>(a.hid) * a.Cin * 2};
        const uint32_t box[3] = {64, 32, 1};
        rc = encode_tmap(&p.tmw1, a.w1, 3, dims, strides, box, ones);
    }
    if (rc == DLF_OK) {  // W2 [C_out][hid] seen as (hid, C_out, 1)
        const uint64_t dims[3] = {static_cast<uint64_t>(a.hid), static_cast<uint64_t>(a.Cout), 1};
        const uint64_t strides[2] = {static_cast<uint64_t>(a.hid) * 2, static_cast<uint64_t>(a.Cout) * a.hid * 2};
        const uint32_t box[3] = {64, static_cast<uint32_t>(p.n_each), 1};
        rc = encode_tmap(&p.tmw2, a.w2, 3, dims, strides, box, ones);
    }
    if (rc) return rc;
    // (never two of these CTAs on an SM: each allocates all of tensor memory)
    const size_t smem = std::max<size_t>(L.smem, 120 * 1024);
    const bool relu6 = p.act2 == DLF_ACT_RELU6 && p.act1 == DLF_ACT_RELU6;
    cudaError_t e = launch_kernel(pick_kernel(a.stride, relu6, t.split), L.n_tiles * t.split, kThreads, smem, s, p);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

}  // namespace dlf
