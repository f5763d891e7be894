// First-layer ("stem") convolution on the tensor cores: C_in <= 4 (the RGB input), kernel up to 11x11, stride 1, 2 or 4,
// up to 64 output channels, bias + activation.
//
// With three input channels a tap is only 6 bytes wide, far below what TMA can address (16-byte strides), so the CTA's own
// threads stage the input patch in shared memory - but nothing more than the patch: no im2col rows are built.  A pixel is
// padded to four channels (8 bytes), two pixels make a 16-byte unit, and the units of a patch row are laid out so that
// neighbouring OUTPUT pixels are neighbouring units.  That is exactly a K-major operand without swizzle: eight pixels of
// the tile's row are one 8 x 16-byte core matrix (128 contiguous bytes), the next row of the tile is `stride` patch rows
// further (the descriptor's stride offset), and the next two kernel columns are another window of the same units, a fixed
// distance away (its leading offset).  Every K = 16 step therefore reads the patch in place; overlapping windows cost
// nothing but the tensor core's own operand reads.
//   stride 1: unit u = pixels u, u + 1 (each pixel stored twice); kernel columns 4i .. 4i+3 = units x + 4i, x + 4i + 2
//   stride 2: unit u = pixels 2u, 2u + 1;                         kernel columns 4i .. 4i+3 = units x + 2i, x + 2i + 1
//   stride 4: even and odd pairs in two planes;                   kernel columns 4i .. 4i+3 = unit x + i of either plane
// Kernel columns past k_w, the fourth channel and output channels past C_out meet zero weights.  The columns past k_w are pixels
// beside the window all the same, and an infinity or a NaN among them times zero is a NaN in every channel: a row whose first
// sum is one is worked out again from the window alone (redo_pixel; one comparison per row where there is none).
//
// Work item = 1 .. 4 tiles of 8 x 16 output pixels (M = 128) side by side that share one patch.  Eight warps build
// patches (two buffers), two warps issue the UMMAs of alternate tiles (N = C_out), four groups of four warps each own one
// accumulator and drain every fourth tile (bias, activation, fp16 rounding, staging tile, TMA store).
// Bound by the patch builders' and epilogue warps' instruction streams (an instruction per warp every eleven cycles, 0.6
// per scheduler and cycle; the output's HBM writes come to a third to a half of the time).  Against the first version,
// which cut im2col rows of K = kh * kw * C_in out of the patch with eight warps that also drained the tiles: 7x7/2 3 -> 64
// at 224x224, batch 32 50.2 -> 27.1 us; 3x3/2 3 -> 32, batch 64 66.0 -> 32.2 us; 3x3 3 -> 64, batch 8 33.3 -> 17.5 us; one
// image of the 7x7/2 layer 9.4 -> 7.3 us; 11x11/4 3 -> 64 (which ran on the CUDA cores) at batch 32 590 -> 23.6 us.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace dlf {

namespace {

constexpr int kGroups = 4;                     // epilogue groups of four warps (one per TMEM lane quarter); group g owns accumulator g
constexpr int kEpiWarps = 4 * kGroups;         // warps 0..15
constexpr int kPatchWarp0 = kEpiWarps;         // warps 16..23 build patches
constexpr int kPatchWarps = 8;
constexpr int kMmaWarp0 = kPatchWarp0 + kPatchWarps;
constexpr int kMmaWarps = 2;                   // issuers, alternate tiles: a lone warp's instruction stream would be the bound
constexpr int kThreads = 32 * (kMmaWarp0 + kMmaWarps);
constexpr int kTileW = 8, kTileH = 16;         // output pixels of one UMMA tile
constexpr int kMaxTiles = 4;                   // tiles side by side in a work item
constexpr int kStage = 128 * 128;              // staging tile: 128 pixels x 64 channels
constexpr int kUnroll = 4;                     // units a patch thread has in flight
constexpr int kMaxDynSmem = 232448 - 1024;     // the 227 KB per CTA less the kernel's static shared memory

struct StemParams {
    const __half* x;
    const __half* w;
    const float* bias;
    int* status;
    int H, W, Ho, Wo, Cout;
    int kh, kw, stride, pad, act;
    int BN, steps;                  // steps: K = 16 UMMAs per kernel row
    int tiles, tiles_w, tiles_h, n_work;   // tiles per work item; work items per row and column of an image
    int units, n_units;             // units per patch row (both planes), units of the patch
    int lp;                         // log2 of the number of planes
    int pitch, plane_bytes, patch_bytes;
    int px_unit;                    // input pixels from one unit to the next
    int a_lbo, a_step, b_lbo, b_step;   // bytes: second half of a K step, next K step
    uint32_t units_magic, kw_magic, per_co_magic;   // quotients by multiplication (see magic())
    int last_word, tail;            // last 32-bit word of the input; 1: only its lower half belongs to the tensor
    int stage_off, patch_off;
};

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, `lbo` bytes between the two core matrices of a
// K = 16 step, `sbo` bytes between groups of eight rows.
__device__ __forceinline__ uint64_t umma_desc_plain(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(lbo >> 4) << 16) | (static_cast<uint64_t>(sbo >> 4) << 32) |
           (static_cast<uint64_t>(1) << 46);
}

__device__ __forceinline__ int quotient(int i, uint32_t magic) { return magic ? static_cast<int>(__umulhi(static_cast<uint32_t>(i), magic)) : i; }

struct ItemOrigin { int wo0, ho0, n; };
__device__ __forceinline__ ItemOrigin decode_item(const StemParams& p, int t) {
    ItemOrigin o;
    o.wo0 = (t % p.tiles_w) * p.tiles * kTileW;
    t /= p.tiles_w;
    o.ho0 = (t % p.tiles_h) * kTileH;
    o.n = t / p.tiles_h;
    return o;
}
// tiles of an item that hold any output pixel
__device__ __forceinline__ int item_tiles(const StemParams& p, const ItemOrigin& o) {
    return min(p.tiles, (p.Wo - o.wo0 + kTileW - 1) / kTileW);
}

// The K = 16 steps of one tile: kernel rows are patch rows, the steps of a row are further windows of the same units.  Sizes
// known at compile time unroll into straight-line issue code (a loop costs its warp about 100 cycles per UMMA).
template <int KH, int STEPS>
__device__ __forceinline__ void issue_tile(uint32_t d_tmem, uint64_t ad, uint64_t bd, uint32_t a_row16, uint32_t a_step16, uint32_t b_step16, uint32_t idesc) {
#pragma unroll
    for (int r = 0; r < KH; r++, ad += a_row16) {
#pragma unroll
        for (int i = 0; i < STEPS; i++, bd += b_step16) umma_f16(d_tmem, ad + static_cast<uint32_t>(i) * a_step16, bd, idesc, (r | i) != 0);
    }
}

// An output pixel's channels by the definition, into its row of the staging tile.
template <int CIN, int ACT>
__device__ __noinline__ void redo_pixel(const __half* x, const __half* w, const float* bias, int H, int W, int kh, int kw, int Cout, int n, int hi0, int wi0, int m, uint8_t* sout) {
    for (int co = 0; co < Cout; co += 2) {
        float v[2] = {0.0f, 0.0f};
        for (int r = 0; r < kh; r++) {
            if (static_cast<unsigned>(hi0 + r) >= static_cast<unsigned>(H)) continue;
            for (int s = 0; s < kw; s++) {
                if (static_cast<unsigned>(wi0 + s) >= static_cast<unsigned>(W)) continue;
                const __half* px = x + ((static_cast<long long>(n) * H + hi0 + r) * W + wi0 + s) * CIN;
                for (int j = 0; j < 2; j++) {
                    const __half* wt = w + (((co + j) * kh + r) * kw + s) * CIN;
                    for (int c = 0; c < CIN; c++) v[j] = fmaf(__half2float(px[c]), __half2float(wt[c]), v[j]);
                }
            }
        }
        *reinterpret_cast<uint32_t*>(sout + m * 128 + (((co >> 3) ^ (m & 7)) << 4) + (co & 7) * 2) = round_act<ACT>(v[0] + bias[co], v[1] + bias[co + 1]);
    }
}

template <int CIN, int ACT>
__global__ void __launch_bounds__(kThreads, 1) stem_tc_kernel(const __grid_constant__ CUtensorMap tmy, const StemParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t wfull_bar, pfull_bar[2], pempty_bar[2], tfull_bar[kGroups], tempty_bar[kGroups];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ __align__(16) float bias_s[64];

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sbase = smem_raw + (base - smem_u32(smem_raw));
    // layout: weights [kh * steps][2][BN][16 B] (padded: see b_step) | staging tiles | two patches
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &abort_s;

    if (threadIdx.x == 0) {
        abort_s = 0;
        mbar_init(&wfull_bar, kEpiWarps);
        for (int i = 0; i < 2; i++) {
            mbar_init(&pfull_bar[i], kPatchWarps);
            mbar_init(&pempty_bar[i], kMmaWarps);
        }
        for (int i = 0; i < kGroups; i++) {
            mbar_init(&tfull_bar[i], 1);
            mbar_init(&tempty_bar[i], 4);
        }
        fence_barrier_init();
        tma_prefetch_desc(&tmy);
    }
    if (warp == kMmaWarp0) {
        tmem_alloc(&tmem_base_s, 64 * kGroups);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_launch_dependents();
    const uint32_t tmem_base = tmem_base_s;

    if (warp >= kMmaWarp0) {
        // ---- UMMA issuers: warp-uniform loops, one elected lane issues; issuer w takes every other tile ----
        const uint32_t w = warp - kMmaWarp0;
        const uint32_t idesc = umma_idesc_f16(p.BN);
        const uint64_t a_desc = umma_desc_plain(base + p.patch_off, p.a_lbo, p.stride * p.pitch);
        const uint64_t b_desc = umma_desc_plain(base, p.b_lbo, 128);
        const uint32_t a_row16 = static_cast<uint32_t>(p.pitch) >> 4, a_step16 = static_cast<uint32_t>(p.a_step) >> 4, b_step16 = static_cast<uint32_t>(p.b_step) >> 4;
        const int shape = p.kh == p.kw ? p.kh : 0;
        uint32_t j = 0, seq = 0, ph = 0;   // ph: phase of this issuer's accumulators (two each, taken in turn)
        bool ok = mbar_wait_warp(&wfull_bar, 0u, abort_flag, p.status, 0x800 | (blockIdx.x << 12));
        for (int t = blockIdx.x; t < p.n_work && ok; t += gridDim.x, j++) {
            const int nt = item_tiles(p, decode_item(p, t));
            const uint32_t b = j & 1u;
            ok = mbar_wait_warp(&pfull_bar[b], (j >> 1) & 1u, abort_flag, p.status, 0x900 | (blockIdx.x << 12));
            if (!ok) break;
            tc_fence_after_sync();
#pragma unroll 1
            for (int k = 0; k < nt; k++, seq++) {
                if ((seq & 1u) != w) continue;
                const uint32_t acc = seq & (kGroups - 1);
                ok = mbar_wait_warp(&tempty_bar[acc], ph ^ 1u, abort_flag, p.status, 0xB00 | (blockIdx.x << 12));
                if (!ok) break;
                if (acc == w + 2) ph ^= 1u;
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * 64u;
                const uint64_t ad = a_desc + ((b * static_cast<uint32_t>(p.patch_bytes) + k * 128u) >> 4);
                if (elect_one()) {
                    if (shape == 3) issue_tile<3, 1>(d_tmem, ad, b_desc, a_row16, a_step16, b_step16, idesc);
                    else if (shape == 5) issue_tile<5, 2>(d_tmem, ad, b_desc, a_row16, a_step16, b_step16, idesc);
                    else if (shape == 7) issue_tile<7, 2>(d_tmem, ad, b_desc, a_row16, a_step16, b_step16, idesc);
                    else if (shape == 11) issue_tile<11, 3>(d_tmem, ad, b_desc, a_row16, a_step16, b_step16, idesc);
                    else {
                        uint64_t arow = ad, bd = b_desc;
#pragma unroll 1
                        for (int r = 0; r < p.kh; r++, arow += a_row16)
#pragma unroll 1
                            for (int i = 0; i < p.steps; i++, bd += b_step16) umma_f16(d_tmem, arow + static_cast<uint32_t>(i) * a_step16, bd, idesc, (r | i) != 0);
                    }
                    umma_commit(&tfull_bar[acc]);
                }
                __syncwarp();
            }
            if (ok && elect_one()) umma_commit(&pempty_bar[b]);   // the patch is free once this issuer's UMMAs have read it
            __syncwarp();
        }
    } else if (warp >= kPatchWarp0) {
        // ---- patch builders ----
        pdl_wait();   // the input may come from the previous kernel
        const uint32_t* x32 = reinterpret_cast<const uint32_t*>(p.x);
        // (a tensor with an odd number of elements ends in half a word)
        const uint32_t tail_word = p.tail ? static_cast<uint32_t>(__half_as_ushort(p.x[2 * static_cast<long long>(p.last_word)])) : 0u;
        const int tid = threadIdx.x - 32 * kPatchWarp0;
        constexpr int kWords = CIN <= 2 ? 2 : 4;   // aligned words that cover a unit's pixels
        uint32_t j = 0;
        for (int t = blockIdx.x; t < p.n_work; t += gridDim.x, j++) {
            const ItemOrigin o = decode_item(p, t);
            const int hi0 = o.ho0 * p.stride - p.pad, wi0 = o.wo0 * p.stride - p.pad;
            const int g0 = ((o.n * p.H + hi0) * p.W + wi0) * CIN, row_halves = p.W * CIN;
            const uint32_t b = j & 1u;
            if (!mbar_wait(&pempty_bar[b], ((j >> 1) & 1u) ^ 1u, abort_flag, p.status, 0xC00 | (blockIdx.x << 12))) break;
            uint8_t* patch = sbase + p.patch_off + b * p.patch_bytes;
#pragma unroll 1
            for (int i0 = tid; i0 < p.n_units; i0 += 32 * kPatchWarps * kUnroll) {
                // a unit = two neighbouring pixels: up to 8 consecutive halves of the tensor, which start on any half; the
                // aligned words that cover them are loaded (all units of the pass in flight together), shifted into place and
                // spread to four channels per pixel
                uint32_t w[kUnroll][4];
                int gw[kUnroll], dst[kUnroll];
                uint32_t flags = 0u;   // per unit: first pixel inside, second pixel inside, odd start
                bool edge = false;     // some of the words lie outside the tensor
#pragma unroll
                for (int u = 0; u < kUnroll; u++) {
                    const int i = i0 + u * 32 * kPatchWarps;
                    const int row = quotient(i, p.units_magic), v = i - row * p.units;
                    const int wi = wi0 + v * p.px_unit;
                    const bool row_ok = static_cast<unsigned>(hi0 + row) < static_cast<unsigned>(p.H) && i < p.n_units;
                    const bool ok0 = row_ok && static_cast<unsigned>(wi) < static_cast<unsigned>(p.W), ok1 = row_ok && static_cast<unsigned>(wi + 1) < static_cast<unsigned>(p.W);
                    const int g = ok0 || ok1 ? g0 + row * row_halves + v * p.px_unit * CIN : 0;   // a unit with no pixel inside reads the tensor's start
                    flags |= ((ok0 ? 1u : 0u) | (ok1 ? 2u : 0u) | ((g & 1) ? 4u : 0u)) << (4 * u);
                    gw[u] = g >> 1;
                    edge = edge || gw[u] < 0 || gw[u] + kWords - 1 > p.last_word - p.tail;
                    dst[u] = i < p.n_units ? (v & ((1 << p.lp) - 1)) * p.plane_bytes + row * p.pitch + (v >> p.lp) * 16 : -1;
                }
                if (!edge) {
#pragma unroll
                    for (int u = 0; u < kUnroll; u++)
#pragma unroll
                        for (int e = 0; e < kWords; e++) w[u][e] = ld_map(x32 + gw[u] + e);
                } else {
#pragma unroll
                    for (int u = 0; u < kUnroll; u++)
#pragma unroll
                        for (int e = 0; e < kWords; e++) {
                            const int k = max(min(gw[u] + e, p.last_word), 0);
                            const uint32_t full = ld_map(x32 + min(k, p.last_word - p.tail));
                            w[u][e] = k > p.last_word - p.tail ? tail_word : full;
                        }
                }
#pragma unroll
                for (int u = 0; u < kUnroll; u++) {
                    const uint32_t f = flags >> (4 * u), sh = (f & 4u) << 2;
                    uint4 q;
                    if (CIN == 1) {
                        const uint32_t a0 = __funnelshift_r(w[u][0], w[u][1], sh);
                        q = make_uint4(a0 & 0xFFFFu, 0u, a0 >> 16, 0u);
                    } else if (CIN == 2) {
                        q = make_uint4(w[u][0], 0u, w[u][1], 0u);
                    } else if (CIN == 3) {
                        const uint32_t a0 = __funnelshift_r(w[u][0], w[u][1], sh), a1 = __funnelshift_r(w[u][1], w[u][2], sh), a2 = __funnelshift_r(w[u][2], w[u][3], sh);
                        q = make_uint4(a0, a1 & 0xFFFFu, __funnelshift_r(a1, a2, 16), a2 >> 16);
                    } else {
                        q = make_uint4(w[u][0], w[u][1], w[u][2], w[u][3]);
                    }
                    if ((f & 3u) != 3u) {
                        if (!(f & 1u)) q.x = q.y = 0u;
                        if (!(f & 2u)) q.z = q.w = 0u;
                    }
                    if (dst[u] >= 0) *reinterpret_cast<uint4*>(patch + dst[u]) = q;
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&pfull_bar[b]);
        }
    } else {
        // ---- the weights, laid out once as the B operand (constants: ahead of the wait for the previous kernel) ----
        const int grp = warp >> 2;
        auto epi_sync = [&]() { asm volatile("bar.sync 5, %0;" ::"n"(32 * kEpiWarps) : "memory"); };
        for (int i = threadIdx.x; i < p.kh * p.steps * p.b_step / 16; i += 32 * kEpiWarps) reinterpret_cast<uint4*>(sbase)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (threadIdx.x < 64) bias_s[threadIdx.x] = threadIdx.x < p.Cout ? __ldg(p.bias + threadIdx.x) : 0.0f;
        {
            const int per_co = p.kh * p.kw * CIN, vecs = p.Cout * per_co / 8;   // (C_out is a multiple of 8)
            constexpr int kVecs = 4;
            bool cleared = false;
            for (int v0 = threadIdx.x; v0 < vecs || !cleared; v0 += 32 * kEpiWarps * kVecs) {
                uint4 wv[kVecs];
#pragma unroll
                for (int u = 0; u < kVecs; u++) wv[u] = __ldg(reinterpret_cast<const uint4*>(p.w) + min(v0 + u * 32 * kEpiWarps, vecs - 1));
                if (!cleared) { epi_sync(); cleared = true; }   // the zeros are all written
#pragma unroll 1
                for (int u = 0; u < kVecs; u++) {
                    const int v = v0 + u * 32 * kEpiWarps;
                    if (v >= vecs) break;
                    int co = quotient(v * 8, p.per_co_magic);
                    const int rem = v * 8 - co * per_co, rs = rem / CIN;
                    int c = rem - rs * CIN, r = quotient(rs, p.kw_magic), s = rs - r * p.kw;
                    const uint4 cur = u == 0 ? wv[0] : (u == 1 ? wv[1] : (u == 2 ? wv[2] : wv[3]));
                    const unsigned short* h = reinterpret_cast<const unsigned short*>(&cur);
#pragma unroll
                    for (int e = 0; e < 8; e++) {
                        *reinterpret_cast<unsigned short*>(sbase + (r * p.steps + (s >> 2)) * p.b_step + ((s >> 1) & 1) * p.b_lbo + co * 16 + (s & 1) * 8 + c * 2) = h[e];
                        if (++c == CIN) { c = 0; if (++s == p.kw) { s = 0; if (++r == p.kh) { r = 0; co++; } } }
                    }
                }
            }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&wfull_bar);
        epi_sync();   // (the bias)
        pdl_wait();   // the output's memory may still be in use

        // ---- epilogue: group g drains every fourth tile ----
        const int q = warp & 3;
        const int m = q * 32 + lane;
        const bool issuer = (threadIdx.x & 127) == 0;
        uint8_t* sout = sbase + p.stage_off + grp * kStage;
        uint32_t seq = 0, ph = 0;
        auto group_sync = [&]() {
            if (grp == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
            else if (grp == 1) asm volatile("bar.sync 2, 128;" ::: "memory");
            else if (grp == 2) asm volatile("bar.sync 3, 128;" ::: "memory");
            else asm volatile("bar.sync 4, 128;" ::: "memory");
        };
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + grp * 64u;
        for (int t = blockIdx.x; t < p.n_work; t += gridDim.x) {
            const ItemOrigin o = decode_item(p, t);
            const int nt = item_tiles(p, o);
#pragma unroll 1
            for (int k = 0; k < nt; k++, seq++) {
                if ((seq & (kGroups - 1)) != static_cast<uint32_t>(grp)) continue;
                // (after a wait that gave up the warp goes on to the end without storing: the others of its group are at the
                // group's barriers, and every later wait returns at once)
                const bool ok = mbar_wait(&tfull_bar[grp], ph, abort_flag, p.status, 0xA00 | (blockIdx.x << 12));
                ph ^= 1u;
                __syncwarp();
                tc_fence_after_sync();
                uint32_t r[32];
                tmem_ld32_issue(taddr, r);
                if (issuer) tma_store_wait_read();
                group_sync();   // the staging tile's last store has read it
                bool redo = false;
#pragma unroll 1
                for (int cc = 0; cc < p.BN; cc += 32) {
                    tmem_ld32_wait(r);
                    if (cc == 0) redo = isnan(__uint_as_float(r[0]));
                    if (cc + 32 >= p.BN) {
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&tempty_bar[grp]);
                    }
#pragma unroll
                    for (int g = 0; g < 4; g++) {
                        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(bias_s + cc + g * 8), b1 = *reinterpret_cast<const ulonglong2*>(bias_s + cc + g * 8 + 4);
                        const float2 v0 = add_f2(r[g * 8 + 0], r[g * 8 + 1], b0.x), v1 = add_f2(r[g * 8 + 2], r[g * 8 + 3], b0.y);
                        const float2 v2 = add_f2(r[g * 8 + 4], r[g * 8 + 5], b1.x), v3 = add_f2(r[g * 8 + 6], r[g * 8 + 7], b1.y);
                        const uint4 out = make_uint4(round_act<ACT>(v0.x, v0.y), round_act<ACT>(v1.x, v1.y), round_act<ACT>(v2.x, v2.y), round_act<ACT>(v3.x, v3.y));
                        const int g8 = (cc >> 3) + g;
                        *reinterpret_cast<uint4*>(sout + m * 128 + (((g8 & 7) ^ (m & 7)) << 4)) = out;
                    }
                    if (cc + 32 < p.BN) {
                        __syncwarp();
                        tmem_ld32_issue(taddr + cc + 32, r);
                    }
                }
                if (redo) {
                    const int wo = o.wo0 + k * kTileW + (m & (kTileW - 1)), ho = o.ho0 + m / kTileW;
                    if (wo < p.Wo && ho < p.Ho)
                        redo_pixel<CIN, ACT>(p.x, p.w, bias_s, p.H, p.W, p.kh, p.kw, p.Cout, o.n, ho * p.stride - p.pad, wo * p.stride - p.pad, m, sout);
                }
                fence_proxy_async_smem();
                group_sync();
                if (issuer && ok) {
                    tma_store_4d(&tmy, sout, 0, o.wo0 + k * kTileW, o.ho0, o.n);
                    tma_store_commit();
                }
            }
        }
        if (issuer) tma_store_wait_read();
    }

    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp0) {
        if (abort_s) __nanosleep(20000);
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 64 * kGroups);
    }
}

// Multiplier for quotient(): i * ceil(2^32 / d) / 2^32 is exact while i < 2^32 / d (here i and d stay below 2^16); 0 for d = 1.
uint32_t magic(int d) { return d <= 1 ? 0u : static_cast<uint32_t>(((1ull << 32) + d - 1) / d); }

// Everything the geometry decides; tiles == 0 if the layer does not fit.
struct Layout {
    int BN, steps, b_lbo, b_step, tiles, rows, units, planes, pitch, plane_bytes, patch_bytes, weight_bytes;
    size_t smem;
};

Layout layout_for(const ConvArgs& a, int tiles) {
    Layout l{};
    l.BN = (a.Cout + 15) / 16 * 16;
    l.steps = (a.kw + 3) / 4;
    l.rows = (kTileH - 1) * a.stride + a.kh;
    l.planes = a.stride == 4 ? 2 : 1;
    // units per plane that the windows of the item's 8 * tiles output columns reach
    const int cols = kTileW * tiles;
    const int per_plane = a.stride == 1 ? cols + 4 * l.steps - 2 : (a.stride == 2 ? cols + 2 * l.steps - 1 : cols + l.steps - 1);
    l.units = per_plane * l.planes;
    l.pitch = per_plane * 16;
    l.plane_bytes = (l.rows * l.pitch + 127) / 128 * 128;
    l.patch_bytes = l.planes * l.plane_bytes;
    // padded so that neighbouring taps of an output channel, which neighbouring threads scatter, fall into different banks
    l.b_lbo = l.BN * 16 + 64;
    l.b_step = 2 * l.b_lbo + 16;
    l.weight_bytes = (a.kh * l.steps * l.b_step + 1023) / 1024 * 1024;
    l.smem = static_cast<size_t>(l.weight_bytes) + kGroups * kStage + 2 * l.patch_bytes + 1024;
    l.tiles = l.smem <= static_cast<size_t>(kMaxDynSmem) && l.rows * l.units < 65536 ? tiles : 0;
    return l;
}

// Tiles per work item: wider items share the halo of the patch, narrower ones spread a small map over more SMs and leave a
// shorter last round.  Cost = rounds of the grid x the slower of an item's UMMAs (or its epilogue) and its patch, plus the
// first patch, which nothing overlaps; in SM clocks.
Layout pick_layout(const ConvArgs& a, int sm_count) {
    Layout best{};
    double best_cost = 0.0;
    for (int tiles = 1; tiles <= kMaxTiles; tiles++) {
        if (tiles > 1 && kTileW * (tiles - 1) >= a.Wo) break;
        const Layout l = layout_for(a, tiles);
        if (l.tiles == 0) continue;
        const long long items = static_cast<long long>((a.Wo + kTileW * tiles - 1) / (kTileW * tiles)) * ((a.Ho + kTileH - 1) / kTileH) * a.N;
        const long long rounds = (items + sm_count - 1) / sm_count;
        const double tile = std::max(a.kh * l.steps * 48.0, l.BN <= 32 ? 180.0 : 300.0), patch = 900.0 + l.rows * l.units * 0.35;
        const double cost = rounds * std::max(tiles * tile, patch) + patch;
        if (best.tiles == 0 || cost < best_cost) {
            best = l;
            best_cost = cost;
        }
    }
    return best;
}

// 32-bit indexing of the input, with room for the patch rows and columns outside the image.
bool input_ok(const ConvArgs& a) {
    const long long row = static_cast<long long>(a.W) * a.Cin;
    const long long total = static_cast<long long>(a.N) * a.H * row;
    return total >= 2 && total + 256 * (row + 256) < 0x7fffffffLL;
}

typedef void (*KernelFn)(const CUtensorMap, const StemParams);
template <int ACT>
KernelFn pick_kernel_act(int cin) {
    switch (cin) {
        case 1: return stem_tc_kernel<1, ACT>;
        case 2: return stem_tc_kernel<2, ACT>;
        case 3: return stem_tc_kernel<3, ACT>;
        default: return stem_tc_kernel<4, ACT>;
    }
}
KernelFn pick_kernel(int cin, int act) {
    return act == DLF_ACT_RELU6 ? pick_kernel_act<2>(cin) : (act == DLF_ACT_RELU ? pick_kernel_act<1>(cin) : pick_kernel_act<0>(cin));
}

}  // namespace

bool stem_tc_supported(const ConvArgs& a) {
    return a.groups == 1 && a.Cin >= 1 && a.Cin <= 4 && a.Cout % 8 == 0 && a.Cout >= 8 && a.Cout <= 64 && a.kh >= 1 && a.kh <= 11 &&
           a.kw >= 1 && a.kw <= 11 && (a.stride == 1 || a.stride == 2 || a.stride == 4) && a.pool == 0 && a.res == nullptr && a.N >= 1 && a.Ho >= 1 &&
           a.Wo >= 1 && input_ok(a) && layout_for(a, 1).tiles > 0;
}

int stem_tc_init() {
    static bool attr_set[kMaxDevices] = {};
    const int dev = current_device_slot();
    if (dev < 0) return DLF_E_UNSUPPORTED;
    if (!attr_set[dev]) {
        for (int v = 0; v < 12; v++) {
            cudaError_t e = cudaFuncSetAttribute(pick_kernel(1 + v / 3, v % 3), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
            if (e != cudaSuccess) return cuda_fail(e);
        }
        attr_set[dev] = true;
    }
    return DLF_OK;
}

int launch_stem_tc(const ConvArgs& a, int sm_count, int* status_dev, cudaStream_t s) {
    if (!stem_tc_supported(a)) return DLF_E_UNSUPPORTED;
    if (!aligned(4, a.x) || !aligned(16, a.y)) return DLF_E_INVALID_ARG;
    int rc = stem_tc_init();
    if (rc) return rc;
    const Layout l = pick_layout(a, sm_count);
    StemParams p{};
    p.x = static_cast<const __half*>(a.x); p.w = static_cast<const __half*>(a.w); p.bias = a.bias; p.status = status_dev;
    p.H = a.H; p.W = a.W; p.Ho = a.Ho; p.Wo = a.Wo; p.Cout = a.Cout;
    p.kh = a.kh; p.kw = a.kw; p.stride = a.stride; p.pad = a.pad; p.act = a.act;
    p.BN = l.BN; p.steps = l.steps; p.tiles = l.tiles;
    p.tiles_w = (a.Wo + kTileW * l.tiles - 1) / (kTileW * l.tiles);
    p.tiles_h = (a.Ho + kTileH - 1) / kTileH;
    const long long n_work = static_cast<long long>(p.tiles_w) * p.tiles_h * a.N;
    if (n_work > 0x7fffffffLL) return DLF_E_UNSUPPORTED;
    p.n_work = static_cast<int>(n_work);
    p.units = l.units; p.n_units = l.rows * l.units;
    p.lp = l.planes == 2 ? 1 : 0;
    p.pitch = l.pitch; p.plane_bytes = l.plane_bytes; p.patch_bytes = l.patch_bytes;
    p.px_unit = a.stride == 1 ? 1 : 2;
    p.a_lbo = a.stride == 1 ? 32 : (a.stride == 2 ? 16 : l.plane_bytes);
    p.a_step = a.stride == 1 ? 64 : (a.stride == 2 ? 32 : 16);
    p.b_lbo = l.b_lbo; p.b_step = l.b_step;
    p.units_magic = magic(l.units); p.kw_magic = magic(a.kw); p.per_co_magic = magic(a.kh * a.kw * a.Cin);
    const long long total = static_cast<long long>(a.N) * a.H * a.W * a.Cin;
    p.last_word = static_cast<int>((total - 1) / 2);
    p.tail = static_cast<int>(total & 1);
    p.stage_off = l.weight_bytes;
    p.patch_off = l.weight_bytes + kGroups * kStage;
    CUtensorMap tmy;
    {
        const uint64_t dims[4] = {static_cast<uint64_t>(a.Cout), static_cast<uint64_t>(a.Wo), static_cast<uint64_t>(a.Ho),
                                  static_cast<uint64_t>(a.N)};
        const uint64_t strides[3] = {static_cast<uint64_t>(a.Cout) * 2, static_cast<uint64_t>(a.Wo) * a.Cout * 2,
                                     static_cast<uint64_t>(a.Ho) * a.Wo * a.Cout * 2};
        const uint32_t box[4] = {64, kTileW, kTileH, 1};
        const uint32_t es[4] = {1, 1, 1, 1};
        rc = encode_tmap(&tmy, a.y, 4, dims, strides, box, es);
        if (rc) return rc;
    }
    const int grid = std::max(1, std::min(sm_count, p.n_work));
    const size_t smem = std::max<size_t>(l.smem, 120 * 1024);   // (one CTA of a persistent grid per SM)
    cudaError_t e = launch_kernel(pick_kernel(a.Cin, a.act), grid, kThreads, smem, s, tmy, p);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

}  // namespace dlf
