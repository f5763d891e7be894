// Implicit-GEMM convolution on tcgen05 for layers too small to fill the chip twice: one output tile per CTA, nothing
// persistent.  What bounds these layers is not a rate but the chain set-up -> first copy -> UMMAs -> drain -> store of one
// tile, so this kernel keeps that chain short: every warp has one job, the weights are on their way before the previous
// kernel has finished, the tile leaves by plain 16-byte stores straight from the registers it was drained into, tensor memory
// is given back while those stores are under way, and the CTA is small enough (416 threads, at most 110 KB of shared memory,
// half of the columns of tensor memory) to be set up beside its predecessor.
//
// A long K (a 3x3 layer on 512 channels has 72 chunks of 64) is shared out over a cluster of SPLIT CTAs that work on the same
// tile.  Their fp32 partial tiles meet in distributed shared memory: CTA d of the cluster adds up, in the order of the ranks,
// and finishes every SPLIT-th run of rows; each warp writes the rows it drained straight into the shared memory of the CTA
// they belong to, and a barrier there counts the bytes (st.async): a CTA waits for its own rows only (a barrier of the whole
// cluster in its place took about 1 us of a layer's 5).  No global scratch, no atomics, the same sum whatever the timing.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "internal.h"
#include "ptx.cuh"

namespace dlf {

namespace {

constexpr int kEpiWarps = 8;                // warps 0..7: warp & 3 = TMEM lane quarter, warp >> 2 = even or odd 16-column groups
constexpr int kProdWarp0 = kEpiWarps;       // warps 8..10 load: warp w takes ring stages w, w + 3, ...
constexpr int kProdWarps = 3;
constexpr int kMmaWarp0 = kProdWarp0 + kProdWarps;
constexpr int kMmaWarps = 2;                // issuers: warp w takes chunks w, w + 2, ... into an accumulator of its own
constexpr int kThreads = 32 * (kMmaWarp0 + kMmaWarps);
constexpr int kMaxBN = 128;
constexpr int kMaxStages = 12;
constexpr int kItems = 4;                   // finished 8-channel vectors per epilogue thread
constexpr int kMaxOut = kItems * 32 * kEpiWarps * 8;   // so that a CTA finishes at most 8192 values
constexpr int kMaxDynSmem = 226 * 1024;     // 227 KB per CTA less the static part
constexpr int kPairSmem = 110 * 1024;       // two CTAs fit an SM: this one is set up while its predecessor's still runs

struct LatParams {
    int N, Ho, Wo, Cout;
    int kw, stride, pad;
    int TW, TH, rows, tiles_w, tiles_h, n_tiles_n, BN;
    int TN;
    int kchunks, kchunks1, ksteps_last;     // 64-channel chunks per tap (both sources), of the first source; UMMAs of the last one
    int total, share;                       // (tap, chunk) pairs of K, and how many a CTA of the cluster takes
    int stride2;
    int stages, a_bytes, stage_bytes, red_off;
    int rows_per, act;
    const float* bias;
    const float* bias2;
    const __half* res;
    __half* out;
    int* status;
};

template <int SPLIT>
__global__ void __cluster_dims__(SPLIT, 1, 1) __launch_bounds__(kThreads, 2)
conv_lat_kernel(const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmw, const __grid_constant__ CUtensorMap tmx2,
                const __grid_constant__ CUtensorMap tmw2, const __grid_constant__ LatParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], tfull_bar, tdone_bar, red_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, red_abort_s;
    __shared__ __align__(16) float bias_s[kMaxBN];

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sbase = smem_raw + (base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &abort_s;
    const int rank = SPLIT > 1 ? static_cast<int>(cluster_rank()) : 0;
    const int tile = SPLIT > 1 ? static_cast<int>(blockIdx.x) / SPLIT : static_cast<int>(blockIdx.x);
    const int co0 = (tile % p.n_tiles_n) * p.BN;
    int mt = tile / p.n_tiles_n;
    const int wo0 = (mt % p.tiles_w) * p.TW;
    mt /= p.tiles_w;
    const int ho0 = (mt % p.tiles_h) * p.TH, n0 = (mt / p.tiles_h) * p.TN;
    const int k_first = rank * p.share, k_count = min(p.share, p.total - k_first);

    if (warp == kProdWarp0 + 1) {
        if (lane < kMaxStages) {
            mbar_init(&full_bar[lane], 1);
            mbar_init(&empty_bar[lane], 1);
        }
        if (lane == 0) {
            abort_s = 0;
            red_abort_s = 0;
            mbar_init(&tfull_bar, kMmaWarps);
            mbar_init(&tdone_bar, kEpiWarps);
            mbar_init(&red_bar, 1);
        }
        fence_barrier_init();
        // the bytes that the cluster's CTAs will send here (before the cluster's barrier, which every sender waits for)
        if (SPLIT > 1 && lane == 0) mbar_expect_tx(&red_bar, static_cast<uint32_t>(SPLIT * max(0, min(p.rows_per, p.rows - rank * p.rows_per)) * p.BN) * 4u);
    }
    if (warp == kProdWarp0 && lane == 0) {
        tma_prefetch_desc(&tmw);
        tma_prefetch_desc(&tmx);
        if (p.kchunks1 < p.kchunks) { tma_prefetch_desc(&tmx2); tma_prefetch_desc(&tmw2); }
    }
    if (warp == kMmaWarp0) {
        tmem_alloc(&tmem_base_s, kMaxBN * kMmaWarps);
        tmem_relinquish();
    }
    if (threadIdx.x < kMaxBN) {
        const int co = co0 + threadIdx.x;
        bias_s[threadIdx.x] = co < p.Cout ? __ldg(p.bias + co) + (p.bias2 ? __ldg(p.bias2 + co) : 0.0f) : 0.0f;
    }
    tc_fence_before_sync();
    __syncthreads();
    if (SPLIT > 1) cluster_arrive();   // first phase: all CTAs of the cluster run (waited for before rows go to the others)
    tc_fence_after_sync();
    pdl_launch_dependents();
    const uint32_t tmem_base = tmem_base_s;

    if (warp >= kProdWarp0 && warp < kMmaWarp0) {
        // ---- producers: warp w owns ring stages w, w + 3, ...; one elected lane issues; the weights of the first ring pass are
        // on their way before the wait for the previous kernel ----
        const int w = warp - kProdWarp0;
        const uint32_t stage_tx = static_cast<uint32_t>(p.rows + p.BN) * 128u;
        const int hi0 = ho0 * p.stride - p.pad, wi0 = wo0 * p.stride - p.pad;
        const int tap0 = k_first / p.kchunks, r0 = tap0 / p.kw;
        // position of a chunk in K, advanced one chunk at a time (a division costs a lone warp about a hundred cycles)
        struct Pos { int tap, r, s, kc; };
        const Pos start{tap0, r0, tap0 - r0 * p.kw, k_first - tap0 * p.kchunks};
        auto advance = [&](Pos& c) {
            if (++c.kc == p.kchunks) {
                c.kc = 0;
                c.tap++;
                if (++c.s == p.kw) { c.s = 0; c.r++; }
            }
        };
        auto load_b = [&](const Pos& c, int st) {
            uint8_t* dst = sbase + st * p.stage_bytes + p.a_bytes;
            if (c.kc >= p.kchunks1) tma_load_3d(dst, &tmw2, &full_bar[st], (c.kc - p.kchunks1) * 64, 0, co0);
            else tma_load_3d(dst, &tmw, &full_bar[st], c.kc * 64, c.tap, co0);
        };
        auto load_a = [&](const Pos& c, int st) {
            uint8_t* dst = sbase + st * p.stage_bytes;
            if (c.kc >= p.kchunks1) tma_load_4d(dst, &tmx2, &full_bar[st], (c.kc - p.kchunks1) * 64, wo0 * p.stride2, ho0 * p.stride2, n0);
            else tma_load_4d(dst, &tmx, &full_bar[st], c.kc * 64, wi0 + c.s, hi0 + c.r, n0);
        };
        const int first_pass = min(p.stages, k_count);
        if (elect_one()) {
            Pos c = start;
            int turn = 0;
#pragma unroll 1
            for (int i = 0; i < first_pass; i++, advance(c)) {
                if (turn == w) {
                    mbar_expect_tx(&full_bar[i], stage_tx);
                    load_b(c, i);
                }
                if (++turn == kProdWarps) turn = 0;
            }
        }
        __syncwarp();
        pdl_wait();
        Pos c = start;
        int turn = 0, st = 0;
        uint32_t ph = 1;
#pragma unroll 1
        for (int i = 0; i < k_count; i++, advance(c)) {
            if (turn == w) {
                if (i >= first_pass && !mbar_wait_warp<true>(&empty_bar[st], ph, abort_flag, p.status, 0xE00 | (blockIdx.x << 12))) break;
                if (elect_one()) {
                    if (i >= first_pass) {
                        mbar_expect_tx(&full_bar[st], stage_tx);
                        load_b(c, st);
                    }
                    load_a(c, st);
                }
                __syncwarp();
            }
            if (++turn == kProdWarps) turn = 0;
            if (++st == p.stages) { st = 0; turn = 0; ph ^= 1u; }
        }
    } else if (warp >= kMmaWarp0) {
        // ---- issuers.  A run of UMMAs holds its warp until it has almost executed, and what the warp does between two runs
        // (the wait, descriptors, the commit) takes as long again: two warps with an accumulator each hide one behind the other
        // (540 -> 290 clocks per chunk of 64 channels); the epilogue adds the two sums ----
        const int w = warp - kMmaWarp0;
        const uint32_t idesc = umma_idesc_f16(p.BN), d_tmem = tmem_base + w * kMaxBN;
        const uint32_t desc0 = umma_desc_lo(base);
        const uint32_t stage16 = static_cast<uint32_t>(p.stage_bytes) >> 4, b16 = static_cast<uint32_t>(p.a_bytes) >> 4;
        const int last = k_count - 1 - ((k_count - 1 - w) & 1);   // this issuer's last chunk (negative: it has none)
        int st = w % p.stages, kc = (k_first + w) % p.kchunks;
        uint32_t ph = static_cast<uint32_t>(w / p.stages) & 1u;
        uint32_t ad = desc0 + static_cast<uint32_t>(st) * stage16;
#pragma unroll 1
        for (int i = w; i < k_count; i += 2) {
            if (!mbar_wait_warp<true>(&full_bar[st], ph, abort_flag, p.status, 0xE10 | (blockIdx.x << 12))) break;
            tc_fence_after_sync();
            const int ksteps = kc == p.kchunks - 1 ? p.ksteps_last : 4;
            const uint32_t bd = ad + b16;
            if (elect_one()) {
                if (ksteps == 4) umma_f16_steps<4>(d_tmem, ad, bd, idesc, i != w);
                else if (ksteps == 3) umma_f16_steps<3>(d_tmem, ad, bd, idesc, i != w);
                else if (ksteps == 2) umma_f16_steps<2>(d_tmem, ad, bd, idesc, i != w);
                else umma_f16_steps<1>(d_tmem, ad, bd, idesc, i != w);
                if (i + p.stages < k_count) umma_commit(&empty_bar[st]);
                if (i == last) umma_commit(&tfull_bar);
            }
            __syncwarp();
            kc += 2;
            if (kc >= p.kchunks) kc -= p.kchunks;
            if (kc >= p.kchunks) kc -= p.kchunks;   // (one chunk per tap)
            st += 2;
            ad += 2 * stage16;
            if (st >= p.stages) { st -= p.stages; ph ^= 1u; ad -= static_cast<uint32_t>(p.stages) * stage16; }
        }
        if (last < 0 && lane == 0) mbar_arrive(&tfull_bar);
    } else {
        // ---- epilogue ----
        const int q = warp & 3, half = warp >> 2;
        [[maybe_unused]] const int bn8 = p.BN >> 3;
        const __half2 lo = act_lo(p.act), hi = act_hi(p.act);
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        const int m = q * 32 + lane;
        // the sums of 16 columns of this thread's row, from both accumulators
        auto drain = [&](int c0, float (&v)[16]) {
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + c0;
            uint32_t r0[16];
            tmem_ld16_issue(taddr, r0);
            if (k_count > 1) {
                uint32_t r1[16];
                tmem_ld16_issue(taddr + kMaxBN, r1);
                tmem_ld16_wait(r0);
                tmem_ld16_wait(r1);
#pragma unroll
                for (int e = 0; e < 16; e++) v[e] = __uint_as_float(r0[e]) + __uint_as_float(r1[e]);
            } else {
                tmem_ld16_wait(r0);
#pragma unroll
                for (int e = 0; e < 16; e++) v[e] = __uint_as_float(r0[e]);
            }
            if (c0 + 32 >= p.BN) {   // this warp's last: tensor memory may go as far as it is concerned
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tdone_bar);
            }
        };
        if (half * 16 >= p.BN && lane == 0) mbar_arrive(&tdone_bar);   // (a tile of 16 columns: the other four warps drain it)
        if (SPLIT == 1) {
            // a thread finishes its own row: no exchange, the first vectors' residual is fetched behind the UMMAs
            const int tw = m % p.TW, t2 = m / p.TW, th = t2 % p.TH, tn = t2 / p.TH;
            const int n = n0 + tn, ho = ho0 + th, wo = wo0 + tw;
            const bool live = m < p.rows && n < p.N && ho < p.Ho && wo < p.Wo;
            const long long row = (((static_cast<long long>(n) * p.Ho + ho) * p.Wo + wo) * p.Cout) + co0;
            const int n_co = p.Cout - co0;
            pdl_wait();
            uint4 rv[kItems] = {zero, zero, zero, zero};
            if (p.res && live) {
#pragma unroll
                for (int it = 0; it < kItems; it++) {
                    const int c = half * 16 + (it >> 1) * 32 + (it & 1) * 8;
                    if (c < p.BN && c < n_co) rv[it] = ld_map(reinterpret_cast<const uint4*>(p.res + row + c));
                }
            }
            const bool ok = mbar_wait<true>(&tfull_bar, 0u, abort_flag, p.status, 0xE20 | (blockIdx.x << 12));
            __syncwarp();
            tc_fence_after_sync();
#pragma unroll
            for (int j = 0; j < kMaxBN / 32; j++) {
                const int c0 = half * 16 + j * 32;
                if (c0 >= p.BN) break;
                float v[16];
                drain(c0, v);
                if (live && ok) {
#pragma unroll
                    for (int g = 0; g < 2; g++) {
                        const int c = c0 + g * 8;
                        if (c >= n_co) break;
                        uint4 res = zero;
                        if (2 * j + g < kItems) res = rv[(2 * j + g) % kItems];
                        else if (p.res) res = ld_map(reinterpret_cast<const uint4*>(p.res + row + c));
                        *reinterpret_cast<uint4*>(p.out + row + c) = finish8(v + g * 8, bias_s + c, res, lo, hi);
                    }
                }
            }
        } else {
            // the vectors this thread will finish: where they go, and their residual (its latency hides behind the UMMAs)
            long long off[kItems];
            uint32_t src[kItems];   // byte offset of the vector's first half in a rank's rows; its second half is 16 bytes beside it
            int bias_at[kItems];
            uint4 rv[kItems];
            const int n_items = p.rows_per * bn8;
            // a row's 16-byte vectors are stored in an order that depends on the row, so that the lanes of a warp (one row each)
            // fall into different banks
            const uint32_t swz = p.BN % 32 == 0 ? 7u : 3u;
#pragma unroll
            for (int it = 0; it < kItems; it++) {
                const int i = static_cast<int>(threadIdx.x) + it * 32 * kEpiWarps;
                off[it] = -1;
                src[it] = 0u;
                bias_at[it] = 0;
                if (i >= n_items) continue;
                const int r = i / bn8, g = i - r * bn8, mo = rank * p.rows_per + r;
                const int tw = mo % p.TW, t2 = mo / p.TW, th = t2 % p.TH, tn = t2 / p.TH;
                const int n = n0 + tn, ho = ho0 + th, wo = wo0 + tw, co = co0 + g * 8;
                src[it] = static_cast<uint32_t>(r * p.BN * 4) + ((static_cast<uint32_t>(2 * g) ^ (static_cast<uint32_t>(r) & swz)) << 4);
                bias_at[it] = g * 8;
                if (mo < p.rows && n < p.N && ho < p.Ho && wo < p.Wo && co < p.Cout)
                    off[it] = ((static_cast<long long>(n) * p.Ho + ho) * p.Wo + wo) * p.Cout + co;
            }
            pdl_wait();
#pragma unroll
            for (int it = 0; it < kItems; it++) rv[it] = p.res && off[it] >= 0 ? ld_map(reinterpret_cast<const uint4*>(p.res + off[it])) : zero;
            const int dest = min(m / p.rows_per, SPLIT - 1), row = m - dest * p.rows_per;
            const uint32_t slab = static_cast<uint32_t>(p.rows_per * p.BN * 4);   // one rank's partial rows
            const uint32_t dst = mapa(base + p.red_off + rank * slab + row * p.BN * 4, dest), dst_bar = mapa(smem_u32(&red_bar), dest);
            bool ok = mbar_wait<true>(&tfull_bar, 0u, abort_flag, p.status, 0xE20 | (blockIdx.x << 12));
            __syncwarp();
            tc_fence_after_sync();
            cluster_wait();   // every CTA of the cluster runs and its barrier expects these rows
#pragma unroll 1
            for (int c0 = half * 16; c0 < p.BN; c0 += 32) {
                float v[16];
                drain(c0, v);
                if (m < p.rows) {   // (sent whatever happened: the other CTAs wait for the bytes)
#pragma unroll
                    for (int e = 0; e < 4; e++)
                        st_async_v4(dst + ((static_cast<uint32_t>((c0 >> 2) + e) ^ (static_cast<uint32_t>(row) & swz)) << 4),
                                    v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3], dst_bar);
                }
                __syncwarp();
            }
            // all rows of this CTA are here.  It must not retire before that, whatever its own part came to, hence a limit above
            // the senders' and a flag of its own.
            ok = mbar_wait<true>(&red_bar, 0u, &red_abort_s, p.status, 0xE30 | (blockIdx.x << 12), 4 * kWaitLimitNs) && ok;
            const uint8_t* red = sbase + p.red_off;
#pragma unroll
            for (int it = 0; it < kItems; it++) {
                if (off[it] < 0 || !ok) continue;
                float4 a = *reinterpret_cast<const float4*>(red + src[it]), b = *reinterpret_cast<const float4*>(red + (src[it] ^ 16u));
#pragma unroll
                for (int sp = 1; sp < SPLIT; sp++) {
                    const float4 a2 = *reinterpret_cast<const float4*>(red + sp * slab + src[it]), b2 = *reinterpret_cast<const float4*>(red + sp * slab + (src[it] ^ 16u));
                    a.x += a2.x; a.y += a2.y; a.z += a2.z; a.w += a2.w;
                    b.x += b2.x; b.y += b2.y; b.z += b2.z; b.w += b2.w;
                }
                const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                *reinterpret_cast<uint4*>(p.out + off[it]) = finish8(v, bias_s + bias_at[it], rv[it], lo, hi);
            }
        }
    }
    __syncwarp();
    if (SPLIT > 1 && warp >= kEpiWarps) cluster_wait();
    if (warp == kMmaWarp0) {
        // tensor memory is given back as soon as it has been read, while the tile is still on its way out
        const bool ok = mbar_wait_warp(&tdone_bar, 0u, &red_abort_s, p.status, 0xE40 | (blockIdx.x << 12), 2 * kWaitLimitNs);
        if (abort_s || !ok) __nanosleep(20000);   // let copies in flight land before the CTA retires
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kMaxBN * kMmaWarps);
    }
}

typedef void (*KernelFn)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const LatParams);
KernelFn pick_kernel(int split) {
    switch (split) {
        case 1: return conv_lat_kernel<1>;
        case 2: return conv_lat_kernel<2>;
        case 4: return conv_lat_kernel<4>;
        default: return conv_lat_kernel<8>;
    }
}

struct Tile { int tw, th, tn; };

// Output tile of at most `cap` pixels: the fewest tiles, then the fewest rows.
Tile pick_tile(int N, int Ho, int Wo, int cap) {
    Tile best{1, 1, 1};
    long long best_tiles = -1;
    int best_rows = 0;
    // (of the heights that make the same number of tile rows the least is never worse, and so for the images; the others are
    // passed over: 540 combinations of four divisions each took a third of a launch's host time)
    for (int tn = 1, parts_n = 0; tn <= std::min(N, cap); tn++) {
        if ((N + tn - 1) / tn == parts_n) continue;
        parts_n = (N + tn - 1) / tn;
        for (int th = 1, parts_h = 0; th <= std::min(Ho, cap / tn); th++) {
            if ((Ho + th - 1) / th == parts_h) continue;
            parts_h = (Ho + th - 1) / th;
            const int tw_max = std::min(Wo, cap / (tn * th)), cols = (Wo + tw_max - 1) / tw_max, tw = (Wo + cols - 1) / cols;
            const int rows = tn * th * tw;
            const long long tiles = static_cast<long long>(cols) * parts_h * parts_n;
            if (best_tiles < 0 || tiles < best_tiles || (tiles == best_tiles && rows < best_rows)) {
                best_tiles = tiles;
                best_rows = rows;
                best = Tile{tw, th, tn};
            }
        }
    }
    return best;
}

struct Choice {
    Tile tile;
    int BN, split, share, stages, rows_per;
    double cost;   // SM clocks between set-up and the last store; negative: none
};

Choice choose(const ConvArgs& a, int total, int sm_count, const int (&max_clusters)[4]) {
    Choice best{};
    best.cost = -1.0;
    const int cout16 = (a.Cout + 15) / 16 * 16;
    for (int cap : {128, 96, 64, 32}) {
        const Tile t = pick_tile(a.N, a.Ho, a.Wo, cap);
        const int rows = t.tw * t.th * t.tn, a_bytes = (rows + 7) / 8 * 1024;
        const long long m_tiles = static_cast<long long>((a.Wo + t.tw - 1) / t.tw) * ((a.Ho + t.th - 1) / t.th) * ((a.N + t.tn - 1) / t.tn);
        for (int bn : {64, 128}) {
            if (bn == 128 && cout16 <= 64) continue;
            const int BN = std::min(cout16, bn), stage = a_bytes + BN * 128;
            const long long tiles = m_tiles * ((cout16 + BN - 1) / BN);
            for (int lg = 0; lg <= 3; lg++) {
                const int split = 1 << lg, share = (total + split - 1) / split, rows_per = (rows + split - 1) / split;
                if (tiles * split > sm_count) break;
                if ((split > 1 && (split - 1) * share >= total) || rows_per * BN > kMaxOut) continue;
                for (int smem : {kPairSmem, kMaxDynSmem}) {
                    const int budget = smem - 1024 - (split > 1 ? split * rows_per * BN * 4 : 0) - (128 * 128 - a_bytes);
                    int stages = std::min({kMaxStages, budget / stage, share});
                    if (stages < share) stages &= ~1;   // the ring goes round: a stage belongs to one issuer
                    if (stages < std::min(share, 2)) continue;
                    if (tiles > (smem > kPairSmem ? max_clusters[lg] : 2 * max_clusters[lg])) continue;   // (a second wave of clusters)
                    // Fitted to about 2000 measured (layer, tile, split) times of 102 layers (ResNet-50's at 1 to 6 images, MobileNetV2's
                    // at 1 and 4, odd ones): a chunk costs what its two issuers take, and with a ring that goes round its part of a
                    // round trip; sharing a tile costs the exchange of its sums; CTAs on more than half of the SMs find the
                    // previous kernel still there, and so do CTAs that fit an SM only once.  The layers chosen by it take 567 us in
                    // all, the best choice for each 558, the constants before these 590.
                    double chunk = 315.0 + 0.45 * BN;
                    if (stages < share) chunk = std::max(chunk, 2500.0 / stages);
                    const double cost = 2000.0 + stage / 366.0 + share * chunk + rows * BN * (lg > 0 ? 0.47 : 0.13) + (lg > 0 ? 760.0 : 0.0) + (lg == 3 ? 160.0 : 0.0) +
                                        (tiles * split > sm_count / 2 ? (lg > 0 ? 1500.0 : 2250.0) : 0.0) + (smem > kPairSmem ? 280.0 : 0.0);
                    if (best.cost < 0 || cost < best.cost) best = Choice{t, BN, split, share, stages, rows_per, cost};
                }
            }
        }
    }
    return best;
}

}  // namespace

// Clusters of 1, 2, 4, 8 CTAs that run at the same time on an otherwise empty device, one CTA per SM (conv_lat_init).
static int g_max_clusters[kMaxDevices][4];

int launch_conv_lat(const ConvArgs& a_in, int sm_count, int* status_dev, cudaStream_t s) {
    const bool dual = a_in.x2 != nullptr;
    if (a_in.pool || !conv_tc_supported(a_in) || (dual && !conv_tc_dual_supported(a_in))) return DLF_E_UNSUPPORTED;
    ConvArgs a = a_in;
    const long long flat_pixels = static_cast<long long>(a.N) * a.H * a.W;
    if (a.kh == 1 && a.kw == 1 && a.stride == 1 && a.pad == 0 && !dual && flat_pixels < (1ll << 31)) {   // no spatial structure: one list of pixels
        a.N = 1; a.H = 1; a.Ho = 1;
        a.W = a.Wo = static_cast<int>(flat_pixels);
    }
    if (static_cast<long long>(a.N) * a.Ho * a.Wo > 128ll * sm_count) return DLF_E_UNSUPPORTED;
    LatParams p{};
    p.kchunks1 = (a.Cin + 63) / 64;
    p.ksteps_last = ((a.Cin - (p.kchunks1 - 1) * 64) + 15) / 16;
    p.kchunks = p.kchunks1 + (dual ? a.Cin2 / 64 : 0);
    p.total = a.kh * a.kw * p.kchunks;
    const int dev = current_device_slot();
    if (dev < 0) return DLF_E_UNSUPPORTED;
    const Choice c = choose(a, p.total, sm_count, g_max_clusters[dev]);
    // Where the tiles fit one wave this kernel is the faster one (64 -> 64 at one 56x56 image 2.6 us against 3.6 in a network, 512
    // -> 128 at six 28x28 images 5.0 against 6.1), except for layers whose kernel rows the persistent kernel loads once: there it
    // takes over when a CTA's share of K is long (256 -> 256 3x3 at six 14x14 images: 9.6 against 9.1).
    const bool row = a.kh == 3 && a.kw == 3 && a.stride == 1 && a.Cin % 64 == 0 && g_conv_row_mode > 0;
    if (g_conv_row_mode > 1 && conv_tc_row_mode(a)) return DLF_E_UNSUPPORTED;   // (asked for)
    if (c.cost < 0 || (row && c.cost > 8600.0 + 117.0 * p.total)) return DLF_E_UNSUPPORTED;
    p.N = a.N; p.Ho = a.Ho; p.Wo = a.Wo; p.Cout = a.Cout;
    p.kw = a.kw; p.stride = a.stride; p.pad = a.pad; p.stride2 = dual ? a.stride2 : 1;
    p.TW = c.tile.tw; p.TH = c.tile.th; p.TN = c.tile.tn;
    p.rows = p.TW * p.TH * p.TN;
    p.tiles_w = (a.Wo + p.TW - 1) / p.TW; p.tiles_h = (a.Ho + p.TH - 1) / p.TH;
    const int tiles_n = (a.N + p.TN - 1) / p.TN;
    p.BN = c.BN;
    p.n_tiles_n = ((a.Cout + 15) / 16 * 16 + c.BN - 1) / c.BN;
    p.share = c.share; p.stages = c.stages; p.rows_per = c.rows_per;
    p.a_bytes = (p.rows + 7) / 8 * 1024;
    p.stage_bytes = p.a_bytes + p.BN * 128;
    // (the UMMA always reads 128 rows: behind a shorter last slab it reads on into memory that must still be this CTA's)
    p.red_off = p.stages * p.stage_bytes + (128 * 128 - p.a_bytes);
    p.act = a.act;
    p.bias = a.bias; p.bias2 = dual ? a.bias2 : nullptr;
    p.res = static_cast<const __half*>(a.res); p.out = static_cast<__half*>(a.y);
    p.status = status_dev;
    CUtensorMap tmx, tmw, tmx2, tmw2;
    auto input_map = [&](CUtensorMap* m, const void* x, int W, int H, int C, int stride) {
        const uint64_t dims[4] = {static_cast<uint64_t>(C), static_cast<uint64_t>(W), static_cast<uint64_t>(H), static_cast<uint64_t>(a.N)};
        const uint64_t strides[3] = {static_cast<uint64_t>(C) * 2, static_cast<uint64_t>(W) * C * 2, static_cast<uint64_t>(H) * W * C * 2};
        const uint32_t box[4] = {64, static_cast<uint32_t>(p.TW * stride), static_cast<uint32_t>(p.TH * stride), static_cast<uint32_t>(p.TN)};
        const uint32_t es[4] = {1, static_cast<uint32_t>(stride), static_cast<uint32_t>(stride), 1};
        return encode_tmap(m, x, 4, dims, strides, box, es);
    };
    auto weight_map = [&](CUtensorMap* m, const void* w, int C, int taps) {
        const uint64_t dims[3] = {static_cast<uint64_t>(C), static_cast<uint64_t>(taps), static_cast<uint64_t>(a.Cout)};
        const uint64_t strides[2] = {static_cast<uint64_t>(C) * 2, static_cast<uint64_t>(taps) * C * 2};
        const uint32_t box[3] = {64, 1, static_cast<uint32_t>(p.BN)};
        const uint32_t es[3] = {1, 1, 1};
        return encode_tmap(m, w, 3, dims, strides, box, es);
    };
    int rc = input_map(&tmx, a.x, a.W, a.H, a.Cin, a.stride);
    if (rc == DLF_OK) rc = weight_map(&tmw, a.w, a.Cin, a.kh * a.kw);
    tmx2 = tmx;
    tmw2 = tmw;
    if (rc == DLF_OK && dual) rc = input_map(&tmx2, a.x2, a.W2, a.H2, a.Cin2, a.stride2);
    if (rc == DLF_OK && dual) rc = weight_map(&tmw2, a.w2, a.Cin2, 1);
    if (rc) return rc;
    const int grid = p.tiles_w * p.tiles_h * tiles_n * p.n_tiles_n * c.split;
    const size_t smem = static_cast<size_t>(p.red_off) + (c.split > 1 ? static_cast<size_t>(c.split) * p.rows_per * p.BN * 4 : 0) + 1024;
    cudaError_t e = launch_kernel(pick_kernel(c.split), grid, kThreads, smem, s, tmx, tmw, tmx2, tmw2, p);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

int conv_lat_init() {
    static bool attr_set[kMaxDevices] = {};
    const int dev = current_device_slot();
    if (dev < 0) return DLF_E_UNSUPPORTED;
    if (!attr_set[dev]) {
        for (int lg = 0; lg <= 3; lg++) {
            cudaError_t e = cudaFuncSetAttribute(pick_kernel(1 << lg), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
            if (e != cudaSuccess) return cuda_fail(e);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1u << lg);
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = kMaxDynSmem;
            int n = 0;
            e = cudaOccupancyMaxActiveClusters(&n, pick_kernel(1 << lg), &cfg);
            if (e != cudaSuccess) return cuda_fail(e);
            g_max_clusters[dev][lg] = n;
        }
        attr_set[dev] = true;
    }
    return DLF_OK;
}

}  // namespace dlf
