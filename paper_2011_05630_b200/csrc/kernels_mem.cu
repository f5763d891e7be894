// CUDA-core kernels for the layers that are bound by memory traffic or too narrow for the
// tensor cores: direct convolution for tiny channel counts (the C = 3 stems), depthwise 3x3,
// max / global-average pooling and the weight-streaming fully connected layer.  All use 128-bit
// accesses along the channel dimension of the NHWC tensors, fp32 arithmetic and a single
// round-to-nearest-even to fp16 per layer.  Grids are sized from the SM-count knob and loop over
// the work with a grid stride.  Launched like the tensor-core kernels with programmatic dependent launch: a kernel's blocks
// start while its predecessor drains, and wait before they read what it wrote.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "internal.h"
#include "ptx.cuh"

namespace dlf {

namespace {

constexpr int kBlocksPerSm = 8;

inline int grid_for(long long work_blocks, int sm_count) {
    long long cap = static_cast<long long>(sm_count) * kBlocksPerSm;
    long long g = work_blocks < cap ? work_blocks : cap;
    return static_cast<int>(g < 1 ? 1 : g);
}

// ---- direct convolution ---------------------------------------------------------------------------
// One thread = one output pixel (after the optional 2x2 pool) x 16 output channels.  The weights
// of the block's 16 channels are staged in shared memory as fp32, one (tap, 64-channel) slab at
// a time, and read as broadcasts.  Summation order is (kh, kw, ci) ascending in fp32.
constexpr int kDirCo = 16;
constexpr int kDirCi = 64;

__global__ void __launch_bounds__(128) conv_direct_kernel(ConvArgs a, long long n_pix, int co_blocks) {
    __shared__ float wsm[kDirCi][kDirCo];
    pdl_launch_dependents();
    pdl_wait();
    const __half* x = static_cast<const __half*>(a.x);
    const __half* w = static_cast<const __half*>(a.w);
    const __half* res = static_cast<const __half*>(a.res);
    __half* y = static_cast<__half*>(a.y);
    const int win = a.pool ? 2 : 1;
    const int Hp = a.Ho / win, Wp = a.Wo / win;
    const int cg = a.Cin / a.groups, og = a.Cout / a.groups;
    const long long pix_blocks = (n_pix + blockDim.x - 1) / blockDim.x;
    const long long total = pix_blocks * co_blocks;
    for (long long blk = blockIdx.x; blk < total; blk += gridDim.x) {
        const int cb = static_cast<int>(blk % co_blocks);
        const long long p = (blk / co_blocks) * blockDim.x + threadIdx.x;
        const int co0 = cb * kDirCo;
        const int g = co0 / og;  // a block of 16 channels never straddles groups (checked on host)
        const bool live = p < n_pix;
        int n = 0, hp = 0, wp = 0;
        if (live) {
            wp = static_cast<int>(p % Wp);
            hp = static_cast<int>((p / Wp) % Hp);
            n = static_cast<int>(p / (static_cast<long long>(Wp) * Hp));
        }
        float best[kDirCo];
        for (int q = 0; q < win * win; q++) {
            const int ho = hp * win + q / win, wo = wp * win + q % win;
            float acc[kDirCo];
#pragma unroll
            for (int j = 0; j < kDirCo; j++) acc[j] = 0.0f;
            for (int r = 0; r < a.kh; r++) {
                for (int s = 0; s < a.kw; s++) {
                    const int hi = ho * a.stride - a.pad + r, wi = wo * a.stride - a.pad + s;
                    const bool inside = live && hi >= 0 && hi < a.H && wi >= 0 && wi < a.W;
                    const __half* xp = x + ((static_cast<long long>(n) * a.H + hi) * a.W + wi) * a.Cin + g * cg;
                    for (int c0 = 0; c0 < cg; c0 += kDirCi) {
                        const int cn = min(kDirCi, cg - c0);
                        __syncthreads();
                        for (int i = threadIdx.x; i < cn * kDirCo; i += blockDim.x) {
                            const int ci = i / kDirCo, j = i % kDirCo;
                            const int co = co0 + j;
                            wsm[ci][j] = co < a.Cout
                                             ? __half2float(w[((static_cast<long long>(co) * a.kh + r) * a.kw + s) * cg + c0 + ci])
                                             : 0.0f;
                        }
                        __syncthreads();
                        if (inside) {
                            for (int ci = 0; ci < cn; ci++) {
                                const float xv = __half2float(xp[c0 + ci]);
#pragma unroll
                                for (int j = 0; j < kDirCo; j++) acc[j] = fmaf(xv, wsm[ci][j], acc[j]);
                            }
                        }
                    }
                }
            }
            if (live) {
#pragma unroll
                for (int j = 0; j < kDirCo; j++) {
                    const int co = co0 + j;
                    if (co < a.Cout) {
                        float v = acc[j] + a.bias[co];
                        if (res) v += __half2float(res[((static_cast<long long>(n) * a.Ho + ho) * a.Wo + wo) * a.Cout + co]);
                        v = __half2float(__float2half_rn(apply_act(v, a.act)));
                        best[j] = (q == 0) ? v : fmaxf(best[j], v);
                    }
                }
            }
        }
        if (live) {
            __half* yp = y + ((static_cast<long long>(n) * Hp + hp) * Wp + wp) * a.Cout + co0;
#pragma unroll
            for (int j = 0; j < kDirCo; j++)
                if (co0 + j < a.Cout) yp[j] = __float2half_rn(best[j]);
        }
    }
}

// ---- depthwise 3x3 ------------------------------------------------------------------------------------
// One thread = 4 channels x one output column x a strip of output rows, walked from top to bottom: every input row of three
// 8-byte vectors is loaded (three rows ahead) once and joins the up to three output rows it touches through multiply-adds that
// take fp16 factors, so an output costs nine of them and 2 to 3 other instructions (with conversions and fp32 factors the same
// walk took 42.3 us for 112x112x32 at 64 images, now 33.8; 16 are its bytes' time); loading a strip's whole window at once
// (the first version: 8 channels x 4 columns of one row) converted every input 4.5 times.  The thread's 36 weights are fetched
// once, before the wait for the previous kernel (the launch makes the total thread count a multiple of C/4, so a thread keeps
// its channels over the whole grid-stride loop).  Lanes run over the channels first, so a warp reads contiguous NHWC runs.
// fp32 accumulation from the bias on in (kh, kw) order, one rounding.
template <int STRIDE>
__global__ void __launch_bounds__(128) dw3x3_kernel(ConvArgs a, long long total, int strips, int rows_per) {
    const int c4n = a.Cout / 4;
    const long long tid = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    const long long nthreads = static_cast<long long>(gridDim.x) * blockDim.x;
    pdl_launch_dependents();
    if (tid >= total) return;
    const int c0 = static_cast<int>(tid % c4n) * 4;
    unsigned short w[9][4];   // (fp16)
    float bias[4];
    {
        uint2 raw[9];   // weights of channels c0 .. c0 + 3: 36 consecutive halves starting at c0 * 9
        const uint2* wp = reinterpret_cast<const uint2*>(static_cast<const __half*>(a.w) + static_cast<long long>(c0) * 9);
#pragma unroll
        for (int k = 0; k < 9; k++) raw[k] = __ldg(wp + k);
        const unsigned short* wv = reinterpret_cast<const unsigned short*>(raw);
#pragma unroll
        for (int t = 0; t < 9; t++)
#pragma unroll
            for (int j = 0; j < 4; j++) w[t][j] = wv[j * 9 + t];
#pragma unroll
        for (int j = 0; j < 4; j++) bias[j] = __ldg(a.bias + c0 + j);
    }
    pdl_wait();   // (the weights above are constants)
    const __half2 lo = act_lo(a.act), hi = act_hi(a.act);   // applied to rounded pairs
    const __half* res = static_cast<const __half*>(a.res);
    const int in_row = a.W * a.Cin, out_row = a.Wo * a.Cout;
    for (long long i = tid; i < total; i += nthreads) {
        long long q = i / c4n;
        const int wo = static_cast<int>(q % a.Wo);
        q /= a.Wo;
        const int strip = static_cast<int>(q % strips), n = static_cast<int>(q / strips);
        const int ho0 = strip * rows_per, rows = min(rows_per, a.Ho - ho0);
        const int wi = wo * STRIDE - a.pad;
        int hi_ = ho0 * STRIDE - a.pad;   // input row that is fetched next
        const bool ok0 = wi >= 0 && wi < a.W, ok1 = wi + 1 >= 0 && wi + 1 < a.W, ok2 = wi + 2 >= 0 && wi + 2 < a.W;
        const __half* src = static_cast<const __half*>(a.x) + (static_cast<long long>(n) * a.H * a.W + wi) * a.Cin + static_cast<long long>(hi_) * in_row + c0;
        long long off = (static_cast<long long>(n) * a.Ho + ho0) * out_row + static_cast<long long>(wo) * a.Cout + c0;
        uint2 raw[3][3];   // the next three input rows
        int left = rows * STRIDE + 3 - STRIDE;   // rows still to fetch
        auto fetch = [&](int slot) {
            const bool row_ok = hi_ >= 0 && hi_ < a.H && left > 0;
            raw[slot][0] = row_ok && ok0 ? ld_map(reinterpret_cast<const uint2*>(src)) : make_uint2(0u, 0u);
            raw[slot][1] = row_ok && ok1 ? ld_map(reinterpret_cast<const uint2*>(src + a.Cin)) : make_uint2(0u, 0u);
            raw[slot][2] = row_ok && ok2 ? ld_map(reinterpret_cast<const uint2*>(src + 2 * a.Cin)) : make_uint2(0u, 0u);
            left--;
            hi_++;
            src += in_row;
        };
        unsigned short x[3][4];
        auto next = [&](int slot) {
#pragma unroll
            for (int s = 0; s < 3; s++) {
                unpack_h2(raw[slot][s].x, x[s][0], x[s][1]);
                unpack_h2(raw[slot][s].y, x[s][2], x[s][3]);
            }
            fetch(slot);
        };
        auto add = [&](float (&acc)[4], int r) {
#pragma unroll
            for (int s = 0; s < 3; s++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[j] = fma_f32_f16(x[s][j], w[r * 3 + s][j], acc[j]);
        };
        auto start = [&](float (&acc)[4]) {
#pragma unroll
            for (int j = 0; j < 4; j++) acc[j] = bias[j];
            add(acc, 0);
        };
        auto store = [&](float (&acc)[4]) {
            if (res != nullptr) {
                const uint2 rv = ld_map(reinterpret_cast<const uint2*>(res + off));
                const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&rv.x)), f1 = __half22float2(*reinterpret_cast<const __half2*>(&rv.y));
                acc[0] += f0.x; acc[1] += f0.y; acc[2] += f1.x; acc[3] += f1.y;
            }
            uint2 o;
            o.x = pack_half2_clamp(acc[0], acc[1], lo, hi);
            o.y = pack_half2_clamp(acc[2], acc[3], lo, hi);
            *reinterpret_cast<uint2*>(static_cast<__half*>(a.y) + off) = o;
            off += out_row;
        };
        float u[4], v[4], t[4];
        fetch(0);
        fetch(1);
        fetch(2);
        if (STRIDE == 1) {
            // input row j is the last row of output j - 2, the middle one of output j - 1, the first one of output j
            next(0); start(u);
            next(1); add(u, 1); start(v);
            int j = 0;
#pragma unroll 1
            while (true) {
                next(2); add(u, 2); store(u);
                if (++j == rows) break;
                add(v, 1); start(t);
                next(0); add(v, 2); store(v);
                if (++j == rows) break;
                add(t, 1); start(u);
                next(1); add(t, 2); store(t);
                if (++j == rows) break;
                add(u, 1); start(v);
            }
        } else {
            next(0); start(u);
            int j = 0;
#pragma unroll 1
            while (true) {
                next(1); add(u, 1); next(2); add(u, 2); store(u);
                if (++j == rows) break;
                start(u);
                next(0); add(u, 1); next(1); add(u, 2); store(u);
                if (++j == rows) break;
                start(u);
                next(2); add(u, 1); next(0); add(u, 2); store(u);
                if (++j == rows) break;
                start(u);
            }
        }
    }
}

// ---- pooling ----------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) maxpool_kernel(const __half* x, __half* y, int N, int H, int W, int C, int k,
                                                      int stride, int pad, int Ho, int Wo, long long total) {
    const int c8n = C / 8;
    pdl_launch_dependents();
    pdl_wait();
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int c8 = static_cast<int>(i % c8n);
        long long p = i / c8n;
        const int wo = static_cast<int>(p % Wo);
        p /= Wo;
        const int ho = static_cast<int>(p % Ho);
        const int n = static_cast<int>(p / Ho);
        __half2 best[4];
        const __half2 ninf = __half2half2(__ushort_as_half(0xFC00));
#pragma unroll
        for (int j = 0; j < 4; j++) best[j] = ninf;
        // clamped taps instead of skipped ones: a tap outside the image re-reads an in-range pixel of the
        // same window (the maximum is unchanged) and the loads carry no branches, so they overlap
        const int h_lo = max(ho * stride - pad, 0), h_hi = min(ho * stride - pad + k - 1, H - 1);
        const int w_lo = max(wo * stride - pad, 0), w_hi = min(wo * stride - pad + k - 1, W - 1);
        for (int r = 0; r < k; r++) {
            const int hi = min(max(ho * stride - pad + r, h_lo), h_hi);
#pragma unroll 3
            for (int s = 0; s < k; s++) {
                const int wi = min(max(wo * stride - pad + s, w_lo), w_hi);
                const uint4 v = ld_map(reinterpret_cast<const uint4*>(x + ((static_cast<long long>(n) * H + hi) * W + wi) * C + c8 * 8));
                const __half2* vh = reinterpret_cast<const __half2*>(&v);
#pragma unroll
                for (int j = 0; j < 4; j++) best[j] = __hmax2(best[j], vh[j]);
            }
        }
        *reinterpret_cast<uint4*>(y + ((static_cast<long long>(n) * Ho + ho) * Wo + wo) * C + c8 * 8) =
            *reinterpret_cast<uint4*>(best);
    }
}

// Mean over (h, w): fp32 sums, one rounding.  A block takes 8 channel vectors (128 contiguous bytes of a pixel) of one image
// and shares the pixels out over 32 groups of threads, whose sums are added in a fixed order; with one thread walking all
// pixels of its vector the kernel waited for one load after another (2048 channels at 7x7, one image 6.2 us in a network, now
// 2.4 us).
constexpr int kAvgVecs = 8, kAvgParts = 32;
__global__ void __launch_bounds__(kAvgVecs * kAvgParts) gavgpool_kernel(const __half* x, __half* y, int HW, int C, int vec_blocks, int total) {
    __shared__ float part[kAvgParts][kAvgVecs * 8 + 4];
    const int v = threadIdx.x % kAvgVecs, q = threadIdx.x / kAvgVecs;
    const float inv = 1.0f / static_cast<float>(HW);
    pdl_launch_dependents();
    pdl_wait();
    for (int blk = blockIdx.x; blk < total; blk += gridDim.x) {
        const int n = blk / vec_blocks, c8 = (blk - n * vec_blocks) * kAvgVecs + v;
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; j++) acc[j] = 0.0f;
        if (c8 * 8 < C) {
            const __half* xp = x + static_cast<long long>(n) * HW * C + c8 * 8;
#pragma unroll 4
            for (int p = q; p < HW; p += kAvgParts) {
                const uint4 u = ld_map(reinterpret_cast<const uint4*>(xp + static_cast<long long>(p) * C));
                const __half* vh = reinterpret_cast<const __half*>(&u);
#pragma unroll
                for (int j = 0; j < 8; j++) acc[j] += __half2float(vh[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < 8; j++) part[q][v * 8 + j] = acc[j];
        __syncthreads();
        if (threadIdx.x < kAvgVecs * 8) {   // one thread per channel
            float sum = 0.0f;
#pragma unroll 8
            for (int k = 0; k < kAvgParts; k++) sum += part[k][threadIdx.x];
            const int c = (blk - n * vec_blocks) * kAvgVecs * 8 + threadIdx.x;
            if (c < C) y[static_cast<long long>(n) * C + c] = __float2half_rn(sum * inv);
        }
        __syncthreads();
    }
}

// ---- fully connected --------------------------------------------------------------------------------------
// A block owns 8 output features and streams their weight rows once per batch tile of NB images; threads stride over K in 128-bit
// pieces, accumulate 8 x NB partial sums in fp32, then reduce.  Bound by latencies: the first weights are on their way before the wait
// for the previous kernel, the next ones while the present ones are worked on, one image pays for one (64 sums of eight images
// were 320 shuffles a thread whatever the batch), and a warp's sums are exchanged in halves.  2048 -> 1000 at one image 5.15 -> 3.1 us,
// at six 5.15 -> 4.1; 4096 -> 1000 at eight 6.7 -> 5.7.
constexpr int kFcFo = 8;

template <int NB>
__global__ void __launch_bounds__(256) fc_kernel(const __half* x, const __half* w, const float* bias, __half* y, int N,
                                                 int K, int M, int act, int o_blocks, int n_blocks) {
    __shared__ float red[8][kFcFo * NB];
    const int k8n = K / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 wv[kFcFo];
    auto load_w = [&](int blk, int k8) {
        const int o0 = (blk % o_blocks) * kFcFo;
#pragma unroll
        for (int i = 0; i < kFcFo; i++) {
            const int o = min(o0 + i, M - 1);
            wv[i] = __ldcs(reinterpret_cast<const uint4*>(w + static_cast<long long>(o) * K) + k8);
        }
    };
    pdl_launch_dependents();
    if (static_cast<int>(threadIdx.x) < k8n && static_cast<int>(blockIdx.x) < o_blocks * n_blocks) load_w(blockIdx.x, threadIdx.x);   // (constants)
    pdl_wait();
    for (int blk = blockIdx.x; blk < o_blocks * n_blocks; blk += gridDim.x) {
        const int o0 = (blk % o_blocks) * kFcFo, n0 = (blk / o_blocks) * NB;
        float acc[kFcFo][NB];
#pragma unroll
        for (int i = 0; i < kFcFo; i++)
#pragma unroll
            for (int j = 0; j < NB; j++) acc[i][j] = 0.0f;
        for (int k8 = threadIdx.x; k8 < k8n; k8 += blockDim.x) {
            uint4 xv[NB], wc[kFcFo];
            auto next_w = [&]() {
                if (k8 + static_cast<int>(blockDim.x) < k8n) load_w(blk, k8 + blockDim.x);
                else if (blk + static_cast<int>(gridDim.x) < o_blocks * n_blocks) load_w(blk + gridDim.x, threadIdx.x);
            };
#pragma unroll
            for (int j = 0; j < NB; j++) {
                const int n = min(n0 + j, N - 1);
                xv[j] = ld_map(reinterpret_cast<const uint4*>(x + static_cast<long long>(n) * K) + k8);
            }
#pragma unroll
            for (int i = 0; i < kFcFo; i++) wc[i] = wv[i];
            if (NB <= 2) next_w();   // (more images leave no registers for it)
#pragma unroll
            for (int e = 0; e < 4; e++) {
                float2 xf[NB];
#pragma unroll
                for (int j = 0; j < NB; j++) xf[j] = __half22float2(reinterpret_cast<const __half2*>(&xv[j])[e]);
#pragma unroll
                for (int i = 0; i < kFcFo; i++) {
                    const float2 wf = __half22float2(reinterpret_cast<const __half2*>(&wc[i])[e]);
#pragma unroll
                    for (int j = 0; j < NB; j++) {
                        acc[i][j] = fmaf(wf.x, xf[j].x, acc[i][j]);
                        acc[i][j] = fmaf(wf.y, xf[j].y, acc[i][j]);
                    }
                }
            }
            if (NB > 2) next_w();
        }
        // A warp's sums: at every step of the exchange a lane keeps half of its values and sends the other half (64 values in 62 shuffles, the
        // same tree as a sum of each by itself in 320); in the end lane l holds values `at`, at + 1, ...
        float v[kFcFo * NB];
#pragma unroll
        for (int i = 0; i < kFcFo * NB; i++) v[i] = acc[i / NB][i % NB];
        int at = 0;
        constexpr int kLeft = kFcFo * NB > 32 ? kFcFo * NB / 32 : 1;   // values of a lane in the end
#pragma unroll
        for (int d = 16, n = kFcFo * NB / 2; d > 0; d >>= 1, n >>= 1) {
            if (n > 0) {
                const bool up = (lane & d) != 0;
#pragma unroll
                for (int i = 0; i < n; i++) {
                    const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
                }
                at += up ? n : 0;
            } else {
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);   // (fewer values than lanes: the last steps add what is there)
            }
        }
#pragma unroll
        for (int i = 0; i < kLeft; i++) red[warp][at + i] = v[i];   // (lanes that hold the same value write the same)
        __syncthreads();
        if (threadIdx.x < kFcFo * NB) {
            float v = 0.0f;
            for (int wq = 0; wq < 8; wq++) v += red[wq][threadIdx.x];
            const int o = o0 + threadIdx.x / NB, n = n0 + threadIdx.x % NB;
            if (o < M && n < N) y[static_cast<long long>(n) * M + o] = __float2half_rn(apply_act(v + bias[o], act));
        }
        __syncthreads();
    }
}

}  // namespace

int launch_conv_direct(const ConvArgs& a, int sm_count, cudaStream_t s) {
    const int og = a.Cout / a.groups;
    if (a.groups > 1 && og % kDirCo != 0) return DLF_E_UNSUPPORTED;
    const int win = a.pool ? 2 : 1;
    const long long n_pix = static_cast<long long>(a.N) * (a.Ho / win) * (a.Wo / win);
    const int co_blocks = (a.Cout + kDirCo - 1) / kDirCo;
    const long long blocks = (n_pix + 127) / 128 * co_blocks;
    if (blocks == 0) return DLF_OK;
    cudaError_t e = launch_kernel(conv_direct_kernel, grid_for(blocks, sm_count), 128, 0, s, a, n_pix, co_blocks);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

int launch_dw3x3(const ConvArgs& a, int sm_count, cudaStream_t s) {
    if (a.kh != 3 || a.kw != 3 || a.groups != a.Cin || a.Cin != a.Cout || a.Cin % 8 || a.pool) return DLF_E_UNSUPPORTED;
    if (a.stride != 1 && a.stride != 2) return DLF_E_UNSUPPORTED;
    if (!aligned(8, a.x, a.res, a.y)) return DLF_E_INVALID_ARG;
    const int c4n = a.Cout / 4;
    static int occ[2] = {0, 0};
    const int v = a.stride == 1 ? 0 : 1;
    if (occ[v] == 0) {
        int n = 0;
        cudaError_t e = v == 0 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dw3x3_kernel<1>, 128, 0)
                               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dw3x3_kernel<2>, 128, 0);
        occ[v] = e != cudaSuccess || n < 1 ? 2 : n;
    }
    // Rows of a strip: long strips load few rows twice, short ones keep all SMs busy on a small map.  A thread's walk costs about
    // 700 clocks per input row at full occupancy (the latency of its loads; about four rows' worth before the first); the cost
    // of a strip length is that times the rounds of the grid, a last round that is not full counting a quarter less.  (Against
    // the longest strip throughout: 96 channels stride 2 at 112x112, batch 64 68 -> 51 us; 24 channels at 51x37, batch 30 6.8 -> 4.3.)
    const long long columns = static_cast<long long>(a.N) * a.Wo * c4n;
    int rows_per = 1;
    double best = -1.0;
    for (int r = 1; r <= a.Ho; r++) {
        const int strips = (a.Ho + r - 1) / r;
        if ((strips - 1) * r >= a.Ho) continue;
        const double threads = static_cast<double>(columns) * strips, rows_in = r * a.stride + 3 - a.stride;
        const double rounds = threads / (static_cast<double>(sm_count) * occ[v] * 128);
        const double cost = (0.75 * std::ceil(rounds) + 0.25 * rounds) * (rows_in + 4.0);
        if (best < 0 || cost < best) {
            best = cost;
            rows_per = r;
        }
    }
    const int strips = (a.Ho + rows_per - 1) / rows_per;
    const long long total = columns * strips;
    if (total == 0) return DLF_OK;
    // the total thread count is a multiple of C/4: a thread keeps its channels (and its weights)
    int step = c4n;
    for (int d = 2; d <= 128; d *= 2)
        if (step % 2 == 0) step /= 2;  // blocks needed for (blocks * 128) % c4n == 0: c4n / gcd(c4n, 128)
    // one resident wave of blocks: a thread fetches its weights once and then walks its strips
    long long blocks = std::min<long long>((total + 127) / 128, static_cast<long long>(sm_count) * occ[v]);
    blocks = std::max<long long>(step, blocks / step * step);
    cudaError_t e = launch_kernel(a.stride == 1 ? dw3x3_kernel<1> : dw3x3_kernel<2>, static_cast<int>(blocks), 128, 0, s, a, total, strips, rows_per);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

int launch_maxpool(const void* x, void* y, int N, int H, int W, int C, int k, int stride, int pad, int Ho, int Wo,
                   int sm_count, cudaStream_t s) {
    if (C % 8) return DLF_E_UNSUPPORTED;
    if (!aligned(16, x, y)) return DLF_E_INVALID_ARG;
    const long long total = static_cast<long long>(N) * Ho * Wo * (C / 8);
    if (total == 0) return DLF_OK;
    cudaError_t e = launch_kernel(maxpool_kernel, grid_for((total + 255) / 256, sm_count), 256, 0, s, static_cast<const __half*>(x),
                                  static_cast<__half*>(y), N, H, W, C, k, stride, pad, Ho, Wo, total);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

int launch_gavgpool(const void* x, void* y, int N, int H, int W, int C, int sm_count, cudaStream_t s) {
    if (C % 8) return DLF_E_UNSUPPORTED;
    if (!aligned(16, x)) return DLF_E_INVALID_ARG;
    const int vec_blocks = (C / 8 + kAvgVecs - 1) / kAvgVecs;
    const long long total = static_cast<long long>(N) * vec_blocks;
    if (total == 0) return DLF_OK;
    if (total > 0x7fffffffLL) return DLF_E_UNSUPPORTED;
    cudaError_t e = launch_kernel(gavgpool_kernel, grid_for(total, sm_count), kAvgVecs * kAvgParts, 0, s, static_cast<const __half*>(x),
                                  static_cast<__half*>(y), H * W, C, vec_blocks, static_cast<int>(total));
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

int launch_fc(const void* x, const void* w, const float* bias, void* y, int N, int K, int M, int act, int sm_count,
              cudaStream_t s) {
    if (K % 8) return DLF_E_UNSUPPORTED;
    if (!aligned(16, x)) return DLF_E_INVALID_ARG;
    if (N == 0) return DLF_OK;
    const int nb = N == 1 ? 1 : (N <= 2 ? 2 : (N <= 4 ? 4 : 8));
    const int o_blocks = (M + kFcFo - 1) / kFcFo, n_blocks = (N + nb - 1) / nb;
    const int grid = grid_for(static_cast<long long>(o_blocks) * n_blocks, sm_count);
    auto* const kernel = nb == 1 ? fc_kernel<1> : (nb == 2 ? fc_kernel<2> : (nb == 4 ? fc_kernel<4> : fc_kernel<8>));
    cudaError_t e = launch_kernel(kernel, grid, 256, 0, s, static_cast<const __half*>(x), static_cast<const __half*>(w), bias,
                                  static_cast<__half*>(y), N, K, M, act, o_blocks, n_blocks);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

// Self-test of the bounded waits: one CTA waits, with the waits' own routine, at a barrier that nothing ever arrives at.
// The wait has to give up after `limit_ns`, record its code in the status word and let the kernel end normally.
__global__ void stall_kernel(int* status, unsigned long long limit_ns) {
    __shared__ uint64_t bar;
    __shared__ int abort_s;
    if (threadIdx.x == 0) {
        abort_s = 0;
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    mbar_wait(&bar, 0u, &abort_s, status, 0xd00, limit_ns);
}

int launch_stall(int* status_dev, unsigned long long limit_ns, cudaStream_t s) {
    stall_kernel<<<1, 64, 0, s>>>(status_dev, limit_ns);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

}  // namespace dlf
