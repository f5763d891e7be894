// Pointwise (1x1, stride 1) convolution with at most 64 input channels: a stream of pixels in, a stream out, with so little
// arithmetic per byte that memory is the only bound there should be.  The tcgen05 kernels spend 1700 clocks of hand-overs per
// 128-pixel tile of such a layer (copy, UMMA, tensor memory, staging tile, TMA store), up to five times its bytes' time; here a
// warp multiplies 16 pixels at a time in registers (mma.m16n8k16) and neither shared nor tensor memory is used.
//
// The order of K and of the output channels is free, so both are chosen for wide accesses: in a block of 32 input channels lane
// c of a quad holds channels 8c .. 8c + 7 of its two pixels - one 16-byte load each, and one 16-byte load per weight row -
// and the output channels are dealt out so that a lane ends up with 2 NT neighbouring ones of a pixel.  A warp keeps the weights
// of 32 output channels in registers; the warps of wider layers share their pixels through L1.  Sums in fp32, then bias,
// residual, activation, one rounding.
// Measured: 32 -> 16 at 112x112, batch 64 41.0 -> 12.6 us (its bytes 11.9), 16 -> 96 there 99 -> 38, 24 -> 24 at 96x96, batch 16
// 17.6 -> 4.5, 64 -> 64 at 28x28, batch 8 3.5 -> 3.1.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace dlf {

namespace {

constexpr int kWarps = 8, kWideWarps = 24;   // of a CTA: where the plan gives the layer all SMs / fewer (see launch_conv_narrow)
constexpr int kTiles = 2;   // 16-pixel tiles a warp has in flight

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// KB: blocks of 32 input channels; NT: eights of output channels of a warp (Cout = 8 NT blocks)
template <int KB, int NT, int ACT, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) conv_narrow_kernel(const __half* x, const __half* __restrict__ w, const float* __restrict__ bias,
                                                                   const __half* res, __half* y, int cin, int cout, int blocks, long long pixels) {
    constexpr int kOwn = 2 * NT;   // neighbouring channels of a pixel that a lane finishes
    // The residual is fetched ahead of the sums where there are many of them (64 -> 64 with a residual at seven 28x28 images 3.5 us
    // against 3.9), and where it is added elsewhere (24 -> 24 with one at 16 images of 96x96 4.6 us against 5.1).
    constexpr bool kResEarly = KB == 2;
    const int warp = threadIdx.x >> 5, block = warp % blocks;   // the warp's block of 8 NT output channels; the warps of a CTA that share pixels
    const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    pdl_launch_dependents();
    uint4 wb[KB][NT];
    float2 b2[NT];
#pragma unroll
    for (int t = 0; t < NT; t++) {
        const int co = block * 8 * NT + (g >> 1) * kOwn + 2 * t + (g & 1);   // column g of the t-th eight
#pragma unroll
        for (int kb = 0; kb < KB; kb++) {
            const int ci = kb * 32 + c * 8;
            wb[kb][t] = ci < cin ? __ldg(reinterpret_cast<const uint4*>(w + co * cin + ci)) : make_uint4(0u, 0u, 0u, 0u);
        }
        b2[t] = make_float2(__ldg(bias + block * 8 * NT + c * kOwn + 2 * t), __ldg(bias + block * 8 * NT + c * kOwn + 2 * t + 1));
    }
    pdl_wait();
    const int groups = static_cast<int>(blockDim.x >> 5) / blocks;   // pixel groups of the CTA
    const long long step = static_cast<long long>(gridDim.x) * groups * 16 * kTiles;
    for (long long p0 = (static_cast<long long>(blockIdx.x) * groups + warp / blocks) * 16 * kTiles; p0 < pixels; p0 += step) {
        uint4 a[kTiles][KB][2];
#pragma unroll
        for (int m = 0; m < kTiles; m++)
#pragma unroll
            for (int h = 0; h < 2; h++)
#pragma unroll
                for (int kb = 0; kb < KB; kb++) {
                    const long long px = p0 + m * 16 + h * 8 + g;
                    const int ci = kb * 32 + c * 8;
                    a[m][kb][h] = px < pixels && ci < cin ? ld_map(reinterpret_cast<const uint4*>(x + px * cin + ci)) : make_uint4(0u, 0u, 0u, 0u);
                }
#pragma unroll
        for (int m = 0; m < kTiles; m++) {
            [[maybe_unused]] __half2 rv[2][NT];
            if (kResEarly && res) {
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const long long px = p0 + m * 16 + h * 8 + g;
#pragma unroll
                    for (int t = 0; t < NT; t++)
                        rv[h][t] = px < pixels ? ld_map(reinterpret_cast<const __half2*>(res + px * cout + block * 8 * NT + c * kOwn + 2 * t)) : __half2();
                }
            }
            float d[NT][4];
#pragma unroll
            for (int t = 0; t < NT; t++) {
                d[t][0] = d[t][1] = d[t][2] = d[t][3] = 0.0f;
#pragma unroll
                for (int kb = 0; kb < KB; kb++) {
                    const uint4 lo = a[m][kb][0], hi = a[m][kb][1], b = wb[kb][t];
                    mma16816(d[t], lo.x, hi.x, lo.y, hi.y, b.x, b.y);
                    mma16816(d[t], lo.z, hi.z, lo.w, hi.w, b.z, b.w);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const long long px = p0 + m * 16 + h * 8 + g;
                if (px >= pixels) continue;
                const long long at = px * cout + block * 8 * NT + c * kOwn;
                uint32_t out[NT];
#pragma unroll
                for (int t = 0; t < NT; t++) {
                    float v0 = d[t][2 * h] + b2[t].x, v1 = d[t][2 * h + 1] + b2[t].y;
                    if (res) {
                        const float2 r = __half22float2(kResEarly ? rv[h][t] : ld_map(reinterpret_cast<const __half2*>(res + at + 2 * t)));
                        v0 += r.x;
                        v1 += r.y;
                    }
                    out[t] = round_act<ACT>(v0, v1);
                }
                if (NT == 4) {
                    *reinterpret_cast<uint4*>(y + at) = make_uint4(out[0], out[1 % NT], out[2 % NT], out[3 % NT]);
                } else if (NT == 2) {
                    *reinterpret_cast<uint2*>(y + at) = make_uint2(out[0], out[1 % NT]);
                } else {
#pragma unroll
                    for (int t = 0; t < NT; t++) *reinterpret_cast<uint32_t*>(y + at + 2 * t) = out[t];
                }
            }
        }
    }
}

typedef void (*KernelFn)(const __half*, const __half*, const float*, const __half*, __half*, int, int, int, long long);
template <int KB, int NT, int WARPS>
KernelFn pick_act(int act) {
    return act == DLF_ACT_RELU6 ? conv_narrow_kernel<KB, NT, 2, WARPS> : (act == DLF_ACT_RELU ? conv_narrow_kernel<KB, NT, 1, WARPS> : conv_narrow_kernel<KB, NT, 0, WARPS>);
}
template <int KB, int WARPS>
KernelFn pick_nt(int nt, int act) {
    switch (nt) {
        case 1: return pick_act<KB, 1, WARPS>(act);
        case 2: return pick_act<KB, 2, WARPS>(act);
        case 3: return pick_act<KB, 3, WARPS>(act);
        default: return pick_act<KB, 4, WARPS>(act);
    }
}

}  // namespace

int launch_conv_narrow(const ConvArgs& a, int sm_count, cudaStream_t s) {
    if (a.kh != 1 || a.kw != 1 || a.stride != 1 || a.pad != 0 || a.groups != 1 || a.pool || a.x2 || a.Cin % 8 || a.Cin > 64) return DLF_E_UNSUPPORTED;
    if (a.Cout % 8 || (a.Cout > 32 && a.Cout % 32) || a.Cout > 32 * kWarps) return DLF_E_UNSUPPORTED;
    const long long pixels = static_cast<long long>(a.N) * a.H * a.W;
    // With two blocks of input channels this kernel's multiply-adds outweigh its bytes once there is enough work to hide the tcgen05
    // kernel's hand-overs: 64 -> 256 at 9000 / 12500 / 16000 / 37632 pixels 3.2 / 4.6 / 5.3 / 8.6 us against 4.5 / 5.6 / 5.2 / 8.0 there,
    // with a residual 4.2 / 6.2 / 7.3 / 12.1 against 4.9 / 5.9 / 5.9 / 8.8.  Up to 64 output channels it stays ahead at any size (64 -> 64 at
    // 100000 pixels 7.1 against 8.3), but for a residual beside a whole 64-channel chunk (37632 / 50000 / 100000 pixels 4.2 / 6.1 / 9.9
    // against 5.3 / 6.1 / 9.0; 40 -> 64 9.3 against 14.3).  The line in the tens of thousands of pixels is where one round of the grid ends.
    if (a.Cin > 32 && (a.Cout > 64 || (a.Cout == 64 && a.Cin == 64 && a.res)) && pixels * a.Cout > 3000000) return DLF_E_UNSUPPORTED;
    // (and on few pixels the cluster kernel, whose weights are on their way before the layer before it ends: a network's six such
    // layers on one 56x56 image take 2.5 us more here)
    if (a.Cin > 32 && pixels < 5000) return DLF_E_UNSUPPORTED;
    int sms = 0;
    const int rc = query_sms(&sms);
    if (rc) return rc;
    // Four CTAs per SM spread over all SMs that are free, so a plan that gives the layer fewer gets one large CTA for each of them.
    // With two blocks of input channels too few warps fit into one: the tcgen05 kernels are as fast there (64 -> 64 with a residual
    // at 33 images of 56x56 on 74 SMs 13.8 us against 16.3, 64 -> 256 with one at three 6.1 against 7.1).
    const bool wide = sm_count < sms;
    if (wide && a.Cin > 32) return DLF_E_UNSUPPORTED;
    const int ctas_sm = wide ? 1 : 4, blocks = std::max(1, a.Cout / 32), groups = (wide ? kWideWarps : kWarps) / blocks;
    const long long ctas = (pixels + 16 * kTiles * groups - 1) / (16 * kTiles * groups);
    const int grid = static_cast<int>(std::min<long long>(ctas, static_cast<long long>(ctas_sm) * sm_count)), nt = std::min(a.Cout / 8, 4);
    const KernelFn fn = a.Cin > 32 ? pick_nt<2, kWarps>(nt, a.act) : (wide ? pick_nt<1, kWideWarps>(nt, a.act) : pick_nt<1, kWarps>(nt, a.act));
    cudaError_t e = launch_kernel(fn, grid, 32 * blocks * groups, 0, s,
                                  static_cast<const __half*>(a.x), static_cast<const __half*>(a.w), a.bias, static_cast<const __half*>(a.res),
                                  static_cast<__half*>(a.y), a.Cin, a.Cout, blocks, pixels);
    return e == cudaSuccess ? DLF_OK : cuda_fail(e);
}

}  // namespace dlf
