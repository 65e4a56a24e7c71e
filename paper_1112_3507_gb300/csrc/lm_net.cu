// The learned warm start / preconditioner network: a 4-level U-Net on NHWC
// images with BF16 activations and weights, FP32 accumulation and FP32
// master weights, trained by Adam.  Every layer's forward and backward pass
// is a kernel here; the host code only sequences them.
//
//   encoder l = 0..3: e_l = relu(conv3(relu(conv3(in_l, A_l)), B_l)),
//                     in_0 = input (3 channels), in_l = avgpool2(e_{l-1})
//   decoder l = 2..0: d_l = relu(conv3(relu(conv3(cat(up2(d_{l+1}), e_l), C_l)), D_l)),
//                     d_3 = e_3
//   output:           y = conv1(d_0, O)
//
// Parameters are stored in one FP32 array in the order A0 a0 B0 b0 ... A3 a3
// B3 b3 C2 c2 D2 d2 C1 c1 D1 d1 C0 c0 D0 d0 O o, conv weights laid out
// [dy][dx][Cin][Cout], so that a host can exchange them with any reference.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/lowmach.h"
#include "lm_common.cuh"
#include "lm_internal.h"
#include "lm_kernels.h"

typedef __nv_bfloat16 bf16;

namespace lm {

constexpr int CT = 16;   // pixel tile edge and channel chunk of the convolution kernels

// ---- 3x3 convolution (forward; backward-data with transposed weights) ----
// out[b,y,x,co] = bias[co] + sum_{dy,dx,ci} in[b, y+dy-1, x+dx-1, ci] W[dy,dx,ci,co]
// Block: a 16x16 pixel tile and a chunk of 16 output channels; the input is
// staged through shared memory 16 channels at a time with a 1-pixel halo
// (zero outside the image).  Each thread accumulates 16 outputs in FP32.
template <typename TI, typename TO>
__global__ void __launch_bounds__(256) k_conv3(const TI* __restrict__ in, int Cin, const bf16* __restrict__ W,
                                               const float* __restrict__ bias, TO* __restrict__ out, int Cout,
                                               int H, int Wd, int relu, int ncoc) {
    __shared__ float xs[CT + 2][CT + 2][CT];
    __shared__ __align__(16) float ws[9][CT][CT];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + CT * ty;
    const int b = blockIdx.z / ncoc, coc = blockIdx.z % ncoc;
    const int x0 = blockIdx.x * CT, y0 = blockIdx.y * CT;
    const int co0 = coc * CT;
    float acc[CT];
#pragma unroll
    for (int c = 0; c < CT; ++c) acc[c] = 0.f;
    const TI* inb = in + (size_t)b * H * Wd * Cin;
    for (int ci0 = 0; ci0 < Cin; ci0 += CT) {
        const int nci = min(CT, Cin - ci0);
        for (int e = tid; e < (CT + 2) * (CT + 2) * CT; e += 256) {
            const int c = e % CT, px = (e / CT) % (CT + 2), py = e / (CT * (CT + 2));
            const int gy = y0 + py - 1, gx = x0 + px - 1;
            float v = 0.f;
            if (c < nci && gy >= 0 && gy < H && gx >= 0 && gx < Wd) v = (float)inb[((size_t)gy * Wd + gx) * Cin + ci0 + c];
            xs[py][px][c] = v;
        }
        for (int e = tid; e < 9 * CT * CT; e += 256) {
            const int co = e % CT, ci = (e / CT) % CT, t = e / (CT * CT);
            float v = 0.f;
            if (ci < nci && co0 + co < Cout) v = __bfloat162float(W[((size_t)t * Cin + ci0 + ci) * Cout + co0 + co]);
            ws[t][ci][co] = v;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int dy = t / 3, dx = t % 3;
#pragma unroll 4
            for (int ci = 0; ci < CT; ++ci) {
                const float v = xs[ty + dy][tx + dx][ci];
                const float4* w4 = reinterpret_cast<const float4*>(&ws[t][ci][0]);
#pragma unroll
                for (int q = 0; q < CT / 4; ++q) {
                    const float4 w = w4[q];
                    acc[4 * q + 0] = fmaf(v, w.x, acc[4 * q + 0]);
                    acc[4 * q + 1] = fmaf(v, w.y, acc[4 * q + 1]);
                    acc[4 * q + 2] = fmaf(v, w.z, acc[4 * q + 2]);
                    acc[4 * q + 3] = fmaf(v, w.w, acc[4 * q + 3]);
                }
            }
        }
        __syncthreads();
    }
    const int gy = y0 + ty, gx = x0 + tx;
    if (gy >= H || gx >= Wd) return;
    TO* o = out + (((size_t)b * H + gy) * Wd + gx) * Cout + co0;
#pragma unroll
    for (int c = 0; c < CT; ++c) {
        if (co0 + c >= Cout) break;
        float v = acc[c] + (bias ? bias[co0 + c] : 0.f);
        if (relu) v = fmaxf(v, 0.f);
        if constexpr (sizeof(TO) == 2) o[c] = __float2bfloat16(v);
        else o[c] = v;
    }
}

// ---- 3x3 convolution on the tensor cores ----------------------------------------
// The convolution as an implicit GEMM: M = pixels, N = output channels, K =
// 9 taps x input channels.  Block: a tile of 16 x 8R pixels, warp w owning R
// pixel rows (R m16 tiles) and all NCB output channels (NCB/8 n8 tiles); K
// runs over chunks of 16 input channels and, within a chunk, the 9 taps.
// mma.sync m16n8k16, BF16 operands, FP32 accumulation; fragments by ldmatrix
// from rows of 16 channels at a 48-byte pitch (eight rows in distinct banks).
//
// With 16 to 112 input and 16 to 64 output channels a block's time is the
// chain of its chunks, so both operands of the next chunk are on their way
// while one is multiplied (two shared-memory buffers, one barrier a chunk):
// the pixels through registers, 16 bytes a load, the weights by cp.async from
// a copy laid out as the tile wants them (k_prep_weights).  Element-wise
// staging with the weights transposed on the way, and no overlap, took 0.94 ms
// for the 14 layers of 16 images of 256^2 against 0.37 ms here; a whole
// inference of one image 0.28 ms against 0.14 ms.
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}
__device__ __forceinline__ void ldmatrix2(uint32_t (&r)[2], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void ldmatrix4t(uint32_t (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

constexpr int CPITCH = 24;                          // elements of a staged row of 16 channels
constexpr int CROW = 2 * CPITCH;                    // its bytes
template <int NCB, bool SPLIT, int R>
constexpr size_t conv_smem() {
    return 2 * ((SPLIT ? 2 : 1) * (8 * R + 2) * 18 + 9 * NCB) * (size_t)CROW;
}

// NCB output channels per block (blockIdx.z = image x channel chunk), of
// Cout in all; Wp: the weights as k_prep_weights lays them out.  SPLIT =
// false: BF16 input, BF16 output with bias and ReLU (the forward pass).
// SPLIT = true: float32 input split into a BF16 high part and a BF16
// remainder, two products per fragment (about 16 mantissa bits of the input
// reach the FP32 accumulator), float32 output with neither bias nor ReLU (the
// backward-data pass of float32 gradients).
template <int NCB, bool SPLIT, int R>
__global__ void __launch_bounds__(256) k_conv3_mma(const void* __restrict__ in_, int Cin, const bf16* __restrict__ Wp,
                                                   const float* __restrict__ bias, void* __restrict__ out_, int Cout,
                                                   int H, int Wd, int relu) {
    constexpr int TXP = 16, TYP = 8 * R, PX = TXP + 2, PY = TYP + 2, NPIX = PX * PY;
    constexpr int XB = (SPLIT ? 2 : 1) * NPIX * CROW, WB = 9 * NCB * CROW;   // bytes of a buffer
    constexpr int QX = (2 * NPIX + 255) / 256;                               // half rows (8 channels) a thread stages
    constexpr int LO = NPIX * CROW;                                          // the remainder tile
    extern __shared__ __align__(16) unsigned char csm[];
    const unsigned xs0 = (unsigned)__cvta_generic_to_shared(csm), ws0 = xs0 + 2 * XB;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nch = Cout / NCB;
    const int b = blockIdx.z / nch, co0 = (blockIdx.z % nch) * NCB;
    const int x0 = blockIdx.x * TXP, y0 = blockIdx.y * TYP;
    const int nk = (Cin + 15) / 16;
    // this thread's half rows: the pixel (NONE: outside the image), position
    constexpr unsigned NONE = ~0u;
    unsigned src[QX];
    int dst[QX];
    const int half = tid & 1;
#pragma unroll
    for (int q = 0; q < QX; ++q) {
        const int e = tid + 256 * q, pix = e >> 1, py = pix / PX, px = pix - py * PX;
        const int gy = y0 + py - 1, gx = x0 + px - 1;
        dst[q] = e < 2 * NPIX ? pix * CROW + half * 16 : -1;
        src[q] = dst[q] >= 0 && gy >= 0 && gy < H && gx >= 0 && gx < Wd ? (unsigned)gy * Wd + gx : NONE;
    }
    const size_t img = (size_t)b * H * Wd * Cin;
    constexpr int NV = SPLIT ? 2 : 1;
    uint4 v[QX][NV];                                // the next chunk's pixels: 8 channels, BF16 or float32
    auto load_x = [&](int c) {
#pragma unroll
        for (int q = 0; q < QX; ++q) {
#pragma unroll
            for (int u = 0; u < NV; ++u) v[q][u] = make_uint4(0, 0, 0, 0);
            if (src[q] == NONE) continue;
            const int ci = 16 * c + 8 * half;
            const size_t at = img + (size_t)src[q] * Cin + ci;
            if (Cin % 8 == 0) {
                if (ci < Cin)
#pragma unroll
                    for (int u = 0; u < NV; ++u)
                        v[q][u] = __ldg(SPLIT ? reinterpret_cast<const uint4*>(static_cast<const float*>(in_) + at) + u
                                              : reinterpret_cast<const uint4*>(static_cast<const bf16*>(in_) + at));
            } else {                                // few or odd channels (the network's input): one by one
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (ci + k < Cin) {
                        if (SPLIT) reinterpret_cast<float*>(&v[q][0])[k] = static_cast<const float*>(in_)[at + k];
                        else reinterpret_cast<bf16*>(&v[q][0])[k] = static_cast<const bf16*>(in_)[at + k];
                    }
            }
        }
    };
    auto store_x = [&](int buf) {
#pragma unroll
        for (int q = 0; q < QX; ++q) {
            if (dst[q] < 0) continue;
            unsigned char* const o = csm + buf * XB + dst[q];
            if (SPLIT) {
                uint4 hi, lo;
                bf16* const h = reinterpret_cast<bf16*>(&hi);
                bf16* const l = reinterpret_cast<bf16*>(&lo);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float f = reinterpret_cast<const float*>(&v[q][0])[k];
                    h[k] = __float2bfloat16(f);
                    l[k] = __float2bfloat16(f - __bfloat162float(h[k]));
                }
                *reinterpret_cast<uint4*>(o) = hi;
                *reinterpret_cast<uint4*>(o + LO) = lo;
            } else {
                *reinterpret_cast<uint4*>(o) = v[q][0];
            }
        }
    };
    auto load_w = [&](int c, int buf) {             // rows co0 .. co0 + NCB - 1 of every tap of the chunk
        const bf16* const w = Wp + ((size_t)c * 9 * Cout + co0) * 16;
        for (int e = tid; e < 9 * NCB * 2; e += 256) {
            const int r = e >> 1, t = r / NCB, co = r - t * NCB;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(ws0 + buf * WB + r * CROW + (e & 1) * 16),
                         "l"(w + ((size_t)t * Cout + co) * 16 + (e & 1) * 8)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[R][NCB / 8][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NCB / 8; ++n) acc[r][n][0] = acc[r][n][1] = acc[r][n][2] = acc[r][n][3] = 0.f;
    // fragment rows of this lane: A, pixel (lane & 15) and channel half
    // (lane >> 4); B, four 8 x 8 blocks (channel half, then output octet)
    const unsigned aoff = ((R * warp) * PX + (lane & 15)) * CROW + (lane >> 4) * 16;
    const unsigned boff = ((lane & 7) + (lane >> 4) * 8) * CROW + ((lane >> 3) & 1) * 16;
    load_x(0);
    load_w(0, 0);
    for (int c = 0; c < nk; ++c) {
        const int buf = c & 1;
        store_x(buf);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (c + 1 < nk) {
            load_x(c + 1);
            load_w(c + 1, buf ^ 1);
        }
        const unsigned xa = xs0 + buf * XB + aoff, wa = ws0 + buf * WB + boff;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            uint32_t a[R][4], al[R][4];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const unsigned p = xa + ((r + t / 3) * PX + t % 3) * CROW;
                ldmatrix4(a[r], p);
                if (SPLIT) ldmatrix4(al[r], p + LO);
            }
#pragma unroll
            for (int n = 0; n < NCB / 8; n += 2) {
                uint32_t w[4];
                if (n + 1 < NCB / 8) {
                    ldmatrix4(w, wa + (t * NCB + n * 8) * CROW);
                } else {                            // an odd octet: lanes 0-15 address its two blocks
                    uint32_t w2[2];
                    ldmatrix2(w2, wa + (t * NCB + n * 8) * CROW - (lane >> 4) * 8 * CROW);
                    w[0] = w2[0], w[1] = w2[1];
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        if (n + m >= NCB / 8) continue;
                        mma_bf16_16816(acc[r][n + m], a[r][0], a[r][1], a[r][2], a[r][3], w[2 * m], w[2 * m + 1]);
                        if (SPLIT)
                            mma_bf16_16816(acc[r][n + m], al[r][0], al[r][1], al[r][2], al[r][3], w[2 * m],
                                           w[2 * m + 1]);
                    }
            }
        }
    }
    const int g = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int gy = y0 + R * warp + r;
        if (gy >= H) continue;
#pragma unroll
        for (int n = 0; n < NCB / 8; ++n) {
            const int co = co0 + n * 8 + 2 * tq;
            const float bb0 = (!SPLIT && bias) ? bias[co] : 0.f, bb1 = (!SPLIT && bias) ? bias[co + 1] : 0.f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {                        // pixel g (c0, c1), pixel g + 8 (c2, c3)
                const int gx = x0 + g + 8 * h;
                if (gx >= Wd) continue;
                float v0 = acc[r][n][2 * h] + bb0, v1 = acc[r][n][2 * h + 1] + bb1;
                const size_t o = (((size_t)b * H + gy) * Wd + gx) * Cout + co;
                if (SPLIT) {
                    *reinterpret_cast<float2*>(static_cast<float*>(out_) + o) = make_float2(v0, v1);
                } else {
                    if (relu) {
                        v0 = fmaxf(v0, 0.f);
                        v1 = fmaxf(v1, 0.f);
                    }
                    __nv_bfloat162 pr;
                    pr.x = __float2bfloat16(v0);
                    pr.y = __float2bfloat16(v1);
                    *reinterpret_cast<__nv_bfloat162*>(static_cast<bf16*>(out_) + o) = pr;
                }
            }
        }
    }
}

template <int NCB, bool SPLIT, int R>
void conv3_launch(const void* in, int Cin, const bf16* Wp, const float* bias, void* out, int Cout, int B, int H, int Wd,
                  int relu, cudaStream_t s) {
    constexpr size_t sm = conv_smem<NCB, SPLIT, R>();      // raised above 48 KB by conv3_allow_smem
    const dim3 grd((Wd + 15) / 16, (H + 8 * R - 1) / (8 * R), B * (Cout / NCB));
    k_conv3_mma<NCB, SPLIT, R><<<grd, 256, sm, s>>>(in, Cin, Wp, bias, out, Cout, H, Wd, relu);
}

template <int NCB, int R>
void conv3_allow() {
    cudaFuncSetAttribute(k_conv3_mma<NCB, false, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)conv_smem<NCB, false, R>());
    cudaFuncSetAttribute(k_conv3_mma<NCB, true, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)conv_smem<NCB, true, R>());
}
void conv3_allow_smem() {
    conv3_allow<8, 1>();
    conv3_allow<8, 2>();
    conv3_allow<16, 1>();
    conv3_allow<16, 2>();
    conv3_allow<32, 1>();
    conv3_allow<32, 2>();
    conv3_allow<40, 1>();
    conv3_allow<48, 1>();
    conv3_allow<56, 1>();
    conv3_allow<64, 1>();
}

// launch the tensor-core convolution for Cout output channels; false when
// Cout has no supported channel chunk (the caller uses the FP32 kernel).
// Output channels a block: the most that divide Cout, for the fewest
// re-readings of a pixel tile; with fewer than two blocks an SM then, the most
// that give two (a block's chain is as long with 8 channels as with 64).  Two
// pixel rows a warp halve the weight fragments' loads where four blocks an SM
// remain.
template <bool SPLIT>
bool conv3_mma(const void* in, int Cin, const bf16* Wp, const float* bias, void* out, int Cout, int B, int H, int Wd,
               int relu, cudaStream_t s) {
    const long long tiles = (long long)B * ((Wd + 15) / 16) * ((H + 7) / 8);
    int ncb = 0;
    for (int c : {64, 56, 48, 40, 32, 16, 8})
        if (Cout % c == 0) {
            ncb = c;
            if (tiles * (Cout / c) >= 2 * 152) break;
        }
    if (!ncb) return false;
    const bool two = ncb <= 32 && tiles * (Cout / ncb) >= 8 * 152;
#define LM_CONV(N)                                                                                     \
    case N:                                                                                            \
        if (two) conv3_launch<N, SPLIT, (N <= 32 ? 2 : 1)>(in, Cin, Wp, bias, out, Cout, B, H, Wd, relu, s); \
        else conv3_launch<N, SPLIT, 1>(in, Cin, Wp, bias, out, Cout, B, H, Wd, relu, s);               \
        break;
    switch (ncb) {
        LM_CONV(64)
        LM_CONV(56)
        LM_CONV(48)
        LM_CONV(40)
        LM_CONV(32)
        LM_CONV(16)
        LM_CONV(8)
    }
#undef LM_CONV
    return true;
}

// The weights' derived layouts, all layers in one launch, formed by the calls
// that change the weights, on their stream, so that a forward or backward pass
// captured in a graph reads the weights of the time it is replayed:
//   wt[t][co][ci] = w[8 - t][ci][co]: the backward-data convolution is a
//     forward convolution of the output gradient with these weights;
//   wp[c][t][co][16]: input channels 16 c .. 16 c + 15 (zero past the last) of
//     each output channel, the rows a tensor-core tile stages; wpt likewise of wt.
struct PrepConv {
    int cin, cout, w;               // channels, offset of w and wt
    int p, pt;                      // offsets of wp and wpt
};
struct PrepTable {
    PrepConv c[14];
};
__global__ void k_prep_weights(PrepTable T, const bf16* __restrict__ w, bf16* __restrict__ wt, bf16* __restrict__ wp,
                               bf16* __restrict__ wpt) {
    const PrepConv c = T.c[blockIdx.y];
    const int n = 9 * c.cin * c.cout, stride = gridDim.x * blockDim.x, e0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int e = e0; e < n; e += stride) {
        const int co = e % c.cout, ci = (e / c.cout) % c.cin, t = e / (c.cin * c.cout);
        wt[c.w + ((8 - t) * c.cout + co) * c.cin + ci] = w[c.w + e];
    }
    const bf16 zero = __float2bfloat16(0.f);
    const int np = (c.cin + 15) / 16 * 9 * c.cout * 16;
    for (int e = e0; e < np; e += stride) {
        const int k = e & 15, r = e >> 4, co = r % c.cout, q = r / c.cout, t = q % 9, ci = q / 9 * 16 + k;
        wp[c.p + e] = ci < c.cin ? w[c.w + (t * c.cin + ci) * c.cout + co] : zero;
    }
    const int npt = (c.cout + 15) / 16 * 9 * c.cin * 16;
    for (int e = e0; e < npt; e += stride) {
        const int k = e & 15, r = e >> 4, ci = r % c.cin, q = r / c.cin, t = q % 9, co = q / 9 * 16 + k;
        wpt[c.pt + e] = co < c.cout ? w[c.w + ((8 - t) * c.cin + ci) * c.cout + co] : zero;
    }
}

// ---- weight gradient on the tensor cores --------------------------------------
// part[grp][t][ci][co] = sum over the group's pixels of in[p + off_t][ci] *
// g[p][co].  Block: 16 input x 16 output channels and a run of 16 x 8 pixel
// tiles; as a GEMM, M = input channels, N = output channels, K = pixels, one
// accumulator per tap, warp w taking the tile's pixel row w.  The input is
// BF16; the float32 gradient is cut into three BF16 parts of 8 significant
// bits each, which add up to it exactly (above 2^-109, where no part is
// subnormal), so each product of the sum is formed without error.  The tensor
// cores cut an accumulator's sum off instead of rounding it, a bias that grows
// with every step: a tile's sums therefore start at zero, smallest parts
// first, which leaves one cut, and are added to the accumulators by float32
// additions; these are added over the warps in float32 and over the groups as
// float pairs (k_reduce_groups).  Sums of one sign over 1, 16, 64 and 256
// images of 256^2 are off by 5e-8 of their value throughout; with the tiles'
// steps in one accumulator they were by 4e-7, 2.7e-6 and 1e-5 (64 images), by
// 2e-7 in the FP32 kernel before (serial FP32 sums over 4096 pixels).  Both
// operands lie in shared memory pixel by pixel, so fragments are read
// transposed (ldmatrix.trans), a tap being a shift of the pixel rows; the next
// tile's loads fly while one is multiplied.
// 16 images of 256^2, all layers: 3.6 ms in FP32, 0.86 ms here.
__global__ void __launch_bounds__(256) k_conv3_dw(const bf16* __restrict__ in, int Cin, const float* __restrict__ g,
                                                  int Cout, float* __restrict__ part, int B, int H, int Wd,
                                                  int tiles_per_group) {
    constexpr int PX = 18, PY = 10, NPIX = PX * PY, NG = 128;
    __shared__ __align__(16) unsigned char sm[(NPIX + 3 * NG) * CROW];
    unsigned char* const gsm = sm + NPIX * CROW;
    const unsigned xs = (unsigned)__cvta_generic_to_shared(sm), gs = xs + NPIX * CROW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ncoc = (Cout + 15) / 16;
    const int ci0 = (blockIdx.x / ncoc) * 16, co0 = (blockIdx.x % ncoc) * 16;
    const int tx_n = (Wd + 15) / 16, ty_n = (H + 7) / 8, ntiles = B * tx_n * ty_n;
    const int first = blockIdx.y * tiles_per_group, last = min(first + tiles_per_group, ntiles);
    uint4 vx[2];                                    // 360 half rows of 8 input channels
    float4 vg[2];                                   // 128 pixels x 4 output channels x 4
    auto load = [&](int tile) {
        const int b = tile / (tx_n * ty_n), r = tile - b * tx_n * ty_n;
        const int y0 = (r / tx_n) * 8, x0 = (r % tx_n) * 16;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            vx[q] = make_uint4(0, 0, 0, 0);
            const int e = tid + 256 * q, pix = e >> 1, py = pix / PX, px = pix - py * PX, ci = ci0 + 8 * (e & 1);
            const int gy = y0 + py - 1, gx = x0 + px - 1;
            if (pix < NPIX && gy >= 0 && gy < H && gx >= 0 && gx < Wd && ci < Cin) {
                const bf16* const p = in + (((size_t)b * H + gy) * Wd + gx) * Cin + ci;
                if (Cin % 8 == 0) {
                    vx[q] = __ldg(reinterpret_cast<const uint4*>(p));
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (ci + k < Cin) reinterpret_cast<bf16*>(&vx[q])[k] = p[k];
                }
            }
            vg[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int pg = e >> 2, co = co0 + 4 * (e & 3), hy = y0 + (pg >> 4), hx = x0 + (pg & 15);
            if (hy < H && hx < Wd && co < Cout) {
                const float* const p = g + (((size_t)b * H + hy) * Wd + hx) * Cout + co;
                if (Cout % 4 == 0) {
                    vg[q] = __ldg(reinterpret_cast<const float4*>(p));
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (co + k < Cout) reinterpret_cast<float*>(&vg[q])[k] = p[k];
                }
            }
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + 256 * q, pix = e >> 1;
            if (pix < NPIX) *reinterpret_cast<uint4*>(sm + pix * CROW + (e & 1) * 16) = vx[q];
            // the three parts: the leading 8 significant bits, of the
            // remainder (exact) the leading 8, and what is left; an infinity
            // or NaN goes whole into the first
            uint32_t part3[3][2];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float r = reinterpret_cast<const float*>(&vg[q])[k];
                const bool fin = isfinite(r);
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    const uint32_t top = __float_as_uint(r) >> 16;
                    const uint32_t bits = (u == 0 || fin) ? (u == 0 && !fin && isnan(r) ? top | 1u : top) : 0u;
                    r = fin ? r - __uint_as_float(top << 16) : 0.f;
                    part3[u][k >> 1] = (k & 1) ? part3[u][k >> 1] | (bits << 16) : bits;
                }
            }
#pragma unroll
            for (int u = 0; u < 3; ++u)
                *reinterpret_cast<uint2*>(gsm + (u * NG + (e >> 2)) * CROW + (e & 3) * 8) =
                    make_uint2(part3[u][0], part3[u][1]);
        }
    };
    float acc[9][2][4];
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int n = 0; n < 2; ++n) acc[t][n][0] = acc[t][n][1] = acc[t][n][2] = acc[t][n][3] = 0.f;
    // rows of the transposed fragments: A, pixels 0-7 | 8-15 (lane >> 4) and
    // channel half (lane >> 3 & 1); B, pixel half (lane >> 3 & 1) and channel half
    const unsigned aoff = xs + (warp * PX + (lane & 7) + 8 * (lane >> 4)) * CROW + ((lane >> 3) & 1) * 16;
    const unsigned boff = gs + (warp * 16 + (lane & 15)) * CROW + (lane >> 4) * 16;
    if (first < last) load(first);
    for (int tile = first; tile < last; ++tile) {
        store();
        __syncthreads();
        if (tile + 1 < last) load(tile + 1);
        uint32_t w[3][4];
#pragma unroll
        for (int u = 0; u < 3; ++u) ldmatrix4t(w[u], boff + u * NG * CROW);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            uint32_t a[4];
            ldmatrix4t(a, aoff + ((t / 3) * PX + t % 3) * CROW);
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                float d[4] = {0.f, 0.f, 0.f, 0.f};          // this tile's sums, the smallest parts first
#pragma unroll
                for (int u = 2; u >= 0; --u)
                    mma_bf16_16816(d, a[0], a[1], a[2], a[3], w[u][2 * n], w[u][2 * n + 1]);
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[t][n][v] += d[v];
            }
        }
        __syncthreads();
    }
    // the sum over the warps, tap by tap (16 x 16 values a warp)
    float* const red = reinterpret_cast<float*>(sm);
    float* const pp = part + (size_t)blockIdx.y * 9 * Cin * Cout;
    const int gq = lane >> 2, tq = lane & 3, ci = ci0 + (tid >> 4), co = co0 + (tid & 15);
#pragma unroll
    for (int t = 0; t < 9; ++t) {
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(red + warp * 256 + (gq + 8 * h) * 16 + n * 8 + 2 * tq) =
                    make_float2(acc[t][n][2 * h], acc[t][n][2 * h + 1]);
        __syncthreads();
        if (ci < Cin && co < Cout) {
            float v = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) v += red[k * 256 + tid];
            pp[((size_t)t * Cin + ci) * Cout + co] = v;
        }
        __syncthreads();
    }
}

// grad[i] = sum over groups of part[grp][i], as float pairs, in a fixed order:
// thread (x, y) of a block adds the groups y, y + 8, ... of value x
__global__ void __launch_bounds__(256) k_reduce_groups(const float* __restrict__ part, int ngroups, int n,
                                                       float* __restrict__ grad) {
    __shared__ double sm[8][32];
    const int i = blockIdx.x * 32 + threadIdx.x;
    FF s{0.f, 0.f};
    if (i < n)
#pragma unroll 4
        for (int k = threadIdx.y; k < ngroups; k += 8) ff_add(s, part[(size_t)k * n + i]);
    sm[threadIdx.y][threadIdx.x] = isfinite(s.hi) ? ff_value(s) : (double)s.hi;   // an infinity's error is NaN
    __syncthreads();
    if (threadIdx.y == 0 && i < n) {
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) v += sm[k][threadIdx.x];
        grad[i] = (float)v;
    }
}

// ---- element-wise forward steps ------------------------------------------------

// out = avgpool2(in) (bf16, NHWC)
__global__ void k_pool(const bf16* __restrict__ in, bf16* __restrict__ out, int B, int H, int Wd, int C) {
    const int Ho = H / 2, Wo = Wd / 2;
    const long long n = (long long)B * Ho * Wo * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = i % C;
        const long long q = i / C;
        const int xo = q % Wo, yo = (q / Wo) % Ho, b = q / ((long long)Wo * Ho);
        const bf16* s = in + (((size_t)b * H + 2 * yo) * Wd + 2 * xo) * C + c;
        const float v = __bfloat162float(s[0]) + __bfloat162float(s[C]) + __bfloat162float(s[(size_t)Wd * C]) +
                        __bfloat162float(s[(size_t)Wd * C + C]);
        out[i] = __float2bfloat16(0.25f * v);
    }
}

// k_pool on 8 channels at a time (C a multiple of 8): 16-byte loads and stores
__global__ void k_pool8(const uint4* __restrict__ in, uint4* __restrict__ out, int B, int H, int Wd, int C8) {
    const int Ho = H / 2, Wo = Wd / 2;
    const long long n = (long long)B * Ho * Wo * C8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C8);
        const long long q = i / C8;
        const int xo = (int)(q % Wo);
        const long long r = q / Wo;
        const int yo = (int)(r % Ho), b = (int)(r / Ho);
        const uint4* s = in + (((size_t)b * H + 2 * yo) * Wd + 2 * xo) * C8 + c;
        const uint4 v[4] = {s[0], s[C8], s[(size_t)Wd * C8], s[(size_t)Wd * C8 + C8]};
        uint4 o;
        const bf16* a0 = reinterpret_cast<const bf16*>(&v[0]);
        const bf16* a1 = reinterpret_cast<const bf16*>(&v[1]);
        const bf16* a2 = reinterpret_cast<const bf16*>(&v[2]);
        const bf16* a3 = reinterpret_cast<const bf16*>(&v[3]);
        bf16* ob = reinterpret_cast<bf16*>(&o);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            ob[e] = __float2bfloat16(0.25f * (__bfloat162float(a0[e]) + __bfloat162float(a1[e]) +
                                              __bfloat162float(a2[e]) + __bfloat162float(a3[e])));
        out[i] = o;
    }
}

// cat = [up2(d) (Cu channels), skip (Cs channels)] at resolution H x W
__global__ void k_up_cat(const bf16* __restrict__ d, const bf16* __restrict__ skip, bf16* __restrict__ cat, int B,
                         int H, int Wd, int Cu, int Cs) {
    const int C = Cu + Cs;
    const long long n = (long long)B * H * Wd * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = i % C;
        const long long q = i / C;
        const int x = q % Wd, y = (q / Wd) % H, b = q / ((long long)Wd * H);
        cat[i] = c < Cu ? d[(((size_t)b * (H / 2) + y / 2) * (Wd / 2) + x / 2) * Cu + c] : skip[q * Cs + (c - Cu)];
    }
}

// k_up_cat on 8 channels at a time (Cu, Cs multiples of 8): 16-byte copies
__global__ void k_up_cat8(const uint4* __restrict__ d, const uint4* __restrict__ skip, uint4* __restrict__ cat, int B,
                          int H, int Wd, int Cu8, int Cs8) {
    const int C8 = Cu8 + Cs8;
    const long long n = (long long)B * H * Wd * C8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C8);
        const long long q = i / C8;
        if (c < Cu8) {
            const int x = (int)(q % Wd);
            const long long r = q / Wd;
            const int y = (int)(r % H), b = (int)(r / H);
            cat[i] = d[(((size_t)b * (H / 2) + y / 2) * (Wd / 2) + x / 2) * Cu8 + c];
        } else {
            cat[i] = skip[q * Cs8 + (c - Cu8)];
        }
    }
}

// y[p] = o + sum_c d[p][c] O[c]
__global__ void k_conv1_fwd(const bf16* __restrict__ d, const float* __restrict__ O, const float* __restrict__ o,
                            float* __restrict__ y, long long P, int C) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        float s = o[0];
        for (int c = 0; c < C; ++c) s = fmaf(__bfloat162float(d[p * C + c]), O[c], s);
        y[p] = s;
    }
}

// ---- element-wise backward steps with per-channel sums ------------------------
//
// Every gradient that enters a convolution's backward pass is masked by the
// layer's ReLU and summed per channel (the bias gradient).  Those sums ride on
// the pass that writes the gradient: a thread keeps V consecutive channels
// over its share of the pixels (16-byte accesses for V = 8) and sums them as
// three floats (TwoSum twice: exact but for a float's rounding of errors of
// errors, 2^-72), then blocks and the final kernel add in float64, in a fixed
// order.  HBM-bound; a float64 addition a term, at 18.5 cycles an SM, made the
// gradient of 16 images of 256^2 350 us longer.  One pass per channel and
// block (a block a channel, each reading every pixel) had taken 4.2 ms of a
// 13.6 ms gradient of those images.
constexpr int ELT_BLOCKS = 4 * 152;

template <int V>
struct FVec;
template <int V>
__device__ __forceinline__ FVec<V> ldf(const float* p);

__device__ __forceinline__ float two_sum(float& s, float x) {      // s + x = (new s) + the returned error
    const float t = __fadd_rn(s, x), bx = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bx)), __fsub_rn(x, bx));
    s = t;
    return e;
}
template <int V>
struct ChanSum {                    // per-channel sums of a thread
    float a[V], b[V], c[V];
    __device__ __forceinline__ ChanSum() {
#pragma unroll
        for (int v = 0; v < V; ++v) a[v] = b[v] = c[v] = 0.f;
    }
    __device__ __forceinline__ void add(int v, float x) {
        c[v] = __fadd_rn(c[v], two_sum(b[v], two_sum(a[v], x)));
    }
    // The totals in float64 of the terms that the thread has stored in out at
    // p0, p0 + step, ... < P of C channels.  A sum that left float32's range on
    // the way, or met an infinity or NaN, is formed again from them.
    __device__ __forceinline__ void totals(double (&t)[V], const float* out, long long p0, long long step, long long P,
                                           int C) const {
        bool lost = false;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            lost |= !isfinite(a[v]);
            t[v] = to_f64(a[v]) + (to_f64(b[v]) + to_f64(c[v]));
        }
        if (!lost) return;
#pragma unroll
        for (int v = 0; v < V; ++v) t[v] = 0.0;
        for (long long p = p0; p < P; p += step) {
            const FVec<V> x = ldf<V>(out + p * C);
#pragma unroll
            for (int v = 0; v < V; ++v) t[v] += (double)x.v[v];
        }
    }
};

// Adds the block's sums into part[blockIdx.x * C + c]: threads of equal
// tid % G hold the same channels (G = C / V groups; threads past nth hold
// none).  256 / C threads share a channel's additions (with one thread a group
// their float64 latencies were two thirds of a pass).
template <int V>
__device__ __forceinline__ void chan_store(const double (&a)[V], int C, int G, int nth, double* __restrict__ part,
                                           double* sm /* 256 V */) {
    const int tid = threadIdx.x;
    __syncthreads();
    if (tid < nth)
#pragma unroll
        for (int v = 0; v < V; ++v) sm[v * 256 + tid] = a[v];
    __syncthreads();
    const int parts = 256 / C, o = tid % C, k = tid / C;
    double t = 0.0;
    if (k < parts)
        for (int e = (o / V) + G * k; e < nth; e += G * parts) t += sm[(o % V) * 256 + e];
    __syncthreads();
    sm[tid] = t;
    __syncthreads();
    if (tid < C) {
        for (int q = 1; q < parts; ++q) t += sm[q * C + tid];
        part[(size_t)blockIdx.x * C + tid] = t;
    }
}

// out[c] = sum over the blocks of part (fixed order), one block per channel
// and array: channel blockIdx.x of array blockIdx.y.
struct ChanOut {
    const double* part;
    float* out;
    int C;
};
__global__ void __launch_bounds__(128) k_chan_final(ChanOut a, ChanOut b, ChanOut c, int nblk) {
    __shared__ double sm[32];
    const ChanOut o = blockIdx.y == 0 ? a : (blockIdx.y == 1 ? b : c);
    if ((int)blockIdx.x >= o.C) return;
    double v[1] = {0.0};
    for (int k = threadIdx.x; k < nblk; k += 128) v[0] += o.part[(size_t)k * o.C + blockIdx.x];
    block_sum<1>(v, sm);
    if (threadIdx.x == 0) o.out[blockIdx.x] = (float)v[0];
}

template <int V>
struct alignas(V * sizeof(float)) FVec {
    float v[V];
};
template <int V>
struct alignas(V * sizeof(bf16)) BVec {
    bf16 v[V];
};
template <int V>
__device__ __forceinline__ FVec<V> ldf(const float* p) {
    return *reinterpret_cast<const FVec<V>*>(p);
}
template <int V>
__device__ __forceinline__ BVec<V> ldb(const bf16* p) {
    return *reinterpret_cast<const BVec<V>*>(p);
}

// The pixel loop of the kernels below: thread's channel group and pixels.  (Their
// grids have up to four blocks an SM, which their registers must leave room for.)
#define LM_PIXELS(V, C, P)                                                        \
    const int G = (C) / (V), nth = 256 / G * G, tid = threadIdx.x;                \
    const int c0 = (tid % G) * (V);                                               \
    const long long step = (long long)gridDim.x * (nth / G);                      \
    const long long p0 = tid < nth ? (long long)blockIdx.x * (nth / G) + tid / G : (P); \
    for (long long p = p0; p < (P); p += step)
// ... and the sums s of what it stored in `out`, through the block into part.
#define LM_SUMS(V, s, out, C, P, part)                                            \
    do {                                                                          \
        double t_[V];                                                             \
        (s).totals(t_, (out) + c0, p0, step, P, C);                               \
        chan_store<V>(t_, C, G, nth, part, sm);                                   \
    } while (0)

// g *= (act > 0); bias sums of the masked g
template <int V>
__global__ void __launch_bounds__(256, 4) k_mask_bias(float* __restrict__ g, const bf16* __restrict__ act, int C,
                                                   long long P, double* __restrict__ part) {
    __shared__ double sm[256 * V];
    ChanSum<V> s;
    LM_PIXELS(V, C, P) {
        const size_t i = p * C + c0;
        FVec<V> x = ldf<V>(g + i);
        const BVec<V> a = ldb<V>(act + i);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (!(__bfloat162float(a.v[v]) > 0.f)) x.v[v] = 0.f;
            s.add(v, x.v[v]);
        }
        *reinterpret_cast<FVec<V>*>(g + i) = x;
    }
    LM_SUMS(V, s, g, C, P, part);
}

// The output layer's backward: gd = gy O masked by d > 0 with its bias sums
// (the layer below), dO = sum_p d gy, do = sum_p gy (part: three arrays of
// blocks x C, blocks x C and blocks x 1).
template <int V>
__global__ void __launch_bounds__(256, 4) k_conv1_bwd(const bf16* __restrict__ d, const float* __restrict__ gy,
                                                   const float* __restrict__ O, float* __restrict__ gd, int C,
                                                   long long P, double* __restrict__ part) {
    __shared__ double sm[256 * V];
    ChanSum<V> sb;
    double sw[V], sg = 0.0;             // products: in float64, where they neither over- nor underflow
    float o[V];
    const int G0 = C / V;
#pragma unroll
    for (int v = 0; v < V; ++v) o[v] = O[(threadIdx.x % G0) * V + v], sw[v] = 0.0;
    LM_PIXELS(V, C, P) {
        const size_t i = p * C + c0;
        const BVec<V> a = ldb<V>(d + i);
        const float y = gy[p];
        const double yd = to_f64(y);
        FVec<V> x;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const float av = __bfloat162float(a.v[v]);
            x.v[v] = av > 0.f ? y * o[v] : 0.f;
            sb.add(v, x.v[v]);
            sw[v] = fma(to_f64(av), yd, sw[v]);
        }
        if (c0 == 0) sg += yd;
        *reinterpret_cast<FVec<V>*>(gd + i) = x;
    }
    const size_t n = (size_t)gridDim.x * C;
    LM_SUMS(V, sb, gd, C, P, part);
    chan_store<V>(sw, C, G, nth, part + n, sm);
    __syncthreads();
    sm[tid] = tid < nth && c0 == 0 ? sg : 0.0;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int k = 0; k < nth; k += G) t += sm[k];
        part[2 * n + blockIdx.x] = t;
    }
}

// The skip half of a concatenation's gradient: gskip = gcat[..., Cu:].
template <int V>
__global__ void k_cat_skip(const float* __restrict__ gcat, float* __restrict__ gskip, long long P, int Cu, int Cs) {
    const int C = Cu + Cs, G = Cs / V;
    const long long n = P * G;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const long long q = e / G;
        const int c = (int)(e - q * G) * V;
        *reinterpret_cast<FVec<V>*>(gskip + q * Cs + c) = ldf<V>(gcat + q * C + Cu + c);
    }
}

// The upsampled half: gd = up_bwd(gcat[..., :Cu]) (sum over the four fine
// pixels) at half resolution, masked by act > 0, with its bias sums.
template <int V>
__global__ void __launch_bounds__(256, 4) k_up_bwd(const float* __restrict__ gcat, const bf16* __restrict__ act,
                                                float* __restrict__ gd, int Ho, int Wo, int Cu, int Cs, long long P,
                                                double* __restrict__ part) {
    __shared__ double sm[256 * V];
    ChanSum<V> s;
    const int Cc = Cu + Cs, Wd = 2 * Wo;
    LM_PIXELS(V, Cu, P) {
        const int xo = (int)(p % Wo);
        const long long r = p / Wo;
        const int yo = (int)(r % Ho);
        const long long b = r / Ho;
        const float* src = gcat + ((b * 2 * Ho + 2 * yo) * Wd + 2 * xo) * Cc + c0;
        const FVec<V> a0 = ldf<V>(src), a1 = ldf<V>(src + Cc), a2 = ldf<V>(src + (size_t)Wd * Cc),
                      a3 = ldf<V>(src + (size_t)Wd * Cc + Cc);
        const BVec<V> a = ldb<V>(act + p * Cu + c0);
        FVec<V> x;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            x.v[v] = __bfloat162float(a.v[v]) > 0.f ? (a0.v[v] + a1.v[v]) + (a2.v[v] + a3.v[v]) : 0.f;
            s.add(v, x.v[v]);
        }
        *reinterpret_cast<FVec<V>*>(gd + p * Cu + c0) = x;
    }
    LM_SUMS(V, s, gd, Cu, P, part);
}

// gacc += pool_bwd(g) (each fine pixel receives a quarter of its parent's
// gradient), masked by act > 0, with its bias sums.
template <int V>
__global__ void __launch_bounds__(256, 4) k_pool_bwd(const float* __restrict__ g, const bf16* __restrict__ act,
                                                  float* __restrict__ gacc, int H, int Wd, int C, long long P,
                                                  double* __restrict__ part) {
    __shared__ double sm[256 * V];
    ChanSum<V> s;
    LM_PIXELS(V, C, P) {
        const int x = (int)(p % Wd);
        const long long r = p / Wd;
        const int y = (int)(r % H);
        const long long b = r / H;
        const size_t i = p * C + c0;
        FVec<V> t = ldf<V>(gacc + i);
        const FVec<V> q = ldf<V>(g + ((b * (H / 2) + y / 2) * (Wd / 2) + x / 2) * C + c0);
        const BVec<V> a = ldb<V>(act + i);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            t.v[v] = __bfloat162float(a.v[v]) > 0.f ? fmaf(0.25f, q.v[v], t.v[v]) : 0.f;
            s.add(v, t.v[v]);
        }
        *reinterpret_cast<FVec<V>*>(gacc + i) = t;
    }
    LM_SUMS(V, s, gacc, C, P, part);
}
#undef LM_PIXELS
#undef LM_SUMS

// gy = 2 (y - t) / n and, with LOSS, loss = mean((y - t)^2) (deterministic grid
// reduction; one block over all pixels had taken 2.1 ms for 16 images of 256^2)
constexpr int LOSS_BLOCKS = 2 * 152;
constexpr int LOSS_WORDS = LOSS_BLOCKS + 2;        // the loss, the blocks' sums, the arrival counter
template <bool LOSS>
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ y, const float* __restrict__ t,
                                             float* __restrict__ gy, long long n, Red red) {
    __shared__ double sm[32];
    double v[1] = {0.0};
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
        const float d = y[i] - t[i];
        gy[i] = 2.f * d / (float)n;
        if (LOSS) {
            const double dd = to_f64(d);
            v[0] = fma(dd, dd, v[0]);
        }
    }
    if (!LOSS) return;
    const int sl[1] = {0};
    if (grid_reduce<1>(v, red, sl, sm) && threadIdx.x == 0) red.scal[0] /= (double)n;
}

// Adam (Kingma & Ba 2015) on the FP32 master weights; refreshes the BF16 copy.
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       bf16* __restrict__ wb, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        wb[i] = __float2bfloat16(wi);
    }
}

__global__ void k_to_bf16(const float* __restrict__ a, bf16* __restrict__ b, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = __float2bfloat16(a[i]);
}

}  // namespace lm

// ============================== the network object ==============================

using namespace lm;

struct lm_net {
    int ch[4] = {16, 32, 48, 64};
    int cin = 3;
    struct Conv {
        int cin, cout, w, b;    // weight / bias offsets in the parameter array
    };
    std::vector<Conv> convs;    // A0 B0 A1 B1 A2 B2 A3 B3 C2 D2 C1 D1 C0 D0
    int oW = 0, ob = 0, nparams = 0;
    float *master = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    bf16 *wb = nullptr, *wt = nullptr;   // BF16 weights and their flipped transposes
    bf16 *wp = nullptr, *wpt = nullptr;  // the same as the tensor-core convolutions stage them
    lm::PrepTable prep{};
    // activations (bf16) and gradients (float) for batch x H x W
    int B = 0, H = 0, W = 0;        // the shape the buffers hold (B images at most)
    int Bf = 0;                     // images of the last forward pass
    std::vector<void*> bufs;        // forward activations (inference)
    std::vector<void*> gbufs;       // gradient buffers, allocated on the first backward pass
    bool grads_ready = false;
    bf16 *x = nullptr, *in_[4] = {}, *a1[4] = {}, *e[4] = {}, *cat[3] = {}, *da1[3] = {}, *d[3] = {};
    float* y = nullptr;
    float *gd0 = nullptr, *gbuf1 = nullptr, *gbuf2 = nullptr, *genc[4] = {}, *gdl[3] = {};
    float* part = nullptr;
    size_t part_n = 0;
    double* sums = nullptr;         // per-channel block sums of the backward pass
    double* dloss = nullptr;        // loss, its block sums and their arrival counter
    std::mutex loss_mu;             // held by a call that uses them, until it has read the loss
    int adam_t = 0;
};

namespace {

#define NCK(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            fprintf(stderr, "lowmach: %s failed: %s\n", #call, cudaGetErrorString(e_));            \
            return e_ == cudaErrorMemoryAllocation ? LM_ERR_OUT_OF_MEMORY : LM_ERR_CUDA;           \
        }                                                                                          \
    } while (0)

int blocks_for(long long n) { return (int)std::min<long long>((n + 255) / 256, 152LL * 16); }

void free_acts(lm_net* N) {
    for (void* p : N->bufs) cudaFree(p);
    for (void* p : N->gbufs) cudaFree(p);
    N->bufs.clear();
    N->gbufs.clear();
    N->grads_ready = false;
    N->B = N->H = N->W = 0;
}

template <class T>
int nalloc(lm_net* N, T** p, size_t count, bool grad = false) {
    NCK(cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T)));
    (grad ? N->gbufs : N->bufs).push_back(*p);
    return LM_OK;
}

// The backward pass's buffers for the current batch shape (only training
// needs them: an inference of a 512^3 grid as 512 images would otherwise
// hold several times its activations in gradients).
int ensure_grads(lm_net* N) {
    if (N->grads_ready) return LM_OK;
    int rc;
    const size_t P0 = (size_t)N->B * N->H * N->W;
    for (int l = 0; l < 4; ++l) {
        const size_t Pl = P0 >> (2 * l);
        const int cl = N->ch[l];
        if ((rc = nalloc(N, &N->genc[l], Pl * cl, true))) return rc;
        // what comes down the decoder: D_0's is gd0, e_3's goes to genc[3]
        if ((l == 1 || l == 2) && (rc = nalloc(N, &N->gdl[l], Pl * cl, true))) return rc;
    }
    size_t gmax = 0;
    for (int l = 0; l < 4; ++l) {
        const size_t Pl = P0 >> (2 * l);
        gmax = std::max(gmax, Pl * (size_t)(N->ch[l] + (l < 3 ? N->ch[l + 1] : 0)));
        gmax = std::max(gmax, Pl * (size_t)(l == 0 ? N->cin : N->ch[l - 1]));
    }
    if ((rc = nalloc(N, &N->gd0, P0 * N->ch[0], true)) || (rc = nalloc(N, &N->gbuf1, gmax, true)) ||
        (rc = nalloc(N, &N->gbuf2, gmax, true)))
        return rc;
    N->part_n = 0;
    for (const auto& c : N->convs) N->part_n = std::max(N->part_n, (size_t)9 * c.cin * c.cout);
    N->part_n *= 256;   // pixel groups of the largest layer; conv_bwd_w takes more of a smaller one
    if ((rc = nalloc(N, &N->part, N->part_n, true))) return rc;
    int cmax = 1;
    for (int c : N->ch) cmax = std::max(cmax, c);
    if ((rc = nalloc(N, &N->sums, (size_t)3 * ELT_BLOCKS * cmax, true))) return rc;
    N->grads_ready = true;
    return LM_OK;
}

int ensure_acts(lm_net* N, int B, int H, int W) {
    if (B <= N->B && H == N->H && W == N->W) return LM_OK;
    free_acts(N);
    int rc;
    const size_t P0 = (size_t)B * H * W;
    if ((rc = nalloc(N, &N->x, P0 * N->cin))) return rc;
    for (int l = 0; l < 4; ++l) {
        const size_t Pl = P0 >> (2 * l);
        const int cl = N->ch[l], cprev = l == 0 ? N->cin : N->ch[l - 1];
        if (l > 0 && (rc = nalloc(N, &N->in_[l], Pl * cprev))) return rc;
        if ((rc = nalloc(N, &N->a1[l], Pl * cl)) || (rc = nalloc(N, &N->e[l], Pl * cl))) return rc;
        if (l < 3) {
            const int cc = N->ch[l + 1] + cl;
            if ((rc = nalloc(N, &N->cat[l], Pl * cc)) || (rc = nalloc(N, &N->da1[l], Pl * cl)) ||
                (rc = nalloc(N, &N->d[l], Pl * cl)))
                return rc;
        }
    }
    N->in_[0] = N->x;
    if ((rc = nalloc(N, &N->y, P0))) return rc;
    N->B = B;
    N->H = H;
    N->W = W;
    return LM_OK;
}

void conv_fwd(lm_net* N, const lm_net::Conv& c, const bf16* in, bf16* out, int B, int H, int W, cudaStream_t s) {
    count_launches(1);
    const bf16* w = N->wb + c.w;
    const float* bias = N->master + c.b;
    const PrepConv& pc = N->prep.c[&c - N->convs.data()];
    if (conv3_mma<false>(in, c.cin, N->wp + pc.p, bias, out, c.cout, B, H, W, 1, s)) return;
    const int ncoc = (c.cout + CT - 1) / CT;
    const dim3 grd((W + CT - 1) / CT, (H + CT - 1) / CT, B * ncoc);
    k_conv3<bf16, bf16><<<grd, dim3(CT, CT), 0, s>>>(in, c.cin, w, bias, out, c.cout, H, W, 1, ncoc);
}

// gin = conv3 backward-data of g (float32, Cout channels) through conv c
void conv_bwd_data(lm_net* N, const lm_net::Conv& c, const float* g, float* gin, int B, int H, int W, cudaStream_t s) {
    count_launches(1);
    const PrepConv& pc = N->prep.c[&c - N->convs.data()];
    if (conv3_mma<true>(g, c.cout, N->wpt + pc.pt, nullptr, gin, c.cin, B, H, W, 0, s)) return;
    const int ncoc = (c.cin + CT - 1) / CT;
    const dim3 grd((W + CT - 1) / CT, (H + CT - 1) / CT, B * ncoc);
    k_conv3<float, float><<<grd, dim3(CT, CT), 0, s>>>(g, c.cout, N->wt + c.w, nullptr, gin, c.cin, H, W, 0, ncoc);
}

// weight and bias gradients of conv c from its input act and output gradient g
void conv_bwd_w(lm_net* N, const lm_net::Conv& c, const bf16* act, const float* g, int B, int H, int W, cudaStream_t s) {
    const int tiles = B * ((W + 15) / 16) * ((H + 7) / 8);
    const int nchunk = ((c.cin + 15) / 16) * ((c.cout + 15) / 16), n = 9 * c.cin * c.cout;
    // four blocks an SM in all, as far as the partials' buffer reaches
    int groups = std::max(1, (int)std::min<long long>(4 * 152 / nchunk, (long long)(N->part_n / n)));
    const int tpg = (tiles + groups - 1) / groups;
    groups = (tiles + tpg - 1) / tpg;
    count_launches(2);
    k_conv3_dw<<<dim3(nchunk, groups), 256, 0, s>>>(act, c.cin, g, c.cout, N->part, B, H, W, tpg);
    k_reduce_groups<<<(n + 31) / 32, dim3(32, 8), 0, s>>>(N->part, groups, n, N->grad + c.w);
}

// V consecutive channels a thread: the widest that divides C (and C2); four at
// most in the passes that would spill with eight in the registers that four
// blocks an SM leave a thread
int chan_width(int C, int C2 = 0, int most = 8) {
    return most >= 8 && C % 8 == 0 && C2 % 8 == 0 ? 8 : (C % 4 == 0 && C2 % 4 == 0 ? 4 : 1);
}
// blocks of a pixel pass over P pixels of C channels, V a thread
int elt_blocks(long long P, int C, int V) {
    const long long per = 256 / (C / V);
    return (int)std::max(1LL, std::min<long long>(ELT_BLOCKS, (P + per - 1) / per));
}
#define LM_BY_WIDTH4(V, CALL)                              \
    do {                                                   \
        if ((V) == 4) { constexpr int W_ = 4; CALL; }      \
        else { constexpr int W_ = 1; CALL; }               \
    } while (0)
#define LM_BY_WIDTH(V, CALL)                               \
    do {                                                   \
        if ((V) == 8) { constexpr int W_ = 8; CALL; }      \
        else LM_BY_WIDTH4(V, CALL);                        \
    } while (0)

// g *= (act > 0), and the bias gradient of conv c (whose output gradient g is)
void mask_bias(lm_net* N, const lm_net::Conv& c, float* g, const bf16* act, long long P, cudaStream_t s) {
    const int V = chan_width(c.cout), nb = elt_blocks(P, c.cout, V);
    const ChanOut o{N->sums, N->grad + c.b, c.cout};
    count_launches(2);
    LM_BY_WIDTH(V, (k_mask_bias<W_><<<nb, 256, 0, s>>>(g, act, c.cout, P, N->sums)));
    k_chan_final<<<dim3(c.cout, 1), 128, 0, s>>>(o, o, o, nb);
}

}  // namespace

namespace lm {

// the derived layouts of the weights, after every change of them
void prepare_weights(lm_net* N, cudaStream_t s) {
    count_launches(1);
    k_prep_weights<<<dim3(32, (unsigned)N->convs.size()), 256, 0, s>>>(N->prep, N->wb, N->wt, N->wp, N->wpt);
}

void net_destroy(lm_net* N);

int net_forward(lm_net* N, const float* xin, float* yout, int B, int H, int W, cudaStream_t s) {
    if (H % 8 || W % 8 || B < 1) return LM_ERR_INVALID_ARG;
    int rc = ensure_acts(N, B, H, W);
    if (rc) return rc;
    N->Bf = B;
    const long long P0 = (long long)B * H * W;
    count_launches(1);
    k_to_bf16<<<blocks_for(P0 * N->cin), 256, 0, s>>>(xin, N->x, P0 * N->cin);
    for (int l = 0; l < 4; ++l) {
        const int Hl = H >> l, Wl = W >> l;
        if (l > 0) {
            count_launches(1);
            const int cp = N->ch[l - 1];
            if (cp % 8 == 0)
                k_pool8<<<blocks_for((long long)B * Hl * Wl * (cp / 8)), 256, 0, s>>>(
                    (const uint4*)N->e[l - 1], (uint4*)N->in_[l], B, H >> (l - 1), W >> (l - 1), cp / 8);
            else
                k_pool<<<blocks_for((long long)B * Hl * Wl * cp), 256, 0, s>>>(N->e[l - 1], N->in_[l], B, H >> (l - 1),
                                                                              W >> (l - 1), cp);
        }
        conv_fwd(N, N->convs[2 * l], N->in_[l], N->a1[l], B, Hl, Wl, s);
        conv_fwd(N, N->convs[2 * l + 1], N->a1[l], N->e[l], B, Hl, Wl, s);
    }
    const bf16* dprev = N->e[3];
    for (int l = 2; l >= 0; --l) {
        const int Hl = H >> l, Wl = W >> l, cu = N->ch[l + 1], cs = N->ch[l];
        count_launches(1);
        if (cu % 8 == 0 && cs % 8 == 0)
            k_up_cat8<<<blocks_for((long long)B * Hl * Wl * ((cu + cs) / 8)), 256, 0, s>>>(
                (const uint4*)dprev, (const uint4*)N->e[l], (uint4*)N->cat[l], B, Hl, Wl, cu / 8, cs / 8);
        else
            k_up_cat<<<blocks_for((long long)B * Hl * Wl * (cu + cs)), 256, 0, s>>>(dprev, N->e[l], N->cat[l], B, Hl,
                                                                                    Wl, cu, cs);
        const int k = 8 + 2 * (2 - l);
        conv_fwd(N, N->convs[k], N->cat[l], N->da1[l], B, Hl, Wl, s);
        conv_fwd(N, N->convs[k + 1], N->da1[l], N->d[l], B, Hl, Wl, s);
        dprev = N->d[l];
    }
    count_launches(1);
    k_conv1_fwd<<<blocks_for(P0), 256, 0, s>>>(N->d[0], N->master + N->oW, N->master + N->ob, yout ? yout : N->y, P0,
                                               N->ch[0]);
    return cudaGetLastError() == cudaSuccess ? LM_OK : LM_ERR_CUDA;
}

int net_backward(lm_net* N, const float* gy, cudaStream_t s) {
    if (int rc = ensure_grads(N)) return rc;
    const int B = N->Bf, H = N->H, W = N->W;     // the images of the last forward pass
    const long long P0 = (long long)B * H * W;
    {   // output layer, and D_0's masked gradient with its bias gradient
        const int C = N->ch[0], V = chan_width(C, 0, 4), nb = elt_blocks(P0, C, V);
        const size_t n = (size_t)nb * C;
        count_launches(2);
        LM_BY_WIDTH4(V, (k_conv1_bwd<W_><<<nb, 256, 0, s>>>(N->d[0], gy, N->master + N->oW, N->gd0, C, P0, N->sums)));
        k_chan_final<<<dim3(C, 3), 128, 0, s>>>(ChanOut{N->sums, N->grad + N->convs[13].b, C},
                                               ChanOut{N->sums + n, N->grad + N->oW, C},
                                               ChanOut{N->sums + 2 * n, N->grad + N->ob, 1}, nb);
    }
    float* gd = N->gd0;                                            // masked: g of D_l's output
    for (int l = 0; l <= 2; ++l) {
        const int Hl = H >> l, Wl = W >> l, cl = N->ch[l], cu = N->ch[l + 1];
        const long long Pl = (long long)B * Hl * Wl;
        const int k = 8 + 2 * (2 - l);
        const lm_net::Conv &Cc = N->convs[k], &Dc = N->convs[k + 1];
        conv_bwd_w(N, Dc, N->da1[l], gd, B, Hl, Wl, s);
        conv_bwd_data(N, Dc, gd, N->gbuf1, B, Hl, Wl, s);          // g of da1
        mask_bias(N, Cc, N->gbuf1, N->da1[l], Pl, s);
        conv_bwd_w(N, Cc, N->cat[l], N->gbuf1, B, Hl, Wl, s);
        conv_bwd_data(N, Cc, N->gbuf1, N->gbuf2, B, Hl, Wl, s);          // g of cat
        // the skip half waits for the encoder's own gradient; the upsampled
        // half goes down masked by d_{l+1} (d_3 = e_3), the next layer's g
        const int V = chan_width(cu, cl), Vu = chan_width(cu, cl, 4), nb = elt_blocks(Pl / 4, cu, Vu);
        const bf16* below = l < 2 ? N->d[l + 1] : N->e[3];
        const lm_net::Conv& next = N->convs[l < 2 ? k - 1 : 7];
        float* gn = l < 2 ? N->gdl[l + 1] : N->genc[3];
        const ChanOut o{N->sums, N->grad + next.b, cu};
        count_launches(3);
        LM_BY_WIDTH(V, (k_cat_skip<W_><<<blocks_for(Pl * (cl / W_)), 256, 0, s>>>(N->gbuf2, N->genc[l], Pl, cu, cl)));
        LM_BY_WIDTH4(Vu, (k_up_bwd<W_><<<nb, 256, 0, s>>>(N->gbuf2, below, gn, Hl / 2, Wl / 2, cu, cl, Pl / 4, N->sums)));
        k_chan_final<<<dim3(cu, 1), 128, 0, s>>>(o, o, o, nb);
        gd = gn;
    }
    for (int l = 3; l >= 0; --l) {                                 // genc[l]: masked g of e_l
        const int Hl = H >> l, Wl = W >> l;
        const long long Pl = (long long)B * Hl * Wl;
        const lm_net::Conv &Ac = N->convs[2 * l], &Bc = N->convs[2 * l + 1];
        conv_bwd_w(N, Bc, N->a1[l], N->genc[l], B, Hl, Wl, s);
        conv_bwd_data(N, Bc, N->genc[l], N->gbuf1, B, Hl, Wl, s);          // g of a1
        mask_bias(N, Ac, N->gbuf1, N->a1[l], Pl, s);
        conv_bwd_w(N, Ac, N->in_[l], N->gbuf1, B, Hl, Wl, s);
        if (l > 0) {
            conv_bwd_data(N, Ac, N->gbuf1, N->gbuf2, B, Hl, Wl, s);      // g of in_l
            const int cp = N->ch[l - 1], V = chan_width(cp), nb = elt_blocks(Pl << 2, cp, V);
            const ChanOut o{N->sums, N->grad + N->convs[2 * l - 1].b, cp};
            count_launches(2);
            LM_BY_WIDTH(V, (k_pool_bwd<W_><<<nb, 256, 0, s>>>(N->gbuf2, N->e[l - 1], N->genc[l - 1], H >> (l - 1),
                                                             W >> (l - 1), cp, Pl << 2, N->sums)));
            k_chan_final<<<dim3(cp, 1), 128, 0, s>>>(o, o, o, nb);
        }
    }
    return cudaGetLastError() == cudaSuccess ? LM_OK : LM_ERR_CUDA;
}

int net_create(const int ch[4], lm_net** out) {
    lm_net* N = new lm_net();
    for (int l = 0; l < 4; ++l) {
        if (ch[l] < 1 || ch[l] > 256) {
            delete N;
            return LM_ERR_INVALID_ARG;
        }
        N->ch[l] = ch[l];
    }
    int off = 0;
    auto conv = [&](int cin, int cout) {
        lm_net::Conv c{cin, cout, off, off + 9 * cin * cout};
        off += 9 * cin * cout + cout;
        N->convs.push_back(c);
    };
    int prev = N->cin;
    for (int l = 0; l < 4; ++l) {
        conv(prev, N->ch[l]);
        conv(N->ch[l], N->ch[l]);
        prev = N->ch[l];
    }
    for (int l = 2; l >= 0; --l) {
        conv(N->ch[l + 1] + N->ch[l], N->ch[l]);
        conv(N->ch[l], N->ch[l]);
    }
    N->oW = off;
    N->ob = off + N->ch[0];
    N->nparams = off + N->ch[0] + 1;
    const size_t n = N->nparams;
    conv3_allow_smem();
    size_t np = 0, npt = 0;
    for (size_t k = 0; k < N->convs.size(); ++k) {
        const lm_net::Conv& c = N->convs[k];
        N->prep.c[k] = PrepConv{c.cin, c.cout, c.w, (int)np, (int)npt};
        np += (size_t)(c.cin + 15) / 16 * 9 * c.cout * 16;
        npt += (size_t)(c.cout + 15) / 16 * 9 * c.cin * 16;
    }
    if (cudaMalloc(&N->wp, np * 2) || cudaMalloc(&N->wpt, npt * 2) || cudaMalloc(&N->master, n * 4) ||
        cudaMalloc(&N->grad, n * 4) || cudaMalloc(&N->m, n * 4) || cudaMalloc(&N->v, n * 4) ||
        cudaMalloc(&N->wb, n * 2) || cudaMalloc(&N->wt, n * 2) || cudaMalloc(&N->dloss, LOSS_WORDS * 8)) {
        net_destroy(N);
        return LM_ERR_OUT_OF_MEMORY;
    }
    cudaMemset(N->master, 0, n * 4);
    cudaMemset(N->grad, 0, n * 4);
    cudaMemset(N->m, 0, n * 4);
    cudaMemset(N->v, 0, n * 4);
    cudaMemset(N->wb, 0, n * 2);
    cudaMemset(N->wt, 0, n * 2);
    cudaMemset(N->wp, 0, np * 2);
    cudaMemset(N->wpt, 0, npt * 2);
    cudaMemset(N->dloss, 0, LOSS_WORDS * 8);
    // the clears run on the default stream, which a caller's stream need not wait for
    if (cudaDeviceSynchronize() != cudaSuccess) {
        net_destroy(N);
        return LM_ERR_CUDA;
    }
    *out = N;
    return LM_OK;
}

void net_destroy(lm_net* N) {
    if (!N) return;
    cudaDeviceSynchronize();
    free_acts(N);
    cudaFree(N->master);
    cudaFree(N->grad);
    cudaFree(N->m);
    cudaFree(N->v);
    cudaFree(N->wb);
    cudaFree(N->wt);
    cudaFree(N->wp);
    cudaFree(N->wpt);
    cudaFree(N->dloss);
    delete N;
}

int net_set_params(lm_net* N, const float* host, int n) {
    if (n != N->nparams) return LM_ERR_INVALID_ARG;
    NCK(cudaMemcpy(N->master, host, sizeof(float) * n, cudaMemcpyHostToDevice));
    count_launches(1);
    k_to_bf16<<<blocks_for(n), 256>>>(N->master, N->wb, n);
    prepare_weights(N, nullptr);
    NCK(cudaMemset(N->m, 0, sizeof(float) * n));
    NCK(cudaMemset(N->v, 0, sizeof(float) * n));
    N->adam_t = 0;
    NCK(cudaDeviceSynchronize());
    return LM_OK;
}

}  // namespace lm

// ================================ features ===================================
// Network input of a 2D grid (rows = z, columns = x) from a field v (the rhs
// or a residual) and the float32 coefficients:
//   ch0 = v / rms(v),  ch1 = log(rho / mean rho),  ch2 = log(1 / (c~ rho h_z^2)) / 10,
// and the output scale s = rms(v) / (mean c~ + mean(1/rho) pi^2): the network
// output times s approximates A^-1 v.

namespace lm {

template <typename TV>
__global__ void __launch_bounds__(NT) k_feat_sums(int N, const TV* __restrict__ v, const float* __restrict__ rho,
                                                  const float* __restrict__ ct, double irs, Red red) {
    __shared__ double sm[4 * 32];
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = blockIdx.x * NT + threadIdx.x; i < N; i += gridDim.x * NT) {
        const double vi = (double)v[i];
        a[0] += vi * vi;
        a[1] += rho[i];
        a[2] += ct[i];
        a[3] += 1.0 / (double)rho[i];
    }
    const int sl[4] = {8, 9, 10, 11};
    if (grid_reduce<4>(a, red, sl, sm) && lin_tid() == 0) {
        const double rms = sqrt(red.scal[8] / N);
        red.scal[12] = rms > 0.0 ? 1.0 / rms : 0.0;                                 // 1 / rms
        red.scal[13] = red.scal[9] / N;                                            // mean rho
        // rho holds rho / rho_scale: mean(1/rho) = mean(1/rho_stored) / rho_scale
        red.scal[14] = rms / (red.scal[10] / N + (red.scal[11] / N) * irs * 9.869604401089358);  // scale s
    }
}

// Pixel of cell idx in the network's image batch: a grid of nx x ny x nz
// cells is ny images (one per x-z slice j) of nz rows and nx columns, so a
// 3D grid is read slice by slice by the 2D network; for a 2D grid (ny = 1)
// the pixel index is the cell index.
__device__ __forceinline__ int net_pixel(int idx, int nx, int ny, int nz) {
    const int i = idx % nx, t = idx / nx, j = t % ny, k = t / ny;
    return (j * nz + k) * nx + i;
}

template <typename TV>
__global__ void k_feat(int N, const TV* __restrict__ v, const float* __restrict__ rho, const float* __restrict__ ct,
                       const double* __restrict__ scal, float ihz2, float* __restrict__ feat, int nx, int ny, int nz) {
    const float irms = (float)scal[12], mrho = (float)scal[13];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const float r = rho[i];
        const int q = net_pixel(i, nx, ny, nz);
        feat[3 * q + 0] = (float)v[i] * irms;
        feat[3 * q + 1] = logf(r / mrho);
        feat[3 * q + 2] = 0.1f * logf(ihz2 / (ct[i] * r));
    }
}

// out = s * y (precision of the destination), y in image order
template <typename TO>
__global__ void k_scale_out(int N, const float* __restrict__ y, const double* __restrict__ scal, TO* __restrict__ out,
                            int nx, int ny, int nz) {
    const double s = scal[14];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
        out[i] = (TO)(s * y[net_pixel(i, nx, ny, nz)]);
}

}  // namespace lm

namespace {

template <typename TV>
int features(lm_grid* g, const TV* v, float* feat, cudaStream_t s) {
    const Red red{g->part, g->scal, g->ctr};
    count_launches(2);
    k_feat_sums<TV><<<g->G, NT, 0, s>>>(g->N, v, g->rho32, g->ct32, 1.0 / g->rho_scale, red);
    // channel 2 is log(1/(c~ rho h^2)) of the true rho = rho_stored * rho_scale
    k_feat<TV><<<blocks_for(g->N), 256, 0, s>>>(g->N, v, g->rho32, g->ct32, g->scal,
                                                (float)(1.0 / (g->h[2] * g->h[2]) / g->rho_scale), feat, g->n[0],
                                                g->n[1], g->n[2]);
    return cudaGetLastError() == cudaSuccess ? LM_OK : LM_ERR_CUDA;
}

uint64_t fnv1a(const unsigned char* p, size_t n) {
    uint64_t h = 1469598103934665603ULL;
    for (size_t i = 0; i < n; ++i) {
        h ^= p[i];
        h *= 1099511628211ULL;
    }
    return h;
}

}  // namespace

namespace lm {

bool net_usable(const lm_grid* g) { return g->net && g->n[0] % 8 == 0 && g->n[2] % 8 == 0; }

// dst = s * NN(features(v)) on grid g, dst float or double: a 2D grid is one
// image; a 3D grid is a batch of ny images, its x-z slices, through the same
// 2D network (the network sees no coupling across y; the flexible-CG
// iteration around it does)
template <typename TV, typename TO>
int net_apply(lm_grid* g, const TV* v, TO* dst, cudaStream_t s) {
    lm_net* N = g->net;
    int rc = features<TV>(g, v, g->feat, s);
    if (rc) return rc;
    rc = net_forward(N, g->feat, g->nny, g->n[1], g->n[2], g->n[0], s);
    if (rc) return rc;
    count_launches(1);
    k_scale_out<TO><<<blocks_for(g->N), 256, 0, s>>>(g->N, g->nny, g->scal, dst, g->n[0], g->n[1], g->n[2]);
    return cudaGetLastError() == cudaSuccess ? LM_OK : LM_ERR_CUDA;
}
template int net_apply<double, double>(lm_grid*, const double*, double*, cudaStream_t);
template int net_apply<float, float>(lm_grid*, const float*, float*, cudaStream_t);

}  // namespace lm

// ================================== C ABI =====================================

extern "C" {

int lm_net_create(const int ch[4], lm_net** out) {
    if (!ch || !out) return LM_ERR_INVALID_ARG;
    return lm::net_create(ch, out);
}

void lm_net_destroy(lm_net* N) { lm::net_destroy(N); }

int lm_net_num_params(const lm_net* N) { return N ? N->nparams : 0; }

int lm_net_set_params(lm_net* N, const float* host, int n) {
    if (!N || !host) return LM_ERR_INVALID_ARG;
    return lm::net_set_params(N, host, n);
}

int lm_net_get_params(lm_net* N, float* host, int n) {
    if (!N || !host || n != N->nparams) return LM_ERR_INVALID_ARG;
    NCK(cudaDeviceSynchronize());
    NCK(cudaMemcpy(host, N->master, sizeof(float) * n, cudaMemcpyDeviceToHost));
    return LM_OK;
}

int lm_net_get_grads(lm_net* N, float* host, int n) {
    if (!N || !host || n != N->nparams) return LM_ERR_INVALID_ARG;
    NCK(cudaDeviceSynchronize());
    NCK(cudaMemcpy(host, N->grad, sizeof(float) * n, cudaMemcpyDeviceToHost));
    return LM_OK;
}

int lm_net_forward(lm_net* N, const float* x, float* y, int B, int H, int W, void* stream) {
    if (!N || !x || !y) return LM_ERR_INVALID_ARG;
    return lm::net_forward(N, x, y, B, H, W, (cudaStream_t)stream);
}

int lm_net_backward(lm_net* N, const float* gy, void* stream) {
    if (!N || !gy || !N->B) return LM_ERR_INVALID_ARG;
    return lm::net_backward(N, gy, (cudaStream_t)stream);
}

int lm_net_mse(lm_net* N, const float* y, const float* t, float* gy, long long n, double* loss, void* stream) {
    if (!N || !y || !t || !gy || n < 1) return LM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (int)std::max<long long>(1, std::min<long long>(LOSS_BLOCKS, (n + 1023) / 1024));
    count_launches(1);
    if (!loss) {
        k_mse<false><<<nb, 256, 0, s>>>(y, t, gy, n, Red{});
        return cudaGetLastError() == cudaSuccess ? LM_OK : LM_ERR_CUDA;
    }
    // one loss at a time: calls on other streams would share the counter
    std::lock_guard<std::mutex> lk(N->loss_mu);
    k_mse<true><<<nb, 256, 0, s>>>(
        y, t, gy, n, Red{N->dloss + 1, N->dloss, (unsigned int*)(N->dloss + 1 + LOSS_BLOCKS)});
    NCK(cudaGetLastError());
    NCK(cudaMemcpyAsync(loss, N->dloss, sizeof(double), cudaMemcpyDeviceToHost, s));
    NCK(cudaStreamSynchronize(s));
    return LM_OK;
}

int lm_net_adam(lm_net* N, float lr, float b1, float b2, float eps, void* stream) {
    if (!N || !(lr > 0.f)) return LM_ERR_INVALID_ARG;
    const int t = ++N->adam_t;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    count_launches(1);
    k_adam<<<blocks_for(N->nparams), 256, 0, (cudaStream_t)stream>>>(N->master, N->grad, N->m, N->v, N->wb,
                                                                     N->nparams, lr, b1, b2, eps, c1, c2);
    lm::prepare_weights(N, (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? LM_OK : LM_ERR_CUDA;
}

// File: "LMUNET01", int32 ch[4], int32 nparams, float32 params[nparams],
// uint64 FNV-1a of the parameter bytes; little-endian.
int lm_net_save(lm_net* N, const char* path) {
    if (!N || !path) return LM_ERR_INVALID_ARG;
    std::vector<float> p(N->nparams);
    int rc = lm_net_get_params(N, p.data(), N->nparams);
    if (rc) return rc;
    FILE* fp = fopen(path, "wb");
    if (!fp) return LM_ERR_INVALID_ARG;
    const uint64_t h = fnv1a((const unsigned char*)p.data(), p.size() * 4);
    const int32_t hdr[5] = {N->ch[0], N->ch[1], N->ch[2], N->ch[3], N->nparams};
    bool ok = fwrite("LMUNET01", 1, 8, fp) == 8 && fwrite(hdr, 4, 5, fp) == 5 &&
              fwrite(p.data(), 4, p.size(), fp) == p.size() && fwrite(&h, 8, 1, fp) == 1;
    ok = (fclose(fp) == 0) && ok;
    return ok ? LM_OK : LM_ERR_INVALID_ARG;
}

int lm_net_load(const char* path, lm_net** out) {
    if (!path || !out) return LM_ERR_INVALID_ARG;
    *out = nullptr;
    FILE* fp = fopen(path, "rb");
    if (!fp) return LM_ERR_NETWORK;
    char magic[8];
    int32_t hdr[5];
    if (fread(magic, 1, 8, fp) != 8 || memcmp(magic, "LMUNET01", 8) || fread(hdr, 4, 5, fp) != 5) {
        fclose(fp);
        return LM_ERR_NETWORK;
    }
    lm_net* N = nullptr;
    if (lm::net_create(hdr, &N) || N->nparams != hdr[4]) {
        fclose(fp);
        lm::net_destroy(N);
        return LM_ERR_NETWORK;
    }
    std::vector<float> p(N->nparams);
    uint64_t h = 0;
    const bool ok = fread(p.data(), 4, p.size(), fp) == p.size() && fread(&h, 8, 1, fp) == 1 &&
                    h == fnv1a((const unsigned char*)p.data(), p.size() * 4);
    fclose(fp);
    if (!ok || lm::net_set_params(N, p.data(), N->nparams)) {
        lm::net_destroy(N);
        return LM_ERR_NETWORK;
    }
    *out = N;
    return LM_OK;
}

int lm_net_features(lm_grid* g, const double* v, float* feat, double* scale, void* stream) {
    if (!g || !v || !feat) return LM_ERR_INVALID_ARG;
    if (!g->have_coefs) return LM_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    int rc = features<double>(g, v, feat, s);
    if (rc) return rc;
    if (scale) {
        NCK(cudaMemcpyAsync(scale, g->scal + 14, sizeof(double), cudaMemcpyDeviceToHost, s));
        NCK(cudaStreamSynchronize(s));
    }
    return LM_OK;
}

}  // extern "C"
