// aqe.cu -- AQE elementwise kernels (Eq. ours, Eq. activation, Eq. weight),
// the fused quantize + bit-plane pack of activations (Eq. inference) and the
// packing of latent weights.  All of them stream HBM: 128-bit loads where the
// layout allows, grids sized from the SM count.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include "common.cuh"

namespace minw {

// ---------------------------------------------------------------------------
// AQE forward / backward, flat fp32 arrays.
// ---------------------------------------------------------------------------

__device__ __forceinline__ float aqe_fwd1(float x, float alpha, float oma, const QParams &q) {
    const float h = level_value(x * q.scale, q);
    return fmaf(alpha, h, oma * x);
}

__global__ void __launch_bounds__(256) aqe_forward_kernel(const float *__restrict__ x,
                                                          float *__restrict__ y, int64_t n,
                                                          float alpha, float oma, QParams q) {
    pdl_trigger();
    pdl_wait();
    const int64_t n4 = n >> 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    float4 *y4 = reinterpret_cast<float4 *>(y);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 v = __ldcs(x4 + i);
        float4 r;
        r.x = aqe_fwd1(v.x, alpha, oma, q);
        r.y = aqe_fwd1(v.y, alpha, oma, q);
        r.z = aqe_fwd1(v.z, alpha, oma, q);
        r.w = aqe_fwd1(v.w, alpha, oma, q);
        __stcs(y4 + i, r);
    }
    for (int64_t i = (n4 << 2) + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        y[i] = aqe_fwd1(x[i], alpha, oma, q);
}

// ---------------------------------------------------------------------------
// Stochastic AQE (Eq. our): alpha sign(a - z) + (1 - alpha) a with z ~ U[-1, 1)
// from a counter-based generator, so that any element's noise is a pure
// function of (seed, offset, index).
// ---------------------------------------------------------------------------

// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC 2011): ten rounds of two
// 64 x 64 -> 128-bit products on the counter, the key bumped by the Weyl
// constants between rounds.
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        const uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
        k0 += W0;
        k1 += W1;
    }
}

// z = (u >> 8) 2^-23 - 1: a point of the 2^-23 grid on [-1, 1), exact in fp32.
__device__ __forceinline__ float noise_of(uint32_t u) { return (float)(u >> 8) * 1.1920928955078125e-7f - 1.0f; }

__device__ __forceinline__ float aqe_sto1(float x, float z, float alpha, float oma) {
    return fmaf(alpha, x > z ? 1.0f : -1.0f, oma * x);      // sign(x - z), sign(0) = -1
}

// Thread = one block of eight elements: one Philox4x64-10 call (counter
// offset + block, key (seed, 0)) gives the eight 32-bit noise words, low half
// of each 64-bit output first; two 128-bit loads and stores.
__global__ void __launch_bounds__(256) aqe_forward_stochastic_kernel(const float *__restrict__ x,
                                                                     float *__restrict__ y, int64_t n,
                                                                     float alpha, float oma, uint64_t seed,
                                                                     uint64_t offset) {
    const int64_t nb = (n + 7) >> 3;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += stride) {
        const int64_t i0 = b << 3;
        const bool whole = i0 + 8 <= n;
        // the loads first, so that they are in flight during the generator's rounds
        float v[8];
        if (whole) {
            const float4 *x4 = reinterpret_cast<const float4 *>(x + i0);
            const float4 v0 = __ldcs(x4), v1 = __ldcs(x4 + 1);
            v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w;
            v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = i0 + j < n ? x[i0 + j] : 0.0f;
        }
        uint64_t c[4] = {offset + (uint64_t)b, 0ull, 0ull, 0ull};
        philox4x64_10(c, seed, 0ull);
        float r[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            r[2 * j] = aqe_sto1(v[2 * j], noise_of((uint32_t)c[j]), alpha, oma);
            r[2 * j + 1] = aqe_sto1(v[2 * j + 1], noise_of((uint32_t)(c[j] >> 32)), alpha, oma);
        }
        if (whole) {
            float4 *y4 = reinterpret_cast<float4 *>(y + i0);
            __stcs(y4, make_float4(r[0], r[1], r[2], r[3]));
            __stcs(y4 + 1, make_float4(r[4], r[5], r[6], r[7]));
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (i0 + j < n) y[i0 + j] = r[j];
        }
    }
}

__device__ __forceinline__ float aqe_bwd1(float x, float g, float two_alpha) {
    return (fabsf(x) <= 1.0f) ? g * two_alpha : 0.0f;
}

__global__ void __launch_bounds__(256) aqe_backward_kernel(const float *__restrict__ x,
                                                           const float *gy, float *gx,
                                                           int64_t n, float two_alpha) {
    pdl_trigger();
    pdl_wait();
    const int64_t n4 = n >> 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    const float4 *g4 = reinterpret_cast<const float4 *>(gy);
    float4 *o4 = reinterpret_cast<float4 *>(gx);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 v = __ldcs(x4 + i);
        float4 g = __ldcs(g4 + i);
        float4 r;
        r.x = aqe_bwd1(v.x, g.x, two_alpha);
        r.y = aqe_bwd1(v.y, g.y, two_alpha);
        r.z = aqe_bwd1(v.z, g.z, two_alpha);
        r.w = aqe_bwd1(v.w, g.w, two_alpha);
        __stcs(o4 + i, r);
    }
    for (int64_t i = (n4 << 2) + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        gx[i] = aqe_bwd1(x[i], gy[i], two_alpha);
}

__global__ void __launch_bounds__(256) aqe_backward_masked_kernel(const uint32_t *__restrict__ mask,
                                                                  const float *gy, float *gx,
                                                                  int64_t n, float two_alpha) {
    pdl_trigger();
    pdl_wait();
    const int64_t n4 = n >> 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float4 *g4 = reinterpret_cast<const float4 *>(gy);
    float4 *o4 = reinterpret_cast<float4 *>(gx);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        const uint32_t m = __ldg(mask + (i >> 3)) >> ((i & 7) * 4);
        float4 g = __ldcs(g4 + i);
        float4 r;
        r.x = (m & 1u) ? g.x * two_alpha : 0.0f;
        r.y = (m & 2u) ? g.y * two_alpha : 0.0f;
        r.z = (m & 4u) ? g.z * two_alpha : 0.0f;
        r.w = (m & 8u) ? g.w * two_alpha : 0.0f;
        __stcs(o4 + i, r);
    }
    for (int64_t i = (n4 << 2) + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t m = (mask[i >> 5] >> (i & 31)) & 1u;
        gx[i] = m ? gy[i] * two_alpha : 0.0f;
    }
}

// ---------------------------------------------------------------------------
// Quantize NCHW activations into a channel-contiguous layout: bit-planes
// [B][H][W][P][NW] (with the AQE forward output and the |x| <= 1 mask of the
// backward from the same load of x), E4M3 codes [B][H][W][C], or E2M1 codes
// [B][H][W][C/2].
//
// HBM bound: 4 B read per element.  A block takes PX pixels x 4 G channels
// of one image, one item of 4 channels x V pixels per thread: all of a
// thread's loads are independent and issue first (four 16-byte loads with
// V = 4, HW % 4 == 0; four 4-byte loads with V = 1), and a warp's loads cover
// whole 128-byte runs of a channel row.  The four channels of a pixel leave
// each thread as one 32-bit word (four E4M3 bytes, four E2M1 nibbles, or one
// nibble per plane in bytes 0 .. P - 1), exchanged through shared memory so
// that one thread assembles the 32 channels of a pixel.  Shared word of
// channel group g of pixel V j + i: [i][j][g], rows of G + 4 words (16-byte
// aligned, no conflict at G = 32, two-way below), or [i][g][j] where one block
// holds all of the channels in fewer than eight groups.  PX is 32 for 128 channels
// and more, and grows to 128 as the channels shrink to 32 and 1024 at 4 (V = 4), so
// that the 256 threads stay busy; images of 16 pixels and fewer (V = 1) take as
// few lanes as they have.  64 x 3 x 224 x 224, 1 bit: 59.7 us with 128 pixels,
// 12.1 with 1024; 256 x 1024 x 1 x 1 with forward and mask 23.5 and 3.6.
// A warp per 32 channels with its channels in a serial loop, as before, had
// one load in flight and few warps on small tensors: 256 x 512 x 14 x 14,
// 3 bits 107 us; 4 x 128 x 32 x 32, 1 bit 21 us (38 and 4 us here; instruction
// issue bounds the first, so plane bits are collected as signs of differences:
// 51 us with a compare and a select each).
// ---------------------------------------------------------------------------

enum QuantOut { OUT_PLANES, OUT_E4M3, OUT_E2M1 };

// A level's representation by selects alone (the thresholds descend, so each test that holds
// overrides the ones before): nested conditionals compile to divergent branches here.
template <int BITS, typename T>
__device__ __forceinline__ T pick(float m, const QParams &q, T zero, T l1, T l2, T l4) {
    if constexpr (BITS == 1) return l1;
    T r = zero;
    if constexpr (BITS == 2) {
        r = (m <= q.thr0) ? r : l1;
    } else {
        r = (m <= q.thr2) ? r : l1;
        r = (m <= q.thr1) ? r : l2;
        r = (m <= q.thr0) ? r : l4;
    }
    return r;
}

// Plane bits of one value's level, bit of plane k at bit 8 k.
template <int BITS>
__device__ __forceinline__ uint32_t plane_bytes(float u, const QParams &q) {
    const uint32_t neg = (u > 0.0f) ? 0u : 1u;
    if constexpr (BITS == 1) return neg;
    return pick<BITS, uint32_t>(fabsf(u), q, 0u, 0x100u | neg, 0x10000u | neg, 0x10100u | neg);
}

// The level's value (level_value with the bit width known: no integer conversion).
template <int BITS>
__device__ __forceinline__ float level_of(float u, const QParams &q) {
    if constexpr (BITS == 2) return ((u > q.thr0) ? 1.0f : 0.0f) - ((u < -q.thr0) ? 1.0f : 0.0f);
    constexpr float one = BITS == 3 ? 0.25f : 1.0f;
    const float s = (u > 0.0f) ? 1.0f : -1.0f;
    return s * pick<BITS, float>(fabsf(u), q, 0.0f, one, 0.5f, 1.0f);
}

// E2M1 nibble or E4M3 byte of the level.
template <int BITS, bool FP4>
__device__ __forceinline__ uint32_t code_of(float u, const QParams &q) {
    const uint32_t neg = (u > 0.0f) ? 0u : (FP4 ? 0x8u : 0x80u);
    constexpr uint32_t c1 = FP4 ? 2u : 0x38u, c2 = FP4 ? 4u : 0x40u, c4 = FP4 ? 6u : 0x48u;
    return pick<BITS, uint32_t>(fabsf(u), q, 0u, c1 | neg, c2 | neg, c4 | neg);
}

// SPLIT: SPLIT_WIDE as above, SPLIT_FEW all channels in fewer than eight groups (at most 16 channels), SPLIT_TINY
// fewer than 32 lanes per pixel run (V = 1, images of at most 16 pixels; a kernel of its own as its bitwise mask
// cost the others' scalar loads 10 %).
enum QuantSplit { SPLIT_WIDE, SPLIT_FEW, SPLIT_TINY };
template <int BITS, int OUT, int V, int SPLIT>
__global__ void __launch_bounds__(256, 4) quantize_kernel(const float *__restrict__ x, int B, int C, int HW, QParams q,
                                                          int lgl, int chunks, int cgs, int64_t total,
                                                          uint32_t *__restrict__ planes, uint8_t *__restrict__ codes,
                                                          float alpha, float oma, float *__restrict__ y,
                                                          uint32_t *__restrict__ mask, int mask_atomic) {
    constexpr bool FEW = SPLIT == SPLIT_FEW;
    __shared__ __align__(16) uint32_t sw[V * (256 + 4 * 32)];
    pdl_trigger();
    pdl_wait();
    const int LN = 1 << lgl, G = 256 >> lgl, PX = V << lgl;      // lanes per pixel run, channel groups, pixels
    const int RS = G + 4, IS = FEW ? 264 : LN * RS;               // shared strides of j and i
    const int NW = (C + 31) >> 5;
    const int j = threadIdx.x & (LN - 1), g = threadIdx.x >> lgl;

    struct Item {
        int64_t b;
        int cg, p0;
    };
    auto item = [&](int64_t t) {
        Item it;
        if (total < (1ll << 31)) {                                // 32-bit divisions
            const uint32_t u = (uint32_t)t, r = u / (uint32_t)cgs;
            it.cg = (int)(u - r * (uint32_t)cgs);
            const uint32_t bb = r / (uint32_t)chunks;
            it.p0 = (int)(r - bb * (uint32_t)chunks) * PX;
            it.b = bb;
        } else {
            const int64_t r = t / cgs;
            it.cg = (int)(t - r * cgs);
            it.b = r / chunks;
            it.p0 = (int)(r - it.b * chunks) * PX;
        }
        return it;
    };
    float nx[4][V];                                               // the next item's values, in flight
    auto load = [&](const Item &it) {
        const int p = it.p0 + V * j, c = it.cg * 4 * G + 4 * g;
        const float *src = x + (it.b * C + c) * HW + p;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = p < HW && c + k < C;                  // V = 4: all four pixels or none
            if constexpr (V == 4) {
                float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (in) f = __ldcs(reinterpret_cast<const float4 *>(src));
                nx[k][0] = f.x; nx[k][1] = f.y; nx[k][2] = f.z; nx[k][3] = f.w;
            } else {
                nx[k][0] = in ? __ldcs(src) : 0.0f;
            }
            src += HW;
        }
    };
    int64_t t = blockIdx.x;
    Item it = item(t);
    load(it);
    while (true) {
        const int cg = it.cg, p0 = it.p0, p = p0 + V * j, c = cg * 4 * G + 4 * g;
        const int64_t b = it.b;
        const bool pin = p < HW;
        const int64_t off = (b * C + c) * HW + p;
        float v[4][V];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < V; ++i) v[k][i] = nx[k][i];
        t += gridDim.x;
        const bool more = t < total;
        if (more) {
            it = item(t);
            load(it);
        }
        uint32_t w[V];
        if constexpr (OUT == OUT_PLANES) {
            // a comparison's bit is the sign of a difference (exact, and +0 at equality), shifted into the
            // pixel's nibble: two instructions; NaN, whose differences carry no sign, takes the selects
            float any = 0.0f;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                uint32_t s0 = 0u, s1 = 0u, s2 = 0u, s3 = 0u;
#pragma unroll
                for (int k = 3; k >= 0; --k) {
                    const float u = v[k][i] * q.scale;
                    asm("max.NaN.f32 %0, %0, %1;\n" : "+f"(any) : "f"(u));
                    if constexpr (BITS == 1) {
                        s0 = __funnelshift_l(__float_as_uint(0.0f - u), s0, 1);              // u > 0
                    } else if constexpr (BITS == 2) {
                        s0 = __funnelshift_l(__float_as_uint(u + q.thr0), s0, 1);            // u < -D
                        s1 = __funnelshift_l(__float_as_uint(q.thr0 - u), s1, 1);            // u > D
                    } else {
                        const float m = fabsf(u);
                        s0 = __funnelshift_l(__float_as_uint(u), s0, 1);                     // u < 0
                        s1 = __funnelshift_l(__float_as_uint(q.thr2 - m), s1, 1);            // |u| > D_3, D_2, D_1
                        s2 = __funnelshift_l(__float_as_uint(q.thr1 - m), s2, 1);
                        s3 = __funnelshift_l(__float_as_uint(q.thr0 - m), s3, 1);
                    }
                }
                if constexpr (BITS == 1) w[i] = s0 ^ 0xFu;
                else if constexpr (BITS == 2) w[i] = s0 | ((s0 | s1) << 8);
                else w[i] = (s0 & s1) | ((s1 & (~s2 | s3)) << 8) | (s2 << 16);
            }
            if (any != any) {
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    w[i] = 0u;
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[i] |= plane_bytes<BITS>(v[k][i] * q.scale, q) << k;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i) w[i] = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    const float u = v[k][i] * q.scale;
                    if constexpr (OUT == OUT_E2M1) w[i] |= code_of<BITS, true>(u, q) << (4 * k);
                    else w[i] |= code_of<BITS, false>(u, q) << (8 * k);
                }
            }
        }
        // this thread's channels of the tensor (planes: bits of channels past C stay zero)
        const int nc = max(0, min(4, C - c)), nst = pin ? nc : 0;
        if constexpr (OUT == OUT_PLANES) {
            const uint32_t cm = ((1u << nc) - 1u) * 0x010101u;
#pragma unroll
            for (int i = 0; i < V; ++i) w[i] &= cm;
        }
#pragma unroll
        for (int i = 0; i < V; ++i) sw[i * IS + (FEW ? (int)threadIdx.x : j * RS + g)] = w[i];
        if constexpr (OUT == OUT_PLANES) {
            if (y != nullptr) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (FEW && k >= nc) break;                    // the same in a whole warp
                    float yv[V];
#pragma unroll
                    for (int i = 0; i < V; ++i)
                        yv[i] = fmaf(alpha, level_of<BITS>(v[k][i] * q.scale, q), oma * v[k][i]);
                    if (k < nst) {
                        float *dst = y + off + (int64_t)k * HW;
                        if constexpr (V == 4) __stcs(reinterpret_cast<float4 *>(dst), make_float4(yv[0], yv[1], yv[2], yv[3]));
                        else __stcs(dst, yv[0]);
                    }
                }
            }
            if (SPLIT == SPLIT_TINY && mask != nullptr) {
                // no 32-pixel runs: bit by bit, four channels at once where their bits are neighbours
                uint32_t mb = 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) mb |= (k < nst && fabsf(v[k][0]) <= 1.0f ? 1u : 0u) << k;
                if (HW == 1 && mb != 0u) {
                    uint32_t *mw = mask + (off >> 5);
                    const uint32_t sh = (uint32_t)off & 31u, hi = __funnelshift_l(mb, 0u, sh);
                    atomicOr(mw, mb << sh);
                    if (hi) atomicOr(mw + 1, hi);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int64_t at = off + (int64_t)k * HW;
                        if ((mb >> k) & 1u) atomicOr(mask + (at >> 5), 1u << (at & 31));
                    }
                }
            } else if (mask != nullptr) {
                // 32 consecutive pixels of a channel row sit in 32 / V neighbouring lanes of one warp; lane k of
                // them stores channel k's word
                uint32_t mk = 0u;
                const int rl = V == 4 ? threadIdx.x & 7 : threadIdx.x & 31;       // lane in the run
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (FEW && k >= nc) break;
                    uint32_t m = 0u;
#pragma unroll
                    for (int i = 0; i < V; ++i) m |= (fabsf(v[k][i]) <= 1.0f ? 1u : 0u) << i;
                    m = pin ? m : 0u;
                    if constexpr (V == 4) {
                        m <<= rl * 4;
                        m |= __shfl_xor_sync(0xffffffffu, m, 1);
                        m |= __shfl_xor_sync(0xffffffffu, m, 2);
                        m |= __shfl_xor_sync(0xffffffffu, m, 4);
                    } else {
                        m = __ballot_sync(0xffffffffu, m);
                    }
                    mk = rl == k ? m : mk;
                }
                const int pr = p - V * rl;                        // the run's first pixel
                if (rl < nc && pr < HW) {
                    const int64_t at = (b * C + c + rl) * HW + pr;
                    uint32_t *mw = mask + (at >> 5);
                    const uint32_t sh = (uint32_t)at & 31u;
                    const uint32_t hi = __funnelshift_l(mk, 0u, sh);     // bits past the first word
                    if (!mask_atomic) {
                        *mw = mk;
                    } else {
                        atomicOr(mw, mk << sh);
                        if (hi) atomicOr(mw + 1, hi);
                    }
                }
            }
        }
        __syncthreads();
        // word wi (32 channels: shared words 8 wi .. + 7) of pixel px; neighbouring threads on neighbouring words
        const int lgn = FEW ? 0 : 5 - lgl, nwi = 1 << lgn;        // 32-channel words per pixel
        for (int e = threadIdx.x; e < PX * nwi; e += 256) {
            const int wi = e & (nwi - 1), px = e >> lgn;
            const int cw = FEW ? 0 : (cg * G >> 3) + wi;
            if (p0 + px >= HW || cw >= NW) continue;
            uint4 a = make_uint4(0u, 0u, 0u, 0u), d = a;
            if constexpr (FEW) {
                const uint32_t *src = sw + (px & (V - 1)) * IS + px / V;
                a.x = src[0];
                if (G > 1) a.y = src[LN];
                if (G > 2) { a.z = src[2 * LN]; a.w = src[3 * LN]; }
            } else {
                const uint32_t *src = sw + (px & (V - 1)) * IS + (px / V) * RS + 8 * wi;
                a = *reinterpret_cast<const uint4 *>(src);
                d = *reinterpret_cast<const uint4 *>(src + 4);
            }
            const uint32_t s[8] = {a.x, a.y, a.z, a.w, d.x, d.y, d.z, d.w};
            const int64_t pix = b * HW + p0 + px;
            if constexpr (OUT == OUT_PLANES) {
                // byte k of each word is plane k's nibble: fold pairs, then fours, then the eight
                const uint32_t e0 = s[0] | (s[1] << 4), e1 = s[2] | (s[3] << 4), e2 = s[4] | (s[5] << 4),
                               e3 = s[6] | (s[7] << 4);           // byte k: 8 channels of plane k
                uint32_t *dst = planes + pix * (BITS * NW) + cw;
#pragma unroll
                for (int k = 0; k < BITS; ++k) {
                    const uint32_t lo = __byte_perm(e0, e1, k | ((4 + k) << 4)), hi = __byte_perm(e2, e3, k | ((4 + k) << 4));
                    dst[k * NW] = __byte_perm(lo, hi, 0x5410);
                }
            } else if constexpr (OUT == OUT_E4M3) {
                uint4 *dst = reinterpret_cast<uint4 *>(codes + pix * C + cw * 32);
                dst[0] = a;
                if (C - cw * 32 > 16) dst[1] = d;
            } else {
                uint4 *dst = reinterpret_cast<uint4 *>(codes + ((pix * C + cw * 32) >> 1));
                *dst = make_uint4(s[0] | (s[1] << 16), s[2] | (s[3] << 16), s[4] | (s[5] << 16), s[6] | (s[7] << 16));
            }
        }
        if (!more) break;
        __syncthreads();
    }
}

template <int OUT>
static minw_status launch_quantize(const float *x, int B, int C, int64_t HW, const QParams &q, uint32_t *planes,
                                   uint8_t *codes, float alpha, float *y, uint32_t *mask, int mask_atomic,
                                   cudaStream_t s) {
    const bool vec = HW % 4 == 0 && minw_host::aligned16(x) && (!y || minw_host::aligned16(y));
    // pixels per block: 32 (lanes 8 x 4 pixels) for more than 64 channels, 64 and 128 below; scalar: 32, or as
    // many as an image of up to 16 has; up to 16 channels in one to four groups where the blocks of one warp a group
    // are more than two per SM, for 9 to 16 channels four (1024 pixels of 3 channels in 38 images 1.8 us, 2.0 in one
    // group; 57 images 2.5 and 2.0; 256 of 16 channels in 228 images 2.3 and 2.7; 304 images 2.6 and 2.0)
    const int sms = minw_host::num_sms() > 0 ? minw_host::num_sms() : 152;
    int lgl = !vec || C <= 32 ? 5 : C <= 64 ? 4 : 3;
    const int px32 = vec ? 128 : 32;
    const int64_t blocks32 = B * ((HW + px32 - 1) / px32);
    if (C <= 8 ? blocks32 > 2 * sms : C <= 16 && blocks32 >= 4 * sms) lgl = C <= 4 ? 8 : C <= 8 ? 7 : 6;
    if (!vec && HW <= 16)
        for (lgl = 0; (1 << lgl) < HW;) ++lgl;
    const int PX = (vec ? 4 : 1) << lgl, CG = 4 * (256 >> lgl);
    const int chunks = (int)((HW + PX - 1) / PX), cgs = (C - 1) / CG + 1;
    const int64_t total = (int64_t)B * chunks * cgs;
    // persistent: four blocks per SM, each with its next item's loads in flight behind the current one
    const dim3 grid((unsigned)(total < 4 * sms ? total : 4 * sms));
    typedef void (*Kernel)(const float *, int, int, int, QParams, int, int, int, int64_t, uint32_t *, uint8_t *, float,
                           float, float *, uint32_t *, int);
    constexpr int F = OUT != OUT_E2M1 ? SPLIT_FEW : SPLIT_WIDE;   // (E2M1 codes have 32 channels and more)
    static const Kernel wide[2][3] = {
        {quantize_kernel<1, OUT, 1, SPLIT_WIDE>, quantize_kernel<2, OUT, 1, SPLIT_WIDE>, quantize_kernel<3, OUT, 1, SPLIT_WIDE>},
        {quantize_kernel<1, OUT, 4, SPLIT_WIDE>, quantize_kernel<2, OUT, 4, SPLIT_WIDE>, quantize_kernel<3, OUT, 4, SPLIT_WIDE>}};
    static const Kernel few[2][3] = {
        {quantize_kernel<1, OUT, 1, F>, quantize_kernel<2, OUT, 1, F>, quantize_kernel<3, OUT, 1, F>},
        {quantize_kernel<1, OUT, 4, F>, quantize_kernel<2, OUT, 4, F>, quantize_kernel<3, OUT, 4, F>}};
    static const Kernel tiny[3] = {quantize_kernel<1, OUT, 1, SPLIT_TINY>, quantize_kernel<2, OUT, 1, SPLIT_TINY>,
                                   quantize_kernel<3, OUT, 1, SPLIT_TINY>};
    const Kernel kern = lgl > 5 ? few[vec][q.bits - 1] : !vec && lgl < 5 ? tiny[q.bits - 1] : wide[vec][q.bits - 1];
    // the pass of a training layer (forward and mask beside the planes) moves 2.5 times the bytes and reads through
    // L1: 256 x 512 x 14 x 14, 2 bits 58.3 -> 40.9 us; alone, the packing is bound by issue, and a change of the
    // carve-out delays a convolution behind it by 1 to 2 us
    const bool stream = y != nullptr && (int64_t)B * C * HW >= (1 << 22);
    if (minw_host::launch_pdl_stream(!stream, kern, grid, dim3(256), 0, s, x, B, C, (int)HW, q,
                                     lgl, chunks, cgs, total, planes, codes, alpha, 1.0f - alpha, y, mask,
                                     mask_atomic) != cudaSuccess)
        return MINW_ECUDA;
    return minw_host::launch_status();
}

// ---------------------------------------------------------------------------
// Weight packing: [O][C][kh][kw] -> [O][kh][kw][P][NW]; one thread per output
// word (the tensor is small and read once).
// ---------------------------------------------------------------------------

template <int P>
__global__ void pack_weights_kernel(const float *__restrict__ w, int O, int C, int kh, int kw,
                                    QParams q, const float *__restrict__ cscale,
                                    uint32_t *__restrict__ planes) {
    const int NW = (C + 31) >> 5;
    const int64_t total = (int64_t)O * kh * kw * NW;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int cw = (int)(t % NW);
        const int tap = (int)((t / NW) % (kh * kw));
        const int o = (int)(t / ((int64_t)NW * kh * kw));
        const float s = cscale ? cscale[o] : q.scale;
        uint32_t wd[P];
#pragma unroll
        for (int k = 0; k < P; ++k) wd[k] = 0u;
        const int cmax = min(32, C - cw * 32);
        for (int c = 0; c < cmax; ++c) {
            const float v = w[((int64_t)o * C + cw * 32 + c) * (kh * kw) + tap];
            const uint32_t pb = level_plane_bits(level_units(v * s, q), P);
#pragma unroll
            for (int k = 0; k < P; ++k) wd[k] |= ((pb >> k) & 1u) << c;
        }
        uint32_t *dst = planes + ((int64_t)o * kh * kw + tap) * (P * NW) + cw;
#pragma unroll
        for (int k = 0; k < P; ++k) dst[k * NW] = wd[k];
    }
}

// Weights [O][C][kh][kw] -> codes [O][kh][kw][C]: one thread per 16 channels
// (E4M3 bytes, or E2M1 nibbles with FP4).
template <bool FP4>
__global__ void weight_codes_kernel(const float *__restrict__ w, int O, int C, int kh, int kw, QParams q,
                                    const float *__restrict__ cscale, uint8_t *__restrict__ codes) {
    const int G = C >> 4;
    const int taps = kh * kw;
    const int64_t total = (int64_t)O * taps * G;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(t % G);
        const int tap = (int)((t / G) % taps);
        const int o = (int)(t / ((int64_t)G * taps));
        const float s = cscale ? cscale[o] : q.scale;
        uint32_t wd[4] = {0u, 0u, 0u, 0u};
        for (int c = 0; c < 16; ++c) {
            const float v = w[((int64_t)o * C + g * 16 + c) * taps + tap];
            const int u = level_units(v * s, q);
            if (FP4)
                wd[c >> 3] |= level_code_e2m1(u) << ((c & 7) * 4);
            else
                wd[c >> 2] |= (uint32_t)level_code_e4m3(u) << ((c & 3) * 8);
        }
        if (FP4)
            *reinterpret_cast<uint2 *>(codes + ((((int64_t)o * taps + tap) * C + g * 16) >> 1)) = make_uint2(wd[0], wd[1]);
        else
            *reinterpret_cast<uint4 *>(codes + ((int64_t)o * taps + tap) * C + g * 16) =
                make_uint4(wd[0], wd[1], wd[2], wd[3]);
    }
}

// Weights [O][C][kh][kw] -> bf16 level values in integer units [O][kh][kw][C]
// (1, 2 or 4 for the 3-bit magnitudes, all exact in bf16): one thread per
// 8 channels, one 128-bit store.
// out [O][kh][kw][Cp]: channels C .. Cp hold 0 (Cp >= C, a multiple of 8).
__global__ void weight_bf16_kernel(const float *__restrict__ w, int O, int C, int Cp, int kh, int kw, QParams q,
                                   const float *__restrict__ cscale, uint16_t *__restrict__ out) {
    const int G = Cp >> 3;
    const int taps = kh * kw;
    const int64_t total = (int64_t)O * taps * G;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(t % G);
        const int tap = (int)((t / G) % taps);
        const int o = (int)(t / ((int64_t)G * taps));
        const float s = cscale ? cscale[o] : q.scale;
        uint32_t wd[4];
        for (int j = 0; j < 4; ++j) {
            const int c = g * 8 + 2 * j;
            const float lo = c < C ? (float)level_units(w[((int64_t)o * C + c) * taps + tap] * s, q) : 0.0f;
            const float hi = c + 1 < C ? (float)level_units(w[((int64_t)o * C + c + 1) * taps + tap] * s, q) : 0.0f;
            wd[j] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
                    ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
        }
        *reinterpret_cast<uint4 *>(out + ((int64_t)o * taps + tap) * Cp + g * 8) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
    }
}

// fp32 NCHW -> bf16 NHWC, round to nearest even, out [B][HW][Cp]: channels
// C .. Cp hold 0 (Cp >= C).  A block takes 64 channels x 32 pixels of one
// image through shared memory: a thread has the loads of eight channels of
// its pixel in flight, and (VEC: Cp % 8 == 0, out 16-byte aligned) each
// pixel's channels leave in 16-byte stores.  256 x 256 x 16 x 16: 24 us with
// 32-channel tiles and 2-byte stores, 17 us here.
template <bool VEC>
__global__ void __launch_bounds__(256) to_bf16_nhwc_kernel(const float *__restrict__ x, int C, int Cp, int HW,
                                                           uint16_t *__restrict__ out) {
    __shared__ float tile[64][33];
    const int b = blockIdx.z, c0 = blockIdx.y * 64, p0 = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = c0 + ty + 8 * k, p = p0 + tx;
        v[k] = (c < C && p < HW) ? __ldg(x + ((int64_t)b * C + c) * HW + p) : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) tile[ty + 8 * k][tx] = v[k];
    __syncthreads();
    if constexpr (VEC) {
        const int g = threadIdx.x & 7, q = threadIdx.x >> 3, p = p0 + q, c = c0 + 8 * g;
        if (p < HW && c < Cp) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                w[e] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(tile[8 * g + 2 * e][q])) |
                       ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(tile[8 * g + 2 * e + 1][q])) << 16);
            *reinterpret_cast<uint4 *>(out + ((int64_t)b * HW + p) * Cp + c) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        for (int i = threadIdx.x; i < 64 * 32; i += 256) {
            const int p = p0 + (i >> 6), c = c0 + (i & 63);
            if (c < Cp && p < HW)
                out[((int64_t)b * HW + p) * Cp + c] = __bfloat16_as_ushort(__float2bfloat16_rn(tile[i & 63][i >> 6]));
        }
    }
}

}  // namespace minw

// ===========================================================================
// Host side
// ===========================================================================

namespace minw_host {

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool valid_quant(const minw_quant *q) {
    if (q == nullptr) return false;
    if (q->bits < 1 || q->bits > 3) return false;
    if (!(q->scale == q->scale)) return false;            // NaN
    if (q->bits == 2 && !(q->thr[0] >= 0.0f)) return false;
    if (q->bits == 3 && !(q->thr[0] >= q->thr[1] && q->thr[1] >= q->thr[2] && q->thr[2] >= 0.0f))
        return false;
    return true;
}

int num_sms() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms = 0;
    }
    return sms;
}

minw_status launch_status() {
    return cudaGetLastError() == cudaSuccess ? MINW_OK : MINW_ECUDA;
}

static int64_t grid_for(int64_t work_items, int threads) {
    const int sms = num_sms() > 0 ? num_sms() : 152;
    int64_t g = (work_items + threads - 1) / threads;
    const int64_t cap = (int64_t)sms * 8;   // 8 resident 256-thread CTAs per SM
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return g;
}

}  // namespace minw_host

using namespace minw;
using namespace minw_host;

extern "C" {

const char *minw_status_string(minw_status s) {
    switch (s) {
        case MINW_OK: return "ok";
        case MINW_EINVAL: return "invalid argument";
        case MINW_EUNSUPPORTED: return "unsupported shape or variant";
        case MINW_ECUDA: return "CUDA error";
        case MINW_ETIMEOUT: return "device-side wait timed out";
        case MINW_EDEVICE: return "no usable sm_103a device";
    }
    return "unknown status";
}

int32_t minw_version(void) { return 100; }

minw_status aqe_forward(const float *x, float *y, int64_t n, float alpha, const minw_quant *q,
                        void *stream) {
    if (n < 0 || !valid_quant(q) || !(alpha >= 0.0f && alpha <= 1.0f)) return MINW_EINVAL;
    if (n == 0) return MINW_OK;
    if (!x || !y || !aligned16(x) || !aligned16(y)) return MINW_EINVAL;
    const QParams qp = to_qparams(q);
    const int64_t g = grid_for(n / 4 + 1, 256);
    return launch_pdl_stream(false, aqe_forward_kernel, dim3((unsigned)g), dim3(256), 0, (cudaStream_t)stream, x, y, n,
                             alpha, 1.0f - alpha, qp) == cudaSuccess ? launch_status() : MINW_ECUDA;
}

minw_status aqe_forward_stochastic(const float *x, float *y, int64_t n, float alpha, uint64_t seed,
                                   uint64_t offset, void *stream) {
    if (n < 0 || !(alpha >= 0.0f && alpha <= 1.0f)) return MINW_EINVAL;
    if (n == 0) return MINW_OK;
    if (!x || !y || !aligned16(x) || !aligned16(y)) return MINW_EINVAL;
    const int64_t g = grid_for((n + 7) / 8, 256);
    aqe_forward_stochastic_kernel<<<(unsigned)g, 256, 0, (cudaStream_t)stream>>>(x, y, n, alpha, 1.0f - alpha, seed,
                                                                                offset);
    return launch_status();
}

minw_status aqe_backward(const float *x, const float *gy, float *gx, int64_t n, float alpha,
                         void *stream) {
    if (n < 0 || !(alpha >= 0.0f && alpha <= 1.0f)) return MINW_EINVAL;
    if (n == 0) return MINW_OK;
    if (!x || !gy || !gx || !aligned16(x) || !aligned16(gy) || !aligned16(gx)) return MINW_EINVAL;
    const int64_t g = grid_for(n / 4 + 1, 256);
    return launch_pdl_stream(false, aqe_backward_kernel, dim3((unsigned)g), dim3(256), 0, (cudaStream_t)stream, x, gy, gx,
                             n, 2.0f * alpha) == cudaSuccess ? launch_status() : MINW_ECUDA;
}

minw_status aqe_backward_masked(const uint32_t *mask, const float *gy, float *gx, int64_t n,
                                float alpha, void *stream) {
    if (n < 0 || !(alpha >= 0.0f && alpha <= 1.0f)) return MINW_EINVAL;
    if (n == 0) return MINW_OK;
    if (!mask || !gy || !gx || !aligned16(gy) || !aligned16(gx)) return MINW_EINVAL;
    const int64_t g = grid_for(n / 4 + 1, 256);
    return launch_pdl_stream(false, aqe_backward_masked_kernel, dim3((unsigned)g), dim3(256), 0, (cudaStream_t)stream,
                             mask, gy, gx, n, 2.0f * alpha) == cudaSuccess ? launch_status() : MINW_ECUDA;
}

minw_status aqe_quantize_pack(const float *x, int32_t B, int32_t C, int32_t H, int32_t W,
                              const minw_quant *q, uint32_t *planes, float alpha, float *y,
                              uint32_t *mask, void *stream) {
    if (B <= 0 || C <= 0 || H <= 0 || W <= 0 || !valid_quant(q)) return MINW_EINVAL;
    if (!x || !planes) return MINW_EINVAL;
    if (y && !(alpha >= 0.0f && alpha <= 1.0f)) return MINW_EINVAL;
    const int64_t HW = (int64_t)H * W;
    if (HW > (1ll << 30) || (int64_t)B * C * HW > (1ll << 40)) return MINW_EUNSUPPORTED;
    const QParams qp = to_qparams(q);
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n = (int64_t)B * C * HW;
    // a 32-pixel run of a channel row fills whole mask words when HW % 32 == 0; else its bits are merged into
    // the two words it may straddle
    const bool mask_atomic = mask && HW % 32 != 0;
    if (mask_atomic) {
        if (cudaMemsetAsync(mask, 0, sizeof(uint32_t) * ((n + 31) / 32), s) != cudaSuccess)
            return MINW_ECUDA;
    }
    return launch_quantize<OUT_PLANES>(x, B, C, HW, qp, planes, nullptr, alpha, y, mask, mask_atomic, s);
}

minw_status minw_pack_weights(const float *w, int32_t O, int32_t C, int32_t kh, int32_t kw,
                              const minw_quant *q, const float *channel_scale, uint32_t *planes,
                              void *stream) {
    if (O <= 0 || C <= 0 || kh <= 0 || kw <= 0 || !valid_quant(q) || !w || !planes)
        return MINW_EINVAL;
    const QParams qp = to_qparams(q);
    const int64_t words = (int64_t)O * kh * kw * ((C + 31) / 32);
    const int64_t g = grid_for(words, 256);
    cudaStream_t s = (cudaStream_t)stream;
    switch (q->bits) {
        case 1: pack_weights_kernel<1><<<(unsigned)g, 256, 0, s>>>(w, O, C, kh, kw, qp, channel_scale, planes); break;
        case 2: pack_weights_kernel<2><<<(unsigned)g, 256, 0, s>>>(w, O, C, kh, kw, qp, channel_scale, planes); break;
        default: pack_weights_kernel<3><<<(unsigned)g, 256, 0, s>>>(w, O, C, kh, kw, qp, channel_scale, planes); break;
    }
    return launch_status();
}

minw_status aqe_quantize_codes(const float *x, int32_t B, int32_t C, int32_t H, int32_t W,
                               const minw_quant *q, uint8_t *codes, void *stream) {
    if (B <= 0 || C <= 0 || H <= 0 || W <= 0 || !valid_quant(q) || !x || !codes) return MINW_EINVAL;
    if (C % 16 != 0 || !aligned16(codes)) return MINW_EUNSUPPORTED;
    const int64_t HW = (int64_t)H * W;
    if (HW > (1ll << 30)) return MINW_EUNSUPPORTED;
    return launch_quantize<OUT_E4M3>(x, B, C, HW, to_qparams(q), nullptr, codes, 0.0f, nullptr, nullptr, 0,
                                     (cudaStream_t)stream);
}

minw_status aqe_quantize_codes_e2m1(const float *x, int32_t B, int32_t C, int32_t H, int32_t W,
                                    const minw_quant *q, uint8_t *codes, void *stream) {
    if (B <= 0 || C <= 0 || H <= 0 || W <= 0 || !valid_quant(q) || !x || !codes) return MINW_EINVAL;
    if (C % 32 != 0 || !aligned16(codes)) return MINW_EUNSUPPORTED;
    const int64_t HW = (int64_t)H * W;
    if (HW > (1ll << 30)) return MINW_EUNSUPPORTED;
    return launch_quantize<OUT_E2M1>(x, B, C, HW, to_qparams(q), nullptr, codes, 0.0f, nullptr, nullptr, 0,
                                     (cudaStream_t)stream);
}

minw_status minw_pack_weight_codes(const float *w, int32_t O, int32_t C, int32_t kh, int32_t kw,
                                   const minw_quant *q, const float *channel_scale, uint8_t *codes,
                                   void *stream) {
    if (O <= 0 || C <= 0 || kh <= 0 || kw <= 0 || !valid_quant(q) || !w || !codes) return MINW_EINVAL;
    if (C % 16 != 0 || !aligned16(codes)) return MINW_EUNSUPPORTED;
    const int64_t items = (int64_t)O * kh * kw * (C / 16);
    const int64_t g = grid_for(items, 256);
    weight_codes_kernel<false><<<(unsigned)g, 256, 0, (cudaStream_t)stream>>>(w, O, C, kh, kw, to_qparams(q),
                                                                             channel_scale, codes);
    return launch_status();
}

minw_status minw_pack_weight_codes_e2m1(const float *w, int32_t O, int32_t C, int32_t kh, int32_t kw,
                                        const minw_quant *q, const float *channel_scale, uint8_t *codes,
                                        void *stream) {
    if (O <= 0 || C <= 0 || kh <= 0 || kw <= 0 || !valid_quant(q) || !w || !codes) return MINW_EINVAL;
    if (C % 16 != 0 || !aligned16(codes)) return MINW_EUNSUPPORTED;
    const int64_t items = (int64_t)O * kh * kw * (C / 16);
    const int64_t g = grid_for(items, 256);
    weight_codes_kernel<true><<<(unsigned)g, 256, 0, (cudaStream_t)stream>>>(w, O, C, kh, kw, to_qparams(q),
                                                                            channel_scale, codes);
    return launch_status();
}

minw_status minw_pack_weight_bf16_pad(const float *w, int32_t O, int32_t C, int32_t kh, int32_t kw, int32_t Cp,
                                      const minw_quant *q, const float *channel_scale, uint16_t *out, void *stream) {
    if (O <= 0 || C <= 0 || kh <= 0 || kw <= 0 || Cp < C || !valid_quant(q) || !w || !out) return MINW_EINVAL;
    if (Cp % 8 != 0 || !aligned16(out)) return MINW_EUNSUPPORTED;
    const int64_t items = (int64_t)O * kh * kw * (Cp / 8);
    const int64_t g = grid_for(items, 256);
    weight_bf16_kernel<<<(unsigned)g, 256, 0, (cudaStream_t)stream>>>(w, O, C, Cp, kh, kw, to_qparams(q),
                                                                     channel_scale, out);
    return launch_status();
}

minw_status minw_pack_weight_bf16(const float *w, int32_t O, int32_t C, int32_t kh, int32_t kw,
                                  const minw_quant *q, const float *channel_scale, uint16_t *out, void *stream) {
    if (C > 0 && C % 8 != 0) return MINW_EUNSUPPORTED;
    return minw_pack_weight_bf16_pad(w, O, C, kh, kw, C, q, channel_scale, out, stream);
}

minw_status minw_to_bf16_nhwc_pad(const float *x, int32_t B, int32_t C, int32_t H, int32_t W, int32_t Cp,
                                  uint16_t *out, void *stream) {
    if (B <= 0 || C <= 0 || H <= 0 || W <= 0 || Cp < C || !x || !out) return MINW_EINVAL;
    const int64_t HW = (int64_t)H * W;
    if (HW > (1ll << 30) || B > 65535 || (Cp + 31) / 32 > 65535) return MINW_EUNSUPPORTED;
    const dim3 grid((unsigned)((HW + 31) / 32), (unsigned)((Cp + 63) / 64), (unsigned)B);
    if (Cp % 8 == 0 && aligned16(out))
        to_bf16_nhwc_kernel<true><<<grid, 256, 0, (cudaStream_t)stream>>>(x, C, Cp, (int)HW, out);
    else
        to_bf16_nhwc_kernel<false><<<grid, 256, 0, (cudaStream_t)stream>>>(x, C, Cp, (int)HW, out);
    return launch_status();
}

minw_status minw_to_bf16_nhwc(const float *x, int32_t B, int32_t C, int32_t H, int32_t W, uint16_t *out,
                              void *stream) {
    return minw_to_bf16_nhwc_pad(x, B, C, H, W, C, out, stream);
}

}  // extern "C"
