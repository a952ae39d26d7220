// conv_wgrad.cu -- the weight gradient of a convolutional training step,
// g_W[o][c][ky][kx] = sum over output pixels n of g~[n][o] a[n at tap][c], on
// the tensor cores straight from the NHWC operands the other products read.
//
// Both operands have the reduced dimension (pixels) outermost and channels
// contiguous, so they are MN-major MMA operands: a TMA box of 64 channels x 64
// pixels is 64 rows of 128 bytes (128-byte swizzle), a pixel per row, and an
// MMA takes 16 rows of it as its K.  The tap shift is a coordinate of the
// activation box (zero outside the image), stride 2 its element stride; no
// patches are written (302 MB written and read again at 256 -> 256 channels,
// 3x3, 256 images of 16 x 16: 165 us of 525), nor a transposed copy of g~.
//
// A CTA accumulates M = 128 MT output channels x N input channels x TPC taps in
// tensor memory (512 columns at most) over a slice of the pixels and writes
// fp32 partial sums [slice][tap][c][o] (lanes along o: whole lines); the
// update kernel adds the slices in order and applies the mask of Eq. weight,
// the step and the clip to W.  More channels per CTA mean fewer reads per
// product: at MT = 2, N = 256 a 64-pixel stage of 64 KB feeds 8 MMAs of N = 256,
// about what an SM's L2 bandwidth allows.
//
// Warp roles (192 threads): warp 0 TMA, warp 1 MMA and tensor memory, warps 2-5
// epilogue.  Every wait is bounded; one that runs out sets this file's error
// flag and the CTA winds down.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "kernels.cuh"

namespace minw {

__device__ int g_wgrad_error = 0;

namespace wg {

constexpr int NT = 192;
constexpr int KPX = 64;                      // pixels per stage
constexpr uint32_t BOX = KPX * 128;          // bytes of one 64-channel box

struct Params {
    int nbx, nby, nbb, bw, bh, bb;           // pixel boxes of bw x bh x bb = 64 output pixels
    int stride, pad, kw, ntaps;
    int MT, N, TPC;                          // 128-channel M tiles, input channels, taps per CTA
    int nm, nn, ntg;                         // M, N and tap groups
    int slices, S;
    uint32_t stage_bytes, idesc, tmem_cols;
    int O, C;
    float *part;                             // [slices][ntaps][C][O]
    long long wait_cycles;
};

__device__ __forceinline__ uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t *b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(b)), "r"(n));
}
__device__ __forceinline__ bool bar_try(uint64_t *b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 100000;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_wait(uint64_t *b, uint32_t parity, long long limit) {
    if (bar_try(b, parity)) return true;
    const long long t0 = clock64();
    while (!bar_try(b, parity)) {
        if (clock64() - t0 > limit) {
            atomicExch(&g_wgrad_error, 1);
            return false;
        }
    }
    return true;
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// MN-major operand in boxes of 64 channels (128-byte rows, 128-byte swizzle):
// the next 64 channels one box on, the next eight pixels 1024 bytes on.
__device__ __forceinline__ uint64_t desc_mn(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(BOX >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p, e;\n .reg .b32 r;\n setp.ne.b32 p, %4, 0;\n elect.sync r|e, 0xffffffff;\n"
                 " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("{\n .reg .pred e;\n .reg .b32 r;\n elect.sync r|e, 0xffffffff;\n"
                 " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(su32(bar))
                 : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(su32(bar))
        : "memory");
}

__global__ void __launch_bounds__(NT, 1)
    conv_wgrad_kernel(const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmA,
                      const __grid_constant__ Params p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (su32(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t full[8], empty[8], tfull;
    __shared__ uint32_t tmem_slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.S; ++s) {
            bar_init(&full[s], 1);
            bar_init(&empty[s], 1);
        }
        bar_init(&tfull, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(&tmem_slot)),
                     "r"(p.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_trigger();

    // (tap group, channel groups, slice) of this CTA; neighbouring CTAs share a slice's pixels
    int u = (int)blockIdx.x;
    const int tg = u % p.ntg;
    u /= p.ntg;
    const int gn = u % p.nn;
    u /= p.nn;
    const int gm = u % p.nm, sl = u / p.nm;
    const long long nk = (long long)p.nbx * p.nby * p.nbb;
    const int kb = (int)(sl * nk / p.slices), ke = (int)((sl + 1) * nk / p.slices);
    const int abox = 2 * p.MT, nbox = p.N / 64;

    if (warp == 0) {
        if (lane == 0) {
            pdl_wait();
            int s = 0, lap = 0, g = 0;
            for (int k = kb; k < ke; ++k, ++g) {
                if (lap > 0 && !bar_wait(&empty[s], (lap - 1) & 1, p.wait_cycles)) break;
                const int xb = k % p.nbx, yb = (k / p.nbx) % p.nby, bb = k / (p.nbx * p.nby);
                const int x = xb * p.bw * p.stride, y = yb * p.bh * p.stride, b = bb * p.bb;
                uint32_t dst = su32(smem) + (uint32_t)s * p.stage_bytes;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(&full[s])),
                             "r"(p.stage_bytes)
                             : "memory");
                for (int i = 0; i < abox; ++i, dst += BOX) tma_load_4d(dst, &tmG, &full[s], (gm * abox + i) * 64, x, y, b);
                for (int t = 0; t < p.TPC; ++t) {
                    const int tap = tg * p.TPC + t, ky = tap / p.kw, kx = tap - ky * p.kw;
                    for (int i = 0; i < nbox; ++i, dst += BOX)
                        tma_load_4d(dst, &tmA, &full[s], (gn * nbox + i) * 64, x - p.pad + kx, y - p.pad + ky, b);
                }
                if (++s == p.S) { s = 0; ++lap; }
            }
            // every load has landed before the CTA can exit
            for (int j = g > p.S ? g - p.S : 0; j < g; ++j)
                if (!bar_wait(&full[j % p.S], (j / p.S) & 1, p.wait_cycles)) break;
        }
    } else if (warp == 1) {
        int s = 0;
        uint32_t phase = 0u, acc = 0u;
        bool alive = true;
        const uint32_t base = su32(smem);
        for (int k = kb; k < ke; ++k) {
            if (!__all_sync(0xffffffffu, bar_wait(&full[s], phase, p.wait_cycles))) { alive = false; break; }
            fence_after();
            const uint64_t ad = desc_mn(base + (uint32_t)s * p.stage_bytes);
            const uint64_t bd = ad + (uint64_t)((uint32_t)abox * BOX >> 4);
            for (int t = 0; t < p.TPC; ++t)
                for (int m = 0; m < p.MT; ++m)
#pragma unroll
                    for (int q = 0; q < KPX / 16; ++q)
                        mma_bf16(tmem + (uint32_t)((t * p.MT + m) * p.N), ad + (uint64_t)((m * 2 * BOX + q * 2048) >> 4),
                                 bd + (uint64_t)(((uint32_t)(t * nbox) * BOX + q * 2048u) >> 4), p.idesc,
                                 q > 0 ? 1u : acc);
            acc = 1u;
            mma_commit(&empty[s]);
            if (++s == p.S) { s = 0; phase ^= 1u; }
        }
        if (alive) mma_commit(&tfull);
    } else {
        pdl_wait();                                       // the partial sums are shared with earlier kernels
        const bool ok = __all_sync(0xffffffffu, bar_wait(&tfull, 0u, p.wait_cycles));
        fence_after();
        const int q = warp & 3;
        for (int t = 0; t < p.TPC && ok; ++t)
            for (int m = 0; m < p.MT; ++m) {
                const int o = (gm * p.MT + m) * 128 + q * 32 + lane;
                float *dst = p.part + ((size_t)sl * p.ntaps + tg * p.TPC + t) * p.C * p.O + o;
                for (int n = 0; n < p.N; n += 32) {
                    uint32_t v[32];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                        "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
                        "[%32];\n"
                        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                          "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
                          "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
                          "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                        : "r"(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((t * p.MT + m) * p.N + n)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                    const int c0 = gn * p.N + n;
                    if (o < p.O) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (c0 + j < p.C) dst[(size_t)(c0 + j) * p.O] = __uint_as_float(v[j]);
                    }
                }
            }
        fence_before();
    }
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(p.tmem_cols));
    }
}

// W [O][C][taps] -= the step: the slices' partial sums added in order, then
// Eq. weight's mask, the update and the clip in the fp32 operations of
// aqe_backward and minw_sgd_clip.  A block takes 32 output channels x 8 RPT
// consecutive (c, tap) of their rows through shared memory, as the partial
// sums run along o and W along (c, tap); a thread has RPT rows of 16 / RPT slices
// in flight (one element and W strided per thread: 35 us at 256 x 256 x 3 x 3 in
// 16 slices; 19 us here, cold).  A small gradient has a slice per SM and few
// blocks: 64 x 39 x 1 x 1, 96 images of 24 x 24, RPT = 4 the step 119.5 us, RPT = 1
// 56.2.
template <int RPT>
__global__ void __launch_bounds__(256) wgrad_update_kernel(const float *__restrict__ part, int slices, int ntaps, int C,
                                                           int O, float lr, float two_alpha, float *__restrict__ W) {
    constexpr int ROWS = 8 * RPT, E = 16 / RPT;
    __shared__ float tile[ROWS][33];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int R = C * ntaps, r0 = blockIdx.x * ROWS;
    const size_t n = (size_t)R * O;
    pdl_wait();                       // (and no early start of a dependent: it may read W before it waits)
    for (int o0 = blockIdx.y * 32; o0 < O; o0 += gridDim.y * 32) {
        float acc[RPT];
        const float *src[RPT];
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = min(r0 + row + 8 * k, R - 1), c = r / ntaps, tap = r - c * ntaps;
            src[k] = part + ((size_t)tap * C + c) * O + min(o0 + lane, O - 1);
            acc[k] = 0.0f;
        }
        int s = 0;
        for (; s + E <= slices; s += E) {
            float v[E][RPT];
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int k = 0; k < RPT; ++k) v[e][k] = __ldcs(src[k] + (size_t)(s + e) * n);
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int k = 0; k < RPT; ++k) acc[k] += v[e][k];
        }
        for (; s < slices; ++s)
#pragma unroll
            for (int k = 0; k < RPT; ++k) acc[k] += __ldcs(src[k] + (size_t)s * n);
#pragma unroll
        for (int k = 0; k < RPT; ++k) tile[row + 8 * k][lane] = acc[k];
        __syncthreads();
        for (int i = threadIdx.x; i < ROWS * 32; i += 256) {
            const int r = i % ROWS, o = i / ROWS;
            if (r0 + r < R && o0 + o < O) {
                float *w = W + (size_t)(o0 + o) * R + r0 + r;
                const float wi = *w;
                const float gm = (fabsf(wi) <= 1.0f) ? tile[r][o] * two_alpha : 0.0f;
                *w = fminf(1.0f, fmaxf(-1.0f, fmaf(-lr, gm, wi)));
            }
        }
        __syncthreads();
    }
}

// Tiles and slices of a shape: pixel boxes that waste least, M of up to 256
// output channels, N of up to 256 input channels, and as many taps as tensor
// memory and a 64 KB stage take (whole groups only); then pixel slices up to
// one CTA per SM, of at least four stages.
static void plan(const WgradArgs &a, Params &p) {
    p = Params{};
    long long best = -1;
    for (int bw = 1; bw <= KPX; bw *= 2)
        for (int bh = 1; bw * bh <= KPX; bh *= 2) {
            const int bb = KPX / (bw * bh);
            const long long n = (long long)((a.Wo + bw - 1) / bw) * ((a.Ho + bh - 1) / bh) * ((a.B + bb - 1) / bb);
            if (best < 0 || n <= best) {                  // ties: the widest rows
                best = n;
                p.bw = bw; p.bh = bh; p.bb = bb;
            }
        }
    p.nbx = (a.Wo + p.bw - 1) / p.bw;
    p.nby = (a.Ho + p.bh - 1) / p.bh;
    p.nbb = (a.B + p.bb - 1) / p.bb;
    p.stride = a.stride; p.pad = a.pad; p.kw = a.kw; p.ntaps = a.kh * a.kw;
    p.O = a.O; p.C = a.C;
    p.MT = a.O > 128 ? 2 : 1;
    p.nm = (a.O + 128 * p.MT - 1) / (128 * p.MT);
    p.nn = (a.C + 255) / 256;
    p.N = ((a.C + p.nn - 1) / p.nn + 63) / 64 * 64;
    p.TPC = 1;
    for (int t = 2; t <= p.ntaps; ++t)
        if (p.ntaps % t == 0 && t * p.MT * p.N <= 512 && (uint32_t)(2 * p.MT + t * (p.N / 64)) * BOX <= 64 * 1024)
            p.TPC = t;
    p.ntg = p.ntaps / p.TPC;
    p.stage_bytes = (uint32_t)(2 * p.MT + p.TPC * (p.N / 64)) * BOX;
    p.S = std::min(8, (int)(216 * 1024 / p.stage_bytes));
    p.tmem_cols = 32;
    while ((int)p.tmem_cols < p.TPC * p.MT * p.N) p.tmem_cols *= 2;
    // D fp32, A and B bf16, both MN-major (bits 15 and 16)
    p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(p.N >> 3) << 17) | (8u << 24);
    const int sms = minw_host::num_sms() > 0 ? minw_host::num_sms() : 152;
    const long long tiles = (long long)p.nm * p.nn * p.ntg;
    long long sl = std::min<long long>(sms / tiles, best / 4);
    p.slices = (int)std::max<long long>(1, sl);
}

}  // namespace wg

size_t conv_wgrad_workspace_bytes(const WgradArgs &a) {
    wg::Params p;
    wg::plan(a, p);
    return sizeof(float) * (size_t)p.slices * p.ntaps * p.C * p.O;
}

minw_status launch_conv_wgrad(const WgradArgs &a, float *part, float lr, float two_alpha, float *W, cudaStream_t s) {
    wg::Params p;
    wg::plan(a, p);
    p.part = part;
    p.wait_cycles = (long long)minw_host::plan_options().wait_cycles;
    minw_host::EncodeTiledFn enc = minw_host::tensor_map_encoder();
    if (enc == nullptr) return MINW_ECUDA;
    CUtensorMap tmG, tmA;
    const cuuint32_t sd = (cuuint32_t)a.stride;
    const cuuint32_t box[4] = {64u, (cuuint32_t)p.bw * sd, (cuuint32_t)p.bh * sd, (cuuint32_t)p.bb};
    const cuuint32_t es[4] = {1u, sd, sd, 1u};
    auto encode = [&](CUtensorMap *m, const uint16_t *ptr, int C, int H, int W_) {
        const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W_, (cuuint64_t)H, (cuuint64_t)a.B};
        const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W_ * C * 2, (cuuint64_t)H * W_ * C * 2};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, const_cast<uint16_t *>(ptr), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (!encode(&tmG, a.gd, a.Op, a.Hd, a.Wd) || !encode(&tmA, a.ab, a.C, a.H, a.W)) return MINW_ECUDA;
    const size_t smem = (size_t)p.S * p.stage_bytes + 1024;
    if (!minw_host::allow_shared(reinterpret_cast<const void *>(wg::conv_wgrad_kernel), 220 * 1024)) return MINW_ECUDA;
    const unsigned grid = (unsigned)(p.nm * p.nn * p.ntg * p.slices);
    if (minw_host::launch_pdl(wg::conv_wgrad_kernel, dim3(grid), dim3(wg::NT), smem, s, tmG, tmA, p) != cudaSuccess)
        return MINW_ECUDA;
    // narrow blocks where there are fewer than two wide ones per SM (the step at 64 images of 16 x 16, 128 -> 256
    // channels, 288 wide blocks: 88.1 -> 83.0 us; above, the same time)
    const int R = p.C * p.ntaps, ob = (p.O + 31) / 32;
    const bool narrow = (long long)((R + 31) / 32) * ob < 2 * (minw_host::num_sms() > 0 ? minw_host::num_sms() : 152);
    const dim3 ugrid((unsigned)(narrow ? (R + 7) / 8 : (R + 31) / 32), (unsigned)std::min(ob, 65535));
    if (minw_host::launch_pdl_stream(false, narrow ? wg::wgrad_update_kernel<1> : wg::wgrad_update_kernel<4>, ugrid,
                                     dim3(256), 0, s, (const float *)part, p.slices, p.ntaps, p.C, p.O, lr, two_alpha,
                                     W) != cudaSuccess)
        return MINW_ECUDA;
    return minw_host::launch_status();
}

int take_wgrad_error() {
    int flag = 0;
    if (cudaMemcpyFromSymbol(&flag, g_wgrad_error, sizeof(int)) != cudaSuccess) return -1;
    if (flag) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_wgrad_error, &zero, sizeof(int)) != cudaSuccess) return -1;
    }
    return flag ? 1 : 0;
}

}  // namespace minw
