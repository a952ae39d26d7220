// wres_fused.cu -- the forward of the weight-only residual network (see
// wonly_nets.cu) as one kernel: a CTA takes one image through the stem, every
// block and the head, with the activations in shared memory, the fp32
// shortcut in registers and the convolutions on the tensor cores.
//
// Layer by layer, each of the 110 convolutions of ResNet-110 is a few tiles of
// 16 .. 64 channels: launches, TMA round trips and re-reads of channels padded
// to 64 set its time (about 16 us each at batch 128), not its products.  Here
// a convolution reads its input in place and the next one starts as soon as
// the last epilogue warp is done.
//
// The activations sit in the padded plane layout of smem_conv.cuh, in which a
// 3x3 convolution's tap is a shifted start address.  The convolution entering
// a stage has stride 2: the last block of the stage before it writes its
// output split by row and column parity, where stride 2 is again contiguous.
//
// Warp roles (320 threads): warps 0-7 epilogue (TMEM lane quarter w & 3, half
// w >> 2 of the channels), warp 8 issues the MMAs, warp 9 streams each
// convolution's weights and BN map (one bulk copy) through two buffers.  An
// epilogue thread meets the same (pixel, channel) outputs in every block of a
// stage, so the fp32 shortcut stays in its registers.
//
// Measured: ResNet-110, 3-bit weights, batch 128: 1857 us layer by layer, 260
// us here (2.4 us per convolution).  What remains is each convolution's chain
// of issue, MMAs, TMEM reads and the barrier to the next one (tensor pipe 15 %
// active, 1.0 instructions a clock): a CTA has one image and nothing to overlap
// it with.
//
// Same operations as the layer-by-layer path: fp32 stem chain, bf16 inputs,
// fp32 accumulation, fmaf BN, one fp32 shortcut add, HardTanh.  Waits are
// bounded; one that runs out sets this file's error flag, after which the
// warps run to the end without waiting.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "smem_conv.cuh"
#include "wres_fused.cuh"

namespace minw {

namespace wfu {

using namespace smc;

constexpr int NT = EPI + 64;
constexpr int R0_BYTES = 40960, R1_BYTES = 36864;            // activation regions (32 x 32 images and smaller)
constexpr int WBUF_BYTES = 9 * 64 * 64 * 2 + 64 * 8;         // the largest convolution with its BN map
constexpr int SMEM_BYTES = R0_BYTES + R1_BYTES + 2 * WBUF_BYTES + 128;
constexpr int MAX_TILES = 8;
constexpr uint32_t D_COL = 256;                              // TMEM column of the shortcut convolution

struct Shared {
    uint64_t wfull[2], wempty[2], tile[MAX_TILES], dbar, act;
    uint32_t tmem;
};

// Streams of the three roles step through the same items: per block conv1,
// [the shortcut convolution entering stages 2 and 3], conv2; item i's weights
// sit in buffer i & 1 in the (i >> 1)-th filling of it.
__device__ __forceinline__ uint32_t item_bytes(int cin, int cout, int taps) {
    return (uint32_t)(taps * cin * cout * 2 + cout * 8);
}

// State of an epilogue thread.
struct Epi {
    const Args &p;
    Shared &sh;
    uint8_t *r0, *r1, *wb;
    uint32_t tmem;         // this warp's lane quarter
    int q, h, lane, b;
    int item = 0;
    uint32_t tph = 0u;     // phase bit of each tile barrier
    uint32_t dph = 0u;
    bool dead = false;

    __device__ __forceinline__ void zero(uint8_t *r, uint32_t bytes) {
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        for (uint32_t i = threadIdx.x * 16u; i < bytes; i += EPI * 16u) *reinterpret_cast<uint4 *>(r + i) = z;
    }
    // this thread's writes are visible to the tensor core; one arrival per warp
    __device__ __forceinline__ void publish() {
        fence_async_smem();
        fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(&sh.act);
    }
    // BN map of the current item's channels [c0, c0 + N), then the buffer's release by this warp
    template <int N>
    __device__ __forceinline__ void bn(int cin, int cout, int taps, int c0, float (&sc)[N], float (&sf)[N]) {
        warp_wait(&sh.wfull[item & 1], (item >> 1) & 1, p.wait_cycles, dead);
        const float *m = reinterpret_cast<const float *>(wb + (item & 1) * WBUF_BYTES + taps * cin * cout * 2);
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const float4 a = *reinterpret_cast<const float4 *>(m + c0 + i);
            const float4 s = *reinterpret_cast<const float4 *>(m + cout + c0 + i);
            sc[i] = a.x; sc[i + 1] = a.y; sc[i + 2] = a.z; sc[i + 3] = a.w;
            sf[i] = s.x; sf[i + 1] = s.y; sf[i + 2] = s.z; sf[i + 3] = s.w;
        }
        __syncwarp();
        if (lane == 0) bar_arrive(&sh.wempty[item & 1]);
        ++item;
    }
    template <int N>
    __device__ __forceinline__ void put(uint8_t *dst, uint32_t plane, const float (&v)[N]) {
#pragma unroll
        for (int k = 0; k < N / 8; ++k) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                w[e] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[8 * k + 2 * e])) |
                       ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[8 * k + 2 * e + 1])) << 16);
            *reinterpret_cast<uint4 *>(dst + k * plane) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    template <int N>
    __device__ __forceinline__ void keep(int index, int C, int S, int c0, int y, int x, const float (&v)[N]) {
        float *dst = p.keep[index] + (((int64_t)b * C + c0) * S + y) * S + x;
#pragma unroll
        for (int i = 0; i < N; ++i) dst[(int64_t)i * S * S] = v[i];
    }
};

// Epilogue side of one stage of n blocks with C channels and at most TM tiles;
// z: the fp32 block output of this thread's pixels and channels (stage 1: the
// stem's on entry).
template <int C, int TM, bool ENTER>
__device__ __forceinline__ void stage(Epi &e, int stg, int S, float (&z)[TM][C / 2]) {
    constexpr int N = C / 2;
    const Args &p = e.p;
    const Geo g(S);
    const int nt = g.tiles(), c0 = e.h * N;
    const int ry = (e.q * 32 + e.lane) >> 3, rx = e.lane & 7;
    const uint32_t cplane = (uint32_t)(c0 / 8);
    for (int j = 0; j < p.n; ++j) {
        const bool enter = ENTER && j == 0, last = j == p.n - 1;
        const int cin = enter ? C / 2 : C;
        float sc[N], sf[N];
        // conv1: HardTanh(BN) into R1
        e.bn<N>(cin, C, 9, c0, sc, sf);
        int y0 = 0, x0 = 0;
#pragma unroll
        for (int t = 0; t < TM; ++t) {
            if (t >= nt) break;
            warp_wait(&e.sh.tile[t], (e.tph >> t) & 1u, p.wait_cycles, e.dead);
            fence_after();
            float a[N];
            tmem_ld<N>(e.tmem + (uint32_t)(t * C + c0), a);
            const int y = y0 + ry, x = x0 + rx;
            x0 += 8;
            if (x0 >= S) { x0 = 0; y0 += 16; }
            if (y < S && x < S) {
#pragma unroll
                for (int i = 0; i < N; ++i) a[i] = fminf(fmaxf(fmaf(a[i], sc[i], sf[i]), -1.0f), 1.0f);
                e.put<N>(e.r1 + cplane * g.plane + g.at(y, x), g.plane, a);
            }
        }
        e.tph ^= (1u << nt) - 1u;
        e.publish();
        if (enter) {
            // the shortcut BN_d(conv_d(x)); with it both convolutions that read R0 have completed
            e.bn<N>(cin, C, 1, c0, sc, sf);
            warp_wait(&e.sh.dbar, e.dph, p.wait_cycles, e.dead);
            e.dph ^= 1u;
            fence_after();
#pragma unroll
            for (int t = 0; t < TM; ++t) {
                if (t >= nt) break;
                tmem_ld<N>(e.tmem + D_COL + (uint32_t)(t * C + c0), z[t]);
#pragma unroll
                for (int i = 0; i < N; ++i) z[t][i] = fmaf(z[t][i], sc[i], sf[i]);
            }
            e.zero(e.r0, (uint32_t)(C / 8) * g.plane);
            epi_sync();
        }
        // conv2: HardTanh(BN + shortcut) into R0, by parity where the next stage reads it
        const bool split = last && stg < 2;
        const Geo hg(S / 2);
        e.bn<N>(C, C, 9, c0, sc, sf);
        if (split) {
            e.zero(e.r0, (uint32_t)(4 * (C / 8)) * hg.plane);
            epi_sync();
        }
        y0 = x0 = 0;
#pragma unroll
        for (int t = 0; t < TM; ++t) {
            if (t >= nt) break;
            warp_wait(&e.sh.tile[t], (e.tph >> t) & 1u, p.wait_cycles, e.dead);
            fence_after();
            float a[N];
            tmem_ld<N>(e.tmem + (uint32_t)(t * C + c0), a);
            const int y = y0 + ry, x = x0 + rx;
            x0 += 8;
            if (x0 >= S) { x0 = 0; y0 += 16; }
            if (y < S && x < S) {
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const float v = fmaf(a[i], sc[i], sf[i]) + z[t][i];
                    z[t][i] = fminf(fmaxf(v, -1.0f), 1.0f);
                }
                if (split)
                    e.put<N>(e.r0 + ((uint32_t)((y & 1) * 2 + (x & 1)) * (C / 8) + cplane) * hg.plane +
                                 hg.at(y >> 1, x >> 1),
                             hg.plane, z[t]);
                else
                    e.put<N>(e.r0 + cplane * g.plane + g.at(y, x), g.plane, z[t]);
                if (p.keep != nullptr) e.keep<N>(1 + stg * p.n + j, C, S, c0, y, x, z[t]);
            }
        }
        e.tph ^= (1u << nt) - 1u;
        if (split) {
            epi_sync();                                  // every convolution that reads R1 has completed
            e.zero(e.r1, (uint32_t)(2 * C / 8) * hg.plane);
        }
        if (!(last && stg == 2)) e.publish();
    }
}

__global__ void __launch_bounds__(NT, 1) wres_fused_kernel(const __grid_constant__ Args p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((128u - (su32(smem_raw) & 127u)) & 127u);
    __shared__ Shared sh;
    uint8_t *r0 = smem, *r1 = smem + R0_BYTES, *wb = smem + R0_BYTES + R1_BYTES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            bar_init(&sh.wfull[i], 1);
            bar_init(&sh.wempty[i], 1 + EPI / 32);
        }
        for (int i = 0; i < MAX_TILES; ++i) bar_init(&sh.tile[i], 1);
        bar_init(&sh.dbar, 1);
        bar_init(&sh.act, EPI / 32);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(su32(&sh.tmem)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = sh.tmem;
    pdl_trigger();

    if (warp == 9) {
        // ---------------- weights: one bulk copy per item, two buffers ----------------
        bool dead = false;
        int item = 0;
        const uint8_t *src = p.blob;
        auto fetch = [&](int cin, int cout, int taps) {
            const int s = item & 1;
            const uint32_t bytes = item_bytes(cin, cout, taps);
            if (item >= 2) warp_wait(&sh.wempty[s], ((item >> 1) - 1) & 1, p.wait_cycles, dead);
            if (!dead && lane == 0) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(&sh.wfull[s])),
                             "r"(bytes)
                             : "memory");
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                        su32(wb + s * WBUF_BYTES)),
                    "l"(src), "r"(bytes), "r"(su32(&sh.wfull[s]))
                    : "memory");
            }
            __syncwarp();
            if (!dead) ++item;
            src += bytes;
        };
        for (int stg = 0, c = 16; stg < 3; ++stg, c *= 2)
            for (int j = 0; j < p.n; ++j) {
                const bool enter = stg > 0 && j == 0;
                fetch(enter ? c / 2 : c, c, 9);
                if (enter) fetch(c / 2, c, 1);
                fetch(c, c, 9);
            }
        // no copy may be in flight when the CTA ends
        bool d2 = false;
        for (int i = item > 2 ? item - 2 : 0; i < item; ++i)
            warp_wait(&sh.wfull[i & 1], (i >> 1) & 1, p.wait_cycles, d2);
    } else if (warp == 8) {
        // ---------------- MMA issuer ----------------
        bool dead = false;
        int item = 0;
        uint32_t actph = 0u;
        const uint32_t a0 = su32(r0), a1 = su32(r1), w0 = su32(wb);
        // one convolution (see issue): weights in, its tiles' MMAs and commits, the buffer's release
        auto conv = [&](auto cin_, auto cout_, auto taps_, auto par_, uint32_t abase, const Geo &g) {
            constexpr int CIN = decltype(cin_)::value, COUT = decltype(cout_)::value, TAPS = decltype(taps_)::value;
            constexpr bool PAR = decltype(par_)::value;
            warp_wait(&sh.wfull[item & 1], (item >> 1) & 1, p.wait_cycles, dead);
            if (!dead) {
                fence_after();
                issue<CIN, COUT, TAPS, PAR>(tmem + (TAPS == 1 ? D_COL : 0u), abase,
                                            w0 + (uint32_t)(item & 1) * WBUF_BYTES, g, TAPS == 9 ? sh.tile : nullptr,
                                            TAPS == 1 ? &sh.dbar : nullptr);
                mma_commit(&sh.wempty[item & 1]);
            }
            ++item;
        };
        auto ready = [&]() {
            warp_wait(&sh.act, actph, p.wait_cycles, dead);
            actph ^= 1u;
            fence_after();
        };
        auto run = [&](auto c_, auto enter_, int S) {
            constexpr int C = decltype(c_)::value;
            constexpr bool ENTER = decltype(enter_)::value;
            const Geo g(S);
            for (int j = 0; j < p.n; ++j) {
                ready();
                if (ENTER && j == 0) {
                    conv(Int<C / 2>{}, c_, Int<9>{}, Int<1>{}, a0, g);
                    conv(Int<C / 2>{}, c_, Int<1>{}, Int<1>{}, a0, g);
                } else {
                    conv(c_, c_, Int<9>{}, Int<0>{}, a0, g);
                }
                ready();
                conv(c_, c_, Int<9>{}, Int<0>{}, a1, g);
            }
        };
        run(Int<16>{}, Int<0>{}, p.hw);
        run(Int<32>{}, Int<1>{}, p.hw / 2);
        run(Int<64>{}, Int<1>{}, p.hw / 4);
    } else {
        // ---------------- epilogue warps: stem, blocks, head ----------------
        Epi e{p, sh, r0, r1, wb, tmem + ((uint32_t)((warp & 3) * 32) << 16), warp & 3, warp >> 2, lane, (int)blockIdx.x};
        const int hw = p.hw, npx = hw * hw;
        const Geo g(hw);
        float *img = reinterpret_cast<float *>(r1);           // [3][hw][hw], then the stem's weights [27][16]
        float *sw = img + 3 * npx;
        e.zero(r0, 2u * g.plane);
        for (int i = threadIdx.x; i < 27 * 16; i += EPI) sw[i] = __ldg(p.stem_wt + i);
        pdl_wait();
        const float *x = p.x + (int64_t)blockIdx.x * 3 * npx;
        for (int i = threadIdx.x; i < 3 * npx; i += EPI) img[i] = __ldg(x + i);
        epi_sync();
        float z1[MAX_TILES][8];
        {
            const int nt = g.tiles(), ntx = g.ntx(), c0 = e.h * 8;
            const int ry = (e.q * 32 + lane) >> 3, rx = lane & 7;
#pragma unroll
            for (int t = 0; t < MAX_TILES; ++t)
#pragma unroll
                for (int i = 0; i < 8; ++i) z1[t][i] = 0.0f;
            // one fmaf chain per output over (c, ky, kx), taps outside the image skipped
            for (int k = 0; k < 27; ++k) {
                const int c = k / 9, dy = (k / 3) % 3 - 1, dx = k % 3 - 1;
                const float4 wa = *reinterpret_cast<const float4 *>(sw + k * 16 + c0);
                const float4 wc = *reinterpret_cast<const float4 *>(sw + k * 16 + c0 + 4);
                const float w[8] = {wa.x, wa.y, wa.z, wa.w, wc.x, wc.y, wc.z, wc.w};
#pragma unroll
                for (int t = 0; t < MAX_TILES; ++t) {
                    if (t >= nt) break;
                    const int y = 16 * (t / ntx) + ry + dy, xx = 8 * (t % ntx) + rx + dx;
                    if (y >= 0 && y < hw && xx >= 0 && xx < hw) {
                        const float v = img[(c * hw + y) * hw + xx];
#pragma unroll
                        for (int i = 0; i < 8; ++i) z1[t][i] = fmaf(v, w[i], z1[t][i]);
                    }
                }
            }
            float sc[8], sf[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                sc[i] = __ldg(p.stem_scale + c0 + i);
                sf[i] = __ldg(p.stem_shift + c0 + i);
            }
#pragma unroll
            for (int t = 0; t < MAX_TILES; ++t) {
                if (t >= nt) break;
                const int y = 16 * (t / ntx) + ry, xx = 8 * (t % ntx) + rx;
                if (y < hw && xx < hw) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float v = fmaf(z1[t][i], sc[i], sf[i]);
                        if (v > 1.0f) v = 1.0f;
                        if (v < -1.0f) v = -1.0f;
                        z1[t][i] = v;
                    }
                    e.put<8>(r0 + (uint32_t)e.h * g.plane + g.at(y, xx), g.plane, z1[t]);
                    if (p.keep != nullptr) e.keep<8>(0, 16, hw, c0, y, xx, z1[t]);
                }
            }
        }
        epi_sync();                                           // the image is read: R1 becomes conv1's output
        e.zero(r1, 2u * g.plane);
        e.publish();
        stage<16, 8, false>(e, 0, hw, z1);
        float z2[2][16];
        stage<32, 2, true>(e, 1, hw / 2, z2);
        float z3[1][32];
        stage<64, 1, true>(e, 2, hw / 4, z3);
        // head: global average (one sum over the pixels in order, one division), fp32 linear layer, BN
        const int S = hw / 4, px = S * S;
        float *act = reinterpret_cast<float *>(r0);           // [64][px + 1]
        float *pooled = act + 64 * (px + 1);
        epi_sync();
        {
            const int y = (e.q * 32 + lane) >> 3, xx = lane & 7;
            if (y < S && xx < S)
#pragma unroll
                for (int i = 0; i < 32; ++i) act[(e.h * 32 + i) * (px + 1) + y * S + xx] = z3[0][i];
        }
        epi_sync();
        if (threadIdx.x < 64) {
            float s = 0.0f;
            for (int i = 0; i < px; ++i) s += act[threadIdx.x * (px + 1) + i];
            pooled[threadIdx.x] = s / (float)px;
        }
        epi_sync();
        for (int o = threadIdx.x; o < p.classes; o += EPI) {
            float acc = 0.0f;
            for (int k = 0; k < 64; ++k) acc = fmaf(pooled[k], __ldg(p.fc_wt + (int64_t)k * p.classes + o), acc);
            acc = acc + 0.0f;
            p.logits[(int64_t)blockIdx.x * p.classes + o] = fmaf(acc, __ldg(p.fc_scale + o), __ldg(p.fc_shift + o));
        }
        fence_before();
    }
    __syncthreads();
    if (warp == 8) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    }
}

// One convolution's item of the stream: its levels wb [O][taps][Cp] as
// [tap][C / 8][O][8], then the BN scale and shift.
__global__ void wres_item_kernel(const uint16_t *__restrict__ wb, const float *__restrict__ scale,
                                 const float *__restrict__ shift, int C, int Cp, int O, int taps,
                                 uint8_t *__restrict__ out) {
    const int n = taps * C * O;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int e = i & 7, o = (i >> 3) % O, r = (i >> 3) / O;
        const int kc = r % (C / 8), tap = r / (C / 8);
        reinterpret_cast<uint16_t *>(out)[i] = wb[((int64_t)o * taps + tap) * Cp + kc * 8 + e];
    }
    float *m = reinterpret_cast<float *>(out + (size_t)n * 2);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < O; i += gridDim.x * blockDim.x) {
        m[i] = scale[i];
        m[O + i] = shift[i];
    }
}

}  // namespace wfu

bool wres_fused_supported(int hw) { return hw >= 8 && hw <= 32 && hw % 4 == 0; }

size_t wres_item_bytes(int C, int O, int taps) { return (size_t)taps * C * O * 2 + (size_t)O * 8; }

minw_status wres_write_item(const uint16_t *wb, const float *scale, const float *shift, int C, int Cp, int O, int taps,
                            uint8_t *out, cudaStream_t s) {
    wfu::wres_item_kernel<<<(taps * C * O + 255) / 256, 256, 0, s>>>(wb, scale, shift, C, Cp, O, taps, out);
    return minw_host::launch_status();
}

minw_status launch_wres_fused(wfu::Args a, int B, cudaStream_t s) {
    a.wait_cycles = (long long)minw_host::plan_options().wait_cycles;
    if (cudaFuncSetAttribute(wfu::wres_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, wfu::SMEM_BYTES) !=
        cudaSuccess)
        return MINW_ECUDA;
    if (minw_host::launch_pdl(wfu::wres_fused_kernel, dim3((unsigned)B), dim3(wfu::NT), (size_t)wfu::SMEM_BYTES, s, a) !=
        cudaSuccess)
        return MINW_ECUDA;
    return minw_host::launch_status();
}

int take_wres_error() {
    int flag = 0;
    if (cudaMemcpyFromSymbol(&flag, smc::g_error, sizeof(int)) != cudaSuccess) return -1;
    if (flag) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(smc::g_error, &zero, sizeof(int)) != cudaSuccess) return -1;
    }
    return flag ? 1 : 0;
}

}  // namespace minw
