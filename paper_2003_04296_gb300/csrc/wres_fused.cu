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
// Shared-memory activations: planes of eight channels, [C / 8][(S + 2)(S + 1)
// + 1 pixels][8] bf16, image pixel (y, x) at (y + 1)(S + 1) + x + 1: one zero
// column serves as the right border of one row and the left border of the
// next, and rows -1 and S are zero.  Without swizzle a matrix descriptor may
// start at any pixel (16 bytes), so the tap (dy, dx) of a 3x3 convolution is
// the same tile with a shifted start address: no im2col.  An MMA tile is 16
// image rows x 8 columns (M = 128: 8-pixel groups, one image row apart), K =
// 16 channels (two planes), N = the output channels.  The convolution entering
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

#include "wres_fused.cuh"

namespace minw {

__device__ int g_wres_error = 0;

namespace wfu {

constexpr int EPI = 256, NT = EPI + 64;
constexpr int R0_BYTES = 40960, R1_BYTES = 36864;            // activation regions (32 x 32 images and smaller)
constexpr int WBUF_BYTES = 9 * 64 * 64 * 2 + 64 * 8;         // the largest convolution with its BN map
constexpr int SMEM_BYTES = R0_BYTES + R1_BYTES + 2 * WBUF_BYTES + 128;
constexpr int MAX_TILES = 8;
constexpr uint32_t D_COL = 256;                              // TMEM column of the shortcut convolution

__device__ __forceinline__ uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t *b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(b)), "r"(n));
}
__device__ __forceinline__ void bar_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(su32(b)) : "memory");
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
// Bounded wait of a whole warp: sets dead (warp-uniform) and the error flag
// after limit SM clocks; returns at once when dead is set.
__device__ __forceinline__ void warp_wait(uint64_t *b, uint32_t parity, long long limit, bool &dead) {
    if (dead) return;
    bool ok = bar_try(b, parity);
    if (!ok) {
        const long long t0 = clock64();
        while (!(ok = bar_try(b, parity)) && clock64() - t0 <= limit) {
        }
    }
    if (!__all_sync(0xffffffffu, ok)) {
        atomicExch(&g_wres_error, 1);
        dead = true;
    }
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(EPI) : "memory"); }

// K-major operand without swizzle: 8-row groups sbo bytes apart (16 bytes per row), K steps of 16 bytes lbo apart.
__device__ __forceinline__ uint64_t desc_ns(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46);
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

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t ta, float (&o)[N]) {
    uint32_t v[N];
    if constexpr (N == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                     : "r"(ta));
    else if constexpr (N == 16)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15}, [%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(ta));
    else
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
              "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
              "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
            : "r"(ta));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = __uint_as_float(v[i]);
}

// One image of S x S pixels in the padded plane layout.
struct Geo {
    int S, Wp;
    uint32_t plane;        // bytes of one plane of eight channels
    __device__ __forceinline__ explicit Geo(int s) : S(s), Wp(s + 1), plane(((s + 2) * (s + 1) + 1) * 16u) {}
    __device__ __forceinline__ uint32_t at(int y, int x) const { return (uint32_t)((y + 1) * Wp + x + 1) * 16u; }
    __device__ __forceinline__ int ntx() const { return (S + 7) >> 3; }
    __device__ __forceinline__ int tiles() const { return ntx() * ((S + 15) >> 4); }
};

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

template <int V>
struct Int {
    static constexpr int value = V;
};

// The MMAs of one convolution, TAPS = 9 or 1 (the shortcut), tile t in TMEM
// columns t COUT (the shortcut's from D_COL).  Each tile's completion goes to
// its barrier (the shortcut's to dbar).  PAR: stride 2 on the parity images:
// input row 2 y + dy has parity dy & 1 and row y (y - 1 for dy = -1).
// Issued by the whole warp with uniform operands; the descriptors differ from
// their first ones by start-address steps (16-byte units) that unroll to one
// addition per MMA, as an N = 16 MMA takes few cycles itself.
template <int CIN, int COUT, int TAPS, bool PAR>
__device__ __forceinline__ void issue(uint32_t tmem, uint32_t abase, uint32_t wbase, const Geo &g, Shared &sh) {
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(COUT >> 3) << 17) | (8u << 24);
    const uint64_t bd0 = desc_ns(wbase, (uint32_t)COUT * 16u, 128u);
    const uint32_t p16 = g.plane >> 4, img = (uint32_t)(CIN / 8) * p16;      // 16-byte units
    const int nt = g.tiles();
    int y0 = 0, x0 = 0;
    for (int t = 0; t < nt; ++t) {
        const uint64_t ad0 = desc_ns(abase + g.at(y0, x0), g.plane, (uint32_t)g.Wp * 16u);
        const uint32_t d = tmem + (TAPS == 1 ? D_COL : 0u) + (uint32_t)(t * COUT);
#pragma unroll
        for (int tap = 0; tap < TAPS; ++tap) {
            const int dy = TAPS == 9 ? tap / 3 - 1 : 0, dx = TAPS == 9 ? tap % 3 - 1 : 0;
            const int oy = PAR ? (dy < 0 ? -1 : 0) : dy, ox = PAR ? (dx < 0 ? -1 : 0) : dx;
            const uint64_t ad = ad0 + (uint64_t)(int64_t)((PAR ? ((dy & 1) * 2 + (dx & 1)) * (int)img : 0) +
                                                          oy * g.Wp + ox);
            const uint64_t bd = bd0 + (uint64_t)(tap * (CIN / 8) * COUT);
#pragma unroll
            for (int k = 0; k < CIN / 16; ++k)
                mma_bf16(d, ad + (uint64_t)(2u * k * p16), bd + (uint64_t)(2 * k * COUT), idesc, tap + k > 0 ? 1u : 0u);
        }
        if (TAPS == 9) mma_commit(&sh.tile[t]);
        x0 += 8;
        if (x0 >= g.S) { x0 = 0; y0 += 16; }
    }
    if (TAPS == 1) mma_commit(&sh.dbar);
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
                issue<CIN, COUT, TAPS, PAR>(tmem, abase, w0 + (uint32_t)(item & 1) * WBUF_BYTES, g, sh);
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
    if (cudaMemcpyFromSymbol(&flag, g_wres_error, sizeof(int)) != cudaSuccess) return -1;
    if (flag) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_wres_error, &zero, sizeof(int)) != cudaSuccess) return -1;
    }
    return flag ? 1 : 0;
}

}  // namespace minw
