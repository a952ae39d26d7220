// smem_conv.cuh -- convolutions on activations held in shared memory, used by
// the one-kernel forwards of the weight-only networks (wres_fused.cu,
// wdense_fused.cu): barriers with bounded waits, the padded plane layout and
// its descriptors, and the MMAs of one convolution.
//
// Layout: planes of eight channels, [C / 8][(S + 2)(S + 1) + 1 pixels][8]
// bf16, image pixel (y, x) at (y + 1)(S + 1) + x + 1: one zero column serves
// as the right border of one row and the left border of the next, and rows -1
// and S are zero.  Without swizzle a matrix descriptor may start at any pixel
// (16 bytes), so the tap (dy, dx) of a 3x3 convolution is the same tile with a
// shifted start address.  An MMA tile is 16 image rows x 8 columns (M = 128:
// 8-pixel groups, one image row apart), K = 16 channels (two planes).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace minw {

namespace smc {

// Set when a bounded wait ran out (one flag per translation unit).
static __device__ int g_error = 0;

constexpr int EPI = 256;               // epilogue threads (warps 0-7)

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
        atomicExch(&g_error, 1);
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

template <int V>
struct Int {
    static constexpr int value = V;
};

// The MMAs of one convolution of TAPS = 9 or 1 taps, tile t in TMEM columns
// tmem + t COUT; each tile's completion goes to tile_bar[t], the whole one's to
// conv_bar (both nullable).  PAR: stride 2 on the parity images:
// input row 2 y + dy has parity dy & 1 and row y (y - 1 for dy = -1).
// Issued by the whole warp with uniform operands; the descriptors differ from
// their first ones by start-address steps (16-byte units) that unroll to one
// addition per MMA, as an N = 16 MMA takes few cycles itself.
template <int CIN, int COUT, int TAPS, bool PAR>
__device__ __forceinline__ void issue(uint32_t tmem, uint32_t abase, uint32_t wbase, const Geo &g, uint64_t *tile_bar,
                                      uint64_t *conv_bar) {
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(COUT >> 3) << 17) | (8u << 24);
    const uint64_t bd0 = desc_ns(wbase, (uint32_t)COUT * 16u, 128u);
    const uint32_t p16 = g.plane >> 4, img = (uint32_t)(CIN / 8) * p16;      // 16-byte units
    const int nt = g.tiles();
    int y0 = 0, x0 = 0;
    for (int t = 0; t < nt; ++t) {
        const uint64_t ad0 = desc_ns(abase + g.at(y0, x0), g.plane, (uint32_t)g.Wp * 16u);
        const uint32_t d = tmem + (uint32_t)(t * COUT);
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
        if (tile_bar != nullptr) mma_commit(tile_bar + t);
        x0 += 8;
        if (x0 >= g.S) { x0 = 0; y0 += 16; }
    }
    if (conv_bar != nullptr) mma_commit(conv_bar);
}


}  // namespace smc

}  // namespace minw
