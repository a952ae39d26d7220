// wdense_fused.cu -- the forward of the weight-only DenseNet-BC (see
// wonly_nets.cu) as one kernel: a CTA takes one image through the stem, every
// bottleneck layer, the transitions and the head.
//
// Layer by layer, the 98 convolutions of DenseNet-100 are narrow (48 and 12
// output channels) and launch and TMA latency set their time.  Here the
// bottleneck activation (4 k channels) never leaves shared memory, and one
// layer's 1x1 convolution runs while the layer before it is still in its
// epilogue, up to the channels that layer adds.
//
// Features stay in global memory (L2), as planes of eight channels [plane][y
// S + x][8]: a block's 216 channels of 32 x 32 pixels do not fit an SM.  The
// 1x1 convolution streams them in stages of up to 16 image rows through a ring
// (bulk copies), each stage feeding the tiles of its rows; tiles are those of
// smem_conv.cuh (16 rows x 8 columns), so a thread meets the same pixels in
// the 1x1 convolution, the 3x3 convolution and the 2x2 pool.  Channels past a
// layer's inputs, up to the padding of K, hold zeros or an earlier pass's
// finite values against zero weights.
//
// TMEM (512 columns): tile t of a 1x1 convolution at t 4 k, of a 3x3 at
// T 4 k + 16 t; a transition takes tiles of one stage of rows at a time, pad16(c / 2)
// columns each, and its weights sit in the bottleneck's region, free by then.
//
// Warp roles (352 threads): warps 0-7 epilogue (lane quarter w & 3, half w >> 2
// of the channels or tiles), warp 8 MMAs, warp 9 feature stages, warp 10
// weights.  Every item (layer or transition) ends with the epilogue warps'
// arrivals on fready, after which its output may be copied.
//
// Measured: DenseNet-100, 3-bit weights, batch 128: 1475 us layer by layer,
// 426 us here.  Block 1 holds most of it: each layer streams its inputs, 256 KB
// per image on average, and 128 CTAs together draw about 5 TB/s from L2.
//
// Same operations as the layer-by-layer path: fp32 stem chain, bf16 features,
// fp32 accumulation, fmaf BN, HardTanh, the pool's order of sums.  Waits are
// bounded; one that runs out sets this file's error flag, after which the
// warps run to the end without waiting.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "smem_conv.cuh"
#include "wdense_fused.cuh"

namespace minw {

namespace dfu {

using namespace smc;

constexpr int NT = EPI + 96;
constexpr int RING = 4;
constexpr uint32_t STAGE_BYTES = 16384;
constexpr int MAX_TILES = 8;
constexpr uint32_t SMEM_LIMIT = 227 * 1024 - 1024;

// Bottleneck region: 4 k channels of an hw x hw image in the plane layout.
__host__ __device__ constexpr uint32_t h_bytes(int k, int hw) {
    return (uint32_t)(k / 2) * (uint32_t)((hw + 2) * (hw + 1) + 1) * 16u;
}
__host__ __device__ constexpr uint32_t item_bytes(int C, int O, int taps) {
    return (uint32_t)taps * (uint32_t)((C + 15) / 16 * 2) * (uint32_t)((O + 15) / 16 * 16) * 16u +
           (uint32_t)((O + 15) / 16 * 16) * 8u;
}

struct Shared {
    uint64_t rfull[RING], rempty[RING], w1full, w1empty, w3full, w3empty, wtfull, hb[2], hready, t3[MAX_TILES], fready;
    uint32_t tmem;
};

// Rows of one block's feature stages: SH rows (16, or the image's fewer), KS K steps (of two planes) per stage.
struct Feat {
    int S, nty;
    __device__ __forceinline__ explicit Feat(int s) : S(s), nty((s + 15) >> 4) {}
    __device__ __forceinline__ int rows(int ty) const { return min(16, S - 16 * ty); }
    __device__ __forceinline__ int ks() const {
        return nty > 1 ? 1 : max(1, min(8, (int)STAGE_BYTES / (S * S * 32)));
    }
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(su32(bar))
                 : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}
__device__ __forceinline__ void bn8(const float *m, int np, int c, float (&sc)[8], float (&sf)[8]) {
#pragma unroll
    for (int i = 0; i < 8; i += 4) {
        const float4 a = *reinterpret_cast<const float4 *>(m + c + i);
        const float4 s = *reinterpret_cast<const float4 *>(m + np + c + i);
        sc[i] = a.x; sc[i + 1] = a.y; sc[i + 2] = a.z; sc[i + 3] = a.w;
        sf[i] = s.x; sf[i + 1] = s.y; sf[i + 2] = s.z; sf[i + 3] = s.w;
    }
}

// K4 = growth / 4: a half of the epilogue warps holds K4 planes of the bottleneck.
template <int K4>
__global__ void __launch_bounds__(NT, 1) wdense_fused_kernel(const __grid_constant__ Args p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((128u - (su32(smem_raw) & 127u)) & 127u);
    __shared__ Shared sh;
    constexpr int K = 4 * K4, N1 = 4 * K;                    // growth, bottleneck channels
    constexpr uint32_t W3_BYTES = item_bytes(N1, K, 9);
    uint8_t *ring = smem, *hbuf = ring + RING * STAGE_BYTES, *w1 = hbuf + ((h_bytes(K, p.hw) + 127u) & ~127u),
            *w3 = w1 + p.w1_bytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t img = blockIdx.x;
    if (threadIdx.x == 0) {
        for (int i = 0; i < RING; ++i) {
            bar_init(&sh.rfull[i], 1);
            bar_init(&sh.rempty[i], 1);
        }
        bar_init(&sh.w1full, 1);
        bar_init(&sh.w3full, 1);
        bar_init(&sh.wtfull, 1);
        bar_init(&sh.w1empty, 1 + EPI / 32);
        bar_init(&sh.w3empty, 1 + EPI / 32);
        for (int i = 0; i < 2; ++i) bar_init(&sh.hb[i], 1);
        bar_init(&sh.hready, EPI / 32);
        for (int i = 0; i < MAX_TILES; ++i) bar_init(&sh.t3[i], 1);
        bar_init(&sh.fready, EPI / 32);
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
        // ---------------- feature stages ----------------
        bool dead = false;
        int s = 0, lap = 0, issued = 0;
        uint32_t fph = 0u;
        for (int b = 0; b < 3; ++b) {
            const Feat f(p.hw >> b);
            const int px = f.S * f.S, KS = f.ks();
            const uint8_t *base = reinterpret_cast<const uint8_t *>(p.F[b] + img * p.planes[b] * px * 8);
            for (int l = 0; l < p.layers + (b < 2); ++l) {
                const int cin = p.cstart[b] + l * K, nk = (cin + 15) >> 4;
                const int from = l == 0 ? 0 : cin - K;        // first channel the item before this one wrote
                bool waited = false;
                for (int ty = 0; ty < f.nty; ++ty) {
                    const uint32_t chunk = (uint32_t)(f.rows(ty) * f.S) * 16u;
                    for (int ks = 0; ks < nk; ks += KS) {
                        const int n = min(KS, nk - ks);
                        if (!waited && 16 * (ks + n) > from) {
                            warp_wait(&sh.fready, fph, p.wait_cycles, dead);
                            fph ^= 1u;
                            waited = true;
                            asm volatile("fence.proxy.async;\n" ::: "memory");
                        }
                        if (lap > 0) warp_wait(&sh.rempty[s], (lap - 1) & 1, p.wait_cycles, dead);
                        if (!dead && lane == 0) {
                            const uint32_t dst = su32(ring) + (uint32_t)s * STAGE_BYTES;
                            expect_tx(&sh.rfull[s], (uint32_t)(2 * n) * chunk);
                            if (f.nty == 1) {                 // whole planes, contiguous
                                bulk_load(dst, base + (size_t)(2 * ks) * px * 16, (uint32_t)(2 * n) * chunk, &sh.rfull[s]);
                            } else {                          // KS == 1: the rows of two planes
                                for (int q = 0; q < 2; ++q)
                                    bulk_load(dst + (uint32_t)q * chunk,
                                              base + ((size_t)(2 * ks + q) * px + (size_t)(16 * ty) * f.S) * 16, chunk,
                                              &sh.rfull[s]);
                            }
                        }
                        __syncwarp();
                        if (!dead) ++issued;
                        if (++s == RING) { s = 0; ++lap; }
                    }
                }
            }
        }
        bool d2 = false;                                      // no copy may be in flight when the CTA ends
        for (int i = max(0, issued - RING); i < issued; ++i)
            warp_wait(&sh.rfull[i % RING], (i / RING) & 1, p.wait_cycles, d2);
    } else if (warp == 10) {
        // ---------------- weights ----------------
        bool dead = false;
        const uint8_t *src = p.blob;
        int n1 = 0, n3 = 0, nt = 0;
        auto fetch = [&](uint64_t *full, uint64_t *empty, int used, uint8_t *dst, uint32_t bytes, int &count) {
            if (used > 0) warp_wait(empty, (used - 1) & 1, p.wait_cycles, dead);
            if (!dead && lane == 0) {
                expect_tx(full, bytes);
                bulk_load(su32(dst), src, bytes, full);
            }
            __syncwarp();
            if (!dead) ++count;
            src += bytes;
        };
        for (int b = 0; b < 3; ++b) {
            for (int l = 0; l < p.layers; ++l) {
                fetch(&sh.w1full, &sh.w1empty, b * p.layers + l, w1, item_bytes(p.cstart[b] + l * K, N1, 1), n1);
                fetch(&sh.w3full, &sh.w3empty, b * p.layers + l, w3, W3_BYTES, n3);
            }
            // the transition's weights replace the bottleneck once the last 3x3 convolution is done
            if (b < 2)
                fetch(&sh.wtfull, &sh.w3empty, (b + 1) * p.layers, hbuf, item_bytes(p.cfin[b], p.cfin[b] / 2, 1), nt);
        }
        bool d2 = false;
        if (n1) warp_wait(&sh.w1full, (n1 - 1) & 1, p.wait_cycles, d2);
        if (n3) warp_wait(&sh.w3full, (n3 - 1) & 1, p.wait_cycles, d2);
        if (nt) warp_wait(&sh.wtfull, (nt - 1) & 1, p.wait_cycles, d2);
    } else if (warp == 8) {
        // ---------------- MMA issuer ----------------
        bool dead = false;
        int s = 0, item = 0, layer = 0;
        uint32_t rph = 0u, hph = 0u;
        const uint32_t rbase = su32(ring);
        // rows ty of a 1x1 convolution with np output columns per tile, tile tx of the rows at column col + tx np
        // (unrolled over the tiles of a row: uniform descriptors plus constants)
        auto rows_n = [&](auto ntx_, const Feat &f, int ty, int cin, uint32_t wbase, int np, uint32_t col) {
            constexpr int NTX = decltype(ntx_)::value;
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(np >> 3) << 17) | (8u << 24);
            uint64_t bd = desc_ns(wbase, (uint32_t)np * 16u, 128u);
            const uint32_t chunk = (uint32_t)(f.rows(ty) * f.S) * 16u, kstep = chunk >> 3, bstep = 2u * (uint32_t)np;
            const int nk = (cin + 15) >> 4, KS = f.ks();
            const uint32_t d = tmem + col;
            const uint64_t adr = desc_ns(rbase, chunk, (uint32_t)f.S * 16u);
            uint32_t acc = 0u;
            for (int ks = 0; ks < nk; ks += KS) {
                const int n = min(KS, nk - ks);
                warp_wait(&sh.rfull[s], rph, p.wait_cycles, dead);
                if (!dead) {
                    fence_after();
                    uint64_t ad = adr + (uint64_t)((uint32_t)s * (STAGE_BYTES >> 4));
                    for (int kk = 0; kk < n; ++kk) {
                        uint32_t dt = d;
#pragma unroll
                        for (int tx = 0; tx < NTX; ++tx) {
                            mma_bf16(dt, ad + (uint64_t)(8 * tx), bd, idesc, acc);
                            dt += (uint32_t)np;
                        }
                        acc = 1u;
                        ad += kstep;
                        bd += bstep;
                    }
                    mma_commit(&sh.rempty[s]);
                }
                if (++s == RING) { s = 0; rph ^= 1u; }
            }
            if (!dead) mma_commit(&sh.hb[ty]);
        };
        auto rows1x1 = [&](const Feat &f, int ty, int cin, uint32_t wbase, int np, uint32_t col) {
            switch ((f.S + 7) >> 3) {
                case 1: rows_n(Int<1>{}, f, ty, cin, wbase, np, col); break;
                case 2: rows_n(Int<2>{}, f, ty, cin, wbase, np, col); break;
                case 3: rows_n(Int<3>{}, f, ty, cin, wbase, np, col); break;
                default: rows_n(Int<4>{}, f, ty, cin, wbase, np, col); break;
            }
        };
        for (int b = 0; b < 3; ++b) {
            const Feat f(p.hw >> b);
            const Geo g(f.S);
            const int ntx = g.ntx();
            const uint32_t col3 = (uint32_t)(g.tiles() * N1);
            for (int l = 0; l < p.layers; ++l, ++item, ++layer) {
                warp_wait(&sh.w1full, layer & 1, p.wait_cycles, dead);
                for (int ty = 0; ty < f.nty; ++ty)
                    rows1x1(f, ty, p.cstart[b] + l * K, su32(w1), N1, (uint32_t)(ty * ntx * N1));
                if (!dead) mma_commit(&sh.w1empty);
                warp_wait(&sh.w3full, layer & 1, p.wait_cycles, dead);
                warp_wait(&sh.hready, hph, p.wait_cycles, dead);
                hph ^= 1u;
                if (!dead) {
                    fence_after();
                    issue<N1, 16, 9, false>(tmem + col3, su32(hbuf), su32(w3), g, sh.t3, &sh.w3empty);
                }
            }
            if (b < 2) {
                // its tiles overlap the last 3x3 convolution's columns: wait for that epilogue
                warp_wait(&sh.wtfull, b & 1, p.wait_cycles, dead);
                warp_wait(&sh.fready, item & 1, p.wait_cycles, dead);
                fence_after();
                const int np = (p.cfin[b] / 2 + 15) / 16 * 16;
                for (int ty = 0; ty < f.nty; ++ty) {
                    rows1x1(f, ty, p.cfin[b], su32(hbuf), np, 0u);
                    warp_wait(&sh.hready, hph, p.wait_cycles, dead);
                    hph ^= 1u;
                    fence_after();
                }
                ++item;
            }
        }
    } else {
        // ---------------- epilogue warps ----------------
        const int q = warp & 3, h = warp >> 2, ry = (q * 32 + lane) >> 3, rx = lane & 7;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        bool dead = false;
        uint32_t hbph = 0u, t3ph = 0u, wtph = 0u;
        int layer = 0;
        auto zero = [&](uint8_t *r, uint32_t bytes) {
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            for (uint32_t i = threadIdx.x * 16u; i < bytes; i += EPI * 16u) *reinterpret_cast<uint4 *>(r + i) = z;
        };
        auto arrive = [&](uint64_t *bar) {
            __syncwarp();
            if (lane == 0) bar_arrive(bar);
        };
        {
            // stem: one fmaf chain per output over (c, ky, kx), taps outside the image skipped
            const int hw = p.hw, npx = hw * hw, c0 = 2 * K;
            const Geo g(hw);
            float *im = reinterpret_cast<float *>(hbuf), *sw = im + 3 * npx;      // then the weights [27][2 k]
            for (int i = threadIdx.x; i < 27 * c0; i += EPI) sw[i] = __ldg(p.stem_wt + i);
            pdl_wait();
            for (int i = threadIdx.x; i < 3 * npx; i += EPI) im[i] = __ldg(p.x + img * 3 * npx + i);
            epi_sync();
            const int nt = g.tiles(), ntx = g.ntx();
            for (int pl = h; pl < K4; pl += 2) {
                float z[MAX_TILES][8];
#pragma unroll
                for (int t = 0; t < MAX_TILES; ++t)
#pragma unroll
                    for (int i = 0; i < 8; ++i) z[t][i] = 0.0f;
                for (int kk = 0; kk < 27; ++kk) {
                    const int c = kk / 9, dy = (kk / 3) % 3 - 1, dx = kk % 3 - 1;
                    float w[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) w[i] = sw[kk * c0 + pl * 8 + i];
#pragma unroll
                    for (int t = 0; t < MAX_TILES; ++t) {
                        if (t >= nt) break;
                        const int y = 16 * (t / ntx) + ry + dy, xx = 8 * (t % ntx) + rx + dx;
                        if (y >= 0 && y < hw && xx >= 0 && xx < hw) {
                            const float v = im[(c * hw + y) * hw + xx];
#pragma unroll
                            for (int i = 0; i < 8; ++i) z[t][i] = fmaf(v, w[i], z[t][i]);
                        }
                    }
                }
                float sc[8], sf[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    sc[i] = __ldg(p.stem_scale + pl * 8 + i);
                    sf[i] = __ldg(p.stem_shift + pl * 8 + i);
                }
                uint16_t *dst = p.F[0] + (img * p.planes[0] + pl) * npx * 8;
#pragma unroll
                for (int t = 0; t < MAX_TILES; ++t) {
                    if (t >= nt) break;
                    const int y = 16 * (t / ntx) + ry, xx = 8 * (t % ntx) + rx;
                    if (y < hw && xx < hw) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float v = fmaf(z[t][i], sc[i], sf[i]);
                            if (v > 1.0f) v = 1.0f;
                            if (v < -1.0f) v = -1.0f;
                            z[t][i] = v;
                        }
                        *reinterpret_cast<uint4 *>(dst + (y * hw + xx) * 8) =
                            make_uint4(pack2(z[t][0], z[t][1]), pack2(z[t][2], z[t][3]), pack2(z[t][4], z[t][5]),
                                       pack2(z[t][6], z[t][7]));
                    }
                }
            }
            asm volatile("fence.proxy.async;\n" ::: "memory");
            arrive(&sh.fready);
            epi_sync();                                        // the image is read
            zero(hbuf, (uint32_t)(N1 / 8) * g.plane);
            epi_sync();
        }
        for (int b = 0; b < 3; ++b) {
            const int S = p.hw >> b, px = S * S;
            const Geo g(S);
            const int nty = (S + 15) >> 4, ntx = g.ntx(), nt = g.tiles();
            const uint32_t col3 = (uint32_t)(nt * N1);
            uint16_t *F = p.F[b] + img * p.planes[b] * px * 8;
            for (int l = 0; l < p.layers; ++l, ++layer) {
                const int cin = p.cstart[b] + l * K;
                // bottleneck: HardTanh(BN) of this half's planes into the padded layout
                {
                    warp_wait(&sh.w1full, layer & 1, p.wait_cycles, dead);
                    const float *m = reinterpret_cast<const float *>(w1 + ((cin + 15) / 16 * 2) * N1 * 16);
                    for (int ty = 0; ty < nty; ++ty) {
                        warp_wait(&sh.hb[ty], (hbph >> ty) & 1u, p.wait_cycles, dead);
                        fence_after();
                        for (int tx = 0; tx < ntx; ++tx) {
                            const int y = 16 * ty + ry, x = 8 * tx + rx;
#pragma unroll
                            for (int pl = 0; pl < K4; ++pl) {
                                const int c = (h * K4 + pl) * 8;
                                float a[8], sc[8], sf[8];
                                tmem_ld<8>(tq + (uint32_t)((ty * ntx + tx) * N1 + c), a);
                                bn8(m, N1, c, sc, sf);
#pragma unroll
                                for (int i = 0; i < 8; ++i) a[i] = fminf(fmaxf(fmaf(a[i], sc[i], sf[i]), -1.0f), 1.0f);
                                if (y < S && x < S)
                                    *reinterpret_cast<uint4 *>(hbuf + (uint32_t)(c >> 3) * g.plane + g.at(y, x)) =
                                        make_uint4(pack2(a[0], a[1]), pack2(a[2], a[3]), pack2(a[4], a[5]),
                                                   pack2(a[6], a[7]));
                            }
                        }
                    }
                    hbph ^= (1u << nty) - 1u;
                    fence_async_smem();
                    fence_before();
                    arrive(&sh.hready);
                    if (lane == 0) bar_arrive(&sh.w1empty);
                }
                // the layer's K new channels, at channel cin of the features; half h takes tiles h, h + 2, ...
                warp_wait(&sh.w3full, layer & 1, p.wait_cycles, dead);
                const float *m = reinterpret_cast<const float *>(w3 + 9 * (N1 / 8) * 16 * 16);
                float sc[K], sf[K];
#pragma unroll
                for (int i = 0; i < K; i += 4) {
                    const float4 a = *reinterpret_cast<const float4 *>(m + i);
                    const float4 d = *reinterpret_cast<const float4 *>(m + 16 + i);
                    sc[i] = a.x; sc[i + 1] = a.y; sc[i + 2] = a.z; sc[i + 3] = a.w;
                    sf[i] = d.x; sf[i + 1] = d.y; sf[i + 2] = d.z; sf[i + 3] = d.w;
                }
                for (int t = h; t < nt; t += 2) {
                    warp_wait(&sh.t3[t], (t3ph >> t) & 1u, p.wait_cycles, dead);
                    fence_after();
                    float a[16];
                    tmem_ld<16>(tq + col3 + (uint32_t)(16 * t), a);
                    const int y = 16 * (t / ntx) + ry, x = 8 * (t % ntx) + rx;
                    if (y < S && x < S) {
                        uint32_t w[K / 2];
#pragma unroll
                        for (int i = 0; i < K; i += 2)
                            w[i / 2] = pack2(fminf(fmaxf(fmaf(a[i], sc[i], sf[i]), -1.0f), 1.0f),
                                             fminf(fmaxf(fmaf(a[i + 1], sc[i + 1], sf[i + 1]), -1.0f), 1.0f));
                        const int pix = y * S + x;
                        if ((cin & 3) == 0) {
#pragma unroll
                            for (int i = 0; i < K; i += 4) {
                                const int c = cin + i;
                                *reinterpret_cast<uint2 *>(F + ((int64_t)(c >> 3) * px + pix) * 8 + (c & 7)) =
                                    make_uint2(w[i / 2], w[i / 2 + 1]);
                            }
                        } else if (cin & 1) {                  // an odd transition width
#pragma unroll
                            for (int i = 0; i < K; ++i) {
                                const int c = cin + i;
                                F[((int64_t)(c >> 3) * px + pix) * 8 + (c & 7)] = (uint16_t)(w[i / 2] >> (16 * (i & 1)));
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < K; i += 2) {
                                const int c = cin + i;
                                *reinterpret_cast<uint32_t *>(F + ((int64_t)(c >> 3) * px + pix) * 8 + (c & 7)) = w[i / 2];
                            }
                        }
                    }
                }
                t3ph ^= (1u << nt) - 1u;
                asm volatile("fence.proxy.async;\n" ::: "memory");
                fence_before();
                arrive(&sh.fready);
                if (lane == 0) bar_arrive(&sh.w3empty);
            }
            if (b < 2) {
                // transition: HardTanh(BN), 2x2 average, the next block's first channels
                const int O = p.cfin[b] / 2, np = (O + 15) / 16 * 16, px2 = px / 4;
                uint16_t *F2 = p.F[b + 1] + img * p.planes[b + 1] * px2 * 8;
                warp_wait(&sh.wtfull, wtph, p.wait_cycles, dead);
                wtph ^= 1u;
                const float *m = reinterpret_cast<const float *>(hbuf + ((p.cfin[b] + 15) / 16 * 2) * np * 16);
                for (int ty = 0; ty < nty; ++ty) {
                    warp_wait(&sh.hb[ty], (hbph >> ty) & 1u, p.wait_cycles, dead);
                    fence_after();
                    for (int tx = 0; tx < ntx; ++tx) {
                        const int y = 16 * ty + ry, x = 8 * tx + rx;
                        for (int c = 8 * h; c < np; c += 16) {
                            float a[8], sc[8], sf[8];
                            tmem_ld<8>(tq + (uint32_t)(tx * np + c), a);
                            bn8(m, np, c, sc, sf);
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                float v = fmaf(a[i], sc[i], sf[i]);
                                if (v > 1.0f) v = 1.0f;
                                if (v < -1.0f) v = -1.0f;
                                // ((v00 + v01) + v10) + v11, then a quarter
                                const float v01 = __shfl_xor_sync(0xffffffffu, v, 1);
                                const float v10 = __shfl_xor_sync(0xffffffffu, v, 8);
                                const float v11 = __shfl_xor_sync(0xffffffffu, v, 9);
                                a[i] = (((v + v01) + v10) + v11) * 0.25f;
                            }
                            if (y < S && x < S && (lane & 9) == 0 && c < O)
                                *reinterpret_cast<uint4 *>(F2 + ((int64_t)(c >> 3) * px2 + (y >> 1) * (S / 2) + (x >> 1)) * 8) =
                                    make_uint4(pack2(a[0], a[1]), pack2(a[2], a[3]), pack2(a[4], a[5]),
                                               pack2(a[6], a[7]));
                        }
                    }
                    if (ty == nty - 1) {
                        // the weights and the BN map are read: the region is the next block's bottleneck
                        epi_sync();
                        const Geo g2(S / 2);
                        zero(hbuf, (uint32_t)(N1 / 8) * g2.plane);
                        epi_sync();
                        asm volatile("fence.proxy.async;\n" ::: "memory");
                    }
                    fence_before();
                    arrive(&sh.hready);
                }
                hbph ^= (1u << nty) - 1u;
                arrive(&sh.fready);
            }
        }
        // head: global average over the bf16 features (one sum over the pixels in order, one division),
        // fp32 linear layer, BN
        epi_sync();
        const int S = p.hw >> 2, px = S * S, C = p.cfin[2];
        float *pooled = reinterpret_cast<float *>(w1);
        const uint16_t *F = p.F[2] + img * p.planes[2] * px * 8;
        for (int c = threadIdx.x; c < C; c += EPI) {
            const unsigned short *src = reinterpret_cast<const unsigned short *>(F) + (int64_t)(c >> 3) * px * 8 + (c & 7);
            float sum = 0.0f;
            for (int i = 0; i < px; ++i) sum += __uint_as_float((uint32_t)__ldcg(src + i * 8) << 16);
            pooled[c] = sum / (float)px;
        }
        epi_sync();
        for (int o = threadIdx.x; o < p.classes; o += EPI) {
            float acc = 0.0f;
            for (int c = 0; c < C; ++c) acc = fmaf(pooled[c], __ldg(p.fc_wt + (int64_t)c * p.classes + o), acc);
            acc = acc + 0.0f;
            p.logits[img * p.classes + o] = fmaf(acc, __ldg(p.fc_scale + o), __ldg(p.fc_shift + o));
        }
        fence_before();
    }
    __syncthreads();
    if (warp == 8) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    }
}

__global__ void wdense_item_kernel(const uint16_t *__restrict__ wb, const float *__restrict__ scale,
                                   const float *__restrict__ shift, int C, int Cp, int O, int taps, int planes, int np,
                                   uint8_t *__restrict__ out) {
    const int n = taps * planes * np * 8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int e = i & 7, o = (i >> 3) % np, r = (i >> 3) / np;
        const int c = (r % planes) * 8 + e, tap = r / planes;
        reinterpret_cast<uint16_t *>(out)[i] =
            (o < O && c < C) ? wb[((int64_t)o * taps + tap) * Cp + c] : (uint16_t)0;
    }
    float *m = reinterpret_cast<float *>(out + (size_t)n * 2);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
        m[i] = i < O ? scale[i] : 0.0f;
        m[np + i] = i < O ? shift[i] : 0.0f;
    }
}

__global__ void wdense_nhwc_kernel(const uint16_t *__restrict__ F, int px, int planes, int c, int row, int64_t total,
                                   uint16_t *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int ch = (int)(i % row);
        const int64_t r = i / row;
        const int pix = (int)(r % px);
        out[i] = ch < c ? F[((r / px * planes + (ch >> 3)) * px + pix) * 8 + (ch & 7)] : (uint16_t)0;
    }
}

// Channels entering and leaving each block.
static void channels(int layers, int k, int (&cs)[3], int (&cf)[3]) {
    int c = 2 * k;
    for (int b = 0; b < 3; ++b) {
        cs[b] = c;
        cf[b] = c + layers * k;
        c = cf[b] / 2;
    }
}

static uint32_t w1_bytes(int layers, int k) {
    int cs[3], cf[3];
    channels(layers, k, cs, cf);
    return (item_bytes(std::max(std::max(cf[0], cf[1]), cf[2]) - k, 4 * k, 1) + 127u) & ~127u;
}

static uint32_t smem_bytes(int hw, int layers, int k) {
    return RING * STAGE_BYTES + ((h_bytes(k, hw) + 127u) & ~127u) + w1_bytes(layers, k) + item_bytes(4 * k, k, 9) + 128u;
}

}  // namespace dfu

bool wdense_fused_supported(int hw, int layers, int k) {
    if (hw < 8 || hw > 32 || hw % 4 != 0 || (k != 4 && k != 8 && k != 12)) return false;
    int cs[3], cf[3];
    dfu::channels(layers, k, cs, cf);
    const uint32_t h = dfu::h_bytes(k, hw);
    // the stem's image and weights, and each transition's weights, fit the bottleneck's region; a transition's
    // tiles of one stage of rows fit the tensor memory, its output columns an MMA
    if (3 * hw * hw * 4 + 27 * 2 * k * 4 > (int)h) return false;
    for (int b = 0; b < 2; ++b) {
        const int np = wdense_pad16(cf[b] / 2);
        if (dfu::item_bytes(cf[b], cf[b] / 2, 1) > h || np > 256 || np * (((hw >> b) + 7) / 8) > 512) return false;
    }
    // tiles read up to 16 rows of 8 columns past an image that is smaller: inside the regions that follow
    return (size_t)cf[2] * 4 <= dfu::w1_bytes(layers, k) && dfu::smem_bytes(hw, layers, k) <= dfu::SMEM_LIMIT;
}

size_t wdense_item_bytes(int C, int O, int taps) { return dfu::item_bytes(C, O, taps); }

minw_status wdense_write_item(const uint16_t *wb, const float *scale, const float *shift, int C, int Cp, int O,
                              int taps, uint8_t *out, cudaStream_t s) {
    const int planes = wdense_planes(C), np = wdense_pad16(O);
    dfu::wdense_item_kernel<<<(taps * planes * np * 8 + 255) / 256, 256, 0, s>>>(wb, scale, shift, C, Cp, O, taps,
                                                                                planes, np, out);
    return minw_host::launch_status();
}

minw_status wdense_planes_to_nhwc(const uint16_t *F, int B, int px, int planes, int c, int row, uint16_t *out,
                                  cudaStream_t s) {
    const int64_t total = (int64_t)B * px * row;
    dfu::wdense_nhwc_kernel<<<(unsigned)std::min<int64_t>((total + 255) / 256, 4096), 256, 0, s>>>(F, px, planes, c, row,
                                                                                                  total, out);
    return minw_host::launch_status();
}

minw_status launch_wdense_fused(dfu::Args a, int B, cudaStream_t s) {
    a.wait_cycles = (long long)minw_host::plan_options().wait_cycles;
    a.w1_bytes = dfu::w1_bytes(a.layers, a.k);
    a.smem = dfu::smem_bytes(a.hw, a.layers, a.k);
    auto kern = a.k == 4 ? dfu::wdense_fused_kernel<1> : a.k == 8 ? dfu::wdense_fused_kernel<2> : dfu::wdense_fused_kernel<3>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dfu::SMEM_LIMIT) != cudaSuccess)
        return MINW_ECUDA;
    if (minw_host::launch_pdl(kern, dim3((unsigned)B), dim3(dfu::NT), (size_t)a.smem, s, a) != cudaSuccess)
        return MINW_ECUDA;
    return minw_host::launch_status();
}

int take_wdense_error() {
    int flag = 0;
    if (cudaMemcpyFromSymbol(&flag, smc::g_error, sizeof(int)) != cudaSuccess) return -1;
    if (flag) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(smc::g_error, &zero, sizeof(int)) != cudaSuccess) return -1;
    }
    return flag ? 1 : 0;
}

}  // namespace minw
