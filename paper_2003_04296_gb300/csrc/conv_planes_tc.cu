// conv_planes_tc.cu -- the bit-plane convolution on the tensor cores: the
// same operands and results as conv_popc.cu (exact int32 accumulators), with
// the planes expanded to E2M1 level codes on the way into shared memory.
//
// The levels {0, +-1, +-2, +-4} are exact in E2M1 and their products and sums
// exact in the fp32 accumulators (|acc| <= 16 K < 2^24, checked by the host),
// so tcgen05.mma kind::mxf4 with unit block scales computes the integer
// product of Table I.  A nibble is sign * 8 + magnitude code * 2, and the
// planes hold exactly those bits: nibble j of register r takes channel bit
// 4 j + r of its word, i.e. one shift and one masked OR per plane and eight
// channels.  The channel order inside a word is permuted that way for both
// operands alike, which leaves the contraction unchanged.
//
// Implicit GEMM: CTA tile = 128 consecutive output pixels (MMA M) x BN output
// channels (MMA N), K = kh kw taps x C/32 words, flattened and taken in chunks
// of four words (128 channels, 64-byte operand rows with the 64-byte swizzle).
// Warp roles (288 threads): warps 0-3 expand activation rows, one pixel per
// thread, warps 4-7 weight rows, one channel per thread; each thread keeps two
// chunks of loads in flight in registers.  Warp 8 issues the MMAs.  After the
// last chunk warps 0-7 run the epilogue from tensor memory: raw accumulators,
// BN, HardTanh + quantize + pack, 2x2 max pool (through shared memory).
// One tile per CTA, two or more CTAs per SM: one CTA's epilogue and set-up
// overlap the other's main loop.
//
// Bound: the expansion's integer instructions (about 6 P per 8 channels and
// operand row) and, for raw outputs, the int32 / fp32 stores.  The popcount
// kernel spends 2 P_a P_w popcounts per 32 products at 16 a clock and SM; on a
// 256 x 512 x 14 x 14, 3x3, 3-bit x 3-bit layer (quantize + convolve, raw and
// fp32 outputs) it took 8.24 ms, this kernel 0.24 ms (0.33 before loads by pairs
// of lanes and BN maps in wide loads); a 4 x 128 x 32 x 32, 1-bit x 1-bit layer 32.8 -> 19.5 us.
//
// Every mbarrier wait is bounded; one that runs out sets this file's error
// flag (read by minw_get_last_device_error) and the CTA winds down.
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.cuh"

namespace minw {

__device__ int g_planes_tc_error = 0;

namespace ptc {

constexpr int BM = 128;
constexpr int NPROD = 256;               // producer / epilogue threads
constexpr int NT = NPROD + 32;
constexpr int ROWB = 64;                 // bytes of one operand row of a chunk: 128 E2M1 channels
constexpr int CW = 4;                    // 32-channel words per chunk
constexpr int SMAX = 6;
constexpr int POOL_LD = BM + 2;          // padded channel row of the pooling stage (pairs of pixels load at once)

struct Params {
    ConvArgs a;
    int BN;                // output channels per tile: 32, 64 or 128
    int ntn;               // channel tiles
    int nchunks;           // K chunks
    int S;                 // ring slots
    uint32_t stage_bytes;  // BM rows then BN rows of ROWB bytes
    uint32_t idesc, tmem_cols;
    long long wait_cycles;
    int stall;             // timeout-path test: the MMA issuer first waits on a barrier nothing completes
};

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
// Bounded wait: false (and the error flag set) after limit SM clocks.
__device__ __forceinline__ bool bar_wait(uint64_t *b, uint32_t parity, long long limit) {
    if (bar_try(b, parity)) return true;
    const long long t0 = clock64();
    while (!bar_try(b, parity)) {
        if (clock64() - t0 > limit) {
            atomicExch(&g_planes_tc_error, 1);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// K-major operand rows of 64 bytes with the 64-byte swizzle (8-row groups 512 bytes apart).
__device__ __forceinline__ uint64_t desc64(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((8 * ROWB) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

// Executed by the whole (converged) issuing warp; one elected lane issues.
__device__ __forceinline__ void mma_f4(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate, uint32_t sfa, uint32_t sfb) {
    asm volatile("{\n .reg .pred p, e;\n .reg .b32 r;\n setp.ne.b32 p, %4, 0;\n elect.sync r|e, 0xffffffff;\n"
                 " @e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n}\n"
                 ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb));
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("{\n .reg .pred e;\n .reg .b32 r;\n elect.sync r|e, 0xffffffff;\n"
                 " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(su32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// E2M1 codes of the 32 channels of one word (P planes at pl[0], pl[CW], ...):
// nibble j of word r is channel 4 j + r.  valid = 0 (1-bit only: a padded tap
// or a word past the last) gives zeros; multi-level planes are then zero.
template <int P>
__device__ __forceinline__ uint4 expand(const uint32_t *pl, bool valid) {
    const uint32_t s = pl[0];
    uint32_t r0 = (s << 3) & 0x88888888u, r1 = (s << 2) & 0x88888888u, r2 = (s << 1) & 0x88888888u,
             r3 = s & 0x88888888u;
    if constexpr (P == 1) {
        const uint32_t one = valid ? 0x22222222u : 0u;   // a zero magnitude with the sign set is -0
        r0 |= one; r1 |= one; r2 |= one; r3 |= one;
    } else {
        const uint32_t m = pl[CW];                       // non-zero mask, or bit 0 of the magnitude code
        r0 |= (m << 1) & 0x22222222u;
        r1 |= m & 0x22222222u;
        r2 |= (m >> 1) & 0x22222222u;
        r3 |= (m >> 2) & 0x22222222u;
        if constexpr (P == 3) {
            const uint32_t c = pl[2 * CW];
            r0 |= (c << 2) & 0x44444444u;
            r1 |= (c << 1) & 0x44444444u;
            r2 |= c & 0x44444444u;
            r3 |= (c >> 1) & 0x44444444u;
        }
    }
    return make_uint4(r0, r1, r2, r3);
}

// One chunk of an operand row in registers: word j of plane p at w[p * CW + j].
template <int P>
struct Chunk {
    uint32_t w[P * CW];
    uint32_t valid;        // bit j: word j lies in the image and before the last word of K
};

// Position of a row's next load in K: tap (ky, kx) and word w of its NW.
struct Cursor {
    int ky, kx, w;
};

// Loads the next chunk of a row.  ACT: an activation row (tap (ky, kx) reads
// pixel (y0 + ky, x0 + kx) of image pix0 where it lies inside), else a weight
// row (consecutive taps).  VEC: NW is a multiple of four, so a chunk lies in
// one tap and each plane's four words are one 16-byte load; otherwise every
// word is placed by itself.
template <int P, bool ACT, bool VEC>
__device__ __forceinline__ void load_chunk(Chunk<P> &ch, Cursor &k, const ConvArgs &a, bool live, int64_t row, int y0,
                                           int x0) {
    ch.valid = 0u;
#pragma unroll
    for (int i = 0; i < P * CW; ++i) ch.w[i] = 0u;
    constexpr int STEP = VEC ? CW : 1;
#pragma unroll
    for (int j = 0; j < CW; j += STEP) {
        const uint32_t *src;
        bool in = live && k.ky < a.kh;
        if constexpr (ACT) {
            const int y = y0 + k.ky, x = x0 + k.kx;
            in = in && y >= 0 && y < a.H && x >= 0 && x < a.W;
            src = a.act + (row + (int64_t)y * a.W + x) * P * a.NW + k.w;
        } else {
            src = a.wgt + (row + k.ky * a.kw + k.kx) * P * a.NW + k.w;
        }
        if (in) {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if constexpr (VEC) {
                    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src + p * a.NW));
                    ch.w[p * CW] = v.x; ch.w[p * CW + 1] = v.y; ch.w[p * CW + 2] = v.z; ch.w[p * CW + 3] = v.w;
                } else {
                    ch.w[p * CW + j] = __ldg(src + p * a.NW);
                }
            }
            ch.valid |= (VEC ? 0xFu : 1u) << j;
        }
        k.w += STEP;
        if (k.w >= a.NW) {
            k.w = 0;
            if (++k.kx == a.kw) { k.kx = 0; ++k.ky; }
        }
    }
}

// Expands a chunk of row r into a ring slot (chunk word j of four at j ^ ((r
// >> 1) & 3): the 64-byte swizzle, and no bank conflict between eight
// neighbouring rows), once the MMAs of the slot's previous lap released it, and
// arrives for the warp.
struct Ring {
    uint8_t *dst;
    uint64_t *full, *empty;
    int r, s, lap;
    bool write, lane0;
};
template <int P>
__device__ __forceinline__ bool put_chunk(const Params &p, Ring &g, const Chunk<P> &c) {
    uint4 v[CW];
#pragma unroll
    for (int j = 0; j < CW; ++j) v[j] = expand<P>(c.w + j, (c.valid >> j) & 1u);
    if (g.lap > 0 && !__all_sync(0xffffffffu, bar_wait(&g.empty[g.s], (g.lap - 1) & 1, p.wait_cycles))) return false;
    if (g.write) {
        uint4 *d = reinterpret_cast<uint4 *>(g.dst + (size_t)g.s * p.stage_bytes + g.r * ROWB);
        const int sw = (g.r >> 1) & 3;
#pragma unroll
        for (int j = 0; j < CW; ++j) d[j ^ sw] = v[j];
    }
    fence_async_smem();
    __syncwarp();
    if (g.lane0) bar_arrive(&g.full[g.s]);
    if (++g.s == p.S) { g.s = 0; ++g.lap; }
    return true;
}

// The producer loop of one thread: every chunk of its row, two in flight.
template <int P, bool ACT, bool VEC>
__device__ __forceinline__ void produce(const Params &p, Ring &g, bool live, int64_t row, int y0, int x0) {
    const ConvArgs &a = p.a;
    Cursor k{0, 0, 0};
    Chunk<P> c[2];
    load_chunk<P, ACT, VEC>(c[0], k, a, live, row, y0, x0);
    load_chunk<P, ACT, VEC>(c[1], k, a, live, row, y0, x0);
    for (int i = 0; i < p.nchunks; i += 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (i + h >= p.nchunks) break;
            if (!put_chunk<P>(p, g, c[h])) return;
            load_chunk<P, ACT, VEC>(c[h], k, a, live, row, y0, x0);
        }
    }
}

// The same where NW is a multiple of eight: an odd and an even lane load the
// two 16-byte halves of eight words of one row and then of another, so that a
// load instruction touches 16 lines instead of 32 (its lines, looked up one a
// clock, held the 512-channel layers), and exchange halves by shuffles.  Lane l
// of the warp holds row (l >> 1) + 16 (l & 1) of its 32.  rowA, yA, xA and
// rowB, yB, xB: rows l >> 1 and (l >> 1) + 16.
template <int P, bool ACT>
__device__ __forceinline__ void produce_pair(const Params &p, Ring &g, bool liveA, int64_t rowA, int yA, int xA, bool liveB,
                                             int64_t rowB, int yB, int xB) {
    const ConvArgs &a = p.a;
    const bool odd = threadIdx.x & 1;
    // each lane's cursor starts at its half and steps by eight words
    Cursor k{0, 0, odd ? CW : 0};
    Chunk<P> A, B;
    auto load = [&]() {
        Cursor ka = k, kb = k;
        load_chunk<P, ACT, true>(A, ka, a, liveA, rowA, yA, xA);
        load_chunk<P, ACT, true>(B, kb, a, liveB, rowB, yB, xB);
        k.w += 2 * CW;
        if (k.w >= a.NW) {
            k.w -= a.NW;
            if (++k.kx == a.kw) { k.kx = 0; ++k.ky; }
        }
    };
    load();
    for (int i = 0; i < p.nchunks; i += 2) {             // nchunks is even: kh kw NW / 4
        // the even lane gives its half of row B for the odd lane's half of row A
        Chunk<P> c0, c1;
#pragma unroll
        for (int j = 0; j < P * CW; ++j) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, odd ? A.w[j] : B.w[j], 1);
            c0.w[j] = odd ? o : A.w[j];
            c1.w[j] = odd ? B.w[j] : o;
        }
        const uint32_t ov = __shfl_xor_sync(0xffffffffu, odd ? A.valid : B.valid, 1);
        c0.valid = odd ? ov : A.valid;
        c1.valid = odd ? B.valid : ov;
        load();
        if (!put_chunk<P>(p, g, c0) || !put_chunk<P>(p, g, c1)) return;
    }
}

// Level planes of BN output y of one channel (bits 0 .. OUTB - 1), the fp32
// chain of the block: HardTanh, prescale, thresholds.
template <int OUTB>
__device__ __forceinline__ uint32_t planes_of_y(float y, const QParams &q) {
    QParams qb = q;
    qb.bits = OUTB;
    y = fminf(fmaxf(y, -1.0f), 1.0f);
    return level_plane_bits(level_units(y * qb.scale, qb), OUTB);
}

// Epilogue of one 32-channel group without pooling: lane = output pixel m.
template <int OUTB>
__device__ __forceinline__ void store_group(const ConvArgs &a, const uint32_t (&v)[32], int o0, long long m) {
    if (m >= a.M) return;
    const int HoWo = a.Ho * a.Wo;
    const long long b = m / HoWo;
    const long long at = (b * a.O + o0) * HoWo + (m - b * HoWo);
    const int nv = min(32, a.O - o0);
    if (a.acc_out != nullptr) {
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (c < nv) __stcs(a.acc_out + at + (long long)c * HoWo, __float2int_rn(__uint_as_float(v[c])));
    }
    if (a.y_out == nullptr && OUTB == 0) return;
    uint32_t w[3] = {0u, 0u, 0u};
    auto one = [&](int c, float sc, float sh) {
        const float y = fmaf(__uint_as_float(v[c]), sc, sh);
        if constexpr (OUTB > 0) {
            const uint32_t pb = planes_of_y<OUTB>(y, a.qo);
#pragma unroll
            for (int u = 0; u < OUTB; ++u) w[u] |= ((pb >> u) & 1u) << c;
        }
        if (a.y_out != nullptr)
            __stcs(a.y_out + at + (long long)c * HoWo, OUTB > 0 ? fminf(fmaxf(y, -1.0f), 1.0f) : y);
    };
    const float *sp = a.scale + o0, *hp = a.shift + o0;
    if (nv == 32 && ((reinterpret_cast<uintptr_t>(sp) | reinterpret_cast<uintptr_t>(hp)) & 15) == 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float4 s = __ldg(reinterpret_cast<const float4 *>(sp) + k), h = __ldg(reinterpret_cast<const float4 *>(hp) + k);
            one(4 * k, s.x, h.x);
            one(4 * k + 1, s.y, h.y);
            one(4 * k + 2, s.z, h.z);
            one(4 * k + 3, s.w, h.w);
        }
    } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            if (c >= nv) break;
            one(c, __ldg(sp + c), __ldg(hp + c));
        }
    }
    if constexpr (OUTB > 0) {
        const int NWo = (a.O + 31) >> 5;
        uint32_t *dst = a.planes_out + m * OUTB * NWo + (o0 >> 5);
#pragma unroll
        for (int u = 0; u < OUTB; ++u) dst[u * NWo] = w[u];
    }
}

// Epilogue of one 32-channel group with the 2x2 max pool: the group's
// accumulators in shared memory [channel][pixel], lane = one of the tile's 32
// pooled pixels (consecutive in the output), warp q of four takes channels 8 q
// .. 8 q + 7: one byte of each plane word, and whole lines of y_out.  With a
// channel per lane and the pixels in turn a 1x1 layer of 32 -> 32 channels, 2 x 2
// bits, 160 images of 32 x 32, took 29.1 us (1-bit planes) and 28.8 (fp32) against
// 25.1 and 18.6 of the popcount kernel; 19.9 and 19.8 here.
template <int OUTB>
__device__ __forceinline__ void store_pooled(const ConvArgs &a, const float *acc, int o0, long long m0, int q,
                                             int lane) {
    const int HoWo = a.Ho * a.Wo, half = a.Wo / 2, HpWp = (a.Ho / 2) * half;
    const int NWo = (a.O + 31) >> 5;
    const int pr = lane / half, r00 = 2 * (pr * a.Wo + lane - pr * half);
    const long long m = m0 + r00;
    if (m >= a.M) return;
    const long long b = m / HoWo;
    const int pix = (int)(m - b * HoWo), yo = pix / a.Wo, xo = pix - yo * a.Wo;
    const long long op = (long long)(yo / 2) * half + xo / 2;
    uint32_t w[3] = {0u, 0u, 0u};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int c = 8 * q + e, o = o0 + c;
        if (o >= a.O) break;
        const float *p = acc + c * POOL_LD + r00;
        const float2 r0 = *reinterpret_cast<const float2 *>(p), r1 = *reinterpret_cast<const float2 *>(p + a.Wo);
        const float y = fmaf(fmaxf(fmaxf(r0.x, r0.y), fmaxf(r1.x, r1.y)), __ldg(a.scale + o), __ldg(a.shift + o));
        if (a.y_out != nullptr)
            a.y_out[(b * a.O + o) * HpWp + op] = OUTB > 0 ? fminf(fmaxf(y, -1.0f), 1.0f) : y;
        if constexpr (OUTB > 0) {
            const uint32_t pb = planes_of_y<OUTB>(y, a.qo);
#pragma unroll
            for (int u = 0; u < OUTB; ++u) w[u] |= ((pb >> u) & 1u) << e;
        }
    }
    if constexpr (OUTB > 0) {
        uint8_t *dst = reinterpret_cast<uint8_t *>(a.planes_out + (b * HpWp + op) * OUTB * NWo + (o0 >> 5)) + q;
#pragma unroll
        for (int u = 0; u < OUTB; ++u) dst[4 * u * NWo] = (uint8_t)w[u];
    }
}

// MODE: loads of single words (0), of four words of a row (1: NW % 4 == 0), of eight by two lanes (2: NW % 8 == 0).
template <int MODE, int OUTB>
__global__ void __launch_bounds__(NT, 2) conv_planes_tc_kernel(const __grid_constant__ Params p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (su32(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t full[SMAX], empty[SMAX], tfull, tstall;
    __shared__ uint32_t tmem_slot;
    const ConvArgs &a = p.a;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tn = (int)(blockIdx.x % (unsigned)p.ntn);
    const long long m0 = (long long)(blockIdx.x / (unsigned)p.ntn) * BM;
    const int o0 = tn * p.BN;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.S; ++s) {
            bar_init(&full[s], NPROD / 32);
            bar_init(&empty[s], 1);
        }
        bar_init(&tfull, 1);
        bar_init(&tstall, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == NPROD / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(&tmem_slot)),
                     "r"(p.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_slot;
    const uint32_t sf = tmem + (uint32_t)p.BN;            // unit scale factors: 32 columns of A's, 32 of B's
    if (warp < 4) {
        // UE8M0 0x7F = 2^0 in every lane of 64 columns, one warp per lane quarter
#pragma unroll
        for (int c = 0; c < 64; c += 8)
            asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};\n" ::"r"(
                             sf + ((uint32_t)(warp * 32) << 16) + (uint32_t)c),
                         "r"(0x7F7F7F7Fu));
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    pdl_trigger();
    pdl_wait();                                           // operands and outputs are shared with earlier kernels

    if (warp == NPROD / 32) {
        bool alive = true;
        if (p.stall && !__all_sync(0xffffffffu, bar_wait(&tstall, 0u, p.wait_cycles))) alive = false;
        const uint64_t ad0 = desc64(su32(smem)), bd0 = desc64(su32(smem) + BM * ROWB);
        const uint32_t step = p.stage_bytes >> 4;
        int s = 0;
        uint32_t phase = 0u, acc = 0u;
        for (int i = 0; alive && i < p.nchunks; ++i) {
            if (!__all_sync(0xffffffffu, bar_wait(&full[s], phase, p.wait_cycles))) { alive = false; break; }
            fence_after();
            const uint64_t off = (uint64_t)((uint32_t)s * step);
            mma_f4(tmem, ad0 + off, bd0 + off, p.idesc, acc, sf, sf + 32u);
            mma_f4(tmem, ad0 + off + 2, bd0 + off + 2, p.idesc, 1u, sf, sf + 32u);
            acc = 1u;
            mma_commit(&empty[s]);
            if (++s == p.S) { s = 0; phase ^= 1u; }
        }
        if (alive) mma_commit(&tfull);
    } else {
        // this thread's row of the operand, and for paired loads the two rows it loads from
        constexpr bool PAIR = MODE == 2;
        const int w32 = (warp & 3) * 32;
        const int rA = PAIR ? w32 + (lane >> 1) : w32 + lane, rB = rA + 16;
        Ring g{warp < 4 ? smem : smem + BM * ROWB, full, empty, PAIR ? (lane & 1 ? rB : rA) : rA, 0, 0, true, lane == 0};
        if (warp < 4) {
            const int HoWo = a.Ho * a.Wo;
            auto place = [&](int r, bool &live, int64_t &row, int &y0, int &x0) {
                const long long m = m0 + r;
                live = m < a.M;
                const int b = live ? (int)(m / HoWo) : 0;
                const int pix = live ? (int)(m - (long long)b * HoWo) : 0;
                const int yo = pix / a.Wo, xo = pix - yo * a.Wo;
                row = (int64_t)b * a.H * a.W;
                y0 = yo * a.stride - a.pad;
                x0 = xo * a.stride - a.pad;
            };
            bool lA, lB = false;
            int64_t wA, wB = 0;
            int yA, xA, yB = 0, xB = 0;
            place(rA, lA, wA, yA, xA);
            if constexpr (PAIR) {
                place(rB, lB, wB, yB, xB);
                if (a.bits_a == 1) produce_pair<1, true>(p, g, lA, wA, yA, xA, lB, wB, yB, xB);
                else if (a.bits_a == 2) produce_pair<2, true>(p, g, lA, wA, yA, xA, lB, wB, yB, xB);
                else produce_pair<3, true>(p, g, lA, wA, yA, xA, lB, wB, yB, xB);
            } else {
                if (a.bits_a == 1) produce<1, true, MODE == 1>(p, g, lA, wA, yA, xA);
                else if (a.bits_a == 2) produce<2, true, MODE == 1>(p, g, lA, wA, yA, xA);
                else produce<3, true, MODE == 1>(p, g, lA, wA, yA, xA);
            }
        } else {
            g.write = g.r < p.BN;
            const int taps = a.kh * a.kw;
            const bool lA = rA < p.BN && o0 + rA < a.O, lB = rB < p.BN && o0 + rB < a.O;
            const int64_t wA = (int64_t)(o0 + rA) * taps, wB = (int64_t)(o0 + rB) * taps;
            if constexpr (PAIR) {
                if (a.bits_w == 1) produce_pair<1, false>(p, g, lA, wA, 0, 0, lB, wB, 0, 0);
                else if (a.bits_w == 2) produce_pair<2, false>(p, g, lA, wA, 0, 0, lB, wB, 0, 0);
                else produce_pair<3, false>(p, g, lA, wA, 0, 0, lB, wB, 0, 0);
            } else {
                if (a.bits_w == 1) produce<1, false, MODE == 1>(p, g, lA, wA, 0, 0);
                else if (a.bits_w == 2) produce<2, false, MODE == 1>(p, g, lA, wA, 0, 0);
                else produce<3, false, MODE == 1>(p, g, lA, wA, 0, 0);
            }
        }
        __syncwarp();
        // a wait that ran out (here or in the MMA warp) leaves tfull open: no output is written
        const bool ok = __all_sync(0xffffffffu, bar_wait(&tfull, 0u, p.wait_cycles));
        fence_after();
        const int q = warp & 3, h = warp >> 2;
        if (!a.pool) {
            for (int g = h; g < p.BN / 32 && ok; g += 2) {
                if (o0 + g * 32 >= a.O) break;
                uint32_t v[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 32), v);
                store_group<OUTB>(a, v, o0 + g * 32, m0 + q * 32 + lane);
            }
        } else {
            // the ring is free: every MMA has completed.  Each half of the warps stages its groups in turn.
            float *stage = reinterpret_cast<float *>(smem) + h * (32 * POOL_LD);
            for (int g = h; g < p.BN / 32; g += 2) {
                if (o0 + g * 32 >= a.O) break;
                if (ok) {
                    uint32_t v[32];
                    tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 32), v);
#pragma unroll
                    for (int c = 0; c < 32; ++c) stage[c * POOL_LD + q * 32 + lane] = __uint_as_float(v[c]);
                }
                asm volatile("bar.sync %0, 128;\n" ::"r"(1 + h) : "memory");
                if (ok) store_pooled<OUTB>(a, stage, o0 + g * 32, m0, q, lane);
                asm volatile("bar.sync %0, 128;\n" ::"r"(1 + h) : "memory");
            }
        }
        fence_before();
    }
    __syncthreads();
    if (warp == NPROD / 32) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(p.tmem_cols));
    }
}

}  // namespace ptc

// Accumulators of magnitude <= 16 kh kw C must stay below 2^24 (exact in fp32);
// outputs are those of the bit-plane entry points (planes, fp32, raw).
bool planes_tc_supported(const ConvArgs &a) {
    if ((long long)a.kh * a.kw * a.C >= (1ll << 20) || a.codes_out != nullptr) return false;
    if (a.pool && ptc::BM % (2 * a.Wo) != 0) return false;
    return (a.M + ptc::BM - 1) / ptc::BM * ((a.O + 31) / 32) < (1ll << 31);
}

minw_status launch_planes_tc(const ConvArgs &a, cudaStream_t s) {
    ptc::Params p{};
    p.a = a;
    const int sms = minw_host::num_sms() > 0 ? minw_host::num_sms() : 152;
    const long long tiles_m = (a.M + ptc::BM - 1) / ptc::BM;
    // channels per tile: as wide as O needs (activation rows are expanded once per
    // channel tile), narrower while that leaves SMs without a tile
    int BN = a.O > 64 ? 128 : a.O > 32 ? 64 : 32;
    while (BN > 32 && tiles_m * ((a.O + BN - 1) / BN) < sms) BN /= 2;
    p.BN = BN;
    p.ntn = (a.O + BN - 1) / BN;
    p.nchunks = (a.kh * a.kw * a.NW + ptc::CW - 1) / ptc::CW;
    p.S = p.nchunks < ptc::SMAX ? p.nchunks : ptc::SMAX;
    p.stage_bytes = (uint32_t)((ptc::BM + BN) * ptc::ROWB);
    // D fp32, A and B E2M1 with UE8M0 scales (kind::mxf4)
    p.idesc = (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | (1u << 23) | ((uint32_t)(ptc::BM >> 4) << 24);
    p.tmem_cols = BN == 128 ? 256u : 128u;                // BN accumulator columns, 64 of scale factors
    p.wait_cycles = (long long)minw_host::plan_options().wait_cycles;
    p.stall = minw_host::take_stall(MINW_STALL_CONV_TC);
    size_t smem = (size_t)p.S * p.stage_bytes;
    const size_t pool = a.pool ? sizeof(float) * 2 * 32 * ptc::POOL_LD : 0;
    if (smem < pool) smem = pool;
    smem += 1024;
    typedef void (*Kernel)(const ptc::Params);
    static const Kernel kernels[3][4] = {
        {ptc::conv_planes_tc_kernel<0, 0>, ptc::conv_planes_tc_kernel<0, 1>, ptc::conv_planes_tc_kernel<0, 2>,
         ptc::conv_planes_tc_kernel<0, 3>},
        {ptc::conv_planes_tc_kernel<1, 0>, ptc::conv_planes_tc_kernel<1, 1>, ptc::conv_planes_tc_kernel<1, 2>,
         ptc::conv_planes_tc_kernel<1, 3>},
        {ptc::conv_planes_tc_kernel<2, 0>, ptc::conv_planes_tc_kernel<2, 1>, ptc::conv_planes_tc_kernel<2, 2>,
         ptc::conv_planes_tc_kernel<2, 3>}};
    const int mode = a.NW % (2 * ptc::CW) == 0 ? 2 : a.NW % ptc::CW == 0 ? 1 : 0;
    const Kernel kern = kernels[mode][a.quant_out ? a.qo.bits : 0];
    constexpr int SMEM_MAX = ptc::SMAX * (ptc::BM + 128) * ptc::ROWB + 1024;
    if (!minw_host::allow_shared(reinterpret_cast<const void *>(kern), SMEM_MAX)) return MINW_ECUDA;
    if (minw_host::launch_pdl(kern, dim3((unsigned)(tiles_m * p.ntn)), dim3(ptc::NT), smem, s, p) != cudaSuccess)
        return MINW_ECUDA;
    return cudaGetLastError() == cudaSuccess ? MINW_OK : MINW_ECUDA;
}

int take_planes_tc_error() {
    int flag = 0;
    if (cudaMemcpyFromSymbol(&flag, g_planes_tc_error, sizeof(int)) != cudaSuccess) return -1;
    if (flag) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_planes_tc_error, &zero, sizeof(int)) != cudaSuccess) return -1;
    }
    return flag ? 1 : 0;
}

}  // namespace minw
