// wdense_fused.cuh -- the one-kernel forward of the weight-only DenseNet-BC
// (wdense_fused.cu) as its builder sees it.
#pragma once

#include "kernels.cuh"

namespace minw {

namespace dfu {

struct Args {
    const float *x;                  // [B][3][hw][hw]
    int hw, layers, k, classes;      // k: growth
    const float *stem_wt;            // [27][2 k]
    const float *stem_scale, *stem_shift;
    const uint8_t *blob;             // every convolution's item (wdense_write_item), in forward order
    uint16_t *F[3];                  // block features, bf16 [B][planes][S S][8]
    int cstart[3], cfin[3], planes[3];
    const float *fc_wt;              // [cfin[2]][classes]
    const float *fc_scale, *fc_shift;
    float *logits;
    uint32_t w1_bytes, smem;         // set by the launcher: the 1x1 weight buffer, dynamic shared memory
    long long wait_cycles;
};

}  // namespace dfu

// Sizes the kernel covers: images of up to 32 x 32, growth 4, 8 or 12, and weights that fit its buffers.
bool wdense_fused_supported(int hw, int layers, int k);
// Planes of eight channels a block's features take (channels padded to a multiple of 16).
inline int wdense_planes(int c) { return (c + 15) / 16 * 2; }
// One convolution's item: bf16 levels [taps][planes of C][Np][8], BN scale [Np], shift [Np]; Np = O
// padded to a multiple of 16, zeros in the padding.
inline int wdense_pad16(int o) { return (o + 15) / 16 * 16; }
size_t wdense_item_bytes(int C, int O, int taps);
minw_status wdense_write_item(const uint16_t *wb, const float *scale, const float *shift, int C, int Cp, int O,
                              int taps, uint8_t *out, cudaStream_t s);
minw_status launch_wdense_fused(dfu::Args a, int B, cudaStream_t s);
// Feature planes of B images as NHWC rows of `row` channels (zeros past the planes).
minw_status wdense_planes_to_nhwc(const uint16_t *F, int B, int px, int planes, int c, int row, uint16_t *out,
                                  cudaStream_t s);
// The kernel's timeout flag (as take_first_error).
int take_wdense_error();

}  // namespace minw
