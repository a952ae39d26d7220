// wres_fused.cuh -- the one-kernel forward of the weight-only residual
// network (wres_fused.cu) as its builder sees it.
#pragma once

#include "kernels.cuh"

namespace minw {

namespace wfu {

struct Args {
    const float *x;                  // [B][3][hw][hw]
    int hw, n, classes;
    const float *stem_wt;            // [27][16]
    const float *stem_scale, *stem_shift;
    const uint8_t *blob;             // every convolution's item (wres_write_item), in forward order
    const float *fc_wt;              // [64][classes]
    const float *fc_scale, *fc_shift;
    float *logits;
    float *const *keep;              // device array: the stem's and every block's fp32 NCHW output (nullable)
    long long wait_cycles;           // set by the launcher
};

}  // namespace wfu

// Image sizes whose activations fit the kernel's shared memory.
bool wres_fused_supported(int hw);
// Bytes of one convolution's item: bf16 levels [taps][C / 8][O][8], BN scale [O], shift [O].
size_t wres_item_bytes(int C, int O, int taps);
minw_status wres_write_item(const uint16_t *wb, const float *scale, const float *shift, int C, int Cp, int O, int taps,
                            uint8_t *out, cudaStream_t s);
minw_status launch_wres_fused(wfu::Args a, int B, cudaStream_t s);
// The kernel's timeout flag (as take_first_error).
int take_wres_error();

}  // namespace minw
