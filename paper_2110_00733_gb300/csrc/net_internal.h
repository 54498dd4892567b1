// net_internal.h -- kernel arguments and launchers of the warm-start network.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace hnet {

// One periodic 3x3x3 convolution.  Input channels are the concatenation
// [src0 (c0s channels, full resolution), src1 (c1s channels, half
// resolution, upsampled by nearest neighbour)]; c0s, c1s multiples of 16,
// c1s = 0 for a single source.  W: [27][cout][c0s + c1s] BF16.  Output
// [voxels][cout], BF16 (out_bf16) or FP32 (out_f32), cout a multiple of 16.
struct ConvArgs {
    int B, n1, n2, n3;
    const __nv_bfloat16 *src0;
    int c0s;
    const __nv_bfloat16 *src1;
    int c1s;
    const __nv_bfloat16 *W;
    const float *bias;      // [cout] or null
    int cout;
    int relu;
    __nv_bfloat16 *out_bf16;
    float *out_f32;
    int *err;               // set when a bounded wait gives up (filled in by the launchers)
};

// Weight gradient of a convolution whose input is described by `in` (sources
// and grid only) and whose output gradient is G [voxels][cout] BF16:
// partial[s][t][cout][c0s + c1s] FP32 over S voxel splits.
struct WgradArgs {
    ConvArgs in;
    const __nv_bfloat16 *G;
    int cout;
    float *partial;
    int S;
};

// the launchers return -1 for a shape that they do not take, -2 without an error
// word, -3 where the device could not be set up
int conv3_forward_tc(const ConvArgs &a, cudaStream_t st);   // tcgen05, cout <= 256
// the word of the current device, or of another, that a bounded wait of a tcgen05
// convolution sets as it gives up (null: it could not be allocated)
int *conv3_tc_error_word();
int *conv3_tc_error_word_of(int dev);
// nonzero if one did on the current device (clears it if asked)
int conv3_tc_error(int clear);
// whether the shape is one of the weight gradient's: channel counts multiples of
// 16, 16 <= cout <= 64, and even grid sizes where there is a second source (its
// half-resolution grid has no voxel for the last plane of an odd one)
bool conv3_wgrad_takes(const WgradArgs &a);
int conv3_wgrad(const WgradArgs &a, cudaStream_t st);   // tcgen05

}  // namespace hnet
