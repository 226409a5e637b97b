// conv_fused_bf16.cu -- instantiates the bfloat16-table tiles of the fused
// conv kernel (conv_fused.cuh); one unit per group so that they compile in
// parallel.
#include "conv_fused.cuh"

namespace qcnn {

static const FusedVariant kPart[] = {
    QCNN_FUSED_BF_SET(4), QCNN_FUSED_BF_SET(8)};

const FusedVariant *fused_variants_bf16(int *n) {
    *n = (int)(sizeof(kPart) / sizeof(kPart[0]));
    return kPart;
}

// 64-channel tiles (4 channels per warp), as conv_fused_plain.cu's: a layer of
// 64 channels gathered half its look-ups for channels that are not there, at 69%
// of the issue slots (with the tables built one position at a time: 3x3 64 -> 64 on
// 8 maps of 56x56 133 us, with this 93; 5x5 32 -> 48 on 16 of 28x28 63 us, 37).
static const FusedVariant kNarrow[] = {
    QCNN_FUSED_BF(4, 4, 1, 4, 16, 1, false, 0.9, 1.3), QCNN_FUSED_BF(4, 4, 1, 8, 16, 1, false, 0.9, 1.3),
    QCNN_FUSED_BF(7, 4, 1, 4, 16, 1, false, 0.9, 1.3), QCNN_FUSED_BF(7, 4, 1, 8, 16, 1, false, 0.9, 1.3)};

const FusedVariant *fused_variants_bf16_narrow(int *n) {
    *n = (int)(sizeof(kNarrow) / sizeof(kNarrow[0]));
    return kNarrow;
}

}  // namespace qcnn
