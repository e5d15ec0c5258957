// Packed H·v kernels in table mode (flips read from an entry table): the multi-block shapes, and single
// blocks with a thread per representative, FP16 vector storage with FP32 arithmetic.
#include "hvp_ops.h"

namespace ftlm {

const HvpOps<float> *hvp_ops_table_f16(int shape) {
    static const HvpOps<float> tab[3] = {FTLM_HVP_OPS_M(float, __half, ShapeIh, 2, false, 1),
                                         FTLM_HVP_OPS_M(float, __half, ShapeOh, 2, false, 1),
                                         FTLM_HVP_OPS_M(float, __half, ShapeTd, 2, false, 1)};
    if (shape < kShapeIh || shape > kShapeTd) return nullptr;  // single blocks: one thread per representative
    return &tab[shape - kShapeIh];
}

const HvpOps<float> *hvp_ops_lane_f16(int shape) {
    static const HvpOps<float> tab[5] = {FTLM_HVP_LANE_OPS(float, __half, 1), FTLM_HVP_LANE_OPS(float, __half, 2),
                                       FTLM_HVP_LANE_OPS(float, __half, 3), FTLM_HVP_LANE_OPS(float, __half, 4),
                                       FTLM_HVP_LANE_OPS(float, __half, 5)};
    if (shape < kShapeD1 || shape > kShapeD5) return nullptr;
    return &tab[shape - kShapeD1];
}

}  // namespace ftlm
