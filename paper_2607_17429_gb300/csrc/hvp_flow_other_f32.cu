// Table-mode H·v with two right-hand sides per lane (hvp_flow.cuh), the full irrep sets of O_h and T_d, FP32 vectors.
#include "hvp_ops.h"

namespace ftlm {

const HvpOps<float> *hvp_ops_flow_other_f32(int shape, int B) {
    using T = float;
    static const HvpOps<float> tab[2][3] = {
        {FTLM_HVP_FLOW_OPS(T, ShapeOh, 4, 0), FTLM_HVP_FLOW_OPS(T, ShapeOh, 8, 0), FTLM_HVP_FLOW_OPS(T, ShapeOh, 16, 0)},
        {FTLM_HVP_FLOW_OPS(T, ShapeTd, 4, 0), FTLM_HVP_FLOW_OPS(T, ShapeTd, 8, 0), FTLM_HVP_FLOW_OPS(T, ShapeTd, 16, 0)}};
    if ((shape != kShapeOh && shape != kShapeTd) || B < 6 || B > 32 || B % 2) return nullptr;
    return &tab[shape == kShapeTd][B <= 8 ? 0 : B <= 16 ? 1 : 2];
}

}  // namespace ftlm
