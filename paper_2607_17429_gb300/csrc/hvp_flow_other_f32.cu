// Table-mode H·v with two right-hand sides per lane (hvp_flow.cuh), the full irrep sets of O_h and T_d, FP32 vectors.
#include "hvp_ops.h"

namespace ftlm {

const HvpOps<float> *hvp_ops_flow_other_f32(int shape, int B) {
    using T = float;
    static const HvpOps<float> oh_fixed[4] = {FTLM_HVP_FLOW_OPS(T, ShapeOh, 4, 8), FTLM_HVP_FLOW_OPS(T, ShapeOh, 8, 16),
                                              FTLM_HVP_FLOW_OPS(T, ShapeOh, 16, 24), FTLM_HVP_FLOW_OPS(T, ShapeOh, 16, 32)};
    static const HvpOps<float> oh_any[3] = {FTLM_HVP_FLOW_OPS(T, ShapeOh, 4, 0), FTLM_HVP_FLOW_OPS(T, ShapeOh, 8, 0),
                                            FTLM_HVP_FLOW_OPS(T, ShapeOh, 16, 0)};
    static const HvpOps<float> td_any[3] = {FTLM_HVP_FLOW_OPS(T, ShapeTd, 4, 0), FTLM_HVP_FLOW_OPS(T, ShapeTd, 8, 0),
                                            FTLM_HVP_FLOW_OPS(T, ShapeTd, 16, 0)};
    return shape == kShapeOh ? flow_pick(B, oh_fixed, oh_any) : shape == kShapeTd ? flow_pick(B, nullptr, td_any) : nullptr;
}

}  // namespace ftlm
