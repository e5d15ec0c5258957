// Table-mode H·v with two right-hand sides per lane (hvp_flow.cuh), the full irrep set of I_h, FP32 vectors.
#include "hvp_ops.h"

namespace ftlm {

const HvpOps<float> *hvp_ops_flow_ih_f32(int B) {
    using T = float;
    static const HvpOps<float> fixed[4] = {FTLM_HVP_FLOW_OPS(T, ShapeIh, 4, 8), FTLM_HVP_FLOW_OPS(T, ShapeIh, 8, 16),
                                           FTLM_HVP_FLOW_OPS(T, ShapeIh, 16, 24), FTLM_HVP_FLOW_OPS(T, ShapeIh, 16, 32)};
    static const HvpOps<float> any[3] = {FTLM_HVP_FLOW_OPS(T, ShapeIh, 4, 0), FTLM_HVP_FLOW_OPS(T, ShapeIh, 8, 0),
                                         FTLM_HVP_FLOW_OPS(T, ShapeIh, 16, 0)};
    return flow_pick(B, fixed, any);
}

}  // namespace ftlm
