// Table-mode H·v with two right-hand sides per lane (hvp_flow.cuh), the full irrep set of I_h, FP16 vectors.
#include "hvp_ops.h"

namespace ftlm {

const HvpOps<float> *hvp_ops_flow_ih_f16(int B) {
    using T = __half;
    static const HvpOps<float> tab[5] = {FTLM_HVP_FLOW_OPS(T, ShapeIh, 4, 8), FTLM_HVP_FLOW_OPS(T, ShapeIh, 4, 0),
                                         FTLM_HVP_FLOW_OPS(T, ShapeIh, 8, 0), FTLM_HVP_FLOW_OPS(T, ShapeIh, 16, 24),
                                         FTLM_HVP_FLOW_OPS(T, ShapeIh, 16, 0)};
    if (B < 6 || B > 32 || B % 2) return nullptr;
    return &tab[B == 8 ? 0 : B < 8 ? 1 : B <= 16 ? 2 : B == 24 ? 3 : 4];
}

}  // namespace ftlm
