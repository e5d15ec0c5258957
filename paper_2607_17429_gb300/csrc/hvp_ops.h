// Compiled packed H·v kernels: one entry per (shape, elements per lane, label width).
#pragma once

#include <string.h>

#include <vector>

#include "hvp_flow.cuh"
#include "hvp_lane.cuh"

namespace ftlm {

// Shape ids: one block of dimension 1..12 (Section 3's limit on d_Gamma; real
// forms of complex and quaternionic irreps count their real dimension), and the
// full real irrep sets of I_h, O_h and T_d in canonical irrep order (dimensions
// ascending).
enum {
    kShapeD1 = 0, kShapeD2, kShapeD3, kShapeD4, kShapeD5, kShapeD6, kShapeD7, kShapeD8, kShapeD9, kShapeD10,
    kShapeD11, kShapeD12, kShapeIh, kShapeOh, kShapeTd, kNumShapes
};
constexpr bool shape_is_single(int shape) { return shape >= kShapeD1 && shape <= kShapeD12; }
constexpr bool shape_is_wide(int shape) { return shape >= kShapeD6 && shape <= kShapeD12; }
using ShapeIh = Shape<1, 1, 3, 3, 3, 3, 4, 4, 5, 5>;
using ShapeOh = Shape<1, 1, 1, 1, 2, 2, 3, 3, 3, 3>;
using ShapeTd = Shape<1, 1, 2, 3, 3>;

template <typename VT>
struct HvpOps {
    int (*occupancy)(const HvpArgs<VT> &, int warps, int nbuf);
    ftlm_status (*launch)(HvpArgs<VT>, const HvpGeom &, cudaStream_t);
    int max_threads;
    int options;     // 1: rho tables in shared memory or read through L1, own rows prefetched or not (else fixed)
    int tile_fixed;  // one thread per representative: the CTA's threads, the most a tile takes (0: warp kernels)
    int most_cols;   // one thread per representative: right-hand sides per thread, at most
    int pad_bytes;   // one thread per representative, B = 1: bytes of a padded row (0: rows stay as they are)
};

#define FTLM_HVP_OPS_M(VT, ST, SH, GPL, HALF, MODE)                                              \
    HvpOps<VT> {                                                                                   \
        &hvp_occupancy_t<VT, ST, SH, GPL, HALF, MODE>, &hvp_launch_t<VT, ST, SH, GPL, HALF, MODE>, \
            hvp_max_threads<VT, SH>(), 1, 0, 0, 0                                                        \
    }
// one thread per representative (table mode, one block; hvp_lane.cuh)
#define FTLM_HVP_LANE_OPS(VT, ST, D) \
    HvpOps<VT> {                                                                                                   \
        &hvp_lane_occupancy_t<VT, ST, D>, &hvp_lane_launch_t<VT, ST, D>, kLaneThreads, 0, kLaneThreads,            \
            lane_most_cols<VT, ST, D>(), lane_pad_bytes<ST, D>()                                                  \
    }
// table mode, multi-block shapes, FP32 arithmetic (hvp_flow.cuh)
#define FTLM_HVP_FLOW_OPS(ST, SH, CL, BC)                                                      \
    HvpOps<float> {                                                                             \
        &hvp_flow_occupancy_t<ST, SH, CL, BC>, &hvp_flow_launch_t<ST, SH, CL, BC>, flow_threads<ST, SH, CL>(), 0, 0, 0, 0 \
    }
#define FTLM_HVP_OPS(VT, ST, SH, GPL, HALF) FTLM_HVP_OPS_M(VT, ST, SH, GPL, HALF, 0)

template <typename VT>
struct HvpPlan {
    HvpArgs<VT> a;
    HvpGeom geo;
    const HvpOps<VT> *ops = nullptr;
    int mode = 0;                     // 0: on-the-fly search; 1: entry table; 2: entry-table build
    uint64_t rows_total = 0;          // packed rows over all parts (profiling)
    std::vector<uint64_t> tile0, ntile;  // per part: first tile and tile count
};

// packed.cu
template <typename VT>
void hvp_part_of(const ftlm_sector *s, const PackedSet *ps, const ftlm_basis *const *blocks, const void *x, void *y,
                 HvpPart<VT> &p);
// esize: bytes of a stored vector element (sizeof(VT), or 2 for FP16 storage with VT = float)
template <typename VT>
ftlm_status hvp_plan(const ftlm_sector *s, const PackedSet *ps, std::vector<HvpPart<VT>> &parts, int B, int esize,
                     HvpPlan<VT> &plan, cudaStream_t tune_stream);
// padded copy of the parts' rows for a plan on the one-thread kernel at B = 1: bytes it needs (0: none), and its
// use (x: the first part's rows, the others' following; out: that many bytes).  Below 2^18 rows the vector sits in
// L2 and the copy's launch costs what it saves (2.5e5 rows of five: 91 us without, 88 with).
template <typename VT>
size_t hvp_pad_bytes(const HvpPlan<VT> &plan, uint64_t n_rows) {
    return plan.a.B == 1 && n_rows >= (1u << 18) ? (size_t)n_rows * plan.ops->pad_bytes : 0;
}
// bytes of one padded row at B right-hand sides of esize bytes (0: the block has none)
size_t hvp_pad_row_bytes(const ftlm_sector *s, const PackedSet *ps, int B, int esize);
template <typename VT>
ftlm_status hvp_launch_plan(const HvpPlan<VT> &plan, double *dot_part, cudaStream_t stream, bool timed);
// the part as the build kernel sees it (no vectors, no blocks)
template <typename VT>
void hvp_copy_flips(const HvpPart<VT> &p, HvpPart<float> &b) {
    memset(&b, 0, sizeof(b));
    b.n_reps = p.n_reps;
    b.n_all = p.n_all;
    b.rec = p.rec;
    b.bucket = p.bucket;
    b.n_buckets = p.n_buckets;
    b.bucket_shift = p.bucket_shift;
    b.n_sid = p.n_sid;
    b.rep0 = p.rep0;
    b.ent = p.ent;
    b.ecnt = p.ecnt;
    b.estride = p.estride;
}
// pieces of a plan (packed.cu): sector-wide arguments, geometry, tile order
template <typename VT>
void hvp_fill_common(const ftlm_sector *s, const PackedSet *ps, int B, int esize, HvpArgs<VT> &a);
template <typename VT>
ftlm_status hvp_choose_geom(const HvpOps<VT> *ops, HvpArgs<VT> a, bool tma, HvpGeom &geo);
template <typename VT>
void hvp_retile(HvpPlan<VT> &plan, std::vector<HvpPart<VT>> &parts);
// entries.cu: flips of the parts' representatives (rep0 .. rep0 + n_reps - 1) into ent, ecnt and estride of each part;
// d_parts: device copy of the parts when there are several
constexpr size_t kSplitBytes = 128u << 20;  // entry workspace of one H·v on the search path
inline int flip_stride(const ftlm_sector *s) { return s->grp.n_bonds() * (s->two_s == 1 ? 1 : 2); }
ftlm_status flips_build(const ftlm_sector *s, std::vector<HvpPart<float>> &parts, const HvpPart<float> *d_parts, int *err,
                        HvpPlan<float> &plan);
// scratch of one call, from a pool of at most kPoolBytes kept between calls (packed.cu)
ftlm_status scratch_alloc(void **p, size_t bytes, cudaStream_t stream);
void scratch_trim();
// entries.cu: the sector's optional entry table
ftlm_status entry_table_build(ftlm_sector *s, cudaStream_t stream);
void entry_table_free(ftlm_sector *s);

// null if the combination is not compiled (gpl: 2 for |G| <= 64, 4 for |G| <= 128)
const HvpOps<float> *hvp_ops_single_f32(int shape, int gpl, bool half);
const HvpOps<float> *hvp_ops_multi_f32(int shape, int gpl, bool half);
const HvpOps<double> *hvp_ops_single_f64(int shape, int gpl, bool half);
const HvpOps<double> *hvp_ops_multi_f64(int shape, int gpl, bool half);
const HvpOps<float> *hvp_ops_single_f16(int shape, int gpl, bool half);  // FP16 storage, FP32 arithmetic
const HvpOps<float> *hvp_ops_multi_f16(int shape, int gpl, bool half);
// one block of dimension 6..12 (label search with 4 elements per lane, any |G| <= 128):
// kind 0 search, 1 table (FP64), 2 table with one thread per representative (FP64: B = 1)
const HvpOps<float> *hvp_ops_wide_f32(int shape, bool half, int kind);
const HvpOps<double> *hvp_ops_wide_f64(int shape, bool half, int kind);
const HvpOps<float> *hvp_ops_wide_f16(int shape, bool half, int kind);
// table mode (flips from an entry table), shapes D1..D5 (FP64), I_h, O_h, T_d; esize 8, 4 or 2
const HvpOps<double> *hvp_ops_table_f64(int shape);
const HvpOps<float> *hvp_ops_table_f32(int shape);
const HvpOps<float> *hvp_ops_table_f16(int shape);
// table mode of the multi-block shapes for an even B in 6..32 (hvp_flow.cuh): lanes per flip and the ops
constexpr int flow_lanes(int B) { return B <= 8 ? 4 : B <= 16 ? 8 : 16; }
// Multiples of eight, whose rows are whole 32-byte sectors in FP32, have B as a compile-time constant (row strides as
// immediates).  FP32, ms a call without and with: ten icosidodecahedron irreps, B = 8 6.34, 5.79; 16 10.41, 9.91; 24
// 17.6, 16.9; s = 1 dodecahedron, M = 8, B = 32 3.37, 3.27; s = 2 cuboctahedron, M = 0, 8 1.29, 1.27; 16 2.02, 1.98; 24
// 3.93, 3.70; 32 3.97, 3.73.  T_d's sectors are too small to show it.
inline const HvpOps<float> *flow_pick(int B, const HvpOps<float> *fixed, const HvpOps<float> *any) {
    if (B < 6 || B > 32 || B % 2) return nullptr;
    return fixed && B % 8 == 0 ? &fixed[B / 8 - 1] : &any[B <= 8 ? 0 : B <= 16 ? 1 : 2];
}
const HvpOps<float> *hvp_ops_flow_ih_f32(int B);
const HvpOps<float> *hvp_ops_flow_ih_f16(int B);
const HvpOps<float> *hvp_ops_flow_other_f32(int shape, int B);
const HvpOps<float> *hvp_ops_flow_other_f16(int shape, int B);
// table mode, one thread per representative: single blocks (shapes D1..D5), FP64 at B = 1
const HvpOps<double> *hvp_ops_lane_f64(int shape);
const HvpOps<float> *hvp_ops_lane_f32(int shape);
const HvpOps<float> *hvp_ops_lane_f16(int shape);
// build mode (writes the entry table; no gathers or outputs)
const HvpOps<float> *hvp_ops_build(int gpl, bool half);

}  // namespace ftlm
