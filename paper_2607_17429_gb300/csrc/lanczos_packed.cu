// FTLM Lanczos chains on packed sets (Section 2.2 of arXiv 2607.17429), batched
// through one packed H·v launch per step, every launch of the step loop overlapping
// the end of the one before (while profiling, captured in a CUDA graph).
//
// The vectors are kept unnormalised: u_j with v_j = s_j u_j.  One step j is
//   A  y = H u_j (packed H·v) with <u_j, y> per (block, chain) fused into
//      the H·v epilogue;
//   fA alpha_j = s_j^2 <u_j, y>; coefficients (s_j, alpha_j s_j, beta_j s_{j-1});
//   U  w = s_j y - alpha_j s_j u_j - beta_j s_{j-1} u_{j-1}  (= H v_j - alpha_j v_j
//      - beta_j v_{j-1}), written over y, with |w|^2 per (block, chain);
//   fB beta_{j+1} = |w|, stop test, s_{j+1} = 1 / beta_{j+1}, u_{j+1} = w.
// Dot products and norms: exact products, double-float sums per representative
// and lane (FP32 vectors) or FP64 (FP64 vectors), FP64 across lanes and CTAs in a
// fixed order, so repeated runs give identical coefficients.  A chain stops
// after step j when beta_{j+1} <= tol (|alpha_j| + beta_j) (tol 1e-12 for FP64,
// 1e-6 for FP32 vectors) or when j + 1 = min(n_steps, dim).
//
// Several packed sets of the same group and shape (for instance every S^z
// sector of a cluster) run as the parts of one launch per kernel (two for the
// H·v when only some of them have a flip table).
#include <string.h>

#include <algorithm>
#include <vector>

#include "hvp_ops.h"
#include "lanczos_packed.h"
#include "philox.cuh"
#include "ritz_thermo.cuh"

namespace ftlm {

void hv_profile_add(double ms, uint64_t rows);
unsigned long long wait_limit_cycles();

namespace {

constexpr int kLzThreads = 256;

template <typename VT>
struct LzPart {
    uint64_t n_reps;
    uint64_t tile0;
    const HvRec *rec;
    const uint8_t *ntab;           // [n_sid][K] n_k(sid)
    const VT *V[kPMaxK];           // block k: [n_sid][d_k][d_k] (Eq. 11), lifts the start vectors
    const uint64_t *boff[kPMaxK];  // block k's row offsets [n_reps] (start-vector counters)
    uint32_t key1[kPMaxK];         // Philox key word 1 of block k (block id)
    int entry0;                    // index of (part, block 0, chain 0) in the state arrays: p * K * B
    void *y;                       // start vectors: output, of the storage type
};

template <typename VT>
struct LzArgs {
    int n_parts;
    LzPart<VT> part0;
    const LzPart<VT> *parts;
    uint64_t n_tiles;
    int tile_reps;
    int B, BT, lgBT;
    int W, dims[kPMaxK], zoff[kPMaxK];
    int rng;
    uint32_t chain0, key0;
    double *norm_part;     // [n_parts][gridDim.x][K][B]
};

// Start vectors u_0 (Philox per block row index and chain, lifted by V_k(r)),
// with |u_0|^2 per (block, chain) as per-CTA partials.  Rows of representative
// r: r W + Z_k + gamma.
template <typename VT, typename ST, int K>
__global__ void __launch_bounds__(kLzThreads) lzp_start(const __grid_constant__ LzArgs<VT> a) {
    __shared__ double red[kPMaxK * 32];
    const int warps = blockDim.x >> 5;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int B = a.B, BT = a.BT;
    const int Q = 32 >> a.lgBT;
    const int b = lane & (BT - 1), fg = lane >> a.lgBT;
    for (int i = threadIdx.x; i < K * B; i += blockDim.x) red[i] = 0.0;
    __syncthreads();
    DotAcc<VT> acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k].zero();
    int cur = -1;
    auto flush = [&](int p) {
        double v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            v[k] = acc[k].value();
            for (int w = BT; w < 32; w <<= 1) v[k] += __shfl_xor_sync(kFullMask, v[k], w);
        }
        for (int w = 0; w < warps; ++w) {
            __syncthreads();
            if (wid == w && lane < B) {
#pragma unroll
                for (int k = 0; k < K; ++k) red[k * B + lane] += v[k];
            }
        }
        __syncthreads();
        double *dst = a.norm_part + ((size_t)p * gridDim.x + blockIdx.x) * K * B;
        for (int i = threadIdx.x; i < K * B; i += blockDim.x) {
            dst[i] = red[i];
            red[i] = 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k].zero();
    };
    for (uint64_t t = blockIdx.x; t < a.n_tiles; t += gridDim.x) {
        int p = 0;
        if (a.n_parts > 1) {
            int lo = 0, hi = a.n_parts - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.parts[mid].tile0 <= t)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            p = lo;
        }
        const LzPart<VT> &P = a.n_parts == 1 ? a.part0 : a.parts[p];
        if (p != cur) {
            if (cur >= 0) flush(cur);
            cur = p;
        }
        const uint64_t r0 = (t - P.tile0) * (uint64_t)a.tile_reps;
        const uint64_t r1 = min(r0 + (uint64_t)a.tile_reps, P.n_reps);
        for (uint64_t rep = r0 + wid; rep < r1; rep += warps) {
            const HvRec rr = P.rec[rep];
            const int sid = (int)rr.sid;
            if (b >= B) continue;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int D = a.dims[k];
                for (int gam = fg; gam < D; gam += Q) {
                    const size_t e = ((size_t)rr.idx * a.W + a.zoff[k] + gam) * B + b;
                    const uint64_t row0 = __ldg(P.boff[k] + rep);
                    VT v;
                    if (sid == 0) {
                        v = start_value_t<VT>(row0 + (uint64_t)gam, a.chain0 + (uint32_t)b, a.key0, P.key1[k], a.rng);
                    } else {  // lift the n_k(r) coefficients: V_k(r) x_k(r)
                        const int nk = __ldg(P.ntab + sid * K + k);
                        const VT *Vr = P.V[k] + ((size_t)sid * D + gam) * D;
                        v = (VT)0;
                        for (int q = 0; q < nk; ++q)
                            v += __ldg(Vr + q) * start_value_t<VT>(row0 + (uint64_t)q, a.chain0 + (uint32_t)b,
                                                                   a.key0, P.key1[k], a.rng);
                    }
                    const ST sv = st_put<VT, ST>(v);
                    static_cast<ST *>(P.y)[e] = sv;
                    const VT vs = st_get<VT, ST>(sv);  // norms of the values as stored
                    acc[k].add(vs, vs);
                }
            }
        }
    }
    if (cur >= 0) flush(cur);
}

// The update on the flat packed vector, 4 streams of W B elements per representative (HBM bound).
// Rows of every representative are consecutive W-row segments, so element e of a part has row
// (e / B) mod W and chain e mod B; a CTA covers W B 2^k elements at a time, VEC neighbours per thread
// (four chains of one row with 8- or 16-byte loads when B is a multiple of four, else one), so every
// thread keeps its (row, chains), hence one block, one set of coefficients and VEC accumulators.  A CTA
// takes one run of representatives of one part; a part's runs depend on the part alone, so a set gives
// the same sums in any mix.  Per run the elements of equal (row, chain) meet in a fixed tree and a
// block's rows are added in order.  (Every CTA walking every part, with 256 terms scanned per (block,
// chain): 1.17 ms a step for the six s = 3/2 icosahedron sectors M = 0..5 at 24 chains, 0.12 ms now;
// the icosidodecahedron's 5.3 GB a step at 8 chains 0.84 ms before, 0.74 ms now.)
constexpr int kUpdElems = 1024;  // elements of a CTA at a time, at most (W B <= 1024)
constexpr int kUpdThreads = 1024;  // threads per SM aimed at
constexpr int kUpdMinSteps = 8;    // loop steps of a run, at least (its reduction costs about two)

template <typename VT>
struct LzUpd {
    int n_parts, W, B, K, has_prev, n_sub;  // n_sub: representatives side by side in a CTA (a power of two)
    int zrow[kPMaxK + 1];       // first row of each block in a segment, then W
    int blk_of_row[32];         // block of each row of a segment
    const uint64_t *run0, *run_reps;  // [n_parts]: first run of each part, representatives per run
    const uint64_t *elem0;      // [n_parts + 1] first element of each part in the vectors
    const int *entry0;          // [n_parts] p * K * B
    void *y;                    // in: H u_j, out: w (storage type)
    const void *u, *up;
    const VT *coef;             // [entries][3]
    double *norm_part;          // [runs][K][B]
};

// VEC neighbouring stored elements, one load or store
template <typename VT, typename ST, int VEC>
__device__ __forceinline__ void upd_load(const ST *p, VT (&v)[VEC]) {
    if constexpr (VEC == 1) {
        v[0] = st_get<VT, ST>(*p);
    } else {
        alignas(16) ST s[VEC];
        constexpr int BYTES = VEC * (int)sizeof(ST);
        if constexpr (BYTES == 8) {
            *reinterpret_cast<uint2 *>(s) = *reinterpret_cast<const uint2 *>(p);
        } else {
#pragma unroll
            for (int i = 0; i < BYTES / 16; ++i) reinterpret_cast<uint4 *>(s)[i] = reinterpret_cast<const uint4 *>(p)[i];
        }
#pragma unroll
        for (int i = 0; i < VEC; ++i) v[i] = st_get<VT, ST>(s[i]);
    }
}
template <typename ST, int VEC>
__device__ __forceinline__ void upd_store(ST *p, const ST (&s)[VEC]) {
    constexpr int BYTES = VEC * (int)sizeof(ST);
    if constexpr (VEC == 1) {
        *p = s[0];
    } else if constexpr (BYTES == 8) {
        *reinterpret_cast<uint2 *>(p) = *reinterpret_cast<const uint2 *>(s);
    } else {
#pragma unroll
        for (int i = 0; i < BYTES / 16; ++i) reinterpret_cast<uint4 *>(p)[i] = reinterpret_cast<const uint4 *>(s)[i];
    }
}

template <typename VT, typename ST, int VEC>
__global__ void __launch_bounds__(VEC == 1 ? kUpdElems : kUpdElems / VEC) lzp_update(const __grid_constant__ LzUpd<VT> a) {
    __shared__ double red[kUpdElems];
    const int B = a.B, WB = a.W * a.B, K = a.K, tid = threadIdx.x;
    const int tb = tid * VEC % WB, k = a.blk_of_row[tb / B], b = tb % B;
    let_next_start();
    const uint64_t run = blockIdx.x + prior_done(), T = (uint64_t)blockDim.x * VEC;
    int p = 0;
    for (int hi = a.n_parts - 1; p < hi;) {  // last part whose first run is <= run (parts without runs come before it)
        const int mid = (p + hi + 1) >> 1;
        if (a.run0[mid] <= run)
            p = mid;
        else
            hi = mid - 1;
    }
    ST *__restrict__ y = static_cast<ST *>(a.y);
    const ST *__restrict__ u = static_cast<const ST *>(a.u);
    const ST *__restrict__ up = static_cast<const ST *>(a.up);
    const uint64_t len = a.run_reps[p] * (uint64_t)WB, start = a.elem0[p] + (run - a.run0[p]) * len;
    const uint64_t end = min(a.elem0[p + 1], start + len);
    const VT *c = a.coef + ((size_t)a.entry0[p] + k * B + b) * 3;
    VT cy[VEC], cu[VEC], cp[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        cy[v] = c[3 * v];
        cu[v] = c[3 * v + 1];
        cp[v] = a.has_prev ? c[3 * v + 2] : (VT)0;
    }
    DotAcc<VT> acc[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v].zero();
    auto step = [&](uint64_t e, const VT(&yv)[VEC], const VT(&uv)[VEC], const VT(&pv)[VEC]) {
        alignas(16) ST ws[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            ws[v] = st_put<VT, ST>(cy[v] * yv[v] - cu[v] * uv[v] - cp[v] * pv[v]);
            const VT w = st_get<VT, ST>(ws[v]);
            acc[v].add(w, w);
        }
        upd_store<ST, VEC>(y + e, ws);
    };
    constexpr int U = VEC == 1 ? 4 : 2;  // steps in flight per thread
    uint64_t e = start + (uint64_t)tid * VEC;
    for (; e + (U - 1) * T < end; e += U * T) {
        VT yv[U][VEC], uv[U][VEC], pv[U][VEC];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            upd_load<VT, ST, VEC>(y + e + q * T, yv[q]);
            upd_load<VT, ST, VEC>(u + e + q * T, uv[q]);
#pragma unroll
            for (int v = 0; v < VEC; ++v) pv[q][v] = (VT)0;
            if (a.has_prev) upd_load<VT, ST, VEC>(up + e + q * T, pv[q]);
        }
#pragma unroll
        for (int q = 0; q < U; ++q) step(e + q * T, yv[q], uv[q], pv[q]);
    }
    for (; e < end; e += T) {
        VT yv[VEC], uv[VEC], pv[VEC];
        upd_load<VT, ST, VEC>(y + e, yv);
        upd_load<VT, ST, VEC>(u + e, uv);
#pragma unroll
        for (int v = 0; v < VEC; ++v) pv[v] = (VT)0;
        if (a.has_prev) upd_load<VT, ST, VEC>(up + e, pv);
        step(e, yv, uv, pv);
    }
#pragma unroll
    for (int v = 0; v < VEC; ++v) red[tid * VEC + v] = acc[v].value();
    __syncthreads();
    for (int h = a.n_sub >> 1; h; h >>= 1) {
        for (int i = tid; i < h * WB; i += blockDim.x) red[i] += red[i + h * WB];
        __syncthreads();
    }
    for (int i = tid; i < K * B; i += blockDim.x) {
        const int kk = i / B, bb = i % B;
        double sum = 0.0;
        for (int r = a.zrow[kk]; r < a.zrow[kk + 1]; ++r) sum += red[r * B + bb];
        a.norm_part[(size_t)run * K * B + i] = sum;
    }
}

struct LzState {
    double *alpha, *beta;       // [n_steps][entries]
    double *s, *s_prev, *bprev; // [entries]
    double *sig;                // [entries] power-of-two scale of the stored u_{j+1} (FP16 storage; else 1)
    const double *rms_rows;     // [n_parts * K] sqrt(packed rows of the block) / (16 Hmax): the scale target
    int *active, *steps;        // [entries]
    const int *m_max;           // [n_parts * K]
    double *coef64;             // [entries][3]
    float *coef32;              // [entries][3]
};

// The partials of a part: n rows of [K][B], the i-th in row base + (first + i) mod wrap.  `first` is the CTA of
// the part's first tile, so the order is that of its own tiles, whatever part came before.
struct LzFin {
    uint64_t base, wrap, first, n;
};

// One CTA per part and 32 (block, chain) entries: a lane per entry, eight warps over slices of the
// part's partials (fixed association: it depends on their count only).
// mode 0: start-vector norms; 1: alpha_j and the update coefficients; 2: beta_{j+1}.
// With `scaled` (FP16 storage) the update writes sigma w instead of w, sigma the
// per-block power of two 2^floor(log2(sqrt(rows) / (16 Hmax))) with Hmax = |J|
// n_bonds s(s+1) >= |H|: since |w| = beta_{j+1} <= |H v_j| <= Hmax, the stored
// components have a root mean square at most 1/16 and no component can exceed
// sqrt(rows) / 16, independently of the block dimension (the subnormal range of
// FP16 that a fixed scale would reach in large blocks is avoided).  sigma
// multiplies the three coefficients, beta_{j+1} = |sigma w| / sigma, and the next
// scale s_{j+1} = 1 / |sigma w| (v_{j+1} = sigma w / (sigma beta_{j+1})).  Without
// it sigma = 1 and the recurrence is unchanged.
constexpr int kFinSlices = 8;

__global__ void __launch_bounds__(32 * kFinSlices)
    lzp_finalize(int mode, int j, int K, int B, const LzFin *fin, const double *part, LzState st, double tol, int scaled) {
    let_next_start();
    const int p = blockIdx.x + (int)prior_done(), KB = K * B;
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5, t = blockIdx.y * 32 + lane;
    __shared__ double sl_sum[kFinSlices][32];
    const int k = t / B, b = t % B;
    const size_t e = ((size_t)p * K + k) * B + b;
    const LzFin fp = fin[p];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (t < KB) {
        auto at = [&](uint64_t i) {
            uint64_t c = fp.first + i;
            if (c >= fp.wrap) c -= fp.wrap;
            return part[(fp.base + c) * KB + t];
        };
        constexpr uint64_t S = kFinSlices;
        const uint64_t n = fp.n;
        uint64_t i = (uint64_t)sl;
        for (; i + 3 * S < n; i += 4 * S) {  // four interleaved running sums: loads in flight
            const double v0 = at(i), v1 = at(i + S), v2 = at(i + 2 * S), v3 = at(i + 3 * S);
            acc[0] += v0;
            acc[1] += v1;
            acc[2] += v2;
            acc[3] += v3;
        }
        if (i < n) acc[0] += at(i);  // at most three left
        if (i + S < n) acc[1] += at(i + S);
        if (i + 2 * S < n) acc[2] += at(i + 2 * S);
    }
    sl_sum[sl][lane] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    __syncthreads();
    if (sl != 0 || t >= KB) return;
    double sum = sl_sum[0][lane];
    for (int q = 1; q < kFinSlices; ++q) sum += sl_sum[q][lane];
    const size_t E = (size_t)gridDim.x * K * B;
    if (mode == 0) {
        const double n = sqrt(sum);
        const bool on = n > 0.0 && st.m_max[p * K + k] > 0;
        st.s[e] = on ? 1.0 / n : 0.0;
        st.s_prev[e] = 0.0;
        st.bprev[e] = 0.0;
        st.sig[e] = 1.0;
        st.active[e] = on ? 1 : 0;
        st.steps[e] = 0;
    } else if (mode == 1) {
        double c0 = 0.0, c1 = 0.0, c2 = 0.0, al = 0.0;
        if (st.active[e]) {
            const double s = st.s[e];
            al = s * s * sum;
            c0 = s;
            c1 = al * s;
            c2 = j > 0 ? st.bprev[e] * st.s_prev[e] : 0.0;
            double sig = 1.0;
            if (scaled) {
                const double ex = floor(log2(st.rms_rows[p * K + k]));
                sig = ldexp(1.0, (int)fmin(fmax(ex, -100.0), 100.0));
            }
            st.sig[e] = sig;
            c0 *= sig;
            c1 *= sig;
            c2 *= sig;
        }
        st.alpha[(size_t)j * E + e] = al;
        st.coef64[3 * e] = c0;
        st.coef64[3 * e + 1] = c1;
        st.coef64[3 * e + 2] = c2;
        st.coef32[3 * e] = (float)c0;
        st.coef32[3 * e + 1] = (float)c1;
        st.coef32[3 * e + 2] = (float)c2;
    } else {
        if (!st.active[e]) {
            st.beta[(size_t)j * E + e] = 0.0;
            return;
        }
        const double bn = sqrt(sum);           // |sigma w| of the stored vector
        const double be = bn / st.sig[e];      // beta_{j+1} = |w|
        const double al = st.alpha[(size_t)j * E + e];
        st.beta[(size_t)j * E + e] = be;
        if (j + 1 >= st.m_max[p * K + k] || be <= tol * (fabs(al) + st.bprev[e])) {
            st.active[e] = 0;
            st.steps[e] = j + 1;
        } else {
            st.s_prev[e] = st.s[e];
            st.s[e] = 1.0 / bn;
            st.bprev[e] = be;
        }
    }
}

// flips of a part in fixed-stride slots at `at`, counts behind them
template <typename VT>
void lz_use_flips(HvpPart<VT> &part, uint8_t *at, int stride) {
    part.eoff = nullptr;
    part.ent = reinterpret_cast<HvEntry *>(at);
    part.ecnt = at + (size_t)part.n_reps * stride * sizeof(HvEntry);
    part.estride = stride;
}

template <typename VT, typename ST>
ftlm_status lzp_start_launch(int K, const LzArgs<VT> &a, int grid, cudaStream_t st) {
    count_launch();
    switch (K) {
        case 1: lzp_start<VT, ST, 1><<<grid, kLzThreads, 0, st>>>(a); break;
        case 5: lzp_start<VT, ST, 5><<<grid, kLzThreads, 0, st>>>(a); break;
        case 10: lzp_start<VT, ST, 10><<<grid, kLzThreads, 0, st>>>(a); break;
        default: return fail(FTLM_EUNSUPPORTED, "no recurrence kernel for %d blocks", K);
    }
    FTLM_CUDA(cudaGetLastError());
    return FTLM_OK;
}


}  // namespace

// Searching once and reading the flips in every step replaces a search per step (six s = 3/2
// icosahedron sectors at 24 chains, 14 steps: 35.5 ms with a search in every H·v, 22.6 ms so; one block of
// the 4x6 lattice at 4 chains: 2.0 and 1.4 ms).  The table has fixed-stride slots, eight bytes per possible
// flip.  It is built where it takes at most twice the call's vectors, or 64 MB: single blocks of few
// rows on large sectors (one chain of the s = 3/2 dodecahedron: 480 bytes a representative for 60 of
// vectors) keep searching.
size_t lanczos_flip_bytes(const ftlm_sector *sec, const PackedSet *ps, int B, int esize) {
    if (sec->d_ent) return 0;
    const size_t bytes = (size_t)sec->n_reps * ((size_t)flip_stride(sec) * sizeof(HvEntry) + 1);
    const size_t vectors = 3 * (size_t)ps->rows * B * esize;
    return bytes <= std::max<size_t>(64u << 20, 2 * vectors) ? (bytes + 255) / 256 * 256 : 0;
}

size_t lanczos_spare_bytes(const ftlm_sector *sec, const PackedSet *ps, int B, int esize) {
    const size_t flips = lanczos_flip_bytes(sec, ps, B, esize);
    return flips + (flips || sec->d_ent ? (size_t)sec->n_reps * hvp_pad_row_bytes(sec, ps, B, esize) : 0);
}

// A launch over the parts with flip tables and one over those without run in turn in every step: a large
// sector that keeps searching leaves the others their tables (and their sums: the kernel of a part, and so its
// bits, do not depend on what runs with it).  Five icosidodecahedron sectors at four chains of dimension 3,
// one of them above the bound, 14 steps: 31.1 ms with a search in every part, 24.4 so.
template <typename VT>
struct LzHv {
    int p0 = 0, n = 0;           // parts
    HvpPlan<VT> plan[3];         // of the three rotations: x = vb[j % 3], y = vb[(j + 1) % 3]
    std::vector<HvpPart<VT>> parts[3];
    ScratchBuf<HvpPart<VT>> d_parts[3];
    size_t row = 0;              // first row of its dot partials
};

// spare: in, whether the call may take memory that it can do without (flip tables, padded rows); out, whether it did
template <typename VT, typename ST>
ftlm_status lanczos_packed_st(const std::vector<LzSetIn> &sets_in, int R, int n_steps, uint64_t seed, int rng,
                              cudaStream_t stream, double *alpha, double *beta, int *steps_done, bool &spare) {
    constexpr bool kScaled = sizeof(ST) < sizeof(VT);
    const int P = (int)sets_in.size();
    const PackedSet *ps0 = sets_in[0].ps;
    const int K = ps0->K;
    const size_t out_n = (size_t)P * K * R;
    for (size_t i = 0; i < out_n; ++i) steps_done[i] = 0;
    for (size_t i = 0; i < out_n * n_steps; ++i) alpha[i] = beta[i] = 0.0;
    const int Bmax = std::min(R, kMaxB);
    auto limit = [&](const LzSetIn &in, int k) {
        const int lim = in.n_steps > 0 ? std::min(in.n_steps, n_steps) : n_steps;
        return (int)std::min<uint64_t>((uint64_t)lim, in.blocks[k]->dim);
    };
    int m_all = 0;
    uint64_t rows = 0;
    for (const LzSetIn &in : sets_in) {
        rows += in.ps->rows;
        for (int k = 0; k < K; ++k) m_all = std::max(m_all, limit(in, k));
    }
    if (m_all == 0) return FTLM_OK;
    ScratchBuf<ST> vb[3];
    for (int q = 0; q < 3; ++q) FTLM_CUDA(vb[q].alloc(std::max<uint64_t>(rows, 1) * Bmax, stream));
    // ---- flips of the sectors without an entry table, searched once for all steps; parts with tables first
    ScratchBuf<uint8_t> flips;
    std::vector<LzSetIn> sets;
    std::vector<int> orig;        // place of each part in sets_in
    std::vector<size_t> flip_at;  // a part's place in flips
    int n_table = 0;
    {
        std::vector<size_t> by(P);
        size_t total = 0;
        for (int i = 0; i < P && spare; ++i)
            if (sets_in[i].spare)
                total += by[i] = lanczos_flip_bytes(sets_in[i].sec, sets_in[i].ps, Bmax, (int)sizeof(ST));
        if (total && flips.alloc(total, stream) != cudaSuccess) {
            cudaGetLastError();
            by.assign(P, 0);
        }
        size_t at = 0;
        for (bool table : {true, false})
            for (int i = 0; i < P; ++i) {
                if ((sets_in[i].sec->d_ent || by[i]) != table) continue;
                sets.push_back(sets_in[i]);
                orig.push_back(i);
                flip_at.push_back(by[i] ? at : SIZE_MAX);
                at += by[i];
                n_table += table;
            }
    }
    const bool may_pad = spare;
    spare = flips.p != nullptr;
    std::vector<uint64_t> row0(P + 1, 0);
    std::vector<int> m_max((size_t)P * K);
    for (int p = 0; p < P; ++p) {
        row0[p + 1] = row0[p] + sets[p].ps->rows;
        for (int k = 0; k < K; ++k) m_max[(size_t)p * K + k] = limit(sets[p], k);
    }
    const size_t E = (size_t)P * K * Bmax;
    ScratchBuf<double> dstate;
    ScratchBuf<float> fstate;
    ScratchBuf<int> istate;
    FTLM_CUDA(dstate.alloc(2 * (size_t)n_steps * E + 7 * E + (size_t)P * K, stream));
    FTLM_CUDA(fstate.alloc(3 * E, stream));
    FTLM_CUDA(istate.alloc(2 * E + (size_t)P * K, stream));
    LzState st;
    st.alpha = dstate.p;
    st.beta = dstate.p + (size_t)n_steps * E;
    st.s = st.beta + (size_t)n_steps * E;
    st.s_prev = st.s + E;
    st.bprev = st.s_prev + E;
    st.coef64 = st.bprev + E;
    st.sig = st.coef64 + 3 * E;
    st.rms_rows = st.sig + E;
    {
        std::vector<double> rr((size_t)P * K);
        for (int p = 0; p < P; ++p) {
            const ftlm_sector *sp = sets[p].sec;
            const double sp1 = 0.5 * sp->two_s * (0.5 * sp->two_s + 1.0);
            const double hmax = std::max(1e-300, fabs(sp->grp.J) * sp->grp.n_bonds() * sp1);  // >= |H|
            for (int k = 0; k < K; ++k)
                rr[(size_t)p * K + k] = sqrt((double)sp->n_reps * ps0->dims[k]) / (16.0 * hmax);
        }
        FTLM_CUDA(cudaMemcpyAsync(st.sig + E, rr.data(), rr.size() * 8, cudaMemcpyHostToDevice, stream));
    }
    st.coef32 = fstate.p;
    st.active = istate.p;
    st.steps = istate.p + E;
    st.m_max = istate.p + 2 * E;
    FTLM_CUDA(cudaMemcpyAsync(istate.p + 2 * E, m_max.data(), m_max.size() * sizeof(int), cudaMemcpyHostToDevice,
                              stream));
    ScratchBuf<int> derr;
    FTLM_CUDA(derr.alloc(1, stream));
    FTLM_CUDA(cudaMemsetAsync(derr.p, 0, sizeof(int), stream));
    ScratchBuf<HvpPart<float>> d_fparts;
    if (flips.p) {
        std::vector<HvpPart<float>> fparts;
        for (int p = 0; p < n_table; ++p) {
            if (flip_at[p] == SIZE_MAX) continue;
            HvpPart<VT> part;
            hvp_part_of<VT>(sets[p].sec, sets[p].ps, sets[p].blocks, nullptr, nullptr, part);
            lz_use_flips(part, flips.p + flip_at[p], flip_stride(sets[p].sec));
            fparts.emplace_back();
            hvp_copy_flips(part, fparts.back());
        }
        if (fparts.size() > 1) FTLM_CUDA(d_fparts.alloc(fparts.size(), stream));
        HvpPlan<float> build;
        ftlm_status sb = flips_build(sets[0].sec, fparts, d_fparts.p, derr.p, build);
        if (sb != FTLM_OK) return sb;
        if (fparts.size() > 1)
            FTLM_CUDA(cudaMemcpyAsync(d_fparts.p, fparts.data(), fparts.size() * sizeof(HvpPart<float>),
                                      cudaMemcpyHostToDevice, stream));
        if ((sb = hvp_launch_plan<float>(build, nullptr, stream, false)) != FTLM_OK) return sb;
    }
    int dev = 0, sms = kNumSMs;
    FTLM_CUDA(cudaGetDevice(&dev));
    FTLM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const double tol = sizeof(ST) == 8 ? 1e-12 : (sizeof(ST) == 4 ? 1e-6 : 1e-3);
    const char *ng = getenv("FTLM_NO_GRAPH");
    const bool use_graph = !(ng && strcmp(ng, "1") == 0);
    std::vector<double> ha, hb;
    std::vector<int> hs;

    for (int chain0 = 0; chain0 < R; chain0 += Bmax) {
        const int B = std::min(Bmax, R - chain0);
        const size_t EB = (size_t)P * K * B;  // entries of this batch
        LzHv<VT> hv[2];
        hv[0].n = hv[1].p0 = n_table;
        hv[1].n = P - n_table;
        ScratchBuf<uint8_t> pad;  // padded rows of the vector an H·v gathers from (B = 1)
        bool no_pad = !may_pad;
        for (int p = 0; p < n_table; ++p) no_pad = no_pad || !sets[p].spare;
        size_t hv_rows = 0;  // rows of dot partials
        for (LzHv<VT> &h : hv) {
            if (h.n == 0) continue;
            const uint64_t reps0 = row0[h.p0] / ps0->W, reps = row0[h.p0 + h.n] / ps0->W - reps0;
            for (int q = 0; q < 3; ++q) {
                HvpPlan<VT> &plan = h.plan[q];
                h.parts[q].resize(h.n);
                for (int i = 0; i < h.n; ++i) {
                    const int p = h.p0 + i;
                    hvp_part_of<VT>(sets[p].sec, sets[p].ps, sets[p].blocks, vb[q].p + row0[p] * B,
                                    vb[(q + 1) % 3].p + row0[p] * B, h.parts[q][i]);
                    if (flip_at[p] != SIZE_MAX)
                        lz_use_flips(h.parts[q][i], flips.p + flip_at[p], flip_stride(sets[p].sec));
                }
                ftlm_status s0 = hvp_plan<VT>(sets[h.p0].sec, ps0, h.parts[q], B, (int)sizeof(ST), plan, stream);
                if (s0 != FTLM_OK) return s0;
                const size_t pb = hvp_pad_bytes(plan, reps);
                if (pb && !pad.p && !no_pad && pad.alloc(pb, stream) != cudaSuccess) {
                    cudaGetLastError();
                    no_pad = true;
                }
                spare = spare || pad.p;
                if (pb && !no_pad) {  // the parts' rows follow one another in the vector
                    plan.a.pad_x = vb[q].p + row0[h.p0] * B;
                    plan.a.pad_out = pad.p;
                    plan.a.pad_n = reps;
                    for (int i = 0; i < h.n; ++i)
                        h.parts[q][i].xpad = pad.p + (row0[h.p0 + i] / ps0->W - reps0) * (size_t)plan.ops->pad_bytes;
                    if (h.n == 1) plan.a.part0.xpad = h.parts[q][0].xpad;
                }
                plan.a.err = derr.p;  // this call's own error word (launches on the same sector may run concurrently)
                plan.rows_total = row0[h.p0 + h.n] - row0[h.p0];
                if (h.n > 1) {
                    FTLM_CUDA(h.d_parts[q].alloc(h.n, stream));
                    FTLM_CUDA(cudaMemcpyAsync(h.d_parts[q].p, h.parts[q].data(), h.n * sizeof(HvpPart<VT>),
                                              cudaMemcpyHostToDevice, stream));
                    plan.a.parts = h.d_parts[q].p;
                }
            }
            h.row = hv_rows;
            hv_rows += (size_t)h.n * h.plan[0].geo.grid;
        }
        ScratchBuf<double> hv_part, lz_part;
        FTLM_CUDA(hv_part.alloc(hv_rows * K * B, stream));
        ScratchBuf<LzFin> fin;  // partials of the H·v, of the start vectors and of the update
        FTLM_CUDA(fin.alloc(3 * (size_t)P, stream));
        std::vector<LzFin> hfin(3 * (size_t)P);
        auto cta_partials = [](uint64_t tile0, uint64_t ntile, uint64_t row, int local, int grid) {
            const uint64_t g = (uint64_t)grid;  // CTA t mod grid took tile t and wrote [local part][CTA]
            return LzFin{row + (uint64_t)local * g, g, tile0 % g, std::min(ntile, g)};
        };
        for (const LzHv<VT> &h : hv)
            for (int i = 0; i < h.n; ++i)
                hfin[h.p0 + i] = cta_partials(h.plan[0].tile0[i], h.plan[0].ntile[i], h.row, i, h.plan[0].geo.grid);
        // ---- recurrence kernels: tiles of 64 representatives, up to 8 CTAs per SM
        const int lz_tile = 64;
        std::vector<uint64_t> lz_tile0(P + 1, 0);
        for (int p = 0; p < P; ++p) lz_tile0[p + 1] = lz_tile0[p] + (sets[p].sec->n_reps + lz_tile - 1) / lz_tile;
        const uint64_t lz_tiles = lz_tile0[P];
        const int lz_grid = (int)std::max<uint64_t>(1, std::min<uint64_t>(lz_tiles, (uint64_t)sms * 8));
        FTLM_CUDA(lz_part.alloc((size_t)P * lz_grid * K * B, stream));
        for (int p = 0; p < P; ++p)
            hfin[P + p] = cta_partials(lz_tile0[p], lz_tile0[p + 1] - lz_tile0[p], 0, p, lz_grid);
        std::vector<LzPart<VT>> lparts(P);  // start vectors
        ScratchBuf<LzPart<VT>> d_lparts;
        LzArgs<VT> la;
        for (int p = 0; p < P; ++p) {
            LzPart<VT> &lp = lparts[p];
            memset(&lp, 0, sizeof(lp));
            lp.n_reps = sets[p].sec->n_reps;
            lp.tile0 = lz_tile0[p];
            lp.rec = sets[p].sec->d_rec;
            lp.ntab = sets[p].ps->d_ntab;
            for (int k = 0; k < K; ++k) {
                lp.V[k] = sizeof(VT) == 8 ? reinterpret_cast<const VT *>(sets[p].blocks[k]->d_V)
                                          : reinterpret_cast<const VT *>(sets[p].blocks[k]->d_Vf);
                lp.boff[k] = sets[p].blocks[k]->d_off;
                lp.key1[k] = (uint32_t)sets[p].block_ids[k];
            }
            lp.entry0 = p * K * B;
            lp.y = vb[0].p + row0[p] * B;
        }
        memset(&la, 0, sizeof(la));
        la.n_parts = P;
        if (P == 1) {
            la.part0 = lparts[0];
        } else {
            FTLM_CUDA(d_lparts.alloc(P, stream));
            FTLM_CUDA(cudaMemcpyAsync(d_lparts.p, lparts.data(), P * sizeof(LzPart<VT>), cudaMemcpyHostToDevice,
                                      stream));
            la.parts = d_lparts.p;
        }
        la.W = ps0->W;
        la.n_tiles = lz_tiles;
        la.tile_reps = lz_tile;
        la.B = B;
        la.BT = hv[n_table ? 0 : 1].plan[0].a.BT;
        la.lgBT = hv[n_table ? 0 : 1].plan[0].a.lgBT;
        {
            int z = 0;
            for (int k = 0; k < K; ++k) {
                la.dims[k] = ps0->dims[k];
                la.zoff[k] = z;
                z += ps0->dims[k];
            }
        }
        la.rng = rng;
        la.chain0 = (uint32_t)chain0;
        la.key0 = (uint32_t)seed;
        la.norm_part = lz_part.p;
        // flat update: W B 2^k elements per CTA at a time, one run of representatives per CTA
        const int WB = ps0->W * B, up_vec = B % 4 == 0 ? 4 : 1;
        int n_sub = 1;
        while (2 * n_sub * WB <= (up_vec == 4 ? kUpdElems : kUpdElems / 2)) n_sub *= 2;
        const int up_threads = n_sub * WB / up_vec;
        const uint64_t up_ctas = (uint64_t)sms * std::max(1, std::min(8, kUpdThreads / up_threads));
        std::vector<uint64_t> elem0(P + 1), ut(2 * (size_t)P);  // runs: first, representatives
        std::vector<int> ent(P);
        uint64_t up_runs = 0;
        for (int p = 0; p <= P; ++p) elem0[p] = row0[p] * (uint64_t)B;
        for (int p = 0; p < P; ++p) {
            const uint64_t n = sets[p].sec->n_reps, steps = (n + n_sub - 1) / n_sub;
            const uint64_t len = n_sub * std::max<uint64_t>(kUpdMinSteps, (steps + up_ctas - 1) / up_ctas);
            ent[p] = p * K * B;
            ut[p] = up_runs;
            ut[P + p] = len;
            const uint64_t runs = (n + len - 1) / len;
            hfin[2 * P + p] = LzFin{up_runs, runs, 0, runs};
            up_runs += runs;
        }
        ScratchBuf<double> up_part;
        FTLM_CUDA(up_part.alloc(std::max<uint64_t>(1, up_runs) * K * B, stream));
        ScratchBuf<uint64_t> d_elem0, d_ut;
        ScratchBuf<int> d_ent;
        FTLM_CUDA(d_elem0.alloc(P + 1, stream));
        FTLM_CUDA(d_ut.alloc(2 * (size_t)P, stream));
        FTLM_CUDA(d_ent.alloc(P, stream));
        FTLM_CUDA(cudaMemcpyAsync(d_elem0.p, elem0.data(), (P + 1) * 8, cudaMemcpyHostToDevice, stream));
        FTLM_CUDA(cudaMemcpyAsync(d_ut.p, ut.data(), 2 * (size_t)P * 8, cudaMemcpyHostToDevice, stream));
        FTLM_CUDA(cudaMemcpyAsync(fin.p, hfin.data(), hfin.size() * sizeof(LzFin), cudaMemcpyHostToDevice, stream));
        FTLM_CUDA(cudaMemcpyAsync(d_ent.p, ent.data(), P * sizeof(int), cudaMemcpyHostToDevice, stream));
        const dim3 fin_grid(P, (K * B + 31) / 32);
        constexpr int kFinThreads = 32 * kFinSlices;
        LzUpd<VT> ua[3];
        for (int q = 0; q < 3; ++q) {
            LzUpd<VT> &U = ua[q];
            memset(&U, 0, sizeof(U));
            U.n_parts = P;
            U.W = ps0->W;
            U.B = B;
            U.K = K;
            int r = 0;
            for (int k = 0; k < K; ++k)
                for (int d = 0; d < ps0->dims[k]; ++d) U.blk_of_row[r++] = k;
            for (int k = 0; k < K; ++k) U.zrow[k + 1] = U.zrow[k] + ps0->dims[k];
            U.n_sub = n_sub;
            U.run0 = d_ut.p;
            U.run_reps = d_ut.p + P;
            U.elem0 = d_elem0.p;
            U.entry0 = d_ent.p;
            U.y = vb[(q + 1) % 3].p;
            U.u = vb[q].p;
            U.up = vb[(q + 2) % 3].p;
            U.coef = sizeof(VT) == 8 ? reinterpret_cast<const VT *>(st.coef64)
                                     : reinterpret_cast<const VT *>(st.coef32);
            U.norm_part = up_part.p;
        }
        // ---- start vectors and their norms
        ftlm_status s1 = lzp_start_launch<VT, ST>(K, la, lz_grid, stream);
        if (s1 != FTLM_OK) return s1;
        count_launch();
        lzp_finalize<<<fin_grid, kFinThreads, 0, stream>>>(0, 0, K, B, fin.p + P, lz_part.p, st, tol, kScaled);
        FTLM_CUDA(cudaGetLastError());
        // ---- the step loop (while profiling: captured once on a private stream, replayed once on the caller's)
        // Each launch overlaps the end of the one before: jobs of 8 to 14 steps on small sectors take 533, 745 and
        // 801 us a call, 583, 813 and 821 with the steps in a graph that is built for one replay, 627, 856
        // and 906 in a graph with overlap (its construction costs more), 22.3 ms in the large batch either way.
        // Profiling events between the launches keep them apart, and there the graph is the faster form.
        const bool prof = profiling_on(), overlap = !prof;
        std::vector<cudaEvent_t> ev;
        auto steps = [&](cudaStream_t ss, bool capture) -> ftlm_status {
            for (int j = 0; j < m_all; ++j) {
                const int q = j % 3;
                if (prof) {
                    cudaEvent_t e0, e1;
                    FTLM_CUDA(cudaEventCreate(&e0));
                    FTLM_CUDA(cudaEventCreate(&e1));
                    ev.push_back(e0);
                    ev.push_back(e1);
                    FTLM_CUDA(capture ? cudaEventRecordWithFlags(e0, ss, cudaEventRecordExternal)
                                      : cudaEventRecord(e0, ss));
                }
                for (LzHv<VT> &h : hv) {
                    if (h.n == 0) continue;
                    h.plan[q].a.overlap = overlap && j > 0;
                    ftlm_status s2 = hvp_launch_plan<VT>(h.plan[q], hv_part.p + h.row * K * B, ss, false);
                    if (s2 != FTLM_OK) return s2;
                }
                if (prof)
                    FTLM_CUDA(capture ? cudaEventRecordWithFlags(ev.back(), ss, cudaEventRecordExternal)
                                      : cudaEventRecord(ev.back(), ss));
                count_launch();
                FTLM_CUDA(launch_overlapped(overlap, lzp_finalize, fin_grid, kFinThreads, 0, ss, 1, j, K, B, fin.p,
                                            hv_part.p, st, tol, kScaled));
                LzUpd<VT> U = ua[q];
                U.has_prev = j > 0;
                count_launch();
                FTLM_CUDA(launch_overlapped(overlap, up_vec == 4 ? lzp_update<VT, ST, 4> : lzp_update<VT, ST, 1>,
                                            (unsigned)up_runs, up_threads, 0, ss, U));
                count_launch();
                FTLM_CUDA(launch_overlapped(overlap, lzp_finalize, fin_grid, kFinThreads, 0, ss, 2, j, K, B, fin.p + 2 * P,
                                            up_part.p, st, tol, kScaled));
            }
            return FTLM_OK;
        };
        if (prof) profile_flip_counter();  // allocated before the capture (no allocation while capturing)
        if (prof && use_graph) {
            cudaStream_t cap = nullptr;
            FTLM_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
            cudaGraph_t graph = nullptr;
            cudaGraphExec_t exec = nullptr;
            cudaError_t ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
            if (ce != cudaSuccess) {
                cudaStreamDestroy(cap);
                return fail(FTLM_ECUDA, "graph capture: %s", cudaGetErrorString(ce));
            }
            ftlm_status s3 = steps(cap, true);
            ce = cudaStreamEndCapture(cap, &graph);  // always end the capture, even after a failed launch
            cudaStreamDestroy(cap);
            if (s3 != FTLM_OK) {
                if (graph) cudaGraphDestroy(graph);
                return s3;
            }
            if (ce != cudaSuccess) return fail(FTLM_ECUDA, "graph capture: %s", cudaGetErrorString(ce));
            ce = cudaGraphInstantiate(&exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ce != cudaSuccess) return fail(FTLM_ECUDA, "graph instantiate: %s", cudaGetErrorString(ce));
            ce = cudaGraphLaunch(exec, stream);
            cudaError_t ce2 = cudaStreamSynchronize(stream);
            cudaGraphExecDestroy(exec);
            if (ce != cudaSuccess || ce2 != cudaSuccess)
                return fail(FTLM_ECUDA, "graph launch: %s", cudaGetErrorString(ce != cudaSuccess ? ce : ce2));
        } else {
            ftlm_status s3 = steps(stream, false);
            if (s3 != FTLM_OK) return s3;
            FTLM_CUDA(cudaStreamSynchronize(stream));
        }
        if (prof) {
            for (size_t i = 0; i + 1 < ev.size(); i += 2) {
                float ms = 0.f;
                if (cudaEventElapsedTime(&ms, ev[i], ev[i + 1]) == cudaSuccess) hv_profile_add(ms, rows * B);
            }
            for (auto e : ev) cudaEventDestroy(e);
        }
        // ---- results of the batch
        ha.resize((size_t)n_steps * E);
        hb.resize((size_t)n_steps * E);
        hs.resize(E);
        FTLM_CUDA(cudaMemcpyAsync(ha.data(), st.alpha, (size_t)n_steps * E * 8, cudaMemcpyDeviceToHost, stream));
        FTLM_CUDA(cudaMemcpyAsync(hb.data(), st.beta, (size_t)n_steps * E * 8, cudaMemcpyDeviceToHost, stream));
        FTLM_CUDA(cudaMemcpyAsync(hs.data(), st.steps, E * sizeof(int), cudaMemcpyDeviceToHost, stream));
        FTLM_CUDA(cudaStreamSynchronize(stream));
        {
            int err = 0;
            FTLM_CUDA(cudaMemcpyAsync(&err, derr.p, sizeof(int), cudaMemcpyDeviceToHost, stream));
            FTLM_CUDA(cudaStreamSynchronize(stream));
            if (err) {
                if (err & kErrWaitTimeout) return fail(FTLM_ETIMEOUT, "a bounded device wait gave up in H·v");
                return fail(FTLM_EINTERNAL, "device bounds check tripped in H·v (code %d)", err);
            }
        }
        for (int p = 0; p < P; ++p)
            for (int k = 0; k < K; ++k)
                for (int b = 0; b < B; ++b) {
                    const size_t e = ((size_t)p * K + k) * B + b;
                    const size_t o = ((size_t)orig[p] * K + k) * R + chain0 + b;
                    const int m = hs[e];
                    steps_done[o] = m;
                    for (int jj = 0; jj < m; ++jj) {
                        alpha[o * n_steps + jj] = ha[(size_t)jj * EB + e];
                        beta[o * n_steps + jj] = hb[(size_t)jj * EB + e];
                    }
                }
    }
    return FTLM_OK;
}

// A call that runs out of memory with flip tables or padded rows runs again without them.
template <typename VT, typename ST>
ftlm_status lanczos_packed_any(const std::vector<LzSetIn> &sets, int R, int n_steps, uint64_t seed, int rng,
                               cudaStream_t stream, double *alpha, double *beta, int *steps_done) {
    bool spare = true;
    ftlm_status st = lanczos_packed_st<VT, ST>(sets, R, n_steps, seed, rng, stream, alpha, beta, steps_done, spare);
    if (st != FTLM_ENOMEM || !spare) return st;
    cudaGetLastError();
    scratch_trim();
    spare = false;
    return lanczos_packed_st<VT, ST>(sets, R, n_steps, seed, rng, stream, alpha, beta, steps_done, spare);
}

template <typename VT>
ftlm_status lanczos_packed(const std::vector<LzSetIn> &sets, int R, int n_steps, uint64_t seed, int rng,
                           cudaStream_t stream, double *alpha, double *beta, int *steps_done, int esize) {
    if (esize == (int)sizeof(VT))
        return lanczos_packed_any<VT, VT>(sets, R, n_steps, seed, rng, stream, alpha, beta, steps_done);
    if constexpr (sizeof(VT) == 4) {
        if (esize == 2)
            return lanczos_packed_any<float, __half>(sets, R, n_steps, seed, rng, stream, alpha, beta, steps_done);
    }
    return fail(FTLM_EINVAL, "no %d-byte storage for this arithmetic type", esize);
}

template ftlm_status lanczos_packed<float>(const std::vector<LzSetIn> &, int, int, uint64_t, int, cudaStream_t,
                                           double *, double *, int *, int);
template ftlm_status lanczos_packed<double>(const std::vector<LzSetIn> &, int, int, uint64_t, int, cudaStream_t,
                                            double *, double *, int *, int);

}  // namespace ftlm
