// Table-mode H·v of one block (K = 1) with a thread per output representative and CV right-hand sides:
// Eqs. 15-16 in the pull form with the flips read from an entry table (Section 3).  A warp of the search
// or table kernel works on one representative at a time; with d B small most of its lanes idle and
// each representative is a chain of dependent memory round trips (record, entry offsets, entries,
// gathers).  Here every thread walks its own representative's entries, so a warp keeps 32 / (B / CV) such
// chains in flight.  CV is 1 for B = 1 and odd B, else 2 or 4 neighbouring right-hand sides, one vector
// load per row.  The contributions are summed in entry order, a few apart at a time (the warp
// kernels sum them per flip group and then across groups), so results agree with theirs to rounding.
//
// Blocks of dimension 1, 3, 4, 5 of the icosidodecahedron at M = 0, FP32, from the table: B = 1 0.19 to 0.40 ms;
// B = 8 2.6 to 3.1 ms with a warp per representative, 0.29 to 1.29 ms here; B = 32 7.2 to 9.1 ms, 0.9 to 4.3 ms.
// Bound by L1 sector look-ups of the gathers for rows of less than 32 bytes (B = 1: about one per cycle
// and SM), by the entries' and gathers' latency above.
#pragma once

#include "hvp.cuh"

namespace ftlm {

constexpr int kLaneThreads = 256;
// flips whose entries and rows are loaded before the first is summed
__host__ __device__ constexpr int lane_flips(int D, int CV) { return D * CV <= 4 ? 4 : D * CV <= 16 ? 2 : 1; }
// Flips summed apart before they meet the rest.  FP32 vectors: four, since one chain over all flips carries up to
// 1.6 times the error of a warp's short sums (icosidodecahedron, d = 5, B = 8: 6.7e-8 with a warp per representative,
// 9.4e-8 in one chain, 6.9e-8 in fours; B = 24 9.4, 9.4 and 6.9e-8; complete graph of 11 sites, d = 10, 14.1 and 9.5e-8).
// FP16 vectors round each output to 2^-11 and FP64 operations bind: as many as are loaded at a time.
template <typename ST, int FL>
__host__ __device__ constexpr int lane_sum() {
    return sizeof(ST) == 4 ? 4 : FL;
}
// right-hand sides per thread, at most `most`: the sums and accumulators of FP32 vectors fill the registers with four
// columns from dimension 5 on (d = 5, B = 8: 1.66 ms with four columns, 1.29 with two)
inline int lane_cols(int B, int most) { return B % 4 == 0 && most == 4 ? 4 : B % 2 == 0 ? 2 : 1; }
template <typename VT, typename ST, int D>
constexpr int lane_most_cols() {
    return sizeof(VT) == 8 ? 1 : D <= 4 || sizeof(ST) == 2 ? 4 : 2;
}

__host__ __device__ constexpr int lane_gcd(int a, int b) { return b == 0 ? a : lane_gcd(b, a % b); }

// Element j of a span of 32-bit words (j a compile-time constant after unrolling).
template <typename ST>
__device__ __forceinline__ ST span_elem(const uint32_t *w, int j) {
    if constexpr (sizeof(ST) == 2) {
        return __ushort_as_half((unsigned short)(w[j >> 1] >> (16 * (j & 1))));
    } else if constexpr (sizeof(ST) == 4) {
        return __uint_as_float(w[j]);
    } else {
        return __hiloint2double((int)w[2 * j + 1], (int)w[2 * j]);
    }
}

// The D stored elements of row r of x (D * sizeof(ST) bytes from byte r * D * sizeof(ST)).  A row
// starts at a multiple of gcd(D * sizeof(ST), 16) bytes past a 16-byte boundary, so the L aligned
// 16-byte words from that boundary cover it: L vector loads per lane instead of D scalar ones, a
// warp's gather then takes about 32 L sector lookups in L1 instead of 32 D.  The row is picked
// out of the words by its offset (selects over the possible offsets, no local memory).  Rows
// whose covering words would pass the end of x (n_elems elements), or an x that is not 16-byte
// aligned, take scalar loads.
template <typename VT, typename ST, int D>
__device__ __forceinline__ void lane_row(const ST *__restrict__ x, uint64_t r, uint64_t n_elems, bool vec,
                                         VT (&u)[D]) {
    constexpr int E = (int)sizeof(ST), RB = D * E, PER = 16 / E;
    constexpr int G = lane_gcd(RB, 16);
    constexpr int L = (16 - G + RB + 15) / 16;  // words covering a row at the largest offset
    constexpr int STEP = G / E, NOFF = 16 / G;  // offsets 0, STEP, ..., (NOFF - 1) STEP elements
    const uint64_t e0 = r * D, w0 = e0 / PER;
    if (vec && (w0 + L) * PER <= n_elems) {
        uint32_t w[4 * L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(x) + w0 + l);
            w[4 * l] = v.x;
            w[4 * l + 1] = v.y;
            w[4 * l + 2] = v.z;
            w[4 * l + 3] = v.w;
        }
        const int off = (int)(e0 - w0 * PER);
#pragma unroll
        for (int g = 0; g < D; ++g) u[g] = st_get<VT, ST>(span_elem<ST>(w, g));
#pragma unroll
        for (int k = 1; k < NOFF; ++k) {
            const bool hit = off == k * STEP;
#pragma unroll
            for (int g = 0; g < D; ++g) {
                const VT v = st_get<VT, ST>(span_elem<ST>(w, k * STEP + g));
                u[g] = hit ? v : u[g];
            }
        }
    } else {
#pragma unroll
        for (int g = 0; g < D; ++g) u[g] = st_get<VT, ST>(__ldg(x + e0 + g));
    }
}

// Rows whose size is no power of two straddle sectors: a copy of x with rows padded to the next one (PB bytes, 32
// at most) is made before the launch, and a row then is one aligned load (256 bits for PB = 32) and one
// sector (s = 3/2 dodecahedron, M = 14, d = 5: 3.84 -> 3.66 ms in FP32, 3.71 -> 3.1 in FP16; what remains is the
// rate of random sectors, 1.1e11 a second here).  0: the rows are aligned already or too long, or FP64,
// whose operations bind.
template <typename ST, int D>
__host__ __device__ constexpr int lane_pad_bytes() {
    int pb = 1;
    while (pb < D * (int)sizeof(ST)) pb *= 2;
    return pb == D * (int)sizeof(ST) || pb > 32 || sizeof(ST) == 8 ? 0 : pb;
}
template <int PB>
struct PadRow {
    uint32_t w[PB / 4];
};
template <typename ST, int D, int PB>
__device__ __forceinline__ PadRow<PB> pad_row(const ST *v) {
    PadRow<PB> r;
#pragma unroll
    for (int i = 0; i < PB / 4; ++i) r.w[i] = 0u;
#pragma unroll
    for (int g = 0; g < D; ++g) {
        if constexpr (sizeof(ST) == 2) {
            r.w[g >> 1] |= (uint32_t)__half_as_ushort(v[g]) << (16 * (g & 1));
        } else {  // FP64 rows are not padded
            r.w[g] = __float_as_uint(v[g]);
        }
    }
    return r;
}

// one thread per row: D elements in, PB bytes out (bandwidth of both)
template <typename ST, int D, int PB>
__global__ void __launch_bounds__(256) lane_pad_kernel(const ST *__restrict__ x, uint64_t n, void *out) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    ST v[D];
#pragma unroll
    for (int g = 0; g < D; ++g) v[g] = __ldg(x + i * D + g);
    const PadRow<PB> r = pad_row<ST, D, PB>(v);
    uint32_t *o = reinterpret_cast<uint32_t *>(static_cast<char *>(out) + i * PB);
    if constexpr (PB == 8) {
        *reinterpret_cast<uint2 *>(o) = make_uint2(r.w[0], r.w[1]);
    } else {
#pragma unroll
        for (int k = 0; k < PB / 16; ++k)
            reinterpret_cast<uint4 *>(o)[k] = make_uint4(r.w[4 * k], r.w[4 * k + 1], r.w[4 * k + 2], r.w[4 * k + 3]);
    }
}

// row r of the padded copy
template <typename VT, typename ST, int D, int PB>
__device__ __forceinline__ void padded_row(const void *xpad, uint64_t r, VT (&u)[D]) {
    const char *p = static_cast<const char *>(xpad) + r * PB;
    uint32_t w[PB / 4];
    if constexpr (PB == 8) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
        w[0] = v.x, w[1] = v.y;
    } else if constexpr (PB == 16) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
        w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
    } else {
        asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
            : "l"(p));
    }
#pragma unroll
    for (int g = 0; g < D; ++g) u[g] = st_get<VT, ST>(span_elem<ST>(w, g));
}

// CV neighbouring stored elements of row r, columns c .. c + CV - 1
template <typename VT, typename ST, int CV>
__device__ __forceinline__ void lane_cols_load(const ST *__restrict__ x, size_t e, bool vec, VT (&u)[CV]) {
    if constexpr (CV > 1) {
        constexpr int BYTES = CV * (int)sizeof(ST);
        if (vec) {
            alignas(16) ST s[CV];
            if constexpr (BYTES == 4)
                *reinterpret_cast<uint32_t *>(s) = __ldg(reinterpret_cast<const uint32_t *>(x + e));
            else if constexpr (BYTES == 8)
                *reinterpret_cast<uint2 *>(s) = __ldg(reinterpret_cast<const uint2 *>(x + e));
            else
                *reinterpret_cast<uint4 *>(s) = __ldg(reinterpret_cast<const uint4 *>(x + e));
#pragma unroll
            for (int v = 0; v < CV; ++v) u[v] = st_get<VT, ST>(s[v]);
            return;
        }
    }
#pragma unroll
    for (int v = 0; v < CV; ++v) u[v] = st_get<VT, ST>(__ldg(x + e + v));
}

// ONE: a single right-hand side (rows of D consecutive elements); PB: bytes of the padded copy's rows, 0 for none
template <typename VT, typename ST, int D, int CV, bool ONE, int PB>
__global__ void __launch_bounds__(kLaneThreads) hvp_lane_kernel(const __grid_constant__ HvpArgs<VT> a) {
    constexpr int RP = rho_row(D), FL = ONE ? 2 : lane_flips(D, CV), SUM = lane_sum<ST, FL>();
    extern __shared__ __align__(128) uint8_t smem[];
    VT *s_rho = reinterpret_cast<VT *>(smem);  // rho(g) of the block, [G][D][RP]
    uint8_t *s_bond = smem + (((size_t)a.rho_total * sizeof(VT) + 15) & ~(size_t)15);
    __shared__ double red[kLaneThreads];
    let_next_start();
    for (int i = threadIdx.x; i < a.rho_total; i += blockDim.x) s_rho[i] = a.rhoT[i];
    for (int i = threadIdx.x; i < 2 * a.n_bonds; i += blockDim.x) s_bond[i] = a.bonds[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int B = ONE ? 1 : a.B, tpr = ONE ? 1 : B / CV, per_cta = kLaneThreads / tpr;  // threads per representative
    const int lrep = (int)threadIdx.x / tpr, col = ((int)threadIdx.x - lrep * tpr) * CV;
    const VT halfJ = sizeof(VT) == 8 ? (VT)1 : a.J * (VT)0.5;  // as in hvp_kernel: FP64 scales the sums
    const VT zscale = sizeof(VT) == 8 ? a.J * (VT)0.5 : (VT)1;
    const bool want_dot = a.dot_part != nullptr;
    DotAcc<VT> dacc[CV];
#pragma unroll
    for (int v = 0; v < CV; ++v) dacc[v].zero();
    int cur_part = -1;
    unsigned long long n_flips = 0;  // profiling: one atomic per warp at the end
    auto flush = [&](int p) {        // CTA sums of the per-thread <x, y> per column, a fixed tree over representatives
#pragma unroll
        for (int v = 0; v < CV; ++v) {
            __syncthreads();
            red[threadIdx.x] = dacc[v].value();
            int top = 1;
            while (2 * top < per_cta) top *= 2;
            for (int h = top; h; h >>= 1) {
                __syncthreads();
                if (lrep < h && lrep + h < min(per_cta, 2 * h)) red[threadIdx.x] += red[threadIdx.x + h * tpr];
            }
            __syncthreads();
            if (lrep == 0) a.dot_part[((size_t)p * gridDim.x + blockIdx.x) * B + col + v] = red[threadIdx.x];
            dacc[v].zero();
        }
    };
    for (uint64_t t = blockIdx.x + prior_done(); t < a.n_tiles; t += gridDim.x) {
        int p = 0;
        if (a.n_parts > 1) {
            int lo = 0, hi = a.n_parts - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (__ldg(&a.parts[mid].tile0) <= t)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            p = lo;
        }
        if (want_dot && p != cur_part) {
            if (cur_part >= 0) flush(cur_part);
            cur_part = p;
        }
        const HvpPart<VT> &P = a.n_parts == 1 ? a.part0 : a.parts[p];
        const uint64_t rep = (t - P.tile0) * (uint64_t)P.tile_reps + lrep;
        if (rep >= P.n_reps || lrep >= P.tile_reps) continue;
        const ST *__restrict__ x = static_cast<const ST *>(P.x);
        ST *__restrict__ y = static_cast<ST *>(P.y);
        const uint64_t n_elems = P.n_all * (uint64_t)D;
        const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
        const uint64_t at = P.rep0 + rep;  // in the sector
        const HvRec rr = P.rec[at];
        const int sid = (int)rr.sid;
        const size_t seg = at * D * B + col;
        if (sid != 0 && __ldg(P.wtab + sid) == 0) {
#pragma unroll
            for (int g = 0; g < D; ++g)
#pragma unroll
                for (int v = 0; v < CV; ++v) y[seg + (size_t)g * B + v] = st_put<VT, ST>((VT)0);
            continue;
        }
        const uint64_t lab = rr.label;
        uint64_t e0, e1;
        if (P.ecnt) {
            e0 = rep * (uint64_t)P.estride;
            e1 = e0 + __ldg(P.ecnt + rep);
        } else {
            e0 = __ldg(P.eoff + at);
            e1 = __ldg(P.eoff + at + 1);
        }
        int diag4 = 0;
        if (a.two_s == 1) {  // every bond is +1/4 or, when it flips, -1/4
            diag4 = a.n_bonds - 2 * (int)(e1 - e0);
        } else {
            for (int e = 0; e < a.n_bonds; ++e)
                diag4 += (2 * (int)hvp_digit(lab, s_bond[2 * e], a.bits) - a.two_s) *
                         (2 * (int)hvp_digit(lab, s_bond[2 * e + 1], a.bits) - a.two_s);
        }
        const VT diag = a.J * (VT)diag4 * (VT)0.25;
        if (col == 0) n_flips += e1 - e0;
        VT z[D][CV];
#pragma unroll
        for (int g = 0; g < D; ++g)
#pragma unroll
            for (int v = 0; v < CV; ++v) z[g][v] = (VT)0;
        // one flip: coefficient of Eq. 3 times sqrt|Stab r'| (the 1/sqrt|Stab r| comes last), gather of
        // the target's rows; flips are summed in entry order
        auto coef = [&](uint2 raw) {
            const uint32_t g8 = raw.y & 255u, es = (raw.y >> 8) & 255u, sidf = raw.y >> 16;
            VT c = halfJ;
            if (a.two_s != 1) {
                const int b = (int)(es & 127u);
                const int ai = (int)hvp_digit(lab, s_bond[2 * b], a.bits);
                const int aj = (int)hvp_digit(lab, s_bond[2 * b + 1], a.bits);
                c = halfJ * ((es & 128u) == 0 ? a.up[ai] * a.dn[aj] : a.dn[ai] * a.up[aj]);
            }
            VT cf = c * __ldg(P.sqrtS + sidf);
            if ((g8 & 128u) && (a.neg & 1u)) cf = -cf;  // (g*, 1) in a Gamma- block
            return cf;
        };
        auto gather = [&](uint64_t r, VT(&u)[D][CV]) {
            if constexpr (ONE) {
                VT w[D];
                if constexpr (PB > 0)
                    padded_row<VT, ST, D, PB>(P.xpad, r, w);
                else
                    lane_row<VT, ST, D>(x, r, n_elems, vec, w);
#pragma unroll
                for (int g = 0; g < D; ++g) u[g][0] = w[g];
            } else {
#pragma unroll
                for (int g = 0; g < D; ++g) lane_cols_load<VT, ST, CV>(x, (r * D + g) * B + col, vec, u[g]);
            }
        };
        // cf rho(g*)^T u, the first of a sum or added to it
        auto contract = [&](uint2 raw, VT cf, const VT(&u)[D][CV], VT(&s)[D][CV], bool first) {
            const VT *R = s_rho + (size_t)(raw.y & 127u) * D * RP;
            VT acc[D][CV];
#pragma unroll
            for (int ga = 0; ga < D; ++ga) {
                VT row[RP];
                load_row<VT, RP>(R + ga * RP, row);
#pragma unroll
                for (int be = 0; be < D; ++be)
#pragma unroll
                    for (int v = 0; v < CV; ++v) acc[be][v] = ga == 0 ? row[be] * u[0][v] : acc[be][v] + row[be] * u[ga][v];
            }
#pragma unroll
            for (int be = 0; be < D; ++be)
#pragma unroll
                for (int v = 0; v < CV; ++v) s[be][v] = first ? cf * acc[be][v] : s[be][v] + cf * acc[be][v];
        };
        // FP32 vectors: SUM flips (or the last few) are summed in s, then added to z; FP16 vectors: those of a step;
        // FP64, whose operations bind, adds to z at once
        constexpr bool kApart = sizeof(ST) == 4, kStep = sizeof(ST) == 2;
        VT s[D][CV];
        VT(&sum)[D][CV] = kApart || kStep ? s : z;
        auto add_sum = [&]() {
#pragma unroll
            for (int g = 0; g < D; ++g)
#pragma unroll
                for (int v = 0; v < CV; ++v) {
                    z[g][v] += s[g][v];
                    s[g][v] = (VT)0;
                }
        };
#pragma unroll
        for (int g = 0; g < D; ++g)
#pragma unroll
            for (int v = 0; v < CV; ++v) s[g][v] = (VT)0;
        const uint2 *ent = reinterpret_cast<const uint2 *>(P.ent);
        uint64_t e = e0;
        auto step = [&](auto N) {  // N gathers in flight
            constexpr int n = decltype(N)::value;
            uint2 r[n];
            VT u[n][D][CV];
#pragma unroll
            for (int q = 0; q < n; ++q) r[q] = __ldg(ent + e + q);
#pragma unroll
            for (int q = 0; q < n; ++q) gather(r[q].x, u[q]);
#pragma unroll
            for (int q = 0; q < n; ++q) contract(r[q], coef(r[q]), u[q], sum, kStep && q == 0);
            if (kStep) add_sum();
            e += n;
        };
        while (e + SUM <= e1) {
#pragma unroll
            for (int h = 0; h < SUM; h += FL) step(std::integral_constant<int, FL>{});
            if (kApart) add_sum();
        }
        if (FL == 2 && SUM == 4 && e + 2 <= e1) step(std::integral_constant<int, 2>{});
        while (e < e1) step(std::integral_constant<int, 1>{});
        if (kApart) add_sum();
        VT xo[D][CV];
        gather(at, xo);
#pragma unroll
        for (int v = 0; v < CV; ++v) {
            VT val[D];
            if (sid == 0) {
#pragma unroll
                for (int g = 0; g < D; ++g) val[g] = sizeof(VT) == 8 ? z[g][v] * zscale : z[g][v];
            } else {  // projector onto the range of V(r), and 1/sqrt|Stab r|
                const VT inv_sq = zscale * __ldg(P.sqrtS + P.n_sid + sid);
                const VT *Pr = P.Pj[0] + (size_t)sid * D * D;
#pragma unroll
                for (int g = 0; g < D; ++g) {
                    VT w = (VT)0;
#pragma unroll
                    for (int be = 0; be < D; ++be) w += __ldg(Pr + g * D + be) * z[be][v];
                    val[g] = w * inv_sq;
                }
            }
#pragma unroll
            for (int g = 0; g < D; ++g) z[g][v] = val[g] + diag * xo[g][v];
        }
#pragma unroll
        for (int g = 0; g < D; ++g) {
            alignas(16) ST ys[CV];
#pragma unroll
            for (int v = 0; v < CV; ++v) {
                ys[v] = st_put<VT, ST>(z[g][v]);
                if (want_dot) dacc[v].add(xo[g][v], st_get<VT, ST>(ys[v]));
            }
            if (CV * sizeof(ST) == 16 && vec && (reinterpret_cast<uintptr_t>(y) & 15) == 0) {
                *reinterpret_cast<uint4 *>(y + seg + (size_t)g * B) = *reinterpret_cast<const uint4 *>(ys);
            } else {
#pragma unroll
                for (int v = 0; v < CV; ++v) y[seg + (size_t)g * B + v] = ys[v];
            }
        }
    }
    if (want_dot && cur_part >= 0) flush(cur_part);
    if (a.flips) {
        for (int o = 16; o; o >>= 1) n_flips += __shfl_xor_sync(kFullMask, n_flips, o);
        if (lane == 0 && n_flips) atomicAdd(a.flips, n_flips);
    }
}

template <typename VT, typename ST, int D>
size_t hvp_lane_smem(const HvpArgs<VT> &a) {
    return (((size_t)a.rho_total * sizeof(VT) + 15) & ~(size_t)15) + (size_t)2 * a.n_bonds + 16;
}

// CV for the plan's B (FP64: one right-hand side only), PB with a padded copy
template <typename VT, typename ST, int D, class F>
auto lane_dispatch(const HvpArgs<VT> &a, F f) {
    using std::false_type;
    using std::true_type;
    constexpr int PB = lane_pad_bytes<ST, D>();
    if constexpr (sizeof(VT) == 4) {
        constexpr int most = lane_most_cols<VT, ST, D>();
        const int cols = lane_cols(a.B, most);
        if constexpr (most == 4)
            if (a.B > 1 && cols == 4)
                return f(std::integral_constant<int, 4>{}, false_type{}, std::integral_constant<int, 0>{});
        if (a.B > 1 && cols == 2)
            return f(std::integral_constant<int, 2>{}, false_type{}, std::integral_constant<int, 0>{});
        if (a.B > 1) return f(std::integral_constant<int, 1>{}, false_type{}, std::integral_constant<int, 0>{});
    }
    if (PB > 0 && a.pad_n) return f(std::integral_constant<int, 1>{}, true_type{}, std::integral_constant<int, PB>{});
    return f(std::integral_constant<int, 1>{}, true_type{}, std::integral_constant<int, 0>{});
}

template <typename VT, typename ST, int D>
int hvp_lane_occupancy_t(const HvpArgs<VT> &a, int warps, int) {
    if (warps * 32 != kLaneThreads) return 0;
    return lane_dispatch<VT, ST, D>(a, [&](auto CV, auto ONE, auto PB) {
        return hvp_fit_occupancy<
            hvp_lane_kernel<VT, ST, D, decltype(CV)::value, decltype(ONE)::value, decltype(PB)::value>>(
            warps, hvp_lane_smem<VT, ST, D>(a));
    });
}

template <typename VT, typename ST, int D>
ftlm_status hvp_lane_launch_t(HvpArgs<VT> a, const HvpGeom &geo, cudaStream_t stream) {
    constexpr int PB = lane_pad_bytes<ST, D>();
    if constexpr (PB > 0) {
        if (a.pad_n) {
            lane_pad_kernel<ST, D, PB><<<(unsigned)((a.pad_n + 255) / 256), 256, 0, stream>>>(
                static_cast<const ST *>(a.pad_x), a.pad_n, a.pad_out);
            count_launch();
            FTLM_CUDA(cudaGetLastError());
        }
    }
    if (hvp_lane_smem<VT, ST, D>(a) > 48 * 1024 && hvp_lane_occupancy_t<VT, ST, D>(a, kLaneThreads / 32, 1) < 1)
        return fail(FTLM_EUNSUPPORTED, "rho table does not fit in shared memory");  // raises the padded kernel's limit
    count_launch();
    const cudaError_t e = lane_dispatch<VT, ST, D>(a, [&](auto CV, auto ONE, auto PBC) {
        return launch_overlapped(
            a.overlap, hvp_lane_kernel<VT, ST, D, decltype(CV)::value, decltype(ONE)::value, decltype(PBC)::value>,
            (unsigned)geo.grid, kLaneThreads, hvp_lane_smem<VT, ST, D>(a), stream, a);
    });
    FTLM_CUDA(e);
    return FTLM_OK;
}

}  // namespace ftlm
