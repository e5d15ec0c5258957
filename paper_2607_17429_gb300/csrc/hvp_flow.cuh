// Table-mode H·v of the multi-block shapes with FP32 arithmetic (Eqs. 15-16 in the pull form, flips
// read from an entry table): one warp per output representative, as in hvp.cuh, with the work laid out
// for few instructions and few shared-memory wavefronts per flip.
//
// What bound the kernel of hvp.cuh on the ten irreps of I_h at B = 8 (icosidodecahedron, M = 0, 9.2 ms):
// 164 warp instructions and 50 shared-memory wavefronts per flip, with one group of four gathers in
// flight per warp.  Here:
//  - a lane takes two neighbouring right-hand sides (CL = ceil(B / 2) rounded up to a power of two lanes
//    per flip, Q = 32 / CL flips at a time), so a rho element serves two columns and eight flips' rho
//    rows share a wavefront (a 16-byte shared load costs two wavefronts for up to sixteen addresses
//    when lane pairs agree, an 8-byte load one);
//  - rho(g) of all blocks is one record (stride 4 mod 8 words: records start in different banks), so a
//    flip needs one base address; pairs of rows go through fma.rn.f32x2.  A flip's products are summed before
//    they meet the accumulators, which keeps the rounding of the kernel of hvp.cuh; but where 64 accumulators fill
//    the registers (W = 32) blocks of dimension 1 to 3 scale the gathered values and add every product to them
//    (icosidodecahedron at B = 8: error 6.6e-8 in hvp.cuh, 6.9e-8 with every product added in 5.86 ms, 6.4e-8 so in
//    5.78, 6.2e-8 with every block's sums first in 6.41);
//  - entries stay in registers (lane j holds flips j and 32 + j) and reach the others by shuffles;
//  - the record, the entry offsets and the entries of the next representative are loaded while the
//    present one is worked on, and its first gathers are issued as soon as the last of this one's are,
//    so the copies never drain between representatives;
//  - the flip groups' sums are combined by a reduce-scatter (each step halves the rows a lane keeps),
//    which leaves every lane R = ceil(W / Q) rows of its two columns to finish.
// Icosidodecahedron, M = 0, ten irreps, FP32: B = 8 9.16 -> 5.8 ms, B = 16 16.7 -> 9.9, B = 24 29.9 -> 16.9 (with
// the contraction left out 4.5, 9.6 and 16.2 ms: at B = 24 the 25 GB of gathers that miss L2 bind, at
// B = 8 gathers and contraction take 4.5 and 4.4 ms and overlap in part).
//
// x and y start on a pair of elements (own rows and outputs move as pairs); hvp_plan takes the kernel of hvp.cuh otherwise.
#pragma once

#include "hvp.cuh"

namespace ftlm {

// rho record of a shape: offset of block k, elements, stride between group elements
__host__ __device__ constexpr int flow_block_elems(int D) { return D == 1 ? 1 : D == 2 ? 4 : D == 3 ? 12 : D == 4 ? 16 : 28; }
template <class SH, int k>
struct FlowOff {
    static constexpr int prev = FlowOff<SH, k - 1>::value + flow_block_elems(SH::template D<k - 1>);
    static constexpr int value = k < SH::K && SH::template D<(k < SH::K ? k : 0)> == 1 ? prev : (prev + 3) / 4 * 4;
};
template <class SH>
struct FlowOff<SH, 0> {
    static constexpr int value = 0;
};
template <class SH>
__host__ __device__ constexpr int flow_stride() {
    constexpr int n = (FlowOff<SH, SH::K>::value + 3) / 4;
    return 4 * (n % 2 ? n : n + 1);
}
// accumulators: pairs of rows, then the odd rows; first pair and first odd row of block k
template <class SH, int k>
struct FlowPair {
    static constexpr int value = FlowPair<SH, k - 1>::value + SH::template D<k - 1> / 2;
};
template <class SH>
struct FlowPair<SH, 0> {
    static constexpr int value = 0;
};

template <typename ST, class SH, int CL>
__host__ __device__ constexpr int flow_threads() {
    // W = 32: 64 accumulators and the loads in flight want 255 registers; eight such warps with two
    // staging buffers each beat sixteen that spill (I_h, FP32, B = 8: 5.9 ms against 6.8).  FP16 segments
    // leave room for two buffers at sixteen warps, which hide the conversions better (6.1 against 6.4 ms).
    // CL = 16 ends with W / 2 rows per lane.
    return SH::W > 20 ? (sizeof(ST) == 2 ? 512 : 256) : CL == 16 ? 384 : 512;
}

struct FlowLayout {
    size_t o_bond, o_red, o_bar, o_stage, per_warp, total;
};
__host__ __device__ inline FlowLayout flow_layout(int G, int stride, int n_bonds, int K, int B, int warps, int nbuf,
                                                  size_t stage_bytes) {
    FlowLayout L;
    size_t o = (size_t)G * stride * 4;
    L.o_bond = o;
    o = (o + 2 * (size_t)n_bonds + 15) & ~(size_t)15;
    L.o_red = o;
    o += (size_t)K * B * 8;
    o = (o + 15) & ~(size_t)15;
    L.o_bar = o;
    o += (size_t)warps * 8 * kMaxBuf;
    o = (o + 127) & ~(size_t)127;
    L.o_stage = o;
    L.per_warp = ((size_t)nbuf * stage_bytes + 127) & ~(size_t)127;
    L.total = o + (size_t)warps * L.per_warp;
    return L;
}

// two neighbouring stored elements as floats, and back
template <typename ST>
__device__ __forceinline__ float2 flow_load2(const ST *p) {
    if constexpr (std::is_same<ST, __half>::value)
        return __half22float2(*reinterpret_cast<const __half2 *>(p));
    else
        return *reinterpret_cast<const float2 *>(p);
}

// pair q of rows of both columns: a rho pair times the gathered row
template <int N>
__device__ __forceinline__ void flow_acc(unsigned long long (&ap)[2][N], int q, bool first, unsigned long long rr, float2 xv) {
    const unsigned long long u0 = f2_pack(xv.x, xv.x), u1 = f2_pack(xv.y, xv.y);
    ap[0][q] = first ? f2_mul(rr, u0) : f2_fma(rr, u0, ap[0][q]);
    ap[1][q] = first ? f2_mul(rr, u1) : f2_fma(rr, u1, ap[1][q]);
}

// N rows per column held by every lane -> N / 2 after the exchange with the lane M groups of CL away
template <int CL, int N, int M>
__device__ __forceinline__ void flow_reduce(float *z0, float *z1, int f) {
    if constexpr (M >= 1) {
        const bool up = (f & M) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const float s0 = up ? z0[i] : z0[i + N / 2], s1 = up ? z1[i] : z1[i + N / 2];
            const float k0 = up ? z0[i + N / 2] : z0[i], k1 = up ? z1[i + N / 2] : z1[i];
            z0[i] = k0 + __shfl_xor_sync(kFullMask, s0, M * CL);
            z1[i] = k1 + __shfl_xor_sync(kFullMask, s1, M * CL);
        }
        flow_reduce<CL, N / 2, M / 2>(z0, z1, f);
    }
}

// BC: the number of right-hand sides when it is a compile-time constant, else 0
template <typename ST, class SH, int CL, int BC>
__global__ void __launch_bounds__(flow_threads<ST, SH, CL>(), 1) hvp_flow_kernel(const __grid_constant__ HvpArgs<float> a) {
    constexpr int K = SH::K, W = SH::W, Q = 32 / CL, R = (W + Q - 1) / Q;
    constexpr int S = flow_stride<SH>();
    constexpr int NP = FlowPair<SH, K>::value, NS = W - 2 * NP;  // row pairs and odd rows
    extern __shared__ __align__(128) uint8_t smem[];
    const int B = BC ? BC : a.B;
    const int warps = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cq = lane & (CL - 1), f = lane / CL;
    const bool col = 2 * cq < B;
    const int nbuf = a.nbuf;
    const size_t stage_bytes = (size_t)a.stage_elems * sizeof(ST);
    const FlowLayout L = flow_layout(a.G, S, a.n_bonds, K, B, warps, nbuf, stage_bytes);
    let_next_start();
    float *s_rho = reinterpret_cast<float *>(smem);
    uint8_t *s_bond = smem + L.o_bond;
    double *red = reinterpret_cast<double *>(smem + L.o_red);
    static_for<K>([&](auto kc) {
        constexpr int k = decltype(kc)::value, D = SH::template D<k>, RP = rho_row(D);
        constexpr int P = D == 2 ? 2 : 4;
        float *dst = s_rho + FlowOff<SH, k>::value;
        const float *src = a.rhoT + a.rho_off[k];
        for (int i = threadIdx.x; i < a.G * D * D; i += blockDim.x) {
            const int g = i / (D * D), ga = i / D % D, be = i % D;
            dst[g * S + (D == 1 ? 0 : be < 4 ? ga * P + be : 20 + ga)] = src[(g * D + ga) * RP + be];
        }
    });
    for (int i = threadIdx.x; i < 2 * a.n_bonds; i += blockDim.x) s_bond[i] = a.bonds[i];
    for (int i = threadIdx.x; i < K * B; i += blockDim.x) red[i] = 0.0;
    if (lane < kMaxBuf) mbar_init(smem_u32(smem + L.o_bar + 8 * (kMaxBuf * wid + lane)), 1);
    fence_mbar_init();
    fence_proxy_async_smem();
    __syncthreads();
    const uint32_t bar0 = smem_u32(smem + L.o_bar + 8 * kMaxBuf * wid);
    ST *stage = reinterpret_cast<ST *>(smem + L.o_stage + (size_t)wid * L.per_warp);
    const uint32_t stage_s = smem_u32(stage);
    const float halfJ = a.J * 0.5f;
    const bool want_dot = a.dot_part != nullptr;
    uint32_t parity = 0, pending = 0;  // bit i: phase parity of buffer i; copies in flight into it
    int head = 0, tail = 0;            // buffer to consume next, to fill next
    bool dead = false;                 // a wait ran out: no more work for this warp
    DotAcc32 dacc[R][2];
#pragma unroll
    for (int i = 0; i < R; ++i) dacc[i][0].zero(), dacc[i][1].zero();
    unsigned long long n_flips = 0;
    int cur_part = -1;

    // CTA-wide flush of the per-lane dot accumulators into the partials of part pt
    auto flush = [&](int pt) {
        static_for<K>([&](auto kc) {
            constexpr int k = decltype(kc)::value, Zk = SH::template Z<k>, D = SH::template D<k>;
            double v0 = 0.0, v1 = 0.0;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int r = f * R + i;
                if (r >= Zk && r < Zk + D) {
                    v0 += dacc[i][0].value();
                    v1 += dacc[i][1].value();
                }
            }
            for (int w = CL; w < 32; w <<= 1) {
                v0 += __shfl_xor_sync(kFullMask, v0, w);
                v1 += __shfl_xor_sync(kFullMask, v1, w);
            }
            for (int w = 0; w < warps; ++w) {  // fixed order over warps: deterministic sums
                __syncthreads();
                if (wid == w && f == 0 && col) {
                    red[k * B + 2 * cq] += v0;
                    red[k * B + 2 * cq + 1] += v1;
                }
            }
        });
        __syncthreads();
        double *dst = a.dot_part + ((size_t)pt * gridDim.x + blockIdx.x) * K * B;
        for (int i = threadIdx.x; i < K * B; i += blockDim.x) {
            dst[i] = red[i];
            red[i] = 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < R; ++i) dacc[i][0].zero(), dacc[i][1].zero();
    };

    for (uint64_t t = blockIdx.x + prior_done(); t < a.n_tiles;) {
        int p = 0;
        if (a.n_parts > 1) {  // last part whose first tile is <= t
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
        const HvpPart<float> &P = a.n_parts == 1 ? a.part0 : a.parts[p];
        if (want_dot && p != cur_part) {
            if (cur_part >= 0) flush(cur_part);
            cur_part = p;
        }
        const uint64_t n_reps = P.n_reps;
        const int tile_reps = P.tile_reps;
        const uint64_t tl = t - P.tile0, part_tiles = (n_reps + tile_reps - 1) / tile_reps;
        const unsigned n_tile = (unsigned)((part_tiles - tl + gridDim.x - 1) / gridDim.x);  // this CTA's, in the part
        const unsigned sub = (unsigned)((tile_reps + warps - 1) / warps);                   // per tile and warp
        t += (uint64_t)n_tile * gridDim.x;
        if (dead) continue;
        const HvRec *__restrict__ rec = P.rec + P.rep0;
        const HvEntry *ent = P.ent;
        const float *sqrtS = P.sqrtS;
        const ST *__restrict__ x = static_cast<const ST *>(P.x);
        ST *__restrict__ y = static_cast<ST *>(P.y);

        struct Rep {  // one representative's record and its first 64 entries (lane j: flips j and 32 + j)
            uint64_t label, e0;
            uint32_t idx, sid;
            int nf, state;  // state: 0 none, 1 work, 2 no block has rows (y~ = 0)
            uint2 ea, eb;
        };
        unsigned tt = 0;                                  // the next record to load: tile of this CTA,
        int local = wid;                                  // place in the tile,
        uint64_t base = tl * (uint64_t)tile_reps;         // first representative of the tile
        auto load_rec = [&](Rep &q) {
            const uint64_t rep = base + (unsigned)local;
            q.state = tt < n_tile && local < tile_reps && rep < n_reps ? 1 : 0;
            local += warps;
            if (local >= (int)sub * warps) {
                local = wid;
                ++tt;
                base += (uint64_t)gridDim.x * (uint64_t)tile_reps;
            }
            q.nf = 0;
            q.label = q.e0 = 0;
            q.idx = q.sid = 0;
            if (!q.state) return;
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(rec + rep));
            q.label = ((uint64_t)v.y << 32) | v.x;
            q.idx = v.z;
            q.sid = v.w;
            if (P.ecnt) {
                q.e0 = rep * (uint64_t)P.estride;
                q.nf = __ldg(P.ecnt + rep);
            } else {
                q.e0 = __ldg(P.eoff + P.rep0 + rep);
                q.nf = (int)(__ldg(P.eoff + P.rep0 + rep + 1) - q.e0);
            }
        };
        auto load_ent = [&](Rep &q) {
            if (q.state == 1 && q.sid != 0 && __ldg(P.wtab + q.sid) == 0) {
                q.state = 2;
                q.nf = 0;
            }
            q.ea = q.eb = make_uint2(0u, 0u);
            if (lane < q.nf) q.ea = __ldg(reinterpret_cast<const uint2 *>(ent + q.e0 + lane));
            if (lane + 32 < q.nf) q.eb = __ldg(reinterpret_cast<const uint2 *>(ent + q.e0 + 32 + lane));
        };
        // c_a sqrt|Stab r'| of an entry
        auto coef = [&](uint64_t lab, uint2 e) {
            const uint32_t es = (e.y >> 8) & 255u, sidf = e.y >> 16;
            float c = halfJ;
            if (a.two_s != 1) {
                const int b = (int)(es & 127u);
                const int ai = (int)hvp_digit(lab, s_bond[2 * b], a.bits);
                const int aj = (int)hvp_digit(lab, s_bond[2 * b + 1], a.bits);
                c = halfJ * ((es & 128u) == 0 ? a.up[ai] * a.dn[aj] : a.dn[ai] * a.up[aj]);
            }
            return sidf ? c * __ldg(sqrtS + sidf) : c;
        };
        // gathers of flip group gi (Q flips) of q into the next buffer
        auto fill = [&](const Rep &q, int gi) {
            const int j0 = gi * Q;
            const uint32_t held = j0 < 32 ? q.ea.x : q.eb.x;
            if (a.tma) {
                const int j = j0 + lane;
                uint32_t tgt = __shfl_sync(kFullMask, held, (j0 + (lane & (Q - 1))) & 31);
                const bool mine = lane < Q && j < q.nf;
                if (j0 >= 64 && mine) tgt = __ldg(reinterpret_cast<const uint2 *>(ent + q.e0 + j)).x;
                const uint32_t bytes = (uint32_t)(W * B * (int)sizeof(ST));
                const uint32_t bar = bar0 + 8 * tail;
                fence_proxy_async_smem();  // earlier generic reads of the buffer before the async writes
                __syncwarp();
                if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)min(Q, q.nf - j0) * bytes);
                __syncwarp();
                if (mine)
                    bulk_copy_g2s(stage_s + (uint32_t)(tail * stage_bytes) + (uint32_t)(lane * a.slot_elems * (int)sizeof(ST)),
                                  x + (size_t)tgt * W * B, bytes, bar);
            } else {
                const int j = j0 + f;
                uint32_t tgt = __shfl_sync(kFullMask, held, j & 31);
                if (j0 >= 64 && j < q.nf) tgt = __ldg(reinterpret_cast<const uint2 *>(ent + q.e0 + j)).x;
                if (j < q.nf && col) {
                    const ST *src = x + (size_t)tgt * W * B + 2 * cq;
                    ST *dst = stage + (size_t)tail * a.stage_elems + (size_t)f * a.slot_elems + 2 * cq;
                    for (int r = 0; r < W; ++r) {
                        dst[r * B] = __ldg(src + r * B);
                        dst[r * B + 1] = __ldg(src + r * B + 1);
                    }
                }
                __syncwarp();
            }
            pending |= 1u << tail;
            tail = tail + 1 == nbuf ? 0 : tail + 1;
        };

        Rep cur, nxt;
        load_rec(cur);
        load_ent(cur);
        int filled = 0;  // groups of cur whose gathers are issued
        const unsigned n_it = n_tile * sub;
        for (unsigned it = 0; it < n_it && !dead; ++it) {
            load_rec(nxt);
            nxt.ea = nxt.eb = make_uint2(0u, 0u);
            const int ng = (cur.nf + Q - 1) / Q;
            const size_t seg = (size_t)cur.idx * W * B;
            int filled_n = 0;
            n_flips += (unsigned long long)cur.nf;
            const float cfa = coef(cur.label, cur.ea), cfb = coef(cur.label, cur.eb);
            if (cur.state) {  // the own rows are read in the epilogue: start bringing them into L2 now
                const uint32_t bytes = (uint32_t)(W * B * (int)sizeof(ST));
                const char *src = reinterpret_cast<const char *>(x + seg);
                for (uint32_t o = (uint32_t)lane * 128u; o < bytes; o += 32u * 128u) prefetch_l2(src + o);
                if (lane == 31) prefetch_l2(src + bytes - 1);
            }
            unsigned long long zp[2][NP > 0 ? NP : 1];
            float zs[2][NS > 0 ? NS : 1];
#pragma unroll
            for (int i = 0; i < NP; ++i) zp[0][i] = zp[1][i] = 0ull;
#pragma unroll
            for (int i = 0; i < NS; ++i) zs[0][i] = zs[1][i] = 0.f;
            while (filled < ng && filled < nbuf) fill(cur, filled++);
            for (int gi = 0; gi < ng; ++gi) {
                if (a.tma) {
                    if (!mbar_wait_bounded(bar0 + 8 * head, (parity >> head) & 1u, a.wait_limit)) {
                        dead = true;
                        break;
                    }
                    parity ^= 1u << head;
                }
                pending &= ~(1u << head);
                const int j = gi * Q + f;
                const bool hi = gi * Q >= 32;
                float cf = __shfl_sync(kFullMask, hi ? cfb : cfa, j & 31);
                uint32_t g8 = __shfl_sync(kFullMask, (hi ? cur.eb.y : cur.ea.y) & 255u, j & 31);
                if (gi * Q >= 64 && j < cur.nf) {
                    const uint2 e = __ldg(reinterpret_cast<const uint2 *>(ent + cur.e0 + j));
                    cf = coef(cur.label, e);
                    g8 = e.y & 255u;
                }
                if (j < cur.nf && col) {
                    const uint32_t negw = (g8 & 128u) ? a.neg : 0u;  // (g*, 1) in a Gamma- block: -rho(g*)
                    const float *rb = s_rho + (g8 & 127u) * S;
                    const ST *xs = stage + (size_t)head * a.stage_elems + (size_t)f * a.slot_elems + 2 * cq;
                    static_for<K>([&](auto kc) {
                        constexpr int k = decltype(kc)::value, D = SH::template D<k>, Zk = SH::template Z<k>;
                        constexpr int PB = FlowPair<SH, k>::value, SB = Zk - 2 * PB;
                        const float *Rk = rb + FlowOff<SH, k>::value;
                        const float ck = __uint_as_float(__float_as_uint(cf) ^ ((negw << (31 - k)) & 0x80000000u));
                        float odd5[5];
                        if constexpr (D == 5) {
                            const float4 v = *reinterpret_cast<const float4 *>(Rk + 20);
                            odd5[0] = v.x, odd5[1] = v.y, odd5[2] = v.z, odd5[3] = v.w, odd5[4] = Rk[24];
                        }
                        if constexpr (D >= 4 || W <= 20) {  // the flip's sums first (first product a multiply), one addition to z
                            unsigned long long ap[2][D >= 2 ? D / 2 : 1];
                            float as[2];
#pragma unroll
                            for (int ga = 0; ga < D; ++ga) {
                                const float2 xv = flow_load2<ST>(xs + (Zk + ga) * B);
                                float ro = Rk[0];  // rho of the odd row
                                if constexpr (D == 2) {
                                    flow_acc(ap, 0, ga == 0, *reinterpret_cast<const unsigned long long *>(Rk + 2 * ga), xv);
                                } else if constexpr (D > 2) {
                                    const ulonglong2 rr = *reinterpret_cast<const ulonglong2 *>(Rk + 4 * ga);
                                    flow_acc(ap, 0, ga == 0, rr.x, xv);
                                    if constexpr (D >= 4) flow_acc(ap, 1, ga == 0, rr.y, xv);
                                    float pad;
                                    if constexpr (D == 3) f2_unpack(rr.y, ro, pad);
                                    if constexpr (D == 5) ro = odd5[ga];
                                }
                                if constexpr (D % 2) {
                                    as[0] = ga == 0 ? ro * xv.x : fmaf(ro, xv.x, as[0]);
                                    as[1] = ga == 0 ? ro * xv.y : fmaf(ro, xv.y, as[1]);
                                }
                            }
                            const unsigned long long cc = f2_pack(ck, ck);
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
#pragma unroll
                                for (int q = 0; q < D / 2; ++q) zp[c][PB + q] = f2_fma(cc, ap[c][q], zp[c][PB + q]);
                                if constexpr (D % 2) zs[c][SB] = fmaf(ck, as[c], zs[c][SB]);
                            }
                        } else {  // every product straight into z
#pragma unroll
                            for (int ga = 0; ga < D; ++ga) {
                                const float2 xv = flow_load2<ST>(xs + (Zk + ga) * B);
                                const float u0 = xv.x * ck, u1 = xv.y * ck;
                                float ro = Rk[0];
                                if constexpr (D > 1) {
                                    const unsigned long long uu0 = f2_pack(u0, u0), uu1 = f2_pack(u1, u1);
                                    unsigned long long rr;
                                    if constexpr (D == 2) {
                                        rr = *reinterpret_cast<const unsigned long long *>(Rk + 2 * ga);
                                    } else {
                                        const ulonglong2 r4 = *reinterpret_cast<const ulonglong2 *>(Rk + 4 * ga);
                                        float pad;
                                        rr = r4.x;
                                        f2_unpack(r4.y, ro, pad);
                                    }
                                    zp[0][PB] = f2_fma(rr, uu0, zp[0][PB]);
                                    zp[1][PB] = f2_fma(rr, uu1, zp[1][PB]);
                                }
                                if constexpr (D % 2) {
                                    zs[0][SB] = fmaf(ro, u0, zs[0][SB]);
                                    zs[1][SB] = fmaf(ro, u1, zs[1][SB]);
                                }
                            }
                        }
                    });
                }
                __syncwarp();
                head = head + 1 == nbuf ? 0 : head + 1;
                if (gi == 0) load_ent(nxt);
                if (filled < ng)
                    fill(cur, filled++);
                else if (filled_n * Q < nxt.nf && filled_n < nbuf)
                    fill(nxt, filled_n++);
            }
            if (dead) break;
            if (ng == 0) load_ent(nxt);
            if (cur.state == 1) {
                // rows in packed order, padded to a multiple of Q, then the reduce-scatter
                float z[2][R * Q];
                static_for<K>([&](auto kc) {
                    constexpr int k = decltype(kc)::value, D = SH::template D<k>, Zk = SH::template Z<k>;
                    constexpr int PB = FlowPair<SH, k>::value, SB = Zk - 2 * PB;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
#pragma unroll
                        for (int q = 0; q < D / 2; ++q) f2_unpack(zp[c][PB + q], z[c][Zk + 2 * q], z[c][Zk + 2 * q + 1]);
                        if constexpr (D % 2) z[c][Zk + D - 1] = zs[c][SB];
                    }
                });
#pragma unroll
                for (int i = W; i < R * Q; ++i) z[0][i] = z[1][i] = 0.f;
                float diag;
                if (a.two_s == 1) {  // every bond is +1/4 or, when it flips, -1/4
                    diag = a.J * (float)(a.n_bonds - 2 * cur.nf) * 0.25f;
                } else {
                    int d4 = 0;
                    for (int e = lane; e < a.n_bonds; e += 32)
                        d4 += (2 * (int)hvp_digit(cur.label, s_bond[2 * e], a.bits) - a.two_s) *
                              (2 * (int)hvp_digit(cur.label, s_bond[2 * e + 1], a.bits) - a.two_s);
                    diag = a.J * (float)__reduce_add_sync(kFullMask, d4) * 0.25f;
                }
                float2 xo[R];  // the own rows arrive during the exchange
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    xo[i] = make_float2(0.f, 0.f);
                    if (f * R + i < W && col) xo[i] = flow_load2<ST>(x + seg + (size_t)(f * R + i) * B + 2 * cq);
                }
                flow_reduce<CL, R * Q, Q / 2>(z[0], z[1], f);
                if (cur.sid != 0) {  // projector onto the range of V_k(r) and 1 / sqrt|Stab r|
                    const float inv = 1.f / __ldg(sqrtS + cur.sid);
                    float v[2][R];
#pragma unroll
                    for (int i = 0; i < R; ++i) v[0][i] = v[1][i] = 0.f;
                    static_for<K>([&](auto kc) {
                        constexpr int k = decltype(kc)::value, D = SH::template D<k>, Zk = SH::template Z<k>;
                        const float *Pr = P.Pj[k] + (size_t)cur.sid * D * D;
#pragma unroll
                        for (int be = 0; be < D; ++be) {
                            const int row = Zk + be;
                            const float s0 = __shfl_sync(kFullMask, z[0][row % R], row / R * CL + cq);
                            const float s1 = __shfl_sync(kFullMask, z[1][row % R], row / R * CL + cq);
#pragma unroll
                            for (int i = 0; i < R; ++i) {
                                const int gam = f * R + i - Zk;
                                if (gam >= 0 && gam < D) {
                                    const float w = __ldg(Pr + gam * D + be);
                                    v[0][i] += w * s0;
                                    v[1][i] += w * s1;
                                }
                            }
                        }
                    });
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        z[0][i] = v[0][i] * inv;
                        z[1][i] = v[1][i] * inv;
                    }
                }
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    if (f * R + i < W && col) {
                        ST *dst = y + seg + (size_t)(f * R + i) * B + 2 * cq;
                        const float y0 = z[0][i] + diag * xo[i].x, y1 = z[1][i] + diag * xo[i].y;
                        float2 ys;  // the values as stored
                        if constexpr (std::is_same<ST, __half>::value) {
                            const __half2 h = __floats2half2_rn(y0, y1);
                            *reinterpret_cast<__half2 *>(dst) = h;
                            ys = __half22float2(h);
                        } else {
                            ys = make_float2(y0, y1);
                            *reinterpret_cast<float2 *>(dst) = ys;
                        }
                        if (want_dot) {
                            dacc[i][0].add(xo[i].x, ys.x);
                            dacc[i][1].add(xo[i].y, ys.y);
                        }
                    }
                }
            } else if (cur.state == 2) {
                for (int e = lane; e < W * B; e += 32) y[seg + e] = st_put<float, ST>(0.f);
            }
            cur = nxt;
            filled = filled_n;
        }
        if (dead) {  // a wait ran out: record it, let the copies in flight land, only take part in the flushes
            if (lane == 0) atomicOr(a.err, kErrWaitTimeout);
            for (int bi = 0; bi < kMaxBuf; ++bi)
                if (a.tma && ((pending >> bi) & 1u)) mbar_wait_bounded(bar0 + 8 * bi, (parity >> bi) & 1u, kDrainCycles);
            pending = 0;
        }
    }
    if (want_dot && cur_part >= 0) flush(cur_part);
    if (a.flips && lane == 0 && n_flips) atomicAdd(a.flips, n_flips);
}

// ---------------------------------------------------------------- host side

template <typename ST, class SH, int CL, int BC>
size_t flow_smem(const HvpArgs<float> &a, int warps, int nbuf) {
    return flow_layout(a.G, flow_stride<SH>(), a.n_bonds, SH::K, a.B, warps, nbuf, (size_t)a.stage_elems * sizeof(ST)).total;
}

template <typename ST, class SH, int CL, int BC>
int hvp_flow_occupancy_t(const HvpArgs<float> &a, int warps, int nbuf) {
    if (warps * 32 > flow_threads<ST, SH, CL>()) return 0;
    return hvp_fit_occupancy<hvp_flow_kernel<ST, SH, CL, BC>>(warps, flow_smem<ST, SH, CL, BC>(a, warps, nbuf));
}

template <typename ST, class SH, int CL, int BC>
ftlm_status hvp_flow_launch_t(HvpArgs<float> a, const HvpGeom &geo, cudaStream_t stream) {
    a.nbuf = geo.nbuf;
    a.tma = geo.tma;
    count_launch();
    FTLM_CUDA(launch_overlapped(a.overlap, hvp_flow_kernel<ST, SH, CL, BC>, (unsigned)geo.grid, geo.warps * 32,
                                flow_smem<ST, SH, CL, BC>(a, geo.warps, geo.nbuf), stream, a));
    return FTLM_OK;
}

}  // namespace ftlm
