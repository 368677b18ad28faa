// qcs_walk.cu -- the walk step, distinguished-point table and re-walk kernels
// of the deterministic-walk T-count search (Di Matteo & Mosca, Sec. 2-3),
// hand-written for sm_103a.
//
// A group of lanes (a warp, or 16 / 4^n lanes for n <= 3) evaluates one step
// f = h o nu o mu of one walk (Sec. 2, Fig. 1):
//   mu : decode the state into a side b and rotations q_1..q_h (Sec. 3, z_b);
//   nu : the exact product V = R^(q_h)..R^(q_1) or W = R^(q_1)^T..R^(q_h)^T
//        [R^(c)^T] C^ over Z[1/sqrt2] (Eq. mitm in channel form), taken modulo
//        right multiplication by Cliffords (Eq. tcount_synthesis);
//   h  : a coset-invariant hash back to an L-bit state.
//
// The hash is defined on the exact product M at exponent K: every column Q
// gets the 16-bit linear fingerprint L_Q = sum_i Ua[i] a_iQ + Ub[i] b_iQ mod
// 2^16, folded to phi_Q = min(L_Q, -L_Q) (so a column's sign does not matter),
// and the multiset of the phi_Q (Q >= 1) is hashed by summing
// smix(base ^ phi_Q), so a permutation of the columns does not matter either.
// Because L is linear in M's integer
// numerators and every factor acts linearly on them, L(M e_Q) =
// ((adjoint network) U)^T (M's right factor) e_Q: the kernel pushes the weight
// vector U through the transposed sparse R^ butterflies (4^n entries, h
// stages) instead of pushing all 4^n - 1 columns through them.  The V side is
// then read off directly (its right factor is the identity), and the W side is
// one contraction of the transformed weights with C^, staged in shared memory
// as signed byte quads and contracted by byte-plane dp4a (the n = 4 engine
// of qcs_engine4.cu contracts on the tensor cores instead).  The result is
// bit-identical to hashing the explicitly formed product.
//
// Also here: the distinguished-point table insert and the re-walk of merged
// trails (Sec. 3, Fig. 2), the batched forms of both, the exhaustive level
// pass (Eq. mitm), and the owner binning and insertion of distinguished
// points for a level sharded across ranks.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "qcs_device.cuh"
#include "qcs_internal.h"

namespace qcs {
namespace {

// launch shape of the walk kernels, tuned on GB300 by sweeping warps per CTA,
// lanes per walk, the register cap (minimum resident CTAs) and the
// contraction's unrolling
#ifndef QCS_WARPS
#define QCS_WARPS 8 // warps per CTA, n <= 2
#endif
#ifndef QCS_WARPS3
#define QCS_WARPS3 16 // warps per CTA, n = 3
#endif
#ifndef QCS_LPW3
#define QCS_LPW3 32 // lanes per walk at n = 3 (one walk per warp)
#endif
#ifndef QCS_MIN_BLOCKS3
#define QCS_MIN_BLOCKS3 2 // n = 3: 64 registers, two CTAs of 16 warps (16 walks) per SM
#endif
#ifndef QCS_GEMV_UNROLL
#define QCS_GEMV_UNROLL 2 // 32-bit word contraction (rows per unrolled step / 2)
#endif
#ifndef QCS_QUAD_UNROLL3
#define QCS_QUAD_UNROLL3 16 // byte-quad contraction, n = 3 (16 quads)
#endif
#ifndef QCS_QUAD_UNROLL4
#define QCS_QUAD_UNROLL4 16 // byte-quad contraction, n = 4 (64 quads)
#endif
constexpr int kWarps = QCS_WARPS;
constexpr int kWarps3 = QCS_WARPS3;
constexpr int kGemvUnroll = QCS_GEMV_UNROLL;

// Launch shapes of the walk kernels k_walks and k_walks_batch: warps per CTA
// and the minimum resident CTAs per SM, which caps the registers at 65536 /
// (threads x CTAs).  Shape 0 is the default; the others are chosen at run
// time (qcs_params.launch_shape, qcs_batch_params.launch_shape[n - 1]),
// e.g. by the autotuner.  Every shape evaluates the same walks with the
// same per-walk arithmetic, so the trajectories do not depend on it.
//   n <= 2: 8 warps
//   n = 3 : (16, 2) (8, 4) (32, 1) (16, 1)
//   n = 4 : (16, 1) (24, 1) (32, 1)   (one CTA per SM: C^ takes 128 KB)
//           and shape 3: the tensor-core engine (qcs_engine4.cu; when C^
//           suits it, LevelCtx::Cm; elsewhere shape 3 runs shape 0, whose
//           figures shape_warps gives for it)
__host__ __device__ constexpr int shape_count(int nq) { return nq <= 2 ? 1 : 4; }
__host__ __device__ constexpr int shape_warps(int nq, int s)
{
    return nq <= 2 ? kWarps : nq == 3 ? (s == 1 ? 8 : s == 2 ? 32 : kWarps3) : (s == 1 ? 24 : s == 2 ? 32 : 16);
}
__host__ __device__ constexpr int shape_min_blocks(int nq, int s)
{
    return nq <= 2 ? 1 : nq == 3 ? (s == 1 ? 4 : s >= 2 ? 1 : QCS_MIN_BLOCKS3) : 1;
}

template <int NQ>
struct Geo {
    static constexpr int DIM = 1 << (2 * NQ);            // 4^n rows and columns
    // one walk is evaluated by LPW consecutive lanes of a warp (4^n lanes for
    // n <= 2, QCS_LPW3 at n = 3, the whole warp at n = 4), GROUPS walks per warp
    static constexpr int LPW = DIM < 32 ? DIM : (NQ == 3 ? QCS_LPW3 : 32);
    static constexpr int GROUPS = 32 / LPW;
    static constexpr int RPL = DIM / LPW;                // rows (and columns) per lane
    // n <= 3: C^ staged whole, as byte quads (8 KB at n = 3) or else as low
    // words (32 KB); n = 4: byte quads (128 KB) when every entry fits, else
    // the low words are read through L2
    static constexpr bool C_SMEM = NQ <= 3;
    static constexpr bool CQ_SMEM = NQ == 4;
    static constexpr int WARPS = NQ == 4 ? 16 : NQ == 3 ? kWarps3 : kWarps; // warps per CTA
    static constexpr int THREADS = WARPS * 32;
    static constexpr int WALKS = WARPS * GROUPS;         // walks (lane groups) per CTA
    static constexpr int QUAD_UNROLL = NQ == 4 ? QCS_QUAD_UNROLL4 : QCS_QUAD_UNROLL3;
    static constexpr int COEF_WORDS = DIM * LPW / 2; // rotation masks: a 16-bit word per Pauli and lane
    static constexpr int MAX_CHUNKS = 256;               // hash bases, one per chunk
    // shared memory: weights | C^ | coefficients | chunk bases | exchange buffers
    static constexpr size_t off_C = sizeof(uint2) * DIM;
    static constexpr size_t off_coef =
        off_C + (C_SMEM ? sizeof(uint2) * DIM * DIM : 0) + (CQ_SMEM ? 2 * DIM * DIM : 0);
    static constexpr size_t off_base = off_coef + sizeof(uint32_t) * COEF_WORDS;
    static constexpr size_t off_xchg = off_base + sizeof(uint64_t) * MAX_CHUNKS;
    static constexpr size_t smem_bytes = off_xchg + sizeof(uint2) * WALKS * DIM;
    // the same without C^, for kernels that evaluate V products only:
    // weights | coefficients | chunk bases | exchange buffers
    static constexpr size_t off_coef_v = off_C;
    static constexpr size_t off_base_v = off_coef_v + sizeof(uint32_t) * COEF_WORDS;
    static constexpr size_t off_xchg_v = off_base_v + sizeof(uint64_t) * MAX_CHUNKS;
    static constexpr size_t smem_bytes_v = off_xchg_v + sizeof(uint2) * WALKS * DIM;
};

// One launch shape of the walk kernels (see shape_warps): the CTA's warps,
// its lane groups (walks) and its shared memory, whose exchange buffers
// grow with the walks.
template <int NQ, int S>
struct Shape {
    static constexpr int WARPS = shape_warps(NQ, S);
    static constexpr int THREADS = WARPS * 32;
    static constexpr int WALKS = WARPS * Geo<NQ>::GROUPS;
    static constexpr int MIN_BLOCKS = shape_min_blocks(NQ, S);
    static constexpr size_t smem_bytes = Geo<NQ>::off_xchg + sizeof(uint2) * WALKS * Geo<NQ>::DIM;
};

// Shared-memory views of one CTA (C may point to global memory for n = 4).
template <int NQ>
struct Smem {
    uint2 *U;
    const uint2 *C;
    const uint4 *Cq;  // n >= 3: C^ as byte quads (LevelCtx::Cq layout), or null
    uint32_t *coef;
    uint64_t *base;
    uint2 *xchg; // this lane group's exchange buffer
};

// The lanes evaluating one walk: sub is the lane's index in its group of
// LPW lanes, mask the group's lanes (every shuffle, reduction and warp
// barrier names only the group, so the groups of a warp run independently).
struct Lanes {
    int sub;
    unsigned mask;
};

template <int NQ>
__device__ __forceinline__ Lanes thread_lanes()
{
    constexpr int L = Geo<NQ>::LPW;
    const int lane = threadIdx.x & 31, sub = lane % L;
    return Lanes{sub, (0xFFFFFFFFu >> (32 - L)) << (lane - sub)};
}

// index of the thread's lane group in its CTA
template <int NQ>
__device__ __forceinline__ int group_in_cta()
{
    return (int)(threadIdx.x >> 5) * Geo<NQ>::GROUPS + (int)(threadIdx.x & 31) / Geo<NQ>::LPW;
}

// One adjoint butterfly stage on the weight vector held by the lane group
// (row j = sub + LPW t in registers ua/ub; the group's exchange buffer carries
// the partner rows).  The forward R^(p) maps a row that commutes with p to sqrt2
// times itself, (a, b) -> (2b, a), and an anticommuting row i to
// M_i + s(p, i^p) M_{i^p}; R^(p)^T uses s(p, i) instead, and
// s(p, i^p) = -s(p, i).  The adjoints are (ua, ub) -> (ub, 2 ua) on commuting
// rows and u_j + s(p, j) u_{j^p} (adjoint of R^) or u_j - s(p, j) u_{j^p}
// (adjoint of R^T) on the others.  Commutation and sign come from the
// per-Pauli bit masks staged in shared memory.
template <int NQ, bool ADJ_OF_TRANSPOSE>
__device__ __forceinline__ void adj_stage(uint32_t p, uint32_t (&ua)[Geo<NQ>::RPL],
                                          uint32_t (&ub)[Geo<NQ>::RPL], const Smem<NQ> &sm, Lanes g)
{
    using G = Geo<NQ>;
    uint2 *su = sm.xchg;
#pragma unroll
    for (int t = 0; t < G::RPL; t++) su[g.sub + G::LPW * t] = make_uint2(ua[t], ub[t]);
    __syncwarp(g.mask);
    // this lane's rows of Pauli p: bit t anticommutes, bit 8 + t sign +1
    const uint32_t bits = reinterpret_cast<const uint16_t *>(sm.coef)[p * G::LPW + g.sub];
#pragma unroll
    for (int t = 0; t < G::RPL; t++) {
        const int j = g.sub + G::LPW * t;
        const bool anti = (bits >> t) & 1u;
        const bool plus = (bits >> (8 + t)) & 1u;
        const uint2 v = su[j ^ (int)p];
        const bool add = (plus != ADJ_OF_TRANSPOSE);
        const uint32_t na = add ? ua[t] + v.x : ua[t] - v.x;
        const uint32_t nb = add ? ub[t] + v.y : ub[t] - v.y;
        const uint32_t ca = ub[t], cb = ua[t] << 1;
        ua[t] = anti ? na : ca;
        ub[t] = anti ? nb : cb;
    }
    __syncwarp(g.mask);
}

// d = c + sum_j a_j b_j over the four bytes, a unsigned and b signed (mod 2^32)
__device__ __forceinline__ uint32_t dp4a_us(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// Byte planes of the weights for the byte-quad contraction.  Fingerprints
// live mod 2^16, so a row's weight is u = u_0 + 2^8 u_1 (mod 2^16) with bytes
// u_0, u_1, and sum_i u_i c_i = sum_i u_{i,0} c_i + 2^8 sum_i u_{i,1} c_i
// (mod 2^16): an exact identity whose inner sums are byte dot products.  The
// plane words of quad q (rows 4q .. 4q+3) are written, in place of the rows
// (uint2 per row) in the lane group's exchange buffer, as uint4 number q:
// (a plane 0, a plane 1, b plane 0, b plane 1), each word holding that byte
// of the four rows' weights.
template <int NQ>
__device__ __forceinline__ void weight_planes(uint2 *su, Lanes g)
{
    const int lane = g.sub;
    using G = Geo<NQ>;
    constexpr int JOBS = G::DIM >= 2 * G::LPW ? G::DIM / (2 * G::LPW) : 1; // 2 parts x DIM/4 quads over the lanes
    const uint4 *s4 = reinterpret_cast<const uint4 *>(su);
    uint2 pl[JOBS];
#pragma unroll
    for (int r = 0; r < JOBS; r++) {
        const int job = lane + G::LPW * r, q = job >> 1, part = job & 1;
        const uint4 r01 = s4[2 * q], r23 = s4[2 * q + 1]; // rows 4q, 4q+1 and 4q+2, 4q+3
        const uint32_t u0 = part ? r01.y : r01.x, u1 = part ? r01.w : r01.z;
        const uint32_t u2 = part ? r23.y : r23.x, u3 = part ? r23.w : r23.z;
        const uint32_t lo01 = __byte_perm(u0, u1, 0x5140), lo23 = __byte_perm(u2, u3, 0x5140);
        pl[r] = make_uint2(__byte_perm(lo01, lo23, 0x5410), __byte_perm(lo01, lo23, 0x7632));
    }
    __syncwarp(g.mask);
    uint2 *w2 = su;
#pragma unroll
    for (int r = 0; r < JOBS; r++) w2[lane + G::LPW * r] = pl[r];
    __syncwarp(g.mask);
}

// The fingerprint weights of one decoded point pushed through its side's
// adjoint stages (row j = sub + LPW t in ua, ub): for V (side 0) the result is
// already the column fingerprints, L(V e_Q) = ua[Q]; for W (side 1) it still
// has to be contracted with C^.  All lanes of the group call it with the
// same point.
template <int NQ>
__device__ __forceinline__ void side_weights(int side, uint64_t qpack, uint32_t chunk, const LevelCtx &lv,
                                             const Smem<NQ> &sm, Lanes g, uint32_t (&ua)[Geo<NQ>::RPL],
                                             uint32_t (&ub)[Geo<NQ>::RPL])
{
    using G = Geo<NQ>;
    const Decoded dx{side, qpack};
    const int lane = g.sub;
    const int h = lv.h;

    // The weights enter the side's first adjoint stage from the stage table
    // (fingerprints live mod 2^16, and so does the table): V takes
    // R^(q_h)^* first, W takes (R^(q_1)^T)^* first.  The V side uses it only
    // when further stages follow, so no product is ever a bare lookup; the W
    // side always goes on to the contraction with C^.
    int s0 = 0;
    const uint32_t *tab = nullptr;
    uint32_t e = 0;
    if (h >= (dx.side == 0 ? 2 : 1) && lv.T1[dx.side]) {
        const uint32_t qa = (uint32_t)(dx.qpack >> (8 * (dx.side == 0 ? h - 1 : 0))) & 0xFFu;
        tab = lv.T1[dx.side];
        e = qa - 1;
        s0 = 1;
    }
#pragma unroll
    for (int t = 0; t < G::RPL; t++) {
        const int j = lane + G::LPW * t;
        if (tab) {
            const uint32_t w = __ldg(tab + (size_t)e * G::DIM + j);
            ua[t] = w & 0xFFFFu;
            ub[t] = w >> 16;
        } else {
            const uint2 u = sm.U[j];
            ua[t] = u.x;
            ub[t] = u.y;
        }
    }

    if (dx.side == 0) {
        // V side at exponent K: S R^(q_h)..R^(q_1) with S = multiply by
        // sqrt2^ev.  Weights go through S^* and R^(q_h)^* .. R^(q_1)^*; S^*
        // multiplies every row by the same power of sqrt2, so it commutes
        // with the stages and is applied after the table's.
        const int ev = lv.ev, sh = ev >> 1;
#pragma unroll
        for (int t = 0; t < G::RPL; t++) {
            const uint32_t a = ua[t], b = ub[t];
            ua[t] = (ev & 1) ? shl32(b, sh) : shl32(a, sh);
            ub[t] = (ev & 1) ? shl32(a, sh + 1) : shl32(b, sh);
        }
        for (int j = h - 1 - s0; j >= 0; j--)
            adj_stage<NQ, false>((uint32_t)(dx.qpack >> (8 * j)) & 0xFFu, ua, ub, sm, g);
    } else {
        // W side: R^(q_1)^T .. R^(q_h)^T [R^(c)^T] C^; weights go through
        // (R^(q_1)^T)^* first, ..., (R^(q_h)^T)^*, then (R^(c)^T)^*.
        for (int j = s0; j < h; j++)
            adj_stage<NQ, true>((uint32_t)(dx.qpack >> (8 * j)) & 0xFFu, ua, ub, sm, g);
        if (lv.k & 1) adj_stage<NQ, true>(chunk, ua, ub, sm, g);
    }
}

// The lane's share of the multiset hash: the sum mod 2^64 of
// smix(base ^ phi_Q) over the lane's columns Q = sub + LPW t >= 1, phi_Q the
// sign-folded 16-bit fingerprint of column Q (column 0, the identity, does
// not enter).
template <int NQ>
__device__ __forceinline__ uint64_t lane_column_sum(const uint32_t (&Lc)[Geo<NQ>::RPL], uint64_t base, int lane)
{
    uint64_t acc = 0;
    const uint64_t pre = base ^ (base >> 30);
#pragma unroll
    for (int t = 0; t < Geo<NQ>::RPL; t++) {
        const int Q = lane + Geo<NQ>::LPW * t;
        const uint32_t l = Lc[t] & 0xFFFFu, nl = (0u - l) & 0xFFFFu;
        const uint64_t e = smix_pre(pre, min(l, nl));
        acc += (Q >= 1) ? e : 0ull;
    }
    return acc;
}

// sum mod 2^64 over the lane group from three 32-bit reductions: the high
// words (mod 2^32) and the two 16-bit halves of the low words (no overflow:
// at most 32 terms)
__device__ __forceinline__ uint64_t group_sum64(uint64_t acc, unsigned mask)
{
    const uint32_t lo = (uint32_t)acc, hi = (uint32_t)(acc >> 32);
    const uint32_t s_hi = __reduce_add_sync(mask, hi);
    const uint32_t s_l0 = __reduce_add_sync(mask, lo & 0xFFFFu);
    const uint32_t s_l1 = __reduce_add_sync(mask, lo >> 16);
    return ((uint64_t)s_hi << 32) + ((uint64_t)s_l1 << 16) + (uint64_t)s_l0;
}

// nu and h of one decoded point: the exact product of side `side` (0: V,
// 1: W) for the rotations in qpack (and the chunk, odd k), its column
// fingerprints and their multiset hash with hash base `base`, as a
// full 64-bit value.  All lanes of the group call it with the same point.
template <int NQ>
__device__ uint64_t coset_hash(int side, uint64_t qpack, uint32_t chunk, uint64_t base, const LevelCtx &lv,
                               const Smem<NQ> &sm, Lanes g)
{
    using G = Geo<NQ>;
    const int lane = g.sub;
    uint32_t ua[G::RPL], ub[G::RPL], Lc[G::RPL];
    side_weights<NQ>(side, qpack, chunk, lv, sm, g, ua, ub);
    if (side == 0) {
#pragma unroll
        for (int t = 0; t < G::RPL; t++) Lc[t] = ua[t]; // L(V e_Q) = (U~)_a[Q]
    } else {
        uint2 *su = sm.xchg;
#pragma unroll
        for (int t = 0; t < G::RPL; t++) {
            su[lane + G::LPW * t] = make_uint2(ua[t], ub[t]);
            Lc[t] = 0;
        }
        __syncwarp(g.mask);
        // L(W e_Q) = sum_i U~_a[i] C_a[i][Q] + U~_b[i] C_b[i][Q]; row 0 has
        // zero weight and C[0][Q] = 0 for Q >= 1, so all rows may be summed.
        if (G::DIM >= 64 && sm.Cq) {
            // byte-plane contraction: acc[t][k] = sum over rows of byte k of
            // the weights times C^ (exact byte products), recombined below
            weight_planes<NQ>(su, g);
            const uint4 *w4 = reinterpret_cast<const uint4 *>(su);
            constexpr int CW = G::RPL / 2;
            uint32_t acc[G::RPL][2];
#pragma unroll
            for (int t = 0; t < G::RPL; t++) acc[t][0] = acc[t][1] = 0;
#pragma unroll G::QUAD_UNROLL
            for (int q = 0; q < G::DIM / 4; q++) {
                const uint4 w = w4[q]; // a plane 0, a plane 1, b plane 0, b plane 1
#pragma unroll
                for (int j = 0; j < CW; j++) {
                    const uint4 c = sm.Cq[(q * CW + j) * G::LPW + lane];
                    acc[2 * j][0] = dp4a_us(w.x, c.x, acc[2 * j][0]);
                    acc[2 * j][0] = dp4a_us(w.z, c.y, acc[2 * j][0]);
                    acc[2 * j][1] = dp4a_us(w.y, c.x, acc[2 * j][1]);
                    acc[2 * j][1] = dp4a_us(w.w, c.y, acc[2 * j][1]);
                    acc[2 * j + 1][0] = dp4a_us(w.x, c.z, acc[2 * j + 1][0]);
                    acc[2 * j + 1][0] = dp4a_us(w.z, c.w, acc[2 * j + 1][0]);
                    acc[2 * j + 1][1] = dp4a_us(w.y, c.z, acc[2 * j + 1][1]);
                    acc[2 * j + 1][1] = dp4a_us(w.w, c.w, acc[2 * j + 1][1]);
                }
            }
#pragma unroll
            for (int t = 0; t < G::RPL; t++) Lc[t] = acc[t][0] + (acc[t][1] << 8);
        } else if (G::DIM >= 32) {
            const uint4 *su4 = reinterpret_cast<const uint4 *>(su);
#pragma unroll kGemvUnroll
            for (int i = 0; i < G::DIM; i += 2) {
                const uint4 uu = su4[i >> 1]; // rows i and i + 1
                const uint2 *c0 = sm.C + i * G::DIM + lane * G::RPL;
                const uint2 *c1 = c0 + G::DIM;
#pragma unroll
                for (int t = 0; t < G::RPL; t += 2) {
                    const uint4 a = *reinterpret_cast<const uint4 *>(c0 + t);
                    const uint4 b = *reinterpret_cast<const uint4 *>(c1 + t);
                    Lc[t] += uu.x * a.x + uu.y * a.y + uu.z * b.x + uu.w * b.y;
                    Lc[t + 1] += uu.x * a.z + uu.y * a.w + uu.z * b.z + uu.w * b.w;
                }
            }
        } else {
            for (int i = 0; i < G::DIM; i++) {
                const uint2 u = su[i], c = sm.C[i * G::DIM + lane];
                Lc[0] += u.x * c.x + u.y * c.y;
            }
        }
        __syncwarp(g.mask);
    }

    // sign-invariant 16-bit column fingerprints phi_Q of the columns Q >= 1,
    // hashed as a multiset: the sum mod 2^64 of smix(base ^ phi_Q), a
    // function of the multiset alone
    return smix(group_sum64(lane_column_sum<NQ>(Lc, base, lane), g.mask));
}

// f(x): all lanes of the group call it with the same x; each gets the result.
template <int NQ>
__device__ __forceinline__ uint64_t warp_step(uint64_t x, uint32_t chunk, const LevelCtx &lv, const Smem<NQ> &sm,
                                              Lanes g)
{
    const Decoded dx = decode(x, lv);
    return coset_hash<NQ>(dx.side, dx.qpack, chunk, sm.base[chunk], lv, sm, g) & lv.maskL;
}

// Stage the weights, the rotation coefficients, the per-chunk hash bases and
// (n <= 3) all of C^ into shared memory; returns this warp's views.  WITH_C
// false: the smaller layout without C^ (smem_bytes_v), whose views of C^ are
// null; only V products may then be evaluated.
template <int NQ, bool WITH_C = true>
__device__ __forceinline__ Smem<NQ> stage(const LevelCtx &lv, unsigned char *raw)
{
    using G = Geo<NQ>;
    Smem<NQ> sm;
    sm.U = reinterpret_cast<uint2 *>(raw);
    uint2 *sC = reinterpret_cast<uint2 *>(raw + G::off_C);
    sm.coef = reinterpret_cast<uint32_t *>(raw + (WITH_C ? G::off_coef : G::off_coef_v));
    sm.base = reinterpret_cast<uint64_t *>(raw + (WITH_C ? G::off_base : G::off_base_v));
    sm.xchg = reinterpret_cast<uint2 *>(raw + (WITH_C ? G::off_xchg : G::off_xchg_v)) + group_in_cta<NQ>() * G::DIM;
    for (int i = threadIdx.x; i < G::DIM; i += blockDim.x) sm.U[i] = lv.U[i];
    for (int i = threadIdx.x; i < G::COEF_WORDS; i += blockDim.x) sm.coef[i] = lv.coef[i];
    // base(chunk) = smix(smix(seed_H ^ version) ^ (n | k << 8 | chunk << 16 | K << 32))
    const uint64_t vmix = smix(kSeedH ^ (uint64_t)lv.version);
    for (int c = threadIdx.x; c < G::MAX_CHUNKS; c += blockDim.x) {
        const uint64_t tag = (uint64_t)lv.n | ((uint64_t)lv.k << 8) | ((uint64_t)c << 16) |
                             ((uint64_t)(uint32_t)lv.K << 32);
        sm.base[c] = smix(vmix ^ tag);
    }
    sm.Cq = nullptr;
    if (!WITH_C) {
        sm.C = nullptr;
    } else if (G::C_SMEM) {
        if (lv.Cq && G::DIM >= 64) {
            uint4 *dst = reinterpret_cast<uint4 *>(sC);
            for (int i = threadIdx.x; i < G::DIM * G::DIM * 2 / 16; i += blockDim.x) dst[i] = lv.Cq[i];
            sm.Cq = dst;
        } else {
            const uint4 *src = reinterpret_cast<const uint4 *>(lv.C32);
            uint4 *dst = reinterpret_cast<uint4 *>(sC);
            for (int i = threadIdx.x; i < G::DIM * G::DIM / 2; i += blockDim.x) dst[i] = src[i];
        }
        sm.C = sC;
    } else {
        sm.C = lv.C32;
        if (G::CQ_SMEM && lv.Cq) {
            uint4 *dst = reinterpret_cast<uint4 *>(sC);
            for (int i = threadIdx.x; i < G::DIM * G::DIM * 2 / 16; i += blockDim.x) dst[i] = lv.Cq[i];
            sm.Cq = dst;
        }
    }
    __syncthreads();
    return sm;
}

template <int NQ>
__global__ void __launch_bounds__(Geo<NQ>::THREADS) k_walk_step(LevelCtx lv, uint32_t chunk, const uint64_t *__restrict__ in,
                                                        uint64_t *__restrict__ out, uint8_t *__restrict__ is_dp,
                                                        size_t count)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Smem<NQ> sm = stage<NQ>(lv, smem_raw);
    const Lanes g = thread_lanes<NQ>();
    for (size_t i = (size_t)blockIdx.x * Geo<NQ>::WALKS + group_in_cta<NQ>(); i < count;
         i += (size_t)gridDim.x * Geo<NQ>::WALKS) {
        const uint64_t y = warp_step<NQ>(in[i], chunk, lv, sm, g);
        if (g.sub == 0) {
            out[i] = y;
            if (is_dp) is_dp[i] = (uint8_t)((y >> lv.dshift) == 0);
        }
    }
}

template <typename T>
__device__ __forceinline__ void flush_tally(unsigned long long *counters, TallyOf<T> &t, Lanes g)
{
    if (g.sub == 0) {
        if (t.steps) atomicAdd(&counters[C_STEPS], t.steps);
        if (t.w) atomicAdd(&counters[C_WSTEPS], t.w);
        if (t.dp) atomicAdd(&counters[C_DPS], t.dp);
        if (t.ab) atomicAdd(&counters[C_ABANDONED], t.ab);
        if (t.evicted) atomicAdd(&counters[C_EVICTED], t.evicted);
        if (t.duplicate) atomicAdd(&counters[C_DUPLICATE], t.duplicate);
        if (t.pairs) atomicAdd(&counters[C_PAIRS], t.pairs);
    }
    t = TallyOf<T>();
}

// Advance one walk by w.steps steps (Sec. 3 trails): a trail that reaches a
// distinguished point is stored and a new one starts; a trail longer than
// the cut-off is abandoned.  All lanes of the group call it.
template <int NQ, typename WL>
__device__ __forceinline__ void walk_one(const WL &w, const Smem<NQ> &sm, int local, Lanes g, Tally &t)
{
    WalkState st = w.walks[local];
    const uint32_t walk = w.walk_base + (uint32_t)local; // index among all ranks' walks
    const uint32_t steps = w.steps, max_len = w.max_len;
    const int dshift = w.lv.dshift;
    for (uint32_t s = 0; s < steps; s++) {
        const uint64_t y = warp_step<NQ>(st.cur, st.chunk, w.lv, sm, g);
        t.steps++;
        t.w += st.cur & 1;
        st.len++;
        if ((y >> dshift) == 0) {
            t.dp++;
            if (g.sub == 0) dp_insert(w, y, make_ref(walk, st.seq, st.len), t);
            __syncwarp(g.mask);
            new_trail(st, walk, w.lv);
        } else if (st.len >= max_len) {
            t.ab++;
            new_trail(st, walk, w.lv);
        } else {
            st.cur = y;
        }
    }
    if (g.sub == 0) w.walks[local] = st;
}

template <int NQ, int S>
__global__ void __launch_bounds__(Shape<NQ, S>::THREADS, Shape<NQ, S>::MIN_BLOCKS) k_walks(WalkLaunch w)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Smem<NQ> sm = stage<NQ>(w.lv, smem_raw);
    const Lanes g = thread_lanes<NQ>();
    Tally t;
    for (int walk = blockIdx.x * Shape<NQ, S>::WALKS + group_in_cta<NQ>(); walk < w.n_walks;
         walk += gridDim.x * Shape<NQ, S>::WALKS)
        walk_one<NQ>(w, sm, walk, g, t);
    flush_tally(w.counters, t, g);
}

// Many jobs (targets, each at its own level) in one persistent launch: the
// CTA takes a contiguous range of tasks (job, first walk) of this qubit
// count, restages the job's data when the job changes, and each lane group
// walks one of the task's Shape<NQ, S>::WALKS walks.  The job's launch record is copied to
// shared memory.
template <int NQ, int S>
__global__ void __launch_bounds__(Shape<NQ, S>::THREADS, Shape<NQ, S>::MIN_BLOCKS) k_walks_batch(BatchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ WalkLaunch sw;
    const Lanes g = thread_lanes<NQ>();
    const uint32_t nt = *a.n_tasks;
    int cur = -1;
    Smem<NQ> sm;
    Tally t;
    // a contiguous range of tasks per CTA, so that job changes (restaging) are rare
    const uint32_t t_begin = (uint32_t)(((uint64_t)nt * blockIdx.x) / gridDim.x);
    const uint32_t t_end = (uint32_t)(((uint64_t)nt * (blockIdx.x + 1)) / gridDim.x);
    for (uint32_t task = t_begin; task < t_end; task++) {
        const int job = (int)a.tasks[2 * task];
        const int first = (int)a.tasks[2 * task + 1];
        if (job != cur) {
            if (cur >= 0) flush_tally(sw.counters, t, g);
            __syncthreads(); // every warp is done with the previous job's data
            if (threadIdx.x == 0) sw = a.jobs[job];
            __syncthreads();
            sm = stage<NQ>(sw.lv, smem_raw);
            cur = job;
        }
        const int walk = first + group_in_cta<NQ>();
        if (walk < sw.n_walks) walk_one<NQ>(sw, sm, walk, g, t);
    }
    if (cur >= 0) flush_tally(sw.counters, t, g);
}

__global__ void k_init_walks(WalkLaunch w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= w.n_walks) return;
    WalkState st;
    st.seq = 0;
    st.pad = 0;
    new_trail(st, w.walk_base + (uint32_t)i, w.lv);
    w.walks[i] = st;
}

// DP-owner sharding: the distinguished points received from every rank go
// into this rank's table exactly as the walk's own inserts would.
__global__ void k_insert_points(WalkLaunch w, const Slot *__restrict__ pts, uint32_t count)
{
    Tally t;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const Slot p = pts[i];
        dp_insert(w, p.key, p.ref, t);
    }
    // per-thread tallies (there are no lane groups here)
    if (t.evicted) atomicAdd(&w.counters[C_EVICTED], t.evicted);
    if (t.duplicate) atomicAdd(&w.counters[C_DUPLICATE], t.duplicate);
    if (t.pairs) atomicAdd(&w.counters[C_PAIRS], t.pairs);
}

// owner rank of a distinguished point among n ranks: the high word of a
// second finaliser (independent of the table slot, which takes smix's low
// bits) scaled to [0, n)
__device__ __forceinline__ uint32_t owner_of(uint64_t dp, uint32_t n)
{
    return (uint32_t)(((smix(dp ^ 0xD1B54A32D192ED03ull) >> 32) * (uint64_t)n) >> 32);
}

// Bin points by owner: one counting pass, a prefix over the n owners in
// every block (n <= 1024), then scatter.  Order within a bin is arbitrary
// (the table does not depend on insertion order beyond which trail a slot
// keeps).
__global__ void k_count_owners(const Slot *__restrict__ in, uint32_t count, uint32_t n, uint32_t *counts)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        atomicAdd(&counts[owner_of(in[i].key, n)], 1u);
}

__global__ void k_scatter_owners(const Slot *__restrict__ in, uint32_t count, uint32_t n,
                                 const uint32_t *__restrict__ counts, uint32_t *fill, Slot *out)
{
    extern __shared__ uint32_t start[]; // exclusive prefix of counts
    if (threadIdx.x == 0) {
        uint32_t acc = 0;
        for (uint32_t r = 0; r < n; r++) {
            start[r] = acc;
            acc += counts[r];
        }
    }
    __syncthreads();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const Slot p = in[i];
        const uint32_t r = owner_of(p.key, n);
        out[start[r] + atomicAdd(&fill[r], 1u)] = p;
    }
}

// Sec. 3, Fig. 2: align the longer trail, step both until the images agree,
// and classify the two distinct preimages.  At most `budget` evaluations of f
// (0: no bound); returns false with (a, la, b, lb) advanced when the budget
// ends first, so the re-walk can resume from there.  Lengths are bounded by
// the maximum trail length, so the loops end.
template <int NQ>
__device__ bool rewalk_resume(const LevelCtx &lv, uint32_t chunk, uint64_t &a, uint32_t &la, uint64_t &b,
                              uint32_t &lb, uint32_t budget, const Smem<NQ> &sm, Lanes g, unsigned long long &nf,
                              RewalkOut &r)
{
    r.chunk = chunk;
    if (la > kMaxRewalkLen || lb > kMaxRewalkLen) {
        r.cls = 5;
        r.a = a;
        r.b = b;
        return true;
    }
    if (la < lb) {
        uint64_t tx = a; a = b; b = tx;
        uint32_t tl = la; la = lb; lb = tl;
    }
    // one evaluation of f per iteration through a single call site (the step
    // is large at n = 4; inlining it once keeps the kernel's code compact):
    // align the longer trail, then step a and b in turn
    uint32_t used = 0;
    uint64_t fa = 0;
    bool second = false, checked = false;
    for (;;) {
        uint64_t x;
        if (la > lb) {
            if (budget && used >= budget) return false;
            x = a;
        } else if (!second) {
            // aligned: equal states mean one start lies on the other trail
            // (after a lockstep step this cannot first happen: the images
            // are compared there)
            if (!checked) {
                checked = true;
                if (a == b) {
                    r.cls = 0; // Robin Hood
                    r.a = r.b = a;
                    return true;
                }
            }
            if (lb == 0) {
                r.cls = 5; // no merge
                r.a = a;
                r.b = b;
                return true;
            }
            if (budget && used + 2 > budget) return false;
            x = a;
        } else {
            x = b;
        }
        const uint64_t y = warp_step<NQ>(x, chunk, lv, sm, g);
        used++;
        nf++;
        if (la > lb) {
            a = y;
            la--;
        } else if (!second) {
            fa = y;
            second = true;
        } else {
            second = false;
            if (fa == y) {
                const Decoded da = decode(a, lv), db = decode(b, lv);
                r.a = a;
                r.b = b;
                if (da.side == db.side) r.cls = (da.qpack == db.qpack) ? 1 : 2; // trivial / same side
                else r.cls = 3;                                          // claw candidate
                return true;
            }
            a = fa;
            b = y;
            la--;
            lb--;
        }
    }
}

template <int NQ>
__device__ RewalkOut rewalk_one(const LevelCtx &lv, uint32_t chunk, uint64_t sa, uint32_t la, uint64_t sb,
                                uint32_t lb, const Smem<NQ> &sm, Lanes g, unsigned long long *fevals = nullptr)
{
    RewalkOut r;
    unsigned long long nf = 0;
    rewalk_resume<NQ>(lv, chunk, sa, la, sb, lb, 0, sm, g, nf, r);
    if (fevals) *fevals += nf;
    return r;
}

// Re-walk this CTA's share of one job's queued merges; classes are counted
// per lane group and claw candidates appended to the job's candidate list.
// With `cursor` set, the lane groups take merges one at a time from that
// device counter instead of by a fixed stride, so that a few long trail
// pairs do not leave the rest of the grid idle.
template <int NQ, typename WL>
__device__ __forceinline__ void rewalk_job(const WL &w, const Smem<NQ> &sm, uint32_t p_begin, uint32_t p_end,
                                           uint32_t p_stride, Lanes g, uint32_t *cursor = nullptr)
{
    unsigned long long c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0, c5 = 0; // per class, in registers
    unsigned long long fev = 0;
    auto claim = [&]() -> uint32_t {
        uint32_t v = 0;
        if (g.sub == 0) v = atomicAdd(cursor, 1u);
        return __shfl_sync(g.mask, v, 0, Geo<NQ>::LPW);
    };
    for (uint32_t p = cursor ? claim() : p_begin; p < p_end; p = cursor ? claim() : p + p_stride) {
        // the job's work list: first the re-walks carried from the previous
        // round (batched search), then this launch's queued merges
        const Merge m = load_merge(w, p);
        uint64_t xa = m.a, xb = m.b;
        uint32_t la = m.la, lb = m.lb;
        const uint32_t ca = m.ca;
        RewalkOut r;
        if (ca != m.cb) { // the same value reached in two chunks' functions: no merge
            r.cls = 5;
        } else if (!rewalk_resume<NQ>(w.lv, ca, xa, la, xb, lb, w.rewalk_budget, sm, g, fev, r)) {
            // budget spent: carry the re-walk to the next round (if there is room)
            if (g.sub == 0) carry_merge(w, xa, la, xb, lb, ca);
            continue;
        }
        c0 += r.cls == 0;
        c1 += r.cls == 1;
        c2 += r.cls == 2;
        c3 += r.cls == 3;
        c4 += r.cls == 4;
        c5 += r.cls == 5;
        if (r.cls == 3 && g.sub == 0) {
            append_claw(w, r.a, r.b, ca);
        }
    }
    if (g.sub == 0) {
        const unsigned long long cc[6] = {c0, c1, c2, c3, c4, c5};
#pragma unroll
        for (int c = 0; c < 6; c++)
            if (cc[c]) atomicAdd(&w.counters[C_CLS0 + c], cc[c]);
        if (c3) atomicAdd(&w.counters[C_CANDS], c3);
        if (fev) atomicAdd(&w.counters[C_RSTEPS], fev);
    }
}

// below: lists of this length and longer are left to the quads (k_rewalk_q)
template <int NQ>
__global__ void __launch_bounds__(Geo<NQ>::THREADS) k_rewalk_pairs(WalkLaunch w, uint32_t below)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t cnt = w.pend_in_n + min(*w.qhead, w.qcap);
    if (cnt >= below) return;
    if (cnt <= blockIdx.x * Geo<NQ>::WALKS) return; // no pair for this CTA (uniform)
    const Smem<NQ> sm = stage<NQ>(w.lv, smem_raw);
    rewalk_job<NQ>(w, sm, blockIdx.x * Geo<NQ>::WALKS + group_in_cta<NQ>(), cnt, gridDim.x * Geo<NQ>::WALKS,
                   thread_lanes<NQ>(), w.rw_next);
}

// The batched re-walk: the queued merges of all jobs of this qubit count
// form one index space; each CTA takes a contiguous range of it, so it
// restages a job's data only where its range enters that job.
template <int NQ>
__global__ void __launch_bounds__(Geo<NQ>::THREADS) k_rewalk_batch(BatchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ WalkLaunch sw;
    const uint32_t nj = *a.n_jobs;
    uint64_t total = 0;
    for (uint32_t j = 0; j < nj; j++) {
        const WalkLaunch &w = a.jobs[a.job_ids[j]];
        total += w.pend_in_n + min(*w.qhead, w.qcap);
    }
    const uint64_t lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
    const Lanes g = thread_lanes<NQ>();
    uint64_t base = 0;
    for (uint32_t j = 0; j < nj && base < hi; j++) {
        const int job = (int)a.job_ids[j];
        const uint32_t cnt = a.jobs[job].pend_in_n + min(*a.jobs[job].qhead, a.jobs[job].qcap);
        if (base + cnt <= lo) {
            base += cnt;
            continue;
        }
        const uint32_t p_begin = (uint32_t)(max(lo, base) - base), p_end = (uint32_t)(min(hi, base + cnt) - base);
        base += cnt;
        __syncthreads();
        if (threadIdx.x == 0) sw = a.jobs[job];
        __syncthreads();
        const Smem<NQ> sm = stage<NQ>(sw.lv, smem_raw);
        rewalk_job<NQ>(sw, sm, p_begin + group_in_cta<NQ>(), p_end, Geo<NQ>::WALKS, g);
    }
}

template <int NQ>
__global__ void __launch_bounds__(Geo<NQ>::THREADS) k_rewalk_arrays(LevelCtx lv, uint32_t chunk, const uint64_t *sa,
                                                            const uint32_t *la, const uint64_t *sb,
                                                            const uint32_t *lb, size_t count, int32_t *cls,
                                                            uint64_t *ab)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Smem<NQ> sm = stage<NQ>(lv, smem_raw);
    const Lanes g = thread_lanes<NQ>();
    for (size_t p = (size_t)blockIdx.x * Geo<NQ>::WALKS + group_in_cta<NQ>(); p < count;
         p += (size_t)gridDim.x * Geo<NQ>::WALKS) {
        const RewalkOut r = rewalk_one<NQ>(lv, chunk, sa[p], la[p], sb[p], lb[p], sm, g);
        if (g.sub == 0) {
            cls[p] = r.cls;
            ab[2 * p] = r.a;
            ab[2 * p + 1] = r.b;
        }
    }
}

// Exhaustive level pass (CertArgs): one lane group per point, grid-stride.
// VONLY: the points are V products (a.side == 0), which never touch C^, so
// the CTA stages the smaller layout without it.  A point index is nd base-xi
// digits: the h rotation digits (q_j = digit + 1), then for a W point of odd
// k the chunk digit (chunk = digit + 1).  Each thread divides only for its
// first index and its stride; every further index adds the stride's digits.
template <int NQ, bool VONLY>
__global__ void __launch_bounds__(Geo<NQ>::THREADS) k_certify(CertArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Smem<NQ> sm = stage<NQ, !VONLY>(a.lv, smem_raw);
    const int side = VONLY ? 0 : a.side;
    const Lanes g = thread_lanes<NQ>();
    const uint32_t xi = a.lv.xi;
    const int h = a.lv.h;
    const bool has_chunk = side == 1 && (a.lv.k & 1);
    const int nd = h + (has_chunk ? 1 : 0);
    const uint64_t hmask = h >= 8 ? ~0ull : (1ull << (8 * h)) - 1;
    const uint64_t stride = (uint64_t)gridDim.x * Geo<NQ>::WALKS;
    uint64_t i = (uint64_t)blockIdx.x * Geo<NQ>::WALKS + group_in_cta<NQ>();
    // While i + stride < count, the stride is below xi^nd and its nd digits
    // are exact; otherwise the loop ends before the sum is used.
    uint64_t dig = 0, sdig = 0;
    uint32_t stored = 0;
    if (i < a.count) {
        dig = base_xi_digits(a.first + i, xi, nd);
        sdig = base_xi_digits(stride, xi, nd);
    }
    for (; i < a.count; i += stride, dig = add_base_xi(dig, sdig, xi, nd)) {
        const uint64_t idx = a.first + i;
        const uint64_t qpack = (dig & hmask) + (0x0101010101010101ull & hmask);
        const uint32_t chunk = has_chunk ? (uint32_t)((dig >> (8 * h)) & 0xFFu) + 1 : 0u;
        uint64_t key = coset_hash<NQ>(side, qpack, chunk, a.base, a.lv, sm, g);
        if (key == ~0ull) key = ~0ull - 1; // ~0 marks an empty slot
        if (g.sub == 0) {
            if (a.insert) stored += cert_insert(a, key, idx);
            else cert_probe(a, key, idx);
        }
        __syncwarp(g.mask);
    }
    cert_count(a, stored);
}

int g_num_sms = 0;

// resident CTAs per SM of k_walks<NQ, S> (occupancy, cached)
template <int NQ, int S = 0>
int blocks_per_sm()
{
    static int cached = 0;
    if (!cached) {
        using L = Shape<NQ, S>;
        cudaFuncSetAttribute(k_walks<NQ, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_bytes);
        int b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_walks<NQ, S>, L::THREADS, L::smem_bytes);
        cached = b > 0 ? b : 1;
    }
    return cached;
}

template <int NQ, int S = 0>
unsigned grid_for(size_t units)
{
    const size_t cap = (size_t)num_sms() * (size_t)blocks_per_sm<NQ, S>();
    size_t g = (units + Shape<NQ, S>::WALKS - 1) / Shape<NQ, S>::WALKS;
    if (g > cap) g = cap;
    if (g == 0) g = 1;
    return (unsigned)g;
}

// One entry of LevelCtx::Cm a thread, once per problem: 2 D^2 threads.
template <int NQ>
__global__ void k_operand(const uint2 *__restrict__ C32, uint16_t *__restrict__ Cm)
{
    constexpr uint32_t D = 1u << (2 * NQ), W = D < 32 ? D : 32, R = D / W;
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    uint32_t at, part, row, Q;
    if constexpr (NQ == 4) {
        Q = i & (D - 1);
        part = i >> 16;
        const uint32_t k = (i >> 8) & 255u;
        row = row_of(4, k >> 3, k & 7u);
        at = cm_index(Q, part * D + k);
    } else {
        // fragments of m16n8k16's A, [tile][part][k-step][lane][register][half]:
        // register r holds column lane / 4 (+ 8 for odd r) of the tile, k
        // 2 (lane % 4) (+ 8 for r >= 2) and one more
        constexpr uint32_t T = D / 16;
        const uint32_t half = i & 1u, r = (i >> 1) & 3u, lane = (i >> 3) & 31u, ks = (i >> 8) % T, mt = (i >> 8) / (2 * T);
        const uint32_t m = (lane >> 2) + 8 * (r & 1u);
        part = ((i >> 8) / T) & 1u;
        Q = quad_row(NQ, (m & 7u) >> 1, 4 * mt + (m & 1u) + 2 * (m >> 3));
        row = quad_row(NQ, lane & 3u, 4 * ks + 2 * (r >> 1) + half);
        at = i;
    }
    const uint2 c = C32[row * D + (Q % W) * R + Q / W];
    Cm[at] = row == 0 ? (part ? (uint16_t)0 : kCmBias) : __half_as_ushort(__int2half_rn((int)(part ? c.y : c.x)));
}

template <int NQ>
cudaError_t walk_step_n(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp,
                        size_t count, cudaStream_t s)
{
    // quads, but for short n = 3 lists with C^ in int8, whose one step does
    // not make up for the larger set-up (us a launch: 4096 states 7.6 against
    // 7.3, 16384 10.3 / 14.2, 50021 17.5 / 28; n = 3 with C^ in 32-bit words:
    // 64 7.9 / 9.0, 50021 18 / 44; n = 2: 64 5.2 / 6.3, 50021 8 / 17)
    if ((NQ == 2 || (NQ == 3 && (count >= 8192 || !lv.Cq))) && lv.Cm)
        return launch_walk_step_q(lv, chunk, in, out, is_dp, count, s);
    if (NQ == 4 && lv.Cm) return launch_walk_step_e4(lv, chunk, in, out, is_dp, count, s);
    cudaFuncSetAttribute(k_walk_step<NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Geo<NQ>::smem_bytes);
    k_walk_step<NQ><<<grid_for<NQ>(count), Geo<NQ>::THREADS, Geo<NQ>::smem_bytes, s>>>(lv, (uint32_t)chunk, in, out, is_dp,
                                                                               count);
    return cudaGetLastError();
}

template <int NQ, int S>
cudaError_t walks_ns(const WalkLaunch &w, cudaStream_t s)
{
    using L = Shape<NQ, S>;
    k_walks<NQ, S><<<grid_for<NQ, S>((size_t)w.n_walks), L::THREADS, L::smem_bytes, s>>>(w);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t walks_n(const WalkLaunch &w, cudaStream_t s)
{
    switch (w.shape) {
    case 0:
        if ((NQ == 2 || (NQ == 3 && (uint32_t)w.n_walks >= (w.lv.Cq ? kQuadWalks3 : kQuadWalksWide3))) && w.lv.Cm) return launch_walks_q(w, s);
        return walks_ns<NQ, 0>(w, s);
    case 1: if constexpr (shape_count(NQ) > 1) return walks_ns<NQ, 1>(w, s); break;
    case 2: if constexpr (shape_count(NQ) > 2) return walks_ns<NQ, 2>(w, s); break;
    case 3:
        if constexpr (NQ == 4) return w.lv.Cm ? launch_walks_e4(w, s) : walks_ns<4, 0>(w, s);
        else if constexpr (shape_count(NQ) > 3) return walks_ns<NQ, 3>(w, s);
        break;
    }
    return cudaErrorInvalidValue;
}

// CTAs of the persistent batch walk kernel: every SM x its resident CTAs
template <int NQ, int S>
int batch_grid()
{
    static int g = 0;
    if (!g) {
        using L = Shape<NQ, S>;
        cudaFuncSetAttribute(k_walks_batch<NQ, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_bytes);
        int b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_walks_batch<NQ, S>, L::THREADS, L::smem_bytes);
        g = num_sms() * (b > 0 ? b : 1);
    }
    return g;
}

template <int NQ, int S>
cudaError_t walks_batch_ns(const BatchArgs &a, cudaStream_t s)
{
    using L = Shape<NQ, S>;
    k_walks_batch<NQ, S><<<batch_grid<NQ, S>(), L::THREADS, L::smem_bytes, s>>>(a);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t walks_batch_n(int shape, const BatchArgs &a, cudaStream_t s)
{
    switch (shape) {
    case 0: return walks_batch_ns<NQ, 0>(a, s);
    case 1: if constexpr (shape_count(NQ) > 1) return walks_batch_ns<NQ, 1>(a, s); break;
    case 2: if constexpr (shape_count(NQ) > 2) return walks_batch_ns<NQ, 2>(a, s); break;
    case 3:
        if constexpr (NQ == 4) return walks_batch_ns<4, 0>(a, s); // the jobs that the engine does not take
        else if constexpr (shape_count(NQ) > 3) return walks_batch_ns<NQ, 3>(a, s);
        break;
    }
    return cudaErrorInvalidValue;
}

template <int NQ>
cudaError_t rewalk_batch_n(const BatchArgs &a, cudaStream_t s)
{
    static int g = 0;
    if (!g) {
        cudaFuncSetAttribute(k_rewalk_batch<NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Geo<NQ>::smem_bytes);
        int b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_rewalk_batch<NQ>, Geo<NQ>::THREADS, Geo<NQ>::smem_bytes);
        g = num_sms() * (b > 0 ? b : 1);
    }
    k_rewalk_batch<NQ><<<g, Geo<NQ>::THREADS, Geo<NQ>::smem_bytes, s>>>(a);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t rewalk_pairs_n(const WalkLaunch &w, cudaStream_t s)
{
    // the engine is the faster one from a list of 32 merges on (6 merges: 51
    // against 47 us; 130: 54 / 66; 17320: 115 / 193; 116090: 311 / 869 us at
    // theta 1/2, 431 at 2^-8: 1.25 / 1.42 ms)
    if (NQ == 4 && w.lv.Cm) return launch_rewalk_e4(w, s);
    if (NQ == 2 && w.lv.Cm) return launch_rewalk_q(w, 0, s);
    uint32_t below = ~0u;
    if (NQ == 3 && w.lv.Cm) {
        // by the list's length, which only the device knows: both kernels, and
        // the one whose turn it is not ends at once (4 us).  Where the level's
        // last list was far from the line one of them is enough: a wrong guess
        // costs time, no merge.
        const uint32_t line = w.lv.Cq ? kQuadMerges3 : kQuadMergesWide3;
        if (w.rw_last >= 2 * line) return launch_rewalk_q(w, 0, s);
        if ((uint64_t)w.pend_in_n + w.qcap >= line && (w.rw_last == 0 || w.rw_last >= line / 4)) {
            const cudaError_t e = launch_rewalk_q(w, line, s);
            if (e != cudaSuccess) return e;
            below = line;
        }
    }
    cudaFuncSetAttribute(k_rewalk_pairs<NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)Geo<NQ>::smem_bytes);
    k_rewalk_pairs<NQ><<<grid_for<NQ>(w.qcap), Geo<NQ>::THREADS, Geo<NQ>::smem_bytes, s>>>(w, below);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t rewalk_arrays_n(const LevelCtx &lv, int chunk, const uint64_t *sa, const uint32_t *la,
                            const uint64_t *sb, const uint32_t *lb, size_t count, int32_t *cls, uint64_t *ab,
                            cudaStream_t s)
{
    cudaFuncSetAttribute(k_rewalk_arrays<NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)Geo<NQ>::smem_bytes);
    k_rewalk_arrays<NQ><<<grid_for<NQ>(count), Geo<NQ>::THREADS, Geo<NQ>::smem_bytes, s>>>(lv, (uint32_t)chunk, sa, la,
                                                                                   sb, lb, count, cls, ab);
    return cudaGetLastError();
}

template <int NQ, bool VONLY>
cudaError_t certify_nv(const CertArgs &a, cudaStream_t s)
{
    constexpr size_t smem = VONLY ? Geo<NQ>::smem_bytes_v : Geo<NQ>::smem_bytes;
    static int per_sm = 0;
    if (!per_sm) {
        cudaFuncSetAttribute(k_certify<NQ, VONLY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_certify<NQ, VONLY>, Geo<NQ>::THREADS, smem);
        per_sm = b > 0 ? b : 1;
    }
    const size_t cap = (size_t)num_sms() * (size_t)per_sm;
    size_t grid = (a.count + Geo<NQ>::WALKS - 1) / Geo<NQ>::WALKS;
    if (grid > cap) grid = cap;
    k_certify<NQ, VONLY><<<(unsigned)grid, Geo<NQ>::THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t certify_n(const CertArgs &a, cudaStream_t s)
{
    if constexpr (NQ == 4)
        if (a.side == 1 && a.lv.Cm) return launch_certify_e4(a, s);
    if constexpr (NQ >= 3)
        return a.side == 0 ? launch_certify_v(a, s) : certify_nv<NQ, false>(a, s);
    else
        return a.side == 0 ? certify_nv<NQ, true>(a, s) : certify_nv<NQ, false>(a, s);
}

} // namespace

cudaError_t launch_certify(const CertArgs &a, cudaStream_t s)
{
    if (a.count == 0) return cudaSuccess;
    switch (a.lv.n) {
    case 1: return certify_n<1>(a, s);
    case 2: return certify_n<2>(a, s);
    case 3: return certify_n<3>(a, s);
    case 4: return certify_n<4>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

int num_sms()
{
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    return g_num_sms;
}

int lanes_per_walk(int n) { return n == 4 ? Geo<4>::LPW : n == 3 ? Geo<3>::LPW : n == 2 ? Geo<2>::LPW : Geo<1>::LPW; }

int launch_shapes(int n) { return n == 4 ? shape_count(4) : n == 3 ? shape_count(3) : shape_count(2); }

int shape_warps_of(int n, int shape) { return n == 4 && shape == 3 ? engine4_warps() : shape_warps(n, shape); }

int shape_min_blocks_of(int n, int shape) { return shape_min_blocks(n, shape); }

int walks_per_task(int n, int shape) { return shape_warps(n, shape) * (32 / lanes_per_walk(n)); }

int walk_blocks_per_sm(int n)
{
    switch (n) {
    case 1: return blocks_per_sm<1>();
    case 2: return blocks_per_sm<2>();
    case 3: return blocks_per_sm<3>();
    default: return blocks_per_sm<4>();
    }
}

cudaError_t launch_walk_step(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp,
                             size_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    switch (lv.n) {
    case 1: return walk_step_n<1>(lv, chunk, in, out, is_dp, count, s);
    case 2: return walk_step_n<2>(lv, chunk, in, out, is_dp, count, s);
    case 3: return walk_step_n<3>(lv, chunk, in, out, is_dp, count, s);
    case 4: return walk_step_n<4>(lv, chunk, in, out, is_dp, count, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_init_walks(const WalkLaunch &w, cudaStream_t s)
{
    if (w.n_walks > 0) k_init_walks<<<(w.n_walks + 255) / 256, 256, 0, s>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_operand(int n, const uint2 *C32, uint16_t *Cm, cudaStream_t s)
{
    const unsigned blocks = (2u << (4 * n)) / 256;
    if (n == 2) k_operand<2><<<blocks, 256, 0, s>>>(C32, Cm);
    else if (n == 3) k_operand<3><<<blocks, 256, 0, s>>>(C32, Cm);
    else if (n == 4) k_operand<4><<<blocks, 256, 0, s>>>(C32, Cm);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_insert_points(const WalkLaunch &w, const Slot *pts, uint32_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    const unsigned grid = (unsigned)std::min<uint64_t>(((uint64_t)count + 255) / 256, (uint64_t)num_sms() * 8);
    k_insert_points<<<grid, 256, 0, s>>>(w, pts, count);
    return cudaGetLastError();
}

cudaError_t launch_bin_owners(const Slot *in, uint32_t count, uint32_t n_owners, Slot *out, uint32_t *counts,
                              cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    if (n_owners == 0 || n_owners > 1024) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)std::min<uint64_t>(((uint64_t)count + 255) / 256, (uint64_t)num_sms() * 8);
    k_count_owners<<<grid, 256, 0, s>>>(in, count, n_owners, counts);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the scatter's fill cursors sit right after the counts
    e = cudaMemsetAsync(counts + n_owners, 0, sizeof(uint32_t) * n_owners, s);
    if (e != cudaSuccess) return e;
    k_scatter_owners<<<grid, 256, sizeof(uint32_t) * n_owners, s>>>(in, count, n_owners, counts,
                                                                   counts + n_owners, out);
    return cudaGetLastError();
}

cudaError_t launch_walks(const WalkLaunch &w, cudaStream_t s)
{
    switch (w.lv.n) {
    case 1: return walks_n<1>(w, s);
    case 2: return walks_n<2>(w, s);
    case 3: return walks_n<3>(w, s);
    case 4: return walks_n<4>(w, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_rewalk_pairs(const WalkLaunch &w, cudaStream_t s)
{
    switch (w.lv.n) {
    case 1: return rewalk_pairs_n<1>(w, s);
    case 2: return rewalk_pairs_n<2>(w, s);
    case 3: return rewalk_pairs_n<3>(w, s);
    case 4: return rewalk_pairs_n<4>(w, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_walks_batch(int n, int shape, const BatchArgs &a, cudaStream_t s)
{
    switch (n) {
    case 1: return walks_batch_n<1>(shape, a, s);
    case 2: return walks_batch_n<2>(shape, a, s);
    case 3: return walks_batch_n<3>(shape, a, s);
    case 4: return walks_batch_n<4>(shape, a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_rewalk_batch(int n, const BatchArgs &a, cudaStream_t s)
{
    switch (n) {
    case 1: return rewalk_batch_n<1>(a, s);
    case 2: return rewalk_batch_n<2>(a, s);
    case 3: return rewalk_batch_n<3>(a, s);
    case 4: return rewalk_batch_n<4>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_rewalk_arrays(const LevelCtx &lv, int chunk, const uint64_t *sa, const uint32_t *la,
                                 const uint64_t *sb, const uint32_t *lb, size_t count, int32_t *cls, uint64_t *ab,
                                 cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    switch (lv.n) {
    case 1: return rewalk_arrays_n<1>(lv, chunk, sa, la, sb, lb, count, cls, ab, s);
    case 2: return rewalk_arrays_n<2>(lv, chunk, sa, la, sb, lb, count, cls, ab, s);
    case 3: return rewalk_arrays_n<3>(lv, chunk, sa, la, sb, lb, count, cls, ab, s);
    case 4: return rewalk_arrays_n<4>(lv, chunk, sa, la, sb, lb, count, cls, ab, s);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace qcs
