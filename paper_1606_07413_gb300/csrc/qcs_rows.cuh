// qcs_rows.cuh -- one point's weights on a few lanes: the row layout, the
// adjoint stages and the column finaliser, as the n = 4 engine
// (qcs_engine4.cu) and the exhaustive pass (qcs_certify.cu) use them.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "qcs_internal.h"

namespace qcs {
namespace {

// Rows and stages.
//
// A point's 4^n weight rows sit on 2^(2n - 3) lanes, eight on each: lane l
// holds row_of(n, l, t), t = 0 .. 7 (qcs_internal.h).  t carries the x bit of
// qubit n - 2 and qubit n - 1, the lane the rest, and a Pauli's code (codes_of)
// is laid out the same way: its low 2n - 3 bits are its lane part, the three
// above them its t part.  A stage takes row j to u_j +- u_{j^p} or to sqrt2 u_j, by
// lambda(p, j) in P(p) P(j) = i^lambda P(p^j), which is a sum over the qubits.
// So with the t part of p known at compile time (a switch over its eight
// values) the partner's register and the last qubit's share of lambda are constants,
// and what is left of lambda is one value per lane and x bit of qubit n - 2: a
// word of the stage table, which does not depend on p's last qubit.  About 88
// instructions a stage at n = 4; with the signs and selections looked up row
// by row it was 106.

__host__ __device__ constexpr int lambda1(int px, int pz, int x, int z)
{
    return (px * pz + x * z + 2 * pz * x - (px ^ x) * (pz ^ z)) & 3;
}

// lambda of the lane's rows but for the last qubit's share, for x bit 0, 1 of
// qubit n - 2: byte x is the sign (lambda 0 or 1: +1, 2 or 3: -1; for W the
// other way round), byte 2 + x whether lambda is odd.  code: the low 2n - 2
// bits of the Pauli's code.
template <int NQ>
__device__ __forceinline__ uint32_t stage_word(uint32_t side, uint32_t code, uint32_t l)
{
    // lane bits: z_0 .. z_(n-2), x_0 .. x_(n-3); code bits: the same, then x_(n-2)
    int v = 0;
#pragma unroll
    for (int q = 0; q < NQ - 2; q++)
        v += lambda1((code >> (NQ - 1 + q)) & 1, (code >> q) & 1, (l >> (NQ - 1 + q)) & 1, (l >> q) & 1);
    uint32_t w = 0;
#pragma unroll
    for (int x = 0; x < 2; x++) {
        const uint32_t a =
            (uint32_t)(v + lambda1((code >> (2 * NQ - 3)) & 1, (code >> (NQ - 2)) & 1, x, (l >> (NQ - 2)) & 1)) & 3u;
        w |= (((a >> 1) ^ side) ? 0xFFu : 1u) << (8 * x) | (a & 1u) << (16 + 8 * x);
    }
    return w;
}

// (na, nb) = ODD == (odd != 0) ? (ub, 2 ua) : (ua + s va, ub + s vb)
template <bool ODD>
__device__ __forceinline__ void row_update(uint32_t &ua, uint32_t &ub, uint32_t va, uint32_t vb, uint32_t s,
                                           uint32_t odd)
{
    uint32_t na, nb;
    if (ODD)
        asm("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %7, 0;\n\tmov.b32 %0, %5;\n\tadd.u32 %1, %4, %4;\n\t"
            "@p mad.lo.u32 %0, %2, %6, %4;\n\t@p mad.lo.u32 %1, %3, %6, %5;\n\t}"
            : "=&r"(na), "=&r"(nb)
            : "r"(va), "r"(vb), "r"(ua), "r"(ub), "r"(s), "r"(odd));
    else
        asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %7, 0;\n\tmov.b32 %0, %5;\n\tadd.u32 %1, %4, %4;\n\t"
            "@p mad.lo.u32 %0, %2, %6, %4;\n\t@p mad.lo.u32 %1, %3, %6, %5;\n\t}"
            : "=&r"(na), "=&r"(nb)
            : "r"(va), "r"(vb), "r"(ua), "r"(ub), "r"(s), "r"(odd));
    ua = na;
    ub = nb;
}

// the stage of a Pauli whose t part is PT; s, odd: the lane's sign and parity
// of lambda per x bit of qubit n - 2, without the last qubit's share
template <int PT>
__device__ __forceinline__ void stage_rows(uint32_t (&ua)[8], uint32_t (&ub)[8], int pl, const int (&s)[2],
                                           const uint32_t (&odd)[2])
{
    uint32_t va[8], vb[8];
#pragma unroll
    for (int t = 0; t < 8; t++) {
        va[t] = __shfl_xor_sync(0xFFFFFFFFu, ua[t ^ PT], pl);
        vb[t] = __shfl_xor_sync(0xFFFFFFFFu, ub[t ^ PT], pl);
    }
    const int neg[2] = {-s[0], -s[1]};
#pragma unroll
    for (int t = 0; t < 8; t++) {
        // the last qubit's share of lambda: 0, 1 or 3 (3: the sign turns)
        const int x2 = t & 1, c = lambda1((PT >> 2) & 1, (PT >> 1) & 1, (t >> 2) & 1, (t >> 1) & 1);
        const uint32_t sg = (uint32_t)(c == 3 ? neg[x2] : s[x2]);
        if (c & 1) row_update<true>(ua[t], ub[t], va[t], vb[t], sg, odd[x2]);
        else row_update<false>(ua[t], ub[t], va[t], vb[t], sg, odd[x2]);
    }
}

// side: 0 for V (adjoint of R^), 1 for W (adjoint of R^T); tab: stage_word
// [side][code][lane]; code is the same on the whole warp
template <int NQ>
__device__ __forceinline__ void stage(uint32_t code, uint32_t side, const uint32_t *tab, int lane, uint32_t (&ua)[8],
                                      uint32_t (&ub)[8])
{
    constexpr int LB = 2 * NQ - 3; // lane bits
    const uint32_t w = tab[((side << (LB + 1) | (code & ((2u << LB) - 1u))) << LB) + lane];
    const int pl = (int)(code & ((1u << LB) - 1u));
    const int s[2] = {(int)(int8_t)w, (int)(int8_t)(w >> 8)};
    const uint32_t odd[2] = {w & 0xFF0000u, w & 0xFF000000u};
    switch (code >> LB) {
    case 0: stage_rows<0>(ua, ub, pl, s, odd); break;
    case 1: stage_rows<1>(ua, ub, pl, s, odd); break;
    case 2: stage_rows<2>(ua, ub, pl, s, odd); break;
    case 3: stage_rows<3>(ua, ub, pl, s, odd); break;
    case 4: stage_rows<4>(ua, ub, pl, s, odd); break;
    case 5: stage_rows<5>(ua, ub, pl, s, odd); break;
    case 6: stage_rows<6>(ua, ub, pl, s, odd); break;
    default: stage_rows<7>(ua, ub, pl, s, odd); break;
    }
}

constexpr uint64_t kC1 = 0xBF58476D1CE4E5B9ull, kC2 = 0x94D049BB133111EBull; // SplitMix64's finaliser

// smix(base ^ phi) of one column, phi the sign-folded low 16 bits of l, given
// pre = base ^ (base >> 30) as PH = (pre & ~0xFFFF) * kC1 and pre16 = pre &
// 0xFFFF: (pre ^ phi) * kC1 = PH + (pre16 ^ phi) * kC1, and the second
// product has a 16-bit factor.
__device__ __forceinline__ uint64_t column_hash(uint32_t l, uint64_t PH, uint32_t pre16)
{
    const int s = (int)(int16_t)(uint16_t)l;
    const uint32_t x = (uint32_t)abs(s) ^ pre16;
    uint64_t z = (uint64_t)x * (uint32_t)kC1 + PH;
    z += (uint64_t)(x * (uint32_t)(kC1 >> 32)) << 32;
    z = (z ^ (z >> 27)) * kC2;
    return z ^ (z >> 31);
}

struct alignas(16) HashBase {
    uint64_t PH;         // (pre with its low 16 bits clear) * kC1
    uint32_t pre16, pad; // the low 16 bits of pre
};

__device__ __forceinline__ HashBase hash_base(uint64_t base)
{
    const uint64_t pre = base ^ (base >> 30);
    return HashBase{(pre & ~0xFFFFull) * kC1, (uint32_t)pre & 0xFFFFu, 0};
}

// the weights after the first stage of a point (LevelCtx::T4), as two 16-byte
// loads; the upper halves of ua are never looked at (every sum is mod 2^16)
template <int NQ>
__device__ __forceinline__ void first_stage(const uint4 *tab, uint32_t code, int lane, uint32_t (&ua)[8],
                                            uint32_t (&ub)[8])
{
    const uint4 w0 = __ldg(tab + ((code << (2 * NQ - 3)) + lane) * 2), w1 = __ldg(tab + ((code << (2 * NQ - 3)) + lane) * 2 + 1);
    ua[0] = w0.x; ua[1] = w0.y; ua[2] = w0.z; ua[3] = w0.w;
    ua[4] = w1.x; ua[5] = w1.y; ua[6] = w1.z; ua[7] = w1.w;
#pragma unroll
    for (int t = 0; t < 8; t++) ub[t] = ua[t] >> 16;
}

// Pauli codes (row_of's bit order) of four Pauli indices, one per byte
template <int NQ>
__device__ __forceinline__ uint32_t codes_of(uint32_t q)
{
    if (NQ == 4) return (q & 0x87878787u) | ((q >> 1) & 0x38383838u) | ((q << 3) & 0x40404040u);
    // n = 3: z0 z1 z2 x0 x1 x2 -> z0 z1 x0 x1 z2 x2
    return (q & 0x23232323u) | ((q >> 1) & 0x0C0C0C0Cu) | ((q << 2) & 0x10101010u);
}

} // namespace
} // namespace qcs
