// qcs_certify.cu -- the V products of the exhaustive level pass (CertArgs),
// n = 3 and 4.
//
// A V point's index has its first rotation r_1 as the lowest base-xi digit,
// and r_1 is the last stage that the weights go through: xi consecutive
// points share all stages but the last.  So a warp forms the weights before
// the last stage once per unit of 32 points, whose r_1 share their t part (at
// n = 3: four t parts of eight), and per point only the last stage, of which
// the fingerprints need one part, and its column finalisers remain.  Of those
// the columns that commute with r_1 have the same fingerprints for every r_1:
// their finalisers are formed once per unit, and a point adds a class's sum.
// Except where r_1 has no last-qubit part (a quarter of them) exactly half of
// a lane's columns commute, which half by one bit per lane.  The lanes'
// partial sums of the unit's 32 points go through shared memory, so that one
// lane sums, inserts or probes one point.
//
// What bounds it: issue, about 140 warp instructions a point (881 when every
// point went through all stages and all finalisers on its own, and its key was
// probed by one lane).
#include <cuda_runtime.h>

#include <cstdint>

#include "qcs_device.cuh"
#include "qcs_internal.h"
#include "qcs_rows.cuh"

namespace qcs {
namespace {

namespace cv {
constexpr int kWarps = 24, kThreads = 32 * kWarps;
template <int NQ>
struct Geo {
    static constexpr int LB = 2 * NQ - 3, S = 1 << LB;      // lanes of a point
    static constexpr uint32_t XI = (1u << (2 * NQ)) - 1;
    static constexpr int UNITS = 8 * S / 32;                // units of 32 codes in a block of xi points
    static constexpr int PTS = 32 / S;                      // t parts in a unit
    static constexpr size_t off_sum = sizeof(uint32_t) * (2u << LB) * S; // after V's stage table
    static constexpr size_t sum_pitch = S + 1;              // odd: a lane's row and the lanes' columns without conflicts
    static constexpr size_t smem_bytes = off_sum + sizeof(uint64_t) * kWarps * 32 * sum_pitch;
};
} // namespace cv

// the last qubit's share of lambda for row t and t part PT
__host__ __device__ constexpr int share(int PT, int t)
{
    return lambda1((PT >> 2) & 1, (PT >> 1) & 1, (t >> 2) & 1, (t >> 1) & 1);
}
// the two rows t of x bit x whose share is even (ODD: odd)
__host__ __device__ constexpr int class_row(int PT, int x, bool ODD, int k)
{
    for (int t = x; t < 8; t += 2)
        if (((share(PT, t) & 1) != 0) == ODD && k-- == 0) return t;
    return 0;
}

// The points r_1 = (t part PT, every lane part) of one prefix: partial sums
// to sums[point][lane].  p: the part that is hashed, com: its value on rows
// that commute with r_1 (both before the last stage, scaled).
template <int NQ, int PT>
__device__ __forceinline__ void points(const uint32_t (&p)[8], const uint32_t (&com)[8], const uint32_t *tab,
                                       const HashBase &hb, int lane, uint64_t *sums)
{
    using G = cv::Geo<NQ>;
    constexpr bool kClasses = (PT >> 1) != 0; // r_1 has a last-qubit part
    const int l = lane & (G::S - 1), grp = lane >> G::LB;
    // finalisers of the commuting values, by x bit and class (no classes: all four rows)
    uint64_t sum_e[2], sum_o[2] = {0, 0};
#pragma unroll
    for (int x = 0; x < 2; x++) {
        sum_e[x] = 0;
#pragma unroll
        for (int k = 0; k < (kClasses ? 2 : 4); k++) {
            const int te = kClasses ? class_row(PT, x, false, k) : x + 2 * k;
            const uint64_t e = column_hash(com[te], hb.PH, hb.pre16);
            sum_e[x] += te == 0 && l == 0 ? 0ull : e; // column 0, the identity, does not enter
            if (kClasses) sum_o[x] += column_hash(com[class_row(PT, x, true, k)], hb.PH, hb.pre16);
        }
    }
#pragma unroll 1
    for (int i = grp; i < G::S; i += G::PTS) { // the lane part
        const uint32_t w = tab[(((uint32_t)(PT & 1) << G::LB | (uint32_t)i) << G::LB) + l];
        uint32_t v[8];
#pragma unroll
        for (int t = 0; t < 8; t++) v[t] = __shfl_xor_sync(0xFFFFFFFFu, p[t ^ PT], i);
        uint64_t acc = 0;
#pragma unroll
        for (int x = 0; x < 2; x++) {
            const uint32_t s = (uint32_t)(int)(int8_t)(w >> (8 * x));
            const bool odd = ((w >> (16 + 8 * x)) & 1u) != 0;
            if (kClasses) {
                // odd: the rows of even share anticommute, the others commute
                acc += odd ? sum_o[x] : sum_e[x];
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const int te = class_row(PT, x, false, k), to = class_row(PT, x, true, k);
                    const uint32_t u = odd ? p[te] : p[to], q = odd ? v[te] : v[to];
                    const uint32_t sg = share(PT, to) == 3 ? (odd ? s : 0u - s) : s;
                    acc += column_hash(u + q * sg, hb.PH, hb.pre16);
                }
            } else if (odd) {
#pragma unroll
                for (int k = 0; k < 4; k++)
                    acc += column_hash(p[x + 2 * k] + v[x + 2 * k] * s, hb.PH, hb.pre16);
            } else {
                acc += sum_e[x];
            }
        }
        sums[(size_t)i * G::sum_pitch + l] = acc;
        __syncwarp();
    }
}

template <int NQ>
__global__ void __launch_bounds__(cv::kThreads, 1) k_certify_v(CertArgs a)
{
    using G = cv::Geo<NQ>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *tab = reinterpret_cast<uint32_t *>(smem_raw);
    for (uint32_t i = threadIdx.x; i < (2u << G::LB) * G::S; i += cv::kThreads)
        tab[i] = stage_word<NQ>(0, i >> G::LB, i & (G::S - 1));
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    const int l = lane & (G::S - 1);
    uint64_t *sums = reinterpret_cast<uint64_t *>(smem_raw + G::off_sum) + (size_t)warp * 32 * G::sum_pitch;
    const HashBase hb = hash_base(a.base);
    const int h = a.lv.h, ev = a.lv.ev, sh = (ev >> 1) < 31 ? ev >> 1 : 31;
    // units of the blocks that [first, first + count) touches, an equal
    // contiguous share to each warp
    const uint64_t b0 = a.first / G::XI, blocks = (a.first + a.count - 1) / G::XI - b0 + 1;
    const uint64_t units = blocks * G::UNITS, warps = (uint64_t)gridDim.x * cv::kWarps;
    const uint64_t me = (uint64_t)blockIdx.x * cv::kWarps + (uint64_t)warp;
    const uint64_t end = units * (me + 1) / warps;
    uint32_t stored = 0;
    for (uint64_t u = units * me / warps; u < end; u++) {
        const uint64_t block = b0 + u / G::UNITS;
        const uint32_t part = (uint32_t)(u % G::UNITS);
        // the stages before the last: r_h (the block's highest digit) down to
        // r_2, a code per byte
        uint64_t seq = 0, d = block;
        for (int j = 2; j <= h; j++) {
            seq = seq << 8 | codes_of<NQ>((uint32_t)(d % G::XI) + 1);
            d /= G::XI;
        }
        uint32_t ua[8], ub[8];
        first_stage<NQ>(a.lv.T4[0], (uint32_t)seq & 0xFFu, l, ua, ub);
#pragma unroll 1
        for (int j = 3; j <= h; j++) {
            seq >>= 8;
            stage<NQ>((uint32_t)seq & 0xFFu, 0, tab, l, ua, ub);
        }
        // the fingerprint is the a part after the scaling by sqrt2^ev: an odd
        // ev takes it from the b part
        uint32_t p[8], com[8];
#pragma unroll
        for (int t = 0; t < 8; t++) {
            p[t] = ((ev & 1) ? ub[t] : ua[t]) << sh;
            com[t] = ((ev & 1) ? ua[t] << 1 : ub[t]) << sh;
        }
        uint32_t q; // the lane's own point: its first rotation
        if (NQ == 4) {
            switch (part) {
            case 0: points<NQ, 0>(p, com, tab, hb, lane, sums); break;
            case 1: points<NQ, 1>(p, com, tab, hb, lane, sums); break;
            case 2: points<NQ, 2>(p, com, tab, hb, lane, sums); break;
            case 3: points<NQ, 3>(p, com, tab, hb, lane, sums); break;
            case 4: points<NQ, 4>(p, com, tab, hb, lane, sums); break;
            case 5: points<NQ, 5>(p, com, tab, hb, lane, sums); break;
            case 6: points<NQ, 6>(p, com, tab, hb, lane, sums); break;
            default: points<NQ, 7>(p, com, tab, hb, lane, sums); break;
            }
            q = row_of(NQ, (uint32_t)lane, part);
        } else {
            constexpr size_t step = (size_t)G::S * G::sum_pitch; // the points of one t part
            if (part == 0) {
                points<NQ, 0>(p, com, tab, hb, lane, sums);
                points<NQ, 1>(p, com, tab, hb, lane, sums + step);
                points<NQ, 2>(p, com, tab, hb, lane, sums + 2 * step);
                points<NQ, 3>(p, com, tab, hb, lane, sums + 3 * step);
            } else {
                points<NQ, 4>(p, com, tab, hb, lane, sums);
                points<NQ, 5>(p, com, tab, hb, lane, sums + step);
                points<NQ, 6>(p, com, tab, hb, lane, sums + 2 * step);
                points<NQ, 7>(p, com, tab, hb, lane, sums + 3 * step);
            }
            q = row_of(NQ, (uint32_t)lane & (G::S - 1), part * G::PTS + ((uint32_t)lane >> G::LB));
        }
        __syncwarp();
        uint64_t acc = 0;
#pragma unroll
        for (int j = 0; j < G::S; j++) acc += sums[(size_t)lane * G::sum_pitch + j];
        __syncwarp();
        const uint64_t idx = block * G::XI + (q - 1);
        const bool valid = q != 0 && idx >= a.first && idx - a.first < a.count;
        uint64_t key = smix(acc);
        if (key == ~0ull) key = ~0ull - 1; // ~0 marks an empty slot
        const uint32_t all = all_lanes(); // not kept: a register less in the loops
        if (a.insert) cert_insert_warp(a, all, valid, key, idx, lane, stored);
        else if (valid) cert_probe(a, key, idx);
        __syncwarp(all);
    }
    stored = __reduce_add_sync(all_lanes(), stored);
    if (lane == 0) cert_count(a, stored);
}

template <int NQ>
cudaError_t certify_v_n(const CertArgs &a, cudaStream_t s)
{
    using G = cv::Geo<NQ>;
    const cudaError_t e =
        cudaFuncSetAttribute(k_certify_v<NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::smem_bytes);
    if (e != cudaSuccess) return e;
    const uint64_t units = (a.count / G::XI + 2) * G::UNITS, ctas = (units + cv::kWarps - 1) / cv::kWarps;
    const uint64_t sms = (uint64_t)num_sms();
    k_certify_v<NQ><<<(unsigned)(ctas < sms ? ctas : sms), cv::kThreads, G::smem_bytes, s>>>(a);
    return cudaGetLastError();
}

} // namespace

cudaError_t launch_certify_v(const CertArgs &a, cudaStream_t s)
{
    if (a.count == 0) return cudaSuccess;
    return a.lv.n == 4 ? certify_v_n<4>(a, s) : a.lv.n == 3 ? certify_v_n<3>(a, s) : cudaErrorInvalidValue;
}

} // namespace qcs
