// qcs_quad.cu -- n = 2 and 3: the walk step of eight walks on one warp, four
// lanes (a quad) to a walk, with the contraction by mma.sync.
//
// A quad holds a walk's 4^n fingerprint weights, 4^n / 4 rows to a lane: lane
// q is qubit 0 (z0 | x0 << 1), the rows of a lane are the other qubits.  One
// step:
//  - the weights after the first stage come from a table in shared memory;
//  - a further stage exchanges the rows through shared memory, one word (both
//    parts) a row; the partner of row t is row t ^ p_T of lane q ^ p_L, at a
//    bank of its own lane, so there are no conflicts.  The stage tables give
//    each row's sign and which rows anticommute, per Pauli and lane.
//    V and W walks run the same stages: where W has the chunk's, V takes the
//    identity's, which scales by sqrt2 as its scaling to the level's exponent
//    asks for once anyway;
//  - the contraction is D = A B (m16n8k16, f16 inputs, f32 sums): A holds C^'s
//    columns (fragments in shared memory), B the eight walks' weights as byte
//    planes.  In the lanes that own them the weights already have the B
//    fragment's layout: a k-step is four rows of every lane.  V's column
//    fingerprints are its weights themselves; they go through the same sums
//    by k-steps whose A is the identity, so that D holds every walk's
//    fingerprints in one layout.  W's weights are zero in those k-steps, V's in
//    the others;
//  - each lane hashes the columns it holds of two walks, the sums are exchanged
//    and the quad takes its walk's step.
// The exactness argument is the engine's (qcs_engine4.cu): a weight's byte is
// the f16 subnormal with those bits, and row 0's first k slot puts 0.75 on
// every sum.
//
// What bounds it: issue.  A step costs 145 warp instructions at n = 3 and about
// 50 at n = 2 (379 and 325 with one and two walks to a warp, whose bookkeeping
// ran on all lanes of each).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "qcs_device.cuh"
#include "qcs_internal.h"
#include "qcs_rows.cuh"

namespace qcs {
namespace {

namespace qd {

template <int NQ>
struct Geo {
    static constexpr int D = 1 << (2 * NQ), R = D / 4; // rows of a lane
    static constexpr int KS = R / 4;                   // k-steps of one part
    static constexpr int MT = D / 16;                  // tiles of 16 columns of C^ (as many as KS)
    static constexpr uint32_t XI = D - 1;
    static constexpr int kWarps = NQ == 3 ? 18 : 24, kThreads = 32 * kWarps; // at most
    // shared memory
    static constexpr size_t off_T = sizeof(uint4) * 32 * MT * 2 * KS;     // after C^'s fragments [tile][part, k-step][lane]
    static constexpr size_t off_stage = off_T + sizeof(uint4) * 2 * D * KS * 4; // T: [side][code][k-step][q], four rows
    static constexpr size_t off_anti = off_stage + (size_t)2 * D * 4 * R; // stage: i8 [side][code][q][row]
    static constexpr size_t off_base = off_anti + sizeof(uint32_t) * D * 4; // anti: u32 [code][q], a bit per row
    static constexpr size_t off_x = off_base + sizeof(HashBase) * D;      // HashBase [chunk]
    static constexpr size_t x_warp = sizeof(uint32_t) * 32 * R;           // exchange: u32 [row][lane] per warp
    static constexpr size_t smem_bytes(int warps) { return off_x + x_warp * (size_t)warps; }
};

// the batched kernels: 16 warps, so that nothing spills (n = 3, 12 jobs a round: 24 warps 0.58 ms, 20 0.49, 16 0.46, 12 0.55)
constexpr int kBatchWarps = 16, kBatchThreads = 32 * kBatchWarps, kTaskWalks = 16;

// the lane and row parts of a Pauli's code (row_of's order), as quad_row splits them
template <int NQ>
__device__ __forceinline__ uint32_t code_lane(uint32_t code) // p_L
{
    return NQ == 2 ? code & 3u : (code & 1u) | ((code >> 1) & 2u);
}
template <int NQ>
__device__ __forceinline__ uint32_t code_rows(uint32_t code) // p_T
{
    return NQ == 2 ? code >> 2 : code >> 3 | (code & 2u) << 2;
}
template <int NQ>
__device__ __forceinline__ uint32_t codes(uint32_t q) // of four Pauli indices, one per byte
{
    // n = 2: z0 z1 x0 x1 -> z0 x0 z1 x1
    if (NQ == 2) return (q & 0x09090909u) | ((q >> 1) & 0x02020202u) | ((q << 1) & 0x04040404u);
    return codes_of<3>(q);
}
template <int NQ>
struct Sm {
    const uint4 *frag, *T;
    const unsigned char *stage;
    const uint32_t *anti;
    const HashBase *base;
    uint32_t *x; // this warp's exchange rows
};

// C^'s fragments, the first-stage and stage tables and the chunks' hash bases
// of a level (scale: Level::scale); every thread calls it, a barrier at its
// end.
template <int NQ>
__device__ __forceinline__ Sm<NQ> set_up(const LevelCtx &lv, int scale, unsigned char *raw)
{
    using G = Geo<NQ>;
    uint4 *frag = reinterpret_cast<uint4 *>(raw), *T = reinterpret_cast<uint4 *>(raw + G::off_T);
    HashBase *base = reinterpret_cast<HashBase *>(raw + G::off_base);
    constexpr int nFrag = (int)(G::off_T / sizeof(uint4));
#pragma unroll 4
    for (int i = threadIdx.x; i < nFrag; i += blockDim.x) frag[i] = __ldg(lv.Cm + i);
    constexpr int nT = 2 * G::D * G::KS * 4, nAll = (int)((G::off_base - G::off_T) / sizeof(uint4));
#pragma unroll 4
    for (int i = threadIdx.x; i < nAll; i += blockDim.x) {
        uint4 v = __ldg(lv.quad + i);
        if (i < nT / 2) { // V's scaling by sqrt2^scale commutes with the stages: (a, b) -> (b, 2 a) each
            auto scaled = [&](uint32_t w) {
                const uint32_t a = w & 0xFFFFu, b = w >> 16;
                const int sh = scale >> 1;
                return (scale & 1) ? (shl32(b, sh) & 0xFFFFu) | shl32(a, sh + 1) << 16
                                   : (shl32(a, sh) & 0xFFFFu) | shl32(b, sh) << 16;
            };
            v = make_uint4(scaled(v.x), scaled(v.y), scaled(v.z), scaled(v.w));
        }
        T[i] = v;
    }
    // base(chunk) = smix(smix(seed_H ^ version) ^ (n | k << 8 | chunk << 16 | K << 32))
    const uint64_t vmix = smix(kSeedH ^ (uint64_t)lv.version);
    for (int i = threadIdx.x; i < G::D; i += blockDim.x) {
        const uint64_t tag =
            (uint64_t)lv.n | ((uint64_t)lv.k << 8) | ((uint64_t)i << 16) | ((uint64_t)(uint32_t)lv.K << 32);
        base[i] = hash_base(smix(vmix ^ tag));
    }
    __syncthreads();
    return Sm<NQ>{frag,
                  T,
                  raw + G::off_stage,
                  reinterpret_cast<const uint32_t *>(raw + G::off_anti),
                  base,
                  reinterpret_cast<uint32_t *>(raw + G::off_x + G::x_warp * (threadIdx.x >> 5))};
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint4 &a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// One row of a stage, in place: (ua + m va, ub + m vb) where the row
// anticommutes with the Pauli, else (ub, 2 ua), which m = 1 and the
// differences ub - ua and 2 ua - ub in place of the partner give.  (With the
// result in registers of its own, as in qcs_rows.cuh, the stage loop moves 32
// of them back: 928 against 896 us for 2^16 walks x 64 steps at n = 3.)
__device__ __forceinline__ void row_step(uint32_t &ua, uint32_t &ub, uint32_t va, uint32_t vb, uint32_t m,
                                         uint32_t anti)
{
    asm("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %5, 0;\n\t@p sub.u32 %2, %1, %0;\n\t@p sub.u32 %3, %0, %2;\n\t"
        "mad.lo.u32 %0, %2, %4, %0;\n\tmad.lo.u32 %1, %3, %4, %1;\n\t}"
        : "+r"(ua), "+r"(ub), "+r"(va), "+r"(vb)
        : "r"(m), "r"(anti));
}

// What a level asks of every point (all walks of a warp run the same number
// of stages): V takes q_h .. q_1, then for odd k the identity; W q_1 .. q_h,
// then the chunk.  A V product of fewer than two rotations starts from code
// 0, the untouched weights (its half product then is not one lookup), and so
// does W unless that makes up for the chunk.
template <int NQ>
struct Level {
    int h, ns, sh_v, sh_w, sh_c;
    int scale; // V's remaining power of sqrt2 (it is in the first-stage table)
    uint32_t ell, fmask, mask_lo; // mask_lo: the bytes of up to four rotations
    int sh_rev;
    __device__ __forceinline__ explicit Level(const LevelCtx &lv)
    {
        h = lv.h;
        const int k1 = lv.k & 1, lead_v = h < 2 ? 1 : 0, lead_w = h == 0 || (h == 1 && !k1) ? 1 : 0;
        ns = h + lead_w + k1;
        sh_v = 8 * lead_v;
        sh_w = 8 * lead_w;
        sh_c = 8 * (h + lead_w);
        scale = lv.ev - (h + lead_v < ns ? 1 : 0); // one by V's identity stage
        ell = (uint32_t)lv.ell;
        fmask = lv.fmask;
        mask_lo = h == 0 ? 0u : h >= 4 ? ~0u : (1u << (8 * h)) - 1u;
        sh_rev = h == 0 || h > 4 ? 0 : 32 - 8 * h;
    }
    __device__ __forceinline__ uint64_t chunk_code(uint32_t chunk) const { return (uint64_t)codes<NQ>(chunk) << sh_c; }
    // the stages of state x, a code per byte (cc: its chunk's code in place).
    // The rotation fields are decode's.  Two or four of them are taken at once
    // and those past h masked off: a loop over them, each shifting the last
    // one's rest, took a quarter of an n = 2 step.
    __device__ __forceinline__ uint64_t seq(uint64_t x, uint64_t cc) const
    {
        const bool w = (x & 1) != 0;
        auto field = [&](int j) {
            return (((uint32_t)(x >> (1 + (int)ell * j)) & fmask) * Geo<NQ>::XI >> ell) + 1u;
        };
        uint32_t lo, hi = 0;
        if (h <= 2) {
            lo = (field(0) | field(1) << 8) & mask_lo;
        } else {
            lo = (field(0) | field(1) << 8 | field(2) << 16 | (h > 3 ? field(3) << 24 : 0u)) & mask_lo;
            for (int j = 4; j < h; j++) hi |= field(j) << (8 * (j - 4));
        }
        lo = codes<NQ>(lo);
        hi = codes<NQ>(hi);
        if (h <= 4) {
            // the bytes in reverse order for V; code 0 in front where it leads
            lo = w ? lo << sh_w : __byte_perm(lo, 0, 0x0123) >> sh_rev << sh_v;
        } else if (!w) {
            const uint64_t rev =
                ((uint64_t)__byte_perm(lo, 0, 0x0123) << 32 | __byte_perm(hi, 0, 0x0123)) >> (64 - 8 * h);
            lo = (uint32_t)rev;
            hi = (uint32_t)(rev >> 32);
        }
        const uint64_t r = (uint64_t)hi << 32 | lo;
        return w ? r | cc : r;
    }
};

// f of the quad's state x at its chunk (all lanes of a quad pass the same):
// the full 64-bit hash.  Whole warp.
template <int NQ>
__device__ __forceinline__ uint64_t step(uint64_t seq, int side, uint32_t chunk, const Level<NQ> &L, const Sm<NQ> &sm,
                                         int lane)
{
    using G = Geo<NQ>;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int g = lane >> 2, q = lane & 3;
    // hash bases of the walks whose columns this lane gets: 2q and 2q + 1
    const HashBase h0 = sm.base[__shfl_sync(kAll, chunk, 8 * q)], h1 = sm.base[__shfl_sync(kAll, chunk, 8 * q + 4)];
    uint32_t ua[G::R], ub[G::R];
    {
        const uint4 *t = sm.T + ((size_t)side * G::D + ((uint32_t)seq & 0xFFu)) * G::KS * 4 + q;
#pragma unroll
        for (int s = 0; s < G::KS; s++) {
            const uint4 w = t[4 * s];
            ua[4 * s] = w.x; ua[4 * s + 1] = w.y; ua[4 * s + 2] = w.z; ua[4 * s + 3] = w.w;
        }
#pragma unroll
        for (int t2 = 0; t2 < G::R; t2++) ub[t2] = ua[t2] >> 16; // ua's upper half is never looked at
    }
#pragma unroll 1
    for (int i = 1; i < L.ns; i++) {
        seq >>= 8;
        const uint32_t code = (uint32_t)seq & 0xFFu;
#pragma unroll
        for (int t = 0; t < G::R; t++) sm.x[t * 32 + lane] = __byte_perm(ua[t], ub[t], 0x5410);
        const unsigned char *ms = sm.stage + ((size_t)side * G::D + code) * 4 * G::R + (size_t)q * G::R;
        const uint32_t anti = sm.anti[code * 4 + (uint32_t)q];
        uint32_t m[G::KS];
        if (NQ == 3) {
            const uint4 v = *reinterpret_cast<const uint4 *>(ms);
            m[0] = v.x;
            m[G::KS > 1 ? 1 : 0] = v.y;
            m[G::KS > 2 ? 2 : 0] = v.z;
            m[G::KS > 3 ? 3 : 0] = v.w;
        } else {
            m[0] = *reinterpret_cast<const uint32_t *>(ms);
        }
        __syncwarp();
        const uint32_t at = code_rows<NQ>(code) * 32 + ((uint32_t)lane ^ code_lane<NQ>(code));
        uint32_t v[G::R];
#pragma unroll
        for (int t = 0; t < G::R; t++) v[t] = sm.x[at ^ (uint32_t)(t * 32)];
#pragma unroll
        for (int t = 0; t < G::R; t++)
            row_step(ua[t], ub[t], v[t], v[t] >> 16, (uint32_t)(int)(int8_t)(m[t / 4] >> (8 * (t % 4))),
                     anti & (1u << t));
        __syncwarp();
    }
    // the identity's fragment: columns g and g + 8 against k 2q, 2q + 1 (+ 8)
    const uint32_t one = g == 2 * q ? 0x00003C00u : g == 2 * q + 1 ? 0x3C000000u : 0u;
    const uint4 ident = make_uint4(one, 0, 0, one);
    // the weights as pairs of 16-bit words; V's a parts are its fingerprints
    const uint32_t bias = q == 0 ? 0x6400u : 0u; // row 0's slot of the first k-step
    const uint32_t mw = side ? 0x00FF00FFu : 0u, mv = ~mw & 0x00FF00FFu; // low bytes, or none
    const uint32_t sw = side ? 0x7351u : 0x7454u, sv = side ? 0x7454u : 0x7351u; // high bytes, or none
    uint32_t pa[G::R / 2], pb[G::R / 2];
#pragma unroll
    for (int t = 0; t < G::R; t += 2) {
        pa[t / 2] = __byte_perm(ua[t], ua[t + 1], 0x5410);
        pb[t / 2] = __byte_perm(ub[t], ub[t + 1], 0x5410);
    }
    float d[G::MT][2][4];
#pragma unroll
    for (int mt = 0; mt < G::MT; mt++)
#pragma unroll
        for (int r = 0; r < 8; r++) d[mt][r / 4][r % 4] = 0.f;
#pragma unroll
    for (int s = 0; s < 2 * G::KS; s++) {
        const uint32_t w0 = s < G::KS ? pa[2 * s] : pb[2 * (s - G::KS)];
        const uint32_t w1 = s < G::KS ? pa[2 * s + 1] : pb[2 * (s - G::KS) + 1];
        const uint32_t l0 = s == 0 ? (w0 & mw) | bias : w0 & mw, l1 = w1 & mw;
        const uint32_t u0 = __byte_perm(w0, s == 0 ? bias : 0u, sw), u1 = __byte_perm(w1, 0, sw);
#pragma unroll
        for (int mt = 0; mt < G::MT; mt++) {
            const uint4 a = sm.frag[(mt * 2 * G::KS + s) * 32 + lane];
            mma16816(d[mt][0], a, l0, l1);
            mma16816(d[mt][1], a, u0, u1);
        }
    }
#pragma unroll
    for (int mt = 0; mt < G::MT; mt++) {
        const uint32_t w0 = pa[2 * mt], w1 = pa[2 * mt + 1];
        mma16816(d[mt][0], ident, w0 & mv, w1 & mv);
        mma16816(d[mt][1], ident, __byte_perm(w0, 0, sv), __byte_perm(w1, 0, sv));
    }
    uint64_t s0 = 0, s1 = 0;
#pragma unroll
    for (int mt = 0; mt < G::MT; mt++) {
        // columns g (registers 0, 1) and g + 8 (2, 3) of the tile, walks 2q and 2q + 1
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const uint32_t l = __float_as_uint(d[mt][0][r]) + __float_as_uint(d[mt][1][r]) * 256u;
            uint64_t e = column_hash(l, (r & 1) ? h1.PH : h0.PH, (r & 1) ? h1.pre16 : h0.pre16);
            if (mt == 0 && r < 2 && g == 0) e = 0; // column 0, the identity, does not enter
            if (r & 1) s1 += e;
            else s0 += e;
        }
    }
    // even g keep walk 2q's sum, odd g 2q + 1's; then the sums over the lanes
    // of one parity, and each quad's from the lane that has it
    const bool odd = g & 1;
    uint64_t acc = (odd ? s1 : s0) + __shfl_xor_sync(kAll, odd ? s0 : s1, 4);
    acc += __shfl_xor_sync(kAll, acc, 8);
    acc += __shfl_xor_sync(kAll, acc, 16);
    return smix(__shfl_sync(kAll, acc, 4 * (g & 1) + (g >> 1)));
}

} // namespace qd

// Eight walks from `base` on (those below n), w.steps steps each.  The heads
// (lane 0 of a quad) keep the tallies, in 32 bits: a walk's are at most w.steps.
template <int NQ, typename WL>
__device__ __forceinline__ void walk_eight(const WL &w, uint32_t base, uint32_t n, const qd::Level<NQ> &L,
                                           const qd::Sm<NQ> &sm, int lane)
{
    const LevelCtx &lv = w.lv;
    const uint32_t local = base + (uint32_t)(lane >> 2), walk = w.walk_base + local;
    const bool valid = local < n, head = valid && (lane & 3) == 0;
    WalkState st{};
    if (valid) st = w.walks[local];
    TallyOf<uint32_t> t;
    uint64_t cc = L.chunk_code(st.chunk);
    const uint64_t dp_end = 1ull << lv.dshift, maskL = lv.maskL; // dshift < 64
    const uint32_t steps = w.steps, max_len = w.max_len;
    for (uint32_t s = 0; s < steps; s++) {
        const int side = (int)(st.cur & 1);
        const uint64_t y = qd::step<NQ>(L.seq(st.cur, cc), side, st.chunk, L, sm, lane) & maskL;
        t.w += (uint32_t)side;
        st.len++;
        st.cur = y;
        const bool is_dp = y < dp_end;
        if (is_dp || st.len >= max_len) {
            if (is_dp) {
                t.dp++;
                if (head) dp_insert(w, y, make_ref(walk, st.seq, st.len), t);
            } else {
                t.ab++;
            }
            new_trail<NQ>(st, walk, lv);
            if (head) w.walks[local].start = st.start; // written here, not kept
            cc = L.chunk_code(st.chunk);
        }
        __syncwarp();
    }
    if (head) {
        WalkState *d = &w.walks[local];
        d->cur = st.cur;
        d->len = st.len;
        d->chunk = st.chunk;
        d->seq = st.seq;
    }
    const uint32_t v[7] = {steps, t.w, t.dp, t.ab, t.evicted, t.duplicate, t.pairs};
    const int idx[7] = {C_STEPS, C_WSTEPS, C_DPS, C_ABANDONED, C_EVICTED, C_DUPLICATE, C_PAIRS};
#pragma unroll
    for (int i = 0; i < 7; i++) {
        unsigned long long sum = head ? v[i] : 0u;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (lane == 0 && sum) atomicAdd(&w.counters[idx[i]], sum);
    }
    __syncwarp();
}

template <int NQ>
__global__ void __launch_bounds__(qd::Geo<NQ>::kThreads, 1) k_walks_q(WalkLaunch w)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const qd::Level<NQ> L(w.lv);
    const qd::Sm<NQ> sm = qd::set_up<NQ>(w.lv, L.scale, smem_raw);
    const int lane = threadIdx.x & 31;
    const uint32_t n = (uint32_t)w.n_walks, warps = blockDim.x >> 5;
    for (uint32_t base = 8 * (blockIdx.x + gridDim.x * (threadIdx.x >> 5)); base < n; base += 8 * warps * gridDim.x)
        walk_eight<NQ>(w, base, n, L, sm, lane);
}

template <int NQ>
__global__ void __launch_bounds__(qd::Geo<NQ>::kThreads, 1) k_walk_step_q(LevelCtx lv, uint32_t chunk,
                                                                          const uint64_t *__restrict__ in,
                                                                          uint64_t *__restrict__ out,
                                                                          uint8_t *__restrict__ is_dp, size_t count)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const qd::Level<NQ> L(lv);
    const qd::Sm<NQ> sm = qd::set_up<NQ>(lv, L.scale, smem_raw);
    const int lane = threadIdx.x & 31;
    const size_t warps = blockDim.x >> 5;
    const uint64_t cc = (lv.k & 1) ? L.chunk_code(chunk) : 0ull;
    for (size_t base = 8 * (blockIdx.x + (size_t)gridDim.x * (threadIdx.x >> 5)); base < count;
         base += 8 * warps * gridDim.x) {
        const size_t i = base + (size_t)(lane >> 2);
        const uint64_t x = i < count ? in[i] : 0ull;
        const uint64_t y = qd::step<NQ>(L.seq(x, cc), (int)(x & 1), chunk, L, sm, lane) & lv.maskL;
        if (i < count && (lane & 3) == 0) {
            out[i] = y;
            if (is_dp) is_dp[i] = (uint8_t)((y >> lv.dshift) == 0);
        }
    }
}

// The re-walk of merges (Sec. 3, Fig. 2; the same steps and classes as
// rewalk_resume in qcs_walk.cu), eight at a time on a warp: each quad claims
// merges one after the other from `cursor` (device or shared memory) below cnt
// and evaluates f at one state an iteration: the longer trail until both are
// aligned, then a and b in turn.
template <int NQ, typename WL>
__device__ __forceinline__ void rewalk_eight(const WL &w, uint32_t *cursor, uint32_t cnt, const qd::Level<NQ> &L,
                                             const qd::Sm<NQ> &sm, int lane)
{
    const unsigned kAll = all_lanes(); // 2 % of an n = 3 search
    const LevelCtx &lv = w.lv;
    const bool head = (lane & 3) == 0;
    uint32_t cls[6] = {0, 0, 0, 0, 0, 0}, nf = 0, used = 0;
    uint64_t a = 0, b = 0, fa = 0, cc = 0;
    uint32_t la = 0, lb = 0, chunk = 0;
    bool active = false, second = false, checked = false, more = true;
    // whether the merge needs an evaluation; if not it is classified or carried
    auto settle = [&]() {
        if (la == lb) {
            if (second) return;
            if (!checked) {
                checked = true;
                if (a == b) {
                    cls[0]++; // Robin Hood
                    active = false;
                    return;
                }
            }
            if (lb == 0) {
                cls[5]++; // no merge
                active = false;
                return;
            }
        }
        if (w.rewalk_budget && used + (la > lb ? 0u : 1u) >= w.rewalk_budget) {
            if (head) carry_merge(w, a, la, b, lb, chunk);
            active = false;
        }
    };
    for (;;) {
        // a merge that needs an evaluation for every idle quad, as far as the
        // list goes; the quad's even lanes work out one trail's start and
        // chunk, its odd lanes the other's
        for (;;) {
            const bool need = more && !active;
            const uint32_t m = __ballot_sync(kAll, need && head);
            if (!m) break;
            uint32_t base = 0;
            if (lane == __ffs((int)m) - 1) base = atomicAdd(cursor, (uint32_t)__popc(m));
            base = __shfl_sync(kAll, base, __ffs((int)m) - 1);
            const uint32_t p = base + (uint32_t)__popc(m & ((1u << (lane & ~3)) - 1u));
            const bool got = need && p < cnt;
            if (need && !got) more = false;
            uint64_t s = 0;
            uint32_t ls = 0, cs = 0;
            if (got) {
                if (p < w.pend_in_n) {
                    const Pending q = w.pend_in[p];
                    s = (lane & 1) ? q.b : q.a;
                    ls = (lane & 1) ? q.lb : q.la;
                    cs = q.chunk;
                } else {
                    const Pair P = w.queue[p - w.pend_in_n];
                    uint32_t wi, si;
                    split_ref((lane & 1) ? P.ref_b : P.ref_a, wi, si, ls);
                    s = trail_start(lv, wi, si);
                    cs = trail_chunk<NQ>(lv, s);
                }
            }
            __syncwarp(kAll);
            const uint64_t o = __shfl_xor_sync(kAll, s, 1);
            const uint32_t lo = __shfl_xor_sync(kAll, ls, 1), co = __shfl_xor_sync(kAll, cs, 1);
            if (got) {
                if (cs != co || ls > kMaxRewalkLen || lo > kMaxRewalkLen) {
                    cls[5]++; // the same value reached in two chunks' functions, or too long: no merge
                } else {
                    // a is the longer trail (of equal ones, the first)
                    const bool mine = (lane & 1) ? ls > lo : ls >= lo;
                    a = mine ? s : o;
                    b = mine ? o : s;
                    la = max(ls, lo);
                    lb = min(ls, lo);
                    chunk = cs;
                    cc = L.chunk_code(chunk);
                    used = 0;
                    second = checked = false;
                    active = true;
                    settle();
                }
            }
            __syncwarp(kAll);
        }
        if (!__any_sync(kAll, active)) break;
        const uint64_t x = second ? b : a;
        const uint64_t y = qd::step<NQ>(L.seq(x, cc), (int)(x & 1), chunk, L, sm, lane) & lv.maskL;
        if (active) {
            used++;
            nf++;
            if (la > lb) {
                a = y;
                la--;
                settle();
            } else if (!second) {
                fa = y;
                second = true;
            } else {
                second = false;
                if (fa == y) {
                    // equal rotations: the same fields (decode), so the same stages but for the chunk's
                    const bool claw = ((a ^ b) & 1) != 0, same = !claw && L.seq(a, 0) == L.seq(b, 0);
                    if (claw && head) append_claw(w, a, b, chunk);
                    cls[1] += !claw && same; // trivial
                    cls[2] += !claw && !same; // same side
                    cls[3] += claw;
                    active = false;
                } else {
                    a = fa;
                    b = y;
                    la--;
                    lb--;
                    settle();
                }
            }
        }
        __syncwarp(kAll);
        if (nf >= 0x40000000u) { // tallies are in 32 bits
            if (head) atomicAdd(&w.counters[C_RSTEPS], (unsigned long long)nf);
            nf = 0;
        }
    }
    const uint32_t v[8] = {cls[0], cls[1], cls[2], cls[3], cls[4], cls[5], cls[3], nf};
    const int idx[8] = {C_CLS0, C_CLS0 + 1, C_CLS0 + 2, C_CLS0 + 3, C_CLS0 + 4, C_CLS0 + 5, C_CANDS, C_RSTEPS};
#pragma unroll
    for (int i = 0; i < 8; i++) {
        unsigned long long sum = head ? v[i] : 0u;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) sum += __shfl_xor_sync(kAll, sum, o);
        if (lane == 0 && sum) atomicAdd(&w.counters[idx[i]], sum);
    }
}

template <int NQ>
__global__ void __launch_bounds__(qd::Geo<NQ>::kThreads, 1) k_rewalk_q(WalkLaunch w, uint32_t least)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t cnt = w.pend_in_n + min(*w.qhead, w.qcap);
    if (cnt < least) return; // k_rewalk_pairs takes them
    if (cnt <= 8 * blockIdx.x) return; // no merges for this CTA
    const qd::Level<NQ> L(w.lv);
    const qd::Sm<NQ> sm = qd::set_up<NQ>(w.lv, L.scale, smem_raw);
    rewalk_eight<NQ>(w, w.rw_next, cnt, L, sm, threadIdx.x & 31);
}

// Many jobs in one launch (walk_shares): a job's walks of the CTA's share are
// walked together, eight to a warp, and the tables are set up again where the
// job changes.  No wait of these kernels can run out.
template <int NQ>
__global__ void __launch_bounds__(qd::kBatchThreads, 1) k_walks_batch_q(BatchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ WalkLaunch sw;
    const uint32_t warps = blockDim.x >> 5;
    walk_shares(
        a, blockIdx.x, gridDim.x, 8, qd::kTaskWalks,
        [&](uint32_t job, uint32_t first, uint32_t most) {
            __syncthreads(); // every warp is done with the previous job
            if (threadIdx.x == 0) sw = a.jobs[job];
            __syncthreads();
            const qd::Level<NQ> L(sw.lv);
            const qd::Sm<NQ> sm = qd::set_up<NQ>(sw.lv, L.scale, smem_raw);
            const uint32_t end = min((uint32_t)sw.n_walks, first + most);
            for (uint32_t base = first + 8 * (threadIdx.x >> 5); base < end; base += 8 * warps)
                walk_eight<NQ>(sw, base, end, L, sm, threadIdx.x & 31);
            return true;
        },
        [](uint32_t) {});
}

template <int NQ>
__global__ void __launch_bounds__(qd::kBatchThreads, 1) k_rewalk_batch_q(BatchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ WalkLaunch sw;
    __shared__ uint32_t cursor;
    merge_shares(
        a, blockIdx.x, gridDim.x,
        [&](uint32_t job, uint32_t p0, uint32_t p1) {
            __syncthreads(); // every warp is done with the previous job
            if (threadIdx.x == 0) {
                sw = a.jobs[job];
                cursor = p0;
            }
            __syncthreads();
            const qd::Level<NQ> L(sw.lv);
            const qd::Sm<NQ> sm = qd::set_up<NQ>(sw.lv, L.scale, smem_raw);
            rewalk_eight<NQ>(sw, &cursor, p1, L, sm, threadIdx.x & 31);
            return true;
        },
        [](uint32_t) {});
}

// Grid and warps of a CTA for `groups` warp-loads: warp w of CTA b takes loads
// b + grid w, and every grid * warps-th after it, so that few loads spread over
// the SMs; as many warps as make the rounds even, and at least eight (sixteen
// at n = 3), which also set the CTA up.
template <int NQ>
void shape_for(size_t groups, unsigned *grid, unsigned *warps)
{
    const size_t sms = (size_t)num_sms(), most = (size_t)qd::Geo<NQ>::kWarps;
    const size_t per_sm = std::max<size_t>(1, (groups + sms - 1) / sms), rounds = (per_sm + most - 1) / most;
    *warps = (unsigned)std::max<size_t>(NQ == 3 ? 16 : 8, (per_sm + rounds - 1) / rounds);
    *grid = (unsigned)std::max<size_t>(1, std::min(sms, groups));
}

template <int NQ, typename K>
cudaError_t allow_smem(K k, int warps = qd::Geo<NQ>::kWarps)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qd::Geo<NQ>::smem_bytes(warps));
}

template <int NQ>
cudaError_t walks_q(const WalkLaunch &w, cudaStream_t s)
{
    if (w.n_walks <= 0) return cudaSuccess;
    const cudaError_t e = allow_smem<NQ>(k_walks_q<NQ>);
    if (e != cudaSuccess) return e;
    unsigned grid, warps;
    shape_for<NQ>(((size_t)w.n_walks + 7) / 8, &grid, &warps);
    k_walks_q<NQ><<<grid, 32 * warps, qd::Geo<NQ>::smem_bytes((int)warps), s>>>(w);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t walk_step_q(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp, size_t count,
                        cudaStream_t s)
{
    const cudaError_t e = allow_smem<NQ>(k_walk_step_q<NQ>);
    if (e != cudaSuccess) return e;
    unsigned grid, warps;
    shape_for<NQ>((count + 7) / 8, &grid, &warps);
    k_walk_step_q<NQ><<<grid, 32 * warps, qd::Geo<NQ>::smem_bytes((int)warps), s>>>(lv, (uint32_t)chunk, in, out, is_dp,
                                                                                  count);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t rewalk_q(const WalkLaunch &w, uint32_t least, cudaStream_t s)
{
    using G = qd::Geo<NQ>;
    const cudaError_t e = allow_smem<NQ>(k_rewalk_q<NQ>);
    if (e != cudaSuccess) return e;
    k_rewalk_q<NQ><<<(unsigned)num_sms(), G::kThreads, G::smem_bytes(G::kWarps), s>>>(w, least);
    return cudaGetLastError();
}

template <int NQ>
cudaError_t batch_q(const BatchArgs &a, bool rewalk, cudaStream_t s)
{
    const auto k = rewalk ? k_rewalk_batch_q<NQ> : k_walks_batch_q<NQ>;
    const cudaError_t e = allow_smem<NQ>(k, qd::kBatchWarps);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)num_sms(), qd::kBatchThreads, qd::Geo<NQ>::smem_bytes(qd::kBatchWarps), s>>>(a);
    return cudaGetLastError();
}

} // namespace

cudaError_t launch_rewalk_q(const WalkLaunch &w, uint32_t least, cudaStream_t s)
{
    if (!w.rw_next) return cudaErrorInvalidValue;
    return w.lv.n == 3 ? rewalk_q<3>(w, least, s) : w.lv.n == 2 ? rewalk_q<2>(w, least, s) : cudaErrorInvalidValue;
}

cudaError_t launch_walks_batch_q(int n, const BatchArgs &a, cudaStream_t s)
{
    return n == 3 ? batch_q<3>(a, false, s) : n == 2 ? batch_q<2>(a, false, s) : cudaErrorInvalidValue;
}

cudaError_t launch_rewalk_batch_q(int n, const BatchArgs &a, cudaStream_t s)
{
    return n == 3 ? batch_q<3>(a, true, s) : n == 2 ? batch_q<2>(a, true, s) : cudaErrorInvalidValue;
}

int quad_walks_per_task() { return qd::kTaskWalks; }

cudaError_t launch_walks_q(const WalkLaunch &w, cudaStream_t s)
{
    return w.lv.n == 3 ? walks_q<3>(w, s) : w.lv.n == 2 ? walks_q<2>(w, s) : cudaErrorInvalidValue;
}

cudaError_t launch_walk_step_q(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp,
                               size_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    return lv.n == 3   ? walk_step_q<3>(lv, chunk, in, out, is_dp, count, s)
           : lv.n == 2 ? walk_step_q<2>(lv, chunk, in, out, is_dp, count, s)
                       : cudaErrorInvalidValue;
}

} // namespace qcs
