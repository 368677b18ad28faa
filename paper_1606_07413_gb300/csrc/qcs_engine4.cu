// qcs_engine4.cu -- n = 4: the coset hash of many points at once, with the W
// side's contraction on the fifth-generation tensor cores (tcgen05.mma).
//
// The engine.  A CTA (one per SM) evaluates the hash of 48 points in flight,
// two sets of 24.  Its 19 warps have three roles:
//  - 16 workers, each owning three points (one or two of each set).  Phase A
//    of a set: a point's fingerprint weights go through its adjoint stages
//    (one warp per point); a V point's weights are its column fingerprints,
//    hashed at once; a W point writes its weights as two f16 byte planes, two
//    rows of the set's B operand.  Phase E: the set's product D = C^^T B is
//    read back from tensor memory and hashed, column sums of every W point.
//  - one MMA warp: when all rows of a set are written it issues the product,
//    64 tcgen05.mma (128 x N x 16 each, N = twice the set's W points).
//  - one control warp per set: lane i is what uses slot i's hash (a walk, a
//    re-walked merge, ...).  It takes the set's hashes, decides the slots'
//    next points and publishes them; table inserts and the like follow after
//    that, off the critical path.  All that a walk does besides f runs here
//    on 24 lanes at once instead of once per walk on 32.
// The workers run A(0) A(1) E(0) E(1) in turn: MMA(X) runs beside the other
// set's A, control(X) beside the other set's E.
//
// What bounds it.  A point costs 618 warp instructions; half of them are the
// 255 column finalisers.  Issue is 59 % active, the ALU pipe 59 %, the tensor
// pipe 16 %: fixed-latency and load stalls between the phases take the rest.
// 2^20 walks x 16 steps at level 7: 14.95 ms (1.12 G steps/s), against 26.7 ms
// with mma.sync (12 stage and 8 MMA warps, C^'s fragments through
// tcgen05.ld, the rows through ldmatrix: 1073 instructions a step).
//
// Where C^ sits.  In f16 it is 256 KB.  As the A operand (M = columns of C^,
// K = its 512 numerator rows) its first 128 columns and K-blocks 0-7 of the
// other 128 are in tensor memory (320 of 512 columns), the rest (96 KB) in
// shared memory; that leaves 192 tensor-memory columns for two sets' D (2 x
// 2 x 48 f32 columns) and 96 KB of shared memory for two sets' B.
//
// Exactness.  B holds 1024 + byte (the f16 bits 0x6400 | byte, so no
// conversion), and every sum is an integer below 2^24 in magnitude, so f32
// accumulation is exact.  Row 0 (the identity) has zero weight on both parts,
// so its two K slots are free; their B values are 1024 and their A values are
// 12288 and -sum(c), which adds 1.5 x 2^23 and takes the offset's 1024 sum(c)
// away again: the bits of the f32 result are 0x4B400000 + P, P the integer
// dot product, and its low 16 bits are those of P.  |P| and every partial sum
// stay below 2^22 when a column's absolute sum is at most kMaxColumnSum
// (qcs_internal.h), which the host checks (columns of an orthogonal C^ in
// int8 obey it up to denominator exponent 13).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "qcs_device.cuh"
#include "qcs_internal.h"

namespace qcs {
namespace {

namespace e4 {

constexpr int kWorkers = 16, kSet = 24, kSets = 2;
constexpr int kMmaWarp = kWorkers, kCtlWarp = kWorkers + 1; // control warps kCtlWarp, kCtlWarp + 1
constexpr int kWarps = kWorkers + 1 + kSets, kThreads = 32 * kWarps;
constexpr int kN = 2 * kSet;                // columns of D per set and half
constexpr int kTmemK = 8;                   // K-blocks of C^'s second half held in tensor memory
constexpr int kDcol = 256 + 8 * kTmemK;     // tensor-memory column of D (set X, half h: + 96 X + 48 h)
static_assert(kDcol + kSets * 2 * kN <= 512, "tensor memory");
constexpr uint32_t kInvalid = 1u << 31;

// one point to evaluate, published by the set's control warp
struct alignas(16) Job {
    uint64_t seq;   // the stages in order, one Pauli code (see code_of) per byte
    uint64_t PH;    // (pre with its low 16 bits clear) * the finaliser's first constant
    uint32_t pre16; // the low 16 bits of pre
    uint32_t info;  // stages | side << 8 | row pair << 16, or kInvalid
    uint64_t pad;
};
struct alignas(16) HashBase { // the hash base of a W row pair, for phase E
    uint64_t PH;
    uint32_t pre16, pad;
};

// shared memory
constexpr size_t off_A = 0;                                        // C^, second half, K-blocks 8..31: 6 chunks of 64 K
constexpr size_t off_B = off_A + 6 * 16384;                        // [set]: 8 chunks of 64 K x 48 rows
constexpr size_t off_job = off_B + (size_t)kSets * 8 * kN * 128;   // Job [set][slot]
constexpr size_t off_wb = off_job + sizeof(Job) * kSets * kSet;    // HashBase [set][row pair]
constexpr size_t off_part = off_wb + sizeof(HashBase) * kSets * kSet;   // u64 [set][quadrant and half][row pair]
constexpr size_t off_vsum = off_part + 8 * sizeof(uint64_t) * kSets * kSet; // u64 [set][slot]
constexpr size_t off_chunk = off_vsum + sizeof(uint64_t) * kSets * kSet; // HashBase [chunk]
constexpr size_t off_stage = off_chunk + sizeof(HashBase) * 256;   // stage table: byte [code][lane]
constexpr size_t off_nw = off_stage + 256 * 32;                    // u32 [set]: W points; [2 + set]: the set is done
constexpr size_t off_bar = off_nw + 16;                            // mbarriers: jobs, rows, product, sums [set]
constexpr size_t off_tmem = off_bar + 8 * sizeof(uint64_t);
constexpr size_t smem_bytes = off_tmem + 16;
static_assert(smem_bytes <= 227 * 1024, "shared memory of the n = 4 engine");

// a bounded wait gives up after this many SM clock cycles (about two seconds)
constexpr long long kWaitCycles = 1ll << 32;

constexpr uint64_t kC1 = 0xBF58476D1CE4E5B9ull, kC2 = 0x94D049BB133111EBull; // SplitMix64's finaliser

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- mbarriers: arrive has release and try_wait acquire semantics at CTA scope
__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *b)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(b)) : "memory");
}

// Wait until the phase of parity `ph` has completed; false if the wait ran
// out.  Warp-uniform: true only if every lane saw the phase complete.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t ph)
{
    const uint32_t a = smem_u32(b);
    const long long t0 = clock64();
    bool ok = false;
    for (;;) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(a), "r"(ph)
                     : "memory");
        if (done) {
            ok = true;
            break;
        }
        if (clock64() - t0 > kWaitCycles) break;
    }
    return __all_sync(0xFFFFFFFFu, ok);
}

// ---- tensor memory and products
__device__ __forceinline__ void tmem_alloc(uint32_t *dst)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(dst)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}

__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// 16 lanes x 8 columns: the thread gets row lane / 4 (v[0], v[1]) and row
// lane / 4 + 8 (v[2], v[3]), columns 2 (lane % 4) and + 1
__device__ __forceinline__ void tmem_ld16x256(uint32_t (&v)[4], uint32_t taddr)
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}

// the loads' registers are valid after this; it takes them as operands so
// that no use is scheduled before it
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&a)[4], uint32_t (&b)[4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3])
                 :
                 : "memory");
}

// shared-memory operand: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// D (+)= A B, A in tensor memory (TS) or shared memory (SS); FIRST: D = A B
template <bool FIRST>
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
                 "r"(a), "l"(b), "r"(idesc), "n"(FIRST ? 0 : 1)
                 : "memory");
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, 0, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc)
                 : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// ---- one point on one warp
//
// Lane l holds the eight weight rows row4(l, t) (qcs_internal.h): t carries
// qubit 3's two bits and qubit 2's x bit, the lane the rest, and a Pauli's
// code (code4) is laid out the same way: its low five bits are its lane part,
// its high three its t part.  A stage takes row j to u_j +- u_{j^p} or to
// sqrt2 u_j, by lambda(p, j) in P(p) P(j) = i^lambda P(p^j), which is a sum
// over the qubits.  So with the t part of p known at compile time (a switch
// over its eight values) the partner's register and qubit 3's share of lambda
// are constants, and what is left of lambda is one value per lane and x bit of
// qubit 2: a byte of the stage table per code and lane.

__host__ __device__ constexpr int lambda1(int px, int pz, int x, int z)
{
    return (px * pz + x * z + 2 * pz * x - (px ^ x) * (pz ^ z)) & 3;
}

// lambda of the lane's rows but for qubit 3's share, for x bit 0 (bits 0-1)
// and 1 (bits 2-3) of qubit 2
__device__ __forceinline__ uint32_t stage_byte(uint32_t code, uint32_t l)
{
    // lane bits: z0 z1 z2 x0 x1; code bits: the same, then z3 x3 x2
    uint32_t v = 0;
#pragma unroll
    for (int q = 0; q < 2; q++)
        v += lambda1((code >> (3 + q)) & 1, (code >> q) & 1, (l >> (3 + q)) & 1, (l >> q) & 1);
    const int px2 = (code >> 7) & 1, pz2 = (code >> 2) & 1, z2 = (l >> 2) & 1;
    return ((v + lambda1(px2, pz2, 0, z2)) & 3) | ((v + lambda1(px2, pz2, 1, z2)) & 3) << 2;
}

// m: the multipliers of the partner row, per x bit of qubit 2 (second index)
// for rows whose qubit-3 share of lambda is 0 (m[0]), 1 (m[1]) or 3 (m[2])
template <int PT>
__device__ __forceinline__ void stage_rows(uint32_t (&ua)[8], uint32_t (&ub)[8], int pl, const int (&m)[3][2],
                                           const bool (&odd)[2])
{
    uint32_t na[8], nb[8];
#pragma unroll
    for (int t = 0; t < 8; t++) {
        const int x2 = t >> 2, c = lambda1((PT >> 1) & 1, PT & 1, (t >> 1) & 1, t & 1);
        const uint32_t va = __shfl_xor_sync(0xFFFFFFFFu, ua[t ^ PT], pl);
        const uint32_t vb = __shfl_xor_sync(0xFFFFFFFFu, ub[t ^ PT], pl);
        const bool anti = odd[x2] != ((c & 1) != 0);
        const uint32_t mul = (uint32_t)m[c == 0 ? 0 : c == 1 ? 1 : 2][x2];
        // anticommuting rows: u + s v; commuting rows (multiplier 0): (ub, 2 ua)
        na[t] = va * mul + (anti ? ua[t] : ub[t]);
        nb[t] = vb * mul + (anti ? ub[t] : ua[t] << 1);
    }
#pragma unroll
    for (int t = 0; t < 8; t++) {
        ua[t] = na[t];
        ub[t] = nb[t];
    }
}

// tr: 0 for V (adjoint of R^), 1 for W (adjoint of R^T)
__device__ __forceinline__ void stage(uint32_t code, uint32_t tr, const uint8_t *tab, int lane, uint32_t (&ua)[8],
                                      uint32_t (&ub)[8])
{
    const uint32_t v = tab[code * 32 + lane];
    const int pl = (int)(code & 31);
    int m[3][2];
    bool odd[2];
#pragma unroll
    for (int x = 0; x < 2; x++) {
        odd[x] = ((v >> (2 * x)) & 1u) != 0;
        const int s = 1 - 2 * (int)(((v >> (2 * x + 1)) ^ tr) & 1u); // lambda 0 or 1: +, 2 or 3: - (V)
        m[0][x] = odd[x] ? s : 0;
        m[1][x] = odd[x] ? 0 : s;
        m[2][x] = odd[x] ? 0 : -s;
    }
    switch (code >> 5) {
    case 0: stage_rows<0>(ua, ub, pl, m, odd); break;
    case 1: stage_rows<1>(ua, ub, pl, m, odd); break;
    case 2: stage_rows<2>(ua, ub, pl, m, odd); break;
    case 3: stage_rows<3>(ua, ub, pl, m, odd); break;
    case 4: stage_rows<4>(ua, ub, pl, m, odd); break;
    case 5: stage_rows<5>(ua, ub, pl, m, odd); break;
    case 6: stage_rows<6>(ua, ub, pl, m, odd); break;
    default: stage_rows<7>(ua, ub, pl, m, odd); break;
    }
}

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

__device__ __forceinline__ HashBase hash_base(uint64_t base)
{
    const uint64_t pre = base ^ (base >> 30);
    return HashBase{(pre & ~0xFFFFull) * kC1, (uint32_t)pre & 0xFFFFu, 0};
}

// sum mod 2^64 over the warp from three 32-bit reductions (see group_sum64 in qcs_walk.cu)
__device__ __forceinline__ uint64_t warp_sum64(uint64_t acc)
{
    const uint32_t lo = (uint32_t)acc, hi = (uint32_t)(acc >> 32);
    const uint32_t s_hi = __reduce_add_sync(0xFFFFFFFFu, hi);
    const uint32_t s_l0 = __reduce_add_sync(0xFFFFFFFFu, lo & 0xFFFFu);
    const uint32_t s_l1 = __reduce_add_sync(0xFFFFFFFFu, lo >> 16);
    return ((uint64_t)s_hi << 32) + ((uint64_t)s_l1 << 16) + (uint64_t)s_l0;
}

// the weights after the first stage of a point (LevelCtx::T4), as two 16-byte
// loads; the upper halves of ua are never looked at (every sum is mod 2^16)
__device__ __forceinline__ void first_stage(const uint4 *tab, uint32_t code, int lane, uint32_t (&ua)[8],
                                            uint32_t (&ub)[8])
{
    const uint4 w0 = __ldg(tab + (code * 32 + lane) * 2), w1 = __ldg(tab + (code * 32 + lane) * 2 + 1);
    ua[0] = w0.x; ua[1] = w0.y; ua[2] = w0.z; ua[3] = w0.w;
    ua[4] = w1.x; ua[5] = w1.y; ua[6] = w1.z; ua[7] = w1.w;
#pragma unroll
    for (int t = 0; t < 8; t++) ub[t] = ua[t] >> 16;
}

// The multiset sum of a V point: its weights, scaled by sqrt2^ev, are its
// column fingerprints' a parts (the scaling commutes with the stages, so only
// the part that ends up in a is scaled, once).
__device__ __forceinline__ uint64_t v_column_sum(const uint32_t (&ua)[8], const uint32_t (&ub)[8], int ev,
                                                 uint64_t PH, uint32_t pre16, int lane)
{
    const bool odd = (ev & 1) != 0;
    const int sh = (ev >> 1) < 31 ? ev >> 1 : 31;
    uint64_t acc = 0;
#pragma unroll
    for (int t = 0; t < 8; t++) {
        const uint64_t e = column_hash((odd ? ub[t] : ua[t]) << sh, PH, pre16);
        acc += (t == 0 && lane == 0) ? 0ull : e; // column 0, the identity, does not enter
    }
    return warp_sum64(acc);
}

// Pauli code of index q (row4's bit order)
__device__ __forceinline__ uint32_t code_of(uint32_t q)
{
    return (q & 7u) | ((q >> 4) & 3u) << 3 | ((q >> 3) & 1u) << 5 | ((q >> 7) & 1u) << 6 | ((q >> 6) & 1u) << 7;
}

// The stages of a point: V takes q_h first and goes down to q_1; W takes q_1
// .. q_h, then the chunk.  A product of no rotations starts from code 0, the
// untouched weights; so does V's single rotation (its half product then is
// not one lookup).  Returns the number of stages.
__device__ __forceinline__ int stage_seq(int side, uint64_t qpack, uint32_t chunk, int h, uint64_t *out)
{
    uint64_t seq = 0;
    int ns = 0;
    if (side == 0) {
        if (h <= 1) ns = 1;
        for (int j = h - 1; j >= 0; j--) seq |= (uint64_t)code_of((uint32_t)(qpack >> (8 * j)) & 0xFFu) << (8 * ns++);
    } else {
        if (h == 0) ns = 1;
        for (int j = 0; j < h; j++) seq |= (uint64_t)code_of((uint32_t)(qpack >> (8 * j)) & 0xFFu) << (8 * ns++);
        if (chunk) seq |= (uint64_t)code_of(chunk) << (8 * ns++);
    }
    *out = seq;
    return ns;
}

// ---- roles

struct Cta {
    unsigned char *raw;
    uint64_t *bars; // jobs [2], rows [2], product [2], sums [2]
    uint32_t *nw;   // [2] W points, [2] set done
    uint32_t tmem;
    __device__ Job *jobs(int X) const { return reinterpret_cast<Job *>(raw + off_job) + X * kSet; }
    __device__ HashBase *wb(int X) const { return reinterpret_cast<HashBase *>(raw + off_wb) + X * kSet; }
    __device__ uint64_t *part(int X) const { return reinterpret_cast<uint64_t *>(raw + off_part) + X * 8 * kSet; }
    __device__ uint64_t *vsum(int X) const { return reinterpret_cast<uint64_t *>(raw + off_vsum) + X * kSet; }
    __device__ const HashBase *chunk_base() const { return reinterpret_cast<const HashBase *>(raw + off_chunk); }
    __device__ uint64_t *bar_jobs(int X) const { return bars + X; }
    __device__ uint64_t *bar_rows(int X) const { return bars + 2 + X; }
    __device__ uint64_t *bar_prod(int X) const { return bars + 4 + X; }
    __device__ uint64_t *bar_sums(int X) const { return bars + 6 + X; }
};

// stage table, chunk bases, barriers, tensor memory and C^: every thread calls it
__device__ __forceinline__ Cta cta_begin(const LevelCtx &lv, unsigned char *raw, bool with_chunks)
{
    Cta c;
    c.raw = raw;
    c.bars = reinterpret_cast<uint64_t *>(raw + off_bar);
    c.nw = reinterpret_cast<uint32_t *>(raw + off_nw);
    uint32_t *taddr = reinterpret_cast<uint32_t *>(raw + off_tmem);
    if (threadIdx.x < 32) tmem_alloc(taddr);
    if (threadIdx.x == 32) {
        for (int X = 0; X < kSets; X++) {
            mbar_init(c.bar_jobs(X), 1);
            mbar_init(c.bar_rows(X), kWorkers);
            mbar_init(c.bar_prod(X), 1);
            mbar_init(c.bar_sums(X), kWorkers);
        }
        c.nw[0] = c.nw[1] = c.nw[2] = c.nw[3] = 0;
    }
    uint8_t *tab = raw + off_stage;
    for (int i = threadIdx.x; i < 256 * 32; i += kThreads) tab[i] = (uint8_t)stage_byte(i >> 5, i & 31);
    if (with_chunks) {
        // base(chunk) = smix(smix(seed_H ^ version) ^ (n | k << 8 | chunk << 16 | K << 32))
        const uint64_t vmix = smix(kSeedH ^ (uint64_t)lv.version);
        for (int i = threadIdx.x; i < 256; i += kThreads) {
            const uint64_t tag = (uint64_t)lv.n | ((uint64_t)lv.k << 8) | ((uint64_t)i << 16) |
                                 ((uint64_t)(uint32_t)lv.K << 32);
            reinterpret_cast<HashBase *>(raw + off_chunk)[i] = hash_base(smix(vmix ^ tag));
        }
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    c.tmem = *taddr;
    return c;
}

// two biased bytes of a word of LevelCtx::Cm as an f16 pair: the byte permute
// puts them under 0x64 (1024 + byte in f16), then 1152 is subtracted
__device__ __forceinline__ uint32_t bytes_to_f16x2(uint32_t word, uint32_t sel)
{
    const uint32_t v = __byte_perm(word, 0x64646464u, sel);
    __half2 h = *reinterpret_cast<const __half2 *>(&v);
    h = __hsub2(h, __float2half2_rn(1152.f));
    return *reinterpret_cast<const uint32_t *>(&h);
}

// C^ into tensor and shared memory; every thread calls it, and a barrier follows
__device__ __forceinline__ void load_c(const LevelCtx &lv, const Cta &c)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kBias = 0x7200u; // 12288 in f16: 1024 * 12288 = 1.5 * 2^23
    if (warp < kWorkers) {
        // warp w writes the tensor-memory lanes 32 (w % 4) ..: K-blocks
        // w / 4, w / 4 + 4, .. of its 32 columns of either half
        const uint32_t tq = c.tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        for (int b = warp >> 2; b < 32 + kTmemK; b += kWorkers / 4) {
            const int half = b >= 32, kb = half ? b - 32 : b, Q = 128 * half + 32 * (warp & 3) + lane;
            const uint4 w = __ldg(lv.Cm + Q * 32 + kb);
            uint32_t v[8] = {bytes_to_f16x2(w.x, 0x4140), bytes_to_f16x2(w.x, 0x4342), bytes_to_f16x2(w.y, 0x4140),
                             bytes_to_f16x2(w.y, 0x4342), bytes_to_f16x2(w.z, 0x4140), bytes_to_f16x2(w.z, 0x4342),
                             bytes_to_f16x2(w.w, 0x4140), bytes_to_f16x2(w.w, 0x4342)};
            if (kb == 0) v[0] = (v[0] & 0xFFFF0000u) | kBias;
            if (kb == 16)
                v[0] = (v[0] & 0xFFFF0000u) | __half_as_ushort(__float2half_rn(-(float)lv.Csum[Q]));
            tmem_st8(tq + (half ? 256u : 0u) + 8u * (uint32_t)kb, v);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    // second half, K-blocks kTmemK ..: 16-byte units (8 K) of 128 rows
    constexpr int U0 = 2 * kTmemK, UN = 64 - U0;
    for (int i = threadIdx.x; i < 128 * UN; i += kThreads) {
        const int r = i / UN, u = U0 + i % UN, Q = 128 + r;
        const uint2 w = __ldg(reinterpret_cast<const uint2 *>(lv.Cm + Q * 32) + u);
        uint4 v = make_uint4(bytes_to_f16x2(w.x, 0x4140), bytes_to_f16x2(w.x, 0x4342), bytes_to_f16x2(w.y, 0x4140),
                             bytes_to_f16x2(w.y, 0x4342));
        if (u == 32) v.x = (v.x & 0xFFFF0000u) | __half_as_ushort(__float2half_rn(-(float)lv.Csum[Q]));
        *reinterpret_cast<uint4 *>(c.raw + off_A + (size_t)((u >> 3) - U0 / 8) * 16384 + (r >> 3) * 1024 +
                                   (r & 7) * 128 + (((u & 7) ^ (r & 7)) * 16)) = v;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tmem_fence_before();
}

// phase A of one point
__device__ __forceinline__ void point_a(const LevelCtx &lv, const Cta &c, int X, int slot, int lane)
{
    const Job *jp = c.jobs(X) + slot;
    const uint32_t info = jp->info;
    if (info & kInvalid) return;
    const uint64_t seq = jp->seq;
    const uint32_t side = (info >> 8) & 1u, ns = info & 0xFFu;
    const uint8_t *tab = c.raw + off_stage;
    uint32_t ua[8], ub[8];
    first_stage(lv.T4[side], (uint32_t)seq & 0xFFu, lane, ua, ub);
#pragma unroll 1
    for (uint32_t i = 1; i < ns; i++)
        stage(__shfl_sync(0xFFFFFFFFu, (uint32_t)(seq >> (8 * i)) & 0xFFu, 0), side, tab, lane, ua, ub);
    if (side == 0) {
        const uint64_t sum = v_column_sum(ua, ub, lv.ev, jp->PH, jp->pre16, lane);
        if (lane == 0) c.vsum(X)[slot] = sum;
    } else {
        // rows 2 pos and 2 pos + 1 of B: the low and the high byte plane.  The
        // lane's eight rows are the K indices 8 lane .. of each part, one
        // 16-byte unit; unit u of row r is at unit u ^ (r & 7) of its 128
        // bytes in chunk u / 8.
        const uint32_t r = 2 * (info >> 16);
        unsigned char *b = c.raw + off_B + (size_t)X * 8 * kN * 128 + (size_t)(lane >> 3) * (kN * 128) + (r >> 3) * 1024;
#pragma unroll
        for (int p = 0; p < 2; p++) { // a, b part
            uint32_t lo[4], hi[4];
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const uint32_t w = p ? __byte_perm(ub[2 * e], ub[2 * e + 1], 0x5410)
                                     : __byte_perm(ua[2 * e], ua[2 * e + 1], 0x5410);
                lo[e] = (w & 0x00FF00FFu) | 0x64006400u;
                hi[e] = __byte_perm(w, 0x64646464u, 0x4341);
            }
            unsigned char *d = b + (size_t)p * 4 * (kN * 128);
            const uint32_t u = (uint32_t)lane & 7u, r0 = r & 7u;
            *reinterpret_cast<uint4 *>(d + r0 * 128 + ((u ^ r0) * 16)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            *reinterpret_cast<uint4 *>(d + (r0 + 1) * 128 + ((u ^ (r0 + 1)) * 16)) =
                make_uint4(hi[0], hi[1], hi[2], hi[3]);
        }
    }
}

// Phase E, one unit: the 32 columns of C^ that quadrant qd holds of half h,
// for row pairs 4 g .. 4 g + 3 (lane % 4)
__device__ __forceinline__ void unit_e(const Cta &c, int X, int g, int h, int qd, int lane)
{
    const uint32_t t = c.tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(kDcol + X * 2 * kN + h * kN + 8 * g);
    uint32_t v[2][4];
    tmem_ld16x256(v[0], t);
    tmem_ld16x256(v[1], t + (16u << 16));
    const HashBase hb = c.wb(X)[4 * g + (lane & 3)];
    tmem_wait_ld(v[0], v[1]);
    uint64_t acc = 0;
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
            // the two planes' dot products (their low 16 bits are exact)
            const uint64_t z = column_hash(v[s][2 * e] + v[s][2 * e + 1] * 256u, hb.PH, hb.pre16);
            acc += (s == 0 && e == 0 && h == 0 && qd == 0 && lane < 4) ? 0ull : z; // column 0 does not enter
        }
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 4);
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 8);
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 16);
    if (lane < 4) c.part(X)[(2 * qd + h) * kSet + 4 * g + lane] = acc;
}

// worker warp w; false if a wait ran out
__device__ __forceinline__ bool worker(const LevelCtx &lv, const Cta &c, int w, int lane)
{
    bool done[2] = {false, false};
    uint32_t ph = 0;
    const bool low = w < kWorkers / 2;
    // set 0: slots 2w, 2w + 1 (w < 8) or 8 + w; set 1: the other way round
    while (!(done[0] && done[1])) {
#pragma unroll
        for (int X = 0; X < 2; X++) {
            if (done[X]) continue;
            if (!mbar_wait(c.bar_jobs(X), ph)) return false;
            if (c.nw[2 + X]) {
                done[X] = true;
                continue;
            }
            const bool two = low == (X == 0);
            const int v = low ? w : w - kWorkers / 2;
            const int s0 = two ? 2 * v : kWorkers + v, s1 = two ? s0 + 1 : s0;
#pragma unroll 1
            for (int s = s0; s <= s1; s++) point_a(lv, c, X, s, lane);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(c.bar_rows(X));
        }
        int u0 = w >> 2; // units of both sets in turn over the quadrant's four warps
#pragma unroll
        for (int X = 0; X < 2; X++) {
            if (done[X]) continue;
            if (!mbar_wait(c.bar_prod(X), ph)) return false;
            tmem_fence_after();
            const int units = 2 * ((int)(c.nw[X] + 3) >> 2);
#pragma unroll 1
            for (; u0 < units; u0 += kWorkers / 4) unit_e(c, X, u0 >> 1, u0 & 1, w & 3, lane);
            u0 -= units;
            tmem_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(c.bar_sums(X));
        }
        ph ^= 1u;
    }
    return true;
}

// the MMA warp (the whole warp calls it); false if a wait ran out
__device__ __forceinline__ bool mma_warp(const Cta &c)
{
    bool done[2] = {false, false};
    uint32_t ph = 0;
    const uint64_t a0 = smem_desc(smem_u32(c.raw + off_A));
    while (!(done[0] && done[1])) {
#pragma unroll 1
        for (int X = 0; X < 2; X++) {
            if (X ? done[1] : done[0]) continue;
            if (!mbar_wait(c.bar_jobs(X), ph)) return false;
            if (c.nw[2 + X]) {
                if (X) done[1] = true;
                else done[0] = true;
                continue;
            }
            if (!mbar_wait(c.bar_rows(X), ph)) return false;
            tmem_fence_after();
            const uint32_t nw = c.nw[X];
            if (elect_one()) {
                if (nw) {
                    const uint32_t N = (2 * nw + 15) & ~15u;
                    // f16 x f16 -> f32, both K-major, M = 128
                    const uint32_t idesc = (1u << 4) | ((N >> 3) << 17) | ((128u >> 4) << 24);
                    const uint64_t b0 = smem_desc(smem_u32(c.raw + off_B) + (uint32_t)(X * 8 * kN * 128));
                    const uint32_t d0 = c.tmem + (uint32_t)(kDcol + X * 2 * kN);
#pragma unroll
                    for (int kb = 0; kb < 32; kb++) {
                        const uint64_t b = b0 + (uint64_t)(((kb >> 2) * (kN * 128) + (kb & 3) * 32) >> 4);
                        if (kb == 0) mma_ts<true>(d0, c.tmem + 8 * kb, b, idesc);
                        else mma_ts<false>(d0, c.tmem + 8 * kb, b, idesc);
                    }
#pragma unroll
                    for (int kb = 0; kb < 32; kb++) {
                        const uint64_t b = b0 + (uint64_t)(((kb >> 2) * (kN * 128) + (kb & 3) * 32) >> 4);
                        if (kb == 0) mma_ts<true>(d0 + kN, c.tmem + 256 + 8 * kb, b, idesc);
                        else if (kb < kTmemK) mma_ts<false>(d0 + kN, c.tmem + 256 + 8 * kb, b, idesc);
                        else {
                            const int k2 = kb - kTmemK;
                            mma_ss(d0 + kN, a0 + (uint64_t)(((k2 >> 2) * 16384 + (k2 & 3) * 32) >> 4), b, idesc);
                        }
                    }
                    mma_commit(c.bar_prod(X));
                } else {
                    mbar_arrive(c.bar_prod(X));
                }
            }
            __syncwarp();
        }
        ph ^= 1u;
    }
    return true;
}

// Publish the set's next points: lane i < kSet passes slot i's (valid or
// not).  The row pairs of the W points are numbered here.  Whole warp.
// Returns the lane's row pair.
__device__ __forceinline__ uint32_t publish(const Cta &c, int X, int lane, bool valid, int side, uint64_t qpack,
                                            uint32_t chunk, int h, HashBase hb)
{
    const uint32_t wm = __ballot_sync(0xFFFFFFFFu, valid && side == 1);
    const uint32_t pos = (uint32_t)__popc(wm & ((1u << lane) - 1u));
    if (lane < kSet) {
        Job j;
        j.PH = hb.PH;
        j.pre16 = hb.pre16;
        j.pad = 0;
        j.seq = 0;
        if (valid) {
            const int ns = stage_seq(side, qpack, chunk, h, &j.seq);
            j.info = (uint32_t)ns | (uint32_t)side << 8 | pos << 16;
        } else {
            j.info = kInvalid;
        }
        c.jobs(X)[lane] = j;
        if (valid && side == 1) c.wb(X)[pos] = hb;
    }
    if (lane == 0) c.nw[X] = (uint32_t)__popc(wm);
    __syncwarp();
    if (lane == 0) mbar_arrive(c.bar_jobs(X));
    return pos;
}

__device__ __forceinline__ void publish_done(const Cta &c, int X, int lane)
{
    if (lane == 0) {
        c.nw[2 + X] = 1;
        mbar_arrive(c.bar_jobs(X));
    }
    __syncwarp();
}

// the hash of the lane's slot, after the set's sums are complete
__device__ __forceinline__ uint64_t slot_hash(const Cta &c, int X, int lane, bool valid, int side, uint32_t pos)
{
    uint64_t acc = 0;
    if (valid) {
        if (side == 0) {
            acc = c.vsum(X)[lane];
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) acc += c.part(X)[i * kSet + pos];
        }
    }
    return smix(acc);
}

} // namespace e4

// The level walk.  gsz walks (at most 48, chosen by the host so that every
// CTA steps the same number of groups, as nearly full as that allows) per
// group; a CTA steps its groups one after the other.
__device__ __forceinline__ bool walk_control(const WalkLaunch &w, uint32_t gsz, const e4::Cta &c, int X, int lane)
{
    using namespace e4;
    const LevelCtx &lv = w.lv;
    const uint32_t n_groups = ((uint32_t)w.n_walks + gsz - 1) / gsz;
    const uint32_t slot = (uint32_t)(X * kSet + lane);
    Tally t;
    uint32_t ph = 0;
    bool ok = true;
    for (uint32_t grp = blockIdx.x; grp < n_groups && ok; grp += gridDim.x) {
        const uint32_t local = grp * gsz + slot;
        const bool valid = lane < kSet && slot < gsz && local < (uint32_t)w.n_walks;
        WalkState st{};
        if (valid) st = w.walks[local];
        const uint32_t walk = w.walk_base + local; // index among all ranks' walks
        uint64_t dp = 0, ref = 0;
        bool store = false;
        for (uint32_t s = 0; s < w.steps; s++) {
            const Decoded d = decode(st.cur, lv);
            const uint32_t pos =
                publish(c, X, lane, valid, d.side, d.qpack, st.chunk, lv.h, c.chunk_base()[valid ? st.chunk : 0]);
            // the last step's distinguished points, while the workers run
            if (store) dp_insert(w, dp, ref, t);
            __syncwarp();
            if (!mbar_wait(c.bar_sums(X), ph)) {
                ok = false;
                break;
            }
            ph ^= 1u;
            const uint64_t y = slot_hash(c, X, lane, valid, d.side, pos) & lv.maskL;
            store = false;
            if (valid) {
                t.steps++;
                t.w += (uint32_t)d.side;
                st.len++;
                if ((y >> lv.dshift) == 0) {
                    t.dp++;
                    store = true;
                    dp = y;
                    ref = make_ref(walk, st.seq, st.len);
                    new_trail(st, walk, lv);
                } else if (st.len >= w.max_len) {
                    t.ab++;
                    new_trail(st, walk, lv);
                } else {
                    st.cur = y;
                }
            }
            __syncwarp();
        }
        if (store) dp_insert(w, dp, ref, t);
        if (valid) w.walks[local] = st;
        __syncwarp();
    }
    if (ok) publish_done(c, X, lane);
    unsigned long long v[7] = {t.steps, t.w, t.dp, t.ab, t.evicted, t.duplicate, t.pairs};
    const int idx[7] = {C_STEPS, C_WSTEPS, C_DPS, C_ABANDONED, C_EVICTED, C_DUPLICATE, C_PAIRS};
    for (int i = 0; i < 7; i++) {
#pragma unroll
        for (int o = 16; o; o >>= 1) v[i] += __shfl_xor_sync(0xFFFFFFFFu, v[i], o);
        if (lane == 0 && v[i]) atomicAdd(&w.counters[idx[i]], v[i]);
    }
    return ok;
}

__global__ void __launch_bounds__(e4::kThreads, 1) k_walks_e4(WalkLaunch w, uint32_t gsz)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const e4::Cta c = e4::cta_begin(w.lv, smem_raw, true);
    e4::load_c(w.lv, c);
    __syncthreads();
    e4::tmem_fence_after();
    bool ok;
    if (warp < e4::kWorkers) ok = e4::worker(w.lv, c, warp, lane);
    else if (warp == e4::kMmaWarp) ok = e4::mma_warp(c);
    else ok = walk_control(w, gsz, c, warp - e4::kCtlWarp, lane);
    if (!ok && lane == 0) atomicAdd(w.stall, 1u);
    // every product has completed (its sums were taken) unless a wait ran out
    e4::tmem_fence_before();
    __syncthreads();
    if (warp == 0) {
        e4::tmem_fence_after();
        e4::tmem_dealloc(c.tmem);
    }
}

} // namespace

cudaError_t launch_walks_e4(const WalkLaunch &w, cudaStream_t s)
{
    if (!w.stall) return cudaErrorInvalidValue; // a stalled wait must have somewhere to be counted
    const cudaError_t e =
        cudaFuncSetAttribute(k_walks_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    const uint32_t sms = (uint32_t)num_sms(), full = sms * e4::kSets * e4::kSet, n = (uint32_t)w.n_walks;
    if (n == 0) return cudaSuccess;
    const uint32_t rounds = (n + full - 1) / full;
    const uint32_t gsz = (n + rounds * sms - 1) / (rounds * sms);
    const uint32_t groups = (n + gsz - 1) / gsz;
    k_walks_e4<<<groups < sms ? groups : sms, e4::kThreads, e4::smem_bytes, s>>>(w, gsz);
    return cudaGetLastError();
}

int engine4_warps() { return e4::kWarps; }

} // namespace qcs
