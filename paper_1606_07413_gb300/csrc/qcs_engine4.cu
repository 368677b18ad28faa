// qcs_engine4.cu -- n = 4: the coset hash of many points at once, with the W
// side's contraction on the fifth-generation tensor cores (tcgen05.mma).
//
// The engine.  A CTA (one per SM) evaluates the hash of 72 points in flight,
// three sets of 24.  Its 28 warps have three roles:
//  - 24 workers, each owning one slot of every set.  Phase A of a set: a
//    point's fingerprint weights go through its adjoint stages (one warp per
//    point); a V point's weights are its column fingerprints, hashed at once;
//    a W point writes its weights as two f16 byte planes, two rows of the
//    set's B operand.  Phase E: the set's product D = C^^T B is read back from
//    tensor memory and hashed, column sums of every W point.
//  - one MMA warp: when all rows of a set are written it issues the product,
//    64 tcgen05.mma (128 x N x 16 each, N = twice the set's W points).
//  - one control warp per set: lane i is what uses slot i's hash (a walk).  It
//    takes the set's hashes, decides the slots' next points and publishes
//    them; table inserts and the like follow after that, off the critical
//    path.  All that a walk does besides f runs here on 24 lanes at once
//    instead of once per walk on 32.
//
// What bounds it.  A set's round is a chain: its points through A (about 3000
// cycles, the SM shared with the other sets), the product (1600: 16 cycles a
// tcgen05.mma with A in tensor memory, 40 in shared memory, whatever N), E
// (700), control (800).  With 48 points in flight (two sets of 24, or three
// of 16) that chain was the bound; with 72 it is issue: 75 % active at 582
// warp instructions a point.  The adjoint stages are the largest piece (88
// each, and at level 7 a point has 2.5 on average after the table's: 220), then
// the 255 column finalisers (18 for 32 columns: 144).
// 2^20 walks x 16 steps at level 7: 11.1 ms (1.51 G steps/s); two sets and
// 16 workers 14.9 ms; with mma.sync (12 stage and 8 MMA warps, C^'s fragments
// through tcgen05.ld, the rows through ldmatrix, 1073 instructions) 26.7 ms.
// B has room for 16 W points of a set's 24; more than 16 turn up in 3 % of
// the rounds, and those past 16 wait for the next round.
//
// Where C^ sits.  In f16 it is 256 KB.  As the A operand (M = columns of C^,
// K = its 512 numerator rows) its first 128 columns and K-blocks 0-7 of the
// other 128 are in tensor memory (320 of 512 columns), the rest (96 KB) in
// shared memory; that leaves 192 tensor-memory columns for three sets' D (3 x
// 2 x 32 f32 columns) and 96 KB of shared memory for three sets' B.
//
// Exactness.  B holds a weight's byte as the f16 with those bits, a subnormal
// (byte x 2^-24): no conversion.  C^'s entries are f16 integers (up to 2048),
// so every sum is a multiple of 2^-24.  Row 0 (the identity) has zero weight
// on both parts, so its K slots are free; the first one's B value is 1024 and
// its A value 0.75 / 1024 puts 0.75 on every sum.  While |P| (the integer dot
// product) and its partial sums stay below 2^22, a sum lies in [0.5, 1], whose
// f32 spacing is 2^-24: the accumulation is exact and the result's bits are
// 0x3F400000 + P, its low 16 bits those of P.  That holds when a column's
// absolute sum is at most kMaxColumnSum (qcs_internal.h), which the host
// checks.  (With 1024 + byte in B and 1.5 x 2^23 as the offset the bound was
// 1820, and C^ of 15 rotations went to the 32-bit-word kernels: 2^15 walks x
// 16 steps 15.4 ms there, 0.37 ms here.)
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "qcs_device.cuh"
#include "qcs_internal.h"
#include "qcs_rows.cuh"

namespace qcs {
namespace {

namespace e4 {

constexpr int kSet = 24, kSets = 3, kWorkers = kSet; // a worker owns one slot of each set
constexpr int kPairs = 16;                            // W points of a set that fit one product
static_assert(kWorkers % 4 == 0 && kPairs % 4 == 0 && kPairs / 4 < kWorkers / 4 && kSet <= 32, "units and slots");
constexpr int kMmaWarp = kWorkers, kCtlWarp = kWorkers + 1; // control warps kCtlWarp + set
constexpr int kWarps = kWorkers + 1 + kSets, kThreads = 32 * kWarps;
constexpr int kN = 2 * kPairs;              // columns of D per set and half
constexpr int kTmemK = 8;                   // K-blocks of C^'s second half held in tensor memory
constexpr int kDcol = 256 + 8 * kTmemK;     // tensor-memory column of D (set X, half h: + 2 kN X + kN h)
static_assert(kDcol + kSets * 2 * kN <= 512, "tensor memory");
constexpr uint32_t kInvalid = 1u << 31;
constexpr int kTaskWalks = 24; // of a batch: a third of the slots, for even shares

// one point to evaluate, published by the set's control warp
struct alignas(16) Job {
    uint64_t seq;   // the stages in order, one Pauli code (see code_of) per byte
    uint64_t PH;    // (pre with its low 16 bits clear) * the finaliser's first constant
    uint32_t pre16; // the low 16 bits of pre
    uint32_t info;  // stages | side << 8 | row pair << 16, or kInvalid
    uint64_t pad;
};
// shared memory
constexpr size_t off_A = 0;                                        // C^, second half, K-blocks 8..31: 6 chunks of 64 K
constexpr size_t off_B = off_A + 6 * 16384;                        // [set]: 8 chunks of 64 K x kN rows
constexpr size_t off_job = off_B + (size_t)kSets * 8 * kN * 128;   // Job [set][slot]
constexpr size_t off_wb = off_job + sizeof(Job) * kSets * kSet;    // HashBase [set][row pair]
constexpr int kParts = 16; // partial column sums of a W point
constexpr size_t off_part = off_wb + sizeof(HashBase) * kSets * kPairs; // u64 [set][part][row pair]
constexpr size_t off_vsum = off_part + kParts * sizeof(uint64_t) * kSets * kPairs; // u64 [set][slot]
constexpr size_t off_chunk = off_vsum + sizeof(uint64_t) * kSets * kSet; // HashBase [chunk]
constexpr size_t off_stage = off_chunk + sizeof(HashBase) * 256;   // stage table: u32 [side][code % 64][lane]
constexpr size_t off_nw = off_stage + 2 * 64 * 32 * sizeof(uint32_t);                  // u32 [set]: W points; [4 + set]: the set is done
constexpr size_t off_bar = off_nw + 32;                            // mbarriers: jobs, rows, product, sums [set]
constexpr size_t off_tmem = off_bar + 4 * kSets * sizeof(uint64_t);
constexpr size_t smem_bytes = off_tmem + 16;
static_assert(smem_bytes + sizeof(WalkLaunch) + 64 <= 227 * 1024, "shared memory of the n = 4 engine");

// a bounded wait gives up after this many SM clock cycles (about two seconds)
constexpr long long kWaitCycles = 1ll << 32;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- mbarriers: arrive has release and try_wait acquire semantics at CTA scope
__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_inval(uint64_t *b)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *b)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(b)) : "memory");
}

// One try: whether the phase of parity `ph` has completed, waiting
// (suspended) for at most a system-dependent time.
__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t ph)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(a), "r"(ph)
                 : "memory");
    return done != 0;
}

// Wait until the phase of parity `ph` has completed; false if the wait ran
// out.  Warp-uniform: true only once every lane saw the phase complete.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t ph, uint32_t all = 0xFFFFFFFFu)
{
    const uint32_t a = smem_u32(b);
    if (__all_sync(all, mbar_try(a, ph))) return true;
    const long long t0 = clock64();
    for (;;) {
        if (__all_sync(all, mbar_try(a, ph))) return true;
        // one lane's clock decides for the warp
        if (__shfl_sync(all, clock64() - t0, 0) > kWaitCycles) return false;
    }
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
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[4][4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[0][2]), "+r"(v[0][3]), "+r"(v[1][0]), "+r"(v[1][1]),
                   "+r"(v[1][2]), "+r"(v[1][3]), "+r"(v[2][0]), "+r"(v[2][1]), "+r"(v[2][2]), "+r"(v[2][3]),
                   "+r"(v[3][0]), "+r"(v[3][1]), "+r"(v[3][2]), "+r"(v[3][3])
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

// ---- one point on one warp (the rows and stages of qcs_rows.cuh, n = 4)

// sum mod 2^64 over the warp from three 32-bit reductions (see group_sum64 in qcs_walk.cu)
__device__ __forceinline__ uint64_t warp_sum64(uint64_t acc)
{
    const uint32_t lo = (uint32_t)acc, hi = (uint32_t)(acc >> 32);
    const uint32_t s_hi = __reduce_add_sync(0xFFFFFFFFu, hi);
    const uint32_t s_l0 = __reduce_add_sync(0xFFFFFFFFu, lo & 0xFFFFu);
    const uint32_t s_l1 = __reduce_add_sync(0xFFFFFFFFu, lo >> 16);
    return ((uint64_t)s_hi << 32) + ((uint64_t)s_l1 << 16) + (uint64_t)s_l0;
}

// The multiset sum of a V point: its weights, scaled by sqrt2^ev, are its
// column fingerprints' a parts (the scaling commutes with the stages, so only
// the part that ends up in a is scaled, once).
__device__ __forceinline__ uint64_t v_column_sum(const uint32_t (&ua)[8], const uint32_t (&ub)[8], int ev,
                                                 uint64_t PH, uint32_t pre16, int lane)
{
    const int sh = (ev >> 1) < 31 ? ev >> 1 : 31;
    uint64_t acc = 0;
    auto columns = [&](const uint32_t (&u)[8]) {
#pragma unroll
        for (int t = 0; t < 8; t++) {
            const uint64_t e = column_hash(u[t] << sh, PH, pre16);
            acc += (t == 0 && lane == 0) ? 0ull : e; // column 0, the identity, does not enter
        }
    };
    if (ev & 1) columns(ub);
    else columns(ua);
    return warp_sum64(acc);
}

// The stages of a point in order, a code per byte: V takes q_h first and goes
// down to q_1; W takes q_1 .. q_h, then the chunk.  A product of no rotations
// starts from code 0, the untouched weights; so does V's single rotation (its
// half product then is not one lookup).  What depends on the level alone is
// kept here; the control warps' time from a set's sums to its next points is
// on the sets' critical path.
struct Stages {
    int h, sh_v, sh_rev; // sh_v: shift that puts code 0 first; sh_rev: of the reversed bytes
    uint32_t ns_v, ns_w, sh_c; // stages of a side; shift of the chunk's code
    __device__ __forceinline__ explicit Stages(const LevelCtx &lv)
    {
        h = lv.h;
        sh_v = h == 1 ? 8 : 0;
        sh_rev = 64 - 8 * h;
        ns_v = (uint32_t)(h <= 1 ? h + 1 : h);
        sh_c = (uint32_t)(8 * (h == 0 ? 1 : h));
        ns_w = (uint32_t)(h == 0 ? 1 : h) + (uint32_t)(lv.k & 1);
    }
    __device__ __forceinline__ uint64_t chunk_code(uint32_t chunk) const
    {
        return (uint64_t)codes_of<4>(chunk) << sh_c; // chunk < 256
    }
    // q: the indices, q_1 in the lowest byte; cc: chunk_code
    __device__ __forceinline__ uint64_t seq(int side, uint64_t q, uint64_t cc) const
    {
        const uint32_t lo = codes_of<4>((uint32_t)q), hi = codes_of<4>((uint32_t)(q >> 32));
        if (side) return (((uint64_t)hi << 32) | lo) | cc;
        if (h == 0) return 0;
        const uint64_t rev = ((uint64_t)__byte_perm(lo, 0, 0x0123) << 32) | __byte_perm(hi, 0, 0x0123);
        return (rev >> sh_rev) << sh_v;
    }
};

// ---- roles

struct Cta {
    unsigned char *raw;
    uint64_t *bars; // per set: jobs, rows, product, sums
    uint32_t *nw;   // [set] W points, [4 + set] set done
    uint32_t tmem;
    uint32_t all; // all_lanes, for the control warps
    __device__ Job *jobs(int X) const { return reinterpret_cast<Job *>(raw + off_job) + X * kSet; }
    __device__ HashBase *wb(int X) const { return reinterpret_cast<HashBase *>(raw + off_wb) + X * kPairs; }
    __device__ uint64_t *part(int X) const { return reinterpret_cast<uint64_t *>(raw + off_part) + X * kParts * kPairs; }
    __device__ uint64_t *vsum(int X) const { return reinterpret_cast<uint64_t *>(raw + off_vsum) + X * kSet; }
    __device__ const HashBase *chunk_base() const { return reinterpret_cast<const HashBase *>(raw + off_chunk); }
    __device__ uint64_t *bar_jobs(int X) const { return bars + 4 * X; }
    __device__ uint64_t *bar_rows(int X) const { return bars + 4 * X + 1; }
    __device__ uint64_t *bar_prod(int X) const { return bars + 4 * X + 2; }
    __device__ uint64_t *bar_sums(int X) const { return bars + 4 * X + 3; }
};

// tensor memory and the stage table, once per launch; every thread calls it
__device__ __forceinline__ Cta cta_open(unsigned char *raw)
{
    Cta c;
    c.raw = raw;
    c.bars = reinterpret_cast<uint64_t *>(raw + off_bar);
    c.nw = reinterpret_cast<uint32_t *>(raw + off_nw);
    uint32_t *taddr = reinterpret_cast<uint32_t *>(raw + off_tmem);
    if (threadIdx.x < 32) tmem_alloc(taddr);
    uint32_t *tab = reinterpret_cast<uint32_t *>(raw + off_stage);
    for (int i = threadIdx.x; i < 2 * 64 * 32; i += kThreads)
        tab[i] = stage_word<4>((uint32_t)i >> 11, ((uint32_t)i >> 5) & 63u, (uint32_t)i & 31u);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    c.tmem = *taddr;
    c.all = all_lanes();
    return c;
}

__device__ __forceinline__ void cta_close(const Cta &c)
{
    if (threadIdx.x < 32) tmem_dealloc(c.tmem); // after cta_run's last barrier
}

// the barriers and the chunks' hash bases of a level
__device__ __forceinline__ void level_begin(const LevelCtx &lv, const Cta &c, bool again)
{
    if (threadIdx.x == 0) {
        for (int X = 0; X < kSets; X++) {
            if (again) {
                mbar_inval(c.bar_jobs(X));
                mbar_inval(c.bar_rows(X));
                mbar_inval(c.bar_prod(X));
                mbar_inval(c.bar_sums(X));
            }
            mbar_init(c.bar_jobs(X), 1);
            mbar_init(c.bar_rows(X), kWorkers);
            mbar_init(c.bar_prod(X), 1);
            mbar_init(c.bar_sums(X), kWorkers);
        }
        for (int i = 0; i < 8; i++) c.nw[i] = 0;
    }
    // base(chunk) = smix(smix(seed_H ^ version) ^ (n | k << 8 | chunk << 16 | K << 32))
    const uint64_t vmix = smix(kSeedH ^ (uint64_t)lv.version);
    for (int i = threadIdx.x; i < 256; i += kThreads) {
        const uint64_t tag =
            (uint64_t)lv.n | ((uint64_t)lv.k << 8) | ((uint64_t)i << 16) | ((uint64_t)(uint32_t)lv.K << 32);
        reinterpret_cast<HashBase *>(c.raw + off_chunk)[i] = hash_base(smix(vmix ^ tag));
    }
}

// C^ into tensor and shared memory; every thread calls it, and a barrier follows
__device__ __forceinline__ void load_c(const LevelCtx &lv, const Cta &c)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < kWorkers) {
        // warp w writes the tensor-memory lanes 32 (w % 4) ..: K-blocks
        // w / 4, w / 4 + 4, .. of its 32 columns of either half
        const uint32_t tq = c.tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        for (int b = warp >> 2; b < 32 + kTmemK; b += kWorkers / 4) {
            const uint4 *src = lv.Cm + (size_t)(b * 128 + 32 * (warp & 3) + lane) * 2;
            const uint4 w0 = __ldg(src), w1 = __ldg(src + 1);
            const uint32_t v[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
            tmem_st8(tq + 8u * (uint32_t)b, v);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    // the rest of the second half, as it lies in shared memory
    static_assert(kTmemK == 8, "cm_index");
    const uint4 *src = lv.Cm + (32 + kTmemK) * 256;
    uint4 *dst = reinterpret_cast<uint4 *>(c.raw + off_A);
    for (int i = threadIdx.x; i < 6 * 1024; i += kThreads) dst[i] = __ldg(src + i);
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
    const uint32_t *tab = reinterpret_cast<const uint32_t *>(c.raw + off_stage);
    uint32_t ua[8], ub[8];
    first_stage<4>(lv.T4[side], (uint32_t)seq & 0xFFu, lane, ua, ub);
#pragma unroll 1
    for (uint32_t i = 1; i < ns; i++)
        stage<4>(__shfl_sync(0xFFFFFFFFu, (uint32_t)(seq >> (8 * i)) & 0xFFu, 0), side, tab, lane, ua, ub);
    if (side == 0) {
        const uint64_t sum = v_column_sum(ua, ub, lv.ev, jp->PH, jp->pre16, lane);
        if (lane == 0) c.vsum(X)[slot] = sum;
    } else {
        // rows 2 pos and 2 pos + 1 of B: the low and the high byte plane.  The
        // lane's eight rows are the K indices 8 lane .. of each part, one
        // 16-byte unit; unit u of row r is at unit u ^ (r & 7) of its 128
        // bytes in chunk u / 8.
        const uint32_t r = 2 * (info >> 16), one = lane == 0 ? 0x6400u : 0u; // K slot 0
        unsigned char *b = c.raw + off_B + (size_t)X * 8 * kN * 128 + (size_t)(lane >> 3) * (kN * 128) + (r >> 3) * 1024;
#pragma unroll
        for (int p = 0; p < 2; p++) { // a, b part
            uint32_t lo[4], hi[4];
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const uint32_t w = p ? __byte_perm(ub[2 * e], ub[2 * e + 1], 0x5410)
                                     : __byte_perm(ua[2 * e], ua[2 * e + 1], 0x5410);
                lo[e] = w & 0x00FF00FFu;
                hi[e] = __byte_perm(w, p == 0 && e == 0 ? one : 0u, 0x7351);
                if (p == 0 && e == 0) lo[e] |= one;
            }
            unsigned char *d = b + (size_t)p * 4 * (kN * 128);
            const uint32_t u = (uint32_t)lane & 7u, r0 = r & 7u;
            *reinterpret_cast<uint4 *>(d + r0 * 128 + ((u ^ r0) * 16)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            *reinterpret_cast<uint4 *>(d + (r0 + 1) * 128 + ((u ^ (r0 + 1)) * 16)) =
                make_uint4(hi[0], hi[1], hi[2], hi[3]);
        }
    }
}

// Phase E, one unit: the 64 columns of C^ that quadrant qd holds (32 of each
// half), for row pairs 4 g .. 4 g + 3 (lane % 4).  Each lane sums eight
// columns, lanes 16 apart are added, and the control warp adds the rest.
__device__ __forceinline__ void unit_e(const Cta &c, int X, int g, int qd, int lane)
{
    const uint32_t t = c.tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(kDcol + X * 2 * kN + 8 * g);
    uint32_t v[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++) tmem_ld16x256(v[i], t + (uint32_t)(kN * (i >> 1)) + ((uint32_t)(16 * (i & 1)) << 16));
    const HashBase hb = c.wb(X)[4 * g + (lane & 3)];
    tmem_wait_ld(v);
    uint64_t acc = 0;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
            // the two planes' dot products (their low 16 bits are exact)
            const uint64_t z = column_hash(v[i][2 * e] + v[i][2 * e + 1] * 256u, hb.PH, hb.pre16);
            acc += (i == 0 && e == 0 && qd == 0 && lane < 4) ? 0ull : z; // column 0 does not enter
        }
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 16);
    if (lane < 16) c.part(X)[(4 * qd + (lane >> 2)) * kPairs + 4 * g + (lane & 3)] = acc;
}

// worker warp w: slot w of every set; false if a wait ran out.  The phases run A(0) E(2) A(1) E(0) A(2) E(1): between a set's
// A and its E (the product) and between its E and its next A (the control
// warp) lie another set's A and E.
__device__ __forceinline__ bool worker(const LevelCtx &lv, const Cta &c, int w, int lane)
{
    uint32_t live = (1u << kSets) - 1; // sets that are not done
    uint32_t ph = 0;
    int u = w >> 2; // units of all sets in turn over the quadrant's warps
    for (bool first = true;; first = false) {
#pragma unroll 1
        for (int X = 0; X < kSets; X++) {
            if ((live >> X) & 1u) {
                if (!mbar_wait(c.bar_jobs(X), ph)) return false;
                if (c.nw[4 + X]) live &= ~(1u << X);
            }
            if ((live >> X) & 1u) {
                point_a(lv, c, X, w, lane);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(c.bar_rows(X));
            }
            const int Y = X == 0 ? kSets - 1 : X - 1; // set 2's E is the last iteration's
            if (!((live >> Y) & 1u) || (X == 0 && first)) continue;
            if (!mbar_wait(c.bar_prod(Y), X == 0 ? ph ^ 1u : ph)) return false;
            tmem_fence_after();
            const int units = (int)(c.nw[Y] + 3) >> 2; // at most kPairs / 4, fewer than the quadrant's warps
            if (u < units) unit_e(c, Y, u, w & 3, lane);
            u = u < units ? u + kWorkers / 4 - units : u - units;
            tmem_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(c.bar_sums(Y));
        }
        if (!live) return true;
        ph ^= 1u;
    }
}

// the MMA warp (the whole warp calls it); false if a wait ran out
__device__ __forceinline__ bool mma_warp(const Cta &c)
{
    uint32_t live = (1u << kSets) - 1;
    uint32_t ph = 0;
    const uint64_t a0 = smem_desc(smem_u32(c.raw + off_A));
    while (live) {
#pragma unroll 1
        for (int X = 0; X < kSets; X++) {
            if (!((live >> X) & 1u)) continue;
            bool ok = mbar_wait(c.bar_jobs(X), ph);
            if (ok && c.nw[4 + X]) {
                live &= ~(1u << X);
                continue;
            }
            ok = ok && mbar_wait(c.bar_rows(X), ph);
            if (!ok) {
                // the products in flight (sets before X: this round's, the others': the last)
                for (int Y = 0; Y < kSets; Y++)
                    if ((live >> Y) & 1u) mbar_wait(c.bar_prod(Y), Y < X ? ph : ph ^ 1u);
                return false;
            }
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

// the rotations of a state, as decode's, q_1 in the lowest byte
__device__ __forceinline__ uint64_t rotations(uint64_t x, const LevelCtx &lv)
{
    uint64_t q = 0, f = x >> 1;
#pragma unroll
    for (int j = 0; j < 8; j++)
        if (j < lv.h) {
            q |= (uint64_t)((((uint32_t)f & lv.fmask) * 255u >> lv.ell) + 1u) << (8 * j);
            f >>= lv.ell;
        }
    return q;
}

// Publish the set's next points: lane i < kSet passes slot i's (valid or
// not).  The W points are numbered here; those past kPairs (3 % of a set's
// rounds have any) wait for the next round, where `late` puts them first.
// Whole warp.  Returns whether the lane's point is evaluated this round, and
// its number.
__device__ __forceinline__ bool publish(const Cta &c, int X, int lane, bool valid, bool late, int side, uint64_t seq,
                                        uint32_t ns, HashBase hb, uint32_t *pos_out)
{
    const bool isw = valid && side == 1;
    const uint32_t before = (1u << lane) - 1u;
    const uint32_t all = __ballot_sync(c.all, isw), first = __ballot_sync(c.all, isw && late);
    const uint32_t pos = (uint32_t)(late ? __popc(first & before) : __popc(first) + __popc(all & ~first & before));
    const bool go = valid && (!isw || pos < (uint32_t)kPairs);
    if (lane < kSet) {
        Job *j = c.jobs(X) + lane;
        const uint32_t info = go ? ns | (uint32_t)side << 8 | pos << 16 : kInvalid;
        *reinterpret_cast<uint4 *>(j) =
            make_uint4((uint32_t)seq, (uint32_t)(seq >> 32), (uint32_t)hb.PH, (uint32_t)(hb.PH >> 32));
        *(reinterpret_cast<uint2 *>(j) + 2) = make_uint2(hb.pre16, info);
        if (go && isw)
            *reinterpret_cast<uint4 *>(c.wb(X) + pos) =
                make_uint4((uint32_t)hb.PH, (uint32_t)(hb.PH >> 32), hb.pre16, 0);
    }
    if (lane == 0) c.nw[X] = min((uint32_t)__popc(all), (uint32_t)kPairs);
    __syncwarp(c.all);
    if (lane == 0) mbar_arrive(c.bar_jobs(X));
    *pos_out = pos;
    return go;
}

__device__ __forceinline__ void publish_done(const Cta &c, int X, int lane)
{
    if (lane == 0) {
        c.nw[4 + X] = 1;
        mbar_arrive(c.bar_jobs(X));
    }
    __syncwarp(c.all);
}

// the hash of the lane's slot, after the set's sums are complete
__device__ __forceinline__ uint64_t slot_hash(const Cta &c, int X, int lane, int side, uint32_t pos)
{
    uint64_t acc = c.vsum(X)[lane < kSet ? lane : 0];
    if (side) {
        uint64_t v[kParts];
#pragma unroll
        for (int i = 0; i < kParts; i++) v[i] = c.part(X)[i * kPairs + pos];
#pragma unroll
        for (int o = kParts / 2; o; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; i++) v[i] += v[i + o];
        acc = v[0];
    }
    return smix(acc);
}

// Run the roles over one level's points: ctl(X) is control warp X's part.
// Every thread calls it; false (for all) if a wait ran out.
template <class Ctl>
__device__ __forceinline__ bool cta_run(const LevelCtx &lv, const Cta &c, bool again, Ctl ctl)
{
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    level_begin(lv, c, again);
    load_c(lv, c);
    __syncthreads();
    tmem_fence_after();
    bool ok;
    if (warp < kWorkers) ok = worker(lv, c, warp, lane);
    else if (warp == kMmaWarp) ok = mma_warp(c);
    else ok = ctl(warp - kCtlWarp, lane);
    // every product has completed: its sums were taken, or the MMA warp waited for it
    tmem_fence_before();
    ok = __syncthreads_and(ok) != 0;
    tmem_fence_after();
    return ok;
}

} // namespace e4

// of a batch: the job's round is not complete (the host reads the counter)
__device__ __forceinline__ void count_stall(const BatchArgs &a, uint32_t job)
{
    if (threadIdx.x == 0) atomicAdd(a.jobs[job].stall, 1u);
}

// The level walk: the CTA's slot i (lane * kSets + X) < slots steps walk
// first + i and every stride-th after it below n, one after the other.
template <typename WL>
__device__ __forceinline__ bool walk_control(const WL &w, uint32_t first, uint32_t slots, uint32_t stride, uint32_t n,
                                             const e4::Cta &c, int X, int lane)
{
    using namespace e4;
    const LevelCtx &lv = w.lv;
    const Stages sg(lv);
    const uint32_t slot = (uint32_t)(lane * kSets + X);
    uint32_t local = first + slot; // below 2^25: n <= 2^24, and a slot stops past n
    bool valid = lane < kSet && slot < slots && local < n, late = false, ok = true;
    WalkState st{}, nx{};
    if (valid) st = w.walks[local];
    uint32_t left = w.steps, ph = 0;
    Tally t;
    HashBase hb = c.chunk_base()[st.chunk];
    uint64_t cc = sg.chunk_code(st.chunk), dp = 0, ref = 0;
    bool store = false;
    while (__any_sync(c.all, valid)) {
        const int side = (int)(st.cur & 1);
        uint32_t pos;
        const bool go = publish(c, X, lane, valid, late, side, sg.seq(side, rotations(st.cur, lv), cc),
                                side ? sg.ns_w : sg.ns_v, hb, &pos);
        // while the workers run: the last step's distinguished points, and
        // the slot's next walk if this is its walk's last step
        if (store) dp_insert(w, dp, ref, t);
        store = false;
        late = valid && !go;
        const bool last = st.len + 1 >= w.max_len; // this step ends the trail in any case
        const uint32_t walk = w.walk_base + local; // index among all ranks' walks
        if (go && left == 1 && local + stride < n) nx = w.walks[local + stride];
        __syncwarp(c.all);
        if (!mbar_wait(c.bar_sums(X), ph, c.all)) {
            ok = false;
            break;
        }
        ph ^= 1u;
        const uint64_t y = slot_hash(c, X, lane, go ? side : 0, pos) & lv.maskL;
        if (go) {
            st.cur = y;
            st.len++;
            left--;
            t.steps++;
            t.w += side;
            const bool is_dp = (y >> lv.dshift) == 0;
            if (is_dp || last || left == 0) {
                if (is_dp) {
                    t.dp++;
                    store = true;
                    dp = y;
                    ref = make_ref(walk, st.seq, st.len);
                } else if (last) {
                    t.ab++;
                }
                if (is_dp || last) new_trail<4>(st, walk, lv);
                if (left == 0) {
                    w.walks[local] = st;
                    local += stride;
                    valid = local < n;
                    st = nx;
                    left = w.steps;
                }
                hb = c.chunk_base()[st.chunk];
                cc = sg.chunk_code(st.chunk);
            }
        }
        __syncwarp(c.all);
    }
    if (ok && store) dp_insert(w, dp, ref, t);
    __syncwarp(c.all);
    if (ok) publish_done(c, X, lane);
    unsigned long long v[7] = {t.steps, t.w, t.dp, t.ab, t.evicted, t.duplicate, t.pairs};
    const int idx[7] = {C_STEPS, C_WSTEPS, C_DPS, C_ABANDONED, C_EVICTED, C_DUPLICATE, C_PAIRS};
    for (int i = 0; i < 7; i++) {
#pragma unroll
        for (int o = 16; o; o >>= 1) v[i] += __shfl_xor_sync(c.all, v[i], o);
        if (lane == 0 && v[i]) atomicAdd(&w.counters[idx[i]], v[i]);
    }
    return ok;
}

// gsz (at most kSets * kSet) is chosen by the host so that every slot has the
// same number of walks, as nearly as that allows
__global__ void __launch_bounds__(e4::kThreads, 1) k_walks_e4(WalkLaunch w, uint32_t gsz)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const e4::Cta c = e4::cta_open(smem_raw);
    const bool ok = e4::cta_run(w.lv, c, false, [&](int X, int lane) {
        return walk_control(w, blockIdx.x * gsz, gsz, gsz * gridDim.x, (uint32_t)w.n_walks, c, X, lane);
    });
    if (!ok && threadIdx.x == 0) atomicAdd(w.stall, 1u);
    e4::cta_close(c);
}

// Many jobs in one launch (walk_shares): the CTA runs the engine once for each
// job that its share meets, so C^ is reloaded only where the job changes.
__global__ void __launch_bounds__(e4::kThreads, 1) k_walks_batch_e4(BatchArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ WalkLaunch sw;
    constexpr uint32_t per = e4::kSets * e4::kSet; // slots
    e4::Cta c;
    bool again = false;
    walk_shares(
        a, blockIdx.x, gridDim.x, 1, e4::kTaskWalks,
        [&](uint32_t job, uint32_t first, uint32_t most) {
            if (!again) c = e4::cta_open(smem_raw);
            if (threadIdx.x == 0) sw = a.jobs[job];
            __syncthreads();
            const uint32_t end = min((uint32_t)sw.n_walks, first + most);
            // the slots' shares as even as they can be
            const uint32_t cnt = end > first ? end - first : 0, rounds = (cnt + per - 1) / per;
            const uint32_t slots = rounds ? (cnt + rounds - 1) / rounds : 0;
            const bool ok = e4::cta_run(sw.lv, c, again, [&](int X, int lane) {
                return walk_control(sw, first, slots, slots, end, c, X, lane);
            });
            __syncthreads(); // before sw changes
            again = true;
            return ok;
        },
        [&](uint32_t job) { count_stall(a, job); });
    if (again) e4::cta_close(c);
}

// The re-walk of a level's merges (Sec. 3, Fig. 2; the same steps and classes
// as rewalk_resume in qcs_walk.cu): slot lane * kSets + X re-walks merges
// claimed one after the other from the device cursor, evaluating f at one
// state a round: the longer trail until both are aligned, then a and b in
// turn.  The next merge is claimed and its starts computed while the workers
// run.  cursor (device or shared memory): the next merge; cnt: the list's end;
// slots: slots that take merges (a short list is spread over all CTAs).  A merge to a warp with the dp4a step, a
// search at level 6 (theta 1/2, 2^26 steps) took 240 ms; so it takes 109.
template <typename WL>
__device__ __forceinline__ bool rewalk_control(const WL &w, uint32_t *cursor, uint32_t cnt, uint32_t slots,
                                               const e4::Cta &c, int X, int lane)
{
    using namespace e4;
    const unsigned kAll = c.all;
    const LevelCtx &lv = w.lv;
    const Stages sg(lv);
    const bool mine = lane < kSet && (uint32_t)(lane * kSets + X) < slots;
    uint32_t cls[6] = {0, 0, 0, 0, 0, 0}, ph = 0;
    unsigned long long nf = 0;
    uint64_t a = 0, b = 0, fa = 0, na = 0, nb = 0, cc = 0;
    uint32_t la = 0, lb = 0, chunk = 0, nla = 0, nlb = 0, nchunk = 0, used = 0;
    bool active = false, second = false, checked = false, have = false, more = mine, late = false, ok = true;
    HashBase hb{};

    // give every slot without a next merge one that needs an evaluation, as
    // far as the list goes; the others are classified at once
    auto fetch = [&]() {
        for (;;) {
            const bool need = more && !have;
            const uint32_t m = __ballot_sync(kAll, need);
            if (!m) break;
            uint32_t base = 0;
            if (lane == __ffs((int)m) - 1) base = atomicAdd(cursor, (uint32_t)__popc(m));
            base = __shfl_sync(kAll, base, __ffs((int)m) - 1);
            if (need) {
                const uint32_t p = base + (uint32_t)__popc(m & ((1u << lane) - 1u));
                if (p >= cnt) {
                    more = false;
                } else {
                    const Merge q = load_merge<4>(w, p);
                    const bool bad = q.ca != q.cb || q.la > kMaxRewalkLen || q.lb > kMaxRewalkLen;
                    const bool hood = !bad && q.la == q.lb && q.a == q.b, none = bad || (!hood && (q.la | q.lb) == 0);
                    cls[0] += hood;
                    cls[5] += none;
                    if (!hood && !none) {
                        const bool sw = q.la < q.lb; // a is the longer trail
                        na = sw ? q.b : q.a;
                        nb = sw ? q.a : q.b;
                        nla = sw ? q.lb : q.la;
                        nlb = sw ? q.la : q.lb;
                        nchunk = q.ca;
                        have = true;
                    }
                }
            }
            __syncwarp(c.all);
        }
    };
    // whether the merge goes on; if not it is classified or carried
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
            carry_merge(w, a, la, b, lb, chunk);
            active = false;
        }
    };
    auto take = [&]() {
        if (active || !have) return;
        a = na;
        b = nb;
        la = nla;
        lb = nlb;
        chunk = nchunk;
        hb = c.chunk_base()[chunk];
        cc = sg.chunk_code(chunk);
        used = 0;
        second = checked = have = false;
        active = true;
        settle();
    };
    fetch();
    take();
    __syncwarp(c.all);
    // `more` alone: every merge that was taken was carried at once (a budget of
    // one evaluation and aligned trails), and the list goes on
    while (__any_sync(kAll, active || have || more)) {
        const uint64_t x = second ? b : a;
        const int side = (int)(x & 1);
        uint32_t pos;
        const bool go = publish(c, X, lane, active, late, side, sg.seq(side, rotations(x, lv), cc),
                                side ? sg.ns_w : sg.ns_v, hb, &pos);
        late = active && !go;
        fetch();
        if (!mbar_wait(c.bar_sums(X), ph, c.all)) {
            ok = false;
            break;
        }
        ph ^= 1u;
        const uint64_t y = slot_hash(c, X, lane, go ? side : 0, pos) & lv.maskL;
        if (go) {
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
                    const bool claw = ((a ^ b) & 1) != 0, same = rotations(a, lv) == rotations(b, lv);
                    if (claw) append_claw(w, a, b, chunk);
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
        take();
        __syncwarp(c.all);
    }
    if (ok) publish_done(c, X, lane);
    unsigned long long v[8] = {cls[0], cls[1], cls[2], cls[3], cls[4], cls[5], cls[3], nf};
    const int idx[8] = {C_CLS0, C_CLS0 + 1, C_CLS0 + 2, C_CLS0 + 3, C_CLS0 + 4, C_CLS0 + 5, C_CANDS, C_RSTEPS};
#pragma unroll
    for (int i = 0; i < 8; i++) {
#pragma unroll
        for (int o = 16; o; o >>= 1) v[i] += __shfl_xor_sync(kAll, v[i], o);
        if (lane == 0 && v[i]) atomicAdd(&w.counters[idx[i]], v[i]);
    }
    return ok;
}

__global__ void __launch_bounds__(e4::kThreads, 1) k_rewalk_e4(WalkLaunch w)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t cnt = w.pend_in_n + min(*w.qhead, w.qcap);
    if (cnt <= blockIdx.x) return; // no merge for this CTA
    const e4::Cta c = e4::cta_open(smem_raw);
    const bool ok = e4::cta_run(w.lv, c, false, [&](int X, int lane) {
        return rewalk_control(w, w.rw_next, cnt, (cnt + gridDim.x - 1) / gridDim.x, c, X, lane);
    });
    if (!ok && threadIdx.x == 0) atomicAdd(w.stall, 1u);
    e4::cta_close(c);
}

// The batched re-walk: each CTA takes its share of all jobs' merges
// (merge_shares) and reloads C^ where the share enters another job.
__global__ void __launch_bounds__(e4::kThreads, 1) k_rewalk_batch_e4(BatchArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ WalkLaunch sw;
    __shared__ uint32_t cursor;
    e4::Cta c;
    bool again = false;
    merge_shares(
        a, blockIdx.x, gridDim.x,
        [&](uint32_t job, uint32_t p0, uint32_t p1) {
            if (!again) c = e4::cta_open(smem_raw);
            if (threadIdx.x == 0) {
                sw = a.jobs[job];
                cursor = p0;
            }
            __syncthreads();
            const bool ok = e4::cta_run(sw.lv, c, again, [&](int X, int lane) {
                return rewalk_control(sw, &cursor, p1, p1 - p0, c, X, lane);
            });
            __syncthreads(); // before sw and cursor change
            again = true;
            return ok;
        },
        [&](uint32_t job) { count_stall(a, job); });
    if (again) e4::cta_close(c);
}

// W points of the exhaustive pass: the set takes kPairs points a round (all
// of them need a row pair; which of its slots they sit on turns with the set,
// so that every worker has two points a round), inserts or probes the last
// round's keys and counts its indices on while the workers run.
__device__ __forceinline__ bool certify_control(const CertArgs &a, const e4::Cta &c, int X, int lane)
{
    using namespace e4;
    const Stages sg(a.lv);
    const int my = (lane + kSet - (kSet - kPairs) * X) % kSet, h = a.lv.h;
    const bool mine = lane < kSet && my < kPairs, has_chunk = (a.lv.k & 1) != 0;
    const int nd = h + (has_chunk ? 1 : 0);
    const uint64_t hmask = h >= 8 ? ~0ull : (1ull << (8 * h)) - 1;
    const uint64_t stride = (uint64_t)gridDim.x * kSets * kPairs;
    uint64_t i = ((uint64_t)blockIdx.x * kSets + (uint64_t)X) * kPairs + (uint64_t)my;
    // While i + stride < count, the stride is below xi^nd and its nd digits
    // are exact; otherwise the slot ends before the sum is used.
    const uint64_t sdig = base_xi_digits(stride, 255, nd);
    uint64_t dig = mine && i < a.count ? base_xi_digits(a.first + i, 255, nd) : 0;
    const HashBase hb = hash_base(a.base);
    uint64_t key = 0, idx = 0;
    uint32_t ph = 0, stored = 0;
    bool have = false, valid = mine && i < a.count, ok = true;
    while (__any_sync(c.all, valid)) {
        const uint64_t q = (dig & hmask) + (0x0101010101010101ull & hmask);
        const uint32_t chunk = has_chunk ? (uint32_t)((dig >> (8 * h)) & 0xFFu) + 1 : 0u;
        uint32_t pos;
        publish(c, X, lane, valid, false, 1, sg.seq(1, q, has_chunk ? sg.chunk_code(chunk) : 0), sg.ns_w, hb, &pos);
        if (a.insert) cert_insert_warp(a, c.all, have, key, idx, lane, stored);
        else if (have) cert_probe(a, key, idx);
        __syncwarp(c.all);
        have = valid;
        idx = a.first + i;
        i += stride;
        valid = mine && i < a.count;
        dig = add_base_xi(dig, sdig, 255, nd);
        if (!mbar_wait(c.bar_sums(X), ph, c.all)) {
            ok = false;
            break;
        }
        ph ^= 1u;
        key = slot_hash(c, X, lane, have ? 1 : 0, pos);
        if (key == ~0ull) key = ~0ull - 1; // ~0 marks an empty slot
    }
    if (ok) {
        if (a.insert) cert_insert_warp(a, c.all, have, key, idx, lane, stored);
        else if (have) cert_probe(a, key, idx);
        __syncwarp(c.all);
        publish_done(c, X, lane);
    }
    stored = __reduce_add_sync(c.all, stored);
    if (lane == 0) cert_count(a, stored);
    return ok;
}

__global__ void __launch_bounds__(e4::kThreads, 1) k_certify_e4(CertArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const e4::Cta c = e4::cta_open(smem_raw);
    const bool ok = e4::cta_run(a.lv, c, false, [&](int X, int lane) { return certify_control(a, c, X, lane); });
    if (!ok && threadIdx.x == 0) atomicAdd(a.n_pairs + 1, 1u);
    e4::cta_close(c);
}

// f of a list of states: slot lane * kSets + X of the CTA takes the state of
// that index among the CTA's and every stride-th after it; a state is loaded
// a round before it is published and its image stored a round after.  us a
// launch at level 7 against the dp4a warp-per-state kernel: 16 states 15.5 /
// 19.4 (C^ is read once a CTA here too), 2500 19 / 30, 10000 24 / 53, 50021
// 48 / 164; 33 of the last are the engine's rate and 15 its set-up.
__device__ __forceinline__ bool list_control(const LevelCtx &lv, uint32_t chunk, const uint64_t *in, uint64_t *out,
                                             uint8_t *is_dp, size_t count, uint32_t slots, const e4::Cta &c,
                                             uint64_t *next, int X, int lane)
{
    using namespace e4;
    const Stages sg(lv);
    const uint32_t slot = (uint32_t)(lane * kSets + X);
    const size_t stride = (size_t)slots * gridDim.x;
    const uint64_t cc = (lv.k & 1) ? sg.chunk_code(chunk) : 0ull;
    const HashBase hb = c.chunk_base()[chunk];
    size_t i = (size_t)blockIdx.x * slots + slot, at = 0;
    bool valid = lane < kSet && slot < slots && i < count, late = false, have = false, ok = true;
    uint64_t x = valid ? in[i] : 0ull, nx = 0, y = 0;
    uint32_t ph = 0;
    while (__any_sync(c.all, valid)) {
        const int side = (int)(x & 1);
        uint32_t pos;
        const bool go = publish(c, X, lane, valid, late, side, sg.seq(side, rotations(x, lv), cc),
                                side ? sg.ns_w : sg.ns_v, hb, &pos);
        if (have) {
            out[at] = y;
            if (is_dp) is_dp[at] = (uint8_t)((y >> lv.dshift) == 0);
        }
        if (go && i + stride < count) nx = in[i + stride];
        late = valid && !go;
        __syncwarp(c.all);
        if (!mbar_wait(c.bar_sums(X), ph, c.all)) {
            ok = false;
            break;
        }
        ph ^= 1u;
        y = slot_hash(c, X, lane, go ? side : 0, pos) & lv.maskL;
        have = go;
        at = i;
        if (go) {
            i += stride;
            valid = i < count;
            x = nx;
        }
    }
    if (ok && have) {
        out[at] = y;
        if (is_dp) is_dp[at] = (uint8_t)((y >> lv.dshift) == 0);
    }
    if (lane < kSet) next[slot] = i; // the slot's first state not stored
    __syncwarp(c.all);
    if (ok) publish_done(c, X, lane);
    return ok;
}

// The full hash of one point by one warp alone, no barrier but its own: what
// is left when a bounded wait ran out and the caller has no status to report
// it by.  buf: 512 words of shared memory of the warp's own.
__device__ __noinline__ uint64_t hash_alone(const LevelCtx &lv, const uint32_t *tab, int side, uint64_t seq, int ns,
                                            HashBase hb, uint32_t *buf, int lane)
{
    using namespace e4;
    uint32_t ua[8], ub[8];
    first_stage<4>(lv.T4[side], (uint32_t)seq & 0xFFu, lane, ua, ub);
    for (int i = 1; i < ns; i++) stage<4>((uint32_t)(seq >> (8 * i)) & 0xFFu, (uint32_t)side, tab, lane, ua, ub);
    if (side == 0) return smix(v_column_sum(ua, ub, lv.ev, hb.PH, hb.pre16, lane));
    for (int t = 0; t < 8; t++) {
        buf[8 * lane + t] = ua[t];
        buf[256 + 8 * lane + t] = ub[t];
    }
    __syncwarp();
    uint64_t acc = 0;
    for (int t = 0; t < 8; t++) {
        const int Q = lane + 32 * t;
        const unsigned short *col = reinterpret_cast<const unsigned short *>(lv.Cm);
        uint32_t l = 0;
        for (uint32_t k = 0; k < 512; k++)
            if (k & 255u) // the identity's weights are zero
                l += buf[k] * (uint32_t)(int)__half2float(__ushort_as_half(col[cm_index((uint32_t)Q, k)]));
        if (Q) acc += column_hash(l, hb.PH, hb.pre16);
    }
    __syncwarp();
    return smix(warp_sum64(acc));
}

__global__ void __launch_bounds__(e4::kThreads, 1) k_walk_step_e4(LevelCtx lv, uint32_t chunk, const uint64_t *in,
                                                                  uint64_t *out, uint8_t *is_dp, size_t count,
                                                                  uint32_t slots)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    using namespace e4;
    __shared__ uint64_t next[kSets * kSet];
    const Cta c = cta_open(smem_raw);
    const bool ok = cta_run(lv, c, false, [&](int X, int lane) {
        return list_control(lv, chunk, in, out, is_dp, count, slots, c, next, X, lane);
    });
    if (!ok) { // the call has no status: what is left is evaluated without the engine
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const uint32_t *tab = reinterpret_cast<const uint32_t *>(smem_raw + off_stage);
        uint32_t *buf = reinterpret_cast<uint32_t *>(smem_raw + off_B) + 512 * warp;
        const Stages sg(lv);
        const uint64_t cc = (lv.k & 1) ? sg.chunk_code(chunk) : 0ull;
        for (uint32_t j = (uint32_t)warp; j < slots; j += kWarps)
            for (size_t i = next[j]; i < count; i += (size_t)slots * gridDim.x) {
                const uint64_t x = in[i];
                const int side = (int)(x & 1);
                const uint64_t y = hash_alone(lv, tab, side, sg.seq(side, rotations(x, lv), cc),
                                              (int)(side ? sg.ns_w : sg.ns_v), c.chunk_base()[chunk], buf, lane) &
                                   lv.maskL;
                __syncwarp();
                if (lane == 0) {
                    out[i] = y;
                    if (is_dp) is_dp[i] = (uint8_t)((y >> lv.dshift) == 0);
                }
            }
    }
    cta_close(c);
}

} // namespace

cudaError_t launch_walks_e4(const WalkLaunch &w, cudaStream_t s)
{
    if (!w.stall) return cudaErrorInvalidValue; // a stalled wait must have somewhere to be counted
    const cudaError_t e =
        cudaFuncSetAttribute(k_walks_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    if (w.n_walks <= 0) return cudaSuccess;
    // every slot the same number of walks, as few as the slots allow
    const uint32_t sms = (uint32_t)num_sms(), full = sms * e4::kSets * e4::kSet, n = (uint32_t)w.n_walks;
    const uint32_t rounds = (n + full - 1) / full;
    const uint32_t gsz = (n + rounds * sms - 1) / (rounds * sms);
    const uint32_t ctas = (n + gsz - 1) / gsz;
    k_walks_e4<<<ctas < sms ? ctas : sms, e4::kThreads, e4::smem_bytes, s>>>(w, gsz);
    return cudaGetLastError();
}

cudaError_t launch_rewalk_e4(const WalkLaunch &w, cudaStream_t s)
{
    if (!w.stall || !w.rw_next) return cudaErrorInvalidValue;
    const cudaError_t e =
        cudaFuncSetAttribute(k_rewalk_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    k_rewalk_e4<<<(unsigned)num_sms(), e4::kThreads, e4::smem_bytes, s>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_certify_e4(const CertArgs &a, cudaStream_t s)
{
    if (a.count == 0) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(k_certify_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    const uint64_t ctas = (a.count + e4::kSets * e4::kPairs - 1) / (e4::kSets * e4::kPairs), sms = (uint64_t)num_sms();
    k_certify_e4<<<(unsigned)(ctas < sms ? ctas : sms), e4::kThreads, e4::smem_bytes, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_walk_step_e4(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp,
                                size_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(k_walk_step_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    const size_t sms = (size_t)num_sms(), full = sms * e4::kSets * e4::kSet, rounds = (count + full - 1) / full;
    const size_t slots = (count + rounds * sms - 1) / (rounds * sms), ctas = (count + slots - 1) / slots;
    k_walk_step_e4<<<(unsigned)(ctas < sms ? ctas : sms), e4::kThreads, e4::smem_bytes, s>>>(
        lv, (uint32_t)chunk, in, out, is_dp, count, (uint32_t)slots);
    return cudaGetLastError();
}

cudaError_t launch_walks_batch_e4(const BatchArgs &a, cudaStream_t s)
{
    const cudaError_t e =
        cudaFuncSetAttribute(k_walks_batch_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    k_walks_batch_e4<<<(unsigned)num_sms(), e4::kThreads, e4::smem_bytes, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_rewalk_batch_e4(const BatchArgs &a, cudaStream_t s)
{
    const cudaError_t e =
        cudaFuncSetAttribute(k_rewalk_batch_e4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e4::smem_bytes);
    if (e != cudaSuccess) return e;
    k_rewalk_batch_e4<<<(unsigned)num_sms(), e4::kThreads, e4::smem_bytes, s>>>(a);
    return cudaGetLastError();
}

int engine4_warps() { return e4::kWarps; }

int engine4_walks_per_task() { return e4::kTaskWalks; }

} // namespace qcs
