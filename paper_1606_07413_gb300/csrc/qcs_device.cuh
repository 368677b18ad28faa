// qcs_device.cuh -- device functions shared by the kernels of qcs_walk.cu and
// qcs_engine4.cu: the hash finaliser, the state's decoding, trail starts and
// references, and the distinguished-point table's insert.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "qcs_internal.h"
#include "qcs_shares.h"

namespace qcs {
namespace {

__device__ __forceinline__ uint64_t smix(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// smix(base ^ phi) for phi < 2^30, given pre = base ^ (base >> 30): the
// first xorshift of the finaliser cannot see phi (it shifts by 30), so
// (base ^ phi) ^ ((base ^ phi) >> 30) = pre ^ phi, and the rest follows.
// The same value as smix(base ^ phi), one 64-bit xorshift cheaper per column.
__device__ __forceinline__ uint64_t smix_pre(uint64_t pre, uint32_t phi)
{
    uint64_t z = (pre ^ (uint64_t)phi) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ uint32_t shl32(uint32_t v, int s) { return s >= 32 ? 0u : v << s; }

struct Decoded {
    int side;
    uint64_t qpack; // q_1 .. q_h, 8 bits each (q <= 255)
};

// mu (Sec. 2, the state is a concatenation of per-rotation codes): bit 0 is
// the side; rotation j reads the ell-bit field at bit 1 + ell j and maps its
// value v onto the xi non-identity Paulis as q_j = floor(v xi / 2^ell) + 1.
__device__ __forceinline__ Decoded decode(uint64_t x, const LevelCtx &lv)
{
    Decoded d;
    d.side = (int)(x & 1);
    d.qpack = 0;
    uint64_t f = x >> 1;
    for (int j = 0; j < lv.h; j++) {
        const uint32_t v = (uint32_t)f & lv.fmask;
        d.qpack |= (uint64_t)(((v * lv.xi) >> lv.ell) + 1) << (8 * j);
        f >>= lv.ell;
    }
    return d;
}

// starting state and chunk of trail (walk, seq) in the current version
__device__ __forceinline__ uint64_t trail_start(const LevelCtx &lv, uint32_t walk, uint32_t seq)
{
    seq &= (1u << kRefSeqBits) - 1;
    return smix(lv.seed ^ smix(((uint64_t)walk << 32) | seq) ^ ((uint64_t)lv.version << 40)) & lv.maskL;
}
// NQ: the qubit count where the kernel knows it (the divisions are then by a
// constant), else 0
template <int NQ = 0>
__device__ __forceinline__ uint32_t trail_chunk(const LevelCtx &lv, uint64_t start)
{
    if (!lv.n_chunks) return 0u;
    // n_chunks = xi = 4^n - 1: with v = hi 2^32 + lo and 2^32 = 1 (mod xi)
    // for n = 1, 2, 4 (4^n's powers reach 2^32) and 4 (mod 63) for n = 3
    const uint64_t v = smix(start ^ 0x5851F42D4C957F2Dull);
    const uint32_t xi = NQ ? (1u << (2 * NQ)) - 1u : (uint32_t)lv.n_chunks;
    const uint32_t r32 = (NQ ? NQ : lv.n) == 3 ? 4u : 1u;
    return 1u + ((uint32_t)(v >> 32) % xi * r32 + (uint32_t)v % xi) % xi;
}
__device__ __forceinline__ uint64_t make_ref(uint32_t walk, uint32_t seq, uint32_t len)
{
    return (uint64_t)walk | ((uint64_t)(seq & ((1u << kRefSeqBits) - 1)) << kRefWalkBits) |
           ((uint64_t)len << (kRefWalkBits + kRefSeqBits));
}
__device__ __forceinline__ void split_ref(uint64_t ref, uint32_t &walk, uint32_t &seq, uint32_t &len)
{
    walk = (uint32_t)(ref & ((1u << kRefWalkBits) - 1));
    seq = (uint32_t)((ref >> kRefWalkBits) & ((1u << kRefSeqBits) - 1));
    len = (uint32_t)(ref >> (kRefWalkBits + kRefSeqBits));
}

template <int NQ = 0>
__device__ __forceinline__ void new_trail(WalkState &st, uint32_t walk, const LevelCtx &lv)
{
    st.seq++;
    st.start = trail_start(lv, walk, st.seq);
    st.cur = st.start;
    st.len = 0;
    st.chunk = trail_chunk<NQ>(lv, st.start);
}

// per-walk-group tallies, added to the job's counters by the group's first
// lane (the quads keep theirs in 32 bits: a walk's are at most a launch's steps)
template <typename T>
struct TallyOf {
    T steps = 0, w = 0, dp = 0, ab = 0, evicted = 0, duplicate = 0, pairs = 0;
};
using Tally = TallyOf<unsigned long long>;

// Store the distinguished point (Sec. 3: the triple start, end, length) in
// the slot its value hashes to, keeping the newest trail there (one 128-bit
// atomic exchange, never a wait).  If the slot held the same point from
// another trail the two trails merged: queue them for the re-walk.
template <typename WL, typename T>
__device__ void dp_insert(const WL &w, uint64_t dp, uint64_t ref, TallyOf<T> &c)
{
    if (w.outbox) {
        // DP-owner sharding: the point goes to its owner's table after the exchange
        const uint32_t idx = atomicAdd(w.ohead, 1u);
        if (idx < w.ocap) {
            Slot o;
            o.key = dp;
            o.ref = ref;
            w.outbox[idx] = o;
        }
        return;
    }
    Slot nv;
    nv.key = dp;
    nv.ref = ref;
    Slot *s = &w.table[smix(dp) & w.table_mask];
    const Slot old = atomicExch(s, nv);
    if (old.key == dp) {
        if (old.ref == ref) {
            c.duplicate++;
            return;
        }
        c.pairs++;
        const uint32_t idx = atomicAdd(w.qhead, 1u);
        if (idx < w.qcap) {
            Pair p;
            p.ref_a = old.ref;
            p.ref_b = ref;
            p.dp = dp;
            w.queue[idx] = p;
        }
    } else if (old.key != kEmptyKey) {
        c.evicted++;
    }
}

// All lanes of a warp, as a mask whose value the compiler does not know, so
// that every vote and shuffle under it first brings the warp's lanes together.
// Warps that run a re-walk or the like on every lane need that: under a
// constant full mask the compiled code of the n = 4 engine's budgeted re-walk
// did not, the lanes whose merge was carried in the middle of a round ran on a
// round behind the others, each group voting for itself, merges were lost and
// bounded waits ran out.  It costs the engine 1.5 % (2^20 walks x 16 steps
// 10.95 -> 11.1 ms); its workers' and its MMA warp's waits, which no lane
// reaches alone, keep the constant (with the mask there too 11.9 ms).
__device__ __forceinline__ uint32_t all_lanes()
{
    uint32_t lt, ge;
    asm volatile("mov.u32 %0, %%lanemask_lt;\n\tmov.u32 %1, %%lanemask_ge;" : "=r"(lt), "=r"(ge));
    return lt | ge;
}

constexpr uint32_t kMaxRewalkLen = 1u << 20; // longer trails are reported as no merge

// A merge of a launch's work list: first the re-walks carried from the
// previous launch or round, then this launch's queued merges.  The two states
// with the steps each still has to the shared point, and their trails' chunks
// (different ones: the same value reached in two chunks' functions, no merge).
struct Merge {
    uint64_t a, b;
    uint32_t la, lb, ca, cb;
};
template <int NQ = 0, typename WL>
__device__ __forceinline__ Merge load_merge(const WL &w, uint32_t p)
{
    Merge m;
    if (p < w.pend_in_n) {
        const Pending q = w.pend_in[p];
        m.a = q.a;
        m.b = q.b;
        m.la = q.la;
        m.lb = q.lb;
        m.ca = m.cb = q.chunk;
    } else {
        const Pair P = w.queue[p - w.pend_in_n];
        uint32_t wa, sa, wb, sb;
        split_ref(P.ref_a, wa, sa, m.la);
        split_ref(P.ref_b, wb, sb, m.lb);
        m.a = trail_start(w.lv, wa, sa);
        m.b = trail_start(w.lv, wb, sb);
        m.ca = trail_chunk<NQ>(w.lv, m.a);
        m.cb = trail_chunk<NQ>(w.lv, m.b);
    }
    return m;
}

// budget spent: carry the re-walk to the next launch or round (if there is room)
template <typename WL>
__device__ __forceinline__ void carry_merge(const WL &w, uint64_t a, uint32_t la, uint64_t b, uint32_t lb,
                                            uint32_t chunk)
{
    const uint32_t idx = atomicAdd(w.pend_out_n, 1u);
    if (idx < w.pend_cap) {
        Pending q;
        q.a = a;
        q.b = b;
        q.la = la;
        q.lb = lb;
        q.chunk = chunk;
        q.pad = 0;
        w.pend_out[idx] = q;
    }
}

template <typename WL>
__device__ __forceinline__ void append_claw(const WL &w, uint64_t a, uint64_t b, uint32_t chunk)
{
    const uint32_t idx = atomicAdd(w.ccount, 1u);
    if (idx < w.ccap) {
        Cand c;
        c.a = a;
        c.b = b;
        c.chunk = chunk;
        c.pad = 0;
        w.cands[idx] = c;
    }
}

// The nd low base-xi digits of v, digit j in byte j (xi <= 255).
__device__ __forceinline__ uint64_t base_xi_digits(uint64_t v, uint32_t xi, int nd)
{
    uint64_t r = 0;
    for (int j = 0; j < nd; j++) {
        r |= (v % xi) << (8 * j);
        v /= xi;
    }
    return r;
}

// (d + s) mod xi^nd on packed base-xi digits (digit j in byte j, nd <= 8).
__device__ __forceinline__ uint64_t add_base_xi(uint64_t d, uint64_t s, uint32_t xi, int nd)
{
    uint64_t r = 0;
    uint32_t carry = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        if (j < nd) {
            uint32_t t = (uint32_t)((d >> (8 * j)) & 0xFFu) + (uint32_t)((s >> (8 * j)) & 0xFFu) + carry;
            carry = t >= xi ? 1u : 0u;
            t -= carry * xi;
            r |= (uint64_t)t << (8 * j);
        }
    }
    return r;
}

// Exhaustive pass: the key table.  A key's slots are s, s + d, s + 2d, .. with
// a step d of its own (odd, so the sequence meets every slot); it goes to the
// first empty one, and at most half of the table is full, so there is one.
// The step matters: a point with two equal neighbouring rotations is in the
// coset of the rest, so at h = 3 each single rotation's key is stored some 640
// times.  In one run of slots they held up every probe that met the run
// (16.6 M probes of a 2^25-slot table: 110 ms on the n = 4 engine, 12 ms with
// steps).
struct CertProbe {
    uint64_t s, d;
    __device__ __forceinline__ CertProbe(uint64_t key, uint64_t mask)
    {
        const uint64_t z = smix(key);
        s = z & mask;
        d = (z >> 32) | 1u;
    }
};

__device__ __forceinline__ bool cert_put(const CertArgs &a, uint64_t slot, uint64_t key, uint64_t idx)
{
    if (atomicCAS(reinterpret_cast<unsigned long long *>(&a.table[slot].key), ~0ull, (unsigned long long)key) != ~0ull)
        return false;
    a.table[slot].idx = idx;
    return true;
}

// whether the key was stored (it is unless the table is full)
__device__ __forceinline__ bool cert_insert(const CertArgs &a, uint64_t key, uint64_t idx)
{
    CertProbe p(key, a.mask);
    for (uint64_t probe = 0; probe <= a.mask; probe++, p.s = (p.s + p.d) & a.mask)
        if (cert_put(a, p.s, key, idx)) return true;
    return false;
}

// keys stored by this launch, for the host's check that none was lost
__device__ __forceinline__ void cert_count(const CertArgs &a, uint32_t stored)
{
    if (stored) atomicAdd(reinterpret_cast<unsigned long long *>(a.n_pairs + 2), (unsigned long long)stored);
}

// The same for a whole warp, a point to a valid lane: after a few tries the
// warp looks for each remaining lane's empty slot together, 32 slots at a
// time (the 640th copy of a key alone: as many dependent exchanges; 16.6 M
// points at n = 4: 35 ms lane by lane, 7 ms so).  all: all_lanes(), which
// brings the lanes back together after their tries; a vote that some of them
// missed would lose their keys.  stored counts the lane's keys.
__device__ __forceinline__ void cert_insert_warp(const CertArgs &a, uint32_t all, bool valid, uint64_t key,
                                                 uint64_t idx, int lane, uint32_t &stored)
{
    CertProbe p(key, a.mask);
    bool left = valid;
    for (int probe = 0; probe < 6 && left; probe++, p.s = (p.s + p.d) & a.mask) left = !cert_put(a, p.s, key, idx);
    stored += valid && !left;
    __syncwarp(all);
    uint32_t todo;
    while ((todo = __ballot_sync(all, left)) != 0) {
        const int src = __ffs((int)todo) - 1;
        const uint64_t d = __shfl_sync(all, p.d, src);
        uint64_t at = __shfl_sync(all, p.s, src);
        for (uint64_t probe = 0; probe <= a.mask; probe += 32) {
            const uint64_t k =
                *reinterpret_cast<volatile const uint64_t *>(&a.table[(at + d * (uint64_t)lane) & a.mask].key);
            uint32_t empty = __ballot_sync(all, k == ~0ull);
            bool done = false;
            while (empty && !done) { // another warp may take the slot first
                const uint64_t slot = (at + d * (uint64_t)(__ffs((int)empty) - 1)) & a.mask;
                if (lane == src) done = cert_put(a, slot, key, idx);
                stored += done;
                done = __shfl_sync(all, done, src);
                empty &= empty - 1;
            }
            if (done) break;
            at = (at + 32 * d) & a.mask;
        }
        if (lane == src) left = false;
    }
}

// a probing point's matches are queued
__device__ __forceinline__ void cert_probe(const CertArgs &a, uint64_t key, uint64_t idx)
{
    CertProbe p(key, a.mask);
    for (uint64_t probe = 0; probe <= a.mask; probe++, p.s = (p.s + p.d) & a.mask) {
        const uint64_t k2 = a.table[p.s].key;
        if (k2 == ~0ull) return;
        if (k2 == key) {
            const uint32_t n = atomicAdd(a.n_pairs, 1u);
            if (n < a.cap) {
                a.pairs[2 * (size_t)n] = a.table[p.s].idx;
                a.pairs[2 * (size_t)n + 1] = idx;
            }
        }
    }
}

} // namespace
} // namespace qcs
