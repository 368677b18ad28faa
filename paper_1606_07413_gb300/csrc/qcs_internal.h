// qcs_internal.h -- structures shared by the host library (qcs_api.cpp,
// qcs_exact.cpp) and the CUDA kernels (qcs_walk.cu).  Not part of the ABI.
#pragma once

#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#include "qcs.h"

namespace qcs {

constexpr int kMaxH = 8;              // h = floor(k/2) <= 7 for k <= 15
constexpr uint64_t kEmptyKey = ~0ull; // empty table slot / unwritten meta

// Hash constants of the walk function (written specification, Sec. 2 "h"):
// SplitMix64 output function (Steele, Lea & Flood 2014), its stream increment,
// and two seeds taken from the fractional parts of sqrt2 and sqrt3.
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kSeedU = 0x6A09E667F3BCC908ull;
constexpr uint64_t kSeedH = 0xBB67AE8584CAA73Bull;

// Rows on lanes (qcs_rows.cuh): lane l (2n - 3 bits: z_0 .. z_(n-2), then x_0
// .. x_(n-3) of the row's Pauli index) and t (3 bits: x_(n-2), z_(n-1),
// x_(n-1)) to the row, and a Pauli's code, the same bits in that order (t
// above l).  n >= 2.
__host__ __device__ constexpr uint32_t row_of(int n, uint32_t l, uint32_t t)
{
    const uint32_t z = (l & ((1u << (n - 1)) - 1u)) | ((t >> 1) & 1u) << (n - 1);
    const uint32_t x = (l >> (n - 1)) | (t & 1u) << (n - 2) | ((t >> 2) & 1u) << (n - 1);
    return x << n | z;
}
// Rows on quads (qcs_quad.cu, n = 2 and 3): lane q is qubit 0 (z0 | x0 << 1),
// row t the other qubits: z1 above t8 = (x1 z2 x2) at n = 3, (z1 x1) at n = 2.
// The Pauli index, and the Pauli of a code (row_of's order).
__host__ __device__ constexpr uint32_t quad_row(int n, uint32_t q, uint32_t t)
{
    return n == 2 ? (q & 1u) | (t & 1u) << 1 | (q >> 1) << 2 | (t >> 1) << 3
                  : row_of(3, (q & 1u) | (t >> 3) << 1 | (q >> 1) << 2, t & 7u);
}
__host__ __device__ constexpr uint32_t code_pauli(int n, uint32_t code)
{
    return row_of(n, code & ((1u << (2 * n - 3)) - 1u), code >> (2 * n - 3));
}
// C^ suits the tensor-core kernels (qcs_engine4.cu, qcs_quad.cu) when the
// absolute values of a column's entries add up to at most kMaxColumnSum (the
// weights are bytes: 255 * 16448 < 2^22) and none is above 2048 (exact in
// f16).  By orthogonality a column's squares a^2 + 2 b^2 add up to 2^E, so its
// sum is at most 2^n sqrt(1.5 * 2^E), 14189 at n = 4, E = 19, and an entry at
// most 2^(E / 2).
constexpr int kMaxColumnSum = 16448, kMaxEntry = 2048;
constexpr uint16_t kCmBias = 0x1200; // 0.75 / 1024 in f16
// n = 4: f16 index in LevelCtx::Cm of column Q, K index k (part * 256 + 8 l + t).
// First what goes to tensor memory, columns 0 .. 127 and then K-blocks 0 .. 7
// of the others, 16 K of one column together; then K-blocks 8 .. 31 of columns
// 128 .. 255 as they lie in shared memory (chunks of 64 K x 128 columns, 128
// bytes a column, its 16-byte units exchanged by the 128-byte swizzle).
__host__ __device__ constexpr uint32_t cm_index(uint32_t Q, uint32_t k)
{
    const uint32_t r = Q & 127u;
    return Q < 128 || k < 128
               ? (((Q >> 7) * 32 + (k >> 4)) * 128 + r) * 16 + (k & 15u)
               : 40 * 2048 + ((k >> 6) - 2) * 8192 + (r >> 3) * 512 + (r & 7u) * 64 + ((((k >> 3) ^ r) & 7u) * 8) + (k & 7u);
}

// Everything a warp needs to evaluate one step f of the walk at one level.
struct LevelCtx {
    // C^ numerators mod 2^32 as (a, b), 4^n x 4^n.  With W = lanes_per_walk(n)
    // and R = 4^n / W, row i, column Q = sub + W t sits at i * 4^n + sub * R +
    // t, so one lane's R columns of a row are contiguous.
    const uint2 *C32;
    // n >= 3: C^ as signed byte quads when every entry fits in int8, else
    // null.  Quad q holds rows 4q .. 4q+3 of a column as the bytes 0 .. 3 of
    // one word.  uint4 number (q R/2 + j) W + sub carries, for the columns
    // Q0 = sub + 2 W j and Q1 = Q0 + W, the words (a-quad Q0, b-quad Q0,
    // a-quad Q1, b-quad Q1) (W, R as above).
    const uint4 *Cq;
    // n >= 2, when C^ suits the tensor-core kernels, else null: C^ as their
    // f16 operand, the a and then the b part of every row against every
    // column; the identity's row holds kCmBias and 0.  n = 4
    // (qcs_engine4.cu): ordered by cm_index, K index part * 256 + 8 l + t is
    // row row_of(4, l, t).  n = 2, 3 (qcs_quad.cu): A's fragments, uint4
    // [tile][part][k-step][lane].
    const uint4 *Cm;
    // n >= 2: the weights after the first adjoint stage, as T1, by code: word
    // code * 4^n + 8 l + t is row row_of(n, l, t)'s Ua | Ub << 16 after the
    // Pauli of that code; code 0 holds the weights themselves.
    const uint4 *T4[2];
    // n = 2, 3: the quad kernels' tables (stage_tables): T, uint4 [side][code]
    // [row / 4][lane], the weights after the first stage of a code, Ua | Ub <<
    // 16 of four rows; then the signs, i8 [side][code][lane][row], 1 where the
    // row commutes; then the anticommuting rows, u32 [code][lane], a bit per row
    const uint4 *quad;
    const uint2 *U;    // fingerprint weights (Ua, Ub) per row, 4^n
    // The weights after the first adjoint stage of a side (index 0: V, 1: W),
    // mod 2^16, for every Pauli: entry e = q_a - 1, where q_a is the side's
    // first stage rotation (V: q_h; W: q_1); word e 4^n + row = Ua | Ub << 16.
    const uint32_t *T1[2];
    // rotation masks: for Pauli p and lane sub, the 16-bit word at index
    // p W + sub has bit t set when row sub + W t anticommutes with p and bit
    // 8 + t when the sign s(p, row) is +1 (t < R <= 8).  4^n x W uint16,
    // read as 4^n W / 2 uint32.
    const uint32_t *coef;
    uint64_t xi_h;     // xi^h, the number of rotation tuples per side
    int32_t ell;       // bits of one rotation's field in the state: min(16, (L - 1) / h)
    uint32_t fmask;    // 2^ell - 1
    uint64_t maskL;    // low L bits
    uint32_t xi;       // 4^n - 1
    int32_t n, k, h, K;
    int32_t ev;        // V side is raised from exponent h to K: ev = K - h
    int32_t dshift;    // distinguished iff (x >> dshift) == 0, dshift = L - d_theta
    uint32_t version;
    int32_t n_chunks;  // xi for odd k (trail chunk drawn from its start), 0 for even k
    uint64_t seed;     // seed of trail starting points
};

// A trail is named by a 64-bit reference: walk index (24 bits), its trail
// sequence number (23 bits) and its length (17 bits).  Its starting state and
// chunk are recomputed from (seed, version, walk, sequence), so a
// distinguished point fits in one 16-byte slot.
constexpr int kRefWalkBits = 24, kRefSeqBits = 23, kRefLenBits = 17;
constexpr uint32_t kMaxWalks = 1u << kRefWalkBits;
constexpr uint32_t kMaxTrailLen = (1u << kRefLenBits) - 1;

// One distinguished point (Sec. 3: the triple start, end, length, with the
// start and length folded into the trail reference).  16 bytes, written with
// one 128-bit atomic exchange: the memory keeps the newest trail per slot.
struct alignas(16) Slot {
    unsigned long long key; // the distinguished state, kEmptyKey when free
    unsigned long long ref; // trail reference
};

// Two trails that reached one distinguished point with different starts.
struct Pair {
    unsigned long long ref_a, ref_b, dp;
};

// A merge of a V point and a W point (before the exact check).
struct Cand {
    unsigned long long a, b;
    uint32_t chunk, pad;
};

// A re-walk carried over to the next round (batched search): the two
// states, the steps each trail still has to its shared point, the chunk.
struct Pending {
    unsigned long long a, b;
    uint32_t la, lb, chunk, pad;
};

struct RewalkOut {
    int32_t cls;    // QCS_MERGE_* (claw = candidate before the exact check)
    uint32_t chunk; // chunk of the pair (odd k)
    unsigned long long a, b;
};

// Per-walk state kept in device memory between launches.  32 bytes.
struct WalkState {
    unsigned long long start, cur;
    uint32_t len, chunk, seq, pad;
};

enum Counter {
    C_STEPS = 0,
    C_WSTEPS,      // steps on the W side (these do the 4^n x 4^n contraction)
    C_DPS,
    C_ABANDONED,
    C_EVICTED,     // distinguished points overwritten by another one
    C_DUPLICATE,
    C_PAIRS,       // merges pushed (including overflowed ones)
    C_CANDS,       // claw candidates found by the re-walk (including overflowed ones)
    C_RSTEPS,      // walk steps taken by the re-walk (evaluations of f)
    C_CLS0,        // re-walk classes QCS_MERGE_ROBIN_HOOD .. QCS_MERGE_NO_MERGE at C_CLS0 + class
    C_STALLED = C_CLS0 + 6, // CTAs of the n = 4 engine that gave up on a bounded wait, in a batch once for every job left (low word)
    C_NCOUNTERS
};

struct WalkLaunch {
    LevelCtx lv;
    WalkState *walks;
    int32_t n_walks;    // walks advanced by this launch
    uint32_t steps;     // steps per walk in this launch
    uint32_t max_len;
    Slot *table;
    uint64_t table_mask;
    Pair *queue;
    uint32_t *qhead;
    uint32_t qcap;
    Cand *cands;
    uint32_t *ccount;
    uint32_t ccap;
    unsigned long long *counters;
    // batched search: a re-walk gets rewalk_budget evaluations of f per
    // round (0: no bound); unfinished ones go to pend_out and come back as
    // pend_in in the next round, before that round's new merges
    uint32_t rewalk_budget;
    uint32_t pend_in_n, pend_cap;
    const Pending *pend_in;
    Pending *pend_out;
    uint32_t *pend_out_n;
    int32_t shape;       // launch shape of k_walks (host-side choice; see launch_shapes)
    // DP-owner sharding (Sec. 4.2 collectors): the walks of this launch are
    // walks walk_base .. walk_base + n_walks - 1 of all ranks' walks (trail
    // references and starts use the global index), and with outbox set their
    // distinguished points go to outbox (up to ocap, *ohead counts every one)
    // instead of the local table, for the exchange with their owners
    uint32_t walk_base;
    uint32_t ocap;
    Slot *outbox;
    uint32_t *ohead;
    // single-target re-walk: merges are claimed from this device counter
    // (zeroed before the launch); null: a fixed stride (the batched re-walk)
    uint32_t *rw_next;
    uint32_t rw_last; // merges of the level's last re-walk (0: unknown), for the choice of this one's kernels
    // the n = 4 engine counts here the CTAs that gave up on a bounded wait
    // (the launch's results are then invalid); it refuses to launch without it
    uint32_t *stall;
};

// Many jobs in one launch: per qubit count, the device list of tasks
// (job index, first walk) with walks_per_task(n) walks each, and of job indices.
struct BatchArgs {
    const WalkLaunch *jobs;   // device array indexed by job
    const uint32_t *tasks;    // 2 * n_tasks entries
    const uint32_t *n_tasks;  // device scalar
    const uint32_t *job_ids;  // jobs of this qubit count
    const uint32_t *n_jobs;   // device scalar
};
// Exhaustive meet-in-the-middle pass over one level (Sec. 2 Eq. mitm, the
// collision search's exact counterpart): the points of the smaller side are
// hashed into an open-addressing table of coset keys, then every point of
// the other side probes it and each key match is queued for the exact host
// check.  Point index -> rotations: base-xi digits, q_j = digit_j + 1 (q_1
// the lowest digit); a W index of a level context with odd k is chunk-major,
// chunk = index / xi^h + 1.
struct alignas(16) CertSlot {
    uint64_t key; // ~0: empty
    uint64_t idx; // stored point index
};

struct CertArgs {
    LevelCtx lv;       // the side's level context (lv.h rotations per point)
    int32_t side;      // which product a point is: 0 V, 1 W
    int32_t insert;    // 1: insert the points' keys, 0: probe the table with them
    uint64_t first;    // point indices [first, first + count)
    uint64_t count;
    uint64_t xi_h;     // rotation tuples of the h-rotation W side (chunk stride)
    uint64_t base;     // hash base of the keys, the same for every chunk
    CertSlot *table;
    uint64_t mask;     // table slots - 1 (a power of two, at least twice the stored points)
    uint64_t *pairs;   // key matches (stored index, probing index)
    uint32_t *n_pairs; // [0] matches found (may exceed cap; only cap are stored); [1] the engine's bounded
                       // waits that ran out (the points are then not all evaluated); [2, 3] as one word,
                       // keys stored
    uint32_t cap;
};
cudaError_t launch_certify(const CertArgs &a, cudaStream_t s);
cudaError_t launch_certify_v(const CertArgs &a, cudaStream_t s); // V points at n >= 3 (qcs_certify.cu)
cudaError_t launch_certify_e4(const CertArgs &a, cudaStream_t s); // W points at n = 4 with lv.Cm set (qcs_engine4.cu)
// Host driver of the exhaustive pass (qcs_certify_level); *got = verified claw.
int certify_level(::qcs_problem *P, int k, cudaStream_t s, bool *got);

// The exhaustive pass as a resumable job (the batch engine runs a bounded
// share of it per round): cert_begin allocates and clears the key table,
// cert_advance evaluates points (stored side first, then probing slices,
// each slice's key matches checked exactly) until the pass is done or
// `budget` streamed-point equivalents are spent (*used), and cert_end frees
// the table and folds the pass into the problem's result (QCS_ERR_OVERFLOW:
// done without a claw but inconclusive).  certify_level is the three in a row.
struct CertPass {
    static constexpr uint32_t kCap = 1u << 16;          // key matches read back per slice
    static constexpr uint64_t kSliceMin = 1ull << 20;   // probing points of the first slice
    static constexpr uint64_t kSliceMax = 1ull << 24;   // slices double up to this
    int k = 0, h = 0;
    bool v_heavy = false, done = false, got = false, overflow = false;
    uint64_t xi = 0, xi_h = 0, n_probe = 0, stored = 0, probed = 0, slice = 0;
    uint64_t table_bytes = 0;
    int64_t d2h = 0;
    LevelCtx lv_store{}, lv_probe{};
    CertArgs a{};
    // matches are few and seldom: read into pageable memory (pinning and
    // unpinning 1 MB for each pass took longer than a small level's kernels)
    uint32_t hN[4] = {0, 0, 0, 0};
    uint64_t *hPairs = nullptr;
};
int cert_begin(::qcs_problem *P, int k, cudaStream_t s, CertPass *c);
int cert_advance(::qcs_problem *P, CertPass *c, cudaStream_t s, uint64_t budget, uint64_t *used);
int cert_end(::qcs_problem *P, CertPass *c, cudaStream_t s);
uint64_t exhaustive_points(const ::qcs_problem *P, int k); // V + W points of level k
bool exhaustive_eligible(const ::qcs_problem *P, int k);   // within exhaustive_log2 and device memory

int walks_per_task(int n, int shape); // walks (lane groups) per CTA of the walk kernels of that launch shape
int lanes_per_walk(int n); // lanes of a warp that evaluate one walk (the device layouts follow it)
int launch_shapes(int n);                    // launch shapes of the walk kernels for n qubits
int shape_warps_of(int n, int shape);        // warps per CTA of a launch shape
int shape_min_blocks_of(int n, int shape);   // minimum resident CTAs per SM (the register cap) of a shape

// ---- kernel launchers (qcs_walk.cu); all return cudaError_t of the launch ----
cudaError_t launch_walks_batch(int n, int shape, const BatchArgs &a, cudaStream_t s);
cudaError_t launch_rewalk_batch(int n, const BatchArgs &a, cudaStream_t s);
cudaError_t launch_walk_step(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out,
                             uint8_t *is_dp, size_t count, cudaStream_t s);
cudaError_t launch_init_walks(const WalkLaunch &w, cudaStream_t s);
cudaError_t launch_walks(const WalkLaunch &w, cudaStream_t s);
// C^ (LevelCtx::C32) as the tensor-core kernels' operand (LevelCtx::Cm), n >= 2
cudaError_t launch_operand(int n, const uint2 *C32, uint16_t *Cm, cudaStream_t s);
// n = 4 with lv.Cm set: the level walk on the tensor-core engine (qcs_engine4.cu)
cudaError_t launch_walks_e4(const WalkLaunch &w, cudaStream_t s);
// the re-walk of a level's merges on the engine
cudaError_t launch_rewalk_e4(const WalkLaunch &w, cudaStream_t s);
// f of a list of states on the engine
cudaError_t launch_walk_step_e4(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp,
                                size_t count, cudaStream_t s);
// jobs of a batch on the engine: tasks of engine4_walks_per_task() walks, and the jobs' re-walks
cudaError_t launch_walks_batch_e4(const BatchArgs &a, cudaStream_t s);
cudaError_t launch_rewalk_batch_e4(const BatchArgs &a, cudaStream_t s);
int engine4_warps(); // warps of its CTA
int engine4_walks_per_task();
// n = 2, 3 with lv.Cm set: eight walks to a warp (qcs_quad.cu)
cudaError_t launch_walks_q(const WalkLaunch &w, cudaStream_t s);
// (least: the kernel leaves shorter merge lists alone; their length is known on the device only)
cudaError_t launch_rewalk_q(const WalkLaunch &w, uint32_t least, cudaStream_t s);
// jobs of a batch: tasks of quad_walks_per_task() walks, and the jobs' re-walks
cudaError_t launch_walks_batch_q(int n, const BatchArgs &a, cudaStream_t s);
cudaError_t launch_rewalk_batch_q(int n, const BatchArgs &a, cudaStream_t s);
int quad_walks_per_task();
// below this many n = 3 walks in a launch the warp-per-walk kernels are the
// faster ones (us a launch of 64 steps at theta 2^-8 and 2^-2, quads / them:
// 1000 walks 127 / 94 and 179 / 109, 3000 129 / 144 and 185 / 168, 10000 208 /
// 318 and 257 / 364; 4566 walks x 55 steps at theta 1/2 167 / 164).  At n = 2
// quads always win (200 walks: 53 / 88 and 86 / 112).  Where C^ is not int8
// those kernels take 32-bit words: 1000 walks 126 / 152 and 175 / 152, 3000
// 127 / 228 and 182 / 240.
constexpr uint32_t kQuadWalks3 = 6144, kQuadWalksWide3 = 2048;
// An n = 3 re-walk of fewer merges than this is left to the lane-group kernel:
// a merge is a chain of evaluations of f, a quad's evaluation takes two to
// three times as long as a lane group's, and only enough merges make up for it
// (us, quads / lane groups: theta 1/2, 1600 merges 71 / 36, 29400 70 / 69,
// 47000 98 / 113, 312000 314 / 551; theta 2^-4, 5600 376 / 143, 50300 427 /
// 390, 103000 697 / 775; theta 2^-8, 3980 672 / 228, 40600 1038 / 1215; C^ in
// 32-bit words, theta 2^-4, 9500 303 / 219, 22800 379 / 343, 48500 426 / 551).
// At n = 2 a quad loses little (2360 merges 41 / 32, 29600 43 / 55) and the
// choice, a second launch, costs 4 us: quads always.
constexpr uint32_t kQuadMerges3 = 40960, kQuadMergesWide3 = 20480;
cudaError_t launch_walk_step_q(const LevelCtx &lv, int chunk, const uint64_t *in, uint64_t *out, uint8_t *is_dp,
                               size_t count, cudaStream_t s);
// DP-owner sharding: insert `count` distinguished points {dp, trail ref}
// into w's table (merges queued as by the walk), and bin points by owner
// rank (owner_of in qcs_walk.cu): out gets the points grouped by owner in
// rank order, counts[r] the number for rank r (device arrays; counts has
// 2 n_owners entries, the first n_owners zeroed by the caller, the rest are
// the scatter's cursors)
cudaError_t launch_insert_points(const WalkLaunch &w, const Slot *pts, uint32_t count, cudaStream_t s);
cudaError_t launch_bin_owners(const Slot *in, uint32_t count, uint32_t n_owners, Slot *out, uint32_t *counts,
                              cudaStream_t s);
cudaError_t launch_rewalk_pairs(const WalkLaunch &w, cudaStream_t s);
cudaError_t launch_rewalk_arrays(const LevelCtx &lv, int chunk, const uint64_t *sa, const uint32_t *la,
                                 const uint64_t *sb, const uint32_t *lb, size_t count, int32_t *cls,
                                 uint64_t *ab, cudaStream_t s);
// For the allocation-free walk entry point (qcs_noalloc.cu): the level
// context and trail cut-off that qcs_level_begin would use, and the problem's
// table size; QCS_ERR_ARG when k or dp_bits are out of range.
int noalloc_level(const ::qcs_problem *P, int k, uint32_t version, int dp_bits, LevelCtx *lv,
                  uint32_t *max_len, int *table_log2);
int record_cuda_error(cudaError_t e); // stores the text for qcs_last_cuda_error, returns QCS_ERR_CUDA

// number of resident CTAs of the walk kernel per SM for n qubits (occupancy)
int walk_blocks_per_sm(int n);
int num_sms();

// ---- exact host arithmetic (qcs_exact.cpp) ----
// A matrix over Z[1/sqrt2]: (a + b sqrt2) / sqrt2^E, D x D row-major.
struct PMat {
    int D = 0, E = 0;
    std::vector<int64_t> a, b;
};

// status codes mirror qcs.h; overflow is reported, never wraps
int exact_channel_from_unitary(int n, const int64_t *u, int e, PMat *out);
int exact_unitary_from_circuit(int n, const int32_t *gates, int n_gates, std::vector<int64_t> *u, int *e);
int exact_check_channel(int n, const PMat &C);
void exact_reduce(PMat *M);
bool exact_is_clifford(const PMat &M);
// left-multiply by R^(p) (transpose = false) or R^(p)^T (true); exponent + 1
int exact_rhat_left(int n, uint32_t p, bool transpose, const PMat &M, PMat *out);
// D^ = R^(P_1)^T .. R^(P_t)^T C^; QCS_OK if a signed permutation, else QCS_ERR_MISMATCH
int exact_verify(int n, const PMat &C, const uint32_t *paulis, int t, PMat *Dout);
int pauli_phase(int n, uint32_t p, uint32_t q); // P(p)P(q) = i^lambda P(p^q)
// device tables of the first adjoint stage (LevelCtx::T1), built once per
// device and qubit count and kept for the life of the process
// (*uploaded, when given, grows by the bytes this call copied to the device)
// (t4: LevelCtx::T4, null at n = 1)
// (quad: LevelCtx::quad, null unless n is 2 or 3)
int stage_tables(int n, const uint32_t *t1[2], const uint32_t *t4[2], const uint32_t **quad,
                 int64_t *uploaded = nullptr);

// How a level is walked (Sec. 3 and Appendix): theta, the launch shape, the
// function-version period and the level's step budget.
struct LevelPlan {
    int dp_bits;
    uint32_t walks, steps;
    uint64_t launches_per_version, min_launches;
    uint64_t points;
};

// helpers of the host library shared by qcs_api.cpp and qcs_batch.cpp
uint64_t upow(uint64_t b, int e);
int field_bits(int L, int h);
void decode_state(uint64_t x, int n, int L, int h, uint32_t *q);
LevelCtx make_level(const ::qcs_problem *P, int k, uint32_t version, int dp_bits);
LevelPlan plan_level(const ::qcs_problem *P, int k, const qcs_params &p);
LevelPlan plan_level_n(int D, int k, const qcs_params &p); // D = 4^n
void found(::qcs_problem *P, int k, const uint32_t *paulis, PMat &&Dh); // keeps the first decomposition
void found(::qcs_problem *P, int k, const uint32_t *paulis);              // forms D^ itself
// Exact check of a claw candidate (Eq. tcount_synthesis): paulis gets
// (q_1..q_h, q'_1..q'_h [, c]) from the V rotations qv, the W rotations qw and
// the chunk, and the candidate is a claw iff D^ = R^(P_1)^T..R^(P_k)^T C^ is a
// signed permutation; *Dh gets D^ then.
bool verify_claw(const ::qcs_problem *P, int k, int chunk, const uint32_t *qv, const uint32_t *qw,
                 uint32_t *paulis, PMat *Dh);

} // namespace qcs

// A search problem (include/qcs.h): the exact target and its device copies.
struct qcs_problem {
    int n = 0, D = 0, k_max = 0, device = 0;
    qcs_params p{};
    qcs::PMat C; // reduced, exponent = sde
    // device data
    uint2 *dC32 = nullptr, *dU = nullptr;
    uint32_t *dCq = nullptr; // n >= 3, when every entry of C^ fits in int8
    uint16_t *dCm = nullptr; // n >= 2, when C^ suits the tensor-core kernels: LevelCtx::Cm
    const uint32_t *dT1[2] = {nullptr, nullptr}; // shared stage tables
    const uint32_t *dT4[2] = {nullptr, nullptr}; // and their form by code (LevelCtx::T4)
    const uint32_t *dQuad = nullptr;             // LevelCtx::quad
    uint32_t *dCoef = nullptr;
    qcs::Slot *dTable = nullptr;
    qcs::Pair *dQueue = nullptr;
    uint32_t *dQhead = nullptr; // [0] queued merges, [1] claw candidates, [2] carried re-walks, [3] re-walk cursor
    qcs::Pending *dPend[2] = {nullptr, nullptr}; // carried re-walks (params.rewalk_budget > 0)
    qcs::Cand *dCands = nullptr;
    qcs::WalkState *dWalks = nullptr;
    unsigned long long *dCounters = nullptr;
    // pinned host mirrors
    unsigned long long *hCounters = nullptr;
    qcs::Cand *hCands = nullptr;
    uint32_t *hQhead = nullptr; // mirrors dQhead
    // search state
    std::thread driver;
    std::mutex mu;
    std::condition_variable cv;
    std::atomic<bool> cancel{false};
    bool running = false;
    qcs_result res{};
    std::chrono::steady_clock::time_point t0;
    qcs::PMat Dhat;
    bool have_D = false;
    // the level being stepped (qcs_level_* and the driver)
    struct {
        bool active = false;
        int k = 0, h = 0, dp_bits = 0;
        qcs::WalkLaunch w{};
        int pp = 0;          // dPend[pp] holds the re-walks carried into the next launch
        uint32_t pend_n = 0; // how many
        uint32_t rw_last = 0; // merges of the last collected re-walk
    } lvl;
};
