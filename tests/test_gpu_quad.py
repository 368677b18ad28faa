"""The quad kernels (qcs_quad.cu: n = 2, 3, eight walks to a warp) against the
32-bit-word kernels (c_layout 1), bit for bit: every level from 0 to 15 (no, one
and more rotations per side, one word of stage codes and two), counts around a
warp's eight walks and the least that n = 3 takes there, dense and sparse targets, and ones whose C^ is
beyond int8 and beyond what the quads take."""
import numpy as np
import pytest

import paper_1606_07413_gb300 as Q
from paper_1606_07413_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    from paper_1606_07413_gb300 import build

    build.build()
    assert torch.cuda.is_available()
    return torch.device("cuda:0")


def problem(n, t, layout, k_max=15, **over):
    gates, _ = W.seeded_target(n, t, 3000 + 10 * n + t)
    return Q.Problem.from_circuit(n, gates, k_max, Q.default_params(n, c_layout=layout, **over))


@pytest.mark.parametrize("n,t", [(2, 0), (2, 3), (2, 7), (2, 13), (2, 19), (3, 0), (3, 5), (3, 12), (3, 19),
                                 (3, 24)])
def test_walk_step_at_every_level(dev, n, t):
    bits = {2: 40, 3: 63}[n]
    with problem(n, t, 0, state_bits=bits) as a, problem(n, t, 1, state_bits=bits) as b:
        for k in range(16):
            for count in ((1, 9, 161) if n == 2 else (8192, 8201, 8353)):
                x = torch.from_numpy(W.seeded_states(count, bits, 5 * k + count).view(np.int64)).to(dev)
                chunk = (4 ** n - 1 if count % 64 == 9 else 1 + (7 * k) % (4 ** n - 1)) if k & 1 else 0
                got = []
                for prob in (a, b):
                    y = torch.empty_like(x)
                    dp = torch.empty(count, dtype=torch.uint8, device=dev)
                    prob.walk_step(k, chunk, 4, x, y, dp)
                    got.append((y.cpu().numpy(), dp.cpu().numpy()))
                assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), (k, count)


@pytest.mark.parametrize("n,t,k,walks,steps,dpb", [
    (2, 3, 3, 4096, 40, 6), (2, 3, 2, 1, 9, 2), (2, 5, 5, 8, 9, 2), (2, 7, 11, 9, 9, 2), (2, 5, 4, 40000, 5, 1),
    (3, 5, 5, 7001, 20, 3), (3, 5, 2, 6145, 9, 2), (3, 7, 3, 6144, 9, 2), (3, 9, 13, 6151, 9, 2), (3, 7, 6, 40000, 3, 1),
    (3, 19, 5, 2049, 5, 2), (3, 24, 5, 6300, 5, 2), (3, 5, 5, 6143, 5, 2), (2, 17, 5, 900, 9, 2),
])
def test_level_walk(dev, n, t, k, walks, steps, dpb):
    got = []
    for layout in (0, 1):
        with problem(n, t, layout, walks=walks, table_log2=16) as prob:
            ws = torch.zeros(4 * walks, dtype=torch.int64, device=dev)
            merges = torch.zeros(3 << 16, dtype=torch.int64, device=dev)
            counts = torch.zeros(8, dtype=torch.int64, device=dev)
            for begin in (1, 0):
                prob.level_walk_static(k, 3, dpb, begin, ws, steps, merges, counts)
            torch.cuda.synchronize()
            got.append((ws.cpu().numpy(), counts.cpu().numpy()[:4].tolist()))
    assert got[0][1][0] == walks * steps
    assert got[0][1] == got[1][1]
    assert np.array_equal(got[0][0], got[1][0])


M64 = (1 << 64) - 1


def smix(z):
    z &= M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def trail(ref, seed, version, L, n_chunks):
    walk, seq, length = ref & ((1 << 24) - 1), (ref >> 24) & ((1 << 23) - 1), ref >> 47
    start = smix(seed ^ smix((walk << 32) | seq) ^ (version << 40)) & ((1 << L) - 1)
    return start, (1 + smix(start ^ 0x5851F42D4C957F2D) % n_chunks if n_chunks else 0), length


# lists of a few merges and of many, with and without chunks, and an evaluation
# budget; levels below the target's T-count, so no claw ends the host's check
# of candidates
@pytest.mark.parametrize("n,k,dpb,walks,steps,budget", [
    (3, 4, 3, 40, 40, 0), (3, 4, 1, 20000, 12, 0), (3, 3, 4, 5000, 40, 0), (3, 2, 5, 3000, 90, 0), (3, 4, 3, 9000, 24, 4),
    (2, 4, 2, 33, 30, 0), (2, 3, 3, 4000, 24, 0), (2, 2, 1, 9000, 9, 0),
])
def test_rewalk_classes_equal_the_array_rewalk(dev, n, k, dpb, walks, steps, budget):
    """Every merge of a launch, classified by the level's re-walk and, from its
    two trails' recomputed starts, by qcs_rewalk (one lane group per pair)."""
    L, version, xi = 52, 2, 4 ** n - 1
    with problem(n, 5, 0, walks=walks, table_log2=12, rewalk_budget=budget, state_bits=L) as prob:
        assert prob.sde > k
        prob.level_begin(k, version, dpb)
        prob.level_walk(steps)
        m = prob.level_merges()
        prob.level_rewalk()
        r = prob.level_collect()
        for _ in range(5):
            if not r["rewalk_carried"]:
                break
            prob.level_walk(1)  # the carried re-walks are resumed first
            m = np.concatenate([m, prob.level_merges()])
            prob.level_rewalk()
            r = prob.level_collect()
        got = [r["robin_hood"], r["trivial"], r["same_side"], r["claws"] + r["false_hash"], r["no_merge"]]
        assert len(m) > (500 if walks > 100 else 3) and r["queue_overflow"] == 0
        assert sum(got) + r["rewalk_carried"] == len(m)
        if r["rewalk_carried"]:
            return
        want = np.zeros(6, np.int64)
        by_chunk = {}
        for row in m:
            ta, tb = (trail(int(ref), prob_seed(n), version, L, xi if k & 1 else 0) for ref in row[:2])
            if ta[1] != tb[1]:
                want[5] += 1
            else:
                by_chunk.setdefault(ta[1], []).append((ta[0], ta[2], tb[0], tb[2]))
        for chunk, rows in by_chunk.items():
            x = np.array(rows, np.uint64)
            sa, sb = (torch.from_numpy(np.ascontiguousarray(x[:, i]).view(np.int64)).to(dev) for i in (0, 2))
            la, lb = (torch.from_numpy(x[:, i].astype(np.int32)).to(dev) for i in (1, 3))
            cls = torch.empty(len(rows), dtype=torch.int32, device=dev)
            ab = torch.empty(2 * len(rows), dtype=torch.int64, device=dev)
            prob.rewalk(k, chunk, version, sa, la, sb, lb, cls, ab)
            torch.cuda.synchronize()
            want += np.bincount(cls.cpu().numpy(), minlength=6)
        assert got == [want[0], want[1], want[2], want[3] + want[4], want[5]]


def prob_seed(n):
    return int(Q.default_params(n).seed)


# one small job (its n = 3 walks stay with the warp-per-walk kernels) up to more jobs
# than CTAs, walk counts of one task and of many, one job whose C^ the quads
# do not take, two qubit counts together
@pytest.mark.parametrize("walks,jobs", [(16, [(3, 7)]), (1024, [(3, 7), (3, 6), (3, 9), (3, 24)] * 2 + [(3, 8)]),
                                        (48, [(2, 9)] * 3), (512, [(3, 7), (2, 9)] * 13), (64, [(3, 8)] * 170)])
def test_batched_jobs_walk_the_same(walks, jobs):
    """Walk counters of every job and round against the 32-bit-word kernels."""
    hist = {}
    for layout in (0, 1):
        bp = Q.default_batch_params(max_jobs=len(jobs), walks_per_job=walks, steps_per_round=20, table_log2=10,
                                    queue_capacity=1 << 12, rewalk_budget=6)
        probs = [Q.Problem.from_circuit(n, W.seeded_target(n, t, 900 + i % 7)[0], 15, Q.default_params(
            n, c_layout=layout, seed=5 + i, dp_bits=7, theta_policy=0, exhaustive_log2=0, version_factor=0,
            budget_factor=1 << 20, state_bits=48)) for i, (n, t) in enumerate(jobs)]
        rows = []
        with Q.Batch(bp) as batch:
            ids = [batch.add(p) for p in probs]
            for _ in range(3):
                batch.round()
                rs = [batch.poll(j) for j in ids]
                # n = 2 levels are settled by chance: only the first round's walks are the same
                rows.append([(r["k"], r["steps"], r["w_steps"], r["dps"], r["abandoned"]) for r, (n, _) in zip(rs, jobs)
                             if n == 3 or len(rows) == 0])
        hist[layout] = rows
        for p in probs:
            p.close()
    assert hist[0] == hist[1]
    assert sum(r[1] for r in hist[0][0]) > 0
