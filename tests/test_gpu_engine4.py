"""The n = 4 engine (qcs_engine4.cu) against the dp4a kernels, bit for bit:
walk counts around one and two rounds of every SM, levels with none to three
stages beside the first and with and without the chunk's, targets whose C^ is
sparse, beyond int8, near the largest column sums that the engine takes and
beyond them, where it leaves them to the 32-bit-word kernels."""
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


def walk(dev, shape, t, k, walks, steps, dpb):
    gates, _ = W.seeded_target(4, t, 4000 + t)
    p = Q.default_params(4, walks=walks, table_log2=16, launch_shape=shape)
    with Q.Problem.from_circuit(4, gates, 15, p) as prob:
        ws = torch.zeros(4 * walks, dtype=torch.int64, device=dev)
        merges = torch.zeros(3 * 4096, dtype=torch.int64, device=dev)
        counts = torch.zeros(8, dtype=torch.int64, device=dev)
        prob.level_walk_static(k, 1, dpb, 1, ws, steps, merges, counts)
        torch.cuda.synchronize()
        c = counts.cpu().numpy()
        assert int(c[7]) >> 32 == 0, "a bounded wait ran out"
        return ws.cpu().numpy(), c[:4].tolist()


# 72 slots (three sets of 24, 16 W points each at most) and one CTA per SM:
# 152 x 72 = 10944 walks fill every slot, 10945 are two walks to most slots.
# About 3 % of a full set's rounds have a point that waits for the next one.
@pytest.mark.parametrize("t,k,walks,steps,dpb", [
    (7, 7, 10944, 9, 3), (7, 7, 10945, 2, 12), (7, 7, 21889, 3, 1), (7, 7, 151, 2, 3), (7, 7, 3800, 2, 3),
    (0, 2, 100, 6, 2), (3, 3, 100, 6, 2), (5, 4, 100, 6, 2), (5, 5, 100, 6, 2), (7, 6, 100, 6, 2), (9, 8, 100, 6, 2),
    (9, 9, 100, 6, 2), (7, 15, 100, 4, 2), (13, 7, 500, 8, 2), (12, 13, 500, 8, 2), (15, 7, 10945, 4, 2),
    (17, 6, 500, 4, 2), (19, 7, 3800, 4, 2), (22, 7, 500, 4, 2),
])
def test_engine_walk_equals_the_dp4a_walk(dev, t, k, walks, steps, dpb):
    a, b = walk(dev, 0, t, k, walks, steps, dpb), walk(dev, 3, t, k, walks, steps, dpb)
    assert a[1][0] == walks * steps
    assert np.array_equal(a[0], b[0])
    assert a[1] == b[1]


# lists of one state, around a state to a slot and two, and in place: the
# images are stored a round after they are known
@pytest.mark.parametrize("t", [0, 7, 13, 15, 18, 19])
def test_engine_step_equals_the_dp4a_step(dev, t):
    gates, _ = W.seeded_target(4, t, 4100 + t)
    with Q.Problem.from_circuit(4, gates, 15, Q.default_params(4)) as a, \
            Q.Problem.from_circuit(4, gates, 15, Q.default_params(4, c_layout=1)) as b:
        for k in range(16):
            for count in ((1, 153, 10944, 10945, 32833) if k in (4, 7) else (305,)):
                x = torch.from_numpy(W.seeded_states(count, 64, 9 * k + count).view(np.int64)).to(dev)
                chunk = (255 if count == 153 else 1 + (7 * k) % 255) if k & 1 else 0
                got = []
                for prob in (a, b):
                    y, dp = x.clone(), torch.empty(count, dtype=torch.uint8, device=dev)
                    prob.walk_step(k, chunk, 4, y, y, dp)
                    got.append((y.cpu().numpy(), dp.cpu().numpy()))
                assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), (k, count)


M64 = (1 << 64) - 1


def smix(z):
    z &= M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def trail(ref, seed, version, n_chunks):
    walk, seq, length = ref & ((1 << 24) - 1), (ref >> 24) & ((1 << 23) - 1), ref >> 47
    start = smix(seed ^ smix((walk << 32) | seq) ^ (version << 40))
    return start, (1 + smix(start ^ 0x5851F42D4C957F2D) % n_chunks if n_chunks else 0), length


def classes(r):
    return np.array([r["robin_hood"], r["trivial"], r["same_side"], r["claws"] + r["false_hash"], r["no_merge"]])


# Slots whose merges end at different points of a round (classified, carried
# for their budget, two chunks' functions): every merge is accounted for.
@pytest.mark.parametrize("k,dpb,walks,steps,budget", [(5, 2, 1 << 16, 32, 5), (7, 4, 1 << 17, 32, 9), (6, 3, 1 << 17, 32, 7),
                                                      (4, 1, 1 << 16, 16, 2), (6, 1, 1 << 17, 16, 0)])
def test_engine_rewalk_loses_no_merge(dev, k, dpb, walks, steps, budget):
    gates, _ = W.seeded_target(4, 9, 59)
    p = Q.default_params(4, walks=walks, table_log2=20, rewalk_budget=budget)
    with Q.Problem.from_circuit(4, gates, 15, p) as prob:
        assert prob.sde > k
        prob.level_begin(k, 1, dpb)
        for _ in range(12):
            prob.level_walk(steps)
            prob.level_rewalk()
            r = prob.level_collect()
        assert r["merges"] > 10000 and r["queue_overflow"] == 0 and r["false_hash"] == 0
        assert classes(r).sum() + r["rewalk_carried"] == r["merges"]


# lists shorter than the CTAs, around one merge per slot and far longer, with
# and without chunks, and an evaluation budget; levels below the target's
# T-count, so no claw ends the host's check of candidates
@pytest.mark.parametrize("k,dpb,walks,steps,budget", [
    (4, 4, 400, 30, 0), (4, 4, 3000, 24, 0), (4, 1, 20000, 24, 0), (4, 7, 20000, 60, 0), (5, 3, 12000, 60, 0),
    (2, 2, 5000, 8, 0), (4, 3, 6000, 24, 5),
])
def test_engine_rewalk_classes_equal_the_array_rewalk(dev, k, dpb, walks, steps, budget):
    """Every merge of a launch, classified by the level's re-walk and, from its
    two trails' recomputed starts, by qcs_rewalk (one lane group per pair)."""
    gates, _ = W.seeded_target(4, 7, 4007)
    version = 2
    p = Q.default_params(4, walks=walks, table_log2=16, rewalk_budget=budget)
    with Q.Problem.from_circuit(4, gates, 7, p) as prob:
        prob.level_begin(k, version, dpb)
        prob.level_walk(steps)
        m = prob.level_merges()
        prob.level_rewalk()
        r = prob.level_collect()
        launches = 1
        while r["rewalk_carried"]:  # resumed first in the next launch
            prob.level_walk(1)
            m = np.concatenate([m, prob.level_merges()])
            prob.level_rewalk()
            r = prob.level_collect()
            launches += 1
            if launches == 6:
                break
        got, carried = classes(r), r["rewalk_carried"]
        assert len(m) > (1000 if walks > 400 else 10) and r["queue_overflow"] == 0
        assert got.sum() + carried == len(m)
        if carried:
            return
        want = np.zeros(6, np.int64)
        trails = [[trail(int(ref), p.seed, version, 255 if k & 1 else 0) for ref in row[:2]] for row in m]
        by_chunk = {}
        for ta, tb in trails:
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
        assert np.array_equal(got, [want[0], want[1], want[2], want[3] + want[4], want[5]])


# walks per job around a task (72 walks) and far above; one job whose C^ the
# engine does not take runs beside the others
@pytest.mark.parametrize("walks,targets", [(16, (7, 7, 7)), (64, (7, 6)), (80, (7,) * 5), (2048, (7, 15, 6)),
                                           (144, (7,) * 40)])
def test_batched_jobs_on_the_engine_walk_as_on_dp4a(walks, targets):
    """Walk counters of every job and round, engine (shape 0) against dp4a (shape 1)."""
    hist = {}
    for shape in (0, 1):
        bp = Q.default_batch_params(max_jobs=len(targets), walks_per_job=walks, steps_per_round=24, table_log2=14,
                                    queue_capacity=1 << 12, rewalk_budget=7, launch_shape={4: shape})
        probs = [Q.Problem.from_circuit(4, W.seeded_target(4, t, 4000 + t + 100 * i)[0], min(t, 9), Q.default_params(
            4, state_bits=64, seed=77 + i)) for i, t in enumerate(targets)]
        rows = []
        with Q.Batch(bp) as batch:
            ids = [batch.add(p) for p in probs]
            for _ in range(4):
                batch.round()
                rs = [batch.poll(j) for j in ids]
                rows.append([(r["k"], r["steps"], r["w_steps"], r["dps"], r["abandoned"]) for r in rs])
                for r in rs:
                    assert r["status"] in (Q.SEARCHING, Q.FOUND, Q.BUDGET_EXHAUSTED)
        hist[shape] = rows
        for p in probs:
            p.close()
    assert hist[0] == hist[1]
    assert sum(r[1] for r in hist[0][-1]) > 0
