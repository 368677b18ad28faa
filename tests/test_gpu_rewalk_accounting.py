"""Every merge that a launch queues is accounted for: classified, or carried to
the next launch by its evaluation budget."""
import numpy as np
import pytest

import paper_1606_07413_gb300 as Q
from paper_1606_07413_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def dev():
    from paper_1606_07413_gb300 import build

    build.build()
    assert torch.cuda.is_available()


def classified(r):
    return r["robin_hood"] + r["trivial"] + r["same_side"] + r["claws"] + r["false_hash"] + r["no_merge"]


# A budget of one evaluation advances a longer trail by one step and carries
# aligned merges as they are, so whole rounds of slots are carried when taken.
@pytest.mark.parametrize("n,t,k,dpb,walks", [(4, 9, 6, 1, 1 << 14), (4, 9, 5, 3, 1 << 15), (4, 9, 4, 1, 300), (3, 8, 5, 1, 1 << 14)])
def test_a_budget_of_one_evaluation_loses_no_merge(n, t, k, dpb, walks):
    gates, _ = W.seeded_target(n, t, 59)
    p = Q.default_params(n, walks=walks, table_log2=18, rewalk_budget=1)
    with Q.Problem.from_circuit(n, gates, 15, p) as prob:
        assert prob.sde > k
        prob.level_begin(k, 1, dpb)
        for launch in range(5):
            prob.level_walk(16)
            prob.level_rewalk()
            r = prob.level_collect()
            assert r["queue_overflow"] == 0 and r["false_hash"] == 0
            assert classified(r) + r["rewalk_carried"] == r["merges"], launch
        assert r["merges"] > 100 and r["rewalk_carried"] > 0


def smix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def trails(refs, seed, version, L, n_chunks):
    """Start, chunk and length of the trails that the references name."""
    u = np.uint64
    walk, seq, length = refs & u((1 << 24) - 1), (refs >> u(24)) & u((1 << 23) - 1), refs >> u(47)
    start = smix(u(seed) ^ smix((walk << u(32)) | seq) ^ (u(version) << u(40))) & u((1 << L) - 1)
    chunk = u(1) + smix(start ^ u(0x5851F42D4C957F2D)) % u(n_chunks) if n_chunks else np.zeros(len(refs), u)
    return start, chunk, length


# n = 3 lists as long as the queue, one merge shorter than the quads take, as
# long and longer (40960, and 20480 where C^ is not int8); lists far shorter
# than the queue; a short list after a long one and the other way round; with
# an evaluation budget, whose carried merges count
@pytest.mark.parametrize("t,queue,walks,dpb,budget,steps", [
    (8, 40959, 60000, 1, 0, (12,)), (8, 40960, 60000, 1, 0, (12,)), (8, 60001, 65536, 1, 0, (12,)),
    (8, 50000, 3000, 3, 0, (12,)), (8, 1 << 19, 65536, 1, 0, (12, 1, 1)), (8, 1 << 19, 20000, 2, 0, (1, 1, 30)),
    (8, 1 << 17, 50000, 2, 8, (12, 1, 1, 1)), (19, 20479, 40000, 1, 0, (12,)), (19, 20480, 40000, 1, 0, (12,)),
    (19, 1 << 16, 5000, 2, 0, (12,))])
def test_list_lengths_around_the_quads(t, queue, walks, dpb, budget, steps):
    """Every merge of a list, classified by the level's re-walk and, from its
    two trails' recomputed starts, by qcs_rewalk (one lane group per pair)."""
    k, version, L = 5, 2, 48
    gates, _ = W.seeded_target(3, t, 9)
    p = Q.default_params(3, walks=walks, table_log2=17, rewalk_budget=budget, queue_capacity=queue)
    with Q.Problem.from_circuit(3, gates, 15, p) as prob:
        assert prob.sde > k
        assert (t == 19) == (max(abs(v).max() for v in prob.channel()[:2]) > 127)
        prob.level_begin(k, version, dpb)
        lists, r = [], None
        for count in steps:
            prob.level_walk(count)
            lists.append(prob.level_merges())
            prob.level_rewalk()
            r = prob.level_collect()
        m = np.concatenate(lists).astype(np.uint64)
        lengths = [len(x) for x in lists]
        if len(steps) == 1:
            assert lengths[0] == queue if walks >= 40000 else 500 < lengths[0] < queue
        elif not budget:  # far above the line in one launch, far below it in another
            assert max(lengths) > 2 * 40960 and min(lengths) < 40960 and r["queue_overflow"] == 0
        assert classified(r) + r["rewalk_carried"] == len(m) and r["false_hash"] == 0
        if budget:
            assert r["queue_overflow"] == 0 and r["rewalk_carried"] > 0
            return
        a, b = (trails(m[:, i], p.seed, version, L, 63) for i in (0, 1))
        want = np.zeros(6, np.int64)
        want[5] = int((a[1] != b[1]).sum())
        for chunk in range(1, 64):
            at = (a[1] == chunk) & (b[1] == chunk)
            if not at.any():
                continue
            sa, sb = (torch.from_numpy(v[0][at].view(np.int64)).cuda() for v in (a, b))
            la, lb = (torch.from_numpy(v[2][at].astype(np.int32)).cuda() for v in (a, b))
            cls = torch.empty(len(sa), dtype=torch.int32, device="cuda")
            prob.rewalk(k, chunk, version, sa, la, sb, lb, cls, torch.empty(2 * len(sa), dtype=torch.int64, device="cuda"))
            want += np.bincount(cls.cpu().numpy(), minlength=6)
        got = [r["robin_hood"], r["trivial"], r["same_side"], r["claws"] + r["false_hash"], r["no_merge"]]
        assert got == [want[0], want[1], want[2], want[3] + want[4], want[5]]


def job(n, t, seed, layout, dpb):
    """A problem whose ladder starts at its T-count's level t, where a few
    rounds find no claw, with states so short that trails meet all the time."""
    for s in range(seed, seed + 40):
        prob = Q.Problem.from_circuit(n, W.seeded_target(n, t, s)[0], 7, Q.default_params(
            n, c_layout=layout, theta_policy=0, dp_bits=dpb, exhaustive_log2=0, version_factor=0,
            state_bits=25 if n == 4 else 22))
        if prob.sde == t:
            return prob
        prob.close()
    raise AssertionError("no target with this denominator exponent")


# (n, T-count, layout of C^, -log2 theta) of every job: a CTA for one job alone
# and shares that meet several, on the engine and on quads, trails of different
# lengths, jobs of the general kernels beside them, two qubit counts together
@pytest.mark.parametrize("walks,steps,jobs", [
    (2048, 64, [(4, 7, 0, 1)]),
    (1024, 40, [(4, 7, 0, 1), (4, 6, 0, 2), (4, 7, 0, 4)] * 3),
    (256, 40, [(4, 7, 0, 1), (4, 6, 0, 3)] * 25),
    (1024, 24, [(4, 7, 0, 1), (4, 7, 1, 1), (4, 6, 0, 2), (4, 6, 1, 2)] * 2),
    (2048, 20, [(3, 7, 0, 1), (3, 6, 0, 2), (3, 7, 0, 4)] * 2),
    (512, 20, [(3, 7, 0, 1), (3, 6, 0, 3), (3, 7, 0, 2)] * 18),
    (512, 32, [(3, 7, 0, 1), (3, 7, 1, 1), (4, 7, 0, 2)] * 8),
    (80, 60, [(3, 7, 0, 1), (4, 7, 0, 1)] * 60),
])
def test_batched_rewalks_classify_every_merge_once(walks, steps, jobs):
    probs = [job(n, t, 300 + 50 * i, layout, dpb) for i, (n, t, layout, dpb) in enumerate(jobs)]
    bp = Q.default_batch_params(max_jobs=len(jobs), walks_per_job=walks, steps_per_round=steps, table_log2=16,
                                queue_capacity=1 << 16, rewalk_budget=0)
    searching = merges = 0
    with Q.Batch(bp) as batch:
        ids = [batch.add(p) for p in probs]
        for _ in range(4):
            batch.round()
            for j, (n, t, layout, dpb) in zip(ids, jobs):
                r = batch.poll(j)
                assert r["queue_overflow"] == 0 and r["error"] == 0
                if r["status"] == Q.SEARCHING:  # else the host's check of candidates ended at a claw
                    assert classified(r) == r["merges"], (n, t, layout, dpb)
                    assert r["steps"] == r["launches"] * walks * steps
                    searching += 1
                    merges += r["merges"]
    for p in probs:
        p.close()
    assert searching > 2 * len(jobs) and merges > 100


def test_the_smallest_jobs_stay_within_their_buffers():
    """Jobs of 16 walks whose first level has fewer points than a warp's walks
    take steps for: no more walks than the job has, beside jobs of the next
    kernel class."""
    jobs = [(2, 2, 1)] * 12 + [(3, 5, 1)] * 4 + [(2, 2, 0)] * 12
    probs = [Q.Problem.from_circuit(n, W.seeded_target(n, t, 20 + i)[0], 9, Q.default_params(
        n, c_layout=layout, exhaustive_log2=0)) for i, (n, t, layout) in enumerate(jobs)]
    with Q.Batch(Q.default_batch_params(max_jobs=len(jobs), walks_per_job=16, table_log2=10)) as batch:
        ids = [batch.add(p) for p in probs]
        for _ in range(6):
            before = [batch.poll(j) for j in ids]
            batch.round()
            for a, b in zip(before, (batch.poll(j) for j in ids)):
                assert b["error"] == 0 and b["steps"] - a["steps"] <= 16 * 64
                assert b["status"] in (Q.SEARCHING, Q.FOUND)
                if a["status"] == Q.SEARCHING:
                    assert b["steps"] > a["steps"] or b["status"] == Q.FOUND
    for p in probs:
        p.close()
