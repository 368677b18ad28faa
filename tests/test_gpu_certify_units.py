"""The exhaustive pass where its kernels can go wrong: n = 4 levels on the
tensor-core engine (W points) and in units of 32 points (V points), and
passes cut into small shares, whose ranges begin and end inside a unit."""
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


def anticommute(n, p, q):
    m = (1 << n) - 1
    return (bin((p >> n) & q & m).count("1") + bin(p & m & (q >> n)).count("1")) & 1


def target(n, t, seed):
    """A target of t rotations, neighbours anticommuting, whose T-count is t by
    its denominator exponent; None if this seed's is smaller."""
    rng = np.random.Generator(np.random.PCG64(seed))
    while True:
        p = [int(v) for v in rng.integers(1, 4 ** n, size=t)]
        if all(anticommute(n, p[i], p[i + 1]) for i in range(t - 1)):
            break
    rot = np.asarray([(W.OP_RP, v, 0) for v in p], dtype=np.int32).reshape(-1, 3)
    return np.concatenate([W.clifford_word(rng, n), rot], axis=0)


def problem(n, t, seed, k_max, **over):
    for s in range(seed, seed + 16):
        prob = Q.Problem.from_circuit(n, target(n, t, s), k_max, Q.default_params(n, **over))
        if prob.sde == t:
            return prob
        prob.close()
    raise AssertionError("no target with this denominator exponent")



# below its T-count a level is empty (the denominator exponent bounds it);
# at the T-count the pass finds the one decomposition; two levels above, a
# repeated rotation gives one too
@pytest.mark.parametrize("n,t", [(4, 2), (4, 3), (4, 4), (4, 5), (3, 4), (3, 5), (3, 6)])
def test_levels_around_the_tcount(n, t):
    with problem(n, t, 500 + 10 * n + t, t + 1) as prob:
        for k in range(max(2, t - 2), t):
            assert not prob.certify_level(k)
    with problem(n, t, 500 + 10 * n + t, t + 1) as prob:
        assert prob.certify_level(t)
        r = prob.poll()
        assert r["t_count"] == t
        perm, sign = prob.clifford()  # the library's exact check left a signed permutation
        assert sorted(perm) == list(range(4 ** n)) and set(sign) <= {-1, 1}
    with problem(n, t, 500 + 10 * n + t, t + 1) as prob:
        assert not prob.certify_level(t + 1)  # the parity of the exponents differs


def test_clifford_targets_take_the_chunked_side():
    """sde 0: an odd level's W points carry the chunk rotation."""
    rng = np.random.Generator(np.random.PCG64(9))
    gates = W.clifford_word(rng, 4)
    with Q.Problem.from_circuit(4, gates, 4, Q.default_params(4)) as prob:
        assert prob.sde == 0
        assert not prob.certify_level(3)
        assert prob.certify_level(2)  # two equal rotations


@pytest.mark.parametrize("share", [8, 11, 13])
def test_small_shares_find_the_same(share):
    jobs = [(3, 4, 700), (3, 5, 710), (4, 3, 720), (4, 2, 730), (2, 5, 740)]
    if share >= 13:
        jobs.append((4, 4, 750))
    probs = []
    for n, t, seed in jobs:
        probs.append(Q.Problem.from_circuit(2, W.seeded_target(2, t, seed)[0], t, Q.default_params(
            2, exhaustive_first=1)) if n == 2 else problem(n, t, seed, t, exhaustive_first=1, exhaustive_log2=32))
    with Q.Batch(Q.default_batch_params(max_jobs=8, table_log2=10, walks_per_job=16, cert_points_log2=share)) as batch:
        ids = [batch.add(p) for p in probs]
        for _ in range(20000):
            if batch.round() == 0:
                break
        for (n, t, _), j in zip(jobs, ids):
            r = batch.poll(j)
            assert r["status"] == Q.FOUND and (r["t_count"] == t if n > 2 else r["t_count"] <= t), (n, t, r)
    for p in probs:
        p.close()
