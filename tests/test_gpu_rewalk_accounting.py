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
