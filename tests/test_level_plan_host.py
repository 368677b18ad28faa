"""A level's plan stays within the buffers its parameters size (host arithmetic)."""
import pytest

import paper_1606_07413_gb300 as Q
from paper_1606_07413_gb300 import build as B


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


# batched jobs have 16 walks and a queue of 16 merges at least; small levels
# and queues are where the plan cuts the walks of a launch
@pytest.mark.parametrize("n", [1, 2, 3, 4])
def test_no_more_walks_than_asked_for(n):
    for walks in (1, 16, 24, 31, 32, 33, 48, 4096):
        for queue in (1, 16, 1 << 16):
            for steps in (1, 16, 64):
                for version_factor in (0, 1, 2):
                    p = Q.default_params(n, walks=walks, queue_capacity=queue, steps_per_launch=steps,
                                         version_factor=version_factor, table_log2=18)
                    for k in range(2, 16):
                        pl = Q.plan_level(n, k, p)
                        assert 1 <= pl["walks"] <= walks and 1 <= pl["steps"] <= steps, (walks, queue, steps, k)
