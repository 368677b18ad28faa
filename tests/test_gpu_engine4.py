"""The n = 4 engine (qcs_engine4.cu) against the dp4a kernels, bit for bit:
walk counts around one and two rounds of every SM, levels with none to three
stages beside the first and with and without the chunk's, targets whose C^ is
sparse or near the largest column sums that the engine takes, and one beyond
them, which the engine leaves to the dp4a kernels."""
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
    (9, 9, 100, 6, 2), (7, 15, 100, 4, 2), (13, 7, 500, 8, 2), (12, 13, 500, 8, 2), (15, 7, 500, 4, 2),
])
def test_engine_walk_equals_the_dp4a_walk(dev, t, k, walks, steps, dpb):
    a, b = walk(dev, 0, t, k, walks, steps, dpb), walk(dev, 3, t, k, walks, steps, dpb)
    assert a[1][0] == walks * steps
    assert np.array_equal(a[0], b[0])
    assert a[1] == b[1]
