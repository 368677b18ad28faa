"""The device bytes of a batched job count every layout of C^ that its problem holds."""
import pytest

import paper_1606_07413_gb300 as Q
from paper_1606_07413_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# (a, b) of every entry: int8 quads (n >= 3) and the f16 operand (n >= 2) beside the 32-bit words
@pytest.mark.parametrize("n,extra", [(1, 0), (2, 4), (3, 2 + 4), (4, 2 + 4)])
def test_every_layout_counts(n, extra):
    from paper_1606_07413_gb300 import build

    build.build()
    gates, _ = W.seeded_target(n, 3, 5)
    with Q.Batch(Q.default_batch_params(max_jobs=1)) as batch:
        size = []
        for layout in (0, 1):
            with Q.Problem.from_circuit(n, gates, 3, Q.default_params(n, c_layout=layout)) as prob:
                size.append(batch.job_bytes(prob))
    assert size[0] - size[1] == extra * 16 ** n
