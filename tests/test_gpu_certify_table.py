"""The exhaustive pass's key table: a pass counts the keys that reached it and
is refused unless they are as many as its stored points.  Levels whose stored
side has long chains of equal keys (two equal neighbouring rotations leave the
coset of the rest), in each kernel that stores."""
import pytest

import paper_1606_07413_gb300 as Q
from paper_1606_07413_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# stored sides: n = 4 even levels V in units of 32 points, odd levels W on the
# engine (the general kernel with 32-bit words); n = 3 V in units, W in lane
# groups; n = 2 lane groups
@pytest.mark.parametrize("n,k,layout", [(4, 2, 0), (4, 4, 0), (4, 6, 0), (4, 3, 0), (4, 5, 0), (4, 5, 1), (3, 6, 0),
                                        (3, 8, 0), (3, 5, 0), (3, 7, 1), (2, 6, 0), (2, 9, 0)])
def test_every_stored_point_reaches_the_table(n, k, layout):
    from paper_1606_07413_gb300 import build

    build.build()
    for seed in range(40, 60):
        gates, _ = W.seeded_target(n, k + 1 if n > 2 else k, seed)
        p = Q.default_params(n, exhaustive_log2=34, c_layout=layout)
        with Q.Problem.from_circuit(n, gates, 15, p) as prob:
            if n > 2 and prob.sde <= k:
                continue  # the denominator exponent proves the level empty
            has = prob.certify_level(k)  # an error if a key is missing
            r = prob.poll()
            h = k // 2
            stored, streamed = (4 ** n - 1) ** h, (4 ** n - 1) ** (h + (k & 1))
            assert has or r["cert_points"] == stored + streamed
            assert n == 2 or not has
            return
    raise AssertionError("no target with this denominator exponent")
