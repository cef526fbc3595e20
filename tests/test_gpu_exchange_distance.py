"""The pairs of one exchange attempt of a context by ladder distance.

The context's exchange kernels number the pairs (q, q + d) of a ladder and take
one thread a pair: every pair must be met once, whatever d against R (blocks of
2d cut short by the ladder's end, d = R - 1 with one pair, d = R with none) and
the parity, with the replicas in an order that is not the ladder's.  One CTA
ranks up to 256 replicas, a cluster longer ladders.  Partners, decisions and T
equal the oracle's exactly."""
import numpy as np
import pytest

import oracle as O
from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [5, 130, 256, 300])
@pytest.mark.parametrize("dist", ["3", "half", "last", "beyond"])
def test_pairs_of_any_distance(R, dist):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    d = {"3": 3, "half": R // 2, "last": R - 1, "beyond": R}[dist]
    N, seed = 256, 50 + R
    temps = np.random.default_rng(seed).permutation(inputs.geometric_ladder(0.9, 1.1, R))
    ctx = re.Context(N, inputs.box_length(N), 2.5, temps, seed, exch_distance=d)
    ctx.advance(3)
    for attempt in range(4):
        T, U = ctx.temps(), ctx.energies()[0]
        Tn, _, po, ao, _, _, _ = O.exchange_h(T, np.ones(R), U, seed, attempt, 0, d)
        pg, ag = ctx.exchange(outputs=True)
        assert np.array_equal(pg, po)
        assert np.array_equal(ag, ao)
        assert np.array_equal(ctx.temps(), Tn)
    ctx.close()
