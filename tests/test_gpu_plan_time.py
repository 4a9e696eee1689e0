"""Planning time: proportional to the number of shape groups in either method."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04006_gb300 import api, pq  # noqa: E402
from paper_2403_04006_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def many_shapes(count):
    """Permanents of n = 12..24 with rows and columns repeated 1 to 6 times; most
    have multiplicities of their own."""
    rng = np.random.default_rng(21)
    items = []
    for n in rng.integers(12, 25, count):
        mults = []
        for _ in range(2):
            m, left = [], int(n)
            while left:
                m.append(min(left, int(rng.integers(1, 7))))
                left -= m[-1]
            mults.append(m)
        r, c = mults
        items.append((np.ones((len(r), len(c)), dtype=complex), r, c))
    return W.pack_batch(items)


def test_plain_plan_of_many_shapes():
    """The plain method cuts each group for its own launch, at the same eleven caps
    that the batched method tries for the whole batch, so its plan takes about as
    long: 0.14 s against 0.12 for 12700 groups, and 0.42 where every group copied the
    cuts of all.  Three times as long is allowed for noise."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pq.load_library()
    pb = many_shapes(16384)
    best = {}
    for method in ("batched", "plain"):
        for _ in range(3):
            t = time.perf_counter()
            plan = api.Plan.for_batch(pb, method=method)
            t = time.perf_counter() - t
            plan.close()
            best[method] = min(best.get(method, t), t)
    print({k: round(v, 4) for k, v in best.items()})
    assert best["plain"] <= 3 * best["batched"], best
