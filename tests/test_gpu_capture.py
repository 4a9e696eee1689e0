"""A caller's own graph capture of a forward and a backward in one graph.  The
backward's classes are launched with programmatic dependence on one another, which
the capture records as programmatic edges; the replays give the bits of the
uncaptured calls, also for inputs that change between replays."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04006_gb300 import api, pq  # noqa: E402
from paper_2403_04006_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def test_forward_and_backward_in_one_graph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pq.load_library()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(31)
    items = []
    for q in range(96):  # every register class of the backward, and one wider
        l = 1 + q % 17
        k = min(l, 4)
        r = [l // k + (i < l % k) for i in range(k)]
        B = rng.standard_normal((k, l)) + 1j * rng.standard_normal((k, l))
        items.append((B, r, [1] * l))
    pb = W.pack_batch(items)
    db = api.DeviceBatch(pb, dev)
    go = torch.from_numpy(rng.standard_normal(pb.batch) + 1j * rng.standard_normal(pb.batch)).to(dev)
    plan = api.Plan.for_batch(pb)
    values = [db.mats.clone() * f for f in (1.0, 0.5 - 0.75j, 1.25j)]

    def step():
        return api.permanent_batched(db, plan), api.permanent_backward(db, go, plan)

    want = []
    for v in values:
        db.mats.copy_(v)
        want.append([x.clone() for x in step()])
    assert plan.stats()["launches_backward"] > 8
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = step()
    for v, w in list(zip(values, want)) * 2:
        db.mats.copy_(v)
        graph.replay()
        torch.cuda.synchronize()
        for x, y in zip(got, w):
            assert np.array_equal(x.cpu().numpy().view(np.float64), y.cpu().numpy().view(np.float64))
