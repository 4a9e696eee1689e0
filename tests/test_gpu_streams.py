"""Calls on a stream that does not wait for the default one (torch side streams):
a plan's uploads have to be complete when its kernels read them, whatever the
memory held before.  Every call is made many times over, each time with other
sizes, so that its allocations take over memory that another plan has left; the
results have the bits of the same calls on the default stream."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04006_gb300 import api, pq  # noqa: E402
from paper_2403_04006_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
ROUNDS = 12


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pq.load_library()
    return torch.device("cuda:0")


def hafnians(seed, dev):
    rng = np.random.default_rng(seed)
    ks = rng.integers(1, 7, int(rng.integers(1, 60))).astype(np.int32)
    n = int((ks.astype(np.int64) ** 2).sum())
    mats = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    mo = np.concatenate([[0], np.cumsum(ks.astype(np.int64) ** 2)[:-1]])
    ro = np.concatenate([[0], np.cumsum(ks, dtype=np.int64)[:-1]])
    rep = rng.integers(0, 4, int(ks.sum())).astype(np.int32)
    gam = rng.standard_normal(rep.size) + 1j * rng.standard_normal(rep.size)
    return (torch.from_numpy(mats).to(dev), mo, ks, rep, ro), torch.from_numpy(gam).to(dev)


def both(dev, call, inputs):
    """The call's results on the default stream, then on a side stream."""
    want = [call(x) for x in inputs]
    torch.cuda.synchronize()
    side = torch.cuda.Stream(dev)
    with torch.cuda.stream(side):
        got = [call(x) for x in inputs]
    side.synchronize()
    for w, g in zip(want, got):
        assert np.array_equal(w.cpu().numpy().view(np.uint8), g.cpu().numpy().view(np.uint8))


@pytest.mark.parametrize("loop", [False, True])
def test_hafnians_in_one_call(dev, loop):
    both(dev, lambda x: api.hafnian_repeated(*x[0], gamma=x[1] if loop else None),
         [hafnians(s, dev) for s in range(ROUNDS)])


@pytest.mark.parametrize("loop", [False, True])
def test_hafnian_plan_run_at_once(dev, loop):
    def call(x):
        plan = api.HafnianPlan(*x[0][1:], loop)
        return plan.run(x[0][0], x[1] if loop else None)

    both(dev, call, [hafnians(s, dev) for s in range(ROUNDS)])


def batch(seed, dev):
    rng = np.random.default_rng(seed)
    items = []
    for _ in range(int(rng.integers(1, 40))):
        n = int(rng.integers(2, 10))
        A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        items.append((A, [1] * n, [1] * n) if n % 2 else
                     (A[:n // 2, :n // 2], [2] * (n // 2), [2] * (n // 2)))
    pb = W.pack_batch(items)
    go = rng.standard_normal(len(items)) + 1j * rng.standard_normal(len(items))
    return pb, api.DeviceBatch(pb, dev), torch.from_numpy(go).to(dev)


@pytest.mark.parametrize("method", ["batched", "plain"])
def test_permanents_planned_and_run_at_once(dev, method):
    """The forward, and the first backward call, which plans the backward."""
    def call(x):
        pb, db, go = x
        plan = api.Plan.for_batch(pb, method=method)
        per = api.permanent_batched(db, plan)
        return torch.cat([per, api.permanent_backward(db, go, plan)])

    both(dev, call, [batch(s, dev) for s in range(ROUNDS)])


def test_lossy_planned_and_run_at_once(dev):
    def inputs(seed):
        rng = np.random.default_rng(seed)
        m = 3 + seed % 4
        s = np.array([1, 1, 1] + [0] * (m - 3), dtype=np.int32)
        t = np.concatenate([W.compositions(q, m) for q in range(4)])
        dev_of = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
        return (m, s, t), [dev_of(x) for x in (W.haar_unitary(m, rng), rng.uniform(0.5, 0.9, m),
                                               W.haar_unitary(m, rng))]

    both(dev, lambda x: api.LossyPlan(*x[0]).run(*x[1]), [inputs(s) for s in range(ROUNDS)])
