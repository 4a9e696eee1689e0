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
