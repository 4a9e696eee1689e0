"""Columns whose entries are all subnormal, at the edge of their scale: the largest
subnormal, whose sums lie a few units below a power of two, beside columns of
1e300, so that products are normal numbers."""
import itertools
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from exact import exact_perm_grouped  # noqa: E402
from paper_2403_04006_gb300 import api, pq  # noqa: E402
from paper_2403_04006_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
FORMS = [(m, s) for m in ("batched", "plain") for s in ("shared", "registers")]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pq.load_library()
    return torch.device("cuda:0")


def at_the_bound():
    """One row or two equal rows, every summed entry +-the largest subnormal in
    its real part, its imaginary part or both: the column's sum is its bound,
    a few units below a power of two.  Beside them columns of 1e300, so that
    products are normal numbers."""
    a = (2 ** 52 - 1) * 2.0 ** -1074
    for z in (a, -a, 1j * a, -1j * a, a - 1j * a, -a + 1j * a, -a - 1j * a):
        b = 1e300 - 0.7e300j
        yield np.array([[z, b]]), [4], [2, 2]
        yield np.array([[z, b]]), [2], [1, 1]
        yield np.array([[z, b], [z, b]]), [2, 2], [2, 2]
        yield np.array([[b, z, b], [b, z, b]]), [2, 2], [2, 1, 1]


def near(g, want, tol, least=0.0):
    """|g - want| <= tol max(|want|, least), in exact arithmetic; beyond FP64,
    not finite."""
    if max(abs(w) for w in want) >= 2 ** 1024:
        return not np.isfinite(g)
    if not np.isfinite(g):
        return False
    err2 = (Fraction(g.real) - want[0]) ** 2 + (Fraction(g.imag) - want[1]) ** 2
    size2 = max(want[0] ** 2 + want[1] ** 2, Fraction(least) ** 2)
    return err2 <= Fraction(tol) ** 2 * size2


@pytest.mark.parametrize("method,sums", FORMS)
def test_largest_subnormal(dev, method, sums):
    """All terms have the phase of the permanent and sum to less than twice its
    size in magnitude: 16 n 2^-53 of the permanent."""
    items = list(at_the_bound())
    pb = W.pack_batch(items)
    plan = api.Plan.for_batch(pb, method=method, column_sums=sums)
    got = api.permanent_batched(api.DeviceBatch(pb, dev), plan).cpu().numpy()
    for q, ((B, r, c), g) in enumerate(zip(items, got)):
        assert near(g, exact_perm_grouped(B, r, c), 16 * sum(r) * 2.0 ** -53), (q, g)


@pytest.mark.parametrize("method", ["batched", "plain"])
def test_gradient_at_the_largest_subnormal(dev, method):
    """dper/db_ij = r_i c_j times the permanent with one copy of each less: 16 n
    2^-53 of it, and of the smallest normal number where it is below that."""
    items = list(at_the_bound())
    pb = W.pack_batch(items)
    go = torch.ones(pb.batch, dtype=torch.complex128, device=dev)
    plan = api.Plan.for_batch(pb, method=method)
    got = api.permanent_backward(api.DeviceBatch(pb, dev), go, plan).cpu().numpy()
    for q, (B, r, c) in enumerate(items):
        g = np.conj(got[pb.mat_off[q]:pb.mat_off[q] + B.size].reshape(B.shape))
        for i, j in itertools.product(range(B.shape[0]), range(B.shape[1])):
            r1 = [x - (e == i) for e, x in enumerate(r)]
            c1 = [x - (e == j) for e, x in enumerate(c)]
            want = [r[i] * c[j] * x for x in exact_perm_grouped(B, r1, c1)]
            assert near(g[i, j], want, 16 * sum(r) * 2.0 ** -53, 2.0 ** -1022), (q, i, j, g[i, j])
