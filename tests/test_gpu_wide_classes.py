"""The register-resident forward classes of 22 to 32 product columns: a batch of
one width each, few summed rows of high multiplicity (so that it has few terms),
without repeated columns, with some, and with as many as n <= 48 leaves room for.
Registers and shared memory form the same products in the same order, so with the
same chunks they give the same bits; both are compared with exact rational values,
within 8 n 2^-53 of the mean absolute term."""
import itertools
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from exact import abs_err, exact_perm_grouped  # noqa: E402
from paper_2403_04006_gb300 import api, pq  # noqa: E402
from paper_2403_04006_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def column_mults(l):
    room = 48 - l
    out = [[1] * l, [2] + [1] * (l - 1), [2] * min(l, room) + [1] * max(0, l - room),
           [3, 2, 2] + [1] * (l - 3)]
    if room > l:
        out.append([3] + [2] * (l - 1))
    return [c for c in out if sum(c) <= 48]


def mean_abs_term(B, r, c):
    tot = 0.0
    for g in itertools.product(*[range(x + 1) for x in r]):
        w = math.prod(math.comb(x, q) for x, q in zip(r, g))
        S = np.abs((np.array(r) - 2 * np.array(g)) @ B)
        tot += w * float(np.prod(S ** np.array(c)))
    return tot / 2.0 ** sum(r)


@pytest.mark.parametrize("l", range(21, 33))
def test_wide_register_class(l):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pq.load_library()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(l)
    items = []
    for c in column_mults(l):
        n = sum(c)
        for r in ([n // 2, n - n // 2], [n // 3, n // 3, n - 2 * (n // 3)]):
            B = rng.standard_normal((len(r), l)) + 1j * rng.standard_normal((len(r), l))
            items.append((B / 4.0, r, c))
    pb = W.pack_batch(items)
    db = api.DeviceBatch(pb, dev)
    got = {}
    for method, sums in itertools.product(("batched", "plain"), ("auto", "shared")):
        plan = api.Plan.for_batch(pb, method=method, column_sums=sums, chunk_log2=4)
        assert plan.stats()["column_sums"] == ("registers" if sums == "auto" else "shared")
        got[method, sums] = api.permanent_batched(db, plan).cpu().numpy()
    first = got["batched", "auto"]
    for v in got.values():
        assert np.array_equal(v.view(np.float64), first.view(np.float64))
    for q, (B, r, c) in enumerate(items):
        err = abs_err(complex(first[q]), exact_perm_grouped(B, r, c))
        assert err <= 8 * sum(r) * 2.0 ** -53 * mean_abs_term(B, r, c), (q, err)
