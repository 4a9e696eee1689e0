"""The walks' block-integer arithmetic (permanents and hafnians) where it can go
wrong: low words at the edge of their range, scales over the whole exponent
range, entries that vanish beside the largest, exact zeros, and inputs that have
no scale at all (non-finite, or a bound beyond FP64).  Permanents are compared
with exact rational values; the bound is that of an FP64 evaluation of the Glynn
sum, 8 n 2^-53 of the mean absolute term."""
import itertools
import math

import numpy as np
import pytest

import oracle as O
from paper_2403_04006_gb300 import api, workloads as W
from exact import abs_err, exact_perm_grouped

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return torch.device("cuda:0")


def abs_sum(A):
    """2^-(n-1) sum over sign vectors (first fixed) of prod_j |sum_i d_i a_ij|."""
    n = A.shape[0]
    signs = np.array(np.meshgrid(*[[1.0, -1.0]] * (n - 1), indexing="ij")).reshape(n - 1, -1).T
    d = np.concatenate([np.ones((signs.shape[0], 1)), signs], axis=1)
    return float(np.prod(np.abs(d @ A), axis=1).sum()) / 2 ** (n - 1)


def check(items, dev, method, sums):
    pb = W.pack_batch(items)
    plan = api.Plan.for_batch(pb, method=method, column_sums=sums)
    got = api.permanent_batched(api.DeviceBatch(pb, dev), plan).cpu().numpy()
    for q, ((B, r, c), g) in enumerate(zip(items, got)):
        A = np.repeat(np.repeat(np.asarray(B), r, 0), c, 1)
        err = abs_err(complex(g), exact_perm_grouped(B, r, c))
        assert err <= 8 * A.shape[0] * 2.0 ** -53 * abs_sum(A), (q, g, err)


FORMS = [(m, s) for m in ("batched", "plain") for s in ("shared", "registers")]


@pytest.mark.parametrize("method,sums", FORMS)
def test_low_words_at_the_edge(dev, method, sums):
    """Column sums whose integers have a low word of exactly 2^31 (with a
    column bound in (1, 2) the unit is 2^-61, so 2^-30 is 2^31 units), in the
    real and in the imaginary part, against columns of every size up to 9."""
    rng = np.random.default_rng(1)
    items = []
    for n in range(2, 10):
        for part in (1.0, 1j):
            A = rng.integers(-4, 5, (n, n)) / (8.0 * n) + 1j * rng.integers(-4, 5, (n, n)) / (8.0 * n)
            A[0] += 1.0 + part * 2.0 ** -30
            items.append((A, [1] * n, [1] * n))
        items.append((A[:, :2] if n == 2 else A[:, :n - 1], [1] * n,
                      [1] * 2 if n == 2 else [2] + [1] * (n - 2)))
    check(items, dev, method, sums)


@pytest.mark.parametrize("method,sums", FORMS)
def test_scales_over_the_exponent_range(dev, method, sums):
    """Columns times 2^400, 2^-400 and subnormal columns beside large ones,
    with repeated rows and columns; entries below the unit of their column."""
    rng = np.random.default_rng(2)
    items = []
    for n in (2, 3, 5, 6):
        A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        e = np.where(np.arange(n) % 2 == 0, 400, -400)
        items.append((np.ldexp(A.real, e) + 1j * np.ldexp(A.imag, e), [1] * n, [1] * n))
    A = rng.standard_normal((3, 3)) + 1j * rng.standard_normal((3, 3))
    e = np.array([-1060, 500, 500])
    items.append((np.ldexp(A.real, e) + 1j * np.ldexp(A.imag, e), [1] * 3, [1] * 3))
    A = rng.standard_normal((4, 3)) + 1j * rng.standard_normal((4, 3))
    A[1] *= 1e-17
    A[2] *= 1e-25
    items.append((A, [1, 2, 1, 2], [3, 2, 1]))
    check(items, dev, method, sums)


@pytest.mark.parametrize("method,sums", FORMS)
def test_exact_zeros(dev, method, sums):
    """A zero row, a zero column, and a block structure without a perfect
    matching give exactly zero."""
    rng = np.random.default_rng(3)
    items = []
    for n in (2, 4, 7, 11):
        A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        Z = A.copy()
        Z[n // 2] = 0
        items.append((Z, [1] * n, [1] * n))
        Z = A.copy()
        Z[:, n - 1] = 0
        items.append((Z, [1] * n, [1] * n))
    pb = W.pack_batch(items)
    got = api.permanent_batched(api.DeviceBatch(pb, dev),
                                api.Plan.for_batch(pb, method=method, column_sums=sums))
    assert (got.cpu().numpy() == 0).all()


@pytest.mark.parametrize("method,sums", FORMS)
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 1.7e308])
def test_inputs_without_a_scale(dev, method, sums, bad):
    """An infinite or NaN entry, or a column whose sums overflow FP64, gives a
    result that is not finite; the permanents beside it keep their bits."""
    rng = np.random.default_rng(4)
    items = []
    for n in (1, 3, 6, 10):
        A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        items.append((A, [1] * n, [1] * n))
    clean = W.pack_batch(items)
    want = api.permanent_batched(api.DeviceBatch(clean, dev),
                                 api.Plan.for_batch(clean, method=method, column_sums=sums))
    dirty = []
    for A, r, c in items:
        A = A.copy()
        A[0, 0] = bad
        A[-1, 0] = bad
        dirty.append((A, r, c))
    pb = W.pack_batch(items[:2] + dirty[1:] + items[2:])
    got = api.permanent_batched(api.DeviceBatch(pb, dev),
                                api.Plan.for_batch(pb, method=method, column_sums=sums))
    got, want = got.cpu().numpy(), want.cpu().numpy()
    assert np.array_equal(got[[0, 1, 5, 6]].view(np.float64), want.view(np.float64))
    assert not np.isfinite(got[2:5]).any()


# ------------------------------------------------------------------ hafnians
def haf_items(rng):
    """(B, repetitions, loop weights): sizes from one index up, entries scaled
    by powers of two, one entry far above the others, loop weights far above
    and far below the square root of the entries, and none."""
    out = []
    for k in (1, 2, 3, 4, 5):
        for e, ge in ((0, 0), (200, 100), (-200, -100), (0, 60), (0, -60)):
            B = rng.standard_normal((k, k)) + 1j * rng.standard_normal((k, k))
            B = (B + B.T) / 2
            if k > 1 and e == 0:
                B[0, 1] *= 1e9
                B[1, 0] = B[0, 1]
            gam = rng.standard_normal(k) + 1j * rng.standard_normal(k)
            r = rng.integers(1, 4, k)
            out.append((np.ldexp(B.real, e) + 1j * np.ldexp(B.imag, e), r,
                        np.ldexp(gam.real, ge) + 1j * np.ldexp(gam.imag, ge)))
        out.append((B, r, np.zeros(k, dtype=complex)))
    return out


def run_hafnians(items, dev, loop):
    ks = np.array([B.shape[0] for B, _, _ in items], dtype=np.int32)
    mo = np.concatenate([[0], np.cumsum(ks.astype(np.int64) ** 2)[:-1]])
    ro = np.concatenate([[0], np.cumsum(ks, dtype=np.int64)[:-1]])
    mats = torch.from_numpy(np.concatenate([B.reshape(-1) for B, _, _ in items])).to(dev)
    gam = torch.from_numpy(np.concatenate([g for _, _, g in items])).to(dev)
    rep = np.concatenate([r for _, r, _ in items]).astype(np.int32)
    return api.hafnian_repeated(mats, mo, ks, rep, ro, gamma=gam if loop else None).cpu().numpy()


@pytest.mark.parametrize("loop", [False, True])
def test_hafnian_scales(dev, loop):
    """Against the oracle's double-double sum, within 32 N 2^-53 of the sum of
    the terms' magnitudes (an FP64 evaluation's own bound: N products, the
    updates of q and l, and the accumulation)."""
    items = haf_items(np.random.default_rng(5))
    got = run_hafnians(items, dev, loop)
    for q, ((B, r, g), v) in enumerate(zip(items, got)):
        want, scale = (O.lhaf_grouped(B, g, r, info=True) if loop
                       else O.haf_grouped(B, r, info=True))
        if not np.isfinite(want):  # beyond FP64
            assert not np.isfinite(v)
            continue
        assert abs(v - want) <= 32 * int(sum(r)) * 2.0 ** -53 * max(scale, abs(want)), (q, v, want)


@pytest.mark.parametrize("loop", [False, True])
@pytest.mark.parametrize("bad", [np.inf, np.nan, 1.2e308])
def test_hafnians_without_a_scale(dev, loop, bad):
    """Non-finite entries and sums beyond FP64 give results that are not
    finite; the items beside them keep their bits, a zero matrix gives zero."""
    rng = np.random.default_rng(6)
    items = [x for x in haf_items(rng) if x[0].shape[0] > 1][:6]
    items = [(B, 2 * np.ones_like(r), g) for B, r, g in items]
    want = run_hafnians(items, dev, loop)
    dirty = []
    for B, r, g in items[:2]:
        B = B.copy()
        B[0, 1] = B[1, 0] = bad
        dirty.append((B, r, g))
    zero = (np.zeros((3, 3), dtype=complex), np.array([2, 1, 1]), np.zeros(3, dtype=complex))
    got = run_hafnians(items[:3] + dirty + [zero] + items[3:], dev, loop)
    assert np.array_equal(got[[0, 1, 2, 6, 7, 8]].view(np.float64), want.view(np.float64))
    assert not np.isfinite(got[3:5]).any()
    assert got[5] == 0


# ------------------------------------------------------------------ gradients
def gray_terms(m):
    """Terms when this side is summed: one copy of its least repeated line fixed."""
    return math.prod(int(x) + 1 for x in m) // (min(m) + 1) * min(m)


def grad_abs(B, r, c):
    """c_j times the mean over the sign vectors of |x_i| |prod of the column sums
    without one factor S_j|, rows summed: the size of the gradient's terms."""
    g = np.array(list(itertools.product(*[range(int(x) + 1) for x in r])))
    w = np.prod([[math.comb(int(ri), int(q)) for ri, q in zip(r, row)] for row in g], axis=1)
    x = np.asarray(r) - 2 * g
    S = np.abs(x @ B)
    out = np.zeros(B.shape)
    for j in range(B.shape[1]):
        e = np.asarray(c) - (np.arange(B.shape[1]) == j)
        q = w * np.prod(S ** e, axis=1)
        out[:, j] = c[j] * (np.abs(x) * q[:, None]).sum(axis=0) / 2.0 ** int(sum(r))
    return out


@pytest.mark.parametrize("method", ["batched", "plain"])
def test_gradient_scales(dev, method):
    """dper/db of every product width up to 18, the product side's columns scaled
    by powers of two (scaling the summed side would cancel in any arithmetic of
    53 or 64 bits), repeated rows and columns and zero entries, against the
    oracle's minors, within 16 n 2^-53 of the terms' size (n - 1 products, the
    sums' updates and the accumulation in FP64)."""
    rng = np.random.default_rng(7)
    items, flip = [], []
    for l in list(range(1, 11)) + [12, 13, 14, 15, 16, 17, 18]:
        k = min(l, 5)
        B = rng.standard_normal((k, l)) + 1j * rng.standard_normal((k, l))
        c = [1] * l if l > 8 else list(rng.integers(1, 4, l))
        n = int(sum(c))
        r = [n // k + (i < n % k) for i in range(k)]
        flip.append(gray_terms(c) < gray_terms(r))  # the columns are summed
        e = rng.integers(-60, 61, (k, 1) if flip[-1] else (1, l))
        B = np.ldexp(B.real, e) + 1j * np.ldexp(B.imag, e)
        if l == 7:
            B[1, 2:4] = 0
        items.append((B, r, c))
    pb = W.pack_batch(items)
    go = torch.ones(pb.batch, dtype=torch.complex128, device=dev)
    db = api.DeviceBatch(pb, dev)
    plan = api.Plan.for_batch(pb, method=method)
    got = api.permanent_backward(db, go, plan).cpu().numpy()
    for b, (B, r, c) in enumerate(items):
        if flip[b]:  # the oracle, too, has to sum the side that is not scaled
            want, size = O.perm_grad(B.T, c, r, gold=True).T, grad_abs(B.T, c, r).T
        else:
            want, size = O.perm_grad(B, r, c, gold=True), grad_abs(B, r, c)
        want = np.conj(want)
        g = got[pb.mat_off[b]:pb.mat_off[b] + B.size].reshape(B.shape)
        assert (abs(g - want) <= 16 * sum(r) * 2.0 ** -53 * size).all(), b


@pytest.mark.parametrize("method", ["batched", "plain"])
@pytest.mark.parametrize("bad", [np.inf, np.nan, 1.7e308])
def test_gradients_without_a_scale(dev, method, bad):
    """A non-finite entry makes its permanent's gradient not finite somewhere;
    the gradients beside it keep their bits."""
    rng = np.random.default_rng(8)
    clean = []
    for n in (2, 3, 6, 10, 13):
        clean.append((rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)),
                      [1] * n, [1] * n))
    dirty = []
    for A, r, c in clean:
        A = A.copy()
        A[0, 0] = A[1, 0] = bad
        dirty.append((A, r, c))

    def grads(items):
        pb = W.pack_batch(items)
        go = torch.ones(pb.batch, dtype=torch.complex128, device=dev)
        g = api.permanent_backward(api.DeviceBatch(pb, dev), go, api.Plan.for_batch(pb, method=method))
        g = g.cpu().numpy()
        return [g[o:o + B.size] for o, (B, _, _) in zip(pb.mat_off, items)]

    want = grads(clean)
    got = grads([x for pair in zip(clean, dirty) for x in pair])
    for q in range(len(clean)):
        assert np.array_equal(got[2 * q].view(np.float64), want[q].view(np.float64))
        assert not np.isfinite(got[2 * q + 1]).all()
