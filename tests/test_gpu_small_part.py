"""Values whose imaginary part is far below the real one, or the other way round:
A + i h D with h from 2^-3 down to 1e-200 (a complex step, a small phase), and i
times it.  Each part is compared with its exact rational value, within a bound of
its own: an FP64 evaluation rounds every part of every factor relative to itself,
so the error of the product's parts is at most 8 n 2^-53 of their majorants.  With
R_j and I_j the sums of a column's real and imaginary parts' magnitudes, these are
the even and odd parts in t of prod_j (R_j + t I_j) at t = 1."""
import itertools
import math
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from exact import exact_perm_grouped  # noqa: E402
from paper_2403_04006_gb300 import api, pq  # noqa: E402
from paper_2403_04006_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
STEPS = (2.0 ** -3, 2.0 ** -5, 1e-3, 1e-8, 1e-12, 1e-20, 1e-200)
FORMS = [(m, s) for m in ("batched", "plain") for s in ("shared", "registers")]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pq.load_library()
    return torch.device("cuda:0")


def parts_ok(got, want, f, tol):
    """|part(got) - part(want)| <= tol times the even and odd parts of f at 1, or
    half the smallest subnormal (the rounding of a value below FP64's range)."""
    even, odd = (f(1) + f(-1)) / 2, (f(1) - f(-1)) / 2
    least = Fraction(1, 2 ** 1075)
    return (abs(Fraction(got.real) - want[0]) <= max(Fraction(tol) * even, least)
            and abs(Fraction(got.imag) - want[1]) <= max(Fraction(tol) * odd, least))


def mags(B):
    F = np.vectorize(lambda x: Fraction(abs(float(x))), otypes=[object])
    return F(B.real), F(B.imag)


def perm_majorant(B, r, c):
    """t -> prod_j (R_j + t I_j)^{c_j}, R_j = sum_i r_i |Re b_ij|."""
    re, im = mags(B)
    R = [sum(int(r[i]) * re[i, j] for i in range(B.shape[0])) for j in range(B.shape[1])]
    I = [sum(int(r[i]) * im[i, j] for i in range(B.shape[0])) for j in range(B.shape[1])]
    return lambda t: math.prod((x + t * y) ** int(m) for x, y, m in zip(R, I, c))


def near_axis_items(seed):
    rng = np.random.default_rng(seed)
    out = []
    for h in STEPS:
        for n in range(1, 9):
            A, D = rng.standard_normal((2, n, n))
            B = A + 1j * h * D
            out.append((B if n % 3 else 1j * B, [1] * n, [1] * n))
        B = rng.standard_normal((3, 3)) + 1j * h * rng.standard_normal((3, 3))
        out.append((B, [2, 1, 3], [3, 2, 1]))
        B = rng.standard_normal((2, 4)) + 1j * h * rng.standard_normal((2, 4))
        B[:, 1] *= 1j  # some columns near the one axis, some near the other, some on one
        B[:, 2] = B[:, 2].real
        out.append((B, [4, 3], [2, 2, 2, 1]))
        B = rng.standard_normal((4, 4)) + 1j * h * rng.standard_normal((4, 4))
        out.append((B * np.ldexp(1.0, [300, 200, 200, -650]), [1] * 4, [1] * 4))
    return out


@pytest.mark.parametrize("method,sums", FORMS)
def test_permanents(dev, method, sums):
    items = near_axis_items(11)
    pb = W.pack_batch(items)
    plan = api.Plan.for_batch(pb, method=method, column_sums=sums)
    got = api.permanent_batched(api.DeviceBatch(pb, dev), plan).cpu().numpy()
    for q, ((B, r, c), g) in enumerate(zip(items, got)):
        assert parts_ok(g, exact_perm_grouped(B, r, c), perm_majorant(B, r, c),
                        8 * sum(r) * 2.0 ** -53), (q, g)


def test_one_class_in_registers(dev):
    """A batch of one width, which the planner walks in registers."""
    items = [(B, r, c) for B, r, c in near_axis_items(12) if B.shape == (8, 8)]
    pb = W.pack_batch(items)
    plan = api.Plan.for_batch(pb)
    assert plan.stats()["column_sums"] == "registers"
    got = api.permanent_batched(api.DeviceBatch(pb, dev), plan).cpu().numpy()
    for q, ((B, r, c), g) in enumerate(zip(items, got)):
        assert parts_ok(g, exact_perm_grouped(B, r, c), perm_majorant(B, r, c),
                        8 * sum(r) * 2.0 ** -53), (q, g)


@pytest.mark.parametrize("sums", ["shared", "registers"])
@pytest.mark.parametrize("chunk_log2", [1, 6])
def test_many_tasks_and_long_chunks(dev, sums, chunk_log2):
    """2048 terms of n = 12 in chunks of 2 (32 tasks) and of 64 (two folds)."""
    rng = np.random.default_rng(16)
    items = []
    for h in (1e-3, 1e-12, 1e-200):
        B = rng.standard_normal((12, 12)) + 1j * h * rng.standard_normal((12, 12))
        items += [(B, [1] * 12, [1] * 12), (1j * B[:, :8], [1] * 12, [2] * 4 + [1] * 4)]
    pb = W.pack_batch(items)
    plan = api.Plan.for_batch(pb, column_sums=sums, chunk_log2=chunk_log2)
    got = api.permanent_batched(api.DeviceBatch(pb, dev), plan).cpu().numpy()
    for q, ((B, r, c), g) in enumerate(zip(items, got)):
        assert parts_ok(g, exact_perm_grouped(B, r, c), perm_majorant(B, r, c),
                        8 * sum(r) * 2.0 ** -53), (q, g)


def test_shards(dev):
    """The partial sums of three shards, combined."""
    items = [x for x in near_axis_items(17) if sum(x[1]) == 8]
    pb = W.pack_batch(items)
    db = api.DeviceBatch(pb, dev)
    parts = [api.permanent_partials(db, api.Plan.for_batch(pb, shard=(q, 3))).cpu().numpy()
             for q in range(3)]
    got = api.combine_partials(parts, api.photon_numbers(pb))
    for q, ((B, r, c), g) in enumerate(zip(items, got)):
        assert parts_ok(g, exact_perm_grouped(B, r, c), perm_majorant(B, r, c),
                        8 * sum(r) * 2.0 ** -53), (q, g)


@pytest.mark.parametrize("method", ["batched", "plain"])
def test_gradients(dev, method):
    """dper/db_ij = r_i c_j times the permanent with one copy of each less; two
    more roundings per factor than the permanent has."""
    items = [x for x in near_axis_items(13) if sum(x[1]) <= 6]
    rng = np.random.default_rng(14)
    for h in STEPS:  # one column off the axes: the entries below it stay near one
        B = rng.standard_normal((3, 3)) + 1j * h * rng.standard_normal((3, 3))
        B[:, 2] = rng.standard_normal(3) + 1j * rng.standard_normal(3)
        items.append((B, [1] * 3, [1] * 3))
    pb = W.pack_batch(items)
    go = torch.ones(pb.batch, dtype=torch.complex128, device=dev)
    plan = api.Plan.for_batch(pb, method=method)
    got = api.permanent_backward(api.DeviceBatch(pb, dev), go, plan).cpu().numpy()
    for q, (B, r, c) in enumerate(items):
        g = np.conj(got[pb.mat_off[q]:pb.mat_off[q] + B.size].reshape(B.shape))
        for i, j in itertools.product(range(B.shape[0]), range(B.shape[1])):
            r1 = [x - (e == i) for e, x in enumerate(r)]
            c1 = [x - (e == j) for e, x in enumerate(c)]
            w = r[i] * c[j]
            want = [w * x for x in exact_perm_grouped(B, r1, c1)]
            # the walk forms it from sums with all r_i copies of the row
            f = perm_majorant(B, r, c1)
            assert parts_ok(g[i, j], want, lambda t: w * f(t), 16 * sum(r) * 2.0 ** -53), (q, i, j)


# ------------------------------------------------------------------ hafnians
def exact_haf(B, g, idx):
    """(Loop) hafnian of the expanded index list, exactly: the first index is
    matched with each other one, or with itself (weight g, None: not allowed)."""
    if not idx:
        return Fraction(1), Fraction(0)
    i, rest = idx[0], idx[1:]
    tot = [Fraction(0), Fraction(0)]

    def add(z, sub):
        x, y = Fraction(z.real), Fraction(z.imag)
        tot[0] += x * sub[0] - y * sub[1]
        tot[1] += x * sub[1] + y * sub[0]

    if g is not None:
        add(g[i], exact_haf(B, g, rest))
    for e, j in enumerate(rest):
        add(B[i, j], exact_haf(B, g, rest[:e] + rest[e + 1:]))
    return tot


def haf_majorant(B, g, r):
    """t -> sum_j q^j l^{N-2j} / (j! (N-2j)!) at q = Q_re + t Q_im, l = L_re + t L_im."""
    re, im = mags(B)
    N, k = int(sum(r)), len(r)
    pairs = [(i, j, Fraction(int(r[i]) * (int(r[j]) + (i == j)), 2)) for i in range(k) for j in range(k)]
    q = [sum(w * m[i, j] for i, j, w in pairs) for m in (re, im)]
    gre, gim = mags(np.asarray(g if g is not None else np.zeros(k, dtype=complex)))
    l = [sum(int(r[i]) * m[i] for i in range(k)) for m in (gre, gim)]

    def f(t):
        x, y = q[0] + t * q[1], l[0] + t * l[1]
        low = 0 if g is not None else N // 2
        return sum(x ** j * y ** (N - 2 * j) / (math.factorial(j) * math.factorial(N - 2 * j))
                   for j in range(low, N // 2 + 1))
    return f


def haf_items(seed):
    rng = np.random.default_rng(seed)
    out = []

    def sym(k, h):
        B = rng.standard_normal((k, k)) + 1j * h * rng.standard_normal((k, k))
        return (B + B.T) / 2

    for h in STEPS:
        for k, r in ((2, [1, 1]), (2, [2, 2]), (3, [1, 2, 1]), (4, [1, 1, 1, 1]), (3, [2, 2, 2]),
                     (4, [1, 2, 1, 2])):
            gam = rng.standard_normal(k) + 1j * h * rng.standard_normal(k)
            out.append((sym(k, h), r, gam))
            out.append((1j * sym(k, h), r, gam))
        # small weights off the axes beside real entries, entries beside real weights
        out.append((sym(3, 0.0), [2, 1, 2], h * (rng.standard_normal(3) + 1j * rng.standard_normal(3))))
        out.append((h * sym(3, 1.0), [2, 1, 1], rng.standard_normal(3) + 0j))
        out.append((sym(1, h), [1], rng.standard_normal(1) + 1j * h * rng.standard_normal(1)))
        B = sym(4, h) * 2.0 ** 260
        out.append((B, [1, 1, 2, 2], np.zeros(4, dtype=complex)))
    return out


@pytest.mark.parametrize("loop", [False, True])
def test_diagonal_of_single_indices(dev, loop):
    """An index that occurs once has no pair with itself: its diagonal entry, however
    large, takes nothing from the result (32 N 2^-53 of the majorants of the matrix
    without these entries), unless it is not finite."""
    rng = np.random.default_rng(18)
    items = []
    for size in (1e6, 1e6j, 1e40, -1e40j, 1e300 + 1e300j):
        for k, r in ((2, [1, 1]), (4, [1, 1, 1, 1]), (3, [1, 2, 1]), (4, [2, 1, 1, 2])):
            B = rng.standard_normal((k, k)) + 1j * rng.standard_normal((k, k))
            B = (B + B.T) / 2
            free = B.copy()
            for i in range(k):
                if r[i] == 1:
                    B[i, i], free[i, i] = size * (1.0 + i), 0
            items.append((B, free, r, rng.standard_normal(k) + 1j * rng.standard_normal(k)))
    ks = np.array([B.shape[0] for B, _, _, _ in items], dtype=np.int32)
    mo = np.concatenate([[0], np.cumsum(ks.astype(np.int64) ** 2)[:-1]])
    ro = np.concatenate([[0], np.cumsum(ks, dtype=np.int64)[:-1]])
    mats = torch.from_numpy(np.concatenate([B.reshape(-1) for B, _, _, _ in items])).to(dev)
    gam = torch.from_numpy(np.concatenate([g for _, _, _, g in items])).to(dev)
    rep = np.concatenate([r for _, _, r, _ in items]).astype(np.int32)
    got = api.hafnian_repeated(mats, mo, ks, rep, ro, gamma=gam if loop else None).cpu().numpy()
    for q, ((_, B, r, g), v) in enumerate(zip(items, got)):
        g = g if loop else None
        idx = [i for i, x in enumerate(r) for _ in range(x)]
        assert parts_ok(v, exact_haf(B, g, idx), haf_majorant(B, g, r), 32 * sum(r) * 2.0 ** -53), (q, v)
    mats[0] = float("inf")
    got = api.hafnian_repeated(mats, mo, ks, rep, ro, gamma=gam if loop else None).cpu().numpy()
    assert not np.isfinite(got[0])


@pytest.mark.parametrize("loop", [False, True])
def test_hafnians(dev, loop):
    """32 N 2^-53 of the majorants: N products, the updates of q and l, and the
    accumulation."""
    items = [x for x in haf_items(15) if loop or sum(x[1]) % 2 == 0]
    ks = np.array([B.shape[0] for B, _, _ in items], dtype=np.int32)
    mo = np.concatenate([[0], np.cumsum(ks.astype(np.int64) ** 2)[:-1]])
    ro = np.concatenate([[0], np.cumsum(ks, dtype=np.int64)[:-1]])
    mats = torch.from_numpy(np.concatenate([B.reshape(-1) for B, _, _ in items])).to(dev)
    gam = torch.from_numpy(np.concatenate([g for _, _, g in items])).to(dev)
    rep = np.concatenate([r for _, r, _ in items]).astype(np.int32)
    got = api.hafnian_repeated(mats, mo, ks, rep, ro, gamma=gam if loop else None).cpu().numpy()
    for q, ((B, r, g), v) in enumerate(zip(items, got)):
        g = g if loop else None
        idx = [i for i, x in enumerate(r) for _ in range(x)]
        want = exact_haf(B, g, idx)
        if max(map(abs, want)) >= 2 ** 1024:
            assert not np.isfinite(v), q
            continue
        assert parts_ok(v, want, haf_majorant(B, g, r), 32 * sum(r) * 2.0 ** -53), (q, v)
