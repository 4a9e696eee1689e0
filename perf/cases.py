"""The calls this framework is timed on: what a user of a photonic simulator
asks of it, from a few hundred small permanents to one large one.

Every case is a dict of plain values with a ``kind``:

  bs        probabilities and amplitudes of output patterns, planned
  mesh      Clements mesh -> probabilities -> gradient of a loss (training step)
  ragged    a batch of permanents of uneven size, forward or forward + backward
  power     one k x k permanent, every row and column repeated r times
  sample    the Algorithm A sampler, planned
  lossy     detection probabilities with losses, planned
  hafnian   one (loop) hafnian of a k x k base, every index repeated, planned
  hafnians  a ragged batch of (loop) hafnians, planned inside the call

``exact`` evaluates permanents by Laplace expansion over row multisets and
hafnians by expansion over their first index: sums without the cancellation of
a sign-vector formula, in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2403_04006_gb300 import api
from paper_2403_04006_gb300.workloads import (PermBatch, compositions, haar_unitaries,
                                              haar_unitary, gbs_matrix, sampler_draws)


def listed():
    return [
        # all probabilities of a small interferometer: what a notebook or a
        # test calls in a loop; launches and latency count
        {"name": "bs-m8-n4-all", "kind": "bs", "m": 8, "n": 4, "count": 330, "cap": 4, "every": True},
        # a validation run of a 12-photon experiment: many patterns, one size
        {"name": "bs-m24-n12-4096", "kind": "bs", "m": 24, "n": 12, "count": 4096, "cap": 3,
         "every": False},
        # one training step of a 16-mode mesh
        {"name": "mesh-m16-n8-1024", "kind": "mesh", "m": 16, "n": 8, "count": 1024},
        # simulator back end: a big batch of permanents of every size with
        # repeated rows and columns
        {"name": "ragged-65536", "kind": "ragged", "count": 65536, "nmin": 4, "nmax": 20,
         "backward": False},
        # the same recipe at an ordinary batch size, with gradients
        {"name": "ragged-4096-backward", "kind": "ragged", "count": 4096, "nmin": 4, "nmax": 20,
         "backward": True},
        # one large collision-free amplitude
        {"name": "single-n30", "kind": "power", "k": 30, "r": 1, "method": "batched"},
        # the repeated-permanent benchmark shape, one launch per permanent
        {"name": "repeated-2x-k14-plain", "kind": "power", "k": 14, "r": 2, "method": "plain"},
        # drawing samples from a fixed 16-mode experiment
        {"name": "sample-m16-n8-2000", "kind": "sample", "m": 16, "n": 8, "count": 2000},
        # every detection pattern of a lossy 10-mode experiment
        {"name": "lossy-m10-n5", "kind": "lossy", "m": 10, "n": 5},
        # the repeated-hafnian benchmark shape of Gaussian boson sampling
        {"name": "hafnian-2x-k18", "kind": "hafnian", "k": 18, "r": 2, "loop": False},
        # the loop-hafnian shape (displaced states)
        {"name": "loop-hafnian-2x-k14", "kind": "hafnian", "k": 14, "r": 2, "loop": True},
        # a few hundred small detection events, sizes new at every call
        {"name": "hafnians-300", "kind": "hafnians", "count": 300, "kmax": 8, "rmax": 3,
         "loop": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["bs", "bs", "mesh", "ragged", "ragged", "ragged", "power", "power",
                       "sample", "lossy", "hafnian", "hafnian", "hafnians"])
    if kind == "bs":
        n = rng.randint(2, 14)
        m = rng.randint(n, 40)
        count = _log_int(rng, 64, 8192)
        while count << (n - 1) > 1 << 24:
            count //= 2
        return {"kind": kind, "m": m, "n": n, "count": count, "cap": 3, "every": False}
    if kind == "mesh":
        n = rng.randint(3, 9)
        return {"kind": kind, "m": rng.randint(max(6, n), 20), "n": n,
                "count": _log_int(rng, 64, 2048)}
    if kind == "ragged":
        back = rng.random() < 0.5
        return {"kind": kind, "count": _log_int(rng, 64, 4096 if back else 32768),
                "nmin": rng.randint(2, 6), "nmax": rng.randint(8, 20), "backward": back}
    if kind == "power":
        r = rng.randint(1, 3)
        k = rng.randint(*{1: (12, 28), 2: (5, 16), 3: (4, 12)}[r])
        return {"kind": kind, "k": k, "r": r, "method": rng.choice(["batched", "plain"])}
    if kind == "sample":
        n = rng.randint(4, 10)
        return {"kind": kind, "m": rng.randint(n, 24), "n": n, "count": _log_int(rng, 100, 4000)}
    if kind == "lossy":
        m = rng.randint(4, 10)
        return {"kind": kind, "m": m, "n": rng.randint(2, min(m, 5))}
    if kind == "hafnian":
        loop = rng.random() < 0.5
        r = rng.randint(1, 3)
        k = rng.randint(*{1: (8, 24), 2: (4, 16), 3: (3, 11)}[r])
        if not loop and k * r % 2:
            k += 1
        return {"kind": kind, "k": k, "r": r, "loop": loop}
    return {"kind": kind, "count": _log_int(rng, 20, 600), "kmax": rng.randint(4, 8),
            "rmax": rng.randint(1, 3), "loop": rng.random() < 0.5}


# --------------------------------------------------------------------------
# inputs (host, from the seed alone)
# --------------------------------------------------------------------------
def _gen(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _first_modes(m, n):
    s = np.zeros(m, dtype=np.int32)
    s[:n] = 1
    return s


def _patterns(m, n, count, cap, g):
    """Half collision-free patterns, half of n photons in modes of capacity
    ``cap`` (n of the m cap slots without replacement)."""
    half = count // 2
    t = np.zeros((count, m), dtype=np.int32)
    free = np.argsort(g.random((half, m)), axis=1)[:, :n]
    slot = np.argsort(g.random((count - half, m * cap)), axis=1)[:, :n] // cap
    np.add.at(t, (np.arange(half)[:, None], free), 1)
    np.add.at(t, (np.arange(half, count)[:, None], slot), 1)
    return t


def _parts(n, draws):
    """Multiplicities of every item: parts from {1, 2, 3}, the last clipped so
    that they sum to n[b].  Returns (number of parts, parts row by row)."""
    before = np.cumsum(draws, axis=1) - draws
    p = np.minimum(draws, n[:, None] - before)
    keep = p > 0
    return keep.sum(axis=1).astype(np.int32), p[keep].astype(np.int32)


def _offsets(sizes):
    return (np.cumsum(sizes, dtype=np.int64) - sizes).astype(np.int64)


def _ragged(case, seed, values=True):
    """The batch on the host: n ~ U{nmin..nmax}, rows and columns repeated 1 to
    3 times, each base matrix a random block of one of 64 Haar unitaries of
    2n modes.  Another seed gives the same sizes in another order, so that the
    packed gradients keep their length, and other matrices."""
    g, fixed = _gen(seed), _gen(case["count"])
    order = g.permutation(case["count"])
    n = fixed.integers(case["nmin"], case["nmax"] + 1, size=case["count"])[order]
    parts = fixed.integers(1, 4, size=(2, n.size, case["nmax"]))[:, order]
    k, rm = _parts(n, parts[0])
    l, cm = _parts(n, parts[1])
    sizes = k.astype(np.int64) * l
    off = _offsets(sizes)
    mats = np.zeros(int(sizes.sum()), dtype=np.complex128)
    if values:
        for nn in np.unique(n):
            idx = np.nonzero(n == nn)[0]
            pool = haar_unitaries(min(64, idx.size), 2 * int(nn), g)
            rows = np.argsort(g.random((idx.size, 2 * nn)), axis=1)[:, :nn]
            cols = np.argsort(g.random((idx.size, 2 * nn)), axis=1)[:, :nn]
            which = g.integers(0, pool.shape[0], size=idx.size)
            blocks = pool[which[:, None, None], rows[:, :, None], cols[:, None, :]]
            keep = ((np.arange(nn)[None, :, None] < k[idx, None, None])
                    & (np.arange(nn)[None, None, :] < l[idx, None, None]))
            item, i, j = np.nonzero(keep)
            at = off[idx][item] + i * l[idx][item].astype(np.int64) + j
            mats[at] = blocks[keep]
    return PermBatch(mats, off, k, l, rm, _offsets(k), cm, _offsets(l))


def _grad_out(case, seed):
    g = _gen(seed + 1)
    return g.standard_normal(case["count"]) + 1j * g.standard_normal(case["count"])


def _host(case, seed):
    """The numbers of a case, as numpy arrays."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "bs":
        m, n = case["m"], case["n"]
        t = compositions(n, m) if case["every"] else _patterns(m, n, case["count"], case["cap"], g)
        return {"U": haar_unitary(m, g), "s": _first_modes(m, n), "t": t}
    if kind == "mesh":
        m, n = case["m"], case["n"]
        a = g.uniform(0.0, 2.0 * math.pi, size=(2, m * (m - 1) // 2))
        return {"theta": a[0].copy(), "phi": a[1].copy(), "s": _first_modes(m, n),
                "t": _patterns(m, n, case["count"], 3, g)}
    if kind == "power":
        k = case["k"]
        r = np.full(k, case["r"], dtype=np.int32)
        B = np.ascontiguousarray(haar_unitary(2 * k, g)[:k, :k])
        one = np.zeros(1, dtype=np.int64)
        size = np.full(1, k, dtype=np.int32)
        return {"pb": PermBatch(B.reshape(-1), one, size, size, r, one, r, one)}
    if kind == "sample":
        order, uni = sampler_draws(case["count"], case["n"], seed + 1)
        return {"U": haar_unitary(case["m"], g), "s": _first_modes(case["m"], case["n"]),
                "order": order, "uniforms": uni}
    if kind == "lossy":
        m, n = case["m"], case["n"]
        return {"V": haar_unitary(m, g), "W": haar_unitary(m, g), "eta": g.uniform(0.5, 0.95, m),
                "s": _first_modes(m, n), "t": _lossy_patterns(m, n)}
    if kind == "hafnian":
        k = case["k"]
        gam = (g.standard_normal(k) + 1j * g.standard_normal(k)) * 0.5
        return {"mats": gbs_matrix(k, g).reshape(-1), "mat_off": np.zeros(1, dtype=np.int64),
                "k": np.full(1, k, dtype=np.int32), "rep": np.full(k, case["r"], dtype=np.int32),
                "rep_off": np.zeros(1, dtype=np.int64), "gamma": gam}
    ks = g.integers(1, case["kmax"] + 1, size=case["count"]).astype(np.int32)
    total = int(ks.sum())
    return {"mats": np.concatenate([gbs_matrix(int(k), g).reshape(-1) for k in ks]),
            "mat_off": _offsets(ks.astype(np.int64) ** 2), "k": ks,
            "rep": g.integers(0, case["rmax"] + 1, size=total).astype(np.int32),
            "rep_off": _offsets(ks),
            "gamma": (g.standard_normal(total) + 1j * g.standard_normal(total)) * 0.5}


def _lossy_patterns(m, n):
    return np.concatenate([compositions(q, m) for q in range(n + 1)])


# --------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------
def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "ragged":
        pb = _ragged(case, seed)
        st["db"] = api.DeviceBatch(pb, "cuda")
        st["plan"] = api.Plan.for_batch(pb)
        st["backward"] = case["backward"]
        if case["backward"]:
            st["mats"] = st["db"].mats.clone().requires_grad_(True)
            st["grad_out"] = _dev(_grad_out(case, seed))
        return st
    h = _host(case, seed)
    if kind == "bs":
        st.update(U=_dev(h["U"]), s=_dev(h["s"]), t=_dev(h["t"]),
                  plan=api.Plan.for_bs(case["m"], h["s"], h["t"]))
    elif kind == "mesh":
        st.update(m=case["m"], theta=_dev(h["theta"]).requires_grad_(True),
                  phi=_dev(h["phi"]).requires_grad_(True), s=_dev(h["s"]), t=_dev(h["t"]),
                  plan=api.Plan.for_bs(case["m"], h["s"], h["t"]))
    elif kind == "power":
        st.update(db=api.DeviceBatch(h["pb"], "cuda"),
                  plan=api.Plan.for_batch(h["pb"], method=case["method"]))
    elif kind == "sample":
        st.update(U=_dev(h["U"]), order=h["order"], uniforms=h["uniforms"],
                  plan=api.SamplerPlan(case["m"], h["s"], case["count"]))
    elif kind == "lossy":
        st.update(V=_dev(h["V"]), eta=_dev(h["eta"]), W=_dev(h["W"]),
                  plan=api.LossyPlan(case["m"], h["s"], h["t"]))
    elif kind == "hafnian":
        st.update(mats=_dev(h["mats"]), gamma=_dev(h["gamma"]) if case["loop"] else None,
                  plan=api.HafnianPlan(h["mat_off"], h["k"], h["rep"], h["rep_off"], case["loop"]))
    else:
        st.update(h, mats=_dev(h["mats"]), gamma=_dev(h["gamma"]) if case["loop"] else None)
    return st


def run(st):
    kind = st["kind"]
    if kind == "bs":
        return api.bs_probs(st["U"], st["s"], st["t"], st["plan"])
    if kind == "mesh":
        U = api.ClementsMesh.apply(st["theta"], st["phi"], st["m"])
        p = api.BSProbs.apply(U, st["s"], st["t"], st["plan"])
        grads = torch.autograd.grad(p.sum(), [st["theta"], st["phi"]])
        return p, *grads
    if kind == "ragged" and st["backward"]:
        per = api.Permanent.apply(st["mats"], st["db"], st["plan"])
        return per, *torch.autograd.grad(per, [st["mats"]], [st["grad_out"]])
    if kind in ("ragged", "power"):
        return api.permanent_batched(st["db"], st["plan"])
    if kind == "sample":
        return st["plan"].run(st["U"], st["order"], st["uniforms"])
    if kind == "lossy":
        return st["plan"].run(st["V"], st["eta"], st["W"])
    if kind == "hafnian":
        return st["plan"].run(st["mats"], st["gamma"])
    return api.hafnian_repeated(st["mats"], st["mat_off"], st["k"], st["rep"], st["rep_off"],
                                gamma=st["gamma"])


# --------------------------------------------------------------------------
# work: sign-vector terms times the operations of one term (FMA = 2)
# --------------------------------------------------------------------------
def _terms(mult):
    m = [int(x) for x in mult if x > 0]
    return math.prod(x + 1 for x in m) // (min(m) + 1) * min(m) if m else 1


def _permanent_flops(r, c, backward=False):
    """Column sums 2l, n - 1 complex products and the accumulation; a gradient
    takes two more products per factor and 8 per column to accumulate."""
    r, c = [int(x) for x in r if x > 0], [int(x) for x in c if x > 0]
    tr, tc = _terms(r), _terms(c)
    l, n = (len(c) if tr <= tc else len(r)), sum(r)
    per = 2 * l + 6 * (n - 1) + 2
    return min(tr, tc) * (per + (12 * (n - 1) + 8 * l if backward else 0))


def _hafnian_flops(rep, loop):
    """A Gray step (8) and, per term, q^(N/2) or the loop polynomial."""
    N = int(sum(rep))
    if N == 0 or (not loop and N % 2):
        return 0
    h = max(1, N // 2)
    mults = (h.bit_length() - 1 + bin(h).count("1") - 1) if not loop else h
    return _terms(rep) * (8 + 6 * mults + 2)


def work(case):
    kind = case["kind"]
    if kind == "ragged":
        pb = _ragged(case, 0, values=False)
        back = case["backward"]
        flops = sum(_permanent_flops(r, c, back) for r, c in
                    zip(np.split(pb.row_mult, pb.row_off[1:]), np.split(pb.col_mult, pb.col_off[1:])))
        return {"bytes": 16 * pb.mats.size * (2 if back else 1) + 16 * pb.batch * (2 if back else 1)
                + 4 * (pb.row_mult.size + pb.col_mult.size), "flops": flops}
    if kind == "power":
        r = [case["r"]] * case["k"]
        return {"bytes": 16 * case["k"] ** 2 + 16, "flops": _permanent_flops(r, r)}
    if kind in ("bs", "mesh"):
        m, n = case["m"], case["n"]
        h = _host(case, 0)
        back = kind == "mesh"
        flops = sum(_permanent_flops(t.tolist(), h["s"].tolist(), back) for t in h["t"])
        if back:
            flops += 2 * 2 * 28 * m * m * (m - 1) // 2
        size = (4 * m * (m - 1) // 2 * 8 + 8 * len(h["t"])) if back else 16 * m * m + 24 * len(h["t"])
        return {"bytes": size + 4 * m * (len(h["t"]) + 1), "flops": flops}
    if kind == "sample":
        m, n, b = case["m"], case["n"], case["count"]
        per = sum(q * _permanent_flops([1] * (q - 1), [1] * (q - 1)) + 8 * m * q
                  for q in range(2, n + 1))
        return {"bytes": 16 * m * m + 12 * b * n + 4 * b * m, "flops": b * per}
    if kind == "lossy":
        m, n = case["m"], case["n"]
        perms = math.comb(2 * m + n - 1, n)
        outs = sum(math.comb(q + m - 1, q) for q in range(n + 1))
        return {"bytes": 32 * m * m + 8 * m + 8 * outs + 4 * m * outs,
                "flops": perms * _permanent_flops([1] * n, [1] * n)}
    h = _host(case, 0)
    loop = case["loop"]
    flops = sum(_hafnian_flops(r, loop) for r in np.split(h["rep"], h["rep_off"][1:]))
    return {"bytes": 16 * h["mats"].size + 4 * h["rep"].size + (16 * h["rep"].size if loop else 0)
            + 16 * h["k"].size, "flops": max(flops, 1)}


# --------------------------------------------------------------------------
# exact values in 64 bits
# --------------------------------------------------------------------------
_LIMIT = 800_000_000  # complex products that numpy does in about 20 seconds


def _levels(mult):
    """The multisets g <= mult, grouped by their size: for level q the digits
    (k x states) and, for every i, the place of g - e_i among level q - 1
    (0 where g_i = 0)."""
    mult = np.asarray(mult, dtype=np.int64)
    rad = mult + 1
    stride = np.cumprod(np.concatenate([[1], rad[:-1]]))
    total = int(np.prod(rad))
    code = np.arange(total)
    size = np.zeros(total, dtype=np.int64)
    for s, q in zip(stride, rad):
        size += code // s % q
    order = np.argsort(size, kind="stable")
    start = np.searchsorted(size[order], np.arange(int(mult.sum()) + 2))
    place = np.empty(total, dtype=np.int64)
    place[order] = code - np.repeat(start[:-1], np.diff(start))
    out = []
    for q in range(int(mult.sum()) + 1):
        idx = order[start[q]:start[q + 1]]
        dig = idx[None, :] // stride[:, None] % rad[:, None]
        prev = np.where(dig > 0, place[np.where(dig > 0, idx[None, :] - stride[:, None], 0)], 0)
        out.append((dig, prev, idx))
    return out, place, stride


def _permanent(B, r, c, levels=None, grad=False):
    """per of B with row i repeated r_i and column j c_j times; with ``grad``
    also d per / d B.  F(g), the permanent of the rows g against the first |g|
    column copies, is expanded along its last column."""
    if len(c) and math.prod(int(x) + 1 for x in c) < math.prod(int(x) + 1 for x in r):
        if not grad:
            return _permanent(B.T, c, r)
        v, G = _permanent(B.T, c, r, grad=True)
        return v, G.T
    levels = levels if levels is not None else _levels(r)[0]
    cols = np.repeat(np.arange(len(c)), c)
    F = [np.ones(1, dtype=np.complex128)]
    for q, j in enumerate(cols):
        dig, prev, _ = levels[q + 1]
        F.append(np.einsum("i,is,is->s", B[:, j], dig, F[q][prev]))
    if not grad:
        return F[-1][0]
    G = np.zeros_like(B)
    lam = np.ones(1, dtype=np.complex128)
    for q in range(len(cols) - 1, -1, -1):
        dig, prev, _ = levels[q + 1]
        w = dig * lam
        G[:, cols[q]] += np.einsum("is,is->i", w, F[q][prev])
        w = w * B[:, cols[q]][:, None]
        lam = (np.bincount(prev.ravel(), w.real.ravel(), F[q].size)
               + 1j * np.bincount(prev.ravel(), w.imag.ravel(), F[q].size))
    return F[-1][0], G


def _states(r, c):
    r, c = [int(x) for x in r if x > 0], [int(x) for x in c if x > 0]
    return min((math.prod(x + 1 for x in v) * len(v) for v in (r, c)), default=1)


def _hafnian(B, rep, gamma):
    """Expansion along the first index present: paired with a copy of itself,
    of another index, or (loops) alone."""
    N = int(sum(rep))
    if gamma is None and N % 2:
        return 0.0
    keep = np.nonzero(rep)[0]
    B, rep = B[np.ix_(keep, keep)], np.asarray(rep)[keep]
    gam = None if gamma is None else gamma[keep]
    if N == 0:
        return 1.0
    levels, place, stride = _levels(rep)
    F = [np.ones(1, dtype=np.complex128)]
    for q in range(1, N + 1):
        dig, _, idx = levels[q]
        i = np.argmax(dig > 0, axis=0)
        v = np.zeros(idx.size, dtype=np.complex128)
        if gam is not None:
            v += gam[i] * F[q - 1][place[idx - stride[i]]]
        if q >= 2:
            left = dig.copy()
            left[i, np.arange(idx.size)] -= 1
            for j in range(len(rep)):
                ok = left[j] > 0
                at = place[np.where(ok, idx - stride[i] - stride[j], 0)]
                v += np.where(ok, left[j] * B[i, j] * F[q - 2][np.where(ok, at, 0)], 0.0)
        F.append(v)
    return F[-1][0]


def _norms(s, t):
    """1 / (prod s! prod t!) of every pattern."""
    fact = np.cumprod(np.concatenate([[1.0], np.arange(1.0, 40.0)]))
    return 1.0 / (fact[t].prod(axis=1) * fact[s].prod())


def _probs(A, s, t):
    """Amplitudes per(A_{s,t}) and probabilities of every pattern, A[out][in]."""
    cols = np.nonzero(s)[0]
    amp = np.empty(len(t), dtype=np.complex128)
    for b, row in enumerate(t):
        rows = np.nonzero(row)[0]
        amp[b] = _permanent(A[np.ix_(rows, cols)], row[rows], s[cols])
    return amp, np.abs(amp) ** 2 * _norms(s, t)


def _mesh(theta, phi, m):
    """U = T_{L-1} ... T_0 of the Clements mesh, differentiable."""
    U = torch.eye(m, dtype=torch.complex128)
    q = 0
    for layer in range(m):
        for j in range(layer % 2, m - 1, 2):
            t = torch.cos(theta[q]).to(torch.complex128)
            r = torch.exp(1j * phi[q]) * torch.sin(theta[q])
            q += 1
            a, b = U[j], U[j + 1]
            U = torch.cat([U[:j], (t * a - r.conj() * b)[None], (r * a + t * b)[None], U[j + 2:]])
    return U


def _exact_mesh(case, seed):
    h = _host(case, seed)
    theta = torch.from_numpy(h["theta"]).requires_grad_(True)
    phi = torch.from_numpy(h["phi"]).requires_grad_(True)
    U = _mesh(theta, phi, case["m"])
    A, s, t = U.detach().numpy(), h["s"], h["t"]
    amp, p = _probs(A, s, t)
    cols, norm = np.nonzero(s)[0], _norms(s, t)
    gU = np.zeros_like(A)
    for b, row in enumerate(t):
        rows = np.nonzero(row)[0]
        _, G = _permanent(A[np.ix_(rows, cols)], row[rows], s[cols], grad=True)
        gU[np.ix_(rows, cols)] += 2.0 * norm[b] * amp[b] * G.conj()
    grads = torch.autograd.grad(U, [theta, phi], torch.from_numpy(gU))
    return p, *grads


def exact(case, seed):
    kind = case["kind"]
    if kind == "sample":
        return None
    if kind == "ragged":
        if case["count"] > 5000:
            return None
        pb = _ragged(case, seed)
        items = [pb.item(b) for b in range(pb.batch)]
        back = case["backward"]
        if sum(_states(r, c) * (3 if back else 1) for _, r, c in items) > _LIMIT:
            return None
        if not back:
            return np.array([_permanent(B, r, c) for B, r, c in items])
        go = _grad_out(case, seed)
        both = [_permanent(B, r, c, grad=True) for B, r, c in items]
        return (np.array([v for v, _ in both]),
                np.concatenate([(w * G.conj()).reshape(-1) for w, (_, G) in zip(go, both)]))
    h = _host(case, seed)
    if kind == "power":
        B, r, c = h["pb"].item(0)
        return np.array([_permanent(B, r, c)]) if _states(r, c) * 4 < _LIMIT else None
    if kind in ("bs", "mesh"):
        if sum(_states(t, h["s"]) for t in h["t"]) * (4 if kind == "mesh" else 1) > _LIMIT:
            return None
        if kind == "mesh":
            return _exact_mesh(case, seed)
        amp, p = _probs(h["U"], h["s"], h["t"])
        return p, amp
    if kind == "lossy":
        m, n, s = case["m"], case["n"], h["s"]
        d = np.concatenate([h["V"] @ (np.sqrt(h["eta"])[:, None] * h["W"]),
                            np.sqrt(1.0 - h["eta"])[:, None] * h["W"]])
        lost = [compositions(q, m) for q in range(n + 1)]
        p = np.zeros(len(h["t"]))
        for b, t in enumerate(h["t"]):
            u = lost[n - int(t.sum())]
            full = np.concatenate([np.broadcast_to(t, (len(u), m)), u], axis=1)
            p[b] = _probs(d, s, full)[1].sum()
        return p
    vals = []
    for b, k in enumerate(h["k"]):
        o, ro = int(h["mat_off"][b]), int(h["rep_off"][b])
        rep = h["rep"][ro:ro + k]
        if math.prod(int(x) + 1 for x in rep) * len(rep) * 8 > _LIMIT:
            return None
        gam = h["gamma"][ro:ro + k] if case["loop"] else None
        vals.append(_hafnian(h["mats"][o:o + k * k].reshape(k, k), rep, gam))
    return np.array(vals)
