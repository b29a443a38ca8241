"""Performance cases: the calls that users of this library make.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (a context or a server, the matrices, the multiplicities),
``run`` is one pass through the package's public entry points, ``work`` the
bytes and flops that a pass cannot do without, ``exact`` the outputs in twice
double precision where they are computed numbers and small enough.

Ranges: permanents and Laplace minors of 8 to 30 photons, batches of 16 to
4096 permanents, sampling of 8 to 30 photons in up to 60 modes (ideal and
lossy), 4 to 64 served chains; modes FP64 (0), MIXED (1) and double-float (2).
"""
import math

import numpy as np
import torch

import paper_2309_07027_gb300 as bs

FP64, MIXED, DF64 = bs.BS_FP64, bs.BS_MIXED, bs.BS_DF64


def listed():
    return [
        # one 12-photon permanent with collisions (24-mode unitary, 8 occupied
        # output modes, 576 addends): the smallest call, all latency
        {"name": "perm_12", "kind": "perm", "mults": "3,2,2,1,1,1,1,1", "cols": 12, "m": 24, "mode": FP64},
        # its Laplace minors: one step of a small sampler written by the caller
        {"name": "minors_12", "kind": "minors", "mults": "3,2,2,1,1,1,1", "cols": 12, "m": 24, "mode": FP64},
        # the probability amplitude of one collision-free 23-photon event, odd
        # width, 2^22 addends: an ordinary call
        {"name": "perm_23", "kind": "perm", "mults": ",".join(["1"] * 23), "cols": 23, "m": 60, "mode": FP64},
        # a 30 x 30 permanent, 2^29 addends: the large accurate call
        {"name": "perm_30", "kind": "perm", "mults": ",".join(["1"] * 30), "cols": 30, "m": 60, "mode": FP64},
        # minors of a late sampling step with bunched photons (27 columns)
        {"name": "minors_27_bunched", "kind": "minors", "mults": "3,2,2,2,2" + ",1" * 15, "cols": 27, "m": 60,
         "mode": FP64},
        # the same kind of step in the fast mode: 25 x 26 minors, 2^24 addends
        {"name": "minors_26_mixed", "kind": "minors", "mults": ",".join(["1"] * 25), "cols": 26, "m": 60,
         "mode": MIXED},
        # a small batch of small permanents from host memory (a validation loop)
        {"name": "batch_64", "kind": "batch", "count": 64, "kmin": 10, "kmax": 16, "m": 60, "pattern": 7,
         "mode": FP64},
        # 4096 uneven permanents of 10 to 28 photons kept on the device
        {"name": "batch_4096_mixed", "kind": "batch_dev", "count": 4096, "kmin": 10, "kmax": 28, "m": 60,
         "pattern": 2, "mode": MIXED},
        # 30-photon sampling in 60 modes, accurate mode, a short run
        {"name": "sample_30", "kind": "sample", "n": 30, "m": 60, "eta": 1.0, "samples": 40, "mode": FP64},
        # the same experiment in the fast mode on device tensors, 200 samples
        {"name": "sample_30_mixed", "kind": "sample_dev", "n": 30, "m": 60, "eta": 1.0, "samples": 200,
         "mode": MIXED},
        # lossy sampling (half of the photons lost, one loss mode per photon)
        {"name": "lossy_26_df", "kind": "sample", "n": 26, "m": 60, "eta": 0.5, "samples": 25, "mode": DF64},
        # 48 sampling requests of mixed size answered by one server
        {"name": "serve_48", "kind": "serve", "chains": 48, "nmin": 16, "nmax": 26, "m": 60, "pattern": 4,
         "mode": FP64},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bunched(rng, photons, modes):
    """Photons thrown uniformly into the modes: the occupied modes' counts."""
    counts = {}
    for _ in range(photons):
        i = rng.randrange(modes)
        counts[i] = counts.get(i, 0) + 1
    return ",".join(str(c) for c in counts.values())


def draw(rng):
    kind = rng.choice(["perm", "perm", "minors", "minors", "batch", "batch_dev", "sample", "sample_dev", "serve"])
    mode = rng.choice([FP64, FP64, MIXED, DF64])
    m = rng.randint(40, 60)
    if kind == "perm":
        k = rng.randint(8, 29)
        mults = _bunched(rng, k, m) if rng.random() < 0.5 else ",".join(["1"] * k)
        return {"kind": kind, "mults": mults, "cols": k, "m": m, "mode": mode}
    if kind == "minors":
        k = rng.randint(8, 28)
        mults = _bunched(rng, k - 1, m) if rng.random() < 0.5 else ",".join(["1"] * (k - 1))
        return {"kind": kind, "mults": mults, "cols": k, "m": m, "mode": mode}
    if kind in ("batch", "batch_dev"):
        count = _log_uniform(rng, 16, 2048)
        kmax = rng.randint(11, 20 if mode == FP64 else 24)
        return {"kind": kind, "count": count, "kmin": rng.randint(8, 10), "kmax": kmax, "m": m,
                "pattern": rng.randrange(1 << 20), "mode": mode}
    if kind in ("sample", "sample_dev"):
        n = rng.randint(8, 26)
        return {"kind": kind, "n": n, "m": m, "eta": rng.choice([1.0, 1.0, 0.5, 0.8]),
                "samples": _log_uniform(rng, 8, 300 if n <= 20 else 40), "mode": mode}
    nmin = rng.randint(8, 16)
    return {"kind": "serve", "chains": _log_uniform(rng, 4, 64), "nmin": nmin, "nmax": rng.randint(nmin + 2, 24),
            "m": m, "pattern": rng.randrange(1 << 20), "mode": mode}


# ---------------------------------------------------------------- inputs
def _haar(g, m):
    """Haar-random unitary: QR of a Ginibre matrix, phases of R moved to Q."""
    z = (g.standard_normal((m, m)) + 1j * g.standard_normal((m, m))) / math.sqrt(2.0)
    q, r = np.linalg.qr(z)
    d = np.diagonal(r)
    return q * (d / np.abs(d))


def _mults(case):
    return np.array([int(x) for x in case["mults"].split(",")], dtype=np.int32)


def _one_matrix(case, seed):
    """Rows and columns of one Haar unitary: random output and input modes."""
    g = np.random.Generator(np.random.PCG64(seed))
    u = _haar(g, case["m"])
    rows = g.permutation(case["m"])[:len(_mults(case))]
    cols = g.permutation(case["m"])[:case["cols"]]
    return np.ascontiguousarray(u[np.ix_(rows, cols)])


def _batch_shapes(case):
    """(photons, row multiplicities) of every item; fixed by the case."""
    p = np.random.Generator(np.random.PCG64(case["pattern"]))
    out = []
    for _ in range(case["count"]):
        k = int(p.integers(case["kmin"], case["kmax"] + 1))
        hits = p.integers(0, case["m"], size=k)
        out.append((k, np.unique(hits, return_counts=True)[1].astype(np.int32)))
    return out


def _batch_items(case, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    items, u = [], None
    for t, (k, mult) in enumerate(_batch_shapes(case)):
        if t % 64 == 0:
            u = _haar(g, case["m"])
        rows = g.permutation(case["m"])[:len(mult)]
        cols = g.permutation(case["m"])[:k]
        items.append((np.ascontiguousarray(u[np.ix_(rows, cols)]), mult, np.ones(k, dtype=np.int32)))
    return items


def _interferometer(case, seed):
    """(matrix, occupation, counted rows): the unitary itself, or with loss
    the (m + n) x n isometry with one loss mode per photon."""
    g = np.random.Generator(np.random.PCG64(seed))
    u = _haar(g, case["m"])
    n, eta = case["n"], case["eta"]
    if eta >= 1.0:
        occ = np.zeros(case["m"], dtype=np.int32)
        occ[:n] = 1
        return np.ascontiguousarray(u), occ, case["m"]
    v = np.vstack([math.sqrt(eta) * u[:, :n], math.sqrt(1.0 - eta) * np.eye(n)])
    return np.ascontiguousarray(v), np.ones(n, dtype=np.int32), case["m"]


def _chain_sizes(case):
    p = np.random.Generator(np.random.PCG64(case["pattern"]))
    return [int(x) for x in p.integers(case["nmin"], case["nmax"] + 1, size=case["chains"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        g = np.random.Generator(np.random.PCG64(seed))
        reqs = []
        for n in _chain_sizes(case):
            occ = np.zeros(case["m"], dtype=np.int32)
            occ[:n] = 1
            reqs.append((np.ascontiguousarray(_haar(g, case["m"])), occ, int(g.integers(1 << 30))))
        server = bs.Server(0, mem_budget_bytes=4 << 30, max_active=64, mode=case["mode"])
        return {"case": case, "server": server, "requests": reqs}
    state = {"case": case, "ctx": bs.Context(0)}
    if kind in ("perm", "minors"):
        state["a"] = _one_matrix(case, seed)
        state["rows"] = _mults(case)
        state["cols"] = np.ones(case["cols"], dtype=np.int32)
    elif kind == "batch":
        state["items"] = _batch_items(case, seed)
    elif kind == "batch_dev":
        state["packed"] = state["ctx"].pack_batch(_batch_items(case, seed))
        state["src"] = torch.from_numpy(state["packed"][0]).cuda()
        state["out"] = torch.zeros(case["count"], dtype=torch.complex128, device="cuda")
        state["ctx"].set_stream(torch.cuda.current_stream())
    else:
        state["u"], state["occ"], state["mdet"] = _interferometer(case, seed)
        state["seed"] = int(seed) & 0x7FFFFFFF
        if kind == "sample_dev":
            state["u"] = torch.from_numpy(state["u"]).cuda()
            state["out"] = torch.zeros((case["samples"], state["mdet"]), dtype=torch.int32, device="cuda")
            state["ctx"].set_stream(torch.cuda.current_stream())
    return state


def run(state):
    case = state["case"]
    kind, mode = case["kind"], case["mode"]
    if kind == "perm":
        return np.array(state["ctx"].perm(state["a"], state["rows"], state["cols"], mode=mode))
    if kind == "minors":
        return state["ctx"].laplace_minors(state["a"], state["rows"], state["cols"], mode=mode)
    if kind == "batch":
        return state["ctx"].perm_batch(state["items"], mode=mode)
    if kind == "batch_dev":
        state["ctx"].perm_batch_dev(state["src"], *state["packed"][1:], mode, state["out"])
        return state["out"]
    if kind == "sample":
        return state["ctx"].sample_ex(state["u"], state["occ"], case["samples"], state["seed"],
                                      m_detected=state["mdet"], mode=mode)
    if kind == "sample_dev":
        state["ctx"].sample_dev(state["u"], state["occ"], case["samples"], state["seed"], state["out"],
                                m_detected=state["mdet"], mode=mode)
        return state["out"]
    server = state["server"]
    tickets = [server.submit_sample(u, occ, s) for u, occ, s in state["requests"]]
    return [server.wait_sample(t)[0] for t in tickets]


# ---------------------------------------------------------------- work
def _addends(mults):
    """Addends of the BB/FG sum over rows of these multiplicities: one copy of
    a least repeated row stays fixed."""
    c = 1
    for x in mults:
        c *= int(x) + 1
    p = int(min(mults))
    return c // (p + 1) * p


def _perm_flops(k):
    return 8 * k - 2        # column update 2k, product 6 (k - 1), weighted sum 4


def _minors_flops(k):
    return 22 * k - 22      # update 2k, suffix and prefix products, k sums


def _sample_flops(n, m):
    """One Clifford & Clifford sample: the minors of every step, over the mean
    number of addends of k - 1 photons thrown into m modes."""
    total = 0.0
    for k in range(2, n + 1):
        j = k - 1
        mean = math.exp(math.lgamma(2 * m + j) - math.lgamma(2 * m) - math.lgamma(m + j) + math.lgamma(m))
        total += 0.5 * mean * _minors_flops(k)
    return total


def work(case):
    kind = case["kind"]
    if kind == "perm":
        k, mults = case["cols"], _mults(case)
        return {"bytes": 16 * (len(mults) * k + 1), "flops": _addends(mults) * _perm_flops(k)}
    if kind == "minors":
        k, mults = case["cols"], _mults(case)
        return {"bytes": 16 * (len(mults) * k + k), "flops": _addends(mults) * _minors_flops(k)}
    if kind in ("batch", "batch_dev"):
        shapes = _batch_shapes(case)
        return {"bytes": 16 * sum(k * len(mult) + 1 for k, mult in shapes),
                "flops": sum(_addends(mult) * _perm_flops(k) for k, mult in shapes)}
    if kind in ("sample", "sample_dev"):
        n, m = case["n"], case["m"]
        rows, cols = (m, m) if case["eta"] >= 1.0 else (m + n, n)
        return {"bytes": 16 * rows * cols + 4 * case["samples"] * m, "flops": case["samples"] * _sample_flops(n, rows)}
    m = case["m"]
    sizes = _chain_sizes(case)
    return {"bytes": len(sizes) * (16 * m * m + 4 * m), "flops": sum(_sample_flops(n, m) for n in sizes)}


# ---------------------------------------------------------------- exact values
# Complex numbers in twice double precision: (re, im), each a pair (high, low)
# of doubles, over plain torch tensors (TwoSum and Dekker's TwoProduct).
def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _split(a):
    t = a * 134217729.0
    h = t - (t - a)
    return h, a - h


def _add(x, y):
    s, e = _two_sum(x[0], y[0])
    h = s + (e + (x[1] + y[1]))
    return h, (e + (x[1] + y[1])) - (h - s)


def _mul(x, y):
    p = x[0] * y[0]
    ah, al = _split(x[0])
    bh, bl = _split(y[0])
    e = ((ah * bh - p) + ah * bl + al * bh) + al * bl
    e = e + (x[0] * y[1] + x[1] * y[0])
    h = p + e
    return h, e - (h - p)


def _neg(x):
    return -x[0], -x[1]


def _cadd(x, y):
    return _add(x[0], y[0]), _add(x[1], y[1])


def _cmul(x, y):
    return (_add(_mul(x[0], y[0]), _neg(_mul(x[1], y[1]))), _add(_mul(x[0], y[1]), _mul(x[1], y[0])))


def _sum(x):
    """Pairwise sum of a tensor pair over its only axis."""
    h, l = x
    while h.numel() > 1:
        if h.numel() & 1:
            h, l = torch.cat([h, h.new_zeros(1)]), torch.cat([l, l.new_zeros(1)])
        h, l = _add((h[0::2], l[0::2]), (h[1::2], l[1::2]))
    return h[0].item(), l[0].item()


def _scale(x, w):
    return _mul(x[0], w), _mul(x[1], w)


def _glynn(a, mults, minors):
    """2^(1-n) sum over the sign counts of the rows (the first copy of a least
    repeated row fixed) of sign * binomials * product of column sums: the
    permanent, or for each column the permanent without it."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    k = a.shape[1]
    n = int(mults.sum())
    pin = int(np.argmin(mults))
    digits = [(r, int(mults[r]) - (1 if r == pin else 0)) for r in range(len(mults))]
    digits = [d for d in digits if d[1] > 0]
    total = 1
    for _, c in digits:
        total *= c + 1
    acc = [[0, 0] for _ in range(k if minors else 1)]   # exact integers over 2^200
    step = 1 << 19
    for at in range(0, total, step):
        q = torch.arange(at, min(at + step, total), dtype=torch.int64, device=dev)
        zero = torch.zeros(q.shape, dtype=torch.float64, device=dev)
        coef = {pin: zero + 1.0}
        weight = (zero + 1.0, zero)
        for r, c in digits:
            d = q % (c + 1)
            q = torch.div(q, c + 1, rounding_mode="floor")
            coef[r] = coef.get(r, zero) + (c - 2 * d).to(torch.float64)
            tab = torch.tensor([(-1.0) ** i * math.comb(c, i) for i in range(c + 1)], dtype=torch.float64, device=dev)
            weight = _mul(weight, (tab[d], zero))
        sums = []
        for j in range(k):
            c = ((zero, zero), (zero, zero))
            for r, x in coef.items():
                c = _cadd(c, (_mul((x, zero), (zero + a[r, j].real, zero)), _mul((x, zero), (zero + a[r, j].imag, zero))))
            sums.append(c)
        if minors:
            suffix = [None] * k
            run_ = _scale(((zero + 1.0, zero), (zero, zero)), weight)
            for j in range(k - 1, -1, -1):
                suffix[j] = run_
                run_ = _cmul(run_, sums[j])
            prefix = ((zero + 1.0, zero), (zero, zero))
            terms = []
            for j in range(k):
                terms.append(_cmul(prefix, suffix[j]))
                suffix[j] = None
                if j + 1 < k:
                    prefix = _cmul(prefix, sums[j])
        else:
            p = _scale(sums[0], weight)
            for j in range(1, k):
                p = _cmul(p, sums[j])
            terms = [p]
        for l, t in enumerate(terms):
            for part in (0, 1):
                for v in _sum(t[part]):
                    num, den = v.as_integer_ratio()
                    acc[l][part] += (num << 200) // den
    scale = 1 << (200 + n - 1)
    return np.array([complex(x[0] / scale, x[1] / scale) for x in acc])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("perm", "minors"):
        mults = _mults(case)
        if _addends(mults) * case["cols"] * (3 if kind == "minors" else 1) > 6 << 28:
            return None
        out = _glynn(_one_matrix(case, seed), mults, kind == "minors")
        return out if kind == "minors" else out[0].reshape(())
    if kind in ("batch", "batch_dev"):
        shapes = _batch_shapes(case)
        if case["count"] > 256 or sum(_addends(mult) * k for k, mult in shapes) > 1 << 27:
            return None
        out = np.array([_glynn(a, mult, False)[0] for a, mult, _ in _batch_items(case, seed)])
        return out
    return None     # occupation counts: whole numbers, drawn by the library's own random stream
