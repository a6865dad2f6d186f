"""Performance cases of the sparse spectral library: the calls a user's program
makes, over the sizes and options the library is used at.

Families (``kind``):

  step      Algorithm 1 in one call (lattice, recovery of a and f, stamping set,
            solve) from trigonometric data in device memory to the solution
  recover   recovery of one sum's coefficients on a known candidate set
  identify  recovery without a candidate set (support identification)
  stamp     stamping set, neighbour table and their export
  apply     one application of the stamped Galerkin operator
  solve     one solve on a stamping set that the program keeps
  batch     many uneven systems solved by one call on a batch it keeps
  proxy     Monte Carlo proxy error of a computed solution

``draw`` spreads the same families over their whole ranges.
"""
from math import comb, log2, pi

import numpy as np
import torch

import paper_2302_00752_gb300 as ss


def listed():
    return [
        # The smallest call: a two-dimensional problem on a box lattice of 33^2
        # nodes, |S| of a few hundred.  Launches, read-backs and host work.
        dict(name="step_d2_box", kind="step", d=2, n_cos=4, kmax=4, nnz=0, f_kind="manufactured", pairs=5, f_kmax=6,
             N=2, lattice="box", M_min=33 * 33, solve="fp64"),
        # The ordinary dense-frequency problem: d = 10, forcing of 840 terms from
        # a chosen solution, CBC lattice of 10^6 nodes, |S| = 334,440.
        dict(name="step_d10_cbc", kind="step", d=10, n_cos=10, kmax=8, nnz=0, f_kind="manufactured", pairs=20, f_kmax=8,
             N=3, lattice="cbc", M_min=10**6, solve="fp64"),
        # Multiscale coefficient in three dimensions, prime lattice, mixed
        # precision solve, |S| = 86,272.
        dict(name="step_d3_multiscale", kind="step", d=3, n_cos=9, kmax=1024, nnz=0, f_kind="multiscale", pairs=8,
             f_kmax=1024, N=4, lattice="random", M_min=0, solve="fp32_refined"),
        # The high-dimensional problem, the benchmark's headline: d = 100, lattice
        # of 2^26 nodes, |S| about 1.15 million.  The largest call.
        dict(name="step_d100", kind="step", d=100, n_cos=20, kmax=4, nnz=3, f_kind="pairs", pairs=50, f_kmax=4, N=3,
             lattice="random_smooth", M_min=1 << 26, solve="fp64"),
        # Single-precision recovery of the d = 100 coefficient at the full lattice.
        dict(name="recover_d100_fp32", kind="recover", d=100, n_cos=20, kmax=4, nnz=3, f_kind="pairs", pairs=50,
             f_kmax=4, M_min=1 << 26, precision="fp32"),
        # A forcing of 840 terms whose support is unknown: d + 1 shifted lattices.
        dict(name="identify_d10", kind="identify", d=10, n_cos=10, kmax=8, nnz=0, f_kind="manufactured", pairs=20,
             f_kmax=8, M_min=10**6),
        # A set of about 1e5 frequencies in 30 dimensions, built and exported.
        dict(name="stamp_d30", kind="stamp", d=30, n_cos=15, kmax=8, nnz=0, f_kind="pairs", pairs=10, f_kmax=8, N=3),
        # The operator alone as an outside iteration calls it: double and single.
        dict(name="apply_d10_fp64", kind="apply", d=10, n_cos=10, kmax=8, nnz=0, f_kind="pairs", pairs=20, f_kmax=8, N=4,
             precision="fp64"),
        dict(name="apply_d100_fp32", kind="apply", d=100, n_cos=20, kmax=4, nnz=3, f_kind="pairs", pairs=50, f_kmax=4,
             N=3, precision="fp32"),
        # Another right-hand side on the d = 100 set, mixed precision, to 1e-10.
        dict(name="solve_d100_refined", kind="solve", d=100, n_cos=20, kmax=4, nnz=3, f_kind="pairs", pairs=50, f_kmax=4,
             N=3, precision="fp32_refined", tol=1e-10),
        # 128 uneven systems (d = 6..30, |S| = 1e3..1e5) in one graph-replayed call.
        dict(name="batch_128", kind="batch", n_inst=128, d_lo=6, d_hi=30, s_lo=1000, s_hi=100000,
             precision="fp32_refined"),
        # Monte Carlo proxy at 1000 points on the next stamping level (|S| about
        # 330,000).
        dict(name="proxy_d10", kind="proxy", d=10, n_cos=10, kmax=8, nnz=0, f_kind="pairs", pairs=20, f_kmax=8, N=3,
             points=1000),
    ]


# ------------------------------------------------------------------ ranges


def _count(n_f, n_cos, N):
    """Frequencies reached from n_f points by at most N steps of 2 n_cos +- pairs
    in general position."""
    tot = 0
    for n in range(N + 1):
        for t in range(min(n, n_cos) + 1):
            c = 1 if n == 0 else (comb(n - 1, t - 1) if t >= 1 else 0)
            tot += 2**t * comb(n_cos, t) * c
    return n_f * tot


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _draw_system(rng, s_lo, s_hi, levels=(1, 2, 3, 4)):
    """A problem whose stamping set has a size spread over [s_lo, s_hi]."""
    goal = _log(rng, s_lo, s_hi)
    while True:
        d = rng.choice((2, 3, 4, 5, 7, 10, 17, 30, 64, 100))
        n_cos, pairs, N = rng.randint(1, 20), _log(rng, 1, 50), rng.choice(levels)
        if not goal / 2 <= _count(2 * pairs, n_cos, N) <= min(s_hi, 2 * goal):
            continue
        if d <= 4:
            kmax, nnz = rng.choice((64, 500, 1024)), 0
        elif d <= 30:
            kmax, nnz = rng.randint(5, 12), 0
        else:
            kmax, nnz = rng.randint(3, 5), 3
        return dict(d=d, n_cos=n_cos, kmax=kmax, nnz=nnz, f_kind="pairs", pairs=pairs, f_kmax=kmax, N=N)


def _room(c):
    """A lattice size at which component-by-component search finds a generator soon."""
    return (2 * c["n_cos"] + 1 + 2 * c["pairs"]) ** 2 // 2


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "recover", "identify", "stamp", "apply", "apply", "solve", "batch",
                       "proxy"))
    if kind == "step":
        c = _draw_system(rng, 300, 600000)
        lat = rng.choice(("cbc", "random", "random_smooth"))
        M = max(_log(rng, 2000, 1 << (25 if lat == "random_smooth" else 20)), _room(c))
        return dict(kind=kind, **c, lattice=lat, M_min=M, solve=rng.choice(("fp64", "fp64", "fp32_refined")))
    if kind == "recover":
        c = _draw_system(rng, 300, 600000)
        c.pop("N")
        return dict(kind=kind, **c, M_min=_log(rng, 1 << 17, 1 << 26), precision=rng.choice(("fp64", "fp32")))
    if kind == "identify":
        c = _draw_system(rng, 300, 600000)
        c.pop("N")
        if c["d"] > 10:
            c.update(d=rng.randint(5, 10), kmax=8, f_kmax=8, nnz=0)
        return dict(kind=kind, **c, M_min=max(_log(rng, 5000, 10**6), _room(c)))
    if kind == "stamp":
        return dict(kind=kind, **_draw_system(rng, 300, 800000))
    if kind == "apply":
        return dict(kind=kind, **_draw_system(rng, 300, 1150000), precision=rng.choice(("fp64", "fp32")))
    if kind == "solve":
        p = rng.choice(("fp64", "fp32_refined"))
        return dict(kind=kind, **_draw_system(rng, 300, 1150000), precision=p, tol=1e-12 if p == "fp64" else 1e-10)
    if kind == "batch":
        n = _log(rng, 3, 128)
        return dict(kind=kind, n_inst=n, d_lo=rng.randint(3, 8), d_hi=rng.randint(9, 30), s_lo=rng.randint(300, 1500),
                    s_hi=_log(rng, 5000, 100000), precision=rng.choice(("fp64", "fp32_refined")))
    c = _draw_system(rng, 100, 20000, (1, 2))
    big = _count(2 * c["pairs"], c["n_cos"], c["N"] + 1)
    return dict(kind=kind, **c, points=min(_log(rng, 50, 2000), max(1, 300_000_000 // big)))


# ------------------------------------------------------------------ data


def _freqs(g, n, d, kmax, nnz, taken):
    """n distinct vectors, no two of them +-: uniform in [-kmax, kmax]^d, or nnz
    nonzero coordinates each."""
    out = []
    while len(out) < n:
        if nnz:
            v = np.zeros(d, np.int64)
            v[g.choice(d, size=min(nnz, d), replace=False)] = g.integers(1, kmax + 1, min(nnz, d)) * g.choice([-1, 1], min(nnz, d))
        else:
            v = g.integers(-kmax, kmax + 1, d)
        k = tuple(v.tolist())
        if not any(k) or k in taken or tuple((-v).tolist()) in taken:
            continue
        taken.add(k)
        out.append(v)
    return np.array(out, np.int64).reshape(n, d)


def _shape(c):
    """Generator of the frequencies' shape, one for all seeds of a case, so that
    every seed's stamping set has the same size: the seeds turn it by a
    coordinate permutation and sign flips (``_turn``) and draw the values."""
    return np.random.default_rng([c["d"], c["n_cos"], c["pairs"], c["kmax"], c["f_kmax"], c.get("member", 0)])


def _turn(g, d):
    perm, sign = g.permutation(d), g.choice([-1, 1], d)
    return lambda k: k[:, perm] * sign


def _a_data(g, c, fix, turn):
    """1 + n_cos cosines with sum |c| = 0.5: sum (freq, coef) and its Fourier
    coefficients (freq, val), both +- halves."""
    d, n = c["d"], c["n_cos"]
    p = _freqs(fix, n, d, c["kmax"], c["nnz"], set())
    w = g.uniform(-1, 1, n)
    w *= 0.5 / np.abs(w).sum()
    if c["f_kind"] == "multiscale":  # one axis cosine at each scale, the others at the largest
        p[0], p[1], p[2] = [1, 0, 0], [0, 64, 0], [0, 0, 1024]
        w[3:] *= 0.25 / np.abs(w[3:]).sum()
        w[:3] = [0.25, 0.15, 0.10]
    p = turn(p)
    zero = np.zeros((1, d), np.int64)
    return ((np.vstack([zero, p]), np.concatenate([[1.0], w]).astype(complex)),
            (np.vstack([zero, p, -p]), np.concatenate([[1.0], w / 2, w / 2]).astype(complex)))


def _f_data(g, c, fix, turn, a_hat):
    """The forcing, likewise."""
    d, n = c["d"], c["pairs"]
    if c["f_kind"] == "multiscale":
        taken = set()
        q = np.vstack([_freqs(fix, 1, d, (1, 64, 1024)[j % 3], 0, taken) for j in range(n)])
    else:
        q = _freqs(fix, n, d, c["f_kmax"], c["nnz"], set())
    q = turn(q)
    if c["f_kind"] == "manufactured":  # f = L u for a chosen u
        u = g.standard_normal(n) + 1j * g.standard_normal(n)
        acc = {}
        for l, ul in zip(np.vstack([q, -q]), np.concatenate([u, u.conj()])):
            for p, ap in zip(*a_hat):
                k = l + p
                dot = int(k @ l)
                if dot and k.any():
                    key = tuple(k.tolist())
                    acc[key] = acc.get(key, 0) + 4 * pi**2 * dot * ap * ul
        top = max(abs(v) for v in acc.values())
        acc = {k: v for k, v in acc.items() if abs(v) > 1e-6 * top}
        f_hat = np.array(list(acc), np.int64), np.array(list(acc.values()))
        return f_hat, f_hat
    amp = g.uniform(0.1, 1, n) * g.choice([-1, 1], n)
    coef = np.where(g.integers(0, 2, n) == 1, -1j * amp, amp + 0j)
    return (q, coef), (np.vstack([q, -q]), np.concatenate([coef, coef.conj()]) / 2)


def _data(c, seed):
    g, fix = np.random.default_rng([seed, 11]), _shape(c)
    turn = _turn(g, c["d"])
    a, a_hat = _a_data(g, c, fix, turn)
    f, f_hat = _f_data(g, c, fix, turn, a_hat)
    return a, a_hat, f, f_hat, g


def _cand(a_hat, f_hat):
    return np.unique(np.vstack([a_hat[0], -a_hat[0], f_hat[0], -f_hat[0]]), axis=0)


def _i32(x):
    return torch.as_tensor(np.asarray(x, np.int32)).cuda()


def _c128(x):
    return torch.as_tensor(np.asarray(x, np.complex128)).cuda()


def _lattice(c, g):
    d = c["d"]
    if c["lattice"] == "box":
        side = 33
        return {"kind": "box", "z": np.array([side**j for j in range(d)], np.int64), "M": side**d}
    if c["lattice"] == "cbc":
        return {"kind": "cbc", "raw": g.integers(0, 2**62, size=(d, 64)), "M_min": c["M_min"]}
    return {"kind": "random", "raw": g.integers(0, 2**62, size=(8, d)), "M_min": c["M_min"], "sigma": 0.05,
            "smooth": c["lattice"] == "random_smooth"}


def _batch_members(c):
    """The uneven systems of a batch: odd s_a in 5..41, 5..30 f pairs, N in 2..3,
    sizes within [s_lo, s_hi]."""
    g = np.random.default_rng([c["n_inst"], c["s_lo"], c["s_hi"], 12])
    got = []
    while len(got) < c["n_inst"]:
        n_cos, pairs, N = int(g.integers(2, 21)), int(g.integers(5, 31)), int(g.integers(2, 4))
        if c["s_lo"] <= _count(2 * pairs, n_cos, N) <= c["s_hi"]:
            got.append(dict(d=int(g.integers(c["d_lo"], c["d_hi"] + 1)), n_cos=n_cos, kmax=8, nnz=0, f_kind="pairs",
                            pairs=pairs, f_kmax=8, N=N, member=len(got)))
    return got


def _system(c, seed, N):
    """Stamping set and right-hand side that a program keeps."""
    _, a_hat, _, f_hat, g = _data(c, seed)
    stamp = ss.stamp_build(_i32(a_hat[0]), _c128(a_hat[1]), _i32(f_hat[0]), N)
    f_on, _ = stamp.scatter(_i32(f_hat[0]), _c128(f_hat[1]))
    return stamp, f_on, g


def _vector(n, seed, dtype):
    r = torch.Generator(device="cuda").manual_seed(seed)
    return torch.complex(torch.randn(n, generator=r, device="cuda", dtype=torch.float64),
                         torch.randn(n, generator=r, device="cuda", dtype=torch.float64)).to(dtype)


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c}
    if kind == "batch":
        st["stamps"], st["f"] = [], []
        for i, m in enumerate(_batch_members(c)):
            stamp, f_on, _ = _system(m, 1000 * seed + i, m["N"])
            st["stamps"].append(stamp)
            st["f"].append(f_on)
        st["batch"] = ss.Batch(st["stamps"])
        st["u"] = [torch.empty_like(f) for f in st["f"]]
        return st
    if kind in ("apply", "solve", "proxy"):
        st["stamp"], st["f"], g = _system(c, seed, c["N"])
        if kind == "apply":
            st["u"] = _vector(st["stamp"].size, seed, torch.complex128 if c["precision"] == "fp64" else torch.complex64)
        elif kind == "proxy":
            st["u"], _ = ss.solve(st["stamp"], st["f"], 1e-14, 1000, "fp64")
            st["stamp"].extend(1)
            f = _data(c, seed)[2]
            st["f_freq"], st["f_coef"] = _i32(f[0]), _c128(f[1])
            st["X"] = g.integers(0, 1 << 32, size=(c["points"], c["d"]), dtype=np.uint64).astype(np.uint32)
        return st
    a, a_hat, f, f_hat, g = _data(c, seed)
    if kind == "stamp":
        st["a_freq"], st["a_val"], st["f_freq"] = _i32(a_hat[0]), _c128(a_hat[1]), _i32(f_hat[0])
        return st
    cand = _cand(f_hat if kind == "identify" else a_hat, f_hat)
    if kind == "step":
        if c["lattice"] == "box":  # every frequency of the box
            r = np.arange(-16, 17)
            cand = np.stack(np.meshgrid(*[r] * c["d"], indexing="ij"), -1).reshape(-1, c["d"])
        st["lattice"] = _lattice(c, g)
        st["a_freq"], st["a_coef"], st["f_freq"], st["f_coef"] = _i32(a[0]), _c128(a[1]), _i32(f[0]), _c128(f[1])
        st["cand"] = _i32(cand)
        return st
    # recover: the sum a on the candidates of a and f; identify: the sum f
    h = a if kind == "recover" else f
    st["freq"], st["coef"], st["cand"] = _i32(h[0]), _c128(h[1]), _i32(cand)
    if kind == "recover":
        st["z"], st["M"], _ = ss.lattice_random(st["cand"], g.integers(0, 2**62, size=(16, c["d"])), 0.05, c["M_min"],
                                                smooth=True)
    else:
        st["z"], st["M"] = ss.lattice_cbc(st["cand"], g.integers(0, 2**62, size=(c["d"], 64)), c["M_min"])
        P = 2 * int(np.abs(cand).max()) + 2
        while any(P % q == 0 for q in range(2, int(P**0.5) + 1)):
            P += 1
        st["P"], st["s_max"] = P, 2 * len(f_hat[0]) + 2
    return st


# ------------------------------------------------------------------ the pass


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "step":
        stamp, u, _, z, M = ss.sparse_spectral_solve(st["lattice"], st["a_freq"], st["a_coef"], st["f_freq"],
                                                     st["f_coef"], st["cand"], c["N"], solve_precision=c["solve"])
        size, nnz = stamp.size, stamp.nnz
        stamp.destroy()
        return {"u": u, "z": z, "M": M, "size": size, "nnz": nnz}
    if kind == "recover":
        tau = 1e-9 if c["precision"] == "fp64" else 1e-4
        freq, val = ss.sft_recover(st["z"], st["M"], st["freq"], st["coef"], st["cand"], tau=tau, precision=c["precision"])
        return {"freq": freq, "val": val}
    if kind == "identify":
        freq, val = ss.sft_identify(st["z"], st["M"], st["freq"], st["coef"], st["P"], st["s_max"])
        return {"freq": freq, "val": val}
    if kind == "stamp":
        stamp = ss.stamp_build(st["a_freq"], st["a_val"], st["f_freq"], c["N"])
        freq, level = stamp.export()
        nnz = stamp.nnz
        stamp.destroy()
        return {"freq": freq, "level": level, "nnz": nnz}
    if kind == "apply":
        return {"y": ss.galerkin_apply(st["stamp"], st["u"])}
    if kind == "solve":
        return {"u": ss.solve(st["stamp"], st["f"], c["tol"], 1000, c["precision"])[0]}
    if kind == "batch":
        us, _ = st["batch"].solve(st["f"], st["u"], 1e-12, 1000, c["precision"], use_graph=True)
        return {"u": torch.cat(us)}
    r, f = ss.proxy_mc(st["stamp"], st["u"], st["f_freq"], st["f_coef"], st["X"])
    return {"r": r, "f": f}


# ------------------------------------------------------------------ unavoidable work


def _size(c, N=None):
    n_f = 2 * c["pairs"] * (2 * c["n_cos"] + 1 if c["f_kind"] == "manufactured" else 1)
    n = _count(2 * c["pairs"], c["n_cos"], (c["N"] if N is None else N) + (c["f_kind"] == "manufactured"))
    if c["d"] <= 2:
        n = min(n, (2 * ((N or c["N"]) * c["kmax"] + c["kmax"] + c["f_kmax"]) + 1) ** 2)
    return n, n_f


def _nnz(c, N):
    """Every row on a level below the last has all its neighbours; the others lead
    back.  Counted from both ends of each pair."""
    full = _size(c, N - 1)[0] if N else 0
    return min((2 * c["n_cos"] + 1) * _size(c, N)[0], _size(c, N)[0] + 4 * c["n_cos"] * full)


def _fft(M):
    return 5.0 * M * log2(max(M, 2))


ITERS = 14  # CG iterations to 1e-12 at the data's contrast (sum |c| = 0.5)


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        rows = sum(_size(m)[0] for m in _batch_members(c))
        return {"bytes": 32 * rows, "flops": ITERS * 8 * 6 * rows}
    d = c["d"]
    if kind in ("recover", "identify"):
        n_f = 2 * c["pairs"] * (2 * c["n_cos"] + 1 if c["f_kind"] == "manufactured" else 1)
        M = max(c["M_min"], 20 * (n_f + 2 * c["n_cos"] + 1) ** 2 if kind == "recover" else 0)
        n = 2 * c["n_cos"] + 1 + n_f
        # one length-M transform of the samples, d + 1 of them without candidates
        return {"bytes": (4 * d + 16) * 2 * n, "flops": _fft(M) * (d + 1 if kind == "identify" else 1)}
    size, n_f = _size(c)
    nnz = _nnz(c, c["N"])
    if kind == "step":
        M = max(c["M_min"], 20 * (n_f + 2 * c["n_cos"] + 1) ** 2 if c["lattice"].startswith("random") else 0)
        return {"bytes": (4 * d + 16) * 2 * n_f + 16 * size, "flops": 2 * _fft(M) + ITERS * 8 * nnz}
    if kind == "stamp":
        return {"bytes": 4 * d * n_f + (4 * d + 1) * size + 4 * nnz, "flops": 0}
    if kind == "apply":
        w = 16 if c["precision"] == "fp64" else 8
        return {"bytes": 2 * w * size + 4 * nnz, "flops": 8 * nnz}
    if kind == "solve":
        return {"bytes": 32 * size + 4 * nnz, "flops": ITERS * 8 * nnz}
    big = _size(c, c["N"] + 1)[0]
    return {"bytes": (4 * d + 16) * big + 4 * d * c["points"], "flops": (2.0 * d + 30) * big * c["points"]}


# ------------------------------------------------------------------ the same in 64 bits


class _Set:
    """S^N in canonical order and the operator on it, in plain torch: frequencies
    are compared by a 64-bit linear form with random weights."""

    def __init__(self, a_hat, f_freq, N):
        d = f_freq.shape[1]
        g = np.random.default_rng(99)
        w = torch.as_tensor(g.integers(-(1 << 62), 1 << 62, d) | 1).cuda()

        def form(k):
            out = torch.zeros(k.shape[0], dtype=torch.int64, device="cuda")
            for j in range(d):
                out += k[:, j] * w[j]
            return out

        lex = np.lexsort(a_hat[0].T[::-1])
        p, self.ap = torch.as_tensor(a_hat[0][lex]).cuda(), torch.as_tensor(a_hat[1][lex]).cuda()
        steps = p[(p != 0).any(1)]
        hs = form(steps)
        freq = [torch.as_tensor(np.unique(f_freq, axis=0)).cuda()]
        h = [form(freq[0])]
        for _ in range(N):
            cand = (h[-1][:, None] + hs[None, :]).reshape(-1)
            val, at = torch.sort(cand, stable=True)
            first = torch.ones_like(val, dtype=torch.bool)
            first[1:] = val[1:] != val[:-1]
            first &= ~torch.isin(val, torch.cat(h))
            at = torch.sort(at[first])[0]
            freq.append(freq[-1][at // len(hs)] + steps[at % len(hs)])
            h.append(cand[at])
        self.k, self.p, self.sizes = torch.cat(freq), p, [len(x) for x in h]
        self.n, h = len(self.k), torch.cat(h)
        order = torch.argsort(h)
        hp, hk = form(p), h[order]
        kd = self.k.double()
        k2 = (kd * kd).sum(1)
        self.rows = []
        for j in range(len(p)):
            want = h - hp[j]
            at = torch.searchsorted(hk, want).clamp_(max=self.n - 1)
            row = torch.nonzero(hk[at] == want).reshape(-1)
            dot = k2[row] - kd[row] @ p[j].double()
            self.rows.append((row, order[at[row]], 4 * pi**2 * dot * self.ap[j]))
        self.diag = 4 * pi**2 * k2 * self.ap[(p == 0).all(1)].real
        self.zero = k2 == 0

    def find(self, freq):
        at = {}
        ks = torch.as_tensor(freq).cuda()
        for s in range(0, len(ks), 64):
            hit = (self.k[: self.sizes[0], None, :] == ks[None, s : s + 64]).all(2).nonzero()
            at.update((int(j) + s, int(i)) for i, j in hit)
        return torch.tensor([at[i] for i in range(len(ks))], device="cuda")

    def apply(self, u):
        y = torch.zeros(self.n, dtype=torch.complex128, device="cuda")
        for row, col, coef in self.rows:
            y[row] += coef * u[col]
        return torch.where(self.zero, u, y)

    def rhs(self, f_hat):
        f = torch.zeros(self.n, dtype=torch.complex128, device="cuda")
        f[self.find(f_hat[0])] = torch.as_tensor(f_hat[1]).cuda()
        return f

    def solve(self, f):
        inv = torch.where(self.zero, 1.0, 1.0 / torch.where(self.zero, 1.0, self.diag))
        u, r = torch.zeros_like(f), f.clone()
        z = inv * r
        p, rz, stop = z.clone(), torch.vdot(r, z).real, 1e-31 * torch.vdot(f, f).real
        for _ in range(200):
            q = self.apply(p)
            alpha = rz / torch.vdot(p, q).real
            u += alpha * p
            r -= alpha * q
            if torch.vdot(r, r).real <= stop:
                break
            z = inv * r
            new = torch.vdot(r, z).real
            p = z + (new / rz) * p
            rz = new
        return u


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "stamp":
        return None  # whole numbers
    if kind == "batch":
        us = []
        for i, m in enumerate(_batch_members(c)):
            _, a_hat, _, f_hat, _ = _data(m, 1000 * seed + i)
            s = _Set(a_hat, f_hat[0], m["N"])
            us.append(s.solve(s.rhs(f_hat)))
        return {"u": torch.cat(us)}
    a, a_hat, f, f_hat, g = _data(c, seed)
    if kind == "step":
        s = _Set(a_hat, f_hat[0], c["N"])
        return {"u": s.solve(s.rhs(f_hat)), "z": None, "M": None, "size": None, "nnz": None}
    if kind == "recover":  # kept coefficients in candidate order
        at = {tuple(k): v for k, v in zip(a_hat[0].tolist(), a_hat[1])}
        tau = 1e-9 if c["precision"] == "fp64" else 1e-4
        top = max(abs(v) for v in at.values())
        val = [at[k] for k in map(tuple, _cand(a_hat, f_hat).tolist()) if k in at and abs(at[k]) > tau * top]
        return {"freq": None, "val": np.array(val)}
    if kind == "identify":  # increasing bin, each k (bin at most M / 2) before -k
        st = prepare(case, seed)
        z, M = st["z"], st["M"]
        res = (f_hat[0] @ z.astype(object)) % M
        half = sorted((int(b), v) for b, v in zip(res, f_hat[1]) if 2 * int(b) <= M)
        return {"freq": None, "val": np.array([x for _, v in half for x in (v, np.conj(v))])}
    s = _Set(a_hat, f_hat[0], c["N"])
    if kind == "apply":
        return {"y": s.apply(_vector(s.n, seed, torch.complex128 if c["precision"] == "fp64" else torch.complex64).to(torch.complex128))}
    u = s.solve(s.rhs(f_hat))
    if kind == "solve":
        return {"u": u}
    X = torch.as_tensor(g.integers(0, 1 << 32, size=(c["points"], c["d"]), dtype=np.uint64).astype(np.float64)).cuda()
    t = _Set(a_hat, f_hat[0], c["N"] + 1)
    y = t.apply(torch.cat([u, u.new_zeros(t.n - s.n)]))
    y[t.zero] = 0

    def at_points(k, v):  # sum_k v_k exp(2 pi i k.x), phases reduced exactly
        out = torch.zeros(len(X), dtype=torch.complex128, device="cuda")
        step = max(1, 20_000_000 // len(X))
        for i in range(0, len(k), step):
            ph = torch.remainder(k[i : i + step].double() @ X.T, 2.0**32) * (2 * pi / 2.0**32)
            out += (v[i : i + step, None] * torch.polar(torch.ones_like(ph), ph)).sum(0)
        return out.real

    fx = at_points(torch.as_tensor(f_hat[0]).cuda(), torch.as_tensor(f_hat[1]).cuda())
    return {"r": fx - at_points(t.k, y), "f": fx}
