"""The residual that the solvers report is ||f - L u|| / ||f|| over all rows, the
rows of the colour that the solver eliminates included.

Tolerance: at the level of rounding two evaluations of one residual differ by
their own rounding, which is of its size: a factor 2 either way; above it, by
rounding alone."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


def system(B, d, n_cos, pairs, N, seed):
    g = np.random.default_rng([d, n_cos, pairs, N, seed])

    def freqs(n):
        out, taken = [], set()
        while len(out) < n:
            v = tuple(g.integers(-8, 9, d).tolist())
            if any(v) and v not in taken and tuple(-x for x in v) not in taken:
                taken.add(v)
                out.append(v)
        return np.array(out)

    p, q = freqs(n_cos), freqs(pairs)
    w = g.uniform(-1, 1, n_cos)
    w *= 0.25 / np.abs(w).sum()
    amp = g.uniform(0.1, 1, pairs) * np.exp(2j * np.pi * g.random(pairs))
    stamp = B.stamp_build(np.vstack([np.zeros((1, d), int), p, -p]), np.concatenate([[1.0], w, w]).astype(complex),
                          np.vstack([q, -q]), N)
    return stamp, stamp.scatter(np.vstack([q, -q]), np.concatenate([amp, amp.conj()]))[0]


def check(B, stamp, f, u, reported):
    true = float((f - B.galerkin_apply(stamp, u)).norm() / f.norm())
    assert true / 2 <= reported <= 2 * true + 2.0**-53


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-14), ("df64", 1e-14), ("fp32_refined", 1e-14), ("fp64", 1e-9)])
@pytest.mark.parametrize("half", [True, False])
@pytest.mark.parametrize("block", [512, 1024])
@pytest.mark.parametrize("d,n_cos,pairs,N", [(17, 40, 5, 2), (3, 6, 5, 1), (2, 5, 6, 4)])
def test_one(B, d, n_cos, pairs, N, block, half, precision, tol):
    stamp, f = system(B, d, n_cos, pairs, N, 0)
    stamp.set_symmetry(half)
    stamp.set_solve_config(block, 1, 1)
    u, st = B.solve(stamp, f, tol, 1000, precision, raise_on_error=False)
    check(B, stamp, f, u, st["rel_residual"])
    if stamp.size < 32000 and precision != "df64" and block == 512:
        u = torch.empty_like(f)
        _, st = B.solve_noalloc(stamp, f, u, tol, 1000, precision)
        check(B, stamp, f, u, st["rel_residual"])
    stamp.destroy()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-14), ("fp32_refined", 1e-12)])
@pytest.mark.parametrize("half", [True, False])
def test_batch(B, half, precision, tol):
    sys = [system(B, 3 + i, 2 + 3 * i, 5 + i, 1 + i % 3, i) for i in range(6)]
    b = B.Batch([s for s, _ in sys])
    b.set_symmetry(half)
    us, sts = b.solve([f for _, f in sys], None, tol, 1000, precision)
    for (stamp, f), u, st in zip(sys, us, sts):
        check(B, stamp, f, u, st["rel_residual"])
