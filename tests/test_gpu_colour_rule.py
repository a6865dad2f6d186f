"""Where the solver colours: a set in general position takes about half of plain
CG's iterations; a set of few dimensions, whose rows of one colour mostly touch
each other, runs plain CG, as does one whose masks are dropped in a batch beside
coloured ones.

Which of the two follows from the set: of two neighbours in one of the levels N,
N - 2, ... at least one turns red, so the rows lost are at least a matching of
such pairs and at most the rows in them, and the colours go when the rows lost
are more than a quarter.

Counts: the stopping test is the same, so plain CG in another order of rounding
differs by at most one iteration; the Schur complement's spectrum 1 - mu^2 needs
at most (n + 3) / 2 + 1 of the n iterations that 1 +- mu does."""
import numpy as np
import pytest

from oracle import galerkin as ogal
from oracle import solve as osolve
from oracle import stamp as ostamp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


def system(B, d, kmax, n_cos, pairs, N):
    g = np.random.default_rng([d, kmax, n_cos, pairs, N])

    def freqs(n):
        out = {}
        while len(out) < n:
            v = tuple(g.integers(-kmax, kmax + 1, d).tolist())
            if any(v) and tuple(-x for x in v) not in out:
                out[v] = 1
        return np.array(list(out))

    p, q = freqs(n_cos), freqs(pairs)
    w = g.uniform(0.2, 1, n_cos)
    w *= 0.25 / w.sum()
    amp = g.uniform(0.1, 1, pairs) * np.exp(2j * np.pi * g.random(pairs))
    af, av = np.vstack([np.zeros((1, d), int), p, -p]), np.concatenate([[1.0], w, w]).astype(complex)
    F, fv = np.vstack([q, -q]), np.concatenate([amp, amp.conj()])
    S, level = ostamp.stamp_bfs(af, F, N)
    L = ogal.galerkin_matrix(S, af, av)[0].tocoo()
    level = np.where(np.any(S != 0, axis=1), np.asarray(level), -1)
    cand = (level >= 0) & ((N - level) % 2 == 0)
    pairs_ = [(i, j) for i, j in zip(L.row, L.col) if i < j and cand[i] and level[i] == level[j]]
    used, matched = set(), 0
    for i, j in pairs_:
        if i not in used and j not in used:
            used |= {i, j}
            matched += 1
    kind = None
    if 4 * len({i for e in pairs_ for i in e}) <= cand.sum():
        kind = "coloured"
    elif 4 * matched > cand.sum():
        kind = "plain"
    L = L.tocsr()
    stamp = B.stamp_build(af, av, F, N)
    f, _ = stamp.scatter(F, fv)
    return stamp, f, osolve.pcg(L, f.cpu().numpy(), osolve.jacobi_diag(S, 1.0), tol=1e-12)[1], kind


def check(it, plain, kind):
    if kind == "plain":
        assert abs(it - plain) <= 1
    else:
        assert it <= ((plain + 3) / 2 + 1 if kind == "coloured" else plain + 1)


LOW = [(2, 6, 4, 5, 2), (1, 40, 5, 5, 3), (2, 8, 8, 6, 3)]
GENERAL = [(8, 6, 4, 5, 2), (6, 8, 3, 4, 3)]


def test_both_sides_are_met(B):
    kinds = [system(B, *s)[3] for s in LOW + GENERAL]
    assert "plain" in kinds and "coloured" in kinds


@pytest.mark.parametrize("shape", LOW + GENERAL)
@pytest.mark.parametrize("half", [True, False])
def test_one(B, shape, half):
    stamp, f, plain, kind = system(B, *shape)
    stamp.set_symmetry(half)
    for block in (512, 1024):
        stamp.set_solve_config(block, 1, 1)
        check(B.solve(stamp, f, 1e-12, 1000, "fp64")[1]["inner_iters"], plain, kind)
    stamp.destroy()


@pytest.mark.parametrize("shapes", [LOW, LOW + GENERAL])
@pytest.mark.parametrize("half", [True, False])
def test_batch(B, shapes, half):
    sys = [system(B, *s) for s in shapes]
    b = B.Batch([s[0] for s in sys])
    b.set_symmetry(half)
    _, st = b.solve([s[1] for s in sys], None, 1e-12, 1000, "fp64")
    for (_, _, plain, kind), s in zip(sys, st):
        check(s["inner_iters"], plain, kind)
