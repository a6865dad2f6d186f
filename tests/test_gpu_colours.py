"""The two-colour solver (CG on the Schur complement of the red rows) against a
dense solve, over the sets that it takes and the ones it must leave alone: no
levels, one level, an odd and an even number, more levels than it colours, few
dimensions (rows of one colour that are neighbours of each other), the zero
frequency reached, forcing with and without symmetry, full and half system,
every mode, small and large blocks.

Tolerance: CG stops at ||f - L u|| <= tol ||f||; the error is at most cond(L)
times that in relative terms, and the residual formed here adds its own rounding."""
import numpy as np
import pytest
import torch

from oracle import galerkin as ogal
from oracle import stamp as ostamp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


def system(d, N, sym, cplx):
    rng = np.random.default_rng([d, N, sym, cplx])
    p = rng.integers(-3, 4, size=(3, d))
    p = p[p.any(axis=1)]
    p = np.unique([v if tuple(v) > tuple(-v) else -v for v in p], axis=0)
    c = rng.standard_normal(len(p)) + (1j * rng.standard_normal(len(p)) if cplx else 0.0)
    c = 0.9 * c / (2 * np.abs(c).sum())
    af = np.vstack([np.zeros((1, d), int), p, -p])
    av = np.concatenate([[1.0 + 0j], c, np.conj(c)])
    F = rng.integers(-4, 5, size=(3, d))
    F = np.unique([v if tuple(v) > tuple(-v) else -v for v in F[F.any(axis=1)]], axis=0)
    fv = rng.standard_normal(len(F)) + 1j * rng.standard_normal(len(F))
    if sym:
        F, fv = np.vstack([F, -F]), np.concatenate([fv, np.conj(fv)])
    S, _ = ostamp.stamp_bfs(af, F, N)
    return af, av, F, fv, S, ogal.galerkin_matrix(S, af, av)[0]


@pytest.mark.parametrize("d,N,sym", [(1, 1, True), (1, 17, True), (2, 0, True), (2, 1, False), (2, 2, True), (2, 5, True),
                                     (3, 3, True), (3, 4, False), (4, 4, True)])
@pytest.mark.parametrize("cplx", [False, True])
def test_two_colours(B, d, N, sym, cplx):
    af, av, F, fv, S, L = system(d, N, sym, cplx)
    L = L.toarray() if hasattr(L, "toarray") else np.asarray(L)
    cond = np.linalg.cond(L)
    with B.stamp_build(af, av, F, N) as s:
        f_on, _ = s.scatter(F, fv)
        f = f_on.cpu().numpy()
        assert np.array_equal(s.export()[0].cpu().numpy(), S)
        ref = np.linalg.solve(L, f)
        for half in (True, False):
            s.set_symmetry(half)
            for block in (0, 1024):
                if block:
                    s.set_solve_config(block, 1, 1)
                for prec, tol in (("fp64", 1e-12), ("fp32", 1e-11), ("df64", 1e-11)):
                    u, st = B.solve(s, f_on, tol, 2000, prec)
                    u = u.cpu().numpy()
                    assert st["rel_residual"] <= tol
                    assert np.linalg.norm(f - L @ u) <= (tol + 1e-13) * 1.01 * np.linalg.norm(f)
                    assert np.linalg.norm(u - ref) <= (tol + 1e-13) * cond * np.linalg.norm(ref)
            s.set_solve_config(512, 1, 1)


def test_batch_mixes_coloured_and_not(B):
    sys_ = [system(2, 0, True, False), system(3, 3, True, False), system(1, 17, True, False), system(4, 4, True, True)]
    stamps, fs, refs = [], [], []
    for (af, av, F, fv, S, L), N in zip(sys_, (0, 3, 17, 4)):
        s = B.stamp_build(af, av, F, N)
        f_on, _ = s.scatter(F, fv)
        stamps.append(s)
        fs.append(f_on)
        L = L.toarray() if hasattr(L, "toarray") else np.asarray(L)
        refs.append((L, f_on.cpu().numpy()))
    for prec, tol in (("fp64", 1e-12), ("fp32", 1e-11)):
        us, st = B.Batch(stamps).solve(fs, None, tol, 2000, prec)
        for u, (L, f) in zip(us, refs):
            assert np.linalg.norm(f - L @ u.cpu().numpy()) <= (tol + 1e-13) * 1.01 * np.linalg.norm(f)
    for s in stamps:
        s.destroy()


@pytest.mark.parametrize("s_a", [57, 59, 129])
def test_fill_at_the_step_count_limits(B, s_a):
    # the entry fill by row bit masks takes up to 57 steps, the other one any number
    rng = np.random.default_rng(s_a)
    d, n = 6, (s_a - 1) // 2
    p = np.unique(rng.integers(-3, 4, size=(8 * n, d)), axis=0)
    p = np.array([v for v in p if tuple(v) > tuple(-v)])[:n]
    c = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    c = 0.9 * c / (2 * np.abs(c).sum())
    af, av = np.vstack([np.zeros((1, d), int), p, -p]), np.concatenate([[1.0 + 0j], c, np.conj(c)])
    F = np.array([[1, 0, 2, 0, -1, 0], [-1, 0, -2, 0, 1, 0]])
    S, _ = ostamp.stamp_bfs(af, F, 2)
    L, nnz = ogal.galerkin_matrix(S, af, av)
    u = rng.standard_normal(len(S)) + 1j * rng.standard_normal(len(S))
    with B.stamp_build(af, av, F, 2) as s:
        assert s.nnz == nnz
        y = B.galerkin_apply(s, torch.as_tensor(u).cuda()).cpu().numpy()
        f_on, _ = s.scatter(F, np.array([1 + 1j, 1 - 1j]))
        w, st = B.solve(s, f_on, 1e-12, 1000, "fp64")
    # a row sums at most s_a terms, each rounded three times
    assert np.linalg.norm(y - L @ u) <= s_a * 2.0**-51 * np.linalg.norm(L @ u)
    assert np.linalg.norm(f_on.cpu().numpy() - L @ w.cpu().numpy()) <= 1.2e-12 * np.linalg.norm(f_on.cpu().numpy())
