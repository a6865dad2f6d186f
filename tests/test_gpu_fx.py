"""The fixed-point transforms of the FP64 recovery: every radix, in place and
with two buffers, one and two columns a block, against the closed form of a
trigonometric sum; and the identification that runs two rows per transform,
with an even and an odd number of rows.

Tolerance: a unit is 2^-58 of a scale that is at most twice below sum |c|, a
coefficient collects about one unit of noise (products and divisions round at
half a unit, and noise from before the last pass averages), and its double is
rounded at 2^-53 relative: 2^-53 + 2^-56 of sum |c| in modulus, doubled."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2.0 * (2.0**-53 + 2.0**-56)


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


def problem(B, M, d, n, kmax, seed):
    """n +-pairs with residues +-k.z distinct on a lattice of M nodes."""
    rng = np.random.default_rng([M, d, seed])
    p = np.unique(rng.integers(-kmax, kmax + 1, size=(4 * n, d)), axis=0)
    p = p[p.any(axis=1)]
    p = np.array([v for v in p.tolist() if tuple(v) > tuple(-x for x in v)])
    p = rng.permutation(p)[:n]
    full = np.vstack([p, -p])
    for _ in range(200):
        z = rng.integers(1, M, d)
        if len(np.unique((full @ z) % M)) == len(full) and not np.any((2 * (full @ z)) % M == 0):
            break
    else:
        raise AssertionError("no lattice found")
    c = rng.standard_normal(len(p)) + 1j * rng.standard_normal(len(p))
    return z, p, c, full


@pytest.mark.parametrize("M", [10, 14, 81, 250, 1000, 2 * 3**7, 4 * 7**4, 10**4, 3 * 5**5, 2**13, 8 * 2187, 10**6,
                               2**20 * 3, 2**22])
def test_recover_closed_form(B, M):
    n = 2 if M < 100 else 5 if M < 10**4 else 12
    z, p, c, full = problem(B, M, 3, n, 3 if M < 100 else 40, 1)
    f, v = B.sft_recover(z, M, p, c, full, tau=0.0)
    want = np.concatenate([c, np.conj(c)]) / 2
    assert np.array_equal(f.cpu().numpy(), full)
    assert np.abs(v.cpu().numpy() - want).max() <= TOL * np.abs(c).sum()


@pytest.mark.parametrize("M,d", [(10**4, 2), (10**5, 3), (5**5 * 16, 4), (2**17, 1), (3**9, 5)])
def test_identify_pairs(B, M, d):
    z, p, c, full = problem(B, M, d, 6, 15, 2)
    f, v = B.sft_identify(z, M, p, c, 37, 64)
    res = (full @ z) % M
    val = np.concatenate([c, np.conj(c)]) / 2
    order = [i for b, i in sorted((int(b), i) for i, b in enumerate(res) if 2 * b < M)]
    want_f = np.vstack([full[i] * s for i in order for s in (1, -1)])
    want_v = np.array([x for i in order for x in (val[i], np.conj(val[i]))])
    assert np.array_equal(f.cpu().numpy(), want_f)
    assert np.abs(v.cpu().numpy() - want_v).max() <= TOL * np.abs(c).sum()


@pytest.mark.parametrize("bad", [None, np.nan, np.inf])
def test_every_candidate_and_nonfinite(B, bad):
    """A zero threshold keeps every candidate of a nonzero sum, also bins that
    round to nothing; a sum with a coefficient that is not finite keeps none."""
    M, z = 10**4, np.array([1, 10, 100])
    cand = np.array([[i, j, k] for i in range(-3, 4) for j in range(-3, 4) for k in range(-3, 4)], np.int32)
    p = cand[[200, 250, 300, 310]]
    c = np.array([0.3 - 1j, 0.7 + 0.1j, -0.2 + 0.9j, 1.3 + 0.4j])
    if bad is not None:
        c[1] = bad
    f, v = B.sft_recover(z, M, p, c, cand, tau=0.0)
    assert len(f) == (len(cand) if bad is None else 0)
