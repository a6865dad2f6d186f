"""Small coefficients beside large ones in the FP64 identification, on both sides
of its rule for the number of terms.

Tolerance: an FP64 transform of length M rounds at 2^-53 in each of its about
log2(M) steps, so a bin carries 2^-53 log2(M)^(1/2) M^(-1/2) of the sum's l2 norm
beside its own rounding at 2^-53.  The identification is to be no less exact,
whichever transform it takes: the median error of coefficients over nine decades
stays within that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


@pytest.mark.parametrize("M,n,d", [(10**5, 60, 5), (823543, 420, 3), (10**6, 420, 3), (2**22, 500, 3), (2**22, 2000, 4)])
def test_spread_magnitudes(B, M, n, d):
    rng = np.random.default_rng([M, n, d])
    p = np.unique(rng.integers(-8, 9, size=(4 * n, d)), axis=0)
    p = np.array([v for v in p.tolist() if tuple(v) > tuple(-x for x in v)])
    p, z = rng.permutation(p)[:n], rng.integers(1, M, d)
    keep, seen = [], set()
    for i, k in enumerate(p):
        a = int(k @ z % M)
        if a not in seen and 2 * a % M:
            keep.append(i)
        seen |= {a, M - a}
    p = p[keep]
    c = np.exp(2j * np.pi * rng.random(len(p))) * 10.0 ** (-8.5 * rng.random(len(p)))
    f, v = B.sft_identify(z, M, p, c, 19, 2 * len(p) + 2)
    want = {tuple(k): x for k, x in zip(np.vstack([p, -p]).tolist(), np.concatenate([c, np.conj(c)]) / 2)}
    got = [tuple(k) for k in f.cpu().numpy().tolist()]
    assert len(got) == len(want) and set(got) == set(want)
    want = np.array([want[k] for k in got])
    tol = 2.0**-53 * (np.abs(want) + np.sqrt(np.log2(M) / M) * np.linalg.norm(want))
    assert np.median(np.abs(v.cpu().numpy() - want) / tol) <= 1.0
