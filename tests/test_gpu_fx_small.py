"""Small coefficients beside large ones, and long sums, through the fixed-point
transform of the FP64 recovery: what a bin loses is a unit (2^-58 of the sum's
l1 norm) averaged over a column or a row of the four-step split, not a unit of
the whole sum.

Tolerance: the inverse transform's columns and the forward transform's leave
about half a unit of rounding in each part of their values, white over the L1
and L2 values that a bin averages; both lie within a factor 3 of M^(1/2), so
2^-57 l1 / M^(1/4) covers their sum; and a value rounds at 2^-53.  The few
coefficients whose row or column also holds a large one carry a unit of that, so
the median speaks for spread magnitudes; for equal ones a row holds about n / L1
<= 3 n / M^(1/2) of the l1 norm's n parts, and the root mean square does."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


def recovered(B, M, n, spread):
    rng = np.random.default_rng([M, n])
    k = rng.choice(np.arange(1, (M - 1) // 2), n, replace=False)[:, None]
    c = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    if spread:
        c *= 10.0 ** (-9 * rng.random(n)) / np.abs(c)
    cand = np.vstack([k, -k])
    f, v = B.sft_recover([1], M, k, c, cand, tau=0.0)
    assert np.array_equal(f.cpu().numpy(), cand)
    want = np.concatenate([c, np.conj(c)]) / 2
    return np.abs(v.cpu().numpy() - want), want, np.abs(c).sum()


@pytest.mark.parametrize("M,n", [(10**5, 420), (823543, 420), (10**6, 420), (10**6, 2000), (3**13, 420), (2**22, 420),
                                 (4134375, 2000)])
def test_spread_magnitudes(B, M, n):
    err, want, l1 = recovered(B, M, n, True)
    assert np.median(err / (2.0**-53 * np.abs(want) + 2.0**-57 * l1 / M**0.25)) <= 1.0


@pytest.mark.parametrize("M,n", [(17496, 2000), (10**5, 2000), (10**6, 2000), (823543, 20000), (2**22, 20000)])
def test_long_sums(B, M, n):
    err, want, l1 = recovered(B, M, n, False)
    row = 3.0 * l1 / M**0.5
    assert np.sqrt(np.mean(err**2)) <= (2.0**-53 * np.sqrt(np.mean(np.abs(want) ** 2))
                                        + 2.0**-57 * (l1 / M**0.25 + row))


@pytest.mark.parametrize("M", [10**4, 10**6])
def test_nothing_outside_a_constant(B, M):
    """Every other bin of a constant is exactly zero: not kept at any threshold."""
    cand = np.arange(-200, 201)[:, None]
    f, v = B.sft_recover([1], M, np.zeros((1, 1), int), np.array([1.5 + 0j]), cand, tau=0.0)
    assert f.cpu().numpy().tolist() == [[0]]
    assert v.cpu().numpy().tolist() == [1.5]
