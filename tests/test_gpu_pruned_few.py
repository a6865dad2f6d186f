"""The FP64 recovery on long lattices whose splits have no kernel of their own,
around the number of bins up to which lanes share a bin's columns (256 bins: 64
pairs of candidates), with a last tile that is not whole, and radix 3.

Tolerance: a block adds up its tiles (at most 32 of them at these lengths) and
the blocks are added in 15 + 5 steps, each rounding at 2^-53 of at most sum |c|;
the transform's own rounding stays below 2^-52 of it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [3 * 2**21, 7**8, 3**14, 2**4 * 3**3 * 5**6])
@pytest.mark.parametrize("n", [1, 2, 5, 33, 64, 65])
def test_bins_around_the_shared_columns(M, n):
    from paper_2302_00752_gb300 import binding as B
    rng = np.random.default_rng([M, n])
    k = rng.choice(np.arange(1, (M - 1) // 2), n, replace=False)[:, None]
    c = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    cand = np.vstack([k, -k])
    f, v = B.sft_recover([1], M, k, c, cand, tau=0.0)
    assert np.array_equal(f.cpu().numpy(), cand)
    want = np.concatenate([c, np.conj(c)]) / 2
    assert np.abs(v.cpu().numpy() - want).max() <= (32 + 20 + 2) * 2.0**-53 * np.abs(c).sum()
