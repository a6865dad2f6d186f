"""Recovery on short lattices that are not 7-smooth (samples and bins by direct
FP64 sums) and on 7-smooth ones, with the merging of repeated and mirrored
terms at the edges of its one-block form.

Tolerance: a sample adds at most ceil(T / 16) + 16 products, a bin
ceil(M / 128) + 9, each step rounding at 2^-53 of sum |c|; roots and
coefficients are rounded at 2^-53 (the fixed-point transform stays below the
same bound, see its own test)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2302_00752_gb300 import binding
    return binding


@pytest.mark.parametrize("M,d,pairs,extra,n_terms", [
    (11, 1, 2, 0, 3), (97, 2, 5, 10, 1), (1089, 2, 40, 500, 33), (1994, 3, 20, 100, 512), (3329, 3, 18, 0, 1023),
    (3329, 40, 18, 30, 1024), (32749, 3, 30, 30, 1025), (32749, 7, 64, 0, 100), (1000, 3, 20, 100, 1024),
    (10**4, 100, 30, 10, 60), (20011, 5, 60, 2000, 200)])
def test_recover_direct_and_merge(B, M, d, pairs, extra, n_terms):
    rng = np.random.default_rng([M, d, n_terms])
    # candidates +-k with distinct residues, and zero
    z = rng.integers(1, M, d)
    z[0] = 1
    half, seen = [], {0}
    while len(half) < min(pairs + extra, (M - 1) // 2 - 1):
        k = rng.integers(-20, 21, d)
        k[0] += int(rng.integers(-M // 2, M // 2)) if d < 40 else 0
        r = int(k @ z % M)
        if r in seen or 2 * r == M:
            continue
        seen |= {r, M - r}
        half.append(k)
    half = np.array(half)
    cand = rng.permutation(np.vstack([half, -half, np.zeros((1, d), int)]))
    # terms: support frequencies with either sign, repeated, and zero
    pick = rng.integers(0, min(pairs, len(half)) + 1, n_terms)
    pick[: min(3, n_terms)] = 0
    sup = np.vstack([half, np.zeros((1, d), int)])
    pick[pick == min(pairs, len(half))] = len(half)
    sg = rng.choice([-1, 1], n_terms)
    p = sup[pick] * sg[:, None]
    c = rng.standard_normal(n_terms) + 1j * rng.standard_normal(n_terms)
    want = np.zeros(len(sup), complex)
    np.add.at(want, pick, np.where(sg > 0, c, np.conj(c)))
    val = {tuple(np.zeros(d, int)): want[-1].real}
    for k, v in zip(half, want[:-1]):
        val[tuple(k)], val[tuple(-k)] = v / 2, np.conj(v) / 2
    tol = 2.0**-53 * (-(-n_terms // 16) + -(-M // 128) + 29) * np.abs(c).sum()
    f, v = B.sft_recover(z, M, p, c, cand, tau=1e-10)
    f, v = f.cpu().numpy(), v.cpu().numpy()
    big = 1e-10 * max(abs(x) for x in val.values())
    assert np.array_equal(f, [k for k in cand.tolist() if abs(val[tuple(k)]) > big])
    got = {tuple(k): x for k, x in zip(f.tolist(), v)}
    assert all(abs(x - val[k]) <= tol for k, x in got.items())
    assert all(got[tuple(-i for i in k)] == np.conj(x) for k, x in got.items())
