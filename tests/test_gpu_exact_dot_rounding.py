"""Rounding of the exact dot where one warp resolves the accumulator (at most
28 digits of 32 bits between its lowest and highest nonzero word, as nearly
every dot of a setup has) and at the switch to the walk over more digits:
ties broken far below, borrows and carries through long runs of equal digits,
cancellation to a small remainder, subnormal results.  Every value is the
exact rational sum rounded once; the tolerance is zero."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    G.lib()


def check(terms, rng):
    """terms: pairs (x, y).  Summed by one block, by several blocks, by the
    form without allocation, and with every sign changed."""
    exact = float(sum((Fraction(x) * Fraction(y) for x, y in terms), Fraction(0)))
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    for n in (len(terms), max(5000, len(terms))):
        at = rng.permutation(n)[:len(terms)]
        x, y = np.zeros(n), np.zeros(n)
        x[at], y[at] = [t[0] for t in terms], [t[1] for t in terms]
        for sign in (1.0, -1.0):
            dx, dy = torch.tensor(sign * x, device="cuda"), torch.tensor(y, device="cuda")
            G.airg_dot_exact_noalloc(dx, dy, out)
            got = G.airg_dot_exact(dx, dy), out.item()
            assert got == (sign * exact, sign * exact), (n, sign, got, exact)


def product(e):
    """Factors of 2^e, both normal."""
    return 2.0 ** (e // 2), 2.0 ** (e - e // 2)


# the digit that 2^e falls in changes with e mod 32
@pytest.mark.parametrize("shift", [0, 1, 15, 16, 31])
@pytest.mark.parametrize("gap", [2, 60, 200, 500, 640, 672, 704, 736, 768, 800, 832, 864, 896, 928, 960, 1000])
def test_far_terms(shift, gap):
    """2^e plus or minus half a unit in its last place, plus or minus a term
    `gap` bits below: the last one alone decides the rounding."""
    rng = np.random.default_rng(gap + shift)
    e = 490 - shift
    one, half, ulp = product(e), product(e - 53), product(e - 52)

    def neg(t):
        return -t[0], t[1]

    for low in (product(e - 53 - gap), neg(product(e - 53 - gap))):
        check([one, low], rng)
        for tie in (half, neg(half)):
            check([one, tie, low], rng)
            check([one, ulp, tie, low], rng)       # ties to even the other way
        check([one, neg(one), low], rng)           # all but the last cancels


@pytest.mark.parametrize("n", [3, 32, 33, 500, 1900, 4097])
@pytest.mark.parametrize("spread", [0, 20, 100])
def test_cancellation(n, spread):
    """Random products and their negatives, exponents within `spread` of 0,
    with one small term left over or none."""
    rng = np.random.default_rng(n + spread)
    x = rng.standard_normal(n) * np.exp2(rng.integers(-spread, spread + 1, n).astype(float))
    y = rng.standard_normal(n) * np.exp2(rng.integers(-spread, spread + 1, n).astype(float))
    pairs = list(zip(x, y)) + list(zip(-x, y))
    check(list(zip(x, y)), rng)
    check(pairs, rng)
    for e in (-60, -250, -300):
        check(pairs + [product(e)], rng)
        check(pairs + [(-product(e)[0], product(e)[1]), (2.0 ** 30, 2.0 ** -40)], rng)


def test_subnormal_results():
    """Sums around the smallest subnormals: the last kept bit is 2^-1074."""
    rng = np.random.default_rng(5)
    least, tie, below = product(-1074), product(-1075), product(-1200)
    minus = (-below[0], below[1])
    for terms in ([least], [tie], [tie, below], [tie, minus], [least, tie], [least, tie, minus], [least, tie, below],
                  [product(-1022), (-tie[0], tie[1])], [product(-1022), (-tie[0], tie[1]), minus], [below]):
        check(terms, rng)
