"""The bound on the error of a Cholesky panel's update (kPanelErr, nk_api.cu), from
which the full-rank proof of the SVD solvers takes its margin: the sliced product of 64
columns, in exact integers as the kernel rounds, cuts and drops it (k_ozaki_gemm, kWide),
on the entries that err the most (digits of 255, many bits below the scale) and on random
ones."""
import os
import re
from fractions import Fraction

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_10526_gb300", "csrc",
                   "nk_api.cu")


def _digits(x, e):
    """The 7 base-256 digits of |x| 2^(56 - e) to nearest, first the leading one."""
    y = int(abs(x) * Fraction(2) ** (56 - e) + Fraction(1, 2))
    return [(y >> (8 * (6 - t))) & 255 for t in range(7)], (1 if x >= 0 else -1)


def _error(a, b):
    """|product as computed - exact product| in units of 2^-53 max|a| max|b|."""
    ea, eb = (int(np.frexp(float(max(abs(v) for v in r)))[1]) for r in (a, b))
    got = Fraction(0)
    for x, y in zip(a, b):
        (dx, sx), (dy, sy) = _digits(x, ea), _digits(y, eb)
        v = sum(dx[s] * dy[t] << (8 * (14 - s - t - 2)) for s in range(7) for t in range(7) if s + t + 2 <= 9)
        got += Fraction(sx * sy * v, 1 << 112) * Fraction(2) ** (ea + eb)
    exact = sum(x * y for x, y in zip(a, b))
    window = Fraction(2) ** (ea + eb - 56)  # the recombined value, to nearest
    got = int(got / window + Fraction(1, 2) * (1 if got >= 0 else -1)) * window
    return float(abs(got - exact) / (max(map(abs, a)) * max(map(abs, b))) * 2 ** 53)


def test_the_bound_covers_a_panel():
    bound = float(re.search(r"kPanelErr = ([0-9.]+)", open(SRC).read()).group(1))
    # leading digits 128 (the scale is twice the entry), all others 255; 53 bits each
    worst = Fraction((1 << 52) + (1 << 45) - 1, 1 << 53)
    # eight bits lower, with bits just below half of the last place held
    small = Fraction((1 << 53) - 1 - (1 << 4), 1 << 61)
    g = np.random.default_rng(1)
    cases = [([worst] * 64, [worst] * 64), ([worst] + [small] * 63, [worst] * 64),
             ([worst] + [small] * 63, [worst] + [small] * 63)]
    for _ in range(20):
        cases.append(tuple([Fraction(float(v)) for v in g.normal(size=64)] for _ in range(2)))
    errs = [_error(*c) for c in cases]
    assert max(errs) <= bound, errs
