"""The chunk gather's own sums and reductions (Sec. 3.5), driven on the GPU through
cp_debug_chunk_sum and compared with Python's integers: the 32-bit reduction at the
smallest primes that its bound admits, at the largest, and at its largest coefficient
sums; the one for every prime over both of its quotient shifts.  Words are at the ends
of [-p, p], and sums lie at and beside multiples of p."""
import random

import pytest

import paper_1005_3609_gb300 as cp
from paper_1005_3609_gb300 import _lib

pytestmark = pytest.mark.gpu

MAX_SUM = (1 << 15) - 1


def is_prime(n):
    return n > 1 and all(n % d for d in range(2, int(n ** 0.5) + 1))


def next_prime(n):
    while not is_prime(n):
        n += 1
    return n


def fast_ok(s, p):
    return s <= 8192 and s * 163840 + 65536 + (p * (s + 2) >> 17) + 2 < p


def smallest_fast_prime(s):
    lo, hi = 2, 1 << 31
    while lo < hi:  # the first p within the bound, which is monotone in p
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fast_ok(s, mid) else (mid + 1, hi)
    return next_prime(lo)


def split(s, rng, most):
    """Coefficients of absolute sum s."""
    out = []
    while s:
        out.append(min(s, rng.randint(1, most)) if most < 127 else min(s, 127))
        s -= out[-1]
    return out


def rows(p, s, rng):
    """(coefficients, words): all of one sign or mixed, words at the ends of [-p, p] or random."""
    used = rng.choice([s, s, max(s - 1, 0), s // 2, min(s, 3)])
    c = split(used, rng, rng.choice([127, 127, 3]) if used < 2000 else 127)
    c = [v * rng.choice([[1], [-1], [1, -1]])[0] for v in c] if rng.random() < 0.7 else [rng.choice([v, -v]) for v in c]
    pick = rng.choice([[p], [-p], [p - 1], [p, -p], [p - 1, -p], [0, 1, -1], None])
    x = [rng.choice(pick) if pick else rng.randint(-p, p - 1) for _ in c]
    if c and rng.random() < 0.3:  # the sum at or beside a multiple of p, through the last word
        for want in (0, 1, -1):
            rest = sum(a * b for a, b in zip(c[:-1], x)) % p
            try:
                v = (want - rest) * pow(c[-1], -1, p) % p
            except ValueError:
                break
            x[-1] = v - rng.choice([0, p])
            if rng.random() < 0.5:
                break
    return c, x


def run(cases, any_prime):
    by_edges = {}
    for p, s, c, x in cases:
        n = next(e for e in (0, 1, 4, 32, 300, 3000, 33000) if e >= len(c))
        by_edges.setdefault(n, []).append((p, s, c + [0] * (n - len(c)), x + [0] * (n - len(x))))
    for group in by_edges.values():
        p, s, c, x = ([g[i] for g in group] for i in range(4))
        got = _lib.debug_chunk_sum(c, x, s, p, any_prime=any_prime)
        for pi, si, ci, xi, g in zip(p, s, c, x, got):
            v = sum(a * b for a, b in zip(ci, xi))
            assert -pi <= g < pi and (g - v) % pi == 0, (pi, si, g, v)


def test_32_bit_reduction_within_its_bound():
    rng, cases = random.Random(3), []
    for s in (0, 1, 2, 3, 8, 60, 127, 500, 2000, 5000, 6000):
        p0 = smallest_fast_prime(s)
        assert fast_ok(s, p0) and p0 > 1 << 16
        for p in (p0, next_prime(p0 + 1), next_prime(2 * p0) if p0 < 1 << 29 else p0, 2147483629, 2147483647):
            cases += [(p, s) + rows(p, s, rng) for _ in range(200 if s < 500 else 40)]
    run(cases, False)


def test_reduction_for_every_prime():
    rng, cases = random.Random(4), []
    for p in (2, 3, 5, 7, 251, 257, 32749, 65521, 65537, 131071, next_prime(1 << 17), 1000003, next_prime(1 << 24),
              next_prime(1 << 30), 2147483647):
        for s in (0, 1, 2, 60, 110, 8192, 8193, MAX_SUM):
            cases += [(p, s) + rows(p, s, rng) for _ in range(100 if s < 1000 else 12)]
    run(cases, True)


def test_sums_outside_the_domain_are_refused():
    p = 2147483647
    _lib.debug_chunk_sum([[127]], [[p]], [127], [p])
    for c, x, s, q, any_prime in ((128, 1, 128, p, False), (-128, 1, 128, p, True), (2, 1, 1, p, False),
                                  (1, 101, 1, 97, True), (1, 1, 1 << 15, p, True), (1, 1, 60, 1000003, False),
                                  (1, 1, 8193, p, False), (1, 1, 1, 1, True)):
        with pytest.raises(cp.CPError):
            _lib.debug_chunk_sum([[c]], [[x]], [s], [q], any_prime=any_prime)
