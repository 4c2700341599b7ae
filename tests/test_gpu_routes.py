"""GPU tests of calls that reach the kernels by another route than a plain solve: reads
after an ungraphed pass, small primes, the register tiles, rows without padding lanes."""
import numpy as np
import pytest

import gpu_util
from oracle import tm_exact, tm_generic

pytestmark = pytest.mark.gpu

cp = pytest.importorskip("paper_1005_3609_gb300")


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cp.load()


def is_prime(n):
    return n > 1 and all(n % d for d in range(2, int(n ** 0.5) + 1))


def primes_from(lo, n):
    out = []
    while len(out) < n:
        if is_prime(lo):
            out.append(lo)
        lo += 1
    return out


@pytest.mark.parametrize("n_primes,groups,tile", [(8, 2, 0), (5, 1, 0), (3, 1, 4)])
@pytest.mark.parametrize("lattice", ["square", "triangular"])
def test_ptilde_after_an_ungraphed_pass(lattice, n_primes, groups, tile):
    # the profile pass runs the gathers without the series kernel: residues all the same, before and after a run
    import torch
    primes = gpu_util.seed_primes(n_primes, seed=41)
    with cp.Sweep(lattice, 11, primes, torch.cuda.Stream(), tile=tile, prime_groups=groups) as sw:
        series = None
        for step in ("profile", "run", "profile", "run"):
            getattr(sw, step)()
            for (r, s), res in sw.read_ptilde().items():
                want = tm_exact.ptilde(lattice, r, s)[:sw.n_terms]
                want += [0] * (sw.n_terms - len(want))
                assert res.tolist() == gpu_util.residues_of(want, primes), (step, r, s)
            if step == "run":
                got = sw.read_series()
                assert series is None or np.array_equal(got, series)
                series = got


def test_ptilde_keeps_its_primes_until_the_next_run():
    import torch
    one, two = gpu_util.seed_primes(8, seed=42)[:4], gpu_util.seed_primes(8, seed=42)[4:]
    with cp.Sweep("square", 10, one, torch.cuda.Stream()) as sw:
        for step in ("run", "profile"):
            sw.set_primes(one)
            getattr(sw, step)()
            sw.sync()
            h = sw.read_ptilde()
            sw.set_primes(two)
            after = sw.read_ptilde()
            for (r, s), res in h.items():
                assert np.array_equal(res, after[(r, s)]), (step, r, s)
                want = tm_exact.ptilde("square", r, s)[:sw.n_terms]
                want += [0] * (sw.n_terms - len(want))
                assert res.tolist() == gpu_util.residues_of(want, one), (step, r, s)


def solve(lattice, L, N, primes, D=-1, v=None, tile=0):
    with cp.Strip(lattice, L, primes, max_degree=D, max_rows=N, v=v) as s:
        s.set_tile(tile)
        s.advance(N - 1)
        return s.read()


def solve_ms(lattice, L, N, primes, tile=0, D=-1):
    """Median time of reset, rows and read-out, in ms."""
    import time

    import torch
    with cp.Strip(lattice, L, primes, max_degree=D, max_rows=N) as s:
        s.set_tile(tile)
        ms = []
        for _ in range(9):
            torch.cuda.synchronize()
            t = time.perf_counter()
            s.reset()
            s.advance(N - 1)
            s.read()
            ms.append((time.perf_counter() - t) * 1e3)
    return sorted(ms[2:])[3]


# below the bound of the chunk kernel's 32-bit reduction the sums are put together to 64 bits: both shifts of its
# quotient (2^17), the smallest primes, and large ones beside them
@pytest.mark.parametrize("primes", [[2], [3, 2], [2, 3, 5, 7, 11], primes_from(65500, 4), primes_from(131000, 9),
                                    primes_from(1 << 17, 4), primes_from(1000003, 6), primes_from(15 * 163840, 4),
                                    [2, 2147483647, 131071, 131101, 1073741827]],
                         ids=lambda p: "%d_%d" % (p[0], len(p)))
@pytest.mark.parametrize("lattice", ["square", "triangular"])
def test_small_primes(lattice, primes):
    L, N = 6, 8
    want = gpu_util.residues_of(tm_exact.ptilde(lattice, L, N), primes)
    assert solve(lattice, L, N, primes).tolist() == want
    assert solve(lattice, L, N, primes, D=7).tolist() == [w[:8] for w in want]
    for L, N, D in ((12, 4, 40), (13, 5, -1)):  # heavy rows, split and in several passes
        assert np.array_equal(solve(lattice, L, N, primes, D=D), solve(lattice, L, N, primes, D=D, tile=4)), L


@pytest.mark.parametrize("lattice,v", [("square", 8), ("square", -9), ("square", 10), ("triangular", 4), ("triangular", -3)])
def test_potts_sums_beyond_the_fast_bound(lattice, v):
    # coefficients within a byte, their sums into one state in the hundreds and thousands: no prime below is fast
    for primes in (primes_from(10007, 4), gpu_util.seed_primes(4, seed=43)):
        want = gpu_util.residues_of(tm_generic.ztilde(lattice, 5, 4, v), primes)
        assert solve(lattice, 5, 4, primes, v=v).tolist() == want
        assert np.array_equal(solve(lattice, 9, 5, primes, v=v), solve(lattice, 9, 5, primes, v=v, tile=4))


@pytest.mark.parametrize("lattice", ["square", "triangular"])
def test_small_primes_are_no_slow_case(lattice):
    # the same kernel with a longer reduction (the register kernel took 11 times as long here)
    big, small = gpu_util.seed_primes(8, seed=44), primes_from(1000003, 8)
    assert solve_ms(lattice, 12, 13, small) < 2.5 * solve_ms(lattice, 12, 13, big)


# both depths of the register kernel (launches of fewer and of more blocks), whole and padded prime lanes
@pytest.mark.parametrize("tile", [1, 2, 4, 8])
@pytest.mark.parametrize("lattice", ["square", "triangular"])
def test_register_tiles_agree(lattice, tile):
    for L, N, D, P in ((13, 4, 40, 1), (13, 4, -1, 8), (11, 5, -1, 20), (7, 8, 30, 5)):
        primes = gpu_util.seed_primes(P, seed=45)
        assert np.array_equal(solve(lattice, L, N, primes, D=D, tile=tile), solve(lattice, L, N, primes, D=D)), (L, P)


@pytest.mark.parametrize("tile,ms", [(1, 6.0), (2, 7.5), (4, 9.6), (8, 12.3)])
def test_register_tiles_keep_their_speed(tile, ms):
    # ms: what the tile took on whole rows, before degree windows
    assert solve_ms("square", 12, 13, gpu_util.seed_primes(8, seed=46), tile=tile) < ms
