"""GPU tests of the gathers on degree windows and of the choice between the two
gather kernels: every result bit-exact against the oracle or against the same
strip on the other kernel."""
import numpy as np
import pytest

import gpu_util
from oracle import modp, tm_exact, tm_generic

pytestmark = pytest.mark.gpu

cp = pytest.importorskip("paper_1005_3609_gb300")


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cp.load()


def next_prime(n):
    while any(n % d == 0 for d in range(2, int(n ** 0.5) + 1)):
        n += 1
    return n


def solve(lattice, L, N, primes, D=-1, v=None, tile=0, again=False):
    with cp.Strip(lattice, L, primes, max_degree=D, max_rows=N, v=v) as s:
        s.set_tile(tile)
        if again:  # buffers full of another height's words: none of them may be read
            s.advance(N - 1)
            s.read()
            s.reset()
        s.advance(N - 1)
        return s.read()


# prime counts whose chunks per degree do and do not divide a warp (1..8), padded or not; widths on
# both sides of one pass over a row (128 chunks)
@pytest.mark.parametrize("P", [1, 3, 4, 9, 12, 17, 20, 24, 28, 31])
@pytest.mark.parametrize("lattice", ["square", "triangular"])
def test_prime_lanes_and_passes(lattice, P):
    primes = gpu_util.seed_primes(P, seed=31)
    L, N = 6, 8
    want = gpu_util.residues_of(tm_exact.ptilde(lattice, L, N), primes)
    for tile in (0, 2):
        assert solve(lattice, L, N, primes, tile=tile, again=True).tolist() == want, tile
    for D in (0, 1, 7, 30):
        assert solve(lattice, L, N, primes, D=D).tolist() == [w[:D + 1] for w in want], D


# the chunk kernel's sums need p > S 163840 + ...: primes on both sides of that for these widths' tables
@pytest.mark.parametrize("lattice", ["square", "triangular"])
def test_primes_around_the_fast_reduction_bound(lattice):
    for lo in (1 << 17, 1 << 20, 10 * 163840, 15 * 163840, 64 * 163840, 1 << 27):
        primes = [next_prime(lo)]
        while len(primes) < 4:
            primes.append(next_prime(primes[-1] + 1))
        for L, N in ((5, 6), (9, 5)):
            got = solve(lattice, L, N, primes, D=20)
            for k in (0, 3):
                assert got[k].tolist() == modp.ptilde_heights(lattice, L, [N], 20, primes[k])[N].tolist(), (lo, L)


@pytest.mark.parametrize("lattice,v", [("triangular", 5), ("triangular", -6), ("square", 12), ("square", -11)])
def test_potts_tables_with_coefficients_beyond_a_byte(lattice, v):
    # (1 + v)^2 v or (1 + v) v exceeds 127 in some of the strip's tables and not in others
    primes = gpu_util.seed_primes(4, seed=13)
    want = gpu_util.residues_of(tm_generic.ztilde(lattice, 5, 4, v), primes)
    assert solve(lattice, 5, 4, primes, v=v).tolist() == want


def test_wide_strips_agree_on_both_kernels():
    # the chunk kernel's units (heavy rows split, several passes) against the register kernel's rows
    primes = gpu_util.seed_primes(8, seed=17)
    for lattice, L, N, D in (("square", 13, 6, 70), ("triangular", 13, 5, 60), ("square", 12, 4, -1)):
        assert np.array_equal(solve(lattice, L, N, primes, D=D), solve(lattice, L, N, primes, D=D, tile=4)), (lattice, L)


def test_unpadded_rows_where_padded_ones_do_not_fit():
    import torch
    primes = gpu_util.seed_primes(5, seed=19)
    L, N, D = 12, 4, 13000
    want = solve("square", L, N, primes, D=60)
    vectors = (5798 + 2188) * (D + 1) * 4 * 2 * 1.4  # two vectors and the read-out's, per prime
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(int(free - 6.3 * vectors), dtype=torch.uint8, device="cuda")  # room for 5 lanes, not for 8
    try:
        got = solve("square", L, N, primes, D=D)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(got[:, :61], want) and not got[:, 61:].any()


def test_sweep_changes_primes_across_the_kernels():
    import torch
    stream = torch.cuda.Stream()
    big, small = gpu_util.seed_primes(4, seed=23), [65521, 65519, 131101, 131111]
    with cp.Sweep("square", 11, big, stream) as sw:
        for primes in (big, small, big):
            sw.set_primes(primes)
            sw.run()
            got = sw.read_ptilde()
            for (r, s), res in got.items():
                want = tm_exact.ptilde("square", r, s)[:sw.n_terms]
                want += [0] * (sw.n_terms - len(want))
                assert res.tolist() == gpu_util.residues_of(want, primes), (r, s)
