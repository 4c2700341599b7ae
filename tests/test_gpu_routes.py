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


def gb_used():
    import torch
    free, total = torch.cuda.mem_get_info()
    return (total - free) / 1e9


STATES_12 = 2 * 7986 + 835 + 127  # square width 12, two-site tables: two vectors and the read-out's two


def lane_gb(D):
    """Memory of one prime lane of a square width-12 strip's vectors."""
    return STATES_12 * (D + 1) * 4 / 1e9


class Padding:
    """Two strips of one prime whose padding lanes take all but a thousandth of the share that padding may have."""

    def __enter__(self):
        import torch
        prime = gpu_util.seed_primes(1, seed=48)
        share = torch.cuda.mem_get_info()[1] / 8
        self.D = int(0.4995 * share / (3 * lane_gb(0) * 1e9)) - 1
        self.strips = [cp.Strip("square", 12, prime, max_degree=self.D, max_rows=3) for _ in range(2)]
        return self

    def __exit__(self, *a):
        for s in self.strips:
            s.close()


def test_padding_lanes_leave_room_for_other_strips():
    primes = gpu_util.seed_primes(3, seed=48)
    want = solve("square", 12, 3, primes[:1])[0].tolist()
    with Padding() as pad:
        D, lane = pad.D, lane_gb(pad.D)
        for n, lanes in ((1, 1), (3, 3)):  # the share is taken: their primes alone
            before = gb_used()
            with cp.Strip("square", 12, primes[:n], max_degree=D, max_rows=3) as s:
                assert abs(gb_used() - before - lanes * lane) < 0.1 * lane
                s.advance(2)
                got = s.read()[0]
                assert got[:len(want)].tolist() == want and not got[len(want):].any()
        pad.strips.pop().close()
        before = gb_used()
        with cp.Strip("square", 12, primes[:1], max_degree=D, max_rows=3):  # given back: four lanes again
            assert abs(gb_used() - before - 4 * lane) < 0.1 * lane


@pytest.mark.parametrize("lattice,n_primes,groups", [("square", 5, 1), ("triangular", 2, 2), ("square", 1, 0)])
def test_sweeps_of_unpadded_rows(lattice, n_primes, groups):
    import torch
    primes, stream, out = gpu_util.seed_primes(n_primes, seed=49), torch.cuda.Stream(), []

    def sweep(k):
        before = gb_used()
        with cp.Sweep(lattice, k, primes, stream, prime_groups=groups) as sw:
            used = gb_used() - before
            sw.run()
            return used, sw.read_series(), sw.read_ptilde()

    sweep(31)  # (tables and kernels are there)
    padded = sweep(31)
    with Padding():
        alone = sweep(31)
    Pg = n_primes // max(groups, 1)
    assert alone[0] < padded[0] * (Pg / (Pg + 3 & ~3) + 0.15)
    assert np.array_equal(padded[1], alone[1])
    assert padded[2].keys() == alone[2].keys() and all(np.array_equal(padded[2][x], alone[2][x]) for x in padded[2])


def test_rows_of_the_primes_alone_where_padded_ones_do_not_fit():
    import torch
    primes, D = gpu_util.seed_primes(5, seed=50), 13000
    want = solve("square", 12, 4, primes, D=60)
    torch.cuda.empty_cache()
    lane = lane_gb(D)
    hold = torch.empty(int((torch.cuda.mem_get_info()[0] / 1e9 - 6.5 * lane) * 1e9), dtype=torch.uint8, device="cuda")
    try:
        before = gb_used()
        with cp.Strip("square", 12, primes, max_degree=D, max_rows=4) as s:
            assert abs(gb_used() - before - 5 * lane) < 0.2 * lane
            s.advance(3)
            got = s.read()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(got[:, :61], want) and not got[:, 61:].any()


def test_wide_two_site_tables_keep_their_build_time():
    # triangular width 17 with two-site tables: one table per factor, as before them, took 47.5 to 48.3 ms
    import time

    import torch
    primes, ms = gpu_util.seed_primes(12, seed=51), []
    for _ in range(4):
        cp.load().cp_clear_table_cache()
        torch.cuda.synchronize()
        t = time.perf_counter()
        cp.Strip("triangular", 17, primes, max_degree=40, max_rows=3).close()
        ms.append((time.perf_counter() - t) * 1e3)
    assert min(ms) < 52


@pytest.mark.parametrize("lattice,L", [("square", 14), ("triangular", 13), ("triangular", 14), ("triangular", 15)])
def test_wide_two_site_tables_are_the_product(lattice, L):
    # every way a two-site table is built (eight, two or one thread a source), against one table per factor
    primes, out = gpu_util.seed_primes(4, seed=52), []
    for mode in (3, 0):
        old = cp.set_factor_pairing(mode)
        try:
            out.append(solve(lattice, L, 3, primes, D=12))
        finally:
            cp.set_factor_pairing(old)
    assert np.array_equal(*out)


# rows of one pass of a warp (512 / lanes degrees) and around whole numbers of passes, dealt out by degrees; widths
# without and with heavy rows, whose parts are dealt out again
@pytest.mark.parametrize("lattice", ["square", "triangular"])
@pytest.mark.parametrize("L,N,P", [(1, 300, 32), (2, 90, 12), (4, 60, 32), (7, 40, 16), (10, 30, 32), (11, 20, 28)])
def test_long_rows_dealt_out_by_degrees(lattice, L, N, P):
    primes, span = gpu_util.seed_primes(P, seed=53), 512 // (P + 3 & ~3)
    whole = None
    for D in (-1, span - 1, span, 2 * span - 2, 2 * span, 7 * span, 7 * span + 1):
        got = solve(lattice, L, N, primes, D=D)
        assert np.array_equal(got, solve(lattice, L, N, primes, D=D, tile=4)), D
        if D == -1:
            whole = got
        else:
            n = min(D + 1, whole.shape[1])
            assert np.array_equal(got[:, :n], whole[:, :n]) and not got[:, n:].any(), D
    if L <= 4 and N <= 90:
        want = tm_exact.ptilde(lattice, L, N)
        assert whole.tolist() == gpu_util.residues_of(want, primes)


@pytest.mark.parametrize("L,N,P,ms", [(4, 200, 32, 4.2), (3, 400, 4, 5.7), (7, 171, 16, 12.9), (8, 150, 32, 16.4)])
def test_tall_strips_keep_their_speed(L, N, P, ms):
    # ms: what the rows and the read-out took with a block for the columns of a row (before the chunk kernel)
    assert solve_ms("square", L, N, gpu_util.seed_primes(P, seed=54)) < ms


@pytest.mark.parametrize("lattice,L,v,ms", [("square", 7, 2, 1.65), ("triangular", 7, 2, 1.85), ("square", 9, None, 2.70),
                                            ("triangular", 9, None, 2.32), ("square", 14, None, 7.9)])
def test_small_tables_keep_their_build_time(lattice, L, v, ms):
    # ms: the cold tables and vectors before degree windows; one table per factor (any-v, or rows of 336 bytes)
    import time

    import torch
    primes, stream, got = gpu_util.seed_primes(4, seed=55), torch.cuda.Stream(), []
    for _ in range(40):
        cp.load().cp_clear_table_cache()
        torch.cuda.synchronize()
        t = time.perf_counter()
        cp.Strip(lattice, L, primes, max_degree=20, max_rows=3, v=v, stream=stream).close()
        got.append((time.perf_counter() - t) * 1e3)
    assert min(got) < ms  # (the least of many: a busy host only adds)
