"""GPU tests of calls that reach the kernels by another route than a plain solve: reads
after an ungraphed pass, small primes, the register tiles, rows without padding lanes."""
import numpy as np
import pytest

import gpu_util
from oracle import modp, tm_exact

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
