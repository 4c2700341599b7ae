"""Workloads of the library as its users run them: single rectangles, exact integers, wide
truncated strips, finite-lattice sweeps, a served mix, the any-v Potts strip and a first solve
with nothing cached.  Sizes are those of the configured workloads, the tests and the bench, and
odd ones in between; the primes come from the seed."""
import math

import numpy as np
import torch

import paper_1005_3609_gb300 as cp
import synthetic_inputs


def motzkin(n):
    a, b = 1, 1  # M_0, M_1
    if n < 2:
        return 1
    for k in range(2, n + 1):
        a, b = b, ((2 * k + 1) * b + (3 * k - 3) * a) // (k + 2)
    return b


def listed():
    return [
        # the smallest request a user makes: one little rectangle, exact integers (latency, launches)
        {"name": "integers_square_5x6_p4", "kind": "rect", "lattice": "square", "L": 5, "N": 6, "P": 4, "D": -1, "integers": True},
        # one mid-size rectangle at full degree on 8 primes, residues (the two configured single solves)
        {"name": "solve_square_12x13_p8", "kind": "rect", "lattice": "square", "L": 12, "N": 13, "P": 8, "D": -1, "integers": False},
        {"name": "solve_triangular_13x14_p8", "kind": "rect", "lattice": "triangular", "L": 13, "N": 14, "P": 8, "D": -1, "integers": False},
        # the same square rectangle as exact integers: 10 primes are what the Whitney bound asks for (not a multiple of 4)
        {"name": "integers_square_12x13_p10", "kind": "rect", "lattice": "square", "L": 12, "N": 13, "P": 10, "D": -1, "integers": True},
        # one rectangle, one prime: the plain path a user takes to add a single prime
        {"name": "solve_triangular_12x12_p1", "kind": "rect", "lattice": "triangular", "L": 12, "N": 12, "P": 1, "D": -1, "integers": False},
        # a wide strip truncated to a series order, few rows, an odd number of primes (vectors of a gigabyte)
        {"name": "wide_square_17x4_d40_p5", "kind": "rect", "lattice": "square", "L": 17, "N": 4, "P": 5, "D": 40, "integers": False},
        # the headline sweeps: all rectangles of the band, 16 primes, series as exact integers
        {"name": "sweep_square_k33_p16", "kind": "sweep", "lattice": "square", "k": 33, "P": 16},
        {"name": "sweep_triangular_k33_p16", "kind": "sweep", "lattice": "triangular", "k": 33, "P": 16},
        # a sweep to a low order: many small steps in one graph
        {"name": "sweep_square_k17_p8", "kind": "sweep", "lattice": "square", "k": 17, "P": 8},
        # a burst of mixed requests through the continuous-batching server
        {"name": "serve_mix_32", "kind": "serve", "n": 32, "stream": 1, "L_max": 12},
        # the Potts partition function at v = 2
        {"name": "potts_square_10x10_v2_p8", "kind": "potts", "lattice": "square", "L": 10, "N": 10, "P": 8, "D": -1, "v": 2},
        # a one-off solve in a process that has not used this width yet: the tables are built on the way
        {"name": "first_triangular_12x13_p4", "kind": "first", "lattice": "triangular", "L": 12, "N": 13, "P": 4, "D": -1},
    ]


def draw(rng):
    kind = rng.choice(["rect", "rect", "rect", "wide", "sweep", "serve", "potts", "first"])
    lattice = rng.choice(["square", "triangular"])
    if kind == "rect":
        L = rng.randint(4, 13)
        return {"kind": "rect", "lattice": lattice, "L": L, "N": L + rng.randint(0, 3), "P": int(round(math.exp(rng.uniform(0, math.log(16))))),
                "D": -1, "integers": rng.random() < 0.4}
    if kind == "wide":
        return {"kind": "rect", "lattice": lattice, "L": rng.randint(14, 17), "N": rng.randint(3, 6), "P": rng.randint(1, 12), "D": rng.randint(20, 48),
                "integers": False}
    if kind == "sweep":
        return {"kind": "sweep", "lattice": lattice, "k": rng.randint(12, 29), "P": rng.choice([4, 6, 8, 12, 16])}
    if kind == "serve":
        return {"kind": "serve", "n": int(round(math.exp(rng.uniform(math.log(2), math.log(40))))), "stream": rng.randint(2, 999), "L_max": rng.randint(6, 12)}
    if kind == "potts":
        L = rng.randint(4, 11)
        return {"kind": "potts", "lattice": lattice, "L": L, "N": L + rng.randint(0, 2), "P": rng.randint(2, 12), "D": -1, "v": rng.choice([-2, 1, 2, 3])}
    return {"kind": "first", "lattice": lattice, "L": rng.randint(6, 13), "N": rng.randint(6, 14), "P": rng.choice([1, 4, 8]), "D": rng.choice([-1, 30])}


def n_terms(lattice, k):
    return (2 * k - 2 if k % 2 else 2 * k - 3) if lattice == "square" else k


def requests(case):
    return synthetic_inputs.serving_requests(seed=case["stream"], n=case["n"], L_range=(4, case["L_max"]))


def primes_of(seed, n):
    return cp.select_primes(synthetic_inputs.prime_draws(seed, 64), n)


class State:
    def __init__(self, **kw):
        self.__dict__.update(kw)


def prepare(case, seed):
    """The handles a program keeps: a strip, a sweep or a server, on its own stream, and the primes."""
    kind = case["kind"]
    stream = torch.cuda.Stream()
    if kind == "serve":
        reqs = [(r["lattice"], r["L"], r["N"], primes_of(seed * 1000 + i, r["n_primes"])) for i, r in enumerate(requests(case))]
        return State(case=case, reqs=reqs, stream=stream, server=cp.Server(8 << 30, max_active=64, stream=stream))
    primes = primes_of(seed, case["P"])
    if kind == "sweep":
        sw = cp.Sweep(case["lattice"], case["k"], primes, stream)
        return State(case=case, stream=stream, sweep=sw, limbs=np.zeros((3, sw.n_terms, cp._lib.limbs_for(case["P"])), dtype=np.uint32))
    if kind == "first":
        return State(case=case, stream=stream, primes=primes)
    strip = cp.Strip(case["lattice"], case["L"], primes, max_degree=case["D"], max_rows=case["N"], stream=stream, v=case.get("v"))
    return State(case=case, stream=stream, strip=strip)


def read_integers(strip):
    """The residues, to be kept beside the result, and cp_read_integers as its caller in C sees it: the limbs of every
    coefficient, and the sufficiency flags."""
    residues = strip.read()
    lpc = cp._lib.limbs_for(len(strip.primes))
    limbs = np.zeros((strip.degree + 1, lpc), dtype=np.uint32)
    flags = np.zeros(strip.degree + 1, dtype=np.uint32)
    u32p = cp._lib.u32p
    rc = cp.load().cp_read_integers(strip._h, limbs.ctypes.data_as(u32p), limbs.size, lpc, flags.ctypes.data_as(u32p), None)
    if rc not in (0, cp._lib.CP_EPRIMES):
        raise cp.CPError("cp_read_integers", rc, "")
    return [residues, limbs, flags]


def run(state):
    case = state.case
    kind = case["kind"]
    if kind == "serve":
        sv = state.server
        ids = [sv.submit(*r) for r in state.reqs]
        left = len(ids)
        while left:
            left -= sv.step()[2]
        out = [sv.result(i)[1] for i in ids]
        sv.poll()
        for i in ids:
            sv.release(i)
        return out
    if kind == "sweep":
        sw = state.sweep
        sw.run()
        if case["P"] >= 8:  # enough primes for the series' integers
            sw.series_integers(out=state.limbs)
            return [state.limbs.copy(), sw.read_series()]
        return [sw.read_series()]
    if kind == "first":
        cp.load().cp_clear_table_cache()
        with cp.Strip(case["lattice"], case["L"], state.primes, max_degree=case["D"], max_rows=case["N"], stream=state.stream) as s:
            s.advance(case["N"] - 1)
            return s.read()
    s = state.strip
    s.reset()
    s.advance(case["N"] - 1)
    if case.get("integers"):
        return read_integers(s)
    return s.read()


def strip_work(lattice, L, N, P, D, potts=False):
    """One pass over the state vector per row, up to the degree L h that a strip of height h has: read once, written once;
    two operations for each word of each per-site factor's output."""
    S = math.comb(2 * L, L) // (L + 1) if potts else motzkin(L - 1)
    D = L * N - 1 if D < 0 else D
    words = sum(S * (min(D, L * h) + 1) * P for h in range(1, N))
    return {"bytes": 8 * words + 4 * P * (D + 1), "flops": 2 * L * words}


def work(case):
    kind = case["kind"]
    if kind in ("rect", "potts", "first"):
        return strip_work(case["lattice"], case["L"], case["N"], case["P"], case["D"], kind == "potts")
    if kind == "sweep":
        n = n_terms(case["lattice"], case["k"])
        parts = [strip_work(case["lattice"], r, case["k"] - r, case["P"], n - 1) for r in range(1, case["k"] // 2 + 1)]
    else:
        parts = [strip_work(r["lattice"], r["L"], r["N"], r["n_primes"], -1) for r in requests(case)]
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


def next_prime(n):
    while n < 2 or any(n % d == 0 for d in range(2, math.isqrt(n) + 1)):
        n += 1
    return n


def rectangle_polynomial(lattice, L, N, v, primes, D):
    """sum over edge subsets A of v^|A| w^(|V| - k(A)) modulo each prime, by a plain transfer matrix over the partitions of the front."""
    pr = np.array(primes, dtype=np.int64)[:, None]
    one = np.zeros((len(primes), D + 1), dtype=np.int64)
    one[:, 0] = 1

    def shifted(x):
        y = np.zeros_like(x)
        y[:, 1:] = x[:, :-1]
        return y

    def canon(s):
        m = {}
        return tuple(m.setdefault(x, len(m)) for x in s)

    def add(d, s, x):
        s = canon(s)
        d[s] = (d[s] + x) % pr if s in d else x % pr

    def edge(vec, a, b):
        out = {}
        for s, x in vec.items():
            if s[a] == s[b]:
                add(out, s, x * (1 + v))
            else:
                add(out, s, x)
                add(out, tuple(s[a] if t == s[b] else t for t in s), shifted(x) * v)
        return out

    vec = {tuple(range(L)): one}
    for row in range(N):
        if row:
            for i in range(L):  # old site i, then the new site in its place: vertical edge, diagonal to the old site i + 1
                out = {}
                for s, x in vec.items():
                    add(out, s + (99,), x)
                vec = edge(out, i, L)
                if lattice == "triangular" and i + 1 < L:
                    vec = edge(vec, i + 1, L)
                out = {}
                for s, x in vec.items():
                    add(out, s[:i] + (s[L],) + s[i + 1:L], x)
                vec = out
        for i in range(L - 1):
            vec = edge(vec, i, i + 1)
    return sum(vec.values()) % pr


def exact(case, seed):
    """Residues of a small rectangle by plain numpy in 64 bits; None where that takes long (and for the limbs, which they determine)."""
    if case["kind"] not in ("rect", "potts", "first") or case["L"] > 6 or case["N"] > 9:
        return None
    primes = []
    for d in synthetic_inputs.prime_draws(seed, 64):
        p = next_prime(d)
        if len(primes) < case["P"] and p < 1 << 31 and p not in primes:
            primes.append(p)
    L, N = case["L"], case["N"]
    full = rectangle_polynomial(case["lattice"], L, N, case.get("v", -1), primes, L * N - 1)
    D = L * N - 1 if case["D"] < 0 else case["D"]
    out = np.zeros((len(primes), D + 1), dtype=np.uint32)
    n = min(D + 1, full.shape[1])
    out[:, :n] = full[:, :n]
    return [out, None, None] if case.get("integers") else out
