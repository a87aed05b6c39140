"""The C-ABI library builds, loads and exports every entry point of include/plds.h
(CPU only: no compute calls), and the host-side threshold tables agree with the
oracle's (both compute them with their own exact arithmetic)."""
import ctypes

import numpy as np
import pytest

from paper_2106_03824_gb300 import _build
from paper_2106_03824_gb300 import plds as P


@pytest.fixture(scope="module")
def lib():
    _build.build()
    return P.load()


def test_header_declares_the_boundary():
    names = P.exported_symbols_in_header()
    for must in ("plds_create", "plds_batch_insert", "plds_batch_delete", "plds_coreness",
                 "plds_levels", "plds_destroy", "plds_last_status"):
        assert must in names


def test_library_exports_every_declared_symbol(lib):
    missing = [s for s in P.exported_symbols_in_header() if not hasattr(lib, s)]
    assert not missing, f"symbols declared in plds.h but not exported: {missing}"


def test_library_has_no_oracle_dependency():
    import subprocess
    out = subprocess.run(["nm", "-D", "--defined-only", str(P.LIB_PATH)], capture_output=True, text=True).stdout
    assert "orc_" not in out
    src = "".join(p.read_text() for p in (_build.CSRC).iterdir() if p.is_file())
    assert "oracle" not in src.lower()


def test_invalid_parameters_rejected_without_device(lib):
    # parameter validation happens before any CUDA call
    for args in [(0, 0.4, 3.0), (10, 0.0, 3.0), (10, 0.4, -1.0)]:
        h = lib.plds_create(*args)
        assert not h
        assert lib.plds_last_status() == P.PLDS_EINVAL
    assert lib.plds_batch_insert(None, None, 0) == P.PLDS_EINVAL
    assert lib.plds_levels(None, None) == P.PLDS_EINVAL
    # the single-handle autotuner checks its arguments first as well
    offs = np.array([0, 1], np.int64)
    kinds = np.array([0], np.int32)
    e = np.zeros((1, 2), np.int32)
    best = P.PldsTuning()
    assert lib.plds_autotune(None, e.ctypes.data, offs.ctypes.data, kinds.ctypes.data, 1, 0, 4,
                             ctypes.byref(best)) == P.PLDS_EINVAL


def test_serving_admission_rule(lib):
    """The serving loop's admission rule (pure host function): admit when the pool has
    room or a grown pool holding every used and promised slot fits in free memory;
    otherwise wait while earlier requests are in flight, else reject."""
    A = P.server_admission
    assert A(1000, 400, 100, 500, 0) == 0          # room in the pool, exactly
    assert A(1000, 400, 0, 601, 0) == 2            # no room, nothing in flight, no memory
    assert A(1000, 400, 101, 500, 0) == 1          # no room, but requests in flight
    assert A(1000, 400, 100, 501, 4 * 1001) == 0   # a grown pool of 1001 slots fits
    assert A(1000, 400, 100, 501, 4 * 1001 - 1) == 1
    assert A(1000, 400, 0, 601, 4 * 1001 - 1) == 2
    assert A(1000, 1000, 0, 0, 0) == 0             # deletions and queries need nothing
    assert A(-1, 0, 0, 0, 0) == P.PLDS_EINVAL
    assert A(0, 0, 0, 1, -5) == P.PLDS_EINVAL


def test_tune_search_finds_the_minimum_of_a_separable_cost(lib):
    """Coordinate descent over (thread cutoff, block cutoff, load factor) against a
    fake cost with its minimum at (8, 8192, 5/8): found from the defaults, every
    evaluation inside the candidate lists, no configuration evaluated twice."""
    import math
    seen = []

    def cost(k):
        seen.append(tuple(k.values()))
        return (1.0 + (math.log2(k["thread_max_cap"]) - 3) ** 2 + 0.5 * (math.log2(k["block_cap"]) - 13) ** 2
                + 10 * abs(k["load_num"] / k["load_den"] - 0.625))

    best, n = P.tune_search(cost)
    assert best == {"thread_max_cap": 8, "block_cap": 8192, "load_num": 5, "load_den": 8, "list_cap": 256}
    assert n == len(seen) == len(set(seen))
    for t, b, ln, ld, lc in seen:
        assert t in (4, 8, 16, 32, 64) and b in (1024, 2048, 4096, 8192, 16384)
        assert (ln, ld) in ((1, 2), (5, 8), (3, 4), (7, 8)) and lc in (128, 256, 1024, 1 << 30)


def test_tune_search_budget_and_failure(lib):
    calls = []
    best, n = P.tune_search(lambda k: calls.append(k) or 1.0, max_trials=3)
    assert n == 3 and len(calls) == 3
    assert best == {"thread_max_cap": 16, "block_cap": 4096, "load_num": 3, "load_den": 4,
                    "list_cap": 256}  # flat: defaults kept
    with pytest.raises(P.PldsError) as ex:
        P.tune_search(lambda k: -1.0)
    assert ex.value.code == P.PLDS_EINTERNAL
    # a 1 % gain is below the 2 % threshold: the incumbent stays
    best, _ = P.tune_search(lambda k: 0.99 if k["thread_max_cap"] == 4 else 1.0)
    assert best["thread_max_cap"] == 16


@pytest.mark.parametrize("fixed_cost, picked", [(1.2, 0), (0.99, 0), (0.9, 8)])
def test_tune_search_times_an_unset_cutoff(lib, fixed_cost, picked):
    """From a start with the cutoff left to the handle (-1), that setting (0) is evaluated
    first and stays unless a fixed cutoff costs at least 2 % less."""
    seen = []

    def cost(k):
        seen.append(k["thread_max_cap"])
        c = {0: 1.0, 8: fixed_cost}.get(k["thread_max_cap"], 1.5)
        return c * (0.9 if k["block_cap"] == 2048 else 1.0)

    best, n = P.tune_search(cost, start={"thread_max_cap": -1, "block_cap": 1024})
    assert seen[0] == 0 and n == len(seen)
    assert set(seen) == {0, 4, 8, 16, 32, 64}
    assert best == {"thread_max_cap": picked, "block_cap": 2048, "load_num": 3, "load_den": 4, "list_cap": 256}


def test_opt_levels_per_group_matches_oracle(lib):
    """The library's exact PLDSOpt group size agrees with the oracle's own bignum."""
    from oracle import oracle as O
    rng = np.random.default_rng(2)
    for _ in range(300):
        d = float(rng.choice([0.05, 0.1, 0.2, 0.4, 0.4211, 0.4212, 1.0, 3.2]))
        m = int(rng.integers(0, 2**32))
        assert P.opt_levels_per_group(m, d) == O.opt_levels_per_group(m, d), (m, d)
    assert lib.plds_opt_levels_per_group(2**32, 0.4) == P.PLDS_EINVAL
