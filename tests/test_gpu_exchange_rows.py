"""The gBest rows that blocks exchange carry their generation as a tag.  A row
left from before a run started (zeros of a new handle; rows of a run that
psso_set_gbest or psso_load led elsewhere) is never taken for one of the run."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu

SHAPES = [("sphere", "f64", 100, 30), ("ackley", "f64", 64, 12), ("rastrigin", "f32", 256, 16),
          ("sphere", "f64", 400, 100)]


@pytest.mark.parametrize("fn,precision,N,D", SHAPES)
def test_best_of_a_new_handle(lib, fn, precision, N, D):
    for seed in range(1, 41):
        p = workload.problem(fn, N, D, seed=seed, lattice=precision)
        h = lib.psso_create_ex([p], precision)
        try:
            _, i, row = lib.psso_best(h, 0, D)
        finally:
            lib.psso_destroy(h)
        r = oracle.run_problem(p, 0)
        assert i == r["log_b"][0]
        assert np.array_equal(row, r["P"][i]), seed


def elsewhere(lib, h, p, t):
    """Leads the handle's run to another row at generation t, then on."""
    lib.psso_run(h, t)
    lib.psso_set_gbest(h, 0, -1.0, 0, np.zeros(p["D"]))
    lib.psso_run(h, 9)


@pytest.mark.parametrize("fn,precision,N,D", SHAPES[:3])
def test_reset_after_another_run(lib, fn, precision, N, D):
    for seed in range(1, 21):
        p = workload.problem(fn, N, D, seed=seed, lattice=precision)
        h = lib.psso_create_ex([p], precision)
        try:
            elsewhere(lib, h, p, 5)
            lib.psso_reset(h)
            for _ in range(7):
                lib.psso_run(h, 2)
            X, P, _ = lib.psso_get_state(h, 0, N, D)
        finally:
            lib.psso_destroy(h)
        r = oracle.run_problem(p, 14)
        assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"]), seed


@pytest.mark.parametrize("fn,precision,N,D", SHAPES[:3])
def test_load_after_another_run(lib, fn, precision, N, D):
    for seed in range(1, 21):
        p = workload.problem(fn, N, D, seed=seed, lattice=precision)
        h1 = lib.psso_create_ex([p], precision, single_block_max=4)
        h2 = lib.psso_create_ex([p], precision)
        try:
            elsewhere(lib, h2, p, 5)
            lib.psso_run(h1, 3)
            lib.psso_load(h2, lib.psso_save(h1))
            lib.psso_run(h2, 11)
            X, P, _ = lib.psso_get_state(h2, 0, N, D)
        finally:
            lib.psso_destroy(h1)
            lib.psso_destroy(h2)
        r = oracle.run_problem(p, 14)
        assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"]), seed


def test_reset_after_the_tags_came_round(lib):
    """Generation 3 * 2^16 has generation 0's tag and slot."""
    p = workload.problem("sphere", 100, 30, seed=2, lattice="f64")
    r = oracle.run_problem(p, 0)
    h = lib.psso_create_ex([p], "f64")
    try:
        lib.psso_run(h, 3 * 65536)
        for _ in range(3):
            lib.psso_reset(h)
            _, i, row = lib.psso_best(h, 0, 30)
            assert i == r["log_b"][0] and np.array_equal(row, r["P"][i])
    finally:
        lib.psso_destroy(h)
