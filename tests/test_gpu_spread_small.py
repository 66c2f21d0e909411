"""Small swarms, which run as several pipelined blocks by default: the same
results as in one block, and the calls that a one-block swarm takes
(psso_set_gbest; psso_load of a state saved by a one-block run) still work."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu

FNS = ["sphere", "ackley", "griewank", "schwefel12", "powell"]


@pytest.mark.parametrize("fn", FNS)
@pytest.mark.parametrize("N,D", [(4, 3), (17, 30), (33, 10), (65, 7), (100, 30), (31, 129), (128, 4)])
def test_default_shape_matches_the_oracle(lib, fn, N, D):
    p = workload.problem(fn, N, D, seed=N, lattice="f64", stream=D)
    t = 25
    h = lib.psso_create_ex([p], "f64", log_stride=1, log_capacity=t + 1)
    try:
        lib.psso_run(h, 10)
        lib.psso_run(h, t - 10)
        X, P, pF = lib.psso_get_state(h, 0, N, D)
        log = lib.psso_get_log(h, 0)
    finally:
        lib.psso_destroy(h)
    r = oracle.run_problem(p, t)
    assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"]) and np.array_equal(pF, r["pF"])
    assert np.array_equal(log["index"], r["log_b"]) and np.array_equal(log["value"], r["log_v"])
    assert np.array_equal(log["accepted"], r["log_acc"])


@pytest.mark.parametrize("fn", ["sphere", "ackley", "rosenbrock"])
@pytest.mark.parametrize("N,D", [(17, 30), (33, 10), (100, 30), (31, 129)])
def test_default_shape_same_decisions_fp32(lib, fn, N, D):
    p = workload.problem(fn, N, D, seed=N, lattice="f32", stream=D)
    t = 25
    h = lib.psso_create_ex([p], "f32", log_stride=1, log_capacity=t + 1)
    try:
        lib.psso_run(h, t)
        X, P, _ = lib.psso_get_state(h, 0, N, D)
        log = lib.psso_get_log(h, 0)
    finally:
        lib.psso_destroy(h)
    r = oracle.run_problem(p, t)
    assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"])
    assert np.array_equal(log["index"], r["log_b"]) and np.array_equal(log["accepted"], r["log_acc"])


@pytest.mark.parametrize("lattice,precision", [("f64", "f64"), ("f32", "f64"), ("f32", "f32")])
def test_set_gbest_as_in_one_block(lib, lattice, precision):
    p = workload.problem("ackley", 100, 30, seed=2, lattice=lattice)
    row = np.asarray(p["o"], dtype=np.float64) * 0.5
    if lattice == "f32":
        row = row.astype(np.float32).astype(np.float64)
    out = []
    for cfg in (dict(), dict(single_block_max=100000)):
        h = lib.psso_create_ex([p], precision, **cfg)
        try:
            for value, index in ((0.125, 3), (-5.0, 12345)):
                lib.psso_run(h, 7)
                lib.psso_set_gbest(h, 0, value, index, row)
                v, i, got = lib.psso_best(h, 0, 30)
                assert (v, i) == (value, index) and np.array_equal(got, row)
            lib.psso_run(h, 5)
            X, P, pF = lib.psso_get_state(h, 0, 100, 30)
            out.append((X, P) + lib.psso_best(h, 0, 30) + ((pF,) if precision == "f64" else ()))
        finally:
            lib.psso_destroy(h)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("fn,lattice,precision", [("griewank", "f64", "f64"), ("griewank", "f32", "f64"),
                                                  ("rosenbrock", "f32", "f32")])
@pytest.mark.parametrize("t1", [0, 1, 9])
def test_load_of_a_one_block_state(lib, fn, lattice, precision, t1):
    p = workload.problem(fn, 100, 30, seed=3, lattice=lattice)
    h1 = lib.psso_create_ex([p], precision, single_block_max=100000, log_stride=1, log_capacity=40)
    h2 = lib.psso_create_ex([p], precision, log_stride=1, log_capacity=40)
    other = lib.psso_create_ex([dict(p, N=60)], precision, log_stride=1, log_capacity=40)
    try:
        lib.psso_run(h1, t1)
        blob = lib.psso_save(h1)
        lib.psso_run(h2, 4)
        lib.psso_load(h2, blob)
        lib.psso_run(h2, 11)
        t = t1 + 11
        r = oracle.run_problem(p, t)
        X, P, pF = lib.psso_get_state(h2, 0, 100, 30)
        assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"])
        assert precision == "f32" or np.array_equal(pF, r["pF"])
        log = lib.psso_get_log(h2, 0)
        assert np.array_equal(log["index"], r["log_b"])
        with pytest.raises(lib.PssoError):
            lib.psso_load(other, blob)
    finally:
        for h in (h1, h2, other):
            lib.psso_destroy(h)
