"""States of small swarms saved in one of their two forms (one block, several
pipelined blocks) and loaded by a handle that runs the other: the run goes on
as the oracle's does."""
import struct

import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fn,lattice,precision,N,D", [("ackley", "f64", "f64", 100, 30),
                                                      ("sphere", "f32", "f64", 64, 10),
                                                      ("rosenbrock", "f32", "f32", 250, 16),
                                                      ("rastrigin", "f32", "f32", 100, 30)])
@pytest.mark.parametrize("saver,loader", [(dict(), dict(single_block_max=4)), (dict(), dict(threads_per_block=256)),
                                          (dict(threads_per_block=256), dict()), (dict(single_block_max=4), dict()),
                                          (dict(single_block_max=-1), dict()), (dict(), dict())])
@pytest.mark.parametrize("t1", [0, 9])
def test_state_of_the_other_form(lib, fn, lattice, precision, N, D, saver, loader, t1):
    p = workload.problem(fn, N, D, seed=5, lattice=lattice)
    log = dict(log_stride=1, log_capacity=40)
    if saver.get("single_block_max") == -1 and lib_spreads(lib, p, precision):
        pytest.skip("the default form is the spread one already")
    h1 = lib.psso_create_ex([p], precision, **saver, **log)
    h2 = lib.psso_create_ex([p], precision, **loader, **log)
    try:
        lib.psso_run(h1, t1)
        lib.psso_run(h2, 3)
        lib.psso_load(h2, lib.psso_save(h1))
        lib.psso_run(h2, 8)
        X, P, _ = lib.psso_get_state(h2, 0, N, D)
        got = lib.psso_get_log(h2, 0)
        best = lib.psso_best(h2, 0, D)
    finally:
        lib.psso_destroy(h1)
        lib.psso_destroy(h2)
    r = oracle.run_problem(p, t1 + 8)
    assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"])
    assert np.array_equal(got["index"], r["log_b"])
    assert best[1] == r["log_b"][-1]


def lib_spreads(lib, p, precision):
    h = lib.psso_create_ex([p], precision)
    try:
        return lib.psso_stats(h)["blocks"] > 1
    finally:
        lib.psso_destroy(h)


def test_interval_of_the_gbest_without_an_upper_bound(lib):
    """A saved gBest known by an interval that reaches beyond the floats is
    evaluated by the block that owns its particle."""
    N, D = 250, 16
    p = workload.problem("rastrigin", N, D, seed=6, lattice="f32")
    tried = 0
    for t1 in range(1, 30):
        h1 = lib.psso_create_ex([p], "f32", single_block_max=4, log_stride=1, log_capacity=64)
        h2 = lib.psso_create_ex([p], "f32", log_stride=1, log_capacity=64)
        try:
            lib.psso_run(h1, t1)
            blob = bytearray(lib.psso_save(h1))
            index = int(lib.psso_get_log(h1, 0)["index"][-1])
            at = blob.find(struct.pack("<qq", index, t1))          # GBestDev: idx, gen, ..., lo, hi, ver, has64
            if index < N // 2 or at < 0 or blob[at + 60:at + 64] != bytes(4):
                continue
            tried += 1
            blob[at + 52:at + 56] = struct.pack("<f", float("inf"))
            lib.psso_load(h2, bytes(blob))
            lib.psso_run(h2, 6)
            X, P, _ = lib.psso_get_state(h2, 0, N, D)
        finally:
            lib.psso_destroy(h1)
            lib.psso_destroy(h2)
        r = oracle.run_problem(p, t1 + 6)
        assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"])
    assert tried
