"""Rotated swarms whose GEMM has at most one work item per CTA pair (halves of
tiles, whole tiles, a ragged last one) and more than that: the oracle's
decisions."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu


# the first four: the arg-min block's smallest and largest sizes
@pytest.mark.parametrize("N,D", [(1, 32), (5, 33), (129, 300), (1025, 32),
                                 (130, 32), (257, 33), (2000, 63), (10000, 65), (9000, 129), (20000, 65)])
@pytest.mark.parametrize("fn", ["rot_ellipsoid", "rot_rastrigin", "rot_ackley"])
def test_same_decisions(lib, fn, N, D):
    p = workload.problem(fn, N, D, seed=D, lattice="f32")
    t = 4
    h = lib.psso_create_ex([p], "f32", tensor_rotation=1, log_stride=1, log_capacity=t + 1)
    try:
        lib.psso_run(h, t)
        X, P, _ = lib.psso_get_state(h, 0, N, D)
        log = lib.psso_get_log(h, 0)
    finally:
        lib.psso_destroy(h)
    r = oracle.run_problem(p, t, nthreads=8)
    assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"])
    assert np.array_equal(log["index"], r["log_b"]) and np.array_equal(log["accepted"], r["log_acc"])
