"""Swarms whose fitness overflows: FP64 sums that reach infinity, and FP32
fitness beyond the floats' range (decided in FP64).  The oracle's decisions in
every form a swarm runs in; no particle left out of the arg-min."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu


def check(lib, ps, precision, **cfg):
    t = 6
    h = lib.psso_create_ex(ps, precision, log_stride=1, log_capacity=t + 1, **cfg)
    try:
        lib.psso_run(h, t)
        got = [lib.psso_get_state(h, k, p["N"], p["D"])[:2] + (lib.psso_get_log(h, k)["index"],)
               for k, p in enumerate(ps)]
    finally:
        lib.psso_destroy(h)
    for p, (X, P, index) in zip(ps, got):
        r = oracle.run_problem(p, t)
        assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"]), p["fn"]
        assert np.array_equal(index, r["log_b"]), p["fn"]


@pytest.mark.parametrize("fn", ["sphere", "rastrigin", "rosenbrock"])
@pytest.mark.parametrize("N,D,cfg", [(3, 3, {}), (100, 30, {}), (100, 30, dict(single_block_max=4)), (700, 100, {}),
                                     (700, 100, dict(pipeline=2)), (40, 20, dict(batch_stream=1)),
                                     (40, 200, dict(batch_stream=1))])
def test_fp64_infinite_fitness(lib, fn, N, D, cfg):
    ps = [workload.problem(fn, N, D, seed=2, lattice="f64", bounds=(-1e200, 1e200), shift_range=(0.0, 0.0))]
    check(lib, ps, "f64", **cfg)


@pytest.mark.parametrize("fn", ["sphere", "rastrigin", "rosenbrock"])
@pytest.mark.parametrize("N,D,cfg", [(3, 3, {}), (64, 20, {}), (250, 16, {}), (400, 100, {}),
                                     (400, 100, dict(pipeline=2)), (40, 20, dict(batch_stream=1)),
                                     (40, 200, dict(batch_stream=1))])
def test_fp32_beyond_the_floats(lib, fn, N, D, cfg):
    b = float(np.float32(1e30))
    ps = [workload.problem(fn, N, D, seed=2, lattice="f32", bounds=(-b, b), shift_range=(0.0, 0.0))]
    check(lib, ps, "f32", **cfg)


@pytest.mark.parametrize("fn", ["rot_ellipsoid", "rot_rastrigin"])
def test_rotated_fp32_beyond_the_floats(lib, fn):
    b = float(np.float32(1e25))
    ps = [workload.problem(fn, 150, 40, seed=3, lattice="f32", bounds=(-b, b), shift_range=(0.0, 0.0))]
    check(lib, ps, "f32", tensor_rotation=1)
    check(lib, ps, "f32", tensor_rotation=-1)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("fn", ["ackley", "rot_ackley"])
def test_ackley_far_from_its_optimum(lib, fn, precision):
    """Ackley where its exponential has left the normal doubles (rows beyond
    about 3500 in magnitude), and on both sides of the exponents at which it
    becomes 0 against 1."""
    rng = np.random.default_rng(4)
    D = 20
    X = np.concatenate([s * rng.uniform(-1.0, 1.0, (30, D))
                        for s in (100.0, 250.0, 330.0, 400.0, 1e3, 4e3, 1e4, 1e6, 1e10, 1e18)])
    X = X.astype(np.float32).astype(np.float64)
    M = workload.rotation(D, 3) if fn == "rot_ackley" else None
    o = np.zeros(D)
    f, err = lib.psso_evaluate(fn, X, o, None, M, precision=precision)
    want = np.array([oracle.fitness(fn, x, o, None, M) for x in X])
    if precision == "f64":
        assert np.array_equal(f, want)
    else:
        assert np.all(np.abs(f - want) <= err)


def test_fp32_ackley_beyond_the_floats(lib):
    b = float(np.float32(1e30))
    for N, D, cfg in [(3, 3, {}), (250, 16, {}), (400, 100, {}), (40, 20, dict(batch_stream=1))]:
        check(lib, [workload.problem("ackley", N, D, seed=2, lattice="f32", bounds=(-b, b), shift_range=(0.0, 0.0))],
              "f32", **cfg)
