"""The batched row kernel with several slices per warp task (large handles):
ragged tasks, rows around one chunk, one slice and eight slices, both FP64
lattices (the certified FP32 filter in front of the FP64 fitness) and FP32 with
recheck, in both interval orders -- equal to the persistent kernel's run of the
same swarms."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

# (N, D): 16 swarms, more than 8 * 2 * 152 * 32 slices of 128 variables in all
SIZES = [(100003, 3), (30001, 1), (40001, 17), (9001, 128), (20000, 129), (3001, 1000), (7, 1000),
         (33, 10), (5003, 255), (5000, 256), (4999, 257), (64, 5), (2000, 64), (2500, 65), (1, 130),
         (1201, 900)]
FNS = ["rastrigin", "ackley", "rosenbrock", "sphere", "ellipsoid"]


@pytest.mark.parametrize("lattice,precision", [("f64", "f64"), ("f32", "f64"), ("f32", "f32")])
def test_large_tasks_match_the_persistent_kernel(lib, lattice, precision):
    ps = []
    for k, (N, D) in enumerate(SIZES):
        order = "paper" if k % 3 == 2 else "gpx"
        C = dict(Cg=0.8, Cp=0.6, Cw=0.3) if order == "paper" else dict(Cg=0.4, Cp=0.7, Cw=0.9)
        # narrow shifts: the runs reach values where accepts and near ties are common
        ps.append(workload.problem(FNS[k % 5], N, D, seed=40 + k, lattice=lattice, stream=k, order=order,
                                   shift_range=(-0.5, 0.5), **C))
    t = 4
    out = []
    for mode in (1, -1):
        h = lib.psso_create_ex(ps, precision, batch_stream=mode, log_stride=1, log_capacity=t + 1)
        try:
            lib.psso_run(h, t)
            out.append([lib.psso_get_state(h, k, p["N"], p["D"]) + (lib.psso_get_log(h, k),)
                        for k, p in enumerate(ps)])
        finally:
            lib.psso_destroy(h)
    for k, (a, b) in enumerate(zip(*out)):
        for q in range(2 if precision == "f32" else 3):      # X, P (and the FP64 pBest values)
            assert np.array_equal(a[q], b[q]), (ps[k]["fn"], SIZES[k], q)
        for key in ("index", "accepted"):
            assert np.array_equal(a[3][key], b[3][key]), (ps[k]["fn"], SIZES[k], key)


@pytest.mark.parametrize("fn", ["rastrigin", "ackley", "rosenbrock"])
def test_filter_at_extreme_scales(lib, fn):
    """FP64 fitness where the FP32 filter's floats over- and underflow, or the
    whole swarm sits on one value: same runs as without the filter."""
    ps = []
    for k, (lb, ub) in enumerate([(-1e30, 1e30), (-1e18, 1e18), (-1e-25, 1e-25), (-1e-45, 1e-45),
                                  (-1e-3, 1e-3), (-3.0, 5e7)] * 3):
        ps.append(workload.problem(fn, 40, 20 + 60 * (k % 3), seed=k + 1, lattice="f64", stream=k,
                                   bounds=(lb, ub), shift_range=(0.25 * lb, 0.25 * ub)))
    t = 12
    out = []
    for mode in (1, -1):
        h = lib.psso_create_ex(ps, "f64", batch_stream=mode)
        try:
            lib.psso_run(h, t)
            out.append([lib.psso_get_state(h, k, p["N"], p["D"]) for k, p in enumerate(ps)])
        finally:
            lib.psso_destroy(h)
    for k, (a, b) in enumerate(zip(*out)):
        for q in range(3):
            assert np.array_equal(a[q], b[q], equal_nan=True), (ps[k]["lb"], q)
