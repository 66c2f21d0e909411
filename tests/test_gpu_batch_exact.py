"""The batched arg-min's queue of candidates that the FP32 bounds leave (FP32
fitness with recheck): swarms full of ties and near ties, of one particle, of
more particles than one block's threads, of copies of the gBest row, and after a
gBest put there by psso_set_gbest -- equal to the persistent kernel's runs."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 3), (31, 4), (255, 5), (256, 1), (257, 2), (300, 129), (1025, 3), (4097, 2),
         (3000, 7), (64, 260), (33, 1000), (2049, 1), (129, 33), (700, 64), (5000, 1)]
FNS = ["sphere", "ellipsoid", "rastrigin", "rosenbrock", "ackley"]
# 17 floats per variable: pBests tie and repeat
COARSE = dict(lattice="f32", bounds=(1024.0, 1024.0 + 2.0 ** -9), shift_range=(1024.0, 1024.0))


@pytest.mark.parametrize("shift", [0, 2])
def test_near_ties_match_the_persistent_kernel(lib, shift):
    ps = []
    for k, (N, D) in enumerate(SIZES):
        # no fresh draws in every third swarm, which converges to copies of its gBest row
        C = dict(Cg=0.5, Cp=0.9, Cw=1.0) if k % 3 == 0 else dict(Cg=0.4, Cp=0.7, Cw=0.9)
        ps.append(workload.problem(FNS[(k + shift) % 5], N, D, seed=70 + k, stream=k, **COARSE, **C))
    out = []
    for mode in (1, -1):
        h = lib.psso_create_ex(ps, "f32", batch_stream=mode, log_stride=1, log_capacity=64)
        try:
            lib.psso_run(h, 9)
            lib.psso_run(h, 14)
            out.append([lib.psso_get_state(h, k, p["N"], p["D"])[:2] + (lib.psso_get_log(h, k), lib.psso_best(h, k, p["D"]))
                        for k, p in enumerate(ps)])
        finally:
            lib.psso_destroy(h)
    for k, (a, b) in enumerate(zip(*out)):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), (ps[k]["fn"], SIZES[k])
        for key in ("index", "accepted"):
            assert np.array_equal(a[2][key], b[2][key]), (ps[k]["fn"], SIZES[k], key)
        assert a[3][:2] == b[3][:2] and np.array_equal(a[3][2], b[3][2]), (ps[k]["fn"], SIZES[k])


def test_after_set_gbest(lib):
    """A caller's value for a row that copies then share is not taken over."""
    ps = [workload.problem(FNS[k % 5], 200 + k, 3 + k, seed=k, stream=k, Cg=0.5, Cp=0.9, Cw=1.0, **COARSE) for k in range(16)]
    out = []
    for mode in (1, -1):
        h = lib.psso_create_ex(ps, "f32", batch_stream=mode, single_block_max=100000)
        try:
            lib.psso_run(h, 12)
            for k, p in enumerate(ps):
                v, i, row = lib.psso_best(h, k, p["D"])
                lib.psso_set_gbest(h, k, v - 1.0, i, row)
            lib.psso_run(h, 12)
            out.append([lib.psso_get_state(h, k, p["N"], p["D"])[:2] + (lib.psso_best(h, k, p["D"])[:2],)
                        for k, p in enumerate(ps)])
        finally:
            lib.psso_destroy(h)
    for k, (a, b) in enumerate(zip(*out)):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2], k
