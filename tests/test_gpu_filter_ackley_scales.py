"""FP64 Ackley swarms whose squares reach the denormal floats (positions of
1e-15 to 1e-23): the batched row kernel's FP32 filter takes no decision there
that the FP64 fitness does not take."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["f64", "f32"])
def test_small_scale_ackley_runs(lib, lattice):
    ps = []
    for k, s in enumerate([1e-15, 1e-17, 1e-18, 1e-19, 1e-20, 1e-21, 1e-22, 1e-23] * 2):
        s = float(np.float32(s))
        ps.append(workload.problem("ackley", 200, 20 + 120 * (k // 8), seed=k + 1, lattice=lattice, stream=k,
                                   bounds=(-s, s), shift_range=(-0.25 * s, 0.25 * s)))
    t = 15
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
            assert np.array_equal(a[q], b[q]), (ps[k]["ub"], ps[k]["D"], q)
