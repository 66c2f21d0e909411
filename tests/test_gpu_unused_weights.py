"""Weights passed to a function that has none change nothing, in both batched
fitness calls and in a swarm."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

UNWEIGHTED = ["sphere", "rastrigin", "rosenbrock", "ackley", "hyper_ellipsoid", "schwefel12",
              "griewank", "powell", "schwefel"]
F64_ONLY = ("schwefel12", "griewank", "powell", "schwefel")


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("fn", UNWEIGHTED)
def test_weights_of_an_unweighted_function_are_ignored(lib, fn, precision):
    torch = pytest.importorskip("torch")
    if precision == "f32" and fn in F64_ONLY:
        pytest.skip("FP64 fitness only")
    N, D = 37, 33
    rng = np.random.default_rng(D)
    lb, ub = workload.BOUNDS[fn]
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    X, o = f32(rng.uniform(lb, ub, (N, D))), f32(rng.uniform(0.5 * lb, 0.5 * ub, D))
    w = rng.uniform(2.0, 50.0, D)
    want, _ = lib.psso_evaluate(fn, X, o, precision=precision)
    got, _ = lib.psso_evaluate(fn, X, o, w, precision=precision)
    assert np.array_equal(got, want)
    Xd, od, wd = (torch.from_numpy(a).cuda() for a in (X, o, w))
    f = torch.empty(N, dtype=torch.float64, device="cuda")
    lib.psso_evaluate_noalloc(fn, N, D, Xd.data_ptr(), od.data_ptr(), wd.data_ptr(), precision,
                              f.data_ptr(), None, torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(f.cpu().numpy(), want)
