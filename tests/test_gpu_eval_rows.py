"""psso_evaluate_noalloc and psso_evaluate in FP64 at the edges of the row
kernel's work split (few rows: one row per warp; many: several rows per warp
with a ragged last one; widths around one chunk, 32 chunks and the largest
row), bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu

FNS = ["sphere", "ellipsoid", "rastrigin", "rosenbrock", "ackley", "hyper_ellipsoid", "schwefel12",
       "griewank", "powell", "schwefel"]


@pytest.mark.parametrize("fn", FNS)
@pytest.mark.parametrize("N,D", [(1, 1), (3, 1024), (5, 127), (33, 129), (2433, 5), (2500, 33),
                                 (40007, 3)])
def test_fp64_rows_bitexact(lib, fn, N, D):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(N + D)
    lb, ub = workload.BOUNDS[fn]
    X = rng.uniform(lb, ub, (N, D))
    o = rng.uniform(0.5 * lb, 0.5 * ub, D)
    w = workload.ellipsoid_weights(D) if fn == "ellipsoid" else None
    dev = lambda a: None if a is None else torch.from_numpy(a).cuda()  # noqa: E731
    Xd, od, wd = dev(X), dev(o), dev(w)
    f = torch.full((N,), float("nan"), dtype=torch.float64, device="cuda")
    lib.psso_evaluate_noalloc(fn, N, D, Xd.data_ptr(), od.data_ptr(),
                              None if wd is None else wd.data_ptr(), "f64", f.data_ptr(), None,
                              torch.cuda.current_stream().cuda_stream)
    rows = np.unique(np.concatenate([np.arange(min(N, 200)), rng.integers(0, N, 100), [N - 1]]))
    ref = np.array([oracle.fitness(fn, X[i], o, w) for i in rows])
    assert np.array_equal(f.cpu().numpy()[rows], ref)
    g, err = lib.psso_evaluate(fn, X, o, w)
    assert np.array_equal(g[rows], ref) and not err.any()
