"""FP32 psso_evaluate_noalloc: values that a shift of bits does not convert
(zeros, denormal floats, the float range's ends) and values that are not floats
(NaN for the row, also for a shift that is not one), at the edges of the row
widths the kernel is written for."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


def call(lib, torch, fn, X, o, w):
    N, D = X.shape
    dev = [None if a is None else torch.from_numpy(a).cuda() for a in (X, o, w)]
    f = torch.empty(N, dtype=torch.float64, device="cuda")
    err = torch.empty_like(f)
    ptr = [None if a is None else a.data_ptr() for a in dev]
    lib.psso_evaluate_noalloc(fn, N, D, *ptr, "f32", f.data_ptr(), err.data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
    return f.cpu().numpy(), err.cpu().numpy()


@pytest.mark.parametrize("fn", ["sphere", "ellipsoid", "rosenbrock", "ackley"])
@pytest.mark.parametrize("D", [1, 10, 127, 128, 129, 256, 257, 513, 1021, 1024])
def test_rows_of_floats_and_others(lib, fn, D):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(D)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    X, o = f32(rng.uniform(-2.0, 2.0, (40, D))), f32(rng.uniform(-1.0, 1.0, D))
    w = workload.ellipsoid_weights(D) if fn == "ellipsoid" else None
    X[1] = 0.0
    X[2, ::3] = -0.0
    X[3, ::2] = float(np.float32(1e-45))
    X[4, -1] = float(np.float32(1.1754944e-38))
    want, werr = lib.psso_evaluate(fn, X, o, w, precision="f32")
    for k, bad in enumerate([0.1, np.nan, np.inf, 1e-46, 3.5e38, 1.0 + 2.0 ** -24]):
        X[10 + k, (7 * k) % D] = bad
    f, err = call(lib, torch, fn, X, o, w)
    floats = np.ones(40, dtype=bool)
    floats[[10, 11, 13, 14, 15]] = False                # an infinity is a float
    rows = floats.copy()
    rows[12] = False
    assert np.array_equal(f[rows], want[rows]) and np.array_equal(err[rows], werr[rows])
    assert np.isnan(f[~floats]).all() and np.isnan(err[~floats]).all()
    o[D // 2] = 0.1
    f, err = call(lib, torch, fn, X, o, w)
    assert np.isnan(f).all() and np.isnan(err).all()
