"""Rounding of the FP32 sums behind the rotated fitness of the device-buffer
call (psso_fitness_forward_ws).  With the identity as rotation z is exact, and
a row of one term 1 and terms just below half an ulp of 1 makes every addition
to the running sum round down: a sum in sequence loses one such term an
addition.  Blocks of 32 terms, joined in pairs, and the 64-column sums added
as a tree keep the chain at 32 + 1 + 4 additions."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
# three roundings in a term, then the additions of the longest chain
CHAIN = 3 + 32 + 1 + 4


@pytest.mark.parametrize("fn", ["rot_ellipsoid", "rot_rastrigin"])
@pytest.mark.parametrize("D", [31, 32, 64, 65, 128, 257, 1000, 1024])
@pytest.mark.parametrize("at", [0, 15])
def test_sums_lose_at_most_the_chain(lib, fn, D, at):
    torch = pytest.importorskip("torch")
    N = 10240      # enough rows that a warp sums 64 columns (few: 32)
    scale = 1.0 if fn == "rot_ellipsoid" else 1.0 + 20.0 * np.pi ** 2   # z^2 + 20 sin^2(pi z) for small z
    X = np.full((N, D), np.sqrt(0.96 * U / scale), dtype=np.float32)
    X[np.arange(N), (at + 64 * np.arange(N)) % D] = 1.0
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()  # noqa: E731
    Xd, od, wd, Md = dev(X), dev(np.zeros(D)), dev(np.ones(D)), dev(np.eye(D))
    f = torch.empty(N, device="cuda")
    ws = torch.empty(lib.psso_fitness_workspace_size(fn, N, D), dtype=torch.uint8, device="cuda")
    lib.psso_fitness_forward_ws(fn, N, D, Xd.data_ptr(), od.data_ptr(), wd.data_ptr(), Md.data_ptr(),
                                f.data_ptr(), ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    z = X.astype(np.float64)
    if fn == "rot_rastrigin":
        want = (z * z + 20.0 * np.sin(np.pi * (z - np.rint(z))) ** 2).sum(1)
    else:
        want = (z * z).sum(1)
    err = np.abs(f.cpu().numpy().astype(np.float64) - want)
    assert np.all(err <= CHAIN * U * want), (err / (U * want)).max()
