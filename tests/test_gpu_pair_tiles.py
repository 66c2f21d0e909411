"""Shapes at the edges of the CTA-pair GEMM's tiles (256 rows, 128 columns, cut
into 64 in the last round): the rotated pipeline against the oracle, and the
tensor-core gradients against the warp kernels."""
import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu


# 20001 x 40: 79 row tiles of one 64-column item, several per pair; 12000 x 200:
# whole tiles and a cut last round; 300 x 321: an odd number of 64-column groups
@pytest.mark.parametrize("fn,N,D", [("rot_ellipsoid", 20001, 40), ("rot_rastrigin", 12000, 200),
                                    ("rot_ackley", 300, 321), ("rot_rastrigin", 129, 65),
                                    ("rot_ackley", 257, 128)])
def test_pipeline_same_decisions(lib, fn, N, D):
    p = workload.problem(fn, N, D, seed=11, lattice="f32", shift_range=(-2.0, 2.0))
    t = 2
    h = lib.psso_create_ex([p], "f32", log_stride=1, log_capacity=t + 1)
    try:
        lib.psso_run(h, t)
        X, P, _ = lib.psso_get_state(h, 0, N, D)
        log = lib.psso_get_log(h, 0)
    finally:
        lib.psso_destroy(h)
    r = oracle.run_problem(p, t, nthreads=oracle.max_threads())
    assert np.array_equal(X, r["X"]) and np.array_equal(P, r["P"])
    assert np.array_equal(log["index"], r["log_b"]) and np.array_equal(log["accepted"], r["log_acc"])


@pytest.mark.parametrize("fn", ["rot_ellipsoid", "rot_rastrigin", "rot_ackley"])
@pytest.mark.parametrize("N,D", [(1, 16), (127, 17), (129, 63), (255, 64), (256, 65), (257, 127),
                                 (511, 129), (1025, 192), (40, 193), (2500, 320), (300, 1001)])
def test_gradients_at_tile_edges(lib, fn, N, D):
    """Against the warp kernels: their z carries at most 35 rounding errors of
    sum |M||d| (blocks of 32), the GEMM's about as many, and the gradients'
    derivative in z is at most 20 pi 2 pi of it: 2e-4 of the row's largest
    entry, as between the two implementations elsewhere in the suite."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(N + D)
    p = workload.problem(fn, 4, D, seed=3, lattice="f32", shift_range=(-1.0, 1.0))
    dev = lambda a: None if a is None else torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    X, o, w, M = dev(rng.uniform(-2, 2, (N, D))), dev(p["o"]), dev(p["w"]), dev(p["M"])
    gf = dev(rng.standard_normal(N))
    ptr = lambda v: None if v is None else v.data_ptr()  # noqa: E731
    s = torch.cuda.current_stream().cuda_stream
    res = []
    for tc in (False, True):
        f = torch.full((N,), float("nan"), device="cuda")
        # one element past the end on each side must stay untouched
        buf = torch.full((N * D + 16,), 7.0, device="cuda")
        g = buf[8:8 + N * D]
        args = (fn, N, D, X.data_ptr(), o.data_ptr(), ptr(w), M.data_ptr())
        if tc:
            n = lib.psso_fitness_workspace_size(fn, N, D)
            ws = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
            lib.psso_fitness_forward_ws(*args, f.data_ptr(), ws.data_ptr(), n, s)
            lib.psso_fitness_backward_ws(*args, gf.data_ptr(), g.data_ptr(), ws.data_ptr(), n, s)
        else:
            lib.psso_fitness_forward(*args, f.data_ptr(), s)
            lib.psso_fitness_backward(*args, gf.data_ptr(), g.data_ptr(), s)
        torch.cuda.synchronize()
        assert torch.all(buf[:8] == 7.0) and torch.all(buf[8 + N * D:] == 7.0)
        res.append((f.double().cpu().numpy(), g.reshape(N, D).double().cpu().numpy()))
    (f0, g0), (f1, g1) = res
    assert np.all(np.abs(f1 - f0) <= 1e-4 * np.maximum(np.abs(f0), 1e-3))
    big = np.abs(g0).max(axis=1, keepdims=True)
    assert np.all(np.abs(g1 - g0) <= 2e-4 * big + 1e-30)


def test_gradients_under_capture(lib):
    """The overlapped launches in a CUDA graph, replayed on new inputs: the same
    bits as the calls."""
    torch = pytest.importorskip("torch")
    N, D = 700, 130
    p = workload.problem("rot_ackley", 4, D, seed=3, lattice="f32", shift_range=(-1.0, 1.0))
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    rng = np.random.default_rng(1)
    X, o, M, gf = dev(rng.uniform(-2, 2, (N, D))), dev(p["o"]), dev(p["M"]), dev(rng.standard_normal(N))
    n = lib.psso_fitness_workspace_size("rot_ackley", N, D)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    f, g = torch.empty(N, device="cuda"), torch.empty(N, D, device="cuda")

    def call():
        s = torch.cuda.current_stream().cuda_stream
        args = ("rot_ackley", N, D, X.data_ptr(), o.data_ptr(), None, M.data_ptr())
        lib.psso_fitness_forward_ws(*args, f.data_ptr(), ws.data_ptr(), n, s)
        lib.psso_fitness_backward_ws(*args, gf.data_ptr(), g.data_ptr(), ws.data_ptr(), n, s)

    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for k in range(3):
        X.copy_(dev(rng.uniform(-2, 2, (N, D))))
        gf.copy_(dev(rng.standard_normal(N)))
        graph.replay()
        torch.cuda.synchronize()
        got = f.clone(), g.clone()
        f.zero_(), g.zero_()
        call()
        torch.cuda.synchronize()
        assert torch.equal(got[0], f) and torch.equal(got[1], g), k
