"""Which small single swarms run in one block and which spread over several:
the sizes of which each form is the faster one, and a given block size, with
which the one-block form stays available (to the tuner, too)."""
import pytest

import workload

pytestmark = pytest.mark.gpu


def blocks(lib, precision, N, D, order="gpx", **cfg):
    C = dict(Cg=0.8, Cp=0.6, Cw=0.3) if order == "paper" else dict(Cg=0.4, Cp=0.7, Cw=0.9)
    p = workload.problem("rastrigin", N, D, seed=1, lattice=precision, order=order, **C)
    h = lib.psso_create_ex([p], precision, **cfg)
    try:
        return lib.psso_stats(h)["blocks"]
    finally:
        lib.psso_destroy(h)


@pytest.mark.parametrize("precision,N,D,order,one", [
    ("f32", 64, 10, "gpx", True), ("f32", 64, 16, "gpx", True), ("f32", 64, 20, "gpx", True),
    ("f32", 100, 30, "gpx", True), ("f32", 12, 45, "paper", True), ("f32", 128, 12, "paper", True),
    ("f32", 8, 100, "gpx", False), ("f32", 64, 64, "paper", False), ("f32", 256, 16, "paper", False),
    ("f32", 128, 12, "gpx", False), ("f32", 128, 20, "gpx", False),
    ("f64", 96, 3, "gpx", True), ("f64", 24, 10, "gpx", True), ("f64", 100, 30, "gpx", False),
    ("f64", 8, 30, "gpx", False), ("f64", 64, 10, "paper", False)])
def test_default_shape(lib, precision, N, D, order, one):
    assert (blocks(lib, precision, N, D, order) == 1) == one


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_a_given_block_size_keeps_one_block(lib, precision):
    assert blocks(lib, precision, 100, 30, threads_per_block=256) == 1
    assert blocks(lib, precision, 84, 41, threads_per_block=512) == 1
    assert blocks(lib, precision, 100, 30, threads_per_block=256, single_block_max=-1) > 1
