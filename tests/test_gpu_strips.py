"""The strip kernel (tau1_strip.cu) against the one-thread-per-node kernel, which
shares its arithmetic: the same bits. Sizes where the cut into strips can go
wrong: boxes narrower and wider than a strip by a column or two, strips that
cross the end of a row of columns, one and two columns, rows and planes left
over, periodic and walled faces, media dense enough that the wall list fills up
within one plane."""
import numpy as np
import pytest

import lbm_inputs
from paper_2312_14742_gb300 import Batch, Tau1, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def medium(dims, kind, seed):
    nx, ny, nz = dims
    rnd = np.random.RandomState(seed)
    if kind == "open":
        return np.zeros((nz, ny, nx), np.uint8)
    if kind == "noise":  # every fluid node has walls around it
        return (rnd.rand(nz, ny, nx) < 0.4).astype(np.uint8)
    return (rnd.rand(nz, ny, nx) < 0.05).astype(np.uint8)


@pytest.mark.parametrize("storage,q", [("f32", 19), ("f32", 27), ("f64", 19), ("f64", 27), ("f16s", 19), ("bf16s", 27)])
@pytest.mark.parametrize("dims,per,kind", [
    ((1, 1, 1), (1, 1, 1), "open"), ((2, 5, 3), (1, 1, 1), "few"), ((29, 6, 4), (1, 0, 1), "few"),
    ((30, 7, 5), (0, 1, 1), "few"), ((31, 4, 9), (1, 1, 1), "noise"), ((32, 9, 6), (1, 1, 1), "noise"),
    ((32, 9, 6), (0, 1, 0), "noise"), ((33, 3, 7), (1, 1, 0), "few"), ((59, 10, 3), (1, 1, 1), "noise"),
    ((62, 13, 8), (0, 0, 0), "few"), ((97, 2, 5), (1, 1, 1), "open"), ((5, 61, 3), (1, 1, 1), "few"),
    ((130, 17, 11), (1, 0, 1), "noise")])
def test_strips_give_the_simple_kernels_bits(dims, per, kind, storage, q):
    solid = medium(dims, kind, sum(dims))
    state = lbm_inputs.random_fields(solid.shape, 31, 2e-3, 3e-3, solid)
    g = (1e-5, 2e-6, -3e-6)

    def go(kernel, variant=None):
        with Tau1(q, dims, storage=storage, periodic=per, g=g, kernel=kernel) as t:
            if variant is not None:
                t.set_variant(variant)
            t.set_geometry(solid)
            t.set_fields(*state)
            t.step(5)
            return t.get_fields()

    ref = go("simple")
    for v in range(4 if storage == "f64" else 16):
        for a, b in zip(go("tiled", v), ref):
            assert np.array_equal(a, b, equal_nan=True), v
    if storage == "f16s":
        return  # a batch picks its scales on the device
    # the batched step, from a state at rest
    with Tau1(q, dims, storage=storage, periodic=per, g=g, kernel="simple") as t:
        t.set_geometry(solid)
        t.step(5)
        rest = t.get_fields()
    b = Batch(q, storage, capacity=2, graph_steps=5)
    try:
        slot = b.admit(solid, per, g)
        b.step(5)
        for x, y in zip(b.get_fields(slot), rest):
            assert np.array_equal(x, y, equal_nan=True)
    finally:
        b.close()
