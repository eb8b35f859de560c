"""Compact steps whose strips and node list run beside each other, in both orders:
the dense bits, step after step."""
import numpy as np
import pytest

import lbm_inputs
from paper_2312_14742_gb300 import Tau1, build
from paper_2312_14742_gb300.lbm import LBM_COMPACT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


# few strips and nodes: strips first, in parts of a tile column; a node list of several
# waves: list first, the strips in an even share per SM; many strips: whole columns
@pytest.mark.parametrize("storage,q", [("f32", 19), ("f32", 27), ("f64", 19), ("f16s", 19), ("bf16s", 27)])
@pytest.mark.parametrize("dims,phi", [((64, 48, 30), 0.5), ((192, 192, 96), 0.3), ((256, 256, 80), 0.7)])
def test_both_orders_give_the_dense_bits(dims, phi, storage, q):
    nx, ny, nz = dims
    solid, _ = lbm_inputs.sphere_pack(nx, ny, nz, 6.0, phi, 4100 + nx)
    st = lbm_inputs.random_fields(solid.shape, 4101, 2e-3, 3e-3, solid)

    def go(layout, thr=None):
        with Tau1(q, dims, storage=storage, g=(1e-5, -2e-6, 3e-6), layout=layout) as t:
            if thr is not None:
                t.set_compact_threshold(thr)
            t.set_geometry(solid)
            t.set_fields(*st)
            t.step(25)
            return t.get_fields(), t.compact_info() if layout else None

    ref, _ = go(0)
    for thr in (0.2, 0.35, 0.5, 0.75):
        got, info = go(LBM_COMPACT, thr)
        assert info["tiled_columns"] + info["listed_columns"] > 0
        for a, b in zip(got, ref):
            assert np.array_equal(a, b, equal_nan=True), (thr, info)
