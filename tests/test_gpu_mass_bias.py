"""An FP32 step loses no density on average.

One step of an open periodic box keeps the sum of drho exactly; what FP32 adds is
its rounding, which has to fall to either side alike: a loss that every node takes
in every step grows with the number of steps, however small it is."""
import numpy as np
import pytest

import lbm_inputs
from paper_2312_14742_gb300 import Tau1, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


@pytest.mark.parametrize("kernel", ("tiled", "simple"))
@pytest.mark.parametrize("q", (19, 27))
def test_density_rounds_to_both_sides(q, kernel):
    """A node's drho is 1/36 (D3Q19) or 1/216 (D3Q27) of a sum with less than 100
    roundings of values below 4 or 32, each with an rms of ulp / sqrt(12) = 7e-8 or
    5.5e-7 at most: 2e-8 or 2.6e-8 in all. The mean of N = 128^3 such errors has a
    standard deviation of 1.8e-11 at most; five of them."""
    shape = (128, 128, 128)
    st = lbm_inputs.random_fields(shape, 77, 0.0, 0.1)
    with Tau1(q, shape, storage="f32", kernel=kernel) as t:
        t.set_geometry(np.zeros(shape, np.uint8))
        t.set_fields(*st)
        t.step(1)
        drho = t.get_fields()[0]
    assert abs(float(np.mean(drho))) <= 9e-11
