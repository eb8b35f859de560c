"""The autotune cache gives a choice back only to the kernels and the box it was
timed with."""
import json

import numpy as np
import pytest

from paper_2312_14742_gb300 import Tau1, build, lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def tuned(dims, periodic=(1, 1, 1)):
    with Tau1(19, dims, storage="f32", periodic=periodic, g=(1e-5, 0, 0)) as t:
        t.set_geometry(np.zeros(dims[::-1], np.uint8))
        n0 = t.launch_count
        v, ms = t.autotune(1)
        return v, ms, t.launch_count > n0


def test_entries_of_other_kernels_and_boxes_are_not_used(tmp_path):
    path = tmp_path / "tune.json"
    lbm.lbm_tau1_set_tune_cache(str(path))
    try:
        tuned((64, 48, 40))
        (key,) = json.loads(path.read_text())["entries"]
        # a file of the releases whose variants were tiles: the same key up to the tile fit
        old = key[:key.index("/full") + len("/full")]
        path.write_text('{"version": 1, "entries": {\n "%s": {"variant": 3, "ms_per_step": 1e-09}\n}}\n' % old)
        v, ms, timed = tuned((64, 48, 40))
        assert timed and ms > 1e-8
        entries = json.loads(path.read_text())["entries"]
        assert entries[old]["variant"] == 3 and entries[key]["variant"] == v
        # the same box again, then others of its size bucket
        assert not tuned((64, 48, 40))[2]
        assert tuned((32, 96, 40))[2]
        assert tuned((64, 48, 40), periodic=(0, 1, 1))[2]
    finally:
        lbm.lbm_tau1_set_tune_cache(None)
