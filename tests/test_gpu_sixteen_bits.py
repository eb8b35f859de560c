"""16-bit boxes reproduce recorded results.

Stochastic rounding sends a state whose last bit changed along another path, so
the mean velocity or the permeability of a 16-bit box is reproducible only if
every sum of a step keeps its order and its rounding: each link's equilibrium
with its own two operations, added link by link (tau1_node.cuh). The digests
below are of runs past the first check of the FP16 scales (64 steps); the same
bits have to come from the tiled kernel, the one-thread-per-node kernel, the
compact layout and a batch. The fluid list rounds with its own node numbers."""
import hashlib

import numpy as np
import pytest

import lbm_inputs
from paper_2312_14742_gb300 import Batch, Tau1, build
from paper_2312_14742_gb300.lbm import LBM_COMPACT, LBM_SPARSE

pytestmark = pytest.mark.gpu

G = (1e-5, 2e-6, -3e-6)
# whole tiles of every kernel, and a box that fits none, with walls on two axes
BOXES = {"whole": ((64, 48, 26), (1, 1, 1)), "ragged": ((45, 19, 13), (1, 0, 0))}
STEPS = 70

RECORDED = {
    ("batch", "f16s", 19, "whole"): "f00bcc0feb3aa02a",
    ("batch", "f16s", 19, "ragged"): "48195b7eecee96fd",
    ("batch", "f16s", 27, "whole"): "210c0493a954d288",
    ("batch", "f16s", 27, "ragged"): "61f59c778195c0c1",
    ("batch", "bf16s", 19, "whole"): "237120d305b8eaca",
    ("batch", "bf16s", 19, "ragged"): "dce3a03aba78d00b",
    ("batch", "bf16s", 27, "whole"): "76c0ecfac69f5699",
    ("batch", "bf16s", 27, "ragged"): "b3f7f9e020695886",
    ("dense", "f16s", 19, "whole"): "aea207f1732d9f40",
    ("dense", "f16s", 19, "ragged"): "0fdc90b4c3cd1df0",
    ("dense", "f16s", 27, "whole"): "9d0fa6cebee29032",
    ("dense", "f16s", 27, "ragged"): "601de588485e6cb5",
    ("dense", "bf16s", 19, "whole"): "8691d822864a99aa",
    ("dense", "bf16s", 19, "ragged"): "ec68608b69f43278",
    ("dense", "bf16s", 27, "whole"): "d5e50156730075f6",
    ("dense", "bf16s", 27, "ragged"): "2e425631c97fd12e",
    ("sparse", "f16s", 19, "whole"): "0cd15978ee205d93",
    ("sparse", "f16s", 19, "ragged"): "75a9ec00e8926e4c",
    ("sparse", "f16s", 27, "whole"): "a5d2bbb97fd422e2",
    ("sparse", "f16s", 27, "ragged"): "39c3cf71d74e99ce",
    ("sparse", "bf16s", 19, "whole"): "6dd0c892155127ef",
    ("sparse", "bf16s", 19, "ragged"): "16c0bab9400a19c8",
    ("sparse", "bf16s", 27, "whole"): "12385307ae115665",
    ("sparse", "bf16s", 27, "ragged"): "b9b1d687c181d8d4",
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def digest(fields, mean):
    h = hashlib.sha256()
    for f in fields:
        h.update((np.ascontiguousarray(f) + 0.0).tobytes())  # + 0.0: no sign of zero
    h.update(np.asarray(mean, np.float64).round(15).tobytes())
    return h.hexdigest()[:16]


def medium(box):
    (nx, ny, nz), per = BOXES[box]
    return lbm_inputs.random_mask(nx, ny, nz, 0.1, 900 + nx), per


def single(q, storage, box, layout=0, kernel="auto", variant=None):
    solid, per = medium(box)
    with Tau1(q, BOXES[box][0], storage=storage, periodic=per, g=G, layout=layout, kernel=kernel) as t:
        if variant is not None:
            t.set_variant(variant)
        t.set_geometry(solid)
        t.set_fields(*lbm_inputs.random_fields(solid.shape, 901, 2e-3, 3e-3, solid))
        t.step(STEPS)
        return digest(t.get_fields(), t.reduce()["mean_u_fluid"])


def batch(q, storage):
    """Both boxes together, from rest; the digest of each."""
    b = Batch(q, storage, capacity=2, graph_steps=35)
    try:
        slots = [b.admit(*medium(box), G) for box in BOXES]
        b.step(STEPS)
        stats = b.stats(slots)
        return [digest(b.get_fields(s), [d["permeability"]] + list(d["mean_u_fluid"])) for s, d in zip(slots, stats)]
    finally:
        b.close()


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("q", (19, 27))
@pytest.mark.parametrize("storage", ("f16s", "bf16s"))
def test_single_boxes(storage, q, box):
    want = RECORDED["dense", storage, q, box]
    assert single(q, storage, box) == want
    assert single(q, storage, box, kernel="simple") == want
    assert single(q, storage, box, layout=LBM_COMPACT) == want
    assert single(q, storage, box, layout=LBM_SPARSE) == RECORDED["sparse", storage, q, box]


@pytest.mark.parametrize("q", (19, 27))
@pytest.mark.parametrize("storage", ("f16s", "bf16s"))
def test_batches(storage, q):
    assert batch(q, storage) == [RECORDED["batch", storage, q, box] for box in BOXES]
