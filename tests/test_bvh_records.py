"""The BVH2 records that the kernels read (16-bit planes on a per-scene grid): every record's box
must contain its exact child box, whatever the scene's extent and place."""
import numpy as np
import pytest

from paper_2310_07182_gb300 import binding as cr

FORMS = {
    "one triangle": (1, 1.0, 0.0, (1, 1, 1)),
    "soup": (5000, 1.0, 0.0, (1, 1, 1)),
    "far from the origin": (3000, 1.0, 1e6, (1, 1, 1)),
    "flat": (2000, 1.0, 3.0, (1, 0, 1)),
    "a line": (500, 1.0, 0.0, (0, 0, 1)),
    "a point": (7, 0.0, 2.0, (1, 1, 1)),
    "tiny extent": (1000, 1e-30, 0.0, (1, 1, 1)),
    "subnormal extent": (64, 1e-40, 0.0, (1, 1, 1)),
    "huge extent": (1000, 1e37, 0.0, (1, 1, 1)),
    "thin": (3000, 1.0, 0.0, (1, 1e-4, 1e-7)),
}


@pytest.mark.parametrize("form", FORMS)
def test_records_contain_their_boxes(form):
    n, size, shift, axes = FORMS[form]
    rng = np.random.default_rng(5)
    c = rng.uniform(-1, 1, (n, 1, 3))
    v = (c + rng.uniform(-0.05, 0.05, (n, 3, 3))) * np.array(axes) * size + shift
    rep = cr.cr_debug_bvh_check(v.astype(np.float32).reshape(n, 9), cr.CR_BVH2)
    assert rep["covered2"] == n and rep["violations2"] == 0
