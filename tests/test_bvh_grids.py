"""The BVH2 records where detail is small against the scene: subtrees take grids of their own, so that the
records cull as the exact boxes do (node visits and triangle tests within a tenth of theirs) and
still contain them."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2310_07182_gb300 import binding as cr
from paper_2310_07182_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = next((d for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda")
             if d and os.path.exists(os.path.join(d, "include", "cuda_runtime.h"))), None)


@pytest.mark.skipif(CUDA is None or shutil.which("g++") is None, reason="no g++ or CUDA headers")
def test_visits_are_those_of_the_exact_boxes(tmp_path):
    exe = str(tmp_path / "visits")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", build.INCLUDE, "-I", build.CSRC, "-I",
                    os.path.join(CUDA, "include"), os.path.join(build.CSRC, "bvh_build.cpp"),
                    os.path.join(HERE, "helpers", "bvh_visits_main.cpp"), "-o", exe, "-lpthread"], check=True)
    out = subprocess.run([exe, "100000", "500"], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 10
    for name, n, grids, nodes, nodes_rec, tris, tris_rec in rows:
        assert float(nodes_rec) <= 1.1 * float(nodes) and float(tris_rec) <= 1.1 * float(tris), (name, nodes, nodes_rec, tris, tris_rec)
        assert name in ("even", "ground5") or int(grids) > 1


def _clusters(seed, n, smallest, far):
    """Clusters of triangles whose sizes span the scales from `smallest` to 1, the centre of each near one of the
    next larger cluster's triangles; moved by `far`."""
    rng = np.random.default_rng(seed)
    out, centre = [], np.zeros(3)
    for size in np.geomspace(1.0, smallest, 8):
        c = centre + rng.uniform(-1, 1, (n, 1, 3)) * size
        out.append(c + rng.uniform(-0.03, 0.03, (n, 3, 3)) * size)
        centre = out[-1][rng.integers(n), 0]
    return (np.concatenate(out) + far).astype(np.float32).reshape(-1, 9)


@pytest.mark.parametrize("smallest", [1e-2, 1e-7, 1e-14, 1e-30])
@pytest.mark.parametrize("far", [0.0, 1e3])
@pytest.mark.parametrize("seed", [1, 2])
def test_records_contain_their_boxes_in_every_grid(smallest, far, seed):
    v = _clusters(seed, 700, smallest, far)
    rep = cr.cr_debug_bvh_check(v, cr.CR_BVH2)
    assert rep["covered2"] == len(v) and rep["violations2"] == 0


@pytest.mark.parametrize("scale", [1e-20, 1e20, 1e36])
def test_records_contain_their_boxes_at_any_size(scale):
    v = (_clusters(3, 500, 1e-9, 0.0).astype(np.float64) * scale).astype(np.float32)
    rep = cr.cr_debug_bvh_check(v, cr.CR_BVH2)
    assert rep["covered2"] == len(v) and rep["violations2"] == 0
