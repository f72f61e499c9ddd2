"""The BVH's splits on meshes where a plane split degenerates: nested boxes
(all centroids alike per side), a long row, one huge shell among tiny boxes.
The ray launch over the BVH has to find the oracle's brute-force list."""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes


def _boxes(spec):
    tri, face = [], []
    for k, b in enumerate(spec):
        t, f = scenes.box_mesh(*b, 6 * k)
        tri += t
        face += f
    return np.asarray(tri, np.float32).reshape(-1, 9), np.asarray(face, np.int32)


MESHES = {
    "nested": [(-r, r, -r, r, -r, r) for r in 1.0 + 0.37 * np.arange(20)],
    "row": [(3.0 * k + 1, 3.0 * k + 2, -1, 1, -1, 1) for k in range(40)],
    "shell": [(-90, 95, -70, 80, -1, 3)] + [(0.5 * k, 0.5 * k + 0.1, 1, 1.1, 0, 0.1) for k in range(30)],
    "copies": [(1, 2, 1, 2, 0, 1)] * 3 + [(-5, 5, -5, 5, -2, 2)],
}


@pytest.mark.parametrize("name", sorted(MESHES))
def test_launch_over_degenerate_splits(name, oracle_mod):
    from paper_2310_10578_gb300 import creep
    tri, face = _boxes(MESHES[name])
    tx = np.asarray([0.13, 0.21, 0.17], np.float32)
    sc = scenes.Scene(tri, face, np.zeros((0, 6)), tx, (0, 0, 1), [1e9], np.zeros((1, 3)), name)
    np.testing.assert_array_equal(creep.candidates_mesh(tri, face, tx, 500, 3), oracle_mod.candidates(sc, 500, 3))
