"""The BVH build where the centroids' spread on an axis has no finite
reciprocal, or overflows: the launch over it finds the oracle's brute-force
list.  rt_scene_create takes every finite vertex."""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes


def _mesh(z, n=200):
    rng = np.random.default_rng(3)
    tri = rng.uniform(-5, 5, (n, 3, 3)).astype(np.float32)
    tri[..., 2] = z(rng, (n, 3))
    return tri.reshape(n, 9), np.arange(n, dtype=np.int32) // 4


MESHES = {
    "smallest normals": lambda rng, s: rng.choice(np.asarray([0, 1e-38, 2e-38], np.float32), s),
    "denormals": lambda rng, s: rng.choice(np.asarray([0, 1e-45, 3e-42, 1e-40], np.float32), s),
    "overflowing spread": lambda rng, s: rng.choice(np.asarray([-3e38, 3e38], np.float32), s),
    "overflowing centroids": lambda rng, s: np.where(rng.uniform(size=(s[0], 1)) < 0.5, np.float32(3e38),
                                                     rng.uniform(-1, 1, s).astype(np.float32)),
    "all overflow": lambda rng, s: np.full(s, 3e38, np.float32),
}


@pytest.mark.parametrize("name", sorted(MESHES))
def test_launch_over_extreme_spreads(name, oracle_mod):
    from paper_2310_10578_gb300 import creep
    tri, face = _mesh(MESHES[name])
    tx = np.asarray([0.13, 0.21, 0.17], np.float32)
    sc = scenes.Scene(tri, face, np.zeros((0, 6)), tx, (0, 0, 1), [1e9], np.zeros((1, 3)), name)
    np.testing.assert_array_equal(creep.candidates_mesh(tri, face, tx, 500, 3), oracle_mod.candidates(sc, 500, 3))
