"""The device ray launch over meshes so large that the FP32 filter's products
overflow: its list is the host launch's.  Vertices may be any finite floats."""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e12, 1e14, 1e18])
@pytest.mark.parametrize("boxes", [1, 12])
def test_device_list_equals_host_list(scale, boxes):
    from paper_2310_10578_gb300 import creep
    rng = np.random.default_rng(boxes)
    tri, face = [], []
    for k in range(boxes):
        x, y, z = (0.0, 0.0, 0.0) if k == 0 else rng.uniform(-8, 8, 3)
        r = 10.0 if k == 0 else rng.uniform(0.5, 1.5)
        t, f = scenes.box_mesh(x - r, x + r, y - r, y + r, z - r, z + r, 6 * k)
        tri += t
        face += f
    tri = np.asarray(tri, np.float64).reshape(-1, 3, 3) * scale
    tx = np.asarray([0.13, 0.21, 0.17]) * scale
    sc = scenes.Scene(tri, face, np.zeros((0, 6)), tx, (0, 0, 1), [1e9], np.zeros((1, 3)), "far")
    S = creep.Scene.from_scene(sc)
    want = S.candidates(1500, 3)
    assert len(want) > 20
    S.candidates_device(1500, 3)
    np.testing.assert_array_equal(S.get_candidates(), want)
