"""The device ray launch against the host one at the sizes where its split can
go wrong: fewer rays than a block's warps, ray counts that are no multiple of
them, the largest launch, one to three bounces, a scene below the BVH's size.
The lists are face indices: they are equal, not close."""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rays,order", [(1, 1), (1, 3), (3, 2), (33, 3), (1023, 1), (8192, 2), (5461, 3)])
@pytest.mark.parametrize("small", [True, False])
def test_device_list_equals_host_list(n_rays, order, small):
    from paper_2310_10578_gb300 import creep
    sc = (scenes.room(n_cyl=2, nx=2, ny=2) if small else
          scenes.office(n_rooms=(3, 2), n_furn=90, n_cyl=3, n_sph=1, n_tx=1, nx=4, ny=4, seed=71))
    S = creep.Scene.from_scene(sc)
    S.candidates_device(n_rays, order)
    np.testing.assert_array_equal(S.get_candidates(), S.candidates(n_rays, order))
    S.candidates_device(n_rays, order)          # again into the same buffers
    np.testing.assert_array_equal(S.get_candidates(), S.candidates(n_rays, order))
