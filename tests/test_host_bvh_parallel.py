"""The BVH build of meshes large enough to be built by several threads: the
launch over it finds the oracle's brute-force list, also when callers build at
the same time."""
import concurrent.futures

import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes


@pytest.mark.parametrize("furn", [20, 45, 260])
def test_launch_over_a_large_mesh(furn, oracle_mod):
    from paper_2310_10578_gb300 import creep
    sc = scenes.office(n_rooms=(4, 3), n_furn=furn, n_cyl=1, n_sph=1, n_tx=1, nx=1, ny=1, seed=furn)
    tri = np.ascontiguousarray(sc.tri.reshape(-1, 9))
    want = oracle_mod.candidates(sc, 150, 3)
    with concurrent.futures.ThreadPoolExecutor(6) as ex:
        for got in ex.map(lambda _: creep.candidates_mesh(tri, sc.tri_face, sc.tx, 150, 3), range(12)):
            np.testing.assert_array_equal(got, want)
