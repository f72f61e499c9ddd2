"""Scenes with a BVH at the edges of their culling: bodies that walls hide from
the transmitter, sequences that no receiver of a tile can take, walks shared
by a warp with one receiver, a partial tile, receivers in no order.  Path lists
are equal to the oracle's, fields within the parity bound."""
import numpy as np
import pytest

from parity import compare_fields, compare_paths, gpu_fields
from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(creep, oracle_mod, sc, order, prec):
    S = creep.Scene.from_scene(sc)
    opts = creep.options(max_order=order, precision=prec)
    rx = torch.tensor(sc.rx_soa(), device="cuda")
    E = S.evaluate(rx, opts=opts)
    codes, counts, _ = S.paths(rx, opts=opts)
    ref = oracle_mod.evaluate(sc)
    compare_paths(codes, counts, ref)
    compare_fields(gpu_fields(E), ref, flags=ref.flags, freqs=sc.freqs)
    return ref


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n_rx", [1, 31, 33, 700])
def test_hidden_bodies_and_culled_sequences(oracle_mod, n_rx, prec):
    from paper_2310_10578_gb300 import creep
    sc = scenes.office(n_rooms=(4, 3), n_furn=60, n_cyl=37, n_sph=4, n_tx=1, nx=1, ny=1, seed=90 + n_rx)
    rng = np.random.default_rng(n_rx)
    sc.rx = np.stack([rng.uniform(0.1, 19.9, n_rx), rng.uniform(0.1, 11.9, n_rx), rng.uniform(0.3, 2.9, n_rx)],
                     axis=1).astype(np.float32)
    if n_rx < 64:                                        # some of them in the transmitter's room
        sc.rx[::2, :2] = sc.tx[:2] + rng.uniform(-1.5, 1.5, (len(sc.rx[::2]), 2)).astype(np.float32)
    sc.candidates = oracle_mod.candidates(sc, 2048, 3)
    ref = _check(creep, oracle_mod, sc, 3, prec)
    assert ref.counts.sum() > 0


@pytest.mark.parametrize("prec", [0, 1])
def test_bvh_with_enumerated_faces(oracle_mod, prec):
    """The room with each wall cut into 16 triangles: a BVH, no polygons, and
    every face pair enumerated."""
    from paper_2310_10578_gb300 import creep
    sc = scenes.room(n_cyl=9, nx=19, ny=13, seed=12)
    tri, face = [], []
    for t, f in zip(sc.tri, sc.tri_face):
        a = [t]
        for _ in range(3):
            a = [x for v in a for x in ([v[0], (v[1] + v[2]) / 2, v[2]], [v[0], v[1], (v[1] + v[2]) / 2])]
            a = [np.asarray([v[1], v[2], v[0]], np.float32) for v in a]
        tri += a
        face += [f] * len(a)
    sc = scenes.Scene(np.asarray(tri), np.asarray(face), sc.bodies, sc.tx, sc.pol, sc.freqs, sc.rx, "cut room")
    assert len(sc.tri) > 64
    _check(creep, oracle_mod, sc, 2, prec)
