"""Source and receivers millimetres before one plane.  Where the image's segment
crosses the plane is then uncertain by many times the coordinates' rounding
(image to receiver over the distances of both), so that a crossing near a
face's edge needs FP64.  A free-standing panel turned by 0.5 rad, crossings
within 2 cm of its edges: path lists equal to the oracle's."""
import numpy as np
import pytest

from parity import compare_fields, compare_paths, gpu_fields
from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 3000


def _world(p):
    """Local (along the panel, before it, up) to the scene."""
    p = np.asarray(p, np.float64)
    c, s = np.cos(0.5), np.sin(0.5)
    return np.stack([2 + c * p[..., 0] - s * p[..., 1], 1 + s * p[..., 0] + c * p[..., 1], p[..., 2]], axis=-1)


def _quad(q, f):
    q = _world(q)
    return [[q[0], q[1], q[2]], [q[0], q[2], q[3]]], [f, f]


def _receivers(rng, I, Q, h):
    """Receivers 0.5 to 1 times h before the plane, seen from the image I through the points Q."""
    t = rng.uniform(0.5, 1.0, (len(Q), 1))
    return Q + (Q - I) * t


def _edge_points(rng, side):
    """Points on the panel's plane within 2 cm of its edge u = side, or of its top."""
    near = rng.uniform(-0.02, 0.02, N)
    end = np.stack([side + near, np.zeros(N), rng.uniform(0.2, 2.8, N)], axis=1)
    top = np.stack([rng.uniform(-1, 4.9, N), np.zeros(N), 3 + near], axis=1)
    return np.where(rng.uniform(size=(N, 1)) < 0.5, end, top)


def _scene(kind, h, mesh, u0=-3.0):
    rng = np.random.default_rng(int(1e4 * h))
    edge = [5.0, 5.0]
    bodies, tx = np.zeros((0, 6)), [u0, h, 1.3]
    if kind == "wall":
        # the image's tangent ray reaches the cylinder 0.4 h before the panel's
        # plane: it crosses the plane at u, where the panel's end, slanted, is
        u = u0 + (7 - u0) / 1.4
        edge = [u + 0.02, u - 0.02]
        c = _world([7, 0.3 + 0.4 * h, 0])
        bodies = np.asarray([[scenes.BODY_CYLINDER, c[0], c[1], -0.5, 0.3, 4.0]])
    tri, face = _quad([[-5, 0, 0], [edge[0], 0, 0], [edge[1], 0, 3], [-5, 0, 3]], 0)
    if kind == "one":
        rx = _receivers(rng, np.asarray([-3, -h, 1.3]), _edge_points(rng, 5.0), h)
    elif kind == "wall":
        rx = np.stack([rng.uniform(7.2, 9, N), rng.uniform(0.8, 2, N), rng.uniform(-0.4, 3.4, N)], axis=1)
    else:
        # a second panel across the end of the first, u = 9
        t, f = _quad([[9, -2, -3], [9, 4, -3], [9, 4, 9], [9, -2, 9]], 1)
        tri, face = tri + t, face + f
        if kind == "then far":                       # image -> Q1 on the panel -> the far panel -> receiver
            out = 9 + rng.uniform(0.5, 3, (N, 1))
            Q, I = _edge_points(rng, 5.0), np.asarray([-3, -h, 1.3])
            rx = I + (Q - I) * (out - I[0]) / (Q[:, :1] - I[0])
            rx[:, 0] = 18 - rx[:, 0]
        else:                                        # the far panel first, then grazing along the panel
            tx = [7, h, 1.3]
            rx = _receivers(rng, np.asarray([11, -h, 1.3]), _edge_points(rng, 5.0), h)
    if mesh:                                         # a BVH: 72 triangles more, far away, one face
        for k in range(36):
            a = 0.1 * k
            t, f = _quad([[a, 30, 0], [a + 0.1, 30, 0], [a + 0.1, 30, 1], [a, 30, 1]], max(face) + 1 if k == 0 else face[-1])
            tri, face = tri + t, face + f
    sc = scenes.Scene(tri, face, bodies, _world(tx), (0.2, 0.3, 0.9), [2.4e9], _world(rx), "grazing")
    sc.wall_creep = kind == "wall"
    return sc


# (the wall's crossing is one point for all receivers: several sources)
SOURCES = {"wall": (-3.0, -3.4, -2.7, -2.1, -3.9, -2.4)}
WANT = {"one": (1, 0, 0), "then far": (2, 0, 1), "far first": (2, 1, 0), "wall": (7, 0, 0)}


@pytest.mark.parametrize("prec", [1])
@pytest.mark.parametrize("mesh", [False, True])
@pytest.mark.parametrize("h", [1e-3, 5e-3, 1e-2])
@pytest.mark.parametrize("kind", sorted(WANT))
def test_crossings_near_edges(oracle_mod, kind, h, mesh, prec):
    from paper_2310_10578_gb300 import creep
    for u0 in SOURCES.get(kind, (-3.0,)):
        sc = _scene(kind, h, mesh, u0)
        ref = oracle_mod.evaluate(sc)
        want = WANT[kind]
        on = np.sum(np.concatenate(ref.paths) == np.uint64(want[0] << 56 | want[1] << 28 | want[2]))
        assert 100 < on < N - 100                    # some crossings on the panel, some off it
        S = creep.Scene.from_scene(sc)
        opts = creep.options(max_order=2, precision=prec,
                             enable=creep.RT_EN_ALL | (creep.RT_EN_WALL_CREEP if sc.wall_creep else 0))
        rx = torch.tensor(sc.rx_soa(), device="cuda")
        E = S.evaluate(rx, opts=opts)
        codes, counts, _ = S.paths(rx, opts=opts)
        compare_paths(codes, counts, ref)
        if prec == 1:
            compare_fields(gpu_fields(E), ref, flags=ref.flags, freqs=sc.freqs)
