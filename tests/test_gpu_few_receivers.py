"""How few receivers are split over the GPU changes no result: narrow tiles of
the field kernels, and path lists whose candidates the warps of a block share.
A call for part of the receivers gives the bits of a call for all of them."""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def creep():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_10578_gb300 import creep as c
    c.load()
    return c


def _room(kind):
    sc = scenes.room(n_cyl=33 if kind == "many" else 5, nx=1, ny=1, freqs=np.linspace(2e9, 28e9, 5), seed=6)
    if kind == "mixed":
        for k in range(0, 5, 2):
            sc.bodies[k] = [scenes.BODY_SPHERE, sc.bodies[k, 1], sc.bodies[k, 2], 0.9, sc.bodies[k, 4], 0.0]
    rng = np.random.default_rng(4)
    n = 60011
    sc.rx = np.stack([rng.uniform(0.1, 9.9, n), rng.uniform(0.1, 7.9, n), rng.uniform(0.3, 2.7, n)], 1).astype(np.float32)
    sc.rx[7] = sc.bodies[1, 1:4] + [0.0, 0.0, 0.3]                       # inside a body
    return sc


@pytest.mark.parametrize("kind,prec", [("many", 0), ("mixed", 0), ("mixed", 1)])
def test_part_of_the_receivers(creep, kind, prec):
    sc = _room(kind)
    S = creep.Scene.from_scene(sc)
    rx = torch.tensor(sc.rx_soa(), device="cuda")
    opts = creep.options(max_order=2, precision=prec)
    n = sc.n_rx if prec == 0 else 7001
    rx = rx[:, :n].contiguous()
    E = S.evaluate(rx, opts=opts)
    codes, counts, fl = S.paths(rx, cap=64, opts=opts)
    for lo, m in ((0, 1), (5, 9), (100, 31), (40, 33), (1000, 97), (17, 1217), (0, 5000)):
        part = rx[:, lo:lo + m].contiguous()
        assert torch.equal(S.evaluate(part, opts=opts), E[:, :, lo:lo + m]), (lo, m)
        c, k, f = S.paths(part, cap=64, opts=opts)
        assert torch.equal(k, counts[lo:lo + m]) and torch.equal(f, fl[lo:lo + m]), (lo, m)
        slot = torch.arange(64, device="cuda")[None] < k[:, None]
        assert torch.equal(c[slot], codes[lo:lo + m][slot]), (lo, m)
        Ep, cp, kp, _ = S.evaluate_with_paths(part, cap=64, opts=opts)
        if prec == 0:
            assert torch.equal(Ep, E[:, :, lo:lo + m]) and torch.equal(kp, k)
            assert torch.equal(torch.where(slot, cp, -1).sort(1)[0], torch.where(slot, c, -1).sort(1)[0])


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n_cyl,tilt,enc", [(1, True, 0), (9, False, 2), (40, True, 1), (130, False, 0)])
def test_wall_creep_turned_room(creep, n_cyl, tilt, enc, prec):
    """The wall -> creeping masks where no wall is along an axis, with an oblique
    face, with more than one mask word, and with too many pairs for them:
    path lists equal to the oracle's, fields within the parity bound."""
    from oracle import oracle
    from parity import compare_fields, compare_paths, gpu_fields
    sc = scenes.room(n_cyl=n_cyl, nx=13, ny=9, seed=20 + n_cyl, freqs=(5.8e9,))
    t = 0.5
    R = np.array([[np.cos(t), -np.sin(t), 0.0], [np.sin(t), np.cos(t), 0.0], [0.0, 0.0, 1.0]])
    tri = np.asarray(sc.tri, np.float64).reshape(-1, 3, 3) @ R.T
    face = list(np.asarray(sc.tri_face).reshape(-1))
    if tilt:
        panel = np.array([[3.0, 0.2, 2.9], [7.0, 0.2, 2.9], [5.0, 1.1, 2.2]]) @ R.T
        tri, face = np.concatenate([tri, panel[None]]), face + [max(face) + 1]
    b = np.array(sc.bodies, np.float64)
    b[:, 1:4] = b[:, 1:4] @ R.T
    b[:, 4] *= 0.9                                       # (turned centres are rounded: no two touch)
    rx = (np.asarray(sc.rx, np.float64) @ R.T).astype(np.float32)
    sc = scenes.Scene(tri.astype(np.float32), np.asarray(face), b, (np.asarray(sc.tx) @ R.T).astype(np.float32), sc.pol,
                      sc.freqs, rx, "turned room", max_order=1)
    sc.wall_creep, sc.max_enc = True, enc
    opts = creep.options(max_order=1, precision=prec, enable=creep.RT_EN_ALL | creep.RT_EN_WALL_CREEP, max_encirclements=enc)
    S = creep.Scene.from_scene(sc)
    d = torch.tensor(sc.rx_soa(), device="cuda")
    E = S.evaluate(d, opts=opts)
    codes, counts, _ = S.paths(d, cap=1024, opts=opts)
    ref = oracle.evaluate(sc)
    compare_paths(codes, counts, ref)
    compare_fields(gpu_fields(E), ref, flags=ref.flags, freqs=sc.freqs)
    assert sum(1 for cs in ref.paths for c in cs if (int(c) >> 56) in (6, 7)) > 20
