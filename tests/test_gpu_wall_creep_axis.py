"""Wall -> creeping rays round spheres near the axis through a face's source
image, where the frame of source, centre and receiver is ill-conditioned in
FP32: decided in FP64, lists equal to the oracle's."""
import numpy as np
import pytest

from parity import compare_fields, compare_paths, gpu_fields
from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("enc", [0, 1])
def test_receivers_near_the_image_axes(oracle_mod, enc, prec):
    from paper_2310_10578_gb300 import creep
    sc = scenes.room(n_cyl=0, nx=1, ny=1, freqs=(5.8e9,), seed=5)
    ctr = np.asarray([[3.1, 4.2, 1.4], [6.3, 2.9, 1.1], [7.9, 6.1, 1.7]])
    sc.bodies = np.asarray([[scenes.BODY_SPHERE, *p, 0.35, 0.0] for p in ctr], np.float32)
    tx = np.asarray(sc.tx, np.float64)
    images = [tx * [1, 1, -1], tx * [1, 1, -1] + [0, 0, 6], tx * [-1, 1, 1], tx * [-1, 1, 1] + [20, 0, 0],
              tx * [1, -1, 1], tx * [1, -1, 1] + [0, 16, 0]]
    rng = np.random.default_rng(enc)
    rx = []
    for I in images:
        for p in ctr:
            d = (p - I) / np.linalg.norm(p - I)
            for t in rng.uniform(0.5, 1.6, 60):
                off = np.cross(d, rng.standard_normal(3))
                rx.append(p + d * t + off / np.linalg.norm(off) * t * 10 ** rng.uniform(-5, -3.1))
    rx = np.asarray(rx)
    rx = rx[np.all((rx > 0.05) & (rx < [9.95, 7.95, 2.95]), axis=1)]
    sc.rx = rx.astype(np.float32)
    sc.wall_creep, sc.max_enc, sc.max_order = True, enc, 1
    ref = oracle_mod.evaluate(sc)
    S = creep.Scene.from_scene(sc)
    opts = creep.options(max_order=1, precision=prec, max_encirclements=enc, enable=creep.RT_EN_ALL | creep.RT_EN_WALL_CREEP)
    d = torch.tensor(sc.rx_soa(), device="cuda")
    E = S.evaluate(d, opts=opts)
    codes, counts, _ = S.paths(d, opts=opts)
    compare_paths(codes, counts, ref)
    _, codes, counts, _ = S.evaluate_with_paths(d, opts=opts)
    compare_paths(codes, counts, ref)
    compare_fields(gpu_fields(E), ref, flags=ref.flags, freqs=sc.freqs)
    assert sum(1 for cs in ref.paths for c in cs if (int(c) >> 56) in (6, 7)) > 200
