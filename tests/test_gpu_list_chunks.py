"""Fields with path lists at more frequencies than one planar launch takes:
each path is listed once, as rt_paths lists it."""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nf,chunks", [(16, 4), (17, 4), (33, 4), (5, 1), (64, 4)])
@pytest.mark.parametrize("cand", [False, True])
def test_listed_once(nf, chunks, cand):
    from paper_2310_10578_gb300 import creep
    sc = scenes.room(n_cyl=5, nx=11, ny=9, freqs=np.linspace(2e9, 28e9, nf), seed=8)
    S = creep.Scene.from_scene(sc)
    if cand:
        S.candidates_device(1000, 2)
    p, b, _ = S.shape()
    S.set_shape(p, b, chunks)
    rx = torch.tensor(sc.rx_soa(), device="cuda")
    codes, counts, _ = S.paths(rx, cap=96)
    _, c, k, _ = S.evaluate_with_paths(rx, cap=96)
    assert torch.equal(k, counts)
    slot = torch.arange(96, device="cuda")[None] < k[:, None]
    assert torch.equal(torch.where(slot, c, -1).sort(1)[0], torch.where(slot, codes, -1).sort(1)[0])
