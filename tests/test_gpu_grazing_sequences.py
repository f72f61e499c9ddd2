"""The candidate list's culling per tile with the source and the receivers a
fraction of a millimetre before a plane (the scenes of
test_gpu_grazing_planes): a crossing point's FP32 rounding is then centimetres,
and culling has to keep every sequence that FP64 finds.  Each receiver comes 32
times, so that a tile's box is one point and culls the most it can."""
import numpy as np
import pytest

from parity import compare_fields, compare_paths, gpu_fields
from test_gpu_grazing_planes import WANT, _scene

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mesh", [False, True])
@pytest.mark.parametrize("h", [1.5e-4, 3e-4, 1e-3])
@pytest.mark.parametrize("kind", ["one", "then far", "far first"])
def test_culled_sequences(oracle_mod, kind, h, mesh):
    from paper_2310_10578_gb300 import creep
    sc = _scene(kind, h, mesh)
    seq = [[0, -1, -1]] if kind == "one" else [[0, -1, -1], [1, -1, -1], [0, 1, -1], [1, 0, -1]]
    sc.candidates = np.asarray(seq, np.int32)
    ref = oracle_mod.evaluate(sc)
    want = WANT[kind]
    on = np.sum(np.concatenate(ref.paths) == np.uint64(want[0] << 56 | want[1] << 28 | want[2]))
    assert 100 < on < len(sc.rx) - 100
    S = creep.Scene.from_scene(sc)
    opts = creep.options(max_order=2, precision=creep.RT_PREC_FP64)
    rx = torch.tensor(sc.rx_soa(), device="cuda").repeat_interleave(32, 1)
    E = S.evaluate(rx, opts=opts)[:, :, ::32]
    codes, counts, _ = S.paths(rx, opts=opts)
    compare_paths(codes[::32], counts[::32], ref)
    compare_fields(gpu_fields(E), ref, flags=ref.flags, freqs=sc.freqs)
