"""The adjoint kernel's units: paths of many receivers are sorted by kind, a
window of each list at a time.  A path's contribution does not depend on the
unit it falls in, so the gradient of all receivers is the sum of the
gradients of parts of them, and a list repeated k times gives k times the
gradient.

Tolerance: only the order of FP64 sums differs.  N terms sum to within
N 2^-53 of the sum of their magnitudes; N <= 1.2e6 here, 1.3e-10, and the
magnitudes of a part's gradient may be 10 times less than those of its terms.
"""
import numpy as np
import pytest

from paper_2310_10578_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = 2e-9


@pytest.mark.parametrize("n,fp64,rep", [(1, True, 1), (33, False, 9), (457, True, 3), (915, False, 2),
                                        (14592 + 37, False, 4), (14592 + 37, True, 1)])
def test_parts_sum_to_the_whole(n, fp64, rep):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_10578_gb300 import creep
    sc = scenes.room(n_cyl=3, nx=1, ny=1, freqs=np.asarray([2.4e9, 5.8e9, 10e9, 17e9, 28e9]), seed=3)
    rng = np.random.default_rng(n)
    sc.rx = np.stack([rng.uniform(0.1, 9.9, n), rng.uniform(0.1, 7.9, n), rng.uniform(0.8, 1.6, n)], 1).astype(np.float32)
    S = creep.Scene.from_scene(sc)
    rx = torch.tensor(sc.rx_soa(), device="cuda")
    codes, counts, _ = S.paths(rx, cap=512)
    gE = torch.tensor(rng.standard_normal((5, 3, n, 2)).astype(np.float32), device="cuda")
    opts = creep.options(precision=creep.RT_PREC_FP64 if fp64 else creep.RT_PREC_FP32)
    m = int(counts.max())
    assert m * rep <= 512
    # receiver r's list rep times over, as far as the longest list's slots go
    slot = torch.arange(512, device="cuda")[None]
    c = counts.long().clamp(min=1)[:, None]
    long_codes = torch.gather(codes, 1, (slot % c).expand(n, -1)).contiguous()
    whole = S.backward(rx, long_codes, (counts * rep).contiguous(), gE, opts=opts)
    tot, mag = [torch.zeros_like(x) for x in whole], [torch.zeros_like(x) for x in whole]
    step = 61 if n < 2000 else 1213
    for i in range(0, n, step):
        part = S.backward(rx[:, i:i + step].contiguous(), codes[i:i + step].contiguous(),
                          counts[i:i + step].contiguous(), gE[:, :, i:i + step].contiguous(), opts=opts)
        for t, a, p in zip(tot, mag, part):
            t += rep * p
            a += rep * p.abs()
    for t, a, w in zip(tot, mag, whole):
        assert torch.all((t - w).abs() <= TOL * a)
