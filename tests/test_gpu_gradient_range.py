"""The stencil transpose at the end of float32's range: sums that overflow end as infinities of the
right sign, all others stay what they are."""
import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from test_gpu_reverse import GRAD_REL_L2

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

MAX = float(np.finfo(np.float32).max)


def test_overflowing_sums_are_infinite():
    from paper_2509_14442_gb300 import bos

    sc = S.blob_cube(n=8, width=256, height=256, steps=24)
    sc = sc.replace(light=S.Light(0, S.smooth_pattern(64, 64, 3)))
    ctx = bos.Context(0)
    ctx.set_scene(sc, bos.BOS_PREC_FP32_COMP)
    I, _, _ = ctx.render(save_for_backward=True)
    g = ctx.backward(torch.ones_like(I)).cpu().numpy().astype(np.float64)
    # the sums before d deta / dT = -K / T^2, and a seed that takes the largest to 1.5 of the range
    # (the accumulators, which the stencil divides by 2 h = 1/4, to at most half of it)
    factor = -(sc.grid.rho0 * sc.grid.G * sc.grid.T0) / sc.T.astype(np.float64) ** 2
    tot = g / factor
    seed = float(np.float32(1.5 * MAX / np.abs(tot).max()))
    assert seed < 0.01 * MAX
    big = ctx.backward(torch.full_like(I, seed)).cpu().numpy()
    ctx.status()
    ctx.close()
    tot = tot * seed
    slack = GRAD_REL_L2 * np.abs(tot).max()          # two sums of the same terms in another order
    over, under = np.abs(tot) > MAX + slack, np.abs(tot) < MAX - slack
    assert over.sum() > 0 and under.sum() > 0.5 * tot.size
    assert np.array_equal(big[over], np.sign(g[over]) * np.inf)
    assert np.isfinite(big[under]).all()
    assert np.abs(big[under] / factor[under] - tot[under]).max() <= slack
