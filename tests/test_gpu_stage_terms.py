"""Which rays the adjoint may reverse without their stage terms: steps of eight cells with a layer
between a step's middle and its end, which the difference of the first two stages does not see."""
import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from helpers import with_camera
from test_gpu_march import SAME_POINT
from test_gpu_reverse import GRAD_REL_L2, gradient_error

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def layer(after, n=32, steps=4, slope=0.02):
    """A gradient of eta across the rays (along x) from node `after` + 1 on, none before: the first
    two stages of every step lie on the same side."""
    sc = S.blob_cube(n=n, width=23, height=19, steps=steps)
    # nearly parallel rays: along x the index changes by less than SAME_POINT allows
    sc = with_camera(sc, fx=3000.0, fy=3000.0)
    g = sc.grid
    x = (np.arange(n) + 0.5) / n - 0.5
    on = (np.arange(n) > after).astype(np.float64)
    K = g.rho0 * g.G * g.T0
    eta0 = K / g.T0
    g = g.__class__(**{**g.__dict__, "G": g.G * 0.04 / eta0})           # deta = 0.04 at T0
    T = g.T0 / (1.0 + (slope / 0.04) * on[:, None] * x[None, :])
    # stage points of a step are steps of n / (2 steps) cells apart; the nodes of the start's and the
    # middle's cells are on one side, those of the end's on the other
    u = np.arange(2 * steps + 1) * n / (2 * steps) - 0.5
    near = [set(range(min(max(int(np.floor(v)), 0), n - 2), min(max(int(np.floor(v)), 0), n - 2) + 2)) for v in u]
    k = next(i for i in range(1, 2 * steps, 2) if max(near[i]) < after and min(near[i + 1]) > after)
    assert not any({after, after + 1} & near[i] for i in range(k + 1))
    # taking the one acceleration for the other moves the second stage's point by this much
    assert slope / (24.0 * steps ** 2) * n > 100 * SAME_POINT
    return sc.replace(grid=g, T=np.broadcast_to(T, (n, n, n)).astype(np.float32), light=S.Light(0, S.smooth_pattern(64, 64, 3)))


@pytest.mark.parametrize("after", [5, 13, 21, 29])
def test_layer_between_mid_step_and_step_end(bos, orc, after):
    assert gradient_error(bos, orc, layer(after), bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2
