"""The reversing adjoint on rays of more than 2^20 steps, whose line is set up anew on the way: the
ray enters in a far cell of another brick and ends in cell (0, 0, 0) or beside it, so that a cell
or a brick kept from before the set-up would be taken for the new one."""
import dataclasses

import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# N float32 additions of half an ulp each at most, all of one sign: N 2^-25 of the sum.  Two sums
# follow one another (a ray's adjoint, and the sensitivities of a cell's corners).
def bound(N):
    return 2 * N * 2.0 ** -25


def backwards(cell, steps, integrator, gain):
    """A cube of 20^3 cells seen along -y before a smooth wall at y = 0, an index field `gain` times
    air's; the rays end in the column of cells `cell` (x, z)."""
    h = 1.0 / 20.0
    x, z = ((c + 0.5) * h for c in cell)
    sc = S.blob_cube(n=20, width=2, height=2, steps=steps)
    T = S.blob_field(sc.grid, np.array([x + 0.12, 0.1, z + 0.09]), 0.2, 8.0)
    cam = dataclasses.replace(sc.camera, pos=(x, 2.5, z), fwd=(0.0, -1.0, 0.0), up=(0.0, 0.0, 1.0), fx=400.0, fy=400.0,
                              cx=1.0, cy=1.0)
    wall = dataclasses.replace(sc.wall, origin=(0.0, 0.0, 0.0), normal=(0.0, -1.0, 0.0))
    return sc.replace(T=T, camera=cam, wall=wall, light=S.Light(0, S.smooth_pattern(64, 64, 3)),
                      grid=dataclasses.replace(sc.grid, G=gain * sc.grid.G),
                      integ=dataclasses.replace(sc.integ, integrator=integrator, ckpt_every=64))


@pytest.mark.parametrize("integrator", [0, 2])
@pytest.mark.parametrize("cell,extra,gain", [((0, 0), 37, 1.0), ((0, 0), 1 << 16, 1.0), ((3, 1), 37, 800.0)])
def test_gradient_across_line_changes(orc, cell, extra, gain, integrator):
    from paper_2509_14442_gb300 import bos

    N = (1 << 20) + extra
    sc = backwards(cell, N, integrator, gain)
    w = np.random.default_rng(8).standard_normal((2, 2)).astype(np.float32)
    ctx = bos.Context(0)
    ctx.set_scene(sc, bos.BOS_PREC_FP32_COMP)
    ctx.render(save_for_backward=True)
    g = ctx.backward(torch.as_tensor(w, device="cuda")).cpu().numpy().astype(np.float64)
    ctx.status()
    ctx.close()
    ref = orc.grad(sc, w.astype(np.float64))
    for part in (slice(None), slice(0, 1)):      # the whole field; the layer in which the rays end
        a, b = g[:, part], ref[:, part]
        assert np.linalg.norm(b) > 0
        assert np.linalg.norm(a - b) <= bound(N) * np.linalg.norm(b), part
