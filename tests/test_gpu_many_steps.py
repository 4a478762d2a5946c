"""The quasi-linear adjoint beyond 2^24 steps, where a float32 count of the steps stops growing: a
thin slab whose smallest cell sets 1.5 2^24 steps along its long axis, against the oracle's
gradient in 4096 steps (64 cells: the quadrature's own error is below 1e-6)."""
import dataclasses

import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CELLS = 64


def slab(steps):
    """1 m x 1 m x thin, seen along +y by one pixel; `steps` of 1.01e-3 of its thin cell."""
    thin = 4.0 / (1.01e-3 * steps)
    sc = S.blob_cube(n=4, width=1, height=1)
    grid = dataclasses.replace(sc.grid, n=(8, CELLS, 4), extent=(1.0, 1.0, thin))
    # T falls along x, more steeply at mid-way: a gradient across the ray at every point
    x, y = (np.arange(8) + 0.5) / 8.0, (np.arange(CELLS) + 0.5) / CELLS
    T = 293.0 + 8.0 * x[None, :] * (0.5 + y * (1.0 - y))[:, None]
    cam = dataclasses.replace(sc.camera, pos=(0.45, -1.5, 0.5 * thin), fx=1.0, fy=1.0, cx=0.5, cy=0.5)
    wall = dataclasses.replace(S.back_wall(grid), size_v=1.0, origin=(0.0, 1.0, -0.5))
    return sc.replace(grid=grid, T=np.broadcast_to(T, (4, CELLS, 8)).astype(np.float32), camera=cam, wall=wall,
                      light=S.Light(0, S.smooth_pattern(64, 64, 3)),
                      integ=dataclasses.replace(sc.integ, fixed_steps=0, max_step_vox=1.01e-3, integrator=2))


def test_gradient_beyond_2_to_the_24_steps(orc):
    from paper_2509_14442_gb300 import bos

    N = 3 << 23
    sc = slab(N)
    w = np.ones((1, 1), np.float32)
    ctx = bos.Context(0)
    ctx.set_scene(sc, bos.BOS_PREC_FP32_COMP)
    ctx.render(save_for_backward=True)
    g = ctx.backward(torch.as_tensor(w, device="cuda")).cpu().numpy().astype(np.float64)
    assert ctx.last_ray_steps() > 1.4 * 2 ** 24
    ctx.status()
    ctx.close()
    ref = orc.grad(sc.replace(integ=dataclasses.replace(sc.integ, fixed_steps=4096)), w.astype(np.float64))
    # two float32 sums, a ray's adjoint and a cell's 2 N / CELLS samples: half an ulp per addition
    bound = 2 * (2 * N / CELLS) * 2.0 ** -25
    assert np.linalg.norm(ref) > 0
    assert np.linalg.norm(g - ref) <= bound * np.linalg.norm(ref)
