"""A NaN temperature: a ray that meets it has NaN sensitivities from there back to the cell where
it enters the grid, not in some other cell."""
import dataclasses

import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("light", ["texture", "refracted"])
@pytest.mark.parametrize("prec", ["FP32_COMP", "BF16_COMP"])
def test_nan_reaches_the_entry_cells(prec, light):
    from paper_2509_14442_gb300 import bos

    if light == "texture":
        sc = S.blob_cube(n=16, width=40, height=33, steps=48)
    else:
        sc = S.room((20, 18, 16), 40, 33, 1, 6400)
        sc = sc.replace(light=S.Light(2, sc.light.pattern, sc.light.proj, connect_iters=1))
    # (a checkpoint on the way would give the reversal a finite state again)
    sc = sc.replace(integ=dataclasses.replace(sc.integ, ckpt_every=64))
    n, o, h, c = np.array(sc.grid.n), np.array(sc.grid.origin), np.array(sc.grid.spacing()), sc.camera
    hot = n // 2
    T = np.array(sc.T)
    T[hot[2], hot[1], hot[0]] = np.nan
    ctx = bos.Context(0)
    ctx.set_scene(sc.replace(T=T), getattr(bos, "BOS_PREC_" + prec))
    I, _, _ = ctx.render(save_for_backward=True)
    g = ctx.backward(torch.ones_like(I)).cpu().numpy()
    ctx.status()
    ctx.close()
    # camera rays that pass within 0.4 cells of the node, and the cells in which they enter (y face)
    assert c.fwd == (0.0, 1.0, 0.0) and c.up == (0.0, 0.0, 1.0)
    py, px = np.mgrid[0:c.height, 0:c.width]
    d = np.stack([(px + 0.5 - c.cx) / c.fx, np.ones(px.shape), -(py + 0.5 - c.cy) / c.fy], -1).reshape(-1, 3)
    pos = np.array(c.pos)
    at = lambda y: (pos + (y - pos[1]) * d - o) / h - 0.5
    meets = (np.abs(at(o[1] + (hot[1] + 0.5) * h[1]) - hot) < 0.4).all(1)
    u = at(o[1])
    i = np.clip(np.floor(u).astype(int), 0, n - 2)
    clear = (np.abs(u - np.floor(u) - 0.5)[:, [0, 2]] < 0.45).all(1)      # not on a face of the entry cell
    assert (meets & clear).any()
    for x, y, z in i[meets & clear]:
        assert np.isnan(g[z, y, x]), (x, y, z)
