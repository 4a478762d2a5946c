"""The cell-marching Sharma tracer (renders without checkpoints) against the FP64 oracle at
the sizes where its shortcuts could go wrong: cells that are never left or always
extrapolated, many half steps per cell, uneven cells, rays that cross cells along every
axis, steep fields in which a step's last point and the next step's first one are distinct
points, and step counts beyond the length of one line set-up."""
import dataclasses

import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from helpers import DISP_REL_TOL, I_ABS_TOL, bf16_round, errors, gpu_render, with_camera

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SAME_POINT = 2.0 ** -24     # cells: the tracer's bound for taking two stage points as one


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def steep(n=16, steps=12, gain=40.0):
    """Few steps through a blob whose index field is `gain` times air's."""
    sc = S.blob_cube(n=n, width=45, height=38, steps=steps)
    g = dataclasses.replace(sc.grid, G=sc.grid.G * gain)
    de = g.rho0 * g.G * g.T0 / sc.T.astype(np.float64)
    h = g.extent[0] / n
    grad = np.gradient(de, h)
    # a - b = (dt^2 / 6) (D(p1) - D(p2)), half a step apart along y
    along_y = max(np.abs(np.diff(d, axis=1)).max() for d in grad) / h * (0.5 / steps)
    assert (1.0 / steps) ** 2 / 6.0 * along_y / h > 10 * SAME_POINT
    return sc.replace(grid=g)


def diagonal():
    """A wide view from a corner: rays cross cells along all three axes."""
    sc = S.blob_cube(n=21, width=53, height=47, steps=64)
    f, r = np.array([0.5, 0.75, 0.0]), None
    f[2] = -np.sqrt(1.0 - (f ** 2).sum())
    r = np.cross(f, [0.0, 0.0, 1.0])
    r /= np.linalg.norm(r)
    up = np.cross(r, f)
    return with_camera(sc, pos=(-0.4, -0.7, 1.3), fwd=tuple(f), up=tuple(up), fx=60.0, fy=60.0)


SCENES = {
    "two_cells": lambda: S.blob_cube(n=2, width=19, height=17, steps=9),
    "fine_steps": lambda: S.blob_cube(n=16, width=24, height=20, steps=3000),
    "uneven_cells": lambda: S.room((97, 31, 13), 83, 61, 2, 6101),
    "three_samples": lambda: S.room((40, 36, 30), 61, 47, 3, 6102),
    "diagonal": diagonal,
    "steep": steep,
    "long_line": lambda: S.blob_cube(n=4, width=3, height=2, steps=(1 << 20) + 37),
}


@pytest.mark.parametrize("light", ["plain", "refracted"])
@pytest.mark.parametrize("name", sorted(SCENES))
def test_march_matches_oracle(bos, orc, name, light):
    sc = SCENES[name]()
    if light == "refracted":
        if sc.light.mode == 0:
            pytest.skip("the refracted connection needs a projector")
        sc = sc.replace(light=S.Light(2, sc.light.pattern, sc.light.proj, connect_iters=1))
    o = orc.render(sc, nsteps=True)
    g = gpu_render(sc, bos.BOS_PREC_FP32_COMP)
    assert light == "refracted" or g["steps"] == int(o["nsteps"].sum())
    e = errors(g, o)
    assert e["disp_max"] > 0 and e["disp_rel"] <= DISP_REL_TOL and e["I_abs"] <= I_ABS_TOL, e


@pytest.mark.parametrize("name", ["steep", "uneven_cells"])
def test_march_bf16_matches_oracle_on_the_bf16_field(bos, orc, name):
    sc = SCENES[name]()
    de = orc.deta_from_T(sc.grid, sc.T.astype(np.float64))
    field = orc.NodeField(bf16_round(de), bf16_round(orc.grad_from_deta(sc.grid, de)))
    e = errors(gpu_render(sc, bos.BOS_PREC_BF16_COMP), orc.render(sc, field=field))
    assert e["disp_max"] > 0 and e["disp_rel"] <= DISP_REL_TOL and e["I_abs"] <= I_ABS_TOL, e
