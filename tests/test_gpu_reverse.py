"""The Sharma adjoint that reverses rays without their stage terms, and its hand-over to the
segment-recomputing kernel, against the FP64 oracle's discrete adjoint: steep fields (every
tile handed over, and some), rays that end far off their lines (states taken from the
checkpoints), edge cells, uneven cells, lanes that loop over samples, and pixel lists."""
import dataclasses

import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from test_gpu_march import SCENES, diagonal, steep

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# float32 rounding over N ~ 500 steps, 2^-24 sqrt(N) ~ 1.3e-6 per node, and the atomics' order
GRAD_REL_L2 = 1e-5


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def bent(K=16):
    """An index field 800 times air's in fine steps: rays end ~3.5 mm (a ninth of a cell) off
    their lines, while a step's stage points stay within 1e-8 cells of one another."""
    sc = S.blob_cube(n=32, width=37, height=29, steps=512)
    return sc.replace(grid=dataclasses.replace(sc.grid, G=800.0 * sc.grid.G),
                      integ=dataclasses.replace(sc.integ, ckpt_every=K))


def partly_steep():
    """A plume 30 times as hot on a coarse grid: tiles through it are handed over, others not."""
    sc = S.room((24, 20, 18), 90, 70, 1, 6201)
    T = (S.T_AMBIENT + 30.0 * (sc.T.astype(np.float64) - S.T_AMBIENT)).astype(np.float32)
    return sc.replace(T=T)


ALL = {
    "steep": steep,
    "partly_steep": partly_steep,
    "diagonal": diagonal,
    "two_cells": SCENES["two_cells"],
    "uneven_cells": SCENES["uneven_cells"],
    "three_samples": SCENES["three_samples"],
    **{f"bent_K{K}": (lambda K=K: bent(K)) for K in (1, 5, 16, 64)},
}


def smooth(sc):
    """The scene before a smooth pattern (a binary one's gradient is a sum over few pixels)."""
    th, tw = sc.light.pattern.shape
    return sc.replace(light=S.Light(sc.light.mode, S.smooth_pattern(tw, th, 3), sc.light.proj, sc.light.connect_iters))


def gradient_error(bos, orc, sc, prec):
    w = np.random.default_rng(8).standard_normal((sc.camera.height, sc.camera.width)).astype(np.float32)
    ctx = bos.Context(0)
    ctx.set_scene(sc, prec)
    ctx.render(save_for_backward=True)
    g = ctx.backward(torch.as_tensor(w, device="cuda")).cpu().numpy().astype(np.float64)
    ctx.status()
    ctx.close()
    ref = orc.grad(sc, w.astype(np.float64))
    assert np.linalg.norm(ref) > 0
    return float(np.linalg.norm(g - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("name", sorted(ALL))
def test_reversed_adjoint_matches_oracle(bos, orc, name):
    assert gradient_error(bos, orc, smooth(ALL[name]()), bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2


@pytest.mark.parametrize("name", ["steep", "diagonal", "two_cells", "uneven_cells", "three_samples", "bent_K16"])
def test_reversed_quasi_linear_adjoint_matches_oracle(bos, orc, name):
    sc = smooth(ALL[name]())
    sc = sc.replace(integ=dataclasses.replace(sc.integ, integrator=2))
    assert gradient_error(bos, orc, sc, bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2


@pytest.mark.parametrize("name", ["partly_steep", "uneven_cells", "three_samples"])
def test_reversed_refracted_adjoint_matches_oracle(bos, orc, name):
    sc = smooth(ALL[name]())
    sc = sc.replace(light=S.Light(2, sc.light.pattern, sc.light.proj, connect_iters=1))
    assert gradient_error(bos, orc, sc, bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2


def test_hand_over_on_a_pixel_list(bos, orc):
    sc = smooth(partly_steep())
    pix = np.random.default_rng(9).choice(sc.pixels, 333, replace=False).astype(np.int32)
    w = np.random.default_rng(10).standard_normal(pix.size).astype(np.float32)
    ctx = bos.Context(0)
    ctx.set_scene(sc, bos.BOS_PREC_FP32_COMP)
    ctx.render_pixels(torch.as_tensor(pix, device="cuda"), save_for_backward=True)
    g = ctx.backward(torch.as_tensor(w, device="cuda")).cpu().numpy().astype(np.float64)
    ctx.close()
    full = np.zeros(sc.pixels)
    full[pix] = w
    ref = orc.grad(sc, full.reshape(sc.camera.height, sc.camera.width))
    assert np.linalg.norm(g - ref) <= GRAD_REL_L2 * np.linalg.norm(ref)
