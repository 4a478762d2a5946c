"""The float64 tracer and its adjoint with the cell polynomial and the per-cell corner sums,
against the FP64 oracle where they could go wrong: cells never left or always extrapolated,
several steps per cell and several cells per step, uneven cells, rays that cross cells along
every axis, steep fields, lanes that loop over samples."""
import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from helpers import I_ABS_TOL, errors, gpu_render
from test_gpu_adjoint import GRAD_REL_L2_FP64, gpu_grad64, rel_l2
from test_gpu_march import SCENES
from test_gpu_reverse import smooth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# displacements come out in float32 (2^-24), from positions whose float64 rounding is far below
DISP_REL_FP64 = 2e-7


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def coarse():
    """Steps of several cells: a step's three points lie in three cells."""
    return S.blob_cube(n=40, width=33, height=35, steps=13)


ALL = {**{k: SCENES[k] for k in ("two_cells", "uneven_cells", "three_samples", "diagonal", "steep")}, "coarse": coarse}


@pytest.mark.parametrize("name", sorted(ALL))
def test_fp64_cells_match_oracle(bos, orc, name):
    sc = smooth(ALL[name]())
    e = errors(gpu_render(sc, bos.BOS_PREC_FP64), orc.render(sc))
    assert e["disp_max"] > 0 and e["disp_rel"] <= DISP_REL_FP64 and e["I_abs"] <= I_ABS_TOL, e
    w = np.random.default_rng(9).standard_normal((sc.camera.height, sc.camera.width))
    ref = orc.grad(sc, w)
    assert np.abs(ref).max() > 0
    assert rel_l2(gpu_grad64(bos, sc, w), ref) <= GRAD_REL_L2_FP64
