"""The quasi-linear tracer through the cell marcher against the FP64 oracle at the sizes where
it could go wrong: cells never left or always extrapolated, many half steps per cell, uneven
cells, rays that cross cells along every axis, lanes that loop over samples, step counts beyond
one line set-up, the bfloat16 store, and the end states that the adjoint reverses from."""
import dataclasses

import numpy as np
import pytest

from helpers import DISP_REL_TOL, I_ABS_TOL, bf16_round, errors, gpu_render
from test_gpu_march import SCENES
from test_gpu_reverse import GRAD_REL_L2, gradient_error, smooth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def quasi(name):
    sc = SCENES[name]()
    return sc.replace(integ=dataclasses.replace(sc.integ, integrator=2))


@pytest.mark.parametrize("name", sorted(SCENES))
def test_quasi_march_matches_oracle(bos, orc, name):
    sc = quasi(name)
    o = orc.render(sc, nsteps=True)
    g = gpu_render(sc, bos.BOS_PREC_FP32_COMP)
    assert g["steps"] == int(o["nsteps"].sum())
    e = errors(g, o)
    assert e["disp_max"] > 0 and e["disp_rel"] <= DISP_REL_TOL and e["I_abs"] <= I_ABS_TOL, e


@pytest.mark.parametrize("name", ["steep", "uneven_cells"])
def test_quasi_march_bf16_matches_oracle_on_the_bf16_field(bos, orc, name):
    sc = quasi(name)
    de = orc.deta_from_T(sc.grid, sc.T.astype(np.float64))
    field = orc.NodeField(bf16_round(de), bf16_round(orc.grad_from_deta(sc.grid, de)))
    e = errors(gpu_render(sc, bos.BOS_PREC_BF16_COMP), orc.render(sc, field=field))
    assert e["disp_max"] > 0 and e["disp_rel"] <= DISP_REL_TOL and e["I_abs"] <= I_ABS_TOL, e


@pytest.mark.parametrize("name", ["diagonal", "three_samples", "two_cells", "uneven_cells"])
def test_quasi_gradient_from_the_marched_end_state(bos, orc, name):
    assert gradient_error(bos, orc, smooth(quasi(name)), bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2
