"""The adjoint's two ways of adding corner sensitivities to the nodes, against the FP64 oracle
on both sides of the rule that chooses between them (lanes per cell of the grid's smallest cross
section), for every light and tracer that has them, with few tiles and many."""
import dataclasses

import pytest

from paper_2509_14442_gb300 import scenes as S
from test_gpu_reverse import GRAD_REL_L2, gradient_error, smooth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


# cells, image: lanes per cell 0.5, 12 exactly (144 tiles of 32 on 16 x 24 cells), just above, 90;
# and 1320 tiles (more than eight per SM) at 10 and 36
SIZES = {"0.5": ((48, 48, 36), (30, 26)), "12": ((32, 24, 16), (96, 48)), "12.2": ((32, 24, 16), (98, 48)),
         "90": ((16, 16, 12), (150, 110)), "many_10": ((72, 72, 58), (264, 160)), "many_36": ((40, 40, 29), (264, 160))}


@pytest.mark.parametrize("kind", ["sharma", "quasi", "refracted"])
@pytest.mark.parametrize("size", sorted(SIZES))
def test_gradient_on_both_sides(bos, orc, size, kind):
    cells, image = SIZES[size]
    sc = smooth(S.room(cells, *image, 1, 6301))
    if kind == "refracted":
        sc = sc.replace(light=S.Light(2, sc.light.pattern, sc.light.proj, connect_iters=1))
    if kind == "quasi":
        sc = sc.replace(integ=dataclasses.replace(sc.integ, integrator=2))
    assert gradient_error(bos, orc, sc, bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2
