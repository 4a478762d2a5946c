"""The float32 and bfloat16 field store against numpy's float64 evaluation, bit for bit, on
fields where its float32 arithmetic has to hand values over to float64: equal and nearly
equal temperatures, neighbours orders of magnitude apart, values at the ends of float32's
range, and temperatures that are zero, negative, infinite or not a number."""
import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from helpers import bf16_round

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def nodes(g, T):
    """(deta, grad eta) in float64: K / T and its central or one-sided differences."""
    with np.errstate(all="ignore"):
        de = (g.rho0 * g.G * g.T0) / T.astype(np.float64)
        cols = [de]
        for a, ax in enumerate((2, 1, 0)):
            h = g.extent[a] / g.n[a]
            n = de.shape[ax]
            lo, hi = np.maximum(np.arange(n) - 1, 0), np.minimum(np.arange(n) + 1, n - 1)
            den = np.where(hi - lo == 2, 2.0 * h, h).reshape([-1 if i == ax else 1 for i in range(3)])
            cols.append((de.take(hi, ax) - de.take(lo, ax)) / den)
    return np.stack(cols, -1)


def fields(rng, shape):
    base = (293.0 + 20.0 * rng.random(shape)).astype(np.float32)
    one = np.full(shape, 293.0, np.float32)
    odd = base.copy()
    odd.reshape(-1)[:: 7] = rng.choice([0.0, -0.0, -293.0, np.inf, -np.inf, np.nan, 1e-30, 1e30, 1e-42], odd.reshape(-1)[:: 7].size)
    return {
        "plain": base,
        "equal": one,
        "one_ulp": np.where(rng.random(shape) < 0.3, np.nextafter(one, np.float32(400)), one),
        "apart": np.exp(rng.uniform(np.log(1e-3), np.log(1e6), shape)).astype(np.float32),
        "wide": np.exp(rng.uniform(np.log(1e-25), np.log(1e25), shape)).astype(np.float32),
        "negative": -base,
        "odd": odd,
    }


@pytest.mark.parametrize("n", [(2, 2, 2), (9, 8, 10), (17, 33, 18)])
@pytest.mark.parametrize("name", ["plain", "equal", "one_ulp", "apart", "wide", "negative", "odd"])
def test_store_bits(bos, n, name):
    g = S.Grid(n=n, origin=(-0.3, 0.2, 0.1), extent=(1.1, 0.7, 0.93), T0=291.3, rho0=1.19, G=2.3e-4)
    T = fields(np.random.default_rng(sum(n)), (n[2], n[1], n[0]))[name]
    want = nodes(g, T)
    ctx = bos.Context(0)
    for prec in ("fp32_comp", "bf16_comp"):
        ctx.set_grid(g, torch.as_tensor(T, device="cuda"), bos.PRECISIONS[prec])
        got = ctx.export_nodes().cpu().numpy()
        with np.errstate(all="ignore"):
            if prec == "fp32_comp":
                ref = want.astype(np.float32)
                same = (got.view(np.uint32) == ref.view(np.uint32)) | (np.isnan(got) & np.isnan(ref))
            else:
                finite = np.isfinite(want) & (np.abs(want) < 3e38) & (np.abs(want) > 1e-37) | (want == 0)
                ref = (bf16_round(np.where(finite, want, 1.0)).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
                same = (got.view(np.uint16) == ref) | ~finite
        assert same.all(), (prec, np.argwhere(~same)[:4])
    ctx.close()
