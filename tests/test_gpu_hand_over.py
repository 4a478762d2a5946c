"""The hand-over of steep tiles to the adjoint kernels that keep stage terms: scenes that have
tiles of both kinds (found on the CPU from the oracle's field), the server's batched pair of
kernels over jobs of several grids, and the bfloat16 store."""
import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S
from test_gpu_reverse import GRAD_REL_L2, gradient_error, smooth
from test_gpu_server import submit

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SAME_REVERSE = 2.0 ** -22     # cells: the tracer's bound for reversing a step from its end state


@pytest.fixture(scope="module")
def bos():
    from paper_2509_14442_gb300 import bos as B
    B.lib()
    return B


def stage_difference(orc, sc):
    """Per pixel (1 ray each): the largest of dt |A - B| / 6 and dt |A - C| / 24 of its steps, in cells."""
    field, h = orc.field_from_T(sc.grid, sc.T), min(sc.grid.spacing())
    rays = [orc.ray_setup(sc, p, 0) for p in range(sc.pixels)]
    d = np.array([r["d"] for r in rays])
    N = np.array([r["N"] if r["traced"] else 0 for r in rays])
    r = np.array(sc.camera.pos) + np.array([q["t_in"] for q in rays])[:, None] * d

    def D(x):
        eta, g = orc.field_eval(sc.grid, field, x)
        return eta[:, None] * g

    eta, _ = orc.field_eval(sc.grid, field, r)
    dt = (np.array([q["ell"] for q in rays]) / np.maximum(N, 1) / eta)[:, None]
    v, out = eta[:, None] * d, np.zeros(len(rays))
    for n in range(int(N.max())):
        A = dt * D(r)
        B = dt * D(r + dt / 2 * v + dt / 8 * A)
        C = dt * D(r + dt * v + dt / 2 * B)
        step = (dt / 6 * np.maximum(np.abs(A - B), np.abs(A - C) / 4)).max(1) / h
        out = np.where(n < N, np.maximum(out, step), out)
        r, v = r + dt * (v + (A + 2 * B) / 6), v + (A + 4 * B + C) / 6
    return out.reshape(sc.camera.height, sc.camera.width)


def tile_kinds(orc, sc):
    """(steep, mild): numbers of 8 x 4 tiles that are clearly handed over, and clearly not."""
    x = stage_difference(orc, sc)
    x = np.pad(x, ((0, -x.shape[0] % 4), (0, -x.shape[1] % 8)))
    m = x.reshape(x.shape[0] // 4, 4, x.shape[1] // 8, 8).max((1, 3))
    return int((m > 2 * SAME_REVERSE).sum()), int((m < 0.5 * SAME_REVERSE).sum())


def heated(n, width, height, seed, gain):
    sc = S.room(n, width, height, 1, seed)
    T = (S.T_AMBIENT + gain * (sc.T.astype(np.float64) - S.T_AMBIENT)).astype(np.float32)
    return smooth(sc.replace(T=T))


def test_both_kinds_of_tile_in_one_launch(bos, orc):
    sc = heated((18, 20, 14), 90, 70, 6204, 60.0)
    steep, mild = tile_kinds(orc, sc)
    assert steep > 0 and mild > 0, (steep, mild)
    assert gradient_error(bos, orc, sc, bos.BOS_PREC_FP32_COMP) <= GRAD_REL_L2


def test_both_kinds_of_tile_on_a_pixel_list(bos, orc):
    sc = heated((18, 20, 14), 90, 70, 6204, 60.0)
    y, x = np.divmod(np.arange(sc.pixels), sc.camera.width)
    order = np.lexsort((x, y, x // 8, y // 4))                # 8 x 4 blocks one after the other
    pix = order[(x[order] < 88) & (y[order] < 68)][40:].astype(np.int32)
    per_tile = [t.max() for t in np.split(stage_difference(orc, sc).ravel()[pix], range(32, pix.size, 32))]
    assert max(per_tile) > 2 * SAME_REVERSE and min(per_tile) < 0.5 * SAME_REVERSE
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


def test_server_batches_steep_and_mild_jobs(bos, orc):
    """Two jobs with steep tiles and one without, on three grids, in one batch."""
    scenes = [heated((20, 20, 15), 66, 90, 6205, 60.0), heated((36, 33, 27), 70, 60, 6202, 1.0),
              heated((20, 22, 16), 81, 50, 6203, 60.0)]
    kinds = [tile_kinds(orc, sc) for sc in scenes]
    assert kinds[0][0] > 0 and kinds[2][0] > 0 and kinds[1][0] == 0, kinds
    reqs = []
    for sc in scenes:
        h, w = sc.camera.height, sc.camera.width
        reqs.append(dict(scene=sc, T=torch.as_tensor(sc.T, device="cuda"), pattern=torch.as_tensor(sc.light.pattern, device="cuda"),
                         I=torch.zeros((h, w), device="cuda"), disp=torch.zeros((h, w, 2), device="cuda"),
                         target=torch.full((h, w), 0.2, device="cuda"),
                         loss=torch.zeros((1,), dtype=torch.float64, device="cuda")))
        reqs[-1]["dLdT"] = torch.zeros_like(reqs[-1]["T"])
    srv = bos.Server(0, 2 << 30, 3)
    tickets = [submit(bos, srv, d) for d in reqs]
    for t in tickets:
        assert srv.wait(t, 60.0) == bos.BOS_OK
    srv.close()
    for d in reqs:
        ref = orc.grad(d["scene"], -2.0 * (d["target"].cpu().numpy().astype(np.float64) - orc.render(d["scene"])["I"]))
        g = d["dLdT"].cpu().numpy().astype(np.float64)
        # the seeds follow from the images, 1e-6 of 0.17 apart: 6e-6 beside the gradient's own rounding
        assert np.linalg.norm(g - ref) <= (GRAD_REL_L2 + 1e-5) * np.linalg.norm(ref)


def test_bfloat16_steps_across_a_layer(bos, orc):
    """A field whose records are bfloat16 numbers (so that the oracle's field is the store's), with a
    layer in the last step: every tile is handed over."""
    n, steps = 32, 4
    sc = S.blob_cube(n=n, width=23, height=19, steps=steps)
    g = sc.grid
    i = np.arange(n)
    deta = 2.0 ** -5 + (i > 29)[:, None] * (i - 16)[None, :] * 2.0 ** -11
    T = np.broadcast_to((g.rho0 * g.G * g.T0) / deta, (n, n, n)).astype(np.float32)
    sc = smooth(sc.replace(T=T))
    assert tile_kinds(orc, sc) == (15, 0)
    assert gradient_error(bos, orc, sc, bos.BOS_PREC_BF16_COMP) <= GRAD_REL_L2
