"""Quasi-linear renders whose end state is kept for the adjoint, bit for bit: the image seeds a
gradient, so its arithmetic is pinned.  The displacements are evaluated here in numpy float32 from
the exported node records: the 32.32 fixed-point line, the trilinear lerps, Sharma's weights with
Kahan sums and the wall hit, each operation rounded as written."""
import dataclasses

import numpy as np
import pytest

from paper_2509_14442_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

f32, f64 = np.float32, np.float64

# a fused multiply-add is formed in float64 here: its product is exact, its sum rounds twice in
# ~2^-29 of the cases; and the line's set-up may fuse float64 operations there.  Ten operations in
# ~200 steps of three components: fewer than one ray in 10^4 either way.
DIFFERENT = 1e-2


def fma(a, b, c):
    return (f64(a) * f64(b) + f64(c)).astype(f32)


def kahan(s, c, y):
    t = s + y
    return t, (t - s) - y


def records(nodes):
    """Node records as float32 (nz, ny, nx, 4)."""
    n = nodes.cpu().numpy()
    return n if n.dtype == f32 else (n.view(np.uint16).astype(np.uint32) << 16).view(f32)


def displacements(sc, rec):
    """(H, W, 2) float32 displacements on the back wall."""
    c, g, w = sc.camera, sc.grid, sc.wall
    pos, fwd, up = (np.array(v, f64) for v in (c.pos, c.fwd, c.up))
    n, h = np.array(g.n), np.array(g.extent, f64) / np.array(g.n)
    px, py = np.meshgrid(np.arange(c.width), np.arange(c.height))
    a, b = ((px.ravel() + 0.5) - c.cx) / c.fx, ((py.ravel() + 0.5) - c.cy) / c.fy
    d = (a[:, None] * np.cross(fwd, up) - b[:, None] * up) + fwd
    d /= np.sqrt((d[:, 0] ** 2 + d[:, 1] ** 2) + d[:, 2] ** 2)[:, None]
    # slabs (no component is zero at a pixel centre of an even-sized image), wall, steps
    lo = np.array(g.origin) - pos
    t0, t1 = lo / d, ((np.array(g.origin) + np.array(g.extent)) - pos) / d
    t_in = np.maximum(np.minimum(t0, t1).max(1), 0.0)
    nw = np.array(w.normal, f64)
    tw = ((np.array(w.origin) - pos) @ nw) / (d @ nw)
    ell = np.minimum(np.maximum(t0, t1).min(1), tw) - t_in
    N = np.full(ell.shape, sc.integ.fixed_steps) if sc.integ.fixed_steps else np.ceil(ell / (sc.integ.max_step_vox * h.min()))
    assert (ell > 0).all()
    sl = ell / N
    U = np.rint(((pos + t_in[:, None] * d - np.array(g.origin)) * (1.0 / h) - 0.5) * 2.0 ** 32).astype(np.int64) + 256
    dU = np.rint(sl[:, None] * d * (1.0 / h) * 2.0 ** 32).astype(np.int64)

    def rhs(U):
        I = (U >> 32).astype(np.int64)
        f = ((U & 0xffffffff) >> 9).astype(f32) * f32(2.0 ** -23)
        i = np.clip(I, 0, n - 2)
        f = f + (I - i).astype(f32)
        at = lambda z, y, x: rec[i[:, 2] + z, i[:, 1] + y, i[:, 0] + x]
        x, y, z = f[:, 0:1], f[:, 1:2], f[:, 2:3]
        e = [[fma(x, at(k, j, 1) - at(k, j, 0), at(k, j, 0)) for j in (0, 1)] for k in (0, 1)]
        e = [fma(y, e[k][1] - e[k][0], e[k][0]) for k in (0, 1)]
        v = fma(z, e[1] - e[0], e[0])
        return v[:, 0], (f32(1.0) + v[:, 0:1]) * v[:, 1:]

    de, D = rhs(U)
    eta = (1.0 + f64(de)).astype(f32)
    dt = (sl.astype(f32) / eta)[:, None]
    A = dt * D
    dr, cr, dv, cv = (np.zeros(d.shape, f32) for _ in range(4))
    six = f32(1.0 / 6.0)
    for k in range(int(N.max())):
        on = (k < N)[:, None]
        B, C = dt * rhs(U + (dU >> 1))[1], dt * rhs(U + dU)[1]
        inc = dt * fma(six, fma(f32(2.0), B, A), dv)
        s = fma(f32(4.0), B, A) + C
        new = (*kahan(dr, cr, inc - cr), *kahan(dv, cv, fma(s, six, -cv)), C, U + dU)
        dr, cr, dv, cv, A, U = (np.where(on, p, q) for p, q in zip(new, (dr, cr, dv, cv, A, U)))
    dr, dv = dr - cr, dv - cv
    # wall hit relative to the straight ray's
    df, nf = d.astype(f32), np.broadcast_to(nw.astype(f32), d.shape)
    dot = lambda p, q: fma(p[:, 2], q[:, 2], fma(p[:, 1], q[:, 1], p[:, 0] * q[:, 0]))
    rest, cd = (tw - t_in - ell).astype(f32), df[:, 1]
    ndr, ndv = dot(nf, dr), dot(nf, dv)
    inv = f32(1.0) / fma(eta, cd, ndv)
    ts, kk = fma(rest, cd, -ndr) * inv, -(fma(rest, ndv, eta * ndr) * inv)
    dx = fma(kk[:, None], df, fma(ts[:, None], dv, dr))
    return dx[:, [0, 2]].reshape(c.height, c.width, 2)


SCENES = {
    "room": lambda: S.room((30, 26, 22), 96, 72, 1, 6301),
    "many_tiles": lambda: S.room((20, 18, 16), 320, 260, 1, 6302),      # more tiles than a small launch has
    "cube": lambda: S.blob_cube(n=12, width=48, height=40, steps=57),
}


@pytest.mark.parametrize("prec", ["FP32_COMP", "BF16_COMP"])
@pytest.mark.parametrize("name", sorted(SCENES))
def test_kept_quasi_linear_displacements_are_the_stage_arithmetic(name, prec):
    from paper_2509_14442_gb300 import bos

    sc = SCENES[name]()
    assert tuple(sc.wall.normal) == (0.0, 1.0, 0.0) and tuple(sc.wall.eu) == (1.0, 0.0, 0.0)
    sc = sc.replace(integ=dataclasses.replace(sc.integ, integrator=2))
    ctx = bos.Context(0)
    ctx.set_scene(sc, getattr(bos, "BOS_PREC_" + prec))
    _, disp, _ = ctx.render(disp=True, save_for_backward=True)
    got, rec = disp.cpu().numpy(), records(ctx.export_nodes())
    ctx.status()
    ctx.close()
    want = displacements(sc, rec)
    moved = np.abs(want).max(-1) > 0
    assert moved.mean() > 0.5
    assert (got[moved] != want[moved]).any(-1).mean() <= DIFFERENT
