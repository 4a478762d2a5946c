"""The work that users of this framework have it do, as cases that can be timed.

A case is one call sequence of a user's program through the public binding
(`paper_2509_14442_gb300.bos`): a frame (field build and render), a gradient step (field
build, render with checkpoints, image loss, adjoint), a minibatch iteration of the voxel
reconstruction, or a handful of requests through the request server.  Sizes are those of the
paper's sensor, of the benchmark's workloads and of the tests, and odd ones between them.

`exact` evaluates the same outputs with plain torch operations in float64: the field
(Gladstone-Dale, central differences, trilinear interpolation), Sharma's Runge-Kutta-Nystroem
steps or the quasi-linear ones, the wall hit, Eq. 2's luminance and weight, and for the
gradients the reverse of every step by automatic differentiation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_14442_gb300 import bos, scenes

DEV = "cuda"
PRECISIONS = {"fp32_comp": bos.BOS_PREC_FP32_COMP, "bf16_comp": bos.BOS_PREC_BF16_COMP, "fp64": bos.BOS_PREC_FP64}


def _case(kind, n, image, spp=1, tracer="sharma", store="fp32_comp", light="projector", steps=0, batch=0, requests=""):
    """A case's plain values.  kind: frame, step (frame + gradient), minibatch or serve; n: cells
    per axis; image: width and height; steps: fixed steps per ray (0: half a cell at most)."""
    return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "width": image[0], "height": image[1], "spp": spp,
            "tracer": tracer, "store": store, "light": light, "steps": steps, "batch": batch, "requests": requests}


def listed():
    return [
        # the smallest gradient step: a 32^3 cube with one hot blob before a textured wall and a
        # 64 x 64 camera with 128 fixed steps per ray; what a user starts with, where launches count
        dict(_case("step", (32, 32, 32), (64, 64), light="texture", steps=128), name="blob_step"),
        # the paper's own sensor: one frame of a 64^3 field, 100 x 100 pixels, 2 rays each, and the
        # no-flow reference image it is compared with
        dict(_case("frame", (64, 64, 64), (100, 100), 2), name="sensor_frame"),
        # one iteration of the paper's reconstruction on that sensor up to the gradient: draw and
        # order 5000 random pixels, build the field, render them with the quasi-linear tracer,
        # image loss and adjoint
        dict(_case("minibatch", (64, 64, 64), (100, 100), 2, tracer="quasi", batch=5000), name="sensor_minibatch"),
        # a frame of a room-scale field as a preview renderer makes it: 4 jittered rays per pixel
        dict(_case("frame", (128, 128, 96), (1024, 1024), 4), name="room_frame"),
        # a new fine field for every small frame (a solver's time steps watched at low
        # resolution): the field build weighs as much as the rays
        dict(_case("frame", (256, 256, 192), (256, 256)), name="fine_field_frame"),
        # the gradient step the benchmark quotes: fine field, one ray per pixel of a 4-megapixel photograph
        dict(_case("step", (256, 256, 192), (2048, 2048)), name="photo_step"),
        # odd everything: cells, image and 3 rays per pixel (a lane walks its samples in turn)
        dict(_case("step", (150, 131, 97), (509, 383), 3), name="ragged_step"),
        # the paper's quasi-linear tracer on the fine field, frame and gradient
        dict(_case("step", (256, 256, 192), (1024, 768), tracer="quasi"), name="quasi_step"),
        # the projector's rays bent by the flow too: two rays per sample, forward and back
        dict(_case("step", (128, 128, 96), (512, 512), light="refracted"), name="refracted_step"),
        # the bfloat16 field store, for fields that would not fit in float32
        dict(_case("step", (192, 192, 144), (768, 768), store="bf16_comp"), name="bf16_step"),
        # float64 throughout, for a user who checks a gradient
        dict(_case("step", (64, 64, 48), (192, 144), store="fp64"), name="fp64_step"),
        # requests of several sizes through the request server, rendered and differentiated together
        dict(_case("serve", (64, 64, 64), (256, 256),
                   requests="64x64x64:256:grad 128x128x96:512:frame 64x64x64:512:grad 128x128x96:1024:frame "
                            "128x128x96:256:grad 64x64x64:1024:frame"), name="serve_mix"),
    ]


def draw(rng):
    """A case of the listed ones' ranges."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def cells(lo, hi):     # a room's proportions, give or take
        n = log_int(lo, hi)
        return (n, max(8, int(n * rng.uniform(0.85, 1.15))), max(8, int(n * rng.uniform(0.65, 0.85))))

    def image(lo, hi):
        w = log_int(lo, hi)
        return (w, max(8, int(w * rng.uniform(0.6, 1.2))))

    kind = rng.choice(["frame", "frame", "step", "step", "quasi", "refracted", "bf16", "minibatch", "blob", "fp64", "serve"])
    if kind == "frame":
        return _case("frame", cells(24, 240), image(60, 1400), rng.choice([1, 1, 2, 3, 4]))
    if kind == "step":
        return _case("step", cells(24, 240), image(60, 1000), rng.choice([1, 1, 2, 3]))
    if kind == "quasi":
        return _case("step", cells(24, 240), image(60, 1200), rng.choice([1, 1, 2]), tracer="quasi")
    if kind == "refracted":
        return _case("step", cells(24, 130), image(60, 600), rng.choice([1, 2]), light="refracted")
    if kind == "bf16":
        return _case("step", cells(24, 200), image(60, 800), store="bf16_comp")
    if kind == "minibatch":
        return _case("minibatch", cells(24, 100), image(64, 400), rng.choice([1, 2, 4]),
                     tracer=rng.choice(["quasi", "quasi", "sharma"]), batch=log_int(200, 12000))
    if kind == "blob":
        n = log_int(16, 64)
        return _case("step", (n, n, n), image(32, 128), light="texture", steps=rng.randint(2 * n, 4 * n))
    if kind == "fp64":
        return _case("step", cells(16, 64), image(32, 200), store="fp64")
    sizes = [f"{n[0]}x{n[1]}x{n[2]}:{log_int(100, 1000)}:{rng.choice(['frame', 'grad'])}"
             for n in (cells(32, 130) for _ in range(rng.randint(3, 8)))]
    return _case("serve", (64, 64, 64), (256, 256), requests=" ".join(sizes))


# ------------------------------------------------------------------ inputs

def _field(grid, seed):
    """A plume from the inlet (a plume seed follows from the case's), made on the GPU."""
    return scenes.plume_field(grid, 4000 + seed, device=DEV).contiguous()


def _scene(case, seed):
    """Geometry and descriptors of a case (host values; the pattern is a small numpy array)."""
    n = (case["nx"], case["ny"], case["nz"])
    integ = scenes.Integrator(fixed_steps=case["steps"], max_step_vox=0.5,
                              integrator=2 if case["tracer"] == "quasi" else 0, ckpt_every=16)
    if case["light"] == "texture":
        sc = scenes.blob_cube(seed=3000 + seed, n=n[0], width=case["width"], height=case["height"], steps=case["steps"])
        return sc.replace(integ=integ)
    sc = scenes.room(n, case["width"], case["height"], case["spp"], seed=5000 + seed, field=False)
    if case["light"] == "refracted":
        sc = sc.replace(light=scenes.Light(2, sc.light.pattern, sc.light.proj, connect_iters=1))
    return sc.replace(integ=integ)


def _noise(shape, seed):
    return torch.randn(shape, generator=torch.Generator(device=DEV).manual_seed(7 * seed + 11), device=DEV)


def _inputs(case, seed):
    """Scene, field, pattern and (for gradients) the photograph: the no-flow image of the scene
    with one per cent of sensor noise."""
    sc = _scene(case, seed)
    if case["light"] == "texture":
        T = torch.as_tensor(sc.T, device=DEV)
    else:
        T = _field(sc.grid, seed)
    out = {"scene": sc, "T": T, "pattern": torch.as_tensor(np.ascontiguousarray(sc.light.pattern), device=DEV)}
    if case["kind"] in ("step", "minibatch"):
        out["target"] = _photograph(sc, out["pattern"], seed)
    return out


def _photograph(sc, pattern, seed):
    cam = sc.camera
    ref = _Tracer(sc, None, pattern).image(straight=True)["I"].view(cam.height, cam.width)
    scale = ref.abs().mean()
    return (ref + 0.01 * scale * _noise(ref.shape, seed).double()).to(torch.float32).contiguous()


def _requests(case):
    out = []
    for r in case["requests"].split():
        n, image, what = r.split(":")
        nx, ny, nz = (int(v) for v in n.split("x"))
        out.append((_case("step" if what == "grad" else "frame", (nx, ny, nz), (int(image), int(image))), what == "grad"))
    return out


def prepare(case, seed):
    if case["kind"] == "serve":
        return _prepare_server(case, seed)
    st = _inputs(case, seed)
    sc = st["scene"]
    ctx = bos.Context(0)
    ctx.set_geometry(sc.camera, sc.wall, sc.light, sc.integ, pattern=st["pattern"])
    st.update(case=case, ctx=ctx, prec=PRECISIONS[case["store"]])
    if case["kind"] == "minibatch":
        st["pix"] = torch.empty(case["batch"], dtype=torch.int32, device=DEV)
        st["seed"] = seed
    return st


def _prepare_server(case, seed):
    st = {"case": case, "server": bos.Server(0, 24 << 30, 6), "jobs": []}
    for i, (sub, grad) in enumerate(_requests(case)):
        job = _inputs(sub, seed + 13 * i)
        cam = job["scene"].camera
        job["I"] = torch.empty((cam.height, cam.width), device=DEV)
        if grad:
            job["loss"] = torch.empty(1, dtype=torch.float64, device=DEV)
            job["dLdT"] = torch.empty_like(job["T"])
        else:
            job["disp"] = torch.empty((cam.height, cam.width, 2), device=DEV)
        sc = job["scene"]
        ptr = lambda k: job[k].data_ptr() if k in job else None
        job["request"] = bos.make_request(sc.grid, bos.BOS_PREC_FP32_COMP, ptr("T"), sc.camera, sc.wall, sc.light,
                                          ptr("pattern"), sc.integ, ptr("I"), ptr("disp"), ptr("target"), ptr("loss"),
                                          ptr("dLdT"))
        st["jobs"].append(job)
    torch.cuda.synchronize()      # the server's streams do not wait for this one
    return st


# ------------------------------------------------------------------ one pass

def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        srv = state["server"]
        tickets = [srv.submit(j["request"]) for j in state["jobs"]]
        for t in tickets:
            status = srv.wait(t, 60.0)
            if status != bos.BOS_OK:
                raise RuntimeError(f"request {t}: status {status}")
        return [[j[k] for k in ("I", "disp", "loss", "dLdT") if k in j] for j in state["jobs"]]
    sc, ctx = state["scene"], state["ctx"]
    if case["kind"] == "minibatch":
        pix = state["pix"]
        stream = torch.cuda.current_stream().cuda_stream
        n, cam = pix.numel(), sc.camera
        bos.bos_sample_pixels(pix.data_ptr(), n, cam.width * cam.height, state["seed"], 0, stream)
        bos.bos_sort_pixels(pix.data_ptr(), n, cam.width, cam.height, stream)
        ctx.set_grid(sc.grid, state["T"], state["prec"])
        I, _ = ctx.render_pixels(pix, save_for_backward=True)
        loss = torch.empty(1, dtype=torch.float64, device=DEV)
        dLdI = torch.empty_like(I)
        bos.bos_loss_l2_pixels(I.data_ptr(), state["target"].data_ptr(), pix.data_ptr(), n, loss.data_ptr(),
                               dLdI.data_ptr(), stream)
        return [pix, I, loss, ctx.backward(dLdI)]
    ctx.set_grid(sc.grid, state["T"], state["prec"])
    if case["kind"] == "frame":
        I, disp, _ = ctx.render(disp=True)
        I_ref, _, _ = ctx.render_reference()
        return [I, disp, I_ref]
    I, disp, _ = ctx.render(disp=True, save_for_backward=True)
    loss, dLdI = bos.loss_l2(I, state["target"])
    if case["store"] == "fp64":
        return [I, disp, loss, ctx.backward_f64(dLdI.double())]
    return [I, disp, loss, ctx.backward(dLdI)]


# ------------------------------------------------------------------ what a pass cannot do without

# Floating-point operations of one ray-step (an FMA counts 2): three field evaluations of
# Sharma's step and its updates, two of the quasi-linear step; the adjoint of a step is its
# field values with derivatives, the transpose of the updates and the sensitivities of the
# corners (no recomputation).
_FORWARD = {"sharma": 356, "quasi": 241}
_ADJOINT = {"sharma": 884, "quasi": 400}


def _work_of(case):
    cells = case["nx"] * case["ny"] * case["nz"]
    pixels = case["width"] * case["height"]
    if case["kind"] == "minibatch":
        rays = case["batch"] * case["spp"]
    else:
        rays = pixels * case["spp"]
    if case["steps"]:
        n = case["steps"]
    else:
        e = scenes.ROOM_EXTENT
        n = math.ceil(e[1] / (0.5 * min(e[0] / case["nx"], e[1] / case["ny"], e[2] / case["nz"])))
    rs = rays * n * (2 if case["light"] == "refracted" else 1)
    nbytes = 4 * cells + 512 * 512 * 4
    flops = _FORWARD[case["tracer"]] * rs + 20 * cells
    if case["kind"] == "frame":
        nbytes += pixels * 16
    elif case["kind"] == "step":
        wide = 8 if case["store"] == "fp64" else 4
        nbytes += pixels * 16 + wide * cells
        flops += _ADJOINT[case["tracer"]] * rs
    else:
        nbytes += case["batch"] * 12 + 4 * cells
        flops += _ADJOINT[case["tracer"]] * rs
    return nbytes, flops


def work(case):
    parts = [_work_of(c) for c, _ in _requests(case)] if case["kind"] == "serve" else [_work_of(case)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------ float64 evaluation in plain torch

def _vec(v):
    return torch.tensor([float(x) for x in v], dtype=torch.float64, device=DEV)


def _dot(a, b):
    return (a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1]) + a[..., 2] * b[..., 2]


def _round_bf16(x):
    m, e = torch.frexp(x)
    return torch.ldexp(torch.round(m * 256.0), e - 8)


def _nodes(T, grid, bf16=False):
    """(deta, grad eta) at the cell centres, (cells, 4), from T (nz, ny, nx) in float64."""
    de = (grid.rho0 * grid.G * grid.T0) / T
    cols = [de]
    for a, dim in enumerate((2, 1, 0)):
        h = grid.extent[a] / grid.n[a]
        n = de.shape[dim]
        lo, hi = de.narrow(dim, 0, n - 2), de.narrow(dim, 2, n - 2)
        first = (de.narrow(dim, 1, 1) - de.narrow(dim, 0, 1)) / h
        last = (de.narrow(dim, n - 1, 1) - de.narrow(dim, n - 2, 1)) / h
        cols.append(torch.cat([first, (hi - lo) / (2.0 * h), last], dim))
    G = torch.stack(cols, -1).reshape(-1, 4)
    return G + (_round_bf16(G.detach()) - G.detach()) if bf16 else G


class _Gather(torch.autograd.Function):
    """Rows of the node table; their sensitivities are summed into `acc`."""

    @staticmethod
    def forward(ctx, hook, G, idx, acc):
        ctx.idx, ctx.acc = idx, acc
        return G[idx]

    @staticmethod
    def backward(ctx, g):
        ctx.acc.index_add_(0, ctx.idx.reshape(-1), g.reshape(-1, 4))
        return None, None, None, None


class _Trace(torch.autograd.Function):
    """N steps of a bundle of rays from (r0, v0); reverses them step by step from kept states."""

    @staticmethod
    def forward(ctx, r0, v0, dt, N, tracer, keep):
        nmax = int(N.max())
        r, v = r0.clone(), v0.clone()
        length = torch.zeros_like(dt)
        states = torch.empty((nmax, r.shape[0], 6), dtype=torch.float64, device=DEV) if keep else None
        for n in range(nmax):
            if keep:
                states[n, :, :3], states[n, :, 3:] = r, v
            act = (n < N)[:, None]
            r2, v2, seg = tracer.step(r, v, dt, r0, v0, n)
            r, v = torch.where(act, r2, r), torch.where(act, v2, v)
            length = length + torch.where(act[:, 0], seg, 0.0)
        ctx.args = (states, N, tracer, nmax)
        ctx.save_for_backward(r0, v0, dt)
        return r, v, length

    @staticmethod
    def backward(ctx, gr, gv, gl):
        states, N, tracer, nmax = ctx.args
        r0, v0, dt = ctx.saved_tensors
        gr, gv = gr.clone(), gv.clone()
        gdt, gr0, gv0 = torch.zeros_like(dt), torch.zeros_like(r0), torch.zeros_like(v0)
        for n in reversed(range(nmax)):
            act = (n < N)[:, None]
            a = act.double()
            leaves = [states[n, :, :3].clone(), states[n, :, 3:].clone(), dt.detach().clone(), r0.detach().clone(),
                      v0.detach().clone()]
            with torch.enable_grad():
                for t in leaves:
                    t.requires_grad_()
                out = tracer.step(*leaves, n)
                g = torch.autograd.grad(out, leaves, [gr * a, gv * a, gl * a[:, 0]], allow_unused=True)
            gr, gv = torch.where(act, g[0], gr), torch.where(act, g[1], gv)
            gdt = gdt + g[2]
            if g[3] is not None:
                gr0, gv0 = gr0 + g[3], gv0 + g[4]
        return gr + gr0, gv + gv0, gdt, None, None, None


class _Tracer:
    def __init__(self, sc, G, pattern, acc=None):
        self.sc, self.G, self.acc = sc, G, acc
        g = sc.grid
        self.o, self.ext = _vec(g.origin), _vec(g.extent)
        self.h = _vec([g.extent[a] / g.n[a] for a in range(3)])
        self.nmax = _vec([g.n[a] - 2 for a in range(3)])
        nx, ny = g.n[0], g.n[1]
        self.stride = torch.tensor([1, nx, nx * ny], dtype=torch.int64, device=DEV)
        self.corners = torch.tensor([i + j * nx + k * nx * ny for k in (0, 1) for j in (0, 1) for i in (0, 1)],
                                    dtype=torch.int64, device=DEV)
        self.quasi = sc.integ.integrator == 2
        self.pattern = pattern.double()
        self.wo, self.eu, self.ev, self.wn = (_vec(v) for v in (sc.wall.origin, sc.wall.eu, sc.wall.ev, sc.wall.normal))

    # ---- field
    def field(self, x):
        u = (x - self.o) / self.h - 0.5
        with torch.no_grad():
            fl = torch.minimum(torch.clamp(torch.floor(u), min=0.0), self.nmax)
            idx = (fl.to(torch.int64) * self.stride).sum(-1)[None, :] + self.corners[:, None]
        f = u - fl
        c = self.G[idx] if self.acc is None else _Gather.apply(x, self.G, idx, self.acc)
        f0, f1, f2 = f[:, 0:1], f[:, 1:2], f[:, 2:3]
        c = c[0::2] + f0 * (c[1::2] - c[0::2])
        c = c[0::2] + f1 * (c[1::2] - c[0::2])
        return c[0] + f2 * (c[1] - c[0])

    def rhs(self, x):
        v = self.field(x)
        return (1.0 + v[:, 0:1]) * v[:, 1:]

    def step(self, r, v, dt, r0, v0, n):
        dt = dt[:, None]
        if self.quasi:
            A, B, C = (dt * self.rhs(r0 + ((n + c) * dt) * v0) for c in (0.0, 0.5, 1.0))
        else:
            A = dt * self.rhs(r)
            B = dt * self.rhs(r + (0.5 * dt) * v + (0.125 * dt) * A)
            C = dt * self.rhs(r + dt * v + (0.5 * dt) * B)
        dr = dt * (v + (A + 2.0 * B) / 6.0)
        return r + dr, v + (A + 4.0 * B + C) / 6.0, torch.sqrt(_dot(dr, dr))

    # ---- rays
    def camera_dirs(self, pix, s):
        c = self.sc.camera
        px, py = (pix % c.width).double(), (pix // c.width).double()
        t1 = t2 = torch.zeros_like(px)
        if c.spp > 1:
            k = pix * c.spp + s + 1

            def const(v):
                return v - (1 << 64) if v >= 1 << 63 else v

            def shr(z, b):
                return (z >> b) & ((1 << (64 - b)) - 1)

            z = k * const(0x9E3779B97F4A7C15) + const(int(c.seed) & ((1 << 64) - 1))
            z = (z ^ shr(z, 30)) * const(0xBF58476D1CE4E5B9)
            z = (z ^ shr(z, 27)) * const(0x94D049BB133111EB)
            z = z ^ shr(z, 31)

            def tent(xi):
                return torch.where(xi < 0.5, torch.sqrt(2.0 * xi) - 1.0, 1.0 - torch.sqrt(2.0 - 2.0 * xi))

            t1 = tent(shr(z, 40).double() / 16777216.0)
            t2 = tent((shr(z, 16) & 0xFFFFFF).double() / 16777216.0)
        a = (((px + 0.5) + t1) - c.cx) / c.fx
        b = (((py + 0.5) + t2) - c.cy) / c.fy
        f, u = c.fwd, c.up
        right = (f[1] * u[2] - f[2] * u[1], f[2] * u[0] - f[0] * u[2], f[0] * u[1] - f[1] * u[0])
        d = torch.stack([(a * right[i] - b * u[i]) + f[i] for i in range(3)], -1)
        return d / torch.sqrt(_dot(d, d))[:, None]

    def segment(self, p, d):
        """Straight wall distance, traced segment [t_in, t_in + ell] and step count of rays p + t d."""
        it, g = self.sc.integ, self.sc.grid
        den = _dot(d, self.wn.expand_as(d))
        q = [self.sc.wall.origin[a] - p[a] for a in range(3)]
        n = self.sc.wall.normal
        tw = ((q[0] * n[0] + q[1] * n[1]) + q[2] * n[2]) / den
        t_in, t_out = torch.zeros_like(tw), torch.full_like(tw, math.inf)
        inside = torch.ones_like(tw, dtype=torch.bool)
        for a in range(3):
            zero = d[:, a] == 0.0
            da = torch.where(zero, torch.ones_like(tw), d[:, a])
            t0 = (g.origin[a] - p[a]) / da
            t1 = ((g.origin[a] + g.extent[a]) - p[a]) / da
            lo, hi = torch.minimum(t0, t1), torch.maximum(t0, t1)
            t_in = torch.where(zero | ~(lo > t_in), t_in, lo)
            t_out = torch.where(zero | ~(hi < t_out), t_out, hi)
            if p[a] < g.origin[a] or p[a] > g.origin[a] + g.extent[a]:
                inside = inside & ~zero
        t_end = torch.where(t_out < tw, t_out, tw)
        ok = (den > 0) & inside & (t_in < t_end)
        ell = torch.where(ok, t_end - t_in, torch.ones_like(tw))
        step = it.max_step_vox * min(g.extent[a] / g.n[a] for a in range(3))
        N = torch.full_like(tw, it.fixed_steps) if it.fixed_steps else torch.ceil(ell.detach() / step)
        return tw, torch.where(ok, t_in, torch.zeros_like(tw)), ell, torch.where(ok, N, 0.0).to(torch.int64)

    def bend(self, p, d, keep):
        """Wall hit, final direction's cosine factor and path length of rays from the pinhole p."""
        tw, t_in, ell, N = self.segment(p, d)
        P = _vec(p)
        rin = P + t_in[:, None] * d
        eta = 1.0 + self.field(rin)[:, 0]
        rN, vN, length = _Trace.apply(rin, eta[:, None] * d, ell / (torch.clamp(N, min=1).double() * eta), N, self, keep)
        vn = _dot(vN, self.wn.expand_as(vN))
        ts = _dot(self.wo - rN, self.wn.expand_as(rN)) / vn
        vl = torch.sqrt(_dot(vN, vN))
        straight = N == 0
        hit = torch.where(straight[:, None], P + tw[:, None] * d, rN + ts[:, None] * vN)
        cosw = torch.where(straight, _dot(d, self.wn.expand_as(d)), vn / vl)
        total = torch.where(straight, tw, (t_in + length) + ts * vl)
        return hit, cosw, total, P + tw[:, None] * d

    def bilinear(self, s, t):
        th, tw = self.pattern.shape
        s, t = s - 0.5, t - 0.5
        fi, fj = torch.floor(s.detach()), torch.floor(t.detach())
        fs, ft = s - fi, t - fj
        i, j = fi.to(torch.int64), fj.to(torch.int64)

        def texel(i, j):
            ok = (i >= 0) & (j >= 0) & (i < tw) & (j < th)
            return torch.where(ok, self.pattern[j.clamp(0, th - 1), i.clamp(0, tw - 1)], 0.0)

        p00, p10, p01, p11 = texel(i, j), texel(i + 1, j), texel(i, j + 1), texel(i + 1, j + 1)
        return (1 - fs) * ((1 - ft) * p00 + ft * p01) + fs * ((1 - ft) * p10 + ft * p11)

    def luminance(self, x):
        sc = self.sc
        if sc.light.mode == 0:
            q = x - self.wo
            th, tw = self.pattern.shape
            return self.bilinear(_dot(q, self.eu.expand_as(q)) / (sc.wall.size_u / tw),
                                 _dot(q, self.ev.expand_as(q)) / (sc.wall.size_v / th))
        P = sc.light.proj
        q = x - _vec(P.pos)
        f, u = _vec(P.fwd), _vec(P.up)
        z = _dot(q, f.expand_as(q))
        xx, yy = _dot(q, torch.linalg.cross(f, u).expand_as(q)), _dot(q, u.expand_as(q))
        return self.bilinear(P.cx + P.fx * xx / z, P.cy - P.fy * yy / z)

    def rays(self, d, straight, keep):
        """Intensity and displacement (wall coordinates) of camera rays of direction d."""
        pos = self.sc.camera.pos
        if straight:
            tw = self.segment(pos, d)[0]
            hit = _vec(pos) + tw[:, None] * d
            return self.luminance(hit) * _dot(d, self.wn.expand_as(d)) / tw, None
        hit, cosw, total, ref = self.bend(pos, d, keep)
        at = hit
        if self.sc.light.mode == 2:      # one aiming round of the projector's ray
            P = self.sc.light.proj.pos
            q = hit - _vec(P)
            y = self.bend(P, q / torch.sqrt(_dot(q, q))[:, None], keep)[0]
            at = hit + (hit - y)
        dx = hit - ref
        disp = torch.stack([_dot(dx, self.eu.expand_as(dx)), _dot(dx, self.ev.expand_as(dx))], -1)
        return self.luminance(at) * cosw / total, disp

    def image(self, pix=None, straight=False, target=None, chunk=1 << 19):
        """Pixel means of I and displacement; with `target` also the image loss, and with an
        accumulator the node sensitivities of that loss."""
        cam = self.sc.camera
        if pix is None:
            pix = torch.arange(cam.width * cam.height, dtype=torch.int64, device=DEV)
        per = max(1, chunk // cam.spp)
        I, D = [], []
        loss = torch.zeros(1, dtype=torch.float64, device=DEV)
        for lo in range(0, pix.numel(), per):
            p = pix[lo:lo + per]
            s = torch.arange(cam.spp, device=DEV).repeat(p.numel())
            d = self.camera_dirs(p.repeat_interleave(cam.spp), s)
            keep = self.acc is not None
            if keep:
                d.requires_grad_()
            with torch.set_grad_enabled(keep):
                Ir, dr = self.rays(d, straight, keep)
                Im = Ir.view(-1, cam.spp).mean(1)
                if target is not None:
                    r = ((target.reshape(-1)[p].double() - Im) ** 2).sum()
                    loss += r.detach()
                    if keep:
                        torch.autograd.grad(r, d)
            I.append(Im.detach())
            if dr is not None:
                D.append(dr.detach().view(-1, cam.spp, 2).mean(1))
        return {"I": torch.cat(I), "disp": torch.cat(D) if D else None, "loss": loss}


def _drawn_pixels(n, pixels, seed):
    """The minibatch of draw 0: splitmix64 outputs k + 1 reduced to [0, pixels), ordered along a Z curve."""
    m = (1 << 64) - 1
    out = []
    for k in range(n):
        z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & m
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
        out.append(((z ^ (z >> 31)) * pixels) >> 64)
    return out


def _z_order(pix, width):
    def key(p):
        x, y, k = p % width, p // width, 0
        for b in range(16):
            k |= ((x >> b) & 1) << (2 * b) | ((y >> b) & 1) << (2 * b + 1)
        return k
    return sorted(pix, key=key)


def _exact_one(case, seed):
    if _work_of(case)[1] > 1e12:      # half a minute and more
        return None
    inp = _inputs(case, seed)
    sc, grid = inp["scene"], inp["scene"].grid
    cam = sc.camera
    cost = _work_of(case)[1]
    grad = case["kind"] in ("step", "minibatch") and cost < 3e11
    bf16 = case["store"] == "bf16_comp"
    T = inp["T"].double().requires_grad_(grad)
    with torch.set_grad_enabled(grad):
        G = _nodes(T, grid, bf16)
    acc = torch.zeros_like(G) if grad else None
    tr = _Tracer(sc, G.detach(), inp["pattern"], acc)
    pix = None
    if case["kind"] == "minibatch":
        drawn = _z_order(_drawn_pixels(case["batch"], cam.width * cam.height, seed), cam.width)
        pix = torch.tensor(drawn, dtype=torch.int64, device=DEV)
    chunk = 1 << 21
    if grad:   # the kept states of a chunk (48 bytes per ray and step) stay within 24 GB
        g = grid.extent
        steps = case["steps"] or 2 * g[1] / min(g[a] / grid.n[a] for a in range(3))
        chunk = max(1 << 12, min(1 << 18, int(24e9 / (48 * steps))))
    o = tr.image(pix, target=inp.get("target"), chunk=chunk)
    dT = torch.autograd.grad(G, T, acc)[0] if grad else None
    shape = (cam.height, cam.width)
    if case["kind"] == "frame":
        ref = _Tracer(sc, None, inp["pattern"]).image(straight=True)
        return [o["I"].view(shape), o["disp"].view(*shape, 2), ref["I"].view(shape)]
    if case["kind"] == "minibatch":
        return [pix.to(torch.int32), o["I"], o["loss"], dT]
    return [o["I"].view(shape), o["disp"].view(*shape, 2), o["loss"], dT]


def exact(case, seed):
    if case["kind"] != "serve":
        return _exact_one(case, seed)
    out = []
    for i, (sub, grad) in enumerate(_requests(case)):
        o = _exact_one(sub, seed + 13 * i)
        out.append([o[0], o[2], o[3]] if grad else o[:2])
    return out
