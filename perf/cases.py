"""Performance cases: what a user of this library has it do, through its public entry points.

Wavefield cases run ``Context.forward`` (synthetic data for one medium) or one evaluation
of the differentiable misfit (``autograd.misfit`` and its backward: forward sweep,
adjoint sweep, gradient integrals). Their time windows are short parts of the 300 to
4000 steps of a whole evaluation; a step does the same work at any time. Network cases
run the kernels of the learned gradient preconditioner layer by layer through the C ABI,
and its U-Net whole.

``exact`` gives the same results in 64 bits: the wave problem element by element on torch
tensors, the convolutions as sums over the 27 taps.
"""
from __future__ import annotations

import ctypes as C
import math
import random

import torch

# ---------------------------------------------------------------------------
# the cases


def listed():
    wave = dict(shots=1, batch=1, checkpoint=0)
    return [
        # forward modelling on the smallest box (8x8x4 elements and a 3-element PML): a few
        # microseconds of work per stage, one persistent launch for the sweep
        dict(name="forward_box_8x8x4", kind="forward", nx=8, ny=8, nz=4, npml=3, steps=100, nrec=5, sweep="persistent",
             medium="bump", **wave),
        # the same sweep as a replayed graph, with three shots in one batch
        dict(name="forward_box_3shots", kind="forward", nx=8, ny=8, nz=4, npml=3, steps=100, nrec=5, sweep="graph",
             medium="bump", shots=3, batch=3, checkpoint=0),
        # one gradient of the preconditioner study's inversions (16x16x8 and a 10-element PML)
        dict(name="gradient_16x16x8", kind="gradient", nx=16, ny=16, nz=8, npml=10, steps=100, nrec=8, sweep="graph",
             medium="grf", **wave),
        # an odd box with a ragged shot group and square-root checkpointing, launched directly
        dict(name="gradient_37x23x18", kind="gradient", nx=37, ny=23, nz=18, npml=6, steps=36, nrec=11, sweep="direct",
             medium="grf", shots=3, batch=2, checkpoint=-1),
        # the single-shot smooth-medium gradient, 64x64x32 and a 10-element PML
        dict(name="gradient_64x64x32", kind="gradient", nx=64, ny=64, nz=32, npml=10, steps=30, nrec=32, sweep="graph",
             medium="grf", **wave),
        # the batched layered gradient, 96x96x48 and a 10-element PML, four shots per launch
        dict(name="gradient_96x96x48", kind="gradient", nx=96, ny=96, nz=48, npml=10, steps=12, nrec=48, sweep="graph",
             medium="layered", shots=4, batch=4, checkpoint=0),
        # convolution layers of the U-Net at widths 28, 56, 112 on the material grid of the
        # 64x64x32 box: a full-resolution encoder layer forward, the decoder layer behind the
        # skip connection backward, a half-resolution layer's weight gradient
        dict(name="conv_forward_28", kind="conv_forward", cin=28, cout=28, D=65, H=129, W=129, relu=True),
        dict(name="conv_data_84_28", kind="conv_backward_data", cin=84, cout=28, D=65, H=129, W=129),
        dict(name="conv_weight_28", kind="conv_backward_weight", cin=28, cout=28, D=65, H=129, W=129),
        dict(name="conv_weight_56", kind="conv_backward_weight", cin=56, cout=56, D=33, H=65, W=65),
        # one network update of the inversion: the whole U-Net on that grid
        dict(name="unet_forward_64x64x32", kind="unet_forward", w0=28, w1=56, w2=112, D=65, H=129, W=129),
        # the gradients of one training sample on the study's grid (17x33x33)
        dict(name="unet_train_16x16x8", kind="unet_gradients", w0=28, w1=56, w2=112, D=17, H=33, W=33),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "gradient", "gradient", "gradient", "conv_forward", "conv_backward_data",
                       "conv_backward_weight", "unet_forward", "unet_gradients"])
    if kind in ("forward", "gradient"):
        c = dict(kind=kind, nx=_log(rng, 6, 96), ny=_log(rng, 6, 96), nz=_log(rng, 4, 48), npml=rng.randint(2, 10))
        c["shots"] = rng.randint(1, 4)
        c["batch"] = rng.randint(1, c["shots"])
        c["checkpoint"] = rng.choice([0, 0, 0, -1, 5]) if kind == "gradient" else 0
        sweeps = 1 if kind == "forward" else (3 if c["checkpoint"] else 2)
        # 45 to 90 million node-steps per sweep at most, between 8 and 100 steps
        c["steps"] = max(8, min(100, int(rng.uniform(90e6, 180e6) / (_nodes(c) * c["shots"] * sweeps))))
        c["nrec"] = rng.randint(3, max(3, min(c["nx"], c["ny"]) // 2))
        c["sweep"] = rng.choice(["graph", "graph", "direct"])
        if kind == "forward" and _nodes(c) < 30000 and rng.random() < 0.5:
            c["sweep"] = "persistent"
        c["medium"] = rng.choice(["grf", "layered", "bump"])
        return c
    if kind == "unet_gradients":
        return dict(kind=kind, w0=rng.randint(8, 32), w1=rng.randint(16, 64), w2=rng.randint(32, 128),
                    D=_log(rng, 9, 25), H=_log(rng, 9, 41), W=_log(rng, 9, 41))
    if kind == "unet_forward":
        return dict(kind=kind, w0=rng.randint(8, 32), w1=rng.randint(16, 64), w2=rng.randint(32, 128),
                    D=_log(rng, 9, 65), H=_log(rng, 9, 129), W=_log(rng, 9, 129))
    c = dict(kind=kind, cin=_log(rng, 2, 112), cout=_log(rng, 2, 112), D=_log(rng, 5, 65), H=_log(rng, 5, 129),
             W=_log(rng, 5, 129))
    if kind == "conv_forward":
        c["relu"] = rng.random() < 0.8
    return c


def _nodes(c):
    return (2 * (c["nx"] + 2 * c["npml"]) + 1) * (2 * (c["ny"] + 2 * c["npml"]) + 1) * (2 * (c["nz"] + c["npml"]) + 1)


def work(case):
    """Bytes: each RK4 step reads its stage inputs and the step start and writes its stage
    outputs once (13 accesses per variable: 27 variables on PML nodes, 6 elsewhere); a
    gradient level reads two displacement fields and updates two FP64 accumulators per
    batch. Network layers: inputs, weights and outputs once. Flops: the convolutions' products
    and sums; per stage and node about 250 (interior) to 400 (PML)."""
    k = case["kind"]
    if k in ("forward", "gradient"):
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        nodes = _nodes(case)
        mat = (2 * nx + 1) * (2 * ny + 1) * (2 * nz + 1)
        pml = nodes - (2 * nx - 1) * (2 * ny - 1) * (2 * nz)
        sweeps = 1 if k == "forward" else (3 if case["checkpoint"] else 2)
        n = case["steps"] * case["shots"]
        b = sweeps * n * 13 * 4 * (27 * pml + 6 * (nodes - pml))
        if k == "gradient":
            b += n * 24 * mat + case["steps"] * -(-case["shots"] // case["batch"]) * 32 * mat
        return {"bytes": b, "flops": sweeps * n * 4 * (400 * pml + 250 * (nodes - pml))}
    vox = case["D"] * case["H"] * case["W"]
    if k.startswith("unet"):
        w0, w1, w2 = case["w0"], case["w1"], case["w2"]
        s1 = -(-case["D"] // 2) * -(-case["H"] // 2) * -(-case["W"] // 2)
        s2 = -(-case["D"] // 4) * -(-case["H"] // 4) * -(-case["W"] // 4)
        pairs = vox * (4 * w0 + w0 * w0 + (w1 + w0) * w0 + w0 * 2) + s1 * (w0 * w1 + w1 * w1 + (w2 + w1) * w1 + w1 * w1) + \
            s2 * (w1 * w2 + w2 * w2)
        grad = k == "unet_gradients"
        return {"bytes": vox * (4 + 2) * (2 + 4 * grad), "flops": 54 * pairs * (3 if grad else 1)}
    cin, cout = case["cin"], case["cout"]
    size = {"conv_forward": 2 * cin + 2 * cout, "conv_backward_data": 4 * cout + 4 * cin,
            "conv_backward_weight": 4 * cout + 2 * cin}[k]
    return {"bytes": vox * size, "flops": 54 * cin * cout * vox}


# ---------------------------------------------------------------------------
# inputs, from the seed alone

RHO, H_EL, ALPHA0, BETA0 = 2000.0, 1.0, 5.0, 400.0


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, device):
    return torch.Generator(device=device).manual_seed(int(seed) * 7919 + 11)


def _smooth_field(shape, corr, gen, device):
    """Gaussian random field of correlation length `corr` nodes, scaled to max |f| = 1."""
    f = torch.fft.fftn(torch.randn(shape, generator=gen, device=device))
    k = [torch.fft.fftfreq(n, device=device) for n in shape]
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    f = torch.fft.ifftn(f * torch.exp(-(math.pi * corr) ** 2 * k2)).real
    f -= f.mean()
    return f / f.abs().max()


def _velocities(case, gen, device):
    """(vs, vp) on the material grid [k][j][i], float32."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (2 * nz + 1, 2 * ny + 1, 2 * nx + 1)
    z, y, x = torch.meshgrid(*(0.5 * H_EL * torch.arange(n, device=device, dtype=torch.float32) for n in shape),
                             indexing="ij")
    r = lambda lo, hi: lo + (hi - lo) * torch.rand((), generator=gen, device=device)  # noqa: E731
    if case["medium"] == "grf":  # smooth random field, 20 % around Vs 200, Vp 400 m/s
        f = 1 + 0.2 * _smooth_field(shape, 16.0, gen, device)
        return 200.0 * f, 400.0 * f
    if case["medium"] == "layered":  # three layers with a sharp fast block, Poisson's ratio 0.3
        d = nz * H_EL * r(0.9, 1.1)
        vs = torch.where(z < d / 3, 150.0, torch.where(z < 2 * d / 3, 250.0, 400.0))
        cx, cy, cz = nx * H_EL * r(0.4, 0.6), ny * H_EL * r(0.4, 0.6), nz * H_EL * r(0.5, 0.8)
        s = 0.17 * min(nx, ny, 2 * nz) * H_EL
        vs = torch.where(((x - cx).abs() <= s) & ((y - cy).abs() <= s) & ((z - cz).abs() <= s), 500.0, vs)
        return vs, vs * math.sqrt(3.5)
    bump = 0.1 * torch.exp(-((x - nx * r(0.3, 0.7)) ** 2 + (y - ny * r(0.3, 0.7)) ** 2 + (z - 0.5 * nz) ** 2) / 4.5)
    f = torch.sqrt(1 + bump)
    return 200.0 * f, 400.0 * f


def _wave_inputs(case, seed):
    """Material, acquisition and observed traces of a wavefield case."""
    dev = _device()
    gen = _gen(seed, dev)
    vs, vp = _velocities(case, gen, dev)
    mu = (RHO * vs * vs).contiguous()
    lam = (RHO * vp * vp - 2 * mu).contiguous()
    rng = random.Random(int(seed) * 31 + 5)
    p, nx, ny = case["npml"], case["nx"], case["ny"]
    src = [(2 * p + rng.randint(1, 2 * nx - 1), 2 * p + rng.randint(1, 2 * ny - 1), 0) for _ in range(case["shots"])]
    dirs = [(rng.uniform(-0.3, 0.3), rng.uniform(-0.3, 0.3), 1.0) for _ in range(case["shots"])]
    n = case["nrec"]
    xs = [2 + round(i * (2 * nx - 4) / (n - 1)) for i in range(n)]
    ys = [2 + round(j * (2 * ny - 4) / (n - 1)) for j in range(n)]
    rec = [(2 * p + i, 2 * p + j, 0) for j in ys for i in xs]
    dt = 0.25 * H_EL / (500.0 * math.sqrt(3.5) if case["medium"] == "layered" else 480.0)
    T = dt * case["steps"]
    f0 = min(60.0, 4.0 / T)
    wavelet = (f0, min(1.5 / f0, 0.4 * T), 1.0e3)
    # smooth traces of the computed ones' size
    t = torch.linspace(0, 1, case["steps"] + 1, device=dev)[None, :, None, None]
    a, b, f = (torch.randn((case["shots"], 1, n * n, 3), generator=gen, device=dev) for _ in range(3))
    f = 1.0 + 3.0 * torch.sigmoid(f)
    obs = (1e-8 * (a * torch.sin(2 * math.pi * f * t) + b * torch.cos(2 * math.pi * f * t) * t)).float().contiguous()
    return dict(lam=lam, mu=mu, src=src, dirs=dirs, rec=rec, dt=dt, wavelet=wavelet, obs=obs)


def _he(cout, cin, gen, dev):
    return torch.randn((cout, cin, 27), generator=gen, device=dev) * math.sqrt(2.0 / (27 * cin))


def _layer_inputs(case, seed):
    """Activations as they leave a ReLU (half of them zero), He-scaled weights, output gradients."""
    dev = _device()
    gen = _gen(seed, dev)
    cin, cout, grid = case["cin"], case["cout"], (case["D"], case["H"], case["W"])
    s = {"w": _he(cout, cin, gen, dev).to(torch.bfloat16), "b": 0.1 * torch.randn(cout, generator=gen, device=dev)}
    if case["kind"] != "conv_backward_data":
        s["x"] = torch.relu(torch.randn((cin, *grid), generator=gen, device=dev)).to(torch.bfloat16)
    if case["kind"] != "conv_forward":
        dy = torch.randn((cout, *grid), generator=gen, device=dev)
        s["dy"] = 1e-4 * dy * (torch.rand((cout, *grid), generator=gen, device=dev) < 0.5)
    return s


_UNET = ("e0a", "e0b", "e1a", "e1b", "ba", "bb", "d1a", "d1b", "d0a", "d0b")


def _unet_channels(case):
    w0, w1, w2 = case["w0"], case["w1"], case["w2"]
    return dict(e0a=(4, w0), e0b=(w0, w0), e1a=(w0, w1), e1b=(w1, w1), ba=(w1, w2), bb=(w2, w2), d1a=(w2 + w1, w1),
                d1b=(w1, w1), d0a=(w1 + w0, w0), d0b=(w0, 2))


def _unet_inputs(case, seed):
    """Trained-network-like weights and a sample: scaled gradients, relative model perturbations."""
    dev = _device()
    gen = _gen(seed, dev)
    grid = (case["D"], case["H"], case["W"])
    weights = {n: (_he(co, ci, gen, dev), 0.05 * torch.randn(co, generator=gen, device=dev))
               for n, (ci, co) in _unet_channels(case).items()}
    amp = (1.0, 1.0, 0.2, 0.2)
    x = torch.stack([a * _smooth_field(grid, 3.0, gen, dev) for a in amp]).contiguous()
    dy = torch.randn((2, *grid), generator=gen, device=dev) * (0.1 / (2 * grid[0] * grid[1] * grid[2]))
    return weights, x, dy


# ---------------------------------------------------------------------------
# a user's program


class State:
    """What a program holds between calls."""

    def __init__(self, **kw):
        self.__dict__.update(kw)


def prepare(case, seed):
    from paper_1504_08340_gb300 import Context, load_library

    k = case["kind"]
    if k in ("forward", "gradient"):
        v = _wave_inputs(case, seed)
        ctx = Context(case["nx"], case["ny"], case["nz"], case["npml"], H_EL, v["dt"], case["steps"], rho=RHO,
                      alpha0=ALPHA0, beta0=BETA0)
        ctx.set_sources(v["src"], v["dirs"], "ricker", v["wavelet"])
        ctx.set_receivers(v["rec"])
        if case["batch"] > 1:
            ctx.set_shot_batch(case["batch"])
        if case["checkpoint"]:
            ctx.set_checkpointing(case["checkpoint"])
        if case["sweep"] == "graph":
            ctx.set_graphs(True)
        elif case["sweep"] == "persistent":
            ctx.set_persistent(True)
        return State(kind=k, ctx=ctx, lam=v["lam"], mu=v["mu"], obs=v["obs"], shots=case["shots"],
                     out=torch.empty(ctx.trace_shape(case["shots"]), dtype=torch.float32, device="cuda"))
    if k.startswith("unet"):
        from paper_1504_08340_gb300.precond import UNet

        weights, x, dy = _unet_inputs(case, seed)
        net = UNet(4, 2, (case["w0"], case["w1"], case["w2"]), (case["D"], case["H"], case["W"]))
        for n, (w, b) in weights.items():
            net.layer[n].w32.copy_(w)
            net.layer[n].w.copy_(w.to(torch.bfloat16))
            net.layer[n].b.copy_(b)
        return State(kind=k, net=net, x=x, dy=dy)
    s = _layer_inputs(case, seed)
    lib = load_library()
    cin, cout, grid = case["cin"], case["cout"], (case["D"], case["H"], case["W"])
    st = State(kind=k, lib=lib, dims=(cin, cout, *grid), relu=int(case.get("relu", False)), **s)
    if k == "conv_forward":
        st.y = torch.empty((cout, *grid), dtype=torch.bfloat16, device="cuda")
    elif k == "conv_backward_data":
        st.dx = torch.empty((cin, *grid), dtype=torch.float32, device="cuda")
    else:
        st.dw = torch.empty((cout, cin, 27), dtype=torch.float32, device="cuda")
        st.db = torch.empty(cout, dtype=torch.float32, device="cuda")
        n = lib.fwi_nn_conv3d_backward_weight_work(*st.dims)
        st.work = torch.empty(int(n), dtype=torch.float32, device="cuda")
    return st


def _p(t):
    return C.c_void_p(t.data_ptr())


def _ok(status):
    if status != 0:
        raise RuntimeError(f"kernel failed with status {status}")


def run(s):
    if s.kind == "forward":
        s.ctx.set_material(s.lam, s.mu)
        return s.ctx.forward(0, s.shots, out=s.out)
    if s.kind == "gradient":
        from paper_1504_08340_gb300.autograd import misfit

        lam, mu = s.lam.detach().requires_grad_(), s.mu.detach().requires_grad_()
        J = misfit(s.ctx, lam, mu, s.obs, 0, s.shots)
        J.backward()
        return {"J": J.item(), "lambda": lam.grad, "mu": mu.grad}
    if s.kind == "unet_forward":
        return s.net.forward(s.net.to_bf16(s.x))["y"]
    if s.kind == "unet_gradients":
        a = s.net.forward(s.net.to_bf16(s.x))
        s.net.backward(a, s.dy)
        return {"y": a["y"], "w": [s.net.layer[n].g_w32 for n in _UNET], "b": [s.net.layer[n].g_b for n in _UNET]}
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    if s.kind == "conv_forward":
        _ok(s.lib.fwi_nn_conv3d_forward(_p(s.x), _p(s.w), _p(s.b), *s.dims, s.relu, _p(s.y), stream))
        return s.y
    if s.kind == "conv_backward_data":
        _ok(s.lib.fwi_nn_conv3d_backward_data(_p(s.dy), _p(s.w), *s.dims, _p(s.dx), stream))
        return s.dx
    _ok(s.lib.fwi_nn_conv3d_backward_weight(_p(s.dy), _p(s.x), *s.dims, _p(s.dw), _p(s.db), _p(s.work), stream))
    return {"dw": s.dw, "db": s.db}


# ---------------------------------------------------------------------------
# the same in 64 bits

_VOIGT = ((0, 5, 4), (5, 1, 3), (4, 3, 2))  # xx yy zz yz xz xy


class Wave:
    """The semi-discrete system of the hybrid formulation, element by element: 27-node
    elements with Lobatto quadrature (points at the nodes), displacements in the interior,
    displacements and stresses in the PML. Node fields are [...][k][j][i]; element fields
    [...][ez][ey][ex][z][y][x] with the element's 27 nodes last."""

    def __init__(self, case, lam, mu, device=None):
        self.dev = dev = device or _device()
        p = case["npml"]
        ne = (case["nz"] + p, case["ny"] + 2 * p, case["nx"] + 2 * p)  # elements along z, y, x
        self.nn = tuple(2 * n + 1 for n in ne)
        self.lo, self.hi = (0, p, p), (case["nz"], p + case["ny"], p + case["nx"])
        f64 = dict(dtype=torch.float64, device=dev)
        al, be = [], []
        for ax in range(3):
            c = torch.arange(self.nn[ax], **f64)
            depth = 0.5 * H_EL * ((2 * self.lo[ax] - c).clamp_min(0) + (c - 2 * self.hi[ax]).clamp_min(0))
            r = (depth / (p * H_EL)) ** 2 if p else depth
            shape = [1, 1, 1]
            shape[ax] = -1
            al.append((1 + ALPHA0 * r).view(shape))
            be.append((BETA0 * r).view(shape))
        (az, ay, ax_), (bz, by, bx) = al, be
        # coefficients of s^2, s, 1, 1/s of the product of the stretch functions
        a = ax_ * ay * az
        self.inv_a = 1 / a
        self.damp = torch.stack([bx * by * bz, ax_ * by * bz + bx * ay * bz + bx * by * az,
                                 ax_ * ay * bz + ax_ * by * az + bx * ay * az]) / a  # d, c, b over a
        # Lambda^{w, p, e}_jj: the two factors across axis j, j = x, y, z
        L = [[B * E, A * E + B * D, A * D] for A, B, D, E in ((ay, by, az, bz), (ax_, bx, az, bz), (ax_, bx, ay, by))]
        self.L = [[v.expand(self.nn) for v in row] for row in L]
        rd = torch.zeros(ne, **f64)
        rd[tuple(slice(self.lo[i], self.hi[i]) for i in range(3))] = 1.0
        self.rd = rd[..., None, None, None]
        w = torch.tensor([1 / 3, 4 / 3, 1 / 3], **f64)
        self.wq = (0.5 * H_EL) ** 3 * w[:, None, None] * w[:, None] * w
        one = torch.ones((*ne, 3, 3, 3), **f64)
        self.inv_mass = 1 / (RHO * a * self._scatter(one * self.wq))
        n_pml = self._scatter(one * (1 - self.rd))
        self.pml = (n_pml > 0).double()
        self.inv_n_pml = 1 / n_pml.clamp_min(1)
        free = torch.ones(self.nn, **f64)
        free[-1], free[:, 0], free[:, -1], free[:, :, 0], free[:, :, -1] = 0, 0, 0, 0, 0
        self.free = free
        idx = [(torch.arange(self.nn[i], device=dev) - 2 * self.lo[i]).clamp(0, 2 * (self.hi[i] - self.lo[i]))
               for i in range(3)]
        self.lam, self.mu = (f.to(**f64)[idx[0]][:, idx[1]][:, :, idx[2]] for f in (lam, mu))

    @staticmethod
    def _elements(f):
        """Node field -> element field (a view)."""
        return f.unfold(-3, 3, 2).unfold(-3, 3, 2).unfold(-3, 3, 2)

    def _scatter(self, e):
        """Element field -> node sums."""
        out = torch.zeros((*e.shape[:-6], *self.nn), dtype=torch.float64, device=self.dev)
        at = [slice(q, n - 2 + q, 2) for n in self.nn for q in range(3)]
        for a in range(3):
            for b in range(3):
                for c in range(3):
                    out[..., at[a], at[3 + b], at[6 + c]] += e[..., a, b, c]
        return out

    @staticmethod
    def _derivative(e, axis):
        """Element-wise derivative along x, y or z (axis 0, 1, 2) at the element's nodes."""
        v0, v1, v2 = e.unbind(-1 - axis)
        return torch.stack([-3 * v0 + 4 * v1 - v2, v2 - v0, v0 - 4 * v1 + 3 * v2], dim=-1 - axis) / H_EL

    def _against_gradient(self, g, axis):
        """sum over the points q of w_q g(q) d phi / d axis (q), by element node."""
        g0, g1, g2 = (self.wq * g).unbind(-1 - axis)
        return torch.stack([-3 * g0 - g1 + g2, 4 * (g0 - g2), -g0 + g1 + 3 * g2], dim=-1 - axis) / H_EL

    def rate(self, Y, load=None):
        """Time derivative of Y = [shot][level 0 history, 1 value, 2 rate][3 displacements,
        6 stresses]; load: (node index arrays k, j, i [shot][point], forces [shot][point][3])."""
        el = self._elements
        u, S = Y[:, :, :3], Y[:, :, 3:]
        G = [self._derivative(el(u), j) for j in range(3)]  # d u / d x_j: [shot][level][i]
        # interior elements: - int sigma : grad phi
        lam, mu = el(self.lam) * self.rd, el(self.mu) * self.rd
        g = [[G[j][:, 1, i] for j in range(3)] for i in range(3)]
        tr = lam * (g[0][0] + g[1][1] + g[2][2])
        force = []
        for i in range(3):
            f = 0.0
            for j in range(3):
                s = mu * (g[i][j] + g[j][i])
                # PML elements: - int (Lambda S) : grad phi
                q = sum(self.L[j][lv] * S[:, lv, _VOIGT[i][j]] for lv in range(3))
                f = f - self._against_gradient((s + tr if i == j else s) + (1 - self.rd) * el(q), j)
            force.append(f)
        force = self._scatter(torch.stack(force, dim=1))
        # PML elements: the stretched strain rates, averaged over the elements around a node
        H = torch.stack([sum(el(self.L[j][lv])[None, None] * G[j][:, lv] for lv in range(3)) for j in range(3)], dim=2)
        H = self._scatter((1 - self.rd) * H) * self.inv_n_pml  # [shot][i][j]
        del G, g
        if load is not None:
            (k, j, i), f = load
            shot = torch.arange(len(k), device=self.dev)[:, None].expand_as(k)
            for c in range(3):
                force[:, c].index_put_((shot, k, j, i), f[..., c], accumulate=True)
        tau = [None] * 6
        trace = self.lam * (H[:, 0, 0] + H[:, 1, 1] + H[:, 2, 2])
        for i in range(3):
            for j in range(i, 3):
                t = self.mu * (H[:, i, j] + H[:, j, i])
                tau[_VOIGT[i][j]] = t + trace if i == j else t
        out = torch.empty_like(Y)
        out[:, 0] = Y[:, 1] * self.pml
        out[:, 1] = Y[:, 2]
        decay = (self.damp[:, None] * Y).sum(dim=1)
        out[:, 2, :3] = (force * self.inv_mass - decay[:, :3]) * self.free
        out[:, 2, 3:] = (torch.stack(tau, dim=1) * self.inv_a - decay[:, 3:]) * self.pml
        return out

    def step(self, Y, dt, loads):
        """One classic RK4 step; loads at t, t + dt/2, t + dt."""
        acc, k = Y.clone(), None
        for w, at, ld in ((1, 0.0, 0), (2, 0.5, 1), (2, 0.5, 1), (1, 1.0, 2)):
            k = self.rate(Y if k is None else Y + at * dt * k, loads[ld])
            acc += (w * dt / 6) * k
        return acc

    def integrand(self, u, w):
        """Node sums over the interior elements of w_q (div w)(div u) and w_q 2 eps(w) : eps(u),
        summed over the shots."""
        U, V = ([self._derivative(self._elements(f), j) for j in range(3)] for f in (u, w))
        div = [sum(g[j][:, j] for j in range(3)) for g in (U, V)]
        e = sum((U[j][:, i] + U[i][:, j]) * (V[j][:, i] + V[i][:, j]) for i in range(3) for j in range(3)) / 2
        both = torch.stack([(div[0] * div[1]).sum(0), e.sum(0)]) * (self.rd * self.wq)
        return self._scatter(both)[(slice(None), *(slice(2 * a, 2 * b + 1) for a, b in zip(self.lo, self.hi)))]


def _ricker(t, f0, t0, amp):
    a = (math.pi * f0 * (t - t0)) ** 2
    return amp * (1 - 2 * a) * math.exp(-a)


def exact_wave(case, v, device=None):
    wave = Wave(case, v["lam"], v["mu"], device)
    dev, dt, N, shots = wave.dev, v["dt"], case["steps"], case["shots"]
    f64 = dict(dtype=torch.float64, device=dev)
    index = lambda pts: tuple(torch.tensor([[q[a] for q in r] for r in pts], device=dev) for a in (2, 1, 0))  # noqa: E731
    at, rec = index([[q] for q in v["src"]]), index([v["rec"]] * shots)
    dirs = torch.tensor(v["dirs"], **f64)[:, None]
    shot = torch.arange(shots, device=dev)[:, None].expand_as(rec[0])
    sample = lambda Y: torch.stack([Y[:, 1, c][(shot, *rec)] for c in range(3)], dim=-1)  # noqa: E731
    Y = torch.zeros((shots, 3, 9, *wave.nn), **f64)
    traces, hist = [sample(Y)], [None]
    grad = case["kind"] == "gradient"
    for n in range(N):
        Y = wave.step(Y, dt, [(at, dirs * _ricker((n + 0.5 * h) * dt, *v["wavelet"])) for h in range(3)])
        traces.append(sample(Y))
        if grad:
            hist.append(Y[:, 1, :3].clone())
    traces = torch.stack(traces, dim=1)
    if not grad:
        return traces
    e = traces - v["obs"].to(dev).double()
    wt = torch.ones(N + 1, **f64)
    wt[0] = wt[-1] = 0.5
    J = 0.5 * dt * float((wt[:, None, None] * e * e).sum())
    # adjoint in reversed time, with the stresses as tau of the adjoint ones: the same
    # system, loaded by the residuals
    W = torch.zeros_like(Y)
    total = 0.0
    for n in range(N):
        a, b = e[:, N - n], e[:, N - n - 1]
        W = wave.step(W, dt, [(rec, a), (rec, 0.5 * (a + b)), (rec, b)])
        if N - n - 1 > 0:
            total = total - dt * wave.integrand(hist[N - n - 1], W[:, 1, :3])
    return {"J": J, "lambda": total[0], "mu": total[1]}


def _taps(D, H, W):
    """(tap, slices of the output grid, slices of the input grid) of the 27 taps."""
    def span(d, n):
        return slice(max(0, -d), n - max(0, d)), slice(max(0, d), n + min(0, d))

    for t in range(27):
        sp = [span(d, n) for d, n in zip((t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1), (D, H, W))]
        if all(s[0].start < s[0].stop for s in sp):
            yield t, tuple(s[0] for s in sp), tuple(s[1] for s in sp)


def _conv(x, w, b):
    y = torch.zeros((w.shape[0], *x.shape[1:]), dtype=torch.float64, device=x.device)
    for t, o, i in _taps(*x.shape[1:]):
        v = x[(slice(None), *i)]
        y[(slice(None), *o)] += (w[:, :, t] @ v.reshape(v.shape[0], -1)).view(w.shape[0], *v.shape[1:])
    return y if b is None else y + b[:, None, None, None]


def _conv_data(dy, w):
    dx = torch.zeros((w.shape[1], *dy.shape[1:]), dtype=torch.float64, device=dy.device)
    for t, o, i in _taps(*dy.shape[1:]):
        v = dy[(slice(None), *o)]
        dx[(slice(None), *i)] += (w[:, :, t].T @ v.reshape(v.shape[0], -1)).view(w.shape[1], *v.shape[1:])
    return dx


def _conv_weight(dy, x):
    dw = torch.zeros((dy.shape[0], x.shape[0], 27), dtype=torch.float64, device=x.device)
    for t, o, i in _taps(*x.shape[1:]):
        a, v = dy[(slice(None), *o)], x[(slice(None), *i)]
        dw[:, :, t] = a.reshape(a.shape[0], -1) @ v.reshape(v.shape[0], -1).T
    return dw


def _cell_counts(grid, dev):
    n = [torch.tensor([min(2, g - 2 * q) for q in range((g + 1) // 2)], dtype=torch.float64, device=dev) for g in grid]
    return n[0][:, None, None] * n[1][None, :, None] * n[2][None, None, :]


def _cell_sum(x):
    D, H, W = x.shape[1:]
    x = torch.nn.functional.pad(x, (0, W % 2, 0, H % 2, 0, D % 2))
    return sum(x[:, a::2, b::2, c::2] for a in (0, 1) for b in (0, 1) for c in (0, 1))


def _cell_spread(x, grid):
    for ax in (1, 2, 3):
        x = x.repeat_interleave(2, dim=ax)
    return x[:, :grid[0], :grid[1], :grid[2]]


def exact_unet(case, weights, x, dy):
    """The U-Net on BF16 weights and input, with the stored activations rounded to BF16 as the
    network defines them and every sum in 64 bits; the gradients with respect to the weights
    and biases when asked."""
    stored = lambda v: v.to(torch.bfloat16).double()  # noqa: E731
    p = {n: (w.to(torch.bfloat16).double(), b.double()) for n, (w, b) in weights.items()}
    a = {}

    def conv(n, v, relu=True):
        y = _conv(v, *p[n])
        a[n] = (v, stored(torch.relu(y)) if relu else y)
        return a[n][1]

    g0 = x.shape[1:]
    e0 = conv("e0b", conv("e0a", stored(x)))
    g1 = tuple((n + 1) // 2 for n in g0)
    c0, c1 = _cell_counts(g0, x.device), _cell_counts(g1, x.device)
    e1 = conv("e1b", conv("e1a", stored(_cell_sum(e0) / c0)))
    bb = conv("bb", conv("ba", stored(_cell_sum(e1) / c1)))
    d1 = conv("d1b", conv("d1a", torch.cat([_cell_spread(bb, g1), e1])))
    y = conv("d0b", conv("d0a", torch.cat([_cell_spread(d1, g0), e0])), relu=False)
    if case["kind"] == "unet_forward":
        return y
    gw, gb = {}, {}

    def back(n, g, need=True):
        v, out = a[n]
        if n != "d0b":
            g = g * (out > 0)
        gw[n], gb[n] = _conv_weight(g, v), g.sum(dim=(1, 2, 3))
        return _conv_data(g, p[n][0]) if need else None

    w1, w2 = case["w1"], case["w2"]
    g = back("d0a", back("d0b", dy.double()))
    g, skip0 = g[:w1], g[w1:]
    g = back("d1a", back("d1b", _cell_sum(g)))
    g, skip1 = g[:w2], g[w2:]
    g = back("ba", back("bb", _cell_sum(g)))
    g = back("e1a", back("e1b", skip1 + _cell_spread(g / c1, g1)))
    back("e0a", back("e0b", skip0 + _cell_spread(g / c0, g0)), need=False)
    return {"y": y, "w": [gw[n] for n in _UNET], "b": [gb[n] for n in _UNET]}


def exact(case, seed):
    k = case["kind"]
    if k in ("forward", "gradient"):
        sweeps = 1 if k == "forward" else 2
        if _nodes(case) * case["shots"] * case["steps"] * sweeps > 400e6:  # over about 20 seconds
            return None
        return exact_wave(case, _wave_inputs(case, seed))
    if k.startswith("unet"):
        return exact_unet(case, *_unet_inputs(case, seed))
    s = _layer_inputs(case, seed)
    if k == "conv_forward":
        y = _conv(s["x"].double(), s["w"].double(), s["b"].double())
        return torch.relu(y) if case["relu"] else y
    if k == "conv_backward_data":
        return _conv_data(s["dy"].double(), s["w"].double())
    return {"dw": _conv_weight(s["dy"].double(), s["x"].double()), "db": s["dy"].double().sum(dim=(1, 2, 3))}
