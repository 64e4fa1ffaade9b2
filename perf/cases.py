"""Performance cases of the registration framework: what its users have it do,
through its public entry points, over the sizes, data types and options that
they use, with a 64-bit restatement of every result in plain torch.

A case is a dict of plain values; ``kind`` says which path it takes:

* ``kernels``: the off-grid kernels alone on a ``kernels_only`` context, as a
  program that brings its own solver calls them: RK2 characteristic, ``fields``
  interpolations at it, 8th-order gradient.
* ``newton``: one linearisation of the Gauss-Newton method through the solver
  interface: gradient, Hessian matvec and spectral preconditioner.
* ``precond``: the two-level zero-velocity preconditioner at a linearisation.
* ``register``: a whole registration with a fixed schedule (``gn``
  Gauss-Newton steps of ``pcg`` PCG iterations each) from v = 0.
* ``evaluate``: the acceptance test of a velocity: objective and mismatch,
  extrema of the Jacobian determinant, and the carried template.
* ``transport``: forward (state) or adjoint solve of one image.
* ``vjp``: differentiable transport as a training step uses it: forward pass
  and gradients of the image and the velocity through autograd.
* ``conv``: one 3x3x3 layer of the warm-start network in training: forward,
  activation gradient, weight and bias gradient, input gradient.
"""
import math

import torch

from paper_2209_08189_gb300 import claire, net

STORAGE = {"f32": claire.STORAGE_F32, "f16": claire.STORAGE_F16, "bf16": claire.STORAGE_BF16}
ORDER = {"cubic": claire.INTERP_CUBIC, "linear": claire.INTERP_LINEAR, "bspline": claire.INTERP_BSPLINE}
BETA_V, BETA_W, SLOPE = 1e-2, 1e-4, 0.1


def _case(kind, n, **kw):
    c = {"kind": kind, "n1": n[0], "n2": n[1], "n3": n[2]}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest grid that tests and examples use: a call is a handful of
        # launches and one read-back, so latency is all of it.
        dict(_case("kernels", (32, 32, 32), interp="cubic", nt=4, fields=1, vmax=0.5), name="kernels_32"),
        # The kernels at the size of a high-resolution scan, three fields
        # (a velocity) carried at once, large CFL number.
        dict(_case("kernels", (512, 512, 512), interp="cubic", nt=4, fields=3, vmax=0.5), name="kernels_512"),
        # The benchmark's grid, half way through a solve: what each outer and
        # inner iteration of a registration consists of.
        dict(_case("newton", (256, 256, 256), interp="cubic", nt=4, storage="f32", lowmem=0, vmax=0.4),
             name="newton_256"),
        # A clinical volume as it comes from a template (not a power of two, no
        # multiple of four along x3), 16-bit storage.
        dict(_case("newton", (182, 218, 182), interp="cubic", nt=4, storage="f16", lowmem=0, vmax=0.4),
             name="newton_182x218x182_f16"),
        # The paper's preconditioner on the benchmark's grid (inner solves on 128^3).
        dict(_case("precond", (256, 256, 256), interp="cubic", nt=4, storage="f32", vmax=0.4), name="precond_256"),
        # A small registration (64^3, the first configuration): five
        # Gauss-Newton steps of ten PCG iterations, many short launches.
        dict(_case("register", (64, 64, 64), interp="cubic", nt=4, storage="f32", precond="spectral", gn=5, pcg=10),
             name="register_64"),
        # The benchmark's registration, two Gauss-Newton steps of five PCG iterations.
        dict(_case("register", (256, 256, 256), interp="cubic", nt=4, storage="f32", precond="spectral", gn=2, pcg=5),
             name="register_256"),
        # Checking a candidate velocity (parameter search, acceptance).
        dict(_case("evaluate", (256, 256, 256), interp="cubic", nt=4, storage="f32", vmax=0.4), name="evaluate_256"),
        # Carrying an image with a known velocity in the paper's clinical
        # setting: 256 x 300 x 256, trilinear, eight time steps.
        dict(_case("transport", (256, 300, 256), interp="linear", nt=8, adjoint=0, vmax=0.5),
             name="transport_256x300x256_linear"),
        # The mismatch term of a training step at the training grid.
        dict(_case("vjp", (128, 128, 128), interp="cubic", nt=4, recompute=0, vmax=0.5), name="vjp_128"),
        # The network's finest layer (16 -> 16 channels) at the training batch.
        dict(_case("conv", (128, 128, 128), batch=4, cin=16, cout=16), name="conv_train_128_16x16"),
        # The decoder layer after the first skip connection (96 -> 32 channels).
        dict(_case("conv", (64, 64, 64), batch=4, cin=96, cout=32), name="conv_train_64_96x32"),
    ]


def _even(rng, lo, hi):
    """An even extent, log-uniform in [lo, hi]; whole multiples of 32 now and then."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    step = rng.choice((2, 2, 4, 32 if x >= 48 else 2))
    return min(hi, max(lo, int(round(x / step)) * step))


def _grid(rng, lo, hi):
    """Three extents near one another, as scans are."""
    base = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    near = lambda: _even(rng, max(lo, 0.75 * base), min(hi, 1.3 * base + 2))
    return tuple(int(max(lo, x // 2 * 2)) for x in (near(), near(), near()))


def draw(rng):
    kind = rng.choice(("kernels", "newton", "newton", "precond", "register", "evaluate", "transport", "vjp", "conv"))
    vmax = round(rng.uniform(0.15, 0.6), 2)
    order = rng.choice(("cubic", "cubic", "linear", "bspline"))
    if kind == "conv":
        level = rng.choice((0, 1, 2, 3))
        base = rng.choice((64, 128))
        chans = (16, 32, 64, 128)
        pairs = [(chans[max(level - 1, 0)], chans[level]), (chans[level], chans[level])]
        if level < 3:
            pairs.append((chans[level] + chans[level + 1], chans[level]))
        cin, cout = rng.choice(pairs)
        return _case("conv", (base >> level,) * 3, batch=rng.choice((1, 2, 3)), cin=cin, cout=cout)
    if kind == "kernels":
        order = "linear" if order == "linear" else "cubic"
        return _case(kind, _grid(rng, 32, 480), interp=order, nt=4, fields=rng.choice((1, 2, 3, 4)), vmax=vmax)
    if kind == "newton":
        sto = "f32" if order == "bspline" else rng.choice(("f32", "f32", "f16", "bf16"))
        return _case(kind, _grid(rng, 32, 240), interp=order, nt=rng.choice((4, 4, 8)), storage=sto,
                     lowmem=rng.choice((0, 0, 1)), vmax=vmax)
    if kind == "precond":
        n = tuple(max(32, x // 4 * 4) for x in _grid(rng, 32, 240))
        return _case(kind, n, interp="cubic", nt=4, storage=rng.choice(("f32", "f16")), vmax=vmax)
    if kind == "register":
        two = rng.choice((False, True))
        n = _grid(rng, 32, 192)
        if two:
            n = tuple(max(32, x // 4 * 4) for x in n)
        return _case(kind, n, interp=rng.choice(("cubic", "linear")), nt=4, storage="f32",
                     precond="two_level" if two else "spectral", gn=rng.choice((1, 2)), pcg=rng.choice((2, 3, 5)))
    if kind == "evaluate":
        return _case(kind, _grid(rng, 32, 240), interp=order, nt=4, storage="f32", vmax=vmax)
    if kind == "transport":
        return _case(kind, _grid(rng, 32, 320), interp=order, nt=rng.choice((4, 8)), adjoint=rng.choice((0, 1)),
                     vmax=vmax)
    return _case(kind, _grid(rng, 32, 192), interp=order, nt=4, recompute=rng.choice((0, 1)), vmax=vmax)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _axes(n):
    return [torch.arange(s, device="cuda", dtype=torch.float32) * (2.0 * math.pi / s) for s in n]


def _velocity(n, g, vmax, kmax=6):
    """Band-limited random field, |k| <= kmax, spectrum ~ 1/sqrt(1 + |k|^2), max |v| = vmax."""
    kmax = min(kmax, min(n) // 6)
    ks = [torch.fft.fftfreq(n[0], 1.0 / n[0], device="cuda"), torch.fft.fftfreq(n[1], 1.0 / n[1], device="cuda"),
          torch.fft.rfftfreq(n[2], 1.0 / n[2], device="cuda")]
    kk = ks[0][:, None, None] ** 2 + ks[1][None, :, None] ** 2 + ks[2][None, None, :] ** 2
    idx = torch.nonzero(((kk >= 1.0) & (kk <= kmax * kmax)).reshape(-1)).reshape(-1)
    amp = 1.0 / torch.sqrt(1.0 + kk.reshape(-1)[idx])
    v = torch.empty((3,) + tuple(n), device="cuda")
    for c in range(3):
        spec = torch.zeros(kk.numel(), dtype=torch.complex64, device="cuda")
        z = torch.randn((2, idx.numel()), device="cuda", generator=g)
        spec[idx] = torch.complex(z[0], z[1]) * amp
        v[c] = torch.fft.irfftn(spec.reshape(kk.shape), s=tuple(n), norm="forward")
    return v * (vmax / torch.sqrt((v * v).sum(0).max()))


def _labels(n, g, shift):
    """Four nested ellipsoids with edges of about a voxel on a zero background
    (the clinical-size workload's label image), seen through a smooth shift."""
    x = _axes(n)
    r = torch.rand(6, device="cuda", generator=g)
    w = 1.5 * 2.0 * math.pi / min(n)
    y = [x[0][:, None, None], x[1][None, :, None], x[2][None, None, :]]
    s = [shift * torch.sin(y[(c + 1) % 3] + 6.0 * r[c]) for c in range(3)]
    q = 0.0
    for c, rad in enumerate((2.2, 1.9, 2.4)):
        q = q + ((y[c] + s[c] - math.pi - 0.2 * (2.0 * r[c] - 1.0)) / (rad * (0.9 + 0.2 * r[3 + c]))) ** 2
    q = torch.sqrt(q)
    m, prev = torch.zeros(tuple(n), device="cuda"), 0.0
    for level, scale in zip((0.2, 0.5, 0.8, 1.0), (1.0, 0.75, 0.5, 0.28)):
        m += (level - prev) * 0.5 * (1.0 + torch.tanh((scale - q) * (2.0 / w)))
        prev = level
    return m


def _images(n, seed):
    """A pair: the labels, and the labels shifted; additive noise of 0.02 on both."""
    g0, g1, g = _gen(seed), _gen(seed), _gen(seed + 7919)
    m0, m1 = _labels(n, g0, 0.0), _labels(n, g1, 0.25)
    noise = lambda: 0.02 * torch.randn(tuple(n), device="cuda", generator=g)
    return (m0 + noise()).contiguous(), (m1 + noise()).contiguous()


def _inputs(case, seed):
    """Device inputs of a case, from its seed alone."""
    n = (case["n1"], case["n2"], case["n3"])
    g = _gen(1000003 * (seed + 1))
    k = case["kind"]
    if k == "conv":
        vol = (case["batch"],) + n
        bf = lambda *s: torch.randn(s, device="cuda", generator=g).to(torch.bfloat16)
        ci, co = case["cin"], case["cout"]
        return {"x": bf(*vol, ci), "dy": bf(*vol, co),
                "w": (torch.randn((co, 27, ci), device="cuda", generator=g) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16),
                "b": 0.1 * torch.randn(co, device="cuda", generator=g)}
    d = {}
    if k != "register":
        d["v"] = _velocity(n, g, case["vmax"])
    if k == "kernels":
        d["f"] = torch.rand((case["fields"],) + n, device="cuda", generator=g)
    else:
        d["m0"], d["m1"] = _images(n, seed)
    if k == "newton":
        d["vt"] = _velocity(n, g, 0.1)
        d["r"] = _velocity(n, g, 0.05, kmax=8) + 1e-3 * torch.randn((3,) + n, device="cuda", generator=g)
    if k == "precond":
        d["r"] = _velocity(n, g, 0.05, kmax=8) + 1e-3 * torch.randn((3,) + n, device="cuda", generator=g)
    if k == "vjp":
        d["gbar"] = d["m0"] - d["m1"]  # a mismatch residual
    return d


def prepare(case, seed):
    n = (case["n1"], case["n2"], case["n3"])
    s = {"case": case, "in": _inputs(case, seed)}
    i, k = s["in"], case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if k == "conv":
        co, _, ci = i["w"].shape
        vol = (case["batch"],) + n
        s["wf"] = torch.empty((ci, 27, co), dtype=torch.bfloat16, device="cuda")
        net.conv3d_flip(i["w"], co, ci, s["wf"], stream)
        s["chunks"] = net.wgrad_chunks(ci, co, vol)
        s["part"] = torch.empty(s["chunks"] * co * 27 * ci, device="cuda")
        s["partb"] = torch.empty(s["chunks"] * co, device="cuda")
        act = lambda c: torch.empty(vol + (c,), dtype=torch.bfloat16, device="cuda")
        s["y"], s["dp"], s["dx"] = act(co), act(co), act(ci)
        s["dw"], s["db"] = torch.empty((co, 27, ci), device="cuda"), torch.empty(co, device="cuda")
        s["stream"] = stream
        return s
    opts = {"interp": ORDER[case["interp"]]}
    if k == "kernels":
        s["ctx"] = claire.Context(n, BETA_V, case["nt"], stream=stream, kernels_only=1, **opts)
        s["d"], s["out"] = torch.empty_like(i["v"]), torch.empty_like(i["f"])
        s["grad"] = torch.empty((3,) + n, device="cuda")
        return s
    opts.update(beta_w=BETA_W, storage=STORAGE[case.get("storage", "f32")], lowmem=case.get("lowmem", 0))
    if k == "register":
        opts.update(gtol=0.0, max_gn=case["gn"], max_pcg=case["pcg"], pcg_fixed=1)
        if case["precond"] == "two_level":
            opts.update(precond=claire.PRECOND_TWO_LEVEL, pc_tol=0.0, pc_maxit=4)
    if k == "precond":
        opts.update(precond=claire.PRECOND_TWO_LEVEL)
    ctx = s["ctx"] = claire.Context(n, BETA_V, case["nt"], stream=stream, **opts)
    if k not in ("transport", "vjp"):
        ctx.set_images(i["m0"], i["m1"])
    if k == "register":
        s["v"] = torch.zeros((3,) + n, device="cuda")
    if k in ("newton", "precond"):
        s["g"], s["z"], s["hv"] = (torch.empty((3,) + n, device="cuda") for _ in range(3))
    if k == "precond":
        ctx.gradient(i["v"], s["g"])
    if k in ("transport", "evaluate"):
        s["out"] = torch.empty(n, device="cuda")
    if k == "vjp":
        i["v"].requires_grad_(True)
        i["m0"].requires_grad_(True)
    return s


def run(state):
    case, i = state["case"], state["in"]
    k = case["kind"]
    if k == "conv":
        st = state["stream"]
        x, dy, y, dp, dx = (net.Act(t, 0, t.shape[-1]) for t in (i["x"], i["dy"], state["y"], state["dp"], state["dx"]))
        net.conv3d(x, i["w"], i["b"], y, SLOPE, 1, st)
        net.leaky_bwd(dy, y, SLOPE, dp, st)
        net.conv3d_wgrad(x, dp, state["chunks"], state["part"], state["partb"], state["dw"], state["db"], st)
        net.conv3d(dp, state["wf"], None, dx, 0.0, 0, st)
        return {"y": state["y"], "dw": state["dw"], "db": state["db"], "dx": state["dx"]}
    ctx = state["ctx"]
    if k == "kernels":
        ctx.backtrace(i["v"], state["d"])
        if case["fields"] == 1:
            ctx.interp(i["f"], state["d"], state["out"], ORDER[case["interp"]])
        else:
            ctx.interp_fields(i["f"], case["fields"], state["d"], state["out"], ORDER[case["interp"]])
        ctx.fd8_grad(i["f"][0], state["grad"])
        return {"d": state["d"], "out": state["out"], "grad": state["grad"]}
    if k == "newton":
        J = ctx.gradient(i["v"], state["g"])
        ctx.hessian_matvec(i["vt"], state["hv"])
        ctx.precond(i["r"], state["z"])
        return {"J": J, "g": state["g"], "hv": state["hv"], "z": state["z"]}
    if k == "precond":
        ctx.precond(i["r"], state["z"])
        return {"z": state["z"]}
    if k == "register":
        state["v"].zero_()
        _, rep = ctx.register(state["v"])
        return {"v": state["v"], "J": rep["J"], "mismatch": rep["mismatch"], "detj": [rep["detj_min"], rep["detj_max"]]}
    if k == "evaluate":
        J, mis = ctx.objective(i["v"])
        lo, hi = ctx.detj(i["v"])
        ctx.transport(i["v"], i["m0"], state["out"])
        return {"J": J, "mismatch": mis, "detj": [lo, hi], "m1": state["out"]}
    if k == "transport":
        ctx.transport(i["v"], i["m0"], state["out"], claire.TRANSPORT_ADJ if case["adjoint"] else claire.TRANSPORT_FWD)
        return {"out": state["out"]}
    out = claire.sl_transport(ctx, i["m0"], i["v"], bool(case["recompute"]))
    gm0, gv = torch.autograd.grad(out, (i["m0"], i["v"]), i["gbar"])
    return {"out": out.detach(), "gm0": gm0, "gv": gv}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Inputs and outputs once; multiplications and additions of the stencils,
    the transforms and the pointwise work."""
    n = (case["n1"], case["n2"], case["n3"])
    N = float(n[0]) * n[1] * n[2]
    k = case["kind"]
    if k == "conv":
        P, ci, co = N * case["batch"], case["cin"], case["cout"]
        return {"bytes": 2.0 * P * (2 * ci + 2 * co) + 6.0 * 27 * ci * co, "flops": 3 * 2.0 * 27 * P * ci * co}
    tap = 150.0 if case["interp"] != "linear" else 25.0   # one interpolated value
    fd, fft = 16.0, 2.5 * 3 * math.log2(N)                # one FD8 derivative; a 3-component real transform
    nt = case["nt"]
    back = 3 * tap + 12
    grad = 2 * back + (2 * nt + 1) * tap + 3 * fd * (nt + 2) + 6 * (nt + 1) + 2 * fft
    mat = 2 * nt * tap + 12 * (nt + 1) + 2 * fft
    if k == "kernels":
        return {"bytes": 4.0 * N * (3 + case["fields"] + 3 + case["fields"] + 3),
                "flops": N * (back + case["fields"] * tap + 3 * fd)}
    if k == "newton":
        return {"bytes": 4.0 * N * (2 + 3 * 3 + 3 * 3), "flops": N * (grad + mat + 2 * fft)}
    if k == "precond":
        return {"bytes": 4.0 * N * (nt + 1 + 3 + 3), "flops": N * (3 * fd + 2 * fft + 10 * fft / 4)}
    if k == "register":
        steps = case["gn"]
        return {"bytes": 4.0 * N * (2 + 3 + 3),
                "flops": N * ((steps + 1) * grad + steps * (case["pcg"] * mat + back + nt * tap) + nt * 3 * tap + 9 * fd)}
    if k == "evaluate":
        return {"bytes": 4.0 * N * (2 + 3 + 1), "flops": N * (3 * back + 5 * nt * tap + 2 * fft + 9 * fd)}
    if k == "transport":
        return {"bytes": 4.0 * N * (1 + 3 + 1), "flops": N * (back + nt * tap + (tap + 3 * fd if case["adjoint"] else 0))}
    return {"bytes": 4.0 * N * (1 + 3 + 1 + 1 + 1 + 3), "flops": N * (2 * back + 3 * nt * tap + 3 * tap + 4 * 3 * tap)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, plain torch
# ---------------------------------------------------------------------------

def _weights(t, order, deriv=False):
    if order == "linear":
        return [torch.full_like(t, -1.0), torch.ones_like(t)] if deriv else [1.0 - t, t]
    if order == "cubic":
        if deriv:
            return [-(3 * t * t - 6 * t + 2) / 6, (3 * t * t - 4 * t - 1) / 2, -(3 * t * t - 2 * t - 2) / 2,
                    (3 * t * t - 1) / 6]
        return [-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2, -(t + 1) * t * (t - 2) / 2,
                (t + 1) * t * (t - 1) / 6]
    if deriv:
        return [-0.5 * (1 - t) ** 2, 1.5 * t * t - 2 * t, -1.5 * t * t + t + 0.5, 0.5 * t * t]
    return [(1 - t) ** 3 / 6, (3 * t ** 3 - 6 * t * t + 4) / 6, (-3 * t ** 3 + 3 * t * t + 3 * t + 1) / 6, t ** 3 / 6]


class _Stencil:
    """Interpolation at x + d (grid units), its transpose and its gradient."""

    def __init__(self, d, order):
        self.n, self.order = tuple(d.shape[1:]), order
        off, m = (0, 2) if order == "linear" else (1, 4)
        self.idx, self.w, self.t = [], [], []
        for c in range(3):
            shape = [1, 1, 1]
            shape[c] = self.n[c]
            node = torch.arange(self.n[c], device="cuda").reshape(shape)
            fl = torch.floor(d[c])
            base = node + fl.to(torch.int64) - off
            stride = (self.n[1] * self.n[2], self.n[2], 1)[c]
            self.idx.append([(base + a) % self.n[c] * stride for a in range(m)])
            self.t.append(d[c] - fl)
            self.w.append(_weights(self.t[c], order))

    def _taps(self, w):
        for a, i in enumerate(self.idx[0]):
            for b, j in enumerate(self.idx[1]):
                ij, wab = i + j, w[0][a] * w[1][b]
                for c, k in enumerate(self.idx[2]):
                    yield ij + k, wab * w[2][c]

    def coef(self, f):
        return _prefilter(f) if self.order == "bspline" else f

    def __call__(self, f):
        f, out = self.coef(f), 0.0
        for q, w in self._taps(self.w):
            out = out + w * torch.take(f, q)
        return out

    def transpose(self, y):
        out = torch.zeros(y.numel(), dtype=torch.float64, device="cuda")
        for q, w in self._taps(self.w):
            out.index_add_(0, q.reshape(-1), (w * y).reshape(-1))
        return self.coef(out.reshape(self.n))

    def gradient(self, f):
        f, out = self.coef(f), []
        for c in range(3):
            w = list(self.w)
            w[c] = _weights(self.t[c], self.order, deriv=True)
            g = 0.0
            for q, ww in self._taps(w):
                g = g + ww * torch.take(f, q)
            out.append(g)
        return torch.stack(out)


def _prefilter(f):
    F = torch.fft.rfftn(f)
    for ax, n in enumerate(f.shape):
        k = torch.arange(F.shape[ax], device="cuda", dtype=torch.float64)
        shape = [1, 1, 1]
        shape[ax] = F.shape[ax]
        F = F / ((2.0 + torch.cos(2.0 * math.pi * k / n)) / 3.0).reshape(shape)
    return torch.fft.irfftn(F, s=tuple(f.shape))


class _Solver:
    """The method in 64 bits on one grid."""

    def __init__(self, n, nt, order):
        self.n, self.nt, self.dt, self.order = tuple(n), nt, 1.0 / nt, order
        self.h = [2.0 * math.pi / s for s in n]
        self.vol = self.h[0] * self.h[1] * self.h[2]
        self.wt = [self.dt * (0.5 if j in (0, nt) else 1.0) for j in range(nt + 1)]
        f8 = dict(device="cuda", dtype=torch.float64)
        ks = [torch.fft.fftfreq(n[0], 1.0 / n[0], **f8), torch.fft.fftfreq(n[1], 1.0 / n[1], **f8),
              torch.fft.rfftfreq(n[2], 1.0 / n[2], **f8)]
        shapes = ((-1, 1, 1), (1, -1, 1), (1, 1, -1))
        self.k = [k.reshape(s) for k, s in zip(ks, shapes)]
        self.u = [torch.where(k.abs() == s / 2, torch.zeros_like(k), k) for k, s in zip(self.k, n)]
        kk = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        self.a, self.c = BETA_V * kk, BETA_W * (1.0 + kk)
        self.nz = kk > 0

    def dot(self, x, y):
        return self.vol * float((x * y).sum())

    def disp(self, v, sign):
        u = torch.stack([v[c] / self.h[c] for c in range(3)])
        s = _Stencil(-sign * self.dt * u, self.order)
        return torch.stack([-0.5 * sign * self.dt * (u[c] + s(u[c])) for c in range(3)])

    def d8(self, f, ax):
        out = 0.0
        for s, c in enumerate((4 / 5, -1 / 5, 4 / 105, -1 / 280), 1):
            out = out + c * (torch.roll(f, -s, ax) - torch.roll(f, s, ax))
        return out / self.h[ax]

    def grad(self, f):
        return torch.stack([self.d8(f, c) for c in range(3)])

    def spectral(self, x, inverse=False):
        X = torch.fft.rfftn(x, dim=(1, 2, 3))
        ud = self.u[0] * X[0] + self.u[1] * X[1] + self.u[2] * X[2]
        if inverse:
            uu = self.u[0] ** 2 + self.u[1] ** 2 + self.u[2] ** 2
            f = torch.where(self.nz, self.c / (self.a + self.c * uu).clamp_min(1e-300), torch.zeros_like(self.c))
            ia = torch.where(self.nz, 1.0 / self.a.clamp_min(1e-300), torch.ones_like(self.a))
            Y = torch.stack([ia * (X[c] - f * self.u[c] * ud) for c in range(3)])
        else:
            Y = torch.stack([self.a * X[c] + self.c * self.u[c] * ud for c in range(3)])
        return torch.fft.irfftn(Y, s=self.n, dim=(1, 2, 3))

    def state(self, v, m0):
        s = _Stencil(self.disp(v, 1), self.order)
        ms = [m0]
        for _ in range(self.nt):
            ms.append(s(ms[-1]))
        return s, ms

    def objective(self, v, m0, m1, ms=None):
        ms = ms or self.state(v, m0)[1]
        mis = 0.5 * self.dot(ms[-1] - m1, ms[-1] - m1)
        return mis + 0.5 * self.dot(v, self.spectral(v)), mis

    def characteristic_adjoint(self, v):
        self.sA = _Stencil(self.disp(v, -1), self.order)
        self.div = self.d8(v[0], 0) + self.d8(v[1], 1) + self.d8(v[2], 2)
        self.divX = self.sA(self.div)

    def adjoint_step(self, lam):
        a = self.sA(lam)
        return a + 0.5 * self.dt * (a * self.divX + (a + self.dt * a * self.divX) * self.div)

    def linearise(self, v, m0, m1):
        self.sS, self.ms = self.state(v, m0)
        self.gms = [self.grad(m) for m in self.ms]
        self.characteristic_adjoint(v)

    def body(self, lam):
        out = self.wt[self.nt] * lam * self.gms[self.nt]
        for j in range(self.nt - 1, -1, -1):
            lam = self.adjoint_step(lam)
            out = out + self.wt[j] * lam * self.gms[j]
        return out

    def gradient(self, v, m1):
        return self.spectral(v) + self.body(m1 - self.ms[-1])

    def matvec(self, vt):
        f = [-(vt * g).sum(0) for g in self.gms]
        mt = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        for j in range(self.nt):
            mt = self.sS(mt + 0.5 * self.dt * f[j]) + 0.5 * self.dt * f[j + 1]
        return self.spectral(vt) + self.body(-mt)

    def detj(self, v):
        d = self.disp(v, 1)
        s, u = _Stencil(d, self.order), torch.zeros_like(v)
        for _ in range(self.nt):
            u = torch.stack([s(u[c]) + d[c] * self.h[c] for c in range(3)])
        F = [[self.d8(u[c], e) + (1.0 if c == e else 0.0) for e in range(3)] for c in range(3)]
        det = (F[0][0] * (F[1][1] * F[2][2] - F[1][2] * F[2][1]) - F[0][1] * (F[1][0] * F[2][2] - F[1][2] * F[2][0])
               + F[0][2] * (F[1][0] * F[2][1] - F[1][1] * F[2][0]))
        return [float(det.min()), float(det.max())]

    def vjp(self, m0, v, gbar):
        u = torch.stack([v[c] / self.h[c] for c in range(3)])
        sp = _Stencil(-self.dt * u, self.order)
        d = torch.stack([-0.5 * self.dt * (u[c] + sp(u[c])) for c in range(3)])
        s, ms = _Stencil(d, self.order), [m0]
        for _ in range(self.nt):
            ms.append(s(ms[-1]))
        mb, db = gbar, torch.zeros_like(v)
        for j in range(self.nt - 1, -1, -1):
            db = db + mb * s.gradient(ms[j])
            mb = s.transpose(mb)
        U = -0.5 * self.dt * db
        ub, yb = U.clone(), torch.zeros_like(v)
        for c in range(3):
            ub[c] += sp.transpose(U[c])
            yb += U[c] * sp.gradient(u[c])
        ub = ub - self.dt * yb
        return ms[-1], mb, torch.stack([ub[c] / self.h[c] for c in range(3)])


class _TwoLevel:
    """The two-level zero-velocity preconditioner at a linearised solver."""

    def __init__(self, s, tol, maxit):
        self.s, self.tol, self.maxit = s, tol, maxit
        self.nc = tuple(x // 2 for x in s.n)
        self.c = _Solver(self.nc, s.nt, s.order)
        self.gbar = self.restrict(sum(w * g for w, g in zip(s.wt, s.gms)))

    def move(self, X, nin, nout):
        h = [x // 2 for x in self.nc]
        out = torch.zeros((3, nout[0], nout[1], nout[2] // 2 + 1), dtype=X.dtype, device="cuda")
        for i in (slice(0, h[0]), slice(-h[0] + 1, None)):
            for j in (slice(0, h[1]), slice(-h[1] + 1, None)):
                out[:, i, j, :h[2]] = X[:, i, j, :h[2]]
        return out * (nout[0] * nout[1] * nout[2] / float(nin[0] * nin[1] * nin[2]))

    def restrict(self, f):
        return torch.fft.irfftn(self.move(torch.fft.rfftn(f, dim=(1, 2, 3)), self.s.n, self.nc), s=self.nc, dim=(1, 2, 3))

    def prolong(self, f):
        return torch.fft.irfftn(self.move(torch.fft.rfftn(f, dim=(1, 2, 3)), self.nc, self.s.n), s=self.s.n, dim=(1, 2, 3))

    def kept(self, f):
        f = torch.fft.irfftn(self.move(torch.fft.rfftn(f, dim=(1, 2, 3)), self.nc, self.nc), s=self.nc, dim=(1, 2, 3))
        return f - f.mean((1, 2, 3), keepdim=True)

    def __call__(self, r):
        c, rc = self.c, self.restrict(r)
        x, q = torch.zeros_like(rc), self.kept(rc)
        r0 = math.sqrt(c.dot(q, q))
        z = c.spectral(q, inverse=True)
        p, rz = z.clone(), c.dot(q, z)
        for it in range(1, self.maxit + 1):
            hp = self.kept(c.spectral(p) + self.gbar * (self.gbar * p).sum(0))
            alpha = rz / c.dot(p, hp)
            x, q = x + alpha * p, q - alpha * hp
            if self.tol > 0 and math.sqrt(c.dot(q, q)) <= self.tol * r0:
                break
            z = c.spectral(q, inverse=True)
            new = c.dot(q, z)
            p, rz = z + new / rz * p, new
        mean = r.mean((1, 2, 3), keepdim=True)
        high = r - self.prolong(rc)
        return self.prolong(x) + self.s.spectral(high, inverse=True) + mean


def _register(s, case, m0, m1):
    v = torch.zeros((3,) + s.n, dtype=torch.float64, device="cuda")
    s.linearise(v, m0, m1)
    g, (J, mis) = s.gradient(v, m1), s.objective(v, m0, m1, s.ms)
    for _ in range(case["gn"]):
        two = case["precond"] == "two_level"
        P = _TwoLevel(s, 0.0, 4) if two else (lambda r: s.spectral(r, inverse=True))
        x, r = torch.zeros_like(v), -g
        z = P(r)
        p, rz = z.clone(), s.dot(r, z)
        for it in range(1, case["pcg"] + 1):
            q = s.matvec(p)
            alpha = rz / s.dot(p, q)
            x, r = x + alpha * p, r - alpha * q
            if it == case["pcg"]:
                break
            zn = P(r)
            new = s.dot(r, zn)
            beta = (new - s.dot(r, z)) / rz if two else new / rz
            p, z, rz = zn + beta * p, zn, new
        step, slope = 1.0, s.dot(g, x)
        while s.objective(v + step * x, m0, m1)[0] > J + 1e-4 * step * slope:
            step *= 0.5
        v = v + step * x
        s.linearise(v, m0, m1)
        g, (J, mis) = s.gradient(v, m1), s.objective(v, m0, m1, s.ms)
    return {"v": v, "J": J, "mismatch": mis, "detj": s.detj(v)}


def _conv64(x, w, taps):
    """sum over taps of x shifted, times w[:, tap, :]^T; channels last."""
    out = 0.0
    for t, (a, b, c) in taps:
        out = out + torch.roll(x, (-a, -b, -c), (1, 2, 3)) @ w[:, t, :].T
    return out


def _exact_conv(i):
    x, dy, w, b = (i[k].double() for k in ("x", "dy", "w", "b"))
    taps = [(t, (t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1)) for t in range(27)]
    y = _conv64(x, w, taps) + b
    y = torch.where(y > 0, y, SLOPE * y)
    dp = torch.where(y > 0, dy, SLOPE * dy)
    flat = dp.reshape(-1, dp.shape[-1])
    dw = torch.stack([flat.T @ torch.roll(x, (-a, -b_, -c), (1, 2, 3)).reshape(-1, x.shape[-1])
                      for _, (a, b_, c) in taps], 1)
    wf = w.flip(1).permute(2, 1, 0)
    return {"y": y, "dw": dw, "db": flat.sum(0), "dx": _conv64(dp, wf, taps)}


def exact(case, seed):
    i, k = _inputs(case, seed), case["kind"]
    if k == "conv":
        return _exact_conv(i)
    i = {name: t.double() for name, t in i.items()}
    s = _Solver((case["n1"], case["n2"], case["n3"]), case["nt"], case["interp"])
    if k == "kernels":
        d = s.disp(i["v"], 1)
        st = _Stencil(d, case["interp"])
        return {"d": d, "out": torch.stack([st(f) for f in i["f"]]), "grad": s.grad(i["f"][0])}
    if k == "newton":
        s.linearise(i["v"], i["m0"], i["m1"])
        J = s.objective(i["v"], i["m0"], i["m1"], s.ms)[0]
        return {"J": J, "g": s.gradient(i["v"], i["m1"]), "hv": s.matvec(i["vt"]), "z": s.spectral(i["r"], inverse=True)}
    if k == "precond":
        s.linearise(i["v"], i["m0"], i["m1"])
        return {"z": _TwoLevel(s, 1e-1, 50)(i["r"])}
    if k == "register":
        return _register(s, case, i["m0"], i["m1"])
    if k == "evaluate":
        _, ms = s.state(i["v"], i["m0"])
        J, mis = s.objective(i["v"], i["m0"], i["m1"], ms)
        return {"J": J, "mismatch": mis, "detj": s.detj(i["v"]), "m1": ms[-1]}
    if k == "transport":
        if not case["adjoint"]:
            return {"out": s.state(i["v"], i["m0"])[1][-1]}
        s.characteristic_adjoint(i["v"])
        lam = i["m0"]
        for _ in range(case["nt"]):
            lam = s.adjoint_step(lam)
        return {"out": lam}
    out, gm0, gv = s.vjp(i["m0"], i["v"], i["gbar"])
    return {"out": out, "gm0": gm0, "gv": gv}
