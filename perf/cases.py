"""The calls this framework is measured on: operator products, whole GKB
solves (2D and 3D, FP64 and mixed, single and batched) and the U-Net's
inference and training passes, each through the public binding.

A case is a dict of plain values:

* ``kind`` "apply": one operator product through a handle (``gkb_apply``) or,
  with ``noalloc``, without one (``gkb_apply_noalloc``); ``op`` is W, A, AT or M;
* ``kind`` "solve": ``gkb_solve`` on an enclosed cavity or (``flow``
  "channel") the inflow/outflow channel with plain CG and a seeded guess;
* ``kind`` "batch": ``gkb_solve_batched`` on ``count`` cavities;
* ``kind`` "unet": ``gkb_unet_forward`` or (``train``) ``gkb_unet_loss_grad``.

``exact`` solves the constant-viscosity systems without the framework: the
component Laplacians of the MAC grid are diagonal in sine bases, so W^-1 is a
few dense transforms and the pressure follows from conjugate gradients on the
Schur complement A^T W^-1 A.
"""
import math

import torch

import paper_2001_10424_gb300 as gk

D, NAT = gk.GKB_BC_DIRICHLET, gk.GKB_BC_NATURAL
OPS = {"W": gk.GKB_OP_W, "A": gk.GKB_OP_A, "AT": gk.GKB_OP_AT, "M": gk.GKB_OP_M}


def _solve(n, precision, gamma, **kw):
    c = {"kind": "solve", "nx": n[0], "ny": n[1], "nz": n[2] if len(n) == 3 else 0, "flow": "cavity",
         "precision": precision, "gamma": gamma, "visc": "const", "degree": 2, "coarse": 8, "variant": 0,
         "host": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a product inside somebody else's loop, no handle, no allocation
        {"name": "noalloc_m_64", "kind": "apply", "noalloc": True, "op": "M", "nx": 64, "ny": 64, "nz": 0,
         "gamma": 100.0, "visc": "const"},
        # operator products of a user's own Krylov method or residual check, at odd sizes: 2D and 3D
        {"name": "apply_m_1023x770", "kind": "apply", "noalloc": False, "op": "M", "nx": 1023, "ny": 770, "nz": 0,
         "gamma": 100.0, "visc": "const"},
        {"name": "apply_m_130x95x77", "kind": "apply", "noalloc": False, "op": "M", "nx": 130, "ny": 95, "nz": 77,
         "gamma": 100.0, "visc": "const"},
        # the Poiseuille channel of the benchmark: natural outflow, unpreconditioned CG to 1e-12, seeded guess
        _solve((32, 32), "fp64", 100.0, name="channel_32", flow="channel"),
        # a small cavity from NumPy buffers with the default options, as in the README
        _solve((96, 64), "fp64", 100.0, name="cavity_96x64_host", host=True),
        # the default benchmark: the 1024^2 cavity for gamma 10 and 1000 in one launch, FP64, its tuned options
        {"name": "cavity_1024_pair_fp64", "kind": "batch", "count": 2, "sides": "fixed", "nx": 1024,
         "precision": "fp64", "gamma": 10.0, "gamma2": 1000.0, "degree": 3, "coarse": 32, "variant": 2},
        # the mixed form of one such solve with the default options
        _solve((1024, 1024), "mixed", 1000.0, name="cavity_1024_mixed"),
        # log-normal viscosity (the learned workload's family), mixed
        _solve((1024, 1024), "mixed", 100.0, name="lognormal_1024_mixed", visc="lognormal"),
        # the 3D cavity, mixed
        _solve((160, 160, 160), "mixed", 100.0, name="cavity3d_160_mixed"),
        # many small cavities of different sizes and viscosities in one launch
        {"name": "batch_24_mixed", "kind": "batch", "count": 24, "sides": "mixed", "nx": 512, "precision": "mixed",
         "gamma": 100.0, "gamma2": 100.0, "degree": 2, "coarse": 8, "variant": 0},
        # the network as the learned coarse correction applies it: one image of its level, tensor cores
        {"name": "unet_forward_512_tc", "kind": "unet", "train": False, "n": 1, "h": 512, "w": 512, "tc": True},
        # one training step's loss and gradient at the learned workload's batch
        {"name": "unet_grad_8x512", "kind": "unet", "train": True, "n": 8, "h": 512, "w": 512, "tc": False},
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _mg_sides(rng, dim, most):
    """Sides that multigrid can coarsen, of at most `most` cells: a small grid, odd or even, times a power of two."""
    k = rng.randint(1, int(math.log2(most // 6)))
    top = min(15 if dim == 2 else 10, most >> k)
    return tuple(rng.randint(5, max(6, top)) << k for _ in range(dim))


def draw(rng):
    kind = rng.choice(["apply", "apply", "solve2", "solve2", "solve3", "channel", "batch", "unet", "train"])
    gamma = round(10.0 ** rng.uniform(0.5, 3.0), 2)
    if kind == "apply":
        noalloc = rng.random() < 0.4
        if rng.random() < 0.5:
            n = (_logint(rng, 20, 700 if noalloc else 1500), _logint(rng, 20, 700 if noalloc else 1500), 0)
        else:
            n = tuple(_logint(rng, 10, 60 if noalloc else 140) for _ in range(3))
        return {"kind": "apply", "noalloc": noalloc, "op": rng.choice(["W", "A", "AT", "M", "M"]), "nx": n[0],
                "ny": n[1], "nz": n[2], "gamma": gamma, "visc": "const"}
    tuned = rng.random() < 0.5
    opts = {"degree": rng.choice([2, 3]) if tuned else 2, "coarse": rng.choice([8, 16, 32]) if tuned else 8,
            "variant": rng.choice([0, 2]) if tuned else 0}
    prec = rng.choice(["fp64", "mixed"])
    if kind == "solve2":
        n = _mg_sides(rng, 2, 1024)
        return _solve(n, prec, gamma, visc=rng.choice(["const", "const", "lognormal"]),
                      host=rng.random() < 0.25, **opts)
    if kind == "solve3":
        n = _mg_sides(rng, 3, 112 if prec == "mixed" else 80)
        return _solve(n, prec, gamma, degree=opts["degree"], variant=opts["variant"])
    if kind == "channel":
        return _solve((rng.randint(16, 48), rng.randint(16, 48)), "fp64", gamma, flow="channel")
    if kind == "batch":
        return dict({"kind": "batch", "count": rng.randint(3, 16), "sides": "mixed", "nx": 32 * rng.randint(3, 12),
                     "precision": prec, "gamma": gamma, "gamma2": gamma}, **opts)
    h, w = 4 * _logint(rng, 8, 128), 4 * _logint(rng, 8, 128)
    return {"kind": "unet", "train": kind == "train", "n": rng.randint(1, 8) if kind == "train" else 1, "h": h,
            "w": w, "tc": kind == "unet" and rng.random() < 0.7}


# ---- inputs ----------------------------------------------------------------

class State:
    """What a program keeps between calls: handles, inputs and output buffers."""

    def __init__(self):
        self.handles, self.net = [], None

    def __del__(self):
        for h in self.handles:
            gk.gkb_destroy(h)
        if self.net is not None:
            gk.gkb_unet_destroy(self.net)


def _sides(case):
    return (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] else ())


def _bc(case, dim):
    return (D, NAT, D, D) if case.get("flow") == "channel" else (D,) * (2 * dim)


def _randn(n, seed, k=0):
    return torch.randn(n, dtype=torch.float64, device="cuda",
                       generator=torch.Generator("cuda").manual_seed(1000003 * seed + k))


def _nvel(n, channel=False):
    return sum(math.prod(n) // n[c] * (n[c] - (0 if channel and c == 0 else 1)) for c in range(len(n)))


def _lognormal(nx, ny, seed):
    """exp of a periodic Gaussian field (unit variance, correlation length 0.05), compact cell order."""
    kx = 2 * math.pi * torch.fft.fftfreq(nx, d=1.0 / nx, dtype=torch.float64, device="cuda")
    ky = 2 * math.pi * torch.fft.fftfreq(ny, d=1.0 / ny, dtype=torch.float64, device="cuda")
    amp = torch.exp(-0.25 * 0.05 ** 2 * (ky[:, None] ** 2 + kx[None, :] ** 2))
    f = torch.fft.ifft2(torch.fft.fft2(_randn(nx * ny, seed, 7).view(ny, nx)) * amp).real
    return torch.exp(f / amp.square().mean().sqrt()).reshape(-1).contiguous()


def _handle(case, n, gamma, mu0=1.0, visc=None, bc=None):
    o = gk.gkb_default_options()
    o.stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "apply":
        o.inner, o.use_graph = gk.GKB_INNER_CG, 0
    else:
        o.precision = gk.GKB_PREC_FP64 if case["precision"] == "fp64" else gk.GKB_PREC_MIXED
        o.smoother_degree, o.coarse_max, o.kernel_variant = case["degree"], case["coarse"], case["variant"]
        o.maxit_inner = 5000
        if case.get("flow") == "channel":
            o.inner, o.tol_inner, o.maxit_inner = gk.GKB_INNER_CG, 1e-12, 20000
    h = gk.gkb_create(o)
    try:
        gk.gkb_set_problem(h, gk.make_grid(n, 1.0 / n[0], bc or (D,) * (2 * len(n))), visc, mu0, gamma, 0.0)
    except Exception:
        gk.gkb_destroy(h)
        raise
    return h


def _batch(case, seed):
    """(side, viscosity, gamma) of every problem of a batch."""
    if case["sides"] == "fixed":
        return [(case["nx"], 1.0, case["gamma"]), (case["nx"], 1.0, case["gamma2"])][:case["count"]]
    # the sizes belong to the case, the viscosities to the inputs
    side = torch.randint(2, case["nx"] // 32 + 1, (case["count"],), generator=torch.Generator().manual_seed(case["count"]))
    xi = torch.randn(case["count"], generator=torch.Generator().manual_seed(seed), dtype=torch.float64)
    return [(32 * int(s), math.exp(0.5 * float(x)), case["gamma"]) for s, x in zip(side, xi)]


CONVS = [(3, 16), (16, 16), (16, 32), (32, 32), (32, 32), (32, 32), (64, 32), (48, 16), (16, 2)]


def _params(seed):
    """The network's flat parameters: He-normal weights, small biases."""
    parts = []
    for k, (ci, co) in enumerate(CONVS):
        parts += [_randn(9 * ci * co, seed, 20 + k) * math.sqrt(2.0 / (9 * ci)), 0.1 * _randn(co, seed, 40 + k)]
    return torch.cat(parts).float()


def _images(case, seed):
    """Images like the harvested pairs: residual channels of unit RMS and a smooth log viscosity; targets."""
    n, h, w = case["n"], case["h"], case["w"]
    r = _randn(n * h * w * 2, seed, 1).view(n, h, w, 2)
    c = _randn(n * (h // 4) * (w // 4), seed, 2).view(n, 1, h // 4, w // 4)
    mu = torch.nn.functional.interpolate(c, size=(h, w), mode="bilinear", align_corners=False)
    x = torch.cat([r, mu.permute(0, 2, 3, 1)], dim=3).float().contiguous()
    t = (0.5 * _randn(n * h * w * 2, seed, 3).view(n, h, w, 2)).float().contiguous()
    return x, t


def prepare(case, seed):
    s = State()
    s.case = case
    if case["kind"] == "apply":
        n = _sides(case)
        m, nc = _nvel(n), math.prod(n)
        s.grid = gk.make_grid(n, 1.0 / n[0])
        s.x = _randn(nc if case["op"] == "A" else m, seed)
        s.y = torch.empty(nc if case["op"] == "AT" else m, dtype=torch.float64, device="cuda")
        if not case["noalloc"]:
            s.handles.append(_handle(case, n, case["gamma"]))
    elif case["kind"] == "solve":
        n = _sides(case)
        ch = case["flow"] == "channel"
        m, nc = _nvel(n, ch), math.prod(n)
        visc = _lognormal(n[0], n[1], seed) if case["visc"] == "lognormal" else None
        h = _handle(case, n, case["gamma"], 1.0, visc, _bc(case, len(n)))
        s.handles.append(h)
        s.w0 = s.p0 = None
        if ch:
            s.g, s.r = _channel_rhs(case, h)
            s.w0, s.p0 = _randn(m, seed), _randn(nc, seed, 1)
        else:
            s.g, s.r = _randn(m, seed), torch.zeros(nc, dtype=torch.float64, device="cuda")
        s.w, s.p = torch.empty_like(s.g), torch.empty_like(s.r)
        if case["host"]:
            s.g, s.r, s.w, s.p = (t.cpu().numpy() for t in (s.g, s.r, s.w, s.p))
    elif case["kind"] == "batch":
        s.g, s.r, s.w, s.p = [], [], [], []
        for i, (side, mu, gamma) in enumerate(_batch(case, seed)):
            s.handles.append(_handle(case, (side, side), gamma, mu))
            s.g.append(_randn(_nvel((side, side)), seed, i))
            s.r.append(torch.zeros(side * side, dtype=torch.float64, device="cuda"))
            s.w.append(torch.empty_like(s.g[-1]))
            s.p.append(torch.empty_like(s.r[-1]))
    else:
        s.net = gk.gkb_unet_create(3, 16, 32, 2, seed, torch.cuda.current_stream().cuda_stream)
        gk.gkb_unet_set_params(s.net, _params(seed))
        s.x, s.t = _images(case, seed)
        s.y = torch.empty_like(s.t)
        s.grad = torch.empty(gk.gkb_unet_num_params(s.net), dtype=torch.float32, device="cuda")
    return s


def _channel_rhs(case, h):
    n = _sides(case)
    m, nc = gk.gkb_layout(h)
    y = (torch.arange(n[1], dtype=torch.float64, device="cuda") + 0.5) / n[1]
    g = torch.zeros(m, dtype=torch.float64, device="cuda")
    r = torch.zeros(nc, dtype=torch.float64, device="cuda")
    gk.gkb_boundary_rhs(h, 0, (4.0 * y * (1.0 - y)).contiguous(), g, r)
    return g, r


def run(s):
    c = s.case
    if c["kind"] == "apply":
        if c["noalloc"]:
            gk.gkb_apply_noalloc(s.grid, 1.0, c["gamma"], 0.0, OPS[c["op"]], s.x, s.y,
                                 torch.cuda.current_stream().cuda_stream)
        else:
            gk.gkb_apply(s.handles[0], OPS[c["op"]], s.x, s.y)
        return s.y
    if c["kind"] == "solve":
        gk.gkb_solve(s.handles[0], s.g, s.r, 1e-8, 5, s.w, s.p, s.w0, s.p0)
        return {"w": s.w, "p": s.p}
    if c["kind"] == "batch":
        gk.gkb_solve_batched(s.handles, s.g, s.r, 1e-8, 5, s.w, s.p)
        return {"w": s.w, "p": s.p}
    if c["train"]:
        loss = gk.gkb_unet_loss_grad(s.net, s.x, s.t, c["n"], c["h"], c["w"], s.grad)
        return {"loss": loss, "grad": s.grad}
    gk.gkb_unet_forward(s.net, s.x, c["n"], c["h"], c["w"], s.y, 1 if c["tc"] else 0)
    return s.y


def work(case):
    """Compulsory bytes and flops: the call's inputs and outputs once; for a
    product its stencil, for a solve one product of its operator, for the
    network its convolutions (three times as many with the gradients)."""
    if case["kind"] == "unet":
        px = case["n"] * case["h"] * case["w"]
        per = 2 * 9 * (3 * 16 + 16 * 16 + 48 * 16 + 16 * 2 + (16 * 32 + 32 * 32 + 64 * 32) / 4 + 2 * 32 * 32 / 16)
        return {"bytes": 4 * px * 5, "flops": per * px * (3 if case["train"] else 1)}
    if case["kind"] == "batch":
        ns = [(side, side) for side, _, _ in _batch(case, 0)]
    else:
        ns = [_sides(case)]
    by = fl = 0
    for n in ns:
        m, nc = _nvel(n, case.get("flow") == "channel"), math.prod(n)
        if case["kind"] == "apply":
            by += 8 * ((nc if case["op"] == "A" else m) + (nc if case["op"] == "AT" else m))
        else:
            by += 16 * (m + nc) + (8 * nc if case.get("visc") == "lognormal" else 0)
        fl += (10.5 if len(n) == 2 else 12.7) * m
    return {"bytes": by, "flops": fl}


# ---- the same in 64 bits, without the framework -----------------------------

def _split(x, n, channel=False):
    """Compact velocity -> per component arrays indexed [(z,) y, x]."""
    out, at = [], 0
    for c in range(len(n)):
        shape = [n[a] - (1 if a == c and not (channel and c == 0) else 0) for a in reversed(range(len(n)))]
        out.append(x[at:at + math.prod(shape)].view(shape))
        at += math.prod(shape)
    return out


def _grad(p, n, h):
    d = len(n)
    return [h ** (d - 1) * torch.diff(p, dim=d - 1 - c) for c in range(d)]


def _negdiv(us, n, h):
    d, out = len(n), 0
    for c in range(d):
        dim = d - 1 - c
        z = torch.zeros_like(us[c].narrow(dim, 0, 1))
        out = out - torch.diff(torch.cat([z, us[c], z], dim=dim), dim=dim)
    return h ** (d - 1) * out


def _visc(us, n, h, mu):
    """W of the enclosed grid: zero normal velocity at the walls, mirrored tangential one."""
    d, out = len(n), []
    for c, u in enumerate(us):
        acc = 2 * d * u
        for a in range(d):
            dim = d - 1 - a
            lo, hi = u.narrow(dim, 0, 1), u.narrow(dim, u.shape[dim] - 1, 1)
            g = torch.cat([lo * (0 if a == c else -1), u, hi * (0 if a == c else -1)], dim=dim)
            k = u.shape[dim]
            acc = acc - g.narrow(dim, 0, k) - g.narrow(dim, 2, k)
        out.append(mu * h ** (d - 2) * acc)
    return out


class _Sine:
    """W^-1 of the enclosed constant-viscosity grid by dense sine transforms."""

    def __init__(self, n, h, mu):
        self.n, d = n, len(n)
        self.q, self.lam = [], []
        for a in range(d):
            k = torch.arange(1, n[a] + 1, dtype=torch.float64, device="cuda")
            j = k - 0.5
            ev = 2 - 2 * torch.cos(math.pi * k / n[a])
            face = torch.sin(math.pi * k[:-1, None] * k[None, :-1] / n[a])
            cell = torch.sin(math.pi * j[:, None] * k[None, :] / n[a])
            self.q.append((face / face.norm(dim=0), cell / cell.norm(dim=0)))
            self.lam.append((ev[:-1], ev))
        self.scale = mu * h ** (d - 2)

    def __call__(self, us):
        d, out = len(self.n), []
        for c, u in enumerate(us):
            den = 0
            for a in range(d):
                shape = [1] * d
                shape[d - 1 - a] = -1
                den = den + self.lam[a][0 if a == c else 1].view(shape)
                u = torch.movedim(torch.tensordot(u, self.q[a][0 if a == c else 1], dims=([d - 1 - a], [0])), -1, d - 1 - a)
            u = u / (self.scale * den)
            for a in range(d):
                u = torch.movedim(torch.tensordot(u, self.q[a][0 if a == c else 1], dims=([d - 1 - a], [1])), -1, d - 1 - a)
            out.append(u)
        return out


def _exact_cavity(n, h, mu, g):
    """(w, p) of [W A; A^T 0][w; p] = [g; 0], p of zero mean."""
    winv, gs = _Sine(n, h, mu), _split(g, n)
    schur = lambda q: _negdiv(winv(_grad(q, n, h)), n, h)  # noqa: E731
    b = _negdiv(winv(gs), n, h)
    p, res = torch.zeros_like(b), b - b.mean()
    dirn, rr, r0 = res.clone(), float(res.square().sum()), float(res.square().sum())
    for _ in range(400):
        if rr <= 1e-28 * r0:
            break
        sd = schur(dirn)
        alpha = rr / float((dirn * sd).sum())
        p, res = p + alpha * dirn, res - alpha * sd
        res = res - res.mean()
        new = float(res.square().sum())
        dirn, rr = res + (new / rr) * dirn, new
    p = p - p.mean()
    w = winv([a - b_ for a, b_ in zip(gs, _grad(p, n, h))])
    return torch.cat([a.reshape(-1) for a in w]), p.reshape(-1)


def _exact_channel(case):
    """The channel's saddle system assembled densely: u faces 1..nx (natural outflow on x = 1), v faces 1..ny-1."""
    nx, ny = case["nx"], case["ny"]
    h = 1.0 / nx
    eye = lambda k: torch.eye(k, dtype=torch.float64, device="cuda")  # noqa: E731

    def chain(k, lo, hi):  # links between neighbours; `lo`, `hi`: conductance of the link to the wall
        t = 2 * eye(k) - torch.diag(torch.ones(k - 1, dtype=torch.float64, device="cuda"), 1)
        t -= torch.diag(torch.ones(k - 1, dtype=torch.float64, device="cuda"), -1)
        t[0, 0] += lo - 1
        t[-1, -1] += hi - 1
        return t

    half = eye(nx)
    half[-1, -1] = 0.5  # the outflow faces' control volumes are halves
    wu = torch.kron(eye(ny), chain(nx, 1, 0)) + torch.kron(chain(ny, 2, 2), half)
    wv = torch.kron(eye(ny - 1), chain(nx, 2, 0)) + torch.kron(chain(ny - 1, 1, 1), eye(nx))
    gu = torch.zeros(nx, nx, dtype=torch.float64, device="cuda")  # u face i+1 between cells i and i+1
    for i in range(nx):
        gu[i, i] = -1
        if i + 1 < nx:
            gu[i, i + 1] = 1
    gv = torch.zeros(ny - 1, ny, dtype=torch.float64, device="cuda")
    for j in range(ny - 1):
        gv[j, j], gv[j, j + 1] = -1, 1
    a = h * torch.cat([torch.kron(eye(ny), gu), torch.kron(gv, eye(nx))])
    m, k = nx * ny + nx * (ny - 1), nx * ny
    big = torch.zeros(m + k, m + k, dtype=torch.float64, device="cuda")
    big[:m, :m] = torch.block_diag(wu, wv)
    big[:m, m:], big[m:, :m] = a, a.T
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny
    inflow = 4 * y * (1 - y)
    rhs = torch.zeros(m + k, dtype=torch.float64, device="cuda")
    rhs[:nx * ny].view(ny, nx)[:, 0] = inflow
    rhs[m:].view(ny, nx)[:, 0] = -h * inflow
    z = torch.linalg.solve(big, rhs)
    z = z + torch.linalg.solve(big, rhs - big @ z)
    return z[:m], z[m:]


def _exact_net(case, seed):
    f = torch.nn.functional

    def forward(par, x):
        at, layers = 0, []
        for ci, co in CONVS:
            w = par[at:at + 9 * ci * co].view(3, 3, ci, co).permute(3, 2, 0, 1)
            layers.append((w, par[at + 9 * ci * co:at + 9 * ci * co + co]))
            at += 9 * ci * co + co
        conv = lambda k, v: f.conv2d(v, layers[k][0], layers[k][1], padding=1)  # noqa: E731
        up = lambda v: f.interpolate(v, scale_factor=2, mode="bilinear", align_corners=False)  # noqa: E731
        v = x.permute(0, 3, 1, 2)
        s1 = conv(1, conv(0, v).relu()).relu()
        s2 = conv(3, conv(2, f.avg_pool2d(s1, 2)).relu()).relu()
        c2 = conv(5, conv(4, f.avg_pool2d(s2, 2)).relu()).relu()
        d1 = conv(6, torch.cat([up(c2), s2], 1)).relu()
        e1 = conv(7, torch.cat([up(d1), s1], 1)).relu()
        return conv(8, e1).permute(0, 2, 3, 1)

    x, t = _images(case, seed)
    par = _params(seed).double()
    if not case["train"]:
        return torch.cat([forward(par, x[i:i + 1].double()) for i in range(case["n"])])
    par.requires_grad_(True)
    total = 0.0
    for i in range(case["n"]):  # one sample at a time: the graph of a sample is freed before the next
        loss = (forward(par, x[i:i + 1].double()) - t[i:i + 1].double()).square().sum() / case["n"]
        loss.backward()
        total += float(loss.detach())
    return {"loss": total, "grad": par.grad}


def exact(case, seed):
    torch.backends.cuda.matmul.allow_tf32 = False
    if case["kind"] == "unet":
        return _exact_net(case, seed)
    if case["kind"] == "batch":
        w, p = [], []
        for i, (side, mu, _) in enumerate(_batch(case, seed)):
            n = (side, side)
            a, b = _exact_cavity(n, 1.0 / side, mu, _randn(_nvel(n), seed, i))
            w.append(a)
            p.append(b)
        return {"w": w, "p": p}
    n = _sides(case)
    h, nc = 1.0 / n[0], math.prod(n)
    if case["kind"] == "apply":
        x = _randn(nc if case["op"] == "A" else _nvel(n), seed)
        if case["op"] == "A":
            y = _grad(x.view(tuple(reversed(n))), n, h)
        else:
            us = _split(x, n)
            if case["op"] == "AT":
                return _negdiv(us, n, h).reshape(-1)
            y = _visc(us, n, h, 1.0)
            if case["op"] == "M":
                extra = _grad(_negdiv(us, n, h) * (case["gamma"] / h ** len(n)), n, h)
                y = [a + b for a, b in zip(y, extra)]
        return torch.cat([a.reshape(-1) for a in y])
    if case["visc"] == "lognormal":
        return None  # no fast solver for a variable coefficient
    if case["flow"] == "channel":
        w, p = _exact_channel(case)
    else:
        w, p = _exact_cavity(n, h, 1.0, _randn(_nvel(n), seed))
    return {"w": w, "p": p}
