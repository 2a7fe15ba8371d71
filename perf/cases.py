"""The work a user of this library has it do, as measurable cases.

Every case goes through the public binding (paper_2501_13046_gb300.mg, .unet): constraint
evaluations of a given state, constraint solves (periodic and Robin boxes, mixed and FP64, single
and batched), and the forward and backward pass of one convolution layer of the learned warm
start.  Sizes and inputs follow the library's own workloads (paper_2501_13046_gb300/fields.py,
tests/, bench.py).

  listed()            the cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs on the GPU and the context a program keeps
  run(state)          one pass; returns its outputs
  work(case)          bytes and operations one pass cannot do without
  exact(case, seed)   the outputs in 64 bits by plain torch (None where there is no such value)
"""
import math

import torch

from paper_2501_13046_gb300 import fields, mg, unet

DEV = "cuda"
F64 = torch.float64
PI = math.pi

# the setting mg_autotune picks for the library's periodic and Robin workloads (V(1,1), omega 1.3)
TUNED = dict(inner_cycles=2, nu_pre=1, nu_post=1, omega=1.3)

# channel pairs (cin, cout) of the network's convolutions
CONV_PAIRS = ((16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (128, 64), (96, 32), (48, 16))


def listed():
    return [
        # constraint norms of a caller's state, no context: the check an evolution code makes every step
        dict(name="norms_32", kind="norms", nx=32, ny=32, nz=32, order=4, bc="periodic"),
        # H and M of a given state on a ragged box with unequal spacings (diagnostics)
        dict(name="fields_ragged", kind="fields", nx=97, ny=80, nz=63, order=4, bc="periodic"),
        # the same for two boosted, spinning punctures in a Robin box (black-hole data diagnostics)
        dict(name="fields_binary_128", kind="fields", nx=128, ny=128, nz=128, order=4, bc="binary"),
        # the smallest complete solve, 2nd order: latency and launches
        dict(name="solve_sine_32", kind="solve", data="sine", nx=32, ny=32, nz=32, order=2, precision="mixed",
             tuned=False, nested=False, accurate=False),
        # a small cosmological solve with the default settings
        dict(name="solve_modes_64", kind="solve", data="modes", nx=64, ny=64, nz=64, order=4, precision="mixed",
             tuned=False, nested=False, accurate=False),
        # the benchmarked solve: 128^3, tuned setting, nested start
        dict(name="solve_modes_128", kind="solve", data="modes", nx=128, ny=128, nz=128, order=4, precision="mixed",
             tuned=True, nested=True, accurate=False),
        # a non-cubic box solved until every field has settled (field_tol with its estimate)
        dict(name="solve_accurate_ragged", kind="solve", data="modes", nx=80, ny=64, nz=48, order=4,
             precision="mixed", tuned=False, nested=False, accurate=True),
        # plain FP64 multigrid, the option without any FP32
        dict(name="solve_fp64_64", kind="solve", data="modes", nx=64, ny=64, nz=64, order=4, precision="fp64",
             tuned=True, nested=False, accurate=False),
        # the largest solve: a puncture in a scalar shell, Robin boundaries
        dict(name="solve_shell_256", kind="solve", data="shell", nx=256, ny=256, nz=256, order=4, precision="mixed",
             tuned=True, nested=True, accurate=False),
        # an ensemble of uneven problems in one call
        dict(name="batch_10", kind="batch", count=10, sizes="48,64,96,128", order=4),
        # the network's widest full-resolution layer at its training size, forward (inference)
        dict(name="conv_fwd_64", kind="conv_fwd", nx=64, ny=64, nz=64, cin=48, cout=16),
        # a middle layer's backward pass (training): ReLU adjoint, bias, weight and input gradients
        dict(name="conv_bwd_32", kind="conv_bwd", nx=32, ny=32, nz=32, cin=96, cout=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _coarsening(rng, lo, hi):
    """Three sizes m_a 2^k with m_a in {3, 4, 5} and one k: every level above the coarsest is even."""
    while True:
        k = rng.randint(2, 6)
        n = [m << k for m in (rng.choice((3, 4, 5)),) * 3]
        if rng.random() < 0.4:
            n = [rng.choice((3, 4, 5)) << k for _ in range(3)]
        if all(lo <= m <= hi for m in n):
            return n


def draw(rng):
    kind = rng.choice(("norms", "fields", "fields", "solve", "solve", "solve", "robin", "batch", "conv_fwd", "conv_bwd"))
    if kind == "norms":
        n = [_log_int(rng, 10, 64) for _ in range(3)]
        return dict(kind="norms", nx=n[0], ny=n[1], nz=n[2], order=rng.choice((2, 4)), bc="periodic")
    if kind == "fields":
        n = [_log_int(rng, 16, 180) for _ in range(3)]
        bc = rng.choice(("periodic", "binary"))
        if bc == "binary":   # even: no cell centre on the axis of the punctures
            n = [n[0], n[1] + n[1] % 2, n[2] + n[2] % 2]
        return dict(kind="fields", nx=n[0], ny=n[1], nz=n[2], order=rng.choice((2, 4, 4)), bc=bc)
    if kind == "solve":
        n = _coarsening(rng, 24, 160)
        small = n[0] * n[1] * n[2] <= 80 ** 3
        return dict(kind="solve", data="modes", nx=n[0], ny=n[1], nz=n[2], order=rng.choice((2, 4, 4)),
                    precision=rng.choice(("mixed", "mixed", "fp64")) if small else "mixed",
                    tuned=rng.random() < 0.6, nested=rng.random() < 0.5, accurate=rng.random() < 0.3)
    if kind == "robin":
        n = rng.choice((3, 4, 5)) << rng.randint(4, 5)
        return dict(kind="solve", data=rng.choice(("shell", "octant", "binary")), nx=n, ny=n, nz=n, order=4,
                    precision="mixed", tuned=True, nested=rng.random() < 0.5, accurate=False)
    if kind == "batch":
        sizes = rng.sample(("32", "48", "64", "80", "96"), 3)
        return dict(kind="batch", count=rng.randint(3, 9), sizes=",".join(sizes), order=4)
    ci, co = rng.choice(CONV_PAIRS)
    n = [8 * rng.randint(1, 10), 8 * rng.randint(1, 10), 2 * rng.randint(1, 32)]   # nx ny nz % 128 == 0
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], cin=ci, cout=co)


# ------------------------------------------------------------------------------------- inputs

class _Context:
    """A library context and the buffers a program keeps with it."""

    def __init__(self, ctx, destroy):
        self.ctx, self._destroy = ctx, destroy

    def __del__(self):
        if self.ctx is not None:
            self._destroy(self.ctx)
            self.ctx = None


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _uniform(seed, count):
    g = torch.Generator()
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return torch.rand(count, generator=g, dtype=F64).tolist()


def _axes(n, lo, hi):
    return [lo[a] + (torch.arange(n[a], dtype=F64, device=DEV) + 0.5) * ((hi[a] - lo[a]) / n[a]) for a in range(3)]


def _mesh(n, lo, hi):
    x, y, z = _axes(n, lo, hi)
    return x[None, None, :], y[None, :, None], z[:, None, None]


def _mode_sum(n, L, modes, offset=0.0):
    """offset + sum A cos(k.x + th) and its gradient; modes: (integer vector, amplitude, phase)."""
    X, Y, Z = _mesh(n, (0.0, 0.0, 0.0), L)
    f = torch.full((n[2], n[1], n[0]), offset, dtype=F64, device=DEV)
    df = [torch.zeros_like(f) for _ in range(3)]
    for nu, A, th in modes:
        kv = [2.0 * PI * nu[a] / L[a] for a in range(3)]
        arg = kv[0] * X + kv[1] * Y + kv[2] * Z + th
        f += A * torch.cos(arg)
        s = torch.sin(arg)
        for a in range(3):
            df[a] -= (A * kv[a]) * s
    return f, df


def _modes(seed, L, a0):
    """The random-mode recipe of the periodic workload: 16 distinct modes, amplitude a0 / |k|."""
    unit = 2.0 * PI   # draw_modes(L = 2 pi) gives the integer vectors
    out = []
    for nu, _, th in fields.draw_modes(seed, unit, 1.0):
        k = math.sqrt(sum((2.0 * PI * nu[a] / L[a]) ** 2 for a in range(3)))
        out.append((nu, a0 / k, th))
    return out


def _scalar_sources(phi, dphi, Pi):
    rho0 = 0.5 * Pi * Pi + 0.5 * phi * phi
    rho2 = 0.5 * (dphi[0] ** 2 + dphi[1] ** 2 + dphi[2] ** 2)
    return rho0.contiguous(), rho2.contiguous(), torch.stack([-Pi * d for d in dphi]).contiguous()


def _problem(n, lo, hi, order, bc, kmode, punctures, src, reflect=0):
    return dict(n=list(n), lo=list(lo), hi=list(hi), order=order, bc=bc, kmode=kmode, K=0.0, punctures=punctures,
                rho0=src[0], rho2=src[1], S=src[2], reflect=reflect)


def _shell_sources(n, lo, hi, A, r0):
    X, Y, Z = _mesh(n, lo, hi)
    r = torch.sqrt(X * X + Y * Y + Z * Z)
    phi = A * torch.exp(-((r - r0) ** 2) / 4.0)
    dr = -phi * (r - r0) / 2.0
    return _scalar_sources(phi, [dr * X / r, dr * Y / r, dr * Z / r], 0.01 * phi)


def _matter(data, n, order, seed):
    """The problem of a workload: 'modes' and 'sine' periodic; 'shell', 'octant', 'binary' Robin."""
    u = _uniform(seed, 4)
    if data == "modes":   # cubic cells, the longest side 32 (the 128^3 workload's box)
        h = 32.0 / max(n)
        L = [h * m for m in n]
        a0 = 3e-5 + 3e-5 * u[0]
        phi, dphi = _mode_sum(n, L, _modes(2 * seed + 1, L, a0), 1.0)
        Pi, _ = _mode_sum(n, L, _modes(2 * seed + 2, L, a0))
        return _problem(n, (0.0,) * 3, L, order, fields.PERIODIC, fields.K_INTEGRABILITY, [],
                        _scalar_sources(phi, dphi, Pi))
    if data == "sine":
        L = [16.0] * 3
        phi, dphi = _mode_sum(n, L, [((1, 0, 0), 0.08 + 0.02 * u[0], 2 * PI * u[1])])
        Pi, _ = _mode_sum(n, L, [((0, 1, 0), 0.04 + 0.01 * u[2], 2 * PI * u[3])])
        return _problem(n, (0.0,) * 3, L, order, fields.PERIODIC, fields.K_INTEGRABILITY, [],
                        _scalar_sources(phi, dphi, Pi))
    if data in ("shell", "octant"):
        half = 64.0 * n[0] / 256 * (2 if data == "octant" else 1)
        r0 = min(10.0, 0.6 * half)
        hi = (half,) * 3
        lo = (0.0,) * 3 if data == "octant" else (-half,) * 3
        src = _shell_sources(n, lo, hi, 0.012 + 0.008 * u[0], r0 * (0.95 + 0.05 * u[1]))
        return _problem(n, lo, hi, order, fields.ROBIN, fields.K_FIXED, [(1.0, (0.0, 0.0, 0.0))], src,
                        7 if data == "octant" else 0)
    half = 16.0
    src = _shell_sources(n, (-half,) * 3, (half,) * 3, 0.006 + 0.004 * u[0], 8.0)
    P, S = 0.15 + 0.05 * u[1], 0.05 + 0.05 * u[2]
    punct = [(0.5, (3.0, 0.0, 0.0), (0.0, P, 0.0), (0.0, 0.0, S)), (0.5, (-3.0, 0.0, 0.0), (0.0, -P, 0.0), (0.0, 0.0, S))]
    return _problem(n, (-half,) * 3, (half,) * 3, order, fields.ROBIN, fields.K_FIXED, punct, src)


def _evaluation(case, seed):
    """Problem and state (u, W) of a constraint evaluation: a state on its way to the solution."""
    n = [case["nx"], case["ny"], case["nz"]]
    v = _uniform(seed + 7, 2)
    if case["bc"] == "periodic":
        L = [32.0, 32.0, 32.0] if n[0] != n[1] else [32.0 * m / max(n) for m in n]
        phi, dphi = _mode_sum(n, L, _modes(2 * seed + 1, L, 5e-5), 1.0)
        Pi, _ = _mode_sum(n, L, _modes(2 * seed + 2, L, 5e-5))
        p = _problem(n, (0.0,) * 3, L, case["order"], fields.PERIODIC, fields.K_INTEGRABILITY, [],
                     _scalar_sources(phi, dphi, Pi))
        u = _mode_sum(n, L, _modes(seed + 11, L, 0.01 + 0.01 * v[0]))[0]
        W = torch.stack([_mode_sum(n, L, _modes(seed + 12 + a, L, 1e-3))[0] for a in range(3)]).contiguous()
        return p, u, W
    p = _matter("binary", n, case["order"], seed)
    X, Y, Z = _mesh(n, p["lo"], p["hi"])
    r2 = X * X + Y * Y + Z * Z
    u = (0.05 + 0.05 * v[0]) / torch.sqrt(1.0 + r2 / 25.0)
    W = torch.stack([0.02 * c * torch.ones_like(r2) / (9.0 + r2) * (1.0 + 0.2 * torch.cos(0.3 * X + v[1]) * torch.sin(
        0.25 * Y - 0.2 * Z)) for c in (X, -Y, Z)]).contiguous()
    return p, u.contiguous(), W


def _config(case, p):
    over = dict(tol=1e-10, max_outer=60)
    if case.get("tuned"):
        over.update(TUNED)
    if case.get("nested"):
        over["nested"] = 1
    if case.get("accurate"):
        over.update(field_tol=1e-10, field_est=1)
    return mg.config_for(p, mg.MG_FP64 if case.get("precision") == "fp64" else mg.MG_MIXED, **over)


def _batch_problems(case, seed):
    """Uneven sizes in a fixed rotation (the work is the same for every seed), fields from the seed."""
    sizes = [int(s) for s in case["sizes"].split(",")]
    return [_matter("modes", [sizes[b % len(sizes)]] * 3, case["order"], seed * 64 + b) for b in range(case["count"])]


def _conv_inputs(case, seed):
    g = _gen(seed)
    nx, ny, nz, ci, co = case["nx"], case["ny"], case["nz"], case["cin"], case["cout"]
    rnd = lambda *s: torch.randn(s, generator=g, device=DEV, dtype=torch.float32)
    x = rnd(nz, ny, nx, ci).clamp_min_(0).bfloat16()                       # activations after a ReLU
    w = rnd(27, co, ci) * math.sqrt(2.0 / (27 * ci))                       # He initialisation
    b = 0.05 * rnd(co)
    d = dict(x=x, w=w, b=b, n=(nx, ny, nz))
    if case["kind"] == "conv_bwd":
        d["y"] = rnd(nz, ny, nx, co).clamp_min_(0).bfloat16()
        d["dy"] = (rnd(nz, ny, nx, co) * 1e-3).bfloat16()
    return d


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "norms":
        p, u, W = _evaluation(case, seed)
        st.update(cfg=mg.config_for(p), p=p, u=u, W=W)
    elif kind == "fields":
        p, u, W = _evaluation(case, seed)
        ctx = mg.mg_create(mg.config_for(p))
        st.update(c=_Context(ctx, mg.mg_destroy), p=p, u=u, W=W, H=torch.empty_like(u), M=torch.empty_like(W))
        mg.mg_set_sources(ctx, p["rho0"], p["rho2"], p["S"][0], p["S"][1], p["S"][2])
    elif kind == "solve":
        p = _matter(case["data"], [case["nx"], case["ny"], case["nz"]], case["order"], seed)
        st.update(c=_Context(mg.mg_create(_config(case, p)), mg.mg_destroy), p=p, u=torch.empty_like(p["rho0"]),
                  W=torch.empty_like(p["S"]))
    elif kind == "batch":
        ps = _batch_problems(case, seed)
        st.update(c=_Context(mg.mg_batch_create([_config(dict(tuned=True), p) for p in ps]), mg.mg_batch_destroy),
                  ps=ps, u=[torch.empty_like(p["rho0"]) for p in ps], W=[torch.empty_like(p["S"]) for p in ps])
    else:
        d = _conv_inputs(case, seed)
        n, ci, co = d["n"], case["cin"], case["cout"]
        st.update(d, cin=ci, cout=co, nvox=n[0] * n[1] * n[2], err=torch.zeros(1, dtype=torch.int32, device=DEV))
        fwd = kind == "conv_fwd"
        st["wp"] = torch.empty((27, co, ci) if fwd else (27, ci, co), dtype=torch.bfloat16, device=DEV)
        unet.pack_weights(d["w"], ci, co, 0 if fwd else 1, st["wp"])
        wsb = unet.conv3d_workspace(n, co if fwd else ci)
        st["ws"] = torch.empty(max(wsb // 4, 4), dtype=torch.float32, device=DEV)
        bf = lambda c: torch.empty((n[2], n[1], n[0], c), dtype=torch.bfloat16, device=DEV)
        if fwd:
            st["y"] = bf(co)
        else:
            st.update(dx=bf(ci), dw=torch.empty((27, co, ci), device=DEV), db=torch.empty(co, device=DEV))
    return st


def _solve(ctx, p, u, W):
    mg.mg_set_sources(ctx, p["rho0"], p["rho2"], p["S"][0], p["S"][1], p["S"][2])
    mg.mg_set_initial_guess(ctx, None, None)
    mg.mg_solve(ctx)
    return mg.mg_get_solution(ctx, u, W)


def run(st):
    kind = st["kind"]
    if kind == "norms":
        p = st["p"]
        norms, K2 = mg.mg_residual_norms_noalloc(st["cfg"], st["u"], st["W"], p["rho0"], p["rho2"], p["S"])
        return dict(norms=norms, K2=K2)
    if kind == "fields":
        mg.mg_set_initial_guess(st["c"].ctx, st["u"], st["W"])
        mg.mg_constraint_fields(st["c"].ctx, st["H"], st["M"])
        return dict(H=st["H"], M=st["M"])
    if kind == "solve":
        K = _solve(st["c"].ctx, st["p"], st["u"], st["W"])
        return dict(u=st["u"], W=st["W"], K=K)
    if kind == "batch":
        bt = st["c"].ctx
        for b, p in enumerate(st["ps"]):
            mg.mg_batch_set_sources(bt, b, p["rho0"], p["rho2"], p["S"][0], p["S"][1], p["S"][2])
            mg.mg_batch_set_initial_guess(bt, b, None, None)
        mg.mg_batch_solve(bt, len(st["ps"]))
        K = [mg.mg_batch_get_solution(bt, b, st["u"][b], st["W"][b]) for b in range(len(st["ps"]))]
        return dict(u=st["u"], W=st["W"], K=K)
    n, ci, co = st["n"], st["cin"], st["cout"]
    if kind == "conv_fwd":
        unet.conv3d_fwd(st["x"], st["wp"], st["b"], st["y"], n, ci, co, True, st["err"], ws=st["ws"])
        return dict(y=st["y"])
    st["dw"].zero_()
    st["db"].zero_()
    unet.relu_bwd(st["dy"], st["y"], co, st["nvox"])
    unet.bias_grad(st["dy"], st["db"], co, st["nvox"])
    unet.conv3d_wgrad(st["x"], st["dy"], st["dw"], n, ci, co, st["err"])
    unet.conv3d_fwd(st["dy"], st["wp"], None, st["dx"], n, co, ci, False, st["err"], ws=st["ws"])
    return dict(dx=st["dx"], dw=st["dw"], db=st["db"])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sizes = [int(s) for s in case["sizes"].split(",")]
        cells = sum(sizes[b % len(sizes)] ** 3 for b in range(case["count"]))
        return dict(bytes=72.0 * cells, flops=179.0 * cells)
    N = case["nx"] * case["ny"] * case["nz"]
    if kind == "norms":     # u, W, rho0, rho2, S read
        return dict(bytes=72.0 * N, flops=179.0 * N)
    if kind == "fields":    # u, W, rho0, rho2, S read, H, M written (the sources stay on the GPU)
        return dict(bytes=104.0 * N, flops=179.0 * N)
    if kind == "solve":     # rho0, rho2, S read, u, W written; one residual certifies the result
        return dict(bytes=72.0 * N, flops=179.0 * N)
    ci, co = case["cin"], case["cout"]
    macs = 27.0 * N * ci * co
    if kind == "conv_fwd":
        return dict(bytes=2.0 * N * (ci + co) + 2.0 * 27 * ci * co + 4.0 * co, flops=2.0 * macs)
    # x, y, dy read, masked dy and dx written; weights read, dw and db written
    return dict(bytes=2.0 * N * (2 * ci + 3 * co) + 6.0 * 27 * ci * co + 4.0 * co, flops=4.0 * macs)


# ------------------------------------------------------------------- 64-bit values, plain torch

def _pad(f, p, comp):
    """f with 2 cells per side from the boundary rule; comp: 0 = u, 1..3 = W_x..W_z."""
    n = p["n"]
    idx = [torch.arange(-2, n[a] + 2, device=DEV) for a in range(3)]
    if p["bc"] == fields.PERIODIC:
        b = [idx[a] % n[a] for a in range(3)]
        return f[b[2]][:, b[1]][:, :, b[0]]
    b, x, xb = [], [], []
    for a in range(3):
        h = (p["hi"][a] - p["lo"][a]) / n[a]
        b.append(idx[a].clamp(0, n[a] - 1))
        x.append(p["lo"][a] + (idx[a].to(F64) + 0.5) * h)
        xb.append(p["lo"][a] + (b[a].to(F64) + 0.5) * h)
    r2 = lambda q: q[2][:, None, None] ** 2 + q[1][None, :, None] ** 2 + q[0][None, None, :] ** 2
    return f[b[2]][:, b[1]][:, :, b[0]] * torch.sqrt(r2(xb) / r2(x))


def _shift(g, o):
    """The box shifted by o = (ox, oy, oz) from a padded array."""
    nz, ny, nx = (s - 4 for s in g.shape)
    return g[2 + o[2]:2 + o[2] + nz, 2 + o[1]:2 + o[1] + ny, 2 + o[0]:2 + o[0] + nx]


def _first(order):
    return {1: 0.5, -1: -0.5} if order == 2 else {1: 8 / 12, -1: -8 / 12, 2: -1 / 12, -2: 1 / 12}


def _second(order):
    return {0: -2.0, 1: 1.0, -1: 1.0} if order == 2 else {0: -30 / 12, 1: 16 / 12, -1: 16 / 12, 2: -1 / 12, -2: -1 / 12}


def _along(a, s):
    return tuple(s if c == a else 0 for c in range(3))


def _stencils(p, u, W):
    """Lap u, the momentum operator of W and At_ij (without the punctures' part)."""
    h = [(p["hi"][a] - p["lo"][a]) / p["n"][a] for a in range(3)]
    o = p["order"]
    G = [_pad(W[A], p, 1 + A) for A in range(3)]
    d2 = lambda g, a: sum(w * _shift(g, _along(a, s)) for s, w in _second(o).items()) / h[a] ** 2
    d1 = lambda g, a: sum(w * _shift(g, _along(a, s)) for s, w in _first(o).items()) / h[a]
    lap_u = sum(d2(_pad(u, p, 0), a) for a in range(3))
    mom = []
    for A in range(3):
        m = sum(d2(G[A], a) * (4 / 3 if a == A else 1.0) for a in range(3))
        for B in range(3):
            if B != A:
                mix = 0.0
                for s, ws in _first(o).items():
                    for t, wt in _first(o).items():
                        off = [0, 0, 0]
                        off[A], off[B] = s, t
                        mix = mix + (ws * wt) * _shift(G[B], off)
                m = m + mix / (3.0 * h[A] * h[B])
        mom.append(m)
    D = [[d1(G[B], a) for B in range(3)] for a in range(3)]
    div = D[0][0] + D[1][1] + D[2][2]
    At = [[D[a][b] + D[b][a] - ((2.0 / 3.0) * div if a == b else 0.0) for b in range(3)] for a in range(3)]
    return lap_u, mom, At


def _background(p):
    """psi without u, and the punctures' Bowen-York curvature (3 x 3 or None)."""
    X, Y, Z = _mesh(p["n"], p["lo"], p["hi"])
    psi = torch.ones((p["n"][2], p["n"][1], p["n"][0]), dtype=F64, device=DEV)
    A = None
    for pun in p["punctures"]:
        d = [c - pun[1][a] for a, c in enumerate((X, Y, Z))]
        r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        psi = psi + pun[0] / (2.0 * r)
        if len(pun) > 2:
            P, S = pun[2], pun[3]
            n = [c / r for c in d]
            Pn = P[0] * n[0] + P[1] * n[1] + P[2] * n[2]
            Sn = [S[1] * n[2] - S[2] * n[1], S[2] * n[0] - S[0] * n[2], S[0] * n[1] - S[1] * n[0]]
            A = A or [[0.0] * 3 for _ in range(3)]
            for a in range(3):
                for b in range(3):
                    A[a][b] = A[a][b] + 1.5 / r ** 2 * (P[a] * n[b] + P[b] * n[a] - ((1.0 if a == b else 0.0) - n[a] * n[b]) * Pn) \
                        + 3.0 / r ** 3 * (Sn[a] * n[b] + Sn[b] * n[a])
    return psi, A


def _constraints(p, u, W):
    """(F_psi, F_W, H, M, K^2, psi)."""
    lap_u, mom, At = _stencils(p, u, W)
    bg, by = _background(p)
    psi = bg + u
    if by is not None:
        At = [[At[a][b] + by[a][b] for b in range(3)] for a in range(3)]
    aa = sum(At[a][b] ** 2 for a in range(3) for b in range(3))
    nonlin = 0.125 * psi ** -7 * aa + 2.0 * PI * (p["rho0"] * psi ** 5 + p["rho2"] * psi)
    periodic = p["bc"] == fields.PERIODIC
    K2 = 12.0 * float(nonlin.sum() / (psi ** 5).sum()) if p["kmode"] == fields.K_INTEGRABILITY else p["K"] ** 2
    src = [8.0 * PI * psi ** 6 * p["S"][a] for a in range(3)]
    Fp = lap_u + nonlin - K2 / 12.0 * psi ** 5
    Fw = torch.stack([mom[a] - src[a] + (src[a].mean() if periodic else 0.0) for a in range(3)])
    return Fp, Fw, -8.0 * psi ** -5 * Fp, psi ** -6 * Fw, K2, psi


def _symbols(p):
    """Fourier symbols: first derivatives (times -i), compact second derivatives, per axis."""
    s, lam = [], []
    for a in range(3):
        n, h = p["n"][a], (p["hi"][a] - p["lo"][a]) / p["n"][a]
        th = 2.0 * PI * torch.arange(n, dtype=F64, device=DEV) / n
        if p["order"] == 2:
            sa, la = torch.sin(th) / h, (2.0 * torch.cos(th) - 2.0) / h ** 2
        else:
            sa = (16.0 * torch.sin(th) - 2.0 * torch.sin(2 * th)) / (12.0 * h)
            la = (-30.0 + 32.0 * torch.cos(th) - 2.0 * torch.cos(2 * th)) / (12.0 * h ** 2)
        shape = [1, 1, 1]
        shape[2 - a] = n
        s.append(sa.view(shape))
        lam.append(la.view(shape))
    return s, lam


def _solve_W(rhs, s, lam):
    """W with Lap W_i + (1/3) d_i d_j W_j = rhs_i and zero means (periodic): 3 x 3 systems in Fourier space."""
    R = [torch.fft.fftn(rhs[a]) for a in range(3)]
    tot = lam[0] + lam[1] + lam[2]
    m = [[(tot + lam[a] / 3.0) if a == b else -s[a] * s[b] / 3.0 + 0.0 * tot for b in range(3)] for a in range(3)]
    c00 = m[1][1] * m[2][2] - m[1][2] * m[1][2]
    c01 = m[0][2] * m[1][2] - m[0][1] * m[2][2]
    c02 = m[0][1] * m[1][2] - m[0][2] * m[1][1]
    c11 = m[0][0] * m[2][2] - m[0][2] * m[0][2]
    c12 = m[0][1] * m[0][2] - m[0][0] * m[1][2]
    c22 = m[0][0] * m[1][1] - m[0][1] * m[0][1]
    det = m[0][0] * c00 + m[0][1] * c01 + m[0][2] * c02
    det[0, 0, 0] = 1.0
    C = [[c00, c01, c02], [c01, c11, c12], [c02, c12, c22]]
    out = []
    for a in range(3):
        f = (C[a][0] * R[0] + C[a][1] * R[1] + C[a][2] * R[2]) / det
        f[0, 0, 0] = 0.0
        out.append(torch.fft.ifftn(f).real)
    return torch.stack(out)


def _gmres(op, b, iters, tol):
    """Restart-free GMRES on flattened tensors (the preconditioned operator is close to the identity)."""
    beta = float(b.norm())
    if beta == 0.0:
        return torch.zeros_like(b)
    V, Hm = [b / beta], torch.zeros((iters + 1, iters), dtype=F64)
    for j in range(iters):
        w = op(V[j])
        for _ in range(2):   # twice is enough: orthogonal to rounding
            for i in range(j + 1):
                c = float((w * V[i]).sum())
                Hm[i, j] += c
                w = w - c * V[i]
        Hm[j + 1, j] = float(w.norm())
        e = torch.zeros(j + 2, dtype=F64)
        e[0] = beta
        y = torch.linalg.lstsq(Hm[:j + 2, :j + 1], e[:, None]).solution[:, 0]
        if float((e - Hm[:j + 2, :j + 1] @ y).norm()) <= tol * beta or float(Hm[j + 1, j]) == 0.0 or j + 1 == iters:
            return sum(float(y[i]) * V[i] for i in range(j + 1))
        V.append(w / float(Hm[j + 1, j]))


def _periodic_root(p):
    """The discrete root (u, W, K) of a periodic problem: Newton in u with K^2 eliminated by the
    integrability condition, inner systems by GMRES on the inverse Laplacian, W solved exactly."""
    s, lam = _symbols(p)
    tot = lam[0] + lam[1] + lam[2]
    safe = tot.clone()
    safe[0, 0, 0] = 1.0

    def inv_lap(r):
        f = torch.fft.fftn(r) / safe
        f[0, 0, 0] = 0.0
        return torch.fft.ifftn(f).real

    u = torch.zeros_like(p["rho0"])
    W = torch.zeros_like(p["S"])
    K2, best = 0.0, math.inf
    for _ in range(30):
        Fp, Fw, _, _, K2, psi = _constraints(p, u, W)
        res = max(float(Fp.abs().max()), float(Fw.abs().max()))
        if res >= best / 2 and best < 1e-11:
            break
        best = min(best, res)
        W = W - _solve_W(Fw, s, lam)
        Fp, Fw, _, _, K2, psi = _constraints(p, u, W)
        aa8 = 0.0
        _, _, At = _stencils(p, u, W)
        aa8 = sum(At[a][b] ** 2 for a in range(3) for b in range(3))
        c = -0.875 * psi ** -8 * aa8 + 2.0 * PI * (5.0 * p["rho0"] * psi ** 4 + p["rho2"]) - 5.0 / 12.0 * K2 * psi ** 4
        z = psi ** 5
        proj = lambda r: r - z * (r.mean() / z.mean())
        u = u + _gmres(lambda e: e + inv_lap(proj(c * e)), -inv_lap(proj(Fp)), 40, 1e-9)
        u = u - u.mean()
    return u, W, -math.sqrt(K2)


def _conv_same(x, w, flip):
    """sum over the 27 taps of x shifted (circular) times w[tap] (cout x cin), in 64 bits."""
    out = None
    for tap in range(27):
        d = (tap // 9 - 1, (tap // 3) % 3 - 1, tap % 3 - 1)
        xs = torch.roll(x, tuple((1 if flip else -1) * c for c in d), (0, 1, 2))
        t = xs.reshape(-1, x.shape[-1]) @ (w[tap] if flip else w[tap].T)
        out = t if out is None else out + t
    return out.reshape(*x.shape[:3], -1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("norms", "fields"):
        p, u, W = _evaluation(case, seed)
        _, _, H, M, K2, _ = _constraints(p, u, W)
        if kind == "fields":
            return dict(H=H, M=M)
        return dict(norms=torch.stack([H.abs().max()] + [M[a].abs().max() for a in range(3)]), K2=K2)
    if kind == "solve":
        p = _matter(case["data"], [case["nx"], case["ny"], case["nz"]], case["order"], seed)
        if p["bc"] != fields.PERIODIC:
            return None   # no quick independent solver for Robin boxes
        u, W, K = _periodic_root(p)
        return dict(u=u, W=W, K=K)
    if kind == "batch":
        roots = [_periodic_root(p) for p in _batch_problems(case, seed)]
        return dict(u=[r[0] for r in roots], W=[r[1] for r in roots], K=[r[2] for r in roots])
    d = _conv_inputs(case, seed)
    x, w = d["x"].double(), d["w"].bfloat16().double()
    if kind == "conv_fwd":
        return dict(y=(_conv_same(x, w, False) + d["b"].double()).clamp_min(0))
    dy = d["dy"].double() * (d["y"] > 0)
    dw = torch.stack([dy.reshape(-1, dy.shape[-1]).T @ torch.roll(
        x, tuple(-c for c in (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)), (0, 1, 2)).reshape(-1, x.shape[-1])
        for t in range(27)])
    return dict(dx=_conv_same(dy, w, True), dw=dw, db=dy.sum((0, 1, 2)))
