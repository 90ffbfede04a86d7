"""Performance cases of the relativistic lattice Boltzmann library.

Each case is work that a user has the library do, through its public entry
points: a forward run (``RLB.init_fields`` / ``step`` / ``macro``), one adjoint
step (``RLB.adjoint_step``) or a whole gradient (``rlb_run`` and its backward
pass).  Sizes and fields are those of the repository's workloads (the 1D shock
tube, the shock on a sphere, the random periodic box) and ragged sizes in
between.  Inputs are built here with torch on the GPU from the seed alone;
``exact`` computes the same outputs in binary64 with plain torch operations.
"""
import math

import torch
from torch.utils.checkpoint import checkpoint

DEV = "cuda:0"
F64 = torch.float64

# velocity order of a state: rest, +-x, +-y, +-z, then the diagonal pairs
_HALF = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1))
E = ((0, 0, 0),) + tuple(v for e in _HALF for v in (e, tuple(-c for c in e)))
WEIGHT = (1 / 3,) + (1 / 18,) * 6 + (1 / 36,) * 12
OPP = (0,) + tuple(i + 1 if i % 2 else i - 1 for i in range(1, 19))
XBC = {"tube": "outflow_both", "sphere": "inflow_outflow", "box": "periodic"}
TAU = {"tube": 0.9, "sphere": 0.8, "box": 0.7}
GAMMA, MASS = 1.2, 0.3  # the general equation of state's gas
BETA_IN = 0.5


def _case(name, task, flow, size, precision, steps, c_l=1.0, eos="ultra"):
    nx, ny, nz = size
    d = dict(task=task, flow=flow, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps, c_l=c_l, eos=eos)
    return dict(d, name=name) if name else d


def listed():
    return [
        # the 1D Riemann problem, the smallest lattice: launches and latency
        _case("tube_steps_f64", "steps", "tube", (1600, 1, 1), "fp64", 200),
        # the gradient study of the 1D problem: many short launches both ways
        _case("tube_gradient_f64", "gradient", "tube", (1600, 1, 1), "fp64", 150),
        # a reduced, ragged sphere as used for parameter scans: held in L2
        _case("small_sphere_steps_f32", "steps", "sphere", (63, 41, 29), "fp32", 100),
        # the paper's 3D shock on a sphere, single and double precision
        _case("sphere_steps_f32", "steps", "sphere", (200, 100, 100), "fp32", 50),
        _case("sphere_steps_f64", "steps", "sphere", (200, 100, 100), "fp64", 10),
        # the benchmark's periodic box, the largest forward run
        _case("box_steps_f32", "steps", "box", (512, 512, 512), "fp32", 12),
        # the same in double precision at a size that production runs use
        _case("box_steps_f64", "steps", "box", (256, 256, 256), "fp64", 5),
        # numerical tachyons (lattice speed 10) on an odd-sized box
        _case("tachyon_steps_f32", "steps", "box", (193, 127, 161), "fp32", 10, c_l=10.0),
        # an ideal gas with rest mass (general equation of state)
        _case("gamma_law_steps_f64", "steps", "box", (128, 128, 128), "fp64", 5, eos="gamma_law"),
        # one adjoint step: the layer of every gradient
        _case("box_adjoint_f32", "adjoint", "box", (256, 256, 256), "fp32", 1),
        _case("sphere_adjoint_f64", "adjoint", "sphere", (200, 100, 100), "fp64", 1),
        # a whole gradient of the sphere run with its recomputation
        _case("sphere_gradient_f32", "gradient", "sphere", (200, 100, 100), "fp32", 30),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size3(rng, cells, aspect):
    """A ragged lattice of about `cells` cells, nx `aspect` times ny and nz."""
    side = (cells / aspect) ** (1 / 3)
    return tuple(max(20, round(s * rng.uniform(0.85, 1.15))) for s in (aspect * side, side, side))


def draw(rng):
    task = rng.choice(("steps", "steps", "steps", "adjoint", "gradient"))
    flow = rng.choice(("tube", "sphere", "box"))
    precision = rng.choice(("fp64", "fp32"))
    c_l, eos = 1.0, "ultra"
    if task == "steps" and flow != "sphere":
        c_l = rng.choice((1.0, 1.0, 10.0))
        if precision == "fp64" and c_l == 1.0 and rng.random() < 0.35:
            eos = "gamma_law"
    if flow == "tube":
        size = (round(_log(rng, 400, 20000)), 1, 1)
    else:
        size = _size3(rng, _log(rng, 1e4, 3e6 if task == "gradient" else 2e7), 2 if flow == "sphere" else 1)
    cells = size[0] * size[1] * size[2]
    if task == "adjoint":
        steps = 1
    else:
        most = (1e8 if task == "steps" else 4e7) / cells / (2 if precision == "fp64" else 1)
        steps = max(2, min(rng.randint(20, 200), round(most)))
    return _case(None, task, flow, size, precision, steps, c_l, eos)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _noise(shape, gen, sigma=8.0):
    """Gaussian-filtered white noise: spectrum and wave vectors."""
    nz, ny, nx = shape
    kz = 2 * math.pi * torch.fft.fftfreq(nz, device=DEV, dtype=F64)[:, None, None]
    ky = 2 * math.pi * torch.fft.fftfreq(ny, device=DEV, dtype=F64)[None, :, None]
    kx = 2 * math.pi * torch.fft.rfftfreq(nx, device=DEV, dtype=F64)[None, None, :]
    white = torch.randn(shape, generator=gen, device=DEV, dtype=F64)
    return torch.fft.rfftn(white).mul_(torch.exp(-0.5 * sigma * sigma * (kx * kx + ky * ky + kz * kz))), (kx, ky, kz)


def _fields(case, seed):
    """Initial n, eps, beta and solid mask (or None) of a case."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    x = torch.arange(nx, device=DEV)
    solid = None
    if case["flow"] == "box":
        phi = torch.fft.irfftn(_noise(shape, gen)[0], s=shape)
        phi -= phi.mean()
        eps = 1.0 + 0.2 * phi / phi.abs().max()
        n = eps ** 0.75
        a = []
        for _ in range(3):
            spec, (kx, ky, kz) = _noise(shape, gen)
            a.append(spec)
        beta = torch.empty((3,) + shape, device=DEV, dtype=F64)
        for c, (k1, i, k2, j) in enumerate(((ky, 2, kz, 1), (kz, 0, kx, 2), (kx, 1, ky, 0))):
            beta[c] = torch.fft.irfftn(1j * k1 * a[i] - 1j * k2 * a[j], s=shape)
        top = torch.stack([b.abs().max() for b in beta]).max()  # |beta| <= sqrt(3) x this
        beta *= 0.3 / (math.sqrt(3.0) * top)
        return n, eps, beta, solid
    shake = torch.rand(shape, generator=gen, device=DEV, dtype=F64) * 2 - 1
    beta = torch.zeros((3,) + shape, device=DEV, dtype=F64)
    if case["flow"] == "tube":
        left = (x < nx // 2).expand(shape)
        strong = case["eos"] == "ultra"
        eps = torch.where(left, 1.0, 1 / 16 if strong else 0.25).to(F64) * (1 + 0.05 * shake)
        n = torch.where(left, 1.0, 1 / 8 if strong else 0.5).to(F64)
        return n, eps, beta, solid
    eps = 1 + 0.02 * shake
    n = torch.full(shape, 0.3, device=DEV, dtype=F64)
    cx, cy, cz = round(60 * nx / 200), ny // 2, nz // 2
    r = 15.0 * min(nx / 200, ny / 100, nz / 100)
    y, z = torch.arange(ny, device=DEV), torch.arange(nz, device=DEV)
    d2 = (x - cx)[None, None, :] ** 2 + (y - cy)[None, :, None] ** 2 + (z - cz)[:, None, None] ** 2
    return n, eps, beta, (d2 <= r * r).to(torch.uint8)


def _inflow(case):
    on = case["flow"] == "sphere"
    return dict(n_in=1.0, eps_in=1.0, beta_in=(BETA_IN if on else 0.0, 0.0, 0.0))


def _reference(v, extra=()):
    """Uniform reference of the single precision storage, as RLB.reference_value."""
    lo, hi = min([float(v.min()), *extra]), max([float(v.max()), *extra])
    return 2 * lo * hi / (lo + hi)


def _references(case, n, eps, solid):
    if solid is not None:
        n, eps = n[solid == 0], eps[solid == 0]
    extra = (1.0,) if case["flow"] == "sphere" else ()
    return dict(n_ref=_reference(n, extra), eps_ref=_reference(eps, extra))


def _rest(case, ref):
    """The 38 reference populations that single precision states are deviations from."""
    c2 = case["c_l"] ** 2
    f = [w * ref["n_ref"] for w in WEIGHT]
    g = [WEIGHT[0] * ref["eps_ref"] * (3 - 2 / c2)] + [w * ref["eps_ref"] / c2 for w in WEIGHT[1:]]
    return torch.tensor(f + g, device=DEV, dtype=F64)


def _adjoint_inputs(case, seed):
    """Full populations in binary64 and lambda of one adjoint step: a flow's
    equilibrium with a small non-equilibrium part, and a smooth lambda."""
    n, eps, beta, solid = _fields(case, seed)
    ref = _references(case, n, eps, solid)
    if case["flow"] != "box":  # off the initial rest state
        shape = n.shape
        phase = [2 * math.pi * torch.arange(s, device=DEV, dtype=F64) / s for s in shape]
        wave = torch.sin(phase[2])[None, None, :] + torch.cos(phase[1])[None, :, None] * torch.sin(phase[0] + 1)[:, None, None]
        beta = beta + 0.1 * torch.stack([wave, wave.roll(3, 2), wave.roll(5, 2)])
    pops = _equilibrium(case, n, eps, beta)
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 77)
    pops *= 1 + 0.003 * (torch.rand(pops.shape, generator=gen, device=DEV, dtype=F64) * 2 - 1)
    pops = _ghosts(case, pops, pops, torch.tensor(_inflow(case)["beta_in"], device=DEV, dtype=F64))
    lam = torch.randn(pops.shape, generator=gen, device=DEV, dtype=F64)
    lam = (lam + lam.roll(1, -1) + lam.roll(1, 0)) / 3
    if solid is not None:
        lam *= solid == 0
    if case["precision"] == "fp32":
        pops = (pops - _rest(case, ref)[:, None, None, None]).float()
        lam = lam.float()
    return pops, lam, solid, ref


def _marker(state, solid):
    """Solid cells of a state carry a NaN payload in every plane."""
    bits, word = (0x7FF8D0D05011D000, torch.int64) if state.dtype == F64 else (0x7FC5011D, torch.int32)
    state.view(word)[:, solid.reshape(-1).nonzero()[:, 0]] = bits


def prepare(case, seed):
    from paper_0912_2913_gb300 import RLB, RunSpec

    nx, ny, nz, flow = case["nx"], case["ny"], case["nz"], case["flow"]
    if case["task"] == "gradient":
        n, eps, beta, solid = _fields(case, seed)
        ref = _references(case, n, eps, solid)
        inflow = _inflow(case)
        spec = RunSpec(nx, ny, nz, case["steps"], case["c_l"], case["precision"], XBC[flow], inflow["n_in"],
                       inflow["eps_in"], solid, ref["n_ref"], ref["eps_ref"], device=DEV)
        tau = torch.tensor(TAU[flow], device=DEV, dtype=F64, requires_grad=True)
        beta_in = torch.tensor(inflow["beta_in"], device=DEV, dtype=F64, requires_grad=True)
        leaves = [tau, beta_in] + [t.requires_grad_() for t in (n, eps, beta)]
        return dict(case=case, spec=spec, leaves=leaves)
    if case["task"] == "adjoint":
        pops, lam, solid, ref = _adjoint_inputs(case, seed)
    else:
        n, eps, beta, solid = _fields(case, seed)
        ref = _references(case, n, eps, solid)
    sim = RLB(nx, ny, nz, TAU[flow], c_l=case["c_l"], precision=case["precision"], xbc=XBC[flow], eos=case["eos"],
              eos_gamma=GAMMA, eos_mass=MASS, device=DEV, **_inflow(case), **ref)
    if case["task"] == "steps":
        return dict(case=case, sim=sim, fields=(n, eps, beta, solid))
    bufs = []
    for t in (pops, lam):
        buf = sim.new_state()
        buf[:, :sim.N] = t.reshape(38, -1)
        bufs.append(buf)
    if solid is not None:
        _marker(bufs[0], solid)
    return dict(case=case, sim=sim, state=bufs[0], lam=bufs[1], out=sim.new_state())


def _loss(n, eps, beta, solid):
    """A scalar of the final fields: mean pressure squared, density and flux."""
    keep = torch.ones_like(eps, dtype=torch.bool) if solid is None else solid == 0
    zero = torch.zeros((), dtype=F64, device=eps.device)
    pick = lambda t: torch.where(keep, t, zero)  # noqa: E731
    return ((pick(eps) / 3) ** 2).sum() + 0.5 * (pick(n) ** 2).sum() + (pick(beta[0]) * pick(eps)).sum()


def run(state):
    case = state["case"]
    if case["task"] == "steps":
        sim = state["sim"]
        sim.init_fields(*state["fields"]).step(case["steps"])
        n, eps, beta, _ = sim.macro()
        return dict(n=n, eps=eps, beta=beta, state=sim.state()[:, :sim.N])
    if case["task"] == "adjoint":
        sim = state["sim"]
        acc = torch.zeros(4, dtype=F64, device=DEV)
        sim.adjoint_step(state["state"], state["lam"], state["out"], acc[0:1], acc[1:4])
        return dict(lam=state["out"][:, :sim.N], dtau=acc[0:1], dbeta_in=acc[1:4])
    from paper_0912_2913_gb300 import rlb_run

    spec, leaves = state["spec"], state["leaves"]
    n, eps, beta = rlb_run(*leaves, spec)
    grads = torch.autograd.grad(_loss(n, eps, beta, spec.solid), leaves)
    return dict(n=n.detach(), eps=eps.detach(), beta=beta.detach(), dtau=grads[0], dbeta_in=grads[1],
                dn0=grads[2], deps0=grads[3], dbeta0=grads[4])


def work(case):
    """Bytes: the populations read and written once per update (an adjoint step
    reads the state and lambda and writes lambda), fields in and out once.
    Floating-point operations of the update as the equations state them."""
    cells = case["nx"] * case["ny"] * case["nz"]
    state = 38 * (8 if case["precision"] == "fp64" else 4) * cells
    step, adjoint = 250 * cells, 500 * cells
    if case["eos"] != "ultra":
        step *= 2
    if case["task"] == "adjoint":
        return dict(bytes=3 * state, flops=adjoint)
    bytes_, flops = case["steps"] * 2 * state + 2 * (40 * cells + state), case["steps"] * step
    if case["task"] == "gradient":
        bytes_ += case["steps"] * 3 * state + 2 * (40 * cells + state)
        flops += case["steps"] * adjoint
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------------------
# The same outputs in binary64 with plain torch operations
# ---------------------------------------------------------------------------
def _equilibrium(case, n, eps, beta, pressure=None):
    c = case["c_l"]
    p = eps / 3 if pressure is None else pressure
    b2 = (beta * beta).sum(0)
    g2 = 1 / (1 - b2)
    ng, h = n * g2.sqrt(), (eps + p) * g2
    out = []
    for i in range(19):
        q = sum(e * b for e, b in zip(E[i], beta) if e)
        out.append(WEIGHT[i] * ng * (1 + 3 * q / c) if i else WEIGHT[0] * ng)
    for i in range(19):
        q = sum(e * b for e, b in zip(E[i], beta) if e)
        if i:
            out.append(WEIGHT[i] * (3 * p / c ** 2 + h * (3 * q / c + (4.5 * q * q - 1.5 * b2) / c ** 2)))
        else:
            out.append(WEIGHT[0] * (3 * h - 3 * p * (2 + c * c) / c ** 2 - 1.5 * h * b2 / c ** 2))
    return torch.stack([o.expand(n.shape) for o in out])


def _recover(case, pops):
    """(n gamma, n, eps, P, beta) of populations."""
    s, e = pops[:19].sum(0), pops[19:].sum(0)
    m = torch.stack([case["c_l"] * sum(E[i][a] * pops[19 + i] for i in range(1, 19) if E[i][a]) for a in range(3)])
    m2 = (m * m).sum(0)
    if case["eos"] == "ultra":
        eps = (4 * e * e - 3 * m2).sqrt() - e
        beta = 3 * m / (3 * e + eps)
        p = eps / 3
    else:
        p = (GAMMA - 1) * (e - MASS * s)
        for _ in range(60):
            w = e + p
            b2 = m2 / (w * w)
            nn = s * (1 - b2).sqrt()
            r = (GAMMA - 1) * (e - m2 / w - MASS * nn) - p
            p = p - r / ((GAMMA - 1) * (b2 - MASS * nn * b2 / (w * (1 - b2))) - 1)
        beta = m / (e + p)
        eps = e - m2 / (e + p)
    return s, s * (1 - (beta * beta).sum(0)).sqrt(), eps, p, beta


def _ghosts(case, new, old, beta_in):
    """The x boundary planes: held inflow state, outflow copies."""
    if case["flow"] == "box":
        return new
    shape = new.shape[1:3]
    first = new[..., 1:2]
    if case["flow"] == "sphere":
        one = torch.ones(shape + (1,), device=DEV, dtype=F64)
        first = _equilibrium(case, one, one, beta_in[:, None, None, None] * one)
    return torch.cat([first, new[..., 1:-1], new[..., -2:-1]], -1)


def _step(case, pops, tau, beta_in, solid):
    bounce = None if solid is None else solid != 0
    pulled = []
    for q in range(38):
        i = q % 19
        ex, ey, ez = E[i]
        v = pops[q].roll((ez, ey, ex), (0, 1, 2)) if i else pops[q]
        if bounce is not None and i:
            v = torch.where(bounce.roll((ez, ey, ex), (0, 1, 2)), pops[q - i + OPP[i]], v)
        pulled.append(v)
    h = torch.stack(pulled)
    s, n, eps, p, beta = _recover(case, h)
    new = h + (_equilibrium(case, n, eps, beta, p) - h) / tau
    if bounce is not None:
        new = torch.where(bounce, pops, new)
    return _ghosts(case, new, pops, beta_in)


def _filled(fields, solid):
    """Fields with benign values in solid cells (they are masked afterwards)."""
    if solid is None:
        return fields
    m = solid != 0
    return [torch.where(m, torch.full_like(t, v), t) for t, v in zip(fields, (0.3, 1.0, 0.0))]


def _cost(case):
    """Cell updates of exact(), an adjoint counted as four."""
    return case["nx"] * case["ny"] * case["nz"] * case["steps"] * (1 if case["task"] == "steps" else 4)


def exact(case, seed):
    cells = case["nx"] * case["ny"] * case["nz"]
    if cells > 2.5e7 or _cost(case) > 4e8 or (case["flow"] == "tube" and case["steps"] > 400):
        return None
    beta_in = torch.tensor(_inflow(case)["beta_in"], device=DEV, dtype=F64)
    tau = torch.tensor(TAU[case["flow"]], device=DEV, dtype=F64)
    if case["task"] == "adjoint":
        pops, lam, solid, ref = _adjoint_inputs(case, seed)
        if case["precision"] == "fp32":
            pops = pops.double() + _rest(case, ref)[:, None, None, None]
        args = [pops.requires_grad_(), tau.requires_grad_(), beta_in.requires_grad_()]
        new = _step(case, *args, solid)
        # a population that nobody pulls has no adjoint; the solid cells keep theirs
        grads = torch.autograd.grad(new, args, lam.double(), allow_unused=True)
        dbeta = grads[2] if grads[2] is not None else torch.zeros(3, device=DEV, dtype=F64)
        return dict(lam=grads[0].reshape(38, cells), dtau=grads[1].reshape(1), dbeta_in=dbeta)
    n, eps, beta, solid = _fields(case, seed)
    ref = _references(case, n, eps, solid)
    grad = case["task"] == "gradient"
    leaves = [tau, beta_in, n, eps, beta]
    if grad:
        leaves = [t.requires_grad_() for t in leaves]
    with torch.set_grad_enabled(grad):
        f = _filled(leaves[2:], solid)
        p = None if case["eos"] == "ultra" else (GAMMA - 1) * (f[1] - MASS * f[0])
        pops = _equilibrium(case, *f, p)
        if case["flow"] == "sphere":
            pops = torch.cat([_ghosts(case, pops, pops, beta_in)[..., :1], pops[..., 1:]], -1)
        for _ in range(case["steps"]):
            if grad:
                pops = checkpoint(lambda a, t, b: _step(case, a, t, b, solid), pops, tau, beta_in, use_reentrant=False)
            else:
                pops = _step(case, pops, tau, beta_in, solid)
        _, n1, e1, _, b1 = _recover(case, pops)
        grads = None
        if grad:
            grads = torch.autograd.grad(_loss(n1, e1, b1, solid), leaves, allow_unused=True)
            grads = [torch.zeros_like(t) if g is None else g for g, t in zip(grads, leaves)]
    nan = torch.full((), math.nan, device=DEV, dtype=F64)
    hide = (lambda t: t.detach()) if solid is None else (lambda t: torch.where(solid != 0, nan, t.detach()))
    out = dict(n=hide(n1), eps=hide(e1), beta=hide(b1))
    if grad:
        return dict(out, dtau=grads[0], dbeta_in=grads[1], dn0=grads[2], deps0=grads[3], dbeta0=grads[4])
    if case["precision"] == "fp32":
        pops = pops - _rest(case, ref)[:, None, None, None]
    return dict(out, state=hide(pops).reshape(38, cells))
