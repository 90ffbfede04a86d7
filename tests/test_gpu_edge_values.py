"""Values and shapes at the edges of what the kernels accept, against the
oracle: an outflow lattice three cells wide, states and lambda of very
different sizes, non-finite and unphysical cells, very large
relaxation times."""
import math

import numpy as np
import pytest
import torch

import oracle
from tests._helpers import oracle_run, rel_errors, tiny_workload

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
TOL = {"fp64": 1e-10, "fp32": 1e-4}


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("prec,env", [("fp64", {}), ("fp64", {"RLB_F64_ARITH": "df"}), ("fp32", {})]
                         + [("fp32", {"RLB_F32_VARIANT": v}) for v in "012345678"])
@pytest.mark.parametrize("c_l", [1.0, 3.0])
def test_three_cells_between_outflow_ghosts(prec, env, c_l, monkeypatch):
    """nx = 3 with outflow at both ends: x = 1 is copied by both ghosts.  The
    context's buffers hold NaN before the initialisation, so a ghost that a
    step leaves unwritten shows."""
    from paper_0912_2913_gb300 import RLB

    for k, v in env.items():
        monkeypatch.setenv(k, v)
    w = tiny_workload(3, 4, 5, 2, seed=42, c_l=c_l)
    ref, _ = oracle_run(w, 12)
    sim = RLB.from_workload(w, prec, device="cuda:0")
    sim.ws[:2 * sim.state_bytes].fill_(0xFF)
    sim.init_fields(w.n, w.eps, w.beta).step(12)
    n, e, b, ok = sim.macro(where="host")
    sim.close()
    assert ok and max(rel_errors((n, e, b), ref)) <= TOL[prec]


def _adjoint_case(w, prec, state=None, lam=None, noalloc=False):
    """lambda_t, dL/dtau, dL/dbeta_in of one adjoint step and the oracle's; the
    state (oracle cells) and lambda as the GPU stores them."""
    from paper_0912_2913_gb300 import RLB
    from paper_0912_2913_gb300 import _native as N

    p = oracle.Params(**w.params())
    sim = RLB.from_workload(w, prec, device="cuda:0").init_fields(w.n, w.eps, w.beta, w.solid)
    rest = 0.0
    if prec == "fp32":
        rest = np.stack(oracle.equilibrium(sim.params.n_ref, sim.params.eps_ref, np.zeros(3), w.c_l))
    st = sim.cells_to_state(_cuda(state - rest))
    li = sim.cells_to_state(_cuda(lam))
    lo = torch.full_like(li, float("nan"))
    acc = torch.zeros(4, dtype=torch.float64, device="cuda")
    if noalloc:
        N.rlb_adjoint_step_noalloc(sim.ctx, st, li, lo, acc[0:1], acc[1:4])
    else:
        sim.adjoint_step(st, li, lo, acc[0:1], acc[1:4])
    got = sim.state_to_cells(lo).double().cpu().numpy()
    lam = sim.state_to_cells(li).double().cpu().numpy()
    state = sim.state_to_cells(st).double().cpu().numpy() + rest
    acc = acc.cpu().numpy()
    sim.close()
    lam_o, dtau_o, dbin_o = oracle.adjoint_step(p, state, lam, w.solid)
    return (got, acc[0], acc[1:]), (lam_o, dtau_o, dbin_o)


@pytest.mark.parametrize("size", [(3, 4, 5), (3, 41, 43)], ids=["small", "large"])
@pytest.mark.parametrize("prec,c_l,env", [("fp64", 1.0, {}), ("fp64", 3.0, {}), ("fp32", 1.0, {}),
                                          ("fp32", 1.0, {"RLB_ADJ_COOP": "0"}), ("fp32", 1.0, {"RLB_ADJ_PIPE": "0"}),
                                          ("fp32", 1.0, {"RLB_ADJ_PIPE": "1"})])
def test_adjoint_of_three_cells_between_outflow_ghosts(size, prec, c_l, env, monkeypatch):
    """The adjoint of that step: mu of x = 1 takes lambda of both ghosts."""
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    w = tiny_workload(*size, 2, seed=8, c_l=c_l)
    p = oracle.Params(**w.params())
    st = oracle.init(p, w.n, w.eps, w.beta)
    oracle.run(p, st, 2)
    lam = np.random.default_rng(1).normal(size=st.shape)
    got, ref = _adjoint_case(w, prec, st, lam)
    tol = 1e-11 if prec == "fp64" else 1e-4
    big = np.abs(lam).max()
    assert np.max(np.abs(got[0] - ref[0])) <= tol * np.abs(ref[0]).max()
    assert abs(got[1] - ref[1]) <= tol * np.prod(size) * big


@pytest.mark.parametrize("size", [(5, 4, 3), (23, 15, 15)], ids=["eight_lanes", "staged"])
@pytest.mark.parametrize("sscale,lscale", [(1e-40, 1e-270), (1e-60, 1e-250), (1e-80, 1e-230), (1e60, 1e240),
                                           (1e-19, 1e-290), (1e-30, 1e-285), (1e-80, 1e-300), (1.0, 1e-290), (1.0, 1e-307),
                                           (1e-80, 1e-240), (1e-170, 1.0), (1e170, 1e-20)])
def test_fp64_adjoint_of_tiny_states_and_lambda(size, sscale, lscale):
    """States and lambda whose products (the terms of dL/dtau) or squares leave
    the range of binary64, and lambda that loses bits itself.  lambda_t is
    linear in lambda and does not depend on the unit of the state, so the
    reference is the oracle's at order one, scaled.  Bounds: 1e-11 of the
    largest values, as there, and 64 smallest subnormals a cell for what
    underflows (57 products of a cell, to half of one each)."""
    w = tiny_workload(*size, 1, seed=3, bmax=0.5)
    p = oracle.Params(**w.params())
    st = oracle.init(p, w.n, w.eps, w.beta)
    oracle.run(p, st, 2)
    lam = np.random.default_rng(2).normal(size=st.shape)
    lam[:, 0] = 0.0
    ref = oracle.adjoint_step(p, st, lam)
    ref = ref[0] * lscale, ref[1] * lscale * sscale, ref[2] * lscale
    st, lam = st * sscale, lam * lscale
    got = _adjoint_case(w, "fp64", st, lam)[0]
    big, tiny, N = np.abs(lam).max(), 5e-324 * 64, np.prod(size)
    assert np.isfinite(got[1]) and np.isfinite(got[0]).all()
    assert np.max(np.abs(got[0] - ref[0])) <= 1e-11 * np.abs(ref[0]).max() + tiny
    assert abs(got[1] - ref[1]) <= 1e-11 * N * big * np.abs(st).max() + N * tiny
    assert np.max(np.abs(got[2] - ref[2])) <= 1e-11 * N * big + N * tiny


def test_dtau_has_no_common_rounding_error():
    """dL/dtau of one FP64 adjoint step for lambda of zero mean: a rounding
    error common to all cells would grow with their number.  The cells' terms
    are formed in binary64 and summed exactly; their own errors change sign
    with lambda, so they have no mean.  Bound: 4 standard deviations of the
    difference, 40 independent roundings a cell of up to half a unit of
    2^-53 of |mu h| on either side."""
    from paper_0912_2913_gb300 import RLB

    nx, ny, nz = 128, 128, 64
    w = tiny_workload(nx, ny, nz, 0, seed=5, tau=1.0, bmax=0.5)
    st = oracle.init(oracle.Params(**w.params()), w.n, w.eps, w.beta)
    rng = np.random.default_rng(11)
    st *= 1 + 0.01 * rng.uniform(-1, 1, st.shape)
    lam = rng.normal(size=st.shape)
    ev = np.asarray(oracle.lattice()[0], int)
    a = np.empty_like(st)  # the state a step gathers st from
    for i in range(19):
        a[..., i] = np.roll(st[..., i], tuple(-ev[i][c] for c in (2, 1, 0)), axis=(0, 1, 2))
    sim = RLB.from_workload(w, "fp64", device="cuda:0").init_fields(w.n, w.eps, w.beta)
    lo, acc = sim.new_state(), torch.zeros(4, dtype=torch.float64, device="cuda")
    sim.adjoint_step(sim.cells_to_state(_cuda(a)), sim.cells_to_state(_cuda(lam)), lo, acc[0:1], acc[1:4])
    got = float(acc[0])
    sim.close()
    f, g = st[..., 0, :], st[..., 1, :]
    E, S = g.sum(-1), f.sum(-1)
    m = [g @ ev[:, k].astype(float) for k in range(3)]
    s = np.sqrt(4 * E * E - 3 * sum(k * k for k in m))
    eps, b = s - E, [3 * k / (2 * E + s) for k in m]
    b2 = sum(k * k for k in b)
    eg = eps / (1 - b2)
    weight = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    want = 0.0
    for i in range(19):
        q = sum(int(ev[i, k]) * b[k] for k in range(3))
        geq = weight[i] * (eps + eg * (6 * q * q - 2 * b2) + 4 * eg * q) if i else weight[0] * (4 * eg - 3 * eps - 2 * eg * b2)
        t = lam[..., 0, i] * (f[..., i] - weight[i] * S * (1 + 3 * q)) + lam[..., 1, i] * (g[..., i] - geq)
        want = math.fsum([want] + t.ravel().tolist())
    sigma = U * np.sqrt(2 * 40 / 12) * np.sqrt(((lam * st) ** 2).sum())
    assert abs(got - want) <= 4 * sigma, (got - want, sigma)


@pytest.mark.parametrize("prec,lscale", [("fp32", 1e-20), ("fp32", 1e-29), ("fp32", 1e-34), ("fp32", 1e-37), ("fp32", 1e-40),
                                         ("fp64", 1e-279), ("fp64", 1e-290), ("fp64", 1e-305), ("fp64", 1e-312)])
def test_field_adjoints_of_tiny_lambda(prec, lscale):
    """Gradients of the initial fields for lambda far below one, zero in part
    of the lattice, and one cell whose f lambdas alone are tiny; bounds as at
    scale one (64 roundings times gamma^2), and 64 smallest subnormals."""
    from paper_0912_2913_gb300 import RLB

    rng = np.random.default_rng(9)
    shape = (3, 5, 41)
    w = tiny_workload(41, 5, 3, 1, seed=9, bmax=0.5)
    p = oracle.Params(**w.params())
    sim = RLB.from_workload(w, prec, device="cuda:0").init_fields(w.n, w.eps, w.beta)
    l0 = rng.normal(size=shape + (2, 19)) * lscale
    l0[0, 1] = 0.0
    l0[1, 1, 7, 1] = rng.normal(size=19)
    ls = sim.cells_to_state(_cuda(l0))
    l0 = sim.state_to_cells(ls).double().cpu().numpy()
    outs = [torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(2)]
    db, acc = torch.empty((3,) + shape, dtype=torch.float64, device="cuda"), torch.zeros(3, dtype=torch.float64, device="cuda")
    sim.adjoint_fields(_cuda(w.n), _cuda(w.eps), _cuda(w.beta), ls, outs[0], outs[1], db, acc)
    ref = oracle.adjoint_fields(p, w.n, w.eps, w.beta, np.ascontiguousarray(l0))
    sim.close()
    gam2 = 1 / (1 - (w.beta * w.beta).sum(0))
    big, bigf, tiny = np.abs(l0).max((-1, -2)) * gam2, np.abs(l0[..., 0, :]).max(-1) * gam2, 5e-324 * 64
    assert np.all(np.abs(outs[0].cpu().numpy() - ref[0]) <= 64 * U * gam2 * bigf + tiny)
    assert np.all(np.abs(outs[1].cpu().numpy() - ref[1]) <= 64 * U * gam2 * big * 8 + tiny)
    assert np.all(np.abs(db.cpu().numpy() - ref[2]) <= 64 * U * gam2 ** 2 * big * 16 * (w.n + w.eps) + tiny)
    assert np.all(np.abs(acc.cpu().numpy() - ref[3]) <= 64 * U * 41 * 15 * np.abs(l0).max() * 16 * 4 + tiny * 615)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_macro_adjoint_of_cells_without_a_gradient(prec):
    """A cell with zero output gradients: lambda is zero where the fields exist
    and not a number where they do not (a non-finite population, |M| > 2E /
    sqrt 3), as zero times the undefined derivative is."""
    from paper_0912_2913_gb300 import RLB

    w = tiny_workload(9, 4, 3, 0, seed=4)
    sim = RLB.from_workload(w, prec, device="cuda:0").init_fields(w.n, w.eps, w.beta)
    s = sim.state()
    s[19 + 3, 5] = float("nan")
    s[19 + 4, 20] = float("inf")
    s[19 + 1, 33], s[19 + 2, 33] = 40.0, -40.0  # |M| beyond E
    s[2, 50] = float("nan")
    z = torch.zeros((3, 4, 9), dtype=torch.float64, device="cuda")
    zb = torch.zeros((3, 3, 4, 9), dtype=torch.float64, device="cuda")
    lam = sim.new_state()
    sim.adjoint_macro(s, z, z, zb, lam)
    nan = torch.isnan(lam[:, :sim.N]).any(0).cpu().numpy()
    rest = lam[:, :sim.N][:, torch.from_numpy(~nan).cuda()]
    sim.close()
    assert set(np.nonzero(nan)[0]) == {5, 20, 33, 50}
    assert bool((rest == 0).all())


@pytest.mark.parametrize("tau", [900.0, 1e4, 1e6, 1e9])
@pytest.mark.parametrize("split", ["0", "1"])
def test_positivity_count_at_large_tau(tau, split, monkeypatch):
    """The positivity decision in binary32 near its threshold at |q| = 1/3, for
    relaxation times far above the usual ones."""
    from paper_0912_2913_gb300 import RLB

    monkeypatch.setenv("RLB_F64_SPLIT", split)
    shape = (4, 8, 64)
    N = int(np.prod(shape))
    rng = np.random.default_rng(3)
    b = np.zeros((3, N))
    grid = np.linspace(0.31, 0.36, N)
    b[0] = grid
    b[:, ::2] = rng.normal(size=(3, N))[:, ::2]
    b[:, ::2] *= grid[::2] / np.abs(b[:, ::2]).sum(0)
    n, e, b = np.ones(shape), np.ones(shape), b.reshape((3,) + shape)
    p = oracle.Params(nx=64, ny=8, nz=4, tau=tau)
    a = oracle.init(p, n, e, b)
    ev = np.asarray(oracle.lattice()[0], int)
    s = np.empty_like(a)
    for i in range(19):
        s[..., i] = np.roll(a[..., i], tuple(-ev[i][c] for c in (2, 1, 0)), axis=(0, 1, 2))
    stats = oracle.Stats()
    oracle.step(p, s, stats=stats)
    sim = RLB(64, 8, 4, tau, precision="fp64", device="cuda:0")
    sim.load_state(sim.cells_to_state(_cuda(s)))
    sim.step(1)
    got = sim.stats()["n_nonpositive_eq"]
    sim.close()
    assert 0.1 * N < stats.n_nonpositive_eq < 0.9 * N
    assert got == stats.n_nonpositive_eq


def test_a_stale_adjoint_ticket_ends_with_the_next_initialisation():
    """The blocks of an FP64 adjoint step draw a ticket of their own context;
    whatever an interrupted or overlapped launch left in it, rlb_init_fields
    starts it afresh, and another context never sees it."""
    from paper_0912_2913_gb300 import RLB
    from paper_0912_2913_gb300 import _native as N

    w = tiny_workload(23, 15, 15, 1, seed=6)
    sims = [RLB.from_workload(w, "fp64", device="cuda:0").init_fields(w.n, w.eps, w.beta) for _ in range(2)]
    lam = [torch.randn(sims[0].state().shape, dtype=torch.float64, device="cuda") for _ in range(3)]

    def sums(sim, noalloc, k=0):
        acc = torch.zeros(4, dtype=torch.float64, device="cuda")
        f = (lambda *a: N.rlb_adjoint_step_noalloc(sim.ctx, *a)) if noalloc else sim.adjoint_step
        f(sim.state(), lam[k], lam[2], acc[0:1], acc[1:4])
        return acc.cpu()

    want = [sums(sims[0], k) for k in (False, True)]
    assert torch.equal(*want)
    for sim in sims:  # other block sums in the arrays
        assert not torch.equal(sums(sim, False, 1), want[0])
        assert not torch.equal(sums(sim, True, 1), want[0])
    # the ticket is the fourth word behind the 2 x 4096 statistics slots
    at = 2 * ((sims[0].state_bytes + 255) // 256 * 256) + 8 * (2 * 4096 + 3)
    sims[0].ws[at] = 3
    for k in (False, True):
        assert torch.equal(sums(sims[1], k), want[0])
    sims[0].init_fields(w.n, w.eps, w.beta)
    for k in (False, True):
        assert torch.equal(sums(sims[0], k), want[0])
    for s in sims:
        s.close()


def test_macro_of_subnormal_deviations():
    """FP32 states whose deviations are binary32 subnormals beside a tiny
    reference: the fields carry them."""
    from paper_0912_2913_gb300 import RLB

    ref = 1e-30
    sim = RLB(16, 2, 1, 0.8, precision="fp32", n_ref=ref, eps_ref=ref, device="cuda:0")
    rng = np.random.default_rng(0)
    d = (rng.uniform(-1, 1, (1, 2, 16, 2, 19)) * 1e-38).astype(np.float32)
    st = sim.cells_to_state(_cuda(d))
    d = sim.state_to_cells(st).double().cpu().numpy()
    assert np.abs(d).max() > 5e-39
    rest = np.stack(oracle.equilibrium(ref, ref, np.zeros(3), 1.0))
    n, e, b, _ = sim.macro(state=st, where="host")
    want = oracle.macro(oracle.Params(nx=16, ny=2, nz=1, tau=0.8), np.ascontiguousarray(d + rest))
    sim.close()
    # the sums of a cell, 19 terms of 1e-30 in the oracle's binary64
    assert np.all(np.abs(n - want[0]) <= 64 * U * ref)
    assert np.all(np.abs(e - want[1]) <= 64 * U * ref)
    assert np.all(np.abs(b - want[2]) <= 64 * U)


@pytest.mark.parametrize("scale", [2.0 ** -115, 2.0 ** -108, 2.0 ** -95])
def test_fp32_init_of_deviations_near_the_subnormals(scale):
    """Initial deviations rounded once to binary32, also where they end among
    the subnormals (binary64 form restated in numpy, operation by operation)."""
    from paper_0912_2913_gb300 import RLB

    rng = np.random.default_rng(2)
    shape, c = (4, 8, 64), 16.0
    n, e = scale * np.exp(rng.uniform(-0.01, 0.01, (2,) + shape))
    b = rng.uniform(-1e-3, 1e-3, (3,) + shape)
    sim = RLB(64, 8, 4, 0.8, c_l=c, precision="fp32", n_ref=scale, eps_ref=scale, device="cuda:0").init_fields(n, e, b)
    got = sim.state_to_cells(sim.state()).cpu().numpy()
    sim.close()
    bx, by, bz = b
    i1, i2 = 1.0 / c, 1.0 / (c * c)
    b2 = bx * bx + by * by + bz * bz
    gam2 = 1.0 / (1.0 - b2)
    ng, eg = n * np.sqrt(gam2), e * gam2
    want = np.empty(shape + (2, 19), np.float32)
    w0 = 1.0 / 3.0
    want[..., 0, 0] = w0 * ng - w0 * scale
    want[..., 1, 0] = w0 * (4.0 * eg - e * (2.0 * i2 + 1.0) - 2.0 * eg * b2 * i2) - w0 * scale * (3.0 - 2.0 * i2)
    for p, q in enumerate((bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz)):
        w = 1.0 / 18.0 if p < 3 else 1.0 / 36.0
        fa = 3.0 * q * i1
        gs, ga = e * i2 + eg * (6.0 * q * q - 2.0 * b2) * i2, eg * 4.0 * q * i1
        for s, i in ((1, 2 * p + 1), (-1, 2 * p + 2)):
            want[..., 0, i] = w * ng * (1.0 + s * fa) - w * scale
            want[..., 1, i] = w * (gs + s * ga) - w * scale * i2
    assert np.array_equal(got.view(np.int32), want.view(np.int32))


def test_macro_of_a_rest_population_far_above_the_others():
    """Moving populations 2^-1000 times the rest one: beta underflows instead
    of wrapping."""
    from paper_0912_2913_gb300 import RLB

    p = oracle.Params(nx=4, ny=1, nz=1, tau=0.8)
    a = oracle.init(p, np.ones((1, 1, 4)), np.ones((1, 1, 4)), np.full((3, 1, 1, 4), 0.1))
    a[..., 1, 1:] *= 2.0 ** np.array([0, -400, -760, -800])[:, None]
    a[..., 1, 0] *= 2.0 ** np.array([0, 200, 300, 400])
    sim = RLB(4, 1, 1, 0.8, precision="fp64", device="cuda:0")
    n, e, b, _ = sim.macro(state=sim.cells_to_state(_cuda(a)), where="host")
    want = oracle.macro(p, a)
    sim.close()
    assert np.all(np.abs(e - want[1]) <= 64 * U * want[1])
    assert np.all(np.abs(b - want[2]) <= 64 * U * np.abs(want[2]) + 5e-324 * 64)


@pytest.mark.parametrize("size", [(16, 16, 16), (64, 64, 4)], ids=["eight_lanes", "staged"])
def test_lambda_has_no_common_rounding_error(size):
    """lambda_t of one FP64 adjoint step for lambda of one sign that grows along
    x, as next to an outflow plane: rounding ties in v_E + e.v_d one way is an
    error that every step repeats.  The reference is formed in extended
    precision.  A value carries three roundings of up to half a unit of 2^-52 of
    the cell's largest lambda (the sums, the conversion, the relaxation); the
    bound is 4 standard deviations of the mean over the cells, with the values
    of a cell taken as fully correlated."""
    from paper_0912_2913_gb300 import RLB

    nx, ny, nz = size
    N, tau = nx * ny * nz, 0.9
    rng = np.random.default_rng(21)
    ev = np.asarray(oracle.lattice()[0], int)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    p = oracle.Params(nx=nx, ny=ny, nz=nz, tau=tau)
    b = np.zeros((3, nz, ny, nx))
    b[0] = rng.uniform(-0.05, 0.05, b[0].shape)
    h = oracle.init(p, *rng.uniform(0.9, 1.1, (2,) + b[0].shape), b)
    h *= 1 + 1e-3 * rng.uniform(-1, 1, h.shape)
    mu = np.empty_like(h)
    mu[..., 0, :] = rng.uniform(1, 2, h.shape[:3])[..., None]
    mu[..., 1, :] = rng.uniform(30, 60, h.shape[:3])[..., None] * np.array([1.0, 2.06, 0.0])[ev[:, 0]]

    # nu = (1 - 1/tau) mu + (d eq / d h)^T mu / tau, cell by cell
    L = np.longdouble
    hl, ml = h.reshape(N, 2, 19).astype(L), mu.reshape(N, 2, 19).astype(L)
    E, S = hl[:, 1].sum(1), hl[:, 0].sum(1)
    M = [(hl[:, 1] * ev[:, k]).sum(1) for k in range(3)]
    s = np.sqrt(4 * E * E - 3 * sum(m * m for m in M))
    eps, D = s - E, 2 * E + s
    u = [3 * m / D for m in M]
    b2 = sum(v * v for v in u)
    g2 = 1 / (1 - b2)
    eg = eps * g2
    aS, ae, dg2, db2, ab = 0, 0, 0, 0, [0, 0, 0]
    for i in range(19):
        q = sum(int(ev[i, k]) * u[k] for k in range(3))
        mf, mg = ml[:, 0, i] * w[i], ml[:, 1, i] * w[i]
        aS = aS + mf * (1 + 3 * q)
        br = 6 * q * q - 2 * b2 + 4 * q if i else 4 - 2 * b2
        ae = ae + mg * ((1 if i else -3) + g2 * br)
        dg2, db2 = dg2 + mg * eps * br, db2 - 2 * mg * eg
        ab = [ab[k] + int(ev[i, k]) * (3 * S * mf + eg * (12 * q + 4) * mg) for k in range(3)]
    ab = [ab[k] + 2 * (db2 + dg2 * g2 * g2) * u[k] for k in range(3)]
    abD = sum(ab[k] * u[k] for k in range(3)) / D
    dE = 4 * E / s - 1
    vE, vd = ae * dE - abD * (3 + dE), [3 * ab[k] / D + 3 * (abD - ae) / s * M[k] for k in range(3)]
    om = L(1.0 / tau)
    want = (1 - om) * ml[:, 1] + om * np.stack([vE + sum(int(ev[i, k]) * vd[k] for k in range(3)) for i in range(19)], 1)

    a = np.empty_like(h)
    for i in range(19):  # the state a step gathers h from
        a[..., i] = np.roll(h[..., i], tuple(-ev[i][c] for c in (2, 1, 0)), axis=(0, 1, 2))
    sim = RLB(nx, ny, nz, tau, precision="fp64", device="cuda:0")
    lo, acc = sim.new_state(), torch.zeros(4, dtype=torch.float64, device="cuda")
    sim.adjoint_step(sim.cells_to_state(_cuda(a)), sim.cells_to_state(_cuda(mu)), lo, acc[0:1], acc[1:4])
    out = sim.state_to_cells(lo).cpu().numpy()
    sim.close()
    got = np.stack([np.roll(out[..., 1, i], tuple(ev[i][c] for c in (2, 1, 0)), axis=(0, 1, 2)).reshape(N) for i in range(19)], 1)
    err = ((got.astype(L) - want) / np.abs(ml[:, 1]).max(1)[:, None]).astype(np.float64)[:, ev[:, 0] > 0].mean(1)
    sigma = 2 * U * np.sqrt(3 / 12)
    assert np.abs(err).max() <= 16 * U
    assert abs(err.mean()) <= 4 * sigma / np.sqrt(N), (err.mean(), sigma / np.sqrt(N))
