"""The FP64 step in block fixed point (csrc/rlb_fixed.cuh, 1 <= c_l <= 2) at
the edges of its range, against the oracle: gathered populations far apart in
size, negative and exactly zero ones, |M| up to and beyond E (cells that take
the binary64 path), extreme exponents, lattice speeds on both sides of the
limits; one thread and eight lanes per cell give the same bits."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

EV = np.asarray(oracle.lattice()[0], int)
# Error bound in units of 2^-53 of a cell's largest population: at |beta| =
# 0.985 the oracle's own eps gamma^2 carries 3 roundings of E times gamma^2 =
# 34; 19 sums and the relaxation stay below 32 units.
UNITS = 1024


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


def _gathered(rng, shape, c_l):
    """Populations (cells, 2, 19) as a step gathers them, one kind per cell."""
    N = int(np.prod(shape))
    b = rng.normal(size=(N, 3))
    b *= (rng.choice([0.0, 0.01, 0.4, 0.7, 0.9, 0.985], N) / np.linalg.norm(b, axis=1))[:, None]
    p = oracle.Params(nx=N, ny=1, nz=1, tau=0.8, c_l=c_l)
    h = oracle.init(p, np.exp(rng.uniform(-3, 3, N)), np.exp(rng.uniform(-3, 3, N)), b.T.copy()).reshape(N, 2, 19)
    h *= 1 + 0.02 * rng.uniform(-1, 1, h.shape)
    kind = rng.integers(0, 6, N)
    small = rng.uniform(size=h.shape) < 0.3
    h[(kind == 1)[:, None, None] & small] = 0.0
    h[(kind == 2)[:, None, None] & small] *= 2.0 ** -45
    h[kind == 3] *= (2.0 ** rng.integers(-200, 200, (kind == 3).sum()))[:, None, None]
    h[:, 1, 1][kind == 4] *= 40.0  # |M| near or above E
    h[N // 2, 1] *= -1.0  # E < 0
    return h.reshape(shape + (2, 19))


def _scatter(h):
    """The state a step gathers h from (periodic): A_i(x - e_i) = h_i(x)."""
    a = np.empty_like(h)
    for i in range(19):
        a[..., i] = np.roll(h[..., i], tuple(-EV[i][c] for c in (2, 1, 0)), axis=(0, 1, 2))
    return a


@pytest.mark.parametrize("c_l", [1.0, 1.7, 2.0, 2.0 + 2 ** -30])
@pytest.mark.parametrize("tau", [0.51, 0.8, 1.0, 30.0])
def test_one_step_of_hard_states(c_l, tau, monkeypatch):
    from paper_0912_2913_gb300 import RLB

    nz, ny, nx = shape = (6, 7, 37)
    h = _gathered(np.random.default_rng(int(8 * c_l + 100 * tau)), shape, c_l)
    a = _scatter(h)
    p = oracle.Params(nx=nx, ny=ny, nz=nz, tau=tau, c_l=c_l)
    stats = oracle.Stats()
    ref = oracle.step(p, a, stats=stats)
    outs = []
    for split in ("0", "1"):
        monkeypatch.setenv("RLB_F64_SPLIT", split)
        sim = RLB(nx, ny, nz, tau, c_l=c_l, precision="fp64", device="cuda:0")
        sim.load_state(sim.cells_to_state(torch.from_numpy(a).cuda()))
        sim.step(1)
        outs.append((sim.state()[:, :sim.N].clone(), sim.stats()))
        got = sim.state_to_cells(sim.state()).cpu().numpy()
        sim.close()
    assert torch.equal(outs[0][0].view(torch.int64), outs[1][0].view(torch.int64))
    assert outs[0][1] == outs[1][1]
    s = outs[0][1]
    assert s["n_unphysical"] == stats.n_unphysical > 0 and s["first_bad"] == stats.first_bad
    assert s["n_nonpositive_eq"] == stats.n_nonpositive_eq
    E, M = h[..., 1, :].sum(-1), c_l * (h[..., 1, :] @ EV.astype(float))
    # |beta| < 0.985, the range of the bound (|M|^2 < 0.986 E^2 there)
    physical = (E > 0) & ((M * M).sum(-1) < 0.985 * E * E)
    assert 0.6 < physical.mean() < 1
    # f scales with its own largest population, g with its own
    for s_ in range(2):
        big = np.abs(h[..., s_, :]).max(-1)[physical]
        err = np.abs(got[..., s_, :] - ref[..., s_, :])[physical].max(-1)
        assert np.all(err <= UNITS * 2.0 ** -53 * big), (s_, (err / big).max() * 2.0 ** 53)


@pytest.mark.parametrize("size", [(5, 4, 3), (23, 15, 15)], ids=["eight_lanes", "staged"])
@pytest.mark.parametrize("xbc", [0, 1, 2])
@pytest.mark.parametrize("c_l,lam_scale", [(1.0, 1.0), (2.0, 1e-200), (2.0 + 2 ** -30, 1.0)])
def test_adjoint_step(size, xbc, c_l, lam_scale):
    """One FP64 adjoint step on lattices of either kernel (at most 32 cells per
    SM: eight lanes per cell), solid cells and every boundary, lambda zero in
    part of the lattice: lambda_t, dL/dtau and
    dL/dbeta_in against the oracle's taped adjoint.  Bound: 1e-11 of the
    largest |lambda| (the sums of a cell, 57 terms, and gamma^2 <= 2 stay
    below 10^3 units of 2^-53)."""
    from paper_0912_2913_gb300 import RLB
    from tests._helpers import tiny_workload

    nx, ny, nz = size
    solids = ((2, 1, 1),) if nx < 10 else ((9, 7, 7), (10, 7, 7), (9, 8, 7))
    w = tiny_workload(nx, ny, nz, xbc, seed=3, c_l=c_l, solid_cells=solids, bmax=0.5)
    p = oracle.Params(**w.params())
    st = oracle.init(p, w.n, w.eps, w.beta, w.solid)
    oracle.run(p, st, 2, solid=w.solid)
    rng = np.random.default_rng(nx + xbc)
    lam = rng.normal(size=st.shape) * lam_scale
    lam[: nz // 2, 0] = 0.0
    lam_o, dtau_o, dbin_o = oracle.adjoint_step(p, st, lam, w.solid)
    sim = RLB.from_workload(w, "fp64", device="cuda:0").init_fields(w.n, w.eps, w.beta, w.solid)
    cells = sim.state_to_cells(sim.state()).cpu().numpy()  # its solid markers
    fluid = w.solid == 0
    cells[fluid] = st[fluid]
    lo = sim.new_state()
    acc = torch.zeros(4, dtype=torch.float64, device="cuda")
    sim.adjoint_step(sim.cells_to_state(torch.from_numpy(cells).cuda()), sim.cells_to_state(torch.from_numpy(lam).cuda()), lo,
                     acc[0:1], acc[1:4])
    got = sim.state_to_cells(lo).cpu().numpy()
    acc = acc.cpu().numpy()
    sim.close()
    assert np.max(np.abs(got - lam_o)) <= 1e-11 * np.max(np.abs(lam_o))
    N = nx * ny * nz
    assert abs(acc[0] - dtau_o) <= 1e-11 * N * np.max(np.abs(lam))
    assert np.max(np.abs(acc[1:] - dbin_o)) <= 1e-11 * N * np.max(np.abs(lam))


@pytest.mark.parametrize("gamma,mass", [(4 / 3, 0.0), (1.2, 0.3), (5 / 3, 0.1), (2.0, 0.0), (1.01, 0.5)])
@pytest.mark.parametrize("c_l", [1.0, 2.0, 2.0 + 2 ** -30])
def test_general_eos_one_step(gamma, mass, c_l):
    """One step and the macroscopic output under the general equation of state
    at the edges of the fixed-point form: the hard states above (unphysical
    ones and |M| near E on the binary64 path).  Bound: the oracle stops its
    iteration at |dP| <= 1e-14 (P + E); 2048 units of 2^-53 of a cell's largest
    population cover that, its roundings and gamma^2 <= 34."""
    from paper_0912_2913_gb300 import RLB

    nz, ny, nx = shape = (4, 7, 37)
    h = _gathered(np.random.default_rng(int(8 * c_l + 100 * gamma)), shape, c_l)
    a = _scatter(h)
    p = oracle.Params(nx=nx, ny=ny, nz=nz, tau=0.8, c_l=c_l, eos=1, eos_gamma=gamma, eos_mass=mass)
    ref = oracle.step(p, a)
    sim = RLB(nx, ny, nz, 0.8, c_l=c_l, precision="fp64", eos="gamma_law", eos_gamma=gamma, eos_mass=mass, device="cuda:0")
    sim.load_state(sim.cells_to_state(torch.from_numpy(a).cuda()))
    n0, e0, b0, _ = sim.macro(state=sim.cells_to_state(torch.from_numpy(h).cuda()), where="host")
    sim.step(1)
    got = sim.state_to_cells(sim.state()).cpu().numpy()
    sim.close()
    rn, re, rb, _ = oracle.macro(p, h)
    E, M, S = h[..., 1, :].sum(-1), c_l * (h[..., 1, :] @ EV.astype(float)), h[..., 0, :].sum(-1)
    # clearly physical: |M| < 0.98 E, a mass share below 0.3 of the rest-frame energy
    ok = (E > 0) & ((M * M).sum(-1) < 0.96 * E * E) & (S > 0) & (mass * S < 0.3 * np.sqrt(np.maximum(E * E - (M * M).sum(-1), 0)))
    ok &= np.isfinite(ref).all((-1, -2))
    assert ok.mean() > 0.05
    for s_ in range(2):
        big = np.abs(h[..., s_, :]).max(-1)[ok]
        err = np.abs(got[..., s_, :] - ref[..., s_, :])[ok].max(-1)
        assert np.all(err <= 2 * UNITS * 2.0 ** -53 * big), (s_, (err / big).max() * 2.0 ** 53)
    tol = 2 * UNITS * 2.0 ** -53
    assert np.all(np.abs(n0 - rn)[ok] <= tol * np.abs(h[..., 0, :]).sum(-1)[ok])
    assert np.all(np.abs(e0 - re)[ok] <= tol * np.abs(h[..., 1, :]).sum(-1)[ok])
    assert np.all(np.abs(b0 - rb)[:, ok] <= tol * (c_l * np.abs(h[..., 1, :]).sum(-1) / E)[ok])
