"""Equilibrium initialisation and macroscopic output (fixed-point sums and
terms, csrc/rlb_fields.cu) against the oracle at the edges of their range:
|beta| from 0 to 0.999 (cells on the binary64 path among them), lattice speeds
on both sides of the limits, fields far from the single precision reference,
extreme magnitudes."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


def _fields(seed, scale, shape=(3, 5, 41)):
    rng = np.random.default_rng(seed)
    N = int(np.prod(shape))
    b = rng.normal(size=(3, N))
    b *= rng.choice([0.0, 1e-9, 0.1, 0.5, 0.9, 0.99, 0.999], N) / np.linalg.norm(b, axis=0)
    n, e = (scale * np.exp(rng.uniform(-3, 3, (2, N))))
    return n.reshape(shape), e.reshape(shape), b.reshape((3,) + shape)


@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e25])
@pytest.mark.parametrize("c_l", [1.0, 2.0, 2.0 + 2 ** -30, 10.0, 17.0])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_init_and_macro(prec, c_l, scale):
    from paper_0912_2913_gb300 import RLB

    n, e, b = _fields(int(10 * c_l), scale)
    shape = n.shape
    p = oracle.Params(nx=shape[2], ny=shape[1], nz=shape[0], tau=0.8, c_l=c_l)
    ref = oracle.init(p, n, e, b)
    n_ref, e_ref = 0.7 * scale, 0.2 * scale
    sim = RLB(shape[2], shape[1], shape[0], 0.8, c_l=c_l, precision=prec, n_ref=n_ref, eps_ref=e_ref, device="cuda:0")
    sim.init_fields(n, e, b)
    got = sim.state_to_cells(sim.state()).double().cpu().numpy()
    gam2 = 1 / (1 - (b * b).sum(0))
    # 1 - |beta|^2 carries a few roundings times gamma^2 on both sides
    big = np.abs(ref).max(-1, keepdims=True)
    tol = 16 * U * gam2[..., None, None] * big
    full = got
    if prec == "fp32":
        rest = oracle.init(oracle.Params(nx=1, ny=1, nz=1, tau=0.8, c_l=c_l), np.full((1, 1, 1), n_ref),
                           np.full((1, 1, 1), e_ref), np.zeros((3, 1, 1, 1)))
        full = got + rest
        # the stored deviation is rounded once to binary32
        tol = tol + 2.0 ** -24 * 1.01 * np.abs(got) + 16 * U * np.abs(rest)
    assert np.all(np.abs(full - ref) <= tol), np.max(np.abs(full - ref) / tol)
    # the macroscopic fields of what is stored
    nn, ee, bb, ok = sim.macro(where="host")
    ref_n, ref_e, ref_b, bad = oracle.macro(p, np.ascontiguousarray(full))
    sim.close()
    E = full[..., 1, :].sum(-1)
    M2 = ((c_l * full[..., 1, :] @ np.asarray(oracle.lattice()[0], float)) ** 2).sum(-1)
    m = (M2 < 0.99 * E * E) & (E > 0)  # eps well resolved in both
    assert m.mean() > 0.5 and ok == (bad == 0)
    cond = (np.abs(full).sum((-1, -2)) / ref_e)[m]  # E / eps and the sums' size
    assert np.all(np.abs(ee - ref_e)[m] <= 32 * U * cond * ref_e[m])
    assert np.all(np.abs(nn - ref_n)[m] <= 32 * U * (cond + np.abs(full[..., 0, :]).sum(-1)[m] / ref_n[m]) * ref_n[m])
    spread = c_l * np.abs(full[..., 1, :]).sum(-1) / E
    assert np.all(np.abs(bb - ref_b)[:, m] <= 32 * U * spread[m])


def test_fp32_init_keeps_the_binary64_bits(monkeypatch):
    """The stored deviations are those of the binary64 equilibria rounded once:
    c_l just above the fixed-point limit runs the binary64 form, and lattice
    speeds scale out of the f populations at |beta| = 0 only, so the check
    restates the binary64 form in numpy, operation by operation."""
    from paper_0912_2913_gb300 import RLB

    n, e, b = _fields(77, 1.0, (16, 64, 128))
    b[:, :8] *= np.minimum(1.0, 0.6 / np.maximum(np.sqrt((b[:, :8] ** 2).sum(0)), 1e-30))
    n_ref, e_ref = 0.4, 0.3
    sim = RLB(128, 64, 16, 0.8, precision="fp32", n_ref=n_ref, eps_ref=e_ref, device="cuda:0")
    sim.init_fields(n, e, b)
    got = sim.state_to_cells(sim.state()).cpu().numpy()
    sim.close()
    bx, by, bz = b
    b2 = bx * bx + by * by + bz * bz
    gam2 = 1.0 / (1.0 - b2)
    ng, eg = n * np.sqrt(gam2), e * gam2
    want = np.empty(n.shape + (2, 19), np.float32)
    w0 = 1.0 / 3.0
    want[..., 0, 0] = w0 * ng - w0 * n_ref
    want[..., 1, 0] = w0 * (4.0 * eg - e * (2.0 * 1.0 + 1.0) - 2.0 * eg * b2 * 1.0) - w0 * e_ref * (3.0 - 2.0)
    for p, q in enumerate((bx, by, bz, bx + by, bx - by, bx + bz, bx - bz, by + bz, by - bz)):
        w = 1.0 / 18.0 if p < 3 else 1.0 / 36.0
        fa = 3.0 * q * 1.0
        gs, ga = e * 1.0 + eg * (6.0 * q * q - 2.0 * b2) * 1.0, eg * 4.0 * q * 1.0
        for s, i in ((1, 2 * p + 1), (-1, 2 * p + 2)):
            want[..., 0, i] = w * ng * (1.0 + s * fa) - w * n_ref
            want[..., 1, i] = w * (gs + s * ga) - w * e_ref * 1.0
    assert np.array_equal(got.view(np.int32), want.view(np.int32))


@pytest.mark.parametrize("c_l", [1.0, 2.0, 2.0 + 2 ** -30])
@pytest.mark.parametrize("gamma,mass", [(1.2, 0.3), (5 / 3, 0.0), (2.0, 0.9)])
def test_general_eos_init(gamma, mass, c_l):
    """Initial equilibria of the general equation of state, pressures from
    below zero to eps among them.  Bound as above; the relative error of
    P / ((eps + P) gamma^2) in the equilibria is covered by 4 units more."""
    from paper_0912_2913_gb300 import RLB

    n, e, b = _fields(int(10 * c_l + 7 * gamma), 1.0)
    p = oracle.Params(nx=41, ny=5, nz=3, tau=0.8, c_l=c_l, eos=1, eos_gamma=gamma, eos_mass=mass)
    ref = oracle.init(p, n, e, b)
    sim = RLB(41, 5, 3, 0.8, c_l=c_l, precision="fp64", eos="gamma_law", eos_gamma=gamma, eos_mass=mass, device="cuda:0")
    sim.init_fields(n, e, b)
    got = sim.state_to_cells(sim.state()).cpu().numpy()
    sim.close()
    gam2 = 1 / (1 - (b * b).sum(0))
    # a pressure formed by cancellation: eps - m n against their size
    size = np.abs(ref).max(-1, keepdims=True) + ((e + mass * n) * gam2)[..., None, None]
    assert np.all(np.abs(got - ref) <= 20 * U * gam2[..., None, None] * size)


@pytest.mark.parametrize("c_l", [1.0, 2.0, 10.0])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_macro_and_field_adjoints(prec, c_l):
    """Adjoints of the macroscopic output and of the initial equilibria over
    the fields above, zero output gradients in part of the lattice and lambda
    of very different sizes.  Bounds: 64 roundings times gamma^2 (the velocity
    terms of eps and n) of the sum of the terms' sizes; stored binary32 lambdas
    one rounding more."""
    from paper_0912_2913_gb300 import RLB

    n, e, b = _fields(int(10 * c_l) + 5, 1.0)
    shape = n.shape
    p = oracle.Params(nx=shape[2], ny=shape[1], nz=shape[0], tau=0.8, c_l=c_l)
    n_ref, e_ref = 0.7, 0.2
    sim = RLB(shape[2], shape[1], shape[0], 0.8, c_l=c_l, precision=prec, n_ref=n_ref, eps_ref=e_ref, device="cuda:0")
    sim.init_fields(n, e, b)
    full = sim.state_to_cells(sim.state()).double().cpu().numpy()
    if prec == "fp32":
        full = full + oracle.init(oracle.Params(nx=1, ny=1, nz=1, tau=0.8, c_l=c_l), np.full((1, 1, 1), n_ref),
                                  np.full((1, 1, 1), e_ref), np.zeros((3, 1, 1, 1)))
    rng = np.random.default_rng(4)
    gn, ge = rng.normal(size=(2,) + shape)
    gb = rng.normal(size=(3,) + shape)
    gn[0] = 0.0
    ge[0, 0] = 0.0
    gb[:, 0] = 0.0
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    lam = sim.new_state()
    sim.adjoint_macro(sim.state(), t(gn), t(ge), t(gb), lam)
    got = sim.state_to_cells(lam).double().cpu().numpy()
    want = oracle.adjoint_macro(p, np.ascontiguousarray(full), gn, ge, gb)
    E, S = full[..., 1, :].sum(-1), full[..., 0, :].sum(-1)
    gam2 = 1 / (1 - (b * b).sum(0))
    size = np.abs(ge) * 9 + (np.abs(gb).sum(0) + np.abs(gn) * np.abs(S) * np.sqrt(gam2)) * (1 + c_l) * 6 / E + np.abs(gn)
    tol = 64 * U * gam2 * size * (np.abs(full).sum((-1, -2)) / np.minimum(np.abs(E), np.abs(S)))
    tol = np.broadcast_to(tol[..., None, None], want.shape)
    if prec == "fp32":
        tol = tol + 2.0 ** -24 * 1.01 * np.abs(got) + 1e-45
    m = gam2 < 40
    assert np.all((np.abs(got - want) <= tol)[m]), np.max((np.abs(got - want) / tol)[m])
    # the initial fields
    l0 = rng.normal(size=got.shape) * np.exp(rng.uniform(-20, 20, size=shape))[..., None, None]
    l0[0, 1] = 0.0
    ls = sim.cells_to_state(t(l0))
    l0 = sim.state_to_cells(ls).double().cpu().numpy()
    outs = [torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(2)]
    db, acc = torch.empty((3,) + shape, dtype=torch.float64, device="cuda"), torch.zeros(3, dtype=torch.float64, device="cuda")
    sim.adjoint_fields(t(n), t(e), t(b), ls, outs[0], outs[1], db, acc)
    ref = oracle.adjoint_fields(p, n, e, b, np.ascontiguousarray(l0))
    sim.close()
    big = np.abs(l0).max((-1, -2)) * gam2
    assert np.all(np.abs(outs[0].cpu().numpy() - ref[0]) <= 64 * U * gam2 * big)
    assert np.all(np.abs(outs[1].cpu().numpy() - ref[1]) <= 64 * U * gam2 * big * 8)
    assert np.all(np.abs(db.cpu().numpy() - ref[2]) <= 64 * U * gam2 ** 2 * big * 16 * (n + e))
