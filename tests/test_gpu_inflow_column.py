"""The inflow column and the solid markers of the FP32 step: both pass through
the gather of their warp, and keep their bits whatever they hold."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(3, 1, 1), (33, 5, 4), (63, 41, 29), (64, 40, 40)]  # both launch shapes of the default rule


@pytest.mark.parametrize("c_l", [1.0, 10.0])
@pytest.mark.parametrize("shape", SHAPES, ids=["%dx%dx%d" % s for s in SHAPES])
def test_inflow_column_and_markers_keep_their_bits(shape, c_l, monkeypatch):
    from paper_0912_2913_gb300 import RLB

    nx, ny, nz = shape
    rng = np.random.default_rng(5)
    n = 1.0 + 0.05 * rng.random((nz, ny, nx))
    beta = 0.02 * rng.random((3, nz, ny, nx))
    solid = np.zeros((nz, ny, nx), np.uint8)
    if nx > 3:
        solid[1, 2, 2] = solid[2, 3, nx - 3] = solid[nz - 1, 0, 5] = solid[2, 2, 7] = 1

    def one(variant):
        if variant is None:
            monkeypatch.delenv("RLB_F32_VARIANT", raising=False)
        else:
            monkeypatch.setenv("RLB_F32_VARIANT", variant)
        with RLB(nx, ny, nz, 0.8, c_l=c_l, precision="fp32", xbc="inflow_outflow", beta_in=(0.1, 0.0, 0.0),
                 device="cuda:0") as sim:
            sim.init_fields(n, n, beta, solid if nx > 3 else None)
            a, b = sim.state().clone(), sim.new_state()
            bits = a.view(torch.int32)
            col = torch.arange(0, sim.N, nx, device=a.device)
            if nx > 3:  # an infinity, a NaN with a payload and a negative zero in cells that only others gather
                for k, v in ((7, 0x7F800000), (8, 0x7FC12345), (9, -2 ** 31)):
                    bits[k + 3, col[k]] = v
            b.fill_(3.0)
            sim.step_into(a, b, counted=True)
            return bits, b.view(torch.int32), col, sim.N, sim.stats()

    a, b, col, N, st = one(None)
    assert torch.equal(a[:, col], b[:, col])
    mark = torch.from_numpy(solid.reshape(-1).astype(bool)).to(a.device)
    assert torch.equal(a[:, :N][:, mark], b[:, :N][:, mark])
    if c_l == 1.0:  # the persistent shape copies the column and tests its markers by loads of their own
        _, ref, _, _, st_ref = one("4")
        assert torch.equal(b[:, :N], ref[:, :N])
        assert (st["n_unphysical"], st["n_nonpositive_eq"]) == (st_ref["n_unphysical"], st_ref["n_nonpositive_eq"])


@pytest.mark.parametrize("eos", ["ultra", "gamma_law"])
@pytest.mark.parametrize("shape", [(3, 1, 1), (33, 5, 4), (64, 40, 40)], ids=str)
def test_inflow_column_keeps_its_bits_fp64(shape, eos):
    from paper_0912_2913_gb300 import RLB

    nx, ny, nz = shape
    rng = np.random.default_rng(6)
    n = 1.0 + 0.05 * rng.random((nz, ny, nx))
    beta = 0.02 * rng.random((3, nz, ny, nx))
    kw = dict(eos="gamma_law", eos_gamma=1.25, eos_mass=0.1) if eos == "gamma_law" else {}
    with RLB(nx, ny, nz, 0.8, precision="fp64", xbc="inflow_outflow", beta_in=(0.1, 0.0, 0.0), device="cuda:0",
             **kw) as sim:
        sim.init_fields(n, n, beta, None)
        a, b = sim.state().clone(), sim.new_state()
        b.fill_(3.0)
        bits, col = a.view(torch.int64), torch.arange(0, sim.N, nx, device=a.device)
        if nx > 3:
            for k, v in ((7, 0x7FF0000000000000), (8, 0x7FF8000012345678), (9, -2 ** 63), (15, 0)):
                bits[k + 3, col[k]] = v
        sim.step_into(a, b, counted=True)
        assert torch.equal(bits[:, col], b.view(torch.int64)[:, col])
        if nx <= 3:
            return
        # away from the column's unusual cells the step is the one of the plain column
        c, d = sim.state().clone(), sim.new_state()
        sim.step_into(c, d)
        inner = torch.arange(sim.N, device=a.device) % nx > 1
        assert torch.equal(b[:, :sim.N][:, inner], d[:, :sim.N][:, inner])
