"""Kernels that the default sizes and lattice speeds do not reach: the
binary64 FP64 step (c_l outside [1, 2]) against the oracle with solids and an
inflow plane, its eight-lane form against its one-thread form, the FP32 launch
shapes chosen by size against each other, and all of them through the
bounds-checking build."""
import json
import os
import subprocess
import sys

import pytest
import torch

import oracle
from tests._helpers import gpu_run, oracle_run, rel_errors, tiny_workload

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LATTICES = [(7, 5, 4, 0, ((3, 2, 2), (4, 2, 2))), (37, 9, 5, 1, ((12, 4, 2), (13, 4, 2), (12, 5, 2))), (9, 6, 4, 2, ((4, 2, 1),)),
            (3, 4, 5, 2, ())]


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


@pytest.mark.parametrize("c_l", [0.9, 3.0])
@pytest.mark.parametrize("size", LATTICES, ids=lambda s: f"{s[0]}x{s[1]}x{s[2]}_bc{s[3]}")
def test_binary64_step_kernels(size, c_l, monkeypatch):
    """k_step_f64 and k_step_f64_split: parity with the oracle, and the same
    values and statistics from both."""
    nx, ny, nz, xbc, solids = size
    w = tiny_workload(nx, ny, nz, xbc, seed=17, c_l=c_l, solid_cells=solids, bmax=0.25, beta_in=(0.2, 0.05, -0.02))
    stats = oracle.Stats()
    ref, _ = oracle_run(w, 20, stats)
    runs = []
    for force in ("0", "1"):
        monkeypatch.setenv("RLB_F64_SPLIT", force)
        got, sim = gpu_run(w, 20, "fp64")
        assert max(rel_errors(got, ref, w.solid)) <= 1e-10
        runs.append((sim.state()[:, :sim.N].clone(), sim.stats()))
        sim.close()
    (s0, st0), (s1, st1) = runs
    assert torch.equal(s0.isnan(), s1.isnan()) and torch.equal(torch.nan_to_num(s0), torch.nan_to_num(s1))
    assert st0 == st1 and st0["n_nonpositive_eq"] == stats.n_nonpositive_eq


@pytest.mark.parametrize("warps", [0.7, 2.9, 3.3, 3.8, 4.2, 6.5, 9.0, 13.0, 16.0])
def test_fp32_launch_shapes_by_size(warps, monkeypatch):
    """The shape that the rule takes (cells per SM from 0.7 to 16 times 128)
    and the plain one give the same bits."""
    from paper_0912_2913_gb300 import RLB

    sm = torch.cuda.get_device_properties(0).multi_processor_count
    ny, nz = 21, 19
    nx = int(warps * 128 * sm / (ny * nz))
    w = tiny_workload(nx, ny, nz, 1, seed=3, solid_cells=((nx // 2, 10, 9), (nx // 2, 11, 9)))
    states = []
    for var in (None, "0"):
        monkeypatch.delenv("RLB_F32_VARIANT", raising=False)
        if var:
            monkeypatch.setenv("RLB_F32_VARIANT", var)
        sim = RLB.from_workload(w, "fp32", device="cuda:0").init_fields(w.n, w.eps, w.beta, w.solid).step(3)
        states.append((sim.state()[:, :sim.N].clone(), sim.stats()))
        sim.close()
    assert torch.equal(states[0][0].view(torch.int32), states[1][0].view(torch.int32)) and states[0][1] == states[1][1]


@pytest.mark.slow
def test_dispatch_meets_no_out_of_range_index():
    from paper_0912_2913_gb300 import build

    build.build(bounds=True)
    env = dict(os.environ, RLB_LIBRARY_VARIANT="bounds")
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "bounds_dispatch_driver.py")], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["library"].startswith("librlb_bounds_")
    assert out["groups"] == {"forward": 0, "adjoint": 0}
    e = out["errors"]
    assert e["forward_fp64"] <= 1e-10 and e["forward_fp32"] <= 1e-4 and e["adjoint"] <= 1e-11, e
