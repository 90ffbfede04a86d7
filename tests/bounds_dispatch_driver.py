"""More of the dispatch through the bounds-checking debug build of librlb.

Run as a program of its own by ``tests/test_gpu_dispatch.py`` with
``RLB_LIBRARY_VARIANT=bounds`` in the environment.  Beside the cases of
``bounds_driver.py``: the default choice of the FP32 step and the launch shapes
that load f early, lattice speeds outside the fixed-point range (the binary64
FP64 step and adjoint, the compensated FP32 step), both FP64 step kernels on
every lattice, and three cells between two outflow ghosts.  It prints one JSON
line: out-of-range indices per group and the parity errors.
"""
import json
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import oracle  # noqa: E402
from tests._helpers import gpu_run, oracle_run, rel_errors, tiny_workload  # noqa: E402

CASES = [(6, 5, 4, 0, ((3, 2, 2),)), (9, 5, 4, 1, ((4, 2, 1), (5, 2, 1))), (9, 5, 4, 2, ((4, 2, 1),)), (3, 4, 5, 2, ()),
         (37, 9, 5, 1, ((12, 4, 2), (13, 4, 2), (12, 5, 2))), (70, 40, 33, 2, ((30, 20, 16), (31, 20, 16)))]
SPEEDS = (0.9, 1.0, 3.0)


def _env(**kw):
    for k in ("RLB_F32_VARIANT", "RLB_F64_SPLIT"):
        os.environ.pop(k, None)
    os.environ.update(kw)


def forward(out):
    from paper_0912_2913_gb300 import _native as N

    worst = {"fp64": 0.0, "fp32": 0.0}
    for nx, ny, nz, xbc, solids in CASES:
        for c_l in SPEEDS:
            w = tiny_workload(nx, ny, nz, xbc, seed=5, c_l=c_l, solid_cells=solids, bmax=0.2, beta_in=(0.2, 0.05, -0.02))
            ref, _ = oracle_run(w, 5)
            runs = [("fp64", dict(RLB_F64_SPLIT="0")), ("fp64", dict(RLB_F64_SPLIT="1")), ("fp64", {}), ("fp32", {})]
            if c_l == 1.0:
                runs += [("fp32", dict(RLB_F32_VARIANT=v)) for v in "678"]
            for prec, env in runs:
                _env(**env)
                got, sim = gpu_run(w, 5, prec)
                sim.close()
                worst[prec] = max(worst[prec], *rel_errors(got, ref, w.solid))
    _env()
    out["groups"]["forward"] = N.rlb_debug_bounds_violations()
    out["errors"].update({"forward_" + k: v for k, v in worst.items()})


def adjoint(out):
    from paper_0912_2913_gb300 import RLB
    from paper_0912_2913_gb300 import _native as N

    worst = 0.0
    rng = np.random.default_rng(1)
    for nx, ny, nz, xbc, solids in CASES:
        for c_l in SPEEDS:
            w = tiny_workload(nx, ny, nz, xbc, seed=6, c_l=c_l, solid_cells=solids, bmax=0.2, beta_in=(0.2, 0.05, -0.02))
            p = oracle.Params(**w.params())
            sim = RLB.from_workload(w, "fp64", device="cuda:0").init_fields(w.n, w.eps, w.beta, w.solid).step(2)
            state = sim.state().clone()
            fluid = (np.ones((nz, ny, nx), bool) if w.solid is None else w.solid == 0)[..., None, None]
            lam = rng.normal(size=(nz, ny, nx, 2, 19)) * fluid
            st = np.where(fluid, sim.state_to_cells(state).cpu().numpy(), oracle.init(p, w.n, w.eps, w.beta, w.solid))
            ref, _, _ = oracle.adjoint_step(p, st, lam, w.solid)
            li = sim.cells_to_state(torch.from_numpy(lam).cuda())
            for step in (N.rlb_adjoint_step, N.rlb_adjoint_step_noalloc):
                lo, acc = torch.zeros_like(li), torch.zeros(4, dtype=torch.float64, device="cuda")
                step(sim.ctx, state, li, lo, acc[0:1], acc[1:4])
                got = sim.state_to_cells(lo).cpu().numpy()
                worst = max(worst, float(np.max(np.abs(got - ref)[np.broadcast_to(fluid, ref.shape)])) / np.abs(ref).max())
            sim.close()
    out["groups"]["adjoint"] = N.rlb_debug_bounds_violations()
    out["errors"]["adjoint"] = worst


def main():
    assert os.environ.get("RLB_LIBRARY_VARIANT") == "bounds"
    from paper_0912_2913_gb300 import _native as N

    out = {"library": os.path.basename(N.library_path()), "groups": {}, "errors": {}}
    N.rlb_debug_bounds_violations()  # starts the count at zero
    forward(out)
    adjoint(out)
    print(json.dumps(out))


if __name__ == "__main__":
    main()
