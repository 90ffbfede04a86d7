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
