"""The device timer of the FP32 apply counts the launches that multiply, and nothing between them: as many as
there were iterations, and no time in which the host let the GPU idle between two solves (the bound is half of
the time slept; the launches themselves take microseconds)."""
import time

import pytest

from gpu_helpers import mesh
from paper_1807_00086_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device_loops", [True, False])
def test_idle_time_is_not_counted(device_loops):
    import torch
    from paper_1807_00086_gb300 import hdg
    vert, elem = mesh(2, 12)
    ne = elem.shape[0]
    s = hdg.Solver(vert, elem, 2, 1.0, inputs.loguniform(ne, 0.5, 2.0, 3), inputs.loguniform(ne, 1.0, 3.0, 4),
                   prec="mixed", rtol=1e-12, device_loops=device_loops)
    s.hdg_condense(300.0)
    r = s.hdg_condensed_rhs(torch.randn(s._fshape, dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda())
    s.hdg_trace_solve(r, s.empty_traces())
    s.hdg_get_stats(reset=True)
    pause, solves, its = 0.03, 5, 0
    for _ in range(solves):
        its += s.hdg_trace_solve(r, s.empty_traces())["iterations"]
        torch.cuda.synchronize()
        time.sleep(pause)
    st = s.hdg_get_stats()
    assert st["dev_apply32_launches"] == its
    assert 0.0 < st["dev_apply32_ms"] < 0.5e3 * pause * solves
