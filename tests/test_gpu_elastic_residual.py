"""Elastic mixed solves at the default tolerance of 1e-13 and a large time step (alpha = 0.2), with a random
right-hand side on the interior faces: a residual in pairs of floats stalls at 1e-13 to 2e-13 of |r| there, the
FP64 blocks give one that is good to about 1e-14, and the refinement converges. The bound: the same product
once more, whose sums may differ by that much."""
import pytest

from gpu_helpers import mesh
from paper_1807_00086_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device_loops", [True, False])
@pytest.mark.parametrize("dim,N,k", [(3, 3, 2), (3, 2, 3), (2, 12, 4), (3, 3, 1)])
def test_default_tolerance_at_a_large_step(dim, N, k, device_loops):
    import torch
    from paper_1807_00086_gb300 import hdg
    vert, elem = mesh(dim, N)
    ne = elem.shape[0]
    s = hdg.Solver(vert, elem, k, 1.0, inputs.loguniform(ne, 0.5, 2.0, 7), lam=inputs.lognormal(ne, 1.5, 0.5, 8),
                   mu=inputs.lognormal(ne, 1.0, 0.5, 9), prec="mixed", device_loops=device_loops)
    s.hdg_condense(0.2)
    g = torch.Generator().manual_seed(5)
    x, r = (torch.randn(s._tshape, dtype=torch.float64, generator=g).cuda() for _ in range(2))
    r = torch.where(s.hdg_trace_apply(x) == 0, torch.zeros_like(r), r)   # boundary entries carry no equation
    lam = s.empty_traces()
    info = s.hdg_trace_solve(r, lam)
    kl = s.hdg_trace_apply(lam)
    res = min(float((r - sg * kl).norm()) for sg in (1.0, -1.0)) / float(r.norm())
    assert info["rel_residual"] <= 1e-13 and res <= 1.2e-13
