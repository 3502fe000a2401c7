"""Packed symmetric copies of the elastic S_K (16 x 16 units): block sizes that fill the last unit, leave
one entry in it or need a single one, one element up to several CTAs, and every per-element degree. A mixed
solve to rtol 1e-12 (inner operator: the FP32 or FP16 copy; residual: the double-float copy) against the
FP64 path, which reads the full blocks: <= 1e-9, the parity bar of the mixed modes."""
import numpy as np
import pytest

from gpu_helpers import mesh, relerr
from paper_1807_00086_gb300 import inputs

pytestmark = pytest.mark.gpu


def _solve(vert, elem, k, prec, **opt):
    import torch
    from paper_1807_00086_gb300 import hdg
    ne = elem.shape[0]
    s = hdg.Solver(vert, elem, k, 1.0, inputs.loguniform(ne, 0.5, 2.0, 7), lam=inputs.lognormal(ne, 1.5, 0.5, 8),
                   mu=inputs.lognormal(ne, 1.0, 0.5, 9), prec=prec, rtol=1e-12, **opt)
    s.hdg_condense(50.0)
    F = torch.randn(s._fshape, dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda()
    lam = s.empty_traces()
    s.hdg_trace_solve(s.hdg_condensed_rhs(F), lam)
    return lam.cpu().numpy()


@pytest.mark.parametrize("dim,N,k", [(2, 1, 4), (2, 5, 4), (2, 2, 3), (3, 1, 1), (3, 1, 2), (3, 2, 3), (3, 3, 2)])
def test_uniform_degree(dim, N, k):
    vert, elem = mesh(dim, N)
    ref = _solve(vert, elem, k, "fp64")
    assert relerr(_solve(vert, elem, k, "mixed"), ref) < 1e-9


@pytest.mark.parametrize("ks", [(1,), (2,), (3,), (4,), (1, 4), (2, 3), (1, 2, 3, 4)])
@pytest.mark.parametrize("prec", ["mixed", "mixed16"])
def test_per_element_degrees(ks, prec):
    vert, elem = mesh(3, 2)
    ek = np.resize(np.array(ks, dtype=np.int32), elem.shape[0])
    ref = _solve(vert, elem, 4, "fp64", elem_k=ek)
    assert relerr(_solve(vert, elem, 4, prec, elem_k=ek), ref) < 1e-9
