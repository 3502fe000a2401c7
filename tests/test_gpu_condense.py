"""Condensation and operator copies on element counts around the kernels' groups (four or two
elements per warp, eight per packing block, 32 per packed group): every S_K against the oracle
(<= 1e-12), and a linear solve through each mixed-precision copy of S_K against the FP64 path
(<= 1e-9, the parity bar of the mixed modes)."""
import numpy as np
import pytest

from gpu_helpers import mesh, relerr
from oracle import acoustic as ac
from paper_1807_00086_gb300 import inputs

pytestmark = pytest.mark.gpu


def _submesh(dim, ne):
    vert, elem = mesh(dim, 5)
    elem = elem[:ne]
    used, inv = np.unique(elem, return_inverse=True)
    return vert[used], inv.reshape(elem.shape).astype(np.int32)


@pytest.mark.parametrize("dim,k", [(2, 1), (2, 2), (2, 4), (3, 1), (3, 3), (3, 4)])
@pytest.mark.parametrize("ne", [1, 3, 9, 33])
def test_partial_groups_schur_and_copies(dim, k, ne):
    import torch
    from paper_1807_00086_gb300 import hdg
    vert, elem = _submesh(dim, ne)
    rho, c = inputs.loguniform(ne, 0.5, 2.0, 3), inputs.loguniform(ne, 1.0, 3.0, 4)
    prob = ac.build_problem(vert, elem, k, 1.0, rho, c)
    alpha = 37.0
    cond = ac.condense(prob, alpha)
    F = torch.tensor(inputs.random_state(ne, (dim + 1) * prob.Np, 11), device="cuda")
    ref = None
    for prec, R in (("fp64", 1), ("mixed", 1), ("mixed16", 1), ("mixed", 4), ("mixed", 32)):
        s = hdg.Solver(vert, elem, k, 1.0, rho, c, prec=prec, rtol=1e-12, nrhs=R)
        s.hdg_condense(alpha)
        S = s.hdg_get_schur().cpu().numpy()
        assert relerr(S, np.array(cond.S)) < 1e-12
        FR = F if R == 1 else F[:, :, None].expand(-1, -1, R).contiguous()
        r = s.hdg_condensed_rhs(FR)
        lam = s.empty_traces()
        s.hdg_trace_solve(r, lam)
        u = s.hdg_recover(FR, lam).cpu().numpy()
        if ref is None:
            ref = u
        for j in range(R):
            assert relerr(u if R == 1 else u[:, :, j], ref) < 1e-9, (prec, R, j)
