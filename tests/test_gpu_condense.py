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


@pytest.mark.parametrize("dim,k", [(2, 2), (3, 1), (3, 3), (3, 4)])
@pytest.mark.parametrize("over", [0, 1, 3])
def test_either_side_of_the_small_mesh_rule(dim, k, over):
    """The last meshes with a CTA per element (4 or 8 elements per SM), and the first whose elements share a warp
    (partial last ones). The recovery checks the coefficients that either kernel leaves for the local solves."""
    import torch
    from paper_1807_00086_gb300 import hdg
    ne = (8 if dim == 3 and k < 4 else 4) * torch.cuda.get_device_properties(0).multi_processor_count + over
    vert, elem = mesh(dim, 20 if dim == 2 else 6)
    elem = elem[:ne]
    used, inv = np.unique(elem, return_inverse=True)
    vert, elem = vert[used], inv.reshape(elem.shape).astype(np.int32)
    rho, c = inputs.loguniform(ne, 0.5, 2.0, 3), inputs.loguniform(ne, 1.0, 3.0, 4)
    prob = ac.build_problem(vert, elem, k, 1.0, rho, c)
    cond = ac.condense(prob, 37.0)
    s = hdg.Solver(vert, elem, k, 1.0, rho, c)
    s.hdg_condense(37.0)
    assert relerr(s.hdg_get_schur().cpu().numpy(), np.array(cond.S)) < 1e-12
    F = inputs.random_state(ne, s.n, 11).reshape(ne, s.n)
    lam = inputs.random_traces(s.n_faces, s.Nf, 5).reshape(s.n_faces, s.Nf)
    u = s.hdg_recover(torch.tensor(F, device="cuda"), torch.tensor(lam, device="cuda")).cpu().numpy()
    assert relerr(u, ac.recover(prob, cond, F, lam)) < 1e-12


@pytest.mark.parametrize("dim,k", [(2, 1), (2, 2), (2, 3), (2, 4), (3, 1), (3, 2), (3, 3), (3, 4)])
def test_both_kernels_agree_at_the_rule(dim, k):
    """Up to a number of elements per SM a CTA condenses one element, above it a warp several: on both sides of
    that line, with every number of elements in the last warp, the last elements' S_K and local solves against
    those of a mesh of these elements alone (<= 1e-12: the same formulas in another order)."""
    import torch
    from paper_1807_00086_gb300 import hdg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    line = (6 if dim == 3 and k in (2, 3) else 4) * sms
    N = 1
    while (2 * N * N if dim == 2 else 6 * N ** 3) < line + 4:
        N += 1
    vert, elem = mesh(dim, N)
    rho, c = inputs.loguniform(line + 4, 0.5, 2.0, 3), inputs.loguniform(line + 4, 1.0, 3.0, 4)
    n = (dim + 1) * ((k + 1) * (k + 2) // 2 if dim == 2 else (k + 1) * (k + 2) * (k + 3) // 6)
    F = inputs.random_state(line + 4, n, 11)

    def blocks(ids):
        used, inv = np.unique(elem[ids], return_inverse=True)
        s = hdg.Solver(vert[used], inv.reshape(elem[ids].shape).astype(np.int32), k, 1.0, rho[ids], c[ids])
        s.hdg_condense(37.0)
        u = s.hdg_recover(torch.tensor(F[ids], device="cuda"), s.empty_traces())
        return s.hdg_get_schur().cpu().numpy(), u.cpu().numpy()

    for ne in range(line, line + 5):
        S, u = blocks(np.arange(ne))
        Sl, ul = blocks(np.arange(ne - 7, ne))
        assert relerr(S[-7:], Sl) < 1e-12 and relerr(u[-7:], ul) < 1e-12
