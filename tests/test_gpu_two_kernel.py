"""The two-kernel FP32 Krylov iteration (direction formed in the operator's gather; update of all vectors
in one pass): one column and column blocks of 4, 8 and 16, on the smallest meshes (two triangles, one
cube), ragged element counts and more elements than one wave of CTAs holds, with the device-driven,
graph and plain host loops. A mixed solve to rtol 1e-12 against the FP64 path: <= 1e-9, the parity bar of
the mixed modes. A loop cut off by maxit runs exactly maxit updates a sweep, whichever loop drives it."""
import numpy as np
import pytest

from gpu_helpers import mesh, relerr
from paper_1807_00086_gb300 import inputs

pytestmark = pytest.mark.gpu


LOOPS = (dict(device_loops=True), dict(device_loops=False), dict(device_loops=False, use_graphs=True))


def _solve(vert, elem, k, alpha, F, **opt):
    import torch
    from paper_1807_00086_gb300 import hdg
    st = torch.cuda.Stream()   # a graph capture needs a stream of its own
    torch.cuda.synchronize()
    ne = elem.shape[0]
    rho, c = inputs.loguniform(ne, 0.5, 2.0, 3), inputs.loguniform(ne, 1.0, 3.0, 4)
    s = hdg.Solver(vert, elem, k, 1.0, rho, c, rtol=1e-12, stream=st, **opt)
    with torch.cuda.stream(st):
        s.hdg_condense(alpha)
        lam = s.empty_traces()
        info = s.hdg_trace_solve(s.hdg_condensed_rhs(F), lam)
    torch.cuda.synchronize()
    return lam.cpu().numpy(), info


def _rhs(ne, n, R, seed=11):
    import torch
    F = inputs.random_state(ne, n * R, seed).reshape((ne, n, R) if R > 1 else (ne, n))
    return torch.tensor(F, device="cuda")


def _n(dim, k):
    return (dim + 1) * ((k + 1) * (k + 2) // 2 if dim == 2 else (k + 1) * (k + 2) * (k + 3) // 6)


@pytest.mark.parametrize("R", [1, 4, 8, 16])
@pytest.mark.parametrize("dim,N,k", [(2, 1, 1), (2, 3, 4), (3, 1, 4), (3, 2, 3), (3, 3, 2)])
def test_mixed_solve_matches_fp64(dim, N, k, R):
    vert, elem = mesh(dim, N)
    F = _rhs(elem.shape[0], _n(dim, k), R)
    ref, _ = _solve(vert, elem, k, 300.0, F, prec="fp64", nrhs=R)
    for loops in LOOPS:
        lam, info = _solve(vert, elem, k, 300.0, F, prec="mixed", nrhs=R, **loops)
        assert relerr(lam, ref) < 1e-9, loops


@pytest.mark.parametrize("N,R", [(290, 1), (75, 16)])
def test_more_elements_than_one_wave(N, R):
    """k = 1 triangles: 168,200 elements for one column, 11,250 for sixteen."""
    vert, elem = mesh(2, N)
    F = _rhs(elem.shape[0], _n(2, 1), R)
    ref, _ = _solve(vert, elem, 1, 3000.0, F, prec="fp64", nrhs=R)
    lam, _ = _solve(vert, elem, 1, 3000.0, F, prec="mixed", nrhs=R)
    assert relerr(lam, ref) < 1e-9


@pytest.mark.parametrize("R", [1, 4])
def test_columns_without_right_hand_side_stay_zero(R):
    vert, elem = mesh(2, 4)
    F = _rhs(elem.shape[0], _n(2, 2), R)
    if R > 1:
        F[:, :, 1] = 0.0
    else:
        F.zero_()
    lam, _ = _solve(vert, elem, 2, 300.0, F, prec="mixed", nrhs=R)
    assert np.all((lam[:, :, 1] if R > 1 else lam) == 0.0) and np.all(np.isfinite(lam))


@pytest.mark.parametrize("R", [1, 4])
def test_maxit_bounds_every_sweep(R):
    vert, elem = mesh(2, 6)
    F = _rhs(elem.shape[0], _n(2, 2), R)
    ref, _ = _solve(vert, elem, 2, 300.0, F, prec="fp64", nrhs=R)
    seen = set()
    for loops in LOOPS:
        lam, info = _solve(vert, elem, 2, 300.0, F, prec="mixed", nrhs=R, maxit=4, max_sweeps=200, **loops)
        assert relerr(lam, ref) < 1e-9, loops
        assert info["iterations"] <= 4 * info["sweeps"]
        seen.add((info["iterations"], info["sweeps"]))
    assert len(seen) == 1
