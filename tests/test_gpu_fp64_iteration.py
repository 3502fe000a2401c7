"""The FP64 Krylov iteration runs in two kernels where the operator has at most four CTAs per SM and in four
above: element counts that fill the last CTA of the two-kernel form exactly, and one more. A solve ends within
its tolerance (by the operator's own product; the bound is twice the tolerance, which the recurrence's drift of
about 1e-13 does not reach), n updates suffice where n are reported and n - 1 do not, and the device-driven
and the host loop give the same bits."""
import numpy as np
import pytest

from gpu_helpers import mesh
from paper_1807_00086_gb300 import inputs

pytestmark = pytest.mark.gpu

RTOL = 1e-8
# dim, k, elastic, trace entries of an element
SHAPES = [(2, 1, False, 6), (3, 2, False, 24), (2, 4, True, 30), (3, 3, True, 120)]


def _solver(dim, k, elastic, ne, **opt):
    import torch
    from paper_1807_00086_gb300 import hdg
    N = 1
    while (2 * N * N if dim == 2 else 6 * N ** 3) < ne:
        N += 1
    vert, elem = mesh(dim, N)
    elem = elem[:ne]
    used, inv = np.unique(elem, return_inverse=True)
    vert, elem = vert[used], inv.reshape(elem.shape).astype(np.int32)
    rho = inputs.loguniform(ne, 0.5, 2.0, 7)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    if elastic:
        return hdg.Solver(vert, elem, k, 1.0, rho, lam=inputs.lognormal(ne, 1.5, 0.5, 8),
                          mu=inputs.lognormal(ne, 1.0, 0.5, 9), rtol=RTOL, stream=st, **opt)
    return hdg.Solver(vert, elem, k, 1.0, rho, inputs.loguniform(ne, 1.0, 3.0, 4), rtol=RTOL, stream=st, **opt)


def _solve(s, elastic):
    import torch
    with torch.cuda.stream(s.stream):
        s.hdg_condense(50.0 if elastic else 300.0)
        F = torch.randn(s._fshape, dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda()
        r, lam = s.hdg_condensed_rhs(F), s.empty_traces()
        info = s.hdg_trace_solve(r, lam)
        kl = s.hdg_trace_apply(lam)
    torch.cuda.synchronize()
    return r, lam, kl, info


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("dim,k,elastic,m", SHAPES)
def test_both_forms(dim, k, elastic, m, extra):
    import torch
    from paper_1807_00086_gb300 import hdg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ne = 4 * sms * max(1, 128 // m) + extra
    got = []
    for loops in (True, False):
        r, lam, kl, info = _solve(_solver(dim, k, elastic, ne, device_loops=loops), elastic)
        res = min(float((r - sg * kl).norm()) for sg in (1.0, -1.0)) / float(r.norm())
        assert res <= 2 * RTOL and info["rel_residual"] <= RTOL
        n = info["iterations"]
        assert n > 2
        got.append((n, lam.cpu().numpy()))
        assert _solve(_solver(dim, k, elastic, ne, device_loops=loops, maxit=n), elastic)[3]["iterations"] == n
        with pytest.raises(hdg.HDGError) as err:
            _solve(_solver(dim, k, elastic, ne, device_loops=loops, maxit=n - 1), elastic)
        assert err.value.status == -4
    assert got[0][0] == got[1][0] and np.array_equal(got[0][1], got[1][1])
