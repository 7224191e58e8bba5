"""2D tiles with and without their check-free form: the finest grid's nodes times the problems decide (200k
in complex64, 55k in complex128), so a problem alone takes the one and two of them together the other.
Equal bit for bit, through whole cycles and the kernels one by one."""
import pytest
import torch

from paper_2506_18694_gb300 import hh

pytestmark = pytest.mark.gpu
S, D = hh.SOMMERFELD, hh.DIRICHLET
DT = {hh.HH_C128: torch.complex128, hh.HH_C64: torch.complex64}


@pytest.mark.parametrize("prec,n,levels", [
    (hh.HH_C64, 316, 3), (hh.HH_C64, 352, 4), (hh.HH_C64, 440, 4), (hh.HH_C128, 168, 4), (hh.HH_C128, 232, 3)])
@pytest.mark.parametrize("bc", [(S, S, S, S), (D, S, S, D)])
@pytest.mark.parametrize("o", [dict(), dict(fuse_sweeps=0, nu_pre=3), dict(nu_post=1)],
                         ids=["default", "separate", "post1"])
def test_one_problem_alone_and_in_a_pair(libhh, prec, n, levels, bc, o):
    k = 9.0
    opt = dict(precision=prec, levels=levels, restart=1, coarse_kernel=1, **o)
    with hh.Problem(2, n, k, 0.0, k, bc, hh.default_options(**opt)) as p, \
            hh.Problem(2, n, [k, k], 0.0, [k, k], bc, hh.default_options(**opt)) as q:
        g = torch.Generator(device="cuda").manual_seed(n)
        r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g)
        x = torch.randn(p.size(), dtype=DT[prec], device="cuda", generator=g)
        b = r.to(DT[prec])
        two = lambda v: torch.cat([v, v])
        for a, c in ((p.precondition(r), q.precondition(two(r))), (p.vcycle(b), q.vcycle(two(b))),
                     (p.jacobi(0, b, x), q.jacobi(0, two(b), two(x))),
                     (p.residual_restrict(0, b, x), q.residual_restrict(0, two(b), two(x))),
                     (p.apply(0, "AL", x), q.apply(0, "AL", two(x)))):
            assert torch.equal(two(a), c)
