"""Waits of the cluster-resident kernels that run out on purpose (a limit of one poll): the kernel gives
up at once and returns, the call reports it, and the next problems' results are right.  Every CTA of the
cluster gives up, at passes that differ; sizes have one to three distributed levels."""
import pytest
import torch

from paper_2506_18694_gb300 import hh

pytestmark = pytest.mark.gpu
S, D = hh.SOMMERFELD, hh.DIRICHLET
BC = (S, S, D, S)

CASES = [(64, 4, hh.HH_C64), (128, 5, hh.HH_C64), (256, 4, hh.HH_C64), (104, 2, hh.HH_C64), (32, 4, hh.HH_C128),
         (128, 4, hh.HH_C128)]


def _problem(n, levels, prec, nb=1, **kw):
    ks = [5.0 + b for b in range(nb)] if nb > 1 else 5.0
    return hh.Problem(2, n, ks, 0.0, ks, BC, hh.default_options(precision=prec, levels=levels, restart=2, **kw))


@pytest.mark.parametrize("nb", [1, 3])
@pytest.mark.parametrize("n,levels,prec", CASES)
def test_precondition_reports_a_wait_that_ran_out(libhh, n, levels, prec, nb):
    g = torch.Generator(device="cuda").manual_seed(n)
    with _problem(n, levels, prec, nb) as p, _problem(n, levels, prec, nb, coarse_kernel=1) as q, \
            _problem(n, levels, prec, nb, sync_spin_limit=1) as s:
        r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g)
        for _ in range(3):
            for call in (lambda: s.precondition(r), lambda: s.solve(r, 1e-8)):
                with pytest.raises(hh.HHError) as e:
                    call()
                assert e.value.status == hh.HH_ERR_TIMEOUT
        assert torch.equal(p.precondition(r), q.precondition(r))


@pytest.mark.parametrize("nb", [1, 3])
def test_vcycle_leaves_no_unfinished_result(libhh, nb):
    """hh_vcycle does not block: where its wait ran out, x is NaN and the next blocking call says so (here
    one whose own loop is not resident, and whose result is right)."""
    n, o = 136, dict(precision=hh.HH_C128, levels=4, restart=2)  # complex128 loop beyond the resident form's size
    ks = [5.0 + b for b in range(nb)] if nb > 1 else 5.0
    g = torch.Generator(device="cuda").manual_seed(n)
    with hh.Problem(2, n, ks, 0.0, ks, BC, hh.default_options(**o)) as p, \
            hh.Problem(2, n, ks, 0.0, ks, BC, hh.default_options(sync_spin_limit=1, **o)) as s:
        r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g)
        for _ in range(2):
            x = s.vcycle(r.to(torch.complex64))
            assert torch.isnan(x.real).all() and torch.isnan(x.imag).all()
            with pytest.raises(hh.HHError, match="hh_vcycle") as e:
                s.precondition(r)
            assert e.value.status == hh.HH_ERR_TIMEOUT
            assert torch.equal(s.precondition(r), p.precondition(r))
        assert torch.isfinite(torch.view_as_real(p.vcycle(r.to(torch.complex64)))).all()
