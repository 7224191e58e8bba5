"""Cluster-resident cycles and HSS loops of small 2D problems (one launch, every level in distributed
shared memory) against the separate kernels of the same arithmetic: equal bit for bit.

Sizes cover one CTA (all levels replicated), clusters with one to three distributed levels, odd
coarsest levels, rows that do not divide evenly over the CTAs, two rounds of items, r read back from
global memory (257^2), and level counts 2 to 5."""
import pytest
import torch

from paper_2506_18694_gb300 import hh

pytestmark = pytest.mark.gpu
S, D = hh.SOMMERFELD, hh.DIRICHLET

CASES = [
    # n, levels, k, tags, nu_coarse
    (2, 2, 3.0, (S, S, S, S), 8),
    (4, 3, 3.0, (S, D, S, S), 8),
    (24, 4, 9.5, (S, D, S, S), 1),
    (32, 4, 10.0, (D, D, D, D), 8),
    (40, 4, 12.0, (D, S, S, D), 7),
    (64, 4, 14.0, (S, S, S, S), 8),
    (88, 4, 16.0, (S, S, D, S), 8),
    (104, 2, 10.0, (S, S, S, S), 8),
    (128, 5, 20.0, (D, S, S, S), 5),
    (200, 4, 11.0, (S, S, S, D), 8),
    (256, 4, 20.0, (S, D, S, S), 8),
]


@pytest.mark.parametrize("prec", [hh.HH_C64, hh.HH_C128], ids=["c64", "c128"])
@pytest.mark.parametrize("n,levels,k,bc,nuc", CASES, ids=[str(c[0]) for c in CASES])
def test_resident_equals_separate_kernels(libhh, prec, n, levels, k, bc, nuc):
    dt = torch.complex64 if prec == hh.HH_C64 else torch.complex128
    o = dict(precision=prec, levels=levels, nu_coarse=nuc, restart=2)
    g = torch.Generator(device="cuda").manual_seed(n)
    # coarse_kernel = 1 asks for the separate kernels' cluster solve of the coarsest level
    with hh.Problem(2, n, k, 0.0, k, bc, hh.default_options(**o)) as p, \
            hh.Problem(2, n, k, 0.0, k, bc, hh.default_options(coarse_kernel=1, **o)) as q:
        r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g)
        for _ in range(2):  # (the second pass starts from the first one's buffers)
            assert torch.equal(p.precondition(r), q.precondition(r))
            assert torch.equal(p.vcycle(r.to(dt)), q.vcycle(r.to(dt)))


@pytest.mark.parametrize("n,nb", [(32, 3), (64, 7), (64, 12), (96, 20)])
def test_resident_batch(libhh, n, nb):
    """A batch with uneven HSS lengths: as many clusters as problems while the device holds them."""
    ks = [4.0 + (3 * b) % 7 for b in range(nb)]
    g = torch.Generator(device="cuda").manual_seed(nb)
    with hh.Problem(2, n, ks, 0.0, ks, (S, S, D, S), hh.default_options(restart=2)) as p, \
            hh.Problem(2, n, ks, 0.0, ks, (S, S, D, S), hh.default_options(restart=2, coarse_kernel=1)) as q:
        r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g)
        assert torch.equal(p.precondition(r), q.precondition(r))
