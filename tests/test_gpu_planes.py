"""3D grids of few tiles: one or two planes per tile, and the correction interpolated in the first
post-sweep, against four planes per tile and separate passes (tile_rows = 4).  The same sums in the same
order: equal bit for bit.  41^3 takes one plane, 49^3 and 57^3 two, 65^3 four on level 0."""
import pytest
import torch

from paper_2506_18694_gb300 import hh

pytestmark = pytest.mark.gpu
S, D = hh.SOMMERFELD, hh.DIRICHLET


@pytest.mark.parametrize("n,levels,nu_post,bc", [
    (2, 2, 2, (S, S, S, S, D, S)),
    (8, 3, 1, (D, S, S, D, S, S)),
    (30, 2, 3, (S, D, D, S, S, D)),
    (40, 4, 2, (S, S, S, S, D, S)),
    (48, 4, 2, (D, D, S, D, D, D)),
    (56, 4, 1, (S, S, S, S, S, S)),
    (64, 4, 2, (S, S, D, S, D, S)),
])
@pytest.mark.parametrize("nb", [1, 3])
def test_planes_and_fused_prolongation(libhh, n, levels, nu_post, bc, nb):
    k = 5.0 if nb == 1 else [3.0, 5.0, 4.0]
    out = []
    for rows in (0, 4):
        o = hh.default_options(levels=levels, nu_post=nu_post, restart=2, tile_rows=rows)
        g = torch.Generator(device="cuda").manual_seed(n)
        with hh.Problem(3, n, k, 0.0, k, bc, o) as p:
            r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g)
            out.append([p.precondition(r), p.precondition(r), p.vcycle(r.to(torch.complex64))])
    for a, b in zip(*out):
        assert torch.equal(a, b)
