"""The GMRES smoothing step of a 2D level in one launch, over the sizes where its split changes: one
CTA, clusters of 2 to 16 (bands of uneven height), one, two and five nodes a thread, the largest
band that fits shared memory and the first that does not (separate kernels), one to eight
iterations (one and two groups of basis vectors).  A two-level cycle smooths from 0 and from an
iterate.  Tolerances as in the cycle tests of this smoother: the oracle orthogonalises by modified
Gram-Schmidt, so 1e-10 relative in complex128 and 2e-4 in complex64.
"""
import numpy as np
import pytest
import torch

from oracle import hh_oracle as O
from nodewise import rel
from paper_2506_18694_gb300 import hh, inputs

pytestmark = pytest.mark.gpu

S, D = O.SOMMERFELD, O.DIRICHLET
TOL = {hh.HH_C128: 1e-10, hh.HH_C64: 2e-4}
DT = {hh.HH_C128: torch.complex128, hh.HH_C64: torch.complex64}


@pytest.mark.parametrize("prec", [hh.HH_C64, hh.HH_C128])
@pytest.mark.parametrize("n,its,bc", [
    (4, 1, (S, S, S, S)), (20, 5, (D, S, S, S)), (24, 8, (S, S, D, D)), (34, 4, (S, D, S, S)),
    (50, 5, (S, S, S, D)), (66, 3, (D, S, D, S)), (130, 5, (S, S, S, S)), (194, 2, (S, D, S, S)),
    (264, 5, (S, S, S, S)), (264, 6, (S, S, S, D)),
])
def test_step_matches_oracle(libhh, prec, n, its, bc):
    g = O.Grid(2, n, bc)
    k = 0.4 * n
    prob = O.Problem(g, k, 0.0, 0.5 * k, O.Options(smoother="gmres", levels=2, nu_pre=its, nu_post=its,
                                                   nu_coarse=its))
    b = inputs.random_complex(g.N, 4100 + n) * g.free()
    ref = prob.vcycle(0, b)
    o = hh.default_options(precision=prec, smoother=hh.HH_SMOOTH_GMRES, levels=2, nu_pre=its, nu_post=its,
                           nu_coarse=its)
    with hh.Problem(2, n, k, 0.0, 0.5 * k, bc, o) as p:
        x = p.vcycle(torch.from_numpy(b).to(DT[prec]).cuda()).cpu().numpy().astype(np.complex128)
    assert rel(x, ref) <= TOL[prec]
