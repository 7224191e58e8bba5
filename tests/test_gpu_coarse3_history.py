"""A 3D result does not depend on what the process ran before: which coarsest levels run in a cluster (whose
sums go in another order than the separate sweeps') is decided by the grid alone.  17^3 and 6^3 coarsest
nodes, beyond one CTA's and within."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import sys, torch
from paper_2506_18694_gb300 import hh
S, D = hh.SOMMERFELD, hh.DIRICHLET
n = int(sys.argv[2])
if sys.argv[1] == "c128":
    with hh.Problem(2, 16, 3.0, 0.0, 3.0, (S,) * 4, hh.default_options(precision=hh.HH_C128, levels=2)) as p:
        p.vcycle(torch.ones(p.size(), dtype=torch.complex128, device="cuda"))
with hh.Problem(3, n, 5.0, 0.0, 5.0, (S, S, S, S, D, S), hh.default_options(levels=2, restart=1)) as p:
    g = torch.Generator(device="cuda").manual_seed(1)
    x = p.vcycle(torch.randn(p.size(), dtype=torch.complex64, device="cuda", generator=g))
print(torch.view_as_real(x).cpu().numpy().tobytes().hex())
"""


@pytest.mark.parametrize("n", [32, 10])
def test_result_does_not_depend_on_the_first_precision(libhh, n):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = [subprocess.run([sys.executable, "-c", CODE, first, str(n)], cwd=root, check=True, timeout=300,
                          capture_output=True, text=True).stdout for first in ("c64", "c128")]
    assert out[0] == out[1]
