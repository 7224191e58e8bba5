"""Which 3D coarsest levels run in a cluster: in a process whose first problem is complex128, a level
beyond one CTA (17^3 here) stays with separate sweeps, whose sums run in another order."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch
from paper_2506_18694_gb300 import hh
S, D = hh.SOMMERFELD, hh.DIRICHLET
with hh.Problem(2, 16, 3.0, 0.0, 3.0, (S, S, S, S), hh.default_options(precision=hh.HH_C128, levels=2)) as p:
    p.vcycle(torch.ones(p.size(), dtype=torch.complex128, device="cuda"))
out = []
for most in (100000, 0):
    o = hh.default_options(levels=2, restart=1, coarse_cluster_nodes=most)
    with hh.Problem(3, 32, 5.0, 0.0, 5.0, (S, S, S, S, D, S), o) as p:
        g = torch.Generator(device="cuda").manual_seed(1)
        out.append(p.vcycle(torch.randn(p.size(), dtype=torch.complex64, device="cuda", generator=g)))
assert torch.equal(out[0], out[1])
"""


def test_level_beyond_one_cta_after_a_complex128_problem(libhh):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", CODE], cwd=root, check=True, timeout=300)
