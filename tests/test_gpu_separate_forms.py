"""The separate kernels on small 2D problems, which otherwise run cluster-resident: packed launches, packs
that hold members of both kinds, tuned shapes, graph replays.  coarse_kernel = 1 asks for them (so does
a size beyond the resident form's); the number of launches shows which form ran."""
import numpy as np
import pytest
import torch

from paper_2506_18694_gb300 import hh, inputs

pytestmark = pytest.mark.gpu
S, D = hh.SOMMERFELD, hh.DIRICHLET
TOL = 1e-9
SEP = dict(coarse_kernel=1)


def _loop_launches(n, k=12.0, **o):
    """launches of one outer iteration: 12 HSS steps, 7 kernels each, or one resident loop"""
    with hh.Problem(2, n, k, 0.0, k, (S,) * 4, hh.default_options(max_outer=1, **o)) as p:
        b = torch.ones(p.size(), dtype=torch.complex128, device="cuda")
        return p.solve(b, TOL)[1].kernel_launches


@pytest.mark.parametrize("n,o,resident", [
    (32, {}, True), (256, {}, True), (264, {}, False), (128, dict(precision=hh.HH_C128), True),
    (136, dict(precision=hh.HH_C128), False), (32, SEP, False), (128, SEP, False), (32, dict(fuse_sweeps=0), False),
])
def test_which_form_runs(libhh, n, o, resident):
    assert (_loop_launches(n, **o) < 50) == resident


# n, k, bc, options: resident and packed members in turn
MEMBERS = [
    (64, 12.0, (S, S, S, S), {}),
    (96, 20.0, (D, S, S, D), SEP),
    (320, 9.0, (S, S, D, S), {}),
    (128, 9.0, (S, S, D, S), {}),
    (40, 6.0, (S, D, S, S), SEP),
    (264, 11.0, (S, S, S, S), {}),
    (72, 15.0, (S, S, S, S), {}),
]


def _source(i):
    rng = np.random.default_rng(300 + i)
    return inputs.gaussian_source(2, MEMBERS[i][0], tuple(rng.uniform(0.2, 0.8, 2)), 0.05, complex(1.0, 0.3))


@pytest.fixture(scope="module")
def lone(libhh):
    out = []
    for i, (n, k, bc, o) in enumerate(MEMBERS):
        with hh.Problem(2, n, k, 0.0, k, bc, hh.default_options(**o)) as p:
            out.append(p.solve_host(_source(i), TOL, nodal=True))
    return out


@pytest.mark.parametrize("members", [[1, 4], [1, 2, 4, 5], list(range(7))], ids=["small", "packed", "mixed"])
@pytest.mark.parametrize("capacity", [2, 7])
def test_pack_equals_lone_solves(libhh, lone, members, capacity):
    queue, slot_of, got, probs = list(members), {}, {}, {}
    with hh.Pack(capacity=capacity) as pk:
        while queue or slot_of:
            while queue and pk.members() < capacity:
                i = queue.pop(0)
                n, k, bc, o = MEMBERS[i]
                probs[i] = hh.Problem(2, n, k, 0.0, k, bc, hh.default_options(**o))
                slot_of[pk.add(probs[i], _source(i), TOL, nodal=True)] = i
            for s in pk.run():
                i = slot_of.pop(s)
                got[i] = pk.take(s)
                probs.pop(i).close()
    assert sorted(got) == members
    for i, (u, info) in got.items():
        ul, il = lone[i]
        assert np.array_equal(u, ul), i
        assert info.outer_its == il.outer_its and info.rel_residual == il.rel_residual <= TOL, i


@pytest.mark.parametrize("n,nb,prec", [(128, 1, hh.HH_C64), (128, 1, hh.HH_C128), (64, 4, hh.HH_C64), (320, 1, hh.HH_C64)])
def test_tuned_and_replayed_equal_plain(libhh, n, nb, prec):
    ks = [10.0 + 5 * b for b in range(nb)] if nb > 1 else 20.0
    g = torch.Generator(device="cuda").manual_seed(n)
    out = []
    for graphs, tune in ((1, False), (0, False), (1, True), (0, True)):
        o = hh.default_options(levels=3, precision=prec, restart=2, use_graphs=graphs, **SEP)
        with hh.Problem(2, n, ks, 0.0, ks, (D, S, S, S), o) as p:
            if tune:
                assert p.autotune()
            r = torch.randn(p.size(), dtype=torch.complex128, device="cuda", generator=g.manual_seed(n))
            out += [p.precondition(r), p.precondition(r)]
    assert all(torch.equal(z, out[0]) for z in out[1:])
