"""The phases of a stage over different element ranges: the gradient phase in
two parts and the flux phase in one, or the other way round, are the same
kernels on the same elements as whole phases, so the states agree bit for bit."""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
from frinputs import box_hex, ics, mixed_box
from frtest import lib_state
from paper_2408_16509_gb300 import partition

pytestmark = pytest.mark.gpu

FAR = ("state", 1.0, 0.4, 0.1, 0.0, 1.0 / 1.4 / 0.09)
BCS = {0: FAR, 1: ("extrap",), 2: FAR, 3: ("extrap",)}
SPECS = {"hex": lambda: box_hex((5, 4, 3), perturb=0.1),
         "mixed": lambda: mixed_box(n=4, x_pri=0.34, x_tet=0.67, perturb=0.05)}


def _run(case, prec, order, parts):
    """One step of a two-part mesh, both parts in this process; parts: the
    ranges that phase 1 and phase 2 are launched in."""
    import torch
    subs, _, _ = partition.split(SPECS[case](), 2, "weighted", halo_last=True)
    gs = [fr.FRMesh(s, order, physics="ns", mu=0.02, prandtl=0.71,
                    bcs=partition.exchange_bcs(BCS), precision=prec) for s in subs]
    faces = [g.exchange_faces() for g in gs]
    nv = {0: 5, 1: 15 if prec == "fp64" else 5}
    dt = torch.float64 if prec == "fp64" else torch.float32
    for r, g in enumerate(gs):
        g.set_variant("sumfact")
        g.set_solution(lib_state(g, ics.flow3d))
    n = [int(g.exchange_setup(r, faces).sum()) for r, g in enumerate(gs)]
    assert n[0] == n[1] > 0
    for st in range(4):
        for phase, what in ((1, 0), (2, 1)):
            bufs = [torch.zeros((n[0], nv[what]), dtype=dt, device="cuda") for _ in gs]
            torch.cuda.synchronize()  # the handles have streams of their own
            for g, b in zip(gs, bufs):
                g.exchange_pack(what, b)
                g.sync()
            for r, g in enumerate(gs):
                g.exchange_unpack(what, bufs[1 - r])
                for p in parts[phase - 1]:
                    g.rk_stage("rk4", 2e-4, st, phase, p)
                g.sync()
    return [g.get_solution() for g in gs]


@pytest.mark.parametrize("case,prec,order", [("hex", "fp64", 2), ("hex", "fp64", 3),
                                             ("hex", "fp32", 2), ("hex", "mixed", 3),
                                             ("mixed", "fp64", 2), ("mixed", "fp32", 3)])
def test_phases_over_different_parts_are_bitwise_equal(case, prec, order):
    whole = _run(case, prec, order, ((0,), (0,)))
    for parts in (((1, 2), (0,)), ((0,), (1, 2))):
        got = _run(case, prec, order, parts)
        for a, b in zip(whole, got):
            for t in a:
                assert np.array_equal(a[t], b[t])
