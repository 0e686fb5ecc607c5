"""Which side of an interface a flux point is on, where it matters (LDG, beta not
zero): the gradient kernels take the solution's jump from both traces and
decide the side by comparing the flux points' numbers.  Kernels and meshes that
test_gpu_ldg.py does not run; tolerances as there (FP64 right-hand sides 1e-12,
FP32 solutions 1e-6)."""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
import test_gpu_phase_parts as phases
from frinputs import box_hex, ics, mixed_box
from frtest import lib_state, oracle_state, rel_l2, rel_l2_rhs
from oracle import rk
from oracle.fr import FRSystem
from oracle.mesh import FRMesh as OracleMesh

pytestmark = pytest.mark.gpu
LDG = (0.5, 0.1)


@pytest.fixture(scope="module", autouse=True)
def built():
    fr.build()


def _pair(spec, p, precision, bcs=None):
    o = OracleMesh(spec.as_dict(), p)
    osys = FRSystem(o, "ns", gamma=1.4, mu=0.02, pr=0.71, bcs=bcs, ldg=LDG)
    g = fr.FRMesh(spec, p, physics="ns", gamma=1.4, mu=0.02, prandtl=0.71, bcs=bcs,
                  precision=precision)
    g.set_viscous_scheme(*LDG)
    g.set_variant("sumfact")
    g.set_solution(lib_state(g, ics.flow3d))
    return osys, g, oracle_state(o, ics.flow3d)


@pytest.mark.parametrize("p", [1, 2, 3])
def test_fp32_prisms_and_tetrahedra(p):
    osys, g, u = _pair(mixed_box(n=3, x_pri=0.34, x_tet=0.67, perturb=0.05), p, "fp32",
                       phases.BCS)
    for _ in range(2):
        u = rk.step(osys.rhs, u, 1e-3, "rk45")
    g.rk_step("rk45", 1e-3, 2)
    assert rel_l2(g.get_solution(), u).max() < 1e-6


@pytest.mark.parametrize("n", [(3, 1, 2), (1, 1, 3), (2, 2, 1)])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_elements_that_are_their_own_neighbour(n, p):
    # one cell along a periodic direction: both sides of its faces are one element
    spec = box_hex(n, perturb=0.0)
    osys, g, u = _pair(spec, p, "fp64")
    assert rel_l2_rhs(g.rhs(), osys.rhs(u)).max() < 1e-12
    osys, g, u = _pair(spec, p, "fp32")
    u = rk.step(osys.rhs, u, 1e-4, "rk45")
    g.rk_step("rk45", 1e-4, 1)
    assert rel_l2(g.get_solution(), u).max() < 1e-6


@pytest.mark.parametrize("case,prec,order", [("hex", "fp64", 2), ("hex", "fp64", 3),
                                             ("hex", "fp32", 2), ("mixed", "fp64", 2),
                                             ("mixed", "fp32", 3)])
def test_element_ranges(case, prec, order, monkeypatch):
    # a range of elements counts its flux points from the whole mesh's start
    make = fr.FRMesh

    def biased(*a, **kw):
        g = make(*a, **kw)
        g.set_viscous_scheme(*LDG)
        return g
    monkeypatch.setattr(phases.fr, "FRMesh", biased)
    whole = phases._run(case, prec, order, ((0,), (0,)))
    got = phases._run(case, prec, order, ((1, 2), (0,)))
    for a, b in zip(whole, got):
        for t in a:
            assert np.array_equal(a[t], b[t])
