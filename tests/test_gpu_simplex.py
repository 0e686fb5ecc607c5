"""The register-blocked FP32 kernels of tetrahedra and prisms
(csrc/fr_simplex.cuh) at every order, against the FP64 oracle and the dense
kernels.

Sizes: 3^3 cells give 18 prisms and 54 tetrahedra (a ragged last group for
most group sizes, fewer groups than SMs: groups of few elements), 12^3 cells
more groups than resident CTAs at p = 3 (the loop over groups).

Tolerances: those of FP32 parity, 2e-5 relative L2 on a right-hand side
against the oracle; after three steps 1e-6 against the dense kernels (both
round each right-hand side, of which a step of 2e-4 adds a small part).
"""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
from frinputs import ics, mixed_box
from frtest import lib_state, oracle_state, rel_l2, rel_l2_rhs
from oracle.fr import FRSystem
from oracle.mesh import FRMesh as OracleMesh

pytestmark = pytest.mark.gpu

FAR = ("state", 1.0, 0.4, 0.1, 0.0, 1.0 / 1.4 / 0.09)
BCS = {0: FAR, 1: ("extrap",), 2: FAR, 3: ("extrap",)}


@pytest.fixture(scope="module", autouse=True)
def built():
    fr.build()


def _mesh(spec, p, physics, variant):
    g = fr.FRMesh(spec, p, physics=physics, mu=0.02, prandtl=0.71, bcs=BCS,
                  precision="fp32")
    g.set_variant(variant)
    g.set_solution(lib_state(g, ics.flow3d))
    return g


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("physics", ["euler", "ns"])
def test_rhs_against_oracle(p, physics):
    spec = mixed_box(n=3, x_pri=0.34, x_tet=0.67, perturb=0.05)
    o = OracleMesh(spec.as_dict(), p)
    osys = FRSystem(o, physics, mu=0.02, pr=0.71, bcs=BCS)
    r = _mesh(spec, p, physics, "sumfact").rhs()
    err = rel_l2_rhs(r, osys.rhs(oracle_state(o, ics.flow3d)))
    assert err.max() < 2e-5, err


@pytest.mark.parametrize("p,n,scheme", [(1, 3, "rk45"), (2, 3, "rk4"), (3, 3, "rk45"),
                                        (4, 3, "rk4"), (3, 12, "rk45"), (2, 12, "rk4")])
def test_steps_and_any_tile(p, n, scheme):
    spec = mixed_box(n=n, x_pri=0.2 if n > 3 else 0.34, x_tet=0.6, perturb=0.05)
    g, h = _mesh(spec, p, "ns", "sumfact"), _mesh(spec, p, "ns", "dense")
    for m in (g, h):
        m.rk_step(scheme, 2e-4, 3)
    assert rel_l2(g.get_solution(), h.get_solution()).max() < 1e-6
    # one CTA per SM instead of as many as fit: the same sums
    t = _mesh(spec, p, "ns", "sumfact")
    t.rhs()
    t.set_schedule(tiles={"pri": (1, 1), "tet": (1, 1)})
    t.rk_step(scheme, 2e-4, 3)
    a, b = g.get_solution(), t.get_solution()
    for k in a:
        assert np.array_equal(a[k], b[k])
