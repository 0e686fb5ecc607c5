"""States far from one: Euler fluxes are homogeneous of degree one in the
conserved state, so a state scaled by a power of two gives a right-hand side
scaled by it bit for bit, as long as values, fluxes and their products with the
metric are normal numbers.  A scale of 2^66 in FP32 (2^600 in FP64) leaves the
squares of the momenta outside the type's range, and the state and its fluxes
well inside.
"""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
from frinputs import box_hex, ics, mixed_box
from frtest import lib_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    fr.build()


@pytest.mark.parametrize("mesh,variant", [("hex", "sumfact"), ("hex", "dense"),
                                          ("mixed", "sumfact"), ("mixed", "dense")])
@pytest.mark.parametrize("precision,shift", [("fp32", 66), ("fp32", -66),
                                             ("fp64", 600), ("fp64", -600)])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_power_of_two_scaling_is_exact(mesh, variant, precision, shift, p):
    if mesh == "hex":
        g = fr.FRMesh(box_hex((3, 2, 2), perturb=0.1), p, physics="euler", precision=precision)
    else:
        g = fr.FRMesh(mixed_box(6), p, physics="euler", precision=precision,
                      bcs={t: ("extrap",) for t in range(4)})
    g.set_variant(variant)
    typ = np.float32 if precision == "fp32" else np.float64
    u = {t: v.astype(typ).astype(np.float64) for t, v in lib_state(g, ics.flow3d).items()}
    g.set_solution(u)
    a = g.rhs()
    g.set_solution({t: np.ldexp(v, shift) for t, v in u.items()})
    b = g.rhs()
    for t in a:
        assert np.abs(a[t]).max() > 0
        assert np.array_equal(np.ldexp(a[t], shift), b[t])
