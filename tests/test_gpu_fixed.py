"""The FP64 hexahedron kernels whose line operators are fixed-point sums
(csrc/fr_hexfx.cuh) against the FP64 oracle, where their fields can go wrong:
large ranges within an element, fields that vanish, extreme scales, NaN.

Tolerances: the parity bounds of FP64 right-hand sides (1e-12 per variable,
5e-12 at p = 4, see test_gpu_parity.py) hold for the oracle's own rounding; a
fixed-point field resolves 2^-59 of its largest value in the element, so a
spread of 2^8 within an element leaves it below FP64 rounding (2^-53).  Scaling
a state by a power of two shifts the fields' exponents only: the result is the
same bit for bit.
"""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
from frinputs import box_hex
from frtest import rel_l2_rhs
from oracle.elements import Hex
from oracle.fr import FRSystem
from oracle.mesh import FRMesh as OracleMesh

pytestmark = pytest.mark.gpu

N = (3, 2, 5)  # 30 elements: a ragged last CTA for every tile above 1 but 2, 3


@pytest.fixture(scope="module", autouse=True)
def built():
    fr.build()


def _rough(p, seed, family="gl", slope=0.32):
    """Density and pressure linear in each element's reference coordinates
    (a range of 49 within an element at slope 0.32), constant random velocity
    per element, a little noise per point: jumps of order one at every face,
    and admissible traces (linear fields are interpolated exactly, where a
    random value per point extrapolates to negative densities)."""
    rng = np.random.default_rng(seed)
    el = Hex(p, family)
    ne = N[0] * N[1] * N[2]

    def field():
        c = np.exp(rng.uniform(-1.0, 1.0, (ne, 1)))
        s = rng.choice([-1.0, 1.0], (ne, 3)) * slope
        noise = rng.uniform(-1e-3, 1e-3, (ne, el.nupts))
        return c * (1.0 + s @ el.upts.T + noise)
    rho, pr = field(), field()
    v = rng.normal(size=(ne, 1, 3))
    u = np.empty((ne, el.nupts, 5))
    u[..., 0] = rho
    u[..., 1:4] = rho[..., None] * v
    u[..., 4] = pr / 0.4 + 0.5 * rho * (v ** 2).sum(-1)
    return u


def _handle(p, physics, family="gl", **kw):
    return fr.FRMesh(box_hex(N, perturb=0.1), p, physics=physics, mu=0.02, prandtl=0.71,
                     family=family, **kw)


def _oracle(p, physics, family="gl", **kw):
    m = OracleMesh(box_hex(N, perturb=0.1).as_dict(), p, family=family)
    return FRSystem(m, physics, mu=0.02, pr=0.71, **kw)


@pytest.mark.parametrize("p", [2, 3, 4])
@pytest.mark.parametrize("physics", ["euler", "ns"])
@pytest.mark.parametrize("family", ["gl", "gll"])
def test_rough_state(p, physics, family):
    g = _handle(p, physics, family)
    u = _rough(p, seed=p, family=family)
    g.set_solution({"hex": u})
    err = rel_l2_rhs(g.rhs(), _oracle(p, physics, family).rhs({"hex": u}))
    assert err.max() < (5e-12 if p == 4 else 1e-12), err


@pytest.mark.parametrize("p", [2, 4])
def test_fields_that_vanish(p):
    # gas at rest: zero mass flux and momentum, one variable's fields all zero
    g = _handle(p, "ns")
    u = _rough(p, seed=7, slope=0.2)
    u[..., 4] -= 0.5 * (u[..., 1:4] ** 2).sum(-1) / u[..., 0]
    u[..., 1:4] = 0.0
    g.set_solution({"hex": u})
    err = rel_l2_rhs(g.rhs(), _oracle(p, "ns").rhs({"hex": u}))
    assert err.max() < 5e-12, err


@pytest.mark.parametrize("p", [2, 3, 4])
@pytest.mark.parametrize("shift", [-400, 400])
def test_power_of_two_scaling_is_exact(p, shift):
    # Euler fluxes are homogeneous of degree one in the conserved state
    g = _handle(p, "euler")
    u = _rough(p, seed=3)
    g.set_solution({"hex": u})
    a = g.rhs()["hex"]
    g.set_solution({"hex": np.ldexp(u, shift)})
    b = g.rhs()["hex"]
    assert np.array_equal(np.ldexp(a, shift), b)


@pytest.mark.parametrize("p", [2, 3, 4])
def test_tiles_and_rk_registers(p):
    # every tile gives the same bits, also through the RK epilogue and u_f
    g = _handle(p, "ns")
    g.set_variant("sumfact")
    u = _rough(p, seed=5, slope=0.1)
    out = []
    for tile in (0, 1, 2):
        g.set_schedule({"hex": (tile, tile)})
        g.set_solution({"hex": u})
        g.rk_step("rk45", 1e-5, 2)
        out.append(g.get_solution()["hex"])
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


@pytest.mark.parametrize("p", [2, 3, 4])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_state_is_reported(p, bad):
    g = _handle(p, "ns")
    u = _rough(p, seed=9)
    g.set_solution({"hex": u})
    ok = g.rhs()["hex"]
    u2 = u.copy()
    u2[11, 4, 4] = bad
    g.set_solution({"hex": u2})
    with pytest.raises(fr.FRError) as e:
        g.rhs()
    assert e.value.name == "FR_ENONFINITE"
    g.set_solution({"hex": u})
    assert np.array_equal(g.rhs()["hex"], ok)


def test_antialiased_flux():
    g = _handle(3, "ns")
    g.set_antialias(9)
    u = _rough(3, seed=13, slope=0.2)
    g.set_solution({"hex": u})
    err = rel_l2_rhs(g.rhs(), _oracle(3, "ns", antialias=9).rhs({"hex": u}))
    assert err.max() < 1e-12, err
