"""The vertex-metric family of hexahedra (FP32 values) at every order, against the
FP64 oracle: at p = 1 an element has fewer threads (8) than vertex coordinates
(24).  Tolerance as in test_gpu_parity: FP32 solutions 1e-6 per variable."""
import pytest

import paper_2408_16509_gb300 as fr
from frinputs import box_hex, ics
from frtest import lib_state, oracle_state, rel_l2
from oracle import rk
from oracle.fr import FRSystem
from oracle.mesh import FRMesh as OracleMesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("physics", ["euler", "ns"])
@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("variant", ["sumfact_vertex", "sumfact"])
def test_steps_at_every_order(p, physics, precision, variant):
    fr.build()
    spec = box_hex((4, 3, 5), perturb=0.1)
    o = OracleMesh(spec.as_dict(), p)
    osys = FRSystem(o, physics, gamma=1.4, mu=0.02, pr=0.71)
    g = fr.FRMesh(spec, p, physics=physics, mu=0.02, prandtl=0.71, precision=precision)
    g.set_variant(variant)
    g.set_solution(lib_state(g, ics.flow3d))
    u = oracle_state(o, ics.flow3d)
    for _ in range(2):
        u = rk.step(osys.rhs, u, 1e-3, "rk45")
    g.rk_step("rk45", 1e-3, 2)
    assert rel_l2(g.get_solution(), u).max() < 1e-6
