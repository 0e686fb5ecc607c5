"""The autotuner on a stream that cannot be captured: the legacy default stream
(handle 1).  Steps are graph replays there only where they have to be; a
profiled step launches kernel by kernel and needs no capture, and neither may
the choice of the schedule before it."""
import numpy as np
import pytest

import paper_2408_16509_gb300 as fr
from frinputs import box_hex, ics, mixed_box
from frtest import lib_state

pytestmark = pytest.mark.gpu
LEGACY_STREAM = 1


@pytest.mark.parametrize("mesh", ["hex", "mixed"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_profiled_step_on_the_legacy_stream(mesh, precision):
    fr.build()
    spec = box_hex((3, 2, 2)) if mesh == "hex" else mixed_box(4)
    bcs = {} if mesh == "hex" else {t: ("extrap",) for t in range(4)}

    def handle():
        g = fr.FRMesh(spec, 2, physics="ns", mu=0.01, prandtl=0.71, precision=precision, bcs=bcs)
        g.set_solution(lib_state(g, ics.flow3d))
        return g
    g = handle()
    g.set_stream(LEGACY_STREAM)
    prof = g.profile_step("rk4", 1e-4)
    assert prof["volume"][1] == 4 * len(g.types)
    got = g.get_solution()
    g.set_stream(None)
    g.rk_step("rk4", 1e-4, 1)
    # the same step on the handle's own stream, with the schedule tuned there
    h = handle()
    h.rk_step("rk4", 1e-4, 1)
    ref = h.get_solution()
    tol = 1e-12 if precision == "fp64" else 1e-5
    for t in ref:
        assert np.abs(got[t] - ref[t]).max() < tol * np.abs(ref[t]).max()
