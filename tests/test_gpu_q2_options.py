"""FP64 quadrilaterals under the run options that move the departure time or its formula, on the maps whose metrics vary from node to
node: the derivative passes take the metrics of the arrival time, whatever map the propagation evaluated."""
import pytest

import oracle as O
from paper_2002_04353_gb300 import inputs as I
from test_gpu_q2 import CASES, _check64, _eq_state, _pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, O.FLAG_MIDPOINT, O.FLAG_LITERAL_VG, O.FLAG_MIDPOINT | O.FLAG_LITERAL_VG],
                         ids=["plain", "midpoint", "literal_vg", "both"])
@pytest.mark.parametrize("name", ["box_sine", "omesh_blended"])
def test_run_options_on_deforming_maps(name, flags):
    mesh, motion = CASES[name]()
    flow = I.flow_params(0.1, T_inf=0.3, Re=500.0, chord=200.0)
    flow.flags = flags
    o, s = _pair(mesh, motion, flow, state=_eq_state(mesh, flow, 0.01, 5))
    for k in range(2):
        o.step(3)
        s.lb_step(3)
        _check64(o, s, f"{name} flags {flags} after {3 * (k + 1)} steps")
