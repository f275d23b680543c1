"""The mixed form's packed pair pass with the options that the default form
leaves out: the literal F_sn, the collision model and both, against the CPU
FP64 oracle, on a vessel whose lists have odd and even lengths."""
import numpy as np
import pytest

import oracle
from paper_2405_03980_gb300 import _binding as B
from paper_2405_03980_gb300 import synth
from paper_2405_03980_gb300.sim import Simulation

pytestmark = pytest.mark.gpu

LITERAL = B.SPH_SN_LITERAL
L2_TOL = 2e-5   # relative L2 of the FP32 fields, the bound the mixed form is held to


@pytest.mark.parametrize("extra", [LITERAL, B.SPH_COLLISION, LITERAL | B.SPH_COLLISION])
def test_options_in_the_packed_pair_pass(extra):
    c = synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9)
    flags = B.SPH_FLAGS_DEFAULT | extra
    c.params = dict(c.params, col_dist=0.9, col_e=0.4, flags=flags)
    sim = Simulation(c, precision=B.SPH_MIXED)
    o = oracle.Sim(c.params, c.pos, c.vel, c.spin, c.species, flags=flags)
    fl = c.species < 2
    st = sim.state_arrays()
    for f, ref in (("acc", o.acc), ("dspin", o.dspin)):
        e = np.linalg.norm(st[f][fl] - ref[fl]) / np.linalg.norm(ref[fl])
        assert e <= L2_TOL, (f, e)
    sim.close()
