"""The optional pair terms by themselves, in both forms against the CPU FP64
oracle: the literal F_sn, the collision model and the two together, with every
other term off, so that nothing else hides them.  The vessel's lists have odd
and even lengths, and pairs with the wall are among those that collide."""
import numpy as np
import pytest

import oracle
from paper_2405_03980_gb300 import _binding as B
from paper_2405_03980_gb300 import synth
from paper_2405_03980_gb300.sim import Simulation

pytestmark = pytest.mark.gpu

LITERAL = B.SPH_TERM_SN | B.SPH_SN_LITERAL


def vessel():
    """A jittered vessel with velocity noise, and a collision distance in the
    widest gap of its pair distances between 0.96 and 1.0, so that FP32
    positions decide every pair as FP64 ones do."""
    c = synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9, jitter=0.12, vel_noise=0.2)
    c.spin += np.random.default_rng(3).normal(0.0, 0.2, c.spin.shape) * (c.species < 2)[:, None]
    d = c.pos[:, None] - c.pos[None]
    d[..., 2] -= 11.0 * np.round(d[..., 2] / 11.0)
    r = np.sqrt((d * d).sum(-1))
    near = np.unique(r[(r > 0.96) & (r < 1.0)])
    k = int(np.argmax(np.diff(near)))
    assert near[k + 1] - near[k] > 2e-5
    c.params = dict(c.params, C_l=0.5, col_dist=float(near[k] + near[k + 1]) / 2, col_e=0.4)
    hit = (r > 0) & (r < c.params["col_dist"])
    assert hit[c.species < 2].sum() > 1000 and hit[c.species < 2][:, c.species == 2].sum() > 20
    return c


@pytest.mark.parametrize("flags", [LITERAL, B.SPH_COLLISION, LITERAL | B.SPH_COLLISION])
@pytest.mark.parametrize("precision,tol", [(B.SPH_FP64, 1e-12), (B.SPH_MIXED, 2e-5)])
def test_optional_terms_alone(flags, precision, tol):
    """acc within the form's bound (relative L2; the mixed form's 2e-5, FP64's
    1e-12); no torque; and the wall torque that the options exert."""
    c = vessel()
    o = oracle.Sim(c.params, c.pos, c.vel, c.spin, c.species, flags=flags)
    fl = c.species < 2
    lengths = np.diff(oracle.neighbors(oracle.make_params(c.params), c.pos)[0])[fl]
    assert (lengths % 2 == 1).any() and (lengths % 2 == 0).any() and np.linalg.norm(o.acc[fl]) > 1
    sim = Simulation(c, precision=precision, flags=flags)
    st = sim.state_arrays()
    e = np.linalg.norm(st["acc"][fl] - o.acc[fl]) / np.linalg.norm(o.acc[fl])
    print(flags, precision, e)
    assert e <= tol
    assert not st["dspin"].any() and not o.dspin.any()
    tw, ow = np.array(sim.diagnostics()["T_wall"]), np.array(o.diagnostics()["T_wall"])
    assert np.abs(ow).max() > 1e-3
    assert np.abs(tw - ow).max() <= 100 * tol * np.abs(ow).max()
    sim.close()
