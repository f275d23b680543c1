"""Edges of the FP64 form's fixed-point neighbour passes, per particle against
the oracle or an evaluation in extended precision."""
import numpy as np
import pytest

import oracle
from paper_2405_03980_gb300 import synth
from test_gpu_fp64 import _cuda, per_particle_check, sim_of  # noqa: F401

pytestmark = pytest.mark.gpu


def box_of(pos, species, half, seed=1, sigma=0.2, **kw):
    """Fluid particles in a box of the given half widths in x and y and height
    8 (periodic), with random velocities and spins."""
    rng = np.random.default_rng(seed)
    prm = synth.workload_params(4.0, 8, 0.1)
    prm.update(box_lo=(-half[0], -half[1], 0.0), box_hi=(half[0], half[1], 8.0), C_T=0.5, C_l=0.3)
    prm.update(kw)
    n = len(species)
    return synth.Cylinder(R=4.0, H=8, dx=1.0, Omega=0.1, f_v=0.5, seed=seed,
                          pos=np.ascontiguousarray(pos, dtype=np.float64),
                          vel=rng.normal(0.0, sigma, (n, 3)), spin=rng.normal(0.0, sigma, (n, 3)),
                          species=np.asarray(species, dtype=np.uint8), params=prm)


def neighbours_equal(sim, c):
    off, nbr = sim.neighbors()
    off_o, nbr_o = oracle.neighbors(oracle.make_params(c.params), c.pos)
    return np.array_equal(off, off_o) and np.array_equal(nbr, nbr_o)


@pytest.mark.parametrize("m,cap", [(60, 64), (100, 104), (150, 152)])
def test_prefiltered_lists_past_the_capacity(m, cap):
    """Two flat clusters a little more than 2h apart on a long axis, where the
    FP32 prefilter passes every pair between them: each particle has 2m - 1
    prefiltered neighbours (119, within the staging of 168; 199 and 299, past
    it), more than its list holds, of which m - 1 are neighbours and fit."""
    rng = np.random.default_rng(m)
    g = np.stack(np.meshgrid(np.arange(13), np.arange(13), indexing="ij"), -1).reshape(-1, 2)[:m]
    one = np.zeros((m, 3))
    one[:, 1:] = (g - 6) * 0.02 + [0.0, 4.0]
    pos = np.concatenate([one, one + [2.602, 0.0, 0.0]])
    pos += rng.uniform(-5e-4, 5e-4, pos.shape)
    c = box_of(pos, rng.integers(0, 2, 2 * m), (5.5e4, 8.0))
    r = np.linalg.norm(pos[:m, None] - pos[None, m:], axis=2)
    assert 2.6 < r.min() and r.max() < 2.64
    sim = sim_of(c, nbr_cap=cap)
    print(per_particle_check(sim.state_arrays(), c, 0))
    assert neighbours_equal(sim, c)
    sim.close()
