"""The FP64 form's fixed-point neighbour passes where they leave their common
route: pairs nearer than fixed point resolves, more neighbours than its sums
hold, a box in which the FP32 prefilter is too wide, velocities whose sizes
differ by many orders.  Each state is compared with the oracle per particle,
to 1e-12 of the particle's absolute pair sums (the FP64 form's bar)."""
import numpy as np
import pytest

import oracle
from paper_2405_03980_gb300 import synth
from test_gpu_fp64 import _cuda, per_particle_check, sim_of  # noqa: F401

pytestmark = pytest.mark.gpu


def vessel(pos, vel, spin, species, box, nz=8.0, **kw):
    prm = synth.workload_params(4.0, int(nz), 0.1)
    prm.update(box_lo=(-box[0], -box[1], 0.0), box_hi=(box[0], box[1], nz), C_T=0.5, C_l=0.3, **kw)
    return synth.Cylinder(R=4.0, H=int(nz), dx=1.0, Omega=0.1, f_v=0.4, seed=4, pos=pos, vel=vel,
                          spin=spin, species=species, params=prm)


def state(kind):
    pos, vel, spin, sp = synth.periodic_block(8, 8, 8, seed=3, f_v=0.5, vel_sigma=0.2)
    pos = pos - [4.0, 4.0, 0.0]
    rng = np.random.default_rng(5)
    box, kw = (8.0, 8.0), {}
    if kind == "near":  # pairs from 0.3 dx down to coincidence, some across the period
        for k, r in enumerate((0.3, 0.2, 0.05, 0.02, 1e-3, 1e-6, 1e-12, 0.0) * 4):
            e = rng.normal(size=3)
            pos[2 * k + 1] = pos[2 * k] + r * e / np.linalg.norm(e)
        pos[100, 2] = 1e-9
        pos[101] = pos[100] + [0.01, 0.0, 8.0 - 2e-9]
        pos[:, 2] %= 8.0
    elif kind == "long lists":  # more than 160 neighbours
        pos[:300] = rng.uniform(-1.6, 1.6, size=(300, 3)) + [0.0, 0.0, 4.0]
        kw["nbr_cap"] = 512
    elif kind == "wide box":
        box = (1.0e5, 8.0)
    elif kind == "fast particles":
        vel *= 1e-4
        vel[::97] = rng.normal(size=vel[::97].shape) * 1e6
        spin[::83] *= 1e5
    elif kind == "slow particles":
        vel *= 1e-44
        spin *= 1e-60
    elif kind == "at rest":
        vel[:], spin[:] = 0.0, 0.0
    return vessel(pos, vel, spin, sp, box, **kw)


@pytest.mark.parametrize("kind", ["near", "long lists", "wide box", "fast particles",
                                  "slow particles", "at rest"])
def test_states_off_the_common_route(kind):
    c = state(kind)
    sim = sim_of(c)
    st = sim.state_arrays()
    p = oracle.make_params(c.params)
    if kind == "at rest":  # no spin torque at all
        assert not st["dspin"].any()
        rho, P = oracle.density(p, c.pos, c.species)
        acc, _, _, sc = oracle.forces(p, c.pos, c.vel, c.spin, c.species, rho, P, scale=True)
        assert (np.linalg.norm(st["acc"] - acc, axis=1) <= 1e-12 * sc[:, 0]).all()
    else:
        print(kind, per_particle_check(st, c, 0))
    off, nbr = sim.neighbors()
    off_o, nbr_o = oracle.neighbors(p, st["pos"])
    assert np.array_equal(off, off_o) and np.array_equal(nbr, nbr_o)
    sim.close()


def test_wall_torque_and_options_share_the_lists():
    """Lists hold inviscid, viscous and wall neighbours in that order; the
    optional terms' FP64 loops read the same lists: with a collision distance
    below every pair distance they must give the fixed-point pass's forces and
    wall torque (both within 1e-12 of the oracle's)."""
    from paper_2405_03980_gb300 import _binding as B
    c = synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9)
    d = synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9)
    d.params = dict(d.params, col_dist=1e-3, flags=B.SPH_FLAGS_DEFAULT | B.SPH_COLLISION)
    a, b = sim_of(c), sim_of(d)
    a.step(2)
    b.step(2)
    sa, sb, da, db = a.state_arrays(), b.state_arrays(), a.diagnostics(), b.diagnostics()
    for k in sa:
        assert np.abs(sa[k] - sb[k]).max() <= 2e-12 * np.abs(sb[k]).max(), k
    tw = np.abs(db["T_wall"]).max()
    assert np.abs(np.subtract(da["T_wall"], db["T_wall"])).max() <= 1e-11 * tw
    a.close()
    b.close()


@pytest.mark.parametrize("partner", [(21.0, 40), (36.0, 70)])
def test_lane_counts_give_the_same_bits(partner):
    """The lanes that share a list (eight below 2^15 particles in all, four
    below 2^18, then two) and the partition's tiles change no bit: a small
    vessel alone and batched with one that takes the batch past each bound."""
    a = synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9)
    b = synth.cylinder(*partner, Omega=0.1, f_v=0.3, seed=10)
    assert a.n < 1 << 15 and (1 << 15 < a.n + b.n < 1 << 18 or a.n + b.n > 1 << 18)
    solo, both = sim_of(a), sim_of([a, b])
    solo.step(2)
    both.step(2)
    x, y = solo.state_arrays(), both.state_arrays()
    for k in x:
        assert np.array_equal(x[k], y[k][:a.n]), k
    dx, dy = solo.diagnostics(), both.diagnostics(0)
    assert dx["T_wall"] == dy["T_wall"] and dx["L_orb"] == dy["L_orb"]
    solo.close()
    both.close()
