"""Edges of the FP64 form's fixed-point neighbour passes, per particle against
the oracle or an evaluation in extended precision."""
import numpy as np
import pytest

import oracle
from paper_2405_03980_gb300 import _binding as B
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


def exact_sites(c, m):
    """Acceleration and spin change of every particle, and the sums of the
    magnitudes of their pair terms, for consecutive groups of m particles that
    see nothing but each other, in extended precision."""
    L = np.longdouble
    q, p = c.params, oracle.make_params(c.params)
    n = len(c.species)
    h, aD = L(q["h"]), L(oracle.W(p, 0.0))
    mass = np.where(c.species == 0, oracle.mass(p, 0), oracle.mass(p, 1)).astype(L).reshape(-1, m)
    inv = (c.species == 0).reshape(-1, m)
    x, v, w = (a.astype(L).reshape(-1, m, 3) for a in (c.pos, c.vel, c.spin))
    d = x[:, :, None] - x[:, None]
    r = np.sqrt((d * d).sum(-1))
    t = 1 - r / (2 * h)
    t[t < 0] = 0
    self_ = np.eye(m, dtype=bool)[None]
    W = aD * t**4 * (5 - 4 * t)
    rho = (W * mass[:, None]).sum(-1)
    P = L(q["p0"]) * (rho / L(q["rho0"])) ** int(q["alpha_P"]) - L(q["beta_P"])
    V, Pr = mass / rho, P / rho**2
    F = 5 * aD / h**2 * t**3 * ~self_
    W = W * ~self_
    VV = V[:, :, None] * V[:, None]
    u = v[:, :, None] - v[:, None]
    dv = (d * u).sum(-1)
    s = (w[:, :, None] + w[:, None]) / 2
    u = u + np.cross(d, s)
    unlike = inv[:, :, None] != inv[:, None]
    vv = ~inv[:, :, None] & ~inv[:, None]
    A, Bv = 10 * (L(q["eta_bar"]) - L(0.6) * L(q["eta_r"])), 4 * L(q["eta_r"])
    r2 = np.where(self_, 1, r * r)
    along = (mass[:, :, None] * mass[:, None] * (Pr[:, :, None] + Pr[:, None]) * F
             + vv * (Bv - A) * VV * F * dv / r2)
    bu = np.where(unlike, -L(q["C_l"]) * VV * W, -(vv * Bv * VV * F))
    aT = unlike * L(q["C_T"]) * VV * F
    rot = bu[..., None] * u
    f = along[..., None] * d + rot + aT[..., None] * d * np.array([1, 1, 0])
    tau = -np.cross(d, rot) / 2
    I = L(q["inertia_coef"]) * mass * L(q["dx"]) ** 2
    out = []
    for g, k in ((f, mass), (tau, I)):
        out += [(g.sum(2) / k[..., None]).reshape(n, 3), (np.linalg.norm(g.astype(float), axis=-1).sum(2) / k.astype(float)).reshape(n)]
    return out


def sites(kind, t, seed):
    """Groups of particles 9 apart.  "pairs": two particles of any species at
    r = 2h (1 - t).  "one unlike": an inviscid particle among seven others and
    one viscous particle at that distance, on which alone its torque hangs."""
    rng = np.random.default_rng(seed)
    S = len(t)
    e = rng.normal(size=(S, 8, 3))
    e /= np.linalg.norm(e, axis=-1, keepdims=True)
    far = 2.6 * (1 - t)[:, None] * e[:, 0]
    if kind == "pairs":
        off, sp = np.stack([np.zeros((S, 3)), far], 1), rng.integers(0, 2, (S, 2))
    else:
        off = np.concatenate([np.zeros((S, 1, 3)), rng.uniform(0.9, 1.6, (S, 7, 1)) * e[:, 1:],
                              far[:, None]], 1)
        sp = np.zeros((S, 9), dtype=int)
        sp[:, 8] = 1
    k = int(np.ceil(np.sqrt(S)))
    at = np.stack([np.arange(S) % k - k / 2, np.arange(S) // k - k / 2, np.zeros(S)], 1) * 9.0
    off = off + at[:, None] + [0.0, 0.0, 4.0]
    return off.reshape(-1, 3), sp.ravel(), off.shape[1], (9.0 * k / 2 + 9.0,) * 2


@pytest.mark.parametrize("kind", ["pairs", "one unlike"])
def test_sums_that_hang_on_pairs_near_the_cutoff(kind):
    """Force and torque relative to their own pair terms, whatever t.  The
    fixed-point r is within 2^-58.6 of 2h (positions to a unit of 2^-62 each,
    r^2 to three of 2^-60), which t^4 turns into 2^-56.6 / t; the coefficients
    (density, Tait power, volumes) are FP64 operations, some forty of 2^-53."""
    t = 10.0 ** np.random.default_rng(2).uniform(-6.0, -0.3, 900)
    pos, sp, m, half = sites(kind, t, 4)
    c = box_of(pos, sp, half)
    sim = sim_of(c)
    st = sim.state_arrays()
    acc, sa, dsp, sd = exact_sites(c, m)
    for f, ref, s in (("acc", acc, sa), ("dspin", dsp, sd)):
        e = np.linalg.norm((st[f] - ref).astype(float), axis=1)
        assert np.array_equal(e[s == 0], np.zeros((s == 0).sum()))
        tt = np.repeat(t, m)
        rows = s > 0
        if kind == "one unlike":
            rows &= np.arange(len(s)) % m == 0   # the particle in the middle
            tt = tt if f == "dspin" else np.full(len(s), 0.3)
        bound = 5e-15 + 2.0**-56 / tt
        worst = (e[rows] / s[rows] / bound[rows]).max()
        print(kind, f, "largest error over its bound", worst)
        assert rows.sum() > 200 and worst <= 1.0
    sim.close()


def test_lists_of_a_thousand_neighbours():
    """The sums hold every list that the capacity admits."""
    rng = np.random.default_rng(11)
    e = rng.normal(size=(1000, 3))
    pos = 1.25 * e / np.linalg.norm(e, axis=1)[:, None] * rng.uniform(0, 1, (1000, 1)) ** (1 / 3)
    c = box_of(pos + [0.0, 0.0, 4.0], rng.integers(0, 2, 1000), (8.0, 8.0))
    sim = sim_of(c, nbr_cap=1024)
    print(per_particle_check(sim.state_arrays(), c, 0))
    assert neighbours_equal(sim, c)
    sim.close()


@pytest.mark.parametrize("ratio", [1e-7, 1e-3, 0.2, 6.0, 1e4])
@pytest.mark.parametrize("kind", ["pairs", "one unlike"])
def test_species_of_different_mass(kind, ratio):
    """Densities, forces and torques where the species' masses differ: a light
    particle's density can hang on the W shape of one heavy neighbour, volumes
    and pressures differ by the ratio and its square.  Where FP64 operations
    form the shapes, r to 1.5 of 2^-53 gives W 6 / t and two more of the
    products, the density enters V and P / rho^2 of both partners: 24 / t in
    all (2^-48 / t allows 32), t the smallest of the group; the coefficients'
    forty operations beside it."""
    t = 10.0 ** np.random.default_rng(2).uniform(-3.0, -0.3, 900)
    pos, sp, m, half = sites(kind, t, 4)
    x = pos.reshape(-1, m, 3)
    near = 1 - np.linalg.norm(x[:, :, None] - x[:, None], axis=-1) / 2.6
    t = np.repeat(np.where(near > 0, near, 1.0).min((1, 2)), m)
    c = box_of(pos, sp, half, mass_ratio=ratio)
    sim = sim_of(c)
    st = sim.state_arrays()
    acc, sa, dsp, sd = exact_sites(c, m)
    for f, ref, s in (("acc", acc, sa), ("dspin", dsp, sd)):
        e = np.linalg.norm((st[f] - ref).astype(float), axis=1)
        rows = s > 0
        worst = (e[rows] / s[rows] / (5e-15 + 2.0**-48 / t[rows])).max()
        print(kind, ratio, f, "largest error over its bound", worst)
        assert rows.sum() > 200 and worst <= 1.0
    sim.close()


@pytest.mark.parametrize("x0", [2e5, 1e6, 2e6, 5e6])
def test_boxes_far_from_the_origin(x0):
    """Where the FP32 prefilter lets pairs through up to 1.1, 1.3, 1.6 and more
    than 2 supports apart: the fixed-point differences hold them (the last
    box: every pair by the FP64 test), and the sets are the exact ones."""
    pos, _, _, sp = synth.periodic_block(8, 8, 8, seed=3, f_v=0.5, jitter=0.3)
    c = box_of(pos - [4.0, 4.0, 0.0] + [x0, 0.0, 0.0], sp, (8.0, 8.0))
    c.params = dict(c.params, box_lo=(x0 - 8.0, -8.0, 0.0), box_hi=(x0 + 8.0, 8.0, 8.0))
    sim = sim_of(c, nbr_cap=128)
    print(x0, per_particle_check(sim.state_arrays(), c, 0))
    assert neighbours_equal(sim, c)
    sim.close()


def test_partition_tiles_change_no_bit():
    """The species partition takes larger tiles from 2^20 particles on: a small
    vessel alone and batched with one that takes the batch past that."""
    a = synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9)
    b = synth.cylinder(60.0, 100, Omega=0.1, f_v=0.3, seed=10)
    assert a.n + b.n > 1 << 20
    solo, both = sim_of(a), sim_of([a, b])
    solo.step(2)
    both.step(2)
    x, y = solo.state_arrays(), both.state_arrays()
    for k in x:
        assert np.array_equal(x[k], y[k][:a.n]), k
    solo.close()
    both.close()


def test_a_batch_keeps_each_instance_on_its_own_pair_pass():
    """An instance without options equals its solo run bit for bit beside one
    whose options, and one whose masses, take the FP64 loops."""
    c = [synth.cylinder(6.3, 11, Omega=0.13, f_v=0.4, seed=9 + k) for k in range(3)]
    c[1].params = dict(c[1].params, flags=B.SPH_FLAGS_DEFAULT | B.SPH_COLLISION)
    c[2].params = dict(c[2].params, mass_ratio=20.0)
    batch = sim_of(c)
    got, at = batch.state_arrays(), 0
    for k in c:
        solo = sim_of(k)
        for f, x in solo.state_arrays().items():
            if "flags" in k.params or k.params["mass_ratio"] == 1.0:
                assert np.array_equal(got[f][at:at + k.n], x), f
            else:  # (the loops are compiled with the batch's options)
                assert np.abs(got[f][at:at + k.n] - x).max() <= 1e-13 * np.abs(x).max(), f
        at += k.n
        solo.close()
    batch.close()


@pytest.mark.parametrize("factor", [1e3, 1e6, 1e10, 1e-10])
def test_particles_far_faster_than_their_neighbours(factor):
    """One particle in fifty faster (or slower) than the rest by the factor:
    forces and torques of the others hang on differences far below the list's
    largest where the fast ones stand near the cutoff (the oracle is within
    1e-13 of extended precision on these states)."""
    pos, vel, spin, sp = synth.periodic_block(10, 10, 8, seed=8, f_v=0.5, jitter=0.2)
    c = box_of(pos - [5.0, 5.0, 0.0], sp, (10.0, 10.0))
    c.vel[::50] *= factor
    c.spin[::50] *= factor
    sim = sim_of(c)
    print(factor, per_particle_check(sim.state_arrays(), c, 0))
    sim.close()


def test_fluid_at_rest_beside_walls_that_turn():
    """A start from rest: among the unlike neighbours of a particle near the
    wall the fluid ones do not move, and the torque hangs on a wall particle
    that may stand at the cutoff (the oracle's shapes there are good to
    8 / t of 2^-53, which allows 1e-12 down to t = 0.001)."""
    c = synth.cylinder(7.0, 11, Omega=0.18, f_v=0.02, seed=3, jitter=0.35, dummy_layers=2)
    fl = c.species < 2
    c.vel[fl] = 0.0
    d = c.pos[fl][:, None] - c.pos[~fl][None]
    d[..., 2] -= 11.0 * np.round(d[..., 2] / 11.0)
    t = 1 - np.sqrt((d * d).sum(-1)) / 2.6
    nearest = t.max(1)
    assert ((nearest > 1e-3) & (nearest < 0.02)).sum() > 5
    sim = sim_of(c)
    st = sim.state_arrays()
    p = oracle.make_params(c.params)
    rho, P = oracle.density(p, c.pos, c.species)
    _, dsp, _, sc = oracle.forces(p, c.pos, c.vel, c.spin, c.species, rho, P, scale=True)
    e = np.linalg.norm(st["dspin"][fl] - dsp[fl], axis=1)
    rows = (sc[fl, 1] > 0) & (nearest > 1e-3)
    print((e[rows] / sc[fl, 1][rows]).max())
    assert (e[rows] <= 1e-12 * sc[fl, 1][rows]).all()
    assert (st["dspin"][fl][sc[fl, 1] == 0] == 0).all()
    sim.close()
