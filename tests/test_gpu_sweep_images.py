"""The plane sweep's choice of y and z images and its FP32 decisions against
the oracle's straight-line brute force: several images of one pair within
reach, trajectories many box lengths long, spheres that exactly touch, and
velocities with a large common part."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build
    from paper_1110_4876_gb300 import rb as m

    build.build()
    return m


def _compare(rb, orc, pos, vel, r, L, **kw):
    n = len(r)
    cfg = dict(box=L, gravity=0, dt=0.2, **kw)
    sim = rb.Sim(collisions=rb.RB_COLL_SWEEP, **cfg)
    sim.set_particles((*pos.T.copy(), *vel.T.copy(), np.ones(n), r))
    p = orc.Params(L=L, gravity=0, dt=0.2, collisions=1, **kw)
    ref = orc.collide_line_brute(p, 0.0, *pos.T.copy(), *vel.T.copy(), r, np.arange(n))
    assert np.array_equal(rb.pair_keys(*sim.pairs()), ref)
    return len(ref)


@pytest.mark.parametrize("ng,zper,Ly,Lz", [((1, 3, 0), 0, 3.0, 40.0), ((2, 2, 2), 1, 5.0, 4.0), ((1, 1, 0), 0, 30.0, 30.0)])
@pytest.mark.parametrize("speed", [1.0, 60.0])
def test_images_within_reach(rb, orc, ng, zper, Ly, Lz, speed):
    g = np.random.default_rng(int(Ly + speed))
    L = (40.0, Ly, Lz)
    n = 150
    pos = g.uniform(-0.5, 0.5, (n, 3)) * np.array(L)
    if not zper:
        pos[:, 2] = g.normal(0.0, 1.0, n)
    vel = g.normal(0.0, speed, (n, 3))
    assert _compare(rb, orc, pos, vel, g.uniform(0.2, 0.7, n), L, boundary=rb.RB_BC_PERIODIC, nghost=ng, z_periodic=zper)


@pytest.mark.parametrize("drift", [0.0, 1e6])
def test_touching_spheres_and_a_common_velocity(rb, orc, drift):
    """A lattice of unit spheres at distance 2 exactly: d^2 = s^2 is no hit;
    moved by one rounding of the positions some are."""
    k = np.arange(6.0)
    pos = np.stack(np.meshgrid(2.0 * k, 2.0 * k, 2.0 * k, indexing="ij"), -1).reshape(-1, 3) - 5.0
    g = np.random.default_rng(3)
    pos[::3] *= 1.0 - 2.0 ** -50
    vel = np.zeros_like(pos)
    vel[::2] = g.normal(0.0, 1e-9, (len(vel[::2]), 3))
    vel[:, 1] += drift
    _compare(rb, orc, pos, vel, np.ones(len(pos)), (64.0,) * 3, boundary=rb.RB_BC_OPEN)
