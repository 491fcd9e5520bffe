"""Resolution order: particles with many contacts, whose pairs are one long
chain, as the lower id, as the higher id and in between."""
import numpy as np
import pytest

from _parity import stepwise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build
    from paper_1110_4876_gb300 import rb as m

    build.build()
    return m


# n - 1 small spheres on one large one; `at` places the large one's id first,
# last or in the middle: its pairs are then all of its lower side, all of its
# higher side, or both.  33 and 1025: a pair past a warp's 32 and a block's 256.
@pytest.mark.parametrize("n,at", [(2, 0), (33, 0), (33, 32), (1025, 0), (1025, 1024), (1025, 500)])
def test_one_body_with_many_contacts(rb, orc, n, at):
    g = np.random.default_rng(n + at)
    u = g.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    pos = 10.0 * u * g.uniform(0.97, 1.03, (n, 1))
    vel = -0.3 * u + g.normal(0.0, 0.2, (n, 3))
    r = g.uniform(0.1, 0.4, n)
    m = g.uniform(0.5, 1.5, n)
    pos[at], vel[at], r[at], m[at] = 0.0, 0.0, 10.0, 50.0
    L = 64.0
    cfg = dict(box=(L, L, L), boundary=rb.RB_BC_OPEN, integrator=rb.RB_INT_LEAPFROG, dt=1e-3, eps=0.6, gravity=0,
               collisions=1)
    sim = rb.Sim(**cfg)
    sim.set_particles((*pos.T.copy(), *vel.T.copy(), m, r))
    p = orc.Params(L=(L, L, L), boundary=0, integrator=0, dt=1e-3, eps=0.6, gravity=0, collisions=1)
    # the large body takes one rounding (2^-53 of its speed) per impulse:
    # n of them against the oracle's form of Eq. 2 stay below 2e-12
    found = stepwise(rb, orc, sim, p, 2, vtol=2e-12)
    assert found >= n // 2


def test_a_speed_that_is_not_a_number_spreads(rb, orc):
    """Two massless bodies in contact leave Eq. 2 with 0/0; the next pair of
    either carries it on to its other body, as in the oracle, and a pair apart
    from them stays as it is."""
    x = np.array([0.0, 1.0, 2.0, 3.0, 10.0, 11.0])
    zero = np.zeros(6)
    vx = np.array([1.0, 0.0, -1.0, -2.0, 1.0, -1.0])
    m, r = np.array([0.0, 0.0, 1.0, 1.0, 1.0, 1.0]), np.full(6, 0.6)
    cfg = dict(eps=0.5, dt=1e-4, gravity=0, collisions=1)
    sim = rb.Sim(box=(64.0,) * 3, boundary=rb.RB_BC_OPEN, **cfg)
    sim.set_particles((x, zero, zero, vx, zero, zero, m, r))
    sim.step(1)
    st = orc.State(orc.Params(L=(64.0,) * 3, boundary=0, integrator=0, **cfg), x, zero, zero, vx, zero, zero, m, r)
    st.step(1)
    got = sim.particles()["vx"]
    assert np.isnan(st.vx[:4]).all() and not np.isnan(st.vx[4:]).any()
    np.testing.assert_allclose(got, st.vx, rtol=1e-15)
