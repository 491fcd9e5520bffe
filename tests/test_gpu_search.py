"""The tree search's shared candidate lists against brute force, bit for bit:
runs of targets that are cut at gaps, lists that fill up, leaf groups of
coincident particles, unequal radii, and more images than one batch of 32.
Each with 4, 8 and 32 targets a warp, which the particle capacity decides: a
simulation that once held more particles keeps the wider runs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build
    from paper_1110_4876_gb300 import rb as m

    build.build()
    return m


def _compare(rb, orc, pos, r, L, boundary, ng, z_periodic=0):
    n = len(r)
    zero = np.zeros(n)
    p = orc.Params(L=(L, L, L), boundary=boundary, nghost=ng, z_periodic=z_periodic, gravity=0, collisions=1, dt=1e-3)
    ref = orc.collide_brute(p, 0.0, *np.ascontiguousarray(pos.T), r, np.arange(n))
    for held in (0, 10_001, 40_001):
        sim = rb.Sim(box=(L, L, L), boundary=boundary, nghost=ng, z_periodic=z_periodic, gravity=0, collisions=1,
                     dt=1e-3)
        if held:
            z = np.zeros(held)
            many = np.random.default_rng(held).uniform(-0.5 * L, 0.5 * L, (3, held))
            sim.set_particles((*many, z, z, z, np.ones(held), np.full(held, 1e-3)))
            sim.pairs()
        sim.set_particles((*np.ascontiguousarray(pos.T), zero, zero, zero, np.ones(n), r))
        assert np.array_equal(rb.pair_keys(*sim.pairs()), ref)
    return len(ref)


@pytest.mark.parametrize("n", [2, 33, 700])
@pytest.mark.parametrize("boundary", [0, 1])
def test_scattered_runs_and_unequal_radii(rb, orc, n, boundary):
    """A quarter of the particles far from a dense clump: neighbours in the
    tree's order lie far apart; radii over two decades."""
    g = np.random.default_rng(n)
    L = 400.0
    pos = g.normal(0.0, 4.0, (n, 3))
    far = g.random(n) < 0.25
    pos[far] = g.uniform(-0.5 * L, 0.5 * L, (int(far.sum()), 3))
    found = _compare(rb, orc, pos, 10.0 ** g.uniform(-1.5, 0.5, n), L, boundary, (1, 1, 0) if boundary else (0, 0, 0))
    assert found or n < 33


@pytest.mark.parametrize("copies", [31, 97])
def test_coincident_groups(rb, orc, copies):
    """Groups of coincident particles beside others: every member is a
    candidate, more than a list holds at once."""
    g = np.random.default_rng(copies)
    pos = g.uniform(-6.0, 6.0, (300, 3))
    pos[50: 50 + copies] = pos[50]
    pos[200: 200 + copies] = pos[200]
    assert _compare(rb, orc, pos, np.full(300, 0.8), 16.0, 1, (1, 1, 0)) > copies ** 2 / 2


def test_more_images_than_a_batch(rb, orc):
    """49 and 27 images of a box only a little larger than the spheres."""
    g = np.random.default_rng(2)
    pos = g.uniform(-2.0, 2.0, (40, 3))
    assert _compare(rb, orc, pos, g.uniform(0.3, 0.9, 40), 4.0, 1, (3, 3, 0)) > 0
    assert _compare(rb, orc, pos, g.uniform(0.3, 0.9, 40), 4.0, 1, (1, 1, 1), 1) > 0
