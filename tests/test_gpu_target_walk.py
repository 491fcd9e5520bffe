"""The walks with one and with two targets per warp against the walk over 32
targets per warp: the same accepted cells, exact terms and tests per target,
forces that differ only in the order of FP32 sums.  Which of them runs depends
on the particle capacity, so a simulation that once held more particles keeps
the other walk."""
import numpy as np
import pytest

from paper_1110_4876_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PAIRS = 3_003     # capacity from which a warp takes two targets (one with the network)
LARGE = 130_001   # capacity from which every walk runs over 32 targets per warp


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build
    from paper_1110_4876_gb300 import rb as m

    build.build()
    return m


def _each(rb, P, pairs, large, w=None, **cfg):
    """(forces, counts) of a fresh simulation and of two of larger capacity."""
    got = []
    for first in (None, pairs, large):
        sim = rb.Sim(**cfg)
        if w is not None:
            rb.rb_load_mlp(sim.h, w, 0.5)
        if first is not None:
            sim.set_particles(first)
            sim.gravity()
        sim.set_particles(P)
        got.append(sim.gravity(counts=True))
    return got


def _check(got, tol):
    b, cb = got[-1]
    den = np.maximum(np.linalg.norm(b, axis=1), 1e-3 * np.sqrt(np.mean(np.sum(b * b, axis=1))) + 1e-300)
    for a, ca in got[:-1]:
        for x, y in zip(ca, cb):
            np.testing.assert_array_equal(x, y)
        assert np.max(np.linalg.norm(a - b, axis=1) / den) <= tol


def _sheet(rb, L, **kw):
    return dict(G=I.G_SI, omega=I.OMEGA, box=(L, L, L), boundary=rb.RB_BC_SHEAR, integrator=rb.RB_INT_SEI,
                dt=I.DT_SHEET, gravity=1, walk=rb.RB_WALK_FP32, **kw)


# one target, partial and full units of targets; images in one and in two
# batches of 32; an opening angle so small that every cell is opened (the
# stack at its limit) and one with the inside rule
@pytest.mark.parametrize("n,theta,ng", [(1, 0.5, 1), (2, 0.5, 1), (33, 0.9, 1), (257, 0.5, 3), (900, 0.02, 1),
                                        (3001, 0.7, 1)])
@pytest.mark.parametrize("quad", [0, 1])
def test_sheet_equals_the_walk_over_32_targets(rb, n, theta, ng, quad):
    L = 120.0
    cfg = _sheet(rb, L, theta=theta, nghost=(ng, ng, 0), quadrupole=quad)
    # sums of n terms in FP32 pieces of at most 16: as between the other
    # launch shapes (2e-5 of each force)
    _check(_each(rb, I.sheet(L, n, 11), I.sheet(L, PAIRS, 12), I.sheet(L, LARGE, 12), **cfg), 2e-5)


@pytest.mark.parametrize("theta", [0.5, 0.9])
def test_softened_cluster(rb, theta):
    P = I.plummer(2500, 4)
    for k in ("x", "y", "z"):
        getattr(P, k)[7] = getattr(P, k)[8]   # a coincident pair, a depth-21 group
    cfg = dict(G=1.0, box=(128.0,) * 3, theta=theta, softening=1e-2, dt=1e-3, gravity=1, walk=rb.RB_WALK_FP32)
    _check(_each(rb, P, I.plummer(PAIRS, 6), I.plummer(LARGE, 5), **cfg), 2e-5)


@pytest.mark.parametrize("n", [5, 2000])
def test_learned_walk(rb, n):
    from paper_1110_4876_gb300 import learned

    L = 110.0
    w = learned.init_weights(3)
    w[-(64 * 3 + 3):-3] = np.random.default_rng(1).normal(0.0, 0.004, 64 * 3)
    cfg = _sheet(rb, L, theta=0.8, nghost=(1, 1, 0))
    cfg["walk"] = rb.RB_WALK_FP32_LEARNED
    # the network's inputs and outputs are the same rows in both
    _check(_each(rb, I.sheet(L, n, 13), I.sheet(L, PAIRS, 12), I.sheet(L, LARGE, 12), w=w, **cfg), 2e-5)


def test_pairs_across_boxes(rb):
    """Batched boxes of odd sizes: pairs of targets that lie in different boxes."""
    sizes = (1, 700, 3, 801, 1601)
    L = 100.0
    cfg = _sheet(rb, L, theta=0.6, nghost=(1, 1, 0))
    boxes = [I.sheet(L, n, 20 + n) for n in sizes]
    sim = rb.Sim(nbox=len(sizes), **cfg)
    for b, P in enumerate(boxes):
        sim.set_particles(P, b)
    rb.rb_compute_gravity(sim.h)
    # each box of the batch against the box alone (one target per warp)
    for b, P in enumerate(boxes):
        alone = rb.Sim(**cfg)
        alone.set_particles(P)
        a, ca = alone.gravity(counts=True)
        x, cx = rb.rb_get_accelerations(sim.h, b), rb.rb_get_counts(sim.h, b)
        _check([(x, cx), (a, ca)], 2e-5)
