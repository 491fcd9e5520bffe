"""Particles that share the Morton bits the sort's passes take (a clump far
smaller than the box): runs put in order by one thread, by one block, and runs
of equal keys, alone and beside the same clump in another box."""
import numpy as np
import pytest

from paper_1110_4876_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build
    from paper_1110_4876_gb300 import rb as m

    build.build()
    return m


def _clumps(n, scale, seed):
    """n particles in clumps of 16, 17 and the rest, each `scale` wide."""
    g = np.random.default_rng(seed)
    P = I.random_cube(n, seed)
    centre = g.uniform(-0.4, 0.4, (3, 3))
    which = np.minimum(np.arange(n) // 16, 2)
    which[32:33] = 1
    for k, f in enumerate(("x", "y", "z")):
        getattr(P, f)[:] = centre[which, k] + scale * getattr(P, f)
    order = g.permutation(n)
    return P.subset(order)


# 2^-13 is the depth the passes sort to; 1e-5 leaves one run per clump, 1e-7
# brings equal keys among them
@pytest.mark.parametrize("n", [40, 300, 2500])
@pytest.mark.parametrize("scale", [1e-3, 1e-5, 1e-7])
def test_forces_of_clumps(rb, orc, n, scale):
    p = orc.Params(G=1.0, L=(1.0,) * 3, theta=0.5, soft=1e-9, gravity=1)
    cfg = dict(G=1.0, box=(1.0,) * 3, theta=0.5, softening=1e-9, gravity=1, walk=rb.RB_WALK_FP64)
    boxes = [_clumps(n, scale, n), _clumps(n, scale, n), _clumps(n // 2, scale, n + 1)]
    ens = rb.Sim(nbox=3, **cfg)
    for b, P in enumerate(boxes):
        ens.set_particles(P, b)
    rb.rb_compute_gravity(ens.h)
    for b, P in enumerate(boxes):
        ref = orc.tree_gravity(p, 0.0, P.x, P.y, P.z, P.m)
        alone = rb.Sim(**cfg)
        alone.set_particles(P)
        den = np.maximum(np.linalg.norm(ref, axis=1), 1e-3 * np.sqrt(np.mean((ref ** 2).sum(1))))
        for a in (alone.gravity(), rb.rb_get_accelerations(ens.h, b)):
            # FP64 on both sides, but a cell's centre near 0.4 is rounded to
            # 2^-54 on each, and the narrowest accepted cells, of a few
            # neighbours, lie scale / 50 away: 3 x 2^-54 x 50 / scale of such a
            # term, below 1e-14 / scale
            assert np.max(np.linalg.norm(a - ref, axis=1) / den) <= 1e-12 + 1e-14 / scale


# passes to depth 13, 15 and 21, by the width of a long box and the number of
# particles that share its cells there
@pytest.mark.parametrize("n,width", [(1500, 1e-4), (3000, 1e-4), (8200, 1e-5)])
def test_long_boxes(rb, orc, n, width):
    g = np.random.default_rng(n)
    L = (1.0, width, 1.0)
    pos = (g.random((n, 3)) - 0.5) * (1.0, width, 1e-6)
    r = g.uniform(0.05, 0.4, n) * width
    zero = np.zeros(n)
    cfg = dict(boundary=1, nghost=(1, 1, 0), gravity=0, collisions=1, dt=1e-3)
    sim = rb.Sim(box=L, **cfg)
    sim.set_particles((*np.ascontiguousarray(pos.T), zero, zero, zero, np.ones(n), r))
    ref = orc.collide_brute(orc.Params(L=L, **cfg), 0.0, *np.ascontiguousarray(pos.T), r, np.arange(n))
    assert len(ref)
    for _ in range(2):
        assert np.array_equal(rb.pair_keys(*sim.pairs()), ref)


def test_a_clump_of_one_long_run(rb, orc):
    """5,000 particles within one cell of depth 13 (and one outside): a run too
    long for one block, after which every key bit is sorted by passes."""
    P = I.random_cube(5000, 3)
    for f in ("x", "y", "z"):
        getattr(P, f)[:-1] = 0.3 + 2e-5 * getattr(P, f)[:-1]
    p = orc.Params(G=1.0, L=(1.0,) * 3, theta=0.5, soft=1e-9, gravity=1)
    ref = orc.tree_gravity(p, 0.0, P.x, P.y, P.z, P.m)
    den = np.maximum(np.linalg.norm(ref, axis=1), 1e-3 * np.sqrt(np.mean((ref ** 2).sum(1))))
    sim = rb.Sim(G=1.0, box=(1.0,) * 3, theta=0.5, softening=1e-9, gravity=1, walk=rb.RB_WALK_FP64)
    for _ in range(3):   # by runs, by passes, by passes on the same buffers
        sim.set_particles(P)
        # as for the clumps above, scale 2e-5
        assert np.max(np.linalg.norm(sim.gravity() - ref, axis=1) / den) <= 1e-12 + 1e-14 / 2e-5


def _clump():
    """5,000 particles within one cell of depth 13: a run that one block puts in
    order, longer than the passes over its bits would take."""
    P = I.random_cube(5000, 3)
    for f in ("x", "y", "z"):
        getattr(P, f)[:] = 0.3 + 2e-5 * getattr(P, f)
    P.r[:] = 1e-9
    return P


def _sim(rb):
    return rb.Sim(box=(1.0,) * 3, gravity=0, collisions=1, dt=1e-9)


def _kernels(rb, sim):
    sim.step(1)
    return sim.stats()["kernels_per_step"]


def test_detecting_pairs_finds_long_runs(rb):
    """Every call that sorts notices the long run: after rb_detect_collisions the
    first step already sorts all bits by passes, as a simulation that only steps
    does from its second step on."""
    stepped, detected = _sim(rb), _sim(rb)
    for s in (stepped, detected):
        s.set_particles(_clump())
    runs, passes = _kernels(rb, stepped), _kernels(rb, stepped)
    assert runs != passes
    detected.pairs()
    assert _kernels(rb, detected) == passes


def test_new_particles_may_lie_apart_again(rb):
    """A set of spread-out particles after a clump is sorted by runs again; after
    a second clump the passes keep every bit."""
    spread = I.random_cube(5000, 3)
    spread.r[:] = 1e-9
    sim = _sim(rb)
    sim.set_particles(spread)
    runs = _kernels(rb, sim)
    sim.set_particles(_clump())
    sim.step(1)
    passes = _kernels(rb, sim)
    assert runs != passes
    sim.set_particles(spread)
    assert _kernels(rb, sim) == runs
    sim.set_particles(_clump())
    sim.step(1)
    assert _kernels(rb, sim) == passes
    sim.set_particles(spread)
    assert _kernels(rb, sim) == passes
