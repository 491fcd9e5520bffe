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
