"""Close pairs among ordinary particles of a unit box, in every form of the FP32
walk: a leaf's term is m d / (d^2 + b^2)^(3/2) alone, finite in FP32 down to
distances of about 1e-13, where r^-5 and r^-7 have long left FP32's range
(below 2.2e-8 and 3.1e-6)."""
import numpy as np
import pytest

from paper_1110_4876_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the form that runs depends on the particle capacity: one target per warp,
# two from 3,000, 32 above 130,000; walk group 4 at any size
FORMS = {"one": (None, 0), "two": (3_003, 0), "union": (130_001, 0), "group": (None, 4)}


@pytest.fixture(scope="module")
def rb():
    from paper_1110_4876_gb300 import build
    from paper_1110_4876_gb300 import rb as m

    build.build()
    return m


def _pairs(gap):
    """300 particles of a unit box, five pairs of them `gap` apart, on either side
    of the plane x = 0, so that no cell but the root holds both of a pair."""
    P = I.random_cube(300, 9)
    for k in range(5):
        a, b = 10 * k, 10 * k + 1
        P.x[a], P.x[b] = -0.5 * gap, 0.5 * gap
        P.y[b], P.z[b] = P.y[a], P.z[a]
    return P


def _check(a, cnt, P, ref, ref_cnt):
    for x, r in zip(cnt, ref_cnt):
        np.testing.assert_array_equal(x, r)
    norm = np.linalg.norm(ref, axis=1)
    close = np.zeros(len(norm), bool)
    close[[10 * k + i for k in range(5) for i in (0, 1)]] = True
    # the ordinary particles' forces beside the pairs' are 1e-12 and less: each
    # against its own, with the floor of the parity tests taken over its kind
    for sel in (close, ~close):
        den = np.maximum(norm[sel], 1e-3 * np.sqrt(np.mean(norm[sel] ** 2)))
        assert np.max(np.linalg.norm((a - ref)[sel], axis=1) / den) <= 1e-5


@pytest.mark.parametrize("gap,soft", [(1e-6, 0.0), (1e-8, 0.0), (1e-6, 1e-9), (1e-8, 1e-9), (0.0, 1e-9)])
@pytest.mark.parametrize("form", FORMS)
def test_forces_of_close_pairs(rb, orc, form, gap, soft):
    capacity, group = FORMS[form]
    P = _pairs(gap)
    sim = rb.Sim(G=1.0, box=(1.0,) * 3, theta=0.5, softening=soft, gravity=1, walk=rb.RB_WALK_FP32)
    rb.rb_set_launch_shape(sim.h, 128, 128, group)
    if capacity:
        sim.set_particles(I.random_cube(capacity, 1))
        sim.gravity()
    sim.set_particles(P)
    a, cnt = sim.gravity(counts=True)
    p = orc.Params(G=1.0, L=(1.0,) * 3, theta=0.5, soft=soft, gravity=1)
    ref, ref_cnt = orc.tree_gravity(p, 0.0, P.x, P.y, P.z, P.m, counts=True)
    _check(a, cnt[:2], P, ref, ref_cnt[:2])


@pytest.mark.parametrize("gap", [1e-6, 1e-8])
def test_learned_walk_of_close_pairs(rb, orc, gap):
    """The network with zero weights adds nothing: the tree's forces at theta."""
    P = _pairs(gap)
    sim = rb.Sim(G=1.0, box=(1.0,) * 3, theta=0.8, gravity=1, walk=rb.RB_WALK_FP32_LEARNED)
    rb.rb_load_mlp(sim.h, np.zeros(rb.RB_MLP_PARAMS, np.float32), 0.5)
    sim.set_particles(P)
    a, cnt = sim.gravity(counts=True)
    p = orc.Params(G=1.0, L=(1.0,) * 3, theta=0.8, gravity=1)
    ref, ref_cnt = orc.tree_gravity(p, 0.0, P.x, P.y, P.z, P.m, counts=True)
    _check(a, cnt[:2], P, ref, ref_cnt[:2])
