"""Accelerations and counts read back in id order: with ids removed through an
open face, into fewer places than ids, per box of a batch, and while other
particles are already staged."""
import ctypes as C

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


def _cfg(rb):
    return dict(G=1.0, box=(1.0,) * 3, theta=0.5, softening=1e-3, dt=0.1, gravity=1, boundary=rb.RB_BC_OPEN,
                walk=rb.RB_WALK_FP64)


def test_removed_ids_and_small_arrays(rb, orc):
    n = 700
    P = I.random_cube(n, 5)
    P.vx[::5] = 100.0   # gone after the first drift half
    sim = rb.Sim(**_cfg(rb))
    sim.set_particles(P)
    sim.step(1)
    left = sim.particles()
    live = len(left["id"])
    assert live < n
    a, (nc, nl, nm) = sim.gravity(counts=True)
    assert a.shape == (live, 3) and len(nc) == live
    p = orc.Params(G=1.0, L=(1.0,) * 3, theta=0.5, soft=1e-3, gravity=1)
    ref = orc.tree_gravity(p, 0.0, left["x"], left["y"], left["z"], left["m"])
    assert np.max(np.abs(a - ref)) <= 1e-11 * np.abs(ref).max()
    assert np.all(nc + nl > 0) and np.all(nm >= nc)
    # exactly as many places as live particles, and one too few
    x = np.zeros(live)
    assert rb.load().rb_get_accelerations(sim.h, 0, live, x.ctypes.data_as(C.c_void_p), None, None) == rb.RB_OK
    assert np.array_equal(x, a[:, 0])
    assert rb.load().rb_get_accelerations(sim.h, 0, live - 1, x.ctypes.data_as(C.c_void_p), None, None) == rb.RB_ERR_ARG


def test_boxes_and_staged_particles(rb):
    sets = [I.random_cube(n, n) for n in (300, 1, 41)]
    ens = rb.Sim(nbox=3, **_cfg(rb))
    for b, P in enumerate(sets):
        ens.set_particles(P, b)
    rb.rb_compute_gravity(ens.h)
    alone = []
    for b, P in enumerate(sets):
        s = rb.Sim(**_cfg(rb))
        s.set_particles(P)
        alone.append(s.gravity())
        assert np.max(np.abs(rb.rb_get_accelerations(ens.h, b) - alone[b])) <= 1e-12 * max(1e-300, np.abs(alone[b]).max())
    # more particles staged for box 1, not yet on the device: the last walk's
    # results stay readable
    ens.set_particles(I.random_cube(5000, 9), 1)
    out = np.zeros((3, 300))
    rc = rb.load().rb_get_accelerations(ens.h, 0, 300, *(v.ctypes.data_as(C.c_void_p) for v in out))
    assert rc == rb.RB_OK
    assert np.max(np.abs(out.T - alone[0])) <= 1e-12 * np.abs(alone[0]).max()
