"""Moments of cells within one range of slots, across a few and across many
ranges, and of leaf groups of coincident particles that cover whole ranges,
against sums over the cells' members."""
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


def _check(rb, P, L, walk, least):
    """Cells of at least `least` members of a tree built over P."""
    sim = rb.Sim(G=1.0, box=(L, L, L), theta=0.9, softening=0.1, gravity=1, walk=walk)
    sim.set_particles(P)
    sim.gravity()
    pos = np.stack([P.x, P.y, P.z], 1)
    # masses and centres are FP64 sums of up to n terms; the quadrupole is
    # summed in FP32 for the FP32 walk (pieces of at most about 100 terms,
    # 2^-24 each and one per level)
    qtol = 1e-11 if walk == rb.RB_WALK_FP64 else 2e-5
    seen = 0
    for depth, ids, M, com, Q in rb.rb_get_tree(sim.h):
        if len(ids) < least:
            continue
        m, x = P.m[ids], pos[ids]
        ref = (m[:, None] * x).sum(0) / m.sum()
        d = x - ref
        d2 = (d * d).sum(1)
        q = np.array([(m * (3 * d[:, 0] ** 2 - d2)).sum(), (m * (3 * d[:, 1] ** 2 - d2)).sum(),
                      (m * (3 * d[:, 2] ** 2 - d2)).sum(), (m * 3 * d[:, 0] * d[:, 1]).sum(),
                      (m * 3 * d[:, 0] * d[:, 2]).sum(), (m * 3 * d[:, 1] * d[:, 2]).sum()])
        w = max(np.ptp(x, axis=0).max(), 1e-9 * L)
        assert abs(M - m.sum()) <= 1e-12 * m.sum()
        assert np.max(np.abs(com - ref)) <= 1e-12 * w + 4e-16 * L
        assert np.max(np.abs(Q - q)) <= qtol * m.sum() * w * w
        seen += 1
    return seen


@pytest.mark.parametrize("walk", [0, 1])
# edges of a range (256) and of a tile of the entry scan (2048)
@pytest.mark.parametrize("n", [2, 255, 256, 257, 700, 2047, 2048, 2049, 5000])
def test_every_cell_of_small_trees(rb, n, walk):
    assert _check(rb, I.random_cube(n, n), 1.0, walk, 2) >= 1


@pytest.mark.parametrize("walk", [0, 1])
def test_cells_across_many_ranges(rb, walk):
    n = 160_000   # 607 ranges of 264 slots
    assert _check(rb, I.random_cube(n, 3), 1.0, walk, 1000) == 1 + 8 + 64


@pytest.mark.parametrize("walk", [0, 1])
def test_coincident_group_over_ranges(rb, walk):
    P = I.random_cube(2000, 8)
    for k in ("x", "y", "z"):
        getattr(P, k)[300:1300] = getattr(P, k)[300]
    assert _check(rb, P, 1.0, walk, 500) >= 2
