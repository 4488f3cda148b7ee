"""The FP64 path's split of the pairs: close ones in FP64, the others in
double-float arithmetic, in one-warp tiles of targets and chunks of sources.

Nodal forces against the oracle at the edges of that split (relative
max-norm <= 1e-11, the bar of every FP64 force): target counts around a warp,
source counts around a staged tile and a chunk, segments along their own
Burgers vector (no edge part to take the frame from), coarse and fine
segments beside each other (both near limits), and nodes so far apart that
the pairs leave the double-float range.
"""

import numpy as np
import pytest

import oracle as O
from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W
from test_zz_no_alloc import forces_noalloc

pytestmark = pytest.mark.gpu
MAT = W.Material().as_tuple()
SIG = np.array([20e6, -35e6, 50e6, 10e6, -5e6, 25e6])


def relmax(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def forces(net):
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.set_network(net)
        return c.get_forces()


@pytest.mark.parametrize("loops,nodes", [(1, 3), (1, 31), (1, 33), (2, 16), (3, 11), (5, 13), (13, 5), (3, 43),
                                         (16, 40)])
def test_forces_at_the_edges_of_tiles_and_chunks(loops, nodes):
    net = W.loop_ensemble(7 * loops + nodes, loops, 0.5e-6, SIG, nodes_per_loop=nodes)
    Fo = O.nodal_forces(MAT, net)
    assert relmax(forces(net), Fo) <= 1e-11
    assert relmax(forces_noalloc(net), Fo) <= 1e-11


def squares(sides, burgers, shift):
    """Square loops in the plane z = k * 7 b with sides along x and y."""
    xyz, n = [], len(sides)
    for k, s in enumerate(sides):
        c = np.array([[0, 0, 0], [s, 0, 0], [s, s, 0], [0, s, 0]], float)
        xyz.append(c + np.array([11.0 * k, 5.0 * k, 7.0 * k]) + shift[k])
    return W.Network(np.concatenate(xyz) * W.BURGERS, 4 * np.arange(n + 1), np.array(burgers, float) * W.BURGERS,
                     np.tile([0.0, 0.0, 1.0], (n, 1)), np.zeros(4 * n, np.uint8), 1e-20, SIG)


def test_screw_segments_and_mixed_segment_lengths():
    """Sides parallel to b (pure screw), to 1e-9 of it, and at 45 degrees; sides of 20 to 3000 b beside one another."""
    b = [[1, 0, 0], [0, 1, 0], [1, 1e-9, 0], [np.sqrt(0.5), np.sqrt(0.5), 0], [1, 0, 0], [0, 1, 0]]
    net = squares([20.0, 300.0, 900.0, 3000.0, 60.0, 5.0], b, np.zeros((6, 3)))
    Fo = O.nodal_forces(MAT, net)
    assert relmax(forces(net), Fo) <= 1e-11


def test_pairs_outside_the_double_float_range():
    """Two pairs of loops 4e6 b apart (the entry point on device arrays sets no extent): each node as the oracle
    has it.  At 4e6 b the positions' own last bit is 5e-10 b, so sides of 300 b keep the comparison at the bar."""
    far = np.zeros((4, 3))
    far[2:] = [4.0e6, -1.0e6, 2.0e6]
    net = squares([300.0, 500.0, 300.0, 500.0], [[1, 0, 0], [0, 1, 0], [0, 1, 0], [1, 0, 0]], far)
    net.xyz = np.round(net.xyz / W.BURGERS) * 2.0 ** -32  # whole multiples of the internal unit: no rounding on the way in
    Fo = O.nodal_forces(MAT, net)
    assert relmax(forces_noalloc(net), Fo) <= 1e-11
