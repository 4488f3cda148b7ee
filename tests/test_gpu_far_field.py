"""What the far pairs alone contribute to the FP64 forces, on the GPU.

The rounding of the close pairs (a segment on itself and its neighbours), 1e-11 of the
largest force, hides the far field in a plain comparison.  It is the same, pair by pair, with
and without a second, distant group of loops; so the forces of two groups together less those of
each group alone are the far field between the groups, in which a difference of FP64
sums of 1e-16 of the force (a few hundred times the far one here) is left.

Bar 1e-9 of the largest cross force against the oracle's same difference: 300 x 64 additions x
1.1e-16 = 2e-12 at most from the sums, 1e-12 from the field (test_df_field.py); without the low
parts of the double-float numbers it would be 2^-24 = 6e-8 or more.
"""

import numpy as np
import pytest

import oracle as O
from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MAT = W.Material().as_tuple()


def join(a, b):
    return W.Network(np.concatenate([a.xyz, b.xyz]), np.concatenate([a.loop_off, a.n_nodes + b.loop_off[1:]]),
                     np.concatenate([a.burgers, b.burgers]), np.concatenate([a.normal, b.normal]),
                     np.concatenate([a.pinned, b.pinned]), a.volume, a.sig_app)


def cross(forces, a, b):
    both = forces(join(a, b))
    return both - np.concatenate([forces(a), forces(b)])


def gpu_forces(net):
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.set_network(net)
        return c.get_forces()


@pytest.mark.parametrize("loops,nodes,gap", [(1, 21, 0.6e-6), (3, 32, 1.5e-6), (8, 40, 4e-6)])
def test_forces_between_distant_groups(loops, nodes, gap):
    a = W.loop_ensemble(31 + loops, loops, 0.3e-6, np.zeros(6), nodes_per_loop=nodes)
    b = W.loop_ensemble(57 + loops, loops, 0.3e-6, np.zeros(6), nodes_per_loop=nodes)
    b.xyz = b.xyz + np.array([gap, -0.4 * gap, 0.7 * gap])
    ref = cross(lambda n: O.nodal_forces(MAT, n), a, b)
    got = cross(gpu_forces, a, b)
    assert np.max(np.abs(got - ref)) <= 1e-9 * np.max(np.abs(ref))
