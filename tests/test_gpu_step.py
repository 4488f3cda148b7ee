"""The fused O(N) phases of a step where their grouping of the nodes changes: up
to 32 nodes of whole loops to a block, a longer loop walked by its block, and
blocks of 32 nodes wherever the loops end once a loop has more than 256.

Bursts of ten steps against the oracle's, lumped and consistent mobility, alone
and as a batch, to the FP64 bars of the burst tests (positions 1e-9, displacements
1e-7, Lp 1e-8, line length 1e-12 relative).
"""

import numpy as np
import pytest

import oracle as O
from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MAT = W.Material().as_tuple()
STEPS, DT = 10, 5e-13
SIG = np.array([20e6, -35e6, 50e6, 10e6, -5e6, 25e6])


def relmax(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / np.max(np.abs(b)))


def network(counts, pinned=False):
    """One loop of each node count, 0.3 to 0.5 um in radius (a segment of 256 nodes is 7 nm or more)."""
    nets = [W.loop_ensemble(900 + 7 * i + n, 1, 2e-6, SIG, nodes_per_loop=n, r_min=3e-7, r_max=5e-7)
            for i, n in enumerate(counts)]
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    pin = np.zeros(off[-1], np.uint8)
    if pinned:
        pin[3::11] = 1
    return W.Network(np.concatenate([t.xyz for t in nets]), off, np.concatenate([t.burgers for t in nets]),
                     np.concatenate([t.normal for t in nets]), pin, 8e-18, SIG)


CASES = [((31,), False), ((32, 33), True), ((255, 5), False), ((256, 3, 40), True), ((257, 7, 31), False),
         ((20, 300, 12), True)]


def check(x, Lp, rho, net, ref):
    assert relmax(x, ref["xyz"]) <= 1e-9
    assert relmax(x - net.xyz, ref["xyz"] - net.xyz) <= 1e-7
    assert relmax(Lp, ref["Lp_avg"]) <= 1e-8
    assert abs(rho / ref["rho_avg"] - 1) <= 1e-12
    pin = net.pinned.astype(bool)
    assert np.all(x[pin] == net.xyz[pin])


@pytest.mark.parametrize("consistent", [False, True])
@pytest.mark.parametrize("counts,pinned", CASES)
def test_burst_at_the_edges_of_the_grouping(counts, pinned, consistent):
    net = network(counts, pinned)
    ref = O.burst(MAT, net, STEPS, DT, consistent_mass=consistent)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.set_network(net)
        c.set_applied_stress(net.sig_app)
        c.set_mobility(consistent)
        Lp, rho = c.advance(STEPS, DT)
        check(c.get_nodes(), Lp, rho, net, ref)


@pytest.mark.parametrize("consistent", [False, True])
@pytest.mark.parametrize("pick", [(0, 1, 3), (0, 4, 5)])  # whole loops to a block, and not
def test_batch_at_the_edges_of_the_grouping(pick, consistent):
    nets = [network(*CASES[k]) for k in pick]
    batch = W.batch_from_networks(nets)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.set_mobility(consistent)
        c.batch_set(batch)
        Lp, rho = c.batch_advance(STEPS, DT)
        x = c.batch_get_nodes()
    for r, net in enumerate(nets):
        ref = O.burst(MAT, net, STEPS, DT, consistent_mass=consistent)
        a, b = batch.node_off[r], batch.node_off[r + 1]
        check(x[a:b], Lp[r], rho[r], net, ref)
