"""An FP64 batch of one large realisation among many tiny ones, and switches of the precision of a
loaded batch: parity with the oracle (1e-11 of the largest force, 1e-9 of positions and rates, the bars
of every FP64 batch) and a bounded work list.
"""

import functools

import numpy as np
import pytest

import oracle as O
from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MAT = W.Material().as_tuple()
SIG = np.array([20e6, -35e6, 50e6, 10e6, -5e6, 25e6])
STEPS, DT = 2, 5e-13


def relmax(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / np.max(np.abs(b)))


@functools.lru_cache(maxsize=None)
def networks():
    nets = [W.loop_ensemble(901, 100, 1.5e-6, SIG, nodes_per_loop=40)]
    nets += [W.loop_ensemble(1000 + r, 1, 0.4e-6, SIG, nodes_per_loop=3 + r % 5) for r in range(96)]
    nets[0].pinned[40:400] = 1
    return nets


def check(nets, batch, F, Lp, rho, x):
    for r in (0, 1, 2, 5, 95, 96):
        nt, n0, n1 = nets[r], batch.node_off[r], batch.node_off[r + 1]
        ref = O.burst(MAT, nt, STEPS, DT)
        Fo = O.nodal_forces(MAT, nt)
        free = nt.pinned == 0
        assert relmax(F[n0:n1][free], Fo[free]) <= 1e-11
        assert relmax(x[n0:n1] - nt.xyz, ref["xyz"] - nt.xyz) <= 1e-9
        assert relmax(Lp[r], ref["Lp_avg"]) <= 1e-9
        assert abs(rho[r] / ref["rho_avg"] - 1) <= 1e-12


def test_one_large_realisation_among_many_tiny_ones():
    nets = networks()
    batch = W.batch_from_networks(nets)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.batch_set(batch)
        info = c.batch_info()
        # 40 chunks, four times the mean one's, x 210 tiles (at equal lengths 114 tiles x 800 chunks)
        assert info["work_items"] <= 8400
        F = c.batch_get_forces()
        Lp, rho = c.batch_advance(STEPS, DT)
        x = c.batch_get_nodes()
    check(nets, batch, F, Lp, rho, x)


def test_precision_of_a_loaded_batch_switched_both_ways():
    """Mixed, then FP64 (whose finer chunks need more partial forces), then mixed again."""
    nets = networks()
    batch = W.batch_from_networks(nets)
    with ptadd.Context(MAT, ptadd.PTADD_MIXED, 0) as c:
        c.batch_set(batch)
        Fm = c.batch_get_forces()
        Lm, _ = c.batch_advance(STEPS, DT)
        c.set_precision(ptadd.PTADD_FP64)
        c.batch_set_nodes(batch.xyz)
        F = c.batch_get_forces()
        Lp, rho = c.batch_advance(STEPS, DT)
        x = c.batch_get_nodes()
        c.set_precision(ptadd.PTADD_MIXED)
        c.batch_set_nodes(batch.xyz)
        assert np.array_equal(c.batch_get_forces(), Fm)
        assert np.array_equal(c.batch_advance(STEPS, DT)[0], Lm)
    check(nets, batch, F, Lp, rho, x)
