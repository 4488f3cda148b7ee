"""Device memory that only one precision or only the consistent mobility uses is made when that is
used: the double-float records (192 bytes per node) with FP64, the FP32 records (64) of a single
network with mixed precision, the consistent system's rows (80) with that mobility.

Sizes are in multiples of 2 MB on the device, so a record of n nodes shows as its bytes less 2 MB at least.
"""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MAT = W.Material().as_tuple()
MB2, DT = 2 << 20, 5e-13
RECORD = {ptadd.PTADD_FP64: 192, ptadd.PTADD_MIXED: 64}


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info(0)[0]


def relmax(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / np.max(np.abs(b)))


@pytest.mark.parametrize("first,second", [(ptadd.PTADD_MIXED, ptadd.PTADD_FP64), (ptadd.PTADD_FP64, ptadd.PTADD_MIXED)])
def test_network_buffers_are_made_when_they_are_used(first, second):
    net = W.loop_ensemble(5, 8192, 8e-6, np.zeros(6), nodes_per_loop=32)
    n = net.n_nodes
    with ptadd.Context(MAT, first, 0) as c:
        c.set_network(net)
        a = free()
        c.set_precision(second)
        b = free()
        c.set_mobility(True)
        d = free()
        assert a - b >= RECORD[second] * n - MB2
        assert b - d >= 80 * n - MB2
        c.set_precision(first)  # both are there now
        c.set_precision(second)
        assert free() == d


def test_batch_buffers_are_made_when_they_are_used():
    batch = W.batch_from_networks([W.loop_ensemble(60 + r, 32, 1.2e-6, np.zeros(6)) for r in range(256)])
    n = batch.xyz.shape[0]
    with ptadd.Context(MAT, ptadd.PTADD_MIXED, 0) as c:
        c.batch_set(batch)
        c.batch_get_forces()
        a = free()
        c.set_precision(ptadd.PTADD_FP64)
        c.batch_get_forces()
        b = free()
        c.set_mobility(True)
        c.batch_advance(1, DT)
        d = free()
    assert a - b >= 192 * n - MB2
    assert b - d >= 80 * n - MB2


@pytest.mark.parametrize("order", [(0, 1, 0), (1, 0, 1)])
def test_results_across_switches(order):
    """Forces and a consistent burst after every switch, as the oracle has them, and a network set in between."""
    sig = np.array([20e6, -35e6, 50e6, 10e6, -5e6, 25e6])
    nets = [W.loop_ensemble(17, 3, 0.5e-6, sig, nodes_per_loop=24), W.loop_ensemble(18, 7, 0.7e-6, sig, nodes_per_loop=30)]
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.set_mobility(True)
        for net in nets:
            c.set_network(net)
            Fo = O.nodal_forces(MAT, net)
            ref = O.burst(MAT, net, 2, DT, consistent_mass=True)
            for mixed in order:
                c.set_precision(ptadd.PTADD_MIXED if mixed else ptadd.PTADD_FP64)
                c.set_nodes(net.xyz)
                assert relmax(c.get_forces(), Fo) <= (1e-4 if mixed else 1e-11)
                Lp, _ = c.advance(2, DT)
                assert relmax(Lp, ref["Lp_avg"]) <= (1e-2 if mixed else 1e-9)


def test_switch_inside_a_capture_and_replay_after_switches():
    """Forces in both precisions captured into one graph, the switch (and its buffers) inside the capture; the graph
    gives the same after the context has been switched on."""
    sig = np.array([20e6, -35e6, 50e6, 10e6, -5e6, 25e6])
    net = W.loop_ensemble(19, 5, 0.6e-6, sig, nodes_per_loop=24)
    with ptadd.Context(MAT, ptadd.PTADD_MIXED, 0) as w:  # the kernels of both are loaded
        w.set_network(net)
        want = {}
        for prec in (ptadd.PTADD_MIXED, ptadd.PTADD_FP64):
            w.set_precision(prec)
            want[prec] = w.get_forces()
    out = {p: torch.zeros((net.n_nodes, 3), dtype=torch.float64, device="cuda") for p in want}
    stream = torch.cuda.Stream()
    with ptadd.Context(MAT, ptadd.PTADD_MIXED, 0) as c:
        c.set_stream(stream.cuda_stream)
        c.set_network(net)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for prec in (ptadd.PTADD_MIXED, ptadd.PTADD_FP64):
                c.set_precision(prec)
                c.get_forces_dev(out[prec].data_ptr())
        for prec in (ptadd.PTADD_MIXED, ptadd.PTADD_FP64, ptadd.PTADD_MIXED):
            c.set_precision(prec)
            for o in out.values():
                o.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            for p, o in out.items():
                assert np.array_equal(o.cpu().numpy(), want[p])
        del graph
