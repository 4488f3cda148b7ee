"""FP64 forces where the double-float far field would leave FP32's range: Burgers vectors many orders of
magnitude from the material's, alone and beside ordinary ones, and cores and segments far below the unit of length.

Nodal forces against the oracle, 1e-11 of the loop's largest (the bar of every FP64 force): the far pairs carry
a per cent or so of them, so a far field lost to underflow, or turned into infinities, misses it by far.
"""

import numpy as np
import pytest

import oracle as O
from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W
from test_zz_no_alloc import forces_noalloc

pytestmark = pytest.mark.gpu
M = W.Material()
MAT = M.as_tuple()
SIG = np.array([20e6, -35e6, 50e6, 10e6, -5e6, 25e6])


def gpu(net, mat=MAT):
    with ptadd.Context(mat, ptadd.PTADD_FP64, 0) as c:
        c.set_network(net)
        return c.get_forces()


def per_loop(F, Fo, off):
    return max(np.max(np.abs(F[a:b] - Fo[a:b])) / np.max(np.abs(Fo[a:b])) for a, b in zip(off, off[1:]))


@pytest.mark.parametrize("scale", [1e-30, 1e-18, 1e-9, 2.0 ** -21, 2.0 ** -19, 2.0 ** 19, 2.0 ** 21, 1e9, 1e18, 1e30])
def test_burgers_vectors_of_any_size(scale):
    net = W.loop_ensemble(71, 3, 0.6e-6, np.zeros(6), nodes_per_loop=24)
    net.burgers = net.burgers * scale
    Fo = O.nodal_forces(MAT, net)
    assert per_loop(gpu(net), Fo, net.loop_off) <= 1e-11
    assert per_loop(forces_noalloc(net), Fo, net.loop_off) <= 1e-11


@pytest.mark.parametrize("scale", [1e-18, 1e-9, 1e9])
def test_one_loop_of_another_size(scale):
    """Loop 1's Burgers vector differs from the others'; every loop's forces to its own scale."""
    net = W.loop_ensemble(72, 4, 0.6e-6, SIG, nodes_per_loop=21)
    net.burgers = net.burgers.copy()
    net.burgers[1] *= scale
    Fo = O.nodal_forces(MAT, net)
    assert per_loop(gpu(net), Fo, net.loop_off) <= 1e-11


@pytest.mark.parametrize("size", [1e-3, 1e-8])
def test_segments_far_below_the_unit(size):
    """Square loops of side `size` b, 40 sides apart, and a core of a tenth of a side."""
    c = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0]], float)
    xyz = np.concatenate([c + 40.0 * np.array([k, k % 2, 0.5 * k]) for k in range(6)]) * (size * M.b)
    b = np.tile([[1.0, 0.0, 0.0], [0.6, 0.8, 0.0]], (3, 1)) * M.b
    net = W.Network(xyz, 4 * np.arange(7), b, np.tile([0.0, 0.0, 1.0], (6, 1)), np.zeros(24, np.uint8), 1e-20, np.zeros(6))
    mat = (M.mu, M.nu, M.b, 0.1 * size * M.b, M.B)
    Fo = O.nodal_forces(mat, net)
    assert per_loop(gpu(net, mat), Fo, net.loop_off) <= 1e-11


@pytest.mark.parametrize("core", [1e-2, 2.0 ** -13, 1e-8, 1e-12])
def test_cores_far_below_the_unit(core):
    """Square loops along the axes on whole multiples of the kernels' unit, 2^-32 m: a point on its own segment's line
    is there without rounding.  (One that is off by its last bit, 1e-13 units, changes the field by 1e-13 / core^2.)"""
    sides, unit = [20.0, 64.0, 300.0, 128.0, 50.0, 200.0], 2.0 ** -32
    xyz = [np.array([[0, 0, 0], [s, 0, 0], [s, s, 0], [0, s, 0]]) + np.array([11.0 * k, 5.0 * k, 7.0 * k])
           for k, s in enumerate(sides)]
    b = np.tile([[1.0, 0.0, 0.0], [0.5, 0.75, 0.0]], (3, 1)) * unit
    net = W.Network(np.concatenate(xyz) * unit, 4 * np.arange(7), b, np.tile([0.0, 0.0, 1.0], (6, 1)),
                    np.zeros(24, np.uint8), 1e-20, SIG)
    mat = (M.mu, M.nu, M.b, core * M.b, M.B)
    Fo = O.nodal_forces(mat, net)
    assert per_loop(gpu(net, mat), Fo, net.loop_off) <= 1e-11
