"""Currents of particles on nodes: nodes whose weight is zero get exactly nothing."""
import numpy as np
import pytest

import paper_2104_11385_gb300 as pic
from paper_2104_11385_gb300 import workloads
from test_gpu_parity import make_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,axis", [(3, 0), (3, 1), (3, 2), (2, 0), (2, 2)])
def test_particle_on_a_node(dim, axis):
    """at rest but for one axis, on nodes along the others: the current of that axis on the
    nodes it sits on, and nothing else"""
    n, b = ((16, 16, 16), (8, 8, 8)) if dim == 3 else ((32, 1, 32), (16, 1, 16))
    wl = workloads.random_plasma(76, dim, n, b, (0.25, 0.25 if dim == 3 else 1.0, 0.25), 1, nspecies=1, npart=1, umax=0.1)
    sp = wl["species"][0]
    for a, (k, v) in enumerate(zip("xyz", ("ux", "uy", "uz"))):
        sp[k][:] = 0.0 if dim == 2 and a == 1 else (4.25 if a == axis else 4.0) * 0.25
        sp[v][:] = 0.1 if a == axis else 0.0
    sim = make_gpu(wl)
    sim.step(1)
    want = [slice(4, 5)] * 3
    if dim == 2:
        want[1] = slice(0, 1)
    for a, c in enumerate((pic.JX, pic.JX + 1, pic.JZ)):
        J = sim.read_field(c).reshape(n[::-1])
        some = np.zeros(J.shape, bool)
        if a == axis:
            some[want[2], want[1], want[0]] = True
        assert np.array_equal(J != 0.0, some), (a, np.argwhere(J != 0.0))
