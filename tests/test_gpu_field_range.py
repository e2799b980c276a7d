"""Fields whose magnitudes differ by many binades inside one staged tile: every
particle sees the fields of its own support, to FP64's accuracy."""
import numpy as np
import pytest

import paper_2104_11385_gb300 as pic
from paper_2104_11385_gb300 import workloads
from test_gpu_parity import make_gpu, make_oracle, rel

pytestmark = pytest.mark.gpu


def plasma(dim, order, keep):
    """random plasma with only the particles for which keep(cells) holds (cells: per active axis)"""
    n, b = ((16, 16, 32), (8, 8, 16)) if dim == 3 else ((32, 1, 64), (16, 1, 32))
    wl = workloads.random_plasma(90 + order, dim, n, b, (0.3, 0.3 if dim == 3 else 1.0, 0.3), order, nspecies=1,
                                 npart=4000, umax=1.0)
    sp = wl["species"][0]
    axes = [a for a in range(3) if dim == 3 or a != 1]
    sel = keep([np.floor(sp["xyz"[a]] / wl["dx"][a]) for a in axes], [n[a] for a in axes])
    for k in list(sp):
        if isinstance(sp[k], np.ndarray):
            sp[k] = sp[k][sel]
    assert sp["x"].size > 500
    return wl


@pytest.mark.parametrize("dim,order,tile", [(3, 1, 4), (3, 1, 8), (3, 2, 8), (3, 3, 4), (2, 1, 16), (2, 2, 8), (2, 3, 16)])
@pytest.mark.parametrize("spike", [1e12, 1e20])
def test_one_cell_far_above_the_rest(dim, order, tile, spike):
    """particles that do not touch the cell move as without it"""
    wl = plasma(dim, order, lambda cell, n: np.any([np.abs(c - 4) > 3 for c in cell], axis=0))
    fields = workloads.random_fields(9, wl["ncell"], amp=0.2)
    clean = make_gpu(wl, fields)
    for c in (0, 4):
        fields[c] = fields[c].copy()
        fields[c].reshape(wl["ncell"][::-1])[4, 4 if dim == 3 else 0, 4] = spike
    sim = make_gpu(wl, fields)
    for s in (sim, clean):
        s.set_launch(tile=tile)
        s.step(1)
    g, r = sim.particles(0), clean.particles(0)
    gi, ri = np.argsort(g["id"]), np.argsort(r["id"])
    for k in ("ux", "uy", "uz", "x", "z"):
        # the two gathers differ by roundings of 2^-53 each: a few 1e-15
        assert rel(g[k][gi], r[k][ri]) < 1e-13, k


@pytest.mark.parametrize("dim", [3, 2])
@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("energy", [False, True])
@pytest.mark.parametrize("binades", [0.7, 3.0])
def test_fields_falling_along_z(dim, order, energy, binades):
    """Fields that fall by so many binades per cell: what each particle gets is
    right relative to itself.  E alone on particles at rest gives u; B alone on
    particles with ux = 1 gives uy and uz."""
    wl = plasma(dim, order, lambda cell, n: np.all([(c >= 4) & (c < m - 4) for c, m in zip(cell, n)], axis=0))
    if energy:
        wl["gather"] = "energy"
    ncell = wl["ncell"]
    ramp = np.broadcast_to(0.2 * 2.0 ** (-binades * np.arange(ncell[2]))[:, None, None], ncell[::-1]).reshape(-1).copy()
    zero = np.zeros_like(ramp)
    sp = wl["species"][0]
    for k in ("ux", "uy", "uz"):
        sp[k] = np.zeros_like(sp[k])
    for fields, ux, keys in (([ramp] * 3 + [zero] * 3, 0.0, ("ux", "uy", "uz")), ([zero] * 4 + [ramp] * 2, 1.0, ("uy", "uz"))):
        sp["ux"] = np.full_like(sp["ux"], ux)
        sim, ref = make_gpu(wl, fields), make_oracle(wl, fields)
        sim.step(1)
        ref.step(1)
        g, r = sim.particles(0), ref.particles(0)
        gi, ri = np.argsort(g["id"]), np.argsort(r["id"])
        for k in keys:
            assert np.all(r[k] != 0.0)
            # a few dozen roundings of 2^-53 (oracle and kernel), no cancellation, and the
            # 9 (27) units of a fixed-point gather from a node that has 2^51 or more: 1.2e-14
            assert np.abs(g[k][gi] / r[k][ri] - 1.0).max() < 1e-13, k


@pytest.mark.parametrize("dim,order,energy,tile,threads", [
    (3, 1, False, 8, 256), (3, 1, True, 8, 256), (3, 2, False, 4, 128), (3, 2, True, 8, 32), (3, 3, False, 8, 256),
    (3, 3, True, 4, 256), (2, 1, False, 16, 64), (2, 1, True, 16, 256), (2, 2, False, 32, 256), (2, 2, True, 16, 256),
    (2, 3, False, 32, 96)])
@pytest.mark.parametrize("corner", [(2, 3, 5), (5, 6, 9), (1, 2, 12)])
def test_weak_patch(dim, order, energy, tile, threads, corner):
    """nodes [corner, corner + 7) hold fields 2^-40 of those around them: particles that
    interpolate from the patch alone see it to FP64's accuracy"""
    wl = plasma(dim, order, lambda cell, n: np.ones(cell[0].size, bool))
    if tile == 32:
        wl["box"] = (32, 1, 32)
    sp = wl["species"][0]
    r = np.random.default_rng(5)
    for a, k in enumerate("xyz"):
        if dim == 3 or a != 1:
            # cells corner + 2 and corner + 3: supports reach 2 nodes below and 3 above
            sp[k] = (corner[a] + 2 + r.uniform(0, 2, sp[k].size)) * wl["dx"][a]
    for k in ("ux", "uy", "uz"):
        sp[k] = np.zeros_like(sp[k])
    if energy:
        wl["gather"] = "energy"
    fields = workloads.random_fields(9, wl["ncell"], amp=0.2)
    s = tuple(slice(c, c + 7) for c in corner)
    patch = [slice(None)] * 3
    patch[0], patch[2] = s[2], s[0]
    if dim == 3:
        patch[1] = s[1]
    for c in range(3):
        fields[c] = fields[c].copy()
        fields[c].reshape(wl["ncell"][::-1])[tuple(patch)] *= 2.0 ** -40
    fields[3:] = [np.zeros_like(f) for f in fields[3:]]
    sim, ref = make_gpu(wl, fields), make_oracle(wl, fields)
    sim.set_launch(tile=tile, threads=threads)
    sim.step(1)
    ref.step(1)
    g, r = sim.particles(0), ref.particles(0)
    gi, ri = np.argsort(g["id"]), np.argsort(r["id"])
    for k in ("ux", "uy", "uz"):
        want = r[k][ri]
        assert 0.0 < np.abs(want).max() < 1e-10
        # dozens of roundings of 2^-53 relative to the patch's fields
        assert np.abs(g[k][gi] - want).max() < 1e-13 * np.abs(want).max(), k


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("order,energy", [(1, False), (1, True), (2, False), (3, True)])
def test_fields_falling_along_x_and_y(axis, order, energy):
    wl = plasma(3, order, lambda cell, n: np.all([(c >= 4) & (c < m - 4) for c, m in zip(cell, n)], axis=0))
    if energy:
        wl["gather"] = "energy"
    ncell = wl["ncell"]
    shape = [1, 1, 1]
    shape[2 - axis] = ncell[axis]
    ramp = np.broadcast_to((0.2 * 8.0 ** -np.arange(ncell[axis])).reshape(shape), ncell[::-1]).reshape(-1).copy()
    sp = wl["species"][0]
    for k in ("ux", "uy", "uz"):
        sp[k] = np.zeros_like(sp[k])
    fields = [ramp] * 3 + [np.zeros_like(ramp)] * 3
    sim, ref = make_gpu(wl, fields), make_oracle(wl, fields)
    sim.step(1)
    ref.step(1)
    g, r = sim.particles(0), ref.particles(0)
    gi, ri = np.argsort(g["id"]), np.argsort(r["id"])
    for k in ("ux", "uy", "uz"):
        assert np.abs(g[k][gi] / r[k][ri] - 1.0).max() < 1e-13, k  # as along z
