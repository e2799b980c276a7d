"""The particle kernel's and the binning's less travelled routes against the
oracle, at the sizes and values where each can go wrong: moves across one cell
face per direction and shape order, fields too small for the fixed-point tile,
weights near the ends of the double range, tiles too large for the particle
staging buffers, boxes far fewer than the SMs, positions at cell faces."""
import numpy as np
import pytest

import oracle as orc
import paper_2104_11385_gb300 as pic
from paper_2104_11385_gb300 import workloads
from test_gpu_parity import compare, make_gpu, make_oracle, rel

pytestmark = pytest.mark.gpu


def boxes(dim, order):
    n = (16, 16, 24) if dim == 3 else (32, 1, 48)
    b = (8, 8, 8) if dim == 3 else (16, 1, 16)
    return workloads.random_plasma(60 + order, dim, n, b, (0.3, 0.3 if dim == 3 else 1.0, 0.35), order, nspecies=1,
                                   npart=3000, umax=3.0)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("dim,axis", [(3, 0), (3, 1), (3, 2), (2, 0), (2, 2)])
def test_moves_along_one_axis(dim, axis, order):
    """fast along one axis, nearly at rest along the others: every crossing is of one face"""
    wl = boxes(dim, order)
    for a, k in enumerate(("ux", "uy", "uz")):
        if a != axis:
            wl["species"][0][k] *= 1e-9
    sim, ref = make_gpu(wl), make_oracle(wl)
    sim.step(3)
    ref.step(3)
    compare(sim, ref, wl)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("scale", [1e-280, 1.0, 1e3])
def test_field_magnitudes(order, scale):
    """1e-280 lies below the fixed-point tile's exponent range: the FP64 gather"""
    wl = boxes(3, order)
    wl["species"][0]["w"] *= min(scale, 1.0)  # the plasma's own fields stay near the given ones
    fields = [scale * f for f in workloads.random_fields(9, wl["ncell"], amp=0.2)]
    sim, ref = make_gpu(wl, fields), make_oracle(wl, fields)
    sim.step(2)
    ref.step(2)
    compare(sim, ref, wl)


@pytest.mark.parametrize("dim,order", [(3, 1), (3, 3), (2, 1), (2, 2)])
@pytest.mark.parametrize("w", [0.0, 1e-290, 1e280])
def test_weights_near_the_ends_of_the_range(dim, order, w):
    wl = boxes(dim, order)
    sp = wl["species"][0]
    sp["w"] = np.where(np.arange(sp["w"].size) % 2 == 0, w, 0.0)
    sim, ref = make_gpu(wl), make_oracle(wl)
    sim.step(1)
    ref.step(1)
    for c in (pic.JX, pic.JX + 1, pic.JZ):
        g, r = sim.read_field(c).reshape(-1), ref.field(c).reshape(-1)
        assert np.all(np.isfinite(g))
        assert rel(g, r) < 1e-10 if np.abs(r).max() > 1e-285 else np.abs(g - r).max() < 1e-295


def test_infinite_field_leaves_the_rest_of_its_tile_alone():
    """a tile holding Inf is gathered in FP64: particles away from it see their own fields"""
    wl = boxes(3, 1)
    sp = wl["species"][0]
    cell = [np.floor(sp[k] / wl["dx"][a]) for a, k in enumerate("xyz")]
    far = np.any([np.abs(v - 4) > 2 for v in cell], axis=0)
    for k in list(sp):
        if isinstance(sp[k], np.ndarray):
            sp[k] = sp[k][far]
    fields = workloads.random_fields(9, wl["ncell"], amp=0.2)
    clean = make_gpu(wl, fields)
    fields[0] = fields[0].copy()
    fields[0].reshape(wl["ncell"][::-1])[4, 4, 4] = np.inf
    sim = make_gpu(wl, fields)
    sim.step(1)
    clean.step(1)
    g, c = sim.particles(0), clean.particles(0)
    gi, ci = np.argsort(g["id"]), np.argsort(c["id"])
    for k in ("ux", "uy", "uz", "x"):
        assert rel(g[k][gi], c[k][ci]) < 1e-13


@pytest.mark.parametrize("order", [2, 3])
def test_tile_without_staging_buffers(order):
    wl = workloads.random_plasma(71, 2, (64, 1, 128), (64, 1, 64), (0.3, 1.0, 0.3), order, nspecies=2, npart=4000,
                                 umax=1.0)
    fields = workloads.random_fields(5, wl["ncell"], amp=0.2)
    sim, ref = make_gpu(wl, fields), make_oracle(wl, fields)
    sim.set_launch(tile=64)
    sim.step(4)
    ref.step(4)
    compare(sim, ref, wl)


@pytest.mark.parametrize("mode", ["none", "queue", "lists"])
@pytest.mark.parametrize("npart", [1, 700, 40000])
def test_few_boxes_shared_by_many_ctas(mode, npart):
    wl = workloads.random_plasma(72, 3, (16, 16, 8), (8, 8, 8), (0.3, 0.3, 0.3), 1, nspecies=2, npart=npart, umax=1.0)
    sim, ref = make_gpu(wl), make_oracle(wl)
    if mode != "none":
        sim.set_lb_params(mode=pic.LB_DYNAMIC, interval=2, theta=0.0, cost=pic.COST_HEURISTIC,
                          sched=pic.SCHED_QUEUE if mode == "queue" else pic.SCHED_LISTS)
    sim.step(5)
    ref.step(5)
    compare(sim, ref, wl)
    _, counts = sim.box_costs(pic.COST_HEURISTIC)
    assert np.array_equal(counts, ref.box_counts(wl["box"]))


@pytest.mark.parametrize("d", [0.25, 0.3, 1.0 / 3.0, 7.0, 1e-3])
def test_bin_positions_at_cell_faces(d):
    """k d and its neighbours, also outside the domain: the boxes of the rounded division"""
    import torch
    from paper_2104_11385_gb300 import sim as S
    n, box = (60, 1, 4096), (3, 1, 512)
    k = np.arange(-4200, 4300, dtype=np.float64)
    x = np.concatenate([k * d, np.nextafter(k * d, -np.inf), np.nextafter(k * d, np.inf), [0.0, -0.0, 1e-300, -1e-300],
                        np.random.default_rng(3).uniform(-1, 2, 5000) * n[2] * d])
    z = x[::-1].copy()
    off_r, perm_r = orc.bin_particles(2, n, (d, 1.0, d), box, x, np.zeros_like(x), z)
    off = torch.empty(len(off_r), dtype=torch.int64, device="cuda")
    perm = torch.empty(x.size, dtype=torch.int64, device="cuda")
    S.bin_particles(2, n, box, (d, 1.0, d), torch.as_tensor(x, device="cuda"), None, torch.as_tensor(z, device="cuda"),
                    off, perm)
    torch.cuda.synchronize()
    off_g, perm_g = off.cpu().numpy(), perm.cpu().numpy()
    assert np.array_equal(off_g, off_r)
    for b in range(len(off_r) - 1):
        assert np.array_equal(np.sort(perm_g[off_r[b]:off_r[b + 1]]), np.sort(perm_r[off_r[b]:off_r[b + 1]]))


@pytest.mark.parametrize("dim,order,precision,ppt", [(3, 1, 1, 1), (3, 2, 1, 2), (2, 3, 1, 1), (2, 1, 1, 2), (3, 1, 3, 1),
                                                     (2, 2, 3, 2)])
def test_steps_in_one_call_and_one_by_one(dim, order, precision, ppt):
    """the steps of one call sort through an order, single calls move the particles:
    the same particles, ids and weights, with some absorbed on the way"""
    n, b = ((16, 16, 32), (8, 8, 8)) if dim == 3 else ((32, 1, 64), (16, 1, 16))
    wl = workloads.random_plasma(80, dim, n, b, (0.3, 0.3 if dim == 3 else 1.0, 0.3), order, nspecies=2, npart=5000,
                                 umax=2.0, absorb=4)
    wl["species"][1]["w"] *= np.linspace(0.5, 2.0, 5000)
    fields = workloads.random_fields(3, n, amp=0.2)
    runs = [make_gpu(wl, fields) for _ in range(3)]
    for s in runs:
        s.set_launch(precision=precision, ppt=ppt)
    runs[0].step(7)
    for _ in range(7):
        runs[1].step(1)
    runs[2].set_lb_params(mode=pic.LB_DYNAMIC, interval=3, theta=0.0, sched=pic.SCHED_QUEUE)
    for k in (2, 4, 1):
        runs[2].step(k)
    tol = 1e-10 if precision == 1 else 3e-5
    ref = make_oracle(wl, fields)
    ref.step(7)
    for s in runs:
        compare(s, ref, wl, tol=tol)


@pytest.mark.parametrize("npart", [9727, 9728, 16384, 16385, 5000003])  # 8 boxes: shared-memory counts from 9728 on (152 SMs)
@pytest.mark.parametrize("one_box", [False, True])
def test_bin_shared_counts(npart, one_box):
    import torch
    from paper_2104_11385_gb300 import sim as S
    n, box, d = (16, 16, 16), (8, 8, 8), 0.3
    r = np.random.default_rng(npart)
    x, y, z = (r.uniform(0.0, (8 if one_box else 16) * d * 0.999, npart) for _ in range(3))
    off = torch.empty(9, dtype=torch.int64, device="cuda")
    perm = torch.empty(npart, dtype=torch.int64, device="cuda")
    S.bin_particles(3, n, box, (d, d, d), *(torch.as_tensor(a, device="cuda") for a in (x, y, z)), off, perm)
    torch.cuda.synchronize()
    cell = [np.floor(a / d).astype(np.int64) // 8 for a in (x, y, z)]
    want = (cell[2] * 2 + cell[1]) * 2 + cell[0]
    off_g, perm_g = off.cpu().numpy(), perm.cpu().numpy()
    assert np.array_equal(off_g, np.concatenate([[0], np.cumsum(np.bincount(want, minlength=8))]))
    assert np.array_equal(want[perm_g], np.repeat(np.arange(8), np.diff(off_g)))
    assert np.array_equal(np.sort(perm_g), np.arange(npart))
