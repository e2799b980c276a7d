"""Small runs under a scheduler: enough work units for every persistent CTA."""
import numpy as np
import pytest
import torch

import paper_2104_11385_gb300 as pic
from paper_2104_11385_gb300 import workloads
from test_gpu_parity import compare, make_gpu, make_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npart", [40000, 130000, 300000])
@pytest.mark.parametrize("sched", [pic.SCHED_QUEUE, pic.SCHED_LISTS])
def test_heavy_boxes_are_cut_for_all_ctas(npart, sched):
    """16 boxes hold every particle; the cut leaves no unit below 256 particles and,
    where there are 256 per CTA, a unit for at least three CTAs of four"""
    wl = workloads.random_plasma(73, 3, (32, 32, 64), (16, 16, 16), (0.3, 0.3, 0.3), 1, nspecies=1, npart=npart, umax=0.5)
    sp = wl["species"][0]
    sp["z"] *= 0.249  # into the first layer of boxes, 4 of 16
    sim = make_gpu(wl)
    ctas = sim.get_launch()["ctas_per_sm"] * torch.cuda.get_device_properties(0).multi_processor_count
    r = sim.rebalance(mode=pic.LB_DYNAMIC, interval=10, theta=0.0, cost=pic.COST_HEURISTIC, sched=sched)
    with_particles = r["n_units"] - 12
    assert with_particles <= max(4, npart // 256)
    if npart >= 256 * ctas:
        assert with_particles >= 0.75 * ctas
    else:
        assert with_particles >= 0.75 * npart / 256
    if npart == 40000:
        ref = make_oracle(wl)
        sim.step(3)
        ref.step(3)
        compare(sim, ref, wl)


@pytest.mark.parametrize("sched", [pic.SCHED_QUEUE, pic.SCHED_LISTS])
def test_units_after_most_particles_left(sched):
    """few boxes, nearly all particles absorbed: a mapping made then is cut for what is left"""
    wl = workloads.random_plasma(75, 3, (16, 16, 32), (8, 8, 16), (0.3, 0.3, 0.3), 1, nspecies=1, npart=20000, umax=0.5,
                                 absorb=6)
    sp = wl["species"][0]
    sp["uz"][:19000] = np.where(sp["z"][:19000] < 4.8, -50.0, 50.0)  # out through the nearer layer
    sim, ref = make_gpu(wl), make_oracle(wl)
    for s in (sim, ref):
        s.step(24)
    assert sim.num_particles(0) < 5000
    sim.rebalance(mode=pic.LB_DYNAMIC, interval=10, theta=0.0, cost=pic.COST_HEURISTIC, sched=sched)
    for s in (sim, ref):
        s.step(3)
    compare(sim, ref, wl)


@pytest.mark.parametrize("sched", [pic.SCHED_QUEUE, pic.SCHED_LISTS])
def test_efficiency_of_shared_units_is_the_mappings(sched):
    """8 boxes shared by all CTAs: E counts the 8 units, one worker each"""
    wl = workloads.random_plasma(77, 3, (16, 16, 16), (8, 8, 8), (0.3, 0.3, 0.3), 1, nspecies=1, npart=20000, umax=0.5)
    sim = make_gpu(wl)
    sim.set_lb_params(mode=pic.LB_DYNAMIC, interval=1000, theta=0.0, cost=pic.COST_HEURISTIC, sched=sched)
    sim.step(1)
    costs, _ = sim.box_costs(pic.COST_HEURISTIC)
    workers = sim.get_launch()["ctas_per_sm"] * torch.cuda.get_device_properties(0).multi_processor_count
    assert sim.efficiency(pic.COST_HEURISTIC) == pytest.approx(costs.sum() / workers / costs.max(), rel=1e-12)
