"""The antenna in the sharded field sub-steps: the E sub-step drives it by itself,
whatever was called between it and the B sub-step before it."""
import numpy as np
import pytest

import paper_2104_11385_gb300 as pic
from paper_2104_11385_gb300 import workloads
from test_gpu_parity import make_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [3, 2])
@pytest.mark.parametrize("between", ["nothing", "settings", "no B step"])
def test_e_substep_by_itself(dim, between):
    n, b = ((16, 16, 48), (8, 8, 16)) if dim == 3 else ((32, 1, 64), (16, 1, 16))
    wl = workloads.random_plasma(301, dim, n, b, (0.3, 0.3 if dim == 3 else 1.0, 0.3), 1, nspecies=1, npart=10, umax=0.1,
                                 absorb=6, laser=True)
    wl["species"][0]["w"][:] = 0.0  # the antenna alone drives the fields
    ref, sim = make_gpu(wl), make_gpu(wl)
    for s in (ref, sim):
        s.shard_set_owner(np.zeros(s.nboxes, np.int32), 0)
        s.set_step(3)
    for stage in (0, 1):
        ref.shard_field_stage(stage)
    if between != "no B step":
        sim.shard_field_stage(0)
    if between == "settings":
        sim.set_cost_capture(clock=True, kernel_time=False)
    sim.shard_field_stage(1)
    want, got = ref.read_field(pic.EX).reshape(-1), sim.read_field(pic.EX).reshape(-1)
    assert np.abs(want).max() > 0.0
    assert np.array_equal(got, want)
