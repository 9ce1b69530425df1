"""A rebuild asked for in the middle of a gic_step call is the next call's: the
substep kernel's later CTAs (several times as many granules as the chip holds
at once) must not take it for their own.  One corner of a loose packing moves,
and passes skin / 2 in the second call, which keeps its lists."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64, shuffled
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [(FP32, 500_000), (FP64, 200_000)])
def test_a_rebuild_asked_for_in_a_call_waits_for_the_next(prec, n):
    prob = shuffled(gi.differentiable_window(n=n, r0=0.001))
    half_skin = 0.5 * 0.05 * float(prob.r.max())
    prob.v[:] = 0.0
    x = prob.positions()
    corner = (x < x.min(0) + 0.25 * (x.max(0) - x.min(0))).all(1)  # first in Morton order
    assert 0 < corner.sum() < n // 8
    prob.v[corner, 0] = 0.6 * half_skin / prob.params.dt_sub
    out = []
    for fused in (True, False):  # no contacts: the order of the granules does not enter
        sim = Simulator.from_problem(prob, prec, fused=fused)
        builds = []
        for _ in range(4):
            sim.run(1)
            builds.append(sim.nb.builds())
        torch.cuda.synchronize()
        assert gic.gic_check_status() == 0
        if fused:
            assert builds[:3] == [1, 1, 2]
        out.append([t.cpu().numpy() for t in sim.positions()])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
