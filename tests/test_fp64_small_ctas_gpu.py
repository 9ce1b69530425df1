"""gic_step's FP64 substep on both sides of the size up to which it takes CTAs of 64
(three per SM of the device), against the separate entry points."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP64, shuffled, subset
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("past", [-1, 0, 1])
def test_fp64_substep_around_the_small_ctas_limit(past):
    n = 3 * 64 * torch.cuda.get_device_properties(0).multi_processor_count + past
    prob = shuffled(subset(gi.differentiable_window(n=40_000, r0=0.001), n))
    out = []
    for fused in (True, False):
        sim = Simulator.from_problem(prob, FP64, fused=fused)
        sim.run(2)  # one call that builds the lists and one that keeps them
        torch.cuda.synchronize()
        assert gic.gic_check_status() == 0
        out.append([t.cpu().numpy() for t in sim.positions()])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
