"""The FP64 substep's tile of fluid samples and its two CTA sizes, against the
separate entry points: both sides of the 38,912 granules up to which CTAs of 64
are taken, CTAs with a partly filled warp, and granules so far apart that the
box of a CTA's samples does not fit the tile."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP64, shuffled, subset
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,spread", [(1, False), (65, False), (38_911, False), (38_912, False), (38_913, False),
                                      (65, True), (300, True)])
def test_fp64_substep_matches_the_separate_calls(n, spread):
    # the same arithmetic in the same order: equal positions and velocities; F_s to
    # the order of the double atomics (at most ~200 terms a sample: 200 * 2^-53 < 1e-12)
    if spread:  # a few of 100,000 granules' places, over the whole domain
        prob = subset(shuffled(gi.differentiable_window(n=100_000, r0=0.001)), n)
    else:
        prob = shuffled(subset(gi.differentiable_window(n=40_000, r0=0.001), n))
    out = []
    for fused in (True, False):
        sim = Simulator.from_problem(prob, FP64, fused=fused)
        sim.run(1)
        torch.cuda.synchronize()
        assert gic.gic_check_status() == 0
        x, v = sim.positions()
        out.append((x.cpu().numpy(), v.cpu().numpy(), [f.cpu().numpy() for f in sim.Fs]))
    (xa, va, Fa), (xb, vb, Fb) = out
    assert np.array_equal(xa, xb) and np.array_equal(va, vb)
    for fa, fb in zip(Fa, Fb):
        assert np.abs(fa - fb).max() <= 1e-12 * max(np.abs(fb).max(), 1e-300)
