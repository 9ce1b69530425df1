"""gic_step with the capillary force takes the granules' moisture ratios from an array
that it fills first; gic_substep interpolates them pair by pair.  The same
values in the same sums: the same bits, in a call that rebuilds and in one that
keeps its lists."""
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64, shuffled, subset
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n", [1, 33, 257, 500])
def test_moisture_array_gives_the_pairwise_ratios(n, prec):
    prob = shuffled(gi.make("wet_block"))
    prob = subset(prob, min(n, prob.n))
    a, b = (Simulator.from_problem(prob, prec) for _ in range(2))
    F = b.fluid
    for call in range(2):  # builds the lists; keeps them
        a.substep(alpha=False, sums=False)
        if call == 0:
            gic.gic_sort(b.grid, b.A, b.B, b.perm, b.table, b.ws)
        gic.gic_substep(b.grid, b.params, b.B, b.table, b.nb, F.u, F.v, F.w, F.p, F.alpha_f, b.A, None, None,
                        (None, None, None), None)
        torch.cuda.synchronize()
        assert gic.gic_check_status() == 0 and a.nb.builds() == b.nb.builds() == 1
        assert torch.equal(a.A.id, b.A.id) and torch.equal(a.A.cell, b.A.cell)
        assert torch.equal(a.A.pos, b.A.pos) and torch.equal(a.A.vel, b.A.vel)
        b.A, b.B = b.B, b.A
