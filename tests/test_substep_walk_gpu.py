"""gic_substep's contact walk over candidate lists (FP32 with float copies of the
positions) against the plain walk of the rows: calls that keep their lists, with and
without alpha_s, dry and wet.  The partners and their order are the same: the same
bits."""
import dataclasses

import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, shuffled, subset
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu

CASES = {
    "partial": lambda: subset(shuffled(gi.make("dense_block")), 301),
    "long_rows": lambda: gi.make("dense_block", n_side=(9, 9, 9), nn_factor=1.6),
    "uneven_rows": lambda: gi.polydisperse_bed(n=20_000),
    "wet": lambda: gi.make("wet_block"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_substep_walks_like_the_rows(name):
    sim = Simulator.from_problem(shuffled(CASES[name]()), FP32)
    F, out = sim.fluid, []
    fields = (F.u, F.v, F.w, F.p, F.alpha_f)
    gic.gic_sort(sim.grid, sim.A, sim.B, sim.perm, sim.table, sim.ws)
    gic.gic_substep(sim.grid, sim.params, sim.B, sim.table, sim.nb, *fields, sim.A2)  # builds
    alpha_s = [torch.zeros_like(sim.alpha_s) for _ in range(2)]
    for alpha, st in ((None, sim.B), (alpha_s[0], sim.B), (None, dataclasses.replace(sim.B, posf=None)),
                      (alpha_s[1], dataclasses.replace(sim.B, posf=None))):
        gic.gic_substep(sim.grid, sim.params, st, sim.table, sim.nb, *fields, sim.A2, None, alpha)
        torch.cuda.synchronize()
        out.append([t.cpu().numpy() for t in (sim.A2.cell, sim.A2.pos, sim.A2.vel)])
    assert gic.gic_check_status() == 0 and sim.nb.builds() == 1
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)
    assert torch.equal(*alpha_s)
