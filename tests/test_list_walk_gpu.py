"""The contact walk over candidate lists (gic_step, with and without alpha_s) against
the plain walk of the rows (a state without its float position copies): rows of
no partner, of fewer and of more than a list holds, and partial warps.  The
partners and their order are the same, so positions and velocities are the same
bits; alpha_s, accumulated where the lists were, is the separate entry point's."""
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
    "one": lambda: subset(gi.make("dense_block"), 1),
    "partial": lambda: subset(shuffled(gi.make("dense_block")), 301),
    "long_rows": lambda: gi.make("dense_block", n_side=(9, 9, 9), nn_factor=1.6),
    "uneven_rows": lambda: gi.polydisperse_bed(n=20_000),
}


@pytest.mark.parametrize("name", list(CASES))
def test_candidate_lists_give_the_rows_own_forces(name):
    sim = Simulator.from_problem(shuffled(CASES[name]()), FP32)
    sim.substep(alpha=False, sums=False)  # builds the lists
    F = sim.fluid
    before = [t.clone() for t in (sim.A.cell, sim.A.pos, sim.A.vel)]
    if name == "long_rows":
        assert int(sim.nb.count.max()) > 10  # entries of the substep's list
    out = []
    alpha_s = torch.zeros_like(sim.alpha_s)
    for alpha, st in ((None, sim.A), (sim.alpha_s, sim.A), (None, dataclasses.replace(sim.A, posf=None))):
        for dst, src in zip((sim.A.cell, sim.A.pos, sim.A.vel), before):
            assert torch.equal(dst, src)
        gic.gic_step(sim.grid, sim.params, st, sim.A2, sim.B, sim.perm, sim.table, sim.ws, sim.nb, F.u, F.v, F.w,
                     F.p, F.alpha_f, alpha, (None, None, None), None)
        torch.cuda.synchronize()
        out.append([t.cpu().numpy() for t in (sim.A2.cell, sim.A2.pos, sim.A2.vel)])
        sim.nb.flags[5] = 0  # this call's request is not the next one's
    assert gic.gic_check_status() == 0 and sim.nb.builds() == 1
    for a, b, c in zip(*out):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    gic.gic_p2g(sim.grid, sim.params, sim.A, sim.A2, sim.f_ex, alpha_s)
    torch.cuda.synchronize()
    assert torch.equal(alpha_s, sim.alpha_s)
