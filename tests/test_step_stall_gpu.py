"""A wait of gic_step's sort that runs out (GIC_STATUS_STALL): the call and the
ones after it make no step and say so, and after gic_neighbors_reset the lists
work as fresh ones do.  The wait is let run out by a limit of no looks at all."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64, shuffled
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _arrays(st):
    return [t for t in (st.cell, st.pos, st.vel, st.id)]  # (posf is derived; gic_pack leaves it unset)


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("name", ["dense_block", "wet_block"])
@pytest.mark.parametrize("built", [False, True])  # on lists that hold no rows yet, and on lists in use
def test_stalled_lists_make_no_step_until_reset(name, prec, built):
    prob = shuffled(gi.make(name))
    fresh = Simulator.from_problem(prob, prec)
    sim = Simulator.from_problem(prob, prec)
    init = sim.A.clone()
    if built:
        sim.run(2)
        sim.nb.flags[5] = 1  # the next call is to rebuild
    else:  # what a C caller's memory may hold: rows that point nowhere
        sim.nb.list.fill_(2**30)
        sim.nb.count.fill_(sim.nb.cap)
        gic.gic_neighbors_reset(sim.nb)
        sim.lists_current = True
    gic.gic_check_status(clear=True)
    before = [t.clone() for t in _arrays(sim.A)]
    rows = sim.nb.list.clone()
    Fs = [f.clone() for f in sim.Fs]
    gic.gic_step_sort(sim.grid, sim.A, sim.B, sim.perm, sim.table, sim.ws, sim.nb, polls=0)
    assert gic.gic_check_status(clear=True) == gic.STATUS_STALL
    for _ in range(2):
        sim.substep()
        assert gic.gic_check_status(clear=True) == gic.STATUS_STALL
        assert all(torch.equal(a, b) for a, b in zip(_arrays(sim.A), before))
    assert torch.equal(sim.nb.list, rows) and all(torch.equal(a, b) for a, b in zip(sim.Fs, Fs))
    assert float(sim.alpha_s.abs().max()) == 0.0
    sim.load_state(init)  # the next gic_step starts from a reset
    sim.run(3)
    fresh.run(3)
    torch.cuda.synchronize()
    assert gic.gic_check_status() == 0
    for a, b in zip(sim.positions(), fresh.positions()):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
    assert torch.equal(sim.alpha_s, fresh.alpha_s) if prec == FP32 else True
