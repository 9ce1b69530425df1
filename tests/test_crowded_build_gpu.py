"""List builds of a state whose cells hold too many granules for the staged
neighbourhood (a contact grid much coarser than the granules): the rows that
gic_neighbors_build and gic_step take from global memory, with and without the
float copies of the positions, against the 27-cell build of gic_contact_verlet."""
import dataclasses

import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, shuffled
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _rows(sim):
    n, cap = sim.nb.n, sim.nb.cap
    used = torch.arange(cap, device="cuda")[None, :] < sim.nb.count[:, None]
    return sim.nb.count.clone(), torch.where(used, sim.nb.list[:n * cap].view(n, cap), -1)


@pytest.mark.parametrize("k_contact", [1, 2])
def test_rows_from_global_memory(k_contact):
    base = gi.make("dense_block", n_side=(12, 12, 12))
    grid = dataclasses.replace(base.grid, k_contact=k_contact)
    cell, q = gi.encode_positions(base.positions(), grid)
    prob = shuffled(dataclasses.replace(base, grid=grid, cell=cell, q=q))
    sim = Simulator.from_problem(prob, FP32)
    gic.gic_sort(sim.grid, sim.A, sim.B, sim.perm, sim.table, sim.ws)
    out = []
    gic.gic_contact_verlet(sim.grid, sim.params, sim.B, sim.table, sim.nb, sim.F_c)
    out.append(_rows(sim))
    gic.gic_neighbors_build(sim.grid, sim.B, sim.table, sim.nb)
    out.append(_rows(sim))
    for posf in (True, False):
        step = Simulator.from_problem(prob, FP32)
        if not posf:
            step.A.posf = step.A2.posf = step.B.posf = None
        step.substep()
        assert step.nb.builds() == 1 and torch.equal(step.perm, sim.perm)
        out.append(_rows(step))
    assert gic.gic_check_status() == 0
    assert int(out[0][0].sum()) > 0
    for count, rows in out[1:]:
        assert torch.equal(count, out[0][0]) and torch.equal(rows, out[0][1])
