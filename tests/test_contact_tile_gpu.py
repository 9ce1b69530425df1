"""gic_contact on the staged neighbourhood (marked cells, candidate lists) against
its general kernel, which walks the 27 cells in global memory: CTAs of one
granule and with a last partial warp, more partners than a candidate list holds,
cells past the staged buffer, radii that differ, and granules so far apart that
no box fits.  The pair law and the order of the partners are the same, so the
forces are the same bits."""
import dataclasses

import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, shuffled, subset
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _crowded():  # a contact grid far coarser than the granules
    prob = gi.make("dense_block", n_side=(10, 10, 10))
    coarse = dataclasses.replace(prob.grid, k_contact=1)
    cell, q = gi.encode_positions(prob.positions(), coarse)
    return dataclasses.replace(prob, grid=coarse, cell=cell, q=q)


CASES = {
    "one": lambda: subset(gi.make("dense_block"), 1),
    "partial": lambda: subset(shuffled(gi.make("dense_block")), 301),
    "partners": lambda: gi.make("dense_block", n_side=(9, 9, 9), nn_factor=1.6),
    "crowded": _crowded,
    "bed": lambda: gi.polydisperse_bed(n=20_000),
    "far": lambda: subset(shuffled(gi.differentiable_window(n=100_000, r0=0.001)), 300),
}


@pytest.mark.parametrize("name", list(CASES))
def test_staged_contact_gives_the_general_kernels_forces(name):
    sim = Simulator.from_problem(shuffled(CASES[name]()), FP32, verlet=False)
    gic.gic_sort(sim.grid, sim.A, sim.B, sim.perm, sim.table, sim.ws)
    out = []
    for st in (sim.B, dataclasses.replace(sim.B, posf=None)):
        F = torch.full_like(sim.F_c, float("nan"))
        gic.gic_contact(sim.grid, sim.params, st, sim.table, F)
        torch.cuda.synchronize()
        assert gic.gic_check_status() == 0
        out.append(F)
    assert torch.equal(*out)
    if name in ("partners", "crowded", "bed"):
        assert bool((out[0] != 0).any())
