"""gic_step's rebuild (the one-launch sort and the list build inside the
substep kernel) against the separate entry points, at the sizes where its
loops change form: a single granule, the edges of a warp, a CTA and a sort
tile, and past the 256 tiles up to which a warp scans a digit's counts."""
import dataclasses

import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64, shuffled, subset
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _lattice(n):
    """n granules of a loose lattice in a random order (half as many again as
    the contact cells hold one each)."""
    prob = gi.differentiable_window(n=max(n, 8), r0=0.002 if n < 100_000 else 0.001)
    return shuffled(subset(prob, n))


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n", [1, 31, 257, 1023, 1025, 4097, 262_145])
def test_step_sorts_and_steps_like_the_separate_calls(n, prec):
    prob = _lattice(n)
    a = Simulator.from_problem(prob, prec)
    b = Simulator.from_problem(prob, prec)
    a.substep()  # gic_step, which rebuilds
    F = b.fluid
    gic.gic_sort(b.grid, b.A, b.B, b.perm, b.table, b.ws)
    gic.gic_substep(b.grid, b.params, b.B, b.table, b.nb, F.u, F.v, F.w, F.p, F.alpha_f, b.A, None, b.alpha_s, b.Fs,
                    b.sums)
    torch.cuda.synchronize()
    assert gic.gic_check_status() == 0
    assert torch.equal(a.perm, b.perm) and torch.equal(a.A.id, b.A.id) and torch.equal(a.A.cell, b.A.cell)
    assert torch.equal(a.A.pos, b.A.pos) and torch.equal(a.A.vel, b.A.vel)  # the same arithmetic in the same order
    assert a.nb.builds() == 1 and int(a.nb.flags.sum()) == 1  # every other list word is back at rest


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("name", ["dense_block", "wet_block"])
def test_overflowing_rows_take_their_forces_from_the_cells(name, prec):
    """Lists of two partners overflow for nearly every granule; the forces then
    come from the 27 cells, in the order of the rows: the same state, bit for
    bit, as lists that hold every partner."""
    prob = shuffled(gi.make(name))
    out = []
    for cap in (2, 96):
        sim = Simulator(prob.grid, prob.params, prob.n, prec, verlet_skin=0.15 * float(prob.r.max()), verlet_cap=cap)
        sim.set_fluid(prob.u, prob.vf, prob.wf, prob.p, prob.alpha_f)
        sim.set_state(prob.cell, prob.q, prob.r, prob.v)
        sim.run(1)
        torch.cuda.synchronize()
        assert gic.gic_check_status() == 0
        assert sim.nb.overflowed() == (cap == 2)
        out.append([t.cpu().numpy() for t in sim.positions()])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_crowded_cells_leave_the_staged_tile():
    """More granules per contact cell than the staged neighbourhood holds (a
    contact grid far coarser than the granules): the build takes the cells from
    global memory, with the same result."""
    prob = shuffled(gi.make("dense_block", n_side=(10, 10, 10)))
    coarse = dataclasses.replace(prob.grid, k_contact=1)
    x = prob.positions()
    cell, q = gi.encode_positions(x, coarse)
    crowded = dataclasses.replace(prob, grid=coarse, cell=cell, q=q)
    a = Simulator.from_problem(crowded, FP32)
    b = Simulator.from_problem(crowded, FP32)
    a.substep()
    F = b.fluid
    gic.gic_sort(b.grid, b.A, b.B, b.perm, b.table, b.ws)
    gic.gic_substep(b.grid, b.params, b.B, b.table, b.nb, F.u, F.v, F.w, F.p, F.alpha_f, b.A, None, b.alpha_s, b.Fs,
                    b.sums)
    torch.cuda.synchronize()
    assert gic.gic_check_status() == 0
    assert torch.equal(a.A.pos, b.A.pos) and torch.equal(a.A.vel, b.A.vel)
