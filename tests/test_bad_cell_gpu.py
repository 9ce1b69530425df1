"""Granules whose cell ids lie beyond the contact grid (a state that was not made
by gic_pack): the calls flag GIC_STATUS_BAD_CELL and take the paths that clamp to
the grid, the shared-memory tiles of the same CTAs included.  The fused calls
against the separate ones, which read the fields from global memory; the packing
is loose, so that the order of the contact sums does not enter."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64, FS_TOL_FP32, shuffled
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _simulators(prec):
    prob = shuffled(gi.differentiable_window(n=3000, r0=0.002))
    nc = prob.grid.nx * prob.grid.k_contact
    assert nc < 1023
    sims = [Simulator.from_problem(prob, prec), Simulator.from_problem(prob, prec, verlet=False, fused=False)]
    for sim in sims:
        for i, c in ((7, (nc, 20, 20)), (900, (20, nc + 3, 20)), (1500, (20, 20, 1023)), (2999, (1023, 1023, 1023))):
            sim.A.cell[i] = c[0] | c[1] << 10 | c[2] << 20
    gic.gic_check_status(clear=True)
    return sims


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_cells_beyond_the_grid_are_flagged_and_clamped(prec):
    fused, separate = _simulators(prec)
    for step in range(3):  # a call that sorts and builds, and two that keep the lists
        for sim in (fused, separate):
            sim.zero_transfer()
            sim.substep()
        assert step > 0 or gic.gic_check_status(clear=True) & gic.STATUS_BAD_CELL
        for a, b in zip(fused.positions(), separate.positions()):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
        a, b = fused.alpha_s.cpu().numpy(), separate.alpha_s.cpu().numpy()
        # FP64: the same deposits in another order; a sample takes those of 8 cells, 34 granules each
        assert np.array_equal(a, b) if prec == FP32 else np.abs(a - b).max() <= 512 * 2.0 ** -52 * np.abs(b).max()
    gic.gic_check_status(clear=True)


def test_exchange_force_of_a_tile_free_cta():
    """F_s of the first substep, in FP32 against FP64 (no tile for the CTAs that hold
    such granules, the tile for the others)."""
    out = []
    for prec in (FP32, FP64):
        fused, separate = _simulators(prec)
        for sim in (fused, separate):
            sim.zero_transfer()
            sim.substep()
        out.append((fused.Fs, separate.Fs))
    gic.gic_check_status(clear=True)
    for f, want, other in zip(out[0][0], *out[1]):
        f, want, other = f.cpu().numpy(), want.cpu().numpy(), other.cpu().numpy()
        assert np.abs(other - want).max() <= 1e-12 * np.abs(want).max()
        assert np.abs(f - want).max() <= FS_TOL_FP32 * np.abs(want).max()


def test_lists_built_with_cells_beyond_the_grid():
    sim, _ = _simulators(FP32)
    gic.gic_sort(sim.grid, sim.A, sim.B, sim.perm, sim.table, sim.ws)
    gic.gic_neighbors_reset(sim.nb)
    gic.gic_contact_verlet(sim.grid, sim.params, sim.B, sim.table, sim.nb, sim.F_c)  # the 27-cell build
    want = sim.nb.count.clone()
    gic.gic_neighbors_reset(sim.nb)
    gic.gic_neighbors_build(sim.grid, sim.B, sim.table, sim.nb)
    torch.cuda.synchronize()
    assert torch.equal(sim.nb.count, want)
    assert gic.gic_check_status(clear=True) == gic.STATUS_BAD_CELL


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_integration_clamps_cells_beyond_the_grid(prec):
    """A granule at rest in such a cell leaves it for the last cell of the grid,
    and the status says so."""
    _, sim = _simulators(prec)
    nc = sim.grid.nx * sim.grid.k_contact
    sim.A.vel.zero_()
    out = gic.State.empty(sim.n, prec)
    zero = [gic.vec4(sim.n, prec) for _ in range(3)]
    gic.gic_integrate(sim.grid, sim.params, sim.A, *zero, out, sim.f_ex)
    torch.cuda.synchronize()
    assert gic.gic_check_status(clear=True) == gic.STATUS_OUT_OF_DOMAIN
    cell = [int(out.cell[i]) for i in (7, 900, 1500, 2999)]
    last = nc - 1
    assert [c & 1023 for c in cell] == [last, 20, 20, last]
    assert [c >> 10 & 1023 for c in cell] == [20, last, 20, last]
    assert [c >> 20 for c in cell] == [20, 20, last, last]
