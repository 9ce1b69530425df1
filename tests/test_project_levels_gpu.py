"""gic_project on grids whose finest two or three levels take grid-wide passes (the
rest run in one CTA), with odd extents on every level and several layers per thread
(and a remainder): the FP64 residual of the pressures by the oracle's operator, and
the iteration counts, which a wrong pass on one level raises (a V-cycle of the same
design needs about 11 iterations per refinement step, 22 without its
over-correction).  The number of grid-wide levels is read from the launches of a
call cut short, so that another threshold cannot take this cover away unseen."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from oracle import projection as pj
from paper_2504_00745_gb300 import gic
from test_project_gpu import TOL, grid_of, run_gpu

pytestmark = pytest.mark.gpu


def _levels(shape):
    n = 1
    while max(shape) > 4:
        shape = tuple((s + 1) // 2 for s in shape)
        n += 1
    return n


def _grid_wide_levels(c):
    """A call with one iteration in one refinement step: 4 + 2 (levels - 1) launches of
    set-up, and per system the right-hand side, the iteration (4 per grid-wide level
    + 3), the update and the residual."""
    dev = torch.device("cuda")
    n = int(np.prod(c.shape))
    t = lambda a, dt: torch.as_tensor(a, dtype=dt, device=dev)
    p1, p2 = (torch.empty(n, dtype=torch.float64, device=dev) for _ in range(2))
    params = gic.make_proj_params(c.dt, c.rho_f, c.open_sides, tol=1e-14, inner_tol=1e-10, max_outer=1, max_inner=1)
    before = gic.launch_count()
    gic.gic_project(grid_of(c.shape, c.dx), params, t(c.alpha_s, torch.float64), t(c.alpha_star, torch.float32),
                    *(t(f, torch.float32) for f in (c.u, c.v, c.w)), p1, p2)
    per_system = (gic.launch_count() - before - 4 - 2 * (_levels(c.shape) - 1)) / 2
    return (per_system - 6) / 4


@pytest.mark.parametrize("shape,open_sides,levels", [((45, 43, 41), (0, 0, 0, 0, 0, 1), 2),
                                                     ((83, 85, 81), (0, 1, 0, 0, 0, 1), 3),
                                                     ((131, 121, 118), (0, 0, 0, 0, 0, 1), 3),
                                                     ((5, 9, 2500), (0, 0, 0, 0, 0, 1), 2)])
def test_grid_wide_levels(shape, open_sides, levels):
    c = gi.projection_case(seed=61, shape=shape, open_sides=open_sides)
    assert _grid_wide_levels(c) >= levels
    out, info = run_gpu(c)
    ap = pj.target_fraction(c.alpha_s)
    A, ops = pj.operator(c.shape, ap, c.open_sides)
    rhs = (pj.rhs_velocity(c.shape, c.dx, c.dt, c.rho_f, ops, c.u, c.v, c.w),
           pj.rhs_density(c.dx, c.dt, c.rho_f, ap, c.alpha_star))
    for s, (p, b) in enumerate(zip((out["p1"], out["p2"]), rhs)):
        assert info.converged[s] == 1
        assert np.linalg.norm(b - A @ p) <= 4 * TOL * np.linalg.norm(b) + 1e-12 * np.abs(A).max() * np.abs(p).max()
        if max(shape) < 1000:  # (a long column is worse conditioned)
            assert info.inner[s] <= 16 * info.outer[s]


def test_repeatable_with_grid_wide_levels():
    c = gi.projection_case(seed=62, shape=(45, 43, 41))
    (a, ia), (b, ib) = run_gpu(c), run_gpu(c)
    for k in a:
        assert np.array_equal(a[k], b[k])
    assert list(ia.inner) == list(ib.inner)
