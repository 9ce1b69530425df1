"""gic_project on long and flat grids, whose passes spread their lanes over layers:
the pressures against the oracle's direct solves within the bound that the final
residual implies, and a column along z at the cost of one along x."""
import time

import numpy as np
import pytest
import scipy.sparse.linalg as spla
import torch

import gic_inputs as gi
from oracle import projection as pj
from test_project_gpu import TOL, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,open_sides", [((3, 2, 700), (0, 0, 0, 0, 0, 1)), ((2, 5, 513), (0, 1, 0, 0, 1, 0)),
                                              ((1, 37, 260), (0, 0, 1, 0, 0, 0)), ((70, 1, 130), (0, 0, 0, 0, 1, 0)),
                                              ((5, 300, 9), (0, 0, 0, 1, 0, 0))])
def test_columns_and_plates_match_the_oracle(shape, open_sides):
    c = gi.projection_case(seed=51, shape=shape, open_sides=open_sides)
    ref = pj.project(c.shape, c.dx, c.alpha_s, c.alpha_star, c.u, c.v, c.w, c.dt, c.rho_f, c.open_sides)
    out, info = run_gpu(c)
    A = ref["A"]
    lmin = spla.eigsh(A.tocsc(), k=1, sigma=0, which="LM", return_eigenvectors=False)[0]
    for s, (p_key, b_key) in enumerate((("p1", "b1"), ("p2", "b2"))):
        b, p = ref[b_key], out[p_key]
        assert info.converged[s] == 1
        res = np.linalg.norm(b - A @ p)
        assert res <= 4 * TOL * np.linalg.norm(b) + 1e-12 * np.abs(A).max() * np.abs(p).max()
        assert np.linalg.norm(p - ref[p_key]) <= res / lmin * 1.01 + 1e-12 * np.linalg.norm(ref[p_key])


def test_a_column_costs_the_same_along_every_axis():
    """One cell wide, 20,000 long: along z within twice its time along x (4.2 times
    when all the lanes were spread over rows)."""
    took = []
    for shape, open_sides in (((20000, 1, 1), (0, 1, 0, 0, 0, 0)), ((1, 1, 20000), (0, 0, 0, 0, 0, 1))):
        c = gi.projection_case(seed=52, shape=shape, open_sides=open_sides)
        times = []
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            _, info = run_gpu(c)
            times.append((time.perf_counter() - t) / sum(info.inner))
        took.append(sorted(times)[3])
    assert took[1] <= 2 * took[0]
