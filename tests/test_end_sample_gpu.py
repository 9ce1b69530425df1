"""A granule beyond the last sample of an axis takes that sample's value exactly:
the sample before it does not enter, however large it is."""
import dataclasses

import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _problem(last_but_one):
    """One layer of granules between the last cell centres and the wall in x; the
    face velocities v and w (centred in x) hold last_but_one times noise in the
    samples before the last."""
    base = gi.random_cloud(n=400)
    g = base.grid
    gen = np.random.default_rng(5)
    x = base.positions()
    x[:, 0] = g.origin[0] + (g.nx - 0.5 * gen.uniform(0.05, 0.95, base.n)) * g.dx
    cell, q = gi.encode_positions(x, g)
    fields = []
    for shape in ((g.nz, g.ny + 1, g.nx), (g.nz + 1, g.ny, g.nx)):
        f = gen.uniform(-0.1, 0.1, shape)
        f[:, :, g.nx - 2] = last_but_one * gen.uniform(-1.0, 1.0, shape[:2])
        fields.append(f.ravel())
    return dataclasses.replace(base, cell=cell, q=q, vf=fields[0], wf=fields[1])


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("fused", [True, False])
def test_the_last_sample_stands_alone_beyond_it(prec, fused):
    out = []
    for last_but_one in (0.0, 1e3):
        sim = Simulator.from_problem(_problem(last_but_one), prec, fused=fused)
        if not fused:
            gic.gic_sort(sim.grid, sim.A, sim.B, sim.perm, sim.table, sim.ws)
            F = sim.fluid
            gic.gic_g2p_couple(sim.grid, sim.params, sim.B, F.u, F.v, F.w, F.p, F.alpha_f, sim.F_fl, sim.a_f)
            out.append([sim.F_fl.cpu().numpy(), sim.a_f.cpu().numpy()])
        else:
            sim.run(1)
            out.append([t.cpu().numpy() for t in sim.positions()])
    torch.cuda.synchronize()
    gic.gic_check_status(clear=True)
    for a, b in zip(*out):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)
