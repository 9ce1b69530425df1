"""The checkpoints of a differentiable window keep one copy of the list rows per
build, not one per checkpoint, and the gradients are those of one long segment."""
import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP64
from paper_2504_00745_gb300.window import GicWindow, Simulator

pytestmark = pytest.mark.gpu


def test_checkpoints_of_one_build_share_their_rows():
    prob = gi.make("dense_block", n_side=(5, 5, 5))
    K, out = 24, []
    for ckpt in (4, K):
        sim = Simulator.from_problem(prob, FP64)
        v0 = torch.tensor(prob.v, dtype=torch.float64, device="cuda", requires_grad=True)
        c, mu = (torch.tensor(float(q), dtype=torch.float64, device="cuda", requires_grad=True)
                 for q in (prob.params.c_drag, prob.params.mu_fric))
        x = GicWindow.apply(v0, c, mu, sim, sim.A.clone(), K, ckpt)
        ctx = x.grad_fn
        if ckpt < K:
            builds = [w[4] for w in ctx.words[1:-1]]  # at every checkpoint after the first
            copies = {id(q["arrays"]) for q in ctx.lists[1:]}
            assert ctx.lists[0]["arrays"] is None and len(builds) == 5
            assert len(copies) == len(set(builds)) < len(builds)
        (x ** 2).sum().backward()
        out.append([t.grad.cpu().numpy() for t in (v0, c, mu)])
    for a, b in zip(*out):  # (c and mu: double atomics in another order)
        assert np.allclose(a, b, rtol=1e-10, atol=1e-12 * np.abs(b).max())
