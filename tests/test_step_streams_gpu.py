"""gic_step's cooperative sort and early-launched substep elsewhere than on one ordinary
stream: on several at once, from two host threads on one, on a stream that owns a part
of the SMs, and in a captured graph.  Every simulator must end in the bits that it has
when it runs alone."""
import ctypes as C
import threading

import numpy as np
import pytest
import torch

import gic_inputs as gi
from gpu_util import FP32, FP64, shuffled
from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import Simulator

pytestmark = pytest.mark.gpu


def _problem(n=60_000):
    """A loose cloud whose granules pass skin / 2 every few substeps."""
    prob = shuffled(gi.differentiable_window(n=n, r0=0.002))
    half_skin = 0.5 * 0.05 * float(prob.r.max())
    prob.v[:, 0] = 0.4 * half_skin / prob.params.dt_sub
    return prob


def _result(sim):
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in sim.positions()] + [sim.alpha_s.cpu().numpy()]


def _alone(prob, prec, steps):
    sim = Simulator.from_problem(prob, prec)
    for _ in range(steps):
        sim.substep(sums=False)
    assert sim.nb.builds() > 2
    return _result(sim)


def _same(a, b, prec):
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    if prec == FP32:  # (FP64 sums alpha_s in the order of the atomics)
        assert np.array_equal(a[2], b[2])


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_two_streams_at_once(prec):
    prob, steps = _problem(), 12
    want = _alone(prob, prec, steps)
    sims = [Simulator.from_problem(prob, prec) for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in sims]
    torch.cuda.synchronize()

    def run(sim, stream):
        torch.cuda.set_device(0)
        for _ in range(steps):
            sim.substep(sums=False, stream=stream)

    threads = [threading.Thread(target=run, args=a) for a in zip(sims, streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for sim in sims:
        _same(_result(sim), want, prec)
    assert gic.gic_check_status() == 0


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_two_threads_on_one_stream(prec):
    prob, steps = _problem(), 12
    want = _alone(prob, prec, steps)
    sims = [Simulator.from_problem(prob, prec) for _ in range(2)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def run(sim):
        torch.cuda.set_device(0)
        for _ in range(steps):
            sim.substep(sums=False, stream=stream)

    threads = [threading.Thread(target=run, args=(sim,)) for sim in sims]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for sim in sims:
        _same(_result(sim), want, prec)
    assert gic.gic_check_status() == 0


class _Partition:
    """A stream that owns at least `sms` SMs of device 0 (a green context)."""

    def __init__(self, sms):
        cu = C.CDLL("libcuda.so.1")
        res, part, left = (C.create_string_buffer(512) for _ in range(3))  # CUdevResource, with room
        groups, desc, ctx, self.stream = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()

        def check(rc):
            if rc:
                pytest.skip(f"no SM partition to be had here (CUresult {rc})")

        check(cu.cuDeviceGetDevResource(0, res, 1))  # 1: CU_DEV_RESOURCE_TYPE_SM
        check(cu.cuDevSmResourceSplitByCount(part, C.byref(groups), res, left, 0, sms))
        check(cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1))
        check(cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, 1))  # 1: CU_GREEN_CTX_DEFAULT_STREAM
        check(cu.cuGreenCtxStreamCreate(C.byref(self.stream), ctx, 1, 0))  # 1: CU_STREAM_NON_BLOCKING
        self.close = lambda: (cu.cuStreamDestroy_v2(self.stream), cu.cuGreenCtxDestroy(ctx))


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_a_stream_with_a_part_of_the_sms(prec):
    prob, steps = _problem(), 12
    want = _alone(prob, prec, steps)
    sim = Simulator.from_problem(prob, prec)
    torch.cuda.synchronize()
    part = _Partition(16)
    try:
        stream = torch.cuda.ExternalStream(part.stream.value)
        for _ in range(steps):
            sim.substep(sums=False, stream=stream)
        _same(_result(sim), want, prec)
        assert gic.gic_check_status() == 0
    finally:
        torch.cuda.synchronize()
        part.close()


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("name", ["loose", "wet_block"])
def test_a_captured_call_replays_like_the_direct_one(name, prec):
    """Two gic_step calls (A -> A2 -> A, the second with alpha_s) in a graph: each
    replay decides anew on the device whether it sorts."""
    prob = _problem() if name == "loose" else shuffled(gi.make(name))
    direct, graphed = (Simulator.from_problem(prob, prec) for _ in range(2))

    def pair(sim, stream=None):
        sim.substep(alpha=False, sums=False, stream=stream)
        sim.substep(stream=stream)

    replays = 5
    for _ in range(replays + 1):
        pair(direct)
    pair(graphed)  # (the first call of a process loads the kernels, which a capture may not)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pair(graphed)
    for _ in range(replays):
        graph.replay()
    _same(_result(graphed), _result(direct), prec)
    assert graphed.nb.builds() == direct.nb.builds() and (name != "loose" or direct.nb.builds() > 2)
    assert gic.gic_check_status() == 0
