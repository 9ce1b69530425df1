"""gic_check_status on a busy stream sleeps between its looks: the wait costs the
host a small part of its length."""
import time

import pytest
import torch

from paper_2504_00745_gb300 import gic

pytestmark = pytest.mark.gpu


def test_a_status_query_leaves_the_core_alone():
    gic.gic_check_status(clear=True)
    torch.cuda.synchronize()
    torch.cuda._sleep(120_000_000)  # clock cycles: some 60 ms
    wall, cpu = time.perf_counter(), time.thread_time()
    assert gic.gic_check_status() == 0
    wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
    assert wall > 0.04 and cpu < 0.2 * wall
