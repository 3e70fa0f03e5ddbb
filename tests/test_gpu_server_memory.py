"""The server's budget bounds all device memory of its running jobs: state and the outcome words of whole runs."""
import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_outcome_words_stay_within_the_budget(S):
    n, R, budget = 2000, 64, 1 << 20  # about four jobs of state
    u, v = W.erdos_renyi(n, 6.0, 7)
    p = graph_problem(S, n, u, v, W.couplings_pm1(u.size, 8), R, 1.0)
    sched = W.linear_schedule(0.2, 2.0, 300)
    c = S.shaken_init(p, 1)  # the kernels' code is loaded outside the measurement, on both routes
    S.shaken_anneal(c, sched)
    ref = S.shaken_observables(c, R)
    S.shaken_free(c)
    b = S.shaken_batch_create()
    c = S.shaken_init(p, 1)
    S.shaken_batch_add(b, c)
    S.shaken_batch_set_timing(b, 1)
    S.shaken_batch_step(b, 40, True)
    S.shaken_free(c)
    S.shaken_batch_free(b)
    before = free_bytes()
    srv = S.shaken_server_create(budget, 256)
    ids = [S.shaken_server_submit(srv, p, s, sched) for s in range(6)]
    S.shaken_server_drain(srv, 120.0)
    held = before - free_bytes()
    assert all(S.shaken_server_poll(srv, i) == 2 for i in ids)
    got = S.shaken_server_result(srv, ids[1], R)[0]  # the job of the same seed
    assert np.array_equal(got["energy"], ref["energy"]) and np.array_equal(got["best_step"], ref["best_step"])
    S.shaken_server_free(srv)
    assert held <= budget + (8 << 20)  # plans, launch graphs and the allocator's granularity
