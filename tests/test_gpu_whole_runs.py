"""Whole runs in one launch per chunk: what a call promises besides its trajectory."""
import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


@pytest.mark.parametrize("L,R,track", [(128, 32, False), (192, 128, True), (32, 64, True)])
def test_multispin_step_returns_before_the_gpu_is_done(S, L, R, track):
    import torch
    stream = torch.cuda.Stream()
    beta = W.beta_grid(R)
    ends = []
    for pieces in ((4, 20000, 1), (1,) * 5 + (20000,)):
        c = S.shaken_init(lattice_problem(S, S.MULTISPIN, L, R, beta), 5, stream)
        S.shaken_set_tracking(c, track)
        for n in pieces:
            S.shaken_step(c, n)
            if n == 20000:
                e = torch.cuda.Event()
                e.record(stream)
                assert not e.query()  # tens of milliseconds of work
        assert S.shaken_get_step(c) == 20005
        obs = S.shaken_observables(c, R)
        ends.append((S.shaken_get_spins(c, R, L * L), obs["best_energy"], obs["best_step"]))
        S.shaken_free(c)
    for a, b in zip(*ends):
        assert np.array_equal(a, b)


def test_launch_count_of_a_cluster_run(S):
    """300 steps of a small MULTISPIN lattice: three launches of at most 128 steps and one that moves the step on."""
    c = S.shaken_init(lattice_problem(S, S.MULTISPIN, 64, 32, 0.5), 5)
    before = S.shaken_launch_count(c)
    S.shaken_step(c, 300)
    assert S.shaken_launch_count(c) - before == 4
    S.shaken_free(c)
