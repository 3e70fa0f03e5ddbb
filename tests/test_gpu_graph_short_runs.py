"""Small +-1 graphs stepped a few steps at a time: a call too short to pay for the set-up of a whole run goes to the
half-step kernels, and calls of any length mix in one trajectory, alone and in a batch with lattices."""
import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


def problem(S, n, R, deg=6.0):
    u, v = W.erdos_renyi(n, deg, n)
    return graph_problem(S, n, u, v, W.couplings_pm1(u.size, n + 1), R, 0.9)


@pytest.mark.parametrize("n,R", [(2000, 32), (8000, 32)])
def test_single_steps_take_the_half_step_kernels(S, n, R):
    c = S.shaken_init(problem(S, n, R), 5)
    at = S.shaken_launch_count(c)
    for _ in range(5):
        S.shaken_step(c, 1)
    assert S.shaken_launch_count(c) - at == 5 * 3  # two half steps and the epilogue each
    at = S.shaken_launch_count(c)
    S.shaken_step(c, 200)
    assert S.shaken_launch_count(c) - at < 200  # whole runs
    for k in (2, 1, 40, 3):
        S.shaken_step(c, k)
    spins = S.shaken_get_spins(c, R, n)
    S.shaken_free(c)
    c = S.shaken_init(problem(S, n, R), 5)
    S.shaken_step(c, 251)
    assert S.shaken_get_step(c) == 251
    assert np.array_equal(S.shaken_get_spins(c, R, n), spins)
    S.shaken_free(c)
