"""Whole runs of small +-1 graphs in thread-block clusters, their draws compared ahead (graph_thresholds_kernel,
graph_ahead_kernel, graph_cluster_kernel), against the half-step kernels (a batch that times its kernels runs
half step by half step): cluster sizes by vertices and groups, runs longer than a chunk of outcome words, a
constant field, saturated thresholds, frozen vertices, both orders, graphs of different sizes in one batch."""
import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


# per batch member: n, mean degree, replicas, q, constant field, beta
@pytest.mark.parametrize("members,order,n", [
    ([(33, 2.0, 32, 1.0, 0.0, 0.9)], 0, 300), ([(2500, 6.0, 64, 1.0, 0.0, 5.0)], 1, 300),
    ([(1200, 4.0, 32, 2.5, 0.3, 0.7)], 0, 40), ([(9000, 5.0, 32, 1.0, -0.2, 40.0)], 0, 70),
    ([(700, 6.0, 32, 1.0, 0.0, 0.0), (2000, 7.0, 160, 0.5, 0.0, 1.0), (31, 3.0, 96, 1.0, 0.0, 2.0)], 1, 33),
    ([(640, 5.0, 1024, 1.0, 0.0, 1.0)], 0, 12)])
def test_cluster_runs_equal_half_steps(S, members, order, n):
    ends = []
    for timed in (0, 1):
        ctxs, batch = [], S.shaken_batch_create()
        for k, (nv, deg, R, q, lam, beta) in enumerate(members):
            u, v = W.erdos_renyi(nv, deg, nv)
            f = (np.arange(nv) % 11 == 5).astype(np.uint8) if k == 0 else None
            c = S.shaken_init(graph_problem(S, nv, u, v, W.couplings_pm1(u.size, nv + 1), R, beta, q=q, lam_c=lam,
                                            frozen=f), 5 + k)
            S.shaken_set_order(c, order)
            S.shaken_batch_add(batch, c)
            ctxs.append(c)
        S.shaken_batch_set_timing(batch, timed)
        S.shaken_batch_step(batch, n, False)
        S.shaken_batch_step(batch, 3, False)
        ends.append([get(c, m[2], m[0]) for c, m in zip(ctxs, members)
                     for get in (S.shaken_get_spins, S.shaken_get_spins_prime)])
        for c in ctxs:
            S.shaken_free(c)
        S.shaken_batch_free(batch)
    for a, b in zip(*ends):
        assert np.array_equal(a, b)
