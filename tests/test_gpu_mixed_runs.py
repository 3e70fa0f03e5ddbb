"""Graphs in whole-run clusters beside other work: batches with lattices and graphs of both routes, tracked and not,
and server jobs that end in the middle of a chunk; every member equals its run alone."""
import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, graph_spins_from_raw, lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


def graph(S, n, R, deg=6.0):
    u, v = W.erdos_renyi(n, deg, n)
    return graph_problem(S, n, u, v, W.couplings_pm1(u.size, n + 1), R, 0.9), R, n


# small: every graph fits a cluster; with a graph of 40000 vertices all go to the half-step kernels
@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("use_graph", [False, True])
def test_batch_of_graphs_and_lattices_equals_alone(S, large, use_graph):
    members = [(graph(S, 700, 32), True), (graph(S, 1500, 64), False),
               ((lattice_problem(S, S.MULTISPIN, 64, 64, W.beta_grid(64)), 64, 64 * 64), True),
               ((lattice_problem(S, S.INT8, 64, 2, [0.4, 0.5]), 2, 64 * 64), False)]
    if large:
        members.append((graph(S, 40000, 32), True))
    pieces = (64, 1, 3, 70, 2)

    def make(k):
        (p, R, n), track = members[k]
        c = S.shaken_init(p, 40 + k)
        S.shaken_set_tracking(c, track)
        return c

    def end(c, k):
        (_, R, n), track = members[k]
        assert S.shaken_get_step(c) == sum(pieces)
        obs = S.shaken_observables(c, R)
        return [obs["energy"], obs["pair_energy"], obs["best_energy"], obs["best_step"], S.shaken_get_spins(c, R, n),
                S.shaken_get_spins_prime(c, R, n)]

    alone = []
    for k in range(len(members)):
        c = make(k)
        S.shaken_step(c, sum(pieces))
        alone.append(end(c, k))
        S.shaken_free(c)
    b = S.shaken_batch_create()
    ctxs = [make(k) for k in range(len(members))]
    for c in ctxs:
        S.shaken_batch_add(b, c)
    for n in pieces:
        S.shaken_batch_step(b, n, use_graph)
    for k, c in enumerate(ctxs):
        for x, y in zip(end(c, k), alone[k]):
            assert np.array_equal(x, y), k
        S.shaken_free(c)
    S.shaken_batch_free(b)


def test_server_jobs_that_end_within_a_chunk(S):
    jobs = []
    for k, (n, R, steps) in enumerate([(500, 32, 100), (900, 64, 37), (2000, 32, 150), (33, 32, 64), (1200, 32, 1)]):
        p, R, n = graph(S, n, R)
        jobs.append((p, 70 + k, W.linear_schedule(0.1, 3.0, steps), R, n))
    srv = S.shaken_server_create(1 << 30, 64)
    S.shaken_server_set_policy(srv, 3e8, 0, keep_states=True)
    ids = [S.shaken_server_submit(srv, p, seed, sched) for p, seed, sched, R, n in jobs]
    S.shaken_server_drain(srv, 120.0)
    for jid, (p, seed, sched, R, n) in zip(ids, jobs):
        res = S.shaken_server_result(srv, jid, R)[0]
        raw = S.shaken_server_result_state(srv, jid, R * n // 8)
        c = S.shaken_init(p, seed)
        S.shaken_anneal(c, sched)
        obs = S.shaken_observables(c, R)
        assert np.array_equal(graph_spins_from_raw(raw, n, R), S.shaken_get_spins(c, R, n))
        for f in ("energy", "pair_energy", "best_energy", "best_step"):
            assert np.array_equal(res[f], obs[f]), f
        S.shaken_free(c)
    S.shaken_server_free(srv)
