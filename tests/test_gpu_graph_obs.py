"""Counting observables of +-1 graphs (graph_obs_kernel, graph_obs_hub_kernel) against numpy sums over
the edges: a single vertex, odd group counts, more groups than a block keeps totals for (direct atomics),
counters that must be flushed before they overflow (degrees up to 255, several vertices a thread), hubs in
both directions, fields (constant and per vertex)."""
import numpy as np
import pytest

from oracle import core
from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


@pytest.mark.parametrize("n,deg,R,lam_c,lam_sd", [
    (1, 0.0, 32, 0.0, 0.0), (333, 7.0, 96, 0.25, 0.0), (3000, 340.0, 2080, 0.0, 0.0), (900, 12.0, 2048, 0.0, 0.1)])
def test_observables_equal_edge_sums(S, n, deg, R, lam_c, lam_sd):
    u, v = W.erdos_renyi(n, deg, 7 + n) if n > 1 else (np.zeros(0, np.int32),) * 2
    if n == 900:  # one hub that all others point to, one that points to all others
        hub = np.arange(1, n - 1, dtype=np.int32)
        u = np.concatenate([u, np.zeros_like(hub), hub])
        v = np.concatenate([v, hub, np.full_like(hub, n - 1)])
    J = W.couplings_pm1(u.size, 8 + n)
    lam = W.fields_normal(n, lam_sd, 9 + n) if lam_sd else None
    q = 0.9
    ctx = S.shaken_init(graph_problem(S, n, u, v, J, R, 0.4, q=q, lam=lam, lam_c=lam_c), 77 + n)
    S.shaken_step(ctx, 1)
    s, p = S.shaken_get_spins(ctx, R, n), S.shaken_get_spins_prime(ctx, R, n)
    o = S.shaken_observables(ctx, R)
    S.shaken_free(ctx)
    tail, head = core.orient(u, v, 0)
    Ji, lf = J.astype(np.int64), np.float64(np.float32(lam_c)) if lam is None else lam.astype(np.float64)
    for r in range(0, R, 32):
        a, b = s[r:r + 32].astype(np.int64), p[r:r + 32].astype(np.int64)
        E, P1 = (Ji * a[:, tail] * a[:, head]).sum(1), (Ji * a[:, tail] * b[:, head]).sum(1)
        cut, L1, L2 = (a[:, tail] != a[:, head]).sum(1), (lf * a).sum(1), (lf * b).sum(1)
        # field sums: fp32 over 32 vertices, fp64 beyond
        tol = 32 * 2.0 ** -24 * np.abs(lf * np.ones(n)).sum() * 4
        w = slice(r, r + 32)
        assert np.array_equal(o["magnetization"][w], a.sum(1) / n) and np.array_equal(o["cut_edges"][w], cut)
        assert np.array_equal(o["cut_weight"][w], 0.5 * (E - Ji.sum()))
        assert np.abs(o["energy"][w] - (-E - 2.0 * L1)).max() <= tol
        pair = -(P1 + q * (a * b).sum(1) + L1 + L2)
        assert np.abs(o["pair_energy"][w] - pair).max() <= tol + 1e-12 * np.abs(pair).max()
