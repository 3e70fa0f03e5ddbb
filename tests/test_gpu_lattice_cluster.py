"""Whole runs of small MULTISPIN lattices in one thread-block cluster per group (lattice_cluster_kernel) against
the oracle: every cluster size (one block to sixteen, by side and number of groups), sides that are no powers
of two, both orders, a frozen frame, collapsed and six-class tables; recorded m and H, best energies, anneals;
runs alternate with the per-half-step kernels (chunks of fewer than four steps)."""
import numpy as np
import pytest

from oracle import core
from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


# short: four steps only (the oracle makes 32 Philox calls an update)
@pytest.mark.parametrize("L,R,q,lam,frozen,order,short", [
    (32, 32, 1.0, 0.0, False, 0, False), (32, 2464, 1.0, 0.0, False, 0, True), (64, 64, 0.1, 0.15, False, 1, False),
    (96, 32, 1.0, 0.0, True, 0, False), (128, 32, 0.7, 0.02, True, 1, False), (160, 32, 1.0, 0.0, False, 0, True),
    (224, 32, 2.0, 0.0, False, 0, True)])
def test_cluster_runs_follow_oracle(S, L, R, q, lam, frozen, order, short):
    fz = W.frozen_frame(L) if frozen else None
    beta = W.beta_grid(R, 0.3, 1.3, 7)
    seed, J = 515 + L + R, 1.0
    ctx = S.shaken_init(lattice_problem(S, S.MULTISPIN, L, R, beta, J, q, lam, fz), seed)
    S.shaken_set_order(ctx, order)
    keep = slice(max(0, R - 32), R)  # the oracle steps the last group (its own lane words)
    o = core.lattice_init(L, R, seed, core.MODE_MULTISPIN, 0, fz)
    prime, t, best = o, 0, np.full(R, np.inf)
    halves = (1, 0) if order else (0, 1)

    def step(b):
        nonlocal o, prime, t
        prime = core.lattice_half(o, J, q, lam, b, seed, t, halves[0], core.MODE_MULTISPIN, fz)
        o = core.lattice_half(prime, J, q, lam, b, seed, t, halves[1], core.MODE_MULTISPIN, fz)
        t += 1

    def check():
        assert np.array_equal(S.shaken_get_spins(ctx, R, L * L).reshape(R, L, L)[keep], o[keep])
        assert np.array_equal(S.shaken_get_spins_prime(ctx, R, L * L).reshape(R, L, L)[keep], prime[keep])

    for n in (4,) if short else (4, 1, 5):  # cluster, tiled, cluster
        S.shaken_step(ctx, n)
        for _ in range(n):
            step(beta)
        check()
    if short:
        S.shaken_free(ctx)
        return
    m, H = S.shaken_step_record(ctx, 4, R)
    for k in range(4):
        x = core.lattice_observables(o[keep], prime[keep], J, q, lam)
        assert np.array_equal(m[k, keep], [v["M"] * (1.0 / (L * L)) for v in x])
        assert np.allclose(H[k, keep], [v["H"] for v in x], rtol=1e-12, atol=0)
        best[keep] = np.minimum(best[keep], H[k, keep])
        step(beta)
    check()
    sched = np.linspace(0.2, 1.5, 5)
    S.shaken_anneal(ctx, sched)
    for b in sched:
        best[keep] = np.minimum(best[keep], [v["H"] for v in core.lattice_observables(o[keep], prime[keep], J, q, lam)])
        step(b)
    check()
    obs = S.shaken_observables(ctx, R)[keep]
    S.shaken_free(ctx)
    best[keep] = np.minimum(best[keep], [v["H"] for v in core.lattice_observables(o[keep], prime[keep], J, q, lam)])
    assert np.allclose(obs["best_energy"], best[keep], rtol=1e-12, atol=0)
