"""Runs of small INT8 / PACKED lattices whose draws are compared ahead of the run (lattice_ahead_kernel,
lattice_follow_kernel) against the oracle: every ring depth and one to four words a thread, four and six field
classes, saturated thresholds, a frozen frame, both orders, runs longer than a chunk of outcome words, and
replicas enough to shorten the chunk; m and H recorded, best energies, anneals."""
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


@pytest.mark.parametrize("enc,L,R,q,lam,beta,frozen,order,n", [
    ("INT8", 32, 1, 1.0, 0.0, 0.40, False, 0, 260), ("PACKED", 32, 3, 0.5, 0.01, 0.7, True, 1, 260),
    ("INT8", 64, 2, 4.0, 0.15, 8.0, False, 0, 40), ("PACKED", 96, 1, 1.0, 0.0, 0.4407, True, 0, 12),
    ("INT8", 160, 1, 2.0, 0.0, 0.48, True, 1, 9), ("PACKED", 192, 1, 1.0, 0.15, 0.48, False, 1, 7),
    ("INT8", 320, 1, 0.5, 0.0, 0.4407, False, 0, 5), ("PACKED", 352, 1, 1.0, 0.0, 0.48, False, 0, 5),
    ("INT8", 352, 1, 2.0, 0.01, 0.48, False, 1, 5)])
def test_ahead_runs_follow_oracle(S, enc, L, R, q, lam, beta, frozen, order, n):
    fz = W.frozen_frame(L) if frozen else None
    seed, J = 77 + L + R, 1.0
    ctx = S.shaken_init(lattice_problem(S, getattr(S, enc), L, R, beta, J, q, lam, fz), seed)
    S.shaken_set_order(ctx, order)
    o = core.lattice_init(L, R, seed, core.MODE_SINGLE, 0, fz)
    prime, t, best, at = o, 0, np.full(R, np.inf), np.zeros(R)
    halves = (1, 0) if order else (0, 1)

    def step(b):
        nonlocal o, prime, t
        prime = core.lattice_half(o, J, q, lam, b, seed, t, halves[0], core.MODE_SINGLE, fz)
        o = core.lattice_half(prime, J, q, lam, b, seed, t, halves[1], core.MODE_SINGLE, fz)
        t += 1

    def energies():
        return core.lattice_observables(o, prime, J, q, lam)

    def check():
        assert np.array_equal(S.shaken_get_spins(ctx, R, L * L).reshape(R, L, L), o)
        assert np.array_equal(S.shaken_get_spins_prime(ctx, R, L * L).reshape(R, L, L), prime)

    for k in (4, 1):  # whole run, half-step kernels
        S.shaken_step(ctx, k)
        for _ in range(k):
            step(beta)
        check()
    m, H = S.shaken_step_record(ctx, n, R)
    for k in range(n):
        x = energies()
        assert np.array_equal(m[k], [v["M"] * (1.0 / (L * L)) for v in x])
        assert np.allclose(H[k], [v["H"] for v in x], rtol=1e-12, atol=0)
        at = np.where(H[k] < best, t, at)
        best = np.minimum(best, H[k])
        step(beta)
    check()
    schedule = W.linear_schedule(0.1, 3.0, 6)
    S.shaken_anneal(ctx, schedule)
    for b in schedule:
        h = np.array([v["H"] for v in energies()])
        at = np.where(h < best, t, at)
        best = np.minimum(best, h)
        step(float(b))
    check()
    obs = S.shaken_observables(ctx, R)  # counts sigma_t of the last step, too
    h = np.array([v["H"] for v in energies()])
    assert np.allclose(obs["energy"], h, rtol=1e-12, atol=0)
    at = np.where(h < best, t, at)
    assert np.allclose(obs["best_energy"], np.minimum(best, h), rtol=1e-12, atol=0)
    assert np.array_equal(obs["best_step"], at)
    S.shaken_free(ctx)


def test_ahead_chunk_of_many_replicas(S):
    """Replicas enough that a chunk of outcome words holds fewer steps than the run: equal to the same
    steps taken one at a time by the half-step kernels."""
    L, R, n = 352, 12, 40
    p = lattice_problem(S, S.PACKED, L, R, 0.48, 1.0, 0.5, 0.0, None)
    a, b = S.shaken_init(p, 9), S.shaken_init(p, 9)
    S.shaken_step(a, n)
    for _ in range(n):
        S.shaken_step(b, 1)
    assert np.array_equal(S.shaken_get_spins(a, R, L * L), S.shaken_get_spins(b, R, L * L))
    assert np.array_equal(S.shaken_get_spins_prime(a, R, L * L), S.shaken_get_spins_prime(b, R, L * L))
    S.shaken_free(a)
    S.shaken_free(b)
