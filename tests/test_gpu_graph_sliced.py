"""The bit-sliced +-1 graph half steps (one inverse temperature, at most 32 threshold classes per vertex)
against the oracle, both as half-step kernels (graph_sliced_kernel) and as whole runs of small graphs in
thread-block clusters (graph_cluster_kernel): every group-word width (1 to 4 words per thread,
rows that leave idle threads), collapsed (q = 1) and two-index classes, degrees on both sides of the
limit, fields, frozen vertices, both orders, and the fused best energies (integers, so equal)."""
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


# degree 20: in-degrees 0 .. ~35 (classes beyond 32 go to the general kernel); beta from 0: T = 2^31 on every
# class, so every lane of the first step is decided by the queue; 288 replicas = 9 groups (1 word per thread, 16
# threads per vertex), 384 = 12 groups (4 words, 3 of 4 threads)
@pytest.mark.parametrize("n,deg,R,q,lam_sd,frozen,reversed_", [
    (1, 0.0, 32, 1.0, 0.0, False, False),
    (300, 3.0, 32, 1.0, 0.0, False, False),
    (257, 20.0, 64, 1.0, 0.0, True, False),
    (300, 8.0, 128, 2.5, 0.0, False, True),
    (129, 20.0, 288, 0.7, 0.3, False, False),
    (200, 6.0, 384, 1.0, 0.2, True, True),
    (40, 60.0, 128, 1.0, 0.0, False, False),
    (900, 9.0, 160, 1.0, 0.0, False, False),
    (700, 5.0, 64, 0.4, 0.2, False, False),
])
@pytest.mark.parametrize("path", ["anneal", "half_steps"])
def test_sliced_steps_bit_exact(S, n, deg, R, q, lam_sd, frozen, reversed_, path):
    u, v = W.erdos_renyi(n, min(deg, n - 1.0), 50 + n) if n > 1 else (np.zeros(0, np.int32),) * 2
    J = W.couplings_pm1(u.size, 51 + n)
    lam = W.fields_normal(n, lam_sd, 52 + n) if lam_sd else np.zeros(n, np.float32)
    f = (np.arange(n) % 7 == 3).astype(np.uint8) if frozen else None
    # a batch that times its kernels runs half step by half step; there beta is the context's own
    sched = np.concatenate([[0.0], W.linear_schedule(0.2, 2.5, 4)]) if path == "anneal" else np.full(4, n % 3 * 0.7)
    seed = 0x5348414B + 31 * n
    ctx = S.shaken_init(graph_problem(S, n, u, v, J, R, sched[0], q=q, lam=lam if lam_sd else None, frozen=f), seed)
    s0 = S.shaken_get_spins(ctx, R, n)
    S.shaken_set_order(ctx, reversed_)
    if path == "anneal":
        S.shaken_anneal(ctx, sched)
    else:
        S.shaken_set_tracking(ctx, True)
        batch = S.shaken_batch_create()
        S.shaken_batch_add(batch, ctx)
        S.shaken_batch_set_timing(batch, 1)
        S.shaken_batch_step(batch, 3, False)
        S.shaken_batch_set_timing(batch, 0)  # the rest as one run
        S.shaken_batch_step(batch, 1, False)
    got, obs = S.shaken_get_spins(ctx, R, n), S.shaken_observables(ctx, R)
    S.shaken_free(ctx)
    if path != "anneal":
        S.shaken_batch_free(batch)
    tail, head = core.orient(u, v, 0)
    Jd, ld = J.astype(np.float64), lam.astype(np.float64)
    o, best = s0, np.full(R, np.inf)
    for t, b in enumerate(sched):
        best = np.minimum(best, [x["H"] for x in core.graph_observables(o, o, tail, head, Jd, ld, q)])
        for half in ((1, 0) if reversed_ else (0, 1)):
            o = core.graph_half(o, tail, head, Jd, True, ld, q, b, seed, t, half, frozen=f, draw=core.DRAW_PLANE)
    assert np.array_equal(got, o)
    best = np.minimum(best, [x["H"] for x in core.graph_observables(o, o, tail, head, Jd, ld, q)])
    if lam_sd == 0.0:
        assert np.array_equal(obs["best_energy"], best)
    else:  # fp32 sums of the fields: at most one rounding of 2^-24 per edge and vertex of the running sum
        tol = (n + u.size) * 2.0 ** -24 * (u.size + 2.0 * np.abs(ld).sum())
        assert np.abs(obs["best_energy"] - best).max() <= tol


@pytest.mark.parametrize("n,R", [(333, 32), (5000, 96), (20000, 32)])
def test_recorded_run_of_small_graph(S, n, R):
    """m and H of every step from a whole run in clusters: one pass of vertices, several, a block's share
    beyond one word per thread; the end state against the oracle's edge sums."""
    u, v = W.erdos_renyi(n, 6.0, n)
    J = W.couplings_pm1(u.size, n + 1)
    a, b = [S.shaken_init(graph_problem(S, n, u, v, J, R, 0.8), 17 + n) for _ in range(2)]
    m, H = S.shaken_step_record(a, 6, R)
    for k in range(6):
        s = S.shaken_get_spins(b, R, n).astype(np.int64)
        assert np.array_equal(m[k], s.sum(1) * (1.0 / n))
        assert np.array_equal(H[k], -(J.astype(np.int64) * s[:, u] * s[:, v]).sum(1))
        S.shaken_step(b, 1)
    assert np.array_equal(S.shaken_get_spins(a, R, n), S.shaken_get_spins(b, R, n))
    S.shaken_free(a)
    S.shaken_free(b)
