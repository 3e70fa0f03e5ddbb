"""Whole runs in one launch per chunk: what a call promises besides its trajectory (it returns before the GPU is done
where the header says so, counts every kernel it launches, leaves a countable state when a chunk is refused), and what
is carried over the end of a chunk: m, H, best energies and their steps, against the same steps taken one at a time
by the half-step kernels."""
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


def refusable(S, kind):
    """Problem, replicas, sites, steps of the run, chunks issued before the refused one."""
    if kind == "graph":
        n = 500
        u, v = W.erdos_renyi(n, 6.0, 3)
        return graph_problem(S, n, u, v, W.couplings_pm1(u.size, 4), 32, 0.8), 32, n, 600, 1
    if kind == "real":  # launch graphs of half steps, then single steps
        n = 300
        u, v = W.erdos_renyi(n, 6.0, 3)
        return graph_problem(S, n, u, v, W.couplings_normal(u.size, 4), 32, 0.8, integer=False), 32, n, 100, 4
    if kind == "multispin":
        return lattice_problem(S, S.MULTISPIN, 64, 64, W.beta_grid(64)), 64, 64 * 64, 300, 1
    if kind == "int8":
        return lattice_problem(S, S.INT8, 64, 2, [0.4, 0.5]), 2, 64 * 64, 600, 1
    if kind == "bits":  # half steps on a bit copy of the bytes
        return lattice_problem(S, S.INT8, 512, 2, [0.4, 0.5]), 2, 512 * 512, 100, 2
    return lattice_problem(S, S.INT8, 512, 1, 0.4), 1, 512 * 512, 65536 + 40, 1  # band


@pytest.mark.parametrize("kind", ["graph", "real", "multispin", "int8", "bits", "band"])
def test_refused_chunk_leaves_the_steps_before_it(S, kind):
    """A run that fails in the middle leaves the state of the steps it counts, and goes on from there."""
    p, R, sites, n, after = refusable(S, kind)
    track = kind not in ("band", "real")  # real couplings: energies are sums in a run-dependent order

    def state(c):
        obs = S.shaken_observables(c, R)
        best = [obs["best_energy"], obs["best_step"]] if track else []
        return best + [S.shaken_get_spins(c, R, sites), S.shaken_get_spins_prime(c, R, sites)]

    def alone(pieces):
        c = S.shaken_init(p, 21)
        S.shaken_set_tracking(c, track)
        for k in pieces:
            S.shaken_step(c, k)
            end = state(c)
        S.shaken_free(c)
        return end

    c = S.shaken_init(p, 21)
    S.shaken_set_tracking(c, track)
    S.shaken_debug_refuse_chunk(c, after)
    with pytest.raises(S.ShakenError) as e:
        S.shaken_step(c, n)
    assert e.value.status == -3
    t = S.shaken_get_step(c)
    assert 0 < t < n
    for x, y in zip(state(c), alone([t])):
        assert np.array_equal(x, y)
    S.shaken_step(c, 1)  # the half-step kernels: the device's step counter
    S.shaken_step(c, n - t - 1)
    for x, y in zip(state(c), alone([t, n - t])):  # a best energy may be seen at the stop, too
        assert np.array_equal(x, y)
    S.shaken_free(c)


@pytest.mark.parametrize("kind", ["graph", "multispin", "int8"])
def test_refused_chunk_of_an_anneal_or_a_recorded_run(S, kind):
    """The context neither anneals nor records any more after the error."""
    p, R, sites, n, after = refusable(S, kind)
    sched = W.linear_schedule(0.1, 2.5, n)
    c = S.shaken_init(p, 22)
    S.shaken_debug_refuse_chunk(c, after)
    with pytest.raises(S.ShakenError):
        S.shaken_anneal(c, sched)
    t = S.shaken_get_step(c)
    S.shaken_debug_refuse_chunk(c, after)
    with pytest.raises(S.ShakenError):
        S.shaken_step_record(c, n, R)
    t2 = S.shaken_get_step(c) - t
    assert 0 < t < n and 0 < t2 < n
    S.shaken_step(c, 7)
    best = S.shaken_observables(c, R)["best_step"]
    assert np.all((best < t + t2) | (best == t + t2 + 7))  # not tracked after the error
    spins = S.shaken_get_spins(c, R, sites)
    S.shaken_free(c)
    c = S.shaken_init(p, 22)
    S.shaken_anneal(c, sched[:t])
    S.shaken_step(c, t2 + 7)
    assert np.array_equal(S.shaken_get_spins(c, R, sites), spins)
    S.shaken_free(c)


@pytest.mark.parametrize("after", [1, 4])
def test_refused_chunk_of_a_batch(S, after):
    """Graph clusters go first (three chunks of 600 steps), then the lattices: each member's own count."""
    members = [refusable(S, "graph"), refusable(S, "int8")]
    n = 600
    b = S.shaken_batch_create()
    ctxs = []
    for k, m in enumerate(members):
        c = S.shaken_init(m[0], 30 + k)
        S.shaken_batch_add(b, c)
        ctxs.append(c)
    S.shaken_debug_refuse_chunk(ctxs[0], after)
    with pytest.raises(S.ShakenError):
        S.shaken_batch_step(b, n, False)
    t = [S.shaken_get_step(c) for c in ctxs]
    assert t == ([256, 0] if after == 1 else [600, 1])
    S.shaken_batch_step(b, 1, False)
    S.shaken_batch_step(b, 50, True)
    for k, (c, m) in enumerate(zip(ctxs, members)):
        assert S.shaken_get_step(c) == t[k] + 51
        ref = S.shaken_init(m[0], 30 + k)
        S.shaken_step(ref, t[k] + 51)
        assert np.array_equal(S.shaken_get_spins(c, m[1], m[2]), S.shaken_get_spins(ref, m[1], m[2]))
        S.shaken_free(ref)
        S.shaken_free(c)
    S.shaken_batch_free(b)


def small_problem(S, kind):
    if kind == "graph":
        n = 500
        u, v = W.erdos_renyi(n, 6.0, 3)
        return graph_problem(S, n, u, v, W.couplings_pm1(u.size, 4), 32, 0.8), 32, n
    if kind == "multispin":
        return lattice_problem(S, S.MULTISPIN, 64, 64, W.beta_grid(64)), 64, 64 * 64
    return lattice_problem(S, S.INT8 if kind == "int8" else S.PACKED, 64, 2, [0.4, 0.5], q=0.7), 2, 64 * 64


@pytest.mark.parametrize("kind", ["graph", "multispin", "int8", "packed"])
def test_recorded_runs_across_chunks_equal_single_steps(S, kind):
    n = 300  # chunks of 128 or 256 steps
    p, R, sites = small_problem(S, kind)
    c = S.shaken_init(p, 11)
    S.shaken_step(c, 3)
    m, H = S.shaken_step_record(c, n, R)
    end = S.shaken_observables(c, R), S.shaken_get_spins(c, R, sites), S.shaken_get_spins_prime(c, R, sites)
    S.shaken_free(c)
    c = S.shaken_init(p, 11)
    S.shaken_step(c, 3)
    for k in range(n):
        m1, H1 = S.shaken_step_record(c, 1, R)
        assert np.array_equal(m1[0], m[k]) and np.array_equal(H1[0], H[k]), k
    ref = S.shaken_observables(c, R), S.shaken_get_spins(c, R, sites), S.shaken_get_spins_prime(c, R, sites)
    S.shaken_free(c)
    for f in ("energy", "pair_energy", "best_energy", "best_step"):
        assert np.array_equal(end[0][f], ref[0][f]), f
    assert np.array_equal(end[1], ref[1]) and np.array_equal(end[2], ref[2])
    low = np.minimum(H.min(axis=0), ref[0]["energy"])
    assert np.array_equal(ref[0]["best_energy"], low)
    first = np.where(H.min(axis=0) <= low, 3 + H.argmin(axis=0), n + 3)
    assert np.array_equal(ref[0]["best_step"], first)


@pytest.mark.parametrize("kind", ["graph", "multispin", "int8", "packed"])
def test_anneals_across_chunks_equal_single_steps(S, kind):
    """Best energy and its step of an anneal of 300 steps against 300 anneals of one step each."""
    p, R, sites = small_problem(S, kind)
    sched = W.linear_schedule(0.1, 2.5, 300)
    ends = []
    for pieces in ([sched], [[b] for b in sched]):
        c = S.shaken_init(p, 12)
        for s in pieces:
            S.shaken_anneal(c, s)
        obs = S.shaken_observables(c, R)
        ends.append((obs["best_energy"], obs["best_step"], S.shaken_get_spins(c, R, sites)))
        S.shaken_free(c)
    for a, b in zip(*ends):
        assert np.array_equal(a, b)
