"""INT8 runs of the half-step kernels on the bit copy of the state against the same steps taken one at a time on the
bytes, and against a PACKED context (the same draws): tails of tiles, several replicas, a frozen frame, both
orders, CUDA-graph replay, annealed and recorded runs."""
import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


@pytest.mark.parametrize("L,R,q,lam,frozen,order,n", [
    (384, 33, 1.0, 0.0, False, 0, 9), (416, 32, 0.5, 0.01, True, 1, 7), (1024, 4, 2.0, 0.0, False, 0, 70),
    (2976, 2, 1.0, 0.15, False, 1, 2)])
def test_bit_copy_runs(S, L, R, q, lam, frozen, order, n):
    fz = W.frozen_frame(L) if frozen else None
    a, b, p = (S.shaken_init(lattice_problem(S, e, L, R, 0.45, 1.0, q, lam, fz), 11) for e in (S.INT8, S.INT8, S.PACKED))
    for c in (a, b, p):
        S.shaken_set_order(c, order)

    def same():
        for get in (S.shaken_get_spins, S.shaken_get_spins_prime):
            x = get(a, R, L * L)
            assert np.array_equal(x, get(b, R, L * L)) and np.array_equal(x, get(p, R, L * L))

    S.shaken_step(a, n)
    S.shaken_step(p, n)
    for _ in range(n):
        S.shaken_step(b, 1)
    same()
    x = [S.shaken_step_record(c, 8, R) for c in (a, p)]
    y = [S.shaken_step_record(b, 1, R) for _ in range(8)]
    assert np.array_equal(x[0][0], x[1][0]) and np.array_equal(x[0][0], np.concatenate([m for m, _ in y]))
    assert np.array_equal(x[0][1], x[1][1]) and np.array_equal(x[0][1], np.concatenate([h for _, h in y]))
    same()
    schedule = W.linear_schedule(0.2, 1.0, 5)
    for c in (a, p):
        S.shaken_anneal(c, schedule)
    for k in range(5):
        S.shaken_anneal(b, schedule[k:k + 1])
    same()
    o = [S.shaken_observables(c, R) for c in (a, b, p)]
    for f in ("magnetization", "energy", "pair_energy", "best_energy", "best_step"):
        assert np.array_equal(o[0][f], o[1][f]) and np.array_equal(o[0][f], o[2][f])
    for c in (a, b, p):
        S.shaken_free(c)
