"""Distinct contexts are independent: two host threads step contexts of different sizes at the same time,
thousands of short whole runs each (kernels that hold the state in shared memory, of a size that is the
context's own), without an error and with the trajectories of the contexts alone."""
import threading

import numpy as np
import pytest

from paper_1904_06257_gb300 import workloads as W
from tests.gpu_util import graph_problem, lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    require_cuda()
    return lib()


def graph(S, n):
    u, v = W.erdos_renyi(n, 6.0, n)
    return graph_problem(S, n, u, v, W.couplings_pm1(u.size, n + 1), 32, 0.9), 32, n


def lattice(S, enc, L):
    R = 32 if enc == S.MULTISPIN else 1
    return lattice_problem(S, enc, L, R, 0.44), R, L * L


@pytest.mark.parametrize("kind", ["graph", "multispin", "int8"])
def test_two_threads_with_contexts_of_different_sizes(S, kind):
    import torch
    if kind == "graph":
        probs = [graph(S, 500), graph(S, 8000)]
    elif kind == "multispin":
        probs = [lattice(S, S.MULTISPIN, 32), lattice(S, S.MULTISPIN, 128)]
    else:
        probs = [lattice(S, S.INT8, 32), lattice(S, S.INT8, 352)]
    calls, steps = 1000, 8

    def run(p, R, n, stream):
        c = S.shaken_init(p, 77, stream)
        for k in range(calls):
            if k % 100 == 50:  # a rebuilt plan asks for its shape again
                S.shaken_set_tracking(c, k % 200 == 50)
            S.shaken_step(c, steps)
        spins = S.shaken_get_spins(c, R, n)
        S.shaken_free(c)
        return spins

    alone = [run(p, R, n, None) for p, R, n in probs]
    streams = [torch.cuda.Stream() for _ in probs]
    got, errors = [None, None], []

    def work(k):
        try:
            got[k] = run(*probs[k], streams[k])
        except Exception as e:  # noqa: BLE001 -- reported below
            errors.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for a, b in zip(got, alone):
        assert np.array_equal(a, b)
