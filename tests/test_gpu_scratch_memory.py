"""Scratch of a run on a nearly full device: the run leaves its caller most of the free memory, and gives the same
trajectory without the scratch."""
import numpy as np
import pytest

from tests.gpu_util import lattice_problem, lib, require_cuda

pytestmark = pytest.mark.gpu


def test_bit_copy_leaves_most_of_the_free_memory():
    require_cuda()
    S = lib()
    import torch
    L, R, steps = 8192, 16, 8
    p = lattice_problem(S, S.INT8, L, R, 0.44)
    c = S.shaken_init(p, 9)
    S.shaken_step(c, steps)  # on the bit copy: a quarter of sigma's bytes, 256 MB
    ref = S.shaken_get_spins(c, R, L * L)
    S.shaken_free(c)
    c = S.shaken_init(p, 9)
    S.shaken_step(c, 1)  # plans and launch shapes
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    block = 1 << 25
    filler = torch.empty((torch.cuda.mem_get_info()[0] - (512 << 20)) // block * block, dtype=torch.uint8,
                         device="cuda")
    free = torch.cuda.mem_get_info()[0]
    S.shaken_step(c, steps - 1)
    S.shaken_sync(c)
    left = torch.cuda.mem_get_info()[0]
    del filler
    torch.cuda.empty_cache()
    got = S.shaken_get_spins(c, R, L * L)
    S.shaken_free(c)
    assert np.array_equal(got, ref)
    assert left >= 0.7 * free  # less a quarter at most, and the allocator's granularity
