"""What a reduced problem holds on the device: its own arrays and nothing of the
reduction's working memory."""
import numpy as np
import pytest

from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem

pytestmark = pytest.mark.gpu


def _held(make, count):
    """Device bytes `count` live results of make() take."""
    import torch
    make()  # one-time set-up
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    keep = [make() for _ in range(count)]
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    assert len(keep) == count
    return taken


def test_reduced_problems_hold_no_scratch(cuda_lib):
    spvar = cuda_lib
    import torch
    inst = I.cubic3d(12, 181)
    p = gpu_problem(inst)
    g = np.random.default_rng(182)
    fixed = torch.from_numpy(np.where(g.random(inst.n) < 0.3, 1 - 2 * g.integers(0, 2, inst.n), 0).astype(np.int8)).cuda()
    count = 240
    created = _held(lambda: gpu_problem(inst), count)
    reduced = _held(lambda: spvar.reduce(p, fixed)[0], count)
    # the same capacities as the problem they come from; the working memory would be 12 bytes a spin and 20 KB each
    assert reduced <= created + count * 12 * inst.n // 4
