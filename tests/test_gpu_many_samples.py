"""GPU parity of samples of small integer-coupler problems at the most replicas
a call takes: 16 quads per work item past two blocks of 8 per SM, byte and
16-bit lanes, degree 6 and 8, a last item of fewer quads.  Every value equals
the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu


def _ring(n, offsets, scale, seed):
    g = np.random.default_rng(seed)
    ei = np.repeat(np.arange(n), len(offsets)).astype(np.int32)
    ej = ((ei + np.tile(offsets, n)) % n).astype(np.int32)
    J = np.rint(scale * g.standard_normal(len(ei))).astype(np.int32)
    x = I.Instance("ring", n, ei, ej, np.where(J == 0, 1, J).astype(np.int32),
                   np.rint(0.2 * scale * g.standard_normal(n)).astype(np.int32))
    x.scale = scale
    return x


@pytest.mark.parametrize("S", [9728, 9732, 12001, 16384])
@pytest.mark.parametrize("n,offsets,scale", [(27, (1, 2, 5), 6), (27, (1, 2, 5), 100), (31, (1, 2, 5, 9), 6),
                                             (31, (1, 2, 5, 9), 100)], ids=["bytes6", "lanes6", "bytes8", "lanes8"])
def test_sample_equals_oracle(cuda_lib, n, offsets, scale, S):
    spvar = cuda_lib
    inst = _ring(n, offsets, scale, 161)
    assert (O.dmax(oracle_problem(inst)) <= 254) == (scale < 10)
    T, seed = 5, 162
    thr = table(inst, T)
    words, e = spvar.sample(gpu_problem(inst), spvar.thresholds_device(thr), thr.shape[1], T, S, seed)
    spins, energies, _ = O.sample(oracle_problem(inst), thr, S, seed)
    assert np.array_equal(e.cpu().numpy(), energies)
    assert np.array_equal(spvar.unpack_spins(words.cpu().numpy(), n), spins)
