"""GPU parity of the SQA item walk at the largest problems a block holds: its
slices fill the opt-in shared memory up to the kernel's static part (144 bytes),
for general and for +-1 couplers."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem

pytestmark = pytest.mark.gpu

OPTIN, STATIC = 227 << 10, 144


def _ring(n, jmax, seed):
    g = np.random.default_rng(seed)
    ei = np.arange(n, dtype=np.int32)
    J = (g.integers(1, jmax + 1, n) * (g.integers(0, 2, n) * 2 - 1)).astype(np.int32)
    if jmax > 1:
        J[0] = J[-1] = jmax  # the flip-cost range does not depend on the draw
    return I.Instance("ring", n, ei, ((ei + 1) % n).astype(np.int32), J, np.zeros(n, np.int32))


# spins, largest coupler, slices, shared memory of the walk in words: the two acceptance rows, the slices (and the
# inverted copy), the spins' data, the energy sums
CASES = {"general": (3215, 2, 16, 12 * 9 + 16 * 3216 + 2 * 3215 + 4 * 16 + 4),
         "pm1": (4459, 1, 4, 12 * 5 + 2 * 4 * 4460 + 5 * 4459 + 4 * 4 + 4)}


@pytest.mark.parametrize("name", list(CASES))
def test_walk_fills_the_block(cuda_lib, name):
    spvar = cuda_lib
    n, jmax, P, words = CASES[name]
    assert OPTIN - 256 < 4 * words <= OPTIN - STATIC  # fits with 144 bytes beside it and not with 256
    inst = _ring(n, jmax, 151)
    T, S, seed = 2, 5, 152
    op = oracle_problem(inst)
    ent = spvar.sqa_table(T, P, 2.0, spvar.gamma_linear(T, 2.5, 0.05), O.dmax(op), 1)
    W = ent.shape[2]
    assert W == 4 * jmax + 1
    words_, e, sl = spvar.sqa_sample(gpu_problem(inst), spvar.table_device(ent), W, T, P, S, seed)
    spins, energies, slices = O.sqa_sample(op, ent, P, S, seed)[:3]
    assert np.array_equal(e.cpu().numpy(), energies)
    assert np.array_equal(sl.cpu().numpy(), slices)
    assert np.array_equal(spvar.unpack_spins(words_.cpu().numpy(), n), spins)
