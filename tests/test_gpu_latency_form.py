"""GPU parity of the +-1 register kernel's latency form, which grids of at most
one 128-thread block per SM take: one to four sweeping warps, two and three
colour classes, degree 8, biases up to the widest byte-lane row, sweep counts
around its buffers (none, one, part of one, several and a remainder), and a sample
in two sweep ranges.  Everything is a whole number
and equals the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu


def _ring(n, offsets, seed, hmax):
    """+-1 couplers to the given offsets of a ring."""
    g = np.random.default_rng(seed)
    ei = np.repeat(np.arange(n), len(offsets)).astype(np.int32)
    ej = ((ei + np.tile(offsets, n)) % n).astype(np.int32)
    J = (g.integers(0, 2, len(ei)) * 2 - 1).astype(np.int32)
    return I.Instance("ring", n, ei, ej, J, g.integers(-hmax, hmax + 1, n).astype(np.int32))


CASES = {
    "one_warp": lambda: I.cubic3d(4, 801),
    "one_warp_odd": lambda: I.cubic3d(3, 802),
    "two_warps_three_classes": lambda: I.cubic3d(5, 803),
    "four_warps": lambda: I.chimera(5, 804),
    "few_spins": lambda: _ring(6, [1], 805, 2),
    "degree8": lambda: _ring(62, [1, 3, 5, 9], 806, 7),
}


@pytest.mark.parametrize("T", [0, 1, 7, 8, 9, 16, 17, 37])
@pytest.mark.parametrize("name", list(CASES))
def test_sample_equals_oracle(cuda_lib, name, T):
    spvar = cuda_lib
    inst = CASES[name]()
    S, seed = 22, 96
    thr = table(inst, max(T, 1))[:T]
    p, dev = gpu_problem(inst), spvar.thresholds_device(table(inst, max(T, 1)))
    words, e = spvar.sample(p, dev, thr.shape[1], T, S, seed)
    spins, energies, _ = O.sample(oracle_problem(inst), thr, S, seed)
    assert np.array_equal(e.cpu().numpy()[:S], energies)
    assert np.array_equal(spvar.unpack_spins(words.cpu().numpy()[:S], inst.n), spins)
    cut = T // 3
    half, _ = spvar.sample_range(p, dev, thr.shape[1], 0, cut, S, seed)
    w2, e2 = spvar.sample_range(p, dev, thr.shape[1], cut, T, S, seed, init=half)
    assert bool((e2 == e).all()) and bool((w2 == words).all())


@pytest.mark.parametrize("name,S", [("one_warp", 2611), ("two_warps_three_classes", 4001), ("four_warps", 1300),
                                    ("one_warp_odd", 16000), ("degree8", 5003), ("chimera9", 8002)])
def test_sample_of_many_quads_equals_oracle(cuda_lib, name, S):
    """Shapes of spvar_sample by the number of quads: several per block, a part
    of the last block, and the quad-group kernel for Chimera C9."""
    spvar = cuda_lib
    inst = I.chimera(9, 807) if name == "chimera9" else CASES[name]()
    T, seed = 3, 97
    thr = table(inst, T)
    words, e = spvar.sample(gpu_problem(inst), spvar.thresholds_device(thr), thr.shape[1], T, S, seed)
    spins, energies, _ = O.sample(oracle_problem(inst), thr, S, seed)
    assert np.array_equal(e.cpu().numpy()[:S], energies)
    assert np.array_equal(spvar.unpack_spins(words.cpu().numpy()[:S], inst.n), spins)


@pytest.mark.parametrize("make,S", [(lambda: I.weak_strong(4, 808), 1300), (lambda: I.weak_strong(6, 809), 5002),
                                    (lambda: I.chimera_u10(3, 810), 9999), (lambda: I.chimera_u10(8, 811), 2501),
                                    (lambda: I.chimera_u10(18, 812), 30), (lambda: I.weak_strong(17, 813), 30)],
                         ids=["ws4", "ws6", "u10_c3", "u10_c8", "u10_c18", "ws17"])
def test_sample_of_16_bit_lanes_equals_oracle(cuda_lib, make, S):
    """The same rule for the 16-bit-lane forms, and the quad-group kernel for
    problems whose classes their blocks do not hold."""
    spvar = cuda_lib
    inst = make()
    T, seed = 3, 98
    thr = table(inst, T)
    words, e = spvar.sample(gpu_problem(inst), spvar.thresholds_device(thr), thr.shape[1], T, S, seed)
    spins, energies, _ = O.sample(oracle_problem(inst), thr, S, seed)
    assert np.array_equal(e.cpu().numpy()[:S], energies)
    assert np.array_equal(spvar.unpack_spins(words.cpu().numpy()[:S], inst.n), spins)
