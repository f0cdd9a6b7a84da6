"""GPU parity of the quad-group +-1 kernel at the edges of its forms: degree 7
and 8, biases up to dmax 30, rows with a threshold of 0, one quad, odd numbers
of quads, classes split over the block, and problems whose records do not fit
shared memory.  Everything is a whole number and equals the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table, with_h

pytestmark = pytest.mark.gpu


def _dense8():
    """36 spins, degree 7 or 8, +-1 couplers, biases in [-2, 2]."""
    n, g = 36, np.random.default_rng(81)
    pairs = sorted({(min(i, (i + k) % n), max(i, (i + k) % n)) for i in range(n) for k in (1, 2, 5, 9)})[:-5]
    ei, ej = (np.array(x, np.int32) for x in zip(*pairs))
    J = (g.integers(0, 2, len(pairs)) * 2 - 1).astype(np.int32)
    return I.Instance("dense8", n, ei, ej, J, g.integers(-2, 3, n).astype(np.int32))


PROBLEMS = {"degree8": _dense8, "cubic_h9": lambda: with_h(I.cubic3d(4, 82), 6, 9), "cubic_odd": lambda: I.cubic3d(5, 83),
            "chimera": lambda: I.chimera(5, 84)}


@pytest.mark.parametrize("replicas,block", [(4, 128), (8, 1024), (16, 128), (28, 256), (32, 512)])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_solve_equals_oracle(cuda_lib, name, replicas, block):
    spvar = cuda_lib
    inst = PROBLEMS[name]()
    T, seed, S = 30, 91, 4 * 11 + 1
    ref = O.solve(oracle_problem(inst), table(inst, T), seed, num_starts=3, fixing_sample_size=S,
                  solving_sample_size=S, elite_threshold=0.2)
    plan = spvar.Plan([gpu_problem(inst)],
                      spvar.make_params(num_starts=3, fixing_sample_size=S, solving_sample_size=S, num_sweeps=T,
                                        elite_threshold=0.2, replicas_per_block=replicas,
                                        sweep_kernel=spvar.SWEEP_PM1Q, sweep_block=block))
    assert plan.shape()["kernel"] == "pm1-quads"
    out = plan.run(seed, device=False)
    assert np.array_equal(out.best_energy, ref.best_e)
    assert np.array_equal(out.fixed.reshape(3, -1), np.asarray(ref.fixed))
    for s in range(3):
        for ph in range(2):
            c = ref.counts[s, ph]
            assert np.array_equal(out.energies[s, ph, :c], ref.energies[s, ph, :c])


@pytest.mark.parametrize("L,S", [(11, 3), (12, 9), (12, 1300), (21, 6)])
def test_sample_equals_oracle(cuda_lib, L, S):
    """spvar_sample of large problems (L = 21: no records, 16-bit byte offsets do not reach)."""
    spvar = cuda_lib
    inst = I.cubic3d(L, 85)
    T, seed = 6, 92
    thr = table(inst, T)
    words, e = spvar.sample(gpu_problem(inst), spvar.thresholds_device(thr), thr.shape[1], T, S, seed)
    spins, energies, _ = O.sample(oracle_problem(inst), thr, min(S, 24), seed)
    assert np.array_equal(e.cpu().numpy()[:24], energies)
    assert np.array_equal(spvar.unpack_spins(words.cpu().numpy()[:24], inst.n), spins)
