"""GPU parity of resumed samples on the quad-group +-1 kernel: a phase in
several sweep launches whose last item per start has one to three quads, so
that a group of two pairs is partly past the item's end.  Everything is a whole
number and equals the oracle's whole run."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [4 * 13, 4 * 14, 4 * 15, 4 * 13 + 1], ids=["one_quad", "two", "three", "odd_samples"])
@pytest.mark.parametrize("chunk", [7, 10])
def test_resumed_groups_equal_oracle(cuda_lib, S, chunk):
    spvar = cuda_lib
    inst = I.cubic3d(5, 121)
    T, seed = 30, 122
    ref = O.solve(oracle_problem(inst), table(inst, T), seed, num_starts=3, fixing_sample_size=S,
                  solving_sample_size=S, elite_threshold=0.2)
    plan = spvar.Plan([gpu_problem(inst)],
                      spvar.make_params(num_starts=3, fixing_sample_size=S, solving_sample_size=S, num_sweeps=T,
                                        elite_threshold=0.2, replicas_per_block=16, sweep_block=128,
                                        sweep_kernel=spvar.SWEEP_PM1Q, sweeps_per_launch=chunk))
    out = plan.run(seed, device=False)
    assert np.array_equal(out.best_energy, ref.best_e)
    assert np.array_equal(out.fixed.reshape(3, -1), np.asarray(ref.fixed))
    for s in range(3):
        for ph in range(2):
            c = ref.counts[s, ph]
            assert np.array_equal(out.energies[s, ph, :c], ref.energies[s, ph, :c])
