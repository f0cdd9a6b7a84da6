"""GPU parity of the SQA register forms on both sides of two blocks an SM, with
64-bit acceptance entries (a sample's own table) and 32-bit ones (a plan's), two
and four colour classes, +-1 and small integer couplers."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem

pytestmark = pytest.mark.gpu

PROBLEMS = {"two_classes": lambda: I.chimera(2, 201), "four_classes": lambda: I.cubic3d(3, 202),
            "integers": lambda: I.chimera_u10(2, 203)}


@pytest.mark.parametrize("S", [40, 1216, 1218], ids=["few", "two_per_sm", "more"])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_sample_equals_oracle(cuda_lib, name, S):
    spvar = cuda_lib
    inst = PROBLEMS[name]()
    op = oracle_problem(inst)
    T, P, seed = 12, 6, 204
    ent = O.sqa_table(T, P, 3.0, O.gamma_linear(T, 3.0, 0.05), O.dmax(op), inst.scale)
    g, e, sl = spvar.sqa_sample(gpu_problem(inst), spvar.table_device(ent), ent.shape[2], T, P, S, seed)
    spins, energies, slices = O.sqa_sample(op, ent, P, S, seed)
    assert np.array_equal(e.cpu().numpy(), energies)
    assert np.array_equal(sl.cpu().numpy(), slices)
    assert np.array_equal(spvar.unpack_spins(g.cpu().numpy(), inst.n), spins)


@pytest.mark.parametrize("starts,S", [(2, 30), (4, 304), (4, 340)], ids=["few", "two_per_sm", "more"])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_plan_equals_oracle(cuda_lib, name, starts, S):
    spvar = cuda_lib
    inst = PROBLEMS[name]()
    sqa = dict(sampler=spvar.SAMPLER_SQA, sqa_slices=4, sqa_beta=2.0, sqa_gamma0=2.5, sqa_gamma1=0.05)
    T, seed = 20, 205
    plan = spvar.Plan([gpu_problem(inst)],
                      spvar.make_params(num_starts=starts, fixing_sample_size=S, solving_sample_size=S, num_sweeps=T,
                                        elite_threshold=0.2, replicas_per_block=4, sweep_block=256,
                                        sweep_kernel=spvar.SWEEP_PM1, **sqa))
    assert plan.shape()["kernel"] == "sqa-register"
    out = plan.run(seed, device=False)
    ref = O.solve(oracle_problem(inst), np.zeros((T, O.dmax(oracle_problem(inst)) + 1), np.uint32), seed,
                  num_starts=starts, fixing_sample_size=S, solving_sample_size=S, elite_threshold=0.2, sampler=1,
                  sqa_slices=4, sqa_beta=2.0, sqa_gamma0=2.5, sqa_gamma1=0.05)
    assert np.array_equal(out.best_energy, ref.best_e)
    assert np.array_equal(out.fixed.reshape(starts, -1), np.asarray(ref.fixed))
    for s in range(starts):
        for ph in range(2):
            c = ref.counts[s, ph]
            assert np.array_equal(out.energies[s, ph, :c], ref.energies[s, ph, :c])
