"""GPU parity of the requested quad-group +-1 kernel at the largest problems a
block holds, and the error where one does not fit: at creation, not at a run."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu


def _ring(n, offsets=(1,), seed=141):
    g = np.random.default_rng(seed)
    ei = np.repeat(np.arange(n), len(offsets)).astype(np.int32)
    ej = ((ei + np.tile(offsets, n)) % n).astype(np.int32)
    return I.Instance("ring", n, ei, ej, (g.integers(0, 2, len(ei)) * 2 - 1).astype(np.int32), np.zeros(n, np.int32))


@pytest.mark.parametrize("offsets", [(1,), (1, 2, 5, 9)], ids=["degree2", "degree8"])
@pytest.mark.parametrize("n", [28200, 28400, 28584])
def test_one_quad_of_a_large_problem(cuda_lib, n, offsets):
    spvar = cuda_lib
    inst = _ring(n, offsets)
    T, S, seed = 3, 5, 142
    plan = spvar.Plan([gpu_problem(inst)],
                      spvar.make_params(num_starts=1, fixing_sample_size=S, solving_sample_size=S, num_sweeps=T,
                                        elite_threshold=0.5, replicas_per_block=4, sweep_kernel=spvar.SWEEP_PM1Q))
    out = plan.run(seed, device=False)
    ref = O.solve(oracle_problem(inst), table(inst, T), seed, num_starts=1, fixing_sample_size=S,
                  solving_sample_size=S, elite_threshold=0.5)
    assert np.array_equal(out.best_energy, ref.best_e)
    assert np.array_equal(out.fixed.reshape(1, -1), np.asarray(ref.fixed))
    c = ref.counts[0, 0]
    assert np.array_equal(out.energies[0, 0, :c], ref.energies[0, 0, :c])


def test_too_large_is_refused_at_creation(cuda_lib):
    spvar = cuda_lib
    inst = _ring(28800)
    prm = spvar.make_params(num_starts=1, fixing_sample_size=4, solving_sample_size=4, num_sweeps=2,
                            replicas_per_block=4, sweep_kernel=spvar.SWEEP_PM1Q)
    with pytest.raises(spvar.SpvarError) as e:
        spvar.Plan([gpu_problem(inst)], prm)
    assert e.value.code == spvar.ELIMIT
    # without a request the general kernel, by trial
    plan = spvar.Plan([gpu_problem(inst)], spvar.make_params(num_starts=1, fixing_sample_size=4, solving_sample_size=4,
                                                              num_sweeps=2))
    assert plan.shape()["kernel"].startswith("general")
    out = plan.run(5, device=False)
    ref = O.solve(oracle_problem(inst), table(inst, 2), 5, num_starts=1, fixing_sample_size=4, solving_sample_size=4,
                  elite_threshold=0.1)
    assert np.array_equal(out.best_energy, ref.best_e)


def test_server_of_large_requests(cuda_lib):
    """The server falls back to the kernels it chooses without the request."""
    spvar = cuda_lib
    for n in (28400, 28800):
        inst = _ring(n)
        prm = spvar.make_params(num_starts=1, fixing_sample_size=4, solving_sample_size=4, num_sweeps=2,
                                replicas_per_block=4, sweep_kernel=spvar.SWEEP_PM1Q)
        srv = spvar.Server(prm, 256 << 20, max_n=n, max_nnz=2 * n, max_degree=2, max_dmax=4, max_requests=1)
        rid = srv.submit(inst, 5)
        while srv.step() > 0:
            pass
        out = srv.result(rid)
        ref = O.solve(oracle_problem(inst), table(inst, 2), 5, num_starts=1, fixing_sample_size=4,
                      solving_sample_size=4, elite_threshold=0.1)
        assert np.array_equal(out.best_energy, ref.best_e)
        srv.close()
