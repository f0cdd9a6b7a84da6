"""GPU tests of the +-1 server's two kernels: few quads in flight run on the
streaming kernel, more on the quad groups, and a step may continue what the
other kernel began.  Each request's result equals the request solved alone, and
one equals the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu

# 4 starts x 50 quads a request: on 152 SMs one or two of equal size are few, three are not
KW = dict(num_starts=4, fixing_sample_size=200, solving_sample_size=120, num_sweeps=60, elite_threshold=0.2)


def _same(a, b):
    assert np.array_equal(a.best_energy, b.best_energy)
    assert np.array_equal(a.fixed, b.fixed)
    assert np.array_equal(a.best_state, b.best_state)
    assert np.array_equal(a.counts, b.counts)
    for s in range(a.counts.shape[0]):
        for p in range(a.counts.shape[1]):
            c = a.counts[s, p]
            assert np.array_equal(a.energies[s, p, :c], b.energies[s, p, :c])


@pytest.mark.parametrize("sps", [0, 17], ids=["phases", "steps17"])
@pytest.mark.parametrize("late", [1, 3, 5], ids=["late1", "late3", "late5"])
def test_requests_that_change_the_load(cuda_lib, sps, late):
    """One request alone, then two to six at once, then the rest of them."""
    spvar = cuda_lib
    insts = [I.cubic3d(6, 171), I.cubic3d(6, 172), I.cubic3d(5, 173), I.cubic3d(6, 174), I.chimera(5, 175),
             I.cubic3d(6, 176)][:1 + late]
    srv = spvar.Server(spvar.make_params(**KW, sweep_kernel=spvar.SWEEP_PM1), 256 << 20, max_n=1000, max_nnz=6000,
                       max_degree=6, max_dmax=12, max_requests=6, sweeps_per_step=sps)
    ids = [srv.submit(insts[0], 300)]
    srv.step()
    ids += [srv.submit(x, 301 + i) for i, x in enumerate(insts[1:])]
    steps = 0
    while srv.step() > 0:
        steps += 1
        assert steps < 100
    for i, (rid, inst) in enumerate(zip(ids, insts)):
        _same(srv.result(rid), spvar.solve(gpu_problem(inst), spvar.make_params(**KW), 300 + i))
    ref = O.solve(oracle_problem(insts[0]), table(insts[0], KW["num_sweeps"], dmax=12), 300, num_starts=4,
                  fixing_sample_size=200, solving_sample_size=120, elite_threshold=0.2)
    out = srv.result(ids[0])
    assert np.array_equal(out.best_energy, ref.best_e)
    assert np.array_equal(out.fixed.reshape(4, -1), ref.fixed)
    srv.close()
