"""GPU parity of the quad-group kernel for integer couplers on work queues: a
general server's default, and a plan's choice for such problems.  Items of
several jobs of uneven size, reduced problems, and samples resumed at odd
sweeps, in byte lanes and in 16-bit lanes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu

KW = dict(num_starts=3, fixing_sample_size=118, solving_sample_size=60, num_sweeps=60, elite_threshold=0.2)


def _gauss(L, seed, scale):
    inst = I.cubic3d(L, seed)
    g = np.random.default_rng(seed)
    j = np.clip(np.rint(scale * g.standard_normal(inst.m)), -4 * scale, 4 * scale).astype(np.int32)
    inst.J = np.where(j == 0, 1, j).astype(np.int32)
    inst.h = np.rint(0.1 * scale * g.standard_normal(inst.n)).astype(np.int32)
    inst.scale = scale
    return inst


def _oracle(inst, seed, dmax=None):
    return O.solve(oracle_problem(inst), table(inst, KW["num_sweeps"], dmax=dmax), seed, num_starts=3,
                   fixing_sample_size=118, solving_sample_size=60, elite_threshold=0.2)


def _equal(out, ref):
    assert np.array_equal(out.best_energy, ref.best_e)
    assert np.array_equal(out.fixed.reshape(3, -1), np.asarray(ref.fixed))
    for s in range(3):
        for ph in range(2):
            c = ref.counts[s, ph]
            assert np.array_equal(out.energies[s, ph, :c], ref.energies[s, ph, :c])


@pytest.mark.parametrize("scale", [4, 100], ids=["bytes", "lanes"])
@pytest.mark.parametrize("sps", [0, 13], ids=["phases", "steps13"])
def test_server_requests_equal_oracle(cuda_lib, scale, sps):
    spvar = cuda_lib
    insts = [_gauss(4, 191, scale), _gauss(7, 192, scale), _gauss(9, 193, scale), _gauss(5, 194, scale)]
    dmax = max(O.dmax(oracle_problem(x)) for x in insts)
    assert (dmax <= 254) == (scale < 10)
    srv = spvar.Server(spvar.make_params(**KW), 256 << 20, max_n=729, max_nnz=6 * 729, max_degree=6, max_dmax=dmax,
                       energy_scale=scale, max_requests=3, sweeps_per_step=sps)
    ids = [srv.submit(insts[0], 401)]      # the smaller tier alone, then all of them
    srv.step()
    ids += [srv.submit(x, 402 + i) for i, x in enumerate(insts[1:])]
    steps = 0
    while srv.step() > 0 or srv.stats()["queued"] > 0:
        steps += 1
        assert steps < 100
    for i, (rid, inst) in enumerate(zip(ids, insts)):
        _equal(srv.result(rid), _oracle(inst, 401 + i))
    srv.close()


@pytest.mark.parametrize("scale", [4, 100], ids=["bytes", "lanes"])
@pytest.mark.parametrize("chunk", [0, 7], ids=["whole", "chunk7"])
def test_plan_equals_oracle(cuda_lib, scale, chunk):
    spvar = cuda_lib
    insts = [_gauss(6, 195, scale), _gauss(3, 196, scale), _gauss(8, 197, scale)]
    plan = spvar.Plan([gpu_problem(x) for x in insts], spvar.make_params(**KW, sweeps_per_launch=chunk))
    out = plan.run([501, 502, 503], device=False)
    at = 0
    for k, inst in enumerate(insts):
        ref = _oracle(inst, 501 + k)
        rows = slice(3 * k, 3 * k + 3)
        assert np.array_equal(out.best_energy[rows], ref.best_e)
        fixed = out.fixed[at:at + 3 * inst.n].reshape(3, -1)
        assert np.array_equal(fixed, np.asarray(ref.fixed))
        at += 3 * inst.n
