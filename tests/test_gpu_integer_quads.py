"""GPU parity of the quad-group kernel for integer couplers, which spvar_sample
takes for couplers of several magnitudes: byte lanes up to dmax 254, 16-bit
lanes from 256 to 16382 (the widest acceptance row), wider problems on the
general kernel, degree 6 and 8, one quad and odd numbers of quads, and a sample
in two sweep ranges.  Everything is a whole number and equals the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu


def _with_dmax(inst, dmax):
    """Spin 0's bias makes the largest flip cost exactly dmax."""
    p = oracle_problem(inst)
    sums = [abs(int(inst.h[i])) + int(np.abs(inst.J[(inst.ei == i) | (inst.ej == i)]).sum()) for i in range(inst.n)]
    assert 2 * max(sums) <= dmax and dmax % 2 == 0
    inst.h[0] += dmax // 2 - sums[0] if inst.h[0] >= 0 else -(dmax // 2 - sums[0])
    assert O.dmax(oracle_problem(inst)) == dmax and p.n == inst.n
    return inst


def _gauss(L, seed, scale):
    inst = I.cubic3d(L, seed)
    g = np.random.default_rng(seed)
    j = np.rint(scale * g.standard_normal(inst.m)).astype(np.int32)
    inst.J = np.where(j == 0, 1, j).astype(np.int32)
    inst.h = np.rint(0.2 * scale * g.standard_normal(inst.n)).astype(np.int32)
    inst.scale = scale
    return inst


def _circulant(seed, jmax, hmax, n=61):
    """Degree 8: offsets 1, 2, 5 and 9 of a ring."""
    g = np.random.default_rng(seed)
    ei = np.repeat(np.arange(n), 4).astype(np.int32)
    ej = ((ei + np.tile([1, 2, 5, 9], n)) % n).astype(np.int32)
    J = (g.integers(1, jmax + 1, 4 * n) * (g.integers(0, 2, 4 * n) * 2 - 1)).astype(np.int32)
    return I.Instance("circulant", n, ei, ej, J, g.integers(-hmax, hmax + 1, n).astype(np.int32))


CASES = {
    "dmax254": (lambda: _with_dmax(_gauss(4, 601, 12), 254), 33),
    "dmax256": (lambda: _with_dmax(_gauss(4, 602, 12), 256), 33),
    "dmax16382": (lambda: _with_dmax(_gauss(4, 603, 300), 16382), 5),
    "dmax16384_general": (lambda: _with_dmax(_gauss(4, 604, 300), 16384), 5),
    "odd_L9": (lambda: _gauss(9, 605, 100), 44),
    "degree8_bytes": (lambda: _circulant(606, 15, 7), 70),
    "degree8_lanes": (lambda: _circulant(607, 90, 30), 1300),
}


@pytest.mark.parametrize("name", list(CASES))
def test_sample_equals_oracle(cuda_lib, name):
    spvar = cuda_lib
    make, S = CASES[name]
    inst = make()
    T, seed = 12, 95
    thr = table(inst, T)
    p, dev = gpu_problem(inst), spvar.thresholds_device(thr)
    words, e = spvar.sample(p, dev, thr.shape[1], T, S, seed)
    spins, energies, _ = O.sample(oracle_problem(inst), thr, min(S, 80), seed)
    assert np.array_equal(e.cpu().numpy()[:80], energies)
    assert np.array_equal(spvar.unpack_spins(words.cpu().numpy()[:80], inst.n), spins)
    half, _ = spvar.sample_range(p, dev, thr.shape[1], 0, 5, S, seed)
    w2, e2 = spvar.sample_range(p, dev, thr.shape[1], 5, T, S, seed, init=half)
    assert bool((e2 == e).all()) and bool((w2 == words).all())


def test_sample_limit_is_the_general_kernels(cuda_lib):
    """A sample whose eight quads per block pass the general kernel's shared
    memory is refused, although the quad-group kernel could hold it."""
    spvar = cuda_lib
    inst = _gauss(20, 608, 100)
    thr = table(inst, 2)
    p, dev = gpu_problem(inst), spvar.thresholds_device(thr)
    with pytest.raises(spvar.SpvarError):
        spvar.sample(p, dev, thr.shape[1], 2, 16000, 1)
    spvar.sample(p, dev, thr.shape[1], 2, 40, 1)
