"""GPU parity of the PTICM kernel's forms at their edges: byte lanes with the
256-byte rows (dmax <= 62) for degree 6 and 8, byte lanes beside them, 16-bit
lanes (dmax > 254, and degree > 8), more than 32 temperatures with cluster
moves from an odd one (two groups of masks), and more spins than two a thread.
Everything is a whole number and equals the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, with_h

pytestmark = pytest.mark.gpu


def _star(n, seed):
    """A hub of degree n - 1 > 8 over a ring."""
    g = np.random.default_rng(seed)
    pairs = sorted({(0, j) for j in range(1, n)} | {(min(j, j % (n - 1) + 1), max(j, j % (n - 1) + 1)) for j in range(1, n)})
    ei, ej = (np.array(x, np.int32) for x in zip(*pairs))
    J = (g.integers(1, 4, len(pairs)) * (g.integers(0, 2, len(pairs)) * 2 - 1)).astype(np.int32)
    return I.Instance("star", n, ei, ej, J, g.integers(-2, 3, n).astype(np.int32))


CASES = {
    "small_deg6": (lambda: with_h(I.cubic3d(4, 501), 1, 20), 7, {}),
    "small_deg8": (lambda: I.random_graph(40, 140, 502, jmax=1, hmax=3), 6, {}),
    "bytes": (lambda: I.chimera_u10(3, 503), 9, {}),
    "lanes16_weak_strong": (lambda: I.weak_strong(3, 504), 6, {}),
    "lanes16_degree": (lambda: _star(14, 505), 5, {}),
    "two_mask_groups": (lambda: I.cubic3d(3, 506), 40, dict(icm_from=3, keep_from=30)),
    "spins_1331": (lambda: I.cubic3d(11, 507), 4, dict(icm_from=0)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_pticm_forms(cuda_lib, name):
    spvar = cuda_lib
    make, R, opt = CASES[name]
    inst = make()
    betas, T = np.geomspace(0.2, 2.5, R), 8 if inst.n > 1000 else 20
    g = spvar.pticm_sample(gpu_problem(inst), betas, T, spvar.energy_range(inst), K=6, num_runs=2, seed=78, start0=2, **opt)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    for run in range(2):
        ref = O.pticm_sample(oracle_problem(inst), betas, T, K=6, seed=78, start=2 + run, **opt)
        assert np.array_equal(spvar.unpack_spins(g["final_states"][run], inst.n), ref["final"])
        assert np.array_equal(g["final_e"][run], ref["final_e"] + inst.offset)
        assert np.array_equal(g["nkept"][run], ref["nkept"])
        for q, nk in enumerate(ref["nkept"]):
            assert np.array_equal(g["kept_e"][run, q, :nk], ref["kept_e"][q, :nk] + inst.offset)
            assert np.array_equal(spvar.unpack_spins(g["kept"][run, q, :nk], inst.n), ref["kept"][q, :nk])
