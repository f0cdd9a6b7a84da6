"""GPU parity of the clustered fold behind spvar.reduce at the edges of its
256-spin chunks: one spin, a chunk less and more by one spin, all eight blocks
of the cluster with one and with several chunks, and the largest problem, with
few and with most spins fixed, the sweep layout compared through the energies of
a sample of the reduced problem; and of the allocation-free form at the edges of
the eight blocks' ranges and of a thread's first and second spin."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1706_07826_gb300 import instances as I

from gpu_cases import gpu_problem, oracle_problem, table

pytestmark = pytest.mark.gpu


def _ring(n, seed):
    """Degree up to 4: a ring and its second neighbours (three colour classes or more)."""
    g = np.random.default_rng(seed)
    if n < 6:
        ei, ej = np.arange(n - 1), np.arange(1, n)
    else:
        ei = np.repeat(np.arange(n), 2)
        ej = (ei + np.tile([1, 2], n)) % n
    J = g.integers(1, 8, len(ei)) * (g.integers(0, 2, len(ei)) * 2 - 1)
    return I.Instance("ring", n, ei.astype(np.int32), ej.astype(np.int32), J.astype(np.int32),
                      g.integers(-5, 6, n).astype(np.int32))


@pytest.mark.parametrize("free", [0.0, 0.15, 0.8])
@pytest.mark.parametrize("n", [1, 2, 7, 9, 1025, 2048, 2049, 8191, 8192, 8193, 16384])
def test_reduce_noalloc_equals_oracle_at_block_edges(cuda_lib, n, free):
    import torch
    spvar = cuda_lib
    inst = _ring(n, 900 + n)
    g = np.random.default_rng(n + 1)
    fixed = np.where(g.random(n) < free, 0, g.choice([-1, 1], n)).astype(np.int8)
    red, _, oon = O.reduce(oracle_problem(inst), fixed)
    gp = gpu_problem(inst)
    z = {k: torch.full((max(s, 1),), -9, dtype=t, device="cuda")
         for k, s, t in (("row_ptr", n + 1, torch.int32), ("col", 2 * inst.m, torch.int32),
                         ("val", 2 * inst.m, torch.int32), ("h", n, torch.int32), ("offset", 1, torch.int64),
                         ("old_of_new", n, torch.int32), ("n_out", 1, torch.int32))}
    spvar.reduce_noalloc(gp, torch.from_numpy(fixed).cuda(), **z)
    d = {k: v.cpu().numpy() for k, v in z.items()}
    m, nnz = red.n, int(red.row_ptr[red.n])
    assert d["n_out"][0] == m and d["offset"][0] == red.offset
    assert np.array_equal(d["row_ptr"][:m + 1], red.row_ptr)
    for k, want, cnt in (("col", red.col, nnz), ("val", red.val, nnz), ("h", red.h, m), ("old_of_new", oon, m)):
        assert np.array_equal(d[k][:cnt], want[:cnt]) and (d[k][cnt:] == -9).all(), k


@pytest.mark.parametrize("free", [0.15, 0.8])
@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 2048, 2049, 4097, 8193, 32768])
def test_reduce_equals_oracle_at_chunk_edges(cuda_lib, n, free):
    import torch
    spvar = cuda_lib
    inst = _ring(n, 700 + n)
    inst.offset = 13
    g = np.random.default_rng(n)
    fixed = np.where(g.random(n) < free, 0, g.choice([-1, 1], n)).astype(np.int8)
    red, colours, oon = O.reduce(oracle_problem(inst), fixed)
    gp = gpu_problem(inst)
    g_red, g_oon = spvar.reduce(gp, torch.from_numpy(fixed).cuda())
    assert np.array_equal(g_oon.cpu().numpy(), oon)
    d = g_red.download()
    assert d["n"] == red.n and d["offset"] == red.offset
    for k in ("row_ptr", "col", "val", "h"):
        assert np.array_equal(d[k], getattr(red, k)), k
    assert np.array_equal(d["colour"], colours[0])
    T, S = 3, 4
    thr = table(inst, T)
    spins, e, _ = O.sample(red, thr, S, 5, colours=colours)
    words, g_e = spvar.sample(g_red, spvar.thresholds_device(thr), thr.shape[1], T, S, 5)
    assert np.array_equal(g_e.cpu().numpy()[:S], e + red.offset)
    if red.n:
        assert np.array_equal(spvar.unpack_spins(words.cpu().numpy()[:S], red.n), spins)
