"""The one-cluster sequence loop over rows and columns that are full or nearly so: rows of
one segment (65 to 256 entries) and of several, every width of the block, entries up to
+-127, residues up to p - 1, against the passes and the oracle; and its time against the
passes', which it replaces."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_0704_2351_gb300 import synth

pytestmark = pytest.mark.gpu

P = 2147483647


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _matrix(rows, cols, lens, vmax, seed):
    """Six entries a row, and a row and a column of each of `lens` entries."""
    rng = np.random.default_rng(seed)
    r, c = np.repeat(np.arange(rows), 6), rng.integers(0, cols, size=6 * rows)
    at = rng.choice(min(rows, cols), size=len(lens), replace=False)
    for k, n in zip(at, lens):
        r = np.concatenate([r, np.full(min(n, cols), k), rng.choice(rows, min(n, rows), replace=False)])
        c = np.concatenate([c, rng.choice(cols, min(n, cols), replace=False), np.full(min(n, rows), k)])
    v = rng.integers(1, vmax + 1, size=len(r)) * (2 * rng.integers(0, 2, size=len(r)) - 1)
    key, first = np.unique(r * cols + c, return_index=True)  # (no sums: entries stay within vmax)
    return synth.csr_from_coo(rows, cols, key // cols, key % cols, v[first])


def _params(wr, m, sym):
    return wr.make_params(P, m, m, 11, projection=wr.WR_PROJ_SYMMETRIC if sym else wr.WR_PROJ_GENERIC, side=0)


@pytest.mark.parametrize("lens", [(65,), (256, 257), (900,), (900, 900, 513, 512, 300, 70, 70)])
@pytest.mark.parametrize("m,sym", [(1, True), (1, False), (2, False), (4, False), (6, False), (16, True), (16, False)])
def test_equals_the_passes_and_the_oracle(wr, lens, m, sym):
    A = _matrix(1000, 900, lens, 127, m + len(lens))
    prm, L, out = _params(wr, m, sym), 133, []
    for passes in (False, True):
        ctx = wr.wr_create(0)
        wr.wr_set_profiling(ctx, passes)
        mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
        S = torch.empty((L, m, m), dtype=torch.int32, device="cuda")
        wr.wr_sequence_device(ctx, mat, prm, S, L)
        out.append(S.cpu().numpy().view(np.uint32))
        wr.wr_matrix_free(mat)
        wr.wr_destroy(ctx)
    assert np.array_equal(out[0], out[1])
    assert np.array_equal(out[0][:7], oracle.sequence(A, oracle.Setup(A, P, m, m, 11, side=0, symmetric=sym), 7))


@pytest.mark.parametrize("lens", [(500,), (250, 250, 250, 250)])
def test_keeps_up_with_the_passes(wr, lens):
    """Blocks of 16, whose products a forced tensor projection leaves on the tensor cores: a
    long row that one warp takes alone makes the loop 1.7 times as slow as the passes (0.7 to
    0.9 times as it is)."""
    A, L, ms = _matrix(500, 450, lens, 3, 5), 257, []
    for mode in (-1, 1):  # 1: the passes
        ctx = wr.wr_create(0)
        wr.wr_set_tensor_projection(ctx, mode)
        mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
        S = torch.empty((L, 16, 16), dtype=torch.int32, device="cuda")
        t = []
        for _ in range(9):
            t0 = time.perf_counter()
            wr.wr_sequence_device(ctx, mat, _params(wr, 16, True), S, L)
            t.append(time.perf_counter() - t0)
        ms.append(1e3 * min(t))
        wr.wr_matrix_free(mat)
        wr.wr_destroy(ctx)
    assert ms[0] < 1.25 * ms[1], ms
