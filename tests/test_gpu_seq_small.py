"""The one-cluster sequence loop of small matrices against the passes (profiling on
takes them) and the oracle: light and long rows, split rows, empty rows and columns,
both sides and projections, block widths up to its limit, lengths around a group of
applications, the exported block, and matrices just too large for it."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_2351_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _matrix(rows, cols, per_row, long_rows, seed):
    """Random rows, some empty ones, and rows and columns of 65 to 700 entries."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 2 * per_row + 1, size=rows)
    r = np.repeat(np.arange(rows), lens)
    c = rng.integers(0, cols - cols // 8, size=len(r))  # the last columns stay empty
    for k in range(long_rows):
        n = min(int(rng.choice([65, 256, 257, 700])), cols, rows)
        r = np.concatenate([r, np.full(n, rng.integers(rows)), rng.choice(rows, n, replace=False)])
        c = np.concatenate([c, rng.choice(cols, n, replace=False), np.full(n, rng.integers(cols))])
    v = rng.integers(1, 4, size=len(r)) * (2 * rng.integers(0, 2, size=len(r)) - 1)
    return synth.csr_from_coo(rows, cols, r, c, v)


def _run(wr, A, prm, L, m, n, plain):
    ctx = wr.wr_create(0)
    wr.wr_set_profiling(ctx, plain)
    mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
    S = torch.empty((L, m, n), dtype=torch.int32, device="cuda")
    N = max(A.rows, A.cols)
    snap, last = (torch.zeros((N, m + n), dtype=torch.int32, device="cuda") for _ in range(2))
    apps, paired = wr.wr_sequence_state_device(ctx, mat, prm, S, L, min(3, L // 2), snap, last)
    out = S.cpu().numpy().view(np.uint32), snap.cpu().numpy(), last.cpu().numpy(), apps, paired
    wr.wr_matrix_free(mat)
    wr.wr_destroy(ctx)
    return out


@pytest.mark.parametrize("rows,cols,per_row,long_rows", [(40, 33, 3, 0), (300, 260, 6, 2), (1000, 900, 8, 3),
                                                         (2000, 1800, 12, 0), (700, 1500, 10, 4)])
@pytest.mark.parametrize("m,sym", [(1, False), (1, True), (2, False), (3, True), (4, False), (7, False), (16, True)])
@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("p,L", [(65521, 9), (2147483647, 140)])
def test_equals_the_passes_and_the_oracle(wr, rows, cols, per_row, long_rows, m, sym, side, p, L):
    A = _matrix(rows, cols, per_row, long_rows, rows + m)
    prm = wr.make_params(p, m, m, 11, projection=wr.WR_PROJ_SYMMETRIC if sym else wr.WR_PROJ_GENERIC, side=side)
    got, ref = _run(wr, A, prm, L, m, m, False), _run(wr, A, prm, L, m, m, True)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
    st = oracle.Setup(A, p, m, m, 11, side=side, symmetric=sym)
    k = min(L, 9)
    assert np.array_equal(got[0][:k], oracle.sequence(A, st, k))


@pytest.mark.parametrize("L", [1, 2, 3, 127, 128, 129, 130, 257])
def test_lengths_around_a_group(wr, L):
    A = _matrix(500, 450, 7, 2, 5)
    prm = wr.make_params(1073741789, 2, 2, 3)
    got, ref = _run(wr, A, prm, L, 2, 2, False), _run(wr, A, prm, L, 2, 2, True)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
