"""Repeated black-box applications whose inputs, seeds and widths change from call to
call, on one matrix and the same buffers: each call's kernels start while the ones
before them drain, and none may see what an earlier call left in the block, the
diagonals or the split rows' sums.  Against the oracle, every call."""
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


def _matrix(rows, cols, long_rows, seed):
    rng = np.random.default_rng(seed)
    r = np.repeat(np.arange(rows), 12)
    c = rng.integers(0, cols, size=len(r))
    for k in range(long_rows):  # a split row and a split column each
        r = np.concatenate([r, np.full(700, rng.integers(rows)), rng.choice(rows, 700, replace=False)])
        c = np.concatenate([c, rng.choice(cols, 700, replace=False), np.full(700, rng.integers(cols))])
    v = rng.integers(1, 4, size=len(r)) * (2 * rng.integers(0, 2, size=len(r)) - 1)
    return synth.csr_from_coo(rows, cols, r, c, v)


@pytest.mark.parametrize("long_rows", [0, 2])
@pytest.mark.parametrize("widths", [(3,), (31,), (8,), (1, 31, 3, 16, 32)])
def test_changing_inputs(wr, long_rows, widths):
    A = _matrix(2000, 1800, long_rows, 7)
    ctx = wr.wr_create(0)
    mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
    rng = np.random.default_rng(1)
    most = max(widths)
    x = torch.empty(A.cols * most, dtype=torch.int32, device="cuda")
    y = torch.empty(A.cols * most + 4, dtype=torch.int32, device="cuda")
    for call in range(10):
        w, seed = widths[call % len(widths)], 5 + call
        v = rng.integers(0, P, size=(A.cols, w)).astype(np.uint32)
        x[:A.cols * w] = torch.from_numpy(v.view(np.int32).ravel()).cuda()
        torch.cuda.synchronize()
        out = y[call % 2:]  # (on a 16-byte boundary the second pass writes it itself)
        wr.wr_blackbox_apply_device(ctx, mat, wr.make_params(P, 1, w, seed, side=0), x, out, w)
        ref = oracle.blackbox_apply(A, P, 0, oracle.derive_diag(seed, oracle.TAG_D1, A.cols, P),
                                    oracle.derive_diag(seed, oracle.TAG_D2, A.rows, P), v)
        got = out[:A.cols * w].cpu().numpy().view(np.uint32).reshape(A.cols, w)
        assert np.array_equal(got, ref), (call, w)
    wr.wr_matrix_free(mat)
    wr.wr_destroy(ctx)
