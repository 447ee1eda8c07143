"""The SpMM pass over rows of every length around its tiles and batches: light
rows of 0..64 entries, long rows around the 32-entry steps and the 256-entry
segments, enough chunks that a block takes several pieces, every lane width,
packed and wide entries, against the oracle's black box."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_2351_gb300 import synth

pytestmark = pytest.mark.gpu

P = 2147483629


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _matrix(rows, cols, vmax, seed):
    rng = np.random.default_rng(seed)
    lens = np.arange(rows) * 7 % 41
    lens[:66] = np.arange(66)
    longs = [65, 95, 96, 97, 127, 128, 129, 191, 255, 256, 257, 511, 513, 700]
    lens[100:100 + len(longs)] = longs
    lens = np.minimum(lens, cols)
    r = np.repeat(np.arange(rows), lens)
    start = rng.integers(0, cols, size=rows)
    within = np.arange(lens.sum()) - np.repeat(np.cumsum(lens) - lens, lens)
    stride = 1 + 2 * (np.arange(rows) % 50)  # distinct columns within a row
    c = (start[r] + within * stride[r]) % cols
    hot = rng.integers(0, rows, size=3000)   # a long column: split rows of the transpose
    r, c = np.concatenate([r, hot]), np.concatenate([c, np.full(len(hot), cols // 2)])
    v = rng.integers(1, vmax + 1, size=len(r)) * (2 * rng.integers(0, 2, size=len(r)) - 1)
    return synth.csr_from_coo(rows, cols, r, c, v)


@pytest.fixture(scope="module")
def matrices():
    return {vmax: _matrix(170000, 131071, vmax, vmax) for vmax in (3, 300)}


@pytest.mark.parametrize("vmax", [3, 300])
@pytest.mark.parametrize("width,lanes", [(1, 1), (2, 2), (4, 1), (4, 4), (7, 2), (8, 4), (8, 8), (16, 2), (16, 4),
                                         (16, 8), (31, 1), (32, 2), (32, 4), (32, 8)])
def test_blackbox_over_row_lengths(wr, matrices, vmax, width, lanes):
    A = matrices[vmax]
    ctx = wr.wr_create(0)
    wr.wr_set_lane_width(ctx, lanes)
    mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
    v = np.random.default_rng(width).integers(0, P, size=(A.cols, width)).astype(np.uint32)
    x = torch.from_numpy(v.view(np.int32)).cuda()
    y = torch.empty_like(x)
    wr.wr_blackbox_apply_device(ctx, mat, wr.make_params(P, 1, width, 5, side=0), x, y, width)
    ref = oracle.blackbox_apply(A, P, 0, oracle.derive_diag(5, oracle.TAG_D1, A.cols, P),
                                oracle.derive_diag(5, oracle.TAG_D2, A.rows, P), v)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), ref)
    wr.wr_matrix_free(mat)
    wr.wr_destroy(ctx)
