"""Fused batches whose Gram products run on the tensor cores: every job's slice of the
shared block (narrow slices of 4 or 8 columns in rows of 16, wider ones on the integer
path), row counts that are whole tiles and others, against the jobs alone."""
import numpy as np
import pytest

from paper_0704_2351_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PRIMES = [1073741789, 1073741783, 1073741741, 1073741723]


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


@pytest.mark.parametrize("rows,cols", [(640, 576), (641, 575), (4160, 4096)])
@pytest.mark.parametrize("m", [2, 3, 4, 8])
@pytest.mark.parametrize("jobs", [2, 3, 4])
def test_slices_of_a_shared_block(wr, rows, cols, m, jobs):
    A = synth.random_sparse(rows, cols, 7, seed=rows + m)
    prms = [wr.make_params(p, m, m, 40 + k, want=wr.WR_WANT_SEQUENCE, seq_len=131) for k, p in enumerate(PRIMES[:jobs])]

    def sequences(mode, fuse):
        ctx = wr.wr_create(0)
        wr.wr_set_tensor_projection(ctx, mode)
        wr.wr_set_batch_fusion(ctx, fuse)
        mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
        out = []
        for r in wr.wr_rank_batch(ctx, [mat] * jobs, prms):
            out.append(wr.wr_result_sequence(r, m, m))
            wr.wr_result_free(r)
        wr.wr_matrix_free(mat)
        wr.wr_destroy(ctx)
        return out

    for a, b in zip(sequences(1, True), sequences(0, False)):
        assert np.array_equal(a, b)
