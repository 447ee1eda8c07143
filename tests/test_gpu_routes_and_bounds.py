"""Which loop a small matrix's sequence takes, by the kernels it launches, on both sides
of the one-cluster loop's limits; and the tensor-core Gram product with every digit of
both factors at its largest over as many rows as a block sums."""
import numpy as np
import pytest
import torch

from paper_0704_2351_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


@pytest.mark.parametrize("rows,per_row,vmax,m,n,sym,one_cluster", [
    (40, 3, 3, 1, 1, False, True), (2000, 12, 3, 1, 1, False, True), (6000, 6, 3, 1, 1, False, True),
    (16000, 6, 3, 1, 1, False, False), (3000, 6, 3, 2, 2, False, True), (9000, 6, 3, 2, 2, False, False),
    (1000, 8, 127, 4, 4, False, True), (1000, 8, 300, 4, 4, False, False), (500, 7, 3, 16, 16, False, True),
    (1000, 7, 3, 16, 16, False, False), (1000, 7, 3, 16, 16, True, True), (2000, 12, 3, 16, 16, True, False),
    (400, 5, 3, 17, 17, True, False), (400, 5, 3, 4, 2, False, False)])
def test_one_cluster_loop_is_taken(wr, rows, per_row, vmax, m, n, sym, one_cluster):
    A = synth.random_sparse(rows, rows - rows // 10, per_row, seed=3, vmax=vmax)
    A.vals[:2] = vmax  # (an entry beyond 127 makes the layout wide)
    prm = wr.make_params(2147483647, m, n, 11, projection=wr.WR_PROJ_SYMMETRIC if sym else wr.WR_PROJ_GENERIC)
    ctx = wr.wr_create(0)
    mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
    L = 257
    S = torch.empty((L, m, n), dtype=torch.int32, device="cuda")
    before = wr.wr_last_timings(ctx)["kernel_launches"]
    wr.wr_sequence_device(ctx, mat, prm, S, L)
    launches = wr.wr_last_timings(ctx)["kernel_launches"] - before
    wr.wr_matrix_free(mat)
    wr.wr_destroy(ctx)
    # 128 applications: two launches of the loop and the set-up, or two passes each at least
    assert launches <= 16 if one_cluster else launches >= 256, launches


@pytest.mark.parametrize("m,stride,yoff", [(8, 8, 0), (8, 16, 8), (16, 32, 16), (32, 32, 0)])
@pytest.mark.parametrize("extra", [0, 1, 64 * 3 + 1])
def test_largest_digits(wr, m, stride, yoff, extra):
    """Residues 0x7EFFFFFF (three digits of 255) in both factors; 2 sms blocks of 507 tiles
    of 64 rows, one short of the most that a block takes, and a little more."""
    p, x = 2147483647, 0x7EFFFFFF
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 2 * sms * 507 * 64 + extra
    t = torch.full((N, stride), x, dtype=torch.int32, device="cuda")
    w = torch.full((N,), 2**32 % p, dtype=torch.int32, device="cuda")  # (times 2^-32: the left factor is x itself)
    G = torch.empty((m, m), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    ctx = wr.wr_create(0)
    wr.wr_set_tensor_projection(ctx, 1)
    wr.wr_gram_device(ctx, p, N, m, m, t, stride, yoff, w, G)
    wr.wr_destroy(ctx)
    want = N * (2**32 % p) * x * x % p
    assert np.array_equal(G.cpu().numpy(), np.full((m, m), want, dtype=np.int32))
