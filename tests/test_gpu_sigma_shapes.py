"""The sigma-basis kernels at the edges of their variants, against the oracle's
M-Basis: block sizes around the row and column classes of the local kernel (m up
to 8, 16, 32; q up to 16, 32, 40, 48, 64), lengths around a chunk, primes of both
fold classes (p <= 2^30 and above), and sequences whose discrepancies lose rank in
some orders of a chunk only, so that the straight elimination and the general one
alternate."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


@pytest.fixture(scope="module")
def ctx(wr):
    c = wr.wr_create(0)
    yield c
    wr.wr_destroy(c)


def _check(wr, ctx, S, p):
    L, m, n = S.shape
    P = torch.empty((L + 2, n, m + n), dtype=torch.int32, device="cuda")
    deg = torch.empty(m + n, dtype=torch.int32, device="cuda")
    dS = torch.from_numpy(np.ascontiguousarray(S).view(np.int32)).cuda()
    torch.cuda.synchronize()
    wr.wr_sigma_basis_device(ctx, dS, L, m, n, p, P, deg, L + 1)
    M, ref = oracle.mbasis(S, p)
    got = P.cpu().numpy().view(np.uint32)
    assert np.array_equal(deg.cpu().numpy(), ref)
    assert np.array_equal(got[:M.shape[0]], M[:, :n, :])
    assert not got[M.shape[0]:].any()


@pytest.mark.parametrize("p", [65521, 1073741789, 1073741827, 1431655777, 2147483647])
@pytest.mark.parametrize("m,n,L", [(1, 2, 129), (4, 4, 64), (7, 9, 63), (8, 9, 66), (8, 32, 40), (9, 7, 65), (1, 32, 35),
                                   (16, 17, 34), (16, 32, 33), (17, 15, 33), (31, 32, 18), (32, 32, 33)])
def test_block_shapes(wr, ctx, m, n, L, p):
    rng = np.random.default_rng(m * 100 + n)
    _check(wr, ctx, rng.integers(0, p, size=(L, m, n)).astype(np.uint32), p)


@pytest.mark.parametrize("m,n", [(3, 3), (8, 8), (16, 16), (20, 12), (32, 32)])
def test_discrepancies_that_lose_rank_in_some_orders(wr, ctx, m, n):
    """Random terms, with zero rows, repeated rows, zero terms and zero columns among them."""
    p = 2147483629
    rng = np.random.default_rng(m)
    L = 70 if m + n <= 32 else 36
    S = rng.integers(0, p, size=(L, m, n)).astype(np.uint32)
    S[0, 0] = 0
    S[1, m - 1] = S[1, 0]
    S[2] = 0
    S[5, :, 0] = 0
    S[9, m // 2:] = 0
    S[20, 1] = S[20, 0]
    S[30] = S[29]
    _check(wr, ctx, S, p)
    S[:, m - 1] = S[:, 0]  # one row of X twice: never full rank
    _check(wr, ctx, S, p)


@pytest.mark.parametrize("m,n", [(9, 9), (12, 6), (15, 20), (17, 17), (23, 10), (24, 24), (25, 7), (30, 31)])
@pytest.mark.parametrize("p", [1073741789, 2147483647])
def test_groups_of_pivot_columns(wr, ctx, m, n, p):
    """m around multiples of the elimination's groups of eight, both primes' folds, and
    residues at the ends of their range."""
    rng = np.random.default_rng(m)
    S = rng.choice(np.array([p - 1, p - 2, 1, p // 2, 12345]), size=(20, m, n)).astype(np.uint32)
    _check(wr, ctx, S, p)
    S = rng.integers(p - 50, p, size=(35, m, n)).astype(np.uint32)
    _check(wr, ctx, S, p)
