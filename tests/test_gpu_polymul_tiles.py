"""Polynomial products whose transforms fill less than one tile of 2^13 values, exactly
one, and one and a part (in each operand and in the product), and sums of lengths
around the stages of the pointwise products with few entries, against the sums of
products reduced one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _product(A, B, p):
    C = np.zeros((len(A) + len(B) - 1, A.shape[1], B.shape[2]), dtype=np.int64)
    for j in range(len(B)):
        for k in range(A.shape[2]):
            C[j:j + len(A)] += A[:, :, k, None] * B[j, k, None, :] % p
        C[j:j + len(A)] %= p
    return C


@pytest.mark.parametrize("p", [65521, 2147483647])
@pytest.mark.parametrize("r,s,t", [(1, 1, 1), (1, 32, 1), (1, 33, 1), (4, 8, 4), (4, 8, 8), (3, 9, 7), (4, 11, 8), (2, 64, 1),
                                   (1, 3, 32), (12, 1, 33)])
@pytest.mark.parametrize("na,nb", [(20, 9), (140, 100), (700, 300)])  # transforms of 32, 256 and 1,024 points
def test_part_tiles(wr, p, r, s, t, na, nb):
    rng = np.random.default_rng(na + s)
    A = rng.integers(0, p, size=(na, r, s), dtype=np.int64)
    B = rng.integers(0, p, size=(nb, s, t), dtype=np.int64)
    A[:, :, -1], B[:, -1, :] = p - 1, p - 1
    ctx = wr.wr_create(0)
    dA, dB = (torch.from_numpy(x.astype(np.int32)).cuda() for x in (A, B))
    C = torch.full((na + nb - 1, r, t), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    wr.wr_polymat_mul_device(ctx, p, dA, na, dB, nb, r, s, t, 0, na + nb - 1, C)
    wr.wr_destroy(ctx)
    assert np.array_equal(C.cpu().numpy().astype(np.int64), _product(A, B, p))
