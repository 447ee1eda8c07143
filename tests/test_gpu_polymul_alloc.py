"""Polynomial products on a context whose allocator refuses the growth of the kept
twiddle table: the call reports it, and every later product, shorter or longer, is
right."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = 2147483629


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _product(wr, ctx, A, B):
    na, nb = A.shape[0], B.shape[0]
    C = torch.full((na + nb - 1, 2, 3), -1, dtype=torch.int32, device="cuda")
    wr.wr_polymat_mul_device(ctx, P, A, na, B, nb, 2, 4, 3, 0, na + nb - 1, C)
    return C.cpu().numpy()


@pytest.mark.parametrize("refusals", [1, 2])
def test_refused_twiddle_table(wr, refusals):
    rng = np.random.default_rng(refusals)

    def operand(n, r, s):
        a = torch.from_numpy(rng.integers(0, P, size=(n, r, s)).astype(np.int32)).cuda()
        torch.cuda.synchronize()
        return a

    short = operand(200, 2, 4), operand(90, 4, 3)
    long = operand(12000, 2, 4), operand(9000, 4, 3)  # transforms of 2^15 points
    clean = wr.wr_create(0)
    want_short, want_long = _product(wr, clean, *short), _product(wr, clean, *long)
    wr.wr_destroy(clean)

    table = {24 << 14}  # the three primes' 2^14 powers, both directions, for 2^15 points
    if refusals == 2:
        table.add(24 << 13)  # and the shorter table that would follow it
    held, refused = {}, []

    def alloc(n, stream):
        if n in table and armed:
            table.discard(n)
            refused.append(n)
            return 0
        t = torch.empty(n, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, n, stream):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    ctx = wr.wr_create(0)
    wr.wr_set_allocator(ctx, alloc, release)
    armed = False
    assert np.array_equal(_product(wr, ctx, *short), want_short)
    armed = True
    with pytest.raises(wr.WrError) as e:
        _product(wr, ctx, *long)
    assert e.value.status == wr.WR_ENOMEM
    if refusals == 2:
        with pytest.raises(wr.WrError):
            _product(wr, ctx, *short)
    assert len(refused) == refusals
    assert np.array_equal(_product(wr, ctx, *short), want_short)
    assert np.array_equal(_product(wr, ctx, *long), want_long)
    assert np.array_equal(_product(wr, ctx, *short), want_short)
    wr.wr_destroy(ctx)
    assert not held
