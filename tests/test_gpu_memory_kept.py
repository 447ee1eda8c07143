"""Freed device memory kept between calls: bounded by 2 GiB, given back by
wr_trim_memory while contexts and matrices live, and by the last context."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = 2147483629
MIB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_is_given_back():
    from paper_0704_2351_gb300 import wr
    n = 1 << 14  # products of 32 x 32 x 32, transforms of 2^15 points: 5 x 128 MiB of buffers
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    A, B = (torch.randint(0, P, (n, 32, 32), generator=g, device="cuda", dtype=torch.int32) for _ in range(2))
    C = [torch.empty((2 * n - 1, 32, 32), dtype=torch.int32, device="cuda") for _ in range(2)]
    other = wr.wr_create(0)
    ctx = wr.wr_create(0)
    before = _free()
    wr.wr_polymat_mul_device(ctx, P, A, n, B, n, 32, 32, 32, 0, 2 * n - 1, C[0])
    kept = before - _free()
    assert 512 * MIB <= kept <= 2048 * MIB + 128 * MIB
    wr.wr_trim_memory(ctx)
    assert before - _free() <= 64 * MIB  # (the twiddle table stays)
    wr.wr_polymat_mul_device(ctx, P, A, n, B, n, 32, 32, 32, 0, 2 * n - 1, C[1])
    wr.wr_destroy(ctx)
    wr.wr_trim_memory(other)
    assert before - _free() <= 64 * MIB
    wr.wr_destroy(other)
    assert torch.equal(C[0], C[1])  # (last: torch keeps its own temporaries)
    with pytest.raises(wr.WrError) as e:
        wr.wr_trim_memory(0)
    assert e.value.status == wr.WR_EINVAL
