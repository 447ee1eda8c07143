"""The Gram product's call forms that its kernels treat apart, against the sum
reduced product by product: weights on any 4-byte boundary, row counts around a tile (64), a drain
(256) and the drains that a block's sums hold, and residues whose digits are all
255 or 0."""
import numpy as np
import pytest
import torch


pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _ref(t, w, m, n, yoff, p):
    G = np.zeros((m, n), dtype=np.int64)
    for k in range(0, len(w), 4096):
        L = t[k:k + 4096, :m].astype(np.int64) * w[k:k + 4096, None].astype(np.int64) % p
        R = t[k:k + 4096, yoff:yoff + n].astype(np.int64)
        G = (G + (L[:, :, None] * R[:, None, :] % p).sum(axis=0)) % p
    return G


@pytest.mark.parametrize("m,stride,yoff", [(8, 16, 8), (16, 16, 0), (32, 64, 32), (32, 32, 0), (20, 32, 0)])
@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("N", [1, 63, 65, 255, 257, 1000, 33000])
def test_weights_on_any_boundary(wr, m, stride, yoff, shift, N):
    p = 2147483647
    rng = np.random.default_rng(N + m)
    t = rng.choice(np.array([0, 1, 255, 0xFFFFFF, 0x7F00FF00, p - 1, 0x7FFFFFFE, 123456789]), size=(N, stride))
    w = rng.integers(0, p, size=N + shift)
    ctx = wr.wr_create(0)
    dt = torch.from_numpy(t.astype(np.int32)).cuda()
    dw = torch.from_numpy(w.astype(np.int32)).cuda()
    G = torch.empty((m, m), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for mode in (0, 1) if m >= 16 or stride <= 16 else (0,):
        wr.wr_set_tensor_projection(ctx, mode)
        wr.wr_gram_device(ctx, p, N, m, m, dt, stride, yoff, dw.data_ptr() + 4 * shift, G)
        assert np.array_equal(G.cpu().numpy().astype(np.int64), _ref(t, w[shift:], m, m, yoff, p)), mode
    wr.wr_destroy(ctx)


def test_more_rows_than_a_blocks_sums_hold(wr):
    """Above 127 drains of 256 rows times two blocks an SM the grid grows."""
    p, m = 2147483629, 16
    N = 11_000_003
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    t = torch.randint(0, p, (N, m), generator=g, device="cuda", dtype=torch.int32)
    t[: N // 2] = p - 1
    w = torch.randint(0, p, (N,), generator=g, device="cuda", dtype=torch.int32)
    G = torch.empty((m, m), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    ctx = wr.wr_create(0)
    out = []
    for mode in (0, 1):
        wr.wr_set_tensor_projection(ctx, mode)
        wr.wr_gram_device(ctx, p, N, m, m, t, m, 0, w, G)
        out.append(G.cpu().clone())
    wr.wr_destroy(ctx)
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("m,stride,yoff", [(32, 32, 0), (20, 32, 0), (32, 64, 32), (16, 32, 16), (8, 8, 0)])
@pytest.mark.parametrize("groups", [1, 2, 3, 5])
def test_groups_of_tiles_in_both_accumulators(wr, m, stride, yoff, groups):
    """Blocks of one to a few groups of four tiles, and of a tile more or less."""
    p = 2147483629
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda")
    g.manual_seed(m + groups)
    ctx = wr.wr_create(0)
    for tiles in (4 * groups - 1, 4 * groups, 4 * groups + 1):
        N = 2 * sms * 64 * tiles - 7
        t = torch.randint(0, p, (N, stride), generator=g, device="cuda", dtype=torch.int32)
        t[: N // 4] = p - 1
        w = torch.randint(0, p, (N,), generator=g, device="cuda", dtype=torch.int32)
        G = torch.empty((m, m), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        out = []
        for mode in (0, 1):
            wr.wr_set_tensor_projection(ctx, mode)
            wr.wr_gram_device(ctx, p, N, m, m, t, stride, yoff, w, G)
            out.append(G.cpu().clone())
        assert torch.equal(out[0], out[1]), tiles
    wr.wr_destroy(ctx)


@pytest.mark.parametrize("m,stride,yoff", [(1, 1, 0), (2, 4, 2), (3, 4, 0), (5, 16, 8), (8, 8, 0), (12, 16, 0), (16, 32, 16),
                                           (32, 32, 0)])
@pytest.mark.parametrize("p", [3, 65521, 1073741789, 2147483647])
def test_integer_products(wr, m, stride, yoff, p):
    """The multiply-add path: both folds, rows around its batches of rows, widths that
    divide a warp and others."""
    ctx = wr.wr_create(0)
    wr.wr_set_tensor_projection(ctx, 0)
    rng = np.random.default_rng(m)
    for N in (1, 31, 300, 20011, 60000):
        t = rng.integers(0, p, size=(N, stride))
        t[: N // 2] = p - 1
        w = rng.integers(0, p, size=N)
        w[: N // 3] = p - 1
        dt = torch.from_numpy(t.astype(np.uint32).view(np.int32)).cuda()
        dw = torch.from_numpy(w.astype(np.uint32).view(np.int32)).cuda()
        G = torch.empty((m, m), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        wr.wr_gram_device(ctx, p, N, m, m, dt, stride, yoff, dw, G)
        assert np.array_equal(G.cpu().numpy().astype(np.int64), _ref(t, w, m, m, yoff, p)), N
    wr.wr_destroy(ctx)
