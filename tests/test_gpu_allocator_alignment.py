"""A caller's allocator whose memory starts on 4-, 8- or 16-byte boundaries: the calls
give what they give with the library's own memory, and every piece goes back as it was
handed out."""
import numpy as np
import pytest

from paper_0704_2351_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = 2147483629


@pytest.fixture(scope="module")
def wr():
    from paper_0704_2351_gb300 import wr as m
    return m


def _calls(wr, ctx):
    rng = np.random.default_rng(2)
    A = synth.planted_sparse(900, 800, 600, row_len=7, seed=3)
    mat = wr.wr_matrix_load_csr(ctx, A.rows, A.cols, A.rowptr, A.colidx, A.vals)
    out = []
    for w in (1, 3, 8):
        x = torch.from_numpy(rng.integers(0, P, size=(A.cols, w)).astype(np.int32)).cuda()
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        wr.wr_blackbox_apply_device(ctx, mat, wr.make_params(P, 1, w, 5, side=0), x, y, w)
        out.append(y.cpu().numpy())
    for m, n in ((1, 1), (8, 4), (16, 16), (17, 17)):
        S = torch.empty((70, m, n), dtype=torch.int32, device="cuda")
        wr.wr_sequence_device(ctx, mat, wr.make_params(P, m, n, 7), S, 70)
        out.append(S.cpu().numpy())
    for m in (4, 20):
        r = wr.wr_rank(ctx, mat, wr.make_params(P, m, m, 9, want=wr.WR_WANT_GENERATOR))
        out += [wr.wr_result_rank(r), wr.wr_result_generator(r, m)[0]]
        wr.wr_result_free(r)
    a, b = (torch.from_numpy(rng.integers(0, P, size=(300, 5, 5)).astype(np.int32)).cuda() for _ in range(2))
    c = torch.empty((599, 5, 5), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    wr.wr_polymat_mul_device(ctx, P, a, 300, b, 300, 5, 5, 5, 0, 599, c)
    out.append(c.cpu().numpy())
    wr.wr_matrix_free(mat)
    return out


@pytest.mark.parametrize("off", [4, 8, 16])
def test_memory_on_any_boundary(wr, off):
    plain = wr.wr_create(0)
    want = _calls(wr, plain)
    wr.wr_destroy(plain)
    held = {}

    def alloc(n, stream):
        t = torch.empty(n + off, dtype=torch.uint8, device="cuda")
        held[t.data_ptr() + off] = (t, n)
        return t.data_ptr() + off

    def release(ptr, n, stream):
        torch.cuda.synchronize()
        assert held.pop(ptr)[1] == n

    ctx = wr.wr_create(0)
    wr.wr_set_allocator(ctx, alloc, release)
    for a, b in zip(_calls(wr, ctx), want):
        assert np.array_equal(a, b)
    wr.wr_destroy(ctx)
    assert not held
