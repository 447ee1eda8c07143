"""Measured cases of the block Wiedemann rank path, through the public binding.

Every case is one call (or the few calls a program makes together) of
paper_0704_2351_gb300.wr on inputs made on the GPU from a seed.  Sizes are
those of the synthetic workloads (paper_0704_2351_gb300/synth.py), the bench
and the tests:

  2,000 x 1,800          12 entries a row, scalar blocks;
  200,000 x 180,000      20 entries a row, power-law columns, blocks of 8;
  1,900,000 x 1,950,000  Poisson(19.5) row lengths, blocks of 32;
  chain matrices         4,000 to 284,000 rows, blocks of 8, several primes;
  served requests        1,000 to 500,000 rows, 10 to 20 entries a row,
                         blocks of 16.

All results are whole numbers (residues, degrees, ranks) and exact.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0704_2351_gb300 import wr

PRIMES = (65521, 65537, 1073741789, 2147483629, 2147483647)
P16, P30, P31 = 65521, 1073741789, 2147483629
EXACT_CELLS = 6e10  # entry products that exact() computes at most


def listed():
    return [
        # the smallest call: one application of the black box of the scalar workload (latency)
        dict(name="apply_2000_w1", kind="apply", rows=2000, cols=1800, per_row=12, skew=False, vmax=3, width=1,
             side=-1, prime=P16),
        # a matrix in host memory is read in and applied once (ingest of the power-law matrix)
        dict(name="load_200k_w8", kind="load", rows=200000, cols=180000, per_row=20, skew=True, vmax=3, width=8,
             side=-1, prime=P30),
        # the iteration of the power-law matrix with independent X (a few graphs of 45,002 terms)
        dict(name="sequence_200k_b8", kind="sequence", rows=200000, cols=180000, per_row=20, skew=True, vmax=3, m=8,
             n=8, symmetric=False, side=-1, prime=P30, terms=513),
        # the largest served request's iteration: block 16, independent X
        dict(name="sequence_500k_b16", kind="sequence", rows=500000, cols=450000, per_row=15, skew=False, vmax=3,
             m=16, n=16, symmetric=False, side=-1, prime=P31, terms=257),
        # the bench step's iteration: block 32, X = Y, the gathered block twice the L2
        dict(name="sequence_1900k_b32", kind="sequence", rows=1900000, cols=1950000, per_row=19.5, skew=False, vmax=4,
             m=32, n=32, symmetric=True, side=-1, prime=P31, terms=129),
        # one projection of the largest workload with independent X (rows of 64 residues)
        dict(name="gram_1900k_b32", kind="gram", N=1900000, m=32, n=32, paired=True, prime=P31),
        # the sigma-basis of blocks of 8 (a quarter of the power-law matrix's orders)
        dict(name="sigma_b8_11252", kind="sigma", m=8, n=8, terms=11252, prime=P30),
        # the sigma-basis of blocks of 32: PM-Basis with its leaves and products
        dict(name="sigma_b32_4098", kind="sigma", m=32, n=32, terms=4098, prime=P31),
        # a basis product of that recursion
        dict(name="product_64_2049", kind="product", r=64, s=64, t=64, na=2049, nb=2049, lo=0, hi=4097, prime=P31),
        # whole rank calls: the scalar workload, and a served request of middle size
        dict(name="rank_2000_b1", kind="rank", rows=2000, cols=1800, per_row=12, rank=1500, m=1, n=1, symmetric=False,
             prime=P30),
        dict(name="rank_20k_b16", kind="rank", rows=20000, cols=18000, per_row=15, rank=17000, m=16, n=16,
             symmetric=False, prime=P31),
        # rank over Q of a chain matrix: four primes in one batch call
        dict(name="batch_6000_b8x4", kind="batch", rows=6000, cols=5000, per_row=10, rank=4200, m=8, n=8, jobs=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, lo, hi):
    rows = _log_int(rng, lo, hi)
    return rows, max(2, int(rows * rng.uniform(0.8, 1.1)))


def draw(rng):
    kind = rng.choice(["apply", "apply", "load", "sequence", "sequence", "sequence", "gram", "sigma", "sigma",
                       "product", "rank", "rank", "batch"])
    prime = rng.choice(PRIMES)
    if kind in ("apply", "load"):
        rows, cols = _shape(rng, 1000, 500000 if kind == "apply" else 300000)
        vmax = rng.choice([3, 3, 3, 4, 300])
        return dict(kind=kind, rows=rows, cols=cols, per_row=rng.randint(10, 20),
                    skew=vmax < 300 and rng.random() < 0.5, vmax=vmax, width=rng.randint(1, 32), side=rng.choice([-1, -1, 0, 1]),
                    prime=prime)
    if kind == "sequence":
        rows, cols = _shape(rng, 1000, 500000)
        m = n = rng.choice([1, 2, 4, 8, 16, 32, rng.randint(1, 32)])
        if rng.random() < 0.2:
            n = rng.randint(1, 32)
        vmax = rng.choice([3, 3, 3, 4, 300])
        return dict(kind=kind, rows=rows, cols=cols, per_row=rng.randint(10, 20),
                    skew=vmax < 300 and rng.random() < 0.4, vmax=vmax, m=m, n=n, symmetric=m == n and rng.random() < 0.4,
                    side=rng.choice([-1, -1, 0, 1]), prime=prime, terms=rng.randint(33, 257))
    if kind == "gram":
        m = rng.choice([1, 4, 8, 16, 32, rng.randint(1, 32)])
        return dict(kind=kind, N=_log_int(rng, 1000, 1950000), m=m, n=m, paired=rng.random() < 0.5, prime=prime)
    if kind == "sigma":
        m = n = rng.choice([1, 2, 4, 8, 16, 32, rng.randint(1, 32)])
        if rng.random() < 0.2:
            n = rng.randint(max(1, m // 2), min(32, 2 * m))
        return dict(kind=kind, m=m, n=n, terms=_log_int(rng, 100, 8000 if m + n <= 32 else 3000), prime=prime)
    if kind == "product":
        r, s, t = (rng.choice([1, 4, 8, 16, 32, 64, rng.randint(1, 64)]) for _ in range(3))
        na, nb = _log_int(rng, 64, 4096), _log_int(rng, 64, 4096)
        full = na + nb - 1
        lo, hi = (0, full) if rng.random() < 0.5 else (nb // 2, nb // 2 + max(1, na // 2))
        return dict(kind=kind, r=r, s=s, t=t, na=na, nb=nb, lo=lo, hi=hi, prime=prime)
    b = rng.choice([2, 4, 8, 16, rng.randint(2, 16)]) if kind == "rank" else rng.choice([2, 4, 8, rng.randint(2, 8)])
    rows, cols = _shape(rng, 1000, 1250 * b if kind == "rank" else 1000 * b)
    case = dict(kind=kind, rows=rows, cols=cols, per_row=rng.randint(8, 15),
                rank=int(min(rows, cols) * rng.uniform(0.7, 0.95)), m=b, n=b)
    if kind == "rank":
        return dict(case, symmetric=rng.random() < 0.3, prime=rng.choice([P30, P31, 2147483647]))
    return dict(case, jobs=rng.randint(2, 4))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFFFFFFFFFF)
    return g


def _rand_int(g, lo, hi, count):
    return torch.randint(lo, hi, (count,), generator=g, device="cuda", dtype=torch.int64)


def _values(g, count, vmax):
    """+-1 (95 %), else +-1 .. +-vmax."""
    sign = 2 * _rand_int(g, 0, 2, count) - 1
    big = _rand_int(g, 1, vmax + 1, count)
    unit = torch.rand(count, generator=g, device="cuda") < 0.95
    return torch.where(unit, sign, sign * big)


def _csr(rows, cols, r, c, v):
    """Sums duplicates, drops zeros; row pointers int64, columns and values int32, on the GPU."""
    key, where = torch.unique(r * cols + c, return_inverse=True)
    val = torch.zeros(len(key), dtype=torch.int64, device="cuda").index_add_(0, where, v)
    key, val = key[val != 0], val[val != 0]
    ptr = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(key // cols, minlength=rows), 0)
    return ptr, (key % cols).to(torch.int32), val.to(torch.int32)


def _random_matrix(case, g):
    """Poisson row lengths; uniform or power-law columns."""
    rows, cols = case["rows"], case["cols"]
    lens = torch.poisson(torch.full((rows,), float(case["per_row"]), device="cuda"), generator=g).to(torch.int64)
    r = torch.repeat_interleave(torch.arange(rows, device="cuda"), lens)
    nnz = len(r)
    if case["skew"]:
        w = torch.arange(1, cols + 1, device="cuda", dtype=torch.float64) ** (-1.0 / 1.1)
        cdf = torch.cumsum(w, 0)
        u = torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
        perm = torch.randperm(cols, generator=g, device="cuda")
        c = perm[torch.searchsorted(cdf, u).clamp_(max=cols - 1)]
    else:
        c = _rand_int(g, 0, cols, nnz)
    return _csr(rows, cols, r, c, _values(g, nnz, case["vmax"]))


def _planted_matrix(rows, cols, rank, per_row, g):
    """`rank` base rows, triangular with +-1 on their pivot columns, and rows that combine three of them."""
    k = per_row - 1
    base = torch.arange(rank, device="cuda")
    off = torch.rand((rank, k), generator=g, device="cuda", dtype=torch.float64)
    after = base[:, None] + 1 + (off * (cols - 1 - base[:, None])).to(torch.int64)  # positions past the pivot's
    pos = torch.cat([base[:, None], after.clamp_(max=cols - 1)], 1)
    val = _values(g, rank * per_row, 3).reshape(rank, per_row)
    val[:, 0] = 2 * _rand_int(g, 0, 2, rank) - 1
    val[:, 1:][pos[:, 1:] <= base[:, None]] = 0
    nd = rows - rank
    pick = _rand_int(g, 0, rank, 3 * nd).reshape(nd, 3)
    coef = (_rand_int(g, 1, 3, 3 * nd) * (2 * _rand_int(g, 0, 2, 3 * nd) - 1)).reshape(nd, 3)
    dpos = pos[pick].reshape(nd, -1)
    dval = (val[pick] * coef[:, :, None]).reshape(nd, -1)
    row_of = torch.randperm(rows, generator=g, device="cuda")
    col_of = torch.randperm(cols, generator=g, device="cuda")
    dep = torch.arange(rank, rows, device="cuda")
    r = torch.cat([base.repeat_interleave(per_row), dep.repeat_interleave(3 * per_row)])
    c = torch.cat([pos.reshape(-1), dpos.reshape(-1)])
    v = torch.cat([val.reshape(-1), dval.reshape(-1)])
    return _csr(rows, cols, row_of[r], col_of[c], v)


class _Handle:
    """A context and the matrix loaded through it, given back with the state."""

    def __init__(self):
        self.ctx, self.mat = wr.wr_create(0), None

    def load(self, rows, cols, csr):
        ptr, ci, va = csr
        torch.cuda.synchronize()
        self.mat = wr.wr_matrix_load_csr_device(self.ctx, rows, cols, len(ci), ptr, ci, va)

    def __del__(self):
        if self.mat is not None:
            wr.wr_matrix_free(self.mat)
        wr.wr_destroy(self.ctx)


def _residues(g, shape, prime):
    return torch.randint(0, prime, shape, generator=g, device="cuda", dtype=torch.int32)


def _padded(n):
    nv = 1
    while nv < n:
        nv *= 2
    return nv


def _draw_seed(seed):
    return 20070704 + seed


def _cols_side(case):
    return case["side"] == 0 or (case["side"] == -1 and case["rows"] >= case["cols"])


def _side_n(case):
    return case["cols"] if _cols_side(case) else case["rows"]


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    st = dict(case=case, h=_Handle())
    ctx = st["h"].ctx
    if kind in ("apply", "load"):
        csr = _random_matrix(case, g)
        N = _side_n(case)
        st["prm"] = wr.make_params(case["prime"], 1, case["width"], _draw_seed(seed), side=case["side"])
        st["x"] = _residues(g, (N, case["width"]), case["prime"])
        st["y"] = torch.empty_like(st["x"])
        if kind == "apply":
            st["h"].load(case["rows"], case["cols"], csr)
        else:
            st["csr"] = [a.cpu().numpy() for a in csr]
    elif kind == "sequence":
        st["h"].load(case["rows"], case["cols"], _random_matrix(case, g))
        proj = wr.WR_PROJ_SYMMETRIC if case["symmetric"] else wr.WR_PROJ_GENERIC
        st["prm"] = wr.make_params(case["prime"], case["m"], case["n"], _draw_seed(seed), projection=proj,
                                   side=case["side"])
        st["S"] = torch.empty((case["terms"], case["m"], case["n"]), dtype=torch.int32, device="cuda")
    elif kind == "gram":
        nv = _padded(case["n"])
        st["stride"], st["yoff"] = (2 * nv, nv) if case["paired"] else (nv, 0)
        st["t"] = _residues(g, (case["N"], st["stride"]), case["prime"])
        st["w"] = _residues(g, (case["N"],), case["prime"])
        st["G"] = torch.empty((case["m"], case["n"]), dtype=torch.int32, device="cuda")
    elif kind == "sigma":
        # the sequence of a planted matrix whose default length is about this one
        m, n, L = case["m"], case["n"], case["terms"]
        N = max(2, (L - 2) * m * n // (m + n))
        rank = max(1, int(0.94 * N))
        st["h"].load(N + N // 16, N, _planted_matrix(N + N // 16, N, rank, 6, g))
        prm = wr.make_params(case["prime"], m, n, _draw_seed(seed))
        st["S"] = torch.empty((L, m, n), dtype=torch.int32, device="cuda")
        wr.wr_sequence_device(ctx, st["h"].mat, prm, st["S"], L)
        st["P"] = torch.empty((L + 2, n, m + n), dtype=torch.int32, device="cuda")
        st["deg"] = torch.empty(m + n, dtype=torch.int32, device="cuda")
    elif kind == "product":
        st["A"] = _residues(g, (case["na"], case["r"], case["s"]), case["prime"])
        st["B"] = _residues(g, (case["nb"], case["s"], case["t"]), case["prime"])
        st["C"] = torch.empty((case["hi"] - case["lo"], case["r"], case["t"]), dtype=torch.int32, device="cuda")
    else:
        st["h"].load(case["rows"], case["cols"],
                     _planted_matrix(case["rows"], case["cols"], case["rank"], case["per_row"], g))
        want = wr.WR_WANT_SEQUENCE | wr.WR_WANT_GENERATOR
        proj = wr.WR_PROJ_SYMMETRIC if case.get("symmetric") else wr.WR_PROJ_GENERIC
        primes = [case["prime"]] if kind == "rank" else [1073741789, 1073741783, 1073741741, 1073741723][:case["jobs"]]
        st["prms"] = [wr.make_params(p, case["m"], case["n"], _draw_seed(seed) + j, projection=proj, want=want)
                      for j, p in enumerate(primes)]
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass

def _take(res, prm):
    gen, deg = wr.wr_result_generator(res, prm.n)
    out = dict(wr.wr_result_info(res), rank=wr.wr_result_rank(res), sequence=wr.wr_result_sequence(res, prm.m, prm.n),
               generator=gen, degrees=deg)
    wr.wr_result_free(res)
    return out


def run(state):
    case, ctx, mat = state["case"], state["h"].ctx, state["h"].mat
    kind = case["kind"]
    if kind == "apply":
        wr.wr_blackbox_apply_device(ctx, mat, state["prm"], state["x"], state["y"], case["width"])
        return state["y"]
    if kind == "load":
        ptr, ci, va = state["csr"]
        new = wr.wr_matrix_load_csr(ctx, case["rows"], case["cols"], ptr, ci, va)
        wr.wr_blackbox_apply_device(ctx, new, state["prm"], state["x"], state["y"], case["width"])
        nnz = wr.wr_matrix_info(new)["nnz"]
        wr.wr_matrix_free(new)
        return dict(nnz=nnz, y=state["y"])
    if kind == "sequence":
        wr.wr_sequence_device(ctx, mat, state["prm"], state["S"], case["terms"])
        return state["S"]
    if kind == "gram":
        wr.wr_gram_device(ctx, case["prime"], case["N"], case["m"], case["n"], state["t"], state["stride"],
                          state["yoff"], state["w"], state["G"])
        return state["G"]
    if kind == "sigma":
        L = case["terms"]
        wr.wr_sigma_basis_device(ctx, state["S"], L, case["m"], case["n"], case["prime"], state["P"], state["deg"],
                                 L + 1)
        return dict(P=state["P"], deg=state["deg"])
    if kind == "product":
        wr.wr_polymat_mul_device(ctx, case["prime"], state["A"], case["na"], state["B"], case["nb"], case["r"],
                                 case["s"], case["t"], case["lo"], case["hi"], state["C"])
        return state["C"]
    if kind == "rank":
        return _take(wr.wr_rank(ctx, mat, state["prms"][0]), state["prms"][0])
    outs = wr.wr_rank_batch(ctx, [mat] * len(state["prms"]), state["prms"])
    return [_take(r, p) for r, p in zip(outs, state["prms"])]


# ------------------------------------------------------------------ what a pass cannot do without

def _iteration_work(rows, cols, nnz, width, m, n, terms, two):
    """One application: both layouts' entries, the two blocks each read and written once, the projections."""
    apps = (terms - 1 + 1) // 2 if two else terms - 1
    io = 2 * (4 * nnz + 8 * width * (rows + cols))
    ops = 2 * (2 * nnz * width) + 2 * m * n * ((rows + cols) if two else min(rows, cols))
    return apps * io, apps * ops


def work(case):
    kind = case["kind"]
    if kind in ("apply", "load", "sequence"):
        rows, cols = case["rows"], case["cols"]
        nnz = rows * case["per_row"]
        if kind == "sequence":
            m, n = case["m"], case["n"]
            two = m == n
            width = n if case["symmetric"] or not two else 2 * n
            b, f = _iteration_work(rows, cols, nnz, width, m, n, case["terms"], two)
            return dict(bytes=b, flops=f)
        b = 2 * 4 * nnz + 4 * case["width"] * 2 * (rows + cols)
        return dict(bytes=b + (8 * nnz + 8 * rows if kind == "load" else 0), flops=4 * nnz * case["width"])
    if kind == "gram":
        nv = _padded(case["n"])
        return dict(bytes=case["N"] * 4 * (nv * (2 if case["paired"] else 1) + 1) + 4 * case["m"] * case["n"],
                    flops=2 * case["N"] * case["m"] * case["n"])
    if kind == "sigma":
        return _sigma_work(case["m"], case["n"], case["terms"])
    if kind == "product":
        r, s, t, na, nb = (case[k] for k in ("r", "s", "t", "na", "nb"))
        size = na + nb
        return dict(bytes=4 * (na * r * s + nb * s * t + (case["hi"] - case["lo"]) * r * t),
                    flops=2 * size * (r * s * t + (r * s + s * t + r * t) * math.log2(size)))
    rows, cols, m, n = case["rows"], case["cols"], case["m"], case["n"]
    N = min(rows, cols)
    L = -(-N // m) + -(-N // n) + 2
    sym = bool(case.get("symmetric"))
    b, f = _iteration_work(rows, cols, rows * case["per_row"], n if sym else 2 * n, m, n, L, True)
    s = _sigma_work(m, n, L)
    jobs = case.get("jobs", 1)
    return dict(bytes=jobs * (b + s["bytes"]), flops=jobs * (f + s["flops"]))


def _sigma_work(m, n, L):
    """The basis by recursive halving: the sequence read and the basis written once, one polynomial product a level."""
    q = m + n
    return dict(bytes=4 * L * (m * n + n * q / 2), flops=2 * L * math.log2(max(2, L)) * (m * q * q + q * q * q / 4))


# ------------------------------------------------------------------ the same in 64 bits

def _mix(x):
    """SplitMix64's output function (uint64 arrays, wrapping)."""
    with np.errstate(over="ignore"):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _stream(seed, tag, count):
    start = np.uint64((tag * 0x9E3779B97F4A7C15) & 0xFFFFFFFFFFFFFFFF) ^ np.uint64(seed)
    with np.errstate(over="ignore"):
        return _mix(_mix(np.asarray([start]))[0] + np.arange(count, dtype=np.uint64))


def _block(seed, tag, rows, width, prime):
    h = _stream(seed, tag, rows * width) % np.uint64(prime)
    return torch.from_numpy(h.astype(np.int64)).cuda().reshape(rows, width)


def _diagonal(seed, tag, count, prime):
    h = np.uint64(1) + _stream(seed, tag, count) % np.uint64(prime - 1)
    return torch.from_numpy(h.astype(np.int64)).cuda()


def _multiply(ptr, ci, va, rows, x, prime):
    """A x mod prime: sums of |value| < 2^9 times residues below 2^31 in int64."""
    out = torch.zeros((rows, x.shape[1]), dtype=torch.int64, device="cuda")
    r = torch.repeat_interleave(torch.arange(rows, device="cuda"), ptr[1:] - ptr[:-1])
    step = max(1, (1 << 27) // x.shape[1])
    for k in range(0, len(ci), step):
        s = slice(k, k + step)
        out.index_add_(0, r[s], va[s].to(torch.int64)[:, None] * x[ci[s].to(torch.int64)])
    return out % prime


def _transposed(ptr, ci, va, rows, cols):
    r = torch.repeat_interleave(torch.arange(rows, device="cuda"), ptr[1:] - ptr[:-1])
    order = torch.argsort(ci.to(torch.int64) * rows + r)
    tp = torch.zeros(cols + 1, dtype=torch.int64, device="cuda")
    tp[1:] = torch.cumsum(torch.bincount(ci.to(torch.int64), minlength=cols), 0)
    return tp, r[order].to(torch.int32), va[order]


def _operator(case, seed, prime):
    """x -> D1 A^T D2 A D1 x mod prime, on the smaller side or the one asked for."""
    rows, cols = case["rows"], case["cols"]
    a = _random_matrix(case, _gen(seed))
    first, second, N, M = (a, _transposed(*a, rows, cols), cols, rows)
    if not _cols_side(case):
        first, second, N, M = second, first, rows, cols
    d1 = _diagonal(_draw_seed(seed), 3, N, prime)[:, None]
    d2 = _diagonal(_draw_seed(seed), 4, M, prime)[:, None]

    def apply(x):
        w = _multiply(*first, M, d1 * x % prime, prime) * d2 % prime
        return _multiply(*second, N, w, prime) * d1 % prime

    return apply, N


def _cross(x, y, w, prime):
    """sum_r w_r x_r^T y_r mod prime, products below 2^62 reduced before they are summed."""
    out = torch.zeros((x.shape[1], y.shape[1]), dtype=torch.int64, device="cuda")
    step = max(1, (1 << 26) // (x.shape[1] * y.shape[1]))
    for k in range(0, len(x), step):
        s = slice(k, k + step)
        left = x[s] if w is None else x[s] * w[s, None] % prime
        out = (out + (left[:, :, None] * y[s][:, None, :] % prime).sum(0)) % prime
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply", "load"):
        apply, N = _operator(case, seed, case["prime"])
        g = _gen(seed)
        csr = _random_matrix(case, g)
        y = apply(_residues(g, (N, case["width"]), case["prime"]).to(torch.int64)).to(torch.int32)
        return y if kind == "apply" else dict(nnz=len(csr[1]), y=y)
    if kind == "sequence":
        prime, m, n = case["prime"], case["m"], case["n"]
        cost = case["rows"] * (2 * case["per_row"] * n + m * n)
        if cost * case["terms"] > EXACT_CELLS:
            return None
        apply, N = _operator(case, seed, prime)
        s = _draw_seed(seed)
        y = _block(s, 2, N, n, prime)
        x = y if case["symmetric"] else _block(s, 1, N, m, prime)
        out = torch.empty((case["terms"], m, n), dtype=torch.int32, device="cuda")
        for k in range(case["terms"]):
            out[k] = _cross(x, y, None, prime).to(torch.int32)
            if k + 1 < case["terms"]:
                y = apply(y)
        return out
    if kind == "gram":
        g, nv = _gen(seed), _padded(case["n"])
        stride, yoff = (2 * nv, nv) if case["paired"] else (nv, 0)
        t = _residues(g, (case["N"], stride), case["prime"]).to(torch.int64)
        w = _residues(g, (case["N"],), case["prime"]).to(torch.int64)
        return _cross(t[:, :case["m"]], t[:, yoff:yoff + case["n"]], w, case["prime"]).to(torch.int32)
    if kind in ("rank", "batch"):  # the planted rank
        one = dict(rank=case["rank"], deg_det=None, codeg=None, sum_delta=None, seq_len=None, sequence=None,
                   generator=None, degrees=None)
        return one if kind == "rank" else [one] * case["jobs"]
    return None
