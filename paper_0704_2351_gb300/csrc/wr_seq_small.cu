// The sequence loop of a small matrix on one cluster of thread blocks (Section 2.5
// step 2; the same passes and projections as wr_spmm.cu, for matrices whose blocks T
// and W fit in shared memory).
//
// A 2,000 x 1,800 matrix with a scalar block spends nothing on its 24,000 entries: an
// application was two passes and a Gram launch of a few microseconds of latency each,
// 9.6 us in all.  Here one launch runs `apps`
// applications: every block of the cluster holds T and W whole in its shared memory and
// the entries of every CS-th chunk of both layouts; a pass computes the block's rows
// from its copy and writes each residue to all the copies (distributed shared memory),
// and a cluster barrier ends it.  The Gram products of the block's rows of W run beside
// pass 2 and those of T beside the next application's pass 1, their sums leaving for
// s_raw one barrier later.  4.2 us an application (two cluster barriers and the
// passes' chains of shared-memory loads).
#include <cuda_runtime.h>

#include <algorithm>

#include "wr_internal.cuh"

namespace wr {

namespace {

constexpr int SS_CLUSTER = 8;    // blocks (the largest portable cluster)
constexpr int SS_THREADS = 512;
constexpr int SS_MAX_PAIRS = 256;  // m n
constexpr int SS_ROW = 1024;     // products of a long row that one warp takes

struct SmallArgs {
    SellView first, second;        // pass 1 (rows of W), pass 2 (rows of T)
    uint32_t *T;                   // N x nv in and out
    const uint32_t *scale1, *scale2;  // D2, D1^2
    const uint32_t *gw1, *gw2;     // Gram weights of W's and T's rows (Montgomery form)
    unsigned long long *s_raw;
    int64_t base, L;               // applications before this launch; terms
    int nv_log, m, n, yoff, apps;
    int cap1, cap2, nvent1;        // entry words a block may hold of each layout's chunks; long entries of the first
    ModP mp;
};

// Rows are kept in the order in which blocks produce them, so that a block's results
// are contiguous and its stores to the other copies whole lines (scattered ones took
// 6 of 8 us a pass): chunk c of a layout belongs to block c mod CS as its chunk
// c / CS, and its row r sits at position ((c mod CS) MC + c / CS) 32 + r; a long row
// (vector part) follows at CP + its first segment, with the block that its target
// picks.  The entries' columns are rewritten to positions when they are loaded.
struct Order {
    int MC, CP, positions;  // chunks a block may have, positions of chunk rows, all positions
};
__host__ __device__ inline Order order_of(int64_t nchunks, int64_t nseg) {
    Order o;
    o.MC = (int)((nchunks + SS_CLUSTER - 1) / SS_CLUSTER);
    o.CP = SS_CLUSTER * o.MC * SELL_C;
    o.positions = o.CP + (int)nseg;
    return o;
}
__device__ __forceinline__ int chunk_pos(const Order &o, int c) {
    return ((c % SS_CLUSTER) * o.MC + c / SS_CLUSTER) * SELL_C;
}
// the output row of segment g when it is the first of its row, else -1
__device__ __forceinline__ int long_row(const SellView &A, int g) {
    const uint32_t t = A.seg_row[g];
    if (g > 0 && A.seg_row[g - 1] == t) return -1;
    return (t & VROW_SPLIT) ? A.split_row[t & ~VROW_SPLIT] : (int)t;
}

// This block's rows of a layout in shared memory.
struct SmallPart {
    int chunks, base, nlong, nsplit;  // its chunks, the position of its first row, its long rows' pieces, rows in pieces
    int *len, *off;           // per chunk
    uint32_t *scale, *gw;     // per chunk row: scale (times R^2: one Montgomery product of
                              // the reduced sum gives scale * sum) and Gram weight
    int *lseg, *lpos, *loff, *llen;  // per piece of a long row (the row, or one of its segments): its first
                              // segment, the row's position, its entries
    int *lsplit;              // the row's sums in lacc (a row in pieces), else -1
    uint32_t *lscale, *lgw;   // the row's on its first piece, else 0 (scale in normal form)
    uint32_t *entries, *lentries;
};

__host__ __device__ inline int part_words(int64_t nchunks, int64_t nseg, int64_t nvent, int cap) {
    return order_of(nchunks, nseg).MC * (2 + 2 * SELL_C) + 7 * (int)nseg + cap + (int)nvent;
}

// rows of several segments whose sums a pass keeps
__host__ __device__ inline int split_sums(int64_t nsplit1, int64_t nsplit2) { return (int)max64(nsplit1, nsplit2); }

__device__ __forceinline__ SmallPart part_at(uint32_t *p, int64_t nchunks, int64_t nseg, int cap) {
    const int c = order_of(nchunks, nseg).MC, l = (int)nseg;
    SmallPart s;
    s.len = (int *)p;
    s.off = s.len + c;
    s.scale = (uint32_t *)(s.off + c);
    s.gw = s.scale + c * SELL_C;
    s.lseg = (int *)(s.gw + c * SELL_C);
    s.lpos = s.lseg + l;
    s.loff = s.lpos + l;
    s.llen = s.loff + l;
    s.lsplit = s.llen + l;
    s.lscale = (uint32_t *)(s.lsplit + l);
    s.lgw = s.lscale + l;
    s.entries = s.lgw + l;
    s.lentries = s.entries + cap;
    return s;
}

// map[row] = position of every row of A's output space
__device__ void map_rows(const SellView &A, int *map) {
    const Order o = order_of(A.nchunks, A.nseg);
    for (int x = threadIdx.x; x < (int)A.nchunks * SELL_C; x += SS_THREADS) {
        const uint32_t r = A.vrow[x];
        if (r != VROW_EMPTY) map[r] = chunk_pos(o, x / SELL_C) + x % SELL_C;
    }
    for (int g = threadIdx.x; g < (int)A.nseg; g += SS_THREADS) {
        const int r = long_row(A, g);
        if (r >= 0) map[r] = o.CP + g;
    }
}

// t (one copy) <- rows in global memory, or back; begin, step: this caller's share
template <bool LOAD>
__device__ void move_rows(const SellView &A, uint32_t *t, uint32_t *rows, int nv_log, int begin, int step) {
    const Order o = order_of(A.nchunks, A.nseg);
    const int nv = 1 << nv_log, n1 = (int)A.nchunks * SELL_C, all = n1 + (int)A.nseg;
    for (int x = begin; x < all << nv_log; x += step) {
        const int y = x >> nv_log, b = x & (nv - 1);
        int r, pos;
        if (y < n1) {
            const uint32_t v = A.vrow[y];
            r = v == VROW_EMPTY ? -1 : (int)v;
            pos = chunk_pos(o, y / SELL_C) + y % SELL_C;
        } else {
            r = long_row(A, y - n1);
            pos = o.CP + y - n1;
        }
        if (r < 0) continue;
        if (LOAD) t[(pos << nv_log) + b] = rows[((int64_t)r << nv_log) + b];
        else rows[((int64_t)r << nv_log) + b] = t[(pos << nv_log) + b];
    }
}

// map, omap: positions of the gathered space's rows and of the output's; counts: three
// shared counters
__device__ void part_load(SmallPart &s, const SellView &A, int cap, int rank, const uint32_t *scale, const uint32_t *gw,
                          const int *map, const int *omap, int *counts, int nv_log, const ModP &mp) {
    const int tid = threadIdx.x, lane = tid & 31;
    const Order o = order_of(A.nchunks, A.nseg);
    s.chunks = A.nchunks > rank ? (int)((A.nchunks - rank + SS_CLUSTER - 1) / SS_CLUSTER) : 0;
    s.base = rank * o.MC * SELL_C;
    if (tid < 3) counts[tid] = 0;
    for (int c = tid; c < s.chunks; c += SS_THREADS) s.len[c] = A.chunk_len[rank + c * SS_CLUSTER];
    __syncthreads();
    if (tid == 0) {
        int f = 0;
        for (int c = 0; c < s.chunks; c++) {
            s.off[c] = f;
            f += s.len[c] * SELL_C;
        }
    }
    for (int x = tid; x < s.chunks * SELL_C; x += SS_THREADS) {
        const uint32_t r = A.vrow[(int64_t)(rank + x / SELL_C * SS_CLUSTER) * SELL_C + x % SELL_C];
        s.scale[x] = r == VROW_EMPTY ? 0u : to_mont(to_mont(scale[r], mp), mp);
        s.gw[x] = r == VROW_EMPTY ? 0u : gw[r];
    }
    for (int g = tid; g < (int)A.nseg; g += SS_THREADS) {
        const uint32_t t = A.seg_row[g];
        const int r = (t & VROW_SPLIT) ? A.split_row[t & ~VROW_SPLIT] : (int)t;
        if (r % SS_CLUSTER != rank) continue;
        const int g0 = omap[r] - o.CP;
        const bool first = g == g0;
        int len = 0;  // the row's entries, counted as far as SS_ROW products
        for (int h = g0; h < (int)A.nseg && A.seg_row[h] == t && len << nv_log <= SS_ROW; h++) len += A.seg_len[h];
        const bool pieces = len << nv_log > SS_ROW && (t & VROW_SPLIT);
        if (!pieces && !first) continue;
        const int k = atomicAdd(&counts[0], 1);
        s.lseg[k] = g;
        s.lpos[k] = omap[r];
        s.lsplit[k] = pieces ? (int)(t & ~VROW_SPLIT) : -1;
        if (pieces && first) atomicAdd(&counts[2], 1);
        s.llen[k] = pieces ? A.seg_len[g] : len;
        s.loff[k] = atomicAdd(&counts[1], s.llen[k]);
        s.lscale[k] = first ? scale[r] : 0u;
        s.lgw[k] = first ? gw[r] : 0u;
    }
    __syncthreads();
    s.nlong = counts[0];
    s.nsplit = counts[2];
    for (int c = tid >> 5; c < s.chunks; c += SS_THREADS / 32) {
        const uint32_t *src = A.entries + A.chunk_off[rank + c * SS_CLUSTER];
        for (int j = lane; j < s.len[c] * SELL_C && s.off[c] + j < cap; j += 32) {
            const uint32_t e = src[j];  // (padding: value 0 at column 0)
            s.entries[s.off[c] + j] = ((uint32_t)map[e >> 8] << 8) | (e & 0xFFu);
        }
    }
    for (int k = tid >> 5; k < s.nlong; k += SS_THREADS / 32) {
        const uint32_t *src = A.ventries + A.seg_start[s.lseg[k]];  // a row's segments are contiguous
        for (int j = lane; j < s.llen[k]; j += 32) {
            const uint32_t e = src[j];
            s.lentries[s.loff[k] + j] = ((uint32_t)map[e >> 8] << 8) | (e & 0xFFu);
        }
    }
    __syncthreads();
}

// The long rows of a pass: a warp a piece, nv lanes side by side along each entry's row of
// x and 32 / nv entries at a time (a warp on one column at a time put its lanes nv words
// apart, on one bank).  Rows of up to SS_ROW products are one piece; longer ones go by
// segments, summed in lacc, for a block barrier more.  64 applications with a full row
// and a full column, before (a warp a row, column after column) and so: 1,000 x 900,
// blocks of 8 2,970 -> 951 us, symmetric blocks of 4 688 -> 439, scalar 421 -> 351,
// symmetric scalar 321 -> 334; a copy of the loop for every width cost matrices without
// long rows 3 % more than it gave.
__device__ __forceinline__ void long_rows(const SmallPart &s, const uint32_t *x, uint32_t *y, unsigned long long *lacc, int nv_log,
                                          const ModP &mp) {
    const int nv = 1 << nv_log, lane = threadIdx.x & 31, b = lane & (nv - 1), e0 = lane >> nv_log, eps = 32 >> nv_log;
    const uint32_t *xb = x + b;
    for (int k = threadIdx.x >> 5; k < s.nlong; k += SS_THREADS / 32) {
        const uint32_t *w = s.lentries + s.loff[k];
        const int len = s.llen[k], split = s.lsplit[k];
        int64_t acc = 0;
        auto products = [&](const uint32_t (&en)[8]) {
            uint32_t v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = xb[(en[u] >> 8) << nv_log];
#pragma unroll
            for (int u = 0; u < 8; u++) acc += (int64_t)(int)(int8_t)(en[u] & 0xFFu) * (int32_t)v[u];
        };
        uint32_t en[8];
        int j = e0;
        for (; j + 7 * eps < len; j += 8 * eps) {
#pragma unroll
            for (int u = 0; u < 8; u++) en[u] = w[j + u * eps];
            products(en);
        }
        if (j < len) {
#pragma unroll
            for (int u = 0; u < 8; u++) en[u] = j + u * eps < len ? w[j + u * eps] : 0u;  // (value 0 at position 0)
            products(en);
        }
        __syncwarp();
#pragma unroll
        for (int h = 16; h > 0; h >>= 1)
            if (h >= nv) acc += __shfl_xor_sync(0xffffffffu, acc, h);
        if (split < 0) {
            const uint32_t o = mulm(red_s64(acc, mp), s.lscale[k], mp);
            for (int c = e0; c < SS_CLUSTER; c += eps) st_cluster(y + (s.lpos[k] << nv_log) + b, (uint32_t)c, o);
        } else if (lane < nv) {
            atomicAdd(&lacc[(split << nv_log) + lane], (unsigned long long)acc);
        }
    }
    if (s.nsplit > 0) {  // (the same for the block)
        __syncthreads();
        for (int it = threadIdx.x; it < s.nlong << nv_log; it += SS_THREADS) {
            const int k = it >> nv_log, c = it & (nv - 1);
            if (s.lsplit[k] < 0 || s.lscale[k] == 0u) continue;  // (scales are units: 0 off the first piece)
            unsigned long long &sum = lacc[(s.lsplit[k] << nv_log) + c];
            const uint32_t o = mulm(red_s64((int64_t)sum, mp), s.lscale[k], mp);
            sum = 0ull;
            for (int d = 0; d < SS_CLUSTER; d++) st_cluster(y + (s.lpos[k] << nv_log) + c, (uint32_t)d, o);
        }
    }
}

// y = scale (A x) for the block's rows, to every block's copy of y; lacc: zero before and after
__device__ __forceinline__ void small_pass(const SmallPart &s, const uint32_t *x, uint32_t *y, unsigned long long *lacc,
                                           int nv_log, const ModP &mp) {
    const uint64_t off = (uint64_t)mp.p << 23;  // (as row_out: |sum| < 2^23 p)
    const int nv = 1 << nv_log;
    for (int it = threadIdx.x; it < s.chunks << (5 + nv_log); it += SS_THREADS) {
        const int c = it >> (5 + nv_log), e = it & ((SELL_C << nv_log) - 1), r = e >> nv_log, b = e & (nv - 1);
        const uint32_t *w = s.entries + s.off[c] + r, *xb = x + b;
        const int len = s.len[c];
        int64_t acc = 0;
        int j = 0;
        for (; j + 4 <= len; j += 4) {
            uint32_t en[4], v[4];
#pragma unroll
            for (int u = 0; u < 4; u++) en[u] = w[(j + u) * SELL_C];
#pragma unroll
            for (int u = 0; u < 4; u++) v[u] = xb[(en[u] >> 8) << nv_log];
#pragma unroll
            for (int u = 0; u < 4; u++) acc += (int64_t)(int)(int8_t)(en[u] & 0xFFu) * (int32_t)v[u];
        }
        for (; j < len; j++) {
            const uint32_t en = w[j * SELL_C];
            acc += (int64_t)(int)(int8_t)(en & 0xFFu) * (int32_t)xb[(en >> 8) << nv_log];
        }
        const uint32_t o = mont_mul(mont_redc((uint64_t)acc + off, mp), s.scale[(c << 5) + r], mp);
        uint32_t *dst = y + ((s.base + (c << 5) + r) << nv_log) + b;
#pragma unroll
        for (int k = 0; k < SS_CLUSTER; k++) st_cluster(dst, (uint32_t)k, o);
    }
    long_rows(s, x, y, lacc, nv_log, mp);
}

// the block's rows' part of sum_r gw_r t_r[0..m)^T t_r[yoff..yoff + n) into sums[m n]
__device__ __forceinline__ void small_gram(const SmallPart &s, const uint32_t *t, int nv_log, int m, int n, int yoff,
                                           unsigned long long *sums, const ModP &mp) {
    int pp_log = 0;
    while ((1 << pp_log) < m * n) pp_log++;
    const int pair = threadIdx.x & ((1 << pp_log) - 1), rg = threadIdx.x >> pp_log, nrg = SS_THREADS >> pp_log;
    const int a = pair / n, b = pair - a * n;
    unsigned long long acc = 0;
    if (pair < m * n)
        for (int x = rg; x < s.chunks * SELL_C + s.nlong; x += nrg) {
            const int k = x - s.chunks * SELL_C;  // (a long row's number)
            const uint32_t *row = t + ((k < 0 ? s.base + x : s.lpos[k]) << nv_log);
            acc = fold1(madw(mont_mul(k < 0 ? s.gw[x] : s.lgw[k], row[a], mp), row[yoff + b], acc), mp.r1);
        }
    acc = red64(acc, mp);
    for (int o = 1 << pp_log; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (pair < m * n && (int)(threadIdx.x & 31) < (1 << pp_log) && acc) atomicAdd(&sums[pair], acc);
}

__global__ void __launch_bounds__(SS_THREADS, 1) k_seq_small(const __grid_constant__ SmallArgs g) {
    extern __shared__ __align__(16) uint32_t ssm[];
    __shared__ unsigned long long sums[2][SS_MAX_PAIRS];
    const int tid = threadIdx.x, rank = (int)cluster_rank(), P = g.m * g.n;
    const ModP mp = g.mp;
    const int nT = order_of(g.second.nchunks, g.second.nseg).positions << g.nv_log;
    const int nW = order_of(g.first.nchunks, g.first.nseg).positions << g.nv_log;
    unsigned long long *lacc = reinterpret_cast<unsigned long long *>(ssm);
    const int nacc = split_sums(g.first.nsplit, g.second.nsplit) << g.nv_log;
    uint32_t *Ts = ssm + 2 * nacc, *Ws = Ts + nT, *p1 = Ws + nW;
    SmallPart s1 = part_at(p1, g.first.nchunks, g.first.nseg, g.cap1);
    SmallPart s2 = part_at(p1 + part_words(g.first.nchunks, g.first.nseg, g.nvent1, g.cap1), g.second.nchunks, g.second.nseg,
                           g.cap2);
    __shared__ int counts[3];
    // the copies' memory holds the positions first (a position per row: they fit)
    map_rows(g.second, (int *)Ts);
    map_rows(g.first, (int *)Ws);
    __syncthreads();
    part_load(s1, g.first, g.cap1, rank, g.scale1, g.gw1, (const int *)Ts, (const int *)Ws, counts, g.nv_log, mp);
    part_load(s2, g.second, g.cap2, rank, g.scale2, g.gw2, (const int *)Ws, (const int *)Ts, counts, g.nv_log, mp);
    for (int x = tid; x < nT + nW; x += SS_THREADS) Ts[x] = 0u;
    for (int x = tid; x < nacc; x += SS_THREADS) lacc[x] = 0ull;
    for (int x = tid; x < 2 * SS_MAX_PAIRS; x += SS_THREADS) sums[x / SS_MAX_PAIRS][x % SS_MAX_PAIRS] = 0ull;
    __syncthreads();
    move_rows<true>(g.second, Ts, g.T, g.nv_log, tid, SS_THREADS);
    // finished sums of term k to s_raw, and back to zero
    auto flush = [&](unsigned long long *q, int64_t k) {
        for (int x = tid; x < P; x += SS_THREADS) {
            const unsigned long long v = q[x];
            q[x] = 0ull;
            if (v && k >= 0 && k < g.L) atomicAdd(g.s_raw + k * P + x, v);
        }
    };
    cluster_arrive();  // every block has loaded T and cleared W before anybody writes a copy
    cluster_wait();
    for (int i = 0; i < g.apps; i++) {
        const int64_t k = 2 * (g.base + i);  // T = D1 A~^(base + i) Y: term k
        if (i > 0) flush(sums[1], k - 1);      // W of the application before
        small_pass(s1, Ts, Ws, lacc, g.nv_log, mp);
        if (i > 0) small_gram(s2, Ts, g.nv_log, g.m, g.n, g.yoff, sums[0], mp);
        cluster_arrive();
        cluster_wait();
        if (i > 0) flush(sums[0], k);
        small_pass(s2, Ws, Ts, lacc, g.nv_log, mp);
        small_gram(s1, Ws, g.nv_log, g.m, g.n, g.yoff, sums[1], mp);
        cluster_arrive();
        cluster_wait();
    }
    const int64_t k = 2 * (g.base + g.apps);
    flush(sums[1], k - 1);
    small_gram(s2, Ts, g.nv_log, g.m, g.n, g.yoff, sums[0], mp);
    __syncthreads();
    flush(sums[0], k);
    move_rows<false>(g.second, Ts, g.T, g.nv_log, rank * SS_THREADS + tid, SS_CLUSTER * SS_THREADS);
}

// A block's entry words of a layout: chunks are sorted by length, so dealing them out in
// turn leaves a block at most one longest chunk above the mean.
int part_cap(const Sell &S) { return (int)(S.nslots / SS_CLUSTER) + LIGHT_MAX * SELL_C; }

size_t small_bytes(const Sell &first, const Sell &second, int nv) {
    return sizeof(uint32_t) *
           ((size_t)(order_of(first.nchunks, first.nseg).positions + order_of(second.nchunks, second.nseg).positions +
                     2 * split_sums(first.nsplit, second.nsplit)) * nv +
            part_words(first.nchunks, first.nseg, first.nvent, part_cap(first)) +
            part_words(second.nchunks, second.nseg, second.nvent, part_cap(second)));
}

// dynamic shared memory beside the kernel's own arrays (the same for every launch, so
// that threads launching at once agree on the kernel's attribute)
size_t max_dynamic(const wr_ctx *ctx) { return std::min<size_t>(ctx->smem_optin, 227 * 1024) - 8 * 1024; }

}  // namespace

// Matrices and blocks that the small loop takes: packed entries, both blocks and a block's
// entries in shared memory, two terms per application, and sizes whose pass is
// shorter than the launches it saves: the limit is the shared memory, near which an
// application of 6,500 x 6,000 with scalar blocks takes 7.1 us against 10.5 and one of
// 1,000 x 900 with blocks of 4 6.2 against 10.6.  (Symmetric blocks of 16, whose products
// the passes take to the tensor cores, meet earlier: 257 terms of 500 x 450 1.62 ms
// against 2.00, of 800 x 720 2.50 against 2.02; of 8, 1,500 x 1,350 1.55 against 1.68,
// 2,000 x 1,800 1.91 against 1.69.)
bool seq_small_fits(const wr_ctx *ctx, const Sell &first, const Sell &second, const Resolved &r) {
    if (!(r.gram || r.paired) || r.m * r.n > SS_MAX_PAIRS) return false;
    if (first.wide || second.wide) return false;
    if ((r.N + r.M) * r.nvs > (int64_t)1 << 16 || first.nslots + second.nslots + first.nvent + second.nvent > (int64_t)1 << 20)
        return false;
    const size_t need = small_bytes(first, second, r.nvs);
    return need <= max_dynamic(ctx);
}

wr_status launch_seq_small(wr_ctx *ctx, const Sell &first, const Sell &second, const Resolved &r, const ModP &mp, uint32_t *T,
                           const uint32_t *scale1, const uint32_t *scale2, const uint32_t *gw1, const uint32_t *gw2,
                           unsigned long long *s_raw, int64_t base, int apps, int64_t L) {
    SmallArgs g{};
    g.first = view(first);
    g.second = view(second);
    g.T = T;
    g.scale1 = scale1;
    g.scale2 = scale2;
    g.gw1 = gw1;
    g.gw2 = gw2;
    g.s_raw = s_raw;
    g.base = base;
    g.L = L;
    while ((1 << g.nv_log) < r.nvs) g.nv_log++;
    g.m = r.m;
    g.n = r.n;
    g.yoff = r.paired ? r.nv : 0;
    g.apps = apps;
    g.cap1 = part_cap(first);
    g.cap2 = part_cap(second);
    g.nvent1 = (int)first.nvent;
    g.mp = mp;
    const size_t smem = small_bytes(first, second, r.nvs);
    WR_CUDA(cudaFuncSetAttribute(k_seq_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_dynamic(ctx)));
    cudaLaunchConfig_t lc{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = SS_CLUSTER;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    lc.gridDim = dim3(SS_CLUSTER);
    lc.blockDim = dim3(SS_THREADS);
    lc.dynamicSmemBytes = smem;
    lc.stream = ctx->stream;
    lc.attrs = &at;
    lc.numAttrs = 1;
    WR_CUDA(cudaLaunchKernelEx(&lc, k_seq_small, g));
    WR_LAUNCHED(ctx);
    return WR_OK;
}

}  // namespace wr
