// sigma-basis of the block Wiedemann sequence and the rank readout
// (Section 2.4 "sigma-basis computations", Section 2.5 steps 3 and 4).
//
// M-Basis (Giorgi, Jeannerod, Villard) computes an order-L sigma-basis M(x)
// of H(x) = [S(x) | -I_m] (m x q, q = m + n) for the shift (0^n, 1^m), one
// order at a time: the discrepancy Delta_k (coefficient k of H M) is
// column-reduced in order of (shifted degree, index), each column by the
// pivots found before it (pivot row = first nonzero row), and the pivot
// columns are multiplied by x.
//
// On the device the orders are processed in chunks of b:
//   window : E_i = coeff_{k0+i}(S P) - [i = 0] Qtop for i < b  (many blocks),
//            where P = first n rows of M and Qtop = coefficient k0 of the
//            last m rows (the only coefficient of those rows that can still
//            matter: their degree is below the shifted degree <= k0 + 1);
//   local  : the b orders of M-Basis on the window alone, building the
//            chunk's transform Mloc (q x q, degree <= b)  (one cluster);
//   apply  : P <- P Mloc  (many blocks).
// The transforms are those of the order-by-order algorithm (the product of
// the same elementary steps), so P and the degrees are bit-identical to it.
// The elimination runs fraction-free (col_j <- d_c col_j - d_j col_c) and
// divides by the accumulated column scale once per order, which removes the
// modular inverses from the sequential part.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "wr_internal.cuh"

namespace wr {

namespace {

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// The starting basis at x^0.  [S | -I_m] (deg_in == nullptr): P = [I_n | 0]
// (the first n rows), degrees (0^n, 1^m), Q = [0 | I_m].  A general residual
// (deg_in given, nr = q rows): P = I_q, the given degrees, Q = 0.
__global__ void k_init_basis(uint32_t *__restrict__ P, int nr, int n, int q, int32_t *__restrict__ deg,
                             const int32_t *__restrict__ deg_in, uint32_t *__restrict__ qtop, int m,
                             int *__restrict__ dmax) {
    for (int t = threadIdx.x; t < m * q || t < q; t += blockDim.x) {
        if (t < nr) P[(size_t)t * q + t] = 1;
        if (t < q) deg[t] = deg_in ? deg_in[t] : (t < n ? 0 : 1);
        if (t < m * q) {
            int a = t / q, c = t % q;
            qtop[t] = (!deg_in && c == n + a) ? 1u : 0u;
        }
    }
    if (threadIdx.x == 0) *dmax = 1;
}

// Early termination test of one chunk.  The generator candidates are the n
// columns of smallest shifted degree (ties by index); the chunk is quiet when
// each has degree <= k0 (so its -Q part lies below the chunk's orders and the
// window's E is its whole discrepancy) and zero discrepancy at every order of
// the chunk.  Such columns are never touched by the chunk's eliminations.
// *count: consecutive quiet orders so far, mirrored to a host-mapped slot.
__global__ void k_quiet(const uint32_t *__restrict__ E, int bb, int m, int n, int q,
                        const int32_t *__restrict__ deg, int64_t k0, long long *__restrict__ count,
                        long long *host_slot) {
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    for (int c = threadIdx.x; c < q; c += blockDim.x) {
        const int dc = deg[c];
        int before = 0;
        for (int c2 = 0; c2 < q; c2++) {
            const int d2 = deg[c2];
            before += (d2 < dc || (d2 == dc && c2 < c)) ? 1 : 0;
        }
        if (before >= n) continue;
        bool nz = dc > k0;
        for (int x = 0; x < bb * m && !nz; x++) nz = E[(size_t)x * q + c] != 0u;
        if (nz) atomicOr(&bad, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const long long v = bad ? 0 : *count + bb;
        *count = v;
        *(volatile long long *)host_slot = v;
    }
}

// ---- block-Toeplitz products mod p: the window and the transform product.
//
// C[R][c] = sum_{v in [v0, v1), f < nf} A[R][(v, f)] B[v nf + f][c] for R < rows,
// c < q, with A[R][(v, f)] = M[(R + (off - v) me) nf + f] (0 outside M's mrows rows):
//   window: R = i m + a, E_i = sum_t S_{k0 + i - t} P_t    (M = S, me = m, off = k0, B = P)
//   apply : R = t nr + r, P'_t = sum_s P_{t - s} Ml_s       (M = P, me = nr, off = 0, B = Ml)
// A block computes 4,096 / NC rows x NC columns (NC = 16, 32 or 64 >= q), a thread
// 4 x 4 of them on 64-bit accumulators; chunks of 16 (v, f) pairs go through double-
// buffered shared memory (rows of A one word apart, so that a thread's operands are
// two 16-byte loads for 16 products).  An accumulator is folded by 2^32 mod p after
// FOLDK products (below p^2 each, on top of a folded value: fold1_products).
// The window's v range is split over blockIdx.y, one partial sum each, added by
// k_sum_parts.  Bound by the 64-bit multiply-adds (a quarter of the issue rate).
// Measured on GB300, average over a whole sigma-basis: q = 64, 4,098 orders in
// 256-order leaves, 16 orders a chunk 55 us a launch (with 512-order leaves and 4
// orders a chunk, one block per SM that held its operands' coefficients whole in
// shared memory, window 141 and product 131 us); q = 16, 11,252 orders, 64 a chunk
// 69 us (window 85, product 154 us).
constexpr int TP_THREADS = 256, TP_K = 16;
constexpr int TP_FOLD = 8;  // (whole groups of a chunk's 16)
static_assert(TP_FOLD <= FOLD_SMALL && TP_K % TP_FOLD == 0 && TP_K % FOLD_BIG == 0, "folds of a chunk");

template <int NC>
struct Toep {
    static constexpr int BR = 4096 / NC;   // rows per block
    static constexpr int TX = NC / 4;
    static constexpr int AW = BR * TP_K / TP_THREADS, BW = NC * TP_K / TP_THREADS;  // words a thread loads
};

struct ToepArgs {
    const uint32_t *M, *B;
    uint32_t *C;
    int64_t rows;       // rows of C (at most, see limit)
    int64_t mrows, off; // rows of M, offset in units of me rows
    int me, nf, q;
    int64_t v0, vend, vper;  // block y: v in [v0 + y vper, v0 + (y + 1) vper) below vend
    int64_t cstride;         // words between the partial sums of consecutive y
    const int *vmax;         // window: vend is also at most *vmax + 1 (the basis degree)
    const int *rmax;         // apply: rows at most (*rmax + 1) me (the new degree)
    const int32_t *degl;     // apply: v at most the largest of the q local degrees
};

template <int NC, int FOLDK>
__global__ void __launch_bounds__(TP_THREADS, 2) k_toeplitz(ToepArgs g, ModP mp) {
    using T = Toep<NC>;
    __shared__ __align__(16) uint32_t As[2][TP_K][T::BR + 4], Bs[2][TP_K][NC + 4];
    const int tid = threadIdx.x;
    int64_t rows = g.rows, vend = g.vend;
    if (g.rmax) rows = min64(rows, ((int64_t)*g.rmax + 1) * g.me);
    const int64_t R0 = (int64_t)blockIdx.x * T::BR;
    if (R0 >= rows) return;
    if (g.vmax) vend = min64(vend, (int64_t)*g.vmax + 1);
    if (g.degl) {
        int d = 0;
        for (int c = tid & 31; c < g.q; c += 32) d = max(d, g.degl[c]);
        d = __reduce_max_sync(0xffffffffu, d);
        vend = min64(vend, (int64_t)d + 1);
    }
    const int64_t va = g.v0 + (int64_t)blockIdx.y * g.vper, vb = min64(va + g.vper, vend);
    const int nf = g.nf, q = g.q;
    const uint32_t fc = mp.r1;  // 2^32 mod p
    const int64_t ka = va * nf, kb = vb * nf;  // (v, f) pairs k = v nf + f
    // this thread's loads of a chunk: pair kl of rows rl, rl + 16, ...; words of B
    const int kl = tid % TP_K, rl = tid / TP_K;
    uint32_t ra[T::AW], rb[T::BW];
    // (v, f) of this thread's pair, advanced by TP_K a chunk
    int64_t v = (ka + kl) / nf;
    int f = (int)((ka + kl) - v * nf);
    auto load = [&](int64_t k) {
        const bool kv = k + kl < kb;
        const int64_t row = R0 + rl + (g.off - v) * g.me;
        const uint32_t *src = g.M + row * nf + f;
#pragma unroll
        for (int u = 0; u < T::AW; u++) {
            const int64_t rr = row + u * (TP_THREADS / TP_K);
            ra[u] = (kv && rr >= 0 && rr < g.mrows) ? __ldg(src + (int64_t)u * (TP_THREADS / TP_K) * nf) : 0u;
        }
#pragma unroll
        for (int u = 0; u < T::BW; u++) {
            const int w = tid + u * TP_THREADS, c = w % NC;
            const int64_t kk = k + w / NC;
            rb[u] = (kk < kb && c < q) ? __ldg(g.B + kk * q + c) : 0u;
        }
        f += TP_K;
        while (f >= nf) { f -= nf; v++; }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int u = 0; u < T::AW; u++) As[b][kl][rl + u * (TP_THREADS / TP_K)] = ra[u];
#pragma unroll
        for (int u = 0; u < T::BW; u++) {
            const int w = tid + u * TP_THREADS;
            Bs[b][w / NC][w % NC] = rb[u];
        }
    };
    unsigned long long acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0ull;
    const int tx = tid % T::TX, ty = tid / T::TX;
    if (ka < kb) {
        load(ka);
        store(0);
        __syncthreads();
        int b = 0;
        for (int64_t k = ka; k < kb; k += TP_K, b ^= 1) {
            const bool more = k + TP_K < kb;
            if (more) load(k + TP_K);
#pragma unroll
            for (int kk = 0; kk < TP_K; kk++) {
                const uint4 a4 = *reinterpret_cast<const uint4 *>(&As[b][kk][4 * ty]);
                const uint4 b4 = *reinterpret_cast<const uint4 *>(&Bs[b][kk][4 * tx]);
                const uint32_t av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) acc[i][j] = madw(av[i], bv[j], acc[i][j]);
                if ((kk + 1) % FOLDK == 0) {
#pragma unroll
                    for (int i = 0; i < 4; i++)
#pragma unroll
                        for (int j = 0; j < 4; j++) acc[i][j] = fold1(acc[i][j], fc);
                }
            }
            if (more) {
                store(b ^ 1);
                __syncthreads();
            }
        }
    }
    uint32_t *out = g.C + (int64_t)blockIdx.y * g.cstride;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int64_t R = R0 + 4 * ty + i;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int c = 4 * tx + j;
            if (R < rows && c < q) out[R * q + c] = red64(acc[i][j], mp);
        }
    }
}

// Esum[x] = sum over the window blocks of Epart[b][x], mod p: 32 entries per
// block, 8 groups of blocks per entry, then a shared-memory sum.
__global__ void __launch_bounds__(256)
    k_sum_parts(int nparts, int64_t E, const uint32_t *__restrict__ Epart, uint32_t *__restrict__ Esum, ModP mp) {
    __shared__ unsigned long long red[8][32];
    const int lx = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t x = (int64_t)blockIdx.x * 32 + lx;
    unsigned long long v = 0;  // < 2^31 * nparts
    if (x < E)
        for (int b = g; b < nparts; b += 8) v += __ldg(Epart + (size_t)b * E + x);
    red[g][lx] = v;
    __syncthreads();
    if (g == 0 && x < E) {
#pragma unroll
        for (int k = 1; k < 8; k++) v += red[k][lx];
        Esum[x] = red64(v, mp);
    }
}

// Orders per chunk unless the context sets it (wr_set_sigma_chunk): the window and
// product launches are spread over more orders by a longer chunk, the local kernel's
// row work per order grows with it.  Measured: q = 16, 11,252 orders 58 / 53 ms
// for 32 / 64; q = 32, 2,254 orders 23.1 / 17.4 / 18.5 ms for 8 / 32 / 64; q = 64,
// 4,098 orders (256-order leaves) 101 / 96 / 105 ms for 8 / 16 / 32.
inline int sigma_chunk_default(int q) {
    return q <= 16 ? 64 : (q <= 32 ? 32 : 16);
}
// PM-Basis by default for sequences longer than SIGMA_PM_MIN_L (q <= 32), with
// leaves of SIGMA_LEAF_DEFAULT orders: the M-Basis's window and product passes grow
// with the square of the length.  M-Basis alone / PM-Basis, ms: q = 2 17,000 orders 34.0 /
// 35.1, 30,000 62.1 / 60.6, 130,000 337 / 264; q = 4 17,000 39.7 / 39.9, 130,000 478 / 303;
// q = 8 17,000 50.5 / 49.4, 130,000 842 / 378; q = 16 11,252 53 / 57 (2,048-order leaves),
// 45,002 387 / 201 (leaves of 2,048 / 8,192: 198 / 221); q = 32 17,000 355 / 174.  Trailing a
// sequence they take its SMs (the rank of the 200,000 x 180,000 matrix: 1,926 ms with the
// M-Basis chunk by chunk; in PM-Basis segments 1,711, 1,729 to 1,813 and 1,917 with 2,048-,
// 4,096- and 8,192-order leaves, the sequence by itself varying by 5 % with the tuner's pick;
// symmetric 1,520 against 1,391, 1,394 to 1,405 and 1,492).  For q > 32 those passes
// cost more per order, so PM-Basis with short leaves takes over early: at q =
// 64, 4,098 orders, 98 / 96 / 105 ms for leaves of 128 / 256 / 512 orders, and
// against the M-Basis alone 12.9 / 12.0 ms at 600 orders, 22.4 / 21.3 at 1,030,
// 44.9 / 34.9 at 1,700; q = 33 10.0 / 11.0 at 1,030, 18.6 / 18.2 at 1,700, 24.5 / 22.5 at 2,100;
// q = 40 (8 x 32) 9.0 / 10.4, 16.2 / 17.2, 20.7 / 21.1, (20 x 20) 14.6 / 15.4, 27.3 / 25.4,
// 36.0 / 31.7; q = 48 24.4 / 16.8, 31.8 / 27.6, 42.8 / 34.7.  wr_set_sigma_leaf chooses the
// leaf explicitly.
constexpr int64_t SIGMA_LEAF_DEFAULT = 4096;
constexpr int64_t SIGMA_PM_MIN_L = 16384;
constexpr int64_t SIGMA_LEAF_WIDE = 256;
constexpr int64_t SIGMA_PM_MIN_L_WIDE = 1024;
constexpr int BAR_T0 = 1, BAR_E = 3;  // named barriers BAR_T0 + (i & 1), BAR_E

__device__ __forceinline__ void named_sync(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int nthreads) {
    __threadfence_block();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// ---- local M-Basis over the window: one cluster of thread blocks, bb orders.
//
// The device keeps the basis in fraction-free form, M_g = M diag(S): the
// elimination of a discrepancy whose columns are scaled by nonzero constants
// picks the same pivots and yields the same reduced columns up to column
// scales, so M_g stays a column-scaled copy of the order-by-order basis.  S
// (per column, product of the scales of all orders) is divided out of P once
// at the end.
//
// An order's transform is new[j] = s_j old[j] + sum_t F[t][j] old[pc[t]], then the
// pivot columns times x.  It multiplies every row of the window (orders i ..), of
// Qtop and of the chunk's transform Ml, each row for itself, so the rows are dealt
// to the blocks of the cluster: block `rank` of CS holds the rows a = rank (mod CS)
// of the window's orders and of Qtop, and the rows x = rank (mod CS) of Ml's
// coefficients.  What the next order needs from everybody is its discrepancy,
// m x q residues: every block writes its rows of it into the shared memory of all
// the others, and after one cluster barrier each block runs the (same) elimination
// for itself.
//
// Roles in a block: the first warps (EW of them) eliminate, the others multiply
// rows.  Per order i
//   elim    Gauss-Jordan by rows on the m x q discrepancy, columns in (degree,
//           index) order, 4 or 8 column slots x MR rows over the EW warps.  A column is frozen (written to FR) at its turn; if it
//           is nonzero outside the pivot rows so far it becomes pivot k, its first
//           such row r_k the pivot row, and every other row of the later columns
//           becomes d_k row - A[row][pc] row_k (fraction-free).  Row r_t then holds
//           the coefficients of the pivot columns, times prod_{t <= i < k} d_i, so
//           with pre_t = d_0 .. d_{t-1}: s_j = pre_k(j), F[t][j] = -pre_t FR[j][r_t]
//           (t < k(j), the pivots before j) -- no inverse, and no transform
//           carried beside the matrix.  With several warps the columns go by groups
//           of one per slot: within a group step by step, the later columns take the
//           group's whole transform as one product.
//   rows    first the block's rows of orders i and i + 1 (the next discrepancy:
//           pivot columns take order i's value, the others order i + 1's), written
//           to all blocks; then, beside the next elimination, the other rows.
// Hand-overs: a named barrier T_i (transform i published; elim arrives, the row
// warps wait) and the cluster barrier of order i (all threads arrive; it completes
// when every block's rows of discrepancy i + 1 are everywhere).  The transform, its
// snapshot of the offsets and the discrepancy are double-buffered; what is
// overwritten two orders later was read before the barrier in between.
// Multiplying column c by x moves no data: window column c is read at row
// ip - sh[c], and Ml column c holds its coefficient s at row base[c] + s.
//
// Bound by the chain of one order (elimination, hand-over, the next discrepancy's rows,
// the cluster barrier) and, at q = 64, by issue: an order is 47,000 warp instructions a
// block, a wide multiply-add taking a scheduler five cycles.  Hence the elimination
// by groups of columns, one copy of the row product's code, sums reduced by three
// multiplications, and 16 blocks where 8 rows a block kept the row warps busy longer
// than the elimination.  An odd pitch for the discrepancy and the transform: with lanes
// a row apart, pitch q put the elimination's loads and the transform's stores on one
// bank (4,700 of 32,000 cycles an order at q = 64).  Measured per order (GB300): q = 16
// 9.6 -> 2.3 us, q = 32 70 -> 4.2 us, q = 64 68 -> 11 us (17 with 8 blocks and 32 steps on
// every later column; at first one block, one elimination warp that also carried the
// transform, or sixteen warps with all rows of the chunk on one SM).  A warp of its own
// for the bookkeeping, beside the elimination, gained nothing: the chain runs through
// the rows (sigma-basis of 11,252 orders at q = 16 52.8 ms without, 53.8 with).
constexpr int LC_SNAP = 228;   // words of an order's snapshot
constexpr int LC_INTS = 1392;  // words of the bookkeeping arrays
__host__ __device__ constexpr int lc_threads(int MR) { return MR == 32 ? 512 : (MR == 16 ? 384 : 256); }
// elimination warps: one for MR = 8 (4 column slots, handed round by shuffles), else 8 column slots
__host__ __device__ constexpr int lc_ew(int MR) { return MR == 8 ? 1 : MR / 4; }
// words of a row warp's pivot residues: 32, or 16 groups of 2 lanes with 8 each
__host__ __device__ constexpr int lc_gs_words(int MR) { return MR == 8 ? 128 : 32; }

// Blocks per cluster for q columns (8 is the largest portable size, 16 the largest): the
// whole sigma-basis with 8 / 16 blocks: q = 32, 2,254 orders 19.6 / 17.4 ms; q = 64, 4,098
// orders 113 / 97 ms; q = 16, 11,252 orders, 4 / 8 blocks 84 / 82 ms with the earlier
// kernels, 16 as 8; up to 8 columns 4 and 8 measure the same
inline int local_cluster(int q) {
    return q > 16 ? 16 : q > 8 ? 8 : 4;
}

struct LcLayout {  // word offsets of the dynamic shared memory (ints and residues are both words)
    int ma, mx;    // most rows of a window order / of an Ml coefficient in a block
    int Es, Ml, qt, disc, F, dg, FR, gs, ints, total;
};
__host__ __device__ inline LcLayout lc_layout(int m, int q, int b, int CS, int MR, int QC) {
    LcLayout l;
    l.ma = (m + CS - 1) / CS;
    l.mx = (q + CS - 1) / CS;
    int o = 0;
    l.Es = o; o += b * l.ma * q;
    l.Ml = o; o += (2 * b + 1) * l.mx * q;
    l.qt = o; o += l.ma * q;
    l.disc = o; o += 2 * m * (QC + 1);
    l.F = o; o += 2 * MR * (QC + 1);  // (rows from m on stay zero)
    l.dg = o; o += 2 * 64;
    l.FR = o; o += q * (MR + 1);
    o = (o + 3) & ~3;  // (16-byte loads)
    l.gs = o; o += (lc_threads(MR) / 32 - lc_ew(MR)) * lc_gs_words(MR);
    l.ints = o; o += LC_INTS;
    l.total = o;
    return l;
}

// (a0 + a1) 2^-32 mod p: folded, each is at most (c + 1)(2^32 - 1) <= 2^63 (c = 2^32 mod
// p), so their sum fits, and folded again it is below p 2^32 (3 multiplications; the
// general reduction mod p takes 8)
__device__ __forceinline__ uint32_t redc_sum(unsigned long long a0, unsigned long long a1, uint32_t fc,
                                             const ModP &mp) {
    const unsigned long long t = fold1(fold1(a0, fc) + fold1(a1, fc), fc);
    const uint32_t u = (uint32_t)(madw((uint32_t)t * mp.pneg, mp.p, t) >> 32);
    return min(u, u - mp.p);
}

// A row times the order's transform in registers (lane: column j and, CPL = 2,
// column j + 32; f[k][t] = F[t][column k], d[k] its diagonal, both in Montgomery form): x[k] the row's
// residues of the lane's columns, gs the row's residues at the pivot columns (shared
// memory, read 4 at a time by the whole group).  Two accumulators a column (even and odd
// t), each folded after FOLDK of its own products.
template <int TM, int CPL, int FOLDK>
__device__ __forceinline__ void row_times(const uint32_t (&f)[CPL][TM], const uint32_t (&d)[CPL], int m,
                                          const uint32_t (&x)[CPL], const uint32_t *gs, uint32_t (&out)[CPL], uint32_t fc,
                                          const ModP &mp) {
    unsigned long long a0[CPL], a1[CPL];
#pragma unroll
    for (int k = 0; k < CPL; k++) {
        a0[k] = (unsigned long long)d[k] * x[k];
        a1[k] = 0ull;
    }
    // (f[k][t] = 0 from the number of pivots on: whole groups of 8, and branches that only
    // depend on a kernel argument)
#pragma unroll
    for (int t0 = 0; t0 < TM; t0 += 8) {
        if (TM == 8 || t0 < m) {
            const uint4 va = *reinterpret_cast<const uint4 *>(gs + t0);
            const uint4 vb = *reinterpret_cast<const uint4 *>(gs + t0 + 4);
            const uint32_t v[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int t = t0 + u;
#pragma unroll
                for (int k = 0; k < CPL; k++) {
                    if ((t & 1) == 0) {
                        a0[k] = madw(f[k][t], v[u], a0[k]);
                        if ((t / 2 + 2) % FOLDK == 0) a0[k] = fold1(a0[k], fc);
                    } else {
                        a1[k] = madw(f[k][t], v[u], a1[k]);
                        if (((t + 1) / 2) % FOLDK == 0) a1[k] = fold1(a1[k], fc);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < CPL; k++) out[k] = redc_sum(a0[k], a1[k], fc, mp);
}

// The update of a pivot step on the lane's residues from k0 on: A[k] <- d A[k] -
// v y with y the pivot row's residue of the same column (nv = p - v; the pivot
// row itself stays).  One block without branches: independent chains.
template <int KR>
__device__ __forceinline__ void pivot_step(uint32_t (&A)[KR], const uint32_t (&y)[KR], int k0, uint32_t d, uint32_t nv,
                                           bool other, uint32_t p, uint32_t pneg) {
#pragma unroll
    for (int k = 0; k < KR; k++) {
        if (k < k0) continue;  // (a constant after unrolling)
        // d x + (p - v) y < 2 p^2 < p 2^32
        const unsigned long long t = madw(nv, y[k], (unsigned long long)d * A[k]);
        const uint32_t u = (uint32_t)(madw((uint32_t)t * pneg, p, t) >> 32);
        A[k] = other ? min(u, u - p) : A[k];
    }
}

template <int MR, int CPL, int QC, int FOLDK>
__global__ void __launch_bounds__(lc_threads(MR), 1)
    k_local(int m, int q, int bb, const uint32_t *__restrict__ E, uint32_t *__restrict__ qtop_g,
            int32_t *__restrict__ deg_g, uint32_t *__restrict__ Ml_g, int32_t *__restrict__ degl_g,
            int *__restrict__ dmax_g, uint32_t *__restrict__ scale_g, int dbase, ModP mp) {
    constexpr int NT = lc_threads(MR), EW = lc_ew(MR), NE = 32 * EW, NWK = NT / 32 - EW;
    constexpr int CL = EW * 32 / MR;        // column slots of the elimination
    constexpr int KR = QC / CL;             // residues a lane of the elimination (q <= QC)
    constexpr int TM = MR;                  // most pivots of an order
    constexpr int PQ = QC + 1;              // odd pitch: the elimination's lanes are rows
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ uint32_t sm[];
    const int CS = (int)cluster_size(), rank = (int)cluster_rank();
    const LcLayout l = lc_layout(m, q, bb, CS, MR, QC);
    uint32_t *Es = sm + l.Es;      // [bb][ma][q]
    uint32_t *Ml = sm + l.Ml;      // [2 bb + 1][mx][q]
    uint32_t *qt = sm + l.qt;      // [ma][q]
    uint32_t *disc = sm + l.disc;  // [2][m][PQ], written by every block
    uint32_t *Fs = sm + l.F;       // [2][MR][PQ]
    uint32_t *dgs = sm + l.dg;     // [2][64]
    uint32_t *FR = sm + l.FR;      // [q][MR + 1] frozen columns by position
    int *deg = (int *)(sm + l.ints);  // [64] degrees, local degrees (before and after the transform), offsets
    int *degl = deg + 64, *dln = degl + 64, *sh = dln + 64, *base = sh + 64;
    int *posc = base + 64;         // [64] column of each position
    int *rk = posc + 64;           // [64] position of each column
    int *kj = rk + 64;             // [64] pivots before the position's turn
    uint32_t *scum = (uint32_t *)(kj + 64);  // [64] column scales of the chunk (Montgomery form)
    uint32_t *preM = scum + 64;    // [33] pre_t in Montgomery form
    int *pr = (int *)(preM + 36);  // [32] pivot rows
    int *snap = pr + 32;           // [2][LC_SNAP]: sh, base, isp [64 each], pc [32], np, D
    int *dmx = snap + 2 * LC_SNAP; // [8]
    int *pdl = dmx + 8;            // [32] the pivots' local degrees before the order
    int *ppos = pdl + 32;          // [32] the pivots' positions
    int *pmax = ppos + 32;         // [33]
    int *degl_n = pmax + 36;       // [64]
    uint32_t *sck = (uint32_t *)(degl_n + 64);  // [64] the order's column scales (Montgomery form)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mq = m * PQ;
    const uint32_t fc = mp.r1;  // 2^32 mod p

    for (int x = tid; x < bb * l.ma * q; x += NT) {
        const int c = x % q, al = x / q % l.ma, i = x / (q * l.ma), a = rank + CS * al;
        uint32_t e = 0;
        if (a < m) {
            e = E[((size_t)i * m + a) * q + c];
            if (i == 0) e = subm(e, qtop_g[a * q + c], mp);
        }
        Es[x] = e;
    }
    for (int x = tid; x < 2 * MR * PQ; x += NT) Fs[x] = 0u;
    for (int x = tid; x < m * q; x += NT) disc[x / q * PQ + x % q] = subm(E[x], qtop_g[x], mp);
    for (int x = tid; x < l.ma * q; x += NT) {
        const int a = rank + CS * (x / q);
        qt[x] = a < m ? qtop_g[a * q + x % q] : 0u;
    }
    for (int x = tid; x < (2 * bb + 1) * l.mx * q; x += NT) {
        const int c = x % q, xl = x / q % l.mx, s = x / (q * l.mx);
        Ml[x] = (s == bb && rank + CS * xl == c) ? 1u : 0u;  // coefficient 0 at row base = bb
    }
    for (int c = tid; c < 64; c += NT) {
        snap[c] = 0;
        snap[64 + c] = bb;
        deg[c] = c < q ? deg_g[c] : 0;
        degl[c] = 0;
        sh[c] = 0;
        base[c] = bb;
        scum[c] = mp.r1;
    }
    __syncthreads();
    cluster_arrive();  // (every block has read qtop_g and set up before anybody writes)
    cluster_wait();

    if (warp < EW) {
        const int a = lane % MR, slot = warp * (32 / MR) + lane / MR;
        auto esync = [&]() {
            if constexpr (EW == 1) __syncwarp();
            else named_sync(BAR_E, NE);
        };
        int D = 0;  // largest local degree
        int QP = 1;
        while (QP < q) QP <<= 1;
        const int parts = QP < NE ? NE / QP : 1, part = tid % parts;  // threads a column
        // positions by (degree, index)
        auto ranks = [&]() {
            for (int c0 = 0; c0 < q; c0 += NE / parts) {
                const int c = c0 + tid / parts, dc = deg[c & 63];
                int r = 0;
#pragma unroll 4
                for (int c2 = part; c2 < q; c2 += parts) {
                    const int d2 = deg[c2];
                    r += (d2 < dc || (d2 == dc && c2 < c)) ? 1 : 0;
                }
                for (int off = 1; off < parts; off <<= 1) r += __shfl_xor_sync(FULL, r, off);
                if (c < q && part == 0) {
                    rk[c] = r;
                    posc[r] = c;
                }
            }
        };
        ranks();
        esync();
        const int nk = (q + CL - 1) / CL, am = a < m ? a : 0;
        // The order's elimination with pivots wherever they are: columns that are zero
        // outside the pivot rows, pivot rows in any order.  Writes what the straight
        // path below writes, through FR; returns the number of pivots.
        auto slow = [&](int i) -> int {
            const uint32_t *dc = disc + (i & 1) * mq;
            uint32_t *F = Fs + (i & 1) * MR * PQ, *dg = dgs + (i & 1) * 64;
            int *sn = snap + (i & 1) * LC_SNAP;
            uint32_t A[KR], y[KR];
#pragma unroll
            for (int k = 0; k < KR; k++) {
                const int pos = CL * k + slot;
                A[k] = to_mont(dc[am * PQ + posc[min(pos, q - 1)]], mp);
                if (pos >= q || a >= m) A[k] = 0u;
            }
            for (int c = tid; c < 64; c += NE) {
                sn[128 + c] = 0;
                dln[c] = degl[c];
            }
            esync();
            uint32_t pre = mp.r1, rmask = m == 32 ? FULL : (1u << m) - 1u;  // rows without a pivot
            int np = 0, pos = 0;
            for (int g4 = 0; g4 < nk; g4++) {
                for (int s = 0; s < CL && pos < q && np < m; s++, pos++) {
                    // the pivot row is nearly always the first row without a pivot: its
                    // residues are fetched before the column is known to have it
                    int fr = __ffs(rmask) - 1;
#pragma unroll
                    for (int k = 0; k < KR; k++) y[k] = __shfl_sync(FULL, A[k], fr, MR);
                    if (slot == s) FR[pos * (MR + 1) + a] = A[0];
                    uint32_t v, d;
                    if constexpr (EW == 1) {
                        v = __shfl_sync(FULL, A[0], s * MR + a);
                        d = __shfl_sync(FULL, A[0], s * MR + fr);
                    } else {
                        esync();
                        v = FR[pos * (MR + 1) + a];
                        d = FR[pos * (MR + 1) + fr];
                    }
                    if (tid == 0) kj[pos] = np;
                    if (d == 0u) {  // another row, or a column that is zero there
                        const uint32_t nz = __ballot_sync(FULL, v != 0u) & rmask;
                        if (nz == 0u) continue;
                        fr = __ffs(nz) - 1;
                        d = __shfl_sync(FULL, v, fr);
#pragma unroll
                        for (int k = 0; k < KR; k++) y[k] = __shfl_sync(FULL, A[k], fr, MR);
                    }
                    if (tid == 0) {
                        pr[np] = fr;
                        ppos[np] = pos;
                        preM[np] = pre;
                    }
                    const uint32_t nv = v != 0u ? mp.p - v : 0u;
                    pivot_step(A, y, 0, d, nv, a != fr, mp.p, mp.pneg);
                    pre = mont_mul(pre, d, mp);
                    rmask &= ~(1u << fr);
                    np++;
                }
                if (np == m || pos >= q) {
                    // the columns not yet frozen, at their final values
#pragma unroll
                    for (int k = 0; k < KR; k++) {
                        const int pk = CL * (g4 + k) + slot;
                        if (pk >= pos && pk < q) {
                            FR[pk * (MR + 1) + a] = A[k];
                            if (a == 0) kj[pk] = np;
                        }
                    }
                    break;
                }
#pragma unroll
                for (int k = 0; k + 1 < KR; k++) A[k] = A[k + 1];
            }
            if (tid == 0) {
                preM[np] = pre;
                sn[224] = np;
                sn[225] = D;
            }
            esync();
            // the pivots' columns, local degrees and scales
            for (int t = tid; t < np; t += NE) {
                const int c = posc[ppos[t]];
                sn[192 + t] = c;
                pdl[t] = degl[c];
                sn[128 + c] = 1;
            }
            esync();
            // publish the transform (Montgomery form) and the local degree bounds
            for (int c0 = 0; c0 < q; c0 += NE / parts) {
                const int j = c0 + tid / parts;
                if (j < q) {
                    const int pj = rk[j], kk = kj[pj];
                    const uint32_t *fj = FR + pj * (MR + 1);
                    int dl = 0;
#pragma unroll 4
                    for (int t = part; t < m; t += parts) {  // (rows from np on: zero)
                        const bool is = t < np;
                        const uint32_t x = mont_mul(fj[is ? pr[t] : 0], is ? preM[t] : 0u, mp);
                        const uint32_t v = t < kk ? x : 0u;
                        F[t * PQ + j] = v != 0u ? mp.p - v : 0u;
                        dl = max(dl, v != 0u ? pdl[t] : 0);
                    }
                    if (dl > 0) atomicMax(&dln[j], dl);
                    if (part == 0) {
                        dg[j] = sck[j] = preM[kk];
                    }
                }
            }
            return np;
        };
        for (int i = 0; i < bb; i++) {
            const uint32_t *dc = disc + (i & 1) * mq;
            uint32_t *F = Fs + (i & 1) * MR * PQ, *dg = dgs + (i & 1) * 64;
            int *sn = snap + (i & 1) * LC_SNAP;
            uint32_t A[KR], y[KR];
            int col[KR];  // the lane's columns
#pragma unroll
            for (int k = 0; k < KR; k++) {
                col[k] = posc[min(CL * k + slot, q - 1)];
                A[k] = to_mont(dc[am * PQ + col[k]], mp);
                if (CL * k + slot >= q || a >= m) A[k] = 0u;
            }
            int np = m;
            // the snapshot's pivots, if nothing vanishes (else the slow path writes its own)
            for (int c = tid; c < q; c += NE) sn[128 + c] = rk[c] < m ? 1 : 0;
            if (tid < m) sn[192 + tid] = posc[tid];
            if (tid == 0) {
                sn[224] = m;
                sn[225] = D;
            }
            // Straight through: position t becomes pivot t with row t its pivot row, as it
            // does unless residues vanish.  Registers keep a column's values from its turn
            // on, so a lane holds row a of every column it has: F and the scales come from
            // registers, with pre_a kept as the lane's own.
            uint32_t pre = mp.r1, pre_a = mp.r1;
            bool bad = m > q;
            if constexpr (EW == 1) {
#pragma unroll
                for (int g = 0; g < MR / CL; g++) {
#pragma unroll
                    for (int s = 0; s < CL; s++) {
                        const int t = CL * g + s;
                        if (t < m) {  // (the same for all)
#pragma unroll
                            for (int k = g; k < KR; k++) y[k] = __shfl_sync(FULL, A[k], t, MR);
                            const uint32_t v = __shfl_sync(FULL, A[g], s * MR + a);
                            const uint32_t d = __shfl_sync(FULL, A[g], s * MR + t);
                            bad |= d == 0u;
                            const uint32_t nv = v != 0u ? mp.p - v : 0u;
                            const uint32_t keep = A[g];
                            pivot_step(A, y, g, d, nv, a != t, mp.p, mp.pneg);
                            if (slot <= s) A[g] = keep;
                            pre_a = a == t ? pre : pre_a;
                            pre = mont_mul(pre, d, mp);
                        }
                    }
                }
            } else {
                // A group of CL columns (one of each slot) at a time.  Its steps change one
                // residue r of a lane: its column's until the column's turn, from then on the
                // coefficients G of that pivot row in the group's transform.  The later
                // columns take the whole transform at once,
                //   row a <- (a a pivot row of the group ? 0 : sg) row a + sum_t G_t[a] row t,
                // sg the product of the group's pivots: 9 products and one reduction instead
                // of 8 steps of two products and a reduction each.
#pragma unroll
                for (int g = 0; g < MR / CL; g++) {
                    const int ns = min(CL, m - CL * g);
                    if (ns > 0) {  // (the same for all)
                        uint32_t r = A[g], sg = mp.r1, sg_a = mp.r1;
#pragma unroll 1
                        for (int s = 0; s < ns; s++) {
                            const int t = CL * g + s;
                            uint32_t *fr = FR + (t & 1) * MR;  // (two slots: a barrier apart)
                            uint32_t yr[1] = {__shfl_sync(FULL, r, t, MR)};
                            if (slot == s) {
                                fr[a] = r;
                                A[g] = r;
                                yr[0] = sg;
                                r = a == t ? sg : 0u;
                            }
                            esync();
                            const uint32_t v = fr[a], d = fr[t];
                            bad |= d == 0u;
                            const uint32_t nv = v != 0u ? mp.p - v : 0u;
                            uint32_t rr[1] = {r};
                            pivot_step(rr, yr, 0, d, nv, a != t, mp.p, mp.pneg);
                            r = rr[0];
                            sg_a = a == t ? sg : sg_a;
                            sg = mont_mul(sg, d, mp);
                        }
                        uint32_t *Gs = FR + 2 * MR;  // [CL][MR] (q >= 10 columns of MR + 1 words)
                        if (slot >= ns) A[g] = r;
                        Gs[slot * MR + a] = slot < ns ? r : 0u;
                        if (a / CL == g && a < m) pre_a = mont_mul(pre, sg_a, mp);
                        const uint32_t dg0 = a / CL == g && a < m ? 0u : sg;
                        pre = mont_mul(pre, sg, mp);
                        esync();
                        uint32_t G[CL];
#pragma unroll
                        for (int u = 0; u < CL; u++) G[u] = Gs[u * MR + a];
#pragma unroll
                        for (int k = g + 1; k < KR; k++) {
                            unsigned long long a0 = (unsigned long long)dg0 * A[k], a1 = 0ull;
#pragma unroll
                            for (int u = 0; u < CL; u++) {
                                const uint32_t yk = __shfl_sync(FULL, A[k], min(CL * g + u, MR - 1), MR);
                                if ((u & 1) == 0) {
                                    a0 = madw(G[u], yk, a0);
                                    if ((u / 2 + 2) % FOLDK == 0) a0 = fold1(a0, fc);
                                } else {
                                    a1 = madw(G[u], yk, a1);
                                    if (((u + 1) / 2) % FOLDK == 0) a1 = fold1(a1, fc);
                                }
                            }
                            A[k] = redc_sum(a0, a1, fc, mp);
                        }
                    }
                }
            }
            if (!bad) {
#pragma unroll
                for (int k = 0; k < KR; k++) {
                    const int pos = CL * k + slot, kk = min(pos, m);
                    if (pos < q && a < m) {
                        const uint32_t v = mont_mul(A[k], pre_a, mp);
                        F[a * PQ + col[k]] = a < kk && v != 0u ? mp.p - v : 0u;
                        if (a == (pos < m ? pos : 0)) {
                            dg[col[k]] = sck[col[k]] = pos < m ? pre_a : pre;
                        }
                    }
                }
            } else {
                np = slow(i);
            }
            if constexpr (EW == 1) __syncwarp();
            named_arrive(BAR_T0 + (i & 1), NE + 32 * NWK);
            // bookkeeping, beside the rows
            if (!bad && warp == 0) {  // pmax[k]: largest local degree of the first k pivots
                int v = lane < m ? degl[posc[lane]] : 0;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int u = __shfl_up_sync(FULL, v, off);
                    if (lane >= off) v = max(v, u);
                }
                pmax[lane + 1] = v;
                if (lane == 0) pmax[0] = 0;
            }
            esync();
            int *sx = snap + ((i + 1) & 1) * LC_SNAP;  // the next order's snapshot
            int Dn = 0;
            for (int c = tid; c < q; c += NE) {
                const int ip = sn[128 + c];
                // local degrees after the transform: exact from the slow path, else the
                // largest of the column's and of the pivots before it (pmax)
                const int pos = rk[c], dl = (bad ? dln[c] : max(degl[c], pmax[min(pos, m)])) + ip;
                deg[c] += ip;
                degl_n[c] = dl;
                sx[c] = sh[c] += ip;
                sx[64 + c] = base[c] -= ip;
                scum[c] = mont_mul(scum[c], sck[c], mp);
                Dn = max(Dn, dl);
            }
            Dn = __reduce_max_sync(FULL, Dn);
            if (lane == 0) dmx[warp] = Dn;
            esync();
#pragma unroll
            for (int w = 0; w < EW; w++) D = max(D, dmx[w]);
            for (int c = tid; c < q; c += NE) degl[c] = degl_n[c];
            ranks();
            esync();
            cluster_arrive();
            cluster_wait();
        }
    } else {
        const int ow = warp - EW;
        int W2 = 1;
        while (W2 < q && W2 < 32) W2 <<= 1;
        const int rpw = 32 / W2, grp = lane / W2, col = lane % W2;
        const int NG = NWK * rpw;          // rows at a time
        uint32_t *gs = sm + l.gs + (ow * rpw + grp) * max(W2, TM);  // the group's pivot residues
        const int wq = l.ma * q, xq = l.mx * q;
        bool cok[CPL];
#pragma unroll
        for (int k = 0; k < CPL; k++) cok[k] = col + 32 * k < q;
        for (int i = 0; i < bb; i++) {
            named_sync(BAR_T0 + (i & 1), NE + 32 * NWK);
            const uint32_t *F = Fs + (i & 1) * MR * PQ, *dg = dgs + (i & 1) * 64;
            const int *sn = snap + (i & 1) * LC_SNAP;
            const int np = sn[224], D = sn[225];
            uint32_t f[CPL][TM], d[CPL];
            int shc[CPL], bsc[CPL];
            bool isp[CPL];
#pragma unroll
            for (int k = 0; k < CPL; k++) {
                const int j = col + 32 * k;
                d[k] = cok[k] ? dg[j] : 0u;
                shc[k] = cok[k] ? sn[j] : 0;
                bsc[k] = cok[k] ? sn[64 + j] : 0;
                isp[k] = cok[k] && sn[128 + j] != 0;
#pragma unroll
                for (int t = 0; t < TM; t++) f[k][t] = F[t * PQ + (cok[k] ? j : 0)];
            }
            // lane t of a group fetches the row's residue at pivot column t
            const bool pok = col < np;
            const int pc = pok ? sn[192 + col] : 0;
            const int shp = pok ? sn[pc] : 0, bsp = pok ? sn[64 + pc] : 0;
            // word offsets of the lane's columns (ad*) and its pivot column (pd*) in row 0 of
            // the window, of Ml and of Qtop
            int adW[CPL], adM[CPL];
#pragma unroll
            for (int k = 0; k < CPL; k++) {
                adW[k] = l.Es + col + 32 * k - shc[k] * wq;
                adM[k] = l.Ml + col + 32 * k + bsc[k] * xq;
            }
            const int pdW = l.Es + pc - shp * wq, pdM = l.Ml + pc + bsp * xq, pdQ = l.qt + pc;
            // Pass 0: the next discrepancy, window rows i and i + 1, to every block.  Pass 1,
            // beside the next elimination: the window's later rows, Qtop (the next one keeps
            // the pivot columns of Qtop T), Ml's coefficients 0 .. D.  One loop over all the
            // rows (those past m or q are zero and stay so): one copy of the product's code.
            uint32_t *dn = disc + ((i + 1) & 1) * mq;
#pragma unroll 1
            for (int ps = 0; ps < 2; ps++) {
                const int w0 = (i + 2 * ps) * l.ma;
                const int nw = ps == 0 ? (i + 1 < bb ? 2 * l.ma : 0) : max(bb - i - 2, 0) * l.ma;
                const int nq = nw + (ps == 0 ? 0 : l.ma);
                const int nr = nq + (ps == 0 || np == 0 ? 0 : (D + 1) * l.mx);
#pragma unroll 1
                for (int r0 = ow * rpw; r0 < nr; r0 += NG) {
                    const int r = r0 + grp;
                    const bool ok = r < nr, inw = r < nw, inm = r >= nq;
                    const int row = (inw ? w0 + r : (inm ? r - nq : r - nw)) * q;
                    uint32_t *rp[CPL], v[CPL], x[CPL];
#pragma unroll
                    for (int k = 0; k < CPL; k++) {
                        rp[k] = sm + row + (inw ? adW[k] : (inm ? adM[k] : l.qt + col + 32 * k));
                        v[k] = ok && cok[k] ? *rp[k] : 0u;
                    }
                    if (pok) gs[col] = ok ? sm[row + (inw ? pdW : (inm ? pdM : pdQ))] : 0u;
                    __syncwarp();
                    row_times<TM, CPL, FOLDK>(f, d, m, v, gs, x, fc, mp);
                    __syncwarp();
                    const int h = r >= l.ma ? 1 : 0, ar = rank + CS * (r - h * l.ma);  // (pass 0)
#pragma unroll
                    for (int k = 0; k < CPL; k++) {
                        if (ok && cok[k]) {
                            *rp[k] = inw || inm || isp[k] ? x[k] : 0u;
                            // row i's pivot columns, row i + 1's others
                            if (ps == 0 && ar < m && isp[k] == (h == 0)) {
                                uint32_t *dst = dn + ar * PQ + col + 32 * k;
                                for (int b = 0; b < CS; b++) st_cluster(dst, (uint32_t)b, x[k]);
                            }
                        }
                    }
                }
                __syncwarp();
                if (ps == 0) cluster_arrive();
            }
            cluster_wait();
        }
    }
    __syncthreads();
    const int qq = q * q;
    for (int y = tid; y < (bb + 1) * l.mx * q; y += NT) {
        const int c = y % q, xl = y / q % l.mx, s = y / (q * l.mx), x = rank + CS * xl;
        if (x < q) Ml_g[(size_t)s * qq + x * q + c] = Ml[((size_t)(base[c] + s) * l.mx + xl) * q + c];
    }
    for (int x = tid; x < l.ma * q; x += NT) {
        const int a = rank + CS * (x / q);
        if (a < m) qtop_g[a * q + x % q] = qt[x];
    }
    if (rank == 0) {
        for (int c = tid; c < q; c += NT) {
            deg_g[c] = deg[c];
            degl_g[c] = degl[c];
            scale_g[c] = mont_mul(scale_g[c], scum[c], mp);
        }
        if (tid == 0) {
            // bound on the polynomial degree of the basis: column c's degree
            // minus the smallest starting degree (the row shifts)
            int d = 0;
            for (int c = 0; c < q; c++) d = max(d, deg[c] - dbase);
            *dmax_g = d;
        }
    }
}

// P[t][r][c] /= S[c] (S in Montgomery form), t <= D
__global__ void k_unscale(uint32_t *__restrict__ P, int n, int q, int64_t D, const uint32_t *__restrict__ scale_g,
                          ModP mp) {
    __shared__ uint32_t inv[64];
    for (int c = threadIdx.x; c < q; c += blockDim.x) inv[c] = from_mont(mont_inv(scale_g[c], mp), mp);
    __syncthreads();
    const int64_t nq = (int64_t)n * q;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < (D + 1) * nq; x += (int64_t)gridDim.x * blockDim.x)
        P[x] = mulm(P[x], inv[x % q], mp);
}

// ---------------------------------------------------------------- readout

// choose the n columns of least (degree, index)
__global__ void k_select(const int32_t *__restrict__ deg, int q, int n, int32_t *__restrict__ sel,
                         int32_t *__restrict__ delta) {
    int c = threadIdx.x;
    if (c >= q) return;
    int rk = 0;
    for (int c2 = 0; c2 < q; c2++) rk += (deg[c2] < deg[c] || (deg[c2] == deg[c] && c2 < c)) ? 1 : 0;
    if (rk < n) {
        sel[rk] = c;
        delta[rk] = deg[c];
    }
}

// G[t][r][j] for t < T: reversed (F) or plain (P) coefficients of the selected columns
__global__ void k_extract(const uint32_t *__restrict__ P, int n, int q, const int32_t *__restrict__ sel,
                          const int32_t *__restrict__ delta, int64_t T, int reversed, int64_t Dcap,
                          uint32_t *__restrict__ G) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T * n * n) return;
    const int64_t t = i / (n * n);
    const int r = (int)((i / n) % n), j = (int)(i % n);
    const int64_t dj = delta[j];
    int64_t src = reversed ? dj - t : t;
    uint32_t v = 0;
    if (src >= 0 && src <= dj && src <= Dcap) v = P[((size_t)src * n + r) * q + sel[j]];
    G[i] = v;
}

// x-adic valuation of det G over F_p[[x]] / x^T: g laid out [(i*n + j)*T + t].
constexpr int VAL_THREADS = 256;

__global__ void __launch_bounds__(VAL_THREADS)
    k_valuation(const uint32_t *__restrict__ G, uint32_t *__restrict__ g, int n, int T,
                int64_t *__restrict__ out, ModP mp) {
    extern __shared__ uint32_t sm[];
    uint32_t *inv = sm;              // T
    uint32_t *mu = inv + T;          // n * T
    int *rdone = (int *)(mu + (size_t)n * T);
    int *cdone = rdone + n;
    __shared__ unsigned long long best;
    const int tid = threadIdx.x;
    for (int64_t i = tid; i < (int64_t)n * n * T; i += blockDim.x) {
        int64_t t = i % T, ij = i / T;
        g[i] = G[(size_t)t * n * n + ij];
    }
    for (int i = tid; i < n; i += blockDim.x) rdone[i] = cdone[i] = 0;
    __syncthreads();
    int prec = T;
    int64_t total = 0;
    for (int step = 0; step < n; step++) {
        if (tid == 0) best = ~0ull;
        __syncthreads();
        // pivot: least valuation, then least (row, col)
        for (int ij = tid; ij < n * n; ij += blockDim.x) {
            const int i = ij / n, j = ij % n;
            if (rdone[i] || cdone[j]) continue;
            const uint32_t *e = g + (size_t)ij * T;
            for (int t = 0; t < prec; t++)
                if (e[t]) {
                    unsigned long long key = ((unsigned long long)t << 40) | ((unsigned long long)i << 20) | j;
                    atomicMin(&best, key);
                    break;
                }
        }
        __syncthreads();
        const unsigned long long key = best;
        if (key == ~0ull) {
            if (tid == 0) *out = -1;
            return;
        }
        const int bv = (int)(key >> 40), bi = (int)((key >> 20) & 0xFFFFF), bj = (int)(key & 0xFFFFF);
        total += bv;
        const int np_ = prec - bv;
        const uint32_t *piv = g + ((size_t)bi * n + bj) * T + bv;  // unit part u
        if (tid == 0) {
            inv[0] = invm(piv[0], mp);
            for (int t = 1; t < np_; t++) {
                unsigned long long acc = 0;
                for (int s = 1; s <= t; s++) acc = red64(acc + (unsigned long long)piv[s] * inv[t - s], mp);
                inv[t] = mulm(subm(0, (uint32_t)acc, mp), inv[0], mp);
            }
        }
        __syncthreads();
        // mu_i = (g[i][bj] / x^bv) * inv  mod x^np_
        for (int w = tid; w < n * np_; w += blockDim.x) {
            const int i = w / np_, t = w % np_;
            if (rdone[i] || i == bi) continue;
            const uint32_t *gi = g + ((size_t)i * n + bj) * T + bv;
            unsigned long long acc = 0;
            for (int s = 0; s <= t; s++) acc = red64(acc + (unsigned long long)gi[s] * inv[t - s], mp);
            mu[(size_t)i * T + t] = (uint32_t)acc;
        }
        __syncthreads();
        // g[i][j] -= mu_i * g[bi][j]  mod x^np_, zero beyond
        for (int w = tid; w < n * n; w += blockDim.x) {
            const int i = w / n, j = w % n;
            if (rdone[i] || i == bi || cdone[j]) continue;
            uint32_t *gij = g + (size_t)w * T;
            const uint32_t *gb = g + ((size_t)bi * n + j) * T;
            const uint32_t *mi = mu + (size_t)i * T;
            for (int t = np_ - 1; t >= 0; t--) {
                unsigned long long acc = 0;
                for (int s = 0; s <= t; s++) acc = red64(acc + (unsigned long long)mi[s] * gb[t - s], mp);
                gij[t] = subm(gij[t], (uint32_t)acc, mp);
            }
            for (int t = np_; t < T; t++) gij[t] = 0;
        }
        __syncthreads();
        if (tid == 0) {
            rdone[bi] = 1;
            cdone[bj] = 1;
        }
        prec = np_;
        __syncthreads();
    }
    if (tid == 0) *out = total;
}

}  // namespace

// Blocked M-Basis over L orders.  [S | -I_m] (d_deg_in == nullptr): S holds
// L x m x n, d_P receives the first nr = n rows of the basis, d_deg the
// shifted degrees.  A general residual F (d_deg_in given): S holds L x m x q,
// nr = q, the basis starts at I_q with the degrees d_deg_in, and dbase is
// their minimum.  *dmax_out (optional): a bound on the basis's polynomial
// degree.
static wr_status mbasis_run(wr_ctx *ctx, const uint32_t *d_S, int64_t L, int m, int nr, int n, uint32_t p,
                            uint32_t *d_P, int32_t *d_deg, const int32_t *d_deg_in, int dbase, int64_t Dcap,
                            int64_t *dmax_out) {
    const int q = m + n;
    const ModP mp = make_modp(p);
    cudaStream_t s = ctx->stream;
    const size_t nq = (size_t)nr * q;
    WR_CUDA(cudaMemsetAsync(d_P, 0, sizeof(uint32_t) * (Dcap + 1) * nq, s));
    DevBuf P2, qtop, dmax, Epart, Ml, degl, scale;
    WR_TRY(dev_alloc(ctx, P2, sizeof(uint32_t) * (Dcap + 1) * nq));
    WR_CUDA(cudaMemsetAsync(P2.ptr, 0, P2.bytes, s));
    WR_TRY(dev_alloc(ctx, qtop, sizeof(uint32_t) * m * q));
    WR_TRY(dev_alloc(ctx, dmax, sizeof(int)));
    k_init_basis<<<1, 256, 0, s>>>(d_P, nr, n, q, d_deg, d_deg_in, qtop.as<uint32_t>(), m, dmax.as<int>());
    WR_LAUNCHED(ctx);

    // chunk size b and tiles: every kernel's shared memory must fit
    const size_t budget = std::min<size_t>(ctx->smem_optin, 227 * 1024) - 1024;
    const int MR = m <= 8 ? 8 : (m <= 16 ? 16 : 32);
    int CS = local_cluster(q);
    const int QC = MR == 8 ? (q <= 16 ? 16 : (q <= 32 ? 32 : 40)) : (q <= 32 ? 32 : (MR == 16 ? 48 : 64));
    const bool big = fold1_products(p) < FOLD_SMALL;
    using LocalFn = void (*)(int, int, int, const uint32_t *, uint32_t *, int32_t *, uint32_t *, int32_t *, int *,
                             uint32_t *, int, ModP);
    LocalFn kloc = nullptr;
#define WR_LOCAL(MRV, CPLV, QCV) kloc = big ? k_local<MRV, CPLV, QCV, FOLD_BIG> : k_local<MRV, CPLV, QCV, FOLD_SMALL>
    if (MR == 8) { if (QC == 16) WR_LOCAL(8, 1, 16); else if (QC == 32) WR_LOCAL(8, 1, 32); else WR_LOCAL(8, 2, 40); }
    else if (MR == 16) { if (QC == 32) WR_LOCAL(16, 1, 32); else WR_LOCAL(16, 2, 48); }
    else { if (QC == 32) WR_LOCAL(32, 1, 32); else WR_LOCAL(32, 2, 64); }
#undef WR_LOCAL
    WR_CUDA(cudaFuncSetAttribute(kloc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget));
    auto local_config = [&](size_t smem, cudaLaunchAttribute &at) {
        cudaLaunchConfig_t lc{};
        at = cudaLaunchAttribute{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)CS;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        lc.gridDim = dim3((unsigned)CS);
        lc.blockDim = dim3((unsigned)lc_threads(MR));
        lc.dynamicSmemBytes = smem;
        lc.stream = s;
        lc.attrs = &at;
        lc.numAttrs = 1;
        return lc;
    };
    if (CS > 8) {
        // more than the portable size: where the device can place such a cluster at all
        cudaLaunchAttribute at;
        int fit = 0;
        if (cudaFuncSetAttribute(kloc, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            [&] {
                const cudaLaunchConfig_t lc = local_config(budget, at);
                return cudaOccupancyMaxActiveClusters(&fit, kloc, &lc);
            }() != cudaSuccess || fit < 1) {
            cudaGetLastError();
            CS = 8;
        }
    }
    auto local_need = [&](int b) { return sizeof(uint32_t) * (size_t)lc_layout(m, q, b, CS, MR, QC).total; };
    int bmax = ctx->sigma_chunk > 0 ? std::min(ctx->sigma_chunk, 64) : sigma_chunk_default(q);
    while (bmax > 1 && local_need(bmax) > budget) bmax--;
    if (local_need(bmax) > budget) return fail(WR_EINVAL, "block sizes too large for shared memory");
    // the window's coefficients split so that about three blocks an SM run
    const int NC = q <= 16 ? 16 : (q <= 32 ? 32 : 64), BR = 4096 / NC;
    const int wtiles = (bmax * m + BR - 1) / BR;
    const int nparts_max = std::max(1, 3 * ctx->num_sms / wtiles);
    WR_TRY(dev_alloc(ctx, Epart, sizeof(uint32_t) * (size_t)nparts_max * bmax * m * q));
    WR_TRY(dev_alloc(ctx, Ml, sizeof(uint32_t) * (size_t)(bmax + 1) * q * q));
    WR_TRY(dev_alloc(ctx, degl, sizeof(int32_t) * q));
    WR_TRY(dev_alloc(ctx, scale, sizeof(uint32_t) * q));
    {
        std::vector<uint32_t> one(q, mp.r1);  // Montgomery form of 1
        WR_CUDA(cudaMemcpyAsync(scale.ptr, one.data(), sizeof(uint32_t) * q, cudaMemcpyHostToDevice, s));
        WR_CUDA(cudaStreamSynchronize(s));
    }
    auto *ktoep = NC == 16 ? (big ? k_toeplitz<16, FOLD_BIG> : k_toeplitz<16, TP_FOLD>)
                  : NC == 32 ? (big ? k_toeplitz<32, FOLD_BIG> : k_toeplitz<32, TP_FOLD>)
                             : (big ? k_toeplitz<64, FOLD_BIG> : k_toeplitz<64, TP_FOLD>);
    DevBuf Esum;
    WR_TRY(dev_alloc(ctx, Esum, sizeof(uint32_t) * (size_t)bmax * m * q));

    uint32_t *Pcur = d_P, *Pnext = P2.as<uint32_t>();
    int64_t Dbound = 1;
    // early termination on a sequence in flight: a quiet-order count per
    // chunk in host-mapped memory; the loop stays ET_LAG chunks ahead of the
    // device and stops once ctx->early_term consecutive orders were quiet
    SeqFeed *feed = d_deg_in ? nullptr : ctx->feed;
    const bool early = feed && ctx->early_term > 0;
    constexpr int ET_RING = 8, ET_LAG = 2;
    long long *et_host = nullptr, *et_host_dev = nullptr;
    cudaEvent_t et_ev[ET_RING] = {};
    DevBuf et_count;
    struct EtCleanup {
        long long *&h;
        cudaEvent_t *ev;
        ~EtCleanup() {
            if (h) cudaFreeHost(h);
            for (int i = 0; i < ET_RING; i++)
                if (ev[i]) cudaEventDestroy(ev[i]);
        }
    } et_cleanup{et_host, et_ev};
    if (early) {
        WR_CUDA(cudaHostAlloc((void **)&et_host, sizeof(long long) * ET_RING, cudaHostAllocMapped));
        for (int i = 0; i < ET_RING; i++) et_host[i] = -1;
        WR_CUDA(cudaHostGetDevicePointer((void **)&et_host_dev, et_host, 0));
        for (int i = 0; i < ET_RING; i++) WR_CUDA(cudaEventCreateWithFlags(&et_ev[i], WAIT_EVENT_FLAGS));
        WR_TRY(dev_alloc(ctx, et_count, sizeof(long long)));
        WR_CUDA(cudaMemsetAsync(et_count.ptr, 0, sizeof(long long), s));
    }
    int64_t Lused = L;
    // profiling: events around the three kernels of every 16th chunk
    cudaEvent_t pe[4] = {nullptr, nullptr, nullptr, nullptr};
    double pw = 0, pl = 0, pa = 0;
    int64_t nchunks = (L + bmax - 1) / bmax, sampled = 0;  // (profiling extrapolates to all L orders)
    if (ctx->profiling)
        for (auto &e : pe) WR_CUDA(cudaEventCreate(&e));
    for (int64_t k0 = 0; k0 < L; k0 += bmax) {
        const int bb = (int)std::min<int64_t>(bmax, L - k0);
        const bool prof = ctx->profiling && ((k0 / bmax) % 16 == 0);
        const int64_t chunk = k0 / bmax;
        if (early && chunk >= ET_LAG) {
            const int slot = (int)((chunk - ET_LAG) % ET_RING);
            WR_CUDA(cudaEventSynchronize(et_ev[slot]));
            if (*(volatile long long *)(et_host + slot) >= ctx->early_term) {
                Lused = k0;  // the generator is stable: the chunks so far are the whole basis
                feed->stop_at.store(k0);
                break;
            }
        }
        // a sequence still in flight: the window reads S rows below k0 + bb
        if (feed) WR_TRY(feed_wait(ctx, feed, std::min<int64_t>(L, k0 + bb)));
        if (prof) WR_CUDA(cudaEventRecord(pe[0], s));
        // window: coefficients [0, min(Dbound, k0 + bb - 1)] split over the parts
        const int64_t tspan = std::min<int64_t>(Dbound, k0 + bb - 1) + 1;
        const int64_t rows = (int64_t)bb * m;
        const int64_t tper = std::max<int64_t>((tspan + nparts_max - 1) / nparts_max, (TP_K + nr - 1) / nr);
        const int nparts = (int)((tspan + tper - 1) / tper);
        {
            const ToepArgs g{d_S, Pcur, Epart.as<uint32_t>(), rows, L * m, k0, m, nr, q, 0, tspan, tper, rows * q,
                             dmax.as<int>(), nullptr, nullptr};
            ktoep<<<dim3((unsigned)((rows + BR - 1) / BR), (unsigned)nparts), TP_THREADS, 0, s>>>(g, mp);
        }
        WR_LAUNCHED(ctx);
        const uint32_t *Ewin = Epart.as<uint32_t>();
        if (nparts > 1) {
            const int64_t E = (int64_t)bb * m * q;
            k_sum_parts<<<(unsigned)((E + 31) / 32), 256, 0, s>>>(nparts, E, Epart.as<uint32_t>(),
                                                                  Esum.as<uint32_t>(), mp);
            WR_LAUNCHED(ctx);
            Ewin = Esum.as<uint32_t>();
        }
        if (early) {
            k_quiet<<<1, 64, 0, s>>>(Ewin, bb, m, n, q, d_deg, k0, et_count.as<long long>(),
                                     et_host_dev + chunk % ET_RING);
            WR_LAUNCHED(ctx);
        }
        if (prof) WR_CUDA(cudaEventRecord(pe[1], s));
        {
            cudaLaunchAttribute at;
            const cudaLaunchConfig_t lc = local_config(local_need(bb), at);
            WR_CUDA(cudaLaunchKernelEx(&lc, kloc, m, q, bb, Ewin, qtop.as<uint32_t>(), d_deg, Ml.as<uint32_t>(),
                                       degl.as<int32_t>(), dmax.as<int>(), scale.as<uint32_t>(), dbase, mp));
        }
        WR_LAUNCHED(ctx);
        if (prof) WR_CUDA(cudaEventRecord(pe[2], s));
        if (Dbound + bb > Dcap + 1) return fail(WR_EINVAL, "sigma-basis degree cap too small");
        const int64_t Dnew = std::min<int64_t>(Dbound + bb, Dcap);
        {
            const int64_t prow = (Dnew + 1) * nr;
            const ToepArgs g{Pcur, Ml.as<uint32_t>(), Pnext, prow, prow, 0, nr, q, q, 0, bb + 1, bb + 1, 0,
                             nullptr, dmax.as<int>(), degl.as<int32_t>()};
            ktoep<<<dim3((unsigned)((prow + BR - 1) / BR)), TP_THREADS, 0, s>>>(g, mp);
        }
        WR_LAUNCHED(ctx);
        if (prof) {
            WR_CUDA(cudaEventRecord(pe[3], s));
            WR_CUDA(cudaEventSynchronize(pe[3]));
            float a = 0, b = 0, c = 0;
            cudaEventElapsedTime(&a, pe[0], pe[1]);
            cudaEventElapsedTime(&b, pe[1], pe[2]);
            cudaEventElapsedTime(&c, pe[2], pe[3]);
            pw += a;
            pl += b;
            pa += c;
            sampled++;
        }
        if (early) WR_CUDA(cudaEventRecord(et_ev[chunk % ET_RING], s));
        std::swap(Pcur, Pnext);
        Dbound = Dnew;
    }
    if (feed) feed->orders_used = Lused;
    if (ctx->profiling) {
        for (auto &e : pe) cudaEventDestroy(e);
        const double scale = sampled ? (double)nchunks / sampled : 0.0;  // extrapolate the samples
        ctx->last.sigma_window_ms += pw * scale;
        ctx->last.sigma_local_ms += pl * scale;
        ctx->last.sigma_apply_ms += pa * scale;
    }
    if (Pcur != d_P)
        WR_CUDA(cudaMemcpyAsync(d_P, Pcur, sizeof(uint32_t) * (Dbound + 1) * nq, cudaMemcpyDeviceToDevice, s));
    // divide the cumulative column scales out of P
    k_unscale<<<(unsigned)std::min<int64_t>(((Dbound + 1) * nq + 255) / 256, (int64_t)ctx->num_sms * 8), 256, 0, s>>>(
        d_P, nr, q, Dbound, scale.as<uint32_t>(), mp);
    WR_LAUNCHED(ctx);
    if (dmax_out) {
        int h = 0;
        WR_CUDA(cudaMemcpyAsync(&h, dmax.ptr, sizeof(int), cudaMemcpyDeviceToHost, s));
        WR_CUDA(sync_stream_blocking(s));
        *dmax_out = std::min<int64_t>(std::max(h, 0), Dbound);
    }
    WR_CUDA(sync_stream_blocking(s));  // (trailing a sequence: as long as the sequence)
    return WR_OK;
}

// F = [S | -I_m]: coefficients [k0, k1) of the L x m x q residual of the whole problem
__global__ void k_build_F(const uint32_t *__restrict__ S, int64_t k0, int64_t k1, int m, int n, uint32_t p,
                          uint32_t *__restrict__ F) {
    const int q = m + n;
    const int64_t total = (k1 - k0) * m * q;
    for (int64_t y = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; y < total; y += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = y + k0 * m * q;
        const int64_t k = x / (m * q);
        const int rem = (int)(x - k * m * q), a = rem / q, c = rem % q;
        F[x] = c < n ? S[((size_t)k * m + a) * n + c] : ((k == 0 && c - n == a) ? p - 1 : 0u);
    }
}

// P[t][r][c] = M[t][r][c] for the first n of the q rows, t <= D
__global__ void k_top_rows(const uint32_t *__restrict__ M, int64_t D, int n, int q, uint32_t *__restrict__ P) {
    const int64_t total = (D + 1) * n * q;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = x / ((int64_t)n * q);
        const int rem = (int)(x - t * n * q);
        P[x] = M[((size_t)t * q + rem / q) * q + rem % q];
    }
}

// PM-Basis (Section 2.4): the sigma-basis of the residual F (d orders, m x q)
// for the starting degrees in d_deg (updated to the final degrees) is M1 M2,
// M1 the basis of the first h orders and M2 that of the residual
// R = (F M1) div x^h mod x^(d-h), the latter started from M1's degrees.  The
// leaves (d <= leaf) run the blocked M-Basis on a general residual; the
// residual and the product are polynomial matrix products by NTT (CRT over
// three FFT primes).  Each leaf's basis is the order-by-order one, so M is.
static wr_status pm_basis_rec(wr_ctx *ctx, const uint32_t *F, int64_t d, int m, int q, uint32_t p,
                              int32_t *d_deg, int64_t leaf, DevBuf &M, int64_t &DM) {
    cudaStream_t s = ctx->stream;
    std::vector<int32_t> h0(q);
    WR_CUDA(cudaMemcpyAsync(h0.data(), d_deg, sizeof(int32_t) * q, cudaMemcpyDeviceToHost, s));
    WR_CUDA(cudaStreamSynchronize(s));
    const int dbase = *std::min_element(h0.begin(), h0.end());
    if (d <= leaf) {
        WR_TRY(dev_alloc(ctx, M, sizeof(uint32_t) * (size_t)(d + 2) * q * q));
        DevBuf degin;
        WR_TRY(dev_alloc(ctx, degin, sizeof(int32_t) * q));
        WR_CUDA(cudaMemcpyAsync(degin.ptr, d_deg, sizeof(int32_t) * q, cudaMemcpyDeviceToDevice, s));
        return mbasis_run(ctx, F, d, m, q, q - m, p, M.as<uint32_t>(), d_deg, degin.as<int32_t>(), dbase, d + 1, &DM);
    }
    int64_t h = ((d / 2 + 63) / 64) * 64;
    if (h >= d) h = d / 2;
    DevBuf M1, M2, R;
    int64_t DM1 = 0, DM2 = 0;
    WR_TRY(pm_basis_rec(ctx, F, h, m, q, p, d_deg, leaf, M1, DM1));
    WR_TRY(dev_alloc(ctx, R, sizeof(uint32_t) * (size_t)(d - h) * m * q));
    WR_TRY(polymat_mul(ctx, F, d, M1.as<uint32_t>(), DM1 + 1, m, q, q, h, d, p, R.as<uint32_t>()));
    WR_TRY(pm_basis_rec(ctx, R.as<uint32_t>(), d - h, m, q, p, d_deg, leaf, M2, DM2));
    R.release();
    // degree of M: at most DM1 + DM2, and at most the largest final degree
    // minus the smallest starting one
    std::vector<int32_t> h1(q);
    WR_CUDA(cudaMemcpyAsync(h1.data(), d_deg, sizeof(int32_t) * q, cudaMemcpyDeviceToHost, s));
    WR_CUDA(cudaStreamSynchronize(s));
    const int64_t bound = (int64_t)*std::max_element(h1.begin(), h1.end()) - dbase;
    DM = std::max<int64_t>(0, std::min<int64_t>(DM1 + DM2, bound));
    WR_TRY(dev_alloc(ctx, M, sizeof(uint32_t) * (size_t)(DM + 2) * q * q));
    WR_CUDA(cudaMemsetAsync(M.ptr, 0, M.bytes, s));
    return polymat_mul(ctx, M1.as<uint32_t>(), DM1 + 1, M2.as<uint32_t>(), DM2 + 1, q, q, q, 0, DM + 1, p,
                       M.as<uint32_t>());
}

static int64_t sigma_leaf_for(const wr_ctx *ctx, int m, int n) {
    return ctx->sigma_leaf > 0 ? ctx->sigma_leaf : (m + n > 32 ? SIGMA_LEAF_WIDE : SIGMA_LEAF_DEFAULT);
}

// PM-Basis (else the blocked M-Basis) for L orders; early termination needs
// the order-by-order basis (PM-Basis splits the orders in halves and so needs
// all of them from the start)
bool sigma_uses_pm(const wr_ctx *ctx, int64_t L, int m, int n, bool early) {
    const int64_t leaf = sigma_leaf_for(ctx, m, n);
    const bool automatic = ctx->sigma_leaf <= 0;
    return !(early || L <= leaf || (automatic && L <= (m + n > 32 ? SIGMA_PM_MIN_L_WIDE : SIGMA_PM_MIN_L)));
}

bool sigma_pm_trailing(const wr_ctx *ctx, int64_t L, int m, int n) {
    return sigma_uses_pm(ctx, L, m, n, ctx->early_term > 0) && L > 2 * sigma_leaf_for(ctx, m, n);
}

wr_status sigma_basis(wr_ctx *ctx, const uint32_t *d_S, int64_t L, int m, int n, uint32_t p,
                      uint32_t *d_P, int32_t *d_deg, int64_t Dcap) {
    if (m < 1 || n < 1 || m > 32 || n > 32) return fail(WR_EINVAL, "block sizes must be in 1..32");
    ctx->last.sigma_window_ms = ctx->last.sigma_local_ms = ctx->last.sigma_apply_ms = 0.0;
    ctx->last.sigma_product_ms = 0.0;
    const int64_t leaf = sigma_leaf_for(ctx, m, n);
    const bool early = ctx->feed && ctx->early_term > 0;
    if (!sigma_uses_pm(ctx, L, m, n, early))
        return mbasis_run(ctx, d_S, L, m, n, n, p, d_P, d_deg, nullptr, 0, Dcap, nullptr);
    const int q = m + n;
    cudaStream_t s = ctx->stream;
    DevBuf F, M;
    WR_TRY(dev_alloc(ctx, F, sizeof(uint32_t) * (size_t)L * m * q));
    auto build_F = [&](int64_t k0, int64_t k1) -> wr_status {
        if (k1 <= k0) return WR_OK;
        const unsigned g = (unsigned)std::min<int64_t>(((k1 - k0) * m * q + 255) / 256, (int64_t)ctx->num_sms * 16);
        k_build_F<<<g, 256, 0, s>>>(d_S, k0, k1, m, n, p, F.as<uint32_t>());
        WR_LAUNCHED(ctx);
        return WR_OK;
    };
    std::vector<int32_t> deg0(q);
    for (int c = 0; c < q; c++) deg0[c] = c < n ? 0 : 1;
    WR_CUDA(cudaMemcpyAsync(d_deg, deg0.data(), sizeof(int32_t) * q, cudaMemcpyHostToDevice, s));
    WR_CUDA(cudaStreamSynchronize(s));
    int64_t DM = 0;
    // Trailing a sequence still in flight: the orders are taken in segments
    // [h_{k-1}, h_k) as the sequence publishes them.  A segment's residual is
    // R_k = (F M) div x^h_{k-1} mod x^(h_k - h_{k-1}) (a middle product of F's
    // coefficients [h_{k-1} - deg M, h_k) and the basis M of the orders before
    // it), its sigma-basis M_k starts from M's degrees, and M <- M M_k:
    // PM-Basis's split at h_{k-1}, applied once per segment.  Each segment is
    // about half of the orders still to come but at most a quarter of all
    // (the first starts when a quarter of the terms are in), down to two
    // leaves, so that what is left after the sequence's last term is one short
    // segment and two products.  (Segments that take every term finished meanwhile, from the
    // first sixteenth on, were measured slower on the 1.9M x 1.95M block-32
    // matrix: their kernels ran beside the SpMM for the whole sequence, each
    // segment with its two products, and cost the SpMM more than the shorter
    // tail saved.)
    if (ctx->feed && L > 2 * leaf) {
        const int64_t seg_min = 2 * leaf;
        std::vector<int32_t> hd(q);
        int64_t hprev = 0;
        for (int k = 0; hprev < L; k++) {
            const int64_t rem = L - hprev;
            const int64_t half = std::min<int64_t>(rem / 2, L / 4);
            const int64_t hk =
                hprev + (rem <= 2 * seg_min ? rem : std::max<int64_t>(seg_min, ((half + 63) / 64) * 64));
            const int64_t d = hk - hprev;
            WR_TRY(feed_wait(ctx, ctx->feed, hk));
            WR_TRY(build_F(hprev, hk));
            DevBuf R, Mk;
            int64_t DMk = 0;
            if (k > 0) {
                // R_i = sum_j F_j M_{i-j}, j in [i - DM, i]: F from hprev - DM on
                const int64_t off = std::max<int64_t>(0, hprev - DM);
                WR_TRY(dev_alloc(ctx, R, sizeof(uint32_t) * (size_t)d * m * q));
                WR_TRY(polymat_mul(ctx, F.as<uint32_t>() + (size_t)off * m * q, hk - off, M.as<uint32_t>(), DM + 1, m,
                                   q, q, hprev - off, hk - off, p, R.as<uint32_t>()));
            }
            WR_TRY(pm_basis_rec(ctx, k > 0 ? R.as<uint32_t>() : F.as<uint32_t>(), d, m, q, p, d_deg, leaf, Mk, DMk));
            R.release();
            if (k == 0) {
                M = std::move(Mk);
                DM = DMk;
            } else {
                WR_CUDA(cudaMemcpyAsync(hd.data(), d_deg, sizeof(int32_t) * q, cudaMemcpyDeviceToHost, s));
                WR_CUDA(cudaStreamSynchronize(s));
                // starting degrees (0^n, 1^m): the smallest is 0
                const int64_t bound = (int64_t)*std::max_element(hd.begin(), hd.end());
                const int64_t DMn = std::max<int64_t>(0, std::min<int64_t>(DM + DMk, bound));
                DevBuf Mn;
                WR_TRY(dev_alloc(ctx, Mn, sizeof(uint32_t) * (size_t)(DMn + 2) * q * q));
                WR_CUDA(cudaMemsetAsync(Mn.ptr, 0, Mn.bytes, s));
                WR_TRY(polymat_mul(ctx, M.as<uint32_t>(), DM + 1, Mk.as<uint32_t>(), DMk + 1, q, q, q, 0, DMn + 1, p,
                                   Mn.as<uint32_t>()));
                M = std::move(Mn);
                DM = DMn;
            }
            hprev = hk;
        }
    } else {
        if (ctx->feed) WR_TRY(feed_wait(ctx, ctx->feed, L));  // PM-Basis reads the whole sequence
        WR_TRY(build_F(0, L));
        WR_TRY(pm_basis_rec(ctx, F.as<uint32_t>(), L, m, q, p, d_deg, leaf, M, DM));
    }
    if (DM > Dcap) return fail(WR_EINVAL, "sigma-basis degree cap too small");
    WR_CUDA(cudaMemsetAsync(d_P, 0, sizeof(uint32_t) * (Dcap + 1) * n * q, s));
    const unsigned g2 = (unsigned)std::min<int64_t>(((DM + 1) * n * q + 255) / 256, (int64_t)ctx->num_sms * 16);
    k_top_rows<<<g2, 256, 0, s>>>(M.as<uint32_t>(), DM, n, q, d_P);
    WR_LAUNCHED(ctx);
    WR_CUDA(cudaStreamSynchronize(s));
    return WR_OK;
}

wr_status det_valuation(wr_ctx *ctx, const uint32_t *d_G, int64_t n, int64_t T, uint32_t p, int64_t *val) {
    if (n <= 0) { *val = 0; return WR_OK; }
    if (n > 64 || T < 1 || T > 4096) return fail(WR_EINVAL, "det valuation: n in 1..64 and T in 1..4096");
    const ModP mp = make_modp(p);
    DevBuf g, out;
    WR_TRY(dev_alloc(ctx, g, sizeof(uint32_t) * n * n * T));
    WR_TRY(dev_alloc(ctx, out, sizeof(int64_t)));
    size_t smem = sizeof(uint32_t) * (T + (size_t)n * T) + sizeof(int) * 2 * n;
    if (smem > 200 * 1024) return fail(WR_EINVAL, "det valuation: precision too large");
    WR_CUDA(cudaFuncSetAttribute(k_valuation, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::max<size_t>(smem, 48 * 1024)));
    k_valuation<<<1, VAL_THREADS, smem, ctx->stream>>>(d_G, g.as<uint32_t>(), (int)n, (int)T,
                                                       out.as<int64_t>(), mp);
    WR_LAUNCHED(ctx);
    WR_CUDA(cudaMemcpyAsync(val, out.ptr, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    WR_CUDA(cudaStreamSynchronize(ctx->stream));
    return WR_OK;
}

wr_status rank_readout(wr_ctx *ctx, const uint32_t *d_P, const int32_t *d_deg, int m, int n, uint32_t p,
                       int64_t Dcap, Readout &out, std::vector<uint32_t> *gen) {
    const int q = m + n;
    cudaStream_t s = ctx->stream;
    DevBuf sel, delta;
    WR_TRY(dev_alloc(ctx, sel, sizeof(int32_t) * n));
    WR_TRY(dev_alloc(ctx, delta, sizeof(int32_t) * n));
    k_select<<<1, 64, 0, s>>>(d_deg, q, n, sel.as<int32_t>(), delta.as<int32_t>());
    WR_LAUNCHED(ctx);
    out.delta.assign(n, 0);
    WR_CUDA(cudaMemcpyAsync(out.delta.data(), delta.ptr, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    WR_CUDA(cudaStreamSynchronize(s));
    int64_t sd = 0, dmax = 0;
    for (int j = 0; j < n; j++) {
        sd += out.delta[j];
        dmax = std::max<int64_t>(dmax, out.delta[j]);
    }
    out.sum_delta = sd;
    out.dmax = dmax;
    // valuations of det P and det F (F_j(x) = x^delta_j P_j(1/x)); double the
    // precision until every pivot is found; coefficients past the degree are
    // zero, so T > n (dmax + 1) decides det = 0.
    int64_t vals[2] = {0, 0};
    for (int which = 0; which < 2; which++) {
        int64_t T = 8;
        for (;;) {
            DevBuf G;
            WR_TRY(dev_alloc(ctx, G, sizeof(uint32_t) * T * n * n));
            k_extract<<<blocks_for(T * n * n, 256), 256, 0, s>>>(d_P, n, q, sel.as<int32_t>(), delta.as<int32_t>(),
                                                                 T, which, Dcap, G.as<uint32_t>());
            WR_LAUNCHED(ctx);
            int64_t v = -1;
            WR_TRY(det_valuation(ctx, G.as<uint32_t>(), n, T, p, &v));
            if (v >= 0) { vals[which] = v; break; }
            if (T > (int64_t)n * (dmax + 1) + 2 || T >= 4096)
                return fail(WR_EPROBFAIL, "generator determinant vanishes (singular generator)");
            T *= 2;
        }
    }
    out.vP = vals[0];
    out.codeg = vals[1];
    out.deg_det = sd - vals[0];
    out.rank = out.deg_det - out.codeg;
    if (gen) {
        const int64_t T = dmax + 1;
        DevBuf G;
        WR_TRY(dev_alloc(ctx, G, sizeof(uint32_t) * T * n * n));
        k_extract<<<blocks_for(T * n * n, 256), 256, 0, s>>>(d_P, n, q, sel.as<int32_t>(), delta.as<int32_t>(),
                                                             T, 1, Dcap, G.as<uint32_t>());
        WR_LAUNCHED(ctx);
        gen->resize((size_t)T * n * n);
        WR_CUDA(cudaMemcpyAsync(gen->data(), G.ptr, sizeof(uint32_t) * gen->size(), cudaMemcpyDeviceToHost, s));
        WR_CUDA(cudaStreamSynchronize(s));
    }
    return WR_OK;
}

}  // namespace wr
