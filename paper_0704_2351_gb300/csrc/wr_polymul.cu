// Products of polynomial matrices mod p by number-theoretic transforms, for
// the PM-Basis sigma-basis (Section 2.4: "PM-Basis ... reduces this
// computation to polynomial matrix multiplication", FFT primes c 2^k + 1, and
// CRT with several FFT primes when the field itself has no large 2^k-th roots
// of unity, with prod p_i > d n p^2).
//
// C = A B with A (r x s) and B (s x t) polynomial matrices whose entries are
// residues mod p, stored coefficient-major ([coef][row][col]).  Each product
// entry is computed exactly as an integer -- a sum of at most
// s * min(deg A, deg B) + s products below p^2 < 2^62, so below 2^88 for
// s <= 64 and degrees below 2^20 -- from its residues modulo three FFT primes
// whose product exceeds 2^89, and then reduced mod p.  Only the coefficients
// [lo, hi) of C are produced; a cyclic transform of length Lz >= hi whose
// wrapped-around part (coefficients at and above Lz folded onto 0..) stays
// below lo gives exactly those (a middle product when lo > 0).
//
// Transforms: X^n - 1 is split as X^2k - c^2 = (X^k - c)(X^k + c) down to linear
// factors, (u, v) -> (u + c v, u - c v) per stage, so that a stage's twiddle c
// depends on the block alone: the pairs of a block share one table entry,
// consecutive blocks read consecutive ones, and one table of the 2^i-th roots
// in bit-reversed order serves every length.  The order of the transform's
// points does not matter to the pointwise products; the inverse undoes the
// stages in reverse.  Residues in Montgomery form.  Up to 2^13 points a
// transform is one pass (registers and shared memory, k_ntt_tile); longer ones
// take their top stages in passes of up to four stages in registers
// (k_ntt_top), each one launch over all polynomials of the batch.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "wr_internal.cuh"

namespace wr {

namespace {

constexpr int NTT_NPRIMES = 3;
constexpr uint32_t NTT_PRIMES[NTT_NPRIMES] = {998244353u, 469762049u, 2013265921u};  // 119 2^23+1, 7 2^26+1, 15 2^27+1
// products between folds in the pointwise sums (P < 2^30, else)
constexpr int PW_FOLD_SMALL = 16, PW_FOLD_BIG = 4;
static_assert(fold1_products(NTT_PRIMES[0]) >= PW_FOLD_SMALL && fold1_products(NTT_PRIMES[1]) >= PW_FOLD_SMALL &&
                  fold1_products(NTT_PRIMES[2]) >= PW_FOLD_BIG,
              "folded sums");
constexpr int NTT_MAX_LOG = 23;  // 2^23 divides every p_i - 1

uint64_t hpow(uint64_t a, uint64_t e, uint64_t m) {
    uint64_t r = 1 % m;
    a %= m;
    while (e) {
        if (e & 1) r = (unsigned __int128)r * a % m;
        a = (unsigned __int128)a * a % m;
        e >>= 1;
    }
    return r;
}

// smallest generator of the multiplicative group mod prime P (checked
// against every prime factor of P - 1)
uint32_t primitive_root(uint32_t P) {
    std::vector<uint64_t> f;
    uint64_t x = P - 1;
    for (uint64_t d = 2; d * d <= x; d++)
        if (x % d == 0) {
            f.push_back(d);
            while (x % d == 0) x /= d;
        }
    if (x > 1) f.push_back(x);
    for (uint32_t g = 2;; g++) {
        bool ok = true;
        for (uint64_t q : f)
            if (hpow(g, (P - 1) / q, P) == 1) { ok = false; break; }
        if (ok) return g;
    }
}

// a (mod p, any p < 2^31) -> Montgomery form mod P, transposed to one
// contiguous run of Lz coefficients per polynomial (zero padded).  Tiles of
// 32 coefficients x 32 entries go through shared memory, so that both the
// reads (along the entries of a coefficient) and the writes (along the
// coefficients of an entry) are coalesced.
constexpr int TR_TILE = 32, TR_ROWS = 8;  // tile edge; thread rows of a 32 x 8 block

__global__ void __launch_bounds__(TR_TILE * TR_ROWS)
    k_ntt_load(const uint32_t *__restrict__ src, int64_t ncoef, int nent, int64_t Lz, uint32_t *__restrict__ dst,
               ModP mP) {
    __shared__ uint32_t tile[TR_TILE][TR_TILE + 1];
    const int tx = threadIdx.x & (TR_TILE - 1), ty = threadIdx.x / TR_TILE;
    const int64_t ktiles = (Lz + TR_TILE - 1) / TR_TILE, etiles = (nent + TR_TILE - 1) / TR_TILE;
    for (int64_t tl = blockIdx.x; tl < ktiles * etiles; tl += gridDim.x) {
        const int64_t k0 = (tl % ktiles) * TR_TILE;
        const int e0 = (int)(tl / ktiles) * TR_TILE;
        __syncthreads();
        if (k0 < ncoef) {
            for (int y = ty; y < TR_TILE; y += TR_ROWS) {
                const int64_t k = k0 + y;
                const int e = e0 + tx;
                // (a r2 < 2^32 P for any 32-bit a: no reduction before the product)
                tile[y][tx] = (k < ncoef && e < nent) ? to_mont(src[(size_t)k * nent + e], mP) : 0u;
            }
        }
        __syncthreads();
        for (int y = ty; y < TR_TILE; y += TR_ROWS) {
            const int e = e0 + y;
            const int64_t k = k0 + tx;
            if (e < nent && k < Lz) dst[(size_t)e * Lz + k] = k0 < ncoef ? tile[tx][y] : 0u;
        }
    }
}

// tw[i] = w^bitrev(i) (Montgomery form, w_m = w R mod P, w a 2^(bits+1)-th root,
// bitrev over `bits` bits) for i < 2^bits, by square and multiply
__global__ void k_twiddles(uint32_t w_m, int bits, uint32_t *__restrict__ tw, ModP mP) {
    const int64_t count = (int64_t)1 << bits;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t r = mP.r1, b = w_m;
        for (uint32_t e = bits ? __brev((uint32_t)i) >> (32 - bits) : 0u; e; e >>= 1) {
            if (e & 1) r = mont_mul(r, b, mP);
            b = mont_mul(b, b, mP);
        }
        tw[i] = r;
    }
}

// residues mod P < 2^31 as the smaller of x and x - P (or x + P) as unsigned
__device__ __forceinline__ uint32_t ntt_add(uint32_t a, uint32_t b, uint32_t P) {
    const uint32_t s = a + b;
    return min(s, s - P);
}
__device__ __forceinline__ uint32_t ntt_sub(uint32_t a, uint32_t b, uint32_t P) {
    const uint32_t d = a - b;
    return min(d, d + P);
}
__device__ __forceinline__ uint32_t ntt_mul(uint32_t a, uint32_t b, uint32_t P, uint32_t pneg) {
    const unsigned long long t = (unsigned long long)a * b;
    const uint32_t k = (uint32_t)t * pneg;
    const uint32_t u = (uint32_t)(madw(k, P, t) >> 32);
    return min(u, u - P);
}

// the 2^K consecutive table entries of a stage, in loads of up to 16 bytes
// (entry blk 2^K of a table aligned to more)
template <int K>
__device__ __forceinline__ void ntt_twiddles(const uint32_t *__restrict__ tw, uint32_t blk, uint32_t (&c)[1 << K]) {
    const uint32_t *p = tw + ((size_t)blk << K);
    if constexpr (K == 0) {
        c[0] = __ldg(p);
    } else if constexpr (K == 1) {
        const uint2 t = __ldg(reinterpret_cast<const uint2 *>(p));
        c[0] = t.x; c[1] = t.y;
    } else {
#pragma unroll
        for (int k = 0; k < (1 << K) / 4; k++) {
            const uint4 t = __ldg(reinterpret_cast<const uint4 *>(p) + k);
            c[4 * k] = t.x; c[4 * k + 1] = t.y; c[4 * k + 2] = t.z; c[4 * k + 3] = t.w;
        }
    }
}

// Stage K of R on 2^R values: 2^K blocks of 2^(R - K) values.
template <int R, int K, bool FWD>
__device__ __forceinline__ void ntt_stage(uint32_t (&v)[1 << R], uint32_t blk, const uint32_t *__restrict__ tw, uint32_t P,
                                          uint32_t pneg) {
    constexpr int half = 1 << (R - 1 - K);
    uint32_t c[1 << K];
    ntt_twiddles<K>(tw, blk, c);
#pragma unroll
    for (int b = 0; b < (1 << K); b++)
#pragma unroll
        for (int i = 0; i < half; i++) {
            uint32_t &x = v[b * 2 * half + i], &y = v[b * 2 * half + i + half];
            if (FWD) {
                const uint32_t m = ntt_mul(y, c[b], P, pneg);
                y = ntt_sub(x, m, P);
                x = ntt_add(x, m, P);
            } else {
                const uint32_t d = ntt_sub(x, y, P);
                x = ntt_add(x, y, P);
                y = ntt_mul(d, c[b], P, pneg);
            }
        }
}

// R stages on 2^R values held in registers; blk: the block that they belong to
// at the first (forward) of these stages.
template <int R, bool FWD>
__device__ __forceinline__ void ntt_stages(uint32_t (&v)[1 << R], uint32_t blk, const uint32_t *__restrict__ tw,
                                           uint32_t P, uint32_t pneg) {
    if constexpr (!FWD && R > 3) ntt_stage<R, 3, FWD>(v, blk, tw, P, pneg);
    if constexpr (!FWD && R > 2) ntt_stage<R, 2, FWD>(v, blk, tw, P, pneg);
    if constexpr (!FWD && R > 1) ntt_stage<R, 1, FWD>(v, blk, tw, P, pneg);
    ntt_stage<R, 0, FWD>(v, blk, tw, P, pneg);
    if constexpr (FWD && R > 1) ntt_stage<R, 1, FWD>(v, blk, tw, P, pneg);
    if constexpr (FWD && R > 2) ntt_stage<R, 2, FWD>(v, blk, tw, P, pneg);
    if constexpr (FWD && R > 3) ntt_stage<R, 3, FWD>(v, blk, tw, P, pneg);
}

// The top K stages (s0 .. s0 + K - 1) of transforms of 2^lg points, in
// registers: one thread per group of 2^K values, lanes along consecutive values.
constexpr int NTT_TOP_THREADS = 256;
template <int K, bool FWD>
__global__ void __launch_bounds__(NTT_TOP_THREADS)
    k_ntt_top(uint32_t *__restrict__ a, int64_t npoly, int lg, int s0, const uint32_t *__restrict__ tw, uint32_t P,
              uint32_t pneg) {
    const int sl = lg - s0 - K;  // log2 of the distance between a group's values
    const int64_t groups = npoly << (lg - K);
    for (int64_t g = (int64_t)blockIdx.x * NTT_TOP_THREADS + threadIdx.x; g < groups;
         g += (int64_t)gridDim.x * NTT_TOP_THREADS) {
        const int64_t hi = g >> sl, low = g & (((int64_t)1 << sl) - 1);  // hi = poly 2^s0 + block
        uint32_t *p = a + (hi << (sl + K)) + low;
        uint32_t v[1 << K];
#pragma unroll
        for (int i = 0; i < (1 << K); i++) v[i] = p[(int64_t)i << sl];
        ntt_stages<K, FWD>(v, (uint32_t)(hi & (((int64_t)1 << s0) - 1)), tw, P, pneg);
#pragma unroll
        for (int i = 0; i < (1 << K); i++) p[(int64_t)i << sl] = v[i];
    }
}

// The last lc stages of transforms of 2^lg points (lc = 13, or lg when lg < 13):
// a block takes a tile of 2^13 values (2^(13-lc) transforms when lc < 13)
// through all of them in two to four steps of R = 2, 3 or 4 stages, each thread
// 16 values in registers, exchanged through shared memory between steps
// (padded by one word in 32).  One read and one write of the data: the first
// step reads global memory, the last one writes it with the values of a step's
// group apart (element i of group g at i 2^(lc-R) + g), which keeps the writes
// coalesced; the inverse reads that order back.  Bound by the butterflies' issue
// (a product mod P, a sum and a difference: 11 instructions).  Measured: 4,096
// transforms of 8,192 points 1,140 -> 200 us (two passes with one
// shared-memory round trip and one scattered twiddle load per stage before).
constexpr int NTT_TILE_LOG = 13;
constexpr int NTT_TILE_THREADS = 512;

struct NttSteps {
    int n;
    int R[4];  // forward order: from the highest bits down
};
__host__ __device__ inline NttSteps ntt_steps(int lc) {
    NttSteps st{(lc + 3) / 4, {0, 0, 0, 0}};
    if (st.n < 2) st.n = 2;
    for (int k = 0, left = lc; k < st.n; k++) {
        st.R[k] = (left + st.n - k - 1) / (st.n - k);
        left -= st.R[k];
    }
    return st;
}

__device__ __forceinline__ int ntt_pad(int e) { return e + (e >> 5); }

// One step: h0 the lowest bit it touches.  SRC / DST: 0 shared memory, 1 the
// tile in natural order, 2 the tile in the transform's order.  SHORT: transforms past
// the end are left out.
template <int R, bool FWD, bool SHORT, int SRC, int DST>
__device__ __forceinline__ void ntt_step(uint32_t *sm, uint32_t *__restrict__ g, int valid, int lc, int h0, uint32_t top,
                                         const uint32_t *__restrict__ tw, uint32_t P, uint32_t pneg) {
    constexpr int NG = 16 >> R;  // groups per thread
#pragma unroll
    for (int u = 0; u < NG; u++) {
        const int gi = threadIdx.x + u * NTT_TILE_THREADS;
        const int base = ((gi >> h0) << (h0 + R)) | (gi & ((1 << h0) - 1));
        const int gp = gi & ((1 << (lc - R)) - 1);  // group within its transform
        const int pbase = ((gi >> (lc - R)) << lc) + gp;
        const uint32_t blk = (top << (lc - h0 - R)) + (uint32_t)((base & ((1 << lc) - 1)) >> (h0 + R));
        if (SHORT && base >> lc << lc >= valid) continue;
        uint32_t v[1 << R];
#pragma unroll
        for (int i = 0; i < (1 << R); i++) {
            const int e = base + (i << h0), pe = pbase + (i << (lc - R));
            if (SRC == 0) v[i] = sm[ntt_pad(e)];
            else if (SRC == 1) v[i] = e < valid ? g[e] : 0u;
            else v[i] = pe < valid ? g[pe] : 0u;
        }
        ntt_stages<R, FWD>(v, blk, tw, P, pneg);
#pragma unroll
        for (int i = 0; i < (1 << R); i++) {
            const int e = base + (i << h0), pe = pbase + (i << (lc - R));
            if (DST == 0) sm[ntt_pad(e)] = v[i];
            else if (DST == 1) { if (e < valid) g[e] = v[i]; }
            else if (pe < valid) g[pe] = v[i];
        }
    }
}

// SHORT: a launch of a single tile that is not full (a product of a few short
// polynomials: 1 x 1 x 1, 100 coefficients, 118 -> 106 us; the test cost launches of
// many tiles 2 %, so their last tile takes the empty transforms along).
template <bool FWD, bool SHORT>
__global__ void __launch_bounds__(NTT_TILE_THREADS, 2)
    k_ntt_tile(uint32_t *__restrict__ a, int64_t words, int lg, int lc, const uint32_t *__restrict__ tw, uint32_t P,
               uint32_t pneg) {
    __shared__ uint32_t sm[(1 << NTT_TILE_LOG) + (1 << (NTT_TILE_LOG - 5))];
    uint32_t *g = a + ((int64_t)blockIdx.x << NTT_TILE_LOG);
    // (the last tile may be short)
    const int valid = (int)min64(words - ((int64_t)blockIdx.x << NTT_TILE_LOG), 1 << NTT_TILE_LOG);
    const uint32_t top = lg > lc ? (uint32_t)(blockIdx.x & ((1u << (lg - lc)) - 1)) : 0u;
    const NttSteps st = ntt_steps(lc);
    int h0 = FWD ? lc : 0;
    for (int k = 0; k < st.n; k++) {
        const int R = st.R[FWD ? k : st.n - 1 - k];
        if (FWD) h0 -= R;
        if (k > 0) __syncthreads();
#define WR_NTT_STEP(SRC, DST)                                                                    \
    {                                                                                            \
        if (R == 4) ntt_step<4, FWD, SHORT, SRC, DST>(sm, g, valid, lc, h0, top, tw, P, pneg);          \
        else if (R == 3) ntt_step<3, FWD, SHORT, SRC, DST>(sm, g, valid, lc, h0, top, tw, P, pneg);     \
        else ntt_step<2, FWD, SHORT, SRC, DST>(sm, g, valid, lc, h0, top, tw, P, pneg);                 \
    }
        if (k == 0) WR_NTT_STEP((FWD ? 1 : 2), 0)
        else if (k + 1 < st.n) WR_NTT_STEP(0, 0)
        else WR_NTT_STEP(0, (FWD ? 2 : 1))
#undef WR_NTT_STEP
        if (!FWD) h0 += R;
    }
}

// pointwise: C_f = A_f B_f (r x s times s x t) at every transform point f.  A
// lane owns a point (rows of 32 consecutive points are 128-byte lines), a
// thread a 4 x 8 tile of C at it, a block of eight warps WR x WC such tiles for
// 8 / (WR WC) groups of 32 points.  The operands of KC values of k are staged in
// shared memory (16-byte asynchronous copies, two stages), so that an A word
// serves 8 WC columns and a B word 4 WR rows per read of L2, and an operand
// costs a conflict-free shared load for 8 or 4 products.  The sums run on
// 64-bit accumulators (one 32 x 32 + 64-bit multiply-add per product), folded by
// 2^32 = r1 (mod P) every FOLDK products: a folded accumulator is below 2^60.3
// for the transform primes (2^32 mod P < 2^28.3), which leaves room for 16
// products below 2^59.8 (P < 2^30) or 4 below 2^61.9.  Bound by the
// multiply-adds.  Measured at 64 x 64 x 64, 8,192 points: 4.65 ms -> 430 us
// (P < 2^30; 480 us with the third prime's folds; before, a
// thread's operands came straight from L1 and L2, with eight warps an SM).
constexpr int PW_RT = 4, PW_CT = 8, PW_WARPS = 8;

__device__ __forceinline__ void cp_async16(uint32_t *dst, const uint32_t *src, bool on) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(on ? 16 : 0)
                 : "memory");
}
template <int WR, int WC, int KC>
struct PwShape {
    static constexpr int FG = PW_WARPS / (WR * WC);
    static constexpr int TR = PW_RT * WR, TC = PW_CT * WC;  // rows and columns of C per block
    static constexpr int STAGE = FG * KC * (TR + TC) * 32;  // words
    static constexpr size_t SMEM = 2 * (size_t)STAGE * 4;
};

template <int WR, int WC, int KC, int FOLDK>
__global__ void __launch_bounds__(32 * PW_WARPS, 2)
    k_ntt_pointwise(const uint32_t *__restrict__ A, const uint32_t *__restrict__ B, uint32_t *__restrict__ C, int r,
                    int s, int t, int64_t Lz, ModP mP) {
    using S = PwShape<WR, WC, KC>;
    extern __shared__ __align__(16) uint32_t pw_sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int fg = warp / (WR * WC), wr = warp / WC % WR, wc = warp % WC;
    const int ntj = (t + S::TC - 1) / S::TC;
    const int i0 = (int)(blockIdx.y / ntj) * S::TR, j0 = (int)(blockIdx.y % ntj) * S::TC;
    const int64_t f0 = (int64_t)blockIdx.x * 32 * S::FG;
    const uint32_t fc = mP.r1;  // 2^32 mod P
    // stage: [group][k][TR rows of A, then TC columns of B][32 points]
    auto load = [&](int k0, int stage) {
        uint32_t *sm = pw_sm + stage * S::STAGE;
        for (int c = threadIdx.x; c < S::STAGE / 4; c += 32 * PW_WARPS) {
            const int row = c >> 3, x = row % (S::TR + S::TC), kg = row / (S::TR + S::TC);
            const int k = k0 + kg % KC;
            const int64_t f = f0 + (kg / KC) * 32 + (c & 7) * 4;
            const bool isa = x < S::TR;
            const int i = i0 + x, j = j0 + x - S::TR;
            const bool on = k < s && f < Lz && (isa ? i < r : j < t);
            const uint32_t *src = !on ? A : (isa ? A + ((size_t)i * s + k) * Lz + f : B + ((size_t)k * t + j) * Lz + f);
            cp_async16(sm + c * 4, src, on);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    unsigned long long acc[PW_RT][PW_CT];
#pragma unroll
    for (int u = 0; u < PW_RT; u++)
#pragma unroll
        for (int v = 0; v < PW_CT; v++) acc[u][v] = 0ull;
    load(0, 0);
    int since = 0;  // products since the last fold
    for (int k0 = 0, st = 0; k0 < s; k0 += KC, st ^= 1) {
        if (k0 + KC < s) {
            load(k0 + KC, st ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const uint32_t *sm = pw_sm + st * S::STAGE + fg * KC * (S::TR + S::TC) * 32 + lane;
        const uint32_t *sa = sm + PW_RT * wr * 32, *sb = sm + (S::TR + PW_CT * wc) * 32;
#pragma unroll
        for (int kk = 0; kk < KC; kk++) {
            uint32_t a[PW_RT], b[PW_CT];
#pragma unroll
            for (int u = 0; u < PW_RT; u++) a[u] = sa[(kk * (S::TR + S::TC) + u) * 32];
#pragma unroll
            for (int v = 0; v < PW_CT; v++) b[v] = sb[(kk * (S::TR + S::TC) + v) * 32];
#pragma unroll
            for (int u = 0; u < PW_RT; u++)
#pragma unroll
                for (int v = 0; v < PW_CT; v++) acc[u][v] = madw(a[u], b[v], acc[u][v]);
            if ((FOLDK < KC && (kk + 1) % FOLDK == 0) || (kk == KC - 1 && (since += KC) >= FOLDK)) {
                since = 0;
#pragma unroll
                for (int u = 0; u < PW_RT; u++)
#pragma unroll
                    for (int v = 0; v < PW_CT; v++) acc[u][v] = fold1(acc[u][v], fc);
            }
        }
        __syncthreads();
    }
    const int64_t f = f0 + fg * 32 + lane;
    if (f >= Lz) return;
#pragma unroll
    for (int u = 0; u < PW_RT; u++)
#pragma unroll
        for (int v = 0; v < PW_CT; v++) {
            const int i = i0 + PW_RT * wr + u, j = j0 + PW_CT * wc + v;
            // folded twice: below 2^57.2, so below P 2^32
            if (i < r && j < t)
                C[((size_t)i * t + j) * Lz + f] = mont_redc(fold1(fold1(acc[u][v], fc), fc), mP);
        }
}

struct CrtConst {
    uint32_t P1, P2, P3;
    uint32_t c12;        // P1^{-1} mod P2                    (these three in the
    uint32_t c123;       // (P1 P2)^{-1} mod P3                Montgomery form of
    uint32_t p1_mod_p3;  // P1 mod P3                          their modulus)
    uint32_t k1, k2, k3; // 1, P1, P1 P2 mod p (Montgomery form)
};

// Garner: the integer x < P1 P2 P3 with x = r_i mod P_i, reduced mod p.
// In: the three inverse transforms (Montgomery form, still times Lz), one
// run of Lz coefficients per entry; out: coefficient-major.  Tiles of 32
// coefficients x 32 entries: coalesced reads along the coefficients of an
// entry, Garner in registers, a shared-memory transpose, coalesced writes
// along the entries of a coefficient.
__global__ void __launch_bounds__(TR_TILE * TR_ROWS)
    k_ntt_crt(const uint32_t *__restrict__ R1, const uint32_t *__restrict__ R2, const uint32_t *__restrict__ R3,
              int nent, int64_t Lz, int64_t lo, int64_t hi, uint32_t *__restrict__ out, uint32_t il1, uint32_t il2,
              uint32_t il3, CrtConst cc, ModP m1, ModP m2, ModP m3, ModP mp) {
    __shared__ uint32_t tile[TR_TILE][TR_TILE + 1];
    const int tx = threadIdx.x & (TR_TILE - 1), ty = threadIdx.x / TR_TILE;
    const int64_t nk = hi - lo;
    const int64_t ktiles = (nk + TR_TILE - 1) / TR_TILE, etiles = (nent + TR_TILE - 1) / TR_TILE;
    for (int64_t tl = blockIdx.x; tl < ktiles * etiles; tl += gridDim.x) {
        const int64_t k0 = lo + (tl % ktiles) * TR_TILE;
        const int e0 = (int)(tl / ktiles) * TR_TILE;
        __syncthreads();
        for (int y = ty; y < TR_TILE; y += TR_ROWS) {
            const int e = e0 + y;
            const int64_t k = k0 + tx;
            uint32_t v = 0;
            if (e < nent && k < hi) {
                const size_t src = (size_t)e * Lz + (size_t)k;
                // mont_mul(v R, Lz^{-1}) = v Lz^{-1} in normal form
                const uint32_t r1 = mont_mul(R1[src], il1, m1);
                const uint32_t r2 = mont_mul(R2[src], il2, m2);
                const uint32_t r3 = mont_mul(R3[src], il3, m3);
                // r1 < P1 < 2.2 P2 and P1 < P3
                uint32_t q1 = r1 >= cc.P2 ? r1 - cc.P2 : r1;
                q1 = q1 >= cc.P2 ? q1 - cc.P2 : q1;
                const uint32_t t2 = mont_mul(subm(r2, q1, m2), cc.c12, m2);
                const uint32_t u = subm(subm(r3, r1, m3), mont_mul(t2, cc.p1_mod_p3, m3), m3);
                const uint32_t t3 = mont_mul(u, cc.c123, m3);
                // r1 + t2 P1 + t3 P1 P2 mod p: r1, t2 < 2^30 (their primes are), so
                // the first two products together stay below p 2^32
                v = addm(mont_redc((uint64_t)r1 * cc.k1 + (uint64_t)t2 * cc.k2, mp), mont_redc((uint64_t)t3 * cc.k3, mp),
                         mp);
            }
            tile[y][tx] = v;
        }
        __syncthreads();
        for (int y = ty; y < TR_TILE; y += TR_ROWS) {
            const int64_t k = k0 + y;
            const int e = e0 + tx;
            if (k < hi && e < nent) out[(size_t)(k - lo) * nent + e] = tile[tx][y];
        }
    }
}

// blocks of the tiled transposes: one per 32 x 32 tile, at most 16 per SM
// (grid-stride beyond)
inline unsigned tr_grid(int64_t nk, int64_t nent, int num_sms) {
    const int64_t tiles = ((nk + TR_TILE - 1) / TR_TILE) * ((nent + TR_TILE - 1) / TR_TILE);
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)num_sms * 16));
}

}  // namespace

// The context's twiddle tables, kept across products: for each transform
// prime, the powers w^bitrev(i) and w^-bitrev(i) (i < 2^(LG-1)) of a 2^LG-th
// root of unity, LG >= lg (entry i is the same for every LG); built on the
// device when a longer transform than the tables serve is first needed.
static wr_status ensure_twiddles(wr_ctx *ctx, int lg) {
    if (ctx->ntt_lg >= lg) return WR_OK;
    const int LG = std::max(lg, 14);
    const int64_t half = (int64_t)1 << (LG - 1);
    ctx->ntt_lg = 0;  // (the old table goes back first: none is there until this one is whole)
    WR_TRY(dev_alloc(ctx, ctx->ntt_tw, sizeof(uint32_t) * (size_t)(2 * NTT_NPRIMES) * half));
    for (int i = 0; i < NTT_NPRIMES; i++) {
        const uint32_t P = NTT_PRIMES[i];
        const ModP mP = make_modp(P);
        const uint64_t g = primitive_root(P);
        const uint64_t w = hpow(g, (P - 1) >> LG, P), wi = hpow(w, P - 2, P);
        const uint32_t wm = (uint32_t)(((unsigned __int128)w << 32) % P), wim = (uint32_t)(((unsigned __int128)wi << 32) % P);
        uint32_t *tw = ctx->ntt_tw.as<uint32_t>() + (size_t)(2 * i) * half;
        const unsigned g2 = (unsigned)std::min<int64_t>((half + 255) / 256, (int64_t)ctx->num_sms * 16);
        k_twiddles<<<g2, 256, 0, ctx->stream>>>(wm, LG - 1, tw, mP);
        WR_LAUNCHED(ctx);
        k_twiddles<<<g2, 256, 0, ctx->stream>>>(wim, LG - 1, tw + half, mP);
        WR_LAUNCHED(ctx);
    }
    ctx->ntt_lg = LG;
    return WR_OK;
}

// All stages of npoly transforms of 2^lg points, in place: the stages above
// the tile's in passes of up to four, and the tile pass.
template <bool FWD>
static wr_status ntt_run(wr_ctx *ctx, uint32_t *a, int64_t npoly, int lg, const uint32_t *tw, const ModP &mP) {
    cudaStream_t st = ctx->stream;
    const int lc = std::min(lg, NTT_TILE_LOG), rem = lg - lc;
    auto top = [&](int s0, int K) -> wr_status {
        const int64_t groups = npoly << (lg - K);
        const unsigned grid = (unsigned)std::min<int64_t>((groups + NTT_TOP_THREADS - 1) / NTT_TOP_THREADS,
                                                          (int64_t)ctx->num_sms * 64);
        auto *k = K == 4 ? k_ntt_top<4, FWD> : (K == 3 ? k_ntt_top<3, FWD> : (K == 2 ? k_ntt_top<2, FWD> : k_ntt_top<1, FWD>));
        k<<<grid, NTT_TOP_THREADS, 0, st>>>(a, npoly, lg, s0, tw, mP.p, mP.pneg);
        WR_LAUNCHED(ctx);
        return WR_OK;
    };
    auto tiles = [&]() -> wr_status {
        const int64_t words = npoly << lg;
        auto *k = words < (1 << NTT_TILE_LOG) ? k_ntt_tile<FWD, true> : k_ntt_tile<FWD, false>;
        k<<<(unsigned)((words + (1 << NTT_TILE_LOG) - 1) >> NTT_TILE_LOG), NTT_TILE_THREADS, 0, st>>>(
            a, words, lg, lc, tw, mP.p, mP.pneg);
        WR_LAUNCHED(ctx);
        return WR_OK;
    };
    if (!FWD) WR_TRY(tiles());
    for (int k = 0; k < (rem + 3) / 4; k++) {
        const int s0 = FWD ? 4 * k : 4 * ((rem + 3) / 4 - 1 - k);
        WR_TRY(top(s0, std::min(4, rem - s0)));
    }
    if (FWD) WR_TRY(tiles());
    return WR_OK;
}

template <int WR, int WC, int KC>
static wr_status pointwise_run(wr_ctx *ctx, const uint32_t *A, const uint32_t *B, uint32_t *C, int r, int s, int t,
                               int64_t Lz, const ModP &mP) {
    using S = PwShape<WR, WC, KC>;
    auto *k = mP.p < (1u << 30) ? k_ntt_pointwise<WR, WC, KC, PW_FOLD_SMALL> : k_ntt_pointwise<WR, WC, KC, PW_FOLD_BIG>;
    WR_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM));
    const int64_t tiles = (int64_t)((r + S::TR - 1) / S::TR) * ((t + S::TC - 1) / S::TC);
    const dim3 g((unsigned)((Lz + 32 * S::FG - 1) / (32 * S::FG)), (unsigned)tiles);
    k<<<g, 32 * PW_WARPS, S::SMEM, ctx->stream>>>(A, B, C, r, s, t, Lz, mP);
    WR_LAUNCHED(ctx);
    return WR_OK;
}

// C[k - lo] = sum_j A_j B_{k-j} (mod p) for lo <= k < hi; A: na coefficients of
// r x s, B: nb coefficients of s x t, C: (hi - lo) x r x t.  All device
// pointers, coefficient-major.
static wr_status polymat_mul_run(wr_ctx *ctx, const uint32_t *A, int64_t na, const uint32_t *B, int64_t nb, int r,
                                 int s, int t, int64_t lo, int64_t hi, uint32_t p, uint32_t *C);

wr_status polymat_mul(wr_ctx *ctx, const uint32_t *A, int64_t na, const uint32_t *B, int64_t nb, int r, int s,
                      int t, int64_t lo, int64_t hi, uint32_t p, uint32_t *C) {
    if (!ctx->profiling) return polymat_mul_run(ctx, A, na, B, nb, r, s, t, lo, hi, p, C);
    // profiling: the product's device time, summed over the sigma-basis
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    WR_CUDA(cudaEventCreate(&e0));
    WR_CUDA(cudaEventCreate(&e1));
    WR_CUDA(cudaEventRecord(e0, ctx->stream));
    const wr_status st = polymat_mul_run(ctx, A, na, B, nb, r, s, t, lo, hi, p, C);
    cudaEventRecord(e1, ctx->stream);
    cudaEventSynchronize(e1);
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    ctx->last.sigma_product_ms += ms;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

static wr_status polymat_mul_run(wr_ctx *ctx, const uint32_t *A, int64_t na, const uint32_t *B, int64_t nb, int r,
                                 int s, int t, int64_t lo, int64_t hi, uint32_t p, uint32_t *C) {
    if (hi <= lo) return WR_OK;
    cudaStream_t st = ctx->stream;
    if (na <= 0 || nb <= 0) {
        WR_CUDA(cudaMemsetAsync(C, 0, sizeof(uint32_t) * (size_t)(hi - lo) * r * t, st));
        return WR_OK;
    }
    // the exact coefficients, at most s min(na, nb) (p - 1)^2, must lie below
    // the product of the transform primes for the remainder step to recover them
    const double bound = (double)s * (double)std::min(na, nb) * (double)(p - 1) * (double)(p - 1);
    if (bound >= 0.999 * (double)NTT_PRIMES[0] * (double)NTT_PRIMES[1] * (double)NTT_PRIMES[2])
        return fail(WR_EINVAL, "polynomial product coefficients exceed the transform primes' product");
    const int64_t full = na + nb - 1;  // coefficients of the exact product
    const int64_t need = std::max<int64_t>(hi, full - lo);
    int lg = 5;  // rows of at least 32 points for the pointwise products
    while (((int64_t)1 << lg) < need) lg++;
    if (lg > NTT_MAX_LOG) return fail(WR_EINVAL, "polynomial product too long for the transform primes");
    const int64_t Lz = (int64_t)1 << lg;
    const int nA = r * s, nB = s * t, nC = r * t;
    const ModP mp = make_modp(p);
    DevBuf bufA, bufB, bufC[NTT_NPRIMES];
    WR_TRY(dev_alloc(ctx, bufA, sizeof(uint32_t) * (size_t)nA * Lz));
    WR_TRY(dev_alloc(ctx, bufB, sizeof(uint32_t) * (size_t)nB * Lz));
    for (int i = 0; i < NTT_NPRIMES; i++) WR_TRY(dev_alloc(ctx, bufC[i], sizeof(uint32_t) * (size_t)nC * Lz));
    WR_TRY(ensure_twiddles(ctx, lg));
    const int LG = ctx->ntt_lg;
    uint32_t il[NTT_NPRIMES];
    ModP mP[NTT_NPRIMES];
    for (int i = 0; i < NTT_NPRIMES; i++) {
        const uint32_t P = NTT_PRIMES[i];
        mP[i] = make_modp(P);
        const uint32_t *tw = ctx->ntt_tw.as<uint32_t>() + (size_t)(2 * i) * ((size_t)1 << (LG - 1));
        const uint32_t *twi = tw + ((size_t)1 << (LG - 1));
        il[i] = (uint32_t)hpow((uint64_t)(Lz % P), P - 2, P);  // Lz^{-1} mod P (normal form)
        k_ntt_load<<<tr_grid(Lz, nA, ctx->num_sms), TR_TILE * TR_ROWS, 0, st>>>(A, na, nA, Lz, bufA.as<uint32_t>(), mP[i]);
        WR_LAUNCHED(ctx);
        k_ntt_load<<<tr_grid(Lz, nB, ctx->num_sms), TR_TILE * TR_ROWS, 0, st>>>(B, nb, nB, Lz, bufB.as<uint32_t>(), mP[i]);
        WR_LAUNCHED(ctx);
        WR_TRY(ntt_run<true>(ctx, bufA.as<uint32_t>(), nA, lg, tw, mP[i]));
        WR_TRY(ntt_run<true>(ctx, bufB.as<uint32_t>(), nB, lg, tw, mP[i]));
        // the tile of C that a block covers: 16 x 16, or less where C is smaller
        // (the block then takes more groups of points)
        // (few entries of C and a long sum: four k a stage, 1 x 64 x 1, 1,000 coefficients
        // 253 -> 241 us; two for up to 8, 2 x 5 x 7, 30,000 coefficients 264 and 271)
        uint32_t *pA = bufA.as<uint32_t>(), *pB = bufB.as<uint32_t>(), *pC = bufC[i].as<uint32_t>();
        if (r <= 4 && t <= 8 && s <= 8) WR_TRY((pointwise_run<1, 1, 2>(ctx, pA, pB, pC, r, s, t, Lz, mP[i])));
        else if (r <= 4 && t <= 8) WR_TRY((pointwise_run<1, 1, 4>(ctx, pA, pB, pC, r, s, t, Lz, mP[i])));
        else if (t <= 8) WR_TRY((pointwise_run<2, 1, 4>(ctx, pA, pB, pC, r, s, t, Lz, mP[i])));
        else if (r <= 8) WR_TRY((pointwise_run<2, 2, 4>(ctx, pA, pB, pC, r, s, t, Lz, mP[i])));
        else WR_TRY((pointwise_run<4, 2, 8>(ctx, pA, pB, pC, r, s, t, Lz, mP[i])));
        WR_TRY(ntt_run<false>(ctx, pC, nC, lg, twi, mP[i]));
    }
    CrtConst cc;
    cc.P1 = NTT_PRIMES[0];
    cc.P2 = NTT_PRIMES[1];
    cc.P3 = NTT_PRIMES[2];
    auto mont = [](uint64_t x, uint32_t m) { return (uint32_t)(((x % m) << 32) % m); };
    cc.c12 = mont(hpow(cc.P1 % cc.P2, cc.P2 - 2, cc.P2), cc.P2);
    cc.c123 = mont(hpow((uint64_t)cc.P1 * cc.P2 % cc.P3, cc.P3 - 2, cc.P3), cc.P3);
    cc.p1_mod_p3 = mont(cc.P1, cc.P3);
    cc.k1 = mont(1, p);
    cc.k2 = mont(cc.P1, p);
    cc.k3 = mont((uint64_t)cc.P1 * cc.P2, p);
    k_ntt_crt<<<tr_grid(hi - lo, nC, ctx->num_sms), TR_TILE * TR_ROWS, 0, st>>>(
        bufC[0].as<uint32_t>(), bufC[1].as<uint32_t>(), bufC[2].as<uint32_t>(), nC, Lz, lo, hi, C, il[0], il[1],
        il[2], cc, mP[0], mP[1], mP[2], mp);
    WR_LAUNCHED(ctx);
    return WR_OK;
}

}  // namespace wr
