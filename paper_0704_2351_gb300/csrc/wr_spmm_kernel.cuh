// The SpMM pass kernel of the black box (Section 2.5 step 2: the sparse
// products A T and A^T W mod p) and its helpers: SELL-C-sigma light chunks
// and warp-per-segment long rows, exact int64 row sums, the diagonal scaling
// and Montgomery reduction as the epilogue, split rows finished by
// k_finalize_split.  Included by wr_spmm.cu only (its launchers and the
// sequence loop live there).
#pragma once

#include <cuda_runtime.h>

#include "wr_internal.cuh"

namespace wr {
namespace {

// W residues per lane, G lanes per gathered row: one warp-wide gather then
// touches 32/G rows, each one contiguous 4*NV-byte run, so the L1 handles one
// tag lookup per row instead of one per lane.
template <int NV, int WW>
struct Lanes {
    static constexpr int W = WW;       // residues per lane
    static constexpr int G = NV / W;   // lanes per row
    static constexpr int RPW = 32 / G; // rows (light) or entries (vector) per warp step
    static_assert(NV % W == 0 && G >= 1 && G <= 32, "lane width must divide the block width");
};
// default residues per lane for a block width (used when nothing is tuned):
// 16 bytes, the fastest on every matrix measured for rows of 32 bytes and more
// (above); 8 for rows of 16
inline int default_lane_width(int nv) { return nv <= 4 ? (nv < 2 ? nv : 2) : 4; }

template <int W>
__device__ __forceinline__ void ldv(const uint32_t *p, uint32_t (&v)[W]) {
    if constexpr (W == 1) {
        v[0] = __ldg(p);
    } else if constexpr (W == 2) {
        uint2 t = __ldg(reinterpret_cast<const uint2 *>(p));
        v[0] = t.x; v[1] = t.y;
    } else {
#pragma unroll
        for (int k = 0; k < W / 4; k++) {
            uint4 t = __ldg(reinterpret_cast<const uint4 *>(p) + k);
            v[4 * k] = t.x; v[4 * k + 1] = t.y; v[4 * k + 2] = t.z; v[4 * k + 3] = t.w;
        }
    }
}

template <int W>
__device__ __forceinline__ void stv(uint32_t *p, const uint32_t (&v)[W]) {
    if constexpr (W == 1) {
        p[0] = v[0];
    } else if constexpr (W == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(v[0], v[1]);
    } else {
#pragma unroll
        for (int k = 0; k < W / 4; k++)
            reinterpret_cast<uint4 *>(p)[k] = make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    }
}

// W residues from memory this kernel also writes (the partial output of the
// previous column slab): plain loads
template <int W>
__device__ __forceinline__ void ldv_rw(const uint32_t *p, uint32_t (&v)[W]) {
    if constexpr (W == 1) {
        v[0] = p[0];
    } else if constexpr (W == 2) {
        const uint2 t = *reinterpret_cast<const uint2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
#pragma unroll
        for (int k = 0; k < W / 4; k++) {
            const uint4 t = reinterpret_cast<const uint4 *>(p)[k];
            v[4 * k] = t.x; v[4 * k + 1] = t.y; v[4 * k + 2] = t.z; v[4 * k + 3] = t.w;
        }
    }
}

// Loads of the matrix's entry words and stores of the output rows, with or
// without the streaming cache hint (CS: evict-first in L1 and L2, ld/st.cs):
// each entry and each output row is touched once per pass, so with the hint
// they stop pushing rows of the gathered block out of L2.  The autotuner
// times both forms per matrix.
template <bool CS>
__device__ __forceinline__ uint32_t lde(const uint32_t *p) {
    if constexpr (CS) return __ldcs(p);
    else return __ldg(p);
}

template <int W, bool CS>
__device__ __forceinline__ void stv_out(uint32_t *p, const uint32_t (&v)[W]) {
    if constexpr (!CS) {
        stv<W>(p, v);
    } else if constexpr (W == 1) {
        __stcs(p, v[0]);
    } else if constexpr (W == 2) {
        __stcs(reinterpret_cast<uint2 *>(p), make_uint2(v[0], v[1]));
    } else {
#pragma unroll
        for (int k = 0; k < W / 4; k++)
            __stcs(reinterpret_cast<uint4 *>(p) + k, make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]));
    }
}

// Entry words: (column << 8) | (uint8)value in the packed layout, the column
// alone in the wide one (values from the int16 array beside the entries).
template <int W>
__device__ __forceinline__ void mac(int64_t (&acc)[W], int a, const uint32_t (&v)[W]) {
#pragma unroll
    for (int w = 0; w < W; w++) acc[w] += (int64_t)a * (int32_t)v[w];
}

// The gathers of a batch: volatile loads keep their program order, so a batch
// of U gathers is in flight before its first product (left to itself the
// compiler interleaves loads and products to stay at 32 registers, with two or
// three gathers in flight).  Plain loads, not the non-coherent ones: under a
// dependent launch (launch_dep) this kernel is resident while the one before it
// still writes the block, and ld.global.nc is defined only for memory that nobody
// writes during the kernel.
template <int W>
__device__ __forceinline__ void gather(const uint32_t *p, uint32_t (&v)[W]) {
    if constexpr (W == 1) {
        asm volatile("ld.global.u32 %0, [%1];" : "=r"(v[0]) : "l"(p));
    } else if constexpr (W == 2) {
        asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "l"(p));
    } else {
#pragma unroll
        for (int k = 0; k < W / 4; k++)
            asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v[4 * k]), "=r"(v[4 * k + 1]), "=r"(v[4 * k + 2]), "=r"(v[4 * k + 3])
                         : "l"(p + 4 * k));
    }
}

// Epilogue of a finished row: y[row] = scale[row] * (sum mod p), or, for a
// row cut into segments, the exact partial sums added into acc64.
// A direct row has at most VSEG = 256 entries of magnitude below 2^15, so
// |sum| < 2^23 p and T = sum + 2^23 p lies in [0, 2^24 p), below p R: one
// Montgomery reduction gives T R^{-1}; with the scale taken to scale R^2 mod p
// (two Montgomery products), mont_mul(T R^{-1}, scale R^2) = sum * scale mod p.
// the modulus and scale of the job owning columns col0.. of a multi-job block
__device__ __forceinline__ void job_of(const MultiEpi &me, int col0, ModP &mp, const uint32_t *&scale) {
    switch (col0 >> me.jw_log) {
        case 0: mp = me.mp[0]; scale = me.scale[0]; break;
        case 1: mp = me.mp[1]; scale = me.scale[1]; break;
        case 2: mp = me.mp[2]; scale = me.scale[2]; break;
        default: mp = me.mp[3]; scale = me.scale[3]; break;
    }
}

// The scale residue of output row tgt (0 for a split or absent row), loaded
// ahead of the row's gathers (a plain load, as the gathers).
template <bool MULTI>
__device__ __forceinline__ uint32_t row_scale(uint32_t tgt, const uint32_t *scale, const MultiEpi &me, int col0) {
    if (tgt & VROW_SPLIT) return 0u;  // (VROW_EMPTY has the bit set)
    if constexpr (MULTI) {
        ModP mp;
        job_of(me, col0, mp, scale);
    }
    return ld_plain(scale + tgt);
}

// part: 0 the whole pass (y = scale (A x)); with column slabs of the matrix
// (passes split by ranges of the gathered rows, so that the rows of x that a
// slab gathers stay in L2) 1 the first slab (y = its sum mod p), 2 a middle
// one (y += its sum), 3 the last (y = scale (y + its sum)); y holds residues
// in between.  sc: row_scale of the row.
template <int W, bool CS, bool MULTI>
__device__ __forceinline__ void row_out(uint32_t tgt, const int64_t (&acc)[W], uint32_t *y, uint32_t sc,
                                        unsigned long long *acc64, int nv, int col0, const ModP &mp_one,
                                        const MultiEpi &me, int part) {
    if (tgt & VROW_SPLIT) {
        unsigned long long *dst = acc64 + (size_t)(tgt & ~VROW_SPLIT) * nv + col0;
#pragma unroll
        for (int w = 0; w < W; w++) atomicAdd(dst + w, (unsigned long long)acc[w]);
    } else {
        ModP mp = mp_one;
        if constexpr (MULTI) {
            const uint32_t *s;
            job_of(me, col0, mp, s);
        }
        const uint64_t off = (uint64_t)mp.p << 23;
        uint32_t o[W];
        uint32_t *yr = y + (size_t)tgt * nv + col0;
        if (part == 0) {
            const uint32_t s2 = to_mont(to_mont(sc, mp), mp);
#pragma unroll
            for (int w = 0; w < W; w++) o[w] = mont_mul(mont_redc((uint64_t)acc[w] + off, mp), s2, mp);
        } else {
            // mont_mul(T R^{-1}, R^2) = T mod p
#pragma unroll
            for (int w = 0; w < W; w++) o[w] = mont_mul(mont_redc((uint64_t)acc[w] + off, mp), mp.r2, mp);
            if (part >= 2) {
                uint32_t prev[W];
                ldv_rw<W>(yr, prev);
#pragma unroll
                for (int w = 0; w < W; w++) o[w] = addm(o[w], prev[w], mp);
            }
            if (part == 3) {
                const uint32_t s1 = to_mont(sc, mp);
#pragma unroll
                for (int w = 0; w < W; w++) o[w] = mont_mul(o[w], s1, mp);
            }
        }
        stv_out<W, CS>(yr, o);
    }
}

// Work of one lane layout: G lanes a row, U gathers in flight per lane, the
// row's entry words in tiles of E.  Rows of up to four lanes hold a tile in
// each lane (LG = 1: a warp's eight or more rows read whole sectors of the
// slot-major entries); wider rows share a tile out, one word a lane, and pass
// the words round by shuffles (LG = G).
//
// What bounds a pass is how many gathers the SM has in flight, so a batch's
// loads are issued together (gather) and the registers are spent on them:
// 64 a thread for 16-byte lanes (32 resident warps x 8 gathers of 16 bytes a
// lane), 51 for narrower ones.  Measured per pass on GB300, against one loop
// that the compiler kept at 32 registers with two or three gathers in flight:
// 1.9M x 1.95M, 40.7M entries, rows of 32 residues from a 250 MB block 740 ->
// 608 us on two GPUs, 586 on a third (3.47 GB of DRAM traffic at 5.6-6.1 TB/s,
// 83-89 % of the copy rate);
// 500,000 x 450,000, rows of 32 from 58 MB 97 -> 79 us; 200,000 x 180,000
// power-law, rows of 16 22.9 and 27.2 -> 21.6 and 26.7 us, rows of 8 18.5 and
// 20.2 -> 17.0 and 20.0 us.  72 registers (7 blocks) and 56 with spills (9 and
// 10 blocks) were slower (500,000: 93 us).
constexpr int SPMM_WARPS = 4;  // warps per block
template <int NV, int WL>
struct Tile {
    static constexpr int G = Lanes<NV, WL>::G;
    static constexpr int LG = G <= 4 ? 1 : G;  // lanes that share out a tile's words
    static constexpr int TE = LG == 1 ? 8 : 1; // words a lane holds
    static constexpr int E = TE * LG;          // entries of a row per tile
    static constexpr int U = WL == 8 ? 4 : 8;  // gathers in flight per lane
    // blocks an SM (6 in the wide layout with LG = 1, whose values take 16 more registers)
    static constexpr int MINB = WL == 8 ? 6 : (WL == 4 ? 8 : 10);
    static_assert(E % U == 0, "whole batches per tile");
};

// The block row of an entry word (part: the lane's byte offset in the row).
// Packed columns are below 2^24 and rows at most 256 bytes, so the offset fits
// 32 bits; the wide layout takes 64.
template <int NV, bool WIDE>
__device__ __forceinline__ const uint32_t *row_at(const uint32_t *x, uint32_t e, uint32_t part) {
    const size_t off = WIDE ? (size_t)e * (NV * 4) + part : (size_t)(uint32_t)((e >> 8) * (NV * 4) + part);
    return reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(x) + off);
}

// B gathers (entries j0 .. j0 + B - 1 of the tile) and their products.  Entry
// words past the row's end are 0 (column 0, value 0): their gathers add nothing
// and hit L1, which costs less than predicating every load.  The entry's value
// is shuffled again for its product instead of being held across the gathers
// (eight registers).
template <int NV, int WL, bool WIDE, int B>
__device__ __forceinline__ void batch(const uint32_t *x, uint32_t part, const uint32_t (&ee)[Tile<NV, WL>::TE],
                                      const int32_t (&wv)[Tile<NV, WL>::TE], int j0, int64_t (&acc)[WL]) {
    constexpr int G = Tile<NV, WL>::LG, W = WL;
    uint32_t v[B][W];
#pragma unroll
    for (int u = 0; u < B; u++) {
        const int j = j0 + u;  // a constant after unrolling
        const uint32_t e = G == 1 ? ee[j / G] : __shfl_sync(0xffffffffu, ee[j / G], j % G, G);
        gather<W>(row_at<NV, WIDE>(x, e, part), v[u]);
    }
#pragma unroll
    for (int u = 0; u < B; u++) {
        const int j = j0 + u;
        int a;
        if constexpr (WIDE) a = G == 1 ? wv[j / G] : __shfl_sync(0xffffffffu, wv[j / G], j % G, G);
        else a = (int)(int8_t)((G == 1 ? ee[j / G] : __shfl_sync(0xffffffffu, ee[j / G], j % G, G)) & 0xFFu);
        mac<W>(acc, a, v[u]);
    }
}

// The products of one tile (its first cnt entries): whole batches of U, the
// rest rounded up to 2, 4 or U gathers.
template <int NV, int WL, bool WIDE>
__device__ __forceinline__ void tile_products(const uint32_t *x, uint32_t part, const uint32_t (&ee)[Tile<NV, WL>::TE],
                                              const int32_t (&wv)[Tile<NV, WL>::TE], int cnt, int64_t (&acc)[WL]) {
    using Tl = Tile<NV, WL>;
#pragma unroll
    for (int j0 = 0; j0 < Tl::E; j0 += Tl::U) {
        const int left = cnt - j0;  // the same for the warp
        if (left > 4 || (Tl::U == 4 && left > 2)) batch<NV, WL, WIDE, Tl::U>(x, part, ee, wv, j0, acc);
        else if (Tl::U == 8 && left > 2) batch<NV, WL, WIDE, 4>(x, part, ee, wv, j0, acc);
        else if (left > 0) batch<NV, WL, WIDE, 2>(x, part, ee, wv, j0, acc);
    }
}

// One SpMM pass, y = scale * (A x) mod p, exact int64 row sums.
// Blocks [0, vblocks): one warp per segment of a long row; its lanes load the
// segment's (contiguous) entries 32 at a time and gather RPW rows per step,
// then a shuffle reduction.
// Blocks [vblocks, ...): G warps per SELL chunk of 32 light rows; warp q of
// the chunk takes rows [q*RPW, (q+1)*RPW), G lanes per row; a block takes
// `pieces` consecutive groups of SPMM_WARPS such warps' work, and each warp
// loads the first tile of its next piece before it gathers for the current
// one, so that a piece costs its gathers' latency alone.
template <int NV, int WL, bool WIDE, bool CS, bool MULTI>
__global__ void __launch_bounds__(32 * SPMM_WARPS, WIDE && Tile<NV, WL>::LG == 1 ? 6 : Tile<NV, WL>::MINB)
    k_spmm(SellView A, const uint32_t *__restrict__ x, uint32_t *__restrict__ y, const uint32_t *__restrict__ scale,
           unsigned long long *__restrict__ acc64, ModP mp, int *__restrict__ term_counter, int64_t vblocks,
           int pieces, MultiEpi me, int part) {
    using Ln = Lanes<NV, WL>;
    using Tl = Tile<NV, WL>;
    constexpr int W = Ln::W, G = Ln::G, RPW = Ln::RPW, TE = Tl::TE, E = Tl::E, U = Tl::U;
    pdl_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane / G, lanepart = lane % G;
    // the pass before this one (its output is x) is done from here on; the first
    // entries are loaded before
    auto begin = [&]() {
        pdl_wait();
        if (term_counter && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(term_counter, 1);
    };
    const uint32_t xpart = lanepart * W * 4;
    int64_t acc[W];
#pragma unroll
    for (int w = 0; w < W; w++) acc[w] = 0;
    if ((int64_t)blockIdx.x < vblocks) {
        const int64_t seg = (int64_t)blockIdx.x * SPMM_WARPS + warp;
        if (seg >= A.nseg) return;  // (thread 0 of block 0 has a segment)
        const uint32_t *e = A.ventries + A.seg_start[seg];
        const int16_t *ev = WIDE ? A.vwvals + A.seg_start[seg] : nullptr;
        const int len = A.seg_len[seg];
        const uint32_t tgt = A.seg_row[seg];
        // 32 NR entries in NR registers across the warp, the next ones
        // prefetched; entry i * RPW + sub of a register is gathered by row group
        // sub in step i (words past the end are 0: column 0, value 0).  NR = 2
        // where one register is at most U / 2 steps
        constexpr int UB = G < U ? G : U;         // steps per batch of one register
        constexpr int NR = 2 * G <= U ? 2 : 1;
        uint32_t cur[NR];
        int32_t cwv[NR];
#pragma unroll
        for (int h = 0; h < NR; h++) {
            const int jh = 32 * h + lane;
            cur[h] = jh < len ? lde<CS>(e + jh) : 0u;
            cwv[h] = WIDE && jh < len ? (int32_t)__ldg(ev + jh) : 0;
        }
        begin();
        for (int j = 0; j < len; j += 32 * NR) {
            uint32_t nxt[NR];
            int32_t nwv[NR];
#pragma unroll
            for (int h = 0; h < NR; h++) {
                const int jn = j + 32 * (NR + h) + lane;
                nxt[h] = jn < len ? lde<CS>(e + jn) : 0u;
                nwv[h] = WIDE && jn < len ? (int32_t)__ldg(ev + jn) : 0;
            }
#pragma unroll
            for (int i0 = 0; i0 < G; i0 += UB) {
                if (j + i0 * RPW >= len) break;
                uint32_t v[NR * UB][W];
#pragma unroll
                for (int u = 0; u < NR * UB; u++) {
                    const int h = u / UB, src = (i0 + u % UB) * RPW + sub;
                    gather<W>(row_at<NV, WIDE>(x, __shfl_sync(0xffffffffu, cur[h], src), xpart), v[u]);
                }
#pragma unroll
                for (int u = 0; u < NR * UB; u++) {
                    const int h = u / UB, src = (i0 + u % UB) * RPW + sub;
                    int a;
                    if constexpr (WIDE) a = __shfl_sync(0xffffffffu, cwv[h], src);
                    else a = (int)(int8_t)(__shfl_sync(0xffffffffu, cur[h], src) & 0xFFu);
                    mac<W>(acc, a, v[u]);
                }
            }
#pragma unroll
            for (int h = 0; h < NR; h++) {
                cur[h] = nxt[h];
                cwv[h] = nwv[h];
            }
        }
#pragma unroll
        for (int off = G; off < 32; off <<= 1)
#pragma unroll
            for (int w = 0; w < W; w++) acc[w] += __shfl_xor_sync(0xffffffffu, acc[w], off);
        if (sub == 0)
            row_out<W, CS, MULTI>(tgt, acc, y, row_scale<MULTI>(tgt, scale, me, lanepart * W), acc64, NV, lanepart * W,
                                  mp, me, part);
        return;
    }
    // (fewer than 2^31 rows: chunk * G + q fits 32 bits)
    const uint32_t nlw = (uint32_t)A.nchunks * G;
    uint32_t lw = (blockIdx.x - (uint32_t)vblocks) * pieces * SPMM_WARPS + warp;
    if (lw >= nlw) {
        if (blockIdx.x == 0) begin();  // (a launch for the counter alone)
        return;
    }
    uint32_t ee[TE];
    int32_t wv[TE];
    // entries [j0, j0 + E) of this lane's row in a chunk of `len` slots at word `at`
    auto load_tile = [&](int64_t at, int j0, int len, uint32_t (&q)[TE], int32_t (&qw)[TE]) {
#pragma unroll
        for (int k = 0; k < TE; k++) {
            const int j = j0 + (Tl::LG == 1 ? k : k * G + lanepart);
            q[k] = j < len ? lde<CS>(A.entries + at + j * SELL_C) : 0u;
            if constexpr (WIDE) qw[k] = j < len ? (int32_t)__ldg(A.wvals + at + j * SELL_C) : 0;
            else qw[k] = 0;
        }
    };
    int len = __ldg(A.chunk_len + lw / G);
    int64_t at = __ldg(A.chunk_off + lw / G) + (lw % G) * RPW + sub;
    load_tile(at, 0, len, ee, wv);
    begin();
    for (int k = pieces;;) {
        const uint32_t vr = __ldg(A.vrow + lw * RPW + sub);  // chunk * 32 + q * RPW + sub
        lw += SPMM_WARPS;
        int len2 = -1;
        int64_t at2 = 0;
        if (--k > 0 && lw < nlw) {
            len2 = __ldg(A.chunk_len + lw / G);
            at2 = __ldg(A.chunk_off + lw / G) + (lw % G) * RPW + sub;
        }
        uint32_t e2[TE];
        int32_t w2[TE];
        int j0 = 0;
        for (; j0 + E < len; j0 += E) {
            load_tile(at, j0 + E, len, e2, w2);
            tile_products<NV, WL, WIDE>(x, xpart, ee, wv, E, acc);
#pragma unroll
            for (int t = 0; t < TE; t++) {
                ee[t] = e2[t];
                wv[t] = w2[t];
            }
        }
        // the last tile, with the next piece's first one and the row's scale in flight
        load_tile(at2, 0, len2, e2, w2);
        const uint32_t sc = row_scale<MULTI>(vr, scale, me, lanepart * W);
        tile_products<NV, WL, WIDE>(x, xpart, ee, wv, len - j0, acc);
        if (vr != VROW_EMPTY) row_out<W, CS, MULTI>(vr, acc, y, sc, acc64, NV, lanepart * W, mp, me, part);
        if (len2 < 0) return;
#pragma unroll
        for (int t = 0; t < TE; t++) {
            ee[t] = e2[t];
            wv[t] = w2[t];
        }
#pragma unroll
        for (int w = 0; w < W; w++) acc[w] = 0;
        len = len2;
        at = at2;
    }
}

// Rows that were cut into segments: their exact int64 sums were added into
// acc64; reduce, scale, store, and clear the accumulator for the next pass.
// (part: as in row_out)
__global__ void k_finalize_split(int64_t nsplit, int nv, const int32_t *__restrict__ split_row,
                                 unsigned long long *__restrict__ acc64, uint32_t *__restrict__ y,
                                 const uint32_t *__restrict__ scale, ModP mp, int part) {
    pdl_launch();
    pdl_wait();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nsplit * nv) return;
    int64_t sid = i / nv;
    int b = (int)(i % nv);
    int32_t r = split_row[sid];
    unsigned long long s = acc64[i];
    acc64[i] = 0;
    uint32_t *yr = y + (size_t)r * nv + b;
    uint32_t v = red_s64((int64_t)s, mp);
    if (part >= 2) v = addm(v, *yr, mp);
    if (part == 0 || part == 3) v = mulm(ld_plain(scale + r), v, mp);
    *yr = v;
}

// the same for a multi-job block: column b is reduced with its job's modulus and scale
__global__ void k_finalize_split_multi(int64_t nsplit, int nv, const int32_t *__restrict__ split_row,
                                       unsigned long long *__restrict__ acc64, uint32_t *__restrict__ y, MultiEpi me) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nsplit * nv) return;
    int64_t sid = i / nv;
    int b = (int)(i % nv);
    int32_t r = split_row[sid];
    unsigned long long s = acc64[i];
    acc64[i] = 0;
    ModP mp;
    const uint32_t *scale;
    job_of(me, b, mp, scale);
    y[(size_t)r * nv + b] = mulm(scale[r], red_s64((int64_t)s, mp), mp);
}

}  // namespace
}  // namespace wr
