// Decode kernels: Y[b][n] = sum_k X[b][k] * table[code(n, k)] for batches up to 32
// (paper Sec. 3.3: dequantisation by lookup table instead of exponentiation).
//
//  * Pair table in shared memory.  Two codes (one byte at 4 bits, one 6-bit
//    field at 3 bits) index a table whose entry is the bf16x2 / f16x2 pair of
//    their dequantised values, signs included; at 8 bits one code per entry.
//    Each entry occupies a 256-byte row holding one copy per lane, so lane l
//    always reads bank l: the lookups of a warp never conflict.  The table starts
//    the dynamic shared memory at the fixed shared address kTabOff, so the byte
//    offset of an entry, byte << 8 | 4 * lane, is one byte permute (prmt) of the
//    code word and the table base is the load's immediate offset.
//  * Multiply-adds on the warp-level tensor-core instruction mma.sync m16n8k16:
//    the looked-up pairs are its A fragments as they are (16 rows, k permuted
//    alike in both operands), and B has 8 columns.  A batch of 1 needs one, so
//    the others hold further segments of k: S segments x 8 / S batch rows, the 16
//    MMA rows being 16 / S weight rows x S segments, of which the products on
//    the matching columns are used.  This is not for the arithmetic rate
//    (tcgen05 has far more, for operands in shared or tensor memory, which the
//    lookups would have to be stored to first) but for the instruction count:
//    one MMA takes the place of 8 fused multiply-adds per lane and of most of the
//    cross-lane reduction, and batches up to 8 cost hardly more than 1.
//  * Each warp owns a span of K and keeps its activations for it in registers;
//    it walks the rows of the CTA's row range, T tiles of code loads in flight,
//    each tile's registers refilled as soon as it is decoded.
//  * fp32 accumulation: single MMAs up to batch 8 (chains of 2 above), their
//    sums and everything after them added with rounding to nearest in a fixed
//    order (bit-identical from run to run).  Longer chains lose bits (the tensor
//    core truncates): against 64 bits fp32 outputs over 4096 k are 0.7e-7 (bf16)
//    and 0.85e-7 (fp16) off, as with fp32 fused multiply-adds (0.7e-7, 0.9e-7);
//    chains of 2 0.7e-7 and 0.9e-7, chains of 8 1.0e-7 and 1.9e-7.
//  * Programmatic dependent launch: a CTA of the next launch on the stream starts
//    as soon as one of these leaves, and issues its first code loads and builds
//    its table meanwhile.  At batch 1 two 8-warp CTAs run per SM for that; larger
//    batches, which hold more activations per lane, fill an SM with one CTA.
//
// What bounds it: nothing is saturated; the busiest unit is the L1 data path, which the
// lookups share with the code and activation loads.  8B gate (14336 x 4096) at batch 1,
// cycles per SM of the 15 300 of a launch in a chain (7.9 us): L1 data path 9 970 (lookups
// and partial sums 7 400, loads 2 570), HBM 8 400 (29.4 MB), instruction issue 7 140 per
// scheduler, and 16 warps to overlap them; the top stall is the wait for loads.  3 bits
// 10 380 and 9 340 (issue), 8 bits 17 260 and 12 430, 4 bits at batch 16 17 150 and 8 300
// (half of it activation loads).  So added instructions cost (an eighth of the codes
// resolved by permutes alone, 7 instructions for 4 codes instead of 4: 2 %) and so does a
// smaller L1 (kCarveout).  Per launch, the latency of a CTA's life (activations after the
// previous launch, first tile, final sum) is 1.6-2.5 us.  Per Llama-3.1-8B layer (q+k+v, o,
// gate+up, down chained, bf16), with fused multiply-adds on the CUDA cores (batches up to 8;
// 5 and more at 3 and 8 bits and 9 and more at 4 in the prefill kernel) before and now:
//   4 bits, batch 1 / 2 / 4 / 8 / 16: 31.1 / 45.6 / 57.0 / 109 / 117 us before,
//     30.6 / 33.9 / 39.5 / 48.7 / 63.0 now;
//   3 bits, batch 1 / 4 / 16: 39.0 / 68.7 / 162 before, 36.0 / 44.2 / 76.4 now;
//   8 bits, batch 1 / 4 / 16: 52.8 / 85.8 / 157 before, 48.7 / 59.1 / 92.3 now.
// Few rows of long K at batches 3-16 have a kernel of their own (few_rows_kernel).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "internal.h"

namespace logq {
namespace {

constexpr int kTabStride = 256;               // bytes per pair-table entry
// Shared address at which dynamic shared memory starts in a kernel without
// static shared memory: the per-CTA reserved area comes first.
constexpr uint32_t kTabOff = 1024;
constexpr uint32_t kLvlOff = 128;             // levels staged in the free half of table row 0
constexpr int kMaxItems = 4;
// Batches from kPartBatch up may share a row range among kMaxParts CTAs (each a
// part of K): a CTA that takes several passes over K reads all of X, at batch 16
// and K = 14336 458 KB against 190 KB of codes.  4096 x 14336 at batch 16 19.8 us
// instead of 23.3; the partial sums need workspace.
constexpr int64_t kPartBatch = 9, kMaxParts = 8;
// Warm-up ranges of this size or more are not prefetched: a launch's end waits for
// the prefetches it issued, and in a chain of launches that costs more than the
// next one gains (4 / 8 / 20 MiB: Llama-3.1-8B step of 128 launches 986 / 986 / 1002 us,
// Llama-3.2-1B step of 64 230.9 / 230.5 / 238.4, at 8 bits 313.9 / 317.5 / 325.4).
constexpr int64_t kPrefetchBytes = 4 << 20;

// One matrix of a grouped launch: all items share X, K, B and the code width.
struct GemvItem {
    const uint8_t* codes;
    void* Y;
    float* part;          // kparts > 1: partial sums [kparts][B][N] (caller's workspace)
    int32_t N;
    int32_t cta_begin;    // first CTA of this item
    int32_t rows_q;       // rows per row range of this item
    int32_t rows_rem;     // its first rows_rem row ranges take one more row
    uint32_t lvl16[16];   // code-indexed 16-bit levels (low half used)
};

struct GemvParams {
    int32_t nitems;
    int32_t K;
    int32_t B;
    int32_t y_dtype;
    const uint16_t* X;
    uint32_t* err;        // workspace error word
    int32_t row_bytes;
    int32_t blocks;       // blocks of a row
    int32_t spans;        // spans of S J blocks covering K
    int32_t kparts;       // CTAs that share a row range, each with part_spans of the spans
    int32_t part_spans;
    int32_t lg_groups;    // log2 of G, the warps sharing one span (row-parallel)
    int32_t span_cols;    // warps / G: spans in flight at once
    int32_t chunk_rows;   // rows reduced per shared-memory pass
    int32_t pitch;        // floats from one set of partial sums to the next
    int32_t wait_codes;   // codes are read only after the previous launch (reads_codes_early)
    const uint8_t* pf;    // optional L2 warm-up range (e.g. the next layer's codes)
    int64_t pf_bytes;
    int64_t pf_share;     // bytes of that range per CTA (multiple of 16)
    GemvItem item[kMaxItems];
};

// 8-bit codes: their 256 code-indexed levels per matrix travel as a second
// kernel parameter of the 8-bit kernels only, so the 3- and 4-bit launches keep
// their small parameter block.
struct Levels8 {
    uint16_t v[kMaxItems][256];
};
struct NoLevels {
    int32_t unused;
};
template <int BITS>
using LevelsT = typename std::conditional<BITS == 8, Levels8, NoLevels>::type;

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Table entry at byte offset off from the table base.  Not volatile, so that
// lookups move freely around the multiply-adds: what keeps them behind the
// table's barrier is that every offset is made from a value defined after it.
__device__ __forceinline__ uint32_t lds_tab(uint32_t off)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(off), "n"(kTabOff));
    return v;
}

// A block is the k that four lanes hold, each its own run: 32 k (12 or 16 bytes of
// codes), at 8 bits 16 k.
__host__ __device__ constexpr int lane_k(int bits) { return bits == 8 ? 16 : 32; }
__host__ __device__ constexpr int lane_words(int bits) { return bits == 3 ? 3 : 4; }
// Batch rows that the 8 NTL columns hold beside S segments.
__host__ __device__ constexpr int batch_cols(int S, int NTL) { return 8 * NTL / S; }
// Accumulator chains per column tile: their length, and how many interleave
// (registers allow fewer for more tiles).
__host__ __device__ constexpr int chain_length(int NTL) { return NTL == 1 ? 1 : 2; }
__host__ __device__ constexpr int chains_for(int bits, int S, int NTL)
{
    return NTL == 1 ? (bits == 4 && S <= 2 ? 4 : 8) : NTL == 2 ? 2 : 1;
}
constexpr int kMaxSmem = 226 * 1024;
// Shared-memory carveout of every shape, in percent of the maximum, which gives 164 KiB:
// room for two CTAs of a 64 KiB table and 17 KiB of partial sums (red_bytes; rows that
// need more are taken in chunks).  The rest of the 256 KiB per SM is L1, which holds
// activations that several warps read and the code loads in flight; one setting for all
// of them spares the SMs a reconfiguration between launches.  8B layer, 58 / 66 / 72 /
// 86 % and the maximum: batch 1 31.7 / 31.6 / 31.9 / 33.6 / 33.4 us, 4 39.6 / 39.6 / 39.7 /
// 42.0 / 41.9, 8 49.4 / 49.5 / 49.5 / 52.9 / 52.9, 16 63.0 / 63.0 / 63.6 / 66.7 / 66.8;
// 8 bits at batch 16 95.2 / 95.2 / 96.2 / 100.2 / 100.1.
constexpr int kCarveout = 66;
// Shared memory of partial sums after a table of tab bytes, per_sm CTAs on an SM: two stay
// within the carveout; one may ask for more.
constexpr int64_t red_bytes(size_t tab, int per_sm)
{
    return (int64_t)(per_sm > 1 ? 164 : 227) * 1024 / per_sm - 1024 - (int64_t)tab;
}

// A lane's codes of a block: 16 bytes, or (3-bit) the three words of a 12-byte
// group.  ALLOC: through L1 as usual; else without an L1 line.
template <bool ALLOC, int NW>
__device__ __forceinline__ void ld_codes(uint32_t (&w)[NW], const uint8_t* p)
{
    if constexpr (NW == 4) {
        if constexpr (ALLOC)
            asm volatile("ld.global.nc.v4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p));
        else
            asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p));
    } else {
#pragma unroll
        for (int i = 0; i < NW; ++i)
            asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(w[i]) : "l"(p + 4 * i));
    }
}

// D (16 x 8, fp32) += A (16 x 16) * B (16 x 8): lane l = 4 g + t holds
//   a0, a1: rows g, g + 8 at the first k pair of t; a2, a3: at the second one;
//   b0, b1: column g at the first / second k pair of t;
//   d0, d1: row g, columns 2t, 2t + 1; d2, d3: row g + 8.
template <bool F16>
__device__ __forceinline__ void mma(float (&d)[4], bool zero, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                    uint32_t b0, uint32_t b1)
{
    const float c0 = zero ? 0.f : d[0], c1 = zero ? 0.f : d[1], c2 = zero ? 0.f : d[2], c3 = zero ? 0.f : d[3];
    if constexpr (F16)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%10,%11,%12,%13};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%10,%11,%12,%13};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

__device__ __forceinline__ void store_y(void* Y, int dtype, int64_t idx, float v)
{
    if (dtype == LOGQ_F32) {
        static_cast<float*>(Y)[idx] = v;
    } else if (dtype == LOGQ_BF16) {
        static_cast<__nv_bfloat16*>(Y)[idx] = __float2bfloat16_rn(v);
    } else {
        static_cast<__half*>(Y)[idx] = __float2half_rn(v);
    }
}

// Value pairs 2q and 2q + 1 (k = 4q .. 4q + 3 of the lane's run) from the pair
// table.  base_lane holds 4 * lane in byte 0 and zeros above, so one byte
// permute yields the entry's offset byte * 256 + 4 * lane.
template <int BITS, int NW>
__device__ __forceinline__ void pairs_of(const uint32_t (&w)[NW], int q, uint32_t base_lane, uint32_t& p0, uint32_t& p1)
{
    if constexpr (BITS == 4) {
        const uint32_t c = w[q >> 1];
        p0 = lds_tab(prmt(c, base_lane, (q & 1) ? 0x7624u : 0x7604u));
        p1 = lds_tab(prmt(c, base_lane, (q & 1) ? 0x7634u : 0x7614u));
    } else if constexpr (BITS == 8) {
        // entry e holds the value of code e in both halves
        const uint32_t c = w[q];
        const uint32_t v0 = lds_tab(prmt(c, base_lane, 0x7604u)), v1 = lds_tab(prmt(c, base_lane, 0x7614u));
        const uint32_t v2 = lds_tab(prmt(c, base_lane, 0x7624u)), v3 = lds_tab(prmt(c, base_lane, 0x7634u));
        p0 = prmt(v0, v1, 0x5410u);
        p1 = prmt(v2, v3, 0x5410u);
    } else {
        // of a group of 32 k: pair i < 15 is the 6-bit field i % 5 of word i / 5; pair 15 the words' top bits
        auto off = [&](int i) -> uint32_t {
            const int w0 = 3 * (i / 16);
            i %= 16;
            if (i == 15)
                return ((w[w0] >> 22) & 0x0300u) | ((w[w0 + 1] >> 20) & 0x0c00u) | ((w[w0 + 2] >> 18) & 0x3000u) | base_lane;
            const uint32_t x = w[w0 + i / 5];
            const int f = i % 5;
            const uint32_t v = f == 0 ? (x << 8) : f == 1 ? (x << 2) : f == 2 ? (x >> 4) : f == 3 ? (x >> 10) : (x >> 16);
            return (v & 0x3f00u) | base_lane;
        };
        p0 = lds_tab(off(2 * q));
        p1 = lds_tab(off(2 * q + 1));
    }
}

// S segments of J blocks per span, NTL column tiles, T tiles of 16 / S rows in flight.
template <int BITS, int S, int J, int NTL, int T, bool F16, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) gemv_kernel(const __grid_constant__ GemvParams p,
                                                        const __grid_constant__ LevelsT<BITS> lv)
{
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr bool HALVES = S >= 4;                          // a row's segments are split over the MMA's two row halves
    constexpr int HS = HALVES ? S / 2 : S;                   // segments per row half
    constexpr int RT = 16 / S, RH = HALVES ? 0 : 8 / S;      // rows per tile; rows from the first half to the second
    constexpr int BC = batch_cols(S, NTL), CB = 8 / S;       // batch rows; batch rows per column tile
    constexpr int NW = lane_words(BITS), BB = 16 * NW;       // words of a lane's codes; code bytes of a block
    constexpr int NENT = (BITS == 3) ? 64 : 256;
    constexpr uint32_t TAB_BYTES = NENT * kTabStride;
    constexpr int LK = lane_k(BITS), BK = 4 * LK, BQ = LK / 4;    // k of a lane's run and of a block; multiply-adds per block
    constexpr int NQ = J * BQ;                               // multiply-adds per tile and column tile
    constexpr int CL = chain_length(NTL), CHAINS = chains_for(BITS, S, NTL), NCH = CHAINS * CL <= NQ ? CHAINS : NQ / CL;
    static_assert(NQ % (NCH * CL) == 0, "whole groups of chains");

    // programmatic dependent launch: the next kernel on the stream may start
    // now.  Its CTAs may run beside this one and do their own prologue
    // meanwhile; they wait for this grid to finish before they touch X or Y.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if ((uint32_t)__cvta_generic_to_shared(smem) != kTabOff) {   // table addressing relies on it
        if (tid == 0) atomicExch(p.err, (uint32_t)LOGQ_ERR_UNSUPPORTED);
        return;
    }
    // this CTA's matrix and its contiguous range of rows
    int m = 0;
#pragma unroll
    for (int i = 1; i < kMaxItems; ++i)
        if (i < p.nitems && (int)blockIdx.x >= p.item[i].cta_begin) m = i;
    const GemvItem& item = p.item[m];
    uint32_t* const lvl = reinterpret_cast<uint32_t*>(smem + kLvlOff);
    if constexpr (BITS != 8)
        if (tid < 16) lvl[tid] = item.lvl16[tid];
    const int cta = (int)blockIdx.x - item.cta_begin;
    const int c = p.kparts == 1 ? cta : cta / p.kparts, kpart = cta - c * p.kparts;
    const int s0 = kpart * p.part_spans, s1 = s0 + p.part_spans < p.spans ? s0 + p.part_spans : p.spans;
    const int r0 = c * item.rows_q + (c < item.rows_rem ? c : item.rows_rem);
    const int r1 = r0 + item.rows_q + (c < item.rows_rem ? 1 : 0);

    // Lane 4 gq + t4 holds k LK t4 .. LK t4 + LK - 1 of a block.  As a holder of
    // activations: column gq of each column tile; column tile nt holds batch rows
    // nt 8 / S .. and for each its S segments.  As a holder of weights: the MMA's
    // rows gq (h = 0) and gq + 8 (h = 1), each a row of the tile and one segment.
    //   S = 8, 4: row gq / HS of the tile, segment h HS + gq % HS; columns 2 i and
    //     2 i + 1 hold batch row i / HS, segments i % HS and HS + i % HS.  A row's
    //     products then stand in d0 (h = 0) and d3 (h = 1) of the lanes with
    //     t4 % HS == gq % HS, batch row t4 / HS.
    //   S = 2, 1: row gq / S + h 8 / S, segment gq % S; column n holds batch row
    //     n / S, segment n % S.  S = 2: d0 or d1 (d2 or d3), by the segment.
    const int gq = lane >> 2, t4 = lane & 3;
    const int rl = gq / HS, aseg = gq % HS;
    const int bseg = HALVES ? (gq & 1) * HS + (gq >> 1) % HS : gq % S;
    const int bcol = HALVES ? (gq >> 1) / HS : gq / S;
    const int G = 1 << p.lg_groups, SC = p.span_cols;
    const int g = warp & (G - 1), scol = warp >> p.lg_groups;
    // (a warp whose first tile starts past the rows would only load activations)
    const bool compute_warp = scol < SC && s0 + scol < s1 && g * RT < r1 - r0;
    struct Tile { uint32_t w[2][J][NW]; };
    Tile ct[T];
    // The span being worked on: address of this lane's codes in row q0.  Blocks
    // past K read the row's first block and are taken as 0.
    struct Span { const uint8_t* codes; int off[2][J]; bool ragged; };
    auto block_of = [&](int s, int h, int j) { return (s * J + j) * S + (HALVES ? h * HS : 0) + aseg; };
    auto span_at = [&](int q0, int s) -> Span {
        Span sp;
        sp.codes = item.codes + (int64_t)(q0 + rl) * p.row_bytes + t4 * (4 * NW);
        sp.ragged = (s + 1) * (S * J) > p.blocks;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int kb = block_of(s, h, j);
                sp.off[h][j] = kb < p.blocks ? kb * BB : 0;
            }
        return sp;
    };
    // codes of the tile at local row lt; rows past the chunk's nrows read its last row
    auto load_tile = [&](Tile& c, const Span& sp, int lt, int nrows) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int last = nrows - 1 - rl, r = lt + h * RH < last ? lt + h * RH : last;
            const uint8_t* rp = sp.codes + (int64_t)r * p.row_bytes;
#pragma unroll
            for (int j = 0; j < J; ++j) ld_codes<S == 1, NW>(c.w[h][j], rp + sp.off[h][j]);
        }
    };
    // 0) the first T tiles' codes of this warp's first (chunk, span) go out first:
    //    their latency hides behind the prologue below.  Codes are weights, not
    //    the previous kernel's output (see the launch contract), or wait_codes is set.
    auto load_first = [&](const Span& sp, int nrows) {
#pragma unroll
        for (int u = 0; u < T; ++u)
            if ((u * G + g) * RT < nrows) load_tile(ct[u], sp, (u * G + g) * RT, nrows);
    };
    auto chunk_of = [&](int q0) { return r1 - q0 > p.chunk_rows ? p.chunk_rows : r1 - q0; };
    int nrows = chunk_of(r0);
    Span sp = span_at(r0, s0 + scol);
    if (BC >= 8 && p.wait_codes)                       // (shapes for up to 4 rows never do)
        asm volatile("griddepcontrol.wait;" ::: "memory");
    if (compute_warp) load_first(sp, nrows);

    // 1) its share of the optional warm-up range
    if (p.pf_bytes > 0) {
        constexpr int64_t piece = 16384;
        const int64_t beg = p.pf_share * blockIdx.x;
        const int64_t end = (beg + p.pf_share < p.pf_bytes) ? beg + p.pf_share : p.pf_bytes;
        for (int64_t off = beg + (int64_t)tid * piece; off < end; off += (int64_t)NT * piece) {
            const int64_t n = (end - off) < piece ? (end - off) : piece;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.pf + off), "r"((uint32_t)n)
                         : "memory");
        }
    }

    // 2) pair table: entry e = (value of its low code) | (value of its high
    //    code) << 16, 32 copies (one per lane) in the first 128 bytes of its
    //    256-byte row.  The 16 levels are staged in the free half of row 0
    //    (indexed parameter reads with per-thread indices would serialise); a
    //    warp makes 32 entries, one per lane, and writes four rows at a time.
    //    8-bit codes: entry e is the value of code e in both halves.
    if constexpr (BITS != 8) __syncthreads();
#pragma unroll
    for (int e0 = 32 * warp; e0 < NENT; e0 += NT) {
        const int e = e0 + lane;
        uint32_t v;
        if constexpr (BITS == 8) v = (uint32_t)lv.v[m][e] * 0x10001u;
        else v = lvl[BITS == 4 ? (e & 15) : (e & 7)] | (lvl[BITS == 4 ? (e >> 4) : (e >> 3)] << 16);
        uint8_t* at = smem + (e0 + (lane >> 3)) * kTabStride + (lane & 7) * 16;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t x = __shfl_sync(0xffffffffu, v, 4 * i + (lane >> 3));
            *reinterpret_cast<uint4*>(at + 4 * i * kTabStride) = make_uint4(x, x, x, x);
        }
    }
    // this lane's partial sums: set (scol, segment) of np, first batch row, row rl
    float* const red0 = reinterpret_cast<float*>(smem + TAB_BYTES);
    const bool holder = !HALVES || t4 % HS == aseg;
    float* const red = red0 + (scol * HS + aseg) * p.pitch + rl * BC + (HALVES ? t4 / HS : S == 2 ? t4 : 2 * t4);
    const uint16_t* const xl = p.X + LK * t4;
    __syncthreads();

    uint32_t base_lane = 4u * (uint32_t)lane;
    asm volatile("" : "+r"(base_lane)::"memory");    // lookups stay behind the barrier
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int q0 = r0;;) {
        if (compute_warp) {
            for (int s = s0 + scol;;) {
                // activations of this span stay in registers (zero outside K and the batch)
                uint32_t xr[NTL][J][LK / 2];
#pragma unroll
                for (int nt = 0; nt < NTL; ++nt) {
                    const int b = nt * CB + bcol;
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const int kb = (s * J + j) * S + bseg;
                        const uint16_t* xp = xl + (int64_t)b * p.K + (int64_t)kb * BK;
                        const bool on = kb < p.blocks && b < p.B;
#pragma unroll
                        for (int i = 0; i < LK / 2; i += 4) {
                            uint4 v = make_uint4(0, 0, 0, 0);
                            if (on) v = *reinterpret_cast<const uint4*>(xp + 2 * i);
                            xr[nt][j][i] = v.x;
                            xr[nt][j][i + 1] = v.y;
                            xr[nt][j][i + 2] = v.z;
                            xr[nt][j][i + 3] = v.w;
                        }
                    }
                }
                // one tile; a row's result for a batch row is added over this warp's spans
                // in its shared-memory slot
                const bool first = s == s0 + scol;
                auto put = [&](float& slot, float v) { slot = first ? v : slot + v; };
                auto run_tile = [&](Tile& c, int lt) {
                    if (sp.ragged) {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int j = 0; j < J; ++j)
                                if (block_of(s, h, j) >= p.blocks)
#pragma unroll
                                    for (int i = 0; i < NW; ++i) c.w[h][j][i] = 0u;
                    }
                    // groups of NCH interleaved chains of CL multiply-adds, chains and groups
                    // added up pairwise with rounding to nearest (the tensor core truncates
                    // its sums); sum[l] holds the sum of 2^l groups
                    constexpr int NG = NQ / (NCH * CL);
                    float acc[NTL][4], sum[5][NTL][4];
                    static_assert(NG <= 32 && (NG & (NG - 1)) == 0, "pairwise over the groups");
#pragma unroll
                    for (int gr = 0; gr < NG; ++gr) {
                        float d[NTL][NCH][4];
#pragma unroll
                        for (int qq = 0; qq < NCH * CL; ++qq) {
                            const int q = gr * NCH * CL + qq;
                            uint32_t a0, a1, a2, a3;
                            pairs_of<BITS, NW>(c.w[0][q / BQ], q % BQ, base_lane, a0, a2);
                            pairs_of<BITS, NW>(c.w[1][q / BQ], q % BQ, base_lane, a1, a3);
#pragma unroll
                            for (int nt = 0; nt < NTL; ++nt)
                                mma<F16>(d[nt][qq % NCH], qq < NCH, a0, a1, a2, a3, xr[nt][q / BQ][2 * (q % BQ)],
                                         xr[nt][q / BQ][2 * (q % BQ) + 1]);
                        }
#pragma unroll
                        for (int nt = 0; nt < NTL; ++nt)
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
#pragma unroll
                                for (int w = NCH / 2; w >= 1; w /= 2)
#pragma unroll
                                    for (int ch = 0; ch < w; ++ch) d[nt][ch][i] += d[nt][ch + w][i];
                                float v = d[nt][0][i];
                                int l = 0;
#pragma unroll
                                for (; (gr >> l) & 1; ++l) v += sum[l][nt][i];
                                if (gr == NG - 1) acc[nt][i] = v;
                                else sum[l][nt][i] = v;
                            }
                    }
                    float* slot = red + lt * BC;
                    if constexpr (HALVES) {
                        if (holder && lt + rl < nrows)
#pragma unroll
                            for (int nt = 0; nt < NTL; ++nt) put(slot[nt * CB], acc[nt][0] + acc[nt][3]);
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (lt + rl + h * RH < nrows)
#pragma unroll
                                for (int nt = 0; nt < NTL; ++nt) {
                                    if constexpr (S == 2) {
                                        put(slot[h * RH * BC + nt * CB], aseg ? acc[nt][2 * h + 1] : acc[nt][2 * h]);
                                    } else {
                                        put(slot[h * RH * BC + nt * CB], acc[nt][2 * h]);
                                        put(slot[h * RH * BC + nt * CB + 1], acc[nt][2 * h + 1]);
                                    }
                                }
                    }
                };
                // T tiles in flight: a tile's registers are refilled as soon as it is decoded
                for (int lt = g * RT; lt < nrows;) {
#pragma unroll
                    for (int u = 0; u < T; ++u) {
                        run_tile(ct[u], lt);
                        if (lt + T * G * RT < nrows) load_tile(ct[u], sp, lt + T * G * RT, nrows);
                        lt += G * RT;
                        if (lt >= nrows) break;
                    }
                }
                s += SC;
                if (s >= s1) break;
                sp = span_at(q0, s);
                load_first(sp, nrows);
            }
        }
        const int n0 = nrows;
        const bool more = r1 - q0 > p.chunk_rows;
        const int q1 = more ? q0 + p.chunk_rows : r1;
        if (more && compute_warp) {           // the next chunk's first codes are in flight during this one's sums
            sp = span_at(q1, s0 + scol);
            load_first(sp, chunk_of(q1));
        }
        __syncthreads();
        // fixed-order sum of each output's partial sums
        const int np = (SC < s1 - s0 ? SC : s1 - s0) * HS;
        for (int i = tid; i < n0 * BC; i += NT) {
            const int row = i / BC, b = i % BC;
            if (b >= p.B) continue;
            float sum = 0.f;
            int k = 0;
            for (; k + 8 <= np; k += 8) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = red0[(k + u) * p.pitch + i];
                sum += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
            }
            for (; k < np; ++k) sum += red0[k * p.pitch + i];
            if (p.kparts == 1) store_y(item.Y, p.y_dtype, (int64_t)b * item.N + q0 + row, sum);
            else item.part[((int64_t)kpart * p.B + b) * item.N + q0 + row] = sum;
        }
        if (!more) break;
        __syncthreads();
        q0 = q1;
        nrows = chunk_of(q0);
    }
}

// ------------------------------------------------------------ few rows ---

// acc_lo / acc_hi += the low / high 16-bit value of w times that of x.
template <bool F16>
__device__ __forceinline__ void fma_pair(float& lo, float& hi, uint32_t w, uint32_t x)
{
    if constexpr (F16)
        asm("{.reg .b16 wl, wh, xl, xh;\n\tmov.b32 {wl, wh}, %2;\n\tmov.b32 {xl, xh}, %3;\n\t"
            "fma.rn.f32.f16 %0, wl, xl, %0;\n\tfma.rn.f32.f16 %1, wh, xh, %1;}"
            : "+f"(lo), "+f"(hi) : "r"(w), "r"(x));
    else
        asm("{.reg .b16 wl, wh, xl, xh;\n\tmov.b32 {wl, wh}, %2;\n\tmov.b32 {xl, xh}, %3;\n\t"
            "fma.rn.f32.bf16 %0, wl, xl, %0;\n\tfma.rn.f32.bf16 %1, wh, xh, %1;}"
            : "+f"(lo), "+f"(hi) : "r"(w), "r"(x));
}

// Sum of each of V per-lane values over the 32 lanes; lane l returns that of value
// l >> (5 - log2 V) (V a power of two up to 32).
template <int V>
__device__ __forceinline__ float reduce_scatter(float (&a)[V], int lane)
{
    int count = V;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        if (count > 1) {
            const int half = count / 2;
            const bool upper = (lane & m) != 0;
#pragma unroll
            for (int i = 0; i < V / 2; ++i)
                if (i < half) {
                    const float send = upper ? a[i] : a[i + half];
                    const float keep = upper ? a[i + half] : a[i];
                    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
                }
            count = half;
        } else {
            a[0] += __shfl_xor_sync(0xffffffffu, a[0], m);
        }
    }
    return a[0];
}

// The pair table, and this CTA's share of the warm-up range below it, as in gemv_kernel.
// (Not shared with it: as functions they cost its batch-1 4-bit instance a spilled register
// and the 8B step 4 %, 979 -> 1018 us.)
template <int BITS, int NT>
__device__ __forceinline__ void build_table(uint8_t* smem, const uint32_t* lvl, const LevelsT<BITS>& lv, int m)
{
    constexpr int NENT = (BITS == 3) ? 64 : 256;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (BITS != 8) __syncthreads();
#pragma unroll
    for (int e0 = 32 * warp; e0 < NENT; e0 += NT) {
        const int e = e0 + lane;
        uint32_t v;
        if constexpr (BITS == 8) v = (uint32_t)lv.v[m][e] * 0x10001u;
        else v = lvl[BITS == 4 ? (e & 15) : (e & 7)] | (lvl[BITS == 4 ? (e >> 4) : (e >> 3)] << 16);
        uint8_t* at = smem + (e0 + (lane >> 3)) * kTabStride + (lane & 7) * 16;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t x = __shfl_sync(0xffffffffu, v, 4 * i + (lane >> 3));
            *reinterpret_cast<uint4*>(at + 4 * i * kTabStride) = make_uint4(x, x, x, x);
        }
    }
}

template <int NT>
__device__ __forceinline__ void warm_share(const GemvParams& p)
{
    if (p.pf_bytes <= 0) return;
    constexpr int64_t piece = 16384;
    const int64_t beg = p.pf_share * blockIdx.x;
    const int64_t end = (beg + p.pf_share < p.pf_bytes) ? beg + p.pf_share : p.pf_bytes;
    for (int64_t off = beg + (int64_t)threadIdx.x * piece; off < end; off += (int64_t)NT * piece) {
        const int64_t n = (end - off) < piece ? (end - off) : piece;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.pf + off), "r"((uint32_t)n) : "memory");
    }
}

// k of a lane's run in the few-rows kernel: 8 bytes of 4-bit codes, 16 of 8-bit ones, a
// 3-bit group.
__host__ __device__ constexpr int few_k(int bits) { return bits == 3 ? 32 : 16; }

// Few rows of long K (few_rows), batches 3 to 16 padded to B: one row at a time per group
// of warps, fused multiply-adds on the CUDA cores.  Each warp owns spans of 32 runs of
// consecutive k; a row's products are summed over its lanes, then over the spans in
// order.  Against the matrix-instruction kernel, whose tiles of 16 / S rows leave most SMs
// idle here while each CTA loads all activations with 64 bytes between its lanes: a row per
// CTA, and activation loads at half the cost in the L1 path (figures at few_rows).  Bound by
// those loads and by latency.
template <int BITS, int B, bool F16, int NT>
__global__ void __launch_bounds__(NT, 1) few_rows_kernel(const __grid_constant__ GemvParams p,
                                                         const __grid_constant__ LevelsT<BITS> lv)
{
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr int LK = few_k(BITS), NW = BITS == 8 ? LK / 4 : BITS == 4 ? LK / 8 : 3;
    constexpr uint32_t TAB_BYTES = (BITS == 3 ? 64 : 256) * kTabStride;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // (see gemv_kernel)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if ((uint32_t)__cvta_generic_to_shared(smem) != kTabOff) {   // table addressing relies on it
        if (tid == 0) atomicExch(p.err, (uint32_t)LOGQ_ERR_UNSUPPORTED);
        return;
    }
    int m = 0;
#pragma unroll
    for (int i = 1; i < kMaxItems; ++i)
        if (i < p.nitems && (int)blockIdx.x >= p.item[i].cta_begin) m = i;
    const GemvItem& item = p.item[m];
    uint32_t* const lvl = reinterpret_cast<uint32_t*>(smem + kLvlOff);
    if constexpr (BITS != 8)
        if (tid < 16) lvl[tid] = item.lvl16[tid];
    const int cta = (int)blockIdx.x - item.cta_begin;
    const int r0 = cta * item.rows_q + (cta < item.rows_rem ? cta : item.rows_rem);
    const int rows = item.rows_q + (cta < item.rows_rem ? 1 : 0);
    const int G = 1 << p.lg_groups, g = warp & (G - 1), scol = warp >> p.lg_groups;
    const bool compute_warp = scol < p.span_cols && g < rows;
    struct Codes { uint32_t w[NW]; };
    // this lane's codes of row r0 + r, span s; runs past K count as 0
    auto load = [&](Codes& c, int r, int s) {
        const int k0 = (s * 32 + lane) * LK;
        const uint8_t* at = item.codes + (int64_t)(r0 + r) * p.row_bytes + k0 / 32 * (4 * BITS) + k0 % 32 * BITS / 8;
        if (k0 >= p.K) {
#pragma unroll
            for (int i = 0; i < NW; ++i) c.w[i] = 0u;
        } else if constexpr (NW == 2) {
            asm volatile("ld.global.nc.L1::no_allocate.v2.b32 {%0,%1}, [%2];" : "=r"(c.w[0]), "=r"(c.w[1]) : "l"(at));
        } else {
            ld_codes<false, NW>(c.w, at);
        }
    };
    if (p.wait_codes) asm volatile("griddepcontrol.wait;" ::: "memory");
    Codes cur;
    if (compute_warp) load(cur, g, scol);
    warm_share<NT>(p);
    build_table<BITS, NT>(smem, lvl, lv, m);
    __syncthreads();
    uint32_t base_lane = 4u * (uint32_t)lane;
    asm volatile("" : "+r"(base_lane)::"memory");    // lookups stay behind the barrier
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float* const red = reinterpret_cast<float*>(smem + TAB_BYTES);       // [span][row][B]
    if (compute_warp)
        for (int s = scol; s < p.spans; s += p.span_cols) {
            const int k0 = (s * 32 + lane) * LK;
            uint32_t xr[B][LK / 2];
#pragma unroll
            for (int b = 0; b < B; ++b)
#pragma unroll
                for (int i = 0; i < LK / 2; i += 4) {
                    uint4 v = make_uint4(0, 0, 0, 0);
                    if (k0 < p.K && b < p.B) v = *reinterpret_cast<const uint4*>(p.X + (int64_t)b * p.K + k0 + 2 * i);
                    xr[b][i] = v.x;
                    xr[b][i + 1] = v.y;
                    xr[b][i + 2] = v.z;
                    xr[b][i + 3] = v.w;
                }
            for (int r = g; r < rows; r += G) {
                Codes next;                          // the next row's, or the next span's first
                const bool same = r + G < rows;
                if (same || s + p.span_cols < p.spans) load(next, same ? r + G : g, same ? s : s + p.span_cols);
                float lo[B], hi[B];
#pragma unroll
                for (int b = 0; b < B; ++b) lo[b] = hi[b] = 0.f;
#pragma unroll
                for (int q = 0; q < LK / 4; ++q) {
                    uint32_t p0, p1;
                    pairs_of<BITS, NW>(cur.w, q, base_lane, p0, p1);
#pragma unroll
                    for (int b = 0; b < B; ++b) {
                        fma_pair<F16>(lo[b], hi[b], p0, xr[b][2 * q]);
                        fma_pair<F16>(lo[b], hi[b], p1, xr[b][2 * q + 1]);
                    }
                }
#pragma unroll
                for (int b = 0; b < B; ++b) lo[b] += hi[b];
                const float sum = reduce_scatter<B>(lo, lane);
                if (lane % (32 / B) == 0) red[(s * rows + r) * B + lane / (32 / B)] = sum;
                cur = next;
            }
        }
    __syncthreads();
    for (int i = tid; i < rows * B; i += NT) {
        const int row = i / B, b = i % B;
        if (b >= p.B) continue;
        float sum = 0.f;
        for (int s = 0; s < p.spans; ++s) sum += red[s * rows * B + i];
        store_y(item.Y, p.y_dtype, (int64_t)b * item.N + r0 + row, sum);
    }
}

// Added to a padded batch: the shape for short rows (shape_key).
constexpr int kShort = 64, kMid = 128;
// Launches of up to this many weights keep to one CTA per SM (per_sm).
constexpr int64_t kOneCta = (int64_t)4 << 20;

// Launch shape of a batch: S segments, J blocks, NTL column tiles,
// T tiles in flight, threads per CTA, CTAs per SM.
struct Shape {
    int S, J, NTL, T, NT, MINB;
};

// Launch of a decode kernel k.  Dynamic shared memory opt-in and carveout: per-device
// function attributes, set once per device.
template <int BITS, typename Kernel>
cudaError_t run_kernel(Kernel k, bool (&configured)[64], const GemvParams& p, const GroupArgs& a, int grid, int threads,
                       size_t smem, cudaStream_t s)
{
    LevelsT<BITS> lv;
    memset(&lv, 0, sizeof lv);
    if constexpr (BITS == 8)
        for (int i = 0; i < a.count; ++i)
            for (int c = 0; c < 256; ++c) lv.v[i][c] = a.item[i].lvl16[c];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, kCarveout);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, p, lv);
}

template <int BITS, int S, int J, int NTL, int T, int NT, int MINB, bool F16>
cudaError_t run(const GemvParams& p, const GroupArgs& a, int grid, size_t smem, cudaStream_t s)
{
    static bool configured[64] = {false};
    return run_kernel<BITS>(gemv_kernel<BITS, S, J, NTL, T, F16, NT, MINB>, configured, p, a, grid, NT, smem, s);
}

template <int BITS, int B, int NT, bool F16>
cudaError_t run_few(const GemvParams& p, const GroupArgs& a, int grid, size_t smem, cudaStream_t s)
{
    static bool configured[64] = {false};
    return run_kernel<BITS>(few_rows_kernel<BITS, B, F16, NT>, configured, p, a, grid, NT, smem, s);
}

// The compiled shapes, per code width and padded batch; calls fn with the
// shape's constants as template arguments.
// Shape of a key (sh), and its launch when p is not NULL.  More segments
// make a warp's loads longer runs of one row (S = 8: 256 bytes per row half),
// fewer leave columns for the batch; J blocks per segment share a row's final sum
// among more multiply-adds where registers hold the activations (16 per column
// tile and block).  Each line was the fastest of the shapes tried for it on the
// Llama-3.1-8B layer (the figures at the top); at 8 bits a block is 64 k, so J
// doubles.
template <int BITS, bool F16>
cudaError_t shape_or_run(int key, Shape* sh, const GemvParams* p, const GroupArgs* a, int grid, size_t smem, cudaStream_t s)
{
#define LOGQ_SHAPE(B, S, J, NTL, T, NT, MINB) \
    case B: \
        *sh = Shape{S, J, NTL, T, NT, MINB}; \
        return p ? run<BITS, S, J, NTL, T, NT, MINB, F16>(*p, *a, grid, smem, s) : cudaSuccess
    if constexpr (BITS == 3) {
        switch (key) {
            LOGQ_SHAPE(1, 8, 1, 1, 6, 256, 2);
            LOGQ_SHAPE(2, 4, 1, 1, 4, 512, 1);
            LOGQ_SHAPE(4, 2, 2, 1, 2, 512, 1);
            LOGQ_SHAPE(8, 1, 2, 1, 2, 512, 1);
            LOGQ_SHAPE(16, 1, 2, 2, 1, 512, 1);
            LOGQ_SHAPE(32, 1, 2, 4, 1, 256, 1);
            LOGQ_SHAPE(kShort + 1, 4, 1, 1, 4, 256, 2);
            LOGQ_SHAPE(kShort + 2, 4, 1, 1, 4, 256, 2);
            LOGQ_SHAPE(kShort + 4, 2, 1, 1, 4, 256, 2);
        }
    } else if constexpr (BITS == 4) {
        switch (key) {
            LOGQ_SHAPE(1, 8, 1, 1, 5, 256, 2);
            LOGQ_SHAPE(2, 4, 1, 1, 4, 512, 1);
            LOGQ_SHAPE(4, 2, 2, 1, 2, 512, 1);
            LOGQ_SHAPE(8, 1, 2, 1, 2, 512, 1);
            LOGQ_SHAPE(16, 1, 4, 2, 2, 256, 1);
            LOGQ_SHAPE(32, 1, 2, 4, 1, 256, 1);
            LOGQ_SHAPE(kShort + 1, 2, 1, 1, 4, 256, 2);
            LOGQ_SHAPE(kMid + 1, 4, 1, 1, 4, 256, 2);
            LOGQ_SHAPE(kShort + 2, 4, 1, 1, 4, 256, 2);
            LOGQ_SHAPE(kShort + 4, 2, 1, 1, 5, 256, 2);
            LOGQ_SHAPE(kShort + 8, 1, 2, 1, 3, 256, 1);
            LOGQ_SHAPE(kShort + 16, 1, 2, 2, 2, 256, 1);
        }
    } else {
        switch (key) {
            LOGQ_SHAPE(1, 8, 2, 1, 3, 256, 2);
            LOGQ_SHAPE(2, 4, 2, 1, 3, 512, 1);
            LOGQ_SHAPE(4, 2, 2, 1, 3, 512, 1);
            LOGQ_SHAPE(8, 2, 2, 2, 2, 512, 1);
            LOGQ_SHAPE(16, 1, 4, 2, 2, 256, 1);
            LOGQ_SHAPE(32, 1, 4, 4, 1, 256, 1);
            LOGQ_SHAPE(kShort + 1, 4, 1, 1, 5, 256, 2);
            LOGQ_SHAPE(kShort + 2, 4, 1, 1, 5, 256, 2);
            LOGQ_SHAPE(kMid + 2, 4, 2, 1, 3, 256, 2);
            LOGQ_SHAPE(kShort + 4, 2, 2, 1, 3, 256, 2);
        }
    }
#undef LOGQ_SHAPE
    return cudaErrorInvalidValue;
}

template <bool F16>
cudaError_t shape_or_run(int bits, int key, Shape* sh, const GemvParams* p, const GroupArgs* a, int grid, size_t smem,
                         cudaStream_t s)
{
    return bits == 8 ? shape_or_run<8, F16>(key, sh, p, a, grid, smem, s)
         : bits == 4 ? shape_or_run<4, F16>(key, sh, p, a, grid, smem, s)
                     : shape_or_run<3, F16>(key, sh, p, a, grid, smem, s);
}

// Key of a call's launch shape: the batch padded to a power of two, plus kShort or kMid for
// short rows.  Those fill a CTA's warps with spans of the wide shapes only by sharing each
// span among several warps, all of which read its activations; shapes with shorter spans
// spare that.  Single launches, us, wide shape / this one (rows x k, batch in brackets):
//   3 bits: 512 x 2048 (1) 2.38 / 1.86, (2) 2.65 / 1.95; 8192 x 512 (1) 2.86 / 2.27, (4) 3.39 /
//     2.5; 2048 x 2048 (2) 3.14 / 2.4, (4) 3.66 / 2.6; 16384 x 2048 (2) 6.6 / 6.35;
//   4 bits: 8192 x 512 (2) 2.42 here, 4096 k (2): 1024 rows 3.0 / 2.4, 28672 rows 14.9 / 14.3;
//     1000 x 3968 (1) 2.32 (kMid), 3.25 with the kShort shape, whose spans take two passes
//     from K = 2176 on; 2048 x 2048 (8) 3.6 / 2.7, (16) 4.9 / 3.45; 4096 x 4096 (16) 7.5, 8.3
//     with the short one;
//   8 bits: 8192 x 512 (1) 3.46 / 2.7; 512 x 2048 (2) 2.84 / 1.9; 16384 x 2048 (2) 9.1 / 8.6, (4)
//     10.8 / 10.0; 6144 x 4096 (2, kMid) 7.6 / 7.2; 2048 x 2048 (1) 2.65 / 2.73, so batch 1
//     only up to 1024 k.
// Batch 1 at 3 and 4 bits: up to 8 M weights (16384 x 2048 in a chain of the 1B shapes 0.06 us
// slower with the short shape, 32768 x 2048 at 3 bits 9.8 / 10.3).
int shape_key(int bits, int64_t B, int64_t rows, int64_t K)
{
    int key = 1;
    while (key < B) key *= 2;
    const bool few = rows * K <= (int64_t)8 << 20;
    if (bits == 4) {
        if (key == 1 && K < 4096 && few) key += K <= 2048 ? kShort : kMid;
        else if (key == 2 ? K <= 4096 : key == 4 ? K <= 2048 : K < 4096 && key >= 8 && key <= 16) key += kShort;
    } else if (bits == 3) {
        if (key == 1 ? K < 4096 && few : key == 2 ? K <= 4096 : key == 4 && K <= 2048) key += kShort;
    } else {
        if (key == 1 ? K <= 1024 : key <= 4 && K <= 2048) key += kShort;
        else if (key == 2 && K <= 4096) key += kMid;
    }
    return key;
}

// CTAs of a launch per SM: as many as fit, but one for small launches of the shapes that
// fit twice, so that the next launch's CTAs find room on every SM from the start (their
// table and first code loads then run beside this launch).  1B step, one CTA per SM for no
// launch / up to 4 M weights (o) / up to 8 M (q/k/v too): batch 1 233.2 / 232.4 / 235.6 us,
// batch 2 265.3 / 256.6 / 258.9, batch 4 286.7 / 279.5 / 284.4.
int per_sm(const Shape& sh, int64_t weights) { return weights <= kOneCta ? 1 : sh.MINB; }

// Whether few_rows_kernel runs a launch.  us, matrix-instruction kernel / few_rows_kernel
// (rows x k, batch in brackets; the line lies where they meet):
//   4 bits: 64 x 4096 (4) 2.58 / 1.85, (8) 3.25 / 2.29, (16) 4.46 / 2.86; 128 x 8192 (8) 5.60 /
//     2.94; 128 x 14336 (16) 13.9 / 7.5; 256 x 4096 (4) 2.68 / 2.22; 384 rows at 3072, 8192 and
//     14336 k (4) 2.42 / 2.37, 3.40 / 3.07, 5.60 / 5.78, (8) 3.30 / 3.00, 5.71 / 4.01, 10.1 / 7.3,
//     (16) 4.42 / 3.65, 8.75 / 6.83, 15.1 / 13.4; 512 x 4096 (8) 3.45 / 3.51; 192 x 2048 (8) 2.28 /
//     2.31;
//   3 bits: 128 x 4096 (4) 2.77 / 2.43, 192 x 8192 3.46 / 3.81;
//   8 bits: 128 x 3072 (4) 2.17 / 2.08, 192 x 3072 2.17 / 2.23, 256 x 4096 2.41 / 2.41, 256 x 14336
//     7.5 / 4.9, 384 x 4096 2.42 / 2.77.
bool few_rows(int bits, int64_t B, int64_t rows, int64_t K)
{
    if (B < 3 || B > (bits == 4 ? 16 : 4) || K <= 2048) return false;
    return rows <= (bits == 4 ? (B <= 4 ? 256 : 384) : bits == 3 || K < 4096 ? 128 : 256);
}

// CTAs per matrix in proportion to the rows, about `grid` in all: at least one each, at
// most one per unit.  Returns their number.
int share_ctas(const GroupArgs& a, int64_t total_rows, const int64_t* units, int grid, int* ctas)
{
    int used = 0;
    for (int i = 0; i < a.count; ++i) {
        int64_t c = (int64_t)grid * a.item[i].N / total_rows;
        if (c < 1) c = 1;
        if (c > units[i]) c = units[i];
        ctas[i] = (int)c;
        used += ctas[i];
    }
    while (used < grid) {               // hand out what rounding left, largest rows per CTA first
        int best = -1;
        double best_load = -1.0;
        for (int i = 0; i < a.count; ++i) {
            if (ctas[i] >= units[i]) continue;
            const double load = (double)a.item[i].N / ctas[i];
            if (load > best_load) { best_load = load; best = i; }
        }
        if (best < 0) break;
        ++ctas[best];
        ++used;
    }
    while (used > grid) {               // too many (minimums): take from the lightest
        int best = -1;
        double best_load = 1e300;
        for (int i = 0; i < a.count; ++i) {
            if (ctas[i] <= 1) continue;
            const double load = (double)a.item[i].N / ctas[i];
            if (load < best_load) { best_load = load; best = i; }
        }
        if (best < 0) break;
        --ctas[best];
        --used;
    }
    return used;
}

// The table lookups address shared memory relative to kTabOff, which is where
// dynamic shared memory starts when a kernel has no static shared memory.
cudaError_t check_shared_base()
{
    static int ok[64] = {0};   // 0 unknown, 1 yes, -1 no
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (ok[dev] == 0) {
        int reserved = -1;
        e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
        if (e != cudaSuccess) return e;
        ok[dev] = (reserved == (int)kTabOff) ? 1 : -1;
    }
    return ok[dev] > 0 ? cudaSuccess : cudaErrorNotSupported;
}

}  // namespace

// Up to 16 rows always (a Llama-3.1-8B layer at 9 / 16 rows, here and in the prefill kernel:
// 4 bits 59.1 / 63.3 and 91.8 / 75.5 us, 3 bits 70.9 / 76.0 and 101 / 94.4, 8 bits 90.9 /
// 92.4 and 103 / 97.0).  17..32 for up to
// 4 M weights in a call: 2048 x 2048 at 17 / 32 rows, 4 bits 5.1 / 6.1 against 6.3 / 6.4,
// 3 bits 5.2 / 6.0 against 6.7, 8 bits 4.7 / 5.2 against 7.3; 3072 x 2048, 4 bits 6.6 /
// 7.6 against 6.4 / 6.6; 4096 x 4096 13.0 / 14.0 against 10.5 / 10.7.
bool gemv_takes(int bits, int64_t B, int64_t rows, int64_t K)
{
    if (bits != 3 && bits != 4 && bits != 8) return false;
    if (B < 1 || B > 32) return false;
    return B <= 16 || rows <= ((int64_t)4 << 20) / K;
}

// Fields that every decode launch shares.
static GemvParams common_params(const GroupArgs& a, int64_t total_rows)
{
    GemvParams p;
    memset(&p, 0, sizeof p);
    p.nitems = a.count;
    p.X = static_cast<const uint16_t*>(a.X);
    p.err = &a.ws->error;
    p.K = (int32_t)a.K;
    p.B = (int32_t)a.B;
    p.y_dtype = a.y_dtype;
    p.wait_codes = reads_codes_early(a.bits, a.B, total_rows * a.K) ? 0 : 1;
    p.row_bytes = (int32_t)(a.K / 32 * (4 * a.bits));
    p.kparts = 1;
    p.pf = static_cast<const uint8_t*>(a.pf);
    p.pf_bytes = (a.pf && a.pf_bytes < kPrefetchBytes) ? a.pf_bytes : 0;
    for (int i = 0; i < a.count; ++i) {
        GemvItem& it = p.item[i];
        it.codes = a.item[i].codes;
        it.Y = a.item[i].Y;
        it.N = (int32_t)a.item[i].N;
        for (int c = 0; c < 16; ++c) it.lvl16[c] = a.item[i].lvl16[c];
    }
    return p;
}

// The launch of few_rows_kernel: warps 8 at batches above 8, else 16, as registers allow.
static cudaError_t launch_few(const GroupArgs& a, int64_t total_rows, cudaStream_t s)
{
    GemvParams p = common_params(a, total_rows);
    const int Bp = a.B <= 4 ? 4 : a.B <= 8 ? 8 : 16, warps = Bp == 16 ? 8 : 16;
    p.spans = (int32_t)((a.K + 32 * few_k(a.bits) - 1) / (32 * few_k(a.bits)));
    while ((warps >> (p.lg_groups + 1)) >= p.spans) ++p.lg_groups;
    p.span_cols = p.spans < (warps >> p.lg_groups) ? p.spans : warps >> p.lg_groups;
    const int sms = sm_count() > 0 ? sm_count() : 148;
    int64_t units[kMaxItems];
    for (int i = 0; i < a.count; ++i) units[i] = a.item[i].N;
    int grid = (int)(total_rows < sms ? total_rows : sms), ctas[kMaxItems] = {0}, begin = 0;
    if (grid < a.count) grid = a.count;
    grid = share_ctas(a, total_rows, units, grid, ctas);
    p.pf_share = p.pf_bytes > 0 ? (((p.pf_bytes + grid - 1) / grid + 15) & ~(int64_t)15) : 0;
    int64_t max_rows = 0;
    for (int i = 0; i < a.count; ++i) {
        GemvItem& it = p.item[i];
        it.cta_begin = begin;
        it.rows_q = (int32_t)(a.item[i].N / ctas[i]);
        it.rows_rem = (int32_t)(a.item[i].N % ctas[i]);
        begin += ctas[i];
        const int64_t rows = it.rows_q + (it.rows_rem ? 1 : 0);
        if (rows > max_rows) max_rows = rows;
    }
    const size_t smem = (size_t)(a.bits == 3 ? 64 : 256) * kTabStride + (size_t)p.spans * max_rows * Bp * 4;
    if (smem > (size_t)kMaxSmem) return cudaErrorNotSupported;
#define LOGQ_FEW(BITS, B, NT) \
    if (a.bits == BITS && Bp == B) \
        return a.x_f16 ? run_few<BITS, B, NT, true>(p, a, grid, smem, s) : run_few<BITS, B, NT, false>(p, a, grid, smem, s)
    LOGQ_FEW(4, 4, 512);
    LOGQ_FEW(4, 8, 512);
    LOGQ_FEW(4, 16, 256);
    LOGQ_FEW(3, 4, 512);
    LOGQ_FEW(8, 4, 512);
#undef LOGQ_FEW
    return cudaErrorInvalidValue;
}

cudaError_t launch_gemv_group(const GroupArgs& a, cudaStream_t s)
{
    if (a.count < 1 || a.count > kMaxItems) return cudaErrorInvalidValue;
    cudaError_t e = check_shared_base();
    if (e != cudaSuccess) return e;
    int64_t total_rows = 0;
    for (int i = 0; i < a.count; ++i) total_rows += a.item[i].N;
    if (few_rows(a.bits, a.B, total_rows, a.K)) {
        e = launch_few(a, total_rows, s);
        if (e != cudaErrorNotSupported) return e;        // (its sums do not fit shared memory)
    }
    const int key = shape_key(a.bits, a.B, total_rows, a.K);
    Shape sh;
    if ((e = shape_or_run<false>(a.bits, key, &sh, nullptr, nullptr, 0, 0, s)) != cudaSuccess) return e;
    GemvParams p = common_params(a, total_rows);
    p.blocks = (int32_t)(a.K / (4 * lane_k(a.bits)));
    p.spans = (p.blocks + sh.S * sh.J - 1) / (sh.S * sh.J);
    // Batches of 9 and more read more activations than codes where a CTA takes
    // several passes over K: with room for partial sums, several CTAs share a row
    // range, one part of the spans each (see the note at kPartBatch).
    const int warps = sh.NT / 32;
    const int passes = (p.spans + warps - 1) / warps;
    int64_t kparts = 1;
    if (a.B >= kPartBatch) {
        const int64_t avail = a.ws_bytes > kWorkspaceBytes ? (int64_t)(a.ws_bytes - kWorkspaceBytes) : 0;
        kparts = avail / (4 * a.B * total_rows);
        if (kparts > kMaxParts) kparts = kMaxParts;
        if (kparts > passes) kparts = passes;
        if (kparts < 1) kparts = 1;
    }
    p.part_spans = (int32_t)((p.spans + kparts - 1) / kparts);
    kparts = (p.spans + p.part_spans - 1) / p.part_spans;
    p.kparts = (int32_t)kparts;
    while ((warps >> (p.lg_groups + 1)) >= p.part_spans) ++p.lg_groups;
    p.span_cols = p.part_spans < (warps >> p.lg_groups) ? p.part_spans : warps >> p.lg_groups;
    // Each matrix's rows are divided among row ranges (kparts CTAs each), in
    // proportion to the rows: at least one range each, at most one per tile.
    const int sms = sm_count() > 0 ? sm_count() : 148;
    const int64_t rt = 16 / sh.S;
    int64_t units[kMaxItems], total_units = 0;
    for (int i = 0; i < a.count; ++i) total_units += (units[i] = (a.item[i].N + rt - 1) / rt);
    const int64_t ranges = (int64_t)sms * per_sm(sh, total_rows * a.K) / kparts;
    int grid = (int)(total_units < ranges ? total_units : ranges);
    if (grid < a.count) grid = a.count;
    int ctas[kMaxItems] = {0};
    const int used = share_ctas(a, total_rows, units, grid, ctas);
    grid = used * (int)kparts;
    p.pf_share = p.pf_bytes > 0 ? (((p.pf_bytes + grid - 1) / grid + 15) & ~(int64_t)15) : 0;
    int64_t max_rows = 0;
    int begin = 0;
    float* part = kparts > 1 ? reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(a.ws) + kWorkspaceBytes) : nullptr;
    for (int i = 0; i < a.count; ++i) {
        GemvItem& it = p.item[i];
        it.cta_begin = begin;
        it.rows_q = (int32_t)(a.item[i].N / ctas[i]);
        it.rows_rem = (int32_t)(a.item[i].N % ctas[i]);
        begin += ctas[i] * (int)kparts;
        it.part = part;
        if (kparts > 1) part += kparts * a.B * a.item[i].N;
        const int64_t rows = it.rows_q + (it.rows_rem ? 1 : 0);
        if (rows > max_rows) max_rows = rows;
    }
    // Partial sums: np sets of one per output, each `pitch` floats from the next.
    // A warp's store covers `run` consecutive outputs of S / 2 sets: a pitch of
    // `run` modulo 32 puts them on different banks.
    const int bc = batch_cols(sh.S, sh.NTL), np = p.span_cols * (sh.S >= 4 ? sh.S / 2 : sh.S);
    const int run = sh.S == 8 ? 2 : sh.S == 4 ? 8 : sh.S == 2 ? 16 : 0;
    const size_t tab = (size_t)(a.bits == 3 ? 64 : 256) * kTabStride;
    const int64_t cap = red_bytes(tab, sh.MINB) / 4;
    auto pitch_for = [&](int64_t rows) { return (rows * bc + 31 - run) / 32 * 32 + run; };
    int64_t chunk = max_rows;
    if (pitch_for(chunk) * np > cap) {
        chunk = (cap / np - 32) / bc;
        const int64_t step = rt << p.lg_groups;                // a tile of every warp
        const int64_t equal = (max_rows + (max_rows + chunk - 1) / chunk - 1) / ((max_rows + chunk - 1) / chunk);
        if (chunk > step) chunk -= chunk % step;
        if ((equal + step - 1) / step * step < chunk) chunk = (equal + step - 1) / step * step;
    }
    if (chunk < 1) return cudaErrorInvalidValue;
    p.chunk_rows = (int32_t)chunk;
    p.pitch = (int32_t)pitch_for(chunk);
    const size_t smem = tab + (size_t)p.pitch * np * 4;
    e = a.x_f16 ? shape_or_run<true>(a.bits, key, &sh, &p, &a, grid, smem, s)
                : shape_or_run<false>(a.bits, key, &sh, &p, &a, grid, smem, s);
    if (e != cudaSuccess || kparts == 1) return e;
    SplitSum sum;
    memset(&sum, 0, sizeof sum);
    sum.n = a.count;
    for (int i = 0; i < a.count; ++i) {
        sum.part[i] = p.item[i].part;
        sum.Y[i] = a.item[i].Y;
        sum.count[i] = a.B * a.item[i].N;
    }
    return launch_split_sum(sum, (int)kparts, a.y_dtype, s);
}

cudaError_t launch_gemv(const LinearArgs& a, cudaStream_t s)
{
    GroupArgs g;
    memset(&g, 0, sizeof g);
    g.count = 1;
    g.item[0].codes = a.codes;
    g.item[0].Y = a.Y;
    g.item[0].N = a.N;
    for (int c = 0; c < 256; ++c) g.item[0].lvl16[c] = a.lvl16[c];
    g.X = a.X;
    g.B = a.B;
    g.K = a.K;
    g.bits = a.bits;
    g.x_f16 = a.x_f16;
    g.y_dtype = a.y_dtype;
    g.ws = a.ws;
    g.ws_bytes = a.ws_bytes;
    return launch_gemv_group(g, s);
}

}  // namespace logq
