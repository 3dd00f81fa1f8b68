// GPTQ with the Log_b quantiser (the calibration the paper runs its
// quantiser in; GPTQ's published procedure, restated).
//
// Factor: Hd = H + damp * mean(diag H) * I (a zero diagonal entry of H, an
// input that never fires, set to 1 first) and U, the upper Cholesky factor of
// Hd^-1 (Hd^-1 = U^T U).  With J the index reversal, let J Hd J = L L^T (lower
// Cholesky).  Then Hd = R R^T with R = J L J upper triangular, Hd^-1 =
// (R^-1)^T R^-1 and R^-1 is upper with a positive diagonal, so U = R^-1 =
// J L^-1 J: one Cholesky factorisation and one triangular inverse, in fp32.
//   - blocked right-looking Cholesky on 64 x 64 blocks: potrf_block factors a
//     diagonal block and replaces it by the inverse of its factor; the panel
//     below becomes L21 = A21 L11^-T and the trailing matrix A22 -= L21 L21^T
//     (both through gptq_rank64_kernel; one CTA of the second updates and factors
//     the next diagonal block while the others update the rest);
//   - the triangular inverse by doubling: with the diagonal blocks already
//     inverted, two neighbouring inverted blocks [A 0; B C] combine to
//     [A^-1 0; -C^-1 B A^-1  C^-1] (two products, batched over all pairs of a
//     level; the triangular operands skip their zero stages);
//   - U is the reversal of L^-1.
//
// Quantise: the columns of W in order; after column j the error
// e = (w_j - level(q_j)) / U_jj is compensated on every later column c by
// w_c -= e * U_jc.  A working copy of W (fp32, [N][K]) in the caller's scratch
// is processed in blocks of 128 columns:
//   gptq_block_kernel: eight lanes per row, lane l holding columns 32 i + 4 l ..
//     + 3 of the row's 128-column slab in registers; the 128 x 128 block of U
//     (zero below the diagonal) in shared memory.  Column by column the lanes
//     take the column's weight from its owner, quantise it (Eq. (1) as
//     m = #{ t : |w| >= thresh[t] }, the boundaries divided among the lanes),
//     form the error and update their registers; rows never synchronise with
//     each other.  The slab's codes are packed at the end and its errors kept
//     (E, [N][128]).
//   the columns after the block, W[:, rest] -= E U[block, rest], through gemm_kernel.
// Every sum has a fixed order, so a run is deterministic.
//
// K = 4096: the factor 7.86 ms with single-buffered 128 x 128 products, a
// two-barriers-per-column diagonal factorisation (60 us a block, alone on the
// GPU) and one warp per row in the column loop, 2.36 ms now; factor and
// quantisation of 4096 rows 11.3 and 4.66 ms.  The fp32 operations (23 G
// multiply-adds in the factor, 34 G in the column updates) take 0.6 and 0.9 ms
// at the FMA rate; the rest is the chain of 64 diagonal blocks and 32 column
// blocks, each waiting for the update before it.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "internal.h"

namespace logq {
namespace {

constexpr int kCols = 128;         // columns per quantisation block (K is a multiple of 128)
constexpr int kRowsPerCta = 16;    // block kernel: eight lanes per row
constexpr int kBlockThreads = 8 * kRowsPerCta;
constexpr int kGK = 16;            // gemm_kernel: terms per shared-memory stage
// Packed pairs of fp32: one instruction for two multiply-adds, each rounded as fmaf.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Programmatic dependent launch: the next kernel of a chain may start as soon as every
// CTA of this one has, and waits itself before it touches what this one reads or
// writes.  The chains here are of 63 x 2 and 32 x 2 kernels of 4-100 us: factor at K =
// 4096 2.45 -> 2.36 ms, with quantisation 4.97 -> 4.66; K = 128 0.15 -> 0.13.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

constexpr int kNb = 64;            // Cholesky block
constexpr size_t kFactorState = 256;   // bytes of factor state ahead of the work matrix

struct GptqTables {
    uint32_t thresh[128];          // fp32 boundaries as bit patterns, 0xffffffff beyond q_max - 1
    float level[128];              // fp32 levels L_0 .. L_qmax
    int32_t bits;
    int32_t qmax;
};

struct FactorState {
    double mean;                   // mean of H's diagonal
    uint32_t not_pd;               // a Cholesky pivot was not positive (or not finite)
};

// Inverse of the Cholesky factor of the 64 x 64 diagonal block at A (lower
// triangle read), written in the block's place with zeros above the diagonal;
// with L, of the block minus L L^T (L its 64 x 64 rows of the last panel, same
// leading dimension).  One CTA of 256 threads; thread (ty, tx) holds the 4 x 4
// elements (ty + 16 i, tx + 16 k) of the block and of a second matrix E (the
// identity at first) in registers.  Elimination step j takes t_ij = a_ij / p times
// row j from the rows i > j of both (p = a_jj): A becomes D L~^T and E the unit
// lower L~^-1 of A = L~ D L~^T, so the factor's inverse is D^-1/2 E.  Four steps go
// in one round of two barriers: the owners of columns j .. j + 3 of A and of rows
// j .. j + 3 of E publish them; 64 threads each carry the four steps out on a row
// of those columns and 64 on a column of those rows, in the order of single steps,
// and publish what each step finds there; then every thread updates its elements.
// What bounds it is this chain of 16 dependent rounds.  The pivots' reciprocals
// are taken of scaled values (sc, exact), so that any positive finite pivot serves.
struct PotrfShared {
    union {
        struct {
            float4 col[kNb];           // [row]: columns j .. j + 3
            float4 row[kNb];           // [column]: rows j .. j + 3 of E
            // per step c, [r % 16][r / 16] as a thread reads its four: multipliers t of the
            // rows, entries of the columns (a_jk = a_kj) and of E's row
            float t[4][16][4], x[4][16][4], e[4][16][4];
        };
        float Lt[kNb][kNb + 4];        // L transposed
    };
    float diag[kNb];
};

__device__ __forceinline__ void potrf_block(float* A, const float* L, int64_t ld, FactorState* st, PotrfShared& sm)
{
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    float a0[4][4], e0[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = ty + 16 * i, c = tx + 16 * k;
            // the upper triangle mirrors the lower one
            a0[i][k] = c <= r ? A[r * ld + c] : A[c * ld + r];
            e0[i][k] = 0.f;
        }
    if (L) {
        for (int i = tid; i < kNb * kNb / 4; i += 256) {
            const int r = i / (kNb / 4), q = i % (kNb / 4);
            const float4 v = *reinterpret_cast<const float4*>(L + r * ld + 4 * q);
            sm.Lt[4 * q + 0][r] = v.x;
            sm.Lt[4 * q + 1][r] = v.y;
            sm.Lt[4 * q + 2][r] = v.z;
            sm.Lt[4 * q + 3][r] = v.w;
        }
        __syncthreads();
#pragma unroll 8
        for (int j = 0; j < kNb; ++j) {
            float lr[4], lc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                lr[i] = sm.Lt[j][ty + 16 * i];
                lc[i] = sm.Lt[j][tx + 16 * i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) e0[i][k] = fmaf(lr[i], lc[k], e0[i][k]);
        }
        __syncthreads();
    }
    f32x2 a[4][2], e[4][2];            // pairs (k, k + 1)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            a[i][k / 2] = pack2(a0[i][k] - e0[i][k], a0[i][k + 1] - e0[i][k + 1]);
            e[i][k / 2] = pack2(ty + 16 * i == tx + 16 * k ? 1.f : 0.f, ty + 16 * i == tx + 16 * (k + 1) ? 1.f : 0.f);
        }
#pragma unroll
    for (int jj = 0; jj < 4; ++jj)
        for (int jm = 0; jm < 16; jm += 4) {
            const int j = 16 * jj + jm;
            if ((tx & ~3) == jm)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float v[2];
                    unpack2(a[i][jj / 2], v[0], v[1]);
                    reinterpret_cast<float*>(&sm.col[ty + 16 * i])[tx - jm] = v[jj % 2];
                }
            if ((ty & ~3) == jm)
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    float v[2];
                    unpack2(e[jj][k / 2], v[0], v[1]);
                    reinterpret_cast<float*>(&sm.row[tx + 16 * k])[ty - jm] = v[0];
                    reinterpret_cast<float*>(&sm.row[tx + 16 * (k + 1)])[ty - jm] = v[1];
                }
            __syncthreads();
            if (tid < 2 * kNb) {
                float d[4][4], rp[4], sc[4], m[4][4];     // d[r][c]: the pivot block at the step of column c; m: its multipliers
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float4 v = sm.col[j + r];
                    d[r][0] = v.x; d[r][1] = v.y; d[r][2] = v.z; d[r][3] = v.w;
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float p = d[c][c];
                    sc[c] = p < 0x1p-64f ? 0x1p64f : p > 0x1p64f ? 0x1p-64f : 1.f;     // keeps 1 / p a normal number
                    rp[c] = 1.f / (p * sc[c]);
                    if (tid == 0) sm.diag[j + c] = p;
#pragma unroll
                    for (int r = c + 1; r < 4; ++r) {
                        m[r][c] = d[r][c] * sc[c] * rp[c];
#pragma unroll
                        for (int q = c + 1; q <= r; ++q) d[r][q] = fmaf(-m[r][c], d[q][c], d[r][q]);
                    }
                }
                const int r = tid % kNb;
                const float4 v = tid < kNb ? sm.col[r] : sm.row[r];
                float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float t[4];
                    if (tid < kNb) {
                        t[c] = r > j + c ? x[c] * sc[c] * rp[c] : 0.f;
                        sm.t[c][r % 16][r / 16] = t[c];
                        sm.x[c][r % 16][r / 16] = x[c];
#pragma unroll
                        for (int q = c + 1; q < 4; ++q) x[q] = fmaf(-t[c], d[q][c], x[q]);
                    } else {
                        sm.e[c][r % 16][r / 16] = x[c];
#pragma unroll
                        for (int q = c + 1; q < 4; ++q) x[q] = fmaf(-m[q][c], x[c], x[q]);
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 tv = *reinterpret_cast<const float4*>(sm.t[c][ty]);
                const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(sm.x[c][tx]);
                const ulonglong2 ev = *reinterpret_cast<const ulonglong2*>(sm.e[c][tx]);
                const float t[4] = {tv.x, tv.y, tv.z, tv.w};
#pragma unroll
                for (int i = jj; i < 4; ++i) {
                    const f32x2 nt = pack2(-t[i], -t[i]);
                    if (jj < 2) a[i][0] = fma2(nt, xv.x, a[i][0]);
                    a[i][1] = fma2(nt, xv.y, a[i][1]);
                    e[i][0] = fma2(nt, ev.x, e[i][0]);
                    if (jj >= 2) e[i][1] = fma2(nt, ev.y, e[i][1]);
                }
            }
        }
    __syncthreads();
    if (tid < kNb && (!(sm.diag[tid] > 0.f) || !isfinite(sm.diag[tid]))) st->not_pd = 1;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            float v[2];
            unpack2(e[i][k / 2], v[0], v[1]);
            const int r = ty + 16 * i, c = tx + 16 * k;
            A[r * ld + c] = c <= r ? v[0] / sqrtf(sm.diag[r]) : 0.f;
            A[r * ld + c + 16] = c + 16 <= r ? v[1] / sqrtf(sm.diag[r]) : 0.f;
        }
}

__global__ void __launch_bounds__(256) gptq_potrf_kernel(float* A, int64_t ld, FactorState* st)
{
    __shared__ PotrfShared sm;
    potrf_block(A, nullptr, ld, st, sm);
}

// C = beta C + alpha A B, A [M][Kd] and B [Kd][N] row-major.  Batched over
// blockIdx.z with element strides sA, sB, sC.  Kd is a multiple of 32; N, the
// leading dimensions and the batch strides are multiples of 4 and the bases
// 16-byte aligned.  TRI_A: A is lower triangular (A[m][k] = 0 for k > m), TRI_B:
// B is lower triangular (B[k][n] = 0 for k < n); the stages that hold only such
// zeros are skipped, the others read the zeros, which must be stored.
struct GemmArgs {
    const float* A;
    const float* B;
    float* C;
    int64_t M, N, Kd;
    int64_t lda, ldb, ldc;
    int64_t sA, sB, sC;
    float alpha, beta;
};

// TM x TN outputs per CTA, RM x 8 per thread.  A warp covers 4 RM rows and 64
// columns, its lanes 4 x 8; a thread's rows are RM / 4 runs of 4 (16 apart), its
// columns two runs of 4 (32 apart), so that a warp's fragment reads are 64
// (rows) and 128 (columns) contiguous bytes.  Both operands are staged k-major
// in two shared-memory buffers of 16 terms: the next stage's loads are in
// flight in registers while one is multiplied, one barrier per stage.  A, which
// arrives k-contiguous, is transposed on the way; its columns are XORed with
// 8 (k / 4 % 4), which keeps the transposed stores (8 rows x 4 runs of k per warp)
// and the fragment reads free of bank conflicts.
// Bound by the fp32 FMA rate; the multiply-adds go in packed pairs, which halves
// the instructions issued for them (the factor at K = 4096 3.7 ms before, 3.2 with
// them and the overlapped diagonal blocks).
// TRI_A takes the rows of tiles with the most terms first, so that the short ones
// fill the last wave; with TRI_B they come first as they are.
template <int TM, int TN, int RM, bool TRI_A, bool TRI_B>
__global__ void __launch_bounds__(TM / RM * TN / 8, 4) gemm_kernel(const __grid_constant__ GemmArgs g)
{
    constexpr int CN = 8;
    constexpr int NT = TM / RM * TN / CN;
    constexpr int WM = TM / (4 * RM);                     // warps along the rows
    constexpr int LA = TM * kGK / 4 / NT, LB = TN * kGK / 4 / NT;   // float4 loads per thread and stage
    static_assert(LA * NT * 4 == TM * kGK && LB * NT * 4 == TN * kGK, "whole loads");
    __shared__ __align__(16) float As[2][kGK][TM];
    __shared__ __align__(16) float Bs[2][kGK][TN];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    int64_t r0 = (int64_t)blockIdx.x * TM, c0 = (int64_t)blockIdx.y * TN;
    if (TRI_A) {          // the longest rows of tiles first
        const unsigned i = blockIdx.x + gridDim.x * blockIdx.y;
        r0 = (int64_t)(gridDim.x - 1 - i / gridDim.y) * TM;
        c0 = (int64_t)(i % gridDim.y) * TN;
    }
    let_next_start();
    wait_for_previous();
    const float* A = g.A + blockIdx.z * g.sA;
    const float* B = g.B + blockIdx.z * g.sB;
    float* C = g.C + blockIdx.z * g.sC;
    int64_t k_begin = 0, k_end = g.Kd;
    if (TRI_B) k_begin = c0 < g.Kd ? c0 / kGK * kGK : g.Kd;
    if (TRI_A && r0 + TM < k_end) k_end = r0 + TM;
    const int m0 = warp % WM * (4 * RM) + lane / 8 * 4, n0 = warp / WM * (8 * CN) + lane % 8 * 4;
    f32x2 acc2[RM][CN / 2];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int k = 0; k < CN / 2; ++k) acc2[i][k] = 0;
    float4 la[LA], lb[LB];
    auto fetch = [&](int64_t k0) {
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int f = tid + i * NT, rr = f / (kGK / 4), q = f % (kGK / 4);
            la[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r0 + rr < g.M) la[i] = *reinterpret_cast<const float4*>(A + (r0 + rr) * g.lda + k0 + 4 * q);
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int f = tid + i * NT;
            lb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int a = f / (TN / 4), q = f % (TN / 4);
            if (c0 + 4 * q < g.N) lb[i] = *reinterpret_cast<const float4*>(B + (k0 + a) * g.ldb + c0 + 4 * q);
        }
    };
    auto stage = [&](int s) {
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int f = tid + i * NT, q = f % (kGK / 4), at = (f / (kGK / 4)) ^ (8 * q);
            As[s][4 * q + 0][at] = la[i].x;
            As[s][4 * q + 1][at] = la[i].y;
            As[s][4 * q + 2][at] = la[i].z;
            As[s][4 * q + 3][at] = la[i].w;
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int f = tid + i * NT;
            *reinterpret_cast<float4*>(&Bs[s][f / (TN / 4)][4 * (f % (TN / 4))]) = lb[i];
        }
    };
    auto multiply = [&](int s) {
#pragma unroll
        for (int a = 0; a < kGK; ++a) {
            const int swz = 8 * (a / 4);
            f32x2 ev[RM], uv[CN / 2];
#pragma unroll
            for (int i = 0; i < RM; i += 4) {
                const float4 e = *reinterpret_cast<const float4*>(&As[s][a][(m0 + 4 * i) ^ swz]);
                ev[i] = pack2(e.x, e.x); ev[i + 1] = pack2(e.y, e.y);
                ev[i + 2] = pack2(e.z, e.z); ev[i + 3] = pack2(e.w, e.w);
            }
#pragma unroll
            for (int k = 0; k < CN; k += 4) {
                const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(&Bs[s][a][n0 + 8 * k]);
                uv[k / 2] = u.x; uv[k / 2 + 1] = u.y;
            }
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int k = 0; k < CN / 2; ++k) acc2[i][k] = fma2(ev[i], uv[k], acc2[i][k]);
        }
    };
    if (k_begin < k_end) {
        fetch(k_begin);
        stage(0);
        __syncthreads();
        int s = 0;
        for (int64_t k0 = k_begin; k0 < k_end; k0 += kGK, s ^= 1) {
            const bool more = k0 + kGK < k_end;
            if (more) fetch(k0 + kGK);
            multiply(s);
            if (more) stage(s ^ 1);
            __syncthreads();
        }
    }
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int64_t rr = r0 + m0 + (i / 4) * 16 + i % 4;
        if (rr >= g.M) continue;
        float acc[CN];
#pragma unroll
        for (int k = 0; k < CN / 2; ++k) unpack2(acc2[i][k], acc[2 * k], acc[2 * k + 1]);
#pragma unroll
        for (int h = 0; h < CN / 4; ++h) {
            const int64_t c = c0 + n0 + 32 * h;
            if (c >= g.N) continue;
            float4* p = reinterpret_cast<float4*>(C + rr * g.ldc + c);
            float4 o;
            if (g.beta == 0.f) {
                o = make_float4(g.alpha * acc[4 * h + 0], g.alpha * acc[4 * h + 1],
                                g.alpha * acc[4 * h + 2], g.alpha * acc[4 * h + 3]);
            } else {
                o = *p;
                o.x = g.beta * o.x + g.alpha * acc[4 * h + 0];
                o.y = g.beta * o.y + g.alpha * acc[4 * h + 1];
                o.z = g.beta * o.z + g.alpha * acc[4 * h + 2];
                o.w = g.beta * o.w + g.alpha * acc[4 * h + 3];
            }
            *p = o;
        }
    }
}

// Products of the Cholesky steps, 64 terms long: C -= A B^T (UPDATE) or C = A B^T with
// A [.][64] and B [.][64] of one leading dimension, TM x 64 outputs per CTA, 4 x 4 per
// thread.  Everything a CTA reads is requested at once (one trip to L2 instead of
// one per stage of 16 terms), then multiplied out of shared memory (layout as in
// gemm_kernel); sizes are multiples of the tile.
//   UPDATE: the trailing matrix's tiles on and below the diagonal, numbered row by
//     row.  The first, the next diagonal block, is factored by its CTA while the
//     others compute.  4032 rows: 47 us with 128 x 128 tiles of four stages.
//   otherwise the panel below a diagonal block, one row of tiles (C may be A).
template <int TM, bool UPDATE>
__global__ void __launch_bounds__(4 * TM, UPDATE ? 3 : 4) gptq_rank64_kernel(const float* A, const float* B, float* C,
                                                                             int64_t ld,
                                                                             FactorState* st)
{
    constexpr int NT = 4 * TM, WM = TM / 16;
    constexpr int LB = kNb * 16 / NT;                     // float4 loads of B per thread (4 of A)
    __shared__ __align__(16) unsigned char smem[sizeof(PotrfShared) > kNb * (TM + kNb) * sizeof(float) && UPDATE
                                                    ? sizeof(PotrfShared) : kNb * (TM + kNb) * sizeof(float)];
    auto& As = *reinterpret_cast<float (*)[kNb][TM]>(smem);
    auto& Bs = *reinterpret_cast<float (*)[kNb][kNb]>(smem + kNb * TM * sizeof(float));
    int64_t r0 = (int64_t)blockIdx.x * TM, c0 = 0;
    let_next_start();
    wait_for_previous();
    if constexpr (UPDATE) {
        static_assert(NT == 256, "the diagonal block's factorisation takes 256 threads");
        if (blockIdx.x == 0) return potrf_block(C, A, ld, st, *reinterpret_cast<PotrfShared*>(smem));
        // tile number = row (row + 1) / 2 + column
        int64_t row = (int64_t)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
        while (row * (row + 1) / 2 > blockIdx.x) --row;
        while ((row + 1) * (row + 2) / 2 <= blockIdx.x) ++row;
        r0 = row * TM;
        c0 = (blockIdx.x - row * (row + 1) / 2) * kNb;
    }
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int m0 = warp % WM * 16 + lane / 8 * 4, n0 = warp / WM * 32 + lane % 8 * 4;
    // a load's row and run of four k: 8 rows x 4 runs per warp
    float4 la[4], lb[LB], o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int f = tid + i * NT;
        la[i] = *reinterpret_cast<const float4*>(A + (r0 + f / 4 % TM) * ld + 4 * (f % 4 + 4 * (f / (4 * TM))));
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
        const int f = tid + i * NT;
        lb[i] = *reinterpret_cast<const float4*>(B + (c0 + f / 4 % kNb) * ld + 4 * (f % 4 + 4 * (f / (4 * kNb))));
    }
    float* c = C + (r0 + m0) * ld + c0 + n0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (UPDATE) o[i] = *reinterpret_cast<const float4*>(c + i * ld);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int f = tid + i * NT, q = f % 4 + 4 * (f / (4 * TM)), at = (f / 4 % TM) ^ (8 * (q % 4));
        As[4 * q + 0][at] = la[i].x;
        As[4 * q + 1][at] = la[i].y;
        As[4 * q + 2][at] = la[i].z;
        As[4 * q + 3][at] = la[i].w;
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
        const int f = tid + i * NT, q = f % 4 + 4 * (f / (4 * kNb)), at = (f / 4 % kNb) ^ (8 * (q % 4));
        Bs[4 * q + 0][at] = lb[i].x;
        Bs[4 * q + 1][at] = lb[i].y;
        Bs[4 * q + 2][at] = lb[i].z;
        Bs[4 * q + 3][at] = lb[i].w;
    }
    __syncthreads();
    f32x2 acc[4][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
#pragma unroll 16
    for (int a = 0; a < kNb; ++a) {
        const int swz = 8 * (a / 4 % 4);
        const float4 e = *reinterpret_cast<const float4*>(&As[a][m0 ^ swz]);
        const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(&Bs[a][n0 ^ swz]);
        const f32x2 ev[4] = {pack2(e.x, e.x), pack2(e.y, e.y), pack2(e.z, e.z), pack2(e.w, e.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i][0] = fma2(ev[i], u.x, acc[i][0]);
            acc[i][1] = fma2(ev[i], u.y, acc[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float v[4];
        unpack2(acc[i][0], v[0], v[1]);
        unpack2(acc[i][1], v[2], v[3]);
        if constexpr (UPDATE)
            *reinterpret_cast<float4*>(c + i * ld) = make_float4(o[i].x - v[0], o[i].y - v[1],
                                                                 o[i].z - v[2], o[i].w - v[3]);
        else
            *reinterpret_cast<float4*>(c + i * ld) = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// mean(diag H) in fp64 (fixed order: strided partial sums, then a tree) and
// the dead-input mask.  One CTA of 1024 threads.
__global__ void __launch_bounds__(1024) gptq_diag_kernel(const float* __restrict__ H, int64_t K,
                                                         FactorState* st, uint8_t* __restrict__ dead)
{
    __shared__ double part[1024];
    const int tid = threadIdx.x;
    double s = 0.0;
    for (int64_t j = tid; j < K; j += 1024) {
        const float h = H[j * K + j];
        s += (double)h;
        if (dead) dead[j] = h == 0.f;
    }
    part[tid] = s;
    __syncthreads();
    for (int w = 512; w >= 1; w >>= 1) {
        if (tid < w) part[tid] += part[tid + w];
        __syncthreads();
    }
    if (tid == 0) {
        st->mean = part[0] / (double)K;
        st->not_pd = 0;
    }
}

// A = J Hd J (rows and columns reversed), damping on the diagonal; zeros above
// it, which the triangular products read.  One row per blockIdx.y step.
__global__ void __launch_bounds__(256) gptq_prep_kernel(const float* __restrict__ H, int64_t K, double damp,
                                                        const FactorState* st, float* __restrict__ A)
{
    const double add = damp * st->mean;
    for (int64_t i = blockIdx.y; i < K; i += gridDim.y) {
        const float* h = H + (K - 1 - i) * K;
        for (int64_t j = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); j < K; j += 4 * (int64_t)gridDim.x * blockDim.x) {
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j <= i) {
                const float4 v = *reinterpret_cast<const float4*>(h + K - 4 - j);
                const float r[4] = {v.w, v.z, v.y, v.x};
                float w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    w[e] = j + e <= i ? r[e] : 0.f;
                    if (j + e == i) w[e] = (float)((r[e] == 0.f ? 1.0 : (double)r[e]) + add);
                }
                o = make_float4(w[0], w[1], w[2], w[3]);
            }
            *reinterpret_cast<float4*>(A + i * K + j) = o;
        }
    }
}

// U[i][j] = Linv[K-1-i][K-1-j] (upper triangular; zeros below the diagonal).
__global__ void __launch_bounds__(256) gptq_reverse_kernel(const float* __restrict__ Li, int64_t K, float* __restrict__ U)
{
    for (int64_t i = blockIdx.y; i < K; i += gridDim.y) {
        const float* l = Li + (K - 1 - i) * K;
        for (int64_t j = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); j < K; j += 4 * (int64_t)gridDim.x * blockDim.x) {
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j + 3 >= i) {
                const float4 v = *reinterpret_cast<const float4*>(l + K - 4 - j);
                o = make_float4(j >= i ? v.w : 0.f, j + 1 >= i ? v.z : 0.f, j + 2 >= i ? v.y : 0.f, v.x);
            }
            *reinterpret_cast<float4*>(U + i * K + j) = o;
        }
    }
}

// Working copy of W with the dead inputs' columns zeroed.
__global__ void gptq_copy_kernel(const float4* __restrict__ W, int64_t n4, int64_t K4,
                                 const uint8_t* __restrict__ dead, float4* __restrict__ Wk)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        float4 v = W[i];
        const int64_t c = 4 * (i % K4);
        if (dead[c + 0]) v.x = 0.f;
        if (dead[c + 1]) v.y = 0.f;
        if (dead[c + 2]) v.z = 0.f;
        if (dead[c + 3]) v.w = 0.f;
        Wk[i] = v;
    }
}

// Bound by the chain of 128 columns (shuffle, compare, divide, update): eight lanes
// per row put four rows into a warp, which shares that chain's instructions among
// them (4096 rows: 24 us a block; one warp per row 30 us).
template <int BITS>
__global__ void __launch_bounds__(kBlockThreads, 3) gptq_block_kernel(float* __restrict__ Wk, int64_t N, int64_t K,
                                                                      const float* __restrict__ U, int64_t j0,
                                                                      const __grid_constant__ GptqTables tb,
                                                                      uint8_t* __restrict__ codes,
                                                                      float* __restrict__ E)
{
    constexpr int kTh = BITS == 8 ? 16 : 1;        // boundaries per lane: 127 or 7 over 8 lanes
    extern __shared__ float4 sm4[];
    float* Ub = reinterpret_cast<float*>(sm4);     // [kCols][kCols], upper triangle of U's block
    __shared__ float lv[128];
    const int tid = threadIdx.x, lane = tid % 32, l8 = lane % 8, base = lane & 24;
    // not from the last block: what follows the call may read codes before it waits,
    // as the linear kernels do
    if (j0 + kCols < K) let_next_start();
    const int64_t r = (int64_t)blockIdx.x * kRowsPerCta + tid / 8;
    if (tid < 128) lv[tid] = tb.level[tid];
    for (int i = tid; i < kCols * kCols / 4; i += kBlockThreads) {
        const int a = i / (kCols / 4), c = 4 * (i % (kCols / 4));
        float4 v = *reinterpret_cast<const float4*>(U + (j0 + a) * K + j0 + c);
        if (c + 0 < a) v.x = 0.f;
        if (c + 1 < a) v.y = 0.f;
        if (c + 2 < a) v.z = 0.f;
        if (c + 3 < a) v.w = 0.f;
        sm4[i] = v;
    }
    uint32_t th[kTh];
#pragma unroll
    for (int b = 0; b < kTh; ++b) th[b] = tb.thresh[l8 + 8 * b];
    wait_for_previous();                           // the update of these columns (U's block is not its output)
    // rows past the end repeat the last one (whole warps take part in the shuffles)
    const int64_t rr = r < N ? r : N - 1;
    f32x2 wv[4][2];                                // this lane's columns 32 i + 4 l8 .. + 3, in pairs
    float ev[4][4];
    uint32_t cv[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const ulonglong2 w4 = *reinterpret_cast<const ulonglong2*>(Wk + rr * K + j0 + 32 * i + 4 * l8);
        wv[i][0] = w4.x; wv[i][1] = w4.y;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
        for (int o = 0; o < 8; ++o)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = 32 * i + 4 * o + k;
                float w0, w1;
                unpack2(wv[i][k / 2], w0, w1);
                const float w = __shfl_sync(0xffffffffu, k % 2 ? w1 : w0, base + o);
                const uint32_t u = __float_as_uint(w) & 0x7fffffffu;
                int m;
                if constexpr (BITS == 4) {
                    m = __popc((__ballot_sync(0xffffffffu, u >= th[0]) >> base) & 0xffu);
                } else {
                    m = 0;
#pragma unroll
                    for (int b = 0; b < kTh; ++b) m += u >= th[b] ? 1 : 0;
                    m += __shfl_xor_sync(0xffffffffu, m, 1);
                    m += __shfl_xor_sync(0xffffffffu, m, 2);
                    m += __shfl_xor_sync(0xffffffffu, m, 4);
                }
                const float deq = m ? (w < 0.f ? -lv[m] : lv[m]) : 0.f;
                const float e = (w - deq) / Ub[j * kCols + j];
                if (l8 == o) {
                    cv[i][k] = w < 0.f && m ? (uint32_t)m | (1u << (BITS - 1)) : (uint32_t)m;
                    ev[i][k] = e;
                }
                const f32x2 ne = pack2(-e, -e);
                // the columns of earlier runs are done (U is zero there)
#pragma unroll
                for (int h = i; h < 4; ++h) {
                    const ulonglong2 u4 = *reinterpret_cast<const ulonglong2*>(&sm4[(j * kCols) / 4 + l8 + 8 * h]);
                    wv[h][0] = fma2(ne, u4.x, wv[h][0]);
                    wv[h][1] = fma2(ne, u4.y, wv[h][1]);
                }
            }
    if (r >= N) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float4*>(E + r * kCols + 32 * i + 4 * l8) = make_float4(ev[i][0], ev[i][1], ev[i][2], ev[i][3]);
        // sign-magnitude codes (the layout of include/logq.h)
        const uint32_t (&c)[4] = cv[i];
        if constexpr (BITS == 4)
            *reinterpret_cast<uint16_t*>(codes + r * (K / 2) + j0 / 2 + 16 * i + 2 * l8) =
                (uint16_t)(c[0] | (c[1] << 4) | (c[2] << 8) | (c[3] << 12));
        else
            *reinterpret_cast<uint32_t*>(codes + r * K + j0 + 32 * i + 4 * l8) =
                c[0] | (c[1] << 8) | (c[2] << 16) | (c[3] << 24);
    }
}

constexpr size_t kBlockSmem = sizeof(float) * kCols * kCols;

template <int BITS>
cudaError_t block_launch(float* Wk, int64_t N, int64_t K, const float* U, int64_t j0, const GptqTables& tb,
                         uint8_t* codes, float* E, cudaStream_t s)
{
    static int configured[64] = {0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(gptq_block_kernel<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBlockSmem);
        if (e != cudaSuccess) return e;
        configured[dev] = 1;
    }
    const unsigned grid = (unsigned)((N + kRowsPerCta - 1) / kRowsPerCta);
    return launch_chained(gptq_block_kernel<BITS>, dim3(grid), kBlockThreads, kBlockSmem, s, Wk, N, K, U, j0, tb, codes, E);
}

template <int TM, int TN, int RM, bool TRI_A, bool TRI_B>
cudaError_t gemm_tiles(const GemmArgs& g, int64_t batch, cudaStream_t s)
{
    const dim3 grid((unsigned)((g.M + TM - 1) / TM), (unsigned)((g.N + TN - 1) / TN), (unsigned)batch);
    return launch_chained(gemm_kernel<TM, TN, RM, TRI_A, TRI_B>, grid, TM / RM * TN / 8, 0, s, g);
}

// Tile of a product: 32 x 64 for 64 columns; 64 x 64 while 128 x 128 tiles would
// number less than two per SM; 64 x 128 beyond that (the column updates of K and
// rows 4096, whole call: 128 x 256 tiles, one CTA per SM, 5.70 ms, 128 x 128, two,
// 5.35, 64 x 128, four, 5.16).
template <bool TRI_A, bool TRI_B>
cudaError_t gemm(const GemmArgs& g, int64_t batch, cudaStream_t s)
{
    if (g.M <= 0 || g.N <= 0 || batch <= 0) return cudaSuccess;
    const int sms = sm_count() > 0 ? sm_count() : 148;
    const int64_t tiles = ((g.M + 127) / 128) * ((g.N + 127) / 128) * batch;
    if (g.N <= 64) return gemm_tiles<32, 64, 4, TRI_A, TRI_B>(g, batch, s);
    if (tiles < 2 * sms) return gemm_tiles<64, 64, 4, TRI_A, TRI_B>(g, batch, s);
    return gemm_tiles<64, 128, 8, TRI_A, TRI_B>(g, batch, s);
}

GemmArgs gemm_args(const float* A, int64_t lda, const float* B, int64_t ldb, float* C, int64_t ldc, int64_t M,
                   int64_t N, int64_t Kd, float alpha, float beta)
{
    GemmArgs g;
    memset(&g, 0, sizeof g);
    g.A = A;
    g.B = B;
    g.C = C;
    g.M = M;
    g.N = N;
    g.Kd = Kd;
    g.lda = lda;
    g.ldb = ldb;
    g.ldc = ldc;
    g.alpha = alpha;
    g.beta = beta;
    return g;
}

// One row of a K x K matrix per blockIdx.y step, four elements per thread.
dim3 row_grid(int64_t K) { return dim3((unsigned)((K + 1023) / 1024), (unsigned)(K < 4096 ? K : 4096)); }

unsigned elementwise_grid(int64_t n)
{
    const int64_t b = (n + 255) / 256;
    return (unsigned)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

// Two neighbouring inverted diagonal blocks -> their combined inverse, for the
// pairs p = p0 .. p0 + count - 1 of one level (top block at p s, `half` rows;
// bottom block of c rows below it).
cudaError_t combine_pairs(float* Lw, int64_t K, int64_t s_, int64_t half, int64_t c, int64_t p0, int64_t count,
                          float* X, cudaStream_t st)
{
    const int64_t t0 = p0 * s_, b0 = t0 + half;
    // X_p = B_p A_p^-1 (A_p^-1 lower triangular)
    GemmArgs g = gemm_args(Lw + b0 * K + t0, K, Lw + t0 * K + t0, K, X, half, c, half, half, 1.f, 0.f);
    g.sA = s_ * K + s_;
    g.sB = s_ * K + s_;
    g.sC = c * half;
    cudaError_t e = gemm<false, true>(g, count, st);
    if (e != cudaSuccess) return e;
    // block (bottom, top) = -C_p^-1 X_p (C_p^-1 lower triangular)
    g = gemm_args(Lw + b0 * K + b0, K, X, half, Lw + b0 * K + t0, K, c, half, c, -1.f, 0.f);
    g.sA = s_ * K + s_;
    g.sB = c * half;
    g.sC = s_ * K + s_;
    return gemm<true, false>(g, count, st);
}

}  // namespace

size_t gptq_factor_scratch_bytes(int64_t K)
{
    return kFactorState + (size_t)(K * K + K * K / 4) * sizeof(float);
}

cudaError_t launch_gptq_factor(const float* H, int64_t K, double damp, float* U, uint8_t* dead, void* scratch,
                               uint32_t* not_pd, cudaStream_t s)
{
    FactorState* st = static_cast<FactorState*>(scratch);
    float* Lw = reinterpret_cast<float*>(static_cast<char*>(scratch) + kFactorState);
    float* X = Lw + K * K;
    gptq_diag_kernel<<<1, 1024, 0, s>>>(H, K, st, dead);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    gptq_prep_kernel<<<row_grid(K), 256, 0, s>>>(H, K, damp, st, Lw);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // Cholesky of J Hd J; diagonal blocks end up inverted
    gptq_potrf_kernel<<<1, 256, 0, s>>>(Lw, K, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int64_t k0 = 0; k0 < K; k0 += kNb) {
        const int64_t k1 = k0 + kNb, m = K - k1;
        if (m <= 0) break;
        // L21 = A21 L11^-T, in place
        float *L11 = Lw + k0 * K + k0, *L21 = Lw + k1 * K + k0, *A22 = Lw + k1 * K + k1;
        e = launch_chained(gptq_rank64_kernel<32, false>, dim3((unsigned)(m / 32)), 128, 0, s, L21, L11, L21, K, st);
        if (e != cudaSuccess) return e;
        // A22 -= L21 L21^T (lower triangle), and the inverse factor of its first block
        const int64_t t = m / kNb;
        e = launch_chained(gptq_rank64_kernel<64, true>, dim3((unsigned)(t * (t + 1) / 2)), 256, 0, s, L21, L21, A22, K, st);
        if (e != cudaSuccess) return e;
    }
    // triangular inverse by doubling
    for (int64_t half = kNb; half < K; half *= 2) {
        const int64_t s_ = 2 * half;
        const int64_t full = K / s_;                    // pairs whose bottom block is complete
        if (full > 0 && (e = combine_pairs(Lw, K, s_, half, half, 0, full, X, s)) != cudaSuccess) return e;
        const int64_t b0 = full * s_ + half;           // a last pair with a shorter bottom block
        if (b0 < K && (e = combine_pairs(Lw, K, s_, half, K - b0, full, 1, X + full * half * half, s)) != cudaSuccess)
            return e;
    }
    gptq_reverse_kernel<<<row_grid(K), 256, 0, s>>>(Lw, K, U);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (not_pd) {
        e = cudaMemcpyAsync(not_pd, &st->not_pd, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return e;
        e = cudaStreamSynchronize(s);
    }
    return e;
}

size_t gptq_scratch_bytes(int64_t N, int64_t K)
{
    return (size_t)(N * K + N * kCols) * sizeof(float);
}

cudaError_t launch_gptq(const float* W, int64_t N, int64_t K, const float* U, const uint8_t* dead, int bits,
                        const float* thresh, const float* level, int qmax, uint8_t* codes, void* scratch,
                        cudaStream_t s)
{
    GptqTables tb;
    memset(&tb, 0, sizeof tb);
    for (int t = 0; t < 128; ++t) {
        uint32_t b = 0xffffffffu;              // above every |w| bit pattern: m never exceeds q_max
        if (t < qmax) memcpy(&b, &thresh[t], 4);
        tb.thresh[t] = b;
        tb.level[t] = t <= qmax ? level[t] : 0.f;
    }
    tb.bits = bits;
    tb.qmax = qmax;
    float* Wk = static_cast<float*>(scratch);
    float* E = Wk + N * K;
    cudaError_t e;
    if (dead) {
        const int64_t n4 = N * K / 4;
        gptq_copy_kernel<<<elementwise_grid(n4), 256, 0, s>>>(reinterpret_cast<const float4*>(W), n4, K / 4, dead,
                                                             reinterpret_cast<float4*>(Wk));
        e = cudaGetLastError();
    } else {
        e = cudaMemcpyAsync(Wk, W, sizeof(float) * (size_t)(N * K), cudaMemcpyDeviceToDevice, s);
    }
    if (e != cudaSuccess) return e;
    for (int64_t j0 = 0; j0 < K; j0 += kCols) {
        e = bits == 8 ? block_launch<8>(Wk, N, K, U, j0, tb, codes, E, s)
                      : block_launch<4>(Wk, N, K, U, j0, tb, codes, E, s);
        if (e != cudaSuccess) return e;
        const int64_t c1 = j0 + kCols;
        if (c1 < K) {   // W[:, c1:] -= E U[j0:c1, c1:]
            e = gemm<false, false>(
                gemm_args(E, kCols, U + j0 * K + c1, K, Wk + c1, K, N, K - c1, kCols, -1.f, 1.f), 1, s);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace logq
