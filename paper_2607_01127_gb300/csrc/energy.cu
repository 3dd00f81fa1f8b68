// Energy-based effective range (paper Sec. 3.2, Eq. (5)): the smallest data
// value t with  sum_{|w_i| <= t} w_i^2  >=  eps * sum_i w_i^2,  and w_max = max |w_i|.
//
// w_min is an order statistic, so it is found by a radix selection over the
// 31-bit pattern u = bits(|w|) (non-negative floats order like their bit
// patterns), three streaming passes over W, one CTA scanning the sums after each:
//   1: energy per exponent u >> 23; also w_max and the non-finite flag;
//   2: within the selected exponent, how many weights share (u >> 11) & 0xfff;
//      their energies lie between the counts times the buckets' ends squared,
//      which leaves a window of a few buckets for the crossing;
//   3: the exact energy of the selected exponent's weights below that window, and
//      how many weights have each value inside it.
// Every value of an exponent e has w^2 = m^2 * 2^(2e - 46) with m the 24-bit
// significand, so energies are kept exactly as integer sums of m^2 (high and low
// 24 bits apart) and counts; only the scans' accumulation across buckets rounds
// (fp64, ascending order of |w|).
//
// The passes read 235 MB for a 14336 x 4096 matrix, 35 us at the measured HBM
// rate; every other pass runs from the end to the start, so that what the pass
// before it left in L2 is read from there.
//   Pass 1: each lane adds its values' m^2 to its own 64-bit cells in shared
//     memory, one per exponent of a 32-exponent window (no collectives, no atomics).
//     Each warp places its window at its CTA's first values and moves it up when it
//     meets a larger exponent.  Values below it are added to the window's first
//     exponent, in whole units of that one's m^2.  The crossing lies above: it holds
//     at least eps of the energy, so for eps >= n 2^-50 (n weights) its exponent is at
//     most 26 below w_max's, a window's start at least 30; and what is cut off, below
//     2^-106 of the total energy per value, is below 2^-56 of what it is compared with.
//     For a smaller eps they are added one by one, with atomics (EXACT).  A cell is
//     folded into registers before 2^16 values (each m^2 < 2^48) could overflow it.
//     14336 x 4096 with 5 % of the rows 1e-14 of the others: 301 us the whole call; 1642
//     with a window that stays at the CTA's first values and atomics for all others.
//   Pass 2: 4096 counts with native 32-bit shared-memory atomics, for the weights
//     of one exponent.
//   Pass 3: registers, and shared-memory atomics for the few weights inside the
//     window.
// When the window does not fit (kWinBuckets), which takes a distribution whose
// crossing lies in a nearly empty stretch above most of its exponent's weights (or
// for 2^32 weights and more), `failed` is set or energy_counts_fit is false, and the
// caller runs the exact form of levels 2 and 3 (energy_hist_kernel): per-bucket energies
// with 64-bit atomics, 4096 sub-buckets and then 2048 single values.
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace logq {
namespace {

constexpr int kHistThreads = 256;
constexpr int kScanThreads = 256;
constexpr int kUnroll = 4;                       // float4 loads in flight per thread

template <int LEVEL> struct Level;
template <> struct Level<1> { static constexpr int NB = 256; };
template <> struct Level<2> { static constexpr int NB = 4096; };
template <> struct Level<3> { static constexpr int NB = 2048; };
static_assert(sizeof(EnergyState::hi) / sizeof(EnergyState::hi[0]) >= 4096, "bucket arrays");

__device__ __forceinline__ float4 ld_stream4(const float4* p)
{
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}

// m^2 of a finite |w| pattern, split into its high and low 24 bits.
__device__ __forceinline__ void msq_parts(uint32_t u, uint32_t& hi, uint32_t& lo)
{
    const uint32_t mant = u & 0x7fffffu;
    const uint32_t m = (u >> 23) ? (mant | 0x800000u) : mant;      // subnormals: no implicit bit
    const unsigned long long sq = (unsigned long long)m * m;         // < 2^48
    hi = (uint32_t)(sq >> 24);
    lo = (uint32_t)(sq & 0xffffffull);
}

template <int LEVEL>
__device__ __forceinline__ void add_one(uint32_t u, uint32_t prefix, unsigned long long* hi,
                                        unsigned long long* lo)
{
    const bool in = u < 0x7f800000u && (LEVEL == 2 ? (u >> 23) == prefix : (u >> 11) == prefix);
    if (!in) return;
    const uint32_t b = LEVEL == 2 ? ((u >> 11) & 0xfffu) : (u & 0x7ffu);
    uint32_t h, l;
    msq_parts(u, h, l);
    if (h | l) {
        atomicAdd(&hi[b], (unsigned long long)h);
        atomicAdd(&lo[b], (unsigned long long)l);
    }
}

// Streams W in the grid's strides: kUnroll loads in flight per thread in whole
// rounds (their number goes to take with each vector; whole warps take part),
// then the rest (-1); from the end to the start when BACK.
template <bool BACK, typename Take>
__device__ __forceinline__ void stream(const float4* __restrict__ W, int64_t n4, Take&& take)
{
    const int64_t nthreads = (int64_t)gridDim.x * kHistThreads;
    const int64_t gtid = (int64_t)blockIdx.x * kHistThreads + threadIdx.x;
    const int64_t rounds = n4 / (nthreads * kUnroll);
    for (int64_t r = 0; r < rounds; ++r) {
        const int64_t base = r * nthreads * kUnroll + gtid;
        float4 v[kUnroll];
#pragma unroll
        for (int j = 0; j < kUnroll; ++j) {
            const int64_t i = base + j * nthreads;
            v[j] = ld_stream4(W + (BACK ? n4 - 1 - i : i));
        }
#pragma unroll
        for (int j = 0; j < kUnroll; ++j) take(v[j], r);
    }
    for (int64_t i = rounds * nthreads * kUnroll + gtid; i < n4; i += nthreads)
        take(ld_stream4(W + (BACK ? n4 - 1 - i : i)), (int64_t)-1);
}

// Exact levels 2 and 3 (see the top of the file).
template <int LEVEL>
__global__ void __launch_bounds__(kHistThreads) energy_hist_kernel(const float4* __restrict__ W, int64_t n4,
                                                                   EnergyState* st)
{
    constexpr int NB = Level<LEVEL>::NB;
    extern __shared__ unsigned long long hist[];              // [2][NB]
    for (int i = threadIdx.x; i < 2 * NB; i += kHistThreads) hist[i] = 0;
    __syncthreads();
    unsigned long long *hi = hist, *lo = hist + NB;
    const uint32_t prefix = st->prefix;
    stream<LEVEL == 3>(W, n4, [&](const float4& v, int64_t) {
        add_one<LEVEL>(__float_as_uint(v.x) & 0x7fffffffu, prefix, hi, lo);
        add_one<LEVEL>(__float_as_uint(v.y) & 0x7fffffffu, prefix, hi, lo);
        add_one<LEVEL>(__float_as_uint(v.z) & 0x7fffffffu, prefix, hi, lo);
        add_one<LEVEL>(__float_as_uint(v.w) & 0x7fffffffu, prefix, hi, lo);
    });
    __syncthreads();
    for (int i = threadIdx.x; i < NB; i += kHistThreads) {
        if (hi[i]) atomicAdd(&st->hi[i], hi[i]);
        if (lo[i]) atomicAdd(&st->lo[i], lo[i]);
    }
}

// 2^k as a double (normal range: k in [-1022, 1023]).
__device__ __forceinline__ double pow2(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }

constexpr int kWin = 32;                      // pass 1: exponents of a CTA's window
constexpr int64_t kFoldRounds = 2048;         // rounds between folds: 2048 x 16 values per lane < 2^16
constexpr int kWinBuckets = 7;                // pass 3: buckets of the window
constexpr int kWinValues = kWinBuckets * 2048;
static_assert(kWinValues % (4 * kScanThreads) == 0, "whole vectors per scanning thread");
constexpr int kBelowHi = 4094, kBelowLo = 4095;   // lo[] slots of pass 3's energy below the window
static_assert(kWinValues * 4 <= 8 * (4096 + 4094), "window counts share the bucket arrays");

// First exponent of a window that reaches up to exponent top.
__device__ __forceinline__ uint32_t window_start(uint32_t top) { return top > kWin ? top - (kWin - 1) : 1u; }

// Pass 1 (see the top of the file).  EXACT: values below a window one by one.
template <bool EXACT>
__global__ void __launch_bounds__(kHistThreads) energy_exponents_kernel(const float4* __restrict__ W, int64_t n4,
                                                                        EnergyState* st, Workspace* ws)
{
    extern __shared__ unsigned long long cells[];     // [warp][kWin][32 lanes]: sums of m^2
    __shared__ unsigned long long shi[256], slo[256];
    __shared__ uint32_t smax;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long* ce = cells + warp * kWin * 32 + lane;
    for (int b = 0; b < kWin; ++b) ce[b * 32] = 0;
    for (int i = threadIdx.x; i < 256; i += kHistThreads) shi[i] = slo[i] = 0;
    if (threadIdx.x == 0) smax = 0;
    __syncthreads();
    // window: up to one exponent above the largest of the CTA's first values
    {
        const int64_t i = (int64_t)blockIdx.x * kHistThreads + threadIdx.x;
        uint32_t m = 0;
        if (i < n4) {
            const float4 v = ld_stream4(W + i);
            const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t u = __float_as_uint(w[e]) & 0x7fffffffu;
                if (u < 0x7f800000u) m = max(m, u);
            }
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) atomicMax(&smax, m);
    }
    __syncthreads();
    uint32_t e_lo = window_start((smax >> 23) + 1);   // exponent field of cell 0 (a normal one), the same for the warp
    unsigned long long acc_hi = 0, acc_lo = 0;        // cell `lane` of this warp, folded so far
    unsigned long long low = 0;                       // this lane's values below the window, in cell 0's unit
    auto add_at = [&](uint32_t e, unsigned long long hi, unsigned long long lo) {
        if (hi) atomicAdd(&shi[e], hi);
        if (lo) atomicAdd(&slo[e], lo);
    };
    auto fold = [&]() {
        __syncwarp();
        // lane l collects cell l from every lane (rotated start), split before the
        // lanes are added up: a cell may hold nearly 2^64
        unsigned long long* row = cells + warp * kWin * 32 + lane * 32;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const unsigned long long x = row[(j + lane) & 31];
            acc_hi += x >> 24;
            acc_lo += x & 0xffffffull;
        }
        __syncwarp();
        for (int b = 0; b < kWin; ++b) ce[b * 32] = 0;
        __syncwarp();
        add_at(e_lo, low >> 24, low & 0xffffffull);
        low = 0;
    };
    uint32_t umax = 0;
    int64_t folded = 0;
    stream<false>(W, n4, [&](const float4& v, int64_t r) {
        const uint32_t u[4] = {__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu,
                               __float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu};
        const uint32_t d[4] = {(u[0] >> 23) - e_lo, (u[1] >> 23) - e_lo, (u[2] >> 23) - e_lo, (u[3] >> 23) - e_lo};
        umax = max(max(umax, max(u[0], u[1])), max(u[2], u[3]));
        const bool inside = max(max(d[0], d[1]), max(d[2], d[3])) < (uint32_t)kWin;
        if (r < 0 ? inside : __all_sync(0xffffffffu, inside)) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t m = (u[e] & 0x7fffffu) | 0x800000u;
                ce[d[e] * 32] += (unsigned long long)m * m;
            }
        } else {
            if (r >= 0) {                             // the whole warp: move the window up?
                uint32_t m = 0;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (u[e] < 0x7f800000u) m = max(m, u[e] >> 23);
                m = __reduce_max_sync(0xffffffffu, m);
                if (m >= e_lo + kWin) {
                    fold();
                    add_at(e_lo + lane, acc_hi, acc_lo);
                    acc_hi = acc_lo = 0;
                    e_lo = window_start(m + 1);
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t ef = u[e] >> 23;
                if (ef - e_lo < (uint32_t)kWin) {
                    const uint32_t m = (u[e] & 0x7fffffu) | 0x800000u;
                    ce[(ef - e_lo) * 32] += (unsigned long long)m * m;
                } else if (u[e] != 0 && u[e] < 0x7f800000u) {
                    uint32_t h, l;
                    msq_parts(u[e], h, l);
                    if (!EXACT && ef < e_lo && e_lo > 1)      // (subnormals stay apart from exponent 1)
                        low += (((unsigned long long)h << 24) | l) >> min(2 * (e_lo - max(ef, 1u)), 63u);
                    else
                        add_at(ef, h, l);
                }
            }
        }
        if (r - folded >= kFoldRounds) {              // the same for every lane of the warp
            fold();
            folded = r;
        }
    });
    __syncwarp();
    fold();
    add_at(e_lo + lane, acc_hi, acc_lo);
    // umax saw non-finite patterns too: they order above every finite one
    umax = __reduce_max_sync(0xffffffffu, umax);
    if (lane == 0) {
        if (umax >= 0x7f800000u) atomicOr(&ws->nonfinite, 1u);
        else atomicMax(&ws->absmax_bits, umax);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += kHistThreads) {
        if (shi[i]) atomicAdd(&st->hi[i], shi[i]);
        if (slo[i]) atomicAdd(&st->lo[i], slo[i]);
    }
}

// Pass 2: weights of the selected exponent per sub-bucket (counts in st->hi, as
// 32-bit words).
__global__ void __launch_bounds__(kHistThreads) energy_count_kernel(const float4* __restrict__ W, int64_t n4,
                                                                    EnergyState* st)
{
    __shared__ uint32_t cnt[4096];
    for (int i = threadIdx.x; i < 4096; i += kHistThreads) cnt[i] = 0;
    __syncthreads();
    const uint32_t prefix = st->prefix;
    stream<true>(W, n4, [&](const float4& v, int64_t) {
        const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t u = __float_as_uint(w[e]) & 0x7fffffffu;
            if ((u >> 23) == prefix && u) atomicAdd(&cnt[(u >> 11) & 0xfffu], 1u);
        }
    });
    __syncthreads();
    uint32_t* out = reinterpret_cast<uint32_t*>(st->hi);
    for (int i = threadIdx.x; i < 4096; i += kHistThreads)
        if (cnt[i]) atomicAdd(&out[i], cnt[i]);
}

// Window of pass 3 from pass 2's counts: bucket b's values lie in [lo_b, lo_(b+1)),
// so the cumulative energies have a lower and an upper bound; the crossing
// bucket is at or after the first whose upper bound reaches eps and at or before the
// first whose lower bound does.  Leaves the window's first bucket in wmin_bits and
// its length in window, and clears the bucket arrays.
__global__ void __launch_bounds__(kScanThreads) energy_window_scan_kernel(EnergyState* st, double eps)
{
    constexpr int PER = 4096 / kScanThreads;
    __shared__ double part[2][2][kScanThreads];
    __shared__ int first, last;
    const int t = threadIdx.x;
    const uint32_t* cnt = reinterpret_cast<const uint32_t*>(st->hi);
    const uint32_t field = st->prefix;
    const int e = (field ? (int)field : 1) - 127;
    const double unit = pow2(2 * e - 46);
    // (significand at the start of bucket b)^2, exact
    auto end_sq = [&](int b) {
        const unsigned long long m = (field ? 8388608ull : 0ull) + 2048ull * b;
        return m * m;
    };
    // This thread's buckets as exact integers (high and low 24 bits of the squares
    // apart), one conversion each: fp64 runs at a 64th of the fp32 rate.
    uint32_t n[PER];
    unsigned long long sum[2][2] = {{0, 0}, {0, 0}};
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        n[j] = cnt[t * PER + j];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const unsigned long long sq = end_sq(t * PER + j + k);
            sum[k][0] += n[j] * (sq >> 24);
            sum[k][1] += n[j] * (sq & 0xffffffull);
        }
    }
    double own[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) part[0][k][t] = own[k] = ((double)sum[k][0] * 16777216.0 + (double)sum[k][1]) * unit;
    int cur = 0;
    if (t == 0) { first = 4096; last = 4096; }
    __syncthreads();
    for (int off = 1; off < kScanThreads; off <<= 1) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
            part[cur ^ 1][k][t] = t >= off ? part[cur][k][t] + part[cur][k][t - off] : part[cur][k][t];
        cur ^= 1;
        __syncthreads();
    }
    // the bounds' own rounding stays far below these margins
    const double target = eps * st->total, below = st->below;
    const double near = target * (1.0 - 0x1p-36), sure = target * (1.0 + 0x1p-36);
    const double base[2] = {below + (t ? part[cur][0][t - 1] : 0.0), below + (t ? part[cur][1][t - 1] : 0.0)};
    // the first of this thread's buckets whose cumulative bound k reaches x
    auto reach = [&](int k, double x) {
        if (!(base[k] + own[k] * (1.0 + 0x1p-40) >= x)) return 4096;
        double cum = base[k];
        for (int j = 0; j < PER; ++j) {
            const int b = t * PER + j;
            cum += (double)cnt[b] * (double)end_sq(b + k) * unit;
            if (cnt[b] && cum >= x) return b;
        }
        return 4096;
    };
    const int f = reach(1, near), l = reach(0, sure);
    if (f < 4096) atomicMin(&first, f);
    if (l < 4096) atomicMin(&last, l);
    __syncthreads();
    uint32_t* words = reinterpret_cast<uint32_t*>(st->hi);
    if (t == 0) {
        // without a sure bucket the crossing may be any up to the last
        const int f0 = first, l0 = last < 4096 ? last : 4095;
        const int len = f0 < 4096 ? l0 - f0 + 1 : 0;
        if (len < 1 || len > kWinBuckets) st->failed = 1;
        st->wmin_bits = (uint32_t)f0;
        st->window = (uint32_t)(len < 1 || len > kWinBuckets ? 0 : len);
    }
    __syncthreads();
    for (int i = t; i < 4 * 4096; i += kScanThreads) words[i] = 0;     // hi and lo, for pass 3
}

// Pass 3 (see the top of the file).
__global__ void __launch_bounds__(kHistThreads) energy_values_kernel(const float4* __restrict__ W, int64_t n4,
                                                                     EnergyState* st)
{
    extern __shared__ uint32_t cnt[];                    // [kWinValues]
    __shared__ unsigned long long shi, slo;
    const uint32_t prefix = st->prefix, len = st->window * 2048u;
    if (len == 0) return;                                // no window: the exact form follows
    const uint32_t win0 = (prefix << 23) | (st->wmin_bits << 11);        // first pattern of the window
    for (uint32_t i = threadIdx.x; i < len; i += kHistThreads) cnt[i] = 0;
    if (threadIdx.x == 0) shi = slo = 0;
    __syncthreads();
    const uint32_t span = win0 - (prefix << 23);
    // energy below the window: one 64-bit sum per lane, split into high and low 24
    // bits before 2^16 values of 2^48 could overflow it
    const uint32_t lead = prefix ? 0x800000u : 0u;
    unsigned long long acc = 0, hi = 0, lo = 0;
    int64_t split = 0;
    stream<false>(W, n4, [&](const float4& v, int64_t r) {
        const float w[4] = {v.x, v.y, v.z, v.w};
        uint32_t in[4];
        bool any = false;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            // offset inside the exponent (wraps for smaller values)
            in[e] = (__float_as_uint(w[e]) & 0x7fffffffu) - (prefix << 23);
            const uint32_t m = in[e] < span ? in[e] | lead : 0u;
            acc += (unsigned long long)m * m;
            any |= in[e] - span < len;
        }
        if (any)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (in[e] - span < len) atomicAdd(&cnt[in[e] - span], 1u);
        if (r - split >= kFoldRounds) {
            hi += acc >> 24;
            lo += acc & 0xffffffull;
            acc = 0;
            split = r;
        }
    });
    hi += acc >> 24;
    lo += acc & 0xffffffull;
    for (int o = 16; o; o >>= 1) {
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&shi, hi);
        atomicAdd(&slo, lo);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (shi) atomicAdd(&st->lo[kBelowHi], shi);
        if (slo) atomicAdd(&st->lo[kBelowLo], slo);
    }
    uint32_t* out = reinterpret_cast<uint32_t*>(st->hi);
    for (uint32_t i = threadIdx.x; i < len; i += kHistThreads)
        if (cnt[i]) atomicAdd(&out[i], cnt[i]);
}

// The first value of the window whose cumulative share reaches eps.
__global__ void __launch_bounds__(kScanThreads) energy_value_scan_kernel(EnergyState* st, double eps)
{
    constexpr int PER = kWinValues / kScanThreads;
    __shared__ double part[2][kScanThreads];
    __shared__ int found;
    const int t = threadIdx.x, len = (int)st->window * 2048;
    if (len == 0) return;
    const uint32_t* cnt = reinterpret_cast<const uint32_t*>(st->hi);
    const uint32_t prefix = st->prefix, start = st->wmin_bits << 11;
    const int e = (prefix ? (int)prefix : 1) - 127;
    const double unit = pow2(2 * e - 46);
    auto sq_of = [&](int i) {
        const uint32_t m = (start + (uint32_t)i) | (prefix ? 0x800000u : 0u);
        return (unsigned long long)m * m;
    };
    unsigned long long hi = 0, lo = 0;                   // exact; one conversion per thread
    const int i0 = t * PER, i1 = i0 + PER < len ? i0 + PER : len;
    for (int i = i0; i < i1; i += 4) {
        const uint4 n4 = *reinterpret_cast<const uint4*>(cnt + i);
        const uint32_t n[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long sq = sq_of(i + k);
            hi += n[k] * (sq >> 24);
            lo += n[k] * (sq & 0xffffffull);
        }
    }
    const double own = ((double)hi * 16777216.0 + (double)lo) * unit;
    part[0][t] = own;
    if (t == 0) found = kWinValues;
    __syncthreads();
    int cur = 0;
    for (int off = 1; off < kScanThreads; off <<= 1) {
        part[cur ^ 1][t] = t >= off ? part[cur][t] + part[cur][t - off] : part[cur][t];
        cur ^= 1;
        __syncthreads();
    }
    const double total = st->total, near = eps * total * (1.0 - 0x1p-40);
    double cum = st->below + ((double)st->lo[kBelowHi] * 16777216.0 + (double)st->lo[kBelowLo]) * unit +
                 (t ? part[cur][t - 1] : 0.0);
    int f = kWinValues;
    if (own > 0.0 && cum + own * (1.0 + 0x1p-40) >= near)
        for (int i = i0; i < i1 && f == kWinValues; ++i) {
            if (cnt[i] == 0) continue;
            const double x = (double)cnt[i] * (double)sq_of(i) * unit;
            cum += x;
            if (x > 0.0 && cum >= near && cum / total >= eps) f = i;
        }
    if (f < kWinValues) atomicMin(&found, f);
    __syncthreads();
    if (t == 0) {
        if (found == kWinValues) st->failed = 1;         // a rounding step short: the exact form settles it
        st->wmin_bits = (prefix << 23) + start + (uint32_t)found;
    }
}

// One CTA: bucket energies in fp64, ascending inclusive scan from the energy
// below the prefix, first bucket whose share reaches eps.
template <int LEVEL>
__global__ void __launch_bounds__(kScanThreads) energy_scan_kernel(EnergyState* st, double eps)
{
    constexpr int NB = Level<LEVEL>::NB;
    constexpr int PER = NB / kScanThreads;               // buckets per thread, contiguous
    __shared__ double part[2][kScanThreads];
    __shared__ int found;
    const int t = threadIdx.x;
    const uint32_t prefix = st->prefix;
    // exponent field of the level's values: the bucket itself (level 1) or the prefix
    auto efield_of = [&](int b) -> uint32_t {
        return LEVEL == 1 ? (uint32_t)b : (LEVEL == 2 ? prefix : (prefix >> 12));
    };
    auto energy = [&](int b) -> double {
        const uint32_t ef = efield_of(b);
        const int e = (ef ? (int)ef : 1) - 127;
        return ((double)st->hi[b] * 16777216.0 + (double)st->lo[b]) * pow2(2 * e - 46);
    };
    double en[PER];
    double mine = 0.0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        en[j] = energy(t * PER + j);
        mine += en[j];
    }
    // fixed-order inclusive scan of the per-thread sums (Hillis-Steele)
    int cur = 0;
    part[0][t] = mine;
    if (t == 0) found = NB;
    __syncthreads();
    for (int off = 1; off < kScanThreads; off <<= 1) {
        const double x = part[cur][t] + (t >= off ? part[cur][t - off] : 0.0);
        part[cur ^ 1][t] = x;
        cur ^= 1;
        __syncthreads();
    }
    if (LEVEL == 1 && t == 0) {
        st->total = part[cur][kScanThreads - 1];
        st->below = 0.0;
    }
    __syncthreads();
    const double total = st->total;
    const double below0 = st->below;
    double cum = below0 + (t > 0 ? part[cur][t - 1] : 0.0);
    double cum_before = 0.0;                             // energy below this thread's crossing bucket
    int mine_found = NB;
    const double near = eps * total * (1.0 - 0x1p-40);   // below this the share is surely < eps
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const double prev = cum;
        cum += en[j];
        if (mine_found == NB && en[j] > 0.0 && cum >= near && cum / total >= eps) {
            mine_found = t * PER + j;
            cum_before = prev;
        }
    }
    atomicMin(&found, mine_found);
    __syncthreads();
    const int b = found;
    auto publish = [&](int bucket, double below) {
        st->below = below;
        const uint32_t np = LEVEL == 1 ? (uint32_t)bucket
                                       : (LEVEL == 2 ? (prefix << 12) | (uint32_t)bucket : (prefix << 11) | (uint32_t)bucket);
        st->prefix = np;
        if (LEVEL == 3) st->wmin_bits = np;
    };
    if (b < NB) {
        if (t == b / PER) publish(b, cum_before);
    } else if (t == 0) {
        // the share stayed a rounding step short of eps inside the parent
        // bucket: the parent's last non-empty value closes it
        int last = 0;
        double run = below0, before = below0;
        for (int i = 0; i < NB; ++i) {
            const double x = energy(i);
            if (x > 0.0) {
                last = i;
                before = run;
            }
            run += x;
        }
        publish(last, before);
    }
}

// Grid of a streaming pass: per_sm CTAs per SM, fewer for small inputs.
int stream_grid(int64_t n4, int per_sm)
{
    const int sms = sm_count() > 0 ? sm_count() : 148;
    const int64_t want = (n4 + kHistThreads * kUnroll - 1) / (kHistThreads * kUnroll), cap = (int64_t)per_sm * sms;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// Dynamic shared memory opt-in, once per kernel and device.
template <typename Kernel>
cudaError_t allow_smem(Kernel k, size_t smem, int (&configured)[64])
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured[dev] = 1;
    }
    return cudaSuccess;
}

template <int LEVEL>
cudaError_t hist(const float4* W, int64_t n4, EnergyState* st, cudaStream_t s)
{
    constexpr size_t smem = 2 * sizeof(unsigned long long) * Level<LEVEL>::NB;
    static int configured[64] = {0};
    cudaError_t e = allow_smem(energy_hist_kernel<LEVEL>, smem, configured);
    if (e != cudaSuccess) return e;
    energy_hist_kernel<LEVEL><<<stream_grid(n4, 3), kHistThreads, smem, s>>>(W, n4, st);
    return cudaGetLastError();
}

template <bool EXACT>
cudaError_t exponents(const float4* W, int64_t n4, EnergyState* st, Workspace* ws, cudaStream_t s)
{
    constexpr size_t smem = (size_t)(kHistThreads / 32) * kWin * 32 * sizeof(unsigned long long);
    static int configured[64] = {0};
    cudaError_t e = allow_smem(energy_exponents_kernel<EXACT>, smem, configured);
    if (e != cudaSuccess) return e;
    energy_exponents_kernel<EXACT><<<stream_grid(n4, 3), kHistThreads, smem, s>>>(W, n4, st, ws);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_energy_range(const float* W, int64_t count, double eps, EnergyState* st, Workspace* ws,
                                cudaStream_t s)
{
    const float4* W4 = reinterpret_cast<const float4*>(W);
    const int64_t n4 = count / 4;
    const size_t bucket_bytes = sizeof st->hi + sizeof st->lo;
    cudaError_t e;
    if ((e = cudaMemsetAsync(st, 0, sizeof(EnergyState), s)) != cudaSuccess) return e;
    const bool exact = eps < (double)count * 0x1p-50;    // (see the top of the file)
    e = exact ? exponents<true>(W4, n4, st, ws, s) : exponents<false>(W4, n4, st, ws, s);
    if (e != cudaSuccess) return e;
    energy_scan_kernel<1><<<1, kScanThreads, 0, s>>>(st, eps);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (!energy_counts_fit(count)) return cudaSuccess;
    static int configured3[64] = {0};
    constexpr size_t smem3 = (size_t)kWinValues * sizeof(uint32_t);
    if ((e = allow_smem(energy_values_kernel, smem3, configured3)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(st->hi, 0, bucket_bytes, s)) != cudaSuccess) return e;
    energy_count_kernel<<<stream_grid(n4, 6), kHistThreads, 0, s>>>(W4, n4, st);
    energy_window_scan_kernel<<<1, kScanThreads, 0, s>>>(st, eps);
    energy_values_kernel<<<stream_grid(n4, 3), kHistThreads, smem3, s>>>(W4, n4, st);
    energy_value_scan_kernel<<<1, kScanThreads, 0, s>>>(st, eps);
    return cudaGetLastError();
}

// Levels 2 and 3 by exact bucket energies, after launch_energy_range left the
// crossing open (its exponent and the energy below it stand).
cudaError_t launch_energy_exact(const float* W, int64_t count, double eps, EnergyState* st, cudaStream_t s)
{
    const float4* W4 = reinterpret_cast<const float4*>(W);
    const int64_t n4 = count / 4;
    const size_t bucket_bytes = sizeof st->hi + sizeof st->lo;
    cudaError_t e;
    if ((e = cudaMemsetAsync(st->hi, 0, bucket_bytes, s)) != cudaSuccess) return e;
    if ((e = hist<2>(W4, n4, st, s)) != cudaSuccess) return e;
    energy_scan_kernel<2><<<1, kScanThreads, 0, s>>>(st, eps);
    if ((e = cudaMemsetAsync(st->hi, 0, bucket_bytes, s)) != cudaSuccess) return e;
    if ((e = hist<3>(W4, n4, st, s)) != cudaSuccess) return e;
    energy_scan_kernel<3><<<1, kScanThreads, 0, s>>>(st, eps);
    return cudaGetLastError();
}

}  // namespace logq
