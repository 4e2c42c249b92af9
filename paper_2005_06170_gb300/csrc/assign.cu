// Steps 1-2 of the estimator on the GPU: catalogue moments and the B-spline
// assignment of mass and momentum to four periodic grids (paper Secs. 2.1-2.2,
// Eq. rawFFTed; the BL kernel's Fourier factor is applied in spectra.cu).
//
// Pipeline (all on one stream):
//   k_hist          the histogram of sort keys (key = x-row, y-row, z-segment of the
//                   cell), from the positions alone.
//   k_scan_*        exclusive scan of the key counts -> segment offsets.
//   k_scatter       writes each particle as a 32-byte record (grid coordinates and the
//                   four deposited values) at the slot an atomic increment of its key's
//                   cursor returns: a counting sort (any order within a key).
//   k_moments       FP64 moments and max |q|, from velocities and masses.
//   k_deposit_home  (FP32, cubic, >= 1/2 particle per cell) each particle deposited
//   + k_home_fixup  once by the tile owning its cell, halos added afterwards; otherwise
//   k_deposit_fx    (FP32), k_deposit_ix (FP64, orders 2 to 5, in integers), k_deposit
//                   (FP64, the rest): one CTA per output tile gathers the particles of every segment whose
//                   stencils reach the tile, accumulates in shared memory, then writes
//                   each node of the tile exactly once. No global atomics, no zero fill.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <utility>

#include "pkmom_internal.cuh"
#include "warp_sums.cuh"

namespace pkmom {

// ------------------------------------------------------------------ checked builds
namespace {
#if PKMOM_CHECKED
__device__ unsigned g_check_word;
__device__ __forceinline__ bool check_index(long long i, long long n, unsigned code)
{
    if (i >= 0 && i < n) return true;
    atomicOr(&g_check_word, code);
    return false;
}
#endif
}  // namespace

unsigned take_check_word_assign()
{
#if PKMOM_CHECKED
    unsigned w = 0;
    if (cudaMemcpyFromSymbol(&w, g_check_word, sizeof w) != cudaSuccess) return 0;
    if (w) {
        const unsigned zero = 0;
        cudaMemcpyToSymbol(g_check_word, &zero, sizeof zero);
    }
    return w;
#else
    return 0;
#endif
}

namespace {
// One index test that fails on purpose: index 1 against a bound of 1. The failed test
// records kChkSelf and no access follows it (checked builds; a no-op otherwise).
__global__ void k_check_selftest(int one)
{
    if (threadIdx.x == 0 && blockIdx.x == 0 && !PK_IN(one, one, kChkSelf)) return;
}
}  // namespace

cudaError_t launch_check_selftest(cudaStream_t s)
{
    k_check_selftest<<<1, 32, 0, s>>>(1);
    return cudaGetLastError();
}
namespace {

// Zeroed with the key table by the histogram's launch: the largest |q| of each field, the
// moments' block counter, and for FP64 2^32 less the high word of the smallest mass and of the
// smallest largest component of a momentum (0: none, subnormals count as zero).
enum { kCtlQmax = 0, kCtlDone = 4, kCtlLow = 5, kCtlWords = 8 };

// Biased exponent of the value behind a word of kCtlLow (none: above all)
__device__ __forceinline__ int exponent_of_least(unsigned word) { return word ? static_cast<int>((~word + 1u) >> 20) : 0x7ff; }
// Biased exponent of an FP64 value, and whether it is zero, in integer arithmetic
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }
__device__ __forceinline__ int high_word(double x) { return __double2hiint(x) & 0x7fffffff; }

constexpr int kHistThreads = 256;
constexpr int kMomentThreads = 256;
constexpr int kLaneParticles = 512;  // particles of one FP32 sum of k_moments

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// A 32-byte FP32 record in one 256-bit access (records_of keeps the records 32-byte aligned):
// the lanes of a warp read records of different lines, and two 128-bit loads of each took
// twice the wavefronts.
__device__ __forceinline__ Record<float> load_record(const Record<float> *p)
{
    Record<float> r;
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(r.u.x), "=f"(r.u.y), "=f"(r.u.z), "=f"(r.u.w), "=f"(r.q.x), "=f"(r.q.y), "=f"(r.q.z), "=f"(r.q.w)
        : "l"(p));
    return r;
}
__device__ __forceinline__ void store_record(Record<float> *p, const Record<float> &r)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(r.u.x), "f"(r.u.y),
                 "f"(r.u.z), "f"(r.u.w), "f"(r.q.x), "f"(r.q.y), "f"(r.q.z), "f"(r.q.w)
                 : "memory");
}
__device__ __forceinline__ void store_record(Record<double> *p, const Record<double> &r) { *p = r; }

// floor(u) wrapped into [0, ng); false for non-finite or huge |u|.
template <typename T>
__device__ __forceinline__ bool cell_of(T u, int ng, int &c)
{
    if (!(fabs(u) < T(1 << 30))) return false;
    int ic = static_cast<int>(floor(u));
    if (static_cast<unsigned>(ic) >= static_cast<unsigned>(ng)) {  // outside the box: wrap
        ic %= ng;
        ic = ic < 0 ? ic + ng : ic;
    }
    c = ic;
    return true;
}

// f(std::integral_constant<int, i>) for i = 0 .. N - 1, each i a compile-time constant
template <class F, int... I>
__device__ __forceinline__ void static_for_seq(F &&f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F &&f)
{
    static_for_seq(f, std::make_integer_sequence<int, N>{});
}

__device__ __forceinline__ int floordiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// A record's fourth coordinate holds its wrapped cell (10 bits per axis, ng <= 1024) as a
// bit pattern.
template <typename T> __device__ __forceinline__ T pack_cell(int c0, int c1, int c2);
template <> __device__ __forceinline__ float pack_cell<float>(int c0, int c1, int c2)
{
    return __int_as_float(c0 | (c1 << 10) | (c2 << 20));
}
template <> __device__ __forceinline__ double pack_cell<double>(int c0, int c1, int c2)
{
    return __longlong_as_double(c0 | (c1 << 10) | (c2 << 20));
}
__device__ __forceinline__ int unpack_cell(float v) { return __float_as_int(v); }
__device__ __forceinline__ int unpack_cell(double v) { return static_cast<int>(__double_as_longlong(v)); }

// The histogram of sort keys: positions only (12 bytes per FP32 particle), one
// fire-and-forget atomic increment per particle; non-finite or huge positions raise
// the data error flag. Two particles per iteration keep more loads in flight.
template <typename T>
__global__ void __launch_bounds__(kHistThreads)
k_hist(const T *__restrict__ x, const T *__restrict__ y, const T *__restrict__ z, int64_t stride, int64_t n,
       T scale, int ng, int sshift, uint32_t *__restrict__ counts, int *__restrict__ err)
{
    const int nseg = ng >> sshift;
    const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
    auto one = [&](int64_t i) {
        const int64_t j = i * stride;
        const T u0 = mul_rn(x[j], scale), u1 = mul_rn(y[j], scale), u2 = mul_rn(z[j], scale);
        int c0, c1, c2;
        if (cell_of(u0, ng, c0) & cell_of(u1, ng, c1) & cell_of(u2, ng, c2)) {
            const int64_t key = (static_cast<int64_t>(c0) * ng + c1) * nseg + (c2 >> sshift);
            if (PK_IN(key, static_cast<int64_t>(ng) * ng * nseg, kChkKey)) atomicAdd(counts + key, 1u);
        } else {
            *err = 1;
        }
    };
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += 2 * step) {
        one(i);
        if (i + step < n) one(i + step);
    }
}

// ------------------------------------------------------------------ scan
constexpr int kScanThreads = 512;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;  // keys per block

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t &total)
{
    __shared__ uint32_t s_w[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? s_w[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        s_w[lane] = w;  // inclusive prefix of warp totals
    }
    __syncthreads();
    const uint32_t warp_base = warp ? s_w[warp - 1] : 0u;
    total = s_w[nw - 1];
    __syncthreads();
    return warp_base + inc - v;
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_reduce(const uint32_t *__restrict__ counts, int64_t nkeys, uint32_t *__restrict__ blocksums)
{
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile + static_cast<int64_t>(threadIdx.x) * kScanItems;
    uint32_t s = 0;
    if (base + kScanItems <= nkeys) {
        const uint4 *v4 = reinterpret_cast<const uint4 *>(counts + base);
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) {
            const uint4 q = v4[k];
            s += q.x + q.y + q.z + q.w;
        }
    } else {
        for (int k = 0; k < kScanItems; ++k)
            if (base + k < nkeys) s += counts[base + k];
    }
    uint32_t total;
    block_exclusive_scan(s, total);
    if (threadIdx.x == 0) blocksums[blockIdx.x] = total;
}

// One block: exclusive scan of the block sums in place; writes the grand total
// to counts[nkeys] (the end offset).
__global__ void __launch_bounds__(1024)
k_scan_top(uint32_t *__restrict__ blocksums, int64_t nblocks, uint32_t *__restrict__ counts, int64_t nkeys)
{
    const int64_t per = (nblocks + blockDim.x - 1) / blockDim.x;
    const int64_t b0 = static_cast<int64_t>(threadIdx.x) * per;
    uint32_t s = 0;
    for (int64_t k = 0; k < per; ++k)
        if (b0 + k < nblocks) s += blocksums[b0 + k];
    uint32_t total;
    uint32_t run = block_exclusive_scan(s, total);
    for (int64_t k = 0; k < per; ++k)
        if (b0 + k < nblocks) {
            const uint32_t v = blocksums[b0 + k];
            blocksums[b0 + k] = run;
            run += v;
        }
    if (threadIdx.x == 0) counts[nkeys] = total;
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_apply(uint32_t *__restrict__ counts, int64_t nkeys, const uint32_t *__restrict__ blocksums)
{
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile + static_cast<int64_t>(threadIdx.x) * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
    const bool full = base + kScanItems <= nkeys;
    if (full) {
        const uint4 *v4 = reinterpret_cast<const uint4 *>(counts + base);
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) {
            const uint4 q = v4[k];
            v[4 * k] = q.x, v[4 * k + 1] = q.y, v[4 * k + 2] = q.z, v[4 * k + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) v[k] = base + k < nkeys ? counts[base + k] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) s += v[k];
    uint32_t total;
    uint32_t run = block_exclusive_scan(s, total) + blocksums[blockIdx.x];
    if (full) {
        uint4 *o4 = reinterpret_cast<uint4 *>(counts + base);
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) {
            uint4 q;
            q.x = run, run += v[4 * k];
            q.y = run, run += v[4 * k + 1];
            q.z = run, run += v[4 * k + 2];
            q.w = run, run += v[4 * k + 3];
            o4[k] = q;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k)
            if (base + k < nkeys) {
                counts[base + k] = run;
                run += v[k];
            }
    }
}

// ------------------------------------------------------------------ moments
// Sums of one lane's particles, in a fixed order: FP32 catalogues in compensated (Kahan) FP32
// pairs, so that neither FP64 work nor a warp reduction runs inside the loop; FP64 ones in
// plain FP64. With unit masses the sums of m and m^2 are the particle count and those of
// m^2 v are those of m v, so only nine of the fourteen are kept.
template <typename T, bool MASS>
struct LaneMoments {
    static constexpr int NV = MASS ? kMomentVals : 9, NG = (NV + 7) / 8;
    T sum[NV], cmp[NV];  // the sum of a value is sum - cmp
    // FP32: max |q| of each field; FP64: the high words of the largest |q| (NaN above all)
    std::conditional_t<sizeof(T) == 4, float, int> qmax[4];
    unsigned low[2];  // FP64: one less than the high words of kCtlLow
    __device__ __forceinline__ LaneMoments()
    {
        clear();
#pragma unroll
        for (int f = 0; f < 4; ++f) qmax[f] = 0;
        low[0] = low[1] = ~0u;
    }
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int k = 0; k < NV; ++k) sum[k] = T(0), cmp[k] = T(0);
    }
    __device__ __forceinline__ void put(int k, T x)
    {
        if constexpr (sizeof(T) == 4) {
            const T y = __fsub_rn(x, cmp[k]);
            const T t = __fadd_rn(sum[k], y);
            cmp[k] = __fsub_rn(__fsub_rn(t, sum[k]), y);
            sum[k] = t;
        } else {
            sum[k] += x;
        }
    }
    // Adds the warp's sums to total, value 8 g + k in lanes 4k .. 4k + 3 of total[g], by warp
    // reduce-scatters (FP32: in float pairs, so that a warp does two FP64 adds instead of 70:
    // FP64 runs at under two lanes a clock per SM on this part). Sums that leave the range of
    // FP32 on the way across the lanes are formed again in FP64.
    __device__ __forceinline__ void add_to(double (&total)[NG]) const
    {
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            double x;
            if constexpr (sizeof(T) == 4) {
                T hi[8], lo[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    hi[k] = 8 * g + k < NV ? sum[8 * g + k < NV ? 8 * g + k : 0] : T(0);
                    lo[k] = 8 * g + k < NV ? -cmp[8 * g + k < NV ? 8 * g + k : 0] : T(0);
                }
                x = warp_scatter_sum8(hi, lo);
                if (__any_sync(0xffffffffu, !isfinite(x))) x = scatter64(g);
            } else {
                x = scatter64(g);
            }
            total[g] += x;
        }
    }
    __device__ __forceinline__ double scatter64(int g) const
    {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = 8 * g + k < NV ? 8 * g + k : 0;
            v[k] = 8 * g + k < NV ? static_cast<double>(sum[i]) : 0.0;
            if constexpr (sizeof(T) == 4) v[k] -= 8 * g + k < NV ? static_cast<double>(cmp[i]) : 0.0;
        }
        return warp_scatter_sum8(v);
    }
    __device__ __forceinline__ void add(T m, T v0, T v1, T v2)
    {
        if constexpr (MASS) {
            const T m2 = m * m, p0 = m * v0, p1 = m * v1, p2 = m * v2;
            top(0, m), top(1, p0), top(2, p1), top(3, p2);
            if constexpr (sizeof(T) == 8) least(0, high_word(m)), least(1, p0, p1, p2);
            put(0, m);
            put(1, m2);
            put(2, p0);
            put(3, p1);
            put(4, p2);
            put(5, m2 * v0);
            put(6, m2 * v1);
            put(7, m2 * v2);
            put(8, m2 * v0 * v0);
            put(9, m2 * v1 * v1);
            put(10, m2 * v2 * v2);
            put(11, m2 * v0 * v1);
            put(12, m2 * v0 * v2);
            put(13, m2 * v1 * v2);
        } else {
            top(1, v0), top(2, v1), top(3, v2);
            if constexpr (sizeof(T) == 8) least(1, v0, v1, v2);
            put(0, v0);
            put(1, v1);
            put(2, v2);
            put(3, v0 * v0);
            put(4, v1 * v1);
            put(5, v2 * v2);
            put(6, v0 * v1);
            put(7, v0 * v2);
            put(8, v1 * v2);
        }
    }
    __device__ __forceinline__ void top(int f, T x)
    {
        if constexpr (sizeof(T) == 4) qmax[f] = fmaxf(qmax[f], fabsf(x));
        else qmax[f] = max(qmax[f], high_word(x));
    }
    __device__ __forceinline__ void least(int k, int word) { low[k] = min(low[k], static_cast<unsigned>(word) - 1u); }
    __device__ __forceinline__ void least(int k, T a, T b, T c)
    {
        least(k, max(high_word(a), max(high_word(b), high_word(c))));
    }
};

// The moments of the catalogue from the warps' sums (total: LaneMoments::add_to) and the lanes'
// maxima: one partial per block, and the last block to finish adds the partials in a fixed
// order into out (pkmom_moments). done: a zeroed counter. As FP64 butterflies in 1216 blocks
// and a separate kernel the same sums took 80 us whatever the catalogue's size.
template <typename T, bool MASS>
__device__ __forceinline__ void finish_moments(LaneMoments<T, MASS> &lm,
                                               const double (&total)[LaneMoments<T, MASS>::NG], int64_t n,
                                               double *__restrict__ partials, unsigned *__restrict__ qmax_bits,
                                               unsigned *__restrict__ done, double *__restrict__ out)
{
    constexpr int NV = LaneMoments<T, MASS>::NV, NG = LaneMoments<T, MASS>::NG;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __shared__ double s_part[kMomentThreads / 32][8 * NG];
    __shared__ bool s_last;
#pragma unroll
    for (int g = 0; g < NG; ++g)
        if ((lane & 3) == 0) s_part[warp][8 * g + (lane >> 2)] = total[g];
    if constexpr (!MASS && sizeof(T) == 4) lm.qmax[0] = 1.0f;
    else if constexpr (!MASS) lm.qmax[0] = 0x3ff00000, lm.low[0] = 0x3ff00000 - 1;
    if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const unsigned low = __reduce_min_sync(0xffffffffu, lm.low[k]);
            if (lane == 0) atomicMax(qmax_bits + kCtlLow + k, ~low);
        }
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        // non-negative floats order like their bit patterns
        unsigned mine;
        if constexpr (sizeof(T) == 4) mine = __float_as_uint(lm.qmax[f]);
        else mine = static_cast<unsigned>(lm.qmax[f]);
        const unsigned bits = __reduce_max_sync(0xffffffffu, mine);
        if (lane == 0) atomicMax(qmax_bits + f, bits);
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double total = 0.0;
        for (int w = 0; w < nw; ++w) total += s_part[w][threadIdx.x];
        partials[static_cast<int64_t>(blockIdx.x) * kMomentWords + threadIdx.x] = total;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // value k by warps k, k + nw, ...; without masses: m v, then m^2 v v^T
    for (int k = warp; k < NV; k += nw) {
        double x = 0.0;
        for (int b = lane; b < static_cast<int>(gridDim.x); b += 32)
            x += __ldcg(partials + static_cast<int64_t>(b) * kMomentWords + k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane != 0) continue;
        if constexpr (MASS) out[k] = x;
        else if (k < 3) out[2 + k] = x, out[5 + k] = x;
        else out[5 + k] = x;
    }
    if (threadIdx.x == 0) {
        if constexpr (!MASS) out[0] = out[1] = static_cast<double>(n);
        out[kMomentVals] = static_cast<double>(n);
        out[kMomentVals + 1] = 0.0;
    }
}

// The catalogue moments and the largest |q| of each deposited field, from velocities
// and masses alone (mass may be null only with MASS false).
template <typename T, bool MASS>
__global__ void __launch_bounds__(kMomentThreads)
k_moments(const T *__restrict__ vx, const T *__restrict__ vy, const T *__restrict__ vz, const T *__restrict__ mass,
          int64_t stride, int64_t n, double *__restrict__ partials, unsigned *__restrict__ qmax_bits,
          unsigned *__restrict__ done, double *__restrict__ out)
{
    LaneMoments<T, MASS> lm;
    double total[LaneMoments<T, MASS>::NG] = {};
    const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
    int count = 0;
    // (the warp's lanes run the same iterations)
    for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i0 - (threadIdx.x & 31) < n;
         i0 += 4 * step) {
        if (sizeof(T) == 4 && count == kLaneParticles / 4) {  // FP32 sums of at most kLaneParticles
            lm.add_to(total);
            lm.clear();
            count = 0;
        }
        ++count;
        T m[4], a[4], b[4], c[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = i0 + k * step;
            const bool ok = i < n;
            const int64_t j = ok ? i * stride : 0;
            m[k] = T(0);
            if constexpr (MASS) m[k] = ok ? mass[i] : T(0);  // absent particles add nothing
            a[k] = ok ? vx[j] : T(0);
            b[k] = ok ? vy[j] : T(0);
            c[k] = ok ? vz[j] : T(0);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) lm.add(m[k], a[k], b[k], c[k]);
    }
    lm.add_to(total);
    finish_moments<T, MASS>(lm, total, n, partials, qmax_bits, done, out);
}

// FP32 interleaved (n, 3) velocities, 16-byte aligned: four particles per thread read
// as three 128-bit loads ((v0x v0y v0z v1x) (v1y v1z v2x v2y) (v2z v3x v3y v3z)), and
// four masses as one. The particles are dealt to `lanes` sums, lane v taking the quads v,
// v + lanes, ..., and lane v < 32 the v-th of the n % 4 last particles, whatever the number
// of threads (a thread takes several lanes, one after another): a compensated sum of
// values that cancel, such as the momentum of a catalogue without bulk flow, depends on how
// they are dealt, and the size of the launch should not matter.
template <bool MASS>
__global__ void __launch_bounds__(kMomentThreads)
k_moments_v3(const float *__restrict__ v, const float *__restrict__ mass, int64_t n, int64_t lanes,
             double *__restrict__ partials, unsigned *__restrict__ qmax_bits, unsigned *__restrict__ done,
             double *__restrict__ out)
{
    const int64_t nq = n / 4;
    const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const float4 *v4 = reinterpret_cast<const float4 *>(v);
    const float4 *m4 = reinterpret_cast<const float4 *>(mass);
    const int64_t used = nq > 32 ? (nq < lanes ? nq : lanes) : 32;  // the other lanes are empty
    LaneMoments<float, MASS> lm;
    double total[LaneMoments<float, MASS>::NG] = {};
    for (int64_t vl = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; vl - (threadIdx.x & 31) < used;
         vl += step) {  // (the warp's lanes run the same iterations; `used` is no multiple of 32)
        lm.clear();
        for (int64_t q = vl < used ? vl : nq; q < nq; q += lanes) {
            const float4 a = v4[3 * q], b = v4[3 * q + 1], c = v4[3 * q + 2];
            float4 mm = make_float4(1.f, 1.f, 1.f, 1.f);
            if constexpr (MASS) mm = m4[q];
            lm.add(mm.x, a.x, a.y, a.z);
            lm.add(mm.y, a.w, b.x, b.y);
            lm.add(mm.z, b.z, b.w, c.x);
            lm.add(mm.w, c.y, c.z, c.w);
        }
        const int64_t i = 4 * nq + vl;
        if (vl < 32 && i < n) {
            float m = 1.f;
            if constexpr (MASS) m = mass[i];
            lm.add(m, v[3 * i], v[3 * i + 1], v[3 * i + 2]);
        }
        lm.add_to(total);
    }
    finish_moments<float, MASS>(lm, total, n, partials, qmax_bits, done, out);
}

// ------------------------------------------------------------------ scatter
// Each particle is written as a 32-byte record at the slot an atomic increment of its
// key's cursor returns: a counting sort (any order within a key).
template <typename T>
__global__ void __launch_bounds__(256)
k_scatter(const T *__restrict__ x, const T *__restrict__ y, const T *__restrict__ z, const T *__restrict__ vx,
          const T *__restrict__ vy, const T *__restrict__ vz, const T *__restrict__ mass, int64_t stride, int64_t n,
          T scale, int ng, int sshift, uint32_t *__restrict__ cursor, Record<T> *__restrict__ rec)
{
    const int nseg = ng >> sshift;
    const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += step) {
        const int64_t j = i * stride;
        const T u0 = mul_rn(x[j], scale), u1 = mul_rn(y[j], scale), u2 = mul_rn(z[j], scale);
        int c0, c1, c2;
        if (!(cell_of(u0, ng, c0) & cell_of(u1, ng, c1) & cell_of(u2, ng, c2))) continue;  // reported by k_hist
        const int64_t key = (static_cast<int64_t>(c0) * ng + c1) * nseg + (c2 >> sshift);
        if (!PK_IN(key, static_cast<int64_t>(ng) * ng * nseg, kChkKey)) continue;
        const uint32_t dst = atomicAdd(cursor + key, 1u);
        if (!PK_IN(dst, n, kChkRecord)) continue;
        const T m = mass ? mass[i] : T(1);
        Record<T> r;
        r.u = Vec4<T>{u0 - floor(u0), u1 - floor(u1), u2 - floor(u2), pack_cell<T>(c0, c1, c2)};
        r.q = Vec4<T>{m, m * vx[j], m * vy[j], m * vz[j]};
        store_record(rec + dst, r);
    }
}

// ------------------------------------------------------------------ deposit
// B-spline weights of order M for a particle at fractional offset t = u - floor(u)
// in its cell; `first` receives the first node relative to floor(u).
// Offset from floor(u) of the first of the M nodes the order-M B-spline reaches for a
// particle at offset t in its cell (the convention of bspline_weights below).
template <int M, typename T>
__host__ __device__ constexpr int bspline_first(T t)
{
    if constexpr (M == 5) return t >= T(0.5) ? -1 : -2;
    else if constexpr (M == 4) return -1;
    else if constexpr (M == 3) return t >= T(0.5) ? 0 : -1;
    else if constexpr (M == 2) return 0;
    else return t >= T(0.5) ? 1 : 0;
}

template <int M, typename T>
__device__ __forceinline__ void bspline_weights(T t, T (&w)[M], int &first)
{
    first = bspline_first<M, T>(t);
    if constexpr (M == 4) {
        const T s = T(1) - t, t2 = t * t, t3 = t2 * t;
        const T sixth = T(1) / T(6);
        w[0] = s * s * s * sixth;
        w[1] = (T(3) * t3 - T(6) * t2 + T(4)) * sixth;
        w[2] = (T(-3) * t3 + T(3) * t2 + T(3) * t + T(1)) * sixth;
        w[3] = t3 * sixth;
    } else if constexpr (M == 5) {
        // the centred quartic B-spline at distances d + 2 .. d - 2 from the nearest node
        const bool up = t >= T(0.5);
        const T d = up ? t - T(1) : t;  // offset from the nearest node, in [-1/2, 1/2)
        const T d2 = d * d;
        auto mid = [](T x) {  // 1/2 <= x <= 3/2
            return (T(55) + x * (T(20) + x * (T(-120) + x * (T(80) + x * T(-16))))) / T(96);
        };
        const T lo = T(1) - T(2) * d, hi = T(1) + T(2) * d;
        w[0] = lo * lo * lo * lo / T(384);
        w[1] = mid(T(1) + d);
        w[2] = T(115) / T(192) - T(5) / T(8) * d2 + T(0.25) * d2 * d2;
        w[3] = mid(T(1) - d);
        w[4] = hi * hi * hi * hi / T(384);
    } else if constexpr (M == 3) {
        const bool up = t >= T(0.5);
        const T d = up ? t - T(1) : t;  // offset from the nearest node, in [-1/2, 1/2)
        const T a = T(0.5) - d, b = T(0.5) + d;
        w[0] = T(0.5) * a * a;
        w[1] = T(0.75) - d * d;
        w[2] = T(0.5) * b * b;
    } else if constexpr (M == 2) {
        w[0] = T(1) - t;
        w[1] = t;
    } else {
        w[0] = T(1);
    }
}

// Coefficients c_0..c_7 of the BL function phi = sum_n c_n B_4(. - n), c_{-n} = c_n
// (cubic order), set once per device by set_bl_coefficients.
__constant__ float c_bl_f[8];
__constant__ double c_bl_d[8];
template <typename T> __device__ __forceinline__ T bl_coef(int n);
template <> __device__ __forceinline__ float bl_coef<float>(int n) { return c_bl_f[n < 0 ? -n : n]; }
template <> __device__ __forceinline__ double bl_coef<double>(int n) { return c_bl_d[n < 0 ? -n : n]; }

// Weights of the BL function truncated to |x| < R cells (the direct real-space
// assignment of Sec. 2.4.1) for a particle at offset t in its cell: nodes floor(u) + k,
// k = 1 - R .. R. phi(t - k) = sum_j b_j(t) c_{j-1-k} with b_j the cubic B-spline
// weights of nodes floor(u) - 1 + j; zero where |t - k| >= R.
template <int R, typename T>
__device__ __forceinline__ void bl_weights(T t, T (&w)[2 * R], int &first)
{
    T b[4];
    int f4;
    bspline_weights<4, T>(t, b, f4);
    first = 1 - R;
#pragma unroll
    for (int i = 0; i < 2 * R; ++i) {
        const int k = 1 - R + i;
        T v = T(0);
#pragma unroll
        for (int j = 0; j < 4; ++j) v += b[j] * bl_coef<T>(j - 1 - k);
        w[i] = fabs(t - T(k)) < T(R) ? v : T(0);
    }
}

template <typename T, int M, int T0, int T1, int T2, int NT>
struct DepositCfg {
    static constexpr int HL = (M % 2 == 0) ? M / 2 : (M + 1) / 2;  // cells below the tile that reach it
    static constexpr int HR = (M % 2 == 0) ? M / 2 - 1 : (M - 1) / 2;
    static constexpr int R0 = T0 + HL + HR, R1 = T1 + HL + HR;
    static constexpr int MAXR = 2 * R0 * R1;  // up to two particle ranges per row
    static constexpr int TN = T0 * T1 * T2;
    static constexpr int IPT = (MAXR + NT - 1) / NT;
    static constexpr size_t smem = 4 * TN * sizeof(T);
};

// Largest product of three B-spline weights of order M: bounds any node value of the
// tile by this times (particles in the tile's reach) times max |q|.
template <int M> constexpr float kMaxWeight3 =
    M == 5 ? 0.2148770f : (M == 4 ? 0.2962963f : (M == 3 ? 0.421875f : 1.0f));
// The same for the BL function: max |phi| = phi(0) = 1.0890, cubed 1.2916.
constexpr float kMaxWeight3BL = 1.2917f;
template <int M, int BLR> constexpr float kMaxW3 = BLR > 0 ? kMaxWeight3BL : kMaxWeight3<M>;

// The particle index ranges of one tile: for every (x, y) cell row within reach of the
// tile, the sort-key segments covering the z cells within reach (one range, or two
// where the reach wraps around the periodic box). Fills s_beg[slot] and the exclusive
// prefix s_pre[slot] of the range lengths; returns the total particle count.
template <class C>
__device__ __forceinline__ uint32_t build_ranges(const uint32_t *__restrict__ offsets, int ng, int sshift, int t0,
                                                 int t1, int t2, int T2, uint32_t *s_beg, uint32_t *s_pre)
{
    const int S = 1 << sshift;
    const int nseg = ng >> sshift;
    const int r0n = C::R0 < ng ? C::R0 : ng;
    const int r1n = C::R1 < ng ? C::R1 : ng;
    const int nrows = r0n * r1n;
    const int zc = (T2 + C::HL + C::HR) < ng ? (T2 + C::HL + C::HR) : ng;
    int slo = 0, shi = nseg - 1;
    bool whole = zc == ng;
    if (!whole) {
        slo = floordiv(t2 - C::HL, S);
        shi = floordiv(t2 - C::HL + zc - 1, S);
        whole = shi - slo + 1 >= nseg;
        if (whole) slo = 0, shi = nseg - 1;
    }
    uint32_t lens[C::IPT];
    uint32_t my = 0;
#pragma unroll
    for (int k = 0; k < C::IPT; ++k) {
        const int slot = threadIdx.x * C::IPT + k;
        uint32_t beg = 0, len = 0;
        if (slot < 2 * nrows) {
            const int r = slot >> 1, second = slot & 1;
            int a0 = t0 - C::HL + r / r1n, a1 = t1 - C::HL + r % r1n;
            a0 = a0 < 0 ? a0 + ng : (a0 >= ng ? a0 - ng : a0);
            a1 = a1 < 0 ? a1 + ng : (a1 >= ng ? a1 - ng : a1);
            const int64_t base = (static_cast<int64_t>(a0) * ng + a1) * nseg;
            int lo = slo, hi = shi;  // segment range of this piece, inclusive
            bool use = !second;
            if (slo < 0) {
                if (second) lo = 0, hi = shi, use = true;
                else lo = slo + nseg, hi = nseg - 1;
            } else if (shi >= nseg) {
                if (second) lo = 0, hi = shi - nseg, use = true;
                else hi = nseg - 1;
            }
            if (use) {
                beg = offsets[base + lo];
                len = offsets[base + hi + 1] - beg;
            }
        }
        if (slot < C::MAXR) s_beg[slot] = beg;
        lens[k] = len;
        my += len;
    }
    uint32_t total;
    uint32_t run = block_exclusive_scan(my, total);
#pragma unroll
    for (int k = 0; k < C::IPT; ++k) {
        const int slot = threadIdx.x * C::IPT + k;
        if (slot < C::MAXR) s_pre[slot] = run;
        run += lens[k];
    }
    if (threadIdx.x == 0) s_pre[C::MAXR] = total;
    __syncthreads();
    return total;
}

// Last slot whose range starts at or before p (p < total).
template <int MAXR>
__device__ __forceinline__ int find_slot(const uint32_t *s_pre, uint32_t p)
{
    int lo = 0, hi = MAXR - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_pre[mid] <= p) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Weights and tile-local node indices (-1 outside the tile) of one particle.
template <typename T, int M, int BLR = 0>
__device__ __forceinline__ void stencil(const Record<T> &r, int ng, int t0, int t1, int t2, int T0, int T1, int T2,
                                        T (&w)[3][M], int (&li)[3][M])
{
    const T t[3] = {r.u.x, r.u.y, r.u.z};  // offsets within the cells
    const int packed = unpack_cell(r.u.w);
    const int tb[3] = {t0, t1, t2};
    const int td[3] = {T0, T1, T2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int c = (packed >> (10 * a)) & 1023;
        int first;
        if constexpr (BLR > 0) bl_weights<BLR, T>(t[a], w[a], first);
        else bspline_weights<M, T>(t[a], w[a], first);
#pragma unroll
        for (int k = 0; k < M; ++k) {
            int l = c + first + k - tb[a];
            l = l < 0 ? l + ng : (l >= ng ? l - ng : l);
            li[a][k] = l < td[a] ? l : -1;
        }
    }
}

// Weight and tile-local index of x node k0 (node floor(u) + 1 - R + k0) of the truncated
// BL stencil, formed on its own (the rolled x loop of the wide stencils); false if the
// node lies outside the tile or beyond the radius.
template <int R, typename T>
__device__ __forceinline__ bool bl_node_x(const Record<T> &r, int ng, int t0, int T0, int k0, T &w, int &l)
{
    const int k = 1 - R + k0;
    int lx = (unpack_cell(r.u.w) & 1023) + k - t0;
    lx = lx < 0 ? lx + ng : (lx >= ng ? lx - ng : lx);
    if (lx >= T0 || !(fabs(r.u.x - T(k)) < T(R))) return false;
    T b[4];
    int f4;
    bspline_weights<4, T>(r.u.x, b, f4);
    T v = T(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) v += b[j] * bl_coef<T>(j - 1 - k);
    w = v;
    l = lx;
    return true;
}

// FP64 tile-gather deposit with FP64 shared-memory atomics, for the cases the fixed-point
// deposit (k_deposit_ix) leaves out. The whole CTA takes part; acc: 4 T0 T1 T2 words.
template <typename T, int M, int T0, int T1, int T2, int NT, int BLR>
__device__ __noinline__ void deposit_fp64_tile(const Record<T> *__restrict__ rec,
                                               const uint32_t *__restrict__ offsets, int ng, int sshift,
                                               T *__restrict__ grids, int64_t grid_elems, T *acc, uint32_t *s_beg,
                                               uint32_t *s_pre)
{
    using C = DepositCfg<T, M, T0, T1, T2, NT>;
    const int ntz = ng / T2, nty = ng / T1;
    int tile = blockIdx.x;
    const int tz = tile % ntz;
    tile /= ntz;
    const int ty = tile % nty;
    const int tx = tile / nty;
    const int t0 = tx * T0, t1 = ty * T1, t2 = tz * T2;
    for (int k = threadIdx.x; k < 4 * C::TN; k += NT) acc[k] = T(0);
    const uint32_t total = build_ranges<C>(offsets, ng, sshift, t0, t1, t2, T2, s_beg, s_pre);

    for (uint32_t p = threadIdx.x; p < total; p += NT) {
        const int slot = find_slot<C::MAXR>(s_pre, p);
        const Record<T> r = rec[s_beg[slot] + (p - s_pre[slot])];
        T w[3][M];
        int li[3][M];
        stencil<T, M, BLR>(r, ng, t0, t1, t2, T0, T1, T2, w, li);
        auto plane = [&](T wx, int lx) {  // the M x M (y, z) nodes of one x node
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) {
                if (li[1][k1] < 0) continue;
                const T w01 = wx * w[1][k1];
                const int b01 = (lx * T1 + li[1][k1]) * T2;
#pragma unroll
                for (int k2 = 0; k2 < M; ++k2) {
                    if (li[2][k2] < 0) continue;
                    const T ww = w01 * w[2][k2];
                    T *a = acc + b01 + li[2][k2];
                    atomicAdd(a, r.q.x * ww);
                    atomicAdd(a + C::TN, r.q.y * ww);
                    atomicAdd(a + 2 * C::TN, r.q.z * ww);
                    atomicAdd(a + 3 * C::TN, r.q.w * ww);
                }
            }
        };
        if constexpr (BLR > 2) {  // wide stencils: rolled x loop (instruction cache)
            T wx;
            int lx;
#pragma unroll 1
            for (int k0 = 0; k0 < M; ++k0)
                if (bl_node_x<BLR, T>(r, ng, t0, T0, k0, wx, lx)) plane(wx, lx);
        } else {
#pragma unroll
            for (int k0 = 0; k0 < M; ++k0)
                if (li[0][k0] >= 0) plane(w[0][k0], li[0][k0]);
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < C::TN; k += NT) {
        const int l2 = k % T2, l01 = k / T2;
        const int l1 = l01 % T1, l0 = l01 / T1;
        const int64_t gi = (static_cast<int64_t>(t0 + l0) * ng + (t1 + l1)) * (ng + 2) + t2 + l2;
        if (!PK_IN(gi, grid_elems, kChkGrid)) continue;
#pragma unroll
        for (int f = 0; f < 4; ++f) grids[f * grid_elems + gi] = acc[f * C::TN + k];
    }
}

template <typename T, int M, int T0, int T1, int T2, int NT, int BLR = 0>
__global__ void __launch_bounds__(NT)
k_deposit(const Record<T> *__restrict__ rec, const uint32_t *__restrict__ offsets,
          const unsigned *__restrict__ /*qmax_bits*/, int ng, int sshift, T *__restrict__ grids, int64_t grid_elems,
          int /*list_cap*/, bool /*sparse*/)
{
    using C = DepositCfg<T, M, T0, T1, T2, NT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_beg[C::MAXR];
    __shared__ uint32_t s_pre[C::MAXR + 1];
    deposit_fp64_tile<T, M, T0, T1, T2, NT, BLR>(rec, offsets, ng, sshift, grids, grid_elems,
                                                 reinterpret_cast<T *>(smem_raw), s_beg, s_pre);
}

// ------------------------------------------------------------------ FP64 in fixed point
// FP64 adds and multiplies run at under two lanes a clock per SM on this part, and a shared
// FP64 atomic at 20 clocks a warp; 32-bit integer multiply-adds run at 64 lanes a clock. So
// FP64 grids of orders 2 to 5 are deposited in integers: offsets in the cell as 63-bit
// fractions, weights as 62-bit ones (two words of 31 bits), values scaled by the largest
// exponent of their field to 62 bits, and each contribution, a 62-bit integer, split into
// words of 22, 22 and 18 bits that are summed by 32-bit shared adds. The sums are exact and
// do not depend on the order. The low words take up to 1023 adds, then their carries are
// moved up; the high words take kIxFlush such chunks, then they are added to 64-bit sums in
// the tile's own grid nodes. Nodes become FP64 by one rounding.
//
// A contribution is off by less than 6 units of 2^-61 of the scale, where FP64 products are
// off by up to 15 roundings of 2^-53 (three weights and three products) of each value. So a
// pass takes the particles whose mass (for the first field) and whose largest momentum
// component (for the others) lie at most kIxGap binary orders below the scale: 6 2^-61 2^9 =
// 2^-49.4 of themselves. What is left goes into another pass, on the scale of the largest
// that is left, added to the nodes in FP64. With equal masses and Gaussian velocities about
// 4 particles in 10^6 make a second pass of their tiles; masses over twelve decades take
// five or six.
constexpr int kIxLow = 22;         // bits of the two low words
constexpr uint32_t kIxChunk = 1016;  // particles between carries (a multiple of 8, below 2^10)
constexpr uint32_t kIxFlush = 7;     // 7 * 1016 contributions below 2^18 in the high word
constexpr int kIxGap = 8;
static_assert(kIxFlush * (kIxChunk * ((1u << 18) + 2)) < (1u << 31) - (1u << 18), "sums of the high word");

// (a b) / 2^63 of 63-bit fractions (at most 2^63 itself)
__device__ __forceinline__ unsigned long long mul63(unsigned long long a, unsigned long long b)
{
    return __umul64hi(a, b) << 1;
}

// Order-M B-spline weights as 63-bit fractions for the offset t (a fraction, at most 2^63);
// the nodes as in bspline_weights.
template <int M>
__device__ __forceinline__ void fixed_weights(unsigned long long t, unsigned long long (&w)[M], int &first)
{
    using u64 = unsigned long long;
    constexpr u64 one = 1ull << 63, half = 1ull << 62;
    constexpr u64 sixth = 0x2aaaaaaaaaaaaaabull;  // 2^64 / 6
    constexpr u64 c24 = 0x0aaaaaaaaaaaaaabull;    // 2^64 / 24
    const bool up = t >= half;
    if constexpr (M == 2) {
        first = 0;
        w[0] = one - t;
        w[1] = t;
    } else if constexpr (M == 4) {
        first = -1;
        const u64 v = one - t, t2 = mul63(t, t), t3 = mul63(t2, t), v2 = mul63(v, v), v3 = mul63(v2, v);
        constexpr u64 two_thirds = 0x5555555555555555ull;
        w[0] = __umul64hi(v3, sixth);
        w[1] = two_thirds - t2 + (t3 >> 1);
        w[2] = two_thirds - v2 + (v3 >> 1);
        w[3] = __umul64hi(t3, sixth);
    } else {
        // b = 1/2 + d and a = 1/2 - d, d the offset from the nearest node
        const u64 b = up ? t - half : t + half, a = one - b, d = up ? one - t : t;
        const u64 a2 = mul63(a, a), b2 = mul63(b, b), d2 = mul63(d, d);
        if constexpr (M == 3) {
            first = up ? 0 : -1;
            w[0] = a2 >> 1;
            w[1] = half + (half >> 1) - d2;
            w[2] = b2 >> 1;
        } else {
            first = up ? -1 : -2;
            const u64 a4 = mul63(a2, a2), b4 = mul63(b2, b2);
            auto mid = [](u64 x, u64 x2, u64 x4) {  // (1 + 4x + 6x^2 + 4x^3 - 4x^4) / 24
                const u64 x3 = mul63(x2, x);
                return (c24 >> 1) + (x2 >> 2) + __umul64hi(x + x3 - x4, sixth);
            };
            w[0] = __umul64hi(a4, c24);
            w[1] = mid(a, a2, a4);
            w[2] = 0x4caaaaaaaaaaaaabull - (d2 >> 1) - (d2 >> 3) + (mul63(d2, d2) >> 2);  // 115/192 - 5/8 d^2 + d^4/4
            w[3] = mid(b, b2, b4);
            w[4] = __umul64hi(b4, c24);
        }
    }
}

// x 2^62 / 2^(biased - 1022) rounded, for a finite x whose biased exponent is at most
// `biased`: below 2^62 in magnitude
__device__ __forceinline__ long long fixed_value(double x, int biased)
{
    const long long bits = __double_as_longlong(x);
    const int e = static_cast<int>(bits >> 52) & 0x7ff;
    long long m = (bits & ((1ll << 52) - 1)) | (e ? 1ll << 52 : 0ll);
    const int left = (e ? e : 1) - max(biased, 1) + 9;
    if (left >= 0) m <<= left;
    else m = left < -62 ? 0 : (m + (1ll << (-left - 1))) >> -left;
    return bits < 0 ? -m : m;
}

// The node sum hi 2^44 + low (0 <= low < 2^44) times 2^scale as FP64, rounded once
__device__ __forceinline__ double fixed_to_double(long long hi, long long low, int scale)
{
    // above 62 bits the lowest bits are dropped, which leaves 61 (hi: below 2^49, n < 2^31)
    const int drop = max(0, 64 - __clzll(hi < 0 ? ~hi : hi) - 18);
    const long long v = (hi << (44 - drop)) + (low >> drop);
    scale += drop;
    if (v == 0) return 0.0;
    const bool neg = v < 0;
    unsigned long long m = neg ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
    const int lz = __clzll(static_cast<long long>(m));
    const int e = 1023 + 63 - lz + scale;  // biased exponent
    m <<= lz;                              // the leading one at bit 63
    if (e < 1 || e > 2045) return scalbn(static_cast<double>(v), scale);
    const unsigned long long rest = m & 0x7ff, q = m >> 11;
    unsigned long long r = (q & ((1ull << 52) - 1)) | (static_cast<unsigned long long>(e) << 52);
    r += (rest > 0x400 || (rest == 0x400 && (q & 1))) ? 1 : 0;  // a carry moves the exponent up
    return __longlong_as_double(static_cast<long long>(r | (neg ? 1ull << 63 : 0ull)));
}

// Three shared-memory adds at byte offsets OFF + j * FS from addr (immediates).
template <int OFF, int FS>
__device__ __forceinline__ void red3(unsigned addr, int v0, int v1, int v2)
{
    asm volatile(
        "red.shared.add.s32 [%0+%4], %1;\n\t"
        "red.shared.add.s32 [%0+%5], %2;\n\t"
        "red.shared.add.s32 [%0+%6], %3;" ::"r"(addr), "r"(v0), "r"(v1), "r"(v2), "n"(OFF), "n"(OFF + FS), "n"(OFF + 2 * FS));
}

// Layout and lane mapping of the fixed-point deposit: 4 fields of 3 words, TNP ints each; one
// particle per warp as in CoopLanes. Order 4: lane (dx, dy, h), four z nodes, fields 2h and
// 2h + 1; order 5: lane (dx, dy) of 25, all z and fields; order 3: lane (dx, dy, dz) of 27,
// all fields; order 2: lane (dx, dy, dz, field). The pitches put the lanes' nodes in
// different banks (checked below); the lanes without a node take the free banks and a weight
// of zero.
template <int M, int T0, int T1, int T2>
struct IxLanes {
    static constexpr int RW = M == 2 ? T2 : M == 3 ? (T2 == 8 ? 11 : 18) : M == 4 && T2 == 8 ? 8 : T2 + 1;
    static constexpr int PX =
        T1 * RW + (M == 2 ? (T2 == 8 ? 16 : 2) : M == 3 ? (T2 == 8 ? 1 : 5) : M == 4 ? (T2 == 8 ? 1 : 0) : T2 == 8 ? 2 : 3);
    static constexpr int TNP = T0 * PX + (M == 2 ? (T2 == 8 ? 2 : 4) : M == 4 ? 2 : 0);
    static constexpr int FRONT = (5 * (PX + RW + 1) + 3) / 4 * 4;
    static constexpr int BACK = 5 * (PX + RW + 1) + 32;
    static constexpr size_t bytes = size_t(FRONT + 12 * TNP + BACK) * sizeof(int);
    static constexpr int NZ = M >= 4 ? M : 1;
    static constexpr int NF = M == 2 ? 1 : M == 4 ? 2 : 4;
    static constexpr int USED = M == 3 ? 27 : M == 5 ? 25 : 32;
    static constexpr int WQ = 6 * M;                 // staged words per particle: 3 M weights of two words,
    static constexpr int QQ = (WQ + 3) / 4 * 4;      // four values of two words, the first node
    static constexpr int STRIDE = QQ + 12;
    static constexpr int NB = 8;
    __host__ __device__ static constexpr int dx(int l) { return M == 2 ? l & 1 : M == 3 ? l / 9 : M == 4 ? (l >> 2) & 3 : l / 5; }
    __host__ __device__ static constexpr int dy(int l) { return M == 2 ? (l >> 1) & 1 : M == 3 ? (l / 3) % 3 : M == 4 ? l & 3 : l % 5; }
    __host__ __device__ static constexpr int dz(int l) { return M == 2 ? (l >> 2) & 1 : M == 3 ? l % 3 : 0; }
    __host__ __device__ static constexpr int field(int l) { return M == 2 ? l >> 3 : M == 4 ? 2 * (l >> 4) : 0; }
    __host__ __device__ static constexpr int node_offset(int l)
    {
        return dx(l) * PX + dy(l) * RW + dz(l) + 3 * field(l) * TNP;
    }
    static constexpr unsigned free_banks()
    {
        unsigned seen = 0;
        for (int l = 0; l < USED; ++l) seen |= 1u << (node_offset(l) & 31);
        return ~seen;
    }
    static constexpr bool banks_distinct()
    {
        int n = 0;
        for (unsigned m = free_banks(); m; m &= m - 1) ++n;
        return n == 32 - USED;
    }
    __device__ static int offset(int lane)
    {
        if (lane < USED) return node_offset(lane);
        unsigned m = free_banks();
        for (int l = USED; l < lane; ++l) m &= m - 1;
        return __ffs(static_cast<int>(m)) - 1;
    }
    // the adds' nodes lie in the padded allocation (see fx_pads_cover)
    static constexpr bool pads_cover()
    {
        constexpr int HL = (M % 2 == 0) ? M / 2 : (M + 1) / 2, HR = (M % 2 == 0) ? M / 2 - 1 : (M - 1) / 2;
        constexpr int lo = -HL + bspline_first<M, float>(0.0f), up = HR - 1 + bspline_first<M, float>(0.5f) + M - 1;
        return lo * (PX + RW + 1) >= -FRONT && (T0 + up) * PX + (T1 + up) * RW + T2 + up + 32 + 11 * TNP < 12 * TNP + BACK;
    }
    static_assert(banks_distinct() && pads_cover() && 3 * M * 2 <= WQ, "lanes in different banks, nodes in the pads");
};

// Whether a particle's mass (heavy) or momentum (fast) is part of the pass whose largest
// exponents are base_m and base_p; what is left for later ones is noted in left.
__device__ __forceinline__ bool in_pass(const double (&q)[4], int base_m, int base_p, int *left, bool &heavy, bool &fast)
{
    const int em = exponent_of(q[0]);
    const int ep = max(exponent_of(q[1]), max(exponent_of(q[2]), exponent_of(q[3])));
    heavy = em <= base_m && em + kIxGap >= base_m;
    fast = ep <= base_p && ep + kIxGap >= base_p;
    if (em + kIxGap < base_m && nonzero(q[0])) atomicMax(left, em + 1);
    if (ep + kIxGap < base_p && (nonzero(q[1]) || nonzero(q[2]) || nonzero(q[3]))) atomicMax(left + 1, ep + 1);
    return heavy || fast;
}

// FP64 tile-gather deposit in fixed point (see above): one particle per warp, its weights
// evaluated by four lanes (three axes and the values) for eight particles at a time, staged in
// shared memory and read back by all lanes. Bound by integer issue. With FP64 products and
// shared FP64 atomics 10^6 uniform particles on 128^3 took 3.58 ms, 10^6 in halos 18 to 20 ms;
// in fixed point 0.97 and 1.46 ms, with lognormal weights (sigma 1) 1.27 and 1.89 ms, with
// weights over twelve decades 1.72 and 2.65 ms.
template <int M, int T0, int T1, int T2, int NT>
__global__ void __launch_bounds__(NT)
k_deposit_ix(const Record<double> *__restrict__ rec, const uint32_t *__restrict__ offsets,
             const unsigned *__restrict__ qmax_bits, int ng, int sshift, double *__restrict__ grids, int64_t grid_elems,
             int /*list_cap*/, bool /*sparse*/)
{
    using C = DepositCfg<double, M, T0, T1, T2, NT>;
    using L = IxLanes<M, T0, T1, T2>;
    constexpr int NW = NT / 32, TNP = L::TNP;
    constexpr unsigned full = 0xffffffffu;
    static_assert(L::bytes >= C::smem, "the FP64 accumulator fits too");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_beg[C::MAXR];
    __shared__ uint32_t s_pre[C::MAXR + 1];
    __shared__ int s_left[2];  // one more than the largest exponent left (mass, momentum), 0: none
    __shared__ __align__(16) int s_stage[NW][L::NB * L::STRIDE];
    __shared__ uint32_t s_queue[NW][L::NB + 32];
    int top[4];  // biased exponent of the largest value of each field
    bool finite = true;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        top[f] = static_cast<int>(qmax_bits[f] >> 20);
        finite = finite && top[f] < 0x7ff;
    }
    // order 2 in FP64 takes no longer than four passes (10^6 particles on 128^3: 0.38 ms; one
    // pass 0.20 ms, weights over twelve decades, six passes, 0.57 ms)
    bool wide = false;
    if constexpr (M == 2)
        wide = top[0] - exponent_of_least(qmax_bits[kCtlLow]) > 3 * (kIxGap + 1) ||
               max(top[1], max(top[2], top[3])) - exponent_of_least(qmax_bits[kCtlLow + 1]) > 3 * (kIxGap + 1);
    if (!finite || wide || ng < C::R0 || ng < C::R1 || ng < T2 + C::HL + C::HR) {
        // infinities and NaN, a wide range of values, or a reach that wraps onto itself
        deposit_fp64_tile<double, M, T0, T1, T2, NT, 0>(rec, offsets, ng, sshift, grids, grid_elems,
                                                        reinterpret_cast<double *>(smem_raw), s_beg, s_pre);
        return;
    }
    const int ntz = ng / T2, nty = ng / T1;
    int tile = blockIdx.x;
    const int tz = tile % ntz;
    tile /= ntz;
    const int ty = tile % nty, tx = tile / nty;
    const int t0 = tx * T0, t1 = ty * T1, t2 = tz * T2;
    int *acc = reinterpret_cast<int *>(smem_raw) + L::FRONT;  // [4 fields][low, middle, high][TNP]
    auto clear = [&]() {
        for (int k = threadIdx.x; k < 3 * TNP; k += NT) reinterpret_cast<int4 *>(acc)[k] = make_int4(0, 0, 0, 0);
        if (threadIdx.x < 2) s_left[threadIdx.x] = 0;
    };
    clear();
    const uint32_t total = build_ranges<C>(offsets, ng, sshift, t0, t1, t2, T2, s_beg, s_pre);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, a = lane & 3, sub = lane >> 2;
    const int corner = a == 0 ? t0 : a == 1 ? t1 : t2, edge = a == 0 ? T0 : a == 1 ? T1 : T2;
    const int pitch = a == 0 ? L::PX : a == 1 ? L::RW : a == 2 ? 1 : 0;
    const bool node = lane < L::USED;
    const int offset = L::offset(lane);
    int *const stage = s_stage[warp];
    const unsigned mine = static_cast<unsigned>(__cvta_generic_to_shared(acc)) + 4 * offset;
    const int *const sx = stage + 2 * (node ? L::dx(lane) : 0), *const sy = stage + 2 * M + 2 * (node ? L::dy(lane) : 0),
              *const sz = stage + 4 * M + 2 * (node ? L::dz(lane) : 0), *const sq = stage + L::QQ + 2 * L::field(lane);

    // value(f, node's word in the low sums, its place in the grid) for every node of the tile
    auto nodes = [&](auto value) {
        for (int k = threadIdx.x; k < C::TN; k += NT) {
            const int l2 = k % T2, l01 = k / T2;
            const int l1 = l01 % T1, l0 = l01 / T1;
            const int64_t gi = (static_cast<int64_t>(t0 + l0) * ng + (t1 + l1)) * (ng + 2) + t2 + l2;
            if (!PK_IN(gi, grid_elems, kChkGrid)) continue;
#pragma unroll
            for (int f = 0; f < 4; ++f)
                value(f, acc + 3 * f * TNP + l0 * L::PX + l1 * L::RW + l2, grids + f * grid_elems + gi);
        }
    };
    int base_p = max(top[1], max(top[2], top[3]));
    for (int pass = 0;; ++pass) {
        auto emit = [&](bool high) {  // high: the grid nodes hold high sums
            nodes([&](int f, int *w, double *g) {
                const long long low = (static_cast<long long>(static_cast<unsigned>(w[TNP])) << kIxLow) +
                                      static_cast<unsigned>(w[0]);
                const long long hi = w[2 * TNP] + (low >> 44) + (high ? __double_as_longlong(*g) : 0ll);
                const double v = fixed_to_double(hi, low & ((1ll << 44) - 1), max(top[f], 1) - 1022 - 62);
                *g = pass ? *g + v : v;
            });
        };
        const int least_m = max(top[0] - kIxGap, 0) << 20, least_p = max(base_p - kIxGap, 0) << 20;
        bool high = false;
        for (uint32_t c0 = 0; c0 < total; c0 += kIxChunk) {
            const uint32_t cnt = min(total - c0, kIxChunk);
            if (c0) {  // carries: after at most 1023 adds
                __syncthreads();
                for (int k = threadIdx.x; k < 4 * TNP; k += NT) {
                    int *w = acc + (k / TNP) * 3 * TNP + k % TNP;
                    const unsigned lo = static_cast<unsigned>(w[0]);
                    const unsigned mid = static_cast<unsigned>(w[TNP]) + (lo >> kIxLow);
                    w[0] = static_cast<int>(lo & ((1u << kIxLow) - 1));
                    w[TNP] = static_cast<int>(mid & ((1u << kIxLow) - 1));
                    w[2 * TNP] += static_cast<int>(mid >> kIxLow);
                }
                __syncthreads();
                if (c0 % (kIxFlush * kIxChunk) == 0) {
                    if (pass) emit(false);
                    nodes([&](int, int *w, double *g) {
                        if (pass) w[0] = w[TNP] = 0;
                        else *g = __longlong_as_double(w[2 * TNP] + (high ? __double_as_longlong(*g) : 0ll));
                        w[2 * TNP] = 0;
                    });
                    high = pass == 0;
                    __syncthreads();
                }
            }
            const uint32_t share = ((cnt + NW - 1) / NW + L::NB - 1) / L::NB * L::NB;
            const uint32_t lo = min(cnt, warp * share), hi = min(cnt, lo + share);
            int slot = lo + sub < hi ? find_slot<C::MAXR>(s_pre, c0 + lo + sub) : 0;
            double v = 0.0, q[4] = {0.0, 0.0, 0.0, 0.0};
            uint32_t at = lo;
            int waiting = 0;  // particles in the queue
            // loads the next particles (at most eight, four lanes each) and returns their number:
            // in the first pass the next ones, later the next of the pass (32 looked at together)
            auto next_group = [&]() -> int {
                if (pass == 0) {
                    const int n = at < hi ? static_cast<int>(min(hi - at, static_cast<uint32_t>(L::NB))) : 0;
                    if (sub < n) {
                        const uint32_t p = c0 + at + sub;
                        while (p >= s_pre[slot + 1]) ++slot;
                        const Record<double> *r = rec + s_beg[slot] + (p - s_pre[slot]);
                        v = reinterpret_cast<const double *>(r)[a];
                        if (a == 3) q[0] = r->q.x, q[1] = r->q.y, q[2] = r->q.z, q[3] = r->q.w;
                    }
                    at += L::NB;
                    return n;
                }
                uint32_t *const queue = s_queue[warp];
                while (waiting < L::NB && at < hi) {
                    bool member = false;
                    uint32_t i = 0;
                    if (at + lane < hi) {
                        const int k = find_slot<C::MAXR>(s_pre, c0 + at + lane);
                        i = s_beg[k] + (c0 + at + lane - s_pre[k]);
                        const Vec4<double> x = rec[i].q;
                        const double y[4] = {x.x, x.y, x.z, x.w};
                        bool heavy, fast;
                        member = in_pass(y, top[0], base_p, s_left, heavy, fast);
                    }
                    const unsigned m = __ballot_sync(full, member);
                    if (member) queue[waiting + __popc(m & ((1u << lane) - 1u))] = i;
                    waiting += __popc(m);
                    at += 32;
                    __syncwarp();
                }
                const int n = min(waiting, L::NB);
                if (sub < n) {
                    const Record<double> *r = rec + queue[sub];
                    v = reinterpret_cast<const double *>(r)[a];
                    if (a == 3) q[0] = r->q.x, q[1] = r->q.y, q[2] = r->q.z, q[3] = r->q.w;
                }
                __syncwarp();
                waiting -= n;
                const uint32_t moved = lane < waiting ? queue[lane + n] : 0u;
                __syncwarp();
                if (lane < waiting) queue[lane] = moved;
                __syncwarp();
                return n;
            };
            for (int nb = next_group(); nb;) {
                // the particles of this pass (lane 3 of four) are staged side by side: nearly always
                // all of them, whole, in the first pass
                bool heavy = true, fast = true;
                unsigned taken = 0x88888888u >> (32 - 4 * nb);
                const bool below = high_word(q[0]) < least_m ||
                                   max(high_word(q[1]), max(high_word(q[2]), high_word(q[3]))) < least_p;
                if (pass || __any_sync(full, a == 3 && sub < nb && below)) {
                    heavy = fast = false;
                    if (a == 3 && sub < nb) in_pass(q, top[0], base_p, s_left, heavy, fast);
                    taken = __ballot_sync(full, heavy || fast);
                    if (!taken) {
                        nb = next_group();
                        continue;
                    }
                }
                const int packed = __shfl_sync(full, unpack_cell(v), lane | 3);
                // the offset in the cell (in [0, 1]) as a 63-bit fraction
                const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(a == 3 ? 0.0 : v));
                const int e = static_cast<int>(bits >> 52) - 1012;
                unsigned long long t = (bits & ((1ull << 52) - 1)) | 1ull << 52;
                t = e >= 0 ? t << e : e > -53 ? t >> -e : 0ull;
                unsigned long long w[M];
                int first;
                fixed_weights<M>(t, w, first);
                int d = ((packed >> (10 * min(a, 2))) & 1023) - corner;
                d = d < -C::HL ? d + ng : (d >= edge + C::HR ? d - ng : d);
                d += first;
                int word = d * pitch;
                word += __shfl_xor_sync(full, word, 1);
                word += __shfl_xor_sync(full, word, 2);
                int *const st = stage + __popc(taken & ((1u << (lane & ~3)) - 1u)) * L::STRIDE;
                if (taken & (8u << (lane & ~3))) {
                    if (a < 3) {
#pragma unroll
                        for (int k = 0; k < M; ++k) {
                            // 62 bits (one itself just below), zero outside the tile
                            const bool in = static_cast<unsigned>(d + k) < static_cast<unsigned>(edge);
                            const unsigned long long x = in ? min(w[k] >> 1, (1ull << 62) - 1) : 0ull;
                            *reinterpret_cast<int2 *>(st + 2 * (a * M + k)) =
                                make_int2(static_cast<int>(x >> 31), static_cast<int>(x & 0x7fffffffu));
                        }
                    } else {
#pragma unroll
                        for (int f = 0; f < 4; ++f) {
                            const long long x = (f ? fast : heavy) ? fixed_value(q[f], top[f]) : 0ll;
                            *reinterpret_cast<int2 *>(st + L::QQ + 2 * f) =
                                make_int2(static_cast<int>(x >> 31), static_cast<int>(x & 0x7fffffffll));
                        }
                        st[L::QQ + 8] = word;
                    }
                }
                __syncwarp();
                nb = next_group();
#pragma unroll 2
                for (int p = 0; p < __popc(taken); ++p) {
                    const int o = p * L::STRIDE;
                    const int2 x = *reinterpret_cast<const int2 *>(sx + o), y = *reinterpret_cast<const int2 *>(sy + o);
                    const unsigned addr = mine + static_cast<unsigned>(4 * stage[L::QQ + 8 + o]);
                    auto mul = [](int2 u, int2 w) {  // u w / 2^62 of values in words of 31 bits
                        const long long cross = static_cast<long long>(u.x) * w.y + static_cast<long long>(u.y) * w.x;
                        return static_cast<long long>(u.x) * w.x + (cross >> 31);
                    };
                    auto split = [](long long u) {
                        return make_int2(static_cast<int>(u >> 31), static_cast<int>(u & 0x7fffffffll));
                    };
                    int2 xy = split(mul(x, y));
                    if (L::USED < 32 && !node) xy = make_int2(0, 0);
                    static_for<L::NZ>([&](auto kc) {
                        constexpr int k = decltype(kc)::value;
                        const int2 ww = split(mul(xy, *reinterpret_cast<const int2 *>(sz + o + 2 * k)));
                        static_for<L::NF>([&](auto fc) {
                            constexpr int f = decltype(fc)::value;
                            const long long c = mul(*reinterpret_cast<const int2 *>(sq + o + 2 * f), ww);
                            if (!PK_IN(stage[L::QQ + 8 + o] + offset + L::FRONT + k + 3 * f * TNP + 2 * TNP,
                                       L::FRONT + 12 * TNP + L::BACK, kChkShared))
                                return;
                            red3<4 * (k + 3 * f * TNP), 4 * TNP>(addr, static_cast<int>(c) & ((1 << kIxLow) - 1),
                                                                 static_cast<int>(c >> kIxLow) & ((1 << kIxLow) - 1),
                                                                 static_cast<int>(c >> (2 * kIxLow)));
                        });
                    });
                }
                __syncwarp();
            }
        }
        __syncthreads();
        const int left_m = s_left[0], left_p = s_left[1];
        emit(high);
        if (left_m == 0 && left_p == 0) break;
        __syncthreads();
        clear();
        top[0] = left_m - 1;  // -1: no mass in the next pass
        top[1] = top[2] = top[3] = base_p = left_p - 1;
        __syncthreads();
    }
}

// Cell-block path of the FP32 deposit for dense tiles (cubic order): one
// warp per occupied cell of the reach; lane l owns stencil nodes (dx, dy, dz) with
// dz = l & 3, dy = (l >> 2) & 3, dx = (l >> 4) and (l >> 4) + 2, evaluates its weight
// pieces by Horner's rule with lane-constant coefficients, sums up to kCellFlush of the
// cell's particles (records read once, broadcast) in FP32 registers and adds the sums to
// the shared accumulator as fixed-point integers (one rounding per sum).
constexpr int kCellFlush = 256;

__device__ __forceinline__ float horner4(const float (&c)[4], float t) { return c[0] + t * (c[1] + t * (c[2] + t * c[3])); }

// coefficients of the cubic B-spline weight of stencil node k (0..3) in t = u - floor(u)
__device__ __forceinline__ void cubic_piece(int k, float (&c)[4])
{
    const float s = 1.0f / 6.0f;
    if (k == 0) c[0] = s, c[1] = -3 * s, c[2] = 3 * s, c[3] = -s;
    else if (k == 1) c[0] = 4 * s, c[1] = 0.f, c[2] = -6 * s, c[3] = 3 * s;
    else if (k == 2) c[0] = s, c[1] = 3 * s, c[2] = 3 * s, c[3] = -3 * s;
    else c[0] = 0.f, c[1] = 0.f, c[2] = 0.f, c[3] = s;
}

__device__ __forceinline__ int round_shift(int v, int d) { return d > 0 ? (v + (1 << (d - 1))) >> d : v; }

// Weight pieces of a lane's two stencil nodes (dx, dx + 2; dy; dz) in the cell-block paths.
struct CellPieces {
    float xa[4], xb[4], y[4], z[4];
};

// Sums of one chunk (at most kCellFlush particles) of a cell for a lane's two stencil
// nodes. Each contribution is rounded once to the fine scale 2^sf (below 2^22 in
// magnitude: one FFMA against 1.5 * 2^23) and added as an integer; the chunk sum is then
// rounded to the tile scale by a right shift of sf - st bits. Integer sums: the result
// does not depend on the order in which the sort left the cell's particles.
// With z >= 0 only the particles of cells at that z count (keys of several cells), at most
// kCellFlush of them; returns where the next chunk starts.
template <int F0 = 0, int NF = 4>
__device__ __forceinline__ uint32_t cell_chunk(const Record<float> *__restrict__ rec, uint32_t i0, uint32_t i1,
                                           const CellPieces &pc, const float (&fine)[4], const int (&shift)[4],
                                           int (&a)[NF], int (&b)[NF], int z = -1)
{
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr int kMagicBits = 0x4B400000;
    int sa[NF], sb[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) sa[f] = 0, sb[f] = 0;
    auto add = [&](const Record<float> &rc) {
        const float wyz = horner4(pc.y, rc.u.y) * horner4(pc.z, rc.u.z);
        const float wa = horner4(pc.xa, rc.u.x) * wyz, wb = horner4(pc.xb, rc.u.x) * wyz;
        const float qv[4] = {rc.q.x, rc.q.y, rc.q.z, rc.q.w};
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const float q = qv[F0 + f] * fine[F0 + f];
            sa[f] += __float_as_int(fmaf(q, wa, kMagic)) - kMagicBits;
            sb[f] += __float_as_int(fmaf(q, wb, kMagic)) - kMagicBits;
        }
    };
    uint32_t i = i0;
    if (z >= 0) {  // the cells of 32 records are read together, then the records of this cell
        const uint32_t lane = threadIdx.x & 31;
        auto cell_z = [&](uint32_t at) { return at + lane < i1 ? unpack_cell(rec[at + lane].u.w) >> 20 : -1; };
        int next = cell_z(i);
        for (int n = 0; i < i1; i += 32) {
            unsigned m = __ballot_sync(0xffffffffu, next == z);
            n += __popc(m);
            if (n > kCellFlush) break;  // the next chunk starts with these
            next = cell_z(i + 32);
            auto take = [&]() {
                const uint32_t k = i + __ffs(static_cast<int>(m)) - 1;
                m &= m - 1u;
                return load_record(rec + k);
            };
            while (__popc(m) >= 4) {  // four loads in flight
                const Record<float> r0 = take(), r1 = take(), r2 = take(), r3 = take();
                add(r0);
                add(r1);
                add(r2);
                add(r3);
            }
            while (m) add(take());
        }
        i1 = i;
    }
    for (; i + 4 <= i1; i += 4) {  // four loads in flight
        const Record<float> r0 = load_record(rec + i), r1 = load_record(rec + i + 1), r2 = load_record(rec + i + 2),
                            r3 = load_record(rec + i + 3);
        add(r0);
        add(r1);
        add(r2);
        add(r3);
    }
    for (; i < i1; ++i) add(load_record(rec + i));
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        a[f] = round_shift(sa[f], shift[F0 + f]);
        b[f] = round_shift(sb[f], shift[F0 + f]);
    }
    return i1;
}

// Fixed-point scales of a tile: 2^st with (bound of any node sum) * 2^st < 2^30, and,
// for the cell-block paths, the fine scale 2^sf with (largest contribution) * 2^sf < 2^22
// and st <= sf. Per-particle paths round at 2^min(st, sf) directly. A node's integer sum
// is then below 2^30 plus half a unit per rounding (fewer than 2^31 particles), which
// fits a signed 32-bit accumulator.
__device__ __forceinline__ void tile_scales(float bound, float cmax, bool cells, float &scale, float &fine, int &shift)
{
    int eb = 0, ec = 0;
    if (bound > 0.f) frexpf(bound, &eb);  // bound < 2^eb
    if (cmax > 0.f) frexpf(cmax, &ec);
    if (!isfinite(bound)) eb = 150;
    if (!isfinite(cmax)) ec = 150;
    auto clampx = [](int e) { return e > 120 ? 120 : (e < -120 ? -120 : e); };
    const int sf = clampx(22 - ec), st = clampx(min(30 - eb, 22 - ec));
    scale = ldexpf(1.0f, st);
    fine = ldexpf(1.0f, sf);
    shift = cells ? min(30, sf - st) : 0;
}

template <int T0, int T1, int T2, int NT>
__device__ __forceinline__ void deposit_cells_path(const Record<float> *__restrict__ rec,
                                                   const uint32_t *__restrict__ offsets, int ng, int sshift, int t0,
                                                   int t1, int t2, int *acc, int fstride, int px, int rw, const float *s_fine,
                                                   const int *s_shift)
{
    constexpr int HL = 2, R0 = T0 + 3, R1 = T1 + 3, RZ = T2 + 3, NW = NT / 32;
    const float fine[4] = {s_fine[0], s_fine[1], s_fine[2], s_fine[3]};
    const int shift[4] = {s_shift[0], s_shift[1], s_shift[2], s_shift[3]};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int dz = lane & 3, dy = (lane >> 2) & 3, dxl = lane >> 4;
    CellPieces pc;
    cubic_piece(dxl, pc.xa);
    cubic_piece(dxl + 2, pc.xb);
    cubic_piece(dy, pc.y);
    cubic_piece(dz, pc.z);
    auto wrapi = [ng](int a) { return a < 0 ? a + ng : (a >= ng ? a - ng : a); };
    for (int c = warp; c < R0 * R1 * RZ; c += NW) {
        const int r = c / RZ, zz = c % RZ;
        const int cx = r / R1 - HL, cy = r % R1 - HL, cz = zz - HL;  // cell relative to the tile
        const int z = wrapi(t2 + cz);
        const int64_t key =
            (static_cast<int64_t>(wrapi(t0 + cx)) * ng + wrapi(t1 + cy)) * (ng >> sshift) + (z >> sshift);
        const uint32_t beg = offsets[key], end = offsets[key + 1];
        if (beg == end) continue;
        const int lxa = cx - 1 + dxl, lxb = lxa + 2, ly = cy - 1 + dy, lz = cz - 1 + dz;
        const bool yz = ly >= 0 && ly < T1 && lz >= 0 && lz < T2;
        const bool ina = yz && lxa >= 0 && lxa < T0, inb = yz && lxb >= 0 && lxb < T0;
        const int oa = lxa * px + ly * rw + lz, ob = (lxa + 2) * px + ly * rw + lz;
        for (uint32_t i0 = beg; i0 < end;) {
            int a[4], b[4];
            i0 = T2 >= 16 && sshift ? cell_chunk(rec, i0, end, pc, fine, shift, a, b, z)
                        : cell_chunk(rec, i0, min(end, i0 + kCellFlush), pc, fine, shift, a, b);
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                if (ina) atomicAdd(acc + f * fstride + oa, a[f]);
                if (inb) atomicAdd(acc + f * fstride + ob, b[f]);
            }
        }
    }
}

// Shared accumulator of the FP32 gather deposit: four fields of TNP ints per tile, node
// (x, y, z) at x * PX + y * RW + z. The pitches are the smallest for which the 32 lanes of
// an add fall on 32 different banks: orders 4 and 5 in the lane mapping of CoopLanes (one
// particle per warp; checked below); the lower orders take an odd row pitch and an odd plane
// pitch, so that the bank of a node, (x PX + y RW + z) mod 32, mixes all three coordinates
// (with PX = 16 mod 32, x would add only its parity).
//
// The listed paths add every stencil node of every particle, with the weights of nodes
// outside the tile set to zero (an add of exactly 0), at an address formed by the same
// linear rule; such a node lies at most 5 nodes below or 4 above the tile on each axis
// (orders 1 to 5), so the allocation has FRONT words of padding before the accumulator and
// at least BACK words after it (the particle list or padding). The zero adds land on
// padding, on other nodes or on list entries, and change none of them.
template <int M, int T0, int T1, int T2>
struct FxLayout {
    static constexpr bool COOP = M == 4 || M == 5;
    static constexpr int RW = M == 4 && T2 == 8 ? 8 : T2 + 1;
    static constexpr int PX = T1 * RW + (M == 4   ? (T2 == 8 ? 1 : T2 == 32 ? (T1 == 8 ? 0 : 4) : 4)
                                         : M == 5 ? (T2 == 8 ? 2 : T2 == 32 ? (T1 == 8 ? 5 : 3) : 5)
                                                  : 3);
    static constexpr int TNP = T0 * PX + (M == 4 ? (T1 == 8 ? 2 : 8) : 0);  // ints per field
    static constexpr int FRONT = (5 * (PX + RW + 1) + 3) / 4 * 4;
    static constexpr int BACK = 4 * PX + (T1 + 4) * RW + T2 + 5;
    static size_t bytes(int list_cap)
    {
        return size_t(FRONT + 4 * TNP + (list_cap > BACK ? list_cap : BACK)) * sizeof(int);
    }
};

// Every node the listed paths add to (weights of nodes outside the tile zero) lies in the
// padded allocation, for particles of cells within reach of the tile, or for which the reach
// test of the list holds (with keys of several cells the runs hold others too, whose
// coordinates can be off by ng: the list and coop_deposit leave those out): node coordinates run from -HL + first(0) to (T + HR - 1) + first(1/2)
// + M - 1 on each axis (first is smallest at t = 0 and largest from t = 1/2 on).
template <int M, int T0, int T1, int T2>
constexpr bool fx_pads_cover()
{
    using Lay = FxLayout<M, T0, T1, T2>;
    constexpr int HL = (M % 2 == 0) ? M / 2 : (M + 1) / 2;
    constexpr int HR = (M % 2 == 0) ? M / 2 - 1 : (M - 1) / 2;
    constexpr int lo = -HL + bspline_first<M, float>(0.0f);
    constexpr int up = HR - 1 + bspline_first<M, float>(0.5f) + M - 1;  // highest coordinate - T
    constexpr long min_lin = static_cast<long>(lo) * (Lay::PX + Lay::RW + 1);
    constexpr long max_lin = static_cast<long>(T0 + up) * Lay::PX + static_cast<long>(T1 + up) * Lay::RW + (T2 + up) +
                             3L * Lay::TNP;
    return min_lin >= -Lay::FRONT && max_lin < 4L * Lay::TNP + Lay::BACK;
}
template <int T0, int T1, int T2>
constexpr bool fx_pads_cover_orders()
{
    return fx_pads_cover<1, T0, T1, T2>() && fx_pads_cover<2, T0, T1, T2>() && fx_pads_cover<3, T0, T1, T2>() &&
           fx_pads_cover<4, T0, T1, T2>() && fx_pads_cover<5, T0, T1, T2>();
}
static_assert(fx_pads_cover_orders<16, 16, 16>() && fx_pads_cover_orders<16, 16, 32>() &&
                  fx_pads_cover_orders<8, 8, 32>() && fx_pads_cover_orders<8, 8, 8>(),
              "the padding of the gather accumulator must cover every node the listed path adds to");

// Pairs of FP32 values in one 64-bit register pair for the paired FP32 FMA of sm_100
// and later (fma.rn.f32x2: two correctly rounded FMAs per instruction issued, each the
// same result as the scalar instruction).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 f2_pack(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Four shared-memory adds at byte offsets OFF + f * FS (f = 0..3) from addr (the offsets
// are immediates).
template <int OFF, int FS>
__device__ __forceinline__ void red4(unsigned addr, int v0, int v1, int v2, int v3)
{
    asm volatile(
        "red.shared.add.s32 [%0+%5], %1;\n\t"
        "red.shared.add.s32 [%0+%6], %2;\n\t"
        "red.shared.add.s32 [%0+%7], %3;\n\t"
        "red.shared.add.s32 [%0+%8], %4;" ::"r"(addr),
        "r"(v0), "r"(v1), "r"(v2), "r"(v3), "n"(OFF), "n"(OFF + FS), "n"(OFF + 2 * FS), "n"(OFF + 3 * FS));
}

template <int OFF, int FS>
__device__ __forceinline__ void red2(unsigned addr, int v0, int v1)
{
    asm volatile(
        "red.shared.add.s32 [%0+%3], %1;\n\t"
        "red.shared.add.s32 [%0+%4], %2;" ::"r"(addr), "r"(v0), "r"(v1), "n"(OFF), "n"(OFF + FS));
}

// Tile-local coordinates of the first stencil node of a particle in the tile's reach,
// where no periodic wrap falls inside the reach (ng >= tile + M cells): the cell offset
// from the tile's corner is taken into [-HL, T + HR).
template <int M, int HL, int HR, int T>
__device__ __forceinline__ int first_node(float t, int cell, int corner, int ng)
{
    int d = cell - corner;
    d = d < -HL ? d + ng : (d >= T + HR ? d - ng : d);
    return d + bspline_first<M, float>(t);
}

// A value on the tile's scale for the listed paths, which add value times weight to nodes
// outside the tile too, relying on weight zero: NaN and infinities, whose product with zero is
// not zero, become the largest value of the scale (finite values are below it: tile_scales).
// Without this a NaN velocity changed other nodes and list entries, that is, record indices.
template <int M>
__device__ __forceinline__ float listed_value(float q, float scale)
{
    constexpr float top = 4194304.0f / kMaxWeight3<M>;  // weights times value below 2^22
    return fminf(fmaxf(q * scale, -top), top);
}

// One particle of the reordered list (see k_deposit_fx): its M^3 stencil nodes at
// immediate offsets from the shared-window address of its first node, with the weights of
// nodes outside the tile set to zero (no branch or predicate per node; see FxLayout). The
// contributions of the nodes in the tile are those of the per-node path.
template <int M, int T0, int T1, int T2, int HL, int HR>
__device__ __forceinline__ void banked_particle(const Record<float> &r, int ng, int t0, int t1, int t2, unsigned acc_s,
                                                float sc0, float sc1, float sc2, float sc3)
{
    using Lay = FxLayout<M, T0, T1, T2>;
    constexpr int RW = Lay::RW, PX = Lay::PX, TNP = Lay::TNP;
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr int kMagicBits = 0x4B400000;
    const int packed = unpack_cell(r.u.w);
    float w[3][M];
    int first;
    bspline_weights<M, float>(r.u.x, w[0], first);
    bspline_weights<M, float>(r.u.y, w[1], first);
    bspline_weights<M, float>(r.u.z, w[2], first);
    const int b0 = first_node<M, HL, HR, T0>(r.u.x, packed & 1023, t0, ng);
    const int b1 = first_node<M, HL, HR, T1>(r.u.y, (packed >> 10) & 1023, t1, ng);
    const int b2 = first_node<M, HL, HR, T2>(r.u.z, (packed >> 20) & 1023, t2, ng);
#pragma unroll
    for (int k = 0; k < M; ++k) {
        w[0][k] = static_cast<unsigned>(b0 + k) < static_cast<unsigned>(T0) ? w[0][k] : 0.0f;
        w[1][k] = static_cast<unsigned>(b1 + k) < static_cast<unsigned>(T1) ? w[1][k] : 0.0f;
        w[2][k] = static_cast<unsigned>(b2 + k) < static_cast<unsigned>(T2) ? w[2][k] : 0.0f;
    }
    // (the first node may lie below the accumulator, inside the front padding)
    // the first node where a particle of the tile's reach can have it (cell offset in
    // [-HL, T + HR) plus the first node's offset from the cell), which FxLayout's padding
    // covers (fx_pads_cover)
    constexpr int LO = -HL + bspline_first<M, float>(0.0f), HI = HR - 1 + bspline_first<M, float>(0.5f);
    if (!PK_IN(b0 - LO, T0 + HI - LO + 1, kChkShared) || !PK_IN(b1 - LO, T1 + HI - LO + 1, kChkShared) ||
        !PK_IN(b2 - LO, T2 + HI - LO + 1, kChkShared))
        return;
    const unsigned base = acc_s + 4u * static_cast<unsigned>(b0 * PX + b1 * RW + b2);
    const float qs[4] = {listed_value<M>(r.q.x, sc0), listed_value<M>(r.q.y, sc1), listed_value<M>(r.q.z, sc2),
                         listed_value<M>(r.q.w, sc3)};
    f32x2 qp[4], zp[(M + 1) / 2];  // each value twice, the z weights in pairs (fma.rn.f32x2)
#pragma unroll
    for (int f = 0; f < 4; ++f) qp[f] = f2_pack(qs[f], qs[f]);
#pragma unroll
    for (int k = 0; k < M; k += 2) zp[k / 2] = f2_pack(w[2][k], k + 1 < M ? w[2][k + 1 < M ? k + 1 : k] : 0.0f);
    const f32x2 mg = f2_pack(kMagic, kMagic);
    auto row = [&](auto k0c, auto k1c) {
        constexpr int k0 = decltype(k0c)::value, k1 = decltype(k1c)::value;
        const float w01 = w[0][k0] * w[1][k1];
        const f32x2 w2 = f2_pack(w01, w01);
        static_for<(M + 1) / 2>([&](auto hc) {
            constexpr int k2 = 2 * decltype(hc)::value;
            const f32x2 ww = f2_mul(w2, zp[k2 / 2]);
            f32x2 t[4];
#pragma unroll
            for (int f = 0; f < 4; ++f) t[f] = f2_fma(qp[f], ww, mg);
            red4<4 * (k0 * PX + k1 * RW + k2), 4 * TNP>(base, static_cast<int>(t[0]) - kMagicBits,
                                                        static_cast<int>(t[1]) - kMagicBits,
                                                        static_cast<int>(t[2]) - kMagicBits,
                                                        static_cast<int>(t[3]) - kMagicBits);
            if constexpr (k2 + 1 < M)
                red4<4 * (k0 * PX + k1 * RW + k2 + 1), 4 * TNP>(base, static_cast<int>(t[0] >> 32) - kMagicBits,
                                                                static_cast<int>(t[1] >> 32) - kMagicBits,
                                                                static_cast<int>(t[2] >> 32) - kMagicBits,
                                                                static_cast<int>(t[3] >> 32) - kMagicBits);
        });
    };
    static_for<M>([&](auto k0c) { static_for<M>([&](auto k1c) { row(k0c, k1c); }); });
}

// One particle per warp (orders 4 and 5). A lane owns fixed stencil nodes of whatever
// particle the warp deposits: order 4: lane (dx, dy, h), the four z nodes of node column
// (dx, dy), fields 2h and 2h + 1; order 5: lane (dx, dy) of 25, five z nodes, all four
// fields. The lanes of an add touch different banks, so an add is one wavefront whatever the
// particles are, where 32 lanes with a particle each serialise on a crowded cell. The
// weights are evaluated once per particle and axis by four lanes (three axes and the scaled
// values) for eight particles at a time, staged in shared memory and read back by all lanes;
// nodes outside the tile get weight zero and add exactly 0 (FxLayout's padding; a predicate
// per add compiled to branches and took twice the instructions). Every contribution is the
// same rounded integer as on the per-node path. Bound by issue and the shared pipe, about 15
// wavefronts a particle of the reach: particles in random cells are faster a particle per
// lane (13), crowded ones here: 8 M particles, 40 % of them in halos, on 256^3: deposit 3.2
// ms a particle per lane, 1.03 ms with this.
template <int M, int T0, int T1, int T2>
struct CoopLanes {
    using Lay = FxLayout<M, T0, T1, T2>;
    static constexpr int NF = M == 4 ? 2 : 4;          // fields per lane
    static constexpr int WP = M == 4 ? 4 : 8;          // staged words per axis
    static constexpr int QW = 3 * WP;                  // the scaled values, then the node word
    static constexpr int STRIDE = M == 4 ? 20 : 32;    // staged words per particle
    static constexpr int NB = 8;                       // particles staged at a time
    // About the wavefronts of a particle. Whole calls with half and twice of it over this: 10 M
    // uniform particles on 200^3 1.05 and 1.01 (order 4), 1.41 and 1.00 (order 5); 1 M in halos on
    // 128^3 1.03 and 1.21, 1.06 and 1.03. On 8^3 tiles, where a particle's visits are mostly zero
    // adds, order 4 with 16, 20 and 26 over a branch per node: lattices of 0.2 a cell on 264^3 1.014,
    // 1.002 and 0.997, uniform ones 0.978, 0.970 and 0.966, in halos 0.77, 0.79 and 0.81
    static constexpr int COST = M == 4 ? (T2 == 8 ? 20 : 16) : 30;
    __host__ __device__ static constexpr int dx(int lane) { return M == 4 ? (lane >> 2) & 3 : lane / 5; }
    __host__ __device__ static constexpr int dy(int lane) { return M == 4 ? lane & 3 : lane % 5; }
    __host__ __device__ static constexpr int half(int lane) { return M == 4 ? lane >> 4 : 0; }
    static constexpr int USED = M == 4 ? 32 : 25;
    __host__ __device__ static constexpr int node_offset(int lane)  // words from the particle's first node
    {
        return dx(lane) * Lay::PX + dy(lane) * Lay::RW + half(lane) * 2 * Lay::TNP;
    }
    // banks no node lane uses (all node lanes' banks differ), and the offset of a lane: that
    // of its node, or for the lanes without one the next free bank
    static constexpr unsigned free_banks()
    {
        unsigned seen = 0;
        for (int l = 0; l < USED; ++l) seen |= 1u << (node_offset(l) & 31);
        return ~seen;
    }
    static constexpr bool banks_distinct()
    {
        int n = 0;
        for (unsigned m = free_banks(); m; m &= m - 1) ++n;
        return n == 32 - USED;
    }
    __device__ static int offset(int lane)
    {
        if (lane < USED) return node_offset(lane);
        unsigned m = free_banks();
        for (int l = USED; l < lane; ++l) m &= m - 1;
        return __ffs(static_cast<int>(m)) - 1;
    }
};
template <int T0, int T1, int T2>
constexpr bool coop_banks_distinct()
{
    return CoopLanes<4, T0, T1, T2>::banks_distinct() && CoopLanes<5, T0, T1, T2>::banks_distinct();
}
static_assert(coop_banks_distinct<16, 16, 16>() && coop_banks_distinct<16, 16, 32>() &&
                  coop_banks_distinct<8, 8, 32>() && coop_banks_distinct<8, 8, 8>(),
              "the lanes of a one-particle-per-warp add must hit different banks");

// Deposits the list positions pos(0 .. count - 1) of one warp; record(p) is the record index
// of position p (called by the four lanes of a particle). stage: NB * STRIDE words of the
// warp. acc: the tile's accumulator (FxLayout).
template <int M, int T0, int T1, int T2, int HL, int HR, class Record_of>
__device__ __forceinline__ void coop_deposit(const Record<float> *__restrict__ rec, Record_of record, uint32_t count,
                                             int ng, int t0, int t1, int t2, int *acc, float *stage, float sc0,
                                             float sc1, float sc2, float sc3)
{
    using C = CoopLanes<M, T0, T1, T2>;
    using Lay = FxLayout<M, T0, T1, T2>;
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr int kMagicBits = 0x4B400000;
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, a = lane & 3, sub = lane >> 2;
    // this lane's axis as a stager
    const int corner = a == 0 ? t0 : a == 1 ? t1 : t2, edge = a == 0 ? T0 : a == 1 ? T1 : T2;
    const int pitch = a == 0 ? Lay::PX : a == 1 ? Lay::RW : a == 2 ? 1 : 0;
    // this lane's nodes as an adder (lanes without a node take a weight of zero)
    const int dx = C::dx(lane), dy = C::dy(lane);
    const unsigned mine = static_cast<unsigned>(__cvta_generic_to_shared(acc)) + 4 * C::offset(lane);
    const float *const sx = stage + (lane < C::USED ? dx : C::WP - 1), *const sy = stage + C::WP + min(dy, M - 1),
                *const sz = stage + 2 * C::WP, *const sq = stage + C::QW + (M == 4 ? 4 * C::half(lane) : 0);

    float v = 0.0f;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](uint32_t at) {
        if (at + sub < count) {
            const Record<float> *r = rec + record(at + sub);
            v = reinterpret_cast<const float *>(r)[a];
            if (a == 3) q = make_float4(r->q.x, r->q.y, r->q.z, r->q.w);
        }
    };
    fetch(0);
    for (uint32_t at = 0; at < count; at += C::NB) {
        const int nb = static_cast<int>(min(count - at, static_cast<uint32_t>(C::NB)));
        // weights of one axis per lane, zero outside the tile
        float w[M];
        int first;
        const int packed = __shfl_sync(full, __float_as_int(v), lane | 3);
        const float t = a == 3 ? 0.0f : v;
        bspline_weights<M, float>(t, w, first);
        int d = ((packed >> (10 * min(a, 2))) & 1023) - corner;
        d = d < -HL ? d + ng : (d >= edge + HR ? d - ng : d);
        d += first;
#pragma unroll
        for (int k = 0; k < M; ++k) w[k] = static_cast<unsigned>(d + k) < static_cast<unsigned>(edge) ? w[k] : 0.0f;
        // the first node, summed over the axes; node 0, with weights of zero, for a particle
        // that does not reach the tile (keys of several cells)
        const unsigned reaches = __ballot_sync(full, a == 3 || (d > -M && d < edge));
        const bool in = ((reaches >> (lane & ~3)) & 15u) == 15u;
        if (!in) w[0] = w[1] = w[2] = w[M - 1] = w[3] = 0.0f;
        int word = in ? d * pitch : 0;
        word += __shfl_xor_sync(full, word, 1);
        word += __shfl_xor_sync(full, word, 2);
        float *const st = stage + sub * C::STRIDE;
        if (sub < nb) {
            if (a < 3) {
                float4 *o = reinterpret_cast<float4 *>(st + a * C::WP);
                o[0] = make_float4(w[0], w[1], w[2], w[3]);
                if constexpr (M == 5) o[1] = make_float4(w[4], 0.f, 0.f, 0.f);
            } else {
                const float wf = __int_as_float(word);
                float4 *o = reinterpret_cast<float4 *>(st + C::QW);
                const float4 qs = make_float4(listed_value<M>(q.x, sc0), listed_value<M>(q.y, sc1),
                                              listed_value<M>(q.z, sc2), listed_value<M>(q.w, sc3));
                if constexpr (M == 4) {
                    o[0] = make_float4(qs.x, qs.y, wf, 0.f);
                    o[1] = make_float4(qs.z, qs.w, wf, 0.f);
                } else {
                    o[0] = qs;
                    st[C::QW + 4] = wf;
                }
            }
        }
        __syncwarp();
        fetch(at + C::NB);
#pragma unroll 4
        for (int p = 0; p < nb; ++p) {
            const int o = p * C::STRIDE;
            const float4 qv = *reinterpret_cast<const float4 *>(sq + o);
            const float w01 = sx[o] * sy[o];
            int c[M][C::NF];
            int word_p;
            if constexpr (M == 4) {
                word_p = __float_as_int(qv.z);
                const float4 wz = *reinterpret_cast<const float4 *>(sz + o);
                const f32x2 ww = f2_pack(w01, w01), mg = f2_pack(kMagic, kMagic);
                const f32x2 wa = f2_mul(ww, f2_pack(wz.x, wz.y)), wb = f2_mul(ww, f2_pack(wz.z, wz.w));
                const float qf[2] = {qv.x, qv.y};
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const f32x2 qq = f2_pack(qf[f], qf[f]);
                    const f32x2 lo = f2_fma(qq, wa, mg), hi = f2_fma(qq, wb, mg);
                    c[0][f] = static_cast<int>(lo), c[1][f] = static_cast<int>(lo >> 32);
                    c[2][f] = static_cast<int>(hi), c[3][f] = static_cast<int>(hi >> 32);
                }
            } else {
                word_p = __float_as_int(sq[o + 4]);
                const float qf[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
                for (int k = 0; k < M; ++k) {
                    const float ww = w01 * sz[o + k];
#pragma unroll
                    for (int f = 0; f < 4; ++f) c[k][f] = __float_as_int(fmaf(qf[f], ww, kMagic));
                }
            }
            const unsigned addr = mine + static_cast<unsigned>(4 * word_p);
            // its last add, of the last field and z node, lies in the padded accumulator
            if (!PK_IN(word_p + C::offset(lane) + Lay::FRONT, Lay::FRONT + (5 - C::NF) * Lay::TNP + Lay::BACK - M,
                       kChkShared))
                continue;
            static_for<M>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                if constexpr (C::NF == 2)
                    red2<4 * k, 4 * Lay::TNP>(addr, c[k][0] - kMagicBits, c[k][1] - kMagicBits);
                else
                    red4<4 * k, 4 * Lay::TNP>(addr, c[k][0] - kMagicBits, c[k][1] - kMagicBits, c[k][2] - kMagicBits,
                                              c[k][3] - kMagicBits);
            });
        }
        __syncwarp();
    }
}

// Tile-gather deposit for FP32 grids with 32-bit integer (fixed-point) shared-memory
// atomics (about three times the throughput of FP32 shared atomics on this part).
//
// Work split: orders 4 and 5, and sparse catalogues at orders 1 to 3, list a tile's
// particles in shared memory, a few thousand at a time, and deposit them a particle per lane
// (banked_particle: the list reordered so that 32 consecutive entries have their first
// stencil nodes in different banks, every node at an immediate offset, nodes outside the
// tile adding exactly 0) or, crowded lists at orders 4 and 5, a particle per warp
// (coop_deposit). The rest (orders 1 to 3 from half a particle per cell on or with a list too
// long, the direct BL stencil, a reach that wraps onto itself) goes node by node: each warp
// walks its own contiguous chunk of the tile's particles, lane j taking the j-th of each 32.
// Tiles with more than two particles per reach cell (cubic order) take the cell-block path.
// The accumulator layout is FxLayout.
//
// Fixed point: field f of the tile uses the scale 2^s_f with
//   B_f 2^s_f < 2^30,   B_f = w3 * min(M^2 * largest row count, particle count) * max |q_f|
// over the tile's reach (w3 = the largest product of three weights; a node receives from
// at most M^2 cell rows, each contributing at most `largest row count` particles, and
// from no more than all of them; max |q_f| over the catalogue), so no node sum can
// overflow, and also max |q_f| w3 2^s_f < 2^22, so that every contribution is rounded to an integer by one FFMA against 1.5 * 2^23 (round to
// nearest even, one rounding of the exact product). The bound depends only on counts
// and maxima, and integer sums do not depend on order: the grids are the same whatever
// order the sort leaves particles of one cell in.
// Ranks within a bank group that the list is ordered by (64: 5 M uniform particles on 256^3 at
// order 4 1.06 times as long, others the same).
constexpr int kListRankMax = 128;

// One tile of the FP32 gather deposit (the body of k_deposit_fx, and of each work item
// of its persistent batched form k_deposit_fx_batch). The whole CTA takes part; its
// shared memory is free again when it returns.
template <int M, int T0, int T1, int T2, int NT, int BLR>
__device__ __forceinline__ void fx_tile(const Record<float> *__restrict__ rec, const uint32_t *__restrict__ offsets,
                                        const unsigned *__restrict__ qmax_bits, int ng, int sshift,
                                        float *__restrict__ grids, int64_t grid_elems, int list_cap, bool sparse,
                                        int tile)
{
    using C = DepositCfg<float, M, T0, T1, T2, NT>;
    using Lay = FxLayout<M, T0, T1, T2>;
    constexpr int RW = Lay::RW, PX = Lay::PX, TNP = Lay::TNP;
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *acc = reinterpret_cast<int *>(smem_raw) + Lay::FRONT;  // [4][T0][PX], FxLayout
    __shared__ uint32_t s_beg[C::MAXR];
    __shared__ uint32_t s_pre[C::MAXR + 1];
    __shared__ unsigned s_rowmax;
    __shared__ float s_scale[4], s_fine[4];
    __shared__ int s_shift[4];
    constexpr bool COOP = BLR == 0 && Lay::COOP;  // one particle per warp (coop_deposit)
    // the list: bank group counts; entries before rank r; bank groups with more than r entries
    __shared__ uint32_t s_bank[32];
    __shared__ uint32_t s_rbase[kListRankMax];
    __shared__ unsigned s_rmask[kListRankMax];
    using Coop = CoopLanes<COOP ? M : 4, T0, T1, T2>;
    __shared__ __align__(16) float s_stage[COOP ? NW : 1][Coop::NB * Coop::STRIDE];

    const int ntz = ng / T2, nty = ng / T1;
    const int tz = tile % ntz;
    tile /= ntz;
    const int ty = tile % nty;
    const int tx = tile / nty;
    const int t0 = tx * T0, t1 = ty * T1, t2 = tz * T2;
    const float qm = threadIdx.x < 4 ? __uint_as_float(qmax_bits[threadIdx.x]) : 0.0f;  // used after the list
    for (int k = threadIdx.x; k < TNP; k += NT) reinterpret_cast<int4 *>(acc)[k] = make_int4(0, 0, 0, 0);
    if (threadIdx.x == 0) s_rowmax = 0;
    if (threadIdx.x < 32) s_bank[threadIdx.x] = 0;
    const uint32_t total = build_ranges<C>(offsets, ng, sshift, t0, t1, t2, T2, s_beg, s_pre);
    if (BLR > 0 && sshift == 0) {
        // the wide BL stencil: a node receives from M consecutive cells of each of M x M
        // cell rows, so bound with the largest count of M consecutive cells of a row
        // (per-cell keys: each row's offsets are cumulative along z)
        const int r0n = C::R0 < ng ? C::R0 : ng, r1n = C::R1 < ng ? C::R1 : ng;
        const int zc = (T2 + C::HL + C::HR) < ng ? (T2 + C::HL + C::HR) : ng;
        for (int r = threadIdx.x; r < r0n * r1n; r += NT) {
            int a0 = t0 - C::HL + r / r1n, a1 = t1 - C::HL + r % r1n;
            a0 = a0 < 0 ? a0 + ng : (a0 >= ng ? a0 - ng : a0);
            a1 = a1 < 0 ? a1 + ng : (a1 >= ng ? a1 - ng : a1);
            const int64_t base = (static_cast<int64_t>(a0) * ng + a1) * ng;
            uint32_t best = 0;
            for (int w0 = 0; w0 + M <= zc; ++w0) {
                int z = t2 - C::HL + w0;
                z = z < 0 ? z + ng : (z >= ng ? z - ng : z);
                const uint32_t c = z + M <= ng ? offsets[base + z + M] - offsets[base + z]
                                               : (offsets[base + ng] - offsets[base + z]) +
                                                     (offsets[base + z + M - ng] - offsets[base]);
                best = c > best ? c : best;
            }
            if (best) atomicMax(&s_rowmax, best);
        }
    } else {
        // largest row count: a row's two pieces are slots 2r and 2r + 1
        for (int r = threadIdx.x; 2 * r + 1 < C::MAXR + 1; r += NT) {
            const uint32_t c = s_pre[2 * r + 2 <= C::MAXR ? 2 * r + 2 : C::MAXR] - s_pre[2 * r];
            if (c) atomicMax(&s_rowmax, c);
        }
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t per_warp = ((total + NW - 1) / NW + 31u) & ~31u;
    const uint32_t wbeg = static_cast<uint32_t>(warp) * per_warp;
    const uint32_t wend = min(wbeg + per_warp, total);
    uint32_t *s_idx = reinterpret_cast<uint32_t *>(acc + 4 * TNP);  // list_cap entries

    __syncthreads();
    constexpr int NREACH = C::R0 * C::R1 * (T2 + C::HL + C::HR);
    const float w3 = kMaxW3<M, BLR> * 1.0001f;
    auto bound = [&](uint32_t rowmax, uint32_t n) {  // of a node sum, in units of max |q_f|
        return w3 * fminf(static_cast<float>(M * M) * static_cast<float>(rowmax), static_cast<float>(n));
    };
    uint32_t reached = total;  // particles in cells of the reach
    constexpr bool RUNS = T2 >= 16;  // smaller tiles have one cell a key (plan_assign)
    if (RUNS && sshift > 0 && T2 + C::HL + C::HR < ng && min(M * M * s_rowmax, total) > 256u) {
        // Keys of several cells: the ranges hold particles below and above the reach too. Up to
        // 256 the bound does not matter (tile_scales); above, the scale must be that of the
        // reach. It is where the runs inside the tile alone give the same power of two (and
        // the same answer to `dense`); otherwise the particles of the reach are counted.
        __shared__ unsigned s_reached, s_inner, s_unsure;
        const uint32_t outer = s_rowmax;
        __syncthreads();
        if (threadIdx.x == 0) s_rowmax = s_reached = s_inner = s_unsure = 0;
        __syncthreads();
        auto row_of = [&](int r) {  // offsets of the runs of a row
            int a0 = t0 - C::HL + r / C::R1, a1 = t1 - C::HL + r % C::R1;
            a0 = a0 < 0 ? a0 + ng : (a0 >= ng ? a0 - ng : a0);
            a1 = a1 < 0 ? a1 + ng : (a1 >= ng ? a1 - ng : a1);
            return offsets + ((static_cast<int64_t>(a0) * ng + a1) * ng >> sshift);
        };
        const int in0 = t2 >> sshift, in1 = (t2 + T2) >> sshift;  // the runs inside the tile
        for (int r = threadIdx.x; r < C::R0 * C::R1; r += NT) {
            const uint32_t *row = row_of(r);
            const uint32_t c = row[in1] - row[in0];
            if (c) atomicAdd(&s_reached, c), atomicMax(&s_inner, c);
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            int lo = 0, hi = 0;
            frexpf(bound(s_inner, s_reached) * qm, &lo);
            frexpf(bound(outer, total) * qm, &hi);
            const bool both_dense = (s_reached > 2u * NREACH) == (total > 2u * NREACH);
            if (lo != hi || (M == 4 && !both_dense)) atomicOr(&s_unsure, 1u);
        }
        __syncthreads();
        const bool unsure = s_unsure;
        __syncthreads();
        if (threadIdx.x == 0) s_rowmax = unsure ? 0u : outer, s_reached = unsure ? 0u : total;
        __syncthreads();
        auto within = [&](uint32_t i) {
            int d = (__float_as_int(rec[i].u.w) >> 20) - t2;
            d = d < -C::HL ? d + ng : (d >= T2 + C::HR ? d - ng : d);
            return d >= -C::HL && d < T2 + C::HR ? 1u : 0u;
        };
        // particles of a range within reach: short ranges by their thread, long ones by the warp
        auto reaching = [&](uint32_t b, uint32_t len) {
            uint32_t c = 0;
            if (len <= 8u)
                for (uint32_t i = 0; i < len; ++i) c += within(b + i);
            for (unsigned lng = __ballot_sync(0xffffffffu, len > 8u); lng; lng &= lng - 1u) {
                const int l = __ffs(static_cast<int>(lng)) - 1;
                const uint32_t lb = __shfl_sync(0xffffffffu, b, l), ln = __shfl_sync(0xffffffffu, len, l);
                uint32_t n = 0;
                for (uint32_t i = lane; i < ln; i += 32) n += within(lb + i);
                n = __reduce_add_sync(0xffffffffu, n);
                if (lane == l) c = n;
            }
            return c;
        };
        // only the runs on either side of the tile hold particles out of reach
        const int below = (C::HL + (1 << sshift) - 1) >> sshift, above = (C::HR + (1 << sshift) - 1) >> sshift;
        const int lo0 = (in0 ? in0 : ng >> sshift) - below, up0 = t2 + T2 == ng ? 0 : in1;
        for (int r0 = 0; r0 < C::R0 * C::R1 && unsure; r0 += NT) {
            const int r = r0 + static_cast<int>(threadIdx.x);
            const bool any = r < C::R0 * C::R1;
            const uint32_t *row = any ? row_of(r) : offsets;
            uint32_t c = any ? row[in1] - row[in0] : 0u;
            c += reaching(row[lo0], any ? row[lo0 + below] - row[lo0] : 0u);
            c += reaching(row[up0], any ? row[up0 + above] - row[up0] : 0u);
            if (c) atomicAdd(&s_reached, c), atomicMax(&s_rowmax, c);
        }
        __syncthreads();
        reached = s_reached;
    }
    // dense tiles (cubic order, more than two particles per reach cell on average) sum
    // each cell's particles in registers first (cell-block path below)
    const bool dense = M == 4 && BLR == 0 && reached > 2u * NREACH && ng >= C::R0 && ng >= C::R1 &&
                       ng >= T2 + C::HL + C::HR;
    // per-field scale from order-independent bounds only (so that the grids, and the
    // spectra, do not depend on the order in which sorted particles share a cell)
    if (threadIdx.x < 4) {
        const int f = threadIdx.x;
        const float m = qm;  // max |q_f| over the catalogue, loaded at the start
        tile_scales(bound(s_rowmax, reached) * m, w3 * m, dense, s_scale[f], s_fine[f], s_shift[f]);
    }
    __syncthreads();
    const float sc0 = s_scale[0], sc1 = s_scale[1], sc2 = s_scale[2], sc3 = s_scale[3];
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr int kMagicBits = 0x4B400000;

    // Tiles with no periodic wrap inside the reach (ng >= tile + M cells) list their
    // particles in shared memory, list_cap at most (and KP per thread) at a time, and add
    // every stencil node at an immediate offset from the first node, nodes outside the tile
    // adding exactly 0. Two ways, chosen by the wavefronts each takes:
    // * a particle per lane (banked_particle): a node's bank is the first node's plus a
    //   constant, so the list is reordered by (rank within its bank group, bank group) and
    //   32 consecutive entries hold distinct first-node banks, or span two ranks: 1.66
    //   wavefronts an add for 860 particles in random cells, 1.4 for 2048;
    // * a particle per warp (coop_deposit): one wavefront an add whatever the particles are.
    //   Taken where one bank holds many of the particles (crowded cells: 32 lanes of one
    //   cell serialise) and for short lists.
    // Each contribution is the same rounded integer as on the per-node path, so the grids do
    // not depend on the order or on the way.
    constexpr int KP = 8;       // listed particles placed per thread
    bool done = false;
    const uint32_t chunk = min(static_cast<uint32_t>(list_cap), static_cast<uint32_t>(KP * NT));
    const bool use_list = M >= 4 || (sparse && total <= chunk);
    const bool long_rows = s_rowmax > 24u;
    const bool unwrapped = ng >= C::R0 && ng >= C::R1 && ng >= T2 + C::HL + C::HR;
    if constexpr (COOP && M == 5 && T0 == 8) {
        // Order 5 on tiles of 8 x 8 rows, crowded (one row holds five times the mean of the
        // rows, or a list is no longer than the particles of 64 cells): a particle per warp
        // straight from the ranges. Listing them first takes as long again here, since a
        // particle is listed by four tiles and a tile's last list is often the whole kernel's
        // tail: whole calls over those with a branch per node and no list, 10^5 particles in
        // halos on 56^3 1.15 listed, 0.77 so; 3.4 10^5 on 72^3 1.16 and 0.81; 4.3 10^6 on 168^3
        // 0.93 and 0.87; a clump of 1.1 10^6 on 200^3 1.5 and 0.92. With eight times the mean
        // 10^5 on 88^3 take 1.10 (0.76 with five). Cubic order and 16^3 tiles, whose halo
        // particles are fewer, are faster listed (2.5 10^6 in halos on 256^3 0.72 against 0.79).
        const bool crowded = s_rowmax * static_cast<uint32_t>(C::R0 * C::R1) > 5u * total || total / NREACH > chunk / 64u;
        if (list_cap > 0 && total > 256u && crowded && unwrapped) {
            const uint32_t share = ((total + NW - 1) / NW + 7u) & ~7u, lo = min(total, warp * share);
            const uint32_t n = min(share, total - lo);
            int slot = static_cast<uint32_t>(lane >> 2) < n ? find_slot<C::MAXR>(s_pre, lo + (lane >> 2)) : 0;
            coop_deposit<M, T0, T1, T2, C::HL, C::HR>(
                rec,
                [&](uint32_t p) {
                    while (lo + p >= s_pre[slot + 1]) ++slot;
                    return s_beg[slot] + (lo + p - s_pre[slot]);
                },
                n, ng, t0, t1, t2, acc, s_stage[warp], sc0, sc1, sc2, sc3);
            done = true;
        }
    }
    if (BLR == 0 && list_cap > 0 && use_list && !dense && !done && unwrapped) {
        for (uint32_t c0 = 0; c0 < total; c0 += chunk) {
            const uint32_t cnt = min(chunk, total - c0);
            if (c0) {
                __syncthreads();  // the last chunk's list and counters are no longer read
                if (threadIdx.x < 32) s_bank[threadIdx.x] = 0;
            }
            // the list in sort order: short ranges by one thread, long ones by a warp
            for (int s0 = 0; s0 < C::MAXR; s0 += NT) {
                const int slot = s0 + static_cast<int>(threadIdx.x);
                uint32_t b = 0, at = 0, len = 0;
                if (slot < C::MAXR) {
                    const uint32_t p0 = s_pre[slot], p1 = s_pre[slot + 1], lo = max(p0, c0), hi = min(p1, c0 + cnt);
                    if (lo < hi) b = s_beg[slot] + (lo - p0), at = lo - c0, len = hi - lo;
                }
                if (long_rows) {  // uniform over the block
                    for (unsigned lng = __ballot_sync(0xffffffffu, len > 8u); lng; lng &= lng - 1u) {
                        const int l = __ffs(static_cast<int>(lng)) - 1;
                        const uint32_t lb = __shfl_sync(0xffffffffu, b, l), la = __shfl_sync(0xffffffffu, at, l),
                                       ln = __shfl_sync(0xffffffffu, len, l);
                        for (uint32_t i = lane; i < ln; i += 32) s_idx[la + i] = lb + i;
                    }
                    if (len > 8u) len = 0;
                }
                for (uint32_t i = 0; i < len; ++i) s_idx[at + i] = b + i;
            }
            __syncthreads();
            uint32_t idx[KP];
            int key[KP];  // bank group | rank << 5, -1 for no particle (or none of its nodes in the tile)
            {
                Vec4<float> u[KP];
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    const uint32_t p = threadIdx.x + k * NT;
                    key[k] = -1;
                    idx[k] = p < cnt ? s_idx[p] : 0u;
                    if (p < cnt) u[k] = rec[idx[k]].u;
                }
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    if (threadIdx.x + k * NT < cnt) {
                        const int packed = unpack_cell(u[k].w);
                        const int b0 = first_node<M, C::HL, C::HR, T0>(u[k].x, packed & 1023, t0, ng);
                        const int b1 = first_node<M, C::HL, C::HR, T1>(u[k].y, (packed >> 10) & 1023, t1, ng);
                        const int b2 = first_node<M, C::HL, C::HR, T2>(u[k].z, (packed >> 20) & 1023, t2, ng);
                        const bool reaches = (M % 2 == 0 && (!RUNS || sshift == 0)) || (b0 > -M && b0 < T0 && b1 > -M && b1 < T1 && b2 > -M && b2 < T2);
                        const int g = (b0 * PX + b1 * RW + b2) & 31;
                        if (reaches) key[k] = g | static_cast<int>(atomicAdd(&s_bank[g], 1u) << 5);
                    }
                }
            }
            __syncthreads();
            const uint32_t bank = s_bank[lane];
            const uint32_t maxc = __reduce_max_sync(0xffffffffu, bank);
            if constexpr (COOP) {
                if (maxc * (4u * M * M * M) > cnt * static_cast<uint32_t>(Coop::COST)) {
                    const uint32_t share = ((cnt + NW - 1) / NW + 7u) & ~7u, lo = min(cnt, warp * share);
                    const uint32_t *mine = s_idx + lo;
                    coop_deposit<M, T0, T1, T2, C::HL, C::HR>(
                        rec, [&](uint32_t p) { return mine[p]; }, min(share, cnt - lo), ng, t0, t1, t2, acc,
                        s_stage[warp], sc0, sc1, sc2, sc3);
                    continue;
                }
            }
            // Only particles that reach the tile go to banked_particle (the pads cover no others):
            // entries before (r, g): sum over groups of min(count, r), then the groups below g
            // with more than r entries; ranks from kListRankMax on come last, group by group
            constexpr uint32_t kRanks = kListRankMax;
            for (uint32_t r = warp; r < min(maxc, kRanks); r += NW) {
                const unsigned m = __ballot_sync(0xffffffffu, bank > r);
                const uint32_t below = __reduce_add_sync(0xffffffffu, bank < r ? bank : r);
                if (lane == 0) s_rmask[r] = m, s_rbase[r] = below;
            }
            const uint32_t len = __reduce_add_sync(0xffffffffu, bank);
            uint32_t last = 0;  // lane g: the place of group g's entry of rank kListRankMax
            if (maxc > kRanks) {
                const uint32_t over = bank > kRanks ? bank - kRanks : 0u;
                uint32_t upto = over;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xffffffffu, upto, o);
                    if (lane >= o) upto += x;
                }
                last = __reduce_add_sync(0xffffffffu, min(bank, kRanks)) + upto - over;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const int g = key[k] & 31, r = key[k] >> 5;
                const uint32_t from = maxc > kRanks ? __shfl_sync(0xffffffffu, last, g) : 0u;
                if (key[k] < 0) continue;
                s_idx[r < kListRankMax ? s_rbase[r] + __popc(s_rmask[r] & ((1u << g) - 1u)) : from + r - kListRankMax] =
                    idx[k];
            }
            __syncthreads();
            const unsigned acc_s = static_cast<unsigned>(__cvta_generic_to_shared(acc));
            uint32_t p = threadIdx.x;  // warp w takes chunks w, w + NW, ... of 32 entries
            Record<float> nxt;
            if (p < len) nxt = load_record(rec + s_idx[p]);
            while (p < len) {
                const Record<float> rc = nxt;
                p += NT;
                if (p < len) nxt = load_record(rec + s_idx[p]);
                banked_particle<M, T0, T1, T2, C::HL, C::HR>(rc, ng, t0, t1, t2, acc_s, sc0, sc1, sc2, sc3);
            }
        }
        done = true;
    }

    if constexpr (M == 4 && BLR == 0) {  // the cell-block path uses B-spline pieces
        if (dense) {
            deposit_cells_path<T0, T1, T2, NT>(rec, offsets, ng, sshift, t0, t1, t2, acc, TNP, PX, RW, s_fine, s_shift);
            done = true;
        }
    }
    // otherwise node by node, one particle per lane
    if (!done) {
        int slot = wbeg + lane < wend ? find_slot<C::MAXR>(s_pre, wbeg + lane) : 0;
        for (uint32_t p = wbeg + lane; p < wend; p += 32) {
            while (p >= s_pre[slot + 1]) ++slot;
            const Record<float> rc = load_record(rec + s_beg[slot] + (p - s_pre[slot]));
            float w[3][M];
            int li[3][M];
            stencil<float, M, BLR>(rc, ng, t0, t1, t2, T0, T1, T2, w, li);
            const float q0 = rc.q.x * sc0, q1 = rc.q.y * sc1, q2 = rc.q.z * sc2, q3 = rc.q.w * sc3;
            // the M x M (y, z) nodes of one x node
            auto plane = [&](float wx, int lx) {
#pragma unroll
                for (int k1 = 0; k1 < M; ++k1) {
                    if (li[1][k1] < 0) continue;
                    const float w01 = wx * w[1][k1];
                    const int b01 = lx * PX + li[1][k1] * RW;
#pragma unroll
                    for (int k2 = 0; k2 < M; ++k2) {
                        if (li[2][k2] < 0) continue;
                        const float ww = w01 * w[2][k2];
                        if (!PK_IN(b01 + li[2][k2], TNP, kChkShared)) continue;
                        int *a = acc + b01 + li[2][k2];
                        atomicAdd(a, __float_as_int(fmaf(q0, ww, kMagic)) - kMagicBits);
                        atomicAdd(a + TNP, __float_as_int(fmaf(q1, ww, kMagic)) - kMagicBits);
                        atomicAdd(a + 2 * TNP, __float_as_int(fmaf(q2, ww, kMagic)) - kMagicBits);
                        atomicAdd(a + 3 * TNP, __float_as_int(fmaf(q3, ww, kMagic)) - kMagicBits);
                    }
                }
            };
            if constexpr (BLR > 2) {
                // wide stencils: a rolled loop over x nodes keeps the code in the
                // instruction cache; each x weight is formed where it is used
                float wx;
                int lx;
#pragma unroll 1
                for (int k0 = 0; k0 < M; ++k0)
                    if (bl_node_x<BLR, float>(rc, ng, t0, T0, k0, wx, lx)) plane(wx, lx);
            } else {
#pragma unroll
                for (int k0 = 0; k0 < M; ++k0)
                    if (li[0][k0] >= 0) plane(w[0][k0], li[0][k0]);
            }
        }
    }
    __syncthreads();
    const float inv[4] = {1.0f / sc0, 1.0f / sc1, 1.0f / sc2, 1.0f / sc3};  // exact: powers of two
    if ((reinterpret_cast<uintptr_t>(grids) & 7u) == 0) {
        // two z-adjacent cells per thread, one 8-byte store per field (ng, the row pitch
        // ng + 2, t2 and the even l2 keep the pair aligned)
        for (int k = threadIdx.x; k < C::TN / 2; k += NT) {
            const int l2 = 2 * (k % (T2 / 2)), l01 = k / (T2 / 2);
            const int l1 = l01 % T1, l0 = l01 / T1;
            const int64_t gi = (static_cast<int64_t>(t0 + l0) * ng + (t1 + l1)) * (ng + 2) + t2 + l2;
            const int ai = l0 * PX + l1 * RW + l2;
            if (!PK_IN(gi + 1, grid_elems, kChkGrid) || !PK_IN(ai + 1, TNP, kChkShared)) continue;
#pragma unroll
            for (int f = 0; f < 4; ++f)
                *reinterpret_cast<float2 *>(grids + f * grid_elems + gi) =
                    make_float2(static_cast<float>(acc[f * TNP + ai]) * inv[f],
                                static_cast<float>(acc[f * TNP + ai + 1]) * inv[f]);
        }
    } else {
        for (int k = threadIdx.x; k < C::TN; k += NT) {
            const int l2 = k % T2, l01 = k / T2;
            const int l1 = l01 % T1, l0 = l01 / T1;
            const int64_t gi = (static_cast<int64_t>(t0 + l0) * ng + (t1 + l1)) * (ng + 2) + t2 + l2;
            const int ai = l0 * PX + l1 * RW + l2;
            if (!PK_IN(gi, grid_elems, kChkGrid) || !PK_IN(ai, TNP, kChkShared)) continue;
#pragma unroll
            for (int f = 0; f < 4; ++f) grids[f * grid_elems + gi] = static_cast<float>(acc[f * TNP + ai]) * inv[f];
        }
    }
}

// (16^3-cell and larger tiles: up to 128 registers, as shared memory already holds them to
// two per SM; 8^3 tiles: 64, for eight per SM)
template <int M, int T0, int T1, int T2, int NT, int BLR = 0>
__global__ void __launch_bounds__(NT, NT >= 512 ? 1 : (NT >= 256 ? 2 : 8))
k_deposit_fx(const Record<float> *__restrict__ rec, const uint32_t *__restrict__ offsets,
             const unsigned *__restrict__ qmax_bits, int ng, int sshift, float *__restrict__ grids, int64_t grid_elems,
             int list_cap, bool sparse)
{
    fx_tile<M, T0, T1, T2, NT, BLR>(rec, offsets, qmax_bits, ng, sshift, grids, grid_elems, list_cap, sparse,
                                    static_cast<int>(blockIdx.x));
}

// Persistent form of the gather deposit over the tiles of many catalogues (the batched
// estimate): each CTA takes the next (catalogue, tile) item from a global counter until
// none is left. Items are independent (each writes its own tile of its own grids), so
// nothing waits on another item; the order items are taken in does not change any
// result. While a tile is deposited the CTA asks L2 to prefetch the key-table rows of
// the item after it (the rows its range search reads first).
template <int M, int T0, int T1, int T2, int NT>
__global__ void __launch_bounds__(NT, NT >= 512 ? 1 : (NT >= 256 ? 2 : 8))
k_deposit_fx_batch(const FxBatch jobs, unsigned long long *__restrict__ counter)
{
    __shared__ long long s_item[2];
    using C = DepositCfg<float, M, T0, T1, T2, NT>;
    auto job_of = [&](long long item) {
        int j = 0;
        while (j + 1 < jobs.n && jobs.job[j + 1].first_tile <= item) ++j;
        return j;
    };
    auto prefetch_rows = [&](long long item) {
        if (item >= jobs.total_tiles) return;
        const FxJob &jb = jobs.job[job_of(item)];
        const int ng = jb.ng, ntz = ng / T2, nty = ng / T1;
        int tile = static_cast<int>(item - jb.first_tile);
        const int tz = tile % ntz;
        tile /= ntz;
        const int ty = tile % nty, tx = tile / nty;
        const int nseg = ng >> jb.sshift;
        for (int r = threadIdx.x; r < C::R0 * C::R1; r += NT) {
            int a0 = tx * T0 - C::HL + r / C::R1, a1 = ty * T1 - C::HL + r % C::R1;
            a0 = a0 < 0 ? a0 + ng : (a0 >= ng ? a0 - ng : a0);
            a1 = a1 < 0 ? a1 + ng : (a1 >= ng ? a1 - ng : a1);
            const uint32_t *row = jb.offsets + (static_cast<int64_t>(a0) * ng + a1) * nseg + ((tz * T2) >> jb.sshift);
            asm volatile("prefetch.L2 [%0];" ::"l"(row));
        }
    };
    if (threadIdx.x == 0) s_item[0] = static_cast<long long>(atomicAdd(counter, 1ull));
    __syncthreads();
    long long item = s_item[0];
    int buf = 0;
    while (item < jobs.total_tiles) {
        if (threadIdx.x == 0) s_item[buf ^ 1] = static_cast<long long>(atomicAdd(counter, 1ull));
        __syncthreads();
        const long long next = s_item[buf ^ 1];
        prefetch_rows(next);
        const FxJob &jb = jobs.job[job_of(item)];
        fx_tile<M, T0, T1, T2, NT, 0>(jb.rec, jb.offsets, jb.qmax, jb.ng, jb.sshift, jb.grids, jb.grid_elems,
                                      jb.list_cap, jb.sparse != 0, static_cast<int>(item - jb.first_tile));
        __syncthreads();
        item = next;
        buf ^= 1;
    }
}

// ------------------------------------------------------------------ home-tile deposit
// FP32 grids, cubic order, catalogues with about half a particle per cell or more.
//
// Each CTA owns a tile of 16^3 cells and deposits only the particles of those cells
// (each particle once), into a shared buffer of the 19^3 nodes their stencils reach
// (nodes -1 .. 17 of the tile on each axis). The 16^3 nodes the tile owns are written
// to the grid; the 2763 halo nodes go to a per-tile scratch area, and k_home_fixup adds
// each neighbour's halo to the owned nodes it overlaps, in a fixed order (so the grids
// do not depend on scheduling).
//
// Lane mapping: a warp takes a block of 2 x 2 cell columns; lane (x, y, m) takes the
// first particles of cells z = 2m, 2m + 1 of its column and sums their contributions
// to each node column's 5 z nodes in registers before adding them (home_pair), two
// fields' roundings per paired FMA (fma.rn.f32x2, each half the scalar FMA's result). The
// buffer's x pitch is 16 modulo 32 banks, its y pitch 19 and its z pitch 1, so the 32
// lanes of every add hit 32 different banks (checked at compile time below): one
// wavefront each. Particles beyond the first of a cell go to a per-warp queue and are
// deposited 32 at a time, one per lane. Bound by the shared pipe and by latency together
// (shared memory holds two tiles per SM). Two cells a lane instead of four add 5 node sums
// for 2 cells instead of 7 for 4, but fit 80 registers instead of 128, so that 24 warps run
// on an SM instead of 16: 512^3 particles on 512^3, deposit 8.99 -> 8.75 ms,
// and with the dy loop of home_pair unrolled and one queue of extra particles 8.04 ms
// (a 500 Mpc/h box; in a 1500 Mpc/h one, less clustered, 8.35 -> 7.12 ms in all).
// Tiles with more than two particles per cell, or 32 in some four consecutive cells of a
// column, take the cell-block path: one warp per cell, each contribution rounded at the
// fine scale (largest contribution < 2^22) and summed exactly, in 64-bit shared
// accumulators (two fields per pass), so that a dense node's error is that of its
// contributions' roundings alone. Tiles with under a quarter particle per cell take one
// particle per lane from the tile's list.
//
// Fixed point as in k_deposit_fx, with bounds over the home tile's own particles (the
// only ones the buffer receives): B_f = w3 * min(16 * largest 4-cell column window count,
// particle count) * max |q_f|.
constexpr int kHomeT = 16;                                      // tile edge in cells (= owned nodes)
constexpr int kHomeB = kHomeT + 3;                              // buffer edge in nodes
constexpr int kHomePY = kHomeB;                                 // buffer y pitch
constexpr int kHomePX = 368;                                    // buffer x pitch
constexpr int kHomeField = kHomeB * kHomePX;                    // ints per field
constexpr int kHomeHalo = kHomeB * kHomeB * kHomeB - kHomeT * kHomeT * kHomeT;  // 2763 halo nodes
constexpr int kHomeNT = 384;                                    // threads (at least one per cell column)
constexpr int kHomeCP = 2;                                      // z-consecutive cells per lane
constexpr int kHomeM = kHomeT / kHomeCP;                        // lanes per cell column
constexpr int kHomeCols = 32 / kHomeM;                          // cell columns per warp step (2 in x)
constexpr int kHomeColY = kHomeCols / 2;
constexpr int kHomeNW = kHomeNT / 32;
constexpr int kHomeQ = 64;                                      // overflow queue entries per warp
constexpr size_t kHomeSmem = size_t(4) * kHomeField * sizeof(int);
static_assert(kHomePX % 32 == 16 && kHomePX >= kHomeB * kHomeB, "x-adjacent cells must be 16 banks apart");
static_assert(kHomeNT >= kHomeT * kHomeT, "one thread per cell column");

// Banks of the first stencil node of the 32 lanes of a block (2 x 2 columns, lane (x, y, m)
// at cells z = 2m, 2m + 1): all different, so that every add of home_pair is one wavefront.
constexpr bool home_pair_banks_distinct()
{
    unsigned seen = 0;
    for (int lane = 0; lane < 32; ++lane) {
        const int m = lane % kHomeM, y = (lane / kHomeM) % kHomeColY, x = lane / (kHomeM * kHomeColY);
        const unsigned bit = 1u << ((x * kHomePX + y * kHomePY + kHomeCP * m) & 31);
        if (seen & bit) return false;
        seen |= bit;
    }
    return true;
}
static_assert(home_pair_banks_distinct(), "the 32 lanes of a home_pair add must hit 32 banks");
// home_pair's largest buffer index on each axis: cell 15 + node offset 3 in x and y, and
// CP + 3 z nodes from the lane's first cell; all inside the 19-node edge
static_assert(kHomeT - 1 + 3 < kHomeB && kHomeT - kHomeCP + kHomeCP + 2 < kHomeB && kHomeT % kHomeCP == 0,
              "home_pair's nodes must lie in the node buffer");

// Halo index of buffer node (bx, by, bz), at least one coordinate in {0, 17, 18}:
// first the three x planes (19 x 19 each), then the y planes of the inner x range
// (16 x 19), then the z planes of the inner x, y range (16 x 16).
__host__ __device__ constexpr int home_side(int b) { return b == 0 ? 0 : b - kHomeT; }  // 0, 17, 18 -> 0, 1, 2
__host__ __device__ constexpr int home_unside(int s) { return s == 0 ? 0 : s + kHomeT; }
__host__ __device__ constexpr int home_halo_index(int bx, int by, int bz)
{
    if (bx == 0 || bx > kHomeT) return (home_side(bx) * kHomeB + by) * kHomeB + bz;
    if (by == 0 || by > kHomeT) return 3 * kHomeB * kHomeB + ((bx - 1) * 3 + home_side(by)) * kHomeB + bz;
    return 3 * kHomeB * kHomeB + 3 * kHomeT * kHomeB + ((bx - 1) * kHomeT + (by - 1)) * 3 + home_side(bz);
}
__host__ __device__ constexpr void home_halo_node(int k, int &bx, int &by, int &bz)
{
    constexpr int nx = 3 * kHomeB * kHomeB, ny = 3 * kHomeT * kHomeB;
    if (k < nx) {
        bz = k % kHomeB;
        const int r = k / kHomeB;
        by = r % kHomeB;
        bx = home_unside(r / kHomeB);
    } else if (k < nx + ny) {
        k -= nx;
        bz = k % kHomeB;
        const int r = k / kHomeB;
        by = home_unside(r % 3);
        bx = r / 3 + 1;
    } else {
        k -= nx + ny;
        bz = home_unside(k % 3);
        const int r = k / 3;
        by = r % kHomeT + 1;
        bx = r / kHomeT + 1;
    }
}

// home_halo_node inverts home_halo_index over the 2763 halo nodes, and every node it
// gives has a coordinate on the halo (0, 17 or 18)
constexpr bool home_halo_bijective()
{
    for (int k = 0; k < kHomeHalo; ++k) {
        int bx = 0, by = 0, bz = 0;
        home_halo_node(k, bx, by, bz);
        const bool inner = bx >= 1 && bx <= kHomeT && by >= 1 && by <= kHomeT && bz >= 1 && bz <= kHomeT;
        if (inner || bx < 0 || bx >= kHomeB || by < 0 || by >= kHomeB || bz < 0 || bz >= kHomeB ||
            home_halo_index(bx, by, bz) != k)
            return false;
    }
    return true;
}
static_assert(home_halo_bijective(), "the halo scratch layout must be a bijection");

// Shared-memory add without a returned value (the accumulators are read only after a
// barrier): addr is a shared-window byte address.
__device__ __forceinline__ void red_shared_add(unsigned addr, int v)
{
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v));
}

// One particle of home cell (cx, cy, cz) (each 0..15) into the node buffer: node
// c - 1 + k of the tile is buffer index c + k.
__device__ __forceinline__ void home_particle(int *acc, const Record<float> &r, int cx, int cy, int cz, float sc0,
                                              float sc1, float sc2, float sc3)
{
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr int kMagicBits = 0x4B400000;
    float wx[4], wy[4], wz[4];
    int first;
    bspline_weights<4, float>(r.u.x, wx, first);
    bspline_weights<4, float>(r.u.y, wy, first);
    bspline_weights<4, float>(r.u.z, wz, first);
    const float q0 = r.q.x * sc0, q1 = r.q.y * sc1, q2 = r.q.z * sc2, q3 = r.q.w * sc3;
    // its last stencil node (3, 3, 3 from the first) must lie in the node buffer
    if (!PK_IN((cx + 3) * kHomePX + (cy + 3) * kHomePY + cz + 3, kHomeField, kChkShared)) return;
    // shared-window byte address of the particle's first stencil node
    const unsigned base = static_cast<unsigned>(__cvta_generic_to_shared(acc)) + 4u * (cx * kHomePX + cy * kHomePY + cz);
#pragma unroll
    for (int k0 = 0; k0 < 4; ++k0) {
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            const float w01 = wx[k0] * wy[k1];
            const unsigned b = base + 4u * (k0 * kHomePX + k1 * kHomePY);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) {
                const float ww = w01 * wz[k2];
                const unsigned a = b + 4 * k2;
                red_shared_add(a, __float_as_int(fmaf(q0, ww, kMagic)) - kMagicBits);
                red_shared_add(a + 4 * kHomeField, __float_as_int(fmaf(q1, ww, kMagic)) - kMagicBits);
                red_shared_add(a + 8 * kHomeField, __float_as_int(fmaf(q2, ww, kMagic)) - kMagicBits);
                red_shared_add(a + 12 * kHomeField, __float_as_int(fmaf(q3, ww, kMagic)) - kMagicBits);
            }
        }
    }
}

// The first particles of the kHomeCP z-consecutive home cells from z = kHomeCP m of column
// (cx, cy), of one lane. For each of the 16 (x, y) stencil node columns the lane sums
// the cells' contributions to the kHomeCP + 3 z nodes it reaches in registers, then adds
// them: 20 shared adds per node column instead of 32 for two particles one by one.
// Each contribution is the same rounded integer as in home_particle (same products, one
// FMA against 1.5 * 2^23, here two fields per paired FMA); the raw bit patterns are summed
// modulo 2^32 and the magic constant is taken off once per node (cnt(i) cells reach z node
// i), so the sums are exact. An empty cell has q = 0 and adds exactly the magic constant.
__device__ __forceinline__ void home_pair(unsigned acc_s, const Record<float> (&r)[kHomeCP], const bool (&has)[kHomeCP], int cx,
                                          int cy, int m, float sc0, float sc1, float sc2, float sc3)
{
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr unsigned kMagicBits = 0x4B400000u;
    constexpr int CP = kHomeCP;
    float wx[CP][4], wy[CP][4], wz[CP][4], q[CP][4];
#pragma unroll
    for (int j = 0; j < CP; ++j) {
        int first;
        bspline_weights<4, float>(has[j] ? r[j].u.x : 0.0f, wx[j], first);
        bspline_weights<4, float>(has[j] ? r[j].u.y : 0.0f, wy[j], first);
        bspline_weights<4, float>(has[j] ? r[j].u.z : 0.0f, wz[j], first);
        q[j][0] = has[j] ? r[j].q.x * sc0 : 0.0f;
        q[j][1] = has[j] ? r[j].q.y * sc1 : 0.0f;
        q[j][2] = has[j] ? r[j].q.z * sc2 : 0.0f;
        q[j][3] = has[j] ? r[j].q.w * sc3 : 0.0f;
    }
    f32x2 qp[CP][2];  // fields (0, 1) and (2, 3) of each cell as pairs
#pragma unroll
    for (int j = 0; j < CP; ++j) qp[j][0] = f2_pack(q[j][0], q[j][1]), qp[j][1] = f2_pack(q[j][2], q[j][3]);
    const f32x2 mg = f2_pack(kMagic, kMagic);
    // buffer index of node (cx - 1 + dx, cy - 1 + dy, CP m - 1 + i) is (cx + dx) PX + (cy + dy) PY + CP m + i.
    // The lane's last node (3, 3 node columns on) must lie in the buffer.
    if (!PK_IN((cx + 3) * kHomePX + (cy + 3) * kHomePY + CP * m + CP + 2, kHomeField, kChkShared)) return;
    unsigned base = acc_s + 4u * static_cast<unsigned>(cx * kHomePX + cy * kHomePY + CP * m);
    // rolled (a short body for the instruction cache): the weights of the current dx are kept in
    // slot 0 by rotating them
#pragma unroll 1
    for (int dx = 0; dx < 4; ++dx) {
        static_for<4>([&](auto dyc) {
            constexpr int dy = decltype(dyc)::value;
            unsigned a[CP + 3][4];
            static_for<CP + 3>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                constexpr unsigned cnt = static_cast<unsigned>((i < CP - 1 ? i : CP - 1) - (i > 3 ? i - 3 : 0) + 1);
#pragma unroll
                for (int f = 0; f < 4; ++f) a[i][f] = 0u - cnt * kMagicBits;
            });
#pragma unroll
            for (int j = 0; j < CP; ++j) {
                const float w01 = wx[j][0] * wy[j][dy];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float ww = w01 * wz[j][k];
                    const f32x2 w2 = f2_pack(ww, ww);
                    const f32x2 t01 = f2_fma(qp[j][0], w2, mg), t23 = f2_fma(qp[j][1], w2, mg);
                    a[j + k][0] += static_cast<unsigned>(t01);
                    a[j + k][1] += static_cast<unsigned>(t01 >> 32);
                    a[j + k][2] += static_cast<unsigned>(t23);
                    a[j + k][3] += static_cast<unsigned>(t23 >> 32);
                }
            }
            static_for<CP + 3>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                red4<4 * (dy * kHomePY + i), 4 * kHomeField>(base, static_cast<int>(a[i][0]), static_cast<int>(a[i][1]),
                                                             static_cast<int>(a[i][2]), static_cast<int>(a[i][3]));
            });
        });
#pragma unroll
        for (int j = 0; j < CP; ++j) {  // next dx in slot 0
            const float t = wx[j][0];
            wx[j][0] = wx[j][1], wx[j][1] = wx[j][2], wx[j][2] = wx[j][3], wx[j][3] = t;
        }
        base += 4u * kHomePX;
    }
}

// A sorted particle of this tile (its cell read from the record); skipped if the record
// does not lie in the tile. One copy for its three call sites (instruction cache).
__device__ __noinline__ void home_listed(int *acc, const Record<float> *__restrict__ rec, uint32_t idx, int t0, int t1,
                                         int t2, float sc0, float sc1, float sc2, float sc3)
{
    const Record<float> r = load_record(rec + idx);
    const int c = unpack_cell(r.u.w);
    const unsigned cx = static_cast<unsigned>((c & 1023) - t0), cy = static_cast<unsigned>(((c >> 10) & 1023) - t1),
                   cz = static_cast<unsigned>(((c >> 20) & 1023) - t2);
    if (cx < kHomeT && cy < kHomeT && cz < kHomeT)
        home_particle(acc, r, static_cast<int>(cx), static_cast<int>(cy), static_cast<int>(cz), sc0, sc1, sc2, sc3);
}

// Dense home tiles: one warp per cell column; lane l owns stencil nodes (dx, dy, dz)
// with dz = l & 3, dy = (l >> 2) & 3, dx = (l >> 4) and (l >> 4) + 2 of the cell at hand, sums
// up to kCellFlush of the cell's particles in registers and adds the sums to 64-bit totals,
// two fields per pass. limbs: the totals are kept as two 32-bit words, the low 16 bits of each
// sum and the rest (a 64-bit shared add takes as long as eight 32-bit ones; a node gets fewer
// than 2^16 sums, see the caller); otherwise as 64-bit words. The column's 17 offsets are
// loaded at once and its records asked for ahead: cell by cell, the two dependent loads of
// each of 4096 cells were most of the time.
template <int F0>
__device__ __forceinline__ void home_cells_path(const Record<float> *__restrict__ rec,
                                                const uint32_t *__restrict__ offsets, int ng, int t0, int t1, int t2,
                                                unsigned char *acc, bool limbs, const float *s_fine)
{
    const float fine[4] = {s_fine[0], s_fine[1], s_fine[2], s_fine[3]};
    const int noshift[4] = {0, 0, 0, 0};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int dz = lane & 3, dy = (lane >> 2) & 3, dxl = lane >> 4;
    auto *acc64 = reinterpret_cast<unsigned long long *>(acc);  // [2][kHomeField]
    int *acc32 = reinterpret_cast<int *>(acc);                  // [2 fields][low, high][kHomeField]
    CellPieces pc;
    cubic_piece(dxl, pc.xa);
    cubic_piece(dxl + 2, pc.xb);
    cubic_piece(dy, pc.y);
    cubic_piece(dz, pc.z);
    auto column_offset = [&](int col) -> uint32_t {  // lane z: offset of cell z of the column
        if (col >= kHomeT * kHomeT || lane > kHomeT) return 0u;
        return offsets[(static_cast<int64_t>(t0 + (col >> 4)) * ng + (t1 + (col & 15))) * ng + t2 + lane];
    };
    uint32_t next = column_offset(warp);
    for (int col = warp; col < kHomeT * kHomeT; col += kHomeNW) {
        const uint32_t o = next;
        next = column_offset(col + kHomeNW);
        const uint32_t first = __shfl_sync(0xffffffffu, o, 0), last = __shfl_sync(0xffffffffu, o, kHomeT);
        for (uint32_t i = first + 4 * lane; i < last && i < first + 512; i += 128)
            asm volatile("prefetch.global.L1 [%0];" ::"l"(rec + i));
        const uint32_t after = __shfl_down_sync(0xffffffffu, o, 1);
        for (unsigned full = __ballot_sync(0xffffffffu, lane < kHomeT && after > o); full; full &= full - 1u) {
            const int cz = __ffs(static_cast<int>(full)) - 1;
            const uint32_t beg = __shfl_sync(0xffffffffu, o, cz), end = __shfl_sync(0xffffffffu, after, cz);
            const int oa = ((col >> 4) + dxl) * kHomePX + ((col & 15) + dy) * kHomePY + cz + dz, ob = oa + 2 * kHomePX;
            if (!PK_IN(ob, kHomeField, kChkShared)) continue;
            for (uint32_t i0 = beg; i0 < end; i0 += kCellFlush) {
                int a[2], b[2];
                cell_chunk<F0, 2>(rec, i0, min(end, i0 + kCellFlush), pc, fine, noshift, a, b);
#pragma unroll
                for (int f = 0; f < 2; ++f) {  // two's complement sums
                    if (limbs) {
                        int *n = acc32 + 2 * f * kHomeField;
                        atomicAdd(n + oa, a[f] & 0xffff);
                        atomicAdd(n + kHomeField + oa, a[f] >> 16);
                        atomicAdd(n + ob, b[f] & 0xffff);
                        atomicAdd(n + kHomeField + ob, b[f] >> 16);
                    } else {
                        unsigned long long *n = acc64 + f * kHomeField;
                        atomicAdd(n + oa, static_cast<unsigned long long>(static_cast<long long>(a[f])));
                        atomicAdd(n + ob, static_cast<unsigned long long>(static_cast<long long>(b[f])));
                    }
                }
            }
        }
    }
}

__global__ void __launch_bounds__(kHomeNT, 2)
k_deposit_home(const Record<float> *__restrict__ rec, const uint32_t *__restrict__ offsets,
               const unsigned *__restrict__ qmax_bits, int ng, float *__restrict__ grids, int64_t grid_elems,
               float *__restrict__ halo)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *acc = reinterpret_cast<int *>(smem_raw);  // [4][kHomeB][kHomePX] (x, y, z of the node buffer)
    // column ranges of the tile (sparse path), reused as the per-warp queues (medium path)
    __shared__ uint32_t s_cols[kHomeNW * kHomeQ > 2 * kHomeT * kHomeT + 1 ? kHomeNW * kHomeQ : 2 * kHomeT * kHomeT + 1];
    uint32_t *s_beg = s_cols, *s_pre = s_cols + kHomeT * kHomeT;
    __shared__ unsigned s_rowmax;
    __shared__ float s_scale[4], s_fine[4];
    __shared__ int s_shift[4];

    const int nt = ng / kHomeT;
    const int tz = blockIdx.x % nt, ty = (blockIdx.x / nt) % nt, tx = blockIdx.x / (nt * nt);
    const int t0 = tx * kHomeT, t1 = ty * kHomeT, t2 = tz * kHomeT;
    const float qm = threadIdx.x < 4 ? __uint_as_float(qmax_bits[threadIdx.x]) : 0.0f;  // used after the scan
    {
        int4 *a4 = reinterpret_cast<int4 *>(acc);
        for (int k = threadIdx.x; k < kHomeField; k += kHomeNT) a4[k] = make_int4(0, 0, 0, 0);  // 4 fields / 4 ints
    }
    if (threadIdx.x == 0) s_rowmax = 0;
    __syncthreads();
    // thread = cell column (x, y) of the tile: its particles are one range of the sort
    uint32_t total;
    {
        const bool col = threadIdx.x < kHomeT * kHomeT;
        const int x = (threadIdx.x >> 4) & 15, y = threadIdx.x & 15;
        const int64_t key = (static_cast<int64_t>(t0 + x) * ng + (t1 + y)) * ng + t2;
        uint32_t o[kHomeT + 1];  // offsets[key + 1] is 16-byte aligned (key_table), keys per column 16
        o[0] = offsets[key];
#pragma unroll
        for (int z = 0; z < kHomeT; z += 4) {
            const uint4 v = *reinterpret_cast<const uint4 *>(offsets + key + 1 + z);
            o[z + 1] = v.x, o[z + 2] = v.y, o[z + 3] = v.z, o[z + 4] = v.w;
        }
        const uint32_t b = o[0], cnt = col ? o[kHomeT] - b : 0u;
        // the column's records are read later, cell by cell: ask L2 for them now (128-byte
        // lines covering the column's contiguous range, at most 32 lines per column)
        {
            const char *r0 = reinterpret_cast<const char *>(rec + b);
            const uint32_t lines = cnt ? min((cnt * 32u + 127u) / 128u + 1u, 32u) : 0u;
            for (uint32_t l = 0; l < lines; ++l) asm volatile("prefetch.L2 [%0];" ::"l"(r0 + 128 * l));
        }
        // a node receives from 4 consecutive cells of a column: the largest such count
        uint32_t win = 0;
#pragma unroll
        for (int z = 0; z + 4 <= kHomeT; ++z) win = max(win, o[z + 4] - o[z]);
        const uint32_t pre = block_exclusive_scan(cnt, total);
        if (col) s_beg[threadIdx.x] = b, s_pre[threadIdx.x] = pre;
        if (threadIdx.x == 0) s_pre[kHomeT * kHomeT] = total;
        if (win) atomicMax(&s_rowmax, win);
    }
    __syncthreads();
    constexpr uint32_t kCells = kHomeT * kHomeT * kHomeT;
    // dense somewhere (32 particles in four consecutive cells) or on average: sum each
    // cell in registers and round once per cell, instead of once per particle
    const bool dense = s_rowmax >= 32u || total > 2u * kCells;
    const bool sparse = !dense && total < kCells / 4u;
    if (threadIdx.x < 4) {
        const int f = threadIdx.x;
        const float m = qm;  // max |q_f| over the catalogue, loaded at the start
        const float w3 = kMaxWeight3<4> * 1.0001f;
        // a node receives from 4 consecutive cells of at most 4 x 4 columns of the tile
        const float reach = fminf(16.0f * static_cast<float>(s_rowmax), static_cast<float>(total));
        tile_scales(w3 * reach * m, w3 * m, dense, s_scale[f], s_fine[f], s_shift[f]);
    }
    __syncthreads();
    const float sc0 = s_scale[0], sc1 = s_scale[1], sc2 = s_scale[2], sc3 = s_scale[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    // owned nodes to the grid, halo nodes to this tile's scratch; value(f, buffer index); the
    // node's place is found once for all fields.
    // Owned rows: eight lanes per (x, y) row, two z nodes each (8-byte stores: the rows
    // start at even offsets, ng + 2 and the tile corner being even, and the grids are
    // 16-byte aligned).
    float *h = halo + static_cast<int64_t>(blockIdx.x) * 4 * kHomeHalo;
    auto emit = [&](auto fields, auto value) {  // fields: the first and one past the last
        constexpr int F0 = decltype(fields)::value / 8, F1 = decltype(fields)::value % 8;
#pragma unroll 2
        for (int rowi = threadIdx.x >> 3; rowi < kHomeT * kHomeT; rowi += kHomeNT / 8) {
            const int zp = 2 * (threadIdx.x & 7);
            const int x = rowi >> 4, y = rowi & 15;
            const int ab = (x + 1) * kHomePX + (y + 1) * kHomePY + zp + 1;
            const int64_t gi = (static_cast<int64_t>(t0 + x) * ng + (t1 + y)) * (ng + 2) + t2 + zp;
            if (!PK_IN(gi + 1, grid_elems, kChkGrid) || !PK_IN(ab + 1, kHomeField, kChkShared)) continue;
#pragma unroll
            for (int f = F0; f < F1; ++f)
                *reinterpret_cast<float2 *>(grids + f * grid_elems + gi) = make_float2(value(f, ab), value(f, ab + 1));
        }
        for (int k = threadIdx.x; k < kHomeHalo; k += kHomeNT) {
            int bx, by, bz;
            home_halo_node(k, bx, by, bz);
            const int ai = bx * kHomePX + by * kHomePY + bz;
            if (!PK_IN(static_cast<int64_t>(blockIdx.x) * 4 * kHomeHalo + (F1 - 1) * kHomeHalo + k,
                       static_cast<int64_t>(gridDim.x) * 4 * kHomeHalo, kChkHalo) ||
                !PK_IN(ai, kHomeField, kChkShared))
                continue;
#pragma unroll
            for (int f = F0; f < F1; ++f) h[f * kHomeHalo + k] = value(f, ai);
        }
    };

    if (dense) {
        // 64-bit sums of the fine-scale contributions, two fields per pass in the same buffer.
        // A node gets one sum from each of 64 cells per kCellFlush particles: up to 2^23
        // particles fewer than 2^16 sums, each below 2^30, so that the low words' sum stays
        // below 2^32 and the high words' below 2^30
        const bool limbs = total <= 1u << 23;
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            if (pass) {
                __syncthreads();
                int4 *a4 = reinterpret_cast<int4 *>(smem_raw);
                for (int k = threadIdx.x; k < kHomeField; k += kHomeNT) a4[k] = make_int4(0, 0, 0, 0);
                __syncthreads();
            }
            if (pass == 0) home_cells_path<0>(rec, offsets, ng, t0, t1, t2, smem_raw, limbs, s_fine);
            else home_cells_path<2>(rec, offsets, ng, t0, t1, t2, smem_raw, limbs, s_fine);
            __syncthreads();
            auto value = [&](int f, int ai) {
                const int k = f & 1;
                const long long v = limbs ? static_cast<long long>(acc[(2 * k + 1) * kHomeField + ai]) * 65536 +
                                                static_cast<unsigned>(acc[2 * k * kHomeField + ai])
                                          : reinterpret_cast<const long long *>(smem_raw)[k * kHomeField + ai];
                return static_cast<float>(v) * (1.0f / s_fine[f]);  // exact: a power of two
            };
            if (pass == 0) emit(std::integral_constant<int, 0 * 8 + 2>{}, value);
            else emit(std::integral_constant<int, 2 * 8 + 4>{}, value);
        }
        return;
    }
    if (sparse) {
        // one particle per lane, warp-contiguous chunks of the tile's list
        const uint32_t per_warp = ((total + kHomeNW - 1) / kHomeNW + 31u) & ~31u;
        const uint32_t wbeg = static_cast<uint32_t>(warp) * per_warp, wend = min(wbeg + per_warp, total);
        int slot = wbeg + lane < wend ? find_slot<kHomeT * kHomeT>(s_pre, wbeg + lane) : 0;
        for (uint32_t p = wbeg + lane; p < wend; p += 32) {
            while (p >= s_pre[slot + 1]) ++slot;
            home_listed(acc, rec, s_beg[slot] + (p - s_pre[slot]), t0, t1, t2, sc0, sc1, sc2, sc3);
        }
    } else {
        uint32_t *q = s_cols + warp * kHomeQ;  // the column ranges are no longer needed
        __syncthreads();
        int qn = 0;  // warp-uniform queue length
        const unsigned acc_s = static_cast<unsigned>(__cvta_generic_to_shared(acc));
        // a block is 2 x kHomeColY cell columns; lane (xl, yl, m) takes the kHomeCP cells from z = kHomeCP m
        constexpr int CP = kHomeCP, BY = kHomeT / kHomeColY;
        const int m = lane % kHomeM, yl = (lane / kHomeM) % kHomeColY, xl = lane / (kHomeM * kHomeColY);
        constexpr int kBlocks = (kHomeT / 2) * BY;
        auto cell_offsets = [&](int blk, uint32_t(&o)[CP + 1]) {  // the offsets of the lane's cells
            if (blk >= kBlocks) {
#pragma unroll
                for (int k = 0; k <= CP; ++k) o[k] = 0;
                return;
            }
            const int cx = 2 * (blk / BY) + xl, cy = kHomeColY * (blk % BY) + yl;
            const int64_t key = (static_cast<int64_t>(t0 + cx) * ng + (t1 + cy)) * ng + (t2 + CP * m);
            const uint2 v = *reinterpret_cast<const uint2 *>(offsets + key + 1);
            o[0] = offsets[key], o[1] = v.x, o[2] = v.y;
        };
        uint32_t on[CP + 1];
        cell_offsets(warp, on);  // loads run one block ahead
        for (int blk = warp; blk < kBlocks; blk += kHomeNW) {
            const int cx = 2 * (blk / BY) + xl, cy = kHomeColY * (blk % BY) + yl;
            uint32_t o[CP + 1];
#pragma unroll
            for (int k = 0; k <= CP; ++k) o[k] = on[k];
            cell_offsets(blk + kHomeNW, on);
            Record<float> r[CP];
            bool has[CP];
#pragma unroll
            for (int k = 0; k < CP; ++k) {
                has[k] = o[k + 1] > o[k];
                r[k] = has[k] ? load_record(rec + o[k]) : Record<float>{};
            }
            home_pair(acc_s, r, has, cx, cy, m, sc0, sc1, sc2, sc3);
            // second and later particles of the cells: the per-warp queue, 32 at a time
            static_assert(CP == 2, "the lane's two cells");
            const uint32_t n0 = has[0] ? o[1] - o[0] - 1u : 0u, n1 = has[1] ? o[2] - o[1] - 1u : 0u;
            for (uint32_t i = 0;; ++i) {
                const bool more = i < n0 + n1;
                const unsigned mk = __ballot_sync(0xffffffffu, more);
                if (!mk) break;
                if (more) q[qn + __popc(mk & ((1u << lane) - 1u))] = i < n0 ? o[0] + 1u + i : o[1] + 1u + (i - n0);
                qn += __popc(mk);
                __syncwarp();
                if (qn >= 32) {
                    home_listed(acc, rec, q[lane], t0, t1, t2, sc0, sc1, sc2, sc3);
                    __syncwarp();
                    if (lane < qn - 32) q[lane] = q[lane + 32];
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
        if (lane < qn) home_listed(acc, rec, q[lane], t0, t1, t2, sc0, sc1, sc2, sc3);
    }
    __syncthreads();
    const float inv[4] = {1.0f / sc0, 1.0f / sc1, 1.0f / sc2, 1.0f / sc3};  // exact: powers of two
    emit(std::integral_constant<int, 0 * 8 + 4>{},
         [&](int f, int ai) { return static_cast<float>(acc[f * kHomeField + ai]) * inv[f]; });
}

// Owned nodes within reach of a neighbouring tile's particles (local index 0, 1 or 15
// on some axis) receive that neighbour's halo values, added in a fixed order. Threads
// take only those 1899 nodes of a tile: the x faces (x in {0, 1, 15}), then the y faces
// of the other x, then the z faces of the rest, z fastest where a face allows.
constexpr int kHomeEdge = 3 * kHomeT * kHomeT + (kHomeT - 3) * 3 * kHomeT + (kHomeT - 3) * (kHomeT - 3) * 3;
__device__ __forceinline__ int home_face(int s) { return s == 2 ? kHomeT - 1 : s; }  // 0, 1, 15

__global__ void __launch_bounds__(256)
k_home_fixup(const float *__restrict__ halo, int ng, float *__restrict__ grids, int64_t grid_elems)
{
    const int nt = ng / kHomeT;
    const int tz = blockIdx.x % nt, ty = (blockIdx.x / nt) % nt, tx = blockIdx.x / (nt * nt);
    auto wrap = [nt](int a) { return a < 0 ? a + nt : (a >= nt ? a - nt : a); };
    // the neighbour offset on one axis whose halo covers local index l (0 if none)
    auto side = [](int l) { return l <= 1 ? -1 : (l == kHomeT - 1 ? 1 : 0); };
    constexpr int nx = 3 * kHomeT * kHomeT, ny = (kHomeT - 3) * 3 * kHomeT;
    for (int k = threadIdx.x; k < kHomeEdge; k += blockDim.x) {
        int x, y, z;
        if (k < nx) {
            x = home_face(k / (kHomeT * kHomeT));
            y = (k / kHomeT) % kHomeT;
            z = k % kHomeT;
        } else if (k < nx + ny) {
            const int r = k - nx;
            x = 2 + r / (3 * kHomeT);
            y = home_face((r / kHomeT) % 3);
            z = r % kHomeT;
        } else {
            const int r = k - nx - ny;
            x = 2 + r / (3 * (kHomeT - 3));
            y = 2 + (r / 3) % (kHomeT - 3);
            z = home_face(r % 3);
        }
        const int64_t gi = (static_cast<int64_t>(tx * kHomeT + x) * ng + (ty * kHomeT + y)) * (ng + 2) + tz * kHomeT + z;
        if (!PK_IN(gi, grid_elems, kChkGrid)) continue;
        float v[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) v[f] = grids[f * grid_elems + gi];
        const int sx = side(x), sy = side(y), sz = side(z);
        // neighbours (dx, dy, dz), each 0 or the axis' side, in a fixed order
#pragma unroll
        for (int c = 1; c < 8; ++c) {
            const int dx = (c & 4) ? sx : 0, dy = (c & 2) ? sy : 0, dz = (c & 1) ? sz : 0;
            if (((c & 4) && !sx) || ((c & 2) && !sy) || ((c & 1) && !sz)) continue;
            const int nb = (wrap(tx + dx) * nt + wrap(ty + dy)) * nt + wrap(tz + dz);
            const int hi = home_halo_index(x - kHomeT * dx + 1, y - kHomeT * dy + 1, z - kHomeT * dz + 1);
            if (!PK_IN(static_cast<int64_t>(nb) * 4 * kHomeHalo + 3 * kHomeHalo + hi,
                       static_cast<int64_t>(gridDim.x) * 4 * kHomeHalo, kChkHalo))
                continue;
            const float *hp = halo + static_cast<int64_t>(nb) * 4 * kHomeHalo + hi;
#pragma unroll
            for (int f = 0; f < 4; ++f) v[f] += hp[f * kHomeHalo];
        }
#pragma unroll
        for (int f = 0; f < 4; ++f) grids[f * grid_elems + gi] = v[f];
    }
}

cudaError_t launch_home(const AssignPlan &pl, const uint32_t *offsets, const unsigned *qmax, const Record<float> *rec,
                        void *grids, float *halo, cudaStream_t s)
{
    constexpr int kMaxDev = 64;
    static bool configured[kMaxDev] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDev || !configured[dev]) {
        e = cudaFuncSetAttribute(k_deposit_home, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kHomeSmem));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(k_deposit_home, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kMaxDev) configured[dev] = true;
    }
    const int ng = pl.ng;
    const unsigned tiles = static_cast<unsigned>((ng / kHomeT) * (ng / kHomeT) * (ng / kHomeT));
    const int64_t grid_elems = static_cast<int64_t>(ng) * ng * (ng + 2);
    auto *g = static_cast<float *>(grids);
    k_deposit_home<<<tiles, kHomeNT, kHomeSmem, s>>>(rec, offsets, qmax, ng, g, grid_elems, halo);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_home_fixup<<<tiles, 256, 0, s>>>(halo, ng, g, grid_elems);
    return cudaGetLastError();
}

struct TileDesc {
    int prec;
    int d[3];
};
constexpr TileDesc kTiles[] = {
    {PKMOM_F32, {16, 16, 16}},  // 0
    {PKMOM_F32, {16, 16, 32}},  // 1
    {PKMOM_F32, {8, 8, 32}},    // 2
    {PKMOM_F32, {8, 8, 8}},     // 3
    {PKMOM_F64, {8, 8, 16}},    // 4
    {PKMOM_F64, {16, 16, 16}},  // 5
    {PKMOM_F64, {8, 8, 8}},     // 6
    {PKMOM_F32, {16, 16, 16}},  // 7: home tiles (cubic order; other orders use tile 0)
};

template <typename T, int M, int T0, int T1, int T2, int NT, int BLR = 0>
cudaError_t launch_deposit_t(const AssignPlan &pl, const uint32_t *offsets, const unsigned *qmax, const Record<T> *rec,
                             void *grids, cudaStream_t s)
{
    using C = DepositCfg<T, M, T0, T1, T2, NT>;
    void (*kern)(const Record<T> *, const uint32_t *, const unsigned *, int, int, T *, int64_t, int, bool);
    size_t smem = C::smem;
    int list_cap = 0;
    if constexpr (sizeof(T) == 4) {
        kern = k_deposit_fx<M, T0, T1, T2, NT, BLR>;
        list_cap = pl.list_cap;
        smem = FxLayout<M, T0, T1, T2>::bytes(list_cap);
    } else if constexpr (M >= 2 && M <= 5 && BLR == 0 && T0 == 8) {
        kern = k_deposit_ix<M, T0, T1, T2, NT>;
        smem = IxLanes<M, T0, T1, T2>::bytes;
    } else {
        kern = k_deposit<T, M, T0, T1, T2, NT, BLR>;
    }
    // the attribute is per device and only needs raising: remember the largest value set
    constexpr int kMaxDev = 64;
    static size_t configured[kMaxDev] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDev || configured[dev] < smem) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kMaxDev) configured[dev] = smem;
    }
    const int ng = pl.ng;
    const int64_t tiles = static_cast<int64_t>(ng / T0) * (ng / T1) * (ng / T2);
    const int64_t grid_elems = static_cast<int64_t>(ng) * ng * (ng + 2);
    kern<<<static_cast<unsigned>(tiles), NT, smem, s>>>(rec, offsets, qmax, ng, pl.sshift, static_cast<T *>(grids),
                                                           grid_elems, list_cap, pl.sparse);
    return cudaGetLastError();
}

template <int M>
cudaError_t launch_deposit_m(const AssignPlan &pl, const uint32_t *offsets, const unsigned *q, const void *rec,
                             void *grids, float *halo, cudaStream_t s)
{
    const auto *rf = static_cast<const Record<float> *>(rec);
    const auto *rd = static_cast<const Record<double> *>(rec);
    switch (pl.tile) {
    case 0: return launch_deposit_t<float, M, 16, 16, 16, 256>(pl, offsets, q, rf, grids, s);
    case 1: return launch_deposit_t<float, M, 16, 16, 32, 512>(pl, offsets, q, rf, grids, s);
    case 2: return launch_deposit_t<float, M, 8, 8, 32, 128>(pl, offsets, q, rf, grids, s);
    case 3: return launch_deposit_t<float, M, 8, 8, 8, 128>(pl, offsets, q, rf, grids, s);
    case 4: return launch_deposit_t<double, M, 8, 8, 16, 256>(pl, offsets, q, rd, grids, s);
    case 5: return launch_deposit_t<double, M, 16, 16, 16, 256>(pl, offsets, q, rd, grids, s);
    case 6: return launch_deposit_t<double, M, 8, 8, 8, 128>(pl, offsets, q, rd, grids, s);
    case 7:
        if constexpr (M == 4) return launch_home(pl, offsets, q, rf, grids, halo, s);
        else return launch_deposit_t<float, M, 16, 16, 16, 256>(pl, offsets, q, rf, grids, s);
    default: return cudaErrorInvalidValue;
    }
}

// The direct truncated-BL deposit (gather tiles 16^3 / 8^3 in FP32, 8x8x16 / 8^3 in FP64).
template <int R>
cudaError_t launch_deposit_bl(const AssignPlan &pl, const uint32_t *offsets, const unsigned *q, const void *rec,
                              void *grids, cudaStream_t s)
{
    constexpr int M = 2 * R;
    const auto *rf = static_cast<const Record<float> *>(rec);
    const auto *rd = static_cast<const Record<double> *>(rec);
    switch (pl.tile) {
    case 0: return launch_deposit_t<float, M, 16, 16, 16, 256, R>(pl, offsets, q, rf, grids, s);
    case 3: return launch_deposit_t<float, M, 8, 8, 8, 128, R>(pl, offsets, q, rf, grids, s);
    case 4: return launch_deposit_t<double, M, 8, 8, 16, 256, R>(pl, offsets, q, rd, grids, s);
    case 6: return launch_deposit_t<double, M, 8, 8, 8, 128, R>(pl, offsets, q, rd, grids, s);
    default: return cudaErrorInvalidValue;
    }
}

// c_n = (1/2 pi) int Sigma_4(w)^{-1/2} e^{i n w} dw by the periodic trapezoid rule on 4096
// points (spectrally accurate for this smooth periodic integrand), with
// Sigma_4(w) = (2416 + 2382 cos w + 240 cos 2w + 2 cos 3w) / 5040 from the integer samples
// of the order-8 B-spline; copied to constant memory once per device.
cudaError_t set_bl_coefficients()
{
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    constexpr int N = 4096;
    constexpr double kPi = 3.14159265358979323846;
    double c[8] = {};
    for (int k = 0; k < N; ++k) {
        const double w = 2.0 * kPi * k / N;
        const double sig = (2416.0 + 2382.0 * std::cos(w) + 240.0 * std::cos(2 * w) + 2.0 * std::cos(3 * w)) / 5040.0;
        const double f = 1.0 / std::sqrt(sig);
        for (int n = 0; n < 8; ++n) c[n] += f * std::cos(n * w);
    }
    float cf[8];
    for (int n = 0; n < 8; ++n) {
        c[n] /= N;
        cf[n] = static_cast<float>(c[n]);
    }
    if ((e = cudaMemcpyToSymbol(c_bl_f, cf, sizeof cf)) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_bl_d, c, sizeof c)) != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) done[dev] = true;
    return cudaSuccess;
}

template <typename T>
const T *tp(const void *p) { return static_cast<const T *>(p); }

}  // namespace

int deposit_tile_count() { return static_cast<int>(sizeof(kTiles) / sizeof(kTiles[0])); }

size_t home_halo_bytes(int ng)
{
    const size_t tiles = size_t(ng / kHomeT) * (ng / kHomeT) * (ng / kHomeT);
    return tiles * 4 * kHomeHalo * sizeof(float);
}

void deposit_tile_shape(int tile, int prec, int dims[3])
{
    dims[0] = dims[1] = dims[2] = 0;
    if (tile < 0 || tile >= deposit_tile_count() || kTiles[tile].prec != prec) return;
    for (int a = 0; a < 3; ++a) dims[a] = kTiles[tile].d[a];
}

// The key table: counts at C = P + 4 words (P = scratch + off_counts; 16-byte aligned
// for the scan's vector accesses). The histogram counts into C[key], the scan turns the
// counts into exclusive offsets in place, and the scatter advances C[key] once per
// particle it places, leaving C[key] = offset[key + 1]. P[3] stays zero, so C - 1 is the
// table offset[0..nkeys] the deposit reads.
size_t key_table_bytes(int64_t nkeys) { return static_cast<size_t>(nkeys + 5) * sizeof(uint32_t); }
uint32_t *key_table(const AssignPlan &pl, void *scratch)
{
    return reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + pl.off_counts) + 4;
}

// The sorted records: on a 32-byte boundary (the scratch is 16-byte aligned; plan_assign
// leaves room for the shift).
void *records_of(const AssignPlan &pl, void *scratch)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(static_cast<char *>(scratch) + pl.off_records);
    return reinterpret_cast<void *>((a + 31) & ~uintptr_t(31));
}
unsigned *control_words(const AssignPlan &pl, void *scratch)
{
    return reinterpret_cast<unsigned *>(static_cast<char *>(scratch) + pl.off_control);
}

cudaError_t launch_hist(const pkmom_catalog &cat, const AssignPlan &pl, double box_L, void *scratch, int *err_flag,
                        cudaStream_t s, LaunchStats &st)
{
    char *sc = static_cast<char *>(scratch);
    uint32_t *counts = key_table(pl, scratch);
    cudaError_t e = cudaMemsetAsync(sc + pl.off_counts, 0, pl.off_records - pl.off_counts, s);
    if (e != cudaSuccess) return e;
    const double scale = static_cast<double>(pl.ng) / box_L;
    if (pl.prec == PKMOM_F32) {
        k_hist<float><<<pl.hist_blocks, kHistThreads, 0, s>>>(tp<float>(cat.x), tp<float>(cat.y), tp<float>(cat.z),
                                                            cat.stride, cat.n, static_cast<float>(scale), pl.ng,
                                                            pl.sshift, counts, err_flag);
    } else {
        k_hist<double><<<pl.hist_blocks, kHistThreads, 0, s>>>(tp<double>(cat.x), tp<double>(cat.y),
                                                             tp<double>(cat.z), cat.stride, cat.n, scale, pl.ng,
                                                             pl.sshift, counts, err_flag);
    }
    st.launches++;
    return cudaGetLastError();
}

size_t control_bytes() { return kCtlWords * sizeof(unsigned); }

cudaError_t launch_scan(const AssignPlan &pl, void *scratch, cudaStream_t s, LaunchStats &st)
{
    char *sc = static_cast<char *>(scratch);
    uint32_t *counts = key_table(pl, scratch);
    auto *bsum = reinterpret_cast<uint32_t *>(sc + pl.off_blocksums);
    const unsigned nb = static_cast<unsigned>(pl.scan_blocks);
    k_scan_reduce<<<nb, kScanThreads, 0, s>>>(counts, pl.nkeys, bsum);
    k_scan_top<<<1, 1024, 0, s>>>(bsum, pl.scan_blocks, counts, pl.nkeys);
    k_scan_apply<<<nb, kScanThreads, 0, s>>>(counts, pl.nkeys, bsum);
    st.launches += 3;
    return cudaGetLastError();
}

namespace {
template <typename T>
void scatter_and_moments(const pkmom_catalog &cat, const AssignPlan &pl, T scale, void *scratch, double *moments_dev,
                         cudaStream_t s)
{
    char *sc = static_cast<char *>(scratch);
    unsigned *ctl = control_words(pl, scratch);
    const T *vx = tp<T>(cat.vx), *vy = tp<T>(cat.vy), *vz = tp<T>(cat.vz), *mass = tp<T>(cat.mass);
    k_scatter<T><<<pl.hist_blocks, 256, 0, s>>>(tp<T>(cat.x), tp<T>(cat.y), tp<T>(cat.z), vx, vy, vz, mass, cat.stride,
                                                cat.n, scale, pl.ng, pl.sshift, key_table(pl, scratch),
                                                static_cast<Record<T> *>(records_of(pl, scratch)));
    auto *partials = reinterpret_cast<double *>(sc + pl.off_partials);
    // four particles a thread at least: the blocks' sums are FP64 work of the last block
    const int64_t want = (cat.n + 4 * kMomentThreads - 1) / (4 * kMomentThreads);
    const unsigned blocks = static_cast<unsigned>(std::min<int64_t>(want, pl.hist_blocks / 2));
    unsigned *qmax = ctl + kCtlQmax, *done = ctl + kCtlDone;
    if constexpr (sizeof(T) == 4) {
        const bool v3 = cat.stride == 3 && vy == vx + 1 && vz == vx + 2 && reinterpret_cast<uintptr_t>(vx) % 16 == 0 &&
                        reinterpret_cast<uintptr_t>(mass) % 16 == 0;
        if (v3) {
            const int64_t lanes = static_cast<int64_t>(pl.hist_blocks) * kMomentThreads;
            if (mass)
                k_moments_v3<true><<<blocks, kMomentThreads, 0, s>>>(vx, mass, cat.n, lanes, partials, qmax, done,
                                                                     moments_dev);
            else
                k_moments_v3<false><<<blocks, kMomentThreads, 0, s>>>(vx, mass, cat.n, lanes, partials, qmax, done,
                                                                      moments_dev);
            return;
        }
    }
    if (mass)
        k_moments<T, true><<<blocks, kMomentThreads, 0, s>>>(vx, vy, vz, mass, cat.stride, cat.n, partials, qmax, done,
                                                             moments_dev);
    else
        k_moments<T, false><<<blocks, kMomentThreads, 0, s>>>(vx, vy, vz, mass, cat.stride, cat.n, partials, qmax, done,
                                                              moments_dev);
}
}  // namespace

cudaError_t launch_scatter(const pkmom_catalog &cat, const AssignPlan &pl, double box_L, void *scratch,
                           double *moments_dev, cudaStream_t s, LaunchStats &st)
{
    const double scale = static_cast<double>(pl.ng) / box_L;
    if (pl.prec == PKMOM_F32) scatter_and_moments<float>(cat, pl, static_cast<float>(scale), scratch, moments_dev, s);
    else scatter_and_moments<double>(cat, pl, scale, scratch, moments_dev, s);
    st.launches += 2;
    return cudaGetLastError();
}

bool batchable_deposit(const AssignPlan &pl)
{
    return pl.prec == PKMOM_F32 && pl.order == 4 && pl.bl_radius == 0 && pl.tile == 0;
}

FxJob deposit_job(const AssignPlan &pl, void *scratch, void *grids)
{
    FxJob j{};
    j.rec = static_cast<const Record<float> *>(records_of(pl, scratch));
    j.offsets = key_table(pl, scratch) - 1;
    j.qmax = control_words(pl, scratch);
    j.grids = static_cast<float *>(grids);
    j.grid_elems = static_cast<int64_t>(pl.ng) * pl.ng * (pl.ng + 2);
    j.ng = pl.ng;
    j.sshift = pl.sshift;
    j.list_cap = pl.list_cap;
    j.sparse = pl.sparse;
    return j;
}

cudaError_t launch_deposit_batch(FxBatch &batch, unsigned long long *counter, int num_sms, cudaStream_t s,
                                 LaunchStats &st)
{
    constexpr int T = 16, NT = 256;
    auto kern = k_deposit_fx_batch<4, T, T, T, NT>;
    long long first = 0;
    int cap = 0;
    for (int k = 0; k < batch.n; ++k) {
        batch.job[k].first_tile = first;
        first += static_cast<long long>(batch.job[k].ng / T) * (batch.job[k].ng / T) * (batch.job[k].ng / T);
        cap = std::max(cap, batch.job[k].list_cap);
    }
    batch.total_tiles = first;
    if (first == 0) return cudaSuccess;
    const size_t smem = FxLayout<4, T, T, T>::bytes(cap);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem)) != cudaSuccess) return e;
    const long long ctas = std::min<long long>(first, static_cast<long long>(std::max(1, per_sm)) * num_sms);
    if ((e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s)) != cudaSuccess) return e;
    kern<<<static_cast<unsigned>(ctas), NT, smem, s>>>(batch, counter);
    st.launches++;
    return cudaGetLastError();
}

cudaError_t launch_deposit(const AssignPlan &pl, void *scratch, void *grids, cudaStream_t s, LaunchStats &st)
{
    char *sc = static_cast<char *>(scratch);
    const uint32_t *offsets = key_table(pl, scratch) - 1;  // offset[0..nkeys] after the scatter
    const unsigned *qmax = control_words(pl, scratch);
    const void *rec = records_of(pl, scratch);
    float *halo = pl.off_halo ? reinterpret_cast<float *>(sc + pl.off_halo) : nullptr;
    cudaError_t e;
    if (pl.bl_radius > 0) {
        if ((e = set_bl_coefficients()) != cudaSuccess) return e;
        switch (pl.bl_radius) {
        case 2: e = launch_deposit_bl<2>(pl, offsets, qmax, rec, grids, s); break;
        case 3: e = launch_deposit_bl<3>(pl, offsets, qmax, rec, grids, s); break;
        case 4: e = launch_deposit_bl<4>(pl, offsets, qmax, rec, grids, s); break;
        default: return cudaErrorInvalidValue;
        }
        st.launches++;
        return e;
    }
    switch (pl.order) {
    case 1: e = launch_deposit_m<1>(pl, offsets, qmax, rec, grids, halo, s); break;
    case 2: e = launch_deposit_m<2>(pl, offsets, qmax, rec, grids, halo, s); break;
    case 3: e = launch_deposit_m<3>(pl, offsets, qmax, rec, grids, halo, s); break;
    case 4: e = launch_deposit_m<4>(pl, offsets, qmax, rec, grids, halo, s); break;
    case 5: e = launch_deposit_m<5>(pl, offsets, qmax, rec, grids, halo, s); break;
    default: return cudaErrorInvalidValue;
    }
    st.launches += (pl.tile == kHomeTile && pl.order == 4) ? 2 : 1;
    return e;
}

}  // namespace pkmom
