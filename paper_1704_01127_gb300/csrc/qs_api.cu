// State management, initial states, FP64 reductions (norm, probabilities,
// entropy / Porter-Thomas moments) and sampling.
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <memory>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "qs_device.cuh"
#include "qs_internal.h"

namespace {
thread_local char g_err[512] = "";

int sm_count_dev()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

int cuda_fail(cudaError_t e, const char *what)
{
    return qs_fail(e == cudaErrorMemoryAllocation ? QS_ENOMEM : QS_ECUDA, "%s: %s", what,
                   cudaGetErrorString(e));
}

#define QS_CUDA(call, what)                          \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

size_t amp_bytes(int dtype) { return dtype == QS_C128 ? 16 : 8; }

// ------------------------------------------------------------------ kernels

template <typename C, typename R>
__global__ void k_fill_uniform(C *psi, uint64_t N, R a)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
        C z;
        z.x = a;
        z.y = 0;
        psi[i] = z;
    }
}

// zeros at every index outside the support {i : (i & ~free) == fix}
template <typename C>
__global__ void k_fill_outside(C *psi, uint64_t N, uint64_t free, uint64_t fix)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
        if ((i & ~free) == fix) continue;
        C z;
        z.x = 0;
        z.y = 0;
        psi[i] = z;
    }
}

template <typename C>
__global__ void k_set_one(C *psi, uint64_t x)
{
    C o;
    o.x = 1;
    o.y = 0;
    psi[x] = o;
}

using qsd::prob;

// p_i = |psi_i|^2 (first <= i < first + count), four steps in flight per thread; VEC = 2:
// two neighbouring complex64 amplitudes per step (16-byte loads and stores).
// 26 qubits: complex64 628 -> 179 us (HBM 159; p is formed in integer operations), complex128 412 -> 266 us
// (HBM 239; its three FP64 operations an amplitude took 348, the squares now run on the integer units).
template <typename C, int VEC>
__global__ void __launch_bounds__(256)
k_probs(const C *__restrict__ psi, uint64_t first, uint64_t count, double *__restrict__ p)
{
    constexpr int kAhead = 4;
    const uint64_t span = (uint64_t)blockDim.x * VEC * kAhead;
    for (uint64_t base = (uint64_t)blockIdx.x * span; base < count; base += (uint64_t)gridDim.x * span) {
        C a[kAhead][VEC];
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint64_t i = base + (uint64_t)(k * blockDim.x + threadIdx.x) * VEC;
            if (i >= count) continue;
            if constexpr (VEC == 2) {
                const float4 w = *reinterpret_cast<const float4 *>(psi + first + i);
                a[k][0] = make_float2(w.x, w.y);
                a[k][1] = make_float2(w.z, w.w);
            } else {
                a[k][0] = psi[first + i];
            }
        }
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint64_t i = base + (uint64_t)(k * blockDim.x + threadIdx.x) * VEC;
            if (i >= count) continue;
            if constexpr (VEC == 2)
                *reinterpret_cast<double2 *>(p + i) = make_double2(prob(a[k][0]), prob(a[k][1]));
            else
                p[i] = prob(a[k][0]);
        }
    }
}

using qsd::ff;
using qsd::ff_abs_double;
using qsd::ff_accumulate;
using qsd::ff_add;
using qsd::ff_p_ln_p;
using qsd::ff_fast_two_sum;
using qsd::ff_sqr_loose;
using qsd::ff_two_sum;
using qsd::FFLogTable;
using qsd::ff_log_table_init;

// The float-float log tables, built once per device (k_fflog_init) and copied
// into shared memory by every block of the statistics kernel.
__device__ __align__(16) FFLogTable g_fflog;

__global__ void k_fflog_init() { ff_log_table_init(g_fflog); }

// p ln p by the FP64 math library, out of the way of the common cases' code
__device__ __noinline__ double p_ln_p_rare(double p) { return p * log(p); }

// Terms of a sum before it goes into the normalised one.  complex64's have no low parts of
// their own and round half as much (32 qubits: 6.06 ms without, 6.15 with 16, 6.04 with 32).
template <typename C> constexpr int kStatsTerms = sizeof(C) == 16 ? 16 : 32;

// Per-thread sums of the statistics; add() takes one amplitude, partials()
// reduces the block (every thread of the block calls it).
struct StatsAcc {
    double d0 = 0, d3 = 0, dent = 0;
    ff f0{0.f, 0.f}, f3{0.f, 0.f}, fent{0.f, 0.f};   // of the terms since the last fold()
    ff g0{0.f, 0.f}, g3{0.f, 0.f}, gent{0.f, 0.f};   // of those before

    // After every kStatsTerms amplitudes: their sums into the normalised ones.
    template <int NSTAT>
    __device__ __forceinline__ void fold()
    {
        g0 = ff_add(g0, f0);
        f0 = ff{0.f, 0.f};
        if (NSTAT == 4) {
            g3 = ff_add(g3, f3);
            gent = ff_add(gent, fent);
            f3 = fent = ff{0.f, 0.f};
        }
    }

    template <int NSTAT>
    __device__ __forceinline__ void add(const double2 a, const FFLogTable &lt)
    {
        // magnitude tests on the high words (integer compares; FP64 compares
        // would run on the FP64 pipe): below 2^30, and 2^-60 or more
        const uint32_t hx = (uint32_t)__double2hiint(a.x) & 0x7FFFFFFFu, hy = (uint32_t)__double2hiint(a.y) & 0x7FFFFFFFu;
        if (max(hx, hy) < 1053u << 20) {
            // |x| and |y| as float-float (values below 2^-60 add less than 2^-120
            // to p and count as zero); p = x^2 + y^2 with the low parts' errors added
            // once, then normalised
            const ff x = hx >= 963u << 20 ? ff_abs_double(hx, (uint32_t)__double2loint(a.x)) : ff{0.f, 0.f};
            const ff y = hy >= 963u << 20 ? ff_abs_double(hy, (uint32_t)__double2loint(a.y)) : ff{0.f, 0.f};
            const ff xx = ff_sqr_loose(x), yy = ff_sqr_loose(y);
            const ff t = ff_two_sum(xx.hi, yy.hi);
            const ff p = ff_fast_two_sum(t.hi, __fadd_rn(t.lo, __fadd_rn(xx.lo, yy.lo)));
            ff_accumulate(f0, p);
            if (NSTAT == 4) {
                ff_accumulate(f3, ff_sqr_loose(p));
                if (p.hi >= 0x1p-79f) {
                    ff_accumulate(fent, ff_p_ln_p(lt, p));
                } else if (p.hi > 0.f) {
                    const double pd = (double)p.hi + (double)p.lo;
                    if (pd >= 2.2250738585072014e-308) dent += pd * log(pd);
                }
            }
        } else {
            // an amplitude of 2^30 or more (unnormalised input): FP64 throughout
            const double p = fma(a.x, a.x, a.y * a.y);
            d0 += p;
            if (NSTAT == 4) {
                d3 = fma(p, p, d3);
                dent += p * log(p);
            }
        }
    }

    template <int NSTAT>
    __device__ __forceinline__ void add(const float2 a, const FFLogTable &)
    {
        // complex64 amplitudes carry FP32 errors (2^-24 relative): p, p^2
        // and the logarithm of p are formed in FP32 (one rounding each, the
        // logarithm a few ulp), and the terms add up in float-float
        const float p = fmaf(a.x, a.x, __fmul_rn(a.y, a.y));
        ff_accumulate(f0, p);
        if (NSTAT == 4) {
            ff_accumulate(f3, __fmul_rn(p, p));
            if (p >= 0x1p-79f && p <= 0x1p100f) {
                ff_accumulate(fent, __fmul_rn(p, __logf(p)));
            } else if (p > 0.f) {
                const double pd = (double)p;
                if (pd >= 2.2250738585072014e-308) dent += p_ln_p_rare(pd);
            }
        }
    }

    // part[blockIdx.x * NSTAT + j]: the block's sums of (p, -p ln p, p, p^2)
    template <int NSTAT>
    __device__ void partials(double *__restrict__ part)
    {
        fold<NSTAT>();
        double acc[NSTAT];
        acc[0] = d0 + ((double)g0.hi + (double)g0.lo);
        if (NSTAT == 4) {
            acc[NSTAT > 1 ? 1 : 0] = -(dent + ((double)gent.hi + (double)gent.lo));
            acc[NSTAT > 2 ? 2 : 0] = acc[0];
            acc[NSTAT > 3 ? 3 : 0] = d3 + ((double)g3.hi + (double)g3.lo);
        }
        __shared__ double red[NSTAT][32];
#pragma unroll
        for (int j = 0; j < NSTAT; j++) {
            double v = acc[j];
            for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if ((threadIdx.x & 31) == 0) red[j][threadIdx.x >> 5] = v;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            int nw = blockDim.x >> 5;
#pragma unroll
            for (int j = 0; j < NSTAT; j++) {
                double v = threadIdx.x < nw ? red[j][threadIdx.x] : 0.0;
                for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (threadIdx.x == 0) part[(size_t)blockIdx.x * NSTAT + j] = v;
            }
        }
    }
};

// The log tables into shared memory (complex128 statistics only).
template <typename C, int NSTAT>
__device__ __forceinline__ void load_fflog(FFLogTable &lt)
{
    if (NSTAT == 4 && sizeof(C) == 16) {
        const uint2 *src = reinterpret_cast<const uint2 *>(&g_fflog);
        uint2 *dst = reinterpret_cast<uint2 *>(&lt);
        for (int i = threadIdx.x; i < (int)(sizeof(FFLogTable) / sizeof(uint2)); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
    }
}

// Per-block FP64 partial sums of (p, -p ln p, p, p^2); NSTAT = 1 or 4.  The
// mean of N p equals the sum of p, and the mean of (N p)^2 is N sum p^2, so
// the moments cost one product per amplitude; the host applies the factor N.
// Everything runs in float-float on the FP32 pipe (GB300's FP64 pipe runs at
// 1/64 of its rate): complex128 amplitudes are split into float-float by bit
// manipulation (the lowest 29 of their 53 bits rounded to 24), complex64 ones give
// p rounded to 32 bits.  p, p^2 and p ln p (table-driven log, ff_p_ln_p) are summed
// per thread in float-float, in sums of 16 or 32 terms that go into normalised ones.
// Errors against exact sums at 28 qubits, relative: random amplitudes 3e-15 (p), 2e-15
// (entropy), 6e-15 (p^2); equal amplitudes, whose rounding errors add up, up to 3e-14
// (1.7e-11 without the sums of 16; 1.4e-13 with each term added to a normalised sum).
// The sums of 16 (complex64: 32) cost at most 0.7% of a pass, within 48 registers: at 54,
// one block less per SM, 1%.  p below 2^-79
// (where the low half of p's float-float form would leave the normal float
// range) takes p ln p from the FP64 math library, and complex128 amplitudes of
// 2^30 or more (unnormalised input) are summed in FP64 throughout; p below the
// normal double range contributes less than 1e-305 and is left out.
template <typename C> constexpr int kStatsAhead = sizeof(C) == 16 ? 4 : 8;   // loads in flight per thread

template <typename C, int NSTAT>
__global__ void __launch_bounds__(256, NSTAT == 4 ? 5 : 8) k_stats_partial(const C *__restrict__ psi, uint64_t N, double *__restrict__ part)
{
    __shared__ __align__(16) FFLogTable lt;
    load_fflog<C, NSTAT>(lt);
    StatsAcc acc;
    // each thread loads kAhead amplitudes (block-strided, so every load of a
    // warp is contiguous) before it adds them up: more loads in flight
    constexpr int kAhead = kStatsAhead<C>;
    constexpr uint32_t kBatches = kStatsTerms<C> / kAhead;
    const uint64_t span = (uint64_t)blockDim.x * kAhead;
    uint32_t batch = 0;
    for (uint64_t base = (uint64_t)blockIdx.x * span; base < N; base += (uint64_t)gridDim.x * span) {
        C av[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint64_t i = base + (uint64_t)k * blockDim.x + threadIdx.x;
            av[k] = i < N ? psi[i] : C{};   // a zero amplitude adds nothing
        }
#pragma unroll
        for (int k = 0; k < kAhead; k++) acc.add<NSTAT>(av[k], lt);
        if (++batch % kBatches == 0) acc.fold<NSTAT>();
    }
    acc.partials<NSTAT>(part);
}

// The blocks' partial sums added up in a fixed order by one block (2432 of them:
// 27 us by one warp, 8 us by 512 threads).
constexpr int kFinalThreads = 512;

template <int NSTAT>
__global__ void __launch_bounds__(kFinalThreads) k_stats_final(const double *__restrict__ part, int nblocks, double *__restrict__ out)
{
    __shared__ double red[NSTAT][kFinalThreads / 32];
    double acc[NSTAT];
#pragma unroll
    for (int j = 0; j < NSTAT; j++) acc[j] = 0;
    for (int b = threadIdx.x; b < nblocks; b += kFinalThreads)
#pragma unroll
        for (int j = 0; j < NSTAT; j++) acc[j] += part[(size_t)b * NSTAT + j];
#pragma unroll
    for (int j = 0; j < NSTAT; j++) {
        double v = acc[j];
        for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[j][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
#pragma unroll
    for (int j = 0; j < NSTAT; j++) {
        double v = threadIdx.x < kFinalThreads / 32 ? red[j][threadIdx.x] : 0.0;
        for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) out[j] = v;
    }
}

std::mutex g_fflog_mu;
bool g_fflog_ready[64] = {false};

// Build the log tables on the current device once (one block, then a wait).
int ensure_fflog(cudaStream_t st)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return qs_fail(QS_EUNSUPPORTED, "statistics: no usable device");
    std::lock_guard<std::mutex> lock(g_fflog_mu);
    if (g_fflog_ready[dev]) return QS_OK;
    k_fflog_init<<<1, 1024, 0, st>>>();
    QS_CUDA(cudaGetLastError(), "log table launch");
    QS_CUDA(cudaStreamSynchronize(st), "log table");
    g_fflog_ready[dev] = true;
    return QS_OK;
}

// ------------------------------------------------------------------ sampling
constexpr uint32_t kFull = 0xffffffffu;

// Pairwise sums over fixed power-of-two blocks (blocks of 1024 amplitudes:
// k_block_sums): lane l of a warp reduces its contiguous len/32 values as a perfect
// binary tree, then the 32 lane results combine as the top five tree levels (lane
// pairs (0,1), (2,3), ... first).

template <typename C>
__device__ double load_p(const C *psi, uint64_t i) { return prob(psi[i]); }
__device__ double load_p(const double *v, uint64_t i) { return v[i]; }

template <typename T>
__device__ double tree_sum_serial(const T *src, uint64_t start, int len)
{
    double buf[32];
    for (int i = 0; i < len; i++) buf[i] = load_p(src, start + i);
    for (int w = len; w > 1; w >>= 1)
        for (int i = 0; i < w / 2; i++) buf[i] = buf[2 * i] + buf[2 * i + 1];
    return buf[0];
}

// The same pairwise tree over LEN values, unrolled: the loads are all issued
// first and the tree stays in registers (the runtime-length form above keeps
// its buffer in local memory).
template <int LEN, typename T>
__device__ __forceinline__ double tree_sum_fixed(const T *src, uint64_t start)
{
    double buf[LEN];
#pragma unroll
    for (int i = 0; i < LEN; i++) buf[i] = load_p(src, start + i);
#pragma unroll
    for (int w = LEN; w > 1; w >>= 1) {
#pragma unroll
        for (int i = 0; i < w / 2; i++) buf[i] = buf[2 * i] + buf[2 * i + 1];
    }
    return buf[0];
}

// One warp per segment of `len` (power of two, >= 32) values; PER > 0: len is
// 32 PER, summed by the unrolled tree.
template <typename T, int PER>
__global__ void k_segment_sums(const T *__restrict__ src, uint64_t nseg, int len, double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const int per = PER > 0 ? PER : len >> 5;
    for (uint64_t seg = warp; seg < nseg; seg += nwarps) {
        const uint64_t start = seg * (uint64_t)len + (uint64_t)lane * per;
        double v;
        if constexpr (PER > 0) v = tree_sum_fixed<PER>(src, start);
        else v = tree_sum_serial(src, start, per);
        for (int o = 1; o < 32; o <<= 1) {
            double w = __shfl_down_sync(0xffffffffu, v, o);
            if ((lane & (2 * o - 1)) == 0) v = v + w;
        }
        if (lane == 0) out[seg] = v;
    }
}

// The pairwise tree over a block of 1024 probabilities, by one warp with contiguous
// loads: rows of 32 amplitudes (complex64: 64, a lane holds a pair and joins it),
// eight rows to a piece.  A piece is summed over lane bits 0 to 2 by halving exchanges
// (a lane keeps half of its rows and hands the other half to its partner: 7
// additions, not 24), which leaves those bits numbering the rows from the top; the
// pieces go on the same way over bits 3 and 4; then the rows are summed over the lanes
// that hold them, lowest row bit first, and the pieces likewise.  Addition commutes,
// so these are the tree's sums bit for bit, 1.125 FP64 additions a value.  (Each lane
// reading its own 32 values needs every 32-byte sector several times over from a
// cache that the warps of an SM overflow.)
template <int N>
__device__ __forceinline__ void halve(double *v, int o)
{
    const bool up = threadIdx.x & o;
#pragma unroll
    for (int i = 0; i < N / 2; i++) {
        const double mine = up ? v[i + N / 2] : v[i], other = up ? v[i] : v[i + N / 2];
        v[i] = mine + __shfl_xor_sync(kFull, other, o);
    }
}

// Rows 0 .. 7 from p on, summed over lane bits 0 to 2; seen(a): every amplitude.
template <typename F>
__device__ __forceinline__ double piece_sum(const float4 *__restrict__ p, F seen)
{
    float4 a[8];
    double v[8];
#pragma unroll
    for (int t = 0; t < 8; t++) a[t] = p[32 * t];
#pragma unroll
    for (int t = 0; t < 8; t++) {
        const float2 x = make_float2(a[t].x, a[t].y), y = make_float2(a[t].z, a[t].w);
        seen(x);
        seen(y);
        v[t] = prob(x) + prob(y);
    }
    halve<8>(v, 1);
    halve<4>(v, 2);
    halve<2>(v, 4);
    return v[0];
}
template <typename F>
__device__ __forceinline__ double piece_sum(const double2 *__restrict__ p, F seen)
{
    double2 a[8];
    double v[8];
#pragma unroll
    for (int t = 0; t < 8; t++) a[t] = p[32 * t];
#pragma unroll
    for (int t = 0; t < 8; t++) {
        seen(a[t]);
        v[t] = prob(a[t]);
    }
    halve<8>(v, 1);
    halve<4>(v, 2);
    halve<2>(v, 4);
    return v[0];
}

// (One piece after another: unrolled altogether, with the statistics, the code leaves
// the instruction cache.)  With the statistics, 29 qubits complex64: 3.33 ms as one
// 32-value run per lane, 1.71 ms.
template <typename C, typename F>
__device__ __forceinline__ double block_sum(const C *__restrict__ psi, F seen)
{
    using V = std::conditional_t<sizeof(C) == 8, float4, double2>;
    constexpr int kPieces = sizeof(C) == 8 ? 2 : 4;
    const V *p = reinterpret_cast<const V *>(psi) + (threadIdx.x & 31);
    double v[kPieces];
#pragma unroll
    for (int j = 0; j < kPieces; j++) v[j] = 0;
#pragma unroll 1
    for (int i = 0; i < kPieces; i++) {
#pragma unroll
        for (int j = 0; j + 1 < kPieces; j++) v[j] = v[j + 1];
        v[kPieces - 1] = piece_sum(p + 256 * i, seen);
    }
    halve<kPieces>(v, 8);
    if constexpr (kPieces == 4) halve<2>(v, 16);
    else v[0] = v[0] + __shfl_xor_sync(kFull, v[0], 16);
    double t = v[0];
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1) t = t + __shfl_xor_sync(kFull, t, o);
    if constexpr (kPieces == 4) t = t + __shfl_xor_sync(kFull, t, 16);
    return t + __shfl_xor_sync(kFull, t, 8);
}

template <typename C>
__global__ void __launch_bounds__(256)
k_block_sums(const C *__restrict__ psi, uint64_t nb, double *__restrict__ out)
{
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t b = warp; b < nb; b += nwarps) {
        const double v = block_sum(psi + b * 1024, [](const C &) {});
        if ((threadIdx.x & 31) == 0) out[b] = v;
    }
}

// The block sums and, from the same loads, the block's partial sums of the
// statistics as k_stats_partial<C, 4> forms them (in another order).  The block
// sums use the FP64 unit, their squares the integer units, the statistics the FP32
// ones (launched for complex64 states); bound by issue slots.
template <typename C>
__global__ void __launch_bounds__(256, 3)
k_block_sums_stats(const C *__restrict__ psi, uint64_t nb, double *__restrict__ out, double *__restrict__ part)
{
    __shared__ __align__(16) FFLogTable lt;
    load_fflog<C, 4>(lt);
    StatsAcc acc;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t b = warp; b < nb; b += nwarps) {
        const double v = block_sum(psi + b * 1024, [&](const C &a) { acc.add<4>(a, lt); });
        acc.fold<4>();   // 32 terms
        if ((threadIdx.x & 31) == 0) out[b] = v;
    }
    acc.partials<4>(part);
}

// Segments shorter than a warp: one thread per segment.
template <typename T>
__global__ void k_segment_sums_small(const T *__restrict__ src, uint64_t nseg, int len, double *__restrict__ out)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t seg = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; seg < nseg; seg += stride)
        out[seg] = tree_sum_serial(src, seg * (uint64_t)len, len);
}

// Sequential sums c <- fl(c + p), p >= 0.  The order of the additions is part of
// the draws' definition, but they need not run one after another: while c
// stays in one binade with unit u in the last place, fl(c + p) = c + u r(p)
// with r(p) = p / u rounded to an integer, whatever c is, unless p / u lies
// exactly half-way (then the parity of c decides).  So a warp rounds 32 values
// to units of c's last place, adds integers in any order, and takes the 32
// additions one by one only where a value ties or the sum reaches the next
// binade.  Bit for bit the sequential sums, without the FP64 pipe and without
// its latency 32 times over.
// r(p) for a sum with exponent field E >= 1; *slow: a tie, or p as large as c.
__device__ __forceinline__ uint64_t chain_term(double p, int E, bool &slow)
{
    const uint64_t b = (uint64_t)__double_as_longlong(p);
    const int e = (int)(b >> 52);
    const uint64_t f = b & 0xFFFFFFFFFFFFFULL, m = e ? f | (1ULL << 52) : f;
    const int sh = E - max(e, 1);
    if (sh >= 54) return 0;                       // below u / 4
    if (sh <= 0) {
        slow = slow || m != 0;                    // c + p leaves the binade (infinities and NaN too)
        return 0;
    }
    const uint64_t t = m + (1ULL << (sh - 1));
    slow = slow || (t << (64 - sh)) == 0;         // exactly half-way
    return t >> sh;
}

// The 32 additions in lane order; *incl: the sum up to this lane's value.
__device__ __forceinline__ double chain_slow(double c, double p, double &incl)
{
    const int lane = threadIdx.x & 31;
    incl = 0.0;
#pragma unroll 8
    for (int k = 0; k < 32; k++) {
        c = c + __shfl_sync(kFull, p, k);
        if (lane == k) incl = c;
    }
    return c;
}

// sum of v < 2^54 over the warp, in every lane (two 27-bit halves, 32 of which fit 32 bits)
__device__ __forceinline__ uint64_t warp_sum54(uint64_t v)
{
    const uint32_t lo = __reduce_add_sync(kFull, (uint32_t)v & 0x7FFFFFFu);
    const uint32_t hi = __reduce_add_sync(kFull, (uint32_t)(v >> 27));
    return (uint64_t)lo + ((uint64_t)hi << 27);
}

// c after this warp's 32 values in lane order; *half: the sum after lane 15's.
__device__ __forceinline__ double chain_add(double c, double p, double &half)
{
    double incl;
    const double end = chain_slow(c, p, incl);
    half = __shfl_sync(kFull, incl, 15);
    return end;
}

// The same for N groups of 32 values, half[k] and full[k] after group k's lanes 15 and
// 31: all N at once while the sum stays in one binade without ties (the terms then
// depend on c's exponent alone), else one group after another, addition by addition.
// 2^e the start of c's binade, u = 2^(e-52): for p < 2^(e-20) - 2^(e-41) a term is the
// low word of fl(2^e + p) (it rounds to at most 2^32 - 2^11 units; the p up to 2^(e-20)
// left out, one value of the high word, can round to 2^32 units, which that word does
// not hold) and a tie needs 20 zero bits at p's end.  Where some value has those (equal
// or real-valued amplitudes) the bits that a term drops are looked at; where some is
// larger, the terms come from chain_term.
template <int N>
__device__ __forceinline__ double chain_add_n(double c, const double *p, double *half, double *full)
{
    const uint64_t cb = (uint64_t)__double_as_longlong(c);
    const int E = (int)(cb >> 52);
    const bool low = (threadIdx.x & 31) < 16;
    const double c0 = __longlong_as_double((long long)(cb & 0x7FF0000000000000ULL));
    const uint32_t top = ((uint32_t)max(E - 20, 1) << 20) - 1u;
    uint32_t v[N], any = 0;
    bool large = E < 64, zeros = false;
#pragma unroll
    for (int k = 0; k < N; k++) {
        const uint32_t h = (uint32_t)__double2hiint(p[k]), l = (uint32_t)__double2loint(p[k]);
        v[k] = (uint32_t)__double2loint(c0 + p[k]);
        any |= v[k];
        large = large || h >= top;
        zeros = zeros || ((l & 0xFFFFFu) == 0 && (h | l) != 0);
    }
    uint64_t at = cb, mid[N], end[N];
    bool slow = false;
    if (!__any_sync(kFull, large)) {
        if (__any_sync(kFull, zeros)) {
#pragma unroll
            for (int k = 0; k < N; k++) {
                const uint64_t b = (uint64_t)__double_as_longlong(p[k]);
                const int sh = E - (int)(b >> 52);   // the term drops p's last sh bits, 21 of them or more
                const uint64_t m = (b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
                slow = slow || (sh < 54 && m << (64 - sh) == 1ULL << 63);
            }
            slow = __any_sync(kFull, slow);
        }
        if (!__any_sync(kFull, any >> 27)) {   // 32 terms add up in 32 bits
#pragma unroll
            for (int k = 0; k < N; k++) {
                mid[k] = at + __reduce_add_sync(kFull, low ? v[k] : 0u);
                end[k] = at = at + __reduce_add_sync(kFull, v[k]);
            }
        } else {
#pragma unroll
            for (int k = 0; k < N; k++) {
                const uint32_t h = low ? v[k] : 0u;
                mid[k] = at + __reduce_add_sync(kFull, h & 0xFFFFu) + ((uint64_t)__reduce_add_sync(kFull, h >> 16) << 16);
                end[k] = at = at + __reduce_add_sync(kFull, v[k] & 0xFFFFu) + ((uint64_t)__reduce_add_sync(kFull, v[k] >> 16) << 16);
            }
        }
    } else {
        slow = E == 0;
#pragma unroll
        for (int k = 0; k < N; k++) {
            const uint64_t r = chain_term(p[k], E, slow);
            mid[k] = at + warp_sum54(low ? r : 0);
            end[k] = at = at + warp_sum54(r);
        }
        slow = __any_sync(kFull, slow);
    }
    if (slow || (int)(at >> 52) != E) {
#pragma unroll 1
        for (int k = 0; k < N; k++) {
#pragma unroll
            for (int j = 0; j < N; j++)
                if (j == k) {
                    c = chain_add(c, p[j], half[j]);
                    full[j] = c;
                }
        }
        return c;
    }
#pragma unroll
    for (int k = 0; k < N; k++) {
        half[k] = __longlong_as_double((long long)mid[k]);
        full[k] = __longlong_as_double((long long)end[k]);
    }
    return full[N - 1];
}

// The same with the sums before and after this lane's value.
__device__ __forceinline__ double chain_scan(double c, double p, double &excl, double &incl)
{
    const int lane = threadIdx.x & 31;
    const uint64_t cb = (uint64_t)__double_as_longlong(c);
    const int E = (int)(cb >> 52);
    bool slow = E == 0;
    const uint64_t r = chain_term(p, E, slow);
    uint64_t v = r;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t w = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += w;
    }
    const uint64_t all = __shfl_sync(kFull, v, 31);
    // r < 2^53 each: 32 of them stay below 2^58
    if (__any_sync(kFull, slow) || (int)((cb + all) >> 52) != E) {
        const double end = chain_slow(c, p, incl);
        excl = __shfl_up_sync(kFull, incl, 1);
        if (lane == 0) excl = c;
        return end;
    }
    excl = __longlong_as_double((long long)(cb + v - r));
    incl = __longlong_as_double((long long)(cb + v));
    return __longlong_as_double((long long)(cb + all));
}

// One warp: out[i] = the sequential sum of v[0 .. i-1] on top of c0 (out[0] = c0).
__device__ __forceinline__ void prefix_chain(const double *__restrict__ v, uint64_t n, double c0, double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    constexpr int kAhead = 8;
    double c = c0;
    for (uint64_t i0 = 0; i0 < n; i0 += 32 * kAhead) {
        double x[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; k++) x[k] = i0 + 32 * k + lane < n ? v[i0 + 32 * k + lane] : 0.0;
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            if (i0 + 32 * k >= n) break;
            double excl, incl;
            c = chain_scan(c, x[k], excl, incl);
            if (i0 + 32 * k + lane < n) out[i0 + 32 * k + lane] = excl;
        }
    }
}

// Q_0 = 0, Q_{s+1} = Q_s + T_s (one warp).  R_{s,0} = Q_s (0 without Q),
// R_{s,j+1} = R_{s,j} + S_{sG+j}, a warp per super-block.  One thread per chain,
// 29 qubits (512 chains of 1024): 37 + 154 us, now 16 + 23 us.
__global__ void k_prefix_super(const double *__restrict__ T, uint64_t ns, double *__restrict__ Q) { prefix_chain(T, ns, 0.0, Q); }

__global__ void __launch_bounds__(128)
k_prefix_blocks(const double *__restrict__ S, const double *__restrict__ Q, uint64_t ns, uint64_t G, double *__restrict__ R)
{
    const uint64_t s = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s < ns) prefix_chain(S + s * G, G, Q ? Q[s] : 0.0, R + s * G);
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t j)
{
    uint64_t z = seed + (j + 1) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// last index in [0, len) with a[idx] <= u (a non-decreasing, a[0] <= u)
__device__ uint64_t last_le(const double *a, uint64_t len, double u)
{
    uint64_t lo = 0, hi = len;   // invariant: a[lo] <= u, answer in [lo, hi)
    while (hi - lo > 1) {
        uint64_t mid = lo + (hi - lo) / 2;
        if (a[mid] <= u) lo = mid; else hi = mid;
    }
    return lo;
}

template <typename C>
__global__ void k_draw(const C *__restrict__ psi, const double *__restrict__ Q, const double *__restrict__ R,
                       uint64_t ns, uint64_t G, uint64_t B, uint64_t seed, int64_t m, uint64_t *__restrict__ out)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += stride) {
        double u = (double)(splitmix64(seed, (uint64_t)j) >> 11) * 0x1.0p-53;
        uint64_t s = last_le(Q, ns, u);
        uint64_t jb = last_le(R + s * G, G, u);
        uint64_t b = s * G + jb;
        double c = R[b];
        uint64_t i = B - 1;
        for (uint64_t x = 0; x < B; x++) {
            c = c + prob(psi[b * B + x]);
            if (c > u) { i = x; break; }
        }
        out[j] = b * B + i;
    }
}

// ---- draws by checkpoints of the running sums (blocks of 1024)
//
// The per-draw scan above adds the probabilities of one block to R_b one after
// another until the sum passes u.  The sums c_{b,x} = R_b + p_{bB} + ... +
// p_{bB+x}, in that order, are the same for every draw of the block and do not
// decrease (p >= 0 and rounding is monotone), so each block that some draw
// falls into is summed once, the sum kept after every kCkRun values, and a draw
// then finds its run among the block's checkpoints and adds up that run alone:
// bit for bit the scan's outcome.
//   k_locate      block of every draw; with few draws for the number of blocks,
//                 the list of the blocks that were hit (slot[b]: b's place in it)
//   k_checkpoints the sums, a warp per block
//   k_draw_run    the draws
// 27 qubits complex64, 10^6 draws: 6.26 ms (a scan per draw) -> 0.94 ms; 29
// qubits, 4096 draws: 441 -> 50 us.  complex128 stored every probability and
// every running sum before (N doubles of scratch).
constexpr int kCkRun = 16;
constexpr int kCks = 1024 / kCkRun;

__global__ void k_locate(const double *__restrict__ Q, const double *__restrict__ R, uint64_t ns, uint64_t G, uint64_t seed,
                         int64_t m, uint32_t *__restrict__ blk, uint32_t *__restrict__ slot, uint32_t *__restrict__ list,
                         uint32_t *__restrict__ n_list, unsigned long long *__restrict__ umax)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; j0 < m; j0 += stride) {
        const int64_t j = j0 + lane;
        uint32_t b = 0;
        bool first = false;
        if (j < m) {
            const double u = (double)(splitmix64(seed, (uint64_t)j) >> 11) * 0x1.0p-53;
            const uint64_t s = last_le(Q, ns, u);
            b = (uint32_t)(s * G + last_le(R + s * G, G, u));
            blk[j] = b;
            if (umax) atomicMax(&umax[b], (unsigned long long)__double_as_longlong(u));   // u >= 0: the bits order as the values
            if (slot) first = atomicExch(&slot[b], 0u) == 0xFFFFFFFFu;
        }
        if (slot) {
            const uint32_t hits = __ballot_sync(0xffffffffu, first);
            uint32_t at = 0;
            if (lane == 0 && hits) at = atomicAdd(n_list, (uint32_t)__popc(hits));
            at = __shfl_sync(0xffffffffu, at, 0) + (uint32_t)__popc(hits & ((1u << lane) - 1u));
            if (first) list[at] = b;
        }
    }
}

// slot[list[i]] = i (after k_locate: every block is in the list once)
__global__ void k_slots(const uint32_t *__restrict__ list, const uint32_t *__restrict__ n_list, uint32_t *__restrict__ slot)
{
    const uint32_t n = *n_list;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) slot[list[i]] = i;
}

template <typename C>
__global__ void __launch_bounds__(128, 8)
k_checkpoints(const C *__restrict__ psi, const double *__restrict__ R, uint32_t nb, const uint32_t *__restrict__ list,
              const uint32_t *__restrict__ n_list, const double *__restrict__ umax, double *__restrict__ ck)
{
    static_assert(kCkRun == 16, "two checkpoints per 32 values");
    const int lane = threadIdx.x & 31;
    const uint32_t n_work = list ? *n_list : nb, nwarps = (gridDim.x * blockDim.x) >> 5;
    constexpr int kAhead = 4;
    for (uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < n_work; w += nwarps) {
        const uint32_t b = list ? list[w] : w;
        const C *p = psi + (uint64_t)b * 1024 + lane;
        const double last = umax ? umax[b] : __longlong_as_double(0x7FF0000000000000LL);
        double c = R[b], keep[2];                     // lane t keeps the checkpoints of values 32 t .. 32 t + 31
        for (int t0 = 0; t0 < 32; t0 += kAhead) {
            C a[kAhead];
#pragma unroll
            for (int t = 0; t < kAhead; t++) a[t] = p[32 * (t0 + t)];
            double q[kAhead], half[kAhead], full[kAhead];
#pragma unroll
            for (int t = 0; t < kAhead; t++) q[t] = prob(a[t]);
            c = chain_add_n<kAhead>(c, q, half, full);
#pragma unroll
            for (int t = 0; t < kAhead; t++)
                if (lane == t0 + t) {
                    keep[0] = half[t];
                    keep[1] = full[t];
                }
            if (c > last) {                           // past every draw of the block: the rest is not searched
                if (lane >= t0 + kAhead) keep[0] = keep[1] = c;
                break;
            }
        }
        *reinterpret_cast<double2 *>(ck + (uint64_t)w * kCks + 2 * lane) = make_double2(keep[0], keep[1]);
    }
}

// Every running sum of every block, for many draws per block (a draw then needs no
// additions).  complex128, 2^18 draws of 12 qubits: 228 -> 156 us a call, 2^20 of 20
// qubits: 521 -> 369 us.
template <typename C>
__global__ void __launch_bounds__(128)
k_running_sums(const C *__restrict__ psi, const double *__restrict__ R, uint32_t nb, double *__restrict__ sums)
{
    const int lane = threadIdx.x & 31;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    constexpr int kAhead = 8;
    for (uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < nb; b += nwarps) {
        const C *p = psi + (uint64_t)b * 1024 + lane;
        double c = R[b];
        for (int t0 = 0; t0 < 32; t0 += kAhead) {
            C a[kAhead];
#pragma unroll
            for (int t = 0; t < kAhead; t++) a[t] = p[32 * (t0 + t)];
#pragma unroll
            for (int t = 0; t < kAhead; t++) {
                double excl, incl;
                c = chain_scan(c, prob(a[t]), excl, incl);
                sums[(uint64_t)b * 1024 + 32 * (t0 + t) + lane] = incl;
            }
        }
    }
}

// kEvery: ck holds every running sum, not one of kCkRun.
template <typename C, bool kEvery>
__global__ void k_draw_run(const C *__restrict__ psi, const double *__restrict__ R, const double *__restrict__ ck,
                           const uint32_t *__restrict__ blk, const uint32_t *__restrict__ slot, uint64_t seed, int64_t m,
                           uint64_t *__restrict__ out)
{
    constexpr int kN = kEvery ? 1024 : kCks;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += stride) {
        const double u = (double)(splitmix64(seed, (uint64_t)j) >> 11) * 0x1.0p-53;
        const uint64_t b = blk[j];
        const double *cb = ck + (uint64_t)(slot ? slot[b] : b) * kN;
        int lo = 0, hi = kN;                 // first run whose last sum passes u
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (cb[mid] > u) hi = mid; else lo = mid + 1;
        }
        int x = 1023;                        // none: the block's last value
        if (kEvery) {
            x = min(lo, 1023);
        } else if (lo < kCks) {
            double c = lo ? cb[lo - 1] : R[b];
            const C *p = psi + b * 1024 + (uint64_t)lo * kCkRun;
            for (x = 0; x < kCkRun - 1; x++) {
                c = c + prob(p[x]);
                if (c > u) break;
            }
            x += lo * kCkRun;
        }
        out[j] = b * 1024 + (uint64_t)x;
    }
}

// 16 blocks of 256 per SM: the float-float work is latency-bound at lower occupancy
// (30 qubits: 7.35 ms with 4 per SM, 6.64 ms with 16).  No block without an amplitude: its
// closing sums are FP64 work all the same (19 qubits: complex64 54 -> 31 us a call, complex128
// 56 -> 43).
constexpr int kStatsBlocksPerSM = 16;

template <typename C>
int stats_grid(uint64_t N, int per_sm)
{
    constexpr uint64_t span = 256 * kStatsAhead<C>;
    return (int)std::min<uint64_t>((N + span - 1) / span, (uint64_t)sm_count_dev() * per_sm);
}

template <typename C>
int stats_impl(qs_state *s, double *out, int nstat)
{
    uint64_t N = 1ULL << s->n;
    const int block = 256, grid = stats_grid<C>(N, kStatsBlocksPerSM);
    void *scr = nullptr;
    int rc = qs_state_scratch(s, sizeof(double) * (size_t)(grid + 1) * 4, &scr);
    if (rc) return rc;
    double *part = (double *)scr, *res = part + (size_t)grid * 4;
    cudaStream_t st = (cudaStream_t)s->stream;
    if (nstat == 4 && (rc = ensure_fflog(st))) return rc;
    if (nstat == 1) {
        k_stats_partial<C, 1><<<grid, block, 0, st>>>((const C *)s->amp, N, part);
        k_stats_final<1><<<1, kFinalThreads, 0, st>>>(part, grid, res);
    } else {
        k_stats_partial<C, 4><<<grid, block, 0, st>>>((const C *)s->amp, N, part);
        k_stats_final<4><<<1, kFinalThreads, 0, st>>>(part, grid, res);
    }
    QS_CUDA(cudaGetLastError(), "stats launch");
    QS_CUDA(cudaMemcpyAsync(out, res, sizeof(double) * nstat, cudaMemcpyDeviceToHost, st), "stats copy");
    QS_CUDA(cudaStreamSynchronize(st), "stats sync");
    if (nstat == 4) out[3] *= (double)N;   // mean of (N p)^2 = N sum p^2
    return QS_OK;
}

// The state's second stream and its fork/join events, made on first use.
int side_stream(qs_state *s, cudaStream_t *out)
{
    if (!s->side) {
        cudaStream_t ss;
        QS_CUDA(cudaStreamCreateWithFlags(&ss, cudaStreamNonBlocking), "side stream");
        cudaEvent_t e[2];
        for (int i = 0; i < 2; i++) {
            cudaError_t err = cudaEventCreateWithFlags(&e[i], cudaEventDisableTiming);
            if (err != cudaSuccess) {
                for (int j = 0; j < i; j++) cudaEventDestroy(e[j]);
                cudaStreamDestroy(ss);
                return cuda_fail(err, "side stream events");
            }
        }
        s->side = ss;
        s->side_ev[0] = e[0];
        s->side_ev[1] = e[1];
    }
    *out = (cudaStream_t)s->side;
    return QS_OK;
}

// stats (optional): also the statistics of qs_stats.  complex64 states with
// blocks of 1024 take them from the same pass over the state as the block sums
// (33.9 ms instead of 7.6 + 29.4 ms for 2^20 draws at 32 qubits).  complex128
// states with blocks of 1024 run the statistics pass (FP32 pipe) on a second
// stream beside the block sums (FP64 pipe), forked from and joined to the
// state's stream (one kernel doing both measured 28.6 ms against 7.2 + 19.7
// ms, its FP64 and FP32 work not overlapping); otherwise stats_impl runs
// first.
template <typename C>
int sample_impl(qs_state *s, uint64_t seed, int64_t m, uint64_t *out, double *stats)
{
    const uint64_t N = 1ULL << s->n;
    const uint64_t B = std::min<uint64_t>(N, 1024), nb = N / B;
    const uint64_t G = std::min<uint64_t>(nb, 1024), ns = nb / G;
    const int sms = sm_count_dev();
    const int gb = (int)std::min<uint64_t>((nb * 32 + 255) / 256, (uint64_t)sms * 16);
    constexpr bool c64 = sizeof(C) == 8;
    const bool fused = c64 && stats && B == 1024;
    const bool beside = !c64 && stats && B == 1024;
    if (stats && !fused && !beside)
        if (int rc = stats_impl<C>(s, stats, 4)) return rc;
    cudaStream_t st = (cudaStream_t)s->stream, ss = nullptr;
    if (fused || beside)
        if (int rc = ensure_fflog(st)) return rc;
    if (beside)
        if (int rc = side_stream(s, &ss)) return rc;
    const int sgrid = stats_grid<C>(N, kStatsBlocksPerSM);   // stats_impl's
    const size_t stats_bytes = beside ? sizeof(double) * ((size_t)sgrid + 1) * 4 : 0;
    const size_t m_slots = (size_t)std::max<int64_t>(m, 1);
    size_t bytes = sizeof(double) * (2 * nb + 2 * ns) + sizeof(uint64_t) * m_slots;
    if (fused) bytes += sizeof(double) * ((size_t)gb * 4 + 4);
    // blocks of 1024: checkpoints of the running sums of every block, or of those
    // hit when the draws cannot hit most of them; without room for them the
    // draws scan their blocks (the same outcomes)
    bool runs = B == 1024 && m > 0;
    const bool listed = m < 2 * (int64_t)nb, every = m >= 128 * (int64_t)nb;
    // a block is summed up to its largest draw where that saves more than the table
    // costs: some 16 draws per block at most (4: a fifth of the sums; 28 qubits
    // complex128, 2^20 draws: checkpoints 1.44 -> 1.31 ms), and many blocks (21 qubits 3% slower)
    const bool part_way = !every && nb >= (1u << 15) && m <= 16 * (int64_t)nb;
    const size_t n_work = listed ? (size_t)std::min<uint64_t>(nb, m_slots) : nb;
    const size_t n_sums = n_work * (every ? 1024 : kCks);
    const size_t runs_bytes = sizeof(double) * (n_sums + (part_way ? nb : 0)) + sizeof(uint32_t) * (m_slots + (listed ? nb + n_work + 1 : 0)) + 16;
    void *scr = nullptr;
    int rc = qs_state_scratch(s, bytes + stats_bytes + (runs ? runs_bytes : 0), &scr);
    if (rc && runs) {
        cudaGetLastError();   // the failed allocation is not an error of the later launches
        runs = false;
        rc = qs_state_scratch(s, bytes + stats_bytes, &scr);
    }
    if (rc) return rc;
    double *S = (double *)scr, *R = S + nb, *T = R + nb, *Q = T + ns;
    uint64_t *dout = (uint64_t *)(Q + ns);
    double *part = (double *)(dout + m_slots), *res = part + (size_t)gb * 4;
    // the statistics' partial sums (complex128), then the draws' tables
    double *spart = (double *)((char *)scr + bytes), *sres = spart + (size_t)sgrid * 4;
    double *ck = (double *)(((uintptr_t)scr + bytes + stats_bytes + 15) & ~(uintptr_t)15);
    double *umax = part_way ? ck + n_sums : nullptr;   // largest draw of each block
    uint32_t *blk = (uint32_t *)(ck + n_sums + (part_way ? nb : 0)), *slot = listed ? blk + m_slots : nullptr;
    uint32_t *list = listed ? slot + nb : nullptr, *n_list = listed ? list + n_work : nullptr;
    const C *psi = (const C *)s->amp;
    if (beside) {
        QS_CUDA(cudaEventRecord((cudaEvent_t)s->side_ev[0], st), "side fork");
        QS_CUDA(cudaStreamWaitEvent(ss, (cudaEvent_t)s->side_ev[0], 0), "side fork");
        k_stats_partial<C, 4><<<sgrid, 256, 0, ss>>>(psi, N, spart);
        k_stats_final<4><<<1, kFinalThreads, 0, ss>>>(spart, sgrid, sres);
        QS_CUDA(cudaGetLastError(), "stats launch");
        QS_CUDA(cudaEventRecord((cudaEvent_t)s->side_ev[1], ss), "side join");
    }
    if (fused) {
        if constexpr (c64) k_block_sums_stats<C><<<gb, 256, 0, st>>>(psi, nb, S, part);
        k_stats_final<4><<<1, kFinalThreads, 0, st>>>(part, gb, res);
    } else if (B == 1024)
        k_block_sums<C><<<gb, 256, 0, st>>>(psi, nb, S);
    else if (B >= 32)
        k_segment_sums<C, 0><<<gb, 256, 0, st>>>(psi, nb, (int)B, S);
    else
        k_segment_sums_small<C><<<1, 32, 0, st>>>(psi, nb, (int)B, S);
    if (ns > 1) {   // G = 1024
        const int gs = (int)std::min<uint64_t>((ns * 32 + 255) / 256, (uint64_t)sms * 16);
        k_segment_sums<double, 32><<<gs, 256, 0, st>>>(S, ns, (int)G, T);
        k_prefix_super<<<1, 32, 0, st>>>(T, ns, Q);
    }
    k_prefix_blocks<<<(int)((ns + 3) / 4), 128, 0, st>>>(S, ns > 1 ? Q : nullptr, ns, G, R);
    const int gd = (int)std::min<int64_t>((m + 127) / 128, (int64_t)sms * 16);
    if (runs) {
        if (listed) QS_CUDA(cudaMemsetAsync(slot, 0xFF, sizeof(uint32_t) * nb, st), "draw table");
        if (listed) QS_CUDA(cudaMemsetAsync(n_list, 0, sizeof(uint32_t), st), "draw table");
        if (umax) QS_CUDA(cudaMemsetAsync(umax, 0, sizeof(double) * nb, st), "draw table");
        k_locate<<<gd, 128, 0, st>>>(Q, R, ns, G, seed, m, blk, slot, list, n_list, (unsigned long long *)umax);
        if (listed) k_slots<<<gd, 128, 0, st>>>(list, n_list, slot);
        const int gr = (int)std::min<uint64_t>((n_work + 3) / 4, (uint64_t)sms * 8);   // one wave
        if (every) {
            k_running_sums<C><<<gr, 128, 0, st>>>(psi, R, (uint32_t)nb, ck);
            k_draw_run<C, true><<<gd, 128, 0, st>>>(psi, R, ck, blk, slot, seed, m, dout);
        } else {
            k_checkpoints<C><<<gr, 128, 0, st>>>(psi, R, (uint32_t)nb, list, n_list, umax, ck);
            k_draw_run<C, false><<<gd, 128, 0, st>>>(psi, R, ck, blk, slot, seed, m, dout);
        }
    } else if (m > 0) {
        k_draw<C><<<gd, 128, 0, st>>>(psi, Q, R, ns, G, B, seed, m, dout);
    }
    QS_CUDA(cudaGetLastError(), "sampling launch");
    if (m > 0)
        QS_CUDA(cudaMemcpyAsync(out, dout, sizeof(uint64_t) * m, cudaMemcpyDeviceToHost, st), "sample copy");
    if (fused)
        QS_CUDA(cudaMemcpyAsync(stats, res, sizeof(double) * 4, cudaMemcpyDeviceToHost, st), "stats copy");
    if (beside) {
        QS_CUDA(cudaStreamWaitEvent(st, (cudaEvent_t)s->side_ev[1], 0), "side join");
        QS_CUDA(cudaMemcpyAsync(stats, sres, sizeof(double) * 4, cudaMemcpyDeviceToHost, st), "stats copy");
    }
    QS_CUDA(cudaStreamSynchronize(st), "sampling sync");
    if (fused || beside) stats[3] *= (double)N;   // mean of (N p)^2 = N sum p^2
    return QS_OK;
}

// Amplitudes at up to kGatherIdx indices, the indices in the launch's own
// parameters (no copy to the device), widened to double2 in the scratch.
constexpr int kGatherIdx = 480;
struct GatherIdx {
    uint64_t at[kGatherIdx];
};

template <typename C>
__global__ void k_gather(const C *__restrict__ psi, const __grid_constant__ GatherIdx ix, int count, double2 *__restrict__ out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= count) return;
    const C a = psi[ix.at[j]];
    out[j] = make_double2(a.x, a.y);
}

// Amplitudes at `count` checked indices to the host: launches of kGatherIdx
// indices into the scratch, one copy per kGatherChunk results.  One 8- or
// 16-byte copy per index, each waiting for the one before, took 22 ms for 2048
// indices, this takes 60 us.
constexpr int64_t kGatherChunk = 1 << 16;

template <typename C>
int gather_impl(qs_state *s, const uint64_t *idx, int64_t count, double *out)
{
    cudaStream_t st = (cudaStream_t)s->stream;
    const bool moved = !qs_loc_identity(s);
    void *scr = nullptr;
    // one copy per index: for one (15 us, a launch and a copy take 21), for up to four on a state
    // that has no scratch yet (60 us, its allocation alone takes 90), and without room for it
    const bool copies = count <= (s->scratch ? 1 : 4);
    if (copies || qs_state_scratch(s, sizeof(double2) * (size_t)std::min(count, kGatherChunk), &scr)) {
        if (!copies) cudaGetLastError();
        for (int64_t j = 0; j < count; j++) {
            C a;
            QS_CUDA(cudaMemcpyAsync(&a, (const C *)s->amp + (moved ? qs_loc_index(s, idx[j]) : idx[j]), sizeof(C),
                                    cudaMemcpyDeviceToHost, st), "qs_get_amplitudes_at");
            QS_CUDA(cudaStreamSynchronize(st), "qs_get_amplitudes_at");
            out[2 * j] = a.x;
            out[2 * j + 1] = a.y;
        }
        return QS_OK;
    }
    for (int64_t c0 = 0; c0 < count; c0 += kGatherChunk) {
        const int64_t n = std::min(kGatherChunk, count - c0);
        for (int64_t j0 = 0; j0 < n; j0 += kGatherIdx) {
            GatherIdx ix;
            const int m = (int)std::min<int64_t>(kGatherIdx, n - j0);
            // the indices in the state's bit order (qubits may sit at other bits)
            for (int j = 0; j < m; j++) ix.at[j] = moved ? qs_loc_index(s, idx[c0 + j0 + j]) : idx[c0 + j0 + j];
            k_gather<C><<<(m + 31) / 32, 32, 0, st>>>((const C *)s->amp, ix, m, (double2 *)scr + j0);
        }
        QS_CUDA(cudaGetLastError(), "qs_get_amplitudes_at");
        QS_CUDA(cudaMemcpyAsync(out + 2 * c0, scr, sizeof(double2) * n, cudaMemcpyDeviceToHost, st), "qs_get_amplitudes_at");
        QS_CUDA(cudaStreamSynchronize(st), "qs_get_amplitudes_at");
    }
    return QS_OK;
}

int make_state(int n, int dtype, void *stream, void *ptr, bool owned, qs_state **out)
{
    qs_state *s = new (std::nothrow) qs_state();
    if (!s) return qs_fail(QS_ENOMEM, "out of host memory");
    s->n = n;
    s->dtype = dtype;
    s->amp = ptr;
    s->owned = owned;
    s->stream = stream;
    cudaGetDevice(&s->device);
    *out = s;
    return QS_OK;
}

}  // namespace

// ---------------------------------------------------------------- internals

int qs_fail(int code, const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

int qs_state_scratch(qs_state *s, size_t bytes, void **out)
{
    if (bytes > s->scratch_bytes) {
        if (s->scratch) {
            cudaStreamSynchronize((cudaStream_t)s->stream);
            cudaFree(s->scratch);
            s->scratch = nullptr;
            s->scratch_bytes = 0;
        }
        size_t want = std::max<size_t>(bytes, 1 << 20);
        cudaError_t e = cudaMalloc(&s->scratch, want);
        if (e != cudaSuccess) {
            s->scratch = nullptr;
            return cuda_fail(e, "scratch allocation");
        }
        s->scratch_bytes = want;
    }
    *out = s->scratch;
    return QS_OK;
}

int qs_state_status(qs_state *s, int **out)
{
    if (!s->status) {
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, 256);
        if (e != cudaSuccess) return cuda_fail(e, "status word");
        e = cudaMemsetAsync(p, 0, 256, (cudaStream_t)s->stream);
        if (e != cudaSuccess) {
            cudaFree(p);
            return cuda_fail(e, "status word");
        }
        s->status = (int *)p;
    }
    *out = s->status;
    return QS_OK;
}

int qs_check_status(qs_state *s)
{
    if (!s->status) return QS_OK;
    int v = 0;
    cudaStream_t st = (cudaStream_t)s->stream;
    QS_CUDA(cudaMemcpyAsync(&v, s->status, sizeof(int), cudaMemcpyDeviceToHost, st), "status read");
    QS_CUDA(cudaStreamSynchronize(st), "status read");
    if (v) {
        cudaMemsetAsync(s->status, 0, sizeof(int), st);
        if (v & 1) return qs_fail(QS_ETIMEOUT, "a kernel's bounded wait ran out (status %d)", v);
        return qs_fail(QS_EINVAL, "amplitudes above ~2^1010 in magnitude: outside the complex128 tensor-core sweep's range");
    }
    return QS_OK;
}

// ------------------------------------------------------------------- C ABI

extern "C" const char *qs_last_error(void) { return g_err; }

extern "C" int qs_alloc(int n, int dtype, void *stream, qs_state **out)
{
    return qs_guard([&]() -> int {
        if (!out || n < 1 || n > QS_MAX_QUBITS || (dtype != QS_C64 && dtype != QS_C128))
            return qs_fail(QS_EINVAL, "qs_alloc: n = %d, dtype = %d not supported", n, dtype);
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, amp_bytes(dtype) << n);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return qs_fail(QS_ENOMEM, "qs_alloc: %zu bytes: %s", amp_bytes(dtype) << n, cudaGetErrorString(e));
        }
        int rc = make_state(n, dtype, stream, p, true, out);
        if (rc) cudaFree(p);
        return rc;
    });
}

extern "C" int qs_wrap(void *dev_ptr, int n, int dtype, void *stream, qs_state **out)
{
    return qs_guard([&]() -> int {
        if (!out || !dev_ptr || ((uintptr_t)dev_ptr & 15) || n < 1 || n > QS_MAX_QUBITS ||
            (dtype != QS_C64 && dtype != QS_C128))
            return qs_fail(QS_EINVAL, "qs_wrap: bad pointer, n or dtype");
        return make_state(n, dtype, stream, dev_ptr, false, out);
    });
}

extern "C" void qs_free(qs_state *s)
{
    if (!s) return;
    if (s->stream) cudaStreamSynchronize((cudaStream_t)s->stream);
    else cudaDeviceSynchronize();
    if (s->owned && s->amp) cudaFree(s->amp);
    if (s->scratch) cudaFree(s->scratch);
    if (s->pinned) cudaFreeHost(s->pinned);
    if (s->status) cudaFree(s->status);
    if (s->side) {
        cudaStreamSynchronize((cudaStream_t)s->side);
        cudaStreamDestroy((cudaStream_t)s->side);
    }
    for (void *e : s->side_ev)
        if (e) cudaEventDestroy((cudaEvent_t)e);
    delete s;
}

extern "C" int qs_set_path(qs_state *s, int path)
{
    return qs_guard([&]() -> int {
        if (!s || path < QS_PATH_AUTO || path > QS_PATH_TENSOR) return qs_fail(QS_EINVAL, "qs_set_path");
        s->path = path;
        return QS_OK;
    });
}

extern "C" int qs_set_phase_fold(qs_state *s, int on)
{
    return qs_guard([&]() -> int {
        if (!s) return qs_fail(QS_EINVAL, "qs_set_phase_fold: null state");
        s->fold_phase = on != 0;
        return QS_OK;
    });
}

extern "C" int qs_num_qubits(const qs_state *s) { return s ? s->n : 0; }
extern "C" int qs_dtype(const qs_state *s) { return s ? s->dtype : -1; }
// the caller reads the buffer directly: the zeros outside the support first
extern "C" void *qs_device_ptr(const qs_state *s)
{
    if (!s) return nullptr;
    if (qs_guard([&]() { return qs_order_set(const_cast<qs_state *>(s), nullptr); })) return nullptr;
    if (qs_materialize(const_cast<qs_state *>(s))) return nullptr;
    return s->amp;
}
extern "C" int qs_set_stream(qs_state *s, void *stream)
{
    return qs_guard([&]() -> int {
        if (!s) return qs_fail(QS_EINVAL, "qs_set_stream: null state");
        if (stream != s->stream) {
            // the new stream starts after everything queued on the old one
            cudaEvent_t ev;
            QS_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming), "qs_set_stream: event");
            cudaError_t e = cudaEventRecord(ev, (cudaStream_t)s->stream);
            if (e == cudaSuccess) e = cudaStreamWaitEvent((cudaStream_t)stream, ev, 0);
            cudaEventDestroy(ev);
            if (e != cudaSuccess) return cuda_fail(e, "qs_set_stream");
        }
        s->stream = stream;
        return QS_OK;
    });
}

// |x>: one amplitude written, the support set to {x}; the zeros elsewhere are
// written by the first call that needs them (qs_materialize), and sweeps on
// the tensor cores never need them (Sec. 3.6 starts from a known state too).
// States on a caller's buffer (qs_wrap) get their zeros at once.
extern "C" int qs_init_basis(qs_state *s, uint64_t x)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp) return qs_fail(QS_EINVAL, "qs_init_basis: null state");
        if (x >> s->n) return qs_fail(QS_EINVAL, "qs_init_basis: index out of range");
        qs_loc_reset(s);   // fresh contents: every qubit at its own bit
        s->perm_invariant = false;
        cudaStream_t st = (cudaStream_t)s->stream;
        if (s->dtype == QS_C128)
            k_set_one<double2><<<1, 1, 0, st>>>((double2 *)s->amp, x);
        else
            k_set_one<float2><<<1, 1, 0, st>>>((float2 *)s->amp, x);
        QS_CUDA(cudaGetLastError(), "qs_init_basis");
        s->sup_free = 0;
        s->sup_fix = x;
        // a wrapped buffer can be read by its owner without a library call: its
        // zeros are written now
        return s->owned ? QS_OK : qs_materialize(s);
    });
}

int qs_basis_move(qs_state *s, uint64_t x)
{
    s->perm_invariant = false;
    cudaStream_t st = (cudaStream_t)s->stream;
    if (s->dtype == QS_C128)
        k_set_one<double2><<<1, 1, 0, st>>>((double2 *)s->amp, x);
    else
        k_set_one<float2><<<1, 1, 0, st>>>((float2 *)s->amp, x);
    QS_CUDA(cudaGetLastError(), "basis move");
    s->sup_free = 0;
    s->sup_fix = x;
    return QS_OK;
}

int qs_materialize(qs_state *s)
{
    if (qs_support_full(s)) return QS_OK;
    const uint64_t N = 1ULL << s->n, all = qs_index_mask(s->n);
    const uint64_t fr = s->sup_free & all, fx = s->sup_fix & ~fr & all;
    int grid = (int)std::min<uint64_t>((N + 255) / 256, (uint64_t)sm_count_dev() * 8);
    cudaStream_t st = (cudaStream_t)s->stream;
    if (s->dtype == QS_C128)
        k_fill_outside<double2><<<grid, 256, 0, st>>>((double2 *)s->amp, N, fr, fx);
    else
        k_fill_outside<float2><<<grid, 256, 0, st>>>((float2 *)s->amp, N, fr, fx);
    QS_CUDA(cudaGetLastError(), "fill outside the support");
    s->sup_free = ~0ULL;
    s->sup_fix = 0;
    return QS_OK;
}

extern "C" int qs_init_uniform(qs_state *s)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp) return qs_fail(QS_EINVAL, "qs_init_uniform: null state");
        qs_loc_reset(s);   // fresh contents: every qubit at its own bit
        uint64_t N = 1ULL << s->n;
        int grid = (int)std::min<uint64_t>((N + 255) / 256, (uint64_t)sm_count_dev() * 8);
        cudaStream_t st = (cudaStream_t)s->stream;
        // 2^{-n/2}: exact power of two for even n; sqrt(0.5) * 2^{-(n-1)/2} for odd n
        double a = (s->n % 2 == 0) ? ldexp(1.0, -s->n / 2) : sqrt(0.5) * ldexp(1.0, -(s->n - 1) / 2);
        if (s->dtype == QS_C128)
            k_fill_uniform<double2, double><<<grid, 256, 0, st>>>((double2 *)s->amp, N, a);
        else
            k_fill_uniform<float2, float><<<grid, 256, 0, st>>>((float2 *)s->amp, N, (float)a);
        QS_CUDA(cudaGetLastError(), "qs_init_uniform");
        s->sup_free = ~0ULL;
        s->sup_fix = 0;
        s->perm_invariant = true;   // every amplitude equal
        return QS_OK;
    });
}

extern "C" int qs_set_amplitudes(qs_state *s, const double *host)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || !host) return qs_fail(QS_EINVAL, "qs_set_amplitudes: null argument");
        qs_loc_reset(s);   // fresh contents: every qubit at its own bit
        s->perm_invariant = false;
        uint64_t N = 1ULL << s->n;
        cudaStream_t st = (cudaStream_t)s->stream;
        if (s->dtype == QS_C128) {
            QS_CUDA(cudaMemcpyAsync(s->amp, host, 16 * N, cudaMemcpyHostToDevice, st), "qs_set_amplitudes");
        } else {
            // a host copy as large as the state (32 GiB at 32 qubits): no throw
            std::unique_ptr<float[]> f(new (std::nothrow) float[2 * N]);
            if (!f) return qs_fail(QS_ENOMEM, "qs_set_amplitudes: out of host memory");
            for (uint64_t i = 0; i < 2 * N; i++) f[i] = (float)host[i];
            QS_CUDA(cudaMemcpyAsync(s->amp, f.get(), 8 * N, cudaMemcpyHostToDevice, st), "qs_set_amplitudes");
        }
        QS_CUDA(cudaStreamSynchronize(st), "qs_set_amplitudes sync");
        s->sup_free = ~0ULL;
        s->sup_fix = 0;
        return QS_OK;
    });
}

extern "C" int qs_get_amplitudes(qs_state *s, double *host)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || !host) return qs_fail(QS_EINVAL, "qs_get_amplitudes: null argument");
        if (int rc = qs_check_status(s)) return rc;
        if (int rc = qs_order_set(s, nullptr)) return rc;   // index order
        if (int rc = qs_materialize(s)) return rc;
        uint64_t N = 1ULL << s->n;
        cudaStream_t st = (cudaStream_t)s->stream;
        if (s->dtype == QS_C128) {
            QS_CUDA(cudaMemcpyAsync(host, s->amp, 16 * N, cudaMemcpyDeviceToHost, st), "qs_get_amplitudes");
            QS_CUDA(cudaStreamSynchronize(st), "qs_get_amplitudes sync");
        } else {
            std::unique_ptr<float[]> f(new (std::nothrow) float[2 * N]);
            if (!f) return qs_fail(QS_ENOMEM, "qs_get_amplitudes: out of host memory");
            QS_CUDA(cudaMemcpyAsync(f.get(), s->amp, 8 * N, cudaMemcpyDeviceToHost, st), "qs_get_amplitudes");
            QS_CUDA(cudaStreamSynchronize(st), "qs_get_amplitudes sync");
            for (uint64_t i = 0; i < 2 * N; i++) host[i] = (double)f[i];
        }
        return QS_OK;
    });
}

extern "C" int qs_get_amplitudes_at(qs_state *s, const uint64_t *idx, int64_t count, double *out)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || count < 0 || (count > 0 && (!idx || !out)))
            return qs_fail(QS_EINVAL, "qs_get_amplitudes_at: bad arguments");
        if (int rc = qs_check_status(s)) return rc;
        if (int rc = qs_materialize(s)) return rc;
        const uint64_t N = 1ULL << s->n;
        for (int64_t j = 0; j < count; j++)
            if (idx[j] >= N) return qs_fail(QS_EINVAL, "qs_get_amplitudes_at: index %lld out of range", (long long)j);
        return s->dtype == QS_C128 ? gather_impl<double2>(s, idx, count, out) : gather_impl<float2>(s, idx, count, out);
    });
}

extern "C" int qs_norm(qs_state *s, double *out)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || !out) return qs_fail(QS_EINVAL, "qs_norm: null argument");
        if (int rc = qs_check_status(s)) return rc;
        if (int rc = qs_materialize(s)) return rc;
        return s->dtype == QS_C128 ? stats_impl<double2>(s, out, 1) : stats_impl<float2>(s, out, 1);
    });
}

extern "C" int qs_stats(qs_state *s, double out[4])
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || !out) return qs_fail(QS_EINVAL, "qs_stats: null argument");
        if (int rc = qs_check_status(s)) return rc;
        if (int rc = qs_materialize(s)) return rc;
        return s->dtype == QS_C128 ? stats_impl<double2>(s, out, 4) : stats_impl<float2>(s, out, 4);
    });
}

extern "C" int qs_probabilities(qs_state *s, double *out, int out_on_device)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || !out) return qs_fail(QS_EINVAL, "qs_probabilities: null argument");
        if (int rc = qs_order_set(s, nullptr)) return rc;   // index order
        if (int rc = qs_materialize(s)) return rc;
        const uint64_t N = 1ULL << s->n;
        cudaStream_t st = (cudaStream_t)s->stream;
        const int sms = sm_count_dev();
        auto launch = [&](uint64_t first, uint64_t count, double *dst) {
            const int grid = (int)std::min<uint64_t>((count + 1023) / 1024, (uint64_t)sms * 8);
            if (s->dtype == QS_C128)
                k_probs<double2, 1><<<grid, 256, 0, st>>>((const double2 *)s->amp, first, count, dst);
            else if (((uintptr_t)dst & 15) == 0)   // 16-byte stores (count is even, the state 16-byte aligned)
                k_probs<float2, 2><<<(grid + 1) / 2, 256, 0, st>>>((const float2 *)s->amp, first, count, dst);
            else
                k_probs<float2, 1><<<grid, 256, 0, st>>>((const float2 *)s->amp, first, count, dst);
        };
        if (out_on_device) {
            launch(0, N, out);
            QS_CUDA(cudaGetLastError(), "qs_probabilities");
            return QS_OK;
        }
        // host output: chunks of at most 2^25 values through the scratch buffer
        const uint64_t chunk = std::min<uint64_t>(N, 1ULL << 25);
        void *scr = nullptr;
        int rc = qs_state_scratch(s, sizeof(double) * chunk, &scr);
        if (rc) return rc;
        for (uint64_t first = 0; first < N; first += chunk) {
            launch(first, chunk, (double *)scr);
            QS_CUDA(cudaGetLastError(), "qs_probabilities");
            QS_CUDA(cudaMemcpyAsync(out + first, scr, sizeof(double) * chunk, cudaMemcpyDeviceToHost, st),
                    "qs_probabilities copy");
        }
        QS_CUDA(cudaStreamSynchronize(st), "qs_probabilities sync");
        return QS_OK;
    });
}

extern "C" int qs_sample(qs_state *s, uint64_t seed, int64_t m, uint64_t *out)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || m < 0 || (m > 0 && !out)) return qs_fail(QS_EINVAL, "qs_sample: bad arguments");
        if (int rc = qs_order_set(s, nullptr)) return rc;   // index order
        if (int rc = qs_materialize(s)) return rc;
        return s->dtype == QS_C128 ? sample_impl<double2>(s, seed, m, out, nullptr)
                                   : sample_impl<float2>(s, seed, m, out, nullptr);
    });
}

extern "C" int qs_sample_stats(qs_state *s, uint64_t seed, int64_t m, uint64_t *out, double *stats)
{
    return qs_guard([&]() -> int {
        if (!s || !s->amp || m < 0 || (m > 0 && !out) || !stats)
            return qs_fail(QS_EINVAL, "qs_sample_stats: bad arguments");
        if (int rc = qs_check_status(s)) return rc;
        if (int rc = qs_order_set(s, nullptr)) return rc;   // index order
        if (int rc = qs_materialize(s)) return rc;
        return s->dtype == QS_C128 ? sample_impl<double2>(s, seed, m, out, stats)
                                   : sample_impl<float2>(s, seed, m, out, stats);
    });
}

extern "C" int qs_synchronize(qs_state *s)
{
    return qs_guard([&]() -> int {
        if (!s) return qs_fail(QS_EINVAL, "qs_synchronize: null state");
        QS_CUDA(cudaStreamSynchronize((cudaStream_t)s->stream), "qs_synchronize");
        return qs_check_status(s);
    });
}

extern "C" int qs_selftest_timeout(qs_state *s)
{
    return qs_guard([&]() -> int {
        if (!s) return qs_fail(QS_EINVAL, "qs_selftest_timeout: null state");
        int rc = qs_launch_wait_selftest(s, 1000);
        if (rc) return rc;
        QS_CUDA(cudaStreamSynchronize((cudaStream_t)s->stream), "qs_selftest_timeout");
        return qs_check_status(s);
    });
}

// --------------------------------------------------------------------------
// Allocation-free statistics (no counterpart in the paper).
//
// For callers that must not allocate device memory: the partial sums live in a
// file-scope device array instead of the state's scratch.  Every call shares
// it, so calls whose kernels overlap on the GPU race on it.
// --------------------------------------------------------------------------
namespace {

constexpr int kStaticStatsBlocks = 1024;   // partial sums per statistic
// 4 statistics per block, plus 4 result slots: 4 * 1025 doubles = 32800 bytes.
static __device__ __align__(256) double g_stats_scratch[4 * (kStaticStatsBlocks + 1)];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
double *g_static_ptr[kMaxDevices] = {nullptr};

// Device address of g_stats_scratch on the current device (looked up once per
// device, with that device current).
int static_scratch(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "qs_stats_static: cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) return qs_fail(QS_EUNSUPPORTED, "qs_stats_static: device %d", dev);
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_stats_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(e, "qs_stats_static: cudaGetSymbolAddress");
        g_static_ptr[dev] = (double *)p;
    }
    *out = g_static_ptr[dev];
    return QS_OK;
}

template <typename C>
int stats_static_impl(const void *amp, int n, void *stream, double *out)
{
    double *scr;
    int rc = static_scratch(&scr);
    if (rc) return rc;
    const uint64_t N = 1ULL << n;
    const int block = 256;
    const int grid = std::min(stats_grid<C>(N, 4), kStaticStatsBlocks);
    double *part = scr, *res = scr + 4 * kStaticStatsBlocks;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = ensure_fflog(st))) return rc;
    // every partial slot in [0, grid) and every result slot is written before it is read
    k_stats_partial<C, 4><<<grid, block, 0, st>>>((const C *)amp, N, part);
    k_stats_final<4><<<1, kFinalThreads, 0, st>>>(part, grid, res);
    QS_CUDA(cudaGetLastError(), "qs_stats_static launch");
    QS_CUDA(cudaMemcpyAsync(out, res, sizeof(double) * 4, cudaMemcpyDeviceToHost, st), "qs_stats_static copy");
    QS_CUDA(cudaStreamSynchronize(st), "qs_stats_static sync");
    out[3] *= (double)N;   // mean of (N p)^2 = N sum p^2
    return QS_OK;
}

}  // namespace

extern "C" int qs_stats_static(const void *dev_amp, int n, int dtype, void *stream, double out[4])
{
    return qs_guard([&]() -> int {
        if (!dev_amp || !out) return qs_fail(QS_EINVAL, "qs_stats_static: null pointer");
        if (n < 1 || n > QS_MAX_QUBITS)
            return qs_fail(QS_EINVAL, "qs_stats_static: n = %d outside [1, %d]", n, QS_MAX_QUBITS);
        if (dtype != QS_C64 && dtype != QS_C128)
            return qs_fail(QS_EINVAL, "qs_stats_static: dtype %d", dtype);
        // the kernel loads whole amplitudes: aligned to their size
        if ((uintptr_t)dev_amp & (amp_bytes(dtype) - 1))
            return qs_fail(QS_EINVAL, "qs_stats_static: pointer not aligned to %zu bytes", amp_bytes(dtype));
        return dtype == QS_C128 ? stats_static_impl<double2>(dev_amp, n, stream, out)
                                : stats_static_impl<float2>(dev_amp, n, stream, out);
    });
}
