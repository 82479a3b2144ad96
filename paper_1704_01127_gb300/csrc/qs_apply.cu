// State sweeps of the hot path: dense k-qubit cluster apply (Sec. 3.2), table
// diagonals and CZ/T phase products (Sec. 2, Sec. 3.5), and the schedule runner.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "qs_device.cuh"
#include "qs_internal.h"
#include "qs_launch.cuh"

namespace {

using qsd::cplx;
using qsd::Targets;
using qsd::group_base;
using qsd::member_offset;

int g_sms = 0;
int sm_count()
{
    if (!g_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

// Dense k-qubit cluster: one thread per group c, the 2^K amplitudes gathered at
// strides 2^{q_j} into registers, v <- U v, scattered back in place.  Each
// complex multiply-accumulate is the pair of real FMA updates of Eqs. (2)-(3):
// acc += (v_R m_R, v_I m_R) then acc += (-v_I m_I, v_R m_I).  U (row-major,
// ascending qubit order) is staged once per CTA in shared memory and read as a
// warp-uniform broadcast.  Consecutive threads take consecutive groups, so for
// targets above bit 4 every gathered row of a warp is one contiguous segment.
template <typename R, int K>
__global__ void __launch_bounds__(128)
k_dense(typename cplx<R>::t *__restrict__ psi, uint64_t n_groups, Targets t,
        const R *__restrict__ Ug)
{
    using C = typename cplx<R>::t;
    constexpr int D = 1 << K;
    __shared__ C Us[D * D];
    chain_start();
    for (int i = threadIdx.x; i < D * D; i += blockDim.x)
        Us[i] = reinterpret_cast<const C *>(Ug)[i];
    __syncthreads();
    chain_wait();
    // complex64, k = 1: four groups' loads in flight per thread (28 qubits: 787 -> 661
    // us); with more members a group has enough of them (k = 2: 643 us, 684 with two
    // groups), and complex128 is bound by the FP64 pipe
    constexpr int G = sizeof(R) == 4 && K == 1 ? 4 : 1;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x * G;
    for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x * G + threadIdx.x; g < n_groups; g += stride) {
        if constexpr (G == 1) {
            qsd::dense_group<R, K>(psi + group_base<K>(g, t), t, Us);
        } else {
            C *p[G], v[G][D];
#pragma unroll
            for (int i = 0; i < G; i++) {
                p[i] = psi + group_base<K>(min(g + (uint64_t)i * blockDim.x, n_groups - 1), t);
                qsd::dense_load<R, K>(p[i], t, v[i]);
            }
#pragma unroll
            for (int i = 0; i < G; i++)
                if (g + (uint64_t)i * blockDim.x < n_groups) qsd::dense_rows<R, K>(p[i], t, Us, v[i]);
        }
    }
}

// The diagonal sweeps split an index into a column (the kDiagRowBits lowest
// bits, one amplitude of complex128 or two of complex64 per thread), a row of
// its chunk and the bits above the chunk; a thread keeps four rows in flight.
constexpr int kDiagThreads = 256;
constexpr int kDiagAhead = 4;
constexpr int kDiagChunkRows = 32;                                           // most rows of a chunk
template <typename R> constexpr int kDiagVec = sizeof(R) == 4 ? 2 : 1;       // amplitudes per thread and row
template <typename R> constexpr int kDiagRowBits = sizeof(R) == 4 ? 9 : 8;   // log2(kDiagThreads * kDiagVec)

// Table diagonal on up to QS_MAX_DIAG_K qubits: psi_i *= d[x(i)], x(i) the
// column's, the row's and the chunk's target bits OR-ed together, each formed
// once per launch, per launch (shared memory) and per chunk.  complex64 is
// bound by HBM (28 qubits: 837 -> 666 us, 95% of the copy rate, with four rows in
// flight instead of one amplitude and its table look-up); complex128 by the
// FP64 pipe (four operations an amplitude, 883 us at 27 qubits: 1022 -> 983 us).
template <typename R>
__global__ void __launch_bounds__(kDiagThreads, 4)
k_diag(typename cplx<R>::t *__restrict__ psi, int n, int L, int k, const int *__restrict__ qg, const R *__restrict__ dg)
{
    using C = typename cplx<R>::t;
    constexpr int VEC = kDiagVec<R>, RB = kDiagRowBits<R>;
    __shared__ int q[QS_MAX_DIAG_K];
    __shared__ int row_x[kDiagChunkRows];
    const C *d = reinterpret_cast<const C *>(dg);
    const int tid = threadIdx.x;
    chain_start();
    if (tid < k) q[tid] = qg[tid];
    __syncthreads();
    auto bits = [&](uint64_t i) {
        int x = 0;
        for (int j = 0; j < k; j++) x |= (int)((i >> q[j]) & 1) << j;
        return x;
    };
    const int rb = min(n, RB), rows = 1 << (L - rb);
    if (tid < rows) row_x[tid] = bits((uint64_t)tid << rb);
    const uint32_t e = (uint32_t)(VEC * tid);
    const bool in = e < (1u << rb);
    int xe[VEC];
#pragma unroll
    for (int v = 0; v < VEC; v++) xe[v] = bits(e + v);
    __syncthreads();
    chain_wait();
    if (!in) return;
    const uint64_t n_chunks = 1ULL << (n - L);
    for (uint64_t ch = blockIdx.x; ch < n_chunks; ch += gridDim.x) {
        const uint64_t h = ch << L;
        const int xh = bits(h);
        for (int r = 0; r < rows; r += kDiagAhead) {
            C v[kDiagAhead][VEC], m[kDiagAhead][VEC];
#pragma unroll
            for (int j = 0; j < kDiagAhead; j++) {
                if (r + j >= rows) break;
                const C *p = psi + h + ((uint64_t)(r + j) << rb) + e;
                const int x = xh | row_x[r + j];
                if constexpr (VEC == 2) {
                    const float4 w = *reinterpret_cast<const float4 *>(p);
                    v[j][0] = make_float2(w.x, w.y);
                    v[j][1] = make_float2(w.z, w.w);
                } else {
                    v[j][0] = *p;
                }
#pragma unroll
                for (int i = 0; i < VEC; i++) m[j][i] = __ldg(&d[x | xe[i]]);
            }
#pragma unroll
            for (int j = 0; j < kDiagAhead; j++) {
                if (r + j >= rows) break;
                C *p = psi + h + ((uint64_t)(r + j) << rb) + e;
                C o[VEC];
#pragma unroll
                for (int i = 0; i < VEC; i++) {
                    o[i].x = v[j][i].x * m[j][i].x - v[j][i].y * m[j][i].y;
                    o[i].y = v[j][i].x * m[j][i].y + v[j][i].y * m[j][i].x;
                }
                if constexpr (VEC == 2)
                    *reinterpret_cast<float4 *>(p) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                else
                    *p = o[0];
            }
        }
    }
}

// Product of T-type phases and CZ signs (Sec. 2, Sec. 3.5): amplitude i gets
// e^{i pi m(i)/4}, m(i) = sum_q c_q i_q + 4 sum_a i_a popc(i & P_a) mod 8, with
// P_a the CZ partners b > a of qubit a.  The index splits into a column e (the
// kDiagRowBits lowest bits, one or two amplitudes per thread), a row r of the
// chunk and the bits h above the chunk:
//   m(i) = m0(e) + m1(r) + m_hi(h) + 4 popc(r & Mr_h) + 4 popc(e & (X_r ^ Me_h)),
// m0 in a register for the whole launch, (m1, X_r) a table of at most 32 rows
// in shared memory, m_hi(h) and the mask M_h (bits below the chunk's top whose
// partner set meets h an odd number of times) formed once per chunk by each
// warp, its lanes taking one term each.
// Bound by HBM (amplitudes with m = 0 are not touched): four rows are in flight
// per thread.  complex128: the factor e^{i pi/4} costs four FP64 operations and
// the FP64 pipe gives two results a clock per SM, so a warp whose lanes are half
// odd and half even pays for all of them.  m is odd exactly where the odd
// coefficients' bits have odd parity; two rows are therefore paired so that
// exactly one of a thread's two amplitudes is odd (the second row's column with
// its lowest odd bit flipped when the rows' parities agree), and one rotation
// serves both: 2 FP64 operations per amplitude, below the HBM time.  Without an odd
// coefficient on the lanes' bits, rows that differ in an odd row bit are paired, or
// else all lanes and rows of a step are alike and the odd steps alone reach the FP64
// pipe (27 qubits, one T gate on qubits 5 to 12 or 26: 1020 to 1070 -> 550 to 580 us).
// 27 qubits complex128, T-type and CZ terms: 1139 -> 680 us (94% of the HBM copy
// rate); 28 qubits complex64: 996 -> 680 us; a phase op on 14 qubits: 53 -> 4 us
// (chunks used to be 2^14 amplitudes with a table entry each, built by every
// CTA; 83 gates on 16 qubits, half of them CZs: 1.79 -> 0.40 ms).
template <typename R>
__global__ void __launch_bounds__(kDiagThreads, 4)
k_phase(typename cplx<R>::t *__restrict__ psi, int n, int L, const qs_phase_dev *__restrict__ ph, int n_act)
{
    using C = typename cplx<R>::t;
    constexpr int VEC = kDiagVec<R>, RB = kDiagRowBits<R>;
    __shared__ uint64_t part[64];
    __shared__ int act[64];
    __shared__ uint32_t row_x[kDiagChunkRows];
    __shared__ uint8_t row_m[kDiagChunkRows];
    chain_start();
    const uint64_t cm[3] = {ph->cmask[0], ph->cmask[1], ph->cmask[2]};
    const qs_phase_term *terms = reinterpret_cast<const qs_phase_term *>(ph + 1);
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < n_act; i += kDiagThreads) {
        part[i] = terms[i].partners;
        act[i] = terms[i].a;
    }
    __syncthreads();
    const int rb = min(n, RB);                       // a state below a row: its own bits
    const int rows = 1 << (L - rb);
    if (tid < rows) {
        const uint64_t r = (uint64_t)tid << rb;
        uint32_t x = 0;
        for (int t = 0; t < n_act && act[t] < rb; t++) x |= ((uint32_t)__popcll(r & part[t]) & 1u) << act[t];
        row_x[tid] = x;
        row_m[tid] = qsd::phase_low(r, cm, act, part, n_act, L);
    }
    const uint32_t e = (uint32_t)(VEC * tid);
    int m0[VEC];
#pragma unroll
    for (int v = 0; v < VEC; v++) m0[v] = qsd::phase_low(e + v, cm, act, part, n_act, rb);
    // complex128: the lowest odd coefficient among the lanes' bits, and the
    // column with that bit flipped
    const uint32_t odd = VEC == 1 ? (uint32_t)cm[0] & 31u : 0u;
    const uint32_t e2 = e ^ (odd & (0u - odd));
    const int m02 = odd ? qsd::phase_low(e2, cm, act, part, n_act, rb) : 0;
    const bool in = e < (1u << rb);
    const bool any_odd = cm[0] != 0;
    // (no such bit, but one of the two lowest row bits: rows that differ in it are paired as they are)
    const uint32_t odd_row = VEC == 1 && odd == 0 ? (uint32_t)(cm[0] >> rb) & (uint32_t)(rows - 1) & 3u : 0u;
    const bool pairs = (odd | odd_row) != 0 && rows > 1 && rb == RB, two_apart = odd_row == 2u;
    __syncthreads();
    chain_wait();
    const uint64_t n_chunks = 1ULL << (n - L);
    // no factor on a chunk's own bits alone: chunks that none of the others reach are passed over
    // (complex128, 27 qubits, T on qubit 26 608 -> 555 us, CZ on 25 and 26 307 -> 184)
    const uint64_t own = (1ULL << L) - 1ULL;
    uint64_t low = (cm[0] | cm[1] | cm[2]) & own;
    for (int t = lane; t < n_act; t += 32)
        if (act[t] < L) low |= part[t] & own;
    const bool flat = !__any_sync(0xffffffffu, low != 0);
    constexpr int kAhead = kDiagAhead;
    for (uint64_t ch = blockIdx.x; ch < n_chunks; ch += gridDim.x) {
        const uint64_t h = ch << L;
        uint32_t Mh = 0, parh = 0;
        for (int t = lane; t < n_act; t += 32) {
            const int a = act[t];
            const uint32_t o = (uint32_t)__popcll(h & part[t]) & 1u;
            if (a >= L) parh ^= (uint32_t)(h >> a) & o;
            else Mh |= o << a;
        }
        Mh = __reduce_or_sync(0xffffffffu, Mh);
        parh = __reduce_xor_sync(0xffffffffu, parh & 1u);
        const int mh = __popcll(h & cm[0]) + 2 * __popcll(h & cm[1]) + 4 * (__popcll(h & cm[2]) + (int)parh);
        const uint32_t Me = Mh & ((1u << rb) - 1u), Mr = Mh >> rb;
        if (!in || (flat && Mh == 0 && (mh & 7) == 0)) continue;
        for (int r = 0; r < rows; r += kAhead) {
            int m[kAhead][VEC];
            C v[kAhead][VEC];
            C *p[kAhead];
#pragma unroll
            for (int j = 0; j < kAhead; j++) {
                const int rj = r + (two_apart ? (j & 1) << 1 | j >> 1 : j);
                const bool ok = rj < rows;
                const int mr = ok ? row_m[rj] + mh + 4 * __popc((uint32_t)rj & Mr) : 0;
                const uint32_t X = ok ? row_x[rj] ^ Me : 0u;
                // the second row of a pair: the column that makes exactly one of the two odd
                bool other = false;
                if (pairs && (j & 1)) other = ok && !((mr ^ m[j - 1][0] ^ m0[0]) & 1);
                const uint32_t ej = other ? e2 : e;
                p[j] = psi + h + ((uint64_t)rj << rb) + ej;
#pragma unroll
                for (int k = 0; k < VEC; k++)
                    m[j][k] = ok ? ((other ? m02 : m0[k]) + mr + 4 * __popc((ej + k) & X)) & 7 : 0;
            }
#pragma unroll
            for (int j = 0; j < kAhead; j++) {
                if constexpr (VEC == 2) {
                    if (m[j][0] | m[j][1]) {
                        const float4 w = *reinterpret_cast<const float4 *>(p[j]);
                        v[j][0] = make_float2(w.x, w.y);
                        v[j][1] = make_float2(w.z, w.w);
                    }
                } else {
                    v[j][0] = C{};
                    if (m[j][0]) v[j][0] = *p[j];
                }
            }
            if (pairs) {
#pragma unroll
                for (int j = 0; j < kAhead; j += 2) {
                    const bool first = m[j][0] & 1;
                    const C t = qsd::eighth_turn(first ? v[j][0] : v[j + 1][0]);
                    if (first) v[j][0] = t;
                    else v[j + 1][0] = t;
                }
            } else if (any_odd) {
                // one branch around all rows: the compiler turns a branch around one row's four
                // FP64 instructions into predicates, and the FP64 pipe takes those too
                int o = VEC == 2;
#pragma unroll
                for (int j = 0; j < kAhead; j++)
#pragma unroll
                    for (int k = 0; k < VEC; k++) o |= m[j][k];
                if (o & 1) {
#pragma unroll
                    for (int j = 0; j < kAhead; j++)
#pragma unroll
                        for (int k = 0; k < VEC; k++)
                            if (m[j][k] & 1) v[j][k] = qsd::eighth_turn(v[j][k]);
                }
            }
#pragma unroll
            for (int j = 0; j < kAhead; j++) {
#pragma unroll
                for (int k = 0; k < VEC; k++) {
                    v[j][k] = qsd::quarter_turns<C>(v[j][k], m[j][k] >> 1);
                }
                if constexpr (VEC == 2) {
                    if (m[j][0] | m[j][1])
                        *reinterpret_cast<float4 *>(p[j]) = make_float4(v[j][0].x, v[j][0].y, v[j][1].x, v[j][1].y);
                } else {
                    if (m[j][0]) *p[j] = v[j][0];
                }
            }
        }
    }
}

int grid_for(uint64_t work, int block, int per_sm)
{
    uint64_t want = (work + block - 1) / block;
    uint64_t cap = (uint64_t)sm_count() * per_sm;
    if (want < 1) want = 1;
    return (int)std::min<uint64_t>(want, cap);
}

template <typename R, int K>
int launch_dense_t(qs_state *s, const int *q, const void *U)
{
    Targets t;
    for (int j = 0; j < K; j++) t.q[j] = q[j];
    uint64_t groups = 1ULL << (s->n - K);
    const int block = 128;
    int grid = grid_for(groups, block, 8);
    // An SM holds up to 16 of these blocks.  Started early they pile up on the SMs that are
    // free first, which costs more than the start gains unless the sweep is little more
    // than a launch.  Three table diagonals and three clusters in turn, us, early start and
    // not: complex128 k = 3, 14 qubits 39, 45; 16 qubits 201, 45; 27 qubits k = 1 13.9,
    // 8.6 ms.  complex64 k = 1, 20 qubits 22, 29; k = 4, 16 qubits 20, 24, 18 qubits 38, 27.
    const bool chain = s->chain && s->n <= (sizeof(R) == 8 ? 14 : K <= 2 ? 20 : 16);
    const cudaError_t e = launch_sweep(s, chain, k_dense<R, K>, grid, block, 0, reinterpret_cast<typename cplx<R>::t *>(s->amp),
                                       groups, t, reinterpret_cast<const R *>(U));
    return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "k_dense launch: %s", cudaGetErrorString(e));
}

template <typename R>
int launch_dense_r(qs_state *s, const int *q, int k, const void *U)
{
    switch (k) {
    case 1: return launch_dense_t<R, 1>(s, q, U);
    case 2: return launch_dense_t<R, 2>(s, q, U);
    case 3: return launch_dense_t<R, 3>(s, q, U);
    case 4: return launch_dense_t<R, 4>(s, q, U);
    case 5: return launch_dense_t<R, 5>(s, q, U);
    default: return qs_fail(QS_EINVAL, "dense cluster of %d qubits", k);
    }
}

}  // namespace

// complex64: clusters of 4 and 5 qubits (a 4-qubit cluster embedded in 5 on
// the tensor cores measured 11.3 ms at 32 qubits against 16.1 ms for the FP32
// CUDA-core sweep, which is FMA-bound there); complex128: every cluster of 2 or
// more qubits (native FP64 runs at 1/58 of the FP32 rate).  Tensor-core sweeps
// need n >= 5.
bool qs_tc_wanted(int dtype, int k, int n)
{
    if (n < 5) return false;
    return dtype == QS_C64 ? k >= 4 : k >= 2;
}

int qs_launch_dense(qs_state *s, const int *sorted_qubits, int k, const void *dev_matrix,
                    const void *dev_tc)
{
    s->perm_invariant = false;
    if (k == 5 && dev_tc) return qs_launch_dense5_tc(s, sorted_qubits, dev_tc, ~0ULL);
    int rc = qs_materialize(s);   // the CUDA-core sweeps read every amplitude
    if (rc) return rc;
    return s->dtype == QS_C128 ? launch_dense_r<double>(s, sorted_qubits, k, dev_matrix)
                               : launch_dense_r<float>(s, sorted_qubits, k, dev_matrix);
}

// Chunk bits of a diagonal sweep: up to 32 rows, fewer (8) where a block would get less
// than four chunks, 4 where less than two, and fewer still where the chunks would not
// fill the GPU (complex128 table, 23 qubits: 79 us with 1.7 chunks a block, 72 so; a
// chunk of few rows costs a phase op its terms: complex64, 23 qubits, 25.3 us with 4 rows,
// 22.8 with 8).
// *grid: its blocks.  Their number is odd where blocks take several chunks: a block's
// chunks then differ in every bit of their number.  (With an even one the blocks split
// by the lowest bit, and one T gate or CZ on that qubit left half of them without
// work: complex128, 27 qubits, T on qubit 13 1080 us, 567 so.)
template <typename R>
static int diag_chunk(int n, int *grid)
{
    const int rb = std::min(n, kDiagRowBits<R>);
    const uint64_t cap = (uint64_t)sm_count() * 4;
    int L = std::min(n, rb + 5);
    while (L > rb && (1ULL << (n - L)) < (L > rb + 3 ? 4 : L > rb + 2 ? 2 : 1) * cap) L--;
    *grid = (int)std::min<uint64_t>(1ULL << (n - L), (cap - 1) | 1);
    return L;
}

template <typename R>
static cudaError_t launch_diag_r(qs_state *s, const int *dev_qubits, int k, const void *dev_table)
{
    int grid;
    const int L = diag_chunk<R>(s->n, &grid);
    return launch_sweep(s, s->chain, k_diag<R>, grid, kDiagThreads, 0, reinterpret_cast<typename cplx<R>::t *>(s->amp), s->n, L, k,
                        dev_qubits, reinterpret_cast<const R *>(dev_table));
}

template <typename R>
static cudaError_t launch_phase_r(qs_state *s, const void *dev_phase, int n_act)
{
    int grid;
    const int L = diag_chunk<R>(s->n, &grid);
    // (complex128 states beyond L2 lose by an early start after a tensor-core sweep: 27 qubits,
    // three of each in turn, 5.47 ms, without 5.18)
    return launch_sweep(s, s->chain && (sizeof(R) == 4 || s->n <= 23), k_phase<R>, grid, kDiagThreads, 0, reinterpret_cast<typename cplx<R>::t *>(s->amp), s->n, L,
                        (const qs_phase_dev *)dev_phase, n_act);
}

int qs_launch_diag(qs_state *s, const int *dev_qubits, int k, const void *dev_table)
{
    s->perm_invariant = false;
    int rc = qs_materialize(s);
    if (rc) return rc;
    const cudaError_t e = s->dtype == QS_C128 ? launch_diag_r<double>(s, dev_qubits, k, dev_table)
                                              : launch_diag_r<float>(s, dev_qubits, k, dev_table);
    return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "k_diag launch: %s", cudaGetErrorString(e));
}

int qs_launch_phase(qs_state *s, const void *dev_phase, int n_act)
{
    s->perm_invariant = false;
    int rc = qs_materialize(s);
    if (rc) return rc;
    const cudaError_t e = s->dtype == QS_C128 ? launch_phase_r<double>(s, dev_phase, n_act)
                                              : launch_phase_r<float>(s, dev_phase, n_act);
    return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "k_phase launch: %s", cudaGetErrorString(e));
}

// ------------------------------------------------------------------ host side

namespace {

// Sorted copy of (qubits, matrix): ascending qubit order, the matrix permuted so
// that bit j of its index belongs to the j-th smallest qubit (Sec. 3.2).
void sort_targets(const int *qubits, int k, const double *U, bool dense, int *qs_out,
                  std::vector<double> &M)
{
    int perm[QS_MAX_DIAG_K];
    for (int j = 0; j < k; j++) perm[j] = j;
    std::sort(perm, perm + k, [&](int a, int b) { return qubits[a] < qubits[b]; });
    for (int j = 0; j < k; j++) qs_out[j] = qubits[perm[j]];
    auto remap = [&](int xn) {
        int xo = 0;
        for (int j = 0; j < k; j++) xo |= ((xn >> j) & 1) << perm[j];
        return xo;
    };
    const int d = 1 << k;
    if (dense) {
        M.resize(2 * d * d);
        for (int r = 0; r < d; r++)
            for (int c = 0; c < d; c++) {
                int ro = remap(r), co = remap(c);
                M[2 * (r * d + c)] = U[2 * (ro * d + co)];
                M[2 * (r * d + c) + 1] = U[2 * (ro * d + co) + 1];
            }
    } else {
        M.resize(2 * d);
        for (int x = 0; x < d; x++) {
            M[2 * x] = U[2 * remap(x)];
            M[2 * x + 1] = U[2 * remap(x) + 1];
        }
    }
}

// Pack FP64 values into the state's real type.
std::vector<uint8_t> to_real(const std::vector<double> &v, int dtype)
{
    std::vector<uint8_t> out;
    if (dtype == QS_C128) {
        out.resize(v.size() * sizeof(double));
        std::memcpy(out.data(), v.data(), out.size());
    } else {
        out.resize(v.size() * sizeof(float));
        float *f = reinterpret_cast<float *>(out.data());
        for (size_t i = 0; i < v.size(); i++) f[i] = (float)v[i];
    }
    return out;
}


int check_state(qs_state *s, const char *who)
{
    if (!s || !s->amp) return qs_fail(QS_EINVAL, "%s: null state", who);
    return QS_OK;
}

// Stage a small operand block in the state's scratch (stream-ordered: the copy
// runs after earlier kernels on the stream have finished reading the slot).
int stage(qs_state *s, const void *host, size_t bytes, void **dev)
{
    void *p = nullptr;
    int rc = qs_state_scratch(s, bytes, &p);
    if (rc) return rc;
    cudaError_t e = cudaMemcpyAsync(p, host, bytes, cudaMemcpyHostToDevice, (cudaStream_t)s->stream);
    if (e != cudaSuccess) return qs_fail(QS_ECUDA, "operand copy: %s", cudaGetErrorString(e));
    *dev = p;
    return QS_OK;
}

int check_qubits(qs_state *s, const int *qubits, int k, int kmax, const char *who)
{
    if (!qubits || k < 1 || k > kmax || k > s->n)
        return qs_fail(QS_EINVAL, "%s: k = %d not in [1, %d] or above n", who, k, kmax);
    uint64_t seen = 0;
    for (int j = 0; j < k; j++) {
        if (qubits[j] < 0 || qubits[j] >= s->n)
            return qs_fail(QS_EINVAL, "%s: qubit %d out of range", who, qubits[j]);
        if ((seen >> qubits[j]) & 1) return qs_fail(QS_EINVAL, "%s: qubit %d repeated", who, qubits[j]);
        seen |= 1ULL << qubits[j];
    }
    return QS_OK;
}

// Which dense clusters go to the tensor cores (qs_tc_wanted): complex64 clusters
// of 4 and 5 qubits, complex128 clusters of 2 or more; smaller ones are
// embedded in 5 qubits.
bool tc_wanted(int dtype, int k, int n) { return qs_tc_wanted(dtype, k, n); }

// U (x) 1: a k-qubit cluster (sorted qubits q, sorted matrix M) as a 5-qubit
// one on q plus the highest qubits not in q; output sorted as well.
void embed5(const int *q, int k, const std::vector<double> &M, int n, std::array<int, 5> &q5,
            std::vector<double> &M5)
{
    uint64_t used = 0;
    for (int j = 0; j < k; j++) used |= 1ULL << q[j];
    // pad with the highest free qubits: low qubits as targets would make the
    // tile gather touch one amplitude per group instead of runs of groups
    uint64_t all = used;
    for (int b = n - 1; b >= 0 && __builtin_popcountll(all) < 5; b--) all |= 1ULL << b;
    int pos[5], j5 = 0;
    for (int b = 0; b < n; b++)
        if ((all >> b) & 1) q5[j5++] = b;
    // position of each original target within q5
    for (int j = 0; j < k; j++)
        for (int i = 0; i < 5; i++)
            if (q5[i] == q[j]) pos[j] = i;
    uint32_t extra = 0;
    for (int i = 0; i < 5; i++)
        if (!((used >> q5[i]) & 1)) extra |= 1u << i;
    const int d = 1 << k;
    M5.assign(2 * 32 * 32, 0.0);
    for (int r5 = 0; r5 < 32; r5++)
        for (int c5 = 0; c5 < 32; c5++) {
            if ((r5 & extra) != (c5 & extra)) continue;
            int r = 0, c = 0;
            for (int j = 0; j < k; j++) {
                r |= ((r5 >> pos[j]) & 1) << j;
                c |= ((c5 >> pos[j]) & 1) << j;
            }
            M5[2 * (r5 * 32 + c5)] = M[2 * (r * d + c)];
            M5[2 * (r5 * 32 + c5) + 1] = M[2 * (r * d + c) + 1];
        }
}

std::vector<uint8_t> tc_pack_for(int dtype, const std::vector<double> &M5)
{
    return dtype == QS_C64 ? qs_pack_tc_c64(M5) : qs_pack_tc_c128(M5);
}

// Fold of phase op ph into the tensor-core sweep on the sorted qubits q5 with
// matrix M5 (qs_post_phase): M5f = D M5, D the diagonal of the phase terms on
// q5 (coefficients and CZ pairs with both ends in q5, Sec. 2), and desc the
// rest: CZ pairs with one or no end in q5 and the coefficients off q5, which
// act on each group as a conditional Z on a target or a phase of the group
// (Sec. 3.5).  False when a coefficient off q5 is odd (its factor is not a
// power of i) or there are more CZ terms off q5 than the kernel holds.
bool fold_phase(int n, const std::array<int, 5> &q5, const std::vector<double> &M5, const qs_op_host &ph,
                std::vector<double> &M5f, std::vector<uint8_t> &desc)
{
    int pos[64];
    std::fill(pos, pos + 64, -1);
    for (int j = 0; j < 5; j++) pos[q5[j]] = j;
    qs_post_phase hdr;
    std::memset(&hdr, 0, sizeof(hdr));
    int cq[5] = {0, 0, 0, 0, 0};        // coefficient of qubit q5[j]
    for (int q = 0; q < n; q++) {
        const int c = ((ph.coeff[q] % 8) + 8) % 8;
        if (pos[q] >= 0) {
            cq[pos[q]] = c;
        } else {
            if (c & 1) return false;
            if (c & 2) hdr.c1 |= 1ULL << q;
            if (c & 4) hdr.c2 |= 1ULL << q;
        }
    }
    uint32_t inner[5] = {0, 0, 0, 0, 0};   // bit j' of inner[j]: CZ (q5[j], q5[j']), j < j', mod 2
    std::vector<uint64_t> partners(n, 0);
    for (const auto &e : ph.edges) {
        const int a = std::min(e.first, e.second), b = std::max(e.first, e.second);
        const int ja = pos[a], jb = pos[b];
        if (ja >= 0 && jb >= 0) inner[ja] ^= 1u << jb;
        else if (ja >= 0) hdr.tp[ja] ^= 1ULL << b;
        else if (jb >= 0) hdr.tp[jb] ^= 1ULL << a;
        else partners[a] ^= 1ULL << b;
    }
    std::vector<qs_phase_term> terms;
    for (int a = 0; a < n; a++)
        if (partners[a]) terms.push_back({partners[a], a, 0});
    if ((int)terms.size() > QS_MAX_POST_TERMS) return false;
    hdr.n_terms = (int32_t)terms.size();
    // row m of M5 times w^{s(m)}, w = e^{i pi / 4}: exact for even s
    const double r = std::sqrt(0.5);
    const double wr[8] = {1, r, 0, -r, -1, -r, 0, r}, wi[8] = {0, r, 1, r, 0, -r, -1, -r};
    M5f.assign(M5.size(), 0.0);
    for (int m = 0; m < 32; m++) {
        int sm = 0;
        for (int j = 0; j < 5; j++)
            if ((m >> j) & 1) sm += cq[j] + 4 * __builtin_popcount(inner[j] & (uint32_t)m);
        sm &= 7;
        for (int x = 0; x < 32; x++) {
            const double a = M5[2 * (m * 32 + x)], b = M5[2 * (m * 32 + x) + 1];
            M5f[2 * (m * 32 + x)] = a * wr[sm] - b * wi[sm];
            M5f[2 * (m * 32 + x) + 1] = a * wi[sm] + b * wr[sm];
        }
    }
    desc.resize(sizeof(hdr) + terms.size() * sizeof(qs_phase_term));
    std::memcpy(desc.data(), &hdr, sizeof(hdr));
    if (!terms.empty()) std::memcpy(desc.data() + sizeof(hdr), terms.data(), terms.size() * sizeof(qs_phase_term));
    return true;
}

// Append bytes to an op's data at a 256-byte boundary; returns their offset.
size_t append_aligned(std::vector<uint8_t> &part, const std::vector<uint8_t> &bytes)
{
    const size_t at = (part.size() + 255) & ~(size_t)255;
    part.resize(at + bytes.size());
    std::memcpy(part.data() + at, bytes.data(), bytes.size());
    return at;
}

// Device image of a schedule for one dtype: every op's data, 256-byte aligned.
std::vector<uint8_t> schedule_blob(const qs_schedule *sc, int dtype, qs_dev_sched &d)
{
    std::vector<uint8_t> blob;
    const size_t nops = sc->ops.size();
    std::vector<size_t> &offset = d.offset, &tc_off = d.tc_off;
    std::vector<std::array<int, 5>> &tc_q = d.tc_q;
    offset.assign(nops, 0);
    d.n_act.assign(nops, 0);
    tc_off.assign(nops, 0);
    d.fold_off.assign(nops, 0);
    d.post_off.assign(nops, 0);
    tc_q.assign(nops, std::array<int, 5>{{0, 0, 0, 0, 0}});
    std::vector<int> &n_act = d.n_act;
    for (size_t i = 0; i < sc->ops.size(); i++) {
        const qs_op_host &op = sc->ops[i];
        std::vector<uint8_t> part;
        if (op.kind == QS_OP_PHASE) {
            part = qs_pack_phase(sc->n, op.coeff, op.edges, &n_act[i]);
        } else if (op.kind == QS_OP_DIAG) {
            std::vector<uint8_t> tab = to_real(op.matrix, dtype);
            part.resize(64 + tab.size());
            std::memcpy(part.data(), op.qubits, sizeof(int) * op.k);
            std::memcpy(part.data() + 64, tab.data(), tab.size());
        } else {
            part = to_real(op.matrix, dtype);
            if (sc->n >= 5) {   // tensor-core operands for every dense op (any path may run it)
                std::vector<double> M5;
                if (op.k == 5) {
                    for (int j = 0; j < 5; j++) tc_q[i][j] = op.qubits[j];
                    M5 = op.matrix;
                } else {
                    embed5(op.qubits, op.k, op.matrix, sc->n, tc_q[i], M5);
                }
                tc_off[i] = append_aligned(part, tc_pack_for(dtype, M5));
                // a phase op right after it can run inside its sweep
                std::vector<double> M5f;
                std::vector<uint8_t> desc;
                if (i + 1 < nops && sc->ops[i + 1].kind == QS_OP_PHASE &&
                    fold_phase(sc->n, tc_q[i], M5, sc->ops[i + 1], M5f, desc)) {
                    d.fold_off[i] = append_aligned(part, tc_pack_for(dtype, M5f));
                    d.post_off[i] = append_aligned(part, desc);
                }
            }
        }
        size_t at = (blob.size() + 255) & ~(size_t)255;
        blob.resize(at + part.size());
        std::memcpy(blob.data() + at, part.data(), part.size());
        offset[i] = at;
    }
    if (blob.empty()) blob.resize(256);
    return blob;
}

int ensure_dev_schedule(qs_state *s, const qs_schedule *csc)
{
    qs_schedule *sc = const_cast<qs_schedule *>(csc);
    qs_dev_sched &d = sc->dev[s->dtype];
    int dev = 0;
    cudaGetDevice(&dev);
    if (d.pool && d.device == dev) return QS_OK;
    if (d.pool) {
        cudaFree(d.pool);
        d.pool = nullptr;
    }
    std::vector<uint8_t> blob = schedule_blob(sc, s->dtype, d);
    cudaError_t e = cudaMalloc(&d.pool, blob.size());
    if (e != cudaSuccess) {
        d.pool = nullptr;
        return qs_fail(QS_ENOMEM, "schedule upload: %s", cudaGetErrorString(e));
    }
    // copied on a stream of its own that waits for nothing, so an upload made
    // ahead of time does not wait for kernels running on other streams
    cudaStream_t cs = nullptr;
    e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d.pool, blob.data(), blob.size(), cudaMemcpyHostToDevice, cs);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
    if (cs) cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
        cudaFree(d.pool);
        d.pool = nullptr;
        return qs_fail(QS_ECUDA, "schedule upload: %s", cudaGetErrorString(e));
    }
    d.bytes = blob.size();
    d.device = dev;
    return QS_OK;
}

// Kernel path of a dense op: the state's setting if not AUTO, else the op's
// planned path if any, else the default policy.  *folded: the phase op after
// it ran inside its tensor-core sweep.
int path_of(const qs_state *s, const qs_op_host &op)
{
    return s->path != QS_PATH_AUTO ? s->path
           : op.path != QS_PATH_AUTO ? op.path
           : (tc_wanted(s->dtype, op.k, s->n) ? QS_PATH_TENSOR : QS_PATH_CUDA_CORES);
}

// Dense ops i and i + 1 as one sweep (qs_pair.cu) when both run on the tensor
// cores and their target qubits fit one super-group; *skip = the ops after i
// that ran inside it (the second cluster, and a phase op folded into it).
bool try_pair(qs_state *s, const qs_schedule *sc, const qs_dev_sched &d, size_t i, int *rc, int *skip)
{
    if (!s->pair_sweeps || s->dtype != QS_C64 || i + 1 >= sc->ops.size()) return false;
    const qs_op_host &a = sc->ops[i], &b = sc->ops[i + 1];
    if (a.kind != QS_OP_DENSE || b.kind != QS_OP_DENSE || !d.tc_off[i] || !d.tc_off[i + 1]) return false;
    if (path_of(s, a) != QS_PATH_TENSOR || path_of(s, b) != QS_PATH_TENSOR) return false;
    if (!qs_pair_possible(s, d.tc_q[i].data(), d.tc_q[i + 1].data())) return false;
    const uint8_t *da = (const uint8_t *)d.pool + d.offset[i], *db = (const uint8_t *)d.pool + d.offset[i + 1];
    const bool fold = s->fold_phase && d.fold_off[i + 1];
    *rc = qs_launch_pair5_tc(s, d.tc_q[i].data(), da + d.tc_off[i], d.tc_q[i + 1].data(),
                             db + (fold ? d.fold_off[i + 1] : d.tc_off[i + 1]), fold ? db + d.post_off[i + 1] : nullptr);
    *skip = fold ? 2 : 1;
    return true;
}

int launch_op_dense(qs_state *s, const qs_dev_sched &d, size_t i, const qs_op_host &op, const uint8_t *data,
                    bool *folded)
{
    *folded = false;
    int path = path_of(s, op);
    if (path == QS_PATH_TENSOR && d.tc_off[i]) {
        uint64_t grow = 0;
        for (int j = 0; j < op.k; j++) grow |= 1ULL << op.qubits[j];
        if (s->fold_phase && d.fold_off[i]) {
            *folded = true;
            return qs_launch_dense5_tc(s, d.tc_q[i].data(), data + d.fold_off[i], grow, data + d.post_off[i]);
        }
        return qs_launch_dense5_tc(s, d.tc_q[i].data(), data + d.tc_off[i], grow);
    }
    return qs_launch_dense(s, op.qubits, op.k, data, nullptr);
}

// Whether a pass is faster than its ops as one sweep each.  Up to 4 MB of state always (every
// sweep is a launch there).  Above, a pass pays for its own read and write of the state
// and its row tables, and saves per op, in microseconds with M = 2^20 amplitudes (fitted to
// runs of 2, 3 and 4 equal ops, complex64 20 to 28 and complex128 19 to 27 qubits):
//   complex64   pass 5 + 3.4 M; a dense op saves 3 + 1.6 M, one factor of a phase op
//               2.2 + (2.2 f - 0.1) M, a longer phase op 2 - M
//   complex128  pass 3 + 10.4 M; a dense op saves 1 (it is bound by the FP64 pipe either
//               way), a T gate 3 + 0.3 M, another factor 3.5 + (4.5 f - 0.6) M, a longer
//               phase op 2 - 2.5 M
// where f is the part of the state that the factor's sweep touches (bits below a 64-byte
// piece save nothing), and a state in L2 has sweeps of half the traffic's time.  24 qubits
// complex128: two phase ops of 24 terms 183 us as sweeps, 462 as a pass, two CZs on high
// qubits 37 and 194; 27 qubits complex64: four CZs on low qubits 1366 and 640, two phase
// ops 686 and 1275.  Circuits gate by gate are passes at every size.
bool pass_pays(const qs_state *s, const qs_pass &p)
{
    const bool c64 = s->dtype == QS_C64;
    const double bytes = (c64 ? 8.0 : 16.0) * std::ldexp(1.0, s->n), M = std::ldexp(1.0, s->n - 20);
    if (bytes <= (4 << 20)) return true;
    const double l2 = bytes <= (96 << 20) ? 0.5 : 1.0;
    double gain = 0;
    for (int i = 0; i < p.n_ops; i++) {
        const qs_pass_op &op = p.op[i];
        if (op.kind == QS_OP_DENSE) {
            gain += c64 ? 3 + 1.6 * l2 * M : 1;
        } else if (op.kind == QS_OP_PHASE) {
            gain += c64 ? 2 - M : 2 - 2.5 * M;
        } else {
            // the factor's index bits: op.data outside the chunk, op.q among its local bits
            double f = std::ldexp(1.0, -__builtin_popcountll(op.data));
            for (int j = 0; j < op.k; j++)
                if (op.q[j] >= (c64 ? 3 : 2)) f /= 2;   // (the lowest local bits are the lowest index bits)
            gain += c64 ? 2.2 + (2.2 * f - 0.1) * l2 * M : op.n_act & 1 ? 3 + 0.3 * M : 3.5 + (4.5 * f - 0.6) * l2 * M;
        }
    }
    return gain > (c64 ? 5 + 3.4 * M : 3 + 10.4 * M);
}

// Ops i, i + 1, ... that run on the CUDA cores as passes (qs_pass.cu), *done of
// them: two or more ops per read and write of the state, a pass of one op, or one
// that does not pay, as sweeps.  A chunk has 2^(n-7) amplitudes, within the kernel's
// 2^8 .. 2^13 (complex64) or 2^12: 128 chunks at least, a CTA each, so a small state
// still fills the GPU.
int run_passes(qs_state *s, const qs_schedule *sc, const qs_dev_sched &d, size_t i, size_t *done)
{
    *done = 0;
    std::vector<qs_pass_in> in;
    for (size_t j = i; j < sc->ops.size(); j++) {
        const qs_op_host &op = sc->ops[j];
        if (op.kind == QS_OP_DIAG || (op.kind == QS_OP_DENSE && path_of(s, op) == QS_PATH_TENSOR && d.tc_off[j])) break;
        const size_t bytes = op.kind == QS_OP_DENSE
                                 ? op.matrix.size() * (s->dtype == QS_C128 ? sizeof(double) : sizeof(float))
                                 : sizeof(qs_phase_dev) + sizeof(qs_phase_term) * (size_t)d.n_act[j];
        in.push_back({op.kind, op.k, d.n_act[j], op.qubits, (uint64_t)(uintptr_t)d.pool + d.offset[j], (uint32_t)bytes,
                      &op});
    }
    if (in.size() < 2) return QS_OK;
    const int wmax = std::max(8, std::min(qs_pass_bits(s->dtype), s->n - 7));
    for (const qs_pass &p : qs_plan_passes(s->n, s->dtype, wmax, in, false)) {
        if (p.n_ops > 1 && pass_pays(s, p)) {
            if (int rc = qs_launch_pass(s, p)) return rc;
            s->chain = !s->pair_sweeps;
            continue;
        }
        for (int j = p.first_op; j < p.first_op + p.n_ops; j++) {
            const qs_pass_in &op = in[j];
            const void *data = (const void *)(uintptr_t)op.data;
            if (int rc = op.kind == QS_OP_DENSE ? qs_launch_dense(s, op.qubits, op.k, data, nullptr)
                                                : qs_launch_phase(s, data, op.n_act))
                return rc;
            s->chain = !s->pair_sweeps;
        }
    }
    *done = in.size();
    return QS_OK;
}

}  // namespace

extern "C" int qs_apply_cluster(qs_state *s, const int *qubits, int k, const double *U)
{
    return qs_guard([&]() -> int {
        int rc = check_state(s, "qs_apply_cluster");
        if (rc) return rc;
        if ((rc = check_qubits(s, qubits, k, QS_MAX_K, "qs_apply_cluster"))) return rc;
        if (!U) return qs_fail(QS_EINVAL, "qs_apply_cluster: null matrix");
        int lq[QS_MAX_K], q[QS_MAX_K];
        for (int j = 0; j < k; j++) lq[j] = qs_loc(s, qubits[j]);   // the qubits' index bits
        std::vector<double> M;
        sort_targets(lq, k, U, true, q, M);
        const bool tc = s->path == QS_PATH_TENSOR ? s->n >= 5
                                                  : s->path == QS_PATH_AUTO && tc_wanted(s->dtype, k, s->n);
        if (tc) {
            std::array<int, 5> q5;
            std::vector<double> M5;
            if (k == 5) {
                for (int j = 0; j < 5; j++) q5[j] = q[j];
                M5 = M;
            } else {
                embed5(q, k, M, s->n, q5, M5);
            }
            std::vector<uint8_t> p = tc_pack_for(s->dtype, M5);
            void *dp = nullptr;
            if ((rc = stage(s, p.data(), p.size(), &dp))) return rc;
            uint64_t grow = 0;
            for (int j = 0; j < k; j++) grow |= 1ULL << q[j];
            return qs_launch_dense5_tc(s, q5.data(), dp, grow);
        }
        std::vector<uint8_t> packed = to_real(M, s->dtype);
        void *dU = nullptr;
        if ((rc = stage(s, packed.data(), packed.size(), &dU))) return rc;
        return qs_launch_dense(s, q, k, dU, nullptr);
    });
}

extern "C" int qs_apply_diag(qs_state *s, const int *qubits, int k, const double *d)
{
    return qs_guard([&]() -> int {
        int rc = check_state(s, "qs_apply_diag");
        if (rc) return rc;
        if ((rc = check_qubits(s, qubits, k, QS_MAX_DIAG_K, "qs_apply_diag"))) return rc;
        if (!d) return qs_fail(QS_EINVAL, "qs_apply_diag: null table");
        int lq[QS_MAX_DIAG_K], q[QS_MAX_DIAG_K];
        for (int j = 0; j < k; j++) lq[j] = qs_loc(s, qubits[j]);   // the qubits' index bits
        std::vector<double> M;
        sort_targets(lq, k, d, false, q, M);
        std::vector<uint8_t> tab = to_real(M, s->dtype);
        std::vector<uint8_t> blob(64 + tab.size());
        std::memcpy(blob.data(), q, sizeof(int) * k);
        std::memcpy(blob.data() + 64, tab.data(), tab.size());
        void *dev = nullptr;
        if ((rc = stage(s, blob.data(), blob.size(), &dev))) return rc;
        return qs_launch_diag(s, (const int *)dev, k, (const uint8_t *)dev + 64);
    });
}

extern "C" int qs_apply_phase(qs_state *s, const int *coeff, int n_edges, const int *edges)
{
    return qs_guard([&]() -> int {
        int rc = check_state(s, "qs_apply_phase");
        if (rc) return rc;
        if (!coeff || n_edges < 0 || (n_edges > 0 && !edges))
            return qs_fail(QS_EINVAL, "qs_apply_phase: bad arguments");
        // coefficients and CZ pairs on the qubits' index bits
        std::vector<int32_t> c(s->n);
        for (int q = 0; q < s->n; q++) c[qs_loc(s, q)] = coeff[q];
        std::vector<std::pair<int, int>> e;
        for (int i = 0; i < n_edges; i++) {
            int a = edges[2 * i], b = edges[2 * i + 1];
            if (a < 0 || a >= s->n || b < 0 || b >= s->n || a == b)
                return qs_fail(QS_EINVAL, "qs_apply_phase: bad edge %d", i);
            e.push_back({qs_loc(s, a), qs_loc(s, b)});
        }
        int n_act;
        std::vector<uint8_t> blob = qs_pack_phase(s->n, c, e, &n_act);
        void *dev = nullptr;
        if ((rc = stage(s, blob.data(), blob.size(), &dev))) return rc;
        return qs_launch_phase(s, dev, n_act);
    });
}

extern "C" int qs_run_circuit(qs_state *s, const qs_schedule *sc)
{
    return qs_guard([&]() -> int {
        int rc = check_state(s, "qs_run_circuit");
        if (rc) return rc;
        if (!sc || sc->n != s->n) return qs_fail(QS_EINVAL, "qs_run_circuit: schedule/state qubit mismatch");
        if ((rc = ensure_dev_schedule(s, sc))) return rc;
        // the schedule's ops name index bits: put the qubits where it expects them
        if ((rc = qs_order_set(s, sc->remap.empty() ? nullptr : sc->remap.data()))) return rc;
        const qs_dev_sched &d = sc->dev[s->dtype];
        struct ChainEnd {                 // whatever ends the run
            qs_state *s;
            ~ChainEnd() { s->chain = false; }
        } chain_end{s};
        for (size_t i = 0; i < sc->ops.size(); i++) {
            const qs_op_host &op = sc->ops[i];
            const uint8_t *data = (const uint8_t *)d.pool + d.offset[i];
            int skip = 0;
            size_t done = 0;
            if ((rc = run_passes(s, sc, d, i, &done))) return rc;
            if (done) {
                i += done - 1;
                continue;
            }
            if (op.kind == QS_OP_DENSE && try_pair(s, sc, d, i, &rc, &skip)) {
                i += skip;         // the ops after it that ran inside the pair's sweep
            } else if (op.kind == QS_OP_DENSE) {
                bool folded;
                rc = launch_op_dense(s, d, i, op, data, &folded);
                if (folded) i++;   // the phase op after it ran inside the sweep
            } else if (op.kind == QS_OP_DIAG) {
                rc = qs_launch_diag(s, (const int *)data, op.k, data + 64);
            } else {
                rc = qs_launch_phase(s, data, d.n_act[i]);
            }
            if (rc) return rc;
            s->chain = !s->pair_sweeps;   // the next op's sweep follows this one directly
        }
        return QS_OK;
    });
}

extern "C" int qs_run_circuit_timed(qs_state *s, const qs_schedule *sc, float *op_ms)
{
    return qs_guard([&]() -> int {
        int rc = check_state(s, "qs_run_circuit_timed");
        if (rc) return rc;
        if (!sc || sc->n != s->n || !op_ms)
            return qs_fail(QS_EINVAL, "qs_run_circuit_timed: bad schedule or output");
        if ((rc = ensure_dev_schedule(s, sc))) return rc;
        // the schedule's ops name index bits (any exchange sweep is not timed)
        if ((rc = qs_order_set(s, sc->remap.empty() ? nullptr : sc->remap.data()))) return rc;
        const qs_dev_sched &d = sc->dev[s->dtype];
        cudaStream_t st = (cudaStream_t)s->stream;
        size_t nops = sc->ops.size();
        std::vector<cudaEvent_t> ev(nops + 1);
        std::vector<char> skipped(nops, 0);
        for (auto &e : ev)
            if (cudaEventCreate(&e) != cudaSuccess) return qs_fail(QS_ECUDA, "event create");
        cudaEventRecord(ev[0], st);
        for (size_t i = 0; i < nops && !rc; i++) {
            const qs_op_host &op = sc->ops[i];
            const uint8_t *data = (const uint8_t *)d.pool + d.offset[i];
            bool folded = false;
            int skip = 0;
            if (op.kind == QS_OP_DENSE && try_pair(s, sc, d, i, &rc, &skip)) {
                // the second cluster (and a phase op folded into it) ran inside the sweep
            } else if (op.kind == QS_OP_DENSE) {
                rc = launch_op_dense(s, d, i, op, data, &folded);
                skip = folded ? 1 : 0;   // the phase op after it ran inside the sweep
            } else if (op.kind == QS_OP_DIAG) {
                rc = qs_launch_diag(s, (const int *)data, op.k, data + 64);
            } else {
                rc = qs_launch_phase(s, data, d.n_act[i]);
            }
            cudaEventRecord(ev[i + 1], st);
            for (int j = 0; j < skip; j++) {
                skipped[++i] = 1;
                cudaEventRecord(ev[i + 1], st);
            }
        }
        if (!rc) {
            cudaError_t e = cudaEventSynchronize(ev[nops]);
            if (e != cudaSuccess) rc = qs_fail(QS_ECUDA, "qs_run_circuit_timed: %s", cudaGetErrorString(e));
            for (size_t i = 0; i < nops && !rc; i++) {
                if (skipped[i]) op_ms[i] = -1.0f;
                else cudaEventElapsedTime(&op_ms[i], ev[i], ev[i + 1]);
            }
        }
        for (auto &e : ev) cudaEventDestroy(e);
        return rc;
    });
}

extern "C" int64_t qs_schedule_upload_bytes(const qs_schedule *sc, int dtype)
{
    int64_t bytes = 0;
    const int rc = qs_guard([&]() -> int {
        if (!sc || (dtype != QS_C64 && dtype != QS_C128)) return qs_fail(QS_EINVAL, "qs_schedule_upload_bytes");
        qs_dev_sched tmp;
        bytes = (int64_t)schedule_blob(sc, dtype, tmp).size();
        return QS_OK;
    });
    return rc == QS_OK ? bytes : rc;
}

extern "C" int qs_set_pair_sweeps(qs_state *s, int on)
{
    return qs_guard([&]() -> int {
        if (!s) return qs_fail(QS_EINVAL, "qs_set_pair_sweeps: null state");
        s->pair_sweeps = on != 0;
        return QS_OK;
    });
}

extern "C" int qs_schedule_remap(qs_schedule *sc, const int *loc)
{
    return qs_guard([&]() -> int {
        if (!sc || !loc) return qs_fail(QS_EINVAL, "qs_schedule_remap: null argument");
        if (!sc->remap.empty()) return qs_fail(QS_EINVAL, "qs_schedule_remap: schedule already remapped");
        const int n = sc->n;
        for (int q = 0; q < n; q++)
            if (loc[q] < 0 || loc[q] >= n || loc[loc[q]] != q)
                return qs_fail(QS_EINVAL, "qs_schedule_remap: loc is not a set of exchanges at qubit %d", q);
        for (qs_op_host &op : sc->ops) {
            if (op.kind == QS_OP_PHASE) {
                std::vector<int32_t> c(n);
                for (int q = 0; q < n; q++) c[loc[q]] = op.coeff[q];
                op.coeff = c;
                for (auto &e : op.edges) e = {loc[e.first], loc[e.second]};
                continue;
            }
            int lq[QS_MAX_DIAG_K], q[QS_MAX_DIAG_K];
            for (int j = 0; j < op.k; j++) lq[j] = loc[op.qubits[j]];
            std::vector<double> M;
            sort_targets(lq, op.k, op.matrix.data(), op.kind == QS_OP_DENSE, q, M);
            for (int j = 0; j < op.k; j++) op.qubits[j] = q[j];
            op.matrix = M;
        }
        for (auto &d : sc->dev) {   // device images describe the old ops
            if (d.pool) cudaFree(d.pool);
            d = qs_dev_sched();
        }
        sc->remap.assign(loc, loc + n);
        return QS_OK;
    });
}

extern "C" int qs_schedule_get_remap(const qs_schedule *sc, int *loc)
{
    return qs_guard([&]() -> int {
        if (!sc || !loc) return qs_fail(QS_EINVAL, "qs_schedule_get_remap: null argument");
        for (int q = 0; q < sc->n; q++) loc[q] = sc->remap.empty() ? q : sc->remap[q];
        return QS_OK;
    });
}

extern "C" int qs_schedule_choose_remap(const qs_schedule *sc, int dtype, int *loc)
{
    return qs_guard([&]() -> int {
        if (!sc || !loc || (dtype != QS_C64 && dtype != QS_C128))
            return qs_fail(QS_EINVAL, "qs_schedule_choose_remap: bad arguments");
        const int n = sc->n;
        for (int q = 0; q < n; q++) loc[q] = q;
        // the index bits whose sweeps cost more (measured): 0-1 for complex128,
        // 0-4 for complex64
        const int nlow = std::min(n, dtype == QS_C128 ? 2 : 5);
        if (n < 5 + nlow) return QS_OK;
        // weight of each qubit: the dense sweeps it is a target of, each
        // counted by the share of the state it covers from |0...0> (the support
        // grows by every dense cluster's qubits)
        std::vector<double> w(n, 0.0);
        uint64_t sup = 0;
        for (const qs_op_host &op : sc->ops) {
            if (op.kind != QS_OP_DENSE) continue;
            for (int j = 0; j < op.k; j++) sup |= 1ULL << op.qubits[j];
            const double share = std::ldexp(1.0, __builtin_popcountll(sup) - n);
            for (int j = 0; j < op.k; j++) w[op.qubits[j]] += share;
        }
        // the nlow lightest qubits go to the low bits (ties: a qubit already
        // there, then the lower qubit)
        std::vector<int> order(n);
        for (int q = 0; q < n; q++) order[q] = q;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
            if (w[a] != w[b]) return w[a] < w[b];
            return (a < nlow) > (b < nlow);
        });
        std::vector<char> chosen(n, 0);
        for (int i = 0; i < nlow; i++) chosen[order[i]] = 1;
        std::vector<int> in, out;              // chosen qubits above, low bits to free
        for (int q = nlow; q < n; q++)
            if (chosen[q]) in.push_back(q);
        for (int b = 0; b < nlow; b++)
            if (!chosen[b]) out.push_back(b);
        for (size_t i = 0; i < in.size() && i < out.size(); i++) {
            loc[in[i]] = out[i];
            loc[out[i]] = in[i];
        }
        return QS_OK;
    });
}

extern "C" int qs_schedule_upload(const qs_schedule *sc, int dtype)
{
    return qs_guard([&]() -> int {
        if (!sc || (dtype != QS_C64 && dtype != QS_C128)) return qs_fail(QS_EINVAL, "qs_schedule_upload");
        qs_state probe;
        probe.n = sc->n;
        probe.dtype = dtype;
        return ensure_dev_schedule(&probe, sc);
    });
}

extern "C" int qs_set_device(int device)
{
    return qs_guard([&]() -> int {
        cudaError_t e = cudaSetDevice(device);
        return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "qs_set_device(%d): %s", device, cudaGetErrorString(e));
    });
}

extern "C" void qs_schedule_free(qs_schedule *sc)
{
    if (!sc) return;
    for (auto &d : sc->dev)
        if (d.pool) cudaFree(d.pool);
    delete sc;
}
