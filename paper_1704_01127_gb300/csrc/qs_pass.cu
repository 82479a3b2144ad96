// Passes: several consecutive CUDA-core ops (dense clusters, phase products) in
// one read and write of the state.
//
// A pass fixes W `local` index bits that hold the targets of all its dense ops;
// the 2^W amplitudes that agree on the other bits (a chunk) go through the ops in
// shared memory, one CTA per chunk (the idea of Sec. 4: several gates while a
// chunk is in fast memory).  The arithmetic per group and per amplitude is that
// of the sweeps (k_dense, k_phase), operation by operation, so a pass gives the
// sweeps' bits.
//
// The lowest kRunBits bits are always local (runs of 64 bytes in memory).  A
// chunk is 64 KB at most (2^13 complex64, 2^12 complex128 amplitudes), so three
// CTAs of 128 threads share an SM (two in complex128): one moves its chunk while
// the others compute.
// What bounds it: the FP32 FMA pipe from k = 4 on in complex64, the FP64 pipe in
// complex128.  Shared memory returns 128 bytes a clock per SM, broadcast or not:
// with one group per thread the rows of U alone take twice the FMAs' time, so a
// complex64 thread carries up to four groups through every row (two for k = 5:
// 128 registers of amplitudes).  Packed FP32 FMAs (fma.rn.f32x2) measured slower:
// they need U's elements twice over, from shared memory or by moves.
// 96 circuits of 16 to 21 qubits, k <= 4, complex64 (102 GFMA, 2.7 ms of the FMA
// pipe; one cluster of CTAs per circuit before): 26.3 -> 6.0 ms, two thirds of the
// issue slots used, two thirds of them by FMAs.  What the kernel holds across an op
// has to stay out of the registers (spills inside the rows: 6.9 ms).  A plain circuit
// of 83 gates on 16 qubits, complex128: 320 -> 90 us (a sweep per gate before); there
// a chunk has 512 amplitudes and the instructions' latency shows, so gates that are one
// factor of a phase product visit just the amplitudes they turn (17 us more with an
// exponent for every amplitude), and even turns have loops without the FP64 pipe (97 us
// without those; 24 qubits, a CZ of a pass 37 -> 11 us, an S gate 70 -> 15).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "qs_device.cuh"
#include "qs_internal.h"
#include "qs_launch.cuh"

namespace {

using qsd::cplx;

template <typename R> constexpr int kRunBits = sizeof(R) == 4 ? 3 : 2;
template <typename R> constexpr int kPassBits = sizeof(R) == 4 ? 13 : 12;    // most local bits
template <typename R> constexpr int kOpBytes = 32 * 32 * 2 * (int)sizeof(R);  // operands held at a time
template <typename R> constexpr int kOneThreads = sizeof(R) == 4 ? 128 : 256;   // a single state's passes

// Where local index l sits in shared memory: the upper bits are folded into the
// bank bits (four of 8-byte, three of 16-byte elements), so that lanes that
// differ in any few neighbouring bits fall in different banks.  Linear:
// place(a ^ b) = place(a) ^ place(b).
template <typename R>
__device__ __forceinline__ uint32_t place(uint32_t l)
{
    if constexpr (sizeof(R) == 4) return l ^ (((l >> 4) ^ (l >> 8) ^ (l >> 12)) & 15u);
    else return l ^ (((l >> 3) ^ (l >> 6) ^ (l >> 9)) & 7u);
}

// The bits of x at the set positions of mask, lowest first.
__device__ __forceinline__ uint64_t deposit(uint64_t x, uint64_t mask)
{
    uint64_t r = 0;
    for (; mask && x; mask &= mask - 1, x >>= 1)
        if (x & 1) r |= mask & (0ULL - mask);
    return r;
}

// Index bits of the local bits above the runs, six at a time.
struct LocalMap {
    uint64_t lo[64], hi[64];
    uint64_t base;   // the chunk's own index bits; here, not in registers that the ops need
    int rb;
    __device__ __forceinline__ uint64_t at(uint32_t l) const
    {
        const uint32_t h = l >> rb;
        return lo[h & 63u] | hi[h >> 6] | (l & ((1u << rb) - 1u));
    }
};

// fma(-a, b, c) with the sign in the FMA itself: written as fmaf(-a, b, c) with a
// from shared memory, the compiler spends an integer instruction on every -a.
__device__ __forceinline__ float fnma(float a, float b, float c)
{
    float r;
    asm("{\n\t.reg .f32 t;\n\tneg.f32 t, %1;\n\tfma.rn.f32 %0, t, %2, %3;\n\t}" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Local index of group g's member 0.
template <int K>
__device__ __forceinline__ uint32_t group_local(uint32_t g, const int *q)
{
#pragma unroll
    for (int j = 0; j < K; j++) {
        const uint32_t lo = g & ((1u << q[j]) - 1u);
        g = ((g ^ lo) << 1) | lo;
    }
    return g;
}

// A dense k-qubit cluster on the chunk, complex64, G groups per thread and turn
// (T G divides the number of groups): the FMA sequence of qsd::dense_group.
template <int K, int G, int T>
__device__ __forceinline__ void dense_groups_g(float2 *sm, int W, const int *q, const float2 *Us)
{
    constexpr int D = 1 << K;
    uint32_t pq[K];
#pragma unroll
    for (int j = 0; j < K; j++) pq[j] = place<float>(1u << q[j]);
    const uint32_t ng = 1u << (W - K);
#pragma unroll 1
    for (uint32_t g0 = threadIdx.x; g0 < ng; g0 += T * G) {
        float2 v[G][D];
        uint32_t pb[G];
#pragma unroll
        for (int i = 0; i < G; i++) {
            pb[i] = place<float>(group_local<K>(g0 + T * i, q));
#pragma unroll
            for (int x = 0; x < D; x++) {
                uint32_t o = 0;
#pragma unroll
                for (int j = 0; j < K; j++)
                    if ((x >> j) & 1) o ^= pq[j];
                v[i][x] = sm[pb[i] ^ o];
            }
        }
        // U's elements two at a time, four ahead (past the last row: the chunk's first
        // bytes, unused)
        const float4 *u = reinterpret_cast<const float4 *>(Us);
        float4 next = u[0], next2 = *++u;
#pragma unroll 1
        for (int r = 0; r < D; r++) {
            float ar[G], ai[G];
#pragma unroll
            for (int i = 0; i < G; i++) ar[i] = ai[i] = 0;
#pragma unroll
            for (int x = 0; x < D; x += 2) {
                const float4 w = next;
                next = next2;
                next2 = *++u;
#pragma unroll
                for (int i = 0; i < G; i++) {
                    ar[i] = fmaf(v[i][x].x, w.x, ar[i]);
                    ai[i] = fmaf(v[i][x].y, w.x, ai[i]);
                    ar[i] = fnma(v[i][x].y, w.y, ar[i]);
                    ai[i] = fmaf(v[i][x].x, w.y, ai[i]);
                }
#pragma unroll
                for (int i = 0; i < G; i++) {
                    ar[i] = fmaf(v[i][x + 1].x, w.z, ar[i]);
                    ai[i] = fmaf(v[i][x + 1].y, w.z, ai[i]);
                    ar[i] = fnma(v[i][x + 1].y, w.w, ar[i]);
                    ai[i] = fmaf(v[i][x + 1].x, w.w, ai[i]);
                }
            }
            uint32_t o = 0;
#pragma unroll
            for (int j = 0; j < K; j++) o ^= (r >> j) & 1 ? pq[j] : 0u;
#pragma unroll
            for (int i = 0; i < G; i++) sm[pb[i] ^ o] = make_float2(ar[i], ai[i]);
        }
    }
}

// The same for any number of groups, one per thread and turn; with fewer groups
// than threads the rows of a group are split over threads.
template <typename R, int K, int T>
__device__ __forceinline__ void dense_groups(typename cplx<R>::t *sm, int W, const int *q, const typename cplx<R>::t *Us)
{
    using C = typename cplx<R>::t;
    constexpr int D = 1 << K;
    uint32_t pq[K];
#pragma unroll
    for (int j = 0; j < K; j++) pq[j] = place<R>(1u << q[j]);
    const uint32_t ng = 1u << (W - K);
    const bool split = ng < T;
    int r0 = 0, r1 = D;
    if (split) {
        const int part = (int)(threadIdx.x >> (W - K)), rows = max(1, (int)((D * ng) / T));
        r0 = min(D, part * rows);
        r1 = min(D, r0 + rows);
    }
#pragma unroll 1
    for (uint32_t g = split ? threadIdx.x & (ng - 1u) : threadIdx.x; g < ng; g += T) {
        const uint32_t pb = place<R>(group_local<K>(g, q));
        C v[D];
#pragma unroll
        for (int x = 0; x < D; x++) {
            uint32_t o = pb;
#pragma unroll
            for (int j = 0; j < K; j++)
                if ((x >> j) & 1) o ^= pq[j];
            v[x] = sm[o];
        }
        if (split) __syncthreads();   // every thread of a group has read it (one turn, all threads)
#pragma unroll (K <= 1 ? 2 : 1)
        for (int r = r0; r < r1; r++) {
            R ar = 0, ai = 0;
            const C *row = Us + r * D;
#pragma unroll
            for (int x = 0; x < D; x++) {
                const C m = row[x];
                ar = fma(v[x].x, m.x, ar);
                ai = fma(v[x].y, m.x, ai);
                ar = fma(-v[x].y, m.y, ar);
                ai = fma(v[x].x, m.y, ai);
            }
            uint32_t o = pb;
#pragma unroll
            for (int j = 0; j < K; j++) o ^= (r >> j) & 1 ? pq[j] : 0u;
            C z;
            z.x = ar;
            z.y = ai;
            sm[o] = z;
        }
    }
}

template <typename R, int K, int T>
__device__ __forceinline__ void dense_chunk(typename cplx<R>::t *sm, int W, const int *q, const typename cplx<R>::t *Us)
{
    if constexpr (sizeof(R) == 4) {
        const uint32_t ng = 1u << (W - K);
        if constexpr (K < 5 && T == 128)
            if (ng >= 4 * T) return dense_groups_g<K, 4, T>(sm, W, q, Us);
        if constexpr (T == 128 || (T == 256 && K < 5))
            if (ng >= 2 * T) return dense_groups_g<K, 2, T>(sm, W, q, Us);
    }
    dense_groups<R, K, T>(sm, W, q, Us);
}

// A phase product on the chunk.  The index splits into a column (as many local
// bits as the CTA has threads), a row of the chunk and the chunk's base; with
// m(x) the exponent of the bits x alone and M(x) the bits whose CZ partners meet
// x an odd number of times,
//   m(x | c) = m(x) + m(c) + 4 popc(c & M(x)),
// x = base and row, formed by one thread per row.  complex128 pairs rows so that
// one FP64 rotation serves two amplitudes, as k_phase does.
template <typename R, int T>
__device__ __forceinline__ void phase_chunk(typename cplx<R>::t *sm, int W, const LocalMap &map, uint64_t base,
                                            const qs_phase_dev *ph, int n_act, uint64_t *row_M, int *row_m)
{
    using C = typename cplx<R>::t;
    constexpr int kT = T == 128 ? 7 : T == 256 ? 8 : 9;
    const qs_phase_term *terms = reinterpret_cast<const qs_phase_term *>(ph + 1);
    const uint64_t c0 = ph->cmask[0], c1 = ph->cmask[1], c2 = ph->cmask[2];
    auto exponent = [&](uint64_t x, uint64_t &M) {
        int m = __popcll(x & c0) + 2 * __popcll(x & c1) + 4 * __popcll(x & c2), par = 0;
        M = 0;
        for (int t = 0; t < n_act; t++) {
            const uint64_t P = terms[t].partners;
            const int a = terms[t].a, o = __popcll(x & P) & 1;
            if ((x >> a) & 1) {
                par ^= o;
                M ^= P;
            }
            M ^= (uint64_t)o << a;
        }
        return m + 4 * par;
    };
    const int tid = threadIdx.x, cb = min(W, kT), rows = 1 << (W - cb);
    const uint32_t col = (uint32_t)tid & ((1u << cb) - 1u);
    const bool in = tid < (1 << cb);
    uint64_t M;
    if (tid < rows) {
        row_m[tid] = exponent(base | map.at((uint32_t)tid << cb), M);
        row_M[tid] = M;
    }
    const uint64_t xc = map.at(col);
    const int mc = exponent(xc, M);
    uint32_t flip = 0;   // complex128: a lane bit whose coefficient is odd
    if constexpr (sizeof(R) == 8)
        for (int j = min(cb, 5) - 1; j >= 0; j--)
            if (map.at(1u << j) & c0) flip = 1u << j;
    uint64_t xc2 = xc;
    int mc2 = mc;
    if (flip) {
        xc2 = map.at(col ^ flip);
        mc2 = exponent(xc2, M);
    }
    __syncthreads();
    if (flip && rows > 1) {
        for (int r = 0; r < rows; r += 2) {
            const int ma = (mc + row_m[r] + 4 * __popcll(xc & row_M[r])) & 7;
            // the second row's column: exactly one of the two amplitudes is odd
            const bool other = !((row_m[r] ^ row_m[r + 1]) & 1);
            const int mb = ((other ? mc2 : mc) + row_m[r + 1] + 4 * __popcll((other ? xc2 : xc) & row_M[r + 1])) & 7;
            C *pa = sm + place<R>(((uint32_t)r << cb) | col);
            C *pb = sm + place<R>(((uint32_t)(r + 1) << cb) | (other ? col ^ flip : col));
            if (!in) continue;
            C a = *pa, b = *pb;
            const C t = qsd::eighth_turn(ma & 1 ? a : b);
            if (ma & 1) a = t;
            else b = t;
            *pa = qsd::quarter_turns<C>(a, ma >> 1);
            *pb = qsd::quarter_turns<C>(b, mb >> 1);
        }
        return;
    }
    auto each_row = [&](auto odd) {
        for (int r = 0; r < rows; r++) {
            const int m = (mc + row_m[r] + 4 * __popcll(xc & row_M[r])) & 7;
            C *p = sm + place<R>(((uint32_t)r << cb) | col);
            if (m && in) *p = decltype(odd)::value ? qsd::rotate8<C, R>(*p, m) : qsd::quarter_turns<C>(*p, m >> 1);
        }
    };
    // (complex128: a loop of their own for even exponents; a branch around an eighth turn alone
    // is made into predicates, and the FP64 pipe takes those instructions too)
    if (sizeof(R) == 4 || c0) each_row(std::true_type{});
    else each_row(std::false_type{});
}

// One factor of a phase op by itself (a T-type gate on one qubit, a CZ): the
// amplitudes whose k (0, 1 or 2) local bits q are set turn by c eighths.  Only those
// are visited, and every lane of an odd turn's FP64 instructions has work.
template <typename R, int T>
__device__ __forceinline__ void turn_chunk(typename cplx<R>::t *sm, int W, int k, int q0, int q1, int c)
{
    using C = typename cplx<R>::t;
    auto with_bit = [](uint32_t l, int q) {
        const uint32_t lo = l & ((1u << q) - 1u);
        return ((l ^ lo) << 1) | lo | 1u << q;
    };
    auto each = [&](auto odd) {
        for (uint32_t h = threadIdx.x; h < (1u << (W - k)); h += T) {
            uint32_t l = h;
            if (k > 0) l = with_bit(l, q0);
            if (k > 1) l = with_bit(l, q1);
            C *p = sm + place<R>(l);
            *p = decltype(odd)::value ? qsd::rotate8<C, R>(*p, c) : qsd::quarter_turns<C>(*p, c >> 1);
        }
    };
    if (sizeof(R) == 4 || (c & 1)) each(std::true_type{});   // two loops as in phase_chunk
    else each(std::false_type{});
}

__device__ __forceinline__ void copy16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Chunk `ch` of a pass on the state psi.  Before wait() nothing of the state is touched.
template <typename R, int T, typename Wait>
__device__ __forceinline__ void run_chunk(const qs_pass &ps, typename cplx<R>::t *__restrict__ psi, uint64_t ch, uint8_t *smem,
                                          Wait wait)
{
    using C = typename cplx<R>::t;
    __shared__ LocalMap map;
    __shared__ uint64_t row_M[1 << (kPassBits<R> - 7)];
    __shared__ int row_m[1 << (kPassBits<R> - 7)];
    const int tid = threadIdx.x, W = ps.W, rb = min(W, kRunBits<R>);
    uint8_t *operands = smem;
    C *sm = reinterpret_cast<C *>(smem + kOpBytes<R>);
    const uint32_t op_a = (uint32_t)__cvta_generic_to_shared(operands);
    // operands of ops o .. o + n - 1, asynchronously
    auto stage = [&](int o, int n) {
        for (int j = o; j < o + n; j++)
            for (uint32_t i = 16u * tid; i < ps.op[j].bytes; i += 16u * T)
                copy16(op_a + ps.op[j].at + i, reinterpret_cast<const uint8_t *>(ps.op[j].data) + i);
    };
    auto staged = [&]() {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    };
    if (ps.n_ops) stage(0, ps.op[0].n_stage);
    {
        uint64_t hi = ps.local, lo6 = 0;   // the local bits above the runs, six at a time
        for (int j = 0; j < rb; j++) hi &= hi - 1;
        for (int j = 0; j < 6 && hi; j++) {
            lo6 |= hi & (0ULL - hi);
            hi &= hi - 1;
        }
        if (tid < 64) map.lo[tid] = deposit(tid, lo6);
        else if (tid < 128) map.hi[tid - 64] = deposit(tid - 64, hi);
        if (tid == 0) {
            map.rb = rb;
            map.base = deposit(ch, ps.outer);
        }
    }
    __syncthreads();
    wait();
    // 16 bytes an access: two complex64 amplitudes (bit 0 is always local)
    constexpr int VEC = sizeof(R) == 4 ? 2 : 1, kAhead = 8;
    const uint32_t units = (1u << W) / VEC;
    const uint64_t outside = ~ps.support;
    const C *from = psi + ps.amp + map.base;
    for (uint32_t u0 = tid; u0 < units; u0 += T * kAhead) {
        uint4 z[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint32_t u = u0 + T * k;
            z[k] = make_uint4(0u, 0u, 0u, 0u);
            if (u >= units) continue;
            const uint64_t o = map.at(VEC * u);
            if (ps.first) {                       // from |0...0>: the one chunk of the first pass
                if (u == 0) {
                    C one;
                    one.x = 1;
                    one.y = 0;
                    *reinterpret_cast<C *>(&z[k]) = one;
                }
            } else if (!(o & outside)) {
                z[k] = __ldcg(reinterpret_cast<const uint4 *>(from + o));
            }
        }
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint32_t u = u0 + T * k;
            if (u >= units) continue;
            const uint32_t l = place<R>(VEC * u);
            if constexpr (VEC == 2) {
                if (l & 1u) z[k] = make_uint4(z[k].z, z[k].w, z[k].x, z[k].y);
                reinterpret_cast<uint4 *>(sm)[l >> 1] = z[k];
            } else {
                reinterpret_cast<uint4 *>(sm)[l] = z[k];
            }
        }
    }
    staged();
    for (int o = 0; o < ps.n_ops; o++) {
        const qs_pass_op &op = ps.op[o];
        if (o && op.n_stage) {
            stage(o, op.n_stage);
            staged();
        }
        const void *data = operands + op.at;
        if (op.kind == QS_OP_DENSE) {
            int q[QS_MAX_K];
#pragma unroll
            for (int j = 0; j < QS_MAX_K; j++) q[j] = op.q[j];
            const C *U = reinterpret_cast<const C *>(data);
            switch (op.k) {
            case 1: dense_chunk<R, 1, T>(sm, W, q, U); break;
            case 2: dense_chunk<R, 2, T>(sm, W, q, U); break;
            case 3: dense_chunk<R, 3, T>(sm, W, q, U); break;
            case 4: dense_chunk<R, 4, T>(sm, W, q, U); break;
            default: dense_chunk<R, 5, T>(sm, W, q, U); break;
            }
        } else if (op.kind == QS_PASS_TURN) {
            if ((map.base & op.data) != op.data) continue;   // the factor's bits outside the chunk: the same for all of it
            turn_chunk<R, T>(sm, W, op.k, op.q[0], op.q[1], op.n_act);
        } else {
            phase_chunk<R, T>(sm, W, map, map.base, reinterpret_cast<const qs_phase_dev *>(data), op.n_act, row_M, row_m);
        }
        __syncthreads();
    }
    C *to = psi + ps.amp + map.base;
    for (uint32_t u = tid; u < units; u += T) {
        const uint32_t l = place<R>(VEC * u);
        uint4 z;
        if constexpr (VEC == 2) {
            z = reinterpret_cast<const uint4 *>(sm)[l >> 1];
            if (l & 1u) z = make_uint4(z.z, z.w, z.x, z.y);
        } else {
            z = reinterpret_cast<const uint4 *>(sm)[l];
        }
        *reinterpret_cast<uint4 *>(to + map.at(VEC * u)) = z;
    }
}

// One state: the pass in the launch's parameters, a CTA per chunk.
template <typename R>
__global__ void __launch_bounds__(kOneThreads<R>, sizeof(R) == 4 ? 3 : 1)
k_pass(const __grid_constant__ qs_pass ps, typename cplx<R>::t *__restrict__ psi)
{
    extern __shared__ __align__(16) uint8_t smem[];
    chain_start();
    run_chunk<R, kOneThreads<R>>(ps, psi, blockIdx.x, smem, [] { chain_wait(); });
}

// Many states: items[i] = (pass, chunk).
template <typename R, int T>
__global__ void __launch_bounds__(T, T == 128 ? (sizeof(R) == 4 ? 3 : 2) : T == 256 ? 2 : 1)
k_pass_items(const qs_pass *__restrict__ passes, const uint2 *__restrict__ items, uint32_t n_items,
             typename cplx<R>::t *__restrict__ amp)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ __align__(16) qs_pass ps;
    chain_start();
    if (blockIdx.x >= n_items) return;
    const uint2 it = items[blockIdx.x];
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(passes + it.x);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&ps);
        for (int i = threadIdx.x; i < (int)(sizeof(qs_pass) / 4); i += T) dst[i] = src[i];
    }
    __syncthreads();
    run_chunk<R, T>(ps, amp, it.y, smem, [] { chain_wait(); });
}

template <typename R>
size_t pass_smem(int W) { return (size_t)kOpBytes<R> + ((size_t)2 * sizeof(R) << W); }

// dynamic shared memory of a kernel, set once per device and kernel
template <typename F>
int allow_smem(F kernel, size_t bytes, bool *ready)
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return qs_fail(QS_EUNSUPPORTED, "device %d", dev);
    if (ready[dev]) return QS_OK;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return qs_fail(QS_ECUDA, "pass smem attribute: %s", cudaGetErrorString(e));
    ready[dev] = true;
    return QS_OK;
}

template <typename R>
int launch_pass_r(qs_state *s, const qs_pass &ps)
{
    static bool ready[64] = {};
    if (int rc = allow_smem(k_pass<R>, pass_smem<R>(kPassBits<R>), ready)) return rc;
    const cudaError_t e = launch_sweep(s, s->chain, k_pass<R>, 1 << (s->n - ps.W), kOneThreads<R>, pass_smem<R>(ps.W), ps,
                                       reinterpret_cast<typename cplx<R>::t *>(s->amp));
    return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "k_pass launch: %s", cudaGetErrorString(e));
}

template <typename R, int T>
int launch_items_t(const qs_pass *passes, const uint2 *items, uint32_t n, void *amp, int W, int C, bool chain, cudaStream_t st)
{
    static bool ready[64] = {};
    if (int rc = allow_smem(k_pass_items<R, T>, pass_smem<R>(kPassBits<R>), ready)) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((n + C - 1) / C * C);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = pass_smem<R>(W);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chain ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_pass_items<R, T>, passes, items, n,
                                             reinterpret_cast<typename cplx<R>::t *>(amp));
    return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "pass launch: %s", cudaGetErrorString(e));
}

template <typename R>
int launch_items_r(const qs_pass *passes, const uint2 *items, uint32_t n, void *amp, int W, int C, int T, bool chain,
                   cudaStream_t st)
{
    return T == 128   ? launch_items_t<R, 128>(passes, items, n, amp, W, C, chain, st)
           : T == 256 ? launch_items_t<R, 256>(passes, items, n, amp, W, C, chain, st)
                      : launch_items_t<R, 512>(passes, items, n, amp, W, C, chain, st);
}

}  // namespace

// A phase op that is one factor: e^{i pi turns / 4} where the one or two index bits
// `bits` are set (a coefficient, or a CZ pair).
static bool single_factor(int n, const qs_op_host &op, uint64_t *bits, int *turns)
{
    uint64_t coeff = 0;
    for (int q = 0; q < n; q++)
        if (op.coeff[q] & 7) coeff |= 1ULL << q;
    const int nc = __builtin_popcountll(coeff);
    if (nc + (int)op.edges.size() != 1) return false;
    *bits = nc ? coeff : 1ULL << op.edges[0].first | 1ULL << op.edges[0].second;
    *turns = nc ? op.coeff[__builtin_ctzll(coeff)] & 7 : 4;
    return true;
}

int qs_pass_bits(int dtype) { return dtype == QS_C128 ? kPassBits<double> : kPassBits<float>; }

std::vector<qs_pass> qs_plan_passes(int n, int dtype, int wmax, const std::vector<qs_pass_in> &ops, bool from_basis)
{
    const int run_bits = dtype == QS_C128 ? kRunBits<double> : kRunBits<float>;
    const uint32_t op_bytes = dtype == QS_C128 ? kOpBytes<double> : kOpBytes<float>;
    const int W = std::min(n, wmax);
    const uint64_t all = qs_index_mask(n), runs = qs_index_mask(std::min(n, run_bits));
    uint64_t support = from_basis ? 0 : all;
    std::vector<qs_pass> out;
    size_t i = 0;
    do {
        qs_pass p;
        std::memset(&p, 0, sizeof(p));
        uint64_t mask = runs;
        const size_t i0 = i;
        for (; i < ops.size() && i - i0 < (size_t)QS_PASS_OPS; i++) {
            uint64_t with = mask;
            if (ops[i].kind == QS_OP_DENSE)
                for (int j = 0; j < ops[i].k; j++) with |= 1ULL << ops[i].qubits[j];
            if (__builtin_popcountll(with) > W) break;
            mask = with;
        }
        for (int b = 0; b < n && __builtin_popcountll(mask) < W; b++) mask |= 1ULL << b;
        p.n_ops = (int32_t)(i - i0);
        p.first_op = (int32_t)i0;
        p.W = W;
        p.first = from_basis && out.empty();
        p.local = mask;
        p.support = support;
        p.outer = support & ~mask;
        support |= mask;
        uint32_t at = op_bytes;   // operand buffer: a new batch of ops whenever the next does not fit
        int batch = 0;
        for (int o = 0; o < p.n_ops; o++) {
            const qs_pass_in &in = ops[i0 + o];
            qs_pass_op &op = p.op[o];
            op.kind = (uint8_t)in.kind;
            op.k = (uint8_t)in.k;
            op.n_act = (uint8_t)in.n_act;
            op.bytes = (uint16_t)in.bytes;
            op.data = in.data;
            auto local = [&](int b) { return (uint8_t)__builtin_popcountll(mask & ((1ULL << b) - 1)); };
            if (in.kind == QS_OP_DENSE)
                for (int j = 0; j < in.k; j++) op.q[j] = local(in.qubits[j]);
            uint64_t bits;
            int turns;
            if (in.kind == QS_OP_PHASE && single_factor(n, *in.op, &bits, &turns)) {
                op.kind = QS_PASS_TURN;
                op.n_act = (uint8_t)turns;
                op.bytes = 0;
                op.data = bits & ~mask;
                op.k = 0;
                for (uint64_t x = bits & mask; x; x &= x - 1) op.q[op.k++] = local(__builtin_ctzll(x));
            }
            const uint32_t need = (op.bytes + 15u) & ~15u;
            if (at + need > op_bytes) {
                at = 0;
                batch = o;
            }
            op.at = (uint16_t)at;
            at += need;
            p.op[batch].n_stage++;
        }
        out.push_back(p);
    } while (i < ops.size());
    return out;
}

int qs_launch_pass(qs_state *s, const qs_pass &ps)
{
    s->perm_invariant = false;
    if (int rc = qs_materialize(s)) return rc;
    return s->dtype == QS_C128 ? launch_pass_r<double>(s, ps) : launch_pass_r<float>(s, ps);
}

int qs_launch_pass_items(int dtype, const void *passes, const void *items, uint32_t n, void *amp, int W, int cluster,
                         int threads, bool chain, void *stream)
{
    const qs_pass *p = (const qs_pass *)passes;
    const uint2 *it = (const uint2 *)items;
    cudaStream_t st = (cudaStream_t)stream;
    return dtype == QS_C128 ? launch_items_r<double>(p, it, n, amp, W, cluster, threads, chain, st)
                            : launch_items_r<float>(p, it, n, amp, W, cluster, threads, chain, st);
}
