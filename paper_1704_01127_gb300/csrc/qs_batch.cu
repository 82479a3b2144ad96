// Batched simulation of many small circuits.
//
// Every circuit keeps its own state (2^n amplitudes) in one device buffer.  Its
// ops are split into passes (qs_pass.cu: several ops per read and write, chunks
// in shared memory); one launch runs pass j of every circuit that has one, a CTA
// per chunk, so the largest circuits spread over the whole GPU and ops of one
// circuit stay ordered by the launches.  From |0...0> only chunks in the support
// so far are visited (zeros elsewhere are neither read nor written until a pass
// covers them).  The arithmetic is the single-state sweeps', so a batch
// reproduces single-state CUDA-core runs bit for bit.  The launch configuration
// (thread-block clusters of C neighbouring chunks, threads per CTA) and the
// cluster bound k_max of the scheduler are chosen by a timing autotuner; the
// launches can be captured once in a CUDA graph and replayed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "qs_device.cuh"
#include "qs_internal.h"

namespace {

using qsd::cplx;

struct BatchCirc {
    int32_t n;
    int32_t pad;
    int64_t amp_off;   // in amplitudes
};

__global__ void k_log_table(qsd::LogTable *t) { qsd::log_table_init(*t); }

// Per-circuit FP64 statistics: a CTA per 2^kStatsBits amplitudes (circuit
// blk[i].x, part blk[i].y), then a warp per circuit over its CTAs' sums.  Bound
// by the FP64 pipe (about 12 operations an amplitude; 102 M amplitudes: 2.1 ms);
// one CTA per circuit, with its own log table, left most SMs idle: 10.2 -> 2.0 ms.
constexpr int kStatsBits = 15;

template <typename R>
__global__ void __launch_bounds__(256)
k_batch_stats(const BatchCirc *__restrict__ circ, const int2 *__restrict__ blk, const qsd::LogTable *__restrict__ table,
              const typename cplx<R>::t *__restrict__ amp, double *__restrict__ part)
{
    using C2 = typename cplx<R>::t;
    __shared__ __align__(16) qsd::LogTable lt;
    __shared__ double red[3][8];
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(table);
        uint4 *dst = reinterpret_cast<uint4 *>(&lt);
        for (int i = threadIdx.x; i < (int)(sizeof(lt) / sizeof(uint4)); i += 256) dst[i] = src[i];
    }
    __syncthreads();
    const int2 at = blk[blockIdx.x];
    const BatchCirc cc = circ[at.x];
    const uint32_t N = 1u << min(cc.n, kStatsBits);
    const C2 *psi = amp + cc.amp_off + ((uint64_t)at.y << kStatsBits);
    double a[3] = {0, 0, 0};   // sum p, -sum p ln p, sum p^2
    constexpr int kAhead = 4;
    for (uint32_t i0 = threadIdx.x; i0 < N; i0 += 256 * kAhead) {
        C2 v[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; k++) v[k] = i0 + 256u * k < N ? psi[i0 + 256u * k] : C2{};
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const double p = qsd::prob(v[k]);
            a[0] += p;
            // p of 2^-1022 or more (an integer compare: FP64 ones run on the FP64 pipe)
            if ((uint32_t)__double2hiint(p) - 0x00100000u <= 0x7FE00000u) a[1] -= p * qsd::log_tab(lt, p);
            a[2] = fma(p, p, a[2]);
        }
    }
#pragma unroll
    for (int j = 0; j < 3; j++) {
        double v = a[j];
        for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[j][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double v = 0;
        for (int w = 0; w < 8; w++) v += red[threadIdx.x][w];
        part[3 * (size_t)blockIdx.x + threadIdx.x] = v;
    }
}

// sum p, entropy, mean of N p (= sum p), mean of (N p)^2 (= N sum p^2)
__global__ void __launch_bounds__(32)
k_batch_stats_final(const BatchCirc *__restrict__ circ, const int *__restrict__ first, const double *__restrict__ part,
                    double *__restrict__ out)
{
    const int c = blockIdx.x, b0 = first[c], b1 = first[c + 1];
    double a[3] = {0, 0, 0};
    for (int b = b0 + (int)threadIdx.x; b < b1; b += 32)
        for (int j = 0; j < 3; j++) a[j] += part[3 * (size_t)b + j];
    for (int j = 0; j < 3; j++)
        for (int o = 16; o; o >>= 1) a[j] += __shfl_down_sync(0xffffffffu, a[j], o);
    if (threadIdx.x == 0) {
        out[4 * c] = out[4 * c + 2] = a[0];
        out[4 * c + 1] = a[1];
        out[4 * c + 3] = a[2] * (double)(1ULL << circ[c].n);
    }
}

uint64_t splitmix64(uint64_t seed, uint64_t j)
{
    uint64_t z = seed + (j + 1) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

}  // namespace

struct qs_batch {
    int dtype = QS_C64;
    int n_circ = 0;
    void *stream = nullptr;
    void *amp = nullptr;
    size_t amp_bytes = 0;
    bool clear = false;             // some circuit has amplitudes that no pass covers: zeroed first
    int W = 0;                      // bits of a chunk
    // passes of all circuits, (pass, chunk) of every CTA by launch, operands
    void *passes = nullptr, *items = nullptr, *circ = nullptr, *pool = nullptr, *stats = nullptr;
    std::vector<size_t> level;      // first item of every launch, then their number
    // statistics: (circuit, part) of every CTA, the first CTA of every circuit, their sums, the log table
    void *sblk = nullptr, *sfirst = nullptr, *spart = nullptr, *slog = nullptr;
    int n_sblk = 0;
    std::vector<int> nq;
    std::vector<uint64_t> amp_off;
    int cluster = 1, block = 256;
    cudaGraphExec_t exec = nullptr;
    int exec_cluster = 0, exec_block = 0;
};

namespace {

template <typename T>
int upload(void **dst, const std::vector<T> &v)
{
    size_t bytes = std::max<size_t>(v.size() * sizeof(T), 16);
    cudaError_t e = cudaMalloc(dst, bytes);
    if (e != cudaSuccess) {
        *dst = nullptr;
        return qs_fail(QS_ENOMEM, "batch upload: %s", cudaGetErrorString(e));
    }
    if (!v.empty() && (e = cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice)) != cudaSuccess)
        return qs_fail(QS_ECUDA, "batch upload: %s", cudaGetErrorString(e));
    return QS_OK;
}

int launch_batch(qs_batch *b, int C, int block)
{
    if (b->clear) {
        const cudaError_t e = cudaMemsetAsync(b->amp, 0, b->amp_bytes, (cudaStream_t)b->stream);
        if (e != cudaSuccess) return qs_fail(QS_ECUDA, "batch clear: %s", cudaGetErrorString(e));
    }
    for (size_t l = 0; l + 1 < b->level.size(); l++) {
        const size_t first = b->level[l], n = b->level[l + 1] - first;
        if (int rc = qs_launch_pass_items(b->dtype, b->passes, (const uint2 *)b->items + first, (uint32_t)n, b->amp, b->W, C,
                                          block, l > 0, b->stream))
            return rc;
    }
    return QS_OK;
}

bool valid_config(int C, int block)
{
    return (C == 1 || C == 2 || C == 4 || C == 8) && (block == 128 || block == 256 || block == 512);
}

}  // namespace

extern "C" int qs_batch_circuit_params(uint64_t seed, int *rows, int *cols, int *cz_cycles)
{
    return qs_guard([&]() -> int {
        if (!rows || !cols || !cz_cycles) return qs_fail(QS_EINVAL, "qs_batch_circuit_params: null output");
        static const int grids[3][2] = {{4, 4}, {4, 5}, {3, 7}};
        const uint64_t r = splitmix64(seed ^ 0x6A09E667F3BCC909ULL, 0);
        const int g = (int)(r % 3);
        *rows = grids[g][0];
        *cols = grids[g][1];
        *cz_cycles = 8 + (int)((r >> 32) % 33);
        return QS_OK;
    });
}

extern "C" int qs_batch_create(int n_circ, const qs_schedule *const *scheds, int dtype, void *stream, qs_batch **out)
{
    return qs_guard([&]() -> int {
        if (!out || n_circ < 1 || !scheds || (dtype != QS_C64 && dtype != QS_C128))
            return qs_fail(QS_EINVAL, "qs_batch_create: bad arguments");
        const size_t rsz = dtype == QS_C128 ? 8 : 4;
        std::vector<BatchCirc> circ(n_circ);
        std::vector<std::vector<qs_pass_in>> in(n_circ);   // operands as offsets into the pool
        std::vector<uint8_t> pool;
        qs_batch *b = new (std::nothrow) qs_batch();
        if (!b) return qs_fail(QS_ENOMEM, "qs_batch_create: out of host memory");
        struct Owner {   // until the batch is handed out
            qs_batch *b;
            ~Owner() { qs_batch_free(b); }
        } owner{b};
        b->dtype = dtype;
        b->n_circ = n_circ;
        b->stream = stream;
        uint64_t amp_total = 0;
        for (int c = 0; c < n_circ; c++) {
            const qs_schedule *sc = scheds[c];
            if (!sc || sc->n < 1 || sc->n > 26)
                return qs_fail(QS_EINVAL, "qs_batch_create: circuit %d must have 1..26 qubits", c);
            if (!sc->remap.empty()) return qs_fail(QS_EINVAL, "qs_batch_create: circuit %d has a remapped schedule", c);
            circ[c].n = sc->n;
            circ[c].amp_off = (int64_t)amp_total;
            b->nq.push_back(sc->n);
            b->amp_off.push_back(amp_total);
            amp_total += ((1ULL << sc->n) + 31) & ~31ULL;   // 256-byte aligned states
            for (const qs_op_host &op : sc->ops) {
                const size_t at = (pool.size() + 255) & ~(size_t)255;
                int n_act = 0;
                if (op.kind == QS_OP_DENSE) {
                    pool.resize(at + op.matrix.size() * rsz);
                    for (size_t i = 0; i < op.matrix.size(); i++) {
                        if (dtype == QS_C128) std::memcpy(pool.data() + at + 8 * i, &op.matrix[i], 8);
                        else {
                            float f = (float)op.matrix[i];
                            std::memcpy(pool.data() + at + 4 * i, &f, 4);
                        }
                    }
                } else if (op.kind == QS_OP_PHASE) {
                    std::vector<uint8_t> ph = qs_pack_phase(sc->n, op.coeff, op.edges, &n_act);
                    pool.resize(at + ph.size());
                    std::memcpy(pool.data() + at, ph.data(), ph.size());
                } else {
                    return qs_fail(QS_EUNSUPPORTED, "qs_batch_create: table diagonals are not batched");
                }
                in[c].push_back({op.kind, op.k, n_act, op.qubits, at, (uint32_t)(pool.size() - at), &op});
            }
        }
        int rc = QS_OK;
        b->amp_bytes = amp_total * 2 * rsz;
        cudaError_t e = cudaMalloc(&b->amp, b->amp_bytes);
        if (e != cudaSuccess) return qs_fail(QS_ENOMEM, "qs_batch_create: states: %s", cudaGetErrorString(e));
        if ((rc = upload(&b->pool, pool))) return rc;
        // the largest chunks (fewest passes) that still give every SM two or more
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        b->W = qs_pass_bits(dtype);
        while (b->W > 9 && (amp_total >> b->W) < 2 * (uint64_t)sms) b->W--;
        std::vector<qs_pass> passes;
        std::vector<std::vector<uint2>> levels;
        for (int c = 0; c < n_circ; c++) {
            for (qs_pass_in &op : in[c]) op.data += (uint64_t)(uintptr_t)b->pool;
            const std::vector<qs_pass> plan = qs_plan_passes(circ[c].n, dtype, b->W, in[c], true);
            for (size_t l = 0; l < plan.size(); l++) {
                if (levels.size() <= l) levels.emplace_back();
                const uint32_t chunks = 1u << __builtin_popcountll(plan[l].outer);
                for (uint32_t ch = 0; ch < chunks; ch++) levels[l].push_back(make_uint2((uint32_t)passes.size(), ch));
                passes.push_back(plan[l]);
                passes.back().amp = circ[c].amp_off;
            }
            const qs_pass &last = passes.back();
            if ((last.support | last.local) != qs_index_mask(circ[c].n)) b->clear = true;
        }
        std::vector<uint2> items;
        for (const std::vector<uint2> &l : levels) {
            b->level.push_back(items.size());
            items.insert(items.end(), l.begin(), l.end());
        }
        b->level.push_back(items.size());
        if (!rc) rc = upload(&b->passes, passes);
        if (!rc) rc = upload(&b->items, items);
        if (!rc) rc = upload(&b->circ, circ);
        std::vector<int2> sblk;
        std::vector<int> sfirst;
        for (int c = 0; c < n_circ; c++) {
            sfirst.push_back((int)sblk.size());
            const int parts = 1 << std::max(0, circ[c].n - kStatsBits);
            for (int p = 0; p < parts; p++) sblk.push_back(make_int2(c, p));
        }
        sfirst.push_back((int)sblk.size());
        b->n_sblk = (int)sblk.size();
        if (!rc) rc = upload(&b->sblk, sblk);
        if (!rc) rc = upload(&b->sfirst, sfirst);
        if (!rc && ((e = cudaMalloc(&b->stats, sizeof(double) * 4 * n_circ)) != cudaSuccess ||
                    (e = cudaMalloc(&b->spart, sizeof(double) * 3 * sblk.size())) != cudaSuccess ||
                    (e = cudaMalloc(&b->slog, sizeof(qsd::LogTable))) != cudaSuccess))
            rc = qs_fail(QS_ENOMEM, "qs_batch_create: stats: %s", cudaGetErrorString(e));
        if (!rc) {
            k_log_table<<<1, 256, 0, (cudaStream_t)stream>>>((qsd::LogTable *)b->slog);
            if ((e = cudaGetLastError()) != cudaSuccess) rc = qs_fail(QS_ECUDA, "qs_batch_create: %s", cudaGetErrorString(e));
        }
        if (rc) return rc;
        *out = b;
        owner.b = nullptr;
        return QS_OK;
    });
}

extern "C" void qs_batch_free(qs_batch *b)
{
    if (!b) return;
    if (b->amp) {
        if (b->stream) cudaStreamSynchronize((cudaStream_t)b->stream);
        else cudaDeviceSynchronize();
    }
    if (b->exec) cudaGraphExecDestroy(b->exec);
    for (void *p : {b->amp, b->passes, b->items, b->circ, b->pool, b->stats, b->sblk, b->sfirst, b->spart, b->slog})
        if (p) cudaFree(p);
    delete b;
}

extern "C" int qs_batch_set_config(qs_batch *b, int cluster_ctas, int threads)
{
    return qs_guard([&]() -> int {
        if (!b || !valid_config(cluster_ctas, threads)) return qs_fail(QS_EINVAL, "qs_batch_set_config");
        b->cluster = cluster_ctas;
        b->block = threads;
        return QS_OK;
    });
}

extern "C" int qs_batch_get_config(const qs_batch *b, int *cluster_ctas, int *threads)
{
    return qs_guard([&]() -> int {
        if (!b || !cluster_ctas || !threads) return qs_fail(QS_EINVAL, "qs_batch_get_config");
        *cluster_ctas = b->cluster;
        *threads = b->block;
        return QS_OK;
    });
}

extern "C" int qs_batch_run(qs_batch *b)
{
    return qs_guard([&]() -> int {
        if (!b) return qs_fail(QS_EINVAL, "qs_batch_run: null batch");
        return launch_batch(b, b->cluster, b->block);
    });
}

extern "C" int qs_batch_run_graph(qs_batch *b)
{
    return qs_guard([&]() -> int {
        if (!b) return qs_fail(QS_EINVAL, "qs_batch_run_graph: null batch");
        cudaStream_t st = (cudaStream_t)b->stream;
        if (!st) return qs_fail(QS_EINVAL, "qs_batch_run_graph: needs a non-default stream");
        if (!b->exec || b->exec_cluster != b->cluster || b->exec_block != b->block) {
            if (b->exec) {
                cudaGraphExecDestroy(b->exec);
                b->exec = nullptr;
            }
            cudaGraph_t g = nullptr;
            cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
            if (e != cudaSuccess) return qs_fail(QS_ECUDA, "graph capture: %s", cudaGetErrorString(e));
            int rc = launch_batch(b, b->cluster, b->block);
            e = cudaStreamEndCapture(st, &g);
            if (rc) {
                if (g) cudaGraphDestroy(g);
                return rc;
            }
            if (e != cudaSuccess) return qs_fail(QS_ECUDA, "graph capture: %s", cudaGetErrorString(e));
            e = cudaGraphInstantiate(&b->exec, g, 0);
            cudaGraphDestroy(g);
            if (e != cudaSuccess) {
                b->exec = nullptr;
                return qs_fail(QS_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
            }
            b->exec_cluster = b->cluster;
            b->exec_block = b->block;
        }
        cudaError_t e = cudaGraphLaunch(b->exec, st);
        return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "graph launch: %s", cudaGetErrorString(e));
    });
}

extern "C" int qs_batch_stats(qs_batch *b, double *out)
{
    return qs_guard([&]() -> int {
        if (!b || !out) return qs_fail(QS_EINVAL, "qs_batch_stats: bad arguments");
        cudaStream_t st = (cudaStream_t)b->stream;
        const BatchCirc *circ = (const BatchCirc *)b->circ;
        const qsd::LogTable *log = (const qsd::LogTable *)b->slog;
        if (b->dtype == QS_C128)
            k_batch_stats<double><<<b->n_sblk, 256, 0, st>>>(circ, (const int2 *)b->sblk, log, (const double2 *)b->amp,
                                                             (double *)b->spart);
        else
            k_batch_stats<float><<<b->n_sblk, 256, 0, st>>>(circ, (const int2 *)b->sblk, log, (const float2 *)b->amp,
                                                            (double *)b->spart);
        k_batch_stats_final<<<b->n_circ, 32, 0, st>>>(circ, (const int *)b->sfirst, (const double *)b->spart, (double *)b->stats);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(out, b->stats, sizeof(double) * 4 * b->n_circ, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "qs_batch_stats: %s", cudaGetErrorString(e));
    });
}

extern "C" int qs_batch_get_amplitudes(qs_batch *b, int i, double *host)
{
    return qs_guard([&]() -> int {
        if (!b || !host || i < 0 || i >= b->n_circ) return qs_fail(QS_EINVAL, "qs_batch_get_amplitudes: bad arguments");
        const uint64_t N = 1ULL << b->nq[i];
        cudaStream_t st = (cudaStream_t)b->stream;
        cudaError_t e;
        if (b->dtype == QS_C128) {
            e = cudaMemcpyAsync(host, (double2 *)b->amp + b->amp_off[i], 16 * N, cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        } else {
            std::vector<float> f(2 * N);
            e = cudaMemcpyAsync(f.data(), (float2 *)b->amp + b->amp_off[i], 8 * N, cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            for (uint64_t j = 0; j < 2 * N; j++) host[j] = f[j];
        }
        return e == cudaSuccess ? QS_OK : qs_fail(QS_ECUDA, "qs_batch_get_amplitudes: %s", cudaGetErrorString(e));
    });
}

// Time every launch configuration (cluster of 1, 2, 4, 8 CTAs x 128, 256, 512
// threads), keep the fastest in the batch and report it.
extern "C" int qs_batch_tune(qs_batch *b, int *cluster_ctas, int *threads, float *ms)
{
    return qs_guard([&]() -> int {
        if (!b) return qs_fail(QS_EINVAL, "qs_batch_tune: null batch");
        cudaStream_t st = (cudaStream_t)b->stream;
        cudaEvent_t e0, e1;
        if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
            return qs_fail(QS_ECUDA, "qs_batch_tune: events");
        float best = 1e30f;
        int bc = 1, bt = 256, rc = QS_OK;
        for (int C : {1, 2, 4, 8})
            for (int T : {128, 256, 512}) {
                if ((rc = launch_batch(b, C, T))) break;   // warm-up
                cudaEventRecord(e0, st);
                for (int r = 0; r < 2 && !rc; r++) rc = launch_batch(b, C, T);
                cudaEventRecord(e1, st);
                if (cudaEventSynchronize(e1) != cudaSuccess) {
                    rc = qs_fail(QS_ECUDA, "qs_batch_tune: sync");
                    break;
                }
                float t = 0;
                cudaEventElapsedTime(&t, e0, e1);
                t /= 2;
                if (t < best) {
                    best = t;
                    bc = C;
                    bt = T;
                }
            }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        if (rc) return rc;
        b->cluster = bc;
        b->block = bt;
        if (cluster_ctas) *cluster_ctas = bc;
        if (threads) *threads = bt;
        if (ms) *ms = best;
        return QS_OK;
    });
}

// Autotune the whole batched path: schedules with k_max in {3, 4, 5}, each
// batch tuned over its launch configurations; the fastest triple is returned.
extern "C" int qs_batch_autotune(int n_circ, const int *n_qubits, const qs_gate *const *gates, const int *n_gates,
                                 int dtype, void *stream, int *k_max, int *cluster_ctas, int *threads, float *ms)
{
    return qs_guard([&]() -> int {
        if (n_circ < 1 || !n_qubits || !gates || !n_gates || !k_max || !cluster_ctas || !threads)
            return qs_fail(QS_EINVAL, "qs_batch_autotune: bad arguments");
        float best = 1e30f;
        int rc = QS_OK;
        for (int km : {3, 4, 5}) {
            std::vector<qs_schedule *> sc(n_circ, nullptr);
            qs_sched_opts o = {km, 1, 1, 0, 1, 1, 1, 1, 0};
            for (int c = 0; c < n_circ && !rc; c++) rc = qs_schedule_build(n_qubits[c], gates[c], n_gates[c], &o, &sc[c]);
            qs_batch *b = nullptr;
            if (!rc) rc = qs_batch_create(n_circ, sc.data(), dtype, stream, &b);
            int C = 1, T = 256;
            float t = 0;
            if (!rc) rc = qs_batch_tune(b, &C, &T, &t);
            if (!rc && t < best) {
                best = t;
                *k_max = km;
                *cluster_ctas = C;
                *threads = T;
            }
            qs_batch_free(b);
            for (qs_schedule *s : sc) qs_schedule_free(s);
            if (rc) return rc;
        }
        if (ms) *ms = best;
        return QS_OK;
    });
}
