// Persistent batched contraction and measurement: many independent chains,
// every site, in one launch.
//
// The kernel is the tcgen05 contraction of tc_contract.cu (TMA producer warp,
// MMA warp, four epilogue warps, two TMEM accumulators) with eight measurement
// warps in two groups, run over one task list: the tiles of every (job, chunk, site)
// segment in round order.  Each task looks up its segment (tensor maps in
// device memory, n-tile width, K extent, scratch pointers), so jobs with
// different bond dimensions, physical dimensions and row counts share the GPU
// in one launch; dependencies between consecutive sites of a job are kept per
// 128-row m-tile with counters in global memory.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "launch.h"
#include "measure.cuh"

namespace fastmps {

namespace {

constexpr int kBM = 128;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kAccStride = 256;
constexpr uint32_t kATileBytes = 16384;      // 128 rows x 128 bytes
constexpr uint32_t kBPlaneBytesMax = 32768;  // 256 rows x 128 bytes
constexpr int kMaxStages = 8;
constexpr int kSmemLimit = 232448;

__device__ __forceinline__ void record_error(int *err, volatile int *abort_flag, int code) {
    *abort_flag = 1;
    atomicCAS(err, 0, code);
}

__device__ __forceinline__ bool mbar_wait_drain(uint64_t *bar, uint32_t parity) {
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (global_ns() - t0 > 200000000ull) return false;
    }
    return true;
}

// ===========================================================================
// Persistent batched kernel: every round of every job in one launch.
//
// The tasks are the tiles of all segments of all rounds in round order.  The
// producer thread of each thread block takes the next task from a global
// counter (atomicAdd), so a block never waits on a task that no running block
// has taken: a task's predecessors come earlier in the order and have been
// taken already.  Before loading a task's left rows it waits -- bounded -- until
// the job's m-tile slot has been measured `step` times (the rows of chunk c at
// site k are written by the measurement of site k-1, and the chunk's scratch
// rows are free once the previous step's measurement has read them).  The
// epilogue stores the FP32 tile and its sums of squares and counts the finished
// tiles of the m-tile; the thread that counts the last one publishes the m-tile
// in the launch's measurement list.  Measurements are handed out like tasks: each
// group of four measurement warps takes the next 128 / parts rows of the list from a global
// counter, in the order of publication, waits (bounded) for them to be published,
// draws, writes the next left rows (Algorithm 2) and adds one to the slot's counter,
// `parts` for every step measured.  Warps: 0 TMA producer,
// 1 MMA issuer, 2-5 epilogue, 6-13 two measurement groups (448 threads).
//
// The list is what keeps a step short: the steps of a chain follow each other, and
// each takes as long as its slowest m-tile.  When the block that finished an m-tile's
// last tile also measured all of it (128 rows, 43 us), some block had several m-tiles
// waiting in every round and a round of 226 m-tiles took 200 us on 152 blocks.
// ===========================================================================
constexpr int kPThreads = 448;
constexpr int kTaskRing = 16;
constexpr int kPBarrierBytes = 3072;
constexpr int kMeasureRows = 32;                   // most rows of one measurement
constexpr int kMeasureGroups = 2;                  // groups of four warps per block
constexpr int kMeasureSums = 896;                  // (row, outcome) sums of a group in shared memory
constexpr int kPMeasureBytes = kMeasureGroups * kMeasureSums * 8;
constexpr int kPStageBytes = 4 * kYWarpBytes;      // scratch staging, one buffer per epilogue warp

struct PParams {
    const PSegment *segs;
    const MeasureArgs *meas;
    int nseg;
    int64_t total_tasks;
    unsigned long long *queue;
    int *measured, *tiles_done;
    unsigned long long *ready;  // [m-tiles of all segments]: (segment + 1) << 32 | m-tile, in order of completion
    int *ready_tail;            // entries published
    unsigned long long *measure_queue;  // next 32-row measurement
    int64_t total_measures;
    int parts;                  // measurements of an m-tile: 128 / parts rows each
    int stages, a_planes, b_planes, nprod;
    uint32_t prod_code, stage_bytes;
    uint64_t limit_ns;
    int stall;
    int *err;
};

// Last segment whose first task is <= t (segments ordered by task_begin).  A block takes tasks in
// increasing order, so the search gallops forward from the block's previous segment `from`.
__device__ __forceinline__ int psegment_of(const PParams &p, int64_t t, int from) {
    int lo = from, hi = from, step = 1;
    while (hi + 1 < p.nseg && p.segs[hi + 1].task_begin <= t) {
        lo = hi + 1;
        hi = hi + step < p.nseg - 1 ? hi + step : p.nseg - 1;
        step <<= 1;
        if (p.segs[hi].task_begin > t) break;
        lo = hi;
    }
    if (p.segs[hi].task_begin <= t) return hi;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.segs[mid].task_begin <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Bounded wait for *cnt >= target (GPU-scope acquire).  Gives up early when any block has recorded
// an error; returns false then or when the limit runs out (*timed_out says which).
__device__ __forceinline__ bool wait_counter(const int *cnt, int target, const PParams &p, bool *timed_out) {
    *timed_out = false;
    if (ld_acquire_gpu(cnt) >= target) return true;
    const uint64_t t0 = global_ns();
    uint32_t iter = 0;
    while (ld_acquire_gpu(cnt) < target) {
        __nanosleep(100);
        if (((++iter) & 31u) == 0u) {
            if (*reinterpret_cast<volatile int *>(p.err) != 0) return false;
            if (global_ns() - t0 > p.limit_ns) {
                *timed_out = true;
                return false;
            }
        }
    }
    return true;
}

// As wait_counter, for a published entry of the measurement list (non-zero).
__device__ __forceinline__ bool wait_entry(const unsigned long long *entry, const PParams &p, unsigned long long *e,
                                           bool *timed_out) {
    *timed_out = false;
    if ((*e = ld_acquire_gpu(entry)) != 0) return true;
    const uint64_t t0 = global_ns();
    uint32_t iter = 0;
    while ((*e = ld_acquire_gpu(entry)) == 0) {
        __nanosleep(100);
        if (((++iter) & 31u) == 0u) {
            if (*reinterpret_cast<volatile int *>(p.err) != 0) return false;
            if (global_ns() - t0 > p.limit_ns) {
                *timed_out = true;
                return false;
            }
        }
    }
    return true;
}

__global__ void __launch_bounds__(kPThreads, 1) tc_batch_persistent_kernel(const PParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);
    uint8_t *ystage = smem + (size_t)p.stages * p.stage_bytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(ystage + kPStageBytes);
    uint64_t *empty = full + p.stages;
    uint64_t *tfull = empty + p.stages;
    uint64_t *tempty = tfull + 2;
    uint64_t *drain = tempty + 2;
    uint64_t *task_full = drain + 1;            // [kTaskRing] task published by the producer
    uint64_t *task_empty = task_full + kTaskRing;  // [kTaskRing] read by the MMA thread and the epilogue
    int64_t *task_id = reinterpret_cast<int64_t *>(task_empty + kTaskRing);  // [kTaskRing]
    int *task_seg = reinterpret_cast<int *>(task_id + kTaskRing);           // [kTaskRing]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(task_seg + kTaskRing);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    int *m_now = reinterpret_cast<int *>(tmem_slot + 4);             // [group][segment or -1, m-tile, part]
    int *m_sstar = m_now + 4 * kMeasureGroups;                       // [group][32]
    float *m_scale = reinterpret_cast<float *>(m_sstar + 32 * kMeasureGroups);  // [group][32]
    double *m_sums = reinterpret_cast<double *>(reinterpret_cast<uint8_t *>(full) + kPBarrierBytes);  // [group][kMeasureSums]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&tfull[0], 1);
        mbar_init(&tfull[1], 1);
        mbar_init(&tempty[0], 128);
        mbar_init(&tempty[1], 128);
        mbar_init(drain, 1);
        for (int r = 0; r < kTaskRing; ++r) {
            mbar_init(&task_full[r], 1);
            mbar_init(&task_empty[r], 2);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer: takes tasks, waits for their left rows ----------------
            int stage = 0;
            uint32_t phase = 0;
            int last_parity[kMaxStages];
            for (int s = 0; s < kMaxStages; ++s) last_parity[s] = -1;
            bool failed = false;
            int seg_cursor = 0;
            for (int64_t seq = 0; !failed; ++seq) {
                const int slot = (int)(seq % kTaskRing);
                const uint32_t tpar = (uint32_t)((seq / kTaskRing) & 1);
                if (!mbar_wait_bounded(&task_empty[slot], tpar ^ 1u, abort_flag, p.limit_ns)) {
                    record_error(p.err, abort_flag, kDevTimeoutProducer);
                    break;
                }
                const int64_t t = (int64_t)atomicAdd(p.queue, 1ull);
                if (t >= p.total_tasks) {
                    task_id[slot] = -1;
                    mbar_arrive(&task_full[slot]);
                    break;
                }
                const int si = psegment_of(p, t, seg_cursor);
                seg_cursor = si;
                const PSegment *sg = &p.segs[si];
                const int64_t lt = t - sg->task_begin;
                const int mt = (int)(lt / sg->num_n_tiles);
                const int nt = (int)(lt - (int64_t)mt * sg->num_n_tiles);
                const int target = (sg->step + p.stall) * p.parts;
                if (target > 0) {
                    bool timed_out;
                    if (!wait_counter(p.measured + sg->slot_base + mt, target, p, &timed_out)) {
                        if (timed_out) record_error(p.err, abort_flag, kDevTimeoutDependency);
                        else *abort_flag = 1;
                        break;
                    }
                    // the rows were written through the generic proxy by another block: order them
                    // before this thread's tensor-memory-access (async proxy) loads
                    fence_proxy_async_global();
                }
                task_id[slot] = t;
                task_seg[slot] = si;
                mbar_arrive(&task_full[slot]);
                const int y_a = sg->row0 + mt * kBM;
                const int y_b = nt * sg->bn;
                for (int kb = 0; kb < sg->num_k_blocks; ++kb) {
                    if (!mbar_wait_bounded(&empty[stage], phase ^ 1u, abort_flag, p.limit_ns)) {
                        record_error(p.err, abort_flag, kDevTimeoutProducer);
                        failed = true;
                        break;
                    }
                    uint8_t *sbase = smem + (size_t)stage * p.stage_bytes;
                    mbar_arrive_expect_tx(&full[stage], sg->tx_bytes);
                    const int x = kb * 64;
                    for (int a = 0; a < p.a_planes; ++a)
                        tma_load_2d(sbase + a * kATileBytes, &sg->tmA[a], &full[stage], x, y_a);
                    uint8_t *bbase = sbase + (size_t)p.a_planes * kATileBytes;
                    for (int b = 0; b < p.b_planes; ++b)
                        tma_load_2d(bbase + b * kBPlaneBytesMax, &sg->tmB[b], &full[stage], x, y_b);
                    last_parity[stage] = (int)phase;
                    if (++stage == p.stages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (*abort_flag)
                for (int s = 0; s < p.stages; ++s)
                    if (last_parity[s] >= 0) mbar_wait_drain(&full[s], (uint32_t)last_parity[s]);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // ---------------- MMA issuer ----------------
            int stage = 0;
            uint32_t phase = 0;
            bool issued = false;
            for (int64_t seq = 0;; ++seq) {
                const int slot = (int)(seq % kTaskRing);
                if (!mbar_wait_bounded(&task_full[slot], (uint32_t)((seq / kTaskRing) & 1), abort_flag,
                                       p.limit_ns)) {
                    record_error(p.err, abort_flag, kDevTimeoutMma);
                    break;
                }
                const int64_t t = task_id[slot];
                const int si = task_seg[slot];
                mbar_arrive(&task_empty[slot]);
                if (t < 0) break;
                const PSegment *sg = &p.segs[si];
                const int buf = (int)(seq & 1);
                const uint32_t use = (uint32_t)(seq >> 1);
                if (!mbar_wait_bounded(&tempty[buf], (use & 1u) ^ 1u, abort_flag, p.limit_ns)) {
                    record_error(p.err, abort_flag, kDevTimeoutMma);
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)buf * kAccStride;
                const uint32_t idesc = sg->idesc;
                bool failed = false;
                for (int kb = 0; kb < sg->num_k_blocks; ++kb) {
                    if (!mbar_wait_bounded(&full[stage], phase, abort_flag, p.limit_ns)) {
                        record_error(p.err, abort_flag, kDevTimeoutMma);
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem + (size_t)stage * p.stage_bytes);
                    const uint32_t sb = sa + (uint32_t)p.a_planes * kATileBytes;
                    for (int q = 0; q < p.nprod; ++q) {
                        const uint32_t pa = (p.prod_code >> (4 * q)) & 3u;
                        const uint32_t pb = (p.prod_code >> (4 * q + 2)) & 3u;
                        const uint64_t ad = sw128_kmajor_desc(sa + pa * kATileBytes);
                        const uint64_t bd = sw128_kmajor_desc(sb + pb * kBPlaneBytesMax);
#pragma unroll
                        for (int k16 = 0; k16 < 4; ++k16)
                            tc_mma_bf16(d_tmem, ad + (uint64_t)(2 * k16), bd + (uint64_t)(2 * k16), idesc,
                                        (kb | q | k16) != 0 ? 1u : 0u);
                    }
                    issued = true;
                    tc_commit(&empty[stage]);
                    if (++stage == p.stages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (failed) break;
                tc_commit(&tfull[buf]);
            }
            if (*abort_flag && issued) {
                tc_commit(drain);
                mbar_wait_drain(drain, 0u);
            }
        }
        __syncwarp();
    } else if (warp < 6) {
        // ---------------- epilogue: warps 2..5 ----------------
        const int quad = warp & 3;
        for (int64_t seq = 0;; ++seq) {
            const int slot = (int)(seq % kTaskRing);
            const bool got = mbar_wait_bounded(&task_full[slot], (uint32_t)((seq / kTaskRing) & 1), abort_flag,
                                               p.limit_ns);
            if (named_bar_any(1, 128, !got)) {
                record_error(p.err, abort_flag, kDevTimeoutEpilogue);
                break;
            }
            const int64_t t = task_id[slot];
            const int si = task_seg[slot];
            named_bar_sync(1, 128);  // every thread has read the slot
            if (threadIdx.x == 64) mbar_arrive(&task_empty[slot]);
            if (t < 0) break;
            const PSegment *sg = &p.segs[si];
            const int64_t lt = t - sg->task_begin;
            const int mt = (int)(lt / sg->num_n_tiles);
            const int nt = (int)(lt - (int64_t)mt * sg->num_n_tiles);
            const int buf = (int)(seq & 1);
            const uint32_t use = (uint32_t)(seq >> 1);
            const bool ready = mbar_wait_bounded(&tfull[buf], use & 1u, abort_flag, p.limit_ns);
            if (named_bar_any(1, 128, !ready)) {
                record_error(p.err, abort_flag, kDevTimeoutEpilogue);
                break;
            }
            tc_fence_after();
            const int row = mt * kBM + quad * 32 + lane;
            const bool valid = row < sg->rows_valid;
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)buf * kAccStride;
            float ss = 0.f;
            const int nch = sg->bn / 32, x0 = nt * sg->bn, y0 = mt * kBM + quad * 32, rows_valid = sg->rows_valid;
            uint8_t *stage = ystage + (uint32_t)quad * kYWarpBytes;
            auto put_chunk = [&](const uint32_t (&r)[32], int ch) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float v = __uint_as_float(r[j]);
                    ss = fmaf(v, v, ss);
                }
                stage_and_store(&sg->tmY, stage, r, lane, x0 + ch * 32, y0, rows_valid, false);
            };
            // the next 32 columns are on their way from tensor memory while a chunk is squared and staged
            uint32_t ra[32], rb[32];
            tmem_ld_32x32b_x32(taddr, ra);
            tc_wait_ld_for(ra);
            for (int ch = 0; ch < nch; ch += 2) {
                const bool two = ch + 1 < nch, more = ch + 2 < nch;
                if (two) tmem_ld_32x32b_x32(taddr + (uint32_t)((ch + 1) * 32), rb);
                put_chunk(ra, ch);
                if (!two) break;
                tc_wait_ld_for(rb);
                if (more) tmem_ld_32x32b_x32(taddr + (uint32_t)((ch + 2) * 32), ra);
                put_chunk(rb, ch + 1);
                if (more) tc_wait_ld_for(ra);
            }
            tc_fence_before();
            mbar_arrive(&tempty[buf]);
            if (valid) sg->P[(int64_t)row * sg->ldP + nt] = ss;
            // count the tile once its scratch stores are complete; the m-tile's last tile puts it on the
            // measurement list
            if (lane == 0) bulk_wait_all();
            named_bar_sync(1, 128);
            if (threadIdx.x == 64) {
                __threadfence();  // the group's stores (ordered by the barrier) before the count
                const int old = atomicAdd(p.tiles_done + sg->done_base + mt, 1);
                if (old == sg->num_n_tiles - 1) {
                    __threadfence();  // every block's tiles of this m-tile before the measurement reads them
                    const int at = atomicAdd(p.ready_tail, 1);
                    st_release_gpu(p.ready + at, (unsigned long long)(si + 1) << 32 | (unsigned)mt);
                }
            }
            __syncwarp();
        }
    } else {
        // ---------------- measurement: warps 6..9 and 10..13, each group on its own ----------------
        const int g = (warp - 6) >> 2;
        const int m = threadIdx.x - 192 - 128 * g;  // thread of the group
        int *now = m_now + 4 * g, *sstar = m_sstar + 32 * g;
        float *scale = m_scale + 32 * g;
        double *sums = m_sums + kMeasureSums * g;
        while (true) {
            if (m == 0) {
                int si = -1;
                const int64_t q = (int64_t)atomicAdd(p.measure_queue, 1ull);
                if (q < p.total_measures) {
                    unsigned long long e = 0;
                    bool timed_out;
                    if (wait_entry(p.ready + q / p.parts, p, &e, &timed_out)) {
                        si = (int)(e >> 32) - 1;
                        now[1] = (int)(unsigned)e;
                        now[2] = (int)(q % p.parts);
                    } else if (timed_out) {
                        record_error(p.err, abort_flag, kDevTimeoutMeasure);
                    }
                }
                now[0] = si;
            }
            named_bar_sync(2 + g, 128);
            const int si = now[0];
            if (si < 0) break;
            const int mt = now[1];
            const MeasureArgs &a = p.meas[si];
            const int part_rows = kBM / p.parts;
            const int r0 = mt * kBM + now[2] * part_rows;
            const int count = min(part_rows, p.segs[si].rows_valid - r0);
            const int d = a.d, T = a.tiles_per_s;
            const bool in_smem = d * part_rows <= kMeasureSums;
            if (in_smem) {
                for (int e = m; e < count * d; e += 128) {
                    const int r = e / d;
                    sums[e] = sum_tiles(a.P + (int64_t)(r0 + r) * a.ldP + (e - r * d) * T, T);
                }
                named_bar_sync(2 + g, 128);
            }
            double Z = 0.0, ws = 0.0;
            bool ok = false;
            const RowSums w{in_smem ? sums + m * d : nullptr, a.P + (int64_t)(r0 + m) * a.ldP, d, T};
            if (m < count) {
                const int s = draw_row(w, sample_uniform(a.seed, a.n_base + (uint64_t)(r0 + m), a.k, a.job), &Z, &ws, &ok);
                sstar[m] = s;
                scale[m] = ok ? rsqrtf((float)ws) : 0.f;
                a.outcomes[r0 + m] = (uint8_t)s;
            }
            named_bar_sync(2 + g, 128);
            // the logarithm (before the rows are released: the next step adds to the same entry)
            if (m < count) measure_finish(a, r0 + m, ws, Z, ok, __ldcg(a.logp + a.row0 + r0 + m), w);
            write_rows_flat<4>(a, m, 128, r0, count, sstar, scale);
            named_bar_sync(2 + g, 128);  // the next left rows are written
            if (m == 0) {
                fence_proxy_async_global();
                red_release_add_gpu(p.measured + p.segs[si].slot_base + mt, 1);
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace

cudaError_t prepare_batch_persistent() {
    return cudaFuncSetAttribute(tc_batch_persistent_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
}

cudaError_t launch_batch_persistent(const PersistentArgs &g, int num_sms, int *d_err, cudaStream_t st) {
    if (g.nseg <= 0 || g.total_tasks <= 0) return cudaSuccess;
    if (g.parts < kBM / kMeasureRows || kBM % g.parts != 0) return cudaErrorInvalidValue;
    if (g.nprod < 1 || g.nprod > kMaxProducts || g.a_planes < 1 || g.a_planes > 3 || g.b_planes < 1 ||
        g.b_planes > 2)
        return cudaErrorInvalidValue;
    PParams p;
    p.segs = g.segs;
    p.meas = g.meas;
    p.nseg = g.nseg;
    p.total_tasks = g.total_tasks;
    p.queue = reinterpret_cast<unsigned long long *>(g.queue);
    p.measured = g.measured;
    p.tiles_done = g.tiles_done;
    p.ready = reinterpret_cast<unsigned long long *>(g.ready);
    p.ready_tail = g.ready_tail;
    p.measure_queue = reinterpret_cast<unsigned long long *>(g.measure_queue);
    p.parts = g.parts;
    p.total_measures = g.total_m_tiles * g.parts;
    p.a_planes = g.a_planes;
    p.b_planes = g.b_planes;
    p.nprod = g.nprod;
    p.prod_code = 0;
    for (int q = 0; q < g.nprod; ++q)
        p.prod_code |= ((uint32_t)g.prod_a[q] | ((uint32_t)g.prod_b[q] << 2)) << (4 * q);
    p.stage_bytes = (uint32_t)g.a_planes * kATileBytes + (uint32_t)g.b_planes * kBPlaneBytesMax;
    p.stages = (kSmemLimit - 1024 - kPBarrierBytes - kPMeasureBytes - kPStageBytes) / (int)p.stage_bytes;
    if (p.stages > kMaxStages) p.stages = kMaxStages;
    if (p.stages < 2) return cudaErrorInvalidConfiguration;
    p.limit_ns = g.wait_limit_ns;
    p.stall = g.stall_test ? 1 : 0;
    p.err = d_err;
    const size_t smem = (size_t)p.stages * p.stage_bytes + 1024 + kPBarrierBytes + kPMeasureBytes + kPStageBytes;
    const int grid = g.total_tasks < num_sms ? (int)g.total_tasks : num_sms;
    tc_batch_persistent_kernel<<<grid, kPThreads, smem, st>>>(p);
    return cudaGetLastError();
}


}  // namespace fastmps
