// batch.cu -- many independent joins in a few launches (hj_join_batch).
//
// Every join partitions on the radix bits that its build size calls for (2048 4-byte or
// 1024 8-byte build tuples per partition at most while 2^11 digits do, at least one bit
// so that every partition is padded and filtered the same way).  Two launches partition
// all relations of all joins at once (one histogram, one scatter over their chunks, each
// relation read in place), one lists the partition pairs, and ONE persistent launch of
// the shared-memory join kernel runs every (join, partition) task, taking tasks from a
// work counter so that joins of very different sizes share the GPU.  The chunk tables
// are made on the host and travel in one copy; the pair buffers are allocated while the
// partitioning runs.  Pairs are placed by exact per-task claims into each join's own
// buffer (the staging sinks), so no compaction is needed.  When the workspace of all
// joins would exceed the HBM budget, joins run in waves.  With four launches to a wave
// there is nothing left for a CUDA graph to shorten (capture and instantiation took
// longer than they saved), so HJ_FLAG_GRAPH changes nothing.
#include <algorithm>
#include <cmath>
#include <memory>
#include <vector>

#include "common.cuh"
#include "emit.cuh"
#include "engine.cuh"

using namespace hj;

namespace {

int join_bits(int width, uint64_t nR) {
    int b = 1;
    while (b < 11 && (nR >> b) > batch_partition_rows(width)) b++;
    return b;
}

// A join of a wave: where its tasks start, and its relations' partition offsets.
struct BatchJoin {
    uint64_t task_at;
    uint64_t r_at, s_at;  // first offset of R's and of S's partitions
    uint32_t join;
    uint32_t bits;
};
struct BatchKeys {
    uint64_t ek1[12], pk1[12];  // by bits
};

// Partition pair i of the wave; its join is the last one whose tasks start at or
// before i.
__global__ void batch_tasks_kernel(const void *rows, const uint64_t *off, const BatchJoin *joins, uint64_t nj,
                                   uint64_t ntasks, BatchKeys keys, int tb, PartTask *tasks) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < ntasks; i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t lo = 0, hi = nj;  // joins[lo].task_at <= i < joins[hi].task_at
        while (hi - lo > 1) {
            const uint64_t mid = (lo + hi) >> 1;
            if (joins[mid].task_at <= i) lo = mid; else hi = mid;
        }
        const BatchJoin j = joins[lo];
        const uint64_t p = i - j.task_at;
        const uint64_t *ro = off + j.r_at + p, *so = off + j.s_at + p;
        PartTask t;
        t.R = (const char *)rows + ro[0] * tb;
        t.S = (const char *)rows + so[0] * tb;
        t.nr = (uint32_t)(ro[1] - ro[0]);
        t.ns = (uint32_t)(so[1] - so[0]);
        t.join = j.join;
        t.p = (uint32_t)p;
        t.b1 = (uint16_t)j.bits;
        t.b2 = 0;
        t.pad = 0;
        t.ek1 = keys.ek1[j.bits];
        t.pk1 = keys.pk1[j.bits];
        t.pk2 = 0;
        tasks[i] = t;
    }
}

// Device work of a wave, which lives until its oversize tasks are done.
struct Wave {
    DevBuf rows, off, tasks, oversize, chunks, joins, counts, totals;
    uint64_t ntasks = 0, nj = 0;
    uint64_t part_rows = 0;  // build rows of a mean partition (the largest), at least the usual ones
    explicit Wave(hj_ctx *c) : rows(c), off(c), tasks(c), oversize(c), chunks(c), joins(c), counts(c), totals(c) {}
};

template <class T> hj_status upload(hj_ctx *c, const std::vector<T> &v, DevBuf &out) {
    HJ_TRY(out.alloc(std::max<size_t>(v.size(), 1) * sizeof(T)));
    if (!v.empty()) HJ_CUDA(c, cudaMemcpyAsync(out.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, c->stream));
    return HJ_OK;
}

// Queue the partitioning of the joins `wj` (pageable host tables: a copy has taken
// them when it returns).
hj_status partition_wave(hj_ctx *c, int W, const hj_rel *Rs, const hj_rel *Ss, const std::vector<int> &wj, Wave &w) {
    const uint64_t tb = tuple_bytes(W), sv = 32 / tb;
    uint64_t total = 0;
    for (int j : wj) total += Rs[j].n + Ss[j].n;
    std::vector<BatchChunk> chunks;
    std::vector<BatchJoin> joins;
    uint64_t rows = 0, h_at = 0, t_at = 0;
    int max_bits = 1;
    bool too_large = false;
    auto relation = [&](const hj_rel &r, int bits) {
        const uint64_t P = 1ull << bits, step = batch_chunk_rows(c, total, bits), at = t_at;
        uint64_t n = 0;
        for (uint64_t lo = 0; lo < r.n; lo += step, ++n) {
            BatchChunk b;
            b.src = (const char *)r.tuples + lo * tb;
            b.obase = rows;
            b.h_at = h_at;
            b.t_at = at;
            b.n = (uint32_t)std::min(step, r.n - lo);
            b.bits = (uint16_t)bits;
            b.lead = lo == 0;
            chunks.push_back(b);
            h_at += P;
        }
        // (run offsets inside a relation are 32-bit)
        if (r.n + n * P * (sv - 1) >= 0xFFFFFFFFull) too_large = true;
        rows = (rows + r.n + n * P * (sv - 1) + 15) / 16 * 16;
        t_at += P + 1;
        return at;
    };
    for (int j : wj) {
        const int bits = join_bits(W, Rs[j].n);
        max_bits = std::max(max_bits, bits);
        w.part_rows = std::max<uint64_t>(w.part_rows, (Rs[j].n + (1ull << bits) - 1) >> bits);
        BatchJoin bj;
        bj.task_at = w.ntasks;
        bj.join = (uint32_t)j;
        bj.bits = (uint32_t)bits;
        bj.r_at = relation(Rs[j], bits);
        bj.s_at = relation(Ss[j], bits);
        joins.push_back(bj);
        w.ntasks += 1ull << bits;
    }
    if (too_large) return set_err(c, HJ_E_UNSUPPORTED, "a relation of a batch padded to whole sectors passes 2^32 rows");
    w.part_rows = std::max(w.part_rows, batch_partition_rows(W));
    w.nj = joins.size();
    HJ_TRY(upload(c, chunks, w.chunks));
    HJ_TRY(upload(c, joins, w.joins));
    HJ_TRY(w.rows.alloc(rows * tb + 64));
    HJ_TRY(w.off.alloc(t_at * 8));
    HJ_TRY(w.counts.alloc(h_at * 8));
    HJ_TRY(w.totals.alloc(t_at * 4));
    HJ_CUDA(c, cudaMemsetAsync(w.totals.p, 0, t_at * 4, c->stream));
    return batch_partition(c, W, w.chunks.as<BatchChunk>(), chunks.size(), max_bits, w.counts.as<uint32_t>(),
                           w.counts.as<uint32_t>() + h_at, w.totals.as<uint32_t>(), w.rows.p, w.off.as<uint64_t>());
}

hj_status join_wave(hj_ctx *c, int W, const JoinSlot *slots, bool agg, bool chk, Wave &w) {
    BatchKeys keys;
    keys.ek1[0] = keys.pk1[0] = 0;
    for (int b = 1; b < 12; ++b) {
        keys.ek1[b] = empty_key2(W, b, 0);
        keys.pk1[b] = pass_pad_key(W, 0, b);
    }
    HJ_TRY(w.tasks.alloc(std::max<uint64_t>(w.ntasks, 1) * sizeof(PartTask)));
    HJ_TRY(w.oversize.alloc(std::max<uint64_t>(w.ntasks, 1) * 4));
    const unsigned grid = (unsigned)std::min<uint64_t>((w.ntasks + 255) / 256, (uint64_t)num_sms(c) * 8);
    HJ_LAUNCH(c, "batch_tasks", batch_tasks_kernel, grid ? grid : 1, 256, 0, w.rows.p, w.off.as<uint64_t>(),
              w.joins.as<BatchJoin>(), w.nj, w.ntasks, keys, (int)tuple_bytes(W), w.tasks.as<PartTask>());
    return partition_join(c, W, agg, w.tasks.as<PartTask>(), w.ntasks, w.ntasks, slots, w.part_rows, chk,
                          w.oversize.as<uint32_t>(), RecArea{nullptr, nullptr, 0}, !agg);
}

bool is_agg(int mode) { return mode == HJ_COUNT || mode == HJ_COUNT_CHECKSUM; }

}  // namespace

extern "C" hj_status hj_join_batch(hj_ctx *c, int n, const hj_rel *Rs, const hj_rel *Ss, const hj_opts *opts,
                                   hj_result *outs) {
    if (!c) return HJ_E_INVALID;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_err(c, cudaGetLastError(), "cudaSetDevice");
    if (n < 0 || (n > 0 && (!Rs || !Ss || !outs))) return set_err(c, HJ_E_INVALID, "bad batch arguments");
    if (n == 0) return HJ_OK;
    hj_opts o{};
    o.mode = HJ_MATERIALIZE;
    if (opts) o = *opts;
    if (o.mode < HJ_COUNT || o.mode > HJ_MATERIALIZE) return set_err(c, HJ_E_INVALID, "bad mode %d", o.mode);
    const int W = Rs[0].width;
    for (int j = 0; j < n; ++j) {
        for (const hj_rel *r : {&Rs[j], &Ss[j]}) {
            if (r->width != W) return set_err(c, HJ_E_INVALID, "join %d: all relations of a batch share one width", j);
            if (r->n && (!r->tuples || ((uintptr_t)r->tuples & 15)))
                return set_err(c, HJ_E_INVALID, "join %d: tuples NULL or not 16-byte aligned", j);
            if (r->n >= 0xFFFFFFFFull) return set_err(c, HJ_E_INVALID, "join %d: relation too large for a batch", j);
        }
        outs[j] = hj_result{};
    }
    if (W != HJ_U32 && W != HJ_U64) return set_err(c, HJ_E_INVALID, "width %d is not 4 or 8", W);
    const bool agg = is_agg(o.mode), mat = o.mode == HJ_MATERIALIZE;
    const bool chk = o.mode == HJ_COUNT_CHECKSUM || (mat && (o.flags & HJ_FLAG_CHECKSUM));
    const uint64_t tb = tuple_bytes(W);

    // per-join output buffers and counters
    std::vector<uint64_t> cap(n, 0);
    std::vector<void *> pairs(n, nullptr);
    auto release_pairs = [&]() {
        for (int j = 0; j < n; ++j) dfree(c, pairs[j]);
    };
    // workspace per join: partitioned copies of R and S, and the pair buffer
    auto need = [&](int j) {
        uint64_t ws = (Rs[j].n + Ss[j].n) * tb * 11 / 10 + 8192 * tb;
        if (mat) ws += (Ss[j].n + 64) * tb;
        return ws;
    };
    // device memory that a wave may take: of what the context's pool holds reserved but
    // unused, and (asked for only when that is not enough) of the free device memory
    uint64_t total = 0;
    for (int j = 0; j < n; ++j)
        if (Rs[j].n && Ss[j].n) total += need(j);
    unsigned long long reserved = 0, used_pool = 0;  // the attributes are 64-bit
    cudaMemPoolGetAttribute(c->pool, cudaMemPoolAttrReservedMemCurrent, &reserved);
    cudaMemPoolGetAttribute(c->pool, cudaMemPoolAttrUsedMemCurrent, &used_pool);
    uint64_t avail = reserved > used_pool ? reserved - used_pool : 0;
    if ((uint64_t)(avail * 0.7) < total) {
        size_t freeb = 0, totalb = 0;
        cudaMemGetInfo(&freeb, &totalb);
        avail += freeb;
    }
    uint64_t budget = (uint64_t)(avail * 0.7);
    if (c->budget) budget = std::min<uint64_t>(budget, c->budget > c->in_use ? (c->budget - c->in_use) * 9 / 10 : 0);

    // waves
    std::vector<std::vector<int>> waves;
    {
        std::vector<int> cur;
        uint64_t used = 0;
        for (int j = 0; j < n; ++j) {
            if (!Rs[j].n || !Ss[j].n) continue;  // empty joins have no pairs
            const uint64_t w = need(j);
            if (!cur.empty() && used + w > budget) {
                waves.push_back(cur);
                cur.clear();
                used = 0;
            }
            cur.push_back(j);
            used += w;
        }
        if (!cur.empty()) waves.push_back(cur);
    }
    DevBuf ctrs(c), slots(c);
    HJ_TRY(ctrs.alloc((uint64_t)n * sizeof(hj_counters)));
    HJ_CUDA(c, cudaMemsetAsync(ctrs.p, 0, (uint64_t)n * sizeof(hj_counters), c->stream));
    std::vector<hj_counters> hc(n);
    bool have_hc = false;
    for (size_t k = 0; k < waves.size(); ++k) {
        const std::vector<int> &wj = waves[k];
        HJ_TRY(zero_counters(c));  // the work counter of the join launch
        Wave w(c);
        hj_status st = partition_wave(c, W, Rs, Ss, wj, w);
        // pair buffers of this wave's joins, while the device partitions
        std::vector<JoinSlot> hs(n, JoinSlot{nullptr, 0, nullptr, 0});
        for (int j : wj) {
            if (mat && st == HJ_OK) {
                cap[j] = (o.out_capacity ? o.out_capacity : Ss[j].n) + 64;
                pairs[j] = dalloc(c, cap[j] * tb, &st);
            }
            hs[j] = JoinSlot{pairs[j], cap[j], ctrs.as<hj_counters>() + j, 0};
        }
        if (st == HJ_OK) st = upload(c, hs, slots);
        if (st == HJ_OK) st = join_wave(c, W, slots.as<JoinSlot>(), agg, chk, w);
        if (st == HJ_OK && k + 1 == waves.size()) {  // the last wave's wait brings the joins' counters too
            if (cudaMemcpyAsync(hc.data(), ctrs.p, (uint64_t)n * sizeof(hj_counters), cudaMemcpyDeviceToHost,
                                c->stream) != cudaSuccess)
                st = set_err(c, HJ_E_CUDA, "reading the joins' counters");
            have_hc = true;
        }
        if (st == HJ_OK) st = read_counters(c);
        if (st == HJ_OK && c->h_ctr->n_oversize) {
            std::vector<JoinSlot> sh(n);
            for (int j = 0; j < n; ++j)
                sh[j] = JoinSlot{pairs[j], cap[j], ctrs.as<hj_counters>() + j, 0};
            st = oversize_fallback(c, W, agg, chk, w.tasks.as<PartTask>(), w.oversize.as<uint32_t>(),
                                   c->h_ctr->n_oversize, sh);
            if (st == HJ_OK) st = read_counters(c);
            have_hc = false;
        }
        if (st == HJ_OK && (c->h_ctr->status & (kStatusTableFull | kStatusTimeout)))
            st = set_err(c, HJ_E_CUDA, "a batch kernel reported status %llu", (unsigned long long)c->h_ctr->status);
        if (st != HJ_OK) {
            release_pairs();
            return st;
        }
    }
    if (!have_hc) {
        HJ_CUDA(c, cudaMemcpyAsync(hc.data(), ctrs.p, (uint64_t)n * sizeof(hj_counters), cudaMemcpyDeviceToHost, c->stream));
        HJ_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    for (int j = 0; j < n; ++j) {
        hj_result &r = outs[j];
        r.count = hc[j].count;
        r.checksum[0] = hc[j].c0;
        r.checksum[1] = hc[j].c1;
        r.width = W;
        r.algo = HJ_ALGO_PHJ;
        r.radix_bits = join_bits(W, Rs[j].n);
        r.passes = 1;
        r.pairs = mat ? pairs[j] : nullptr;
        r.pairs_cap = mat ? cap[j] : 0;
        if (!mat && pairs[j]) dfree(c, pairs[j]);
    }
    // joins with more pairs than their buffer: run again alone at the exact size
    if (mat) {
        for (int j = 0; j < n; ++j) {
            if (outs[j].count <= cap[j] || !Rs[j].n || !Ss[j].n) continue;
            dfree(c, outs[j].pairs);
            outs[j] = hj_result{};
            hj_opts oj = o;
            oj.algo = HJ_ALGO_AUTO;
            oj.flags &= ~(uint64_t)HJ_FLAG_GRAPH;
            oj.out_capacity = hc[j].count;
            hj_status st = hj_join(c, &Rs[j], &Ss[j], &oj, &outs[j]);
            if (st != HJ_OK) {
                for (int i = 0; i < n; ++i) hj_result_free(c, &outs[i]);
                return st;
            }
        }
    }
    return HJ_OK;
}
