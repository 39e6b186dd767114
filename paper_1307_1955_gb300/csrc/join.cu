// join.cu -- build and probe kernels (Alg. 1 steps b1-b4 and p1-p4).
//
//   * table_* : the simple hash join's table in global memory (SHJ), one table
//     shared by all CTAs (Sec. 3.3 prefers one shared table to one per processor).
//   * partition_join : Alg. 2's "apply SHJ on each partition pair" with the table
//     in shared memory; persistent CTAs take partition pairs from a work counter.
//
// Probing is warp-level: each warp streams its share of S in groups of 16-byte
// vectors (the next group is loaded before the current one is probed), looks
// every tuple up, and appends pairs through emit.cuh (no block barrier in the
// probe loop).  A probe key with several build matches (duplicate R keys) is
// walked by the whole warp, 32 consecutive slots at a time -- the GPU answer to
// the divergence that skew causes in steps b3/p3 (Sec. 3.3, workload divergence).
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "common.cuh"
#include "emit.cuh"
#include "engine.cuh"

namespace hj {

// ------------------------------------------------------------------ tuple loads
// Vectors of a warp's probe group (U per lane, lane-interleaved) of an array of n
// tuples, from vector g on; item e of vector u is x[u]'s e-th tuple.  Lanes past the
// end load nothing.  The last vector of a 4-byte relation with an odd number of
// tuples is read with one 8-byte load, so that no read passes the array end.
template <int W, int U> struct Group {
    using Vec = typename Tup<W>::Vec;
    static constexpr int PV = Tup<W>::kPerVec;
    static constexpr int IT = U * PV;
    Vec x[U];
    uint32_t valid;  // one bit per item
    __device__ __forceinline__ void load(const Vec *S, uint64_t g, uint64_t n) {
        const unsigned lane = threadIdx.x & 31;
        const uint64_t nvec = (n + PV - 1) / PV;
        const Vec *p = S + g + lane;
        if (g + 32 * U <= n / PV) {
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = ld_stream(p + 32 * u);
            valid = (1u << IT) - 1u;
            return;
        }
        valid = 0;
        if (g >= nvec) return;
        const uint32_t left = (uint32_t)(nvec - g), whole = (uint32_t)(n / PV - g);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t i = 32 * u + lane;
            if (i < whole) {
                x[u] = ld_stream(p + 32 * u);
                valid |= ((1u << PV) - 1u) << (u * PV);
            } else if (W == 4 && i < left) {
                if constexpr (W == 4) {
                    const uint2 y = *(const uint2 *)(p + 32 * u);
                    x[u] = make_uint4(y.x, y.y, 0u, 0u);
                }
                valid |= 1u << (u * PV);
            }
        }
    }
    __device__ __forceinline__ typename Tup<W>::U key(int i) const {
        if constexpr (W == 4) return i % 2 ? x[i / 2].z : x[i / 2].x;
        else return x[i].x;
    }
    __device__ __forceinline__ typename Tup<W>::U rid(int i) const {
        if constexpr (W == 4) return i % 2 ? x[i / 2].w : x[i / 2].y;
        else return x[i].y;
    }
};

// ----------------------------------------------------------------- table views
// The pair table of common.cuh: nb buckets of one 32-byte sector.
template <int W> struct PairTab {
    using U = typename Tup<W>::U;
    using PS = PairSlot<W>;
    static constexpr uint32_t G = kBucketSlots<W>;
    const typename PS::S *slots;
    uint32_t nb;
    unsigned long long n_allones;
    bool unique;  // no key twice (nor the all-ones key): a match ends the search

    __device__ __forceinline__ uint32_t home(U k) const { return pair_bucket<W>(key_hash<W>(k), nb); }
    __device__ __forceinline__ uint32_t next(uint32_t b) const { return b + 1 == nb ? 0 : b + 1; }
};

// Tuples per lane and probe group.
constexpr int kProbeItems = 2;
constexpr int kProbeCtas = 4;  // per SM

// Per-lane accumulators of a probing warp.
struct ProbeAcc {
    unsigned long long cnt = 0, c0 = 0, c1 = 0;
};

template <int W, bool CHK>
__device__ __forceinline__ void add_check(ProbeAcc &acc, bool has, typename Tup<W>::U rid_r, typename Tup<W>::U rid_s) {
    if (!CHK || !has) return;
    const uint64_t a = mix_a(rid_r), b = mix_b(rid_s);
    acc.c0 += a * b;
    acc.c1 += a + b;
}

// The whole warp emits every build match of probe key kk (probe rid ss).
template <int W, bool CHK>
__device__ __forceinline__ void coop_emit(const PairTab<W> &tab, typename Tup<W>::U kk, typename Tup<W>::U ss,
                                          OutState &st, const OutCtx &oc, ProbeAcc &acc) {
    using PS = PairSlot<W>;
    const unsigned lane = threadIdx.x & 31;
    const uint64_t cap = (uint64_t)tab.nb * PairTab<W>::G, b = (uint64_t)tab.home(kk) * PairTab<W>::G;
    for (uint64_t off = 0; off < cap; off += 32) {
        uint64_t idx = b + off + lane;
        if (idx >= cap) idx -= cap;
        const typename PS::S s = off + lane < cap ? tab.slots[idx] : PS::empty();
        bool end;
        const bool has = run_step<W>(s, &end) && PS::key(s) == kk;
        add_check<W, CHK>(acc, has, PS::rid(s), ss);
        warp_append<W>(st, oc, has, PS::rid(s), ss);
        if (end) break;
    }
    if (kk == Tup<W>::kAllOnes)
        for (unsigned long long i = 0; i < tab.n_allones; i += 32) {
            const bool has = i + lane < tab.n_allones;
            add_check<W, CHK>(acc, has, Tup<W>::kAllOnes, ss);
            warp_append<W>(st, oc, has, Tup<W>::kAllOnes, ss);
        }
}

// A probing warp's queue of runs that go on past a full bucket: the probe's key and
// rid and the run's next bucket.  Fewer than 32 entries wait when a group starts,
// and it adds at most its own items.
template <int W> struct RunQueue {
    using T = typename Tup<W>::U;
    static constexpr uint32_t N = 32 * (kProbeItems + 1);
    T k[N], r[N];
    uint32_t b[N];
};

// Queue the lanes with `on` (key, rid, next bucket); n is the queue's length.
template <int W>
__device__ __forceinline__ void push_runs(RunQueue<W> &q, uint32_t &n, bool on, typename Tup<W>::U k,
                                          typename Tup<W>::U r, uint32_t b) {
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (!m) return;
    if (on) {
        const uint32_t at = n + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
        q.k[at] = k;
        q.r[at] = r;
        q.b[at] = b;
    }
    n += __popc(m);
}

// The last n <= 32 entries (one per lane) take their next bucket: its matches are
// appended, and runs that go on are queued again.
template <int W, bool CHK>
__device__ __forceinline__ void drain_runs(const PairTab<W> &tab, RunQueue<W> &q, uint32_t &qn, uint32_t n,
                                           OutState &st, const OutCtx &oc, ProbeAcc &acc) {
    using T = typename Tup<W>::U;
    constexpr uint32_t G = PairTab<W>::G;
    const unsigned lane = threadIdx.x & 31;
    const bool on = lane < n;
    __syncwarp();
    qn -= n;
    const T k = on ? q.k[qn + lane] : T(0), r = on ? q.r[qn + lane] : T(0);
    const uint32_t b = on ? q.b[qn + lane] : 0;
    __syncwarp();  // read before the queue is refilled
    T bk[G], br[G];
    ld_bucket<W>(tab.slots, b, bk, br);
    bool any = false;
#pragma unroll
    for (uint32_t s = 0; s < G; ++s) {
        const bool has = on && bk[s] == k && (bk[s] & br[s]) != Tup<W>::kAllOnes;
        any |= has;
        add_check<W, CHK>(acc, has, br[s], r);
        warp_append<W>(st, oc, has, br[s], r);
    }
    push_runs<W>(q, qn, on && (bk[G - 1] & br[G - 1]) != Tup<W>::kAllOnes && !(tab.unique && any), k, r, tab.next(b));
}

// Probe one group against a pair table and append its pairs (FULL: every item of
// every lane is a tuple).  A probe is one random sector read from L2 (or HBM): the
// home buckets of all the lane's items are loaded before the first one is looked
// at.  The home bucket is searched without branches.  A run that goes on past it
// (its last slot is taken, a few per cent) is queued, and 32 of them take their next
// bucket together.
// What bounds it: the instructions of a tuple (about 140 thread instructions) and
// the L1 passes of its 32 scattered sectors per load, not DRAM.  2^24 tuples against
// 2^18 (all in L2) took 216 us slot by slot with a branch per slot, 106 us like this;
// 6e6 8-byte tuples against 1e6 took 163 us and 56 us.  Four items per lane, or five
// CTAs per SM for 8-byte tuples, measured slower (more sectors in flight than L1 has
// lines for), and so did buckets of 16 bytes (2.4 times: their runs go on too often).
template <int W, int U, bool CHK, bool FULL>
__device__ __forceinline__ void probe_group_pairs(const PairTab<W> &tab, const Group<W, U> &g, RunQueue<W> &q,
                                                  uint32_t &qn, OutState &st, const OutCtx &oc, ProbeAcc &acc) {
    using T = typename Tup<W>::U;
    constexpr int IT = Group<W, U>::IT;
    constexpr uint32_t G = PairTab<W>::G;
    constexpr T ones = Tup<W>::kAllOnes;
    const unsigned lane = threadIdx.x & 31;
    uint32_t cnt[IT], bkt[IT];
    T first[IT], k[IT], r[IT], bk[IT][G], br[IT][G];
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        k[i] = g.key(i);
        r[i] = g.rid(i);
        bkt[i] = tab.home(k[i]);  // (a bucket of the table whatever the key)
        ld_bucket<W>(tab.slots, bkt[i], bk[i], br[i]);
    }
    bool walk[IT], odd = false;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const bool live = FULL || ((g.valid >> i) & 1u);
        T f = br[i][G - 1];
        uint32_t c = bk[i][G - 1] == k[i];
#pragma unroll
        for (int s = (int)G - 2; s >= 0; --s) {
            const bool m = bk[i][s] == k[i];
            f = m ? br[i][s] : f;
            c += m;
        }
        first[i] = f;
        cnt[i] = live ? c : 0;
        walk[i] = live && (bk[i][G - 1] & br[i][G - 1]) != ones && !(tab.unique && c);
        odd |= live && (c > 1 || k[i] == ones);
    }
    odd = __any_sync(0xffffffffu, odd);
    if (odd) {  // several matches, or the key that empty slots hold too
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            if (k[i] == ones && (FULL || ((g.valid >> i) & 1u))) {
                uint32_t c = 0;
#pragma unroll
                for (int s = (int)G - 1; s >= 0; --s)
                    if (bk[i][s] == ones && br[i][s] != ones) {
                        first[i] = br[i][s];
                        ++c;
                    }
                if (tab.n_allones) {  // tuples kept beside the table
                    if (!c) first[i] = ones;
                    c += (uint32_t)min(tab.n_allones, 2ull);
                }
                cnt[i] = c;
            }
            if (cnt[i] > 1) walk[i] = false;  // (its whole run is walked below)
        }
    }
    if (CHK)
#pragma unroll
        for (int i = 0; i < IT; ++i) add_check<W, CHK>(acc, cnt[i] == 1, first[i], r[i]);
    warp_append_group<W, IT>(st, oc, cnt, first, r);
    if (odd)
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            unsigned multi = __ballot_sync(0xffffffffu, cnt[i] > 1);
            while (multi) {
                const int L = __ffs(multi) - 1;
                multi &= multi - 1;
                coop_emit<W, CHK>(tab, __shfl_sync(0xffffffffu, k[i], L), __shfl_sync(0xffffffffu, r[i], L), st, oc,
                                  acc);
            }
        }
#pragma unroll
    for (int i = 0; i < IT; ++i) push_runs<W>(q, qn, walk[i], k[i], r[i], tab.next(bkt[i]));
    while (qn >= 32) drain_runs<W, CHK>(tab, q, qn, 32, st, oc, acc);
}

// Probe one group against an aggregate table: the home slots of all the lane's
// items are loaded before the first one is looked at; runs that go on are walked
// one by one.
template <int W, int U, bool CHK>
__device__ __forceinline__ void probe_group_agg(const AggSlot<W> *slots, uint64_t cap, const TableSide *side,
                                                const Group<W, U> &g, const PartFilter &pf, ProbeAcc &acc) {
    using T = typename Tup<W>::U;
    constexpr int IT = Group<W, U>::IT;
    AggSlot<W> s[IT];
    uint64_t h[IT];
    auto ld = [&](uint64_t at) {
        AggSlot<W> x;
        if constexpr (W == 4) {
            const ulonglong2 y = __ldg((const ulonglong2 *)slots + at);
            x.key = (uint32_t)y.x;
            x.cnt = (uint32_t)(y.x >> 32);
            x.suma = y.y;
        } else {
            unsigned long long pad;
            asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
                         : "=l"(x.key), "=l"(x.cnt), "=l"(x.suma), "=l"(pad)
                         : "l"(slots + at));
        }
        return x;
    };
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        h[i] = key_hash<W>(g.key(i));
        s[i] = ld(bucket_of<W>(h[i], cap));  // (a slot of the table whatever the key)
    }
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        if (!((g.valid >> i) & 1u) || !pf.keep(h[i])) continue;
        const T k = g.key(i);
        uint64_t n = 0, sa = 0;
        if (k == Tup<W>::kAllOnes) {
            n = side->agg_cnt;
            sa = side->agg_suma;
        } else {
            uint64_t b = bucket_of<W>(h[i], cap);
            for (uint64_t it = 1; s[i].key != k && s[i].key != Tup<W>::kAllOnes && it < cap; ++it) {
                if (++b == cap) b = 0;
                s[i] = ld(b);
            }
            if (s[i].key == k) {
                n = s[i].cnt;
                sa = s[i].suma;
            }
        }
        acc.cnt += n;
        if (CHK && n) {
            const uint64_t b = mix_b(g.rid(i));
            acc.c0 += sa * b;
            acc.c1 += sa + n * b;
        }
    }
}

__device__ __forceinline__ void flush_acc(hj_counters *ctr, ProbeAcc acc, bool with_cnt) {
    acc.cnt = warp_sum(acc.cnt);
    acc.c0 = warp_sum(acc.c0);
    acc.c1 = warp_sum(acc.c1);
    if ((threadIdx.x & 31) == 0) {
        if (with_cnt && acc.cnt) atomicAdd(&ctr->count, acc.cnt);
        if (acc.c0) atomicAdd(&ctr->c0, acc.c0);
        if (acc.c1) atomicAdd(&ctr->c1, acc.c1);
    }
}

// ============================================================ global table (SHJ)

template <int W>
__global__ void agg_table_init(AggSlot<W> *slots, uint64_t cap) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < cap; i += (uint64_t)gridDim.x * blockDim.x) {
        AggSlot<W> s;
        s.key = Tup<W>::kAllOnes;
        s.cnt = 0;
        s.suma = 0;
        if constexpr (W == 8) s.pad = 0;
        slots[i] = s;
    }
}

template <int W, bool AGG>
__global__ void __launch_bounds__(256, 8) table_build_kernel(const void *R, uint64_t n, void *slots, uint64_t cap,
                                                          TableSide *side, hj_counters *ctr, PartFilter pf) {
    constexpr int PV = Tup<W>::kPerVec;
    const uint64_t nvec = (n + PV - 1) / PV;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    bool repeat = false;
    for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < nvec; v += stride) {
        Group<W, 1> g;
        g.load((const typename Tup<W>::Vec *)R, v & ~31ull, n);
#pragma unroll
        for (int e = 0; e < PV; ++e) {
            if (!((g.valid >> e) & 1u)) continue;
            const uint64_t h = key_hash<W>(g.key(e));
            if (!pf.keep(h)) continue;
            const bool ok = AGG ? agg_insert<W>((AggSlot<W> *)slots, cap, side, g.key(e), mix_a(g.rid(e)), h)
                                : pair_insert<W>((typename PairSlot<W>::S *)slots, (uint32_t)(cap / kBucketSlots<W>),
                                                 side, g.key(e), g.rid(e), h, &repeat, kMaxPairWalk, &ctr->status);
            if (!ok) atomicOr(&ctr->status, (unsigned long long)(AGG || cap <= kMaxPairWalk ? kStatusTableFull
                                                                                         : kStatusLongRun));
        }
    }
    if (!AGG && __syncthreads_or(repeat) && threadIdx.x == 0) side->repeats = 1;
}

template <int W> constexpr int kProbeVecs = kProbeItems / Tup<W>::kPerVec;

// Pairs per warp in the probe's shared-memory staging buffer (exact output mode):
// 4 KB, several times a group's pairs, so that the one address all warps claim
// rows from sees an atomic per 512 (256) pairs.
constexpr unsigned kProbeStageBytes = 4096;
template <int W> constexpr unsigned kProbeStage = kProbeStageBytes / (2 * W);

// Shared memory of a probing warp: the staging buffer, then the queue of runs.
template <int W> constexpr unsigned kProbeWarpBytes = kProbeStageBytes + sizeof(RunQueue<W>);

template <int W, bool CHK>
__global__ void __launch_bounds__(256, kProbeCtas) pair_probe_kernel(const void *S, uint64_t n, const void *slots,
                                                            uint32_t nb, const TableSide *side, void *pairs,
                                                            uint64_t pcap, hj_counters *ctr) {
    using Vec = typename Tup<W>::Vec;
    constexpr int PV = Tup<W>::kPerVec, U = kProbeVecs<W>;
    const uint64_t g0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32ull * U);
    const uint64_t stride = (uint64_t)((gridDim.x * blockDim.x) >> 5) * (32 * U);
    const uint64_t nvec = (n + PV - 1) / PV, whole = n / PV / (32 * U) * (32 * U);  // groups below `whole` are full
    extern __shared__ __align__(16) unsigned char tp_smem[];
    unsigned char *mine = tp_smem + (size_t)(threadIdx.x >> 5) * kProbeWarpBytes<W>;
    RunQueue<W> &q = *(RunQueue<W> *)(mine + kProbeStageBytes);
    uint32_t qn = 0;
    OutState st;
    OutCtx oc{pairs, pcap, ctr};
    oc.stage = mine;
    oc.scap = kProbeStage<W>;
    st.used = 0;
    ProbeAcc acc;
    const PairTab<W> tab{(const typename PairSlot<W>::S *)slots, nb, side->n_allones, side->repeats == 0};
    Group<W, U> cur, nxt;
    if (g0 < nvec) cur.load((const Vec *)S, g0, n);
    uint64_t g = g0;
    for (; g < whole; g += stride) {
        nxt.load((const Vec *)S, g + stride, n);
        probe_group_pairs<W, U, CHK, true>(tab, cur, q, qn, st, oc, acc);
        cur = nxt;
    }
    if (g < nvec) probe_group_pairs<W, U, CHK, false>(tab, cur, q, qn, st, oc, acc);  // the last group
    while (qn) drain_runs<W, CHK>(tab, q, qn, min(qn, 32u), st, oc, acc);
    warp_stage_flush<W>(st, oc);
    if (CHK) flush_acc(ctr, acc, false);
}

template <int W, bool CHK>
__global__ void __launch_bounds__(256) agg_probe_kernel(const void *S, uint64_t n, const void *slots, uint64_t cap,
                                                        const TableSide *side, hj_counters *ctr, PartFilter pf) {
    using Vec = typename Tup<W>::Vec;
    constexpr int PV = Tup<W>::kPerVec, U = 4 / PV;
    const uint64_t nvec = (n + PV - 1) / PV;
    const uint64_t g0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32ull * U);
    const uint64_t stride = (uint64_t)((gridDim.x * blockDim.x) >> 5) * (32 * U);
    ProbeAcc acc;
    for (uint64_t g = g0; g < nvec; g += stride) {
        Group<W, U> cur;
        cur.load((const Vec *)S, g, n);
        probe_group_agg<W, U, CHK>((const AggSlot<W> *)slots, cap, side, cur, pf, acc);
    }
    if constexpr (!CHK) {
        flush_acc(ctr, acc, true);
    } else {
        // the CTA's warps add up first: three atomics per warp on one line took a sixth of the
        // call for a small table (2^16 x 2^20 4-byte tuples 80 -> 67 us; one per warp does not
        // show, and without checksums the barrier costs as much)
        __shared__ unsigned long long sums[8][3];
        const unsigned warp = threadIdx.x >> 5;
        acc.cnt = warp_sum(acc.cnt);
        acc.c0 = warp_sum(acc.c0);
        acc.c1 = warp_sum(acc.c1);
        if ((threadIdx.x & 31) == 0) {
            sums[warp][0] = acc.cnt;
            sums[warp][1] = acc.c0;
            sums[warp][2] = acc.c1;
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            unsigned long long x = 0;
            for (unsigned w = 0; w < 8; ++w) x += sums[w][threadIdx.x];
            if (x) atomicAdd(threadIdx.x == 0 ? &ctr->count : threadIdx.x == 1 ? &ctr->c0 : &ctr->c1, x);
        }
    }
}

// One CTA of 256 threads per `per_cta` items, at most `per_sm` CTAs for every SM.
static unsigned items_grid(hj_ctx *c, uint64_t n, uint64_t per_cta, uint64_t per_sm) {
    const uint64_t want = (n + per_cta - 1) / per_cta, most = (uint64_t)num_sms(c) * per_sm;
    return (unsigned)(want < most ? (want ? want : 1) : most);
}

// Largest pair table that takes four slots per tuple (twice L2: larger ones are
// bound by HBM sectors, not by the few longer runs).
constexpr uint64_t kFastTableBytes = 256ull << 20;

// An empty pair table, its side data and (ctr not NULL) a join's counters, all
// but the sticky fault word.
__global__ void __launch_bounds__(256) pair_table_init(ulonglong2 *slots, uint64_t n, TableSide *side, hj_counters *ctr) {
    const uint64_t i0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    for (uint64_t i = i0; i < n; i += (uint64_t)gridDim.x * blockDim.x) slots[i] = make_ulonglong2(~0ull, ~0ull);
    if (i0 < sizeof(TableSide) / 8) ((unsigned long long *)side)[i0] = 0;
    if (ctr && i0 < offsetof(hj_counters, fault) / 8) ((unsigned long long *)ctr)[i0] = 0;
}

uint64_t table_slots(int width, int agg, uint64_t n_build, bool budget) {
    // Capacity: a power of two at least twice the build size (load factor <= 0.5).  A
    // pair table takes four slots per tuple (2 % of 4-byte buckets are then full, 5 %
    // at three: 2^24 probes of 2^18 tuples 106 us against 123 us) unless the context
    // has a memory budget, which keeps the smaller size it always had.
    uint64_t cap = 64;
    while (cap < 2 * n_build + 1) cap <<= 1;
    if (agg) return cap;
    if (!budget && 4 * n_build * 2 * width <= kFastTableBytes) cap = std::max<uint64_t>(64, 4 * n_build);
    // (a bucket's number is 32 bits; the last power of two of 8-byte tuples would have one more)
    const uint64_t g = width == 4 ? kBucketSlots<4> : kBucketSlots<8>;
    return std::min<uint64_t>(cap, 0xFFFFFFFFull * g);
}

hj_status table_create(hj_ctx *c, int width, int agg, uint64_t n_build, hj_table **out, bool zero_ctr) {
    *out = nullptr;
    const uint64_t slot_bytes = agg ? (width == 4 ? sizeof(AggSlot<4>) : sizeof(AggSlot<8>)) : 2ull * width;
    const uint64_t cap = table_slots(width, agg, n_build, c->budget != 0);
    DevBuf slots(c), side(c);
    HJ_TRY(slots.alloc(cap * slot_bytes));
    HJ_TRY(side.alloc(sizeof(TableSide)));
    if (!agg) {
        const uint64_t n = cap * slot_bytes / 16;
        HJ_LAUNCH(c, "pair_table_init", pair_table_init, items_grid(c, n, 1024, 8), 256, 0, slots.as<ulonglong2>(), n,
                  side.as<TableSide>(), zero_ctr ? c->d_ctr : nullptr);
    } else {
        if (zero_ctr) HJ_TRY(zero_counters(c));
        HJ_CUDA(c, cudaMemsetAsync(side.p, 0, sizeof(TableSide), c->stream));
        int grid = num_sms(c) * 4;
        if (width == 4) {
            HJ_LAUNCH(c, "agg_table_init", agg_table_init<4>, grid, 256, 0, slots.as<AggSlot<4>>(), cap);
        } else {
            HJ_LAUNCH(c, "agg_table_init", agg_table_init<8>, grid, 256, 0, slots.as<AggSlot<8>>(), cap);
        }
    }
    hj_table *t = new hj_table();
    t->width = width;
    t->agg = agg;
    t->cap = cap;
    t->slots = slots.release();
    t->side = side.release();
    *out = t;
    return HJ_OK;
}

void table_destroy(hj_ctx *c, hj_table *t) {
    if (!t) return;
    dfree(c, t->slots);
    dfree(c, t->side);
    dfree(c, t->rids);
    delete t;
}

hj_status table_build(hj_ctx *c, hj_table *t, const void *R, uint64_t n, PartFilter pf) {
    if (!n) return HJ_OK;
    const unsigned grid = items_grid(c, n, t->width == 4 ? 512 : 256, 32);
    TableSide *side = (TableSide *)t->side;
#define HJ_TB(WW, AA)                                                                                             \
    HJ_LAUNCH(c, "table_build", (table_build_kernel<WW, AA>), grid, 256, 0, R, n, t->slots, t->cap, side, c->d_ctr, pf)
    if (t->width == 4) {
        if (t->agg) HJ_TB(4, true); else HJ_TB(4, false);
    } else {
        if (t->agg) HJ_TB(8, true); else HJ_TB(8, false);
    }
#undef HJ_TB
    return HJ_OK;
}

hj_status table_probe(hj_ctx *c, const hj_table *t, const void *S, uint64_t n, void *pairs, uint64_t pcap,
                      int checksum, PartFilter pf, hj_counters *ctr) {
    if (!n) return HJ_OK;
    const TableSide *side = (const TableSide *)t->side;
#define HJ_TP(WW, CC)                                                                                               \
    do {                                                                                                            \
        if (t->agg)                                                                                                 \
            HJ_LAUNCH(c, "table_probe", (agg_probe_kernel<WW, CC>), items_grid(c, n, 1024, 8), 256, 0, S, n,        \
                      t->slots, t->cap, side, ctr, pf);                                                             \
        else {                                                                                                      \
            HJ_TRY(allow_max_smem(c, (const void *)pair_probe_kernel<WW, CC>));                                     \
            HJ_LAUNCH(c, "table_probe", (pair_probe_kernel<WW, CC>),                                                \
                      items_grid(c, n, 256 * kProbeItems, kProbeCtas), 256, 8 * kProbeWarpBytes<WW>, S, n,          \
                      t->slots, (uint32_t)(t->cap / kBucketSlots<WW>), side, pairs, pcap, ctr);                     \
        }                                                                                                           \
    } while (0)
    if (t->width == 4) {
        if (checksum) HJ_TP(4, true); else HJ_TP(4, false);
    } else {
        if (checksum) HJ_TP(8, true); else HJ_TP(8, false);
    }
#undef HJ_TP
    return HJ_OK;
}

// ================================================== per-partition join (PHJ)
//
// Persistent CTAs take partition tasks (R_p with a slice of S_p) from ctr->work.
// For each, the CTA builds a table over R_p in shared memory (about three slots
// per build row, multiply-shift buckets so any capacity works), then its warps
// stream the S slice.  Partitions come from the padded partitioner: every
// partition starts and ends on a 32-byte sector, so whole 16-byte vectors can be
// loaded without bounds checks on tuples, and padding tuples (keys of another
// partition) match nothing.  A partition whose table cannot fit (|R_p| too large
// for a pair table, more distinct keys than slots for an aggregate table, or an
// insert walking past kMaxSmemWalk buckets: a heavily repeated key) goes to the
// host's fallback list, joined there with a global key-list table (pairs) or
// aggregate table (counts).

template <int W> struct HashT { using type = uint32_t; };
template <> struct HashT<8> { using type = uint64_t; };

// Bucket of a key inside a partition's shared-memory table: Fibonacci
// multiply-shift of the key.  Keys of one partition already share their
// MurmurHash2 partition digit, so a cheap hash that spreads them is enough here.
template <int W> __device__ __forceinline__ uint32_t part_bucket(typename Tup<W>::U k, uint32_t nb);
template <> __device__ __forceinline__ uint32_t part_bucket<4>(uint32_t k, uint32_t nb) {
    return __umulhi(k * 0x9E3779B1u, nb);
}
template <> __device__ __forceinline__ uint32_t part_bucket<8>(uint64_t k, uint32_t nb) {
    return __umulhi((uint32_t)((k * 0x9E3779B97F4A7C15ull) >> 32), nb);
}

// Bucket hash of a partition's shared-memory aggregate table (the value that
// bucket_of<W> scales to the table): a Fibonacci multiply of the key, for the same
// reason as part_bucket.
template <int W> __device__ __forceinline__ uint64_t part_agg_hash(typename Tup<W>::U k);
template <> __device__ __forceinline__ uint64_t part_agg_hash<4>(uint32_t k) { return (uint32_t)(k * 0x9E3779B1u); }
template <> __device__ __forceinline__ uint64_t part_agg_hash<8>(uint64_t k) { return k * 0x9E3779B97F4A7C15ull; }

template <int W>
__device__ __forceinline__ typename HashT<W>::type hashw(typename Tup<W>::U k) {
    if constexpr (W == 4) return murmur2_u32(k);
    else return murmur2_u64(k);
}

// ----------------------------------------------------------- shared-memory table
// Bucketised open addressing in shared memory for one partition pair.  Bucket b is
// G slots (G = 4 for 4-byte tuples, 2 for 8-byte): its G keys are 16 bytes of the
// key region and its G rids 16 bytes of the rid region (separate regions, so that
// the key loads of random buckets spread over all shared-memory banks).  (Two keys of
// 4 bytes per bucket load in half the time, but one hit in six is then in a bucket
// that overflowed, one in twenty with four, and following those costs more.)
// Every real key of partition p hashes to p, so a key that hashes to another
// partition can never be stored or probed: it marks empty slots (no value of the
// key domain needs reserving).  A key's run starts at its home bucket and moves
// linearly over buckets.  A bucket's 16-bit count says how many inserts tried it:
// the count before its own tells an insert its slot (or, from G on, to move to the
// next bucket), and a lookup stops at the first bucket tried by no more than G.
template <int W> struct SoaTab {
    using T = typename Tup<W>::U;
    static constexpr uint32_t G = 16 / W;
    uint32_t nb;     // buckets
    T empty;
    const uint16_t *cnt;  // inserts that tried the bucket (each once)

    __device__ __forceinline__ bool overflowed(uint32_t b) const { return cnt[b] > G; }
    // keys (half 0) or rids (half 1) of bucket b.  Plain loads through the
    // shared-memory pointers: the compiler orders them with the barriers and may
    // overlap the independent lookups of a thread's items.
    const T *kptr;   // key region: G keys (16 bytes) per bucket
    const T *rptr;   // rid region, same shape
    __device__ __forceinline__ void ld(uint32_t b, uint32_t half, T *v) const {
        const T *p = (half ? rptr : kptr) + b * G;
        if constexpr (W == 4) {
            const uint4 x = *(const uint4 *)p;
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        } else {
            const ulonglong2 x = *(const ulonglong2 *)p;
            v[0] = x.x; v[1] = x.y;
        }
    }
    __device__ __forceinline__ T ld1(uint32_t b, uint32_t half, uint32_t q) const {
        return (half ? rptr : kptr)[b * G + q];
    }
};

// The whole warp emits every build match of key kk (probe rid ss): a window of
// 32 slots (32 / G buckets) per step, up to the first bucket that ends the run.
template <int W, class Sink>
__device__ __forceinline__ void soa_coop_emit(const SoaTab<W> &t, typename Tup<W>::U kk, typename Tup<W>::U ss,
                                              uint32_t home, Sink &sink) {
    using T = typename Tup<W>::U;
    constexpr uint32_t G = SoaTab<W>::G, BPW = 32 / G;
    const unsigned lane = threadIdx.x & 31, jb = lane / G, q = lane % G;
#pragma unroll 1
    for (uint32_t off = 0; off < t.nb; off += BPW) {
        const bool inr = off + jb < t.nb;
        uint32_t b = home + off + jb;
        if (b >= t.nb) b -= t.nb;
        const T key = inr ? t.ld1(b, 0, q) : t.empty;
        const T rid = inr ? t.ld1(b, 1, q) : T(0);
        // (slots fill in order: a bucket whose last one is empty ends the run)
        const unsigned endm = __ballot_sync(0xffffffffu, q == G - 1 && (!inr || key == t.empty || !t.overflowed(b)));
        const bool m = inr && key == kk && lane <= (endm ? (unsigned)(__ffs(endm) - 1) : 31u);
        sink.append(m, rid, ss);
        if (endm) break;
    }
}

// ------------------------------------------------------------------ output sinks
// How a CTA's warps place the pairs of its partition tasks.
//
// ChunkSink: every warp takes whole chunks of the join's pair buffer (emit.cuh);
// partly used chunks are recorded and compacted on the device afterwards.  Used
// for a single join: no extra traffic, a small fix-up at the end.
//
// WarpStageSink, GlobalStageSink: every warp stages its pairs in a private buffer
// and claims exact rows of the join's buffer per buffer-full.  Used for batches of
// joins, where per-warp chunks would leave a partly used chunk per warp per join.
// The join's pair count is the claim cursor (ctr->count).
template <int W> struct ChunkSink {
    using T = typename Tup<W>::U;
    static constexpr bool kCheck = false;
    OutState st;
    OutCtx oc;
    typename PairVec<W>::T *open = nullptr;  // the open chunk (append_found)
    unsigned room = 0;                       // rows of it that append_found may fill without a test
    unsigned join = ~0u;
    const JoinSlot *slots;
    RecArea ra;
    __device__ __forceinline__ void begin_task(unsigned j) {
        if (j == join) return;
        if (join != ~0u) warp_finish(st, oc, ra);
        st = OutState();
        oc = OutCtx{slots[j].pairs, slots[j].pcap, slots[j].ctr, j};
        join = j;
        room = 0;
    }
    __device__ __forceinline__ void append(bool has, T a, T b) {
        warp_append<W>(st, oc, has, a, b);
        open = (typename PairVec<W>::T *)oc.pairs + st.base;
        set_room();
    }
    // one append for all items of a group with a match (at most 32 * IT pairs, so at
    // most one new chunk): item-major positions, so that each store instruction
    // writes consecutive slots; capacity tested once per chunk
    template <int IT>
    __device__ __forceinline__ void append_found(const bool *found, const T *first, const T *r) {
        using P = typename PairVec<W>::T;
        const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
        unsigned m[IT], tot = 0;
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            m[i] = __ballot_sync(0xffffffffu, found[i]);
            tot += __popc(m[i]);
        }
        if (tot <= room) {  // (warp-uniform) the open chunk has room, all of it inside the buffer
            P *dst = open + st.used;
#pragma unroll
            for (int i = 0; i < IT; ++i) {
                if (found[i]) {
                    if constexpr (W == 4) dst[__popc(m[i] & lt)] = make_uint2(first[i], r[i]);
                    else dst[__popc(m[i] & lt)] = make_ulonglong2(first[i], r[i]);
                }
                dst += __popc(m[i]);
            }
            st.used += tot;
            st.pairs += tot;
            room -= tot;
            return;
        }
        const unsigned left = kChunkPairs - st.used;
        unsigned long long nb = 0;
        if (tot > left) {
            if (lane == 0) nb = atomicAdd(&oc.ctr->cursor, (unsigned long long)kChunkPairs);
            nb = __shfl_sync(0xffffffffu, nb, 0);
        }
        const unsigned long long c0 = st.base + st.used;
        unsigned run = 0;
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const unsigned idx = run + __popc(m[i] & lt);
            const unsigned long long pos = idx < left ? c0 + idx : nb + (idx - left);
            if (found[i] && pos < oc.pcap) PairOut<W>::put(oc.pairs, pos, first[i], r[i]);
            run += __popc(m[i]);
        }
        if (tot > left) {
            st.base = nb;
            st.used = tot - left;
            st.claimed = true;
        } else {
            st.used += tot;
        }
        st.pairs += tot;
        open = (P *)oc.pairs + st.base;
        set_room();
    }
    // pairs that fit the open chunk without a test of the buffer's end
    __device__ __forceinline__ void set_room() {
        room = st.claimed && st.base + kChunkPairs <= oc.pcap ? kChunkPairs - st.used : 0u;
    }
    __device__ __forceinline__ void finish() {
        if (join != ~0u) warp_finish(st, oc, ra);
    }
};

// Per-warp staged exact output (batches of joins, whose many joins per launch
// would leave a partly filled chunk per warp and join): each warp collects its
// pairs in a private buffer of scap pairs in shared memory and, when the buffer fills or
// the warp moves on to another join, claims exactly that many rows of the join's buffer
// with one atomic add and
// copies them out with coalesced stores.  Output is dense as written (no
// compaction) and the sink needs no CTA barrier.  scap >= 32 x the items of a
// group, so one flush always makes room.
// (4 KB per warp: 700 us for the 200 joins of batch_partition_rows, 720 us with 2 KB; the
// same staged in global memory, twice the rows per partition, 890 us)
constexpr uint32_t kJoinStageBytes = 4096;
template <int W> struct WarpStageSink {
    using T = typename Tup<W>::U;
    static constexpr bool kCheck = false;
    using P = typename std::conditional<W == 4, uint2, ulonglong2>::type;
    P *stage = nullptr;  // this warp's buffer
    uint32_t scap = 0;
    const JoinSlot *slots = nullptr;
    unsigned join = ~0u;
    uint32_t used = 0;  // warp-uniform
    __device__ __forceinline__ static P mk(T a, T b) {
        if constexpr (W == 4) return make_uint2(a, b);
        else return make_ulonglong2(a, b);
    }
    // all 32 lanes: the staged pairs to exact rows of the join's buffer (pairs past
    // its capacity are dropped; the count stays exact)
    __device__ __forceinline__ void flush() {
        if (!used) return;
        __syncwarp();  // the buffer's stores are visible to every lane
        const unsigned lane = threadIdx.x & 31;
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(&slots[join].ctr->count, (unsigned long long)used);
        b = __shfl_sync(0xffffffffu, b, 0);
        P *out = (P *)slots[join].pairs;
        const unsigned long long pc = slots[join].pcap;
        for (uint32_t i = lane; i < used; i += 32)
            if (b + i < pc) out[b + i] = stage[i];
        __syncwarp();  // read before the buffer is refilled
        used = 0;
    }
    __device__ __forceinline__ void begin_task(unsigned j) {
        if (j == join) return;
        flush();
        join = j;
    }
    __device__ __forceinline__ void append(bool has, T a, T b) {
        const unsigned mask = __ballot_sync(0xffffffffu, has);
        if (!mask) return;
        const unsigned lane = threadIdx.x & 31, k = __popc(mask), rank = __popc(mask & ((1u << lane) - 1u));
        if (used + k > scap) flush();
        if (has) stage[used + rank] = mk(a, b);
        used += k;
    }
    template <int IT>
    __device__ __forceinline__ void append_found(const bool *found, const T *first, const T *r) {
        const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
        unsigned m[IT], tot = 0;
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            m[i] = __ballot_sync(0xffffffffu, found[i]);
            tot += __popc(m[i]);
        }
        if (used + tot > scap) flush();
        P *dst = stage + used;
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            if (found[i]) dst[__popc(m[i] & lt)] = mk(first[i], r[i]);
            dst += __popc(m[i]);
        }
        used += tot;
    }
    __device__ __forceinline__ void finish() { flush(); }
};
// The same with the buffers in global memory (they stay in L2).
template <int W> struct GlobalStageSink : WarpStageSink<W> {};

// Any of them with the checksums of the pairs it takes.
template <int W, class Base> struct CheckSink : Base {
    using T = typename Tup<W>::U;
    static constexpr bool kCheck = true;
    ProbeAcc acc;
    __device__ __forceinline__ void append(bool has, T a, T b) {
        add_check<W, true>(acc, has, a, b);
        Base::append(has, a, b);
    }
    template <int IT> __device__ __forceinline__ void append_found(const bool *found, const T *first, const T *r) {
#pragma unroll
        for (int i = 0; i < IT; ++i) add_check<W, true>(acc, found[i], first[i], r[i]);
        Base::template append_found<IT>(found, first, r);
    }
};
template <int W> using ChunkCheckSink = CheckSink<W, ChunkSink<W>>;
template <int W> using WarpStageCheckSink = CheckSink<W, WarpStageSink<W>>;
template <int W> using GlobalStageCheckSink = CheckSink<W, GlobalStageSink<W>>;

// Longest walk (in buckets) of an insert into a partition's shared-memory table.
constexpr uint32_t kMaxSmemWalk = 64;

// When no more walks than this are left of 32 after three buckets, the warp takes one after
// the other, 32 slots at a time, in place of all at once, a bucket at a time (each key of R
// 4 / 16 / 40 times: 930 / 3300 / 8370 us with 2, 955 / 3150 / 8130 with 4, 975 / 3170 / 7910
// with 8; 16 times 3580 without).  Before that, and with a table of different keys, the
// walks left are short ones, which end sooner together (taken one by one from the first
// bucket on: 2^24 x 2^28 tuples of different keys 2330 -> 2500 us).
constexpr int kLongWalks = 4;

// Entries per warp of the queue of pending run walks (probe keys and rids whose
// run goes on past a full home bucket).
constexpr uint32_t kWalkQ = 64;

// Shared-memory layout of the join kernel: table slots (cap_max x slot bytes), the
// buckets' counts (two bytes each; an aggregate table: its overflow bitmap),
// then each warp's walk queue (kWalkQ keys, kWalkQ rids).
__host__ __device__ constexpr uint32_t bucket_info_bytes(uint32_t cap, int width, bool agg) {
    return agg ? (cap / 2 / 32 + 1) * 4 + 16 : cap * (uint32_t)width / 8;
}
__host__ __device__ constexpr uint32_t walkq_offset(uint32_t cap_max, uint32_t slot_bytes, int width, bool agg) {
    return (cap_max * slot_bytes + bucket_info_bytes(cap_max, width, agg) + 15) / 16 * 16;
}

// Probe rows of the next task asked into L2 (64 KB of 16-byte vectors).
constexpr uint32_t kAheadVecs = 4096;
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// The walks of n <= 32 queued items, one per lane: each lane follows its key's run
// from the bucket after its home and emits every match found there, a bucket per step.
// Walking them one lane at a time as they come would cost a whole warp pass each;
// batched, 32 walks of like length cost about one.
template <int W, bool UNIQ, class Sink>
__device__ __forceinline__ void drain_walks(const SoaTab<W> &tab, const typename Tup<W>::U *qk,
                                            const typename Tup<W>::U *qr, uint32_t n, Sink &sink) {
    using T = typename Tup<W>::U;
    constexpr uint32_t G = SoaTab<W>::G;
    const unsigned lane = threadIdx.x & 31;
    bool active = lane < n;
    const T kk = active ? qk[lane] : tab.empty;
    const T rr = active ? qr[lane] : T(0);
    __syncwarp();  // entries read before the queue is refilled
    uint32_t b = 0;
    if (active) {
        const uint32_t h = part_bucket<W>(kk, tab.nb);
        b = h + 1 == tab.nb ? 0 : h + 1;
    }
#pragma unroll 1
    for (uint32_t it = 1; it < tab.nb; ++it) {
        unsigned on = __ballot_sync(0xffffffffu, active);
        if (!on) break;
        if (!UNIQ && it > 3 && __popc(on) <= kLongWalks) {  // the long runs that are left: 32 slots at a time
#pragma unroll 1
            while (on) {
                const int L = __ffs(on) - 1;
                on &= on - 1;
                soa_coop_emit<W>(tab, __shfl_sync(0xffffffffu, kk, L), __shfl_sync(0xffffffffu, rr, L),
                                 __shfl_sync(0xffffffffu, b, L), sink);
            }
            break;
        }
        T key[G];
        tab.ld(b, 0, key);  // (a bucket of the table whatever the lane)
        uint32_t m = 0;
#pragma unroll
        for (uint32_t q = 0; q < G; ++q) m |= (uint32_t)(active && key[q] == kk) << q;
        const bool any = m != 0;
        if (__any_sync(0xffffffffu, any)) {
            if (UNIQ) {
                sink.append(any, any ? tab.ld1(b, 1, (uint32_t)(__ffs(m) - 1)) : T(0), rr);
                active = active && !any;
            } else {
                T rid[G], sr[G];
                bool hit[G];
                tab.ld(b, 1, rid);
#pragma unroll
                for (uint32_t q = 0; q < G; ++q) {
                    hit[q] = (m >> q) & 1u;
                    sr[q] = rr;
                }
                sink.template append_found<G>(hit, rid, sr);
            }
        }
        // (slots fill in order: an empty one is the last)
        active = active && key[G - 1] != tab.empty && tab.overflowed(b);
        b = b + 1 == tab.nb ? 0 : b + 1;
    }
}

// Whether no key is twice in the table: every thread of the CTA compares the keys
// of its buckets, and of a bucket that overflowed with those its run goes on to.
template <int W, int NT> __device__ __forceinline__ bool keys_repeat(const SoaTab<W> &t) {
    using T = typename Tup<W>::U;
    constexpr uint32_t G = SoaTab<W>::G;
    bool dup = false;
    for (uint32_t b = threadIdx.x; b < t.nb; b += NT) {
        T k[G];
        t.ld(b, 0, k);
#pragma unroll
        for (uint32_t i = 0; i < G; ++i)
#pragma unroll
            for (uint32_t j = i + 1; j < G; ++j) dup |= k[i] == k[j] && k[j] != t.empty;
        uint32_t c = b;
        for (uint32_t it = 1; it < t.nb && t.overflowed(c); ++it) {
            c = c + 1 == t.nb ? 0 : c + 1;
            T o[G];
            t.ld(c, 0, o);
#pragma unroll
            for (uint32_t i = 0; i < G; ++i)
#pragma unroll
                for (uint32_t j = 0; j < G; ++j) dup |= k[i] == o[j] && o[j] != t.empty;
        }
    }
    return dup;
}

// Probe one group of U vectors per lane (FULL: every lane holds tuples in all of them),
// in phases so that the items' shared-memory loads overlap: every item's home bucket
// (keys), then the place of the match (a select per key) and its rid.  Inserts fill a
// bucket's slots in order and move past it only once it is full, so a run goes on past
// the home bucket only if the bucket's last slot is taken AND more inserts tried it than
// it has slots: such items are queued and their runs walked 32 at a time.  With UNIQ (no
// key is twice in the table) a match ends the search; otherwise the further matches of the
// home buckets go out one per item and step.  (A warp that walked one such item after the
// other lived from many warps, 32 of them; with 20, |R| = 2^22 4-byte tuples of each key
// twice / 4 / 16 times with 2^24: 3640 / 3860 / 5860 us, like this 575 / 955 / 3150; each key
// four times with 8 bytes 4260 and 1710.)  With MARK the marker of empty slots may be a key:
// its build rids are the `side` list.
template <int W> struct SideList {
    const typename Tup<W>::U *rids = nullptr;
    uint32_t n = 0;
};
template <int W, int U, bool UNIQ, bool FULL, bool MARK, class Sink>
__device__ __forceinline__ void probe_group_smem(const SoaTab<W> &tab, const typename Tup<W>::Vec *x, const bool *in,
                                                 Sink &sink, unsigned lane, typename Tup<W>::U *wqk,
                                                 typename Tup<W>::U *wqr, uint32_t &qn, const SideList<W> &side) {
    using T = typename Tup<W>::U;
    constexpr int PV = Tup<W>::kPerVec, IT = U * PV;
    constexpr uint32_t G = SoaTab<W>::G;
    T k[IT], r[IT];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if constexpr (W == 4) {
            k[2 * u] = x[u].x; r[2 * u] = x[u].y; k[2 * u + 1] = x[u].z; r[2 * u + 1] = x[u].w;
        } else {
            k[u] = x[u].x; r[u] = x[u].y;
        }
    }
    uint32_t home[IT];
    T kb[IT][G], first[IT];
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        home[i] = part_bucket<W>(k[i], tab.nb);  // < nb for any key: the load is in bounds
        tab.ld(home[i], 0, kb[i]);
    }
    bool found[IT], w[IT], anyw = false;
    uint32_t more = 0;  // further matches in the home buckets: G bits per item
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const bool live = (FULL || in[i]) && !(MARK && k[i] == tab.empty);
        uint32_t sl = home[i] * G + (G - 1), m = (uint32_t)(kb[i][G - 1] == k[i]) << (G - 1);
        bool f = kb[i][G - 1] == k[i];
#pragma unroll
        for (int q = (int)G - 2; q >= 0; --q) {
            const bool h = kb[i][q] == k[i];
            sl = h ? home[i] * G + q : sl;
            f |= h;
            m |= (uint32_t)h << q;
        }
        first[i] = tab.rptr[sl];
        found[i] = live && f;
        if (!UNIQ && live) more |= (m & (m - 1u)) << (i * G);
        w[i] = live && !(UNIQ && f) && kb[i][G - 1] != tab.empty && tab.overflowed(home[i]);
        anyw |= w[i];
    }
    sink.template append_found<IT>(found, first, r);
    if (!UNIQ)
        while (__any_sync(0xffffffffu, more != 0)) {  // (at most G - 1 times)
#pragma unroll
            for (int i = 0; i < IT; ++i) {
                const uint32_t m = (more >> (i * G)) & ((1u << G) - 1u);
                found[i] = m != 0;
                if (m) first[i] = tab.ld1(home[i], 1, (uint32_t)(__ffs(m) - 1));
                more &= ~((m & (0u - m)) << (i * G));
            }
            sink.template append_found<IT>(found, first, r);
        }
    if (MARK && side.n) {
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            unsigned m = __ballot_sync(0xffffffffu, (FULL || in[i]) && k[i] == tab.empty);
            while (m) {
                const int L = __ffs(m) - 1;
                m &= m - 1;
                const T ss = __shfl_sync(0xffffffffu, r[i], L);
                for (uint32_t j = 0; j < side.n; j += 32) {
                    const bool has = j + lane < side.n;
                    sink.append(has, has ? side.rids[j + lane] : T(0), ss);
                }
            }
        }
    }
    if (__any_sync(0xffffffffu, anyw)) {
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const unsigned wm = __ballot_sync(0xffffffffu, w[i]);
            if (!wm) continue;
            if (w[i]) {
                const uint32_t pos = qn + (uint32_t)__popc(wm & ((1u << lane) - 1u));
                wqk[pos] = k[i];
                wqr[pos] = r[i];
            }
            qn += (uint32_t)__popc(wm);
            if (qn >= 32) {
                __syncwarp();
                drain_walks<W, UNIQ>(tab, wqk + (qn - 32), wqr + (qn - 32), 32, sink);
                qn -= 32;
            }
        }
    }
}

// A CTA's probe of a slice of nsv vectors.  What bounds it: instructions and the
// shared-memory pipe (a bucket of random lanes takes 10.3 cycles per warp), each at
// 55 %, and the latency that 20 warps leave open.  Queued are 1 % of the items of a table
// of different keys, 3 % otherwise.  A join of 2^22 with 2^25 4-byte tuples of
// different build keys issues 84e6 warp instructions; one vector per lane, with the
// matches of a bucket counted and several bases per store, took 128e6.
template <int W, int U, bool UNIQ, bool MARK = false, class Sink>
__device__ __forceinline__ void probe_smem(const SoaTab<W> &tab, const typename Tup<W>::Vec *Sv, uint32_t nsv,
                                           Sink &sink, unsigned warp, unsigned nwarps, unsigned lane,
                                           typename Tup<W>::U *wqk, typename Tup<W>::U *wqr,
                                           const SideList<W> &side = SideList<W>()) {
    constexpr int PV = Tup<W>::kPerVec;
    using Vec = typename Tup<W>::Vec;
    const uint32_t gstride = nwarps * 32u * U, whole = nsv / (32u * U) * (32u * U);
    uint32_t g = warp * 32u * U, qn = 0;
    Vec nxt[U];
    if (g < whole)
#pragma unroll
        for (int u = 0; u < U; ++u) nxt[u] = ld_stream(Sv + g + u * 32u + lane);
    for (; g < whole; g += gstride) {
        Vec cur[U];
#pragma unroll
        for (int u = 0; u < U; ++u) cur[u] = nxt[u];
        // (the group in registers covers part of the loads' latency, L2 the rest)
        const uint32_t pv = g + 3u * gstride + lane * 8u;
        if (lane < 4u * U && pv < nsv) prefetch_l2(Sv + pv);
        if (g + gstride < whole)
#pragma unroll
            for (int u = 0; u < U; ++u) nxt[u] = ld_stream(Sv + g + gstride + u * 32u + lane);
        probe_group_smem<W, U, UNIQ, true, MARK>(tab, cur, nullptr, sink, lane, wqk, wqr, qn, side);
    }
    if (g == whole && whole < nsv) {  // the slice's last, partial group, in this warp's turn
        Vec cur[U];
        bool in[U * PV];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool on = g + u * 32u + lane < nsv;
            if (on) cur[u] = ld_stream(Sv + g + u * 32u + lane);
            else cur[u] = Vec{};
#pragma unroll
            for (int e = 0; e < PV; ++e) in[u * PV + e] = on;
        }
        probe_group_smem<W, U, UNIQ, false, MARK>(tab, cur, in, sink, lane, wqk, wqr, qn, side);
    }
    if (qn) {
        __syncwarp();
        drain_walks<W, UNIQ>(tab, wqk, wqr, qn, sink);
    }
}

// Bytes per slot of a partition's shared-memory aggregate table: the key, the
// number of build tuples with that key and, with checksums, the sum of A(rid) over
// them.
__host__ __device__ constexpr uint32_t agg_slot_bytes(int width, int chk) {
    return (uint32_t)width + 4u + (chk ? 8u : 0u);
}

// Aggregate table of one partition in shared memory (Sec. 3.1's key list with each
// rid list folded into a count and a sum): the bucket layout of SoaTab -- G keys
// per 16-byte bucket, a key that hashes to another partition as the empty marker,
// runs that move linearly over buckets with overflow bits -- but one slot per
// distinct key, so a lookup finds at most one slot.  Regions: keys (cap x W
// bytes), sums (cap x 8, with checksums only), counts (cap x 4).
template <int W> struct AggSoa {
    using T = typename Tup<W>::U;
    static constexpr uint32_t G = 16 / W;
    uint32_t nb;
    T empty;
    uint32_t *ovf;
    T *keys;
    unsigned long long *suma;  // null without checksums
    uint32_t *cnt;

    __device__ static AggSoa at(unsigned char *base, uint32_t cap, T empty, uint32_t *ovf, bool chk) {
        AggSoa t;
        t.nb = cap / G;
        t.empty = empty;
        t.ovf = ovf;
        t.keys = (T *)base;
        t.suma = chk ? (unsigned long long *)(base + (size_t)cap * W) : nullptr;
        t.cnt = (uint32_t *)(base + (size_t)cap * (W + (chk ? 8 : 0)));
        return t;
    }
    __device__ __forceinline__ bool overflowed(uint32_t b) const { return (ovf[b >> 5] >> (b & 31)) & 1u; }
    __device__ __forceinline__ void ld(uint32_t b, T *v) const {
        if constexpr (W == 4) {
            const uint4 x = *(const uint4 *)(keys + b * G);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        } else {
            const ulonglong2 x = *(const ulonglong2 *)(keys + b * G);
            v[0] = x.x; v[1] = x.y;
        }
    }
    // Add a build tuple of key k (a = A(rid), used with checksums).  The slot of k is
    // the first slot of its run that holds k, else the first empty one, claimed by
    // CAS: slots only ever go from empty to a key, so two inserts of the same key
    // always meet in one slot.  The 64-bit sum takes two 32-bit adds, the carry out of
    // the low one with the high one (exact modulo 2^64 whatever the order): the shared
    // memory adds 32-bit words of equal keys by itself, while one 64-bit add is a
    // loop of CAS that equal keys repeat.  False if every bucket is full.
    __device__ __forceinline__ bool insert(T k, uint64_t a) const {
        uint32_t b = part_bucket<W>(k, nb);
        for (uint32_t it = 0; it < nb; ++it) {
            volatile T *kb = keys + b * G;
            // each failed CAS follows one more slot of the bucket being filled
            for (uint32_t tries = 0; tries <= G; ++tries) {
                int hit = -1, emp = -1;
#pragma unroll
                for (uint32_t q = 0; q < G; ++q) {
                    const T x = kb[q];
                    if (x == k && hit < 0) hit = (int)q;
                    if (x == empty && emp < 0) emp = (int)q;
                }
                if (hit < 0 && emp >= 0) {
                    const T old = cas_key<W>(keys + b * G + emp, empty, k);
                    if (old != empty && old != k) continue;
                    hit = emp;
                }
                if (hit < 0) break;  // full bucket without k
                atomicAdd(&cnt[b * G + hit], 1u);
                if (suma) {
                    uint32_t *w = (uint32_t *)&suma[b * G + hit];
                    const uint32_t lo = (uint32_t)a, old = atomicAdd(&w[0], lo);
                    atomicAdd(&w[1], (uint32_t)(a >> 32) + (old + lo < lo ? 1u : 0u));
                }
                return true;
            }
            atomicOr(&ovf[b >> 5], 1u << (b & 31));
            b = b + 1 == nb ? 0 : b + 1;
        }
        return false;
    }
    // Slot of key k from bucket b on (the run's continuation), or ~0u.
    __device__ __forceinline__ uint32_t find_from(T k, uint32_t b) const {
        for (uint32_t it = 0; it < nb; ++it) {
            T key[G];
            ld(b, key);
            uint32_t m = 0;
            bool e = false;
#pragma unroll
            for (uint32_t q = 0; q < G; ++q) {
                m |= (uint32_t)(key[q] == k) << q;
                e |= key[q] == empty;
            }
            if (m) return b * G + (uint32_t)(__ffs(m) - 1);
            if (e || !overflowed(b)) return ~0u;
            b = b + 1 == nb ? 0 : b + 1;
        }
        return ~0u;
    }
};

// A CTA's probe of a slice of nsv vectors with a partition's aggregate table: the home
// buckets of all of a lane's items are loaded before the first one is looked at.  No
// partition filter: a padding tuple's key hashes to another partition, so it matches no
// slot.
template <int W>
__device__ __forceinline__ void probe_smem_agg(const AggSoa<W> &at, const typename Tup<W>::Vec *Sv, uint32_t nsv, int chk,
                                               ProbeAcc &acc, unsigned warp, unsigned nwarps, unsigned lane) {
    using T = typename Tup<W>::U;
    using Vec = typename Tup<W>::Vec;
    constexpr int PV = Tup<W>::kPerVec, U = 2, IT = U * PV;
    constexpr uint32_t AG = AggSoa<W>::G;
    const uint32_t gstride = nwarps * 32 * U;
    Vec cur[U], nxt[U];
    uint32_t g = warp * 32 * U;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const uint32_t rel = g + u * 32 + lane;
        if (rel < nsv) cur[u] = ld_stream(Sv + rel);
    }
    for (; g < nsv; g += gstride) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t rel = g + gstride + u * 32 + lane;
            if (rel < nsv) nxt[u] = ld_stream(Sv + rel);
        }
        T k[IT], r[IT];
        bool val[IT];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = g + u * 32 + lane < nsv;
            if constexpr (W == 4) {
                k[2 * u] = cur[u].x; r[2 * u] = cur[u].y; k[2 * u + 1] = cur[u].z; r[2 * u + 1] = cur[u].w;
                val[2 * u] = in;
                val[2 * u + 1] = in;
            } else {
                k[u] = cur[u].x; r[u] = cur[u].y;
                val[u] = in;
            }
        }
        uint32_t home[IT];
        T kb[IT][AG];
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            home[i] = part_bucket<W>(k[i], at.nb);
#pragma unroll
            for (uint32_t q = 0; q < AG; ++q) kb[i][q] = at.empty;
            if (val[i]) at.ld(home[i], kb[i]);
        }
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            uint32_t mm = 0;
            bool e = false;
#pragma unroll
            for (uint32_t q = 0; q < AG; ++q) {
                mm |= (uint32_t)(kb[i][q] == k[i]) << q;
                e |= kb[i][q] == at.empty;
            }
            // (a lane past the slice's end holds a stale key: no slot)
            uint32_t sl = val[i] && mm ? home[i] * AG + (uint32_t)(__ffs(mm) - 1) : ~0u;
            if (val[i] && !mm && !e && at.overflowed(home[i]))  // the run continues (rare)
                sl = at.find_from(k[i], home[i] + 1 == at.nb ? 0 : home[i] + 1);
            if (sl != ~0u) {
                const uint64_t n = at.cnt[sl];
                acc.cnt += n;
                if (chk) {
                    const uint64_t sa = at.suma[sl], bb = mix_b(r[i]);
                    acc.c0 += sa * bb;
                    acc.c1 += sa + n * bb;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) cur[u] = nxt[u];
    }
}

// CTAs per SM of the join kernel's launch shapes.
__host__ __device__ constexpr int join_ctas(int nt) { return nt > 512 ? 1 : 2; }

template <int W, bool AGG, int NT, class Sink>
__global__ void __launch_bounds__(NT, join_ctas(NT)) partition_join_kernel(
    const PartTask *tasks, uint64_t ntasks, uint64_t lead, const JoinSlot *slots, hj_counters *work, uint32_t cap_max,
    RecArea ra, uint32_t *oversize, int chk, uint32_t stage_at, void *stage) {
    using T = typename Tup<W>::U;
    using Vec = typename Tup<W>::Vec;
    constexpr int PV = Tup<W>::kPerVec;
    constexpr uint32_t G = SoaTab<W>::G, AG = AggSoa<W>::G;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_full;
    __shared__ __align__(16) PartTask s_task[2];
    __shared__ unsigned long long s_idx[2];
    __shared__ int s_ahead;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;

    Sink sink;
    if constexpr (std::is_base_of<ChunkSink<W>, Sink>::value) {
        sink.slots = slots;
        sink.ra = ra;
    } else {
        using P = typename WarpStageSink<W>::P;
        if constexpr (std::is_base_of<GlobalStageSink<W>, Sink>::value)
            sink.stage = (P *)((char *)stage + ((size_t)blockIdx.x * nwarps + warp) * kJoinStageBytes);
        else
            sink.stage = (P *)(smem + stage_at + warp * kJoinStageBytes);
        sink.scap = kJoinStageBytes / (2 * W);
        sink.slots = slots;
    }
    // While more than two of the first `lead` tasks per CTA remain, tasks are taken one
    // ahead: during a task's build warp 0 reads the record of the next one (whose index it took at the
    // end of the task before), and during its probe the next one's build rows and first
    // probe rows are asked into L2.  The last tasks are taken as CTAs fall idle.
    constexpr unsigned kTaskWords = sizeof(PartTask) / 4;
    static_assert(kTaskWords <= 32, "a warp reads a task record");
    constexpr unsigned long long kNone = ~0ull;
    unsigned long long idx = kNone;  // warp 0, lane 0: the next task's index, if taken ahead
    if (warp == 0) {
        unsigned long long i = 0;
        if (lane == 0) i = atomicAdd(&work->work, 1ull);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i < ntasks && lane < kTaskWords) ((uint32_t *)&s_task[0])[lane] = ((const uint32_t *)(tasks + i))[lane];
        if (lane == 0) {
            s_idx[0] = i;
            if (i + 2 * gridDim.x < lead) idx = atomicAdd(&work->work, 1ull);
        }
    }
    __syncthreads();
    for (unsigned cur_task = 0;; cur_task ^= 1) {
        if (s_idx[cur_task] >= ntasks) break;
        const uint64_t ti = s_idx[cur_task];
        const PartTask &tk = s_task[cur_task];
        uint32_t rec = 0;  // warp 0: the next task's record, a word per lane
        if (warp == 0) {
            idx = __shfl_sync(0xffffffffu, idx, 0);
            if (idx < ntasks && lane < kTaskWords) rec = ((const uint32_t *)(tasks + idx))[lane];
        }
        auto pass_record = [&]() {
            if (warp != 0) return;
            if (idx != kNone && lane < kTaskWords) ((uint32_t *)&s_task[cur_task ^ 1])[lane] = rec;
            if (lane == 0) s_ahead = idx < ntasks;
        };
        const uint32_t nrv = tk.nr / PV, nsv = tk.ns / PV;
        const Vec *Rv = (const Vec *)tk.R;
        const Vec *Sv = (const Vec *)tk.S;
        const uint64_t nr = tk.nr;  // build rows, padding included
        const PartFilter pf{tk.p, (int)tk.b1, (int)tk.b2, 1};
        const T pk1 = (T)tk.pk1, pk2 = (T)tk.pk2;  // keys of padding rows, besides 0
        hj_counters *jc = slots[tk.join].ctr;
        sink.begin_task(tk.join);
        ProbeAcc acc;
        bool work_p = nsv > 0 && nrv > 0;
        uint32_t cap = 0;
        if (work_p) {
            if (AGG) {
                // about three slots per build row, whole buckets; with duplicate
                // keys fewer slots than rows may do, so no early fallback
                const uint64_t want = (3 * nr + 127) / 128 * 128;
                cap = want < cap_max ? (uint32_t)want : cap_max;
            } else {
                // about three slots per build row (load factor 1/3), whole buckets
                const uint64_t want = (3 * nr + 127) / 128 * 128;
                cap = want < cap_max ? (uint32_t)want : cap_max;
                if (nr >= cap - cap / 5) {  // load factor above 4/5: leave to the fallback
                    if (threadIdx.x == 0) oversize[atomicAdd(&work->n_oversize, 1ull)] = (uint32_t)ti;
                    work_p = false;
                }
            }
        }
        uint32_t *info = (uint32_t *)(smem + (size_t)cap_max * (AGG ? agg_slot_bytes(W, chk) : 2 * W));
        const T top = Tup<W>::kAllOnes;
        const T empty = pf.keep(hashw<W>(top)) ? (T)tk.ek1 : top;
        const SoaTab<W> tab{cap / G, empty, (const uint16_t *)info, (const T *)smem, (const T *)smem + cap};
        const AggSoa<W> at = AggSoa<W>::at(smem, cap, empty, info, chk != 0);
        constexpr int RB = 2;  // build vectors per thread in flight
        Vec rx[RB];
        auto load_r = [&](uint32_t v0) {
#pragma unroll
            for (int u = 0; u < RB; ++u)
                if (v0 + u * NT < nrv) rx[u] = ld_stream(Rv + v0 + u * NT);
        };
        if (!work_p) pass_record();
        if (work_p) {
            if constexpr (!AGG) load_r(threadIdx.x);
            // key region: cap keys (whole 128s); the rid (or sum and count) regions follow
            uint4 e4;
            if constexpr (W == 4) e4 = make_uint4(empty, empty, empty, empty);
            else e4 = make_uint4((uint32_t)empty, (uint32_t)(empty >> 32), (uint32_t)empty, (uint32_t)(empty >> 32));
            for (uint32_t i = threadIdx.x; i < cap * W / 16; i += NT) ((uint4 *)smem)[i] = e4;
            const uint32_t info_words = AGG ? (cap / AG + 31) / 32 : cap / G / 2;
            for (uint32_t i = threadIdx.x; i < info_words; i += NT) info[i] = 0;
            if (AGG) {
                for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x) {
                    at.cnt[i] = 0;
                    if (chk) at.suma[i] = 0;
                }
            }
            if (threadIdx.x == 0) {
                s_full = 0;
            }
            __syncthreads();
            // build over R_p
            if constexpr (AGG) {
                for (uint32_t v = threadIdx.x; v < nrv; v += NT) {
                    const Vec x = ld_stream(Rv + v);
                    T k[2], r[2];
                    if constexpr (W == 4) {
                        k[0] = x.x; r[0] = x.y; k[1] = x.z; r[1] = x.w;
                    } else {
                        k[0] = x.x; r[0] = x.y;
                    }
#pragma unroll
                    for (int e = 0; e < PV; ++e) {
                        // a padding row carries 0 or a pass's second sentinel: only
                        // such keys are hashed to see whether the row is the partition's
                        if ((k[e] == T(0) || k[e] == pk1 || k[e] == pk2) && !pf.keep(hashw<W>(k[e]))) continue;
                        if (!at.insert(k[e], chk ? mix_a(r[e]) : 0)) s_full = 1;
                    }
                }
            } else {
                // An insert takes a count of its home bucket with one atomic add: the
                // count before it is its slot there (load factor 1/3: one in twenty
                // moves on).  The adds of a thread's four tuples are in flight together.
                // A walk past kMaxSmemWalk buckets means a heavily repeated key: the
                // partition goes to the key-list fallback.
                T *kv = (T *)smem;
                const uint32_t lim = tab.nb < kMaxSmemWalk ? tab.nb : kMaxSmemWalk;
                auto tried = [&](uint32_t b) -> uint32_t {
                    const uint32_t sh = (b & 1u) * 16u;
                    return (atomicAdd(&info[b >> 1], 1u << sh) >> sh) & 0xFFFFu;
                };
                for (uint32_t v0 = threadIdx.x; v0 < nrv; v0 += RB * NT) {
                    if (v0 != threadIdx.x) load_r(v0);
                    constexpr int QT = RB * PV;  // tuples of a step
                    T k[QT], r[QT];
                    uint32_t bkt[QT], q[QT];
                    bool in[QT];
#pragma unroll
                    for (int i = 0; i < QT; ++i) {
                        const Vec &x = rx[i / PV];
                        if constexpr (W == 4) {
                            k[i] = i % 2 ? x.z : x.x;
                            r[i] = i % 2 ? x.w : x.y;
                        } else {
                            k[i] = x.x;
                            r[i] = x.y;
                        }
                        // a padding row carries 0 or a pass's second sentinel: only
                        // such keys are hashed to see whether the row is the partition's
                        in[i] = v0 + (i / PV) * NT < nrv &&
                                !((k[i] == T(0) || k[i] == pk1 || k[i] == pk2) && !pf.keep(hashw<W>(k[i])));
                        bkt[i] = part_bucket<W>(k[i], tab.nb);
                        q[i] = in[i] ? tried(bkt[i]) : 0u;
                    }
#pragma unroll
                    for (int i = 0; i < QT; ++i) {
                        if (!in[i]) continue;
                        for (uint32_t it = 1; q[i] >= G && it < lim; ++it) {
                            bkt[i] = bkt[i] + 1 == tab.nb ? 0 : bkt[i] + 1;
                            q[i] = tried(bkt[i]);
                        }
                        if (q[i] < G) {
                            T *slot = &kv[bkt[i] * G + q[i]];
                            slot[0] = k[i];
                            slot[cap] = r[i];  // the same slot of the rid region
                        } else {
                            s_full = 1;
                        }
                    }
                }
            }
            pass_record();
            __syncthreads();
            if (s_ahead) {  // the next task's rows into L2
                const PartTask &nt = s_task[cur_task ^ 1];
                const uint32_t rl = (nt.nr / PV + 7) / 8, sl = (min(nt.ns / PV, kAheadVecs) + 7) / 8;
                for (uint32_t i = threadIdx.x; i < rl + sl; i += NT)
                    prefetch_l2(i < rl ? (const char *)nt.R + (uint64_t)i * 128
                                       : (const char *)nt.S + (uint64_t)(i - rl) * 128);
            }
            bool unique = false;
            if constexpr (!AGG) unique = nsv >= 2 * nrv && !s_full && !__syncthreads_or(keys_repeat<W, NT>(tab));
            if (s_full) {
                if (threadIdx.x == 0) oversize[atomicAdd(&work->n_oversize, 1ull)] = (uint32_t)ti;
            } else if constexpr (AGG) {
                probe_smem_agg<W>(at, Sv, nsv, chk, acc, warp, nwarps, lane);
            } else {
                T *wq = (T *)(smem + walkq_offset(cap_max, 2 * W, W, false)) + (size_t)warp * 2 * kWalkQ;
                if (unique) probe_smem<W, 2, true>(tab, Sv, nsv, sink, warp, nwarps, lane, wq, wq + kWalkQ);
                else probe_smem<W, 2, false>(tab, Sv, nsv, sink, warp, nwarps, lane, wq, wq + kWalkQ);
            }
        }
        if constexpr (AGG) {
            flush_acc(jc, acc, true);
        } else if constexpr (Sink::kCheck) {
            flush_acc(jc, sink.acc, false);
            sink.acc = ProbeAcc();
        }
        if (warp == 0) {
            unsigned long long n = idx;
            if (idx == kNone) {
                if (lane == 0) n = atomicAdd(&work->work, 1ull);
                n = __shfl_sync(0xffffffffu, n, 0);
                if (n < ntasks && lane < kTaskWords)
                    ((uint32_t *)&s_task[cur_task ^ 1])[lane] = ((const uint32_t *)(tasks + n))[lane];
            }
            idx = kNone;
            if (lane == 0) {
                s_idx[cur_task ^ 1] = n;
                if (n + 2 * gridDim.x < lead) idx = atomicAdd(&work->work, 1ull);
            }
        }
        __syncthreads();  // every warp is done with this table and has the next task's record
    }
    if constexpr (!AGG) sink.finish();
}

// ========================================================= small build sides
//
// A build relation that fits shared memory whole needs neither a table in global
// memory nor partitions: every CTA builds its own table of all of R (its rows come from
// L2 after the first CTA) and probes its share of S, in one launch instead of three.  What
// bounds it is the build's latency, then a probe's shared-memory work instead of its L2
// sectors: 4097 x 10007 tuples 39.4 -> 32.8 us, 2500 x 2^23 111 -> 56 us.  All ones mark
// empty slots; R's tuples of that key, which no slot can hold, go to a short list.
constexpr uint32_t kSideRids = 64;
template <int W, int NT>
__global__ void __launch_bounds__(NT, join_ctas(NT)) small_join_kernel(const void *R, uint32_t nr, const void *S,
                                                                       uint64_t ns, uint64_t slice, uint32_t cap,
                                                                       void *pairs, uint64_t pcap, hj_counters *ctr,
                                                                       uint32_t stage_at, uint32_t stage_bytes) {
    using T = typename Tup<W>::U;
    using Vec = typename Tup<W>::Vec;
    constexpr int PV = Tup<W>::kPerVec;
    constexpr uint32_t G = SoaTab<W>::G;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ JoinSlot s_slot;
    __shared__ T s_side[kSideRids];
    __shared__ uint32_t s_nside;
    __shared__ int s_full;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nrv = nr / PV;  // whole vectors
    const T ones = Tup<W>::kAllOnes;
    uint32_t *info = (uint32_t *)(smem + (size_t)cap * 2 * W);
    const SoaTab<W> tab{cap / G, ones, (const uint16_t *)info, (const T *)smem, (const T *)smem + cap};
    constexpr int RB = 2;
    Vec rx[RB];
    auto load_r = [&](uint32_t v0) {
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            const uint32_t v = v0 + u * NT;
            if (v < nrv) rx[u] = ld_stream((const Vec *)R + v);
            else if (W == 4 && v * PV < nr) {
                if constexpr (W == 4) {
                    const uint2 y = ((const uint2 *)R)[2 * v];
                    rx[u] = make_uint4(y.x, y.y, 0u, 0u);
                }
            }
        }
    };
    load_r(threadIdx.x);
    // the build rows that follow and the first probe rows into L2 meanwhile
    for (uint32_t i = RB * NT / 8 + threadIdx.x; i * 8u < nrv; i += NT) prefetch_l2((const Vec *)R + i * 8u);
    const uint64_t nsv = ns / PV, s0 = min(blockIdx.x * slice, nsv), s1 = min(s0 + slice, nsv);
    const Vec *Sv = (const Vec *)S + s0;
    for (uint32_t i = threadIdx.x; i < kAheadVecs / 8 && s0 + i * 8u < s1; i += NT) prefetch_l2(Sv + i * 8u);
    const uint4 e4 = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (uint32_t i = threadIdx.x; i < cap * W / 16; i += NT) ((uint4 *)smem)[i] = e4;
    for (uint32_t i = threadIdx.x; i < cap / G / 2; i += NT) info[i] = 0;
    if (threadIdx.x == 0) {
        s_full = 0;
        s_nside = 0;
        s_slot = JoinSlot{pairs, pcap, ctr, 0};
    }
    __syncthreads();
    T *kv = (T *)smem;
    const uint32_t lim = min(tab.nb, kMaxSmemWalk);
    auto tried = [&](uint32_t b) -> uint32_t {
        const uint32_t sh = (b & 1u) * 16u;
        return (atomicAdd(&info[b >> 1], 1u << sh) >> sh) & 0xFFFFu;
    };
    for (uint32_t v0 = threadIdx.x; v0 * PV < nr; v0 += RB * NT) {
        if (v0 != threadIdx.x) load_r(v0);
        T k[RB * PV], r[RB * PV];
        uint32_t bkt[RB * PV], q[RB * PV];
        bool in[RB * PV];
#pragma unroll
        for (int i = 0; i < RB * PV; ++i) {
            const Vec &x = rx[i / PV];
            if constexpr (W == 4) {
                k[i] = i % 2 ? x.z : x.x;
                r[i] = i % 2 ? x.w : x.y;
            } else {
                k[i] = x.x;
                r[i] = x.y;
            }
            in[i] = (v0 + (i / PV) * NT) * PV + i % PV < nr;
            if (in[i] && k[i] == ones) {
                const uint32_t at = atomicAdd(&s_nside, 1u);
                if (at < kSideRids) s_side[at] = r[i];
                else s_full = 1;
                in[i] = false;
            }
            bkt[i] = part_bucket<W>(k[i], tab.nb);
            q[i] = in[i] ? tried(bkt[i]) : 0u;
        }
#pragma unroll
        for (int i = 0; i < RB * PV; ++i) {
            if (!in[i]) continue;
            for (uint32_t it = 1; q[i] >= G && it < lim; ++it) {
                bkt[i] = bkt[i] + 1 == tab.nb ? 0 : bkt[i] + 1;
                q[i] = tried(bkt[i]);
            }
            if (q[i] < G) {
                T *slot = &kv[bkt[i] * G + q[i]];
                slot[0] = k[i];
                slot[cap] = r[i];
            } else {
                s_full = 1;  // a heavily repeated key
            }
        }
    }
    __syncthreads();
    if (s_full) {
        // (near the walk's limit it depends on the order of a CTA's inserts: one CTA that
        // gives up discards the whole attempt)
        if (threadIdx.x == 0) atomicOr(&ctr->status, (unsigned long long)kStatusLongRun);
        return;
    }
    const SideList<W> side{s_side, s_nside};
    const bool unique = s1 - s0 >= 2 * (uint64_t)nrv && !__syncthreads_or(keys_repeat<W, NT>(tab));
    WarpStageSink<W> sink;
    sink.stage = (typename WarpStageSink<W>::P *)(smem + stage_at + warp * stage_bytes);
    sink.scap = stage_bytes / (2 * W);
    sink.slots = &s_slot;
    sink.begin_task(0);
    T *wq = (T *)(smem + walkq_offset(cap, 2 * W, W, false)) + (size_t)warp * 2 * kWalkQ;
    // (slices are below 2^32 vectors: a relation is)
    if (unique)
        probe_smem<W, 2, true, true>(tab, Sv, (uint32_t)(s1 - s0), sink, warp, NT / 32, lane, wq, wq + kWalkQ, side);
    else
        probe_smem<W, 2, false, true>(tab, Sv, (uint32_t)(s1 - s0), sink, warp, NT / 32, lane, wq, wq + kWalkQ, side);
    if constexpr (W == 4) {  // an odd last tuple
        if (ns % 2 && blockIdx.x + 1 == gridDim.x && warp == 0) {
            Vec x[1];
            const uint2 y = ((const uint2 *)S)[ns - 1];
            x[0] = make_uint4(y.x, y.y, 0u, 0u);
            const bool in[2] = {lane == 0, false};
            uint32_t qn = 0;
            probe_group_smem<W, 1, false, false, true>(tab, x, in, sink, lane, wq, wq + kWalkQ, qn, side);
            if (qn) {
                __syncwarp();
                drain_walks<W, false>(tab, wq, wq + kWalkQ, qn, sink);
            }
        }
    }
    sink.finish();
}

// (what a table of two and a half slots per tuple, 8-byte ones 2.4, holds in a CTA's shared
// memory)
uint64_t small_join_rows(int width) { return width == 4 ? 8192 : 4096; }

hj_status small_join(hj_ctx *c, int width, const void *R, uint64_t nr, const void *S, uint64_t ns, void *pairs,
                     uint64_t pcap, hj_counters *ctr) {
    if (!nr || !ns) return HJ_OK;
    const uint64_t pv = width == 4 ? 2 : 1;
    auto slots_for = [&](int nt, uint64_t stage) {
        const uint64_t total = (join_ctas(nt) == 2 ? (112ull << 10) : (222ull << 10)) - 32,
                       fixed = (uint64_t)(nt / 32) * (kWalkQ * 2 * width + stage);
        return (total - fixed) * 8 / (17 * (uint64_t)width) / 128 * 128;
    };
    // Three slots per tuple, two and a half where that keeps two CTAs on an SM; a probe side
    // that one wide CTA per SM covers is bound by the time to build the table, which
    // twice the threads halve.
    const uint64_t nsv = ns / pv, sms = (uint64_t)num_sms(c);
    const uint64_t want = std::max<uint64_t>((3 * nr + 127) / 128 * 128, 128);
    const bool two = nsv > sms * 1280 && nr * 5 / 2 <= slots_for(320, 2048);
    const int nt = two ? 320 : 640;
    const uint64_t stage = want <= slots_for(nt, 4096) ? 4096 : 2048, cap = std::min(want, slots_for(nt, stage));
    const uint64_t queue_at = walkq_offset((uint32_t)cap, (uint32_t)(2 * width), width, false),
                   stage_at = queue_at + (uint64_t)(nt / 32) * kWalkQ * 2 * width,
                   smem = stage_at + (uint64_t)(nt / 32) * stage;
    const uint64_t grid = std::max<uint64_t>(std::min<uint64_t>(sms * join_ctas(nt), (nsv + 2 * nt - 1) / (2 * nt)), 1);
    const uint64_t slice = std::max<uint64_t>(((nsv + grid - 1) / grid + 63) / 64 * 64, 64);
    const unsigned g = (unsigned)std::max<uint64_t>((nsv + slice - 1) / slice, 1);
#define HJ_SM(WW, NT)                                                                                              \
    do {                                                                                                           \
        auto kern = small_join_kernel<WW, NT>;                                                                     \
        HJ_TRY(allow_max_smem(c, (const void *)kern));                                                             \
        HJ_LAUNCH(c, "small_join", kern, g, NT, smem, R, (uint32_t)nr, S, ns, slice, (uint32_t)cap, pairs, pcap, ctr, \
                  (uint32_t)stage_at, (uint32_t)stage);                                                            \
    } while (0)
    if (width == 4) {
        if (two) HJ_SM(4, 320); else HJ_SM(4, 640);
    } else {
        if (two) HJ_SM(8, 320); else HJ_SM(8, 640);
    }
#undef HJ_SM
    return HJ_OK;
}

// Tasks of one join partitioned into NP padded partitions.  Partition p covers
// rows [roff[p], roff[p+1]) of Rp and [soff[p], soff[p+1]) of Sp.  Its S rows are
// cut into slices of at most `slice` rows (a multiple of the sector's tuples, so
// every slice starts on a sector), one task per slice, all with the whole R_p: a
// partition that skew made large is probed by several CTAs at once, each building
// its own copy of the (small) R_p table.  Task p is the first slice of partition
// p; further slices take indices from NP on, handed out by a counter (*next,
// zero at launch; their order does not matter).
__global__ void make_tasks_kernel(const void *Rp, const uint64_t *roff, const void *Sp, const uint64_t *soff,
                                  uint64_t NP, uint64_t slice, uint64_t tail_from, unsigned long long *next,
                                  uint32_t join, int b1, int b2, uint64_t ek1, uint64_t pk1, uint64_t pk2, int tb,
                                  PartTask *tasks) {
    const uint64_t sv = 32 / (uint64_t)tb;
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < NP; p += (uint64_t)gridDim.x * blockDim.x) {
        PartTask t;
        t.R = (const char *)Rp + roff[p] * tb;
        t.nr = (uint32_t)(roff[p + 1] - roff[p]);
        t.join = join;
        t.p = (uint32_t)p;
        t.b1 = (uint16_t)b1;
        t.b2 = (uint16_t)b2;
        t.pad = 0;
        t.ek1 = ek1;
        t.pk1 = pk1;
        t.pk2 = pk2;
        const uint64_t s0 = soff[p], ns = soff[p + 1] - s0;
        // the partitions of the persistent join's last, partly filled round are
        // probed in two halves, so that the round's idle CTAs take the other halves
        uint64_t sl = slice;
        if (p >= tail_from && ns >= 2 * sv) {
            const uint64_t h = ((ns + 1) / 2 + sv - 1) / sv * sv;
            if (h < sl) sl = h;
        }
        const uint64_t extra = ns > sl ? (ns + sl - 1) / sl - 1 : 0;
        const uint64_t base = extra ? NP + atomicAdd(next, (unsigned long long)extra) : 0;
        for (uint64_t i = 0, at = 0; i == 0 || at < ns; ++i, at += sl) {
            t.S = (const char *)Sp + (s0 + at) * tb;
            t.ns = (uint32_t)(ns - at < sl ? ns - at : sl);
            tasks[i == 0 ? p : base + i - 1] = t;
        }
    }
}

uint64_t task_slice_rows(int width, uint64_t n_s, uint64_t NP) {
    // four times the mean partition, at least 2^16 rows, whole sectors
    const uint64_t sv = 32 / tuple_bytes(width);
    uint64_t sl = 4 * ((n_s + NP - 1) / (NP ? NP : 1));
    if (sl < (1ull << 16)) sl = 1ull << 16;
    return (sl + sv - 1) / sv * sv;
}

uint64_t max_tasks(uint64_t NP, uint64_t s_rows, uint64_t slice) { return NP + s_rows / slice + 1; }

uint64_t tail_split_from(hj_ctx *c, int width, int agg, uint64_t NP, uint64_t expect_r) {
    const uint64_t grid = partition_join_ctas(c, width, agg, expect_r), r = grid ? NP % grid : 0;
    return NP < grid || r == 0 ? NP : NP - r;
}

hj_status make_tasks(hj_ctx *c, const void *Rp, const uint64_t *roff, const void *Sp, const uint64_t *soff,
                     uint64_t NP, uint32_t join, int b1, int b2, int width, uint64_t slice, uint64_t ntasks,
                     PartTask *tasks, uint64_t tail_from) {
    const unsigned grid = (unsigned)((NP + 255) / 256);
    // unused task slots stay empty (no rows; the join skips them), and the slice
    // counter just past the array starts at zero
    HJ_CUDA(c, cudaMemsetAsync(tasks, 0, ntasks * sizeof(PartTask) + 8, c->stream));
    HJ_LAUNCH(c, "make_tasks", make_tasks_kernel, grid ? grid : 1, 256, 0, Rp, roff, Sp, soff, NP, slice, tail_from,
              (unsigned long long *)(tasks + ntasks), join, b1, b2, empty_key2(width, b1, b2),
              pass_pad_key(width, 0, b1), b2 ? pass_pad_key(width, b1, b2) : 0ull, (int)tuple_bytes(width), tasks);
    return HJ_OK;
}

// Second empty-marker candidate for pass bits (b1, b2): the first key below the top
// of the key domain whose partition differs from the top key's.  Padding keys of
// the partitioner come from the bottom of the domain (0, 1, 2, ...), so a probe key
// never equals a marker.
uint64_t empty_key2(int width, int b1, int b2) {
    auto pidx = [&](uint64_t k) {
        uint64_t h = width == 4 ? (uint64_t)murmur2_u32((uint32_t)k) : murmur2_u64(k);
        uint64_t d1 = h & ((1ull << b1) - 1), d2 = b2 ? (h >> b1) & ((1ull << b2) - 1) : 0;
        return (d1 << b2) | d2;
    };
    const uint64_t top = width == 4 ? 0xFFFFFFFFull : ~0ull;
    uint64_t k = top - 1;
    while (pidx(k) == pidx(top)) --k;
    return k;
}

// Join launch shape: two CTAs per SM with tables up to 100 KiB, or one of twice the
// threads with up to 209 KiB (aggregates: 200 KiB) when the expected build partition needs
// the room (load factor about 1/3 either way).  The buckets' counts are part of the 209 KiB:
// 25088 4-byte slots, so that partitions of 18e3 build rows keep off the fallback (2^9
// partitions of 17800 / 18300 / 19000 rows, |S| = 2 |R|: 657 / 747 / 860 us; with 200 KiB
// and a load of at most 3/4 1762 / 4080 / 4220 us).  The aggregate join runs 1024 threads
// per SM, the pair join 640: its probe loop holds four tuples' buckets and needs 96
// registers (with 64, 1024 threads spill into an L1 that the tables leave no room: 2^24 x
// 2^28 1257 us against 828, 896 threads 1181, 768 threads 1072, 576 threads 881).
struct JoinCfg {
    int nt;
    uint64_t smem_limit;
};
static uint64_t join_slot_bytes(int width, int agg, int checksum) {
    return agg ? agg_slot_bytes(width, checksum) : 2ull * width;
}
static JoinCfg join_cfg(int width, int agg, int checksum, uint64_t expect_r) {
    const uint64_t slot = join_slot_bytes(width, agg, checksum);
    const uint64_t need = 3 * (expect_r + 6 * (uint64_t)__builtin_sqrt((double)expect_r + 1.0) + 64) * slot;
    if (need <= (100ull << 10)) return JoinCfg{agg ? 512 : 320, 100ull << 10};
    return JoinCfg{agg ? 1024 : 640, agg ? 200ull << 10 : 209ull << 10};
}

// (two CTAs of an SM then cover each other's waits: 200 joins of 3e7 with 1.2e8 tuples 700 us
// in the join kernel, 765 us at twice the rows, one CTA per SM)
uint64_t batch_partition_rows(int width) { return width == 4 ? 2048 : 1024; }

uint64_t partition_join_warps(hj_ctx *c) { return (uint64_t)num_sms(c) * 32; }
uint64_t partition_join_ctas(hj_ctx *c, int width, int agg, uint64_t expect_r) {
    return (uint64_t)num_sms(c) * join_ctas(join_cfg(width, agg, 1, expect_r).nt);
}

hj_status partition_join(hj_ctx *c, int width, int agg, const PartTask *tasks, uint64_t ntasks, uint64_t lead,
                         const JoinSlot *slots, uint64_t expect_r, int checksum, uint32_t *oversize, RecArea ra,
                         bool staged) {
    if (ntasks == 0) return HJ_OK;
    const uint64_t slot_bytes = join_slot_bytes(width, agg, checksum);
    const JoinCfg cfg = join_cfg(width, agg, checksum, expect_r);
    // Capacity: room for a partition of the expected size plus six standard
    // deviations at load factor 1/3 (whole buckets), within the shape's budget.
    const double mean = (double)expect_r;
    uint64_t want = (uint64_t)(3.0 * (mean + 6.0 * __builtin_sqrt(mean + 1.0) + 64.0));
    want = (want + 127) / 128 * 128;
    const uint64_t bitmap_bytes = 4096;
    // the pair join adds each warp's walk queue, and staged output its buffer when that is in
    // shared memory, within what the shape's CTAs per SM can have
    const uint64_t warps = (uint64_t)(cfg.nt / 32), total_max = join_ctas(cfg.nt) == 2 ? (112ull << 10) : (222ull << 10);
    const uint64_t queues = agg ? 0 : warps * kWalkQ * 2 * width;
    auto slots_beside = [&](uint64_t extra) {
        const uint64_t budget = std::min<uint64_t>(cfg.smem_limit + extra, total_max) - extra;
        return agg ? (budget - bitmap_bytes) / slot_bytes / 128 * 128
                   : (budget - 16) * 8 / (8 * slot_bytes + (uint64_t)width) / 128 * 128;
    };
    uint64_t stage_bytes = staged ? warps * kJoinStageBytes : 0;
    // Staging takes up to 80 KB that a large build partition needs: past a load of 0.46 the
    // buffers go to global memory (u32 14e6 / 2^24 / 18e6 / 22e6 build rows on 2^11
    // partitions 641 / 746 / 797 / 1258 us in shared memory, 678 / 727 / 743 / 953 us in
    // global; u64 6e6 / 7e6 / 8e6 / 10e6 786 / 866 / 1170 / 1893 and 811 / 858 / 1099 / 1217)
    // and the tables hold as many rows as those of a single join.
    const bool in_global = staged && join_ctas(cfg.nt) == 1 && mean > 0.46 * (double)slots_beside(queues + stage_bytes);
    if (in_global) stage_bytes = 0;
    const uint64_t max_slots = slots_beside(queues + stage_bytes);
    uint64_t cap_max = want < max_slots ? want : max_slots;
    if (cap_max < 128) cap_max = 128;
    const size_t smem = (size_t)walkq_offset((uint32_t)cap_max, (uint32_t)slot_bytes, width, agg != 0) +
                        (size_t)(queues + stage_bytes);
    unsigned grid = (unsigned)num_sms(c) * join_ctas(cfg.nt);
    if (grid > ntasks) grid = (unsigned)ntasks;
    DevBuf gstage(c);  // (freed in stream order after the launch)
    if (in_global) HJ_TRY(gstage.alloc((uint64_t)grid * warps * kJoinStageBytes));
#define HJ_PJ(WW, AA, NT, SK)                                                                                         \
    do {                                                                                                              \
        auto kern = partition_join_kernel<WW, AA, NT, SK<WW>>;                                                        \
        HJ_TRY(allow_max_smem(c, (const void *)kern));                                                                \
        HJ_LAUNCH(c, "partition_join", kern, grid, NT, smem, tasks, ntasks, lead, slots, c->d_ctr, (uint32_t)cap_max, \
                  ra, oversize, checksum, (uint32_t)(smem - stage_bytes), gstage.p);                                  \
    } while (0)
#define HJ_PJ_NT(WW, AA, SK)                                             \
    do {                                                                 \
        if (join_ctas(cfg.nt) == 2) HJ_PJ(WW, AA, (AA ? 512 : 320), SK); \
        else HJ_PJ(WW, AA, (AA ? 1024 : 640), SK);                       \
    } while (0)
#define HJ_PJ_SK(WW)                                                     \
    do {                                                                 \
        if (!staged && checksum) HJ_PJ_NT(WW, false, ChunkCheckSink);    \
        else if (!staged) HJ_PJ_NT(WW, false, ChunkSink);                \
        else if (in_global && checksum) HJ_PJ(WW, false, 640, GlobalStageCheckSink); \
        else if (in_global) HJ_PJ(WW, false, 640, GlobalStageSink);      \
        else if (checksum) HJ_PJ_NT(WW, false, WarpStageCheckSink);      \
        else HJ_PJ_NT(WW, false, WarpStageSink);                         \
    } while (0)
    if (width == 4) {
        if (agg) HJ_PJ_NT(4, true, ChunkSink); else HJ_PJ_SK(4);
    } else {
        if (agg) HJ_PJ_NT(8, true, ChunkSink); else HJ_PJ_SK(8);
    }
#undef HJ_PJ
#undef HJ_PJ_NT
#undef HJ_PJ_SK
    return HJ_OK;
}

}  // namespace hj
