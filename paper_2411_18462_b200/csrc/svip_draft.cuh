// Draft side: combining the segment partials of a row, the fine scan that finds the sampled token,
// the draft-step kernel (Algorithm 1 inner loop, Eq. 7) and the row-statistics kernel (first phase of verify).
#pragma once

#include "svip_device.cuh"
#include "svip.h"

namespace svip {

constexpr int kPolicyThreads = 256;

struct SegEntry {
    float m;
    int idx;
    float Z;
    float A;
};

// The entries of a row as rescaled_entries reads them: a block-local table that the warps of the cluster have filled.
struct LocalSegments {
    const SegEntry* all;
    __device__ __forceinline__ SegEntry operator()(int s) const { return all[s]; }
};

// The entries that a lane owns (segments lane * per ...), moved to the row's maximum, which is returned.
template <int kMode, class Source>
__device__ __forceinline__ float rescaled_entries(const Source& src, int nseg, int per, float c, int lane,
                                                  Partial (&e)[kSegPerLane]) {
    float m = neg_inf();
#pragma unroll
    for (int k = 0; k < kSegPerLane; ++k) {
        e[k].m = neg_inf(); e[k].idx = kIntMax; e[k].Z = 0.f; e[k].A = 0.f;
        int s = lane * per + k;
        if (k < per && s < nseg) {
            SegEntry v = src(s);
            e[k].m = v.m; e[k].idx = v.idx; e[k].Z = v.Z; e[k].A = v.A;
        }
        m = fmaxf(m, e[k].m);
    }
    m = warp_max(m);
#pragma unroll
    for (int k = 0; k < kSegPerLane; ++k) {
        if (e[k].m != m) e[k].idx = kIntMax;
        rescale_to<kMode>(e[k], m, c);
    }
    return m;
}

// Selects the segment holding the mass u * Z of the row; returns the row's maximum.  Warp-collective; every warp
// that runs it on the same entries gets the same bits.
template <class Source>
__device__ __forceinline__ float pick_entry(const Source& src, int nseg, float c, float u, int lane, SegPick& pick,
                                            float abs_target = -1.f) {
    const int per = (nseg + 31) / 32;
    Partial e[kSegPerLane];
    const float m = rescaled_entries<1>(src, nseg, per, c, lane, e);
    float mass[kSegPerLane];
#pragma unroll
    for (int k = 0; k < kSegPerLane; ++k) mass[k] = e[k].Z;
    pick = pick_segment(mass, per, nseg, u, lane, abs_target);
    return m;
}

// Merges the nseg segment entries of a row into the row's partial.  Warp-collective.
template <int kMode, class Source>
__device__ __forceinline__ Partial merge_entries(const Source& src, int nseg, float c, int lane) {
    Partial e[kSegPerLane], row;
    row.m = rescaled_entries<kMode>(src, nseg, (nseg + 31) / 32, c, lane, e);
    int idx = kIntMax;
    float Z = 0.f, A = 0.f;
#pragma unroll
    for (int k = 0; k < kSegPerLane; ++k) {
        idx = min(idx, e[k].idx);
        Z += e[k].Z;
        A += e[k].A;
    }
    row.idx = warp_min_int(idx);
    row.Z = kMode >= 1 ? warp_sum(Z) : 0.f;
    row.A = kMode == 2 ? warp_sum(A) : 0.f;
    return row;
}

// The segment entries of a row, pushed by the warps that produced them into every block of the
// cluster (see the exchange primitives in svip_device.cuh).
struct alignas(16) SegExchange {
    SegEntry all[kMaxSeg];     // entry of segment s at index s
    unsigned long long bar;    // mbarrier: completes when S * kWarps entries have landed here
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// To be run by every thread of every block of the cluster before the row is streamed.
__device__ __forceinline__ void exchange_open(SegExchange& ex, int S, int tid) {
    if (S == 1) return;
    if (tid == 0) {
        const uint32_t bar = smem_addr(&ex.bar);
        mbar_init(bar, 1);
        mbar_arrive_expect_tx(bar, static_cast<uint32_t>(S * kWarps * sizeof(SegEntry)));
    }
    cluster_arrive_relaxed();   // a peer pushes only after its cluster_wait(), hence after this initialisation
}

// The calling warp sends the entry of its segment (rank * kWarps + warp) to every block of a cluster of S > 1.
__device__ __forceinline__ void exchange_send(SegExchange& ex, int S, int rank, int warp, int lane, const Partial& t) {
    if (lane < S) {
        const uint32_t dst = map_to_rank(smem_addr(&ex.all[rank * kWarps + warp]), lane);
        const uint32_t bar = map_to_rank(smem_addr(&ex.bar), lane);
        push16(dst, bar, __float_as_uint(t.m), static_cast<uint32_t>(t.idx), __float_as_uint(t.Z), __float_as_uint(t.A));
    }
}

// The calling warp publishes the entry of its segment, the first push after exchange_open().
__device__ __forceinline__ void exchange_push(SegExchange& ex, int S, int rank, int warp, int lane, const Partial& t) {
    if (S == 1) {
        if (lane == 0) { SegEntry& e = ex.all[warp]; e.m = t.m; e.idx = t.idx; e.Z = t.Z; e.A = t.A; }
        return;
    }
    cluster_wait();
    exchange_send(ex, S, rank, warp, lane, t);
}

// Until all entries are here (S > 1; bounded): false if the wait ran out.
__device__ __forceinline__ bool exchange_wait(SegExchange& ex) {
    return mbar_wait_bounded(smem_addr(&ex.bar), 0);
}

// The same exchange for kernels that need several, one after another (rounds 0, 1, ...).  Tables and mbarriers alternate.
// Warp 0 of a block waits for the entries of a round and reads them, then the block passes a barrier, then its warps
// publish their entries of the next round; a block publishes round r + 2 only when it holds all entries of round
// r + 1, so a table is never written while it is read.
struct alignas(16) RoundExchange {
    SegEntry all[2][kMaxSeg];
    unsigned long long bar[2];
};

__device__ __forceinline__ void rounds_arm(RoundExchange& ex, int b, int S) {
    mbar_arrive_expect_tx(smem_addr(&ex.bar[b]), static_cast<uint32_t>(S * kWarps * sizeof(SegEntry)));
}

// To be run by every thread of every block of the cluster; needs no global memory.
__device__ __forceinline__ void rounds_open(RoundExchange& ex, int S, int tid) {
    if (S == 1) return;
    if (tid == 0) {
        mbar_init(smem_addr(&ex.bar[0]), 1);
        mbar_init(smem_addr(&ex.bar[1]), 1);
        rounds_arm(ex, 0, S);
        rounds_arm(ex, 1, S);
    }
    cluster_arrive_relaxed();     // waited for by the publishers of round 0
}

__device__ __forceinline__ void rounds_publish(RoundExchange& ex, int S, int rank, int round, int warp, int lane, const Partial& t) {
    SegEntry* table = ex.all[round & 1];
    if (S == 1) {
        if (lane == 0) { SegEntry& e = table[warp]; e.m = t.m; e.idx = t.idx; e.Z = t.Z; e.A = t.A; }
        return;
    }
    if (round == 0) cluster_wait();
    if (lane < S)
        push16(map_to_rank(smem_addr(&table[rank * kWarps + warp]), lane), map_to_rank(smem_addr(&ex.bar[round & 1]), lane),
               __float_as_uint(t.m), static_cast<uint32_t>(t.idx), __float_as_uint(t.Z), __float_as_uint(t.A));
}

// The entries of the round, once all are here (bounded wait: the status word tells if they are not).  To be called by
// every thread; only warp 0 may read the entries.
__device__ __forceinline__ LocalSegments rounds_wait(RoundExchange& ex, int S, int round, int tid, unsigned* status) {
    const int b = round & 1;
    if (S == 1) {
        __syncthreads();
    } else if (tid < 32) {
        if (!mbar_wait_bounded(smem_addr(&ex.bar[b]), (round >> 1) & 1) && tid == 0) atomicOr(status, SVIP_STATUS_WAIT_TIMEOUT);
        if (tid == 0) rounds_arm(ex, b, S);       // for round + 2, whose first entry comes after this block's next ones
    }
    return LocalSegments{ex.all[b]};
}

// One round whose entries are masses: the segment that holds the mass u * total, the same in every block.
// `pick` is shared scratch.  Ends with a block barrier.
__device__ __forceinline__ void rounds_pick(RoundExchange& ex, int S, int rank, int round, int tid, float mass_of_warp, float u,
                                            SegPick& pick, unsigned* status) {
    const int lane = tid & 31, warp = tid >> 5;
    Partial t;
    t.m = 0.f; t.idx = 0; t.Z = mass_of_warp; t.A = 0.f;
    rounds_publish(ex, S, rank, round, warp, lane, t);
    const LocalSegments entries = rounds_wait(ex, S, round, tid, status);
    if (warp == 0) {
        const int nseg = S * kWarps;
        const int per = (nseg + 31) / 32;
        float mass[kSegPerLane];
#pragma unroll
        for (int k = 0; k < kSegPerLane; ++k) {
            const int s = lane * per + k;
            mass[k] = k < per && s < nseg ? entries.all[s].Z : 0.f;
        }
        const SegPick p = pick_segment(mass, per, nseg, u, lane);
        if (lane == 0) pick = p;
    }
    __syncthreads();
}

// Fine scan of one segment by the whole block.  The functor splits into `load(vi)` (the raw 16-byte
// vectors of element-vector vi) and `weights(vi, raw, w)` (their weights), so that a thread issues all
// its loads at once and keeps them in registers; `element(vi, j)` is the weight of element j of vector
// vi alone.  Each thread sums a run of consecutive vectors, one block scan places the runs, and the warp
// that starts at or below `target` and has a lane whose run ends above it looks at the elements of that run
// side by side, one per lane.  Returns the virtual element index (vector * EPV + element) of the first
// element whose cumulative weight exceeds `target`, else (rounding) the last element with positive weight
// before that point, else -1.  All threads return the same value.
// Bound by its chain of dependent steps, which is why the elements are not walked one after another by one thread,
// warps that start above the target do nothing, and the winner is an integer minimum (512-thread block, 150 vectors in
// shared memory: 1.6 -> 0.9 us).
template <int EPV, class WF>
__device__ __forceinline__ int fine_scan(const WF& wf, int v_lo, int v_hi, float prefix, float target,
                                         ScanShared& sh, int tid, int lane, int warp) {
    constexpr int kRun = 4;
    constexpr unsigned kNone = ~0u;
    const int nv = v_hi - v_lo;
    const int run = min(kRun, max(1, (nv + kThreads - 1) / kThreads));
    if (tid == 0) { sh.key = kNone; sh.lastpos = -1; sh.result = -1; }
    float running = prefix;
    target = fmaxf(target, prefix);     // the segment was picked for it, up to rounding
    for (int cb = v_lo; cb < v_hi; cb += kThreads * run) {
        const int first = cb + tid * run;
        float ls = 0.f;
        int lastv = -1;
        auto add = [&](int vi, const typename WF::Raw& raw) {
            float w[EPV];
            wf.weights(vi, raw, w);
            float sv = 0.f;
#pragma unroll
            for (int j = 0; j < EPV; ++j) sv += w[j];
            if (sv > 0.f) lastv = vi;
            ls += sv;
        };
        if (run == 1) {
            if (first < v_hi) add(first, wf.load(first));
        } else {
            typename WF::Raw raw[kRun];
#pragma unroll
            for (int k = 0; k < kRun; ++k)
                if (k < run && first + k < v_hi) raw[k] = wf.load(first + k);
#pragma unroll
            for (int k = 0; k < kRun; ++k)
                if (k < run && first + k < v_hi) add(first + k, raw[k]);
        }
        const float inc = warp_scan_incl(ls, lane);
        if (cb != v_lo) __syncthreads();   // wsum is free again
        if (lane == 31) sh.wsum[warp] = inc;
        __syncthreads();
        float before = 0.f, total = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float sw = sh.wsum[w];
            if (w < warp) before += sw;
            total += sw;
        }
        if (running + before <= target) {     // warp-uniform; the warps after the one that holds the target stay out
            const float lo = running + (before + (inc - ls));
            const unsigned crossing = __ballot_sync(0xffffffffu, ls > 0.f && lo + ls > target);
            unsigned some = 0;
            if (crossing) {
                // lane (k, j) = (lane / EPV, lane % EPV) takes element j of vector k of the crossing run
                const int src = __ffs(crossing) - 1;
                const float start = __shfl_sync(0xffffffffu, lo, src);
                const int vi = __shfl_sync(0xffffffffu, first, src) + lane / EPV;
                const float e = lane / EPV < run && vi < v_hi ? wf.element(vi, lane % EPV) : 0.f;
                const float cum = start + warp_scan_incl(e, lane);
                some = __ballot_sync(0xffffffffu, e > 0.f);
                const unsigned over = __ballot_sync(0xffffffffu, e > 0.f && cum > target);
                if (lane == (over ? __ffs(over) - 1 : 31 - __clz(some)))
                    atomicMin(&sh.key, static_cast<unsigned>(vi * EPV + lane % EPV));
            }
            if (!some) {      // also where a run has a sum at rounding level but no element of its own
                const int lv = __reduce_max_sync(0xffffffffu, lastv);
                if (lane == 0 && lv >= 0) atomicMax(&sh.lastpos, lv);
            }
        }
        __syncthreads();
        const unsigned key = sh.key;
        if (key != kNone) return static_cast<int>(key);
        running += total;
    }
    // rounding left nothing above the target: the last element with weight
    const int lv = sh.lastpos;
    if (lv < 0) return -1;
    if (tid == 0) {
        float w[EPV];
        wf.weights(lv, wf.load(lv), w);
        int last = -1;
#pragma unroll
        for (int j = 0; j < EPV; ++j)
            if (w[j] > 0.f) last = lv * EPV + j;
        sh.result = last;
    }
    __syncthreads();
    return sh.result;
}

// ------------------------------------------------------------------ draft step

// Control of a drafting loop recorded as a WHILE node of a CUDA graph.  The kernel that closes an
// iteration counts it and tells the graph whether the body runs again: only while sequences are
// still drafting, and never more than `max_iters` times whatever the data say.
struct LoopCtl {
    cudaGraphConditionalHandle handle;
    int* iter;        // iterations done since the loop was entered (NULL: not inside a loop)
    int max_iters;
};

__device__ __forceinline__ void loop_decide(const LoopCtl& loop, int n_active) {
    if (!loop.iter) return;
    const int it = *loop.iter + 1;
    *loop.iter = it;
    cudaGraphSetConditional(loop.handle, (n_active > 0 && it < loop.max_iters) ? 1u : 0u);
}

struct AdvanceArgs {
    int policy;
    const uint8_t* stop;
    const int32_t* gamma;
    int32_t* draft_len;
    uint8_t* active;
    int B, K_cap;
    int32_t* n_active;
    LoopCtl loop;
    unsigned long long* arrived;   // in the draft kernel: sequences done (low word), of them still drafting (high word)
};

// Whether sequence i, now with `len` draft tokens, stops drafting.
__device__ __forceinline__ bool drafting_done(const AdvanceArgs& a, int i, int len, bool stopped) {
    return a.policy == SVIP_POLICY_ENTROPY ? stopped || len >= a.K_cap : len >= min(a.gamma[i], a.K_cap);
}

// What the arrival that makes the counter `sum` (sequences counted in the low word, of them still drafting in the high one)
// means for a batch of B: it closes the iteration if it is the last one.  A counter that runs past the batch holds arrivals
// of another replay of the context's loop: the iteration is closed and the loop ended (nobody goes on), since the counts
// mean nothing any more and a loop that nobody decides would not end.
struct LoopArrival {
    bool closes, overrun;
    int going;
};
__host__ __device__ __forceinline__ LoopArrival loop_arrival(unsigned long long sum, int B) {
    const unsigned n = static_cast<unsigned>(sum);
    LoopArrival r;
    r.closes = n >= static_cast<unsigned>(B);
    r.overrun = n > static_cast<unsigned>(B);
    r.going = r.overrun ? 0 : static_cast<int>(sum >> 32);
    return r;
}

// The policy step of one sequence, taken by the draft kernel that drafted its token (one thread per sequence, those
// that have stopped included).  The last one to arrive knows how many sequences go on and decides the loop.
__device__ __forceinline__ void advance_one(const AdvanceArgs& a, int i, bool drafted, int len, bool stopped, unsigned* status) {
    bool going = false;
    if (drafted) {
        going = !drafting_done(a, i, len, stopped);
        a.draft_len[i] = len;
        if (!going) a.active[i] = 0;
    }
    const unsigned long long mine = 1ull + (going ? 1ull << 32 : 0ull);
    const LoopArrival r = loop_arrival(atomicAdd(a.arrived, mine) + mine, a.B);
    if (r.closes) {
        atomicExch(a.arrived, 0ull);
        if (r.overrun) atomicOr(status, SVIP_STATUS_LOOP_OVERLAP);
        *a.n_active = r.going;
        loop_decide(a.loop, r.going);
    }
}

struct DraftArgs {
    const void* logits;
    long row_stride;
    int V;
    float c;          // log2(e) / T   (T = 1 when greedy)
    float thresh;
    int greedy;
    const float* uniforms;
    int32_t* token;
    float* entropy;
    uint8_t* stop;
    float* row_stats;
    unsigned* status;
    const uint8_t* active;   // NULL, or one flag per row: rows with 0 are skipped
    const float* ext_target; // NULL, or per row the mass to find (units of this row's own Z), see svip_vp_locate
    int token_offset;        // added to the sampled index (vocabulary shard offset)
    const int32_t* pos;      // NULL, or per row the draft position p whose logits are read (svip_draft_step_at)
    long pos_stride;         // elements between the logits of consecutive positions of a row
    long slot_stride;        // uniforms / token / entropy / row_stats live at index p * slot_stride + row
    const float* thr;        // NULL, or per row the truncation threshold: only logits >= thr[row] count
    AdvanceArgs adv;         // position-indexed form in a drafting loop: the policy step, if adv.arrived is not NULL
};

template <int DT>
struct SoftmaxWeights {
    RowGeom g;
    const void* row;
    float c, M;
    float thr = -INFINITY;   // logits below it carry no weight (truncated distributions)
    uint32_t ring = 0;       // ring slots of the warp that streamed the segment, and the vectors that are still there
    int ring_lo = 0, ring_hi = 0;
    typedef uint4 Raw;
    __device__ __forceinline__ Raw load(int vi) const {
        const int o = vi - ring_lo;
        if (o >= 0 && vi < ring_hi) return lds128(ring + (o >> 5) * (kThreads * 16) + (o & 31) * 16);
        return ld_vec(g.base + vi);
    }
    __device__ __forceinline__ void weights(int vi, const Raw& raw, float (&w)[ElemTraits<DT>::kEPV]) const {
        constexpr int EPV = ElemTraits<DT>::kEPV;
        float x[EPV];
        unpack_masked<DT>(raw, vi, g, x);
#pragma unroll
        for (int j = 0; j < EPV; ++j)
            w[j] = x[j] >= thr ? ex2_approx(fmaxf(__fmaf_rn(x[j], c, -M), kArgFloor)) : 0.f;
    }
    __device__ __forceinline__ float element(int vi, int j) const {
        const int i = vi * ElemTraits<DT>::kEPV + j - g.pre;
        if (i < 0 || i >= g.V) return 0.f;
        const int o = vi - ring_lo;
        const float x = o >= 0 && vi < ring_hi
            ? ElemTraits<DT>::lds_one(ring + (o >> 5) * (kThreads * 16) + (o & 31) * 16 + j * ElemTraits<DT>::kBytes)
            : ElemTraits<DT>::load_one(row, i);
        return x >= thr ? ex2_approx(fmaxf(__fmaf_rn(x, c, -M), kArgFloor)) : 0.f;
    }
};

struct RowShared {
    float m;
    SegPick pick;
};

// The draft step of one row by the cluster that shares it: stream the row (Z, A, maximum), push the
// segment partials to every block of the cluster, combine them (every block the same bits), write
// entropy / stop flag / normalisers, and let the block that holds the sampled mass find the token.
// `g` describes the row, `thr` is the truncation threshold when kThr; the caller has opened `ex`.
// No block reads a peer's shared memory, and a block leaves only after every entry aimed at it has landed.
// Launches of up to about 128 rows are bound by the latency of this chain, not by bytes.  Hence: a segment
// that fits the ring is scanned where it lies; the pick of the segment (warp 0 of every block) does not wait
// for the entropy, which warp 1 of block 0 forms beside it; whatever needs no logits is done before the
// predecessor has finished (row geometry, barriers, L2 prefetch).  One step at 1 x 32000 fp32 4.4 -> 3.1 us,
// 1 x 152064 bf16 5.2 -> 3.8, 32 x 152064 8.2 -> 5.9, 128 x 152064 13.9 -> 11.5 (graph of 64 steps).
template <int DT, bool kGreedy, bool kPos, bool kThr>
__device__ __forceinline__ void draft_row(const DraftArgs& a, int S, int rank, int row, int tid, const RowGeom g,
                                          const LaneSpan& span, const uint32_t slot0, const long p, const float thr,
                                          SegExchange& ex) {
    constexpr int EPV = ElemTraits<DT>::kEPV;
    const int lane = tid & 31, warp = tid >> 5;
    const int seg = rank * kWarps + warp;
    __shared__ ScanShared scan;
    __shared__ RowShared res;
    float u = 0.f, ext = -1.f;
    if (!kGreedy && warp == 0) {   // fetched now, used after the stream
        if (a.ext_target) ext = fmaxf(__ldg(a.ext_target + row), 0.f);
        else u = __ldg(a.uniforms + (row + p * a.slot_stride));
    }
    const Partial t = reduce_segment<DT, 2, kGreedy, kThr>(g, span, seg, a.c, lane, slot0, thr);
    pdl_launch_dependents();
    exchange_push(ex, S, rank, warp, lane, t);
    if (S == 1) __syncthreads();
    const LocalSegments entries{ex.all};
    const bool summarises = rank == 0 && warp == 1;
    if (S > 1 && (warp == 0 || summarises) && !exchange_wait(ex) && lane == 0) atomicOr(a.status, SVIP_STATUS_WAIT_TIMEOUT);
    if (summarises) {       // beside the pick and the scan: everything but the sampled token
        const Partial r = merge_entries<2>(entries, S * kWarps, a.c, lane);
        if (lane == 0) {
            const long slot = row + p * a.slot_stride;      // where this row's outputs live
            const bool ok = (r.Z > 0.f) && (fabsf(r.m) <= kMaxLogit);
            float H = 0.f;
            if (ok) H = fmaxf(kLn2 * (log2f(r.Z) - r.A / r.Z), 0.f);
            else atomicOr(a.status, SVIP_STATUS_NONFINITE_ROW);
            if (a.entropy) a.entropy[slot] = H;
            if (a.stop) a.stop[row] = __fsqrt_rn(H) > a.thresh ? 1 : 0;
            if (a.row_stats) { a.row_stats[2 * slot] = r.m; a.row_stats[2 * slot + 1] = r.Z; }
            if (kGreedy || !ok) a.token[slot] = ((r.idx >= 0 && r.idx < a.V) ? r.idx : 0) + a.token_offset;
            // every warp of the cluster has read the position and the flag: their entries are here
            if (kPos && a.adv.arrived) advance_one(a.adv, row, true, static_cast<int>(p) + 1, __fsqrt_rn(H) > a.thresh, a.status);
        }
    }
    if (kGreedy) return;    // warp 0 has seen all entries land, so the block may leave
    if (warp == 0) {
        SegPick pk;
        const float m = pick_entry(entries, S * kWarps, a.c, u, lane, pk, ext);
        if (lane == 0) { res.m = m; res.pick = pk; }
    }
    __syncthreads();        // res is visible block-wide
    const SegPick P = res.pick;
    const bool ok = (P.total > 0.f) && (fabsf(res.m) <= kMaxLogit);
    if (ok && P.seg / kWarps == rank) {
        SoftmaxWeights<DT> wf;
        wf.g = g; wf.c = a.c; wf.M = __fmul_rn(res.m, a.c); wf.thr = thr;
        wf.row = reinterpret_cast<const char*>(g.base) + g.pre * ElemTraits<DT>::kBytes;
        wf.ring = slot0 - tid * 16 + (P.seg % kWarps) * 512;
        int lo, hi;
        seg_range(g, P.seg, lo, hi);
        wf.ring_lo = lo + (lo == 0 && g.pre > 0 ? 1 : 0);
        wf.ring_hi = hi - (hi == g.nvec && ((g.pre + g.V) % EPV) != 0 ? 1 : 0);
        if (wf.ring_hi - wf.ring_lo > 32 * kStages) wf.ring_hi = wf.ring_lo;
        const int virt = fine_scan<EPV>(wf, lo, hi, P.prefix, P.target, scan, tid, lane, warp);
        if (tid == 0) a.token[row + p * a.slot_stride] = (virt >= 0 ? virt - g.pre : 0) + a.token_offset;
    }
}

// kBlocks is the number of blocks the register budget must leave room for on one SM: 2 for
// launches that fit the GPU in one wave (latency matters, registers are free), 3 for launches of
// many waves, where a third resident block streams on while another one is in its epilogue.
// kPos compiles the position-indexed form (svip_draft_step_at) in, kThr the truncated form
// (svip_draft_step_filtered).
template <int DT, bool kGreedy, int kBlocks, bool kPos = false, bool kThr = false>
__global__ void __launch_bounds__(kThreads, kBlocks) draft_step_kernel(DraftArgs a) {
    extern __shared__ __align__(kRingAlign) uint4 ring[];
    cg::cluster_group cluster = cg::this_cluster();
    const int S = cluster.dim_blocks().x;
    const int rank = cluster.block_rank();
    const int row = blockIdx.x / S;
    const int tid = threadIdx.x;

    const char* rp = static_cast<const char*>(a.logits) +
                     static_cast<size_t>(row) * a.row_stride * ElemTraits<DT>::kBytes;
    RowGeom g = make_geom<DT>(rp, a.V, S * kWarps);
    const uint32_t slot0 = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + tid * 16;
    const int lane = tid & 31, seg = rank * kWarps + (tid >> 5);
    LaneSpan span = lane_span<DT>(g, seg, lane);
    __shared__ SegExchange ex;
    exchange_open(ex, S, tid);
    // which rows a masked or position-indexed launch reads is not known yet
    if (!kPos && !a.active && lane == 0) prefetch_segment(g, seg, kRingBytes / kWarps);
    pdl_wait();
    if (a.active && !a.active[row]) {          // the whole cluster leaves together
        if (S > 1) cluster_wait();
        if (kPos && a.adv.arrived && rank == 0 && tid == 0) advance_one(a.adv, row, false, 0, false, a.status);
        return;
    }
    long p = 0;
    if (kPos) {
        p = a.pos[row];
        rp += p * a.pos_stride * ElemTraits<DT>::kBytes;
        g = make_geom<DT>(rp, a.V, S * kWarps);
        span = lane_span<DT>(g, seg, lane);
    }
    const float thr = kThr ? a.thr[row] : neg_inf();
    draft_row<DT, kGreedy, kPos, kThr>(a, S, rank, row, tid, g, span, slot0, p, thr, ex);
}

// ------------------------------------------------------------------ row statistics (verify, phase 1)

struct StatsArgs {
    const void* logits;
    long row_stride;
    int V;
    float c;
    int draft_rows;          // 0: unit = row.  1: unit = (sequence, position) of a draft row
    int K;
    const int32_t* cu;
    long q_seq_stride, q_pos_stride;
    float2* out_stats;       // (m, Z) per row, indexed by target-row number
    int32_t* out_argmax;
    unsigned* status;
    float4* out_partial;     // kMode 2: (m, Z, A, index of the maximum + idx_offset as int bits)
    int idx_offset;
    const float* thr;        // kThr: truncation threshold per row (target rows: by target row; draft rows: by draft row)
};

template <int DT, int kMode, bool kThr = false>
__global__ void __launch_bounds__(kThreads, 2) row_stats_kernel(StatsArgs a) {
    cg::cluster_group cluster = cg::this_cluster();
    const int S = cluster.dim_blocks().x;
    const int rank = cluster.block_rank();
    const int unit = blockIdx.x / S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ SegExchange ex;      // used in block 0, which receives the entries of the whole cluster
    extern __shared__ __align__(kRingAlign) uint4 ring[];
    const uint32_t slot0 = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + tid * 16;

    if (S > 1) {
        if (rank == 0 && tid == 0) {
            mbar_init(smem_addr(&ex.bar), 1);
            mbar_arrive_expect_tx(smem_addr(&ex.bar), static_cast<uint32_t>(S * kWarps * sizeof(SegEntry)));
        }
        cluster_arrive_relaxed();
    }
    const int my_seg = rank * kWarps + warp;
    long in_row = unit;
    int out_row = unit;
    pdl_wait();
    if (a.draft_rows) {
        int i = unit / a.K, j = unit - i * a.K;
        int row0 = a.cu ? a.cu[i] : i * (a.K + 1);
        int Ki = a.cu ? a.cu[i + 1] - row0 - 1 : a.K;
        if (j >= Ki) {         // the whole cluster leaves together
            if (S > 1) cluster_wait();
            return;
        }
        in_row = a.q_seq_stride < 0 ? static_cast<long>(row0 - i + j)
                                    : i * a.q_seq_stride + j * a.q_pos_stride;
        out_row = row0 + j;
    }
    const RowGeom g = make_geom<DT>(static_cast<const char*>(a.logits) +
                                        static_cast<size_t>(in_row) * a.row_stride * ElemTraits<DT>::kBytes, a.V, S * kWarps);
    const float thr = kThr ? a.thr[in_row] : neg_inf();
    const Partial t = reduce_segment<DT, kMode, kMode != 1, kThr>(g, my_seg, a.c, lane, slot0, thr);
    pdl_launch_dependents();
    if (S == 1) {
        if (lane == 0) { SegEntry& e = ex.all[warp]; e.m = t.m; e.idx = t.idx; e.Z = t.Z; e.A = t.A; }
        __syncthreads();
    } else {
        cluster_wait();        // block 0's barrier is ready
        if (lane == 0)
            push16(map_to_rank(smem_addr(&ex.all[my_seg]), 0), map_to_rank(smem_addr(&ex.bar), 0), __float_as_uint(t.m),
                   static_cast<uint32_t>(t.idx), __float_as_uint(t.Z), __float_as_uint(t.A));
    }
    // nothing is sent to the other blocks, and block 0 stays until everything sent to it has landed
    if (rank == 0 && warp == 0) {
        if (S > 1 && !exchange_wait(ex) && lane == 0) atomicOr(a.status, SVIP_STATUS_WAIT_TIMEOUT);
        const Partial r = merge_entries<kMode>(LocalSegments{ex.all}, S * kWarps, a.c, lane);
        if (lane == 0) {
            bool ok = fabsf(r.m) <= kMaxLogit && (kMode == 0 || r.Z > 0.f);
            if (!ok && kMode != 2) atomicOr(a.status, SVIP_STATUS_NONFINITE_ROW);   // a shard may be all masked
            if (kMode == 1) a.out_stats[out_row] = make_float2(r.m, r.Z);
            if (kMode == 2) {
                int gi = ((r.idx >= 0 && r.idx < a.V) ? r.idx : 0) + a.idx_offset;
                a.out_partial[out_row] = make_float4(r.m, ok ? r.Z : 0.f, ok ? r.A : 0.f, __int_as_float(gi));
            }
            if (a.out_argmax) a.out_argmax[out_row] = (r.idx >= 0 && r.idx < a.V) ? r.idx : 0;
        }
    }
}

}  // namespace svip
