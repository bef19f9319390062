// Truncation threshold of a logits row (top-k and nucleus / top-p).
//
// The kept set of a row is {i : l_i >= tau}: tau_k is the k-th largest logit, and inside that set
// tau is the largest logit value v for which the mass of {l_i >= v} reaches top_p of the mass of
// {l_i >= tau_k}; tokens tied with the last kept one are all kept.  The paper applies its length
// policy on top of samplers that truncate but does not define the truncation; these are the
// published definitions (top-k, nucleus sampling) read with a threshold so that the result does not
// depend on the order of equal logits.
//
// One cluster per row.  Top-k with a small k and the nucleus alone take two passes and a handful of candidates (see
// the candidate path below).  Otherwise, and where the candidates do not fit, the value is found by a radix descent over an order-preserving integer
// image of the logits, 8 bits per pass: every pass streams the row once (cp.async ring, as the other
// kernels), histograms the digit of the elements that match the digits already fixed (counts, and
// for the nucleus the masses 2^(l*c - M) in 2^-40 fixed point, so that every sum is an integer and
// the result is the same whatever the order of the additions), the blocks add their histograms up
// through distributed shared memory, and every block takes the same decision from the same sums.
// bf16 rows need two passes per descent, fp32 rows four.
#pragma once

#include "svip_device.cuh"
#include "svip_draft.cuh"

namespace svip {

constexpr int kHistCopies = 8;           // interleaved copies of the histogram: lane l adds into copy l % 8, so
                                         // lanes that meet in one bin mostly hit different words and banks
constexpr float kMassScale = 1099511627776.0f;   // 2^40
constexpr int kPoolCap = 2048;           // candidates of the whole cluster
constexpr int kCandPerBlock = 1024;      // candidates one of several blocks may collect
constexpr int kCounted = 256;            // up to this many group maxima or candidates are put in order by counting
constexpr int kMaxGroups = 2048;         // groups of threads whose maxima give the bound of a top-k

struct ThresholdArgs {
    const void* logits;
    long row_stride;
    int V;
    float c;        // log2(e) / T
    int top_k;      // 1 .. V-1, or 0 when off
    float top_p;    // (0, 1), or >= 1 when off
    float* thr;     // [rows] out: tau as a logit value (-inf: nothing is dropped)
    float2* stats;  // [rows] out or NULL: (largest logit, mass of the kept set relative to it)
    // draft form (kDraft): the whole truncated draft step where the candidates allow it
    const float* uniforms;   // [rows]
    const uint8_t* active;   // NULL, or rows with 0 are skipped
    float thresh;            // h of the stop test
    int32_t* token;          // [rows] out
    float* entropy;          // [rows] out
    uint8_t* stop;           // [rows] out
    unsigned* status;        // device status word
    int sample_den;          // candidate path: the first bound comes from 1/sample_den of every warp segment (1: all)
};

// Monotone image of a float: a < b  <=>  key(a) < key(b).  NaN counts as -inf.
__device__ __forceinline__ uint32_t order_key(float x) {
    x = fmaxf(x, neg_inf());        // NaN -> -inf (the maximum of a NaN and a number is the number)
    x = x + 0.f;                    // -0 -> +0: the two zeros are one value
    const uint32_t u = __float_as_uint(x);
    return u ^ (static_cast<uint32_t>(static_cast<int32_t>(u) >> 31) | 0x80000000u);
}

__device__ __forceinline__ float key_value(uint32_t key) {
    return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
}

// Streams segment `seg` of the row with the calling warp and hands every vector to f(x, vi), with
// the elements outside the row set to -inf.
template <int DT, class F>
__device__ __forceinline__ void stream_segment(const RowGeom& g, int seg, int lane, uint32_t slot0, F&& f) {
    constexpr int EPV = ElemTraits<DT>::kEPV;
    constexpr uint32_t kSlotStride = kThreads * 16;
    int v_lo, v_hi;
    seg_range(g, seg, v_lo, v_hi);
    const int vi0 = v_lo + lane;
    const int n = v_hi > vi0 ? (v_hi - vi0 + 31) >> 5 : 0;
    const uint4* src = g.base + vi0;
#pragma unroll
    for (int s = 0; s < kStages; ++s) {
        if (s < n) cp_async16(slot0 + s * kSlotStride, src + 32 * s);
        cp_async_commit();
    }
    for (int it = 0; it < n; ++it) {
        cp_async_wait<kStages - 1>();
        const uint32_t slot = slot0 + (it & (kStages - 1)) * kSlotStride;
        const uint4 raw = lds128(slot);
        if (it + kStages < n) cp_async16(slot, src + 32 * (it + kStages));
        cp_async_commit();
        float x[EPV];
        unpack_masked<DT>(raw, vi0 + 32 * it, g, x);
        f(x, vi0 + 32 * it);
    }
    cp_async_wait<0>();
}

struct alignas(8) Candidate {
    uint32_t key;         // order_key of the logit
    uint32_t idx;         // its position in the row
};

// What block 0 of the cluster decided about the row, sent to the other blocks.
enum : uint32_t {
    kVerdictDone = 0,     // block 0 writes every output
    kVerdictDescend = 1,  // the candidates do not fit: radix descent over the row
    kVerdictRetry = 2,    // they do not fit a first time: once more with a better bound
    kVerdictStream = 3    // a row without finite mass: the draft step streams it once more at the threshold
};

struct SelectShared {
    union {
        uint32_t priv[3][256][kHistCopies];   // count, mass low word, mass high word; per digit, per copy
        Candidate landing[kPoolCap];          // candidate path, block 0: the peers' candidates, one region per block (the
                                              // candidates of a block alone)
    };
    union {
        alignas(16) float group_max[kMaxGroups];   // candidate path: group maxima of the whole cluster
        Candidate cand[kCandPerBlock];        // then this block's elements at or above the bound
    };
    union {
        struct {
            unsigned long long blk_mass[256]; // this block's histogram, read by the peers
            uint32_t blk_cnt[256];
            uint32_t tot_cnt[256];            // the cluster's histogram
            unsigned long long tot_mass[256];
        };
        uint32_t vec_list[kCandPerBlock];     // candidate path: vectors with an element at or above the bound
    };
    float blk_max;                        // this block's largest logit
    unsigned long long blk_above;         // this block's mass of the elements >= tau_k
    float warp_max[kWarps];
    unsigned long long warp_above[kWarps];
    // candidate path
    SegExchange ex;                       // nucleus alone: maximum and a lower bound of Z of every warp segment of the cluster
    uint4 header[kMaxCluster];            // block 0: x = number of candidates each block collected, (z, y) = mass of its part
    uint4 verdict;                        // x = kVerdict..., y = key of the threshold
    unsigned long long bar_group;         // all group maxima have landed
    unsigned long long bar_pool;          // block 0: headers and candidates of all blocks have landed
    unsigned long long bar_verdict;       // the verdict has landed
    uint32_t n_vec;                       // how many vectors are listed (may exceed the capacity)
    uint32_t n_cand;                      // how many candidates this block found (may exceed the capacity)
    uint32_t bound_key;                   // lower bound of the threshold
    uint32_t better[kMaxCluster];         // ... and what each block makes of the candidates it has, if they do not fit
    uint32_t top_key;
    // decision of a pass (written by warp 0)
    int bin;
    uint32_t cnt_above;
    unsigned long long mass_above;
    unsigned long long mass_total;
    unsigned long long mass_bin;
};

// Block 0's working set while it finishes a row from its candidates; lives in the streaming ring, free by then.
struct PoolScratch {
    Candidate pool[kPoolCap];
    union {
        struct {                                         // up to kCounted candidates
            uint32_t key_desc[kCounted];                 // keys from the largest down ...
            unsigned long long mass_desc[kCounted];      // ... and their masses
            Candidate by_idx[kCounted];                  // candidates in index order ...
            unsigned long long mass_idx[kCounted];       // ... and their masses
        };
        unsigned long long mass[kPoolCap];               // more: the masses of the pool
    };
};
static_assert(sizeof(PoolScratch) <= kRingBytes, "the pool is finished inside the ring");

__device__ __forceinline__ unsigned long long shfl_up_u64(unsigned long long v, int o) {
    uint32_t lo = __shfl_up_sync(0xffffffffu, static_cast<uint32_t>(v), o);
    uint32_t hi = __shfl_up_sync(0xffffffffu, static_cast<uint32_t>(v >> 32), o);
    return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// Adds a mass to a bin of the interleaved histogram copies of the calling lane, as two 32-bit words with carry (64-bit atomics
// on shared memory are loops, which crawl where many candidates share a bin).
__device__ __forceinline__ void add_mass(uint32_t* h_lo, uint32_t* h_hi, uint32_t bin, unsigned long long w) {
    const uint32_t lo = static_cast<uint32_t>(w);
    const uint32_t old = atomicAdd(h_lo + bin * kHistCopies, lo);
    const uint32_t hi = static_cast<uint32_t>(w >> 32) + (old + lo < old ? 1u : 0u);
    if (hi) atomicAdd(h_hi + bin * kHistCopies, hi);
}

// One pass: histogram of digit (key >> shift) & 255 over the elements whose higher digits equal
// those of `prefix` (all elements when first).  kMass adds the masses; kMax also finds the largest
// logit; `key_k` (with kAbove) sums the mass of the elements with key >= key_k.  On return every
// block of the cluster holds the cluster-wide histogram in sh.tot_*.
template <int DT, bool kMass, bool kMax, bool kAbove>
__device__ __forceinline__ void histogram_pass(cg::cluster_group& cluster, const RowGeom& g, int S, int rank,
                                               int tid, uint32_t slot0, uint32_t prefix, int shift, bool first,
                                               float c, float M, uint32_t key_k, SelectShared& sh,
                                               float& row_max, unsigned long long& above) {
    constexpr int EPV = ElemTraits<DT>::kEPV;
    const int lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < kHistCopies * 3 * 256; i += kThreads) (&sh.priv[0][0][0])[i] = 0;
    __syncthreads();
    uint32_t* h_cnt = &sh.priv[0][0][lane % kHistCopies];
    uint32_t* h_lo = &sh.priv[1][0][lane % kHistCopies];
    uint32_t* h_hi = &sh.priv[2][0][lane % kHistCopies];
    float mx = neg_inf();
    unsigned long long ab = 0;
    const uint32_t want = first ? 0u : (prefix >> (shift + 8));
    stream_segment<DT>(g, rank * kWarps + warp, lane, slot0, [&](const float (&x)[EPV], int) {
#pragma unroll
        for (int j = 0; j < EPV; ++j) {
            const uint32_t key = order_key(x[j]);
            if (kMax) mx = fmaxf(mx, x[j]);
            unsigned long long wq = 0;
            if (kMass) {
                const float w = ex2_approx(fmaxf(__fmaf_rn(x[j], c, -M), kArgFloor));
                wq = __float2ull_rz(w * kMassScale);
                if (kAbove && key >= key_k) ab += wq;
            }
            // the nucleus descent is decided by the masses alone, the top-k descent by the counts
            if ((first || (key >> (shift + 8)) == want) && (!kMass || wq)) {
                const uint32_t bin = (key >> shift) & 255u;
                if (!kMass) atomicAdd(h_cnt + bin * kHistCopies, 1u);
                else add_mass(h_lo, h_hi, bin, wq);
            }
        }
    });
    if (kMax) {
        mx = warp_max(mx);
        if (lane == 0) sh.warp_max[warp] = mx;
    }
    if (kAbove) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            uint32_t lo = __shfl_xor_sync(0xffffffffu, static_cast<uint32_t>(ab), o);
            uint32_t hi = __shfl_xor_sync(0xffffffffu, static_cast<uint32_t>(ab >> 32), o);
            ab += (static_cast<unsigned long long>(hi) << 32) | lo;
        }
        if (lane == 0) sh.warp_above[warp] = ab;
    }
    __syncthreads();
    if (tid < 256) {
        uint32_t cn = 0;
        unsigned long long ms = 0;
#pragma unroll
        for (int k = 0; k < kHistCopies; ++k) {
            cn += sh.priv[0][tid][k];
            if (kMass) ms += (static_cast<unsigned long long>(sh.priv[2][tid][k]) << 32) + sh.priv[1][tid][k];
        }
        sh.blk_cnt[tid] = cn;
        sh.blk_mass[tid] = ms;
    }
    if (tid == 0) {
        float m = neg_inf();
        unsigned long long s = 0;
        for (int w = 0; w < kWarps; ++w) {
            if (kMax) m = fmaxf(m, sh.warp_max[w]);
            if (kAbove) s += sh.warp_above[w];
        }
        sh.blk_max = m;
        sh.blk_above = s;
    }
    cluster.sync();
    if (tid < 256) {
        uint32_t cn = 0;
        unsigned long long ms = 0;
        for (int r = 0; r < S; ++r) {
            const SelectShared* peer = cluster.map_shared_rank(&sh, r);
            cn += peer->blk_cnt[tid];
            if (kMass) ms += peer->blk_mass[tid];
        }
        sh.tot_cnt[tid] = cn;
        sh.tot_mass[tid] = ms;
    }
    if (kMax || kAbove) {
        float m = neg_inf();
        unsigned long long s = 0;
        for (int r = 0; r < S; ++r) {
            const SelectShared* peer = cluster.map_shared_rank(&sh, r);
            if (kMax) m = fmaxf(m, peer->blk_max);
            if (kAbove) s += peer->blk_above;
        }
        if (kMax) row_max = m;
        if (kAbove) above = s;
    }
    cluster.sync();   // every peer has read this block's histogram; tot_* is visible block-wide
}

// Warp 0: walks the cluster histogram from the highest digit down and finds the digit at which
// the running count reaches `k_rem` (kByMass false) or the running mass reaches `p_rem`.
template <bool kByMass>
__device__ __forceinline__ void decide(SelectShared& sh, int lane, uint32_t k_rem, unsigned long long p_rem) {
    // lane l owns the digits 255 - 8l ... 248 - 8l, highest first
    uint32_t cn[8];
    unsigned long long ms[8];
    uint32_t csum = 0;
    unsigned long long msum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int bin = 255 - 8 * lane - j;
        cn[j] = sh.tot_cnt[bin];
        ms[j] = sh.tot_mass[bin];
        csum += cn[j];
        msum += ms[j];
    }
    uint32_t cinc = csum;
    unsigned long long minc = msum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t cu = __shfl_up_sync(0xffffffffu, cinc, o);
        const unsigned long long mu = shfl_up_u64(minc, o);
        if (lane >= o) { cinc += cu; minc += mu; }
    }
    uint32_t cbefore = cinc - csum;              // digits above this lane's
    unsigned long long mbefore = minc - msum;
    int hit = -1;
    uint32_t c_at = 0;
    unsigned long long m_at = 0, m_bin = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bool reached = kByMass ? (mbefore + ms[j] >= p_rem) : (cbefore + cn[j] >= k_rem);
        if (hit < 0 && reached && (kByMass ? ms[j] > 0 : cn[j] > 0)) {
            hit = 255 - 8 * lane - j;
            c_at = cbefore;
            m_at = mbefore;
            m_bin = ms[j];
        }
        cbefore += cn[j];
        mbefore += ms[j];
    }
    const unsigned who = __ballot_sync(0xffffffffu, hit >= 0);
    const unsigned long long total = __shfl_sync(0xffffffffu, static_cast<uint32_t>(minc), 31) |
        (static_cast<unsigned long long>(__shfl_sync(0xffffffffu, static_cast<uint32_t>(minc >> 32), 31)) << 32);
    if (who == 0) {
        // nothing reaches the target (an empty histogram): stay at the lowest digit
        if (lane == 0) { sh.bin = 0; sh.cnt_above = 0; sh.mass_above = 0; sh.mass_total = total; sh.mass_bin = 0; }
    } else if (lane == __ffs(who) - 1) {
        sh.bin = hit; sh.cnt_above = c_at; sh.mass_above = m_at; sh.mass_total = total; sh.mass_bin = m_bin;
    }
}

// Inclusive prefix over the lanes of per-lane masses.
__device__ __forceinline__ unsigned long long warp_scan_mass(unsigned long long v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long up = shfl_up_u64(v, o);
        if (lane >= o) v += up;
    }
    return v;
}

// Sum of the integers of the threads before this one, and of all of them.  Two barriers.
__device__ __forceinline__ unsigned long long block_prefix_u64(SelectShared& sh, unsigned long long v, int tid,
                                                               unsigned long long& total) {
    const int lane = tid & 31, warp = tid >> 5;
    const unsigned long long incl = warp_scan_mass(v, lane);
    __syncthreads();   // warp_above may still be read from an earlier use
    if (lane == 31) sh.warp_above[warp] = incl;
    __syncthreads();
    unsigned long long before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        if (w == warp) before = total;
        total += sh.warp_above[w];
    }
    return before + incl - v;
}

// What the statistics output holds for a row: (m, Z~) in the convention of the draft step's row_stats.
__device__ __forceinline__ float2 kept_stats(float row_max, unsigned long long kept_mass, bool finite) {
    return make_float2(row_max, finite ? static_cast<float>(static_cast<double>(kept_mass) / 1099511627776.0) : 0.f);
}

__device__ __forceinline__ unsigned long long mass_of_key(uint32_t key, float c, float M) {
    const float w = ex2_approx(fmaxf(__fmaf_rn(key_value(key), c, -M), kArgFloor));
    return __float2ull_rz(w * kMassScale);
}

// ------------------------------------------------------------------ candidate path
//
// For a top-k with a small k (with or without the nucleus inside it) and for the nucleus alone: a lower bound t0 of
// the threshold from one pass over the row, the elements >= t0 from a second one, everything else from these
// candidates.
//   top-k    the maxima of disjoint groups of threads are distinct elements of the row, so the k-th largest of them
//            is a lower bound of tau_k.  With G groups about -G ln(1 - k/G) elements lie above it (G >= 2k: 1.4 k),
//            so the groups are made as large as that allows, which keeps the exchange small.
//   nucleus  elements of mass below (1 - top_p) Z / V weigh less than (1 - top_p) Z together, so none of them is
//            in the nucleus, and neither with anything below Z in its place: the first pass takes maxima only, and the
//            masses of the threads' maxima stand for Z.  The second pass also sums the masses of all elements, in fixed
//            point and relative to the row's maximum, as the radix descent does: a cut must not depend on how many
//            blocks share the row, nor on which way the row goes (with Z summed in fp32 it did, for running masses within
//            1e-6 of top_p).
// A segment that fits the ring (small launches) is still in shared memory for the second pass.  The blocks push
// their candidates into block 0 of the cluster, which puts up to kCounted of them in order by counting (several threads
// per candidate) and finds tau_k, the nucleus cut and the sample by scans of one warp over the masses; in more these are
// found by radix descents in shared memory.  It tells the other blocks whether they are needed again.  All
// masses are 2^-40 fixed point, so nothing depends on the order in which they are added or candidates arrive.
// Bound by the chain of exchanges for launches of up to about 100 rows, by the two passes over the row above that.
// Rows of 152064 bf16, top-k 50 + top-p 0.9, against cluster barriers with remote reads and a counting finish in every
// block: draft step of 16 rows 18.3 -> 10.1 us, 64 rows 21.5 -> 14.3, 256 rows 41.0 -> 25.1; threshold of 2304 rows
// 243 -> 174 us.  Top-p alone against the radix descent: 1040 rows 521 -> 91 us.

// Block-wide wait for an mbarrier of the exchange: one warp polls, the others sleep at the block barrier.
__device__ __forceinline__ void bar_wait(unsigned long long& bar, uint32_t parity, unsigned* status, int tid) {
    if (tid < 32 && !mbar_wait_bounded(smem_addr(&bar), parity) && tid == 0) atomicOr(status, SVIP_STATUS_WAIT_TIMEOUT);
    __syncthreads();
}

// log2 of how many threads (a power of two, at most 32) can share each of n items in one pass of the block.
__device__ __forceinline__ int share_shift(int n) {
    int k = 0;
    while (k < 5 && (2 * n) << k <= kThreads) ++k;
    return k;
}

// Radix descent over n items of shared memory in bits [low, high) of their keys, at most 8 bits a level; `prefix` holds the
// bits from `high` up, which all items share.  The key of the k_rem-th item from the top (by counts), or the one at which the
// running mass from the top reaches p_rem.  By mass the histogram copies are used, which in the candidate path are the
// landing place of the peers' candidates.  Block-collective; ends with a barrier.
template <bool kByMass, class KeyOf, class MassOf>
__device__ __forceinline__ uint32_t pool_select(SelectShared& sh, int n, uint32_t prefix, int high, int low, uint32_t k_rem,
                                                unsigned long long p_rem, int tid, const KeyOf& key_of, const MassOf& mass_of) {
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll 1
    while (high > low) {
        const int shift = max(high - 8, low);
        const uint32_t digits = (1u << (high - shift)) - 1u;
        if (kByMass) {
            for (int i = tid; i < 256 * kHistCopies; i += kThreads) { (&sh.priv[1][0][0])[i] = 0; (&sh.priv[2][0][0])[i] = 0; }
        }
        if (tid < 256) { sh.tot_cnt[tid] = 0; sh.tot_mass[tid] = 0; }
        __syncthreads();
        for (int i = tid; i < n; i += kThreads) {
            const uint32_t key = key_of(i);
            if (high < 32 && (key >> high) != (prefix >> high)) continue;
            const uint32_t bin = (key >> shift) & digits;
            if (!kByMass) {
                atomicAdd(&sh.tot_cnt[bin], 1u);
            } else {
                const unsigned long long w = mass_of(i);
                if (w) add_mass(&sh.priv[1][0][lane % kHistCopies], &sh.priv[2][0][lane % kHistCopies], bin, w);
            }
        }
        __syncthreads();
        if (kByMass) {
            if (tid < 256) {
                unsigned long long m = 0;
#pragma unroll
                for (int k = 0; k < kHistCopies; ++k)
                    m += (static_cast<unsigned long long>(sh.priv[2][tid][k]) << 32) + sh.priv[1][tid][k];
                sh.tot_mass[tid] = m;
            }
            __syncthreads();
        }
        if (warp == 0) decide<kByMass>(sh, lane, k_rem, p_rem);
        __syncthreads();
        prefix |= static_cast<uint32_t>(sh.bin) << shift;
        k_rem -= sh.cnt_above;
        p_rem -= sh.mass_above;
        high = shift;
    }
    return prefix;
}

// Leaves in sh.bound_key the k-th largest of the n values (as an order key), or somewhat less.  Few values by counting: it is
// the smallest value with fewer than k values above it.  That is quadratic (2048 values: 190 us), so of more the upper 16 bits
// are found by a descent and the others left zero.  Ends with a barrier.  (n <= kMaxGroups, a multiple of 16; 1 <= k <= n.)
__device__ __forceinline__ void kth_largest(SelectShared& sh, int n, uint32_t k, int tid) {
    if (n > kCounted) {
        const auto key_of = [&](int i) { return order_key(sh.group_max[i]); };
        const uint32_t key = pool_select<false>(sh, n, 0u, 32, 16, k, 0ull, tid, key_of, key_of);
        if (tid == 0) sh.bound_key = key;
        __syncthreads();
        return;
    }
    const int shift = share_shift(n), per = 1 << shift, rows = kThreads >> shift;
    const int sub = tid & (per - 1);
    const float4* quads = reinterpret_cast<const float4*>(sh.group_max);
    uint32_t best = 0xffffffffu;
    for (int base = 0; base < n; base += rows) {
        const int i = base + (tid >> shift);
        const float v = i < n ? sh.group_max[i] : neg_inf();
        uint32_t gt = 0;
#pragma unroll 2
        for (int q = sub; q < n / 4; q += per) {
            const float4 w = quads[q];
            gt += (w.x > v) + (w.y > v) + (w.z > v) + (w.w > v);
        }
        for (int o = per >> 1; o > 0; o >>= 1) gt += __shfl_xor_sync(0xffffffffu, gt, o);
        if (i < n && gt < k) best = min(best, order_key(v));
    }
    best = __reduce_min_sync(0xffffffffu, best);
    if ((tid & 31) == 0) atomicMin(&sh.bound_key, best);
    __syncthreads();
}

__device__ __forceinline__ unsigned long long shfl_u64(unsigned long long v, int src) {
    const uint32_t lo = __shfl_sync(0xffffffffu, static_cast<uint32_t>(v), src);
    const uint32_t hi = __shfl_sync(0xffffffffu, static_cast<uint32_t>(v >> 32), src);
    return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// Mass that the nucleus has to reach, of a total mass: at least 1, at most the total.
__device__ __forceinline__ unsigned long long nucleus_target(float top_p, unsigned long long total) {
    unsigned long long want = static_cast<unsigned long long>(ceil(static_cast<double>(top_p) * static_cast<double>(total)));
    if (want < 1) want = 1;
    return want > total ? total : want;
}

// Block 0, warp 0: threshold, statistics and (kDraft) the sample from n <= kCounted candidates, in order both ways
// in `ps`.  Lane l owns the positions [l * per, (l + 1) * per) of both orders.  row_mass: mass of the whole row
// (nucleus alone).  `finite` is false for a row whose maximum is not a number the masses can be taken against.
template <bool kDraft, bool kTopK>
__device__ __forceinline__ void finish_sorted(const PoolScratch& ps, int n, const ThresholdArgs& a, bool use_p,
                                              unsigned long long row_mass, float row_max, float M, bool finite, int row,
                                              int lane) {
    const int per = (n + 31) / 32;
    const int lo = min(lane * per, n), hi = min(lo + per, n);
    unsigned long long sum = 0;
    for (int i = lo; i < hi; ++i) sum += ps.mass_desc[i];
    const unsigned long long before = warp_scan_mass(sum, lane) - sum;
    uint32_t key_t = kTopK ? ps.key_desc[a.top_k - 1] : 0u;
    if (use_p && finite) {
        unsigned long long zk = row_mass;
        if (kTopK) {      // mass of the candidates >= tau_k
            zk = 0;
            for (int i = lo; i < hi; ++i)
                if (ps.key_desc[i] >= key_t) zk += ps.mass_desc[i];
            zk = shfl_u64(warp_scan_mass(zk, lane), 31);
        }
        if (zk > 0) {
            const unsigned long long want = nucleus_target(a.top_p, zk);
            unsigned long long cum = before;
            int at = kIntMax;
            for (int i = lo; i < hi; ++i) {
                cum += ps.mass_desc[i];
                if (cum >= want && at == kIntMax) at = i;
            }
            at = warp_min_int(at);
            if (at == kIntMax) at = n - 1;         // rounding at the very end of the candidates: all of them
            key_t = max(key_t, ps.key_desc[at]);
        }
    }
    if (lane == 0) a.thr[row] = key_t ? key_value(key_t) : neg_inf();
    if (!a.stats && !kDraft) return;
    // kept candidates in index order
    unsigned long long zi = 0;
    long long term = 0;
    for (int i = lo; i < hi; ++i) {
        if (ps.by_idx[i].key < key_t) continue;
        zi += ps.mass_idx[i];
        if (kDraft) {
            const float arg = fmaxf(__fmaf_rn(key_value(ps.by_idx[i].key), a.c, -M), kArgFloor);
            term += __float2ll_rz(ex2_approx(arg) * arg * kMassScale);
        }
    }
    const unsigned long long incl = warp_scan_mass(zi, lane);
    const unsigned long long zt = shfl_u64(incl, 31);
    if (lane == 0 && a.stats) a.stats[row] = kept_stats(row_max, zt, finite);
    if (!kDraft) return;
    const long long aq = static_cast<long long>(shfl_u64(warp_scan_mass(static_cast<unsigned long long>(term), lane), 31));
    const float u = a.uniforms[row];
    const unsigned long long target = static_cast<unsigned long long>(static_cast<double>(u) * static_cast<double>(zt));
    unsigned long long cum = incl - zi;
    int token = -1;
    for (int i = lo; i < hi; ++i) {
        if (ps.by_idx[i].key < key_t) continue;
        const unsigned long long next = cum + ps.mass_idx[i];
        if (cum <= target && target < next) token = static_cast<int>(ps.by_idx[i].idx);
        cum = next;
    }
    if (token >= 0) a.token[row] = token;      // exactly one lane: target < zt
    if (lane == 0) {
        const float Z = static_cast<float>(static_cast<double>(zt) / 1099511627776.0);
        const float A = static_cast<float>(static_cast<double>(aq) / 1099511627776.0);
        const float H = fmaxf(kLn2 * (log2f(Z) - A / Z), 0.f);
        a.entropy[row] = H;
        a.stop[row] = __fsqrt_rn(H) > a.thresh ? 1 : 0;
    }
}

// Block 0 with all candidates of the cluster in ps.pool: finds the threshold and writes what it can.  Returns the
// verdict for the row (kVerdictDone, or kVerdictStream when the draft step has to be streamed at key_out), which
// `tell` passes on to the other blocks as soon as it is certain.
template <int DT, bool kDraft, bool kTopK, class Tell>
__device__ __forceinline__ uint32_t finish_pool(SelectShared& sh, PoolScratch& ps, int n, const ThresholdArgs& a, bool use_p,
                                                unsigned long long row_mass, int row, int tid,
                                                uint32_t& key_out, Tell&& tell) {
    const int lane = tid & 31, warp = tid >> 5;
    if (n <= kCounted) {
        // position of every candidate in both orders, by counting; `per` threads share a candidate
        const int shift = share_shift(n), per = 1 << shift;
        const int sub = tid & (per - 1), i = tid >> shift;
        const Candidate me = i < n ? ps.pool[i] : Candidate{0u, 0u};
        uint32_t above = 0, left = 0, top = 0;
#pragma unroll 4
        for (int j = sub; j < n; j += per) {
            const Candidate o = ps.pool[j];
            above += (o.key > me.key || (o.key == me.key && o.idx < me.idx)) ? 1u : 0u;
            left += o.idx < me.idx ? 1u : 0u;
            top = max(top, o.key);
        }
        for (int o = per / 2; o > 0; o >>= 1) {
            above += __shfl_xor_sync(0xffffffffu, above, o);
            left += __shfl_xor_sync(0xffffffffu, left, o);
        }
        top = __reduce_max_sync(0xffffffffu, top);     // every candidate is seen by some lane of the warp, whatever `per`
        const float row_max = key_value(top);          // the largest candidate is the largest logit of the row
        const bool finite = fabsf(row_max) <= kMaxLogit;
        const float M = finite ? __fmul_rn(row_max, a.c) : 0.f;
        const uint32_t verdict = kDraft && !finite ? kVerdictStream : kVerdictDone;
        if (i < n && sub == 0) {
            const unsigned long long w = mass_of_key(me.key, a.c, M);
            ps.key_desc[above] = me.key;
            ps.mass_desc[above] = w;
            ps.by_idx[left] = me;
            ps.mass_idx[left] = w;
        }
        __syncthreads();
        key_out = kTopK ? ps.key_desc[a.top_k - 1] : 0u;   // what a row without finite mass is cut at
        tell(verdict, key_out);
        if (verdict == kVerdictStream) {
            if (tid == 0) a.thr[row] = key_out ? key_value(key_out) : neg_inf();
        } else if (warp == 0) {
            finish_sorted<kDraft, kTopK>(ps, n, a, use_p, row_mass, row_max, M, finite, row, lane);
        }
        return verdict;
    }
    // a larger set: radix descents, for the threshold in the keys and for the sample in the indices
    if (tid == 0) sh.top_key = 0;
    __syncthreads();
    uint32_t top = 0;
    for (int i = tid; i < n; i += kThreads) top = max(top, ps.pool[i].key);
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) atomicMax(&sh.top_key, top);
    __syncthreads();
    top = sh.top_key;
    const float row_max = key_value(top);          // the largest candidate is the largest logit of the row
    const bool finite = fabsf(row_max) <= kMaxLogit;
    const float M = finite ? __fmul_rn(row_max, a.c) : 0.f;
    const uint32_t verdict = kDraft && !finite ? kVerdictStream : kVerdictDone;
    if (verdict == kVerdictDone) tell(verdict, 0u);
    if (finite)
        for (int i = tid; i < n; i += kThreads) ps.mass[i] = mass_of_key(ps.pool[i].key, a.c, M);     // read by the same thread only
    // the keys lie between the bound and the largest, so they share the bits in which these two agree
    const int high = 32 - __clz(top ^ sh.bound_key);
    const uint32_t shared_bits = high < 32 ? top >> high << high : 0u;
    const int low = DT == kBF16 ? min(16, high) : 0;       // the low 16 bits of a bf16 logit carry nothing: zeros, or
                                                           // ones in the key of a negative one
    const auto whole = [&](uint32_t key) { return DT == kBF16 && !(key & 0x80000000u) ? key | 0xffffu : key; };
    const auto key_of = [&](int i) { return ps.pool[i].key; };
    const auto mass_of = [&](int i) { return ps.mass[i]; };
    const auto total = [&](unsigned long long v) {
        unsigned long long t = 0;
        block_prefix_u64(sh, v, tid, t);
        return t;
    };
    const auto mass_from = [&](uint32_t key) {
        unsigned long long z = 0;
        for (int i = tid; i < n; i += kThreads)
            if (ps.pool[i].key >= key) z += ps.mass[i];
        return total(z);
    };
    uint32_t key_t = kTopK ? whole(pool_select<false>(sh, n, shared_bits, high, low, static_cast<uint32_t>(a.top_k), 0ull, tid,
                                                      key_of, mass_of)) : 0u;
    key_out = key_t;
    if (verdict == kVerdictStream) tell(verdict, key_t);
    if (use_p && finite) {
        const unsigned long long zk = kTopK ? mass_from(key_t) : row_mass;
        if (zk > 0) {
            const unsigned long long all = kTopK ? zk : mass_from(0u);
            unsigned long long want = nucleus_target(a.top_p, zk);
            if (want > all) want = all;                // rounding at the very end of the candidates: all of them
            key_t = max(key_t, whole(pool_select<true>(sh, n, shared_bits, high, low, 0u, want, tid, key_of, mass_of)));
        }
    }
    if (tid == 0) a.thr[row] = key_t ? key_value(key_t) : neg_inf();
    if (verdict == kVerdictStream || (!kDraft && !a.stats)) return verdict;
    const unsigned long long zt = finite ? mass_from(key_t) : 0ull;
    if (tid == 0 && a.stats) a.stats[row] = kept_stats(row_max, zt, finite);
    if (!kDraft) return verdict;
    long long term = 0;
    for (int i = tid; i < n; i += kThreads) {
        if (ps.pool[i].key < key_t) { ps.mass[i] = 0; continue; }
        const float arg = fmaxf(__fmaf_rn(key_value(ps.pool[i].key), a.c, -M), kArgFloor);
        term += __float2ll_rz(ex2_approx(arg) * arg * kMassScale);
    }
    const long long aq = static_cast<long long>(total(static_cast<unsigned long long>(term)));
    // the sample: the first index at which the running mass of the kept candidates exceeds u * zt
    const unsigned long long target = static_cast<unsigned long long>(static_cast<double>(a.uniforms[row]) * static_cast<double>(zt));
    const int idx_bits = 32 - __clz(a.V);
    const auto from_end = [&](int i) { return ~ps.pool[i].idx; };      // the lowest index has the largest key
    const uint32_t found = ~pool_select<true>(sh, n, ~0u << idx_bits, idx_bits, 0, 0u, target + 1, tid, from_end, mass_of);
    if (tid == 0) {
        a.token[row] = static_cast<int32_t>(found);
        const float Z = static_cast<float>(static_cast<double>(zt) / 1099511627776.0);
        const float A = static_cast<float>(static_cast<double>(aq) / 1099511627776.0);
        const float H = fmaxf(kLn2 * (log2f(Z) - A / Z), 0.f);
        a.entropy[row] = H;
        a.stop[row] = __fsqrt_rn(H) > a.thresh ? 1 : 0;
    }
    return verdict;
}

// Sum of the 2^-40 fixed-point masses of elements of a row (those of mass_of_key).  Bound by instructions: nearly all elements
// weigh less than 2^-17, and for these the addition of 2^23 rounded towards zero leaves the integer in the mantissa, two
// elements per instruction on the wide pipe, where a conversion takes the pipe of the exponentials.  A vector with a
// likelier element, or with a NaN (which shows as a sum that no EPV masses have), converts.  Round of 64 sequences with top-p
// 0.95 (5 draft steps, thresholds of 384 rows of 304 KB): 144 us; one element at a time and in one kernel with the top-k
// 173; with the total summed in fp32 in the first pass, in whatever order the launch shape gave, 141.
template <int DT>
struct MassSum {
    float c, M;
    float big;                    // no element below this logit weighs 2^-17 or more
    unsigned long long sum = 0;
    __device__ __forceinline__ MassSum(float c_, float row_max) {
        c = c_;
        M = __fmul_rn(row_max, c_);
        big = (M - 17.01f) / c - 5e-7f * fabsf(row_max);
    }
    __device__ __forceinline__ void one(float x) {
        sum += __float2ull_rz(ex2_approx(fmaxf(__fmaf_rn(x, c, -M), kArgFloor)) * kMassScale);
    }
    __device__ __forceinline__ void vector(const uint4& raw, float vmax) {
        constexpr int EPV = ElemTraits<DT>::kEPV;
        float x[EPV];
        ElemTraits<DT>::unpack(raw, x);
        const f32x2 c2 = pack2(c, c), nm2 = pack2(-M, -M), scale2 = pack2(kMassScale, kMassScale), base2 = pack2(8388608.f, 8388608.f);
        uint32_t s = 0;
#pragma unroll
        for (int j = 0; j < EPV; j += 2) {
            float a0, a1;
            unpack2(fma2(pack2(x[j], x[j + 1]), c2, nm2), a0, a1);
            unpack2(fma2_rz(pack2(ex2_approx(a0), ex2_approx(a1)), scale2, base2), a0, a1);
            s += __float_as_uint(a0) + __float_as_uint(a1);
        }
        s -= EPV * 0x4B000000u;               // EPV masses below 2^23
        if (vmax >= big || s >= EPV * (1u << 23)) {
#pragma unroll
            for (int j = 0; j < EPV; ++j) one(x[j]);
        } else {
            sum += s;
        }
    }
};

// Where a block collects its candidates, and lists the vectors that hold them.
struct CollectInto {
    Candidate* cand;
    uint32_t cap;
    uint32_t* vec_list;
    uint32_t vec_cap;
};

// Collects the elements >= t0v of the block's segments and (kMass) leaves the mass of all elements of every
// warp's segment in sh.warp_above.  `resident`: every segment of the row fits the ring and lies there since pass 1 (a
// property of the row, so the same in every warp: a block barrier depends on it).
template <int DT, bool kMass>
__device__ __forceinline__ void collect(const RowGeom& g, const LaneSpan& s, bool resident, uint32_t slot0, float t0v,
                                        const CollectInto& to, SelectShared& sh, float c, float row_max) {
    constexpr int EPV = ElemTraits<DT>::kEPV;
    MassSum<DT> mass(c, row_max);
    const bool lowest = !(t0v > neg_inf());      // no bound: every element, -inf and NaN (which counts as -inf) among them
    auto place = [&](float x, uint32_t pos, int i) {
        if (pos < to.cap) to.cand[pos] = Candidate{order_key(x), static_cast<uint32_t>(i)};
    };
    // A set that does not fit is of no use, and a flat row has tens of thousands of elements above the bound, each of which
    // would wait for its turn at the counter: collecting ends as soon as that is known, and a vector asks for all its places
    // at once (draft step with Gaussian logits, top-p 0.9: 1 row of 304 KB 39.3 -> 31.7 us, 384 rows of 64 KB 90 -> 70).
    auto over = [&]() { return *static_cast<volatile uint32_t*>(&sh.n_cand) > to.cap; };
    auto has = [&](const uint4& raw) {        // asked once per vector: it also counts its mass
        RawMax<DT> m;
        m.reset();
        m.fold(raw);
        const float top = m.value();
        if (kMass) mass.vector(raw, top);
        return top >= t0v || lowest;
    };
    auto visit = [&](const uint4& raw, int vi) {
        float x[EPV];
        ElemTraits<DT>::unpack(raw, x);
        uint32_t hits = 0;
#pragma unroll
        for (int j = 0; j < EPV; ++j) hits += x[j] >= t0v || lowest ? 1u : 0u;
        if (hits == 0 || over()) return;
        uint32_t pos = atomicAdd(&sh.n_cand, hits);
#pragma unroll
        for (int j = 0; j < EPV; ++j)
            if (x[j] >= t0v || lowest) place(x[j], pos++, vi * EPV + j - g.pre);
    };
    auto edge = [&](int vi) {
        float x[EPV];
        ElemTraits<DT>::unpack(ld_vec(g.base + vi), x);
#pragma unroll
        for (int j = 0; j < EPV; ++j) {
            const int i = vi * EPV + j - g.pre;
            if (i < 0 || i >= g.V) continue;
            if (kMass) mass.one(x[j]);
            if (x[j] >= t0v || lowest) place(x[j], atomicAdd(&sh.n_cand, 1u), i);
        }
    };
    if (resident) {
        const auto look = [&](const uint4& raw, int vi) { if (has(raw)) visit(raw, vi); };
        if constexpr (kMass) revisit_interior(s, slot0, look, over);
        else revisit_interior(s, slot0, look);
    } else {
        // the streaming loop only lists the vectors, which are few, and all threads look at them afterwards: with the
        // elements looked at inside the unrolled loop, 2304 rows of 304 KB took 272 us instead of 174
        auto full = [&]() { return *static_cast<volatile uint32_t*>(&sh.n_vec) > to.vec_cap; };
        stream_interior(s, slot0, [&](const uint4& raw, int vi) {
            if (has(raw) && !full()) {
                const uint32_t pos = atomicAdd(&sh.n_vec, 1u);
                if (pos < to.vec_cap) to.vec_list[pos] = static_cast<uint32_t>(vi);
            }
        }, full);
        __syncthreads();
        const uint32_t nv = sh.n_vec;
        // of a set that does not fit, a top-k still wants as many as there is room for (see candidate_path)
        if (!kMass || nv <= to.vec_cap)
            for (uint32_t i = threadIdx.x; i < min(nv, to.vec_cap); i += kThreads) visit(ld_vec(g.base + to.vec_list[i]), to.vec_list[i]);
        if (nv > to.vec_cap) {
            __syncthreads();
            if (threadIdx.x == 0) atomicAdd(&sh.n_cand, to.cap + 1);
        }
    }
    if (s.head) edge(0);
    if (s.tail) edge(g.nvec - 1);
    if (kMass) {
        const unsigned long long m = warp_scan_mass(mass.sum, threadIdx.x & 31);
        if ((threadIdx.x & 31) == 31) sh.warp_above[threadIdx.x >> 5] = m;
    }
}

// Groups of threads per warp whose maxima bound a top-k: a power of two, at least 2 k in the cluster if there are
// that many threads (as a shift).
__device__ __forceinline__ int group_shift(int S, int k) {
    int g = 0;
    while (g < 5 && (kWarps * S) << g < 2 * k) ++g;
    return g;
}
// The largest number of groups, likewise.
__device__ __forceinline__ int finest_groups(int S) {
    int g = 0;
    while (g < 5 && (kWarps * S) << (g + 1) <= kMaxGroups) ++g;
    return g;
}

// The k-th largest of the maxima of groups of threads, 2^shift groups a warp (`best` is the thread's maximum); the same in
// every block.  The bar_group phase has been opened, in all blocks.
__device__ __forceinline__ uint32_t group_bound(SelectShared& sh, float best, int shift, int S, int seg, int k, uint32_t phase,
                                                unsigned* status, int tid) {
    const int lane = tid & 31, width = 32 >> shift;
    for (int o = width >> 1; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    const int slot = (seg << shift) + (lane >> (5 - shift));
    const bool leads = (lane & (width - 1)) == 0;
    if (S == 1) {
        if (leads) sh.group_max[slot] = best;
        __syncthreads();
    } else {
        if (leads) {
            for (int r = 0; r < S; ++r)
                push4(map_to_rank(smem_addr(&sh.group_max[slot]), r), map_to_rank(smem_addr(&sh.bar_group), r),
                      __float_as_uint(best));
        }
        bar_wait(sh.bar_group, phase, status, tid);
    }
    kth_largest(sh, (kWarps * S) << shift, static_cast<uint32_t>(k), tid);
    return sh.bound_key;
}

// A better bound for a top-k whose candidates do not fit.  The maxima of large groups bound next to nothing where the likely
// tokens are gathered in few warps (a vocabulary in order of frequency), those of half of the row where they are in the
// other half.  Either the maxima of the smallest groups (`finest` >= 0), or the k-th largest of what the blocks have stored,
// which are elements of the row like any others.  Thresholds of rows of 50021 fp32 logits in order of frequency, top-k 50,
// without and with the second attempt: 16 rows 29.6 and 18.0 us, 64 rows 39.9 and 22.1, 300 rows 123 and 42.  A function of
// its own, because its code in line cost every top-k 3 %.
__device__ __noinline__ uint32_t better_bound(SelectShared& sh, const Candidate* cand, uint32_t stored, float best, int finest, int S,
                                              int rank, int k, unsigned* status) {
    const int tid = threadIdx.x;
    uint32_t bound = 0;
    if (finest < 0 && stored >= static_cast<uint32_t>(k)) {
        const auto key_of = [&](int i) { return cand[i].key; };
        bound = pool_select<false>(sh, static_cast<int>(stored), 0u, 32, 16, static_cast<uint32_t>(k), 0ull, tid, key_of, key_of);
    }
    if (S > 1) {
        if (tid == 0) {
            mbar_arrive_expect_tx(smem_addr(&sh.bar_group), static_cast<uint32_t>(finest < 0 ? S * 4 : (kWarps * S * 4) << finest));
            if (rank != 0) mbar_arrive_expect_tx(smem_addr(&sh.bar_verdict), 16);
            if (finest >= 0) sh.bound_key = 0xffffffffu;
        }
        cluster_arrive();
        cluster_wait();
        if (finest >= 0) return group_bound(sh, best, finest, S, rank * kWarps + (tid >> 5), k, 1, status, tid);
        if (tid < S) push4(map_to_rank(smem_addr(&sh.better[rank]), tid), map_to_rank(smem_addr(&sh.bar_group), tid), bound);
        bar_wait(sh.bar_group, 1, status, tid);
        for (int r = 0; r < S; ++r) bound = max(bound, sh.better[r]);
    }
    return bound;
}

// Barriers and counters of the path; needs no global memory, so it runs before the predecessor has finished.
__device__ __forceinline__ void candidate_open(SelectShared& sh, int S, int rank, int top_k, bool use_k, int tid) {
    if (tid == 0) {
        if (S > 1) {
            mbar_init(smem_addr(&sh.ex.bar), 1);
            mbar_init(smem_addr(&sh.bar_group), 1);
            mbar_init(smem_addr(&sh.bar_verdict), 1);
            mbar_init(smem_addr(&sh.bar_pool), S);
            if (use_k) mbar_arrive_expect_tx(smem_addr(&sh.bar_group), static_cast<uint32_t>((kWarps * S * 4) << group_shift(S, top_k)));
            else mbar_arrive_expect_tx(smem_addr(&sh.ex.bar), static_cast<uint32_t>(S * kWarps * sizeof(SegEntry)));
            if (rank != 0) mbar_arrive_expect_tx(smem_addr(&sh.bar_verdict), 16);   // block 0 gives the verdict
        }
        sh.n_cand = 0;
        sh.n_vec = 0;
        sh.bound_key = 0xffffffffu;
    }
    if (S > 1) cluster_arrive_relaxed();     // the peers push only after their cluster_wait()
}

// The whole path for one row, opened by candidate_open(); the same verdict in every block of the cluster.  For the
// nucleus alone row_max receives the largest logit of the row.
template <int DT, bool kDraft, bool kTopK>
__device__ __forceinline__ uint32_t candidate_path(const RowGeom& g, const LaneSpan& span, int S, int rank, int tid,
                                                   uint32_t slot0, const ThresholdArgs& a, bool use_p, int row,
                                                   SelectShared& sh, PoolScratch* scratch, uint32_t& key_out, float& row_max) {
    constexpr int EPV = ElemTraits<DT>::kEPV;
    const int lane = tid & 31, warp = tid >> 5;
    const int seg = rank * kWarps + warp;
    // A block alone collects where the peers' candidates would land.  Otherwise every block collects at home; its first
    // kPoolCap / S candidates are pushed to block 0, which has that much room for each, and fetches the others of a block in
    // whose part of the row the likely tokens are gathered.
    const CollectInto to = S == 1 ? CollectInto{sh.landing, kPoolCap, reinterpret_cast<uint32_t*>(sh.cand), 2 * kCandPerBlock}
                                  : CollectInto{sh.cand, kCandPerBlock, sh.vec_list, kCandPerBlock};
    const uint32_t region = kPoolCap / S;
    const int gs = group_shift(S, a.top_k);
    const int den = kTopK ? a.sample_den : 1;
    // ---- pass 1: the largest logit of every thread, and from these the bound
    const LaneSpan part = den > 1 ? lane_span<DT>(g, seg, lane, den) : span;
    RawMax<DT> m;
    m.reset();
    stream_interior(part, slot0, [&](const uint4& raw, int) { m.fold(raw); });
    float best = m.value();
    if (part.head || part.tail) {
        float x[EPV];
        if (part.head) { unpack_masked<DT>(ld_vec(g.base), 0, g, x); best = fmaxf(best, vec_max<EPV>(x)); }
        if (part.tail) { unpack_masked<DT>(ld_vec(g.base + g.nvec - 1), g.nvec - 1, g, x); best = fmaxf(best, vec_max<EPV>(x)); }
    }
    uint32_t first_bound = 0;
    if constexpr (kTopK) {
        if (S > 1) cluster_wait();
        first_bound = group_bound(sh, best, gs, S, seg, a.top_k, 0, a.status, tid);
    } else {
        Partial t;
        t.m = warp_max(best); t.idx = kIntMax; t.A = 0.f;
        t.Z = warp_sum(best > neg_inf() ? ex2_approx(fmaxf((best - t.m) * a.c, kArgFloor)) : 0.f);
        if (S == 1) {
            if (lane == 0) { SegEntry& e = sh.ex.all[warp]; e.m = t.m; e.idx = t.idx; e.Z = t.Z; e.A = 0.f; }
            __syncthreads();
        } else {
            cluster_wait();
            exchange_send(sh.ex, S, rank, warp, lane, t);
            bar_wait(sh.ex.bar, 0, a.status, tid);
        }
        // every warp forms the same sums from the same entries
        const Partial r = merge_entries<1>(LocalSegments{sh.ex.all}, S * kWarps, a.c, lane);
        row_max = r.m;       // what the radix descent needs first
        if (!(fabsf(r.m) <= kMaxLogit) || !(r.Z > 0.f)) return kVerdictDescend;   // in every block alike
        // no element weighs more than 1, so the nucleus has at least top_p Z of them: a flat row does not fit
        if (a.top_p * r.Z > static_cast<float>(kPoolCap)) return kVerdictDescend;
        // in log2 units, a little low for the roundings of the weights, and of the bound as a logit
        const float cut = log2f((1.f - a.top_p) * r.Z / static_cast<float>(g.V)) - 0.05f;
        if (tid == 0) sh.bound_key = order_key((__fmul_rn(r.m, a.c) + cut) / a.c - 5e-7f * fabsf(r.m));
        __syncthreads();
    }
    // Whether smaller groups are worth a second attempt: if all likely tokens are gathered in as few warps as can hold them, the
    // candidates fit a block all the same.
    const int finest = finest_groups(S);
    const bool finer = S > 1 && den == 1 && finest > gs && (static_cast<long>(a.top_k) * g.vps * EPV >> finest) <= 3 * kCandPerBlock / 2;
    uint32_t parity = 0;
    for (;;) {
        // ---- pass 2: the candidates
        const float t0v = key_value(sh.bound_key);
        pdl_launch_dependents();
        const bool resident = den == 1 && g.vps <= 32 * kStages;
        collect<DT, !kTopK>(g, span, resident, slot0, t0v, to, sh, a.c, row_max);
        __syncthreads();
        uint32_t verdict;
        const uint32_t mine = sh.n_cand;
        unsigned long long my_mass = 0;
        if (!kTopK) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) my_mass += sh.warp_above[w];
        }
        if (S > 1 && rank != 0) {
            const uint32_t sent = mine <= to.cap ? min(mine, region) : 0u;
            const uint32_t bar0 = map_to_rank(smem_addr(&sh.bar_pool), 0);
            for (uint32_t i = tid; i < sent; i += kThreads)
                push8(map_to_rank(smem_addr(&sh.landing[rank * region + i]), 0), bar0, sh.cand[i].key, sh.cand[i].idx);
            if (tid == 0) {
                push16(map_to_rank(smem_addr(&sh.header[rank]), 0), bar0, mine, static_cast<uint32_t>(my_mass),
                       static_cast<uint32_t>(my_mass >> 32), 0u);
                mbar_arrive_expect_tx_remote(bar0, 16u + 8u * sent);
            }
            bar_wait(sh.bar_verdict, parity, a.status, tid);
            verdict = sh.verdict.x;
            key_out = sh.verdict.y;
        } else {
            if (S > 1) {
                if (tid == 0) mbar_arrive_expect_tx(smem_addr(&sh.bar_pool), 0);
                bar_wait(sh.bar_pool, parity, a.status, tid);
            }
            // tells the other blocks, once
            auto tell = [&](uint32_t v, uint32_t key) {
                if (S > 1 && tid >= 1 && tid < S)
                    push16(map_to_rank(smem_addr(&sh.verdict), tid), map_to_rank(smem_addr(&sh.bar_verdict), tid), v, key, 0u, 0u);
            };
            // lane r holds the count of block r; every warp knows all offsets
            const uint4 head = lane > 0 && lane < S ? sh.header[lane] : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t count = lane == 0 ? mine : head.x;
            unsigned long long row_mass = 0;
            if (!kTopK) row_mass = shfl_u64(warp_scan_mass((static_cast<unsigned long long>(head.z) << 32) | head.y, lane), 31) + my_mass;
            uint32_t end = count;
#pragma unroll
            for (int o = 1; o < kMaxCluster; o <<= 1) {
                const uint32_t up = __shfl_up_sync(0xffffffffu, end, o);
                if (lane >= o) end += up;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, end, kMaxCluster - 1);
            const bool fits = !__any_sync(0xffffffffu, count > to.cap) && total <= kPoolCap;
            if (!fits || total < static_cast<uint32_t>(kTopK ? a.top_k : 1)) {
                verdict = kTopK && !fits && parity == 0 && (S == 1 || den > 1 || finer) ? kVerdictRetry : kVerdictDescend;
                tell(verdict, 0u);
            } else {
                // two warps copy the candidates of each block
                const int r = warp & (kMaxCluster - 1);
                const uint32_t nr = __shfl_sync(0xffffffffu, count, r), first = __shfl_sync(0xffffffffu, end, r) - nr;
                const uint32_t here = r == 0 ? nr : min(nr, region);
                const Candidate* from = r == 0 ? to.cand : sh.landing + r * region;
                for (uint32_t t = (warp / kMaxCluster) * 32 + lane; t < here; t += 64) scratch->pool[first + t] = from[t];
                // the block stays, and keeps its candidates, until it hears the verdict
                for (uint32_t t = here + (warp / kMaxCluster) * 32 + lane; t < nr; t += 64) {
                    const uint2 o = ld_remote8(map_to_rank(smem_addr(&sh.cand[t]), r));
                    scratch->pool[first + t] = Candidate{o.x, o.y};
                }
                __syncthreads();
                verdict = finish_pool<DT, kDraft, kTopK>(sh, *scratch, static_cast<int>(total), a, use_p, row_mass, row, tid,
                                                  key_out, tell);
            }
        }
        if (!kTopK || verdict != kVerdictRetry) return verdict;
        // ---- once more with a better bound
        __syncthreads();
        parity = 1;
        const uint32_t bound = better_bound(sh, to.cand, min(mine, to.cap), best, finer ? finest : -1, S, rank, a.top_k, a.status);
        if (bound <= first_bound) return kVerdictDescend;      // in every block alike
        __syncthreads();
        if (tid == 0) {
            sh.n_cand = 0;
            sh.n_vec = 0;
            sh.bound_key = bound;
        }
        __syncthreads();
    }
}

// The streaming draft step of the row at the threshold just found, for the rows the candidates
// could not finish (nucleus alone, large k, heavy ties, no finite mass).  Cluster-collective.
template <int DT>
__device__ __forceinline__ void draft_at_threshold(const ThresholdArgs& a, int S, int rank, int row, int tid,
                                                   const RowGeom& g, uint32_t slot0, float thr) {
    DraftArgs d;
    d.logits = a.logits; d.row_stride = a.row_stride; d.V = a.V; d.c = a.c; d.thresh = a.thresh; d.greedy = 0;
    d.uniforms = a.uniforms; d.token = a.token; d.entropy = a.entropy; d.stop = a.stop;
    d.row_stats = reinterpret_cast<float*>(a.stats); d.status = a.status; d.active = nullptr;
    d.ext_target = nullptr; d.token_offset = 0; d.pos = nullptr; d.pos_stride = 0; d.slot_stride = 0; d.thr = nullptr; d.adv.arrived = nullptr;
    __shared__ SegExchange ex;
    exchange_open(ex, S, tid);
    draft_row<DT, false, false, true>(d, S, rank, row, tid, g, lane_span<DT>(g, rank * kWarps + (tid >> 5), tid & 31), slot0,
                                      0, thr, ex);
}

// kDraft: the truncated draft step in the same launch: from the candidates where that path applies,
// else by streaming the row once more at the threshold just found.  kTopK: with a top_k in [1, V), else the nucleus alone (or
// nothing at all); two kernels rather than one, whose registers did not suffice for both.
template <int DT, bool kDraft, bool kTopK>
__global__ void __launch_bounds__(kThreads, 2) row_threshold_kernel(ThresholdArgs a) {
    constexpr int kLevels = DT == kBF16 ? 2 : 4;   // the low 16 bits of a bf16 logit carry nothing
    extern __shared__ __align__(kRingAlign) uint4 ring[];
    __shared__ SelectShared sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int S = cluster.dim_blocks().x;
    const int rank = cluster.block_rank();
    const int row = blockIdx.x / S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const char* rp = static_cast<const char*>(a.logits) +
                     static_cast<size_t>(row) * a.row_stride * ElemTraits<DT>::kBytes;
    const RowGeom g = make_geom<DT>(rp, a.V, S * kWarps);
    const uint32_t slot0 = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + tid * 16;
    const bool use_p = a.top_p < 1.0f;
    // a small k against the number of threads of the cluster, or the nucleus alone: two passes over the row
    const bool by_candidates = kTopK ? a.top_k <= (S * kThreads) / 4 : use_p;
    const LaneSpan span = lane_span<DT>(g, rank * kWarps + warp, lane);
    if (by_candidates) candidate_open(sh, S, rank, a.top_k, kTopK, tid);
    if (!a.active && lane == 0) prefetch_segment(g, rank * kWarps + warp, kRingBytes / kWarps);
    pdl_wait();
    if (kDraft && a.active && !a.active[row]) {         // the whole cluster leaves together
        if (by_candidates && S > 1) cluster_wait();
        return;
    }

    float row_max = neg_inf();
    unsigned long long above = 0;
    bool have_max = false;
    uint32_t key_k = 0;       // key of tau_k (0: below every key, nothing dropped)

    if (by_candidates) {
        uint32_t key_t = 0;
        const uint32_t verdict = candidate_path<DT, kDraft, kTopK>(g, span, S, rank, tid, slot0, a, use_p, row, sh,
                                                                   reinterpret_cast<PoolScratch*>(ring), key_t, row_max);
        have_max = !kTopK;
        if (verdict == kVerdictDone) return;
        if (kDraft && verdict == kVerdictStream) {
            __syncthreads();       // block 0 is done with the ring in every warp
            draft_at_threshold<DT>(a, S, rank, row, tid, g, slot0, key_t ? key_value(key_t) : neg_inf());
            return;
        }
    }

    if (kTopK) {
        uint32_t prefix = 0, k_rem = static_cast<uint32_t>(a.top_k);
        for (int level = 0; level < kLevels; ++level) {
            const int shift = 24 - 8 * level;
            if (level == 0)
                histogram_pass<DT, false, true, false>(cluster, g, S, rank, tid, slot0, prefix, shift, true, a.c, 0.f,
                                                       0u, sh, row_max, above);
            else
                histogram_pass<DT, false, false, false>(cluster, g, S, rank, tid, slot0, prefix, shift, false, a.c,
                                                        0.f, 0u, sh, row_max, above);
            if (warp == 0) decide<false>(sh, lane, k_rem, 0ull);
            __syncthreads();
            prefix |= static_cast<uint32_t>(sh.bin) << shift;
            k_rem -= sh.cnt_above;
            __syncthreads();   // the decision is read before the next pass overwrites it
        }
        have_max = true;
        // digits below the ones examined: a bf16 logit has them all zero, which the key stores as
        // ones for negative values
        key_k = prefix;
        if (DT == kBF16 && !(prefix & 0x80000000u)) key_k |= 0xffffu;
    }

    uint32_t key_t = key_k;
    if (use_p || (a.stats && !kDraft)) {
        if (!have_max) {
            // the masses are taken relative to the largest logit: find it first
            float mx = neg_inf();
            stream_segment<DT>(g, rank * kWarps + warp, lane, slot0,
                               [&](const float (&x)[ElemTraits<DT>::kEPV], int) {
#pragma unroll
                for (int j = 0; j < ElemTraits<DT>::kEPV; ++j) mx = fmaxf(mx, x[j]);
            });
            mx = warp_max(mx);
            if (lane == 0) sh.warp_max[warp] = mx;
            __syncthreads();
            if (tid == 0) {
                float m = neg_inf();
                for (int w = 0; w < kWarps; ++w) m = fmaxf(m, sh.warp_max[w]);
                sh.blk_max = m;
            }
            cluster.sync();
            float m = neg_inf();
            for (int r = 0; r < S; ++r) m = fmaxf(m, cluster.map_shared_rank(&sh, r)->blk_max);
            row_max = m;
            cluster.sync();
        }
    }
    if (use_p) {
        const bool finite = fabsf(row_max) <= kMaxLogit;
        const float M = finite ? __fmul_rn(row_max, a.c) : 0.f;
        uint32_t prefix = 0;
        unsigned long long p_rem = 0;
        for (int level = 0; level < kLevels; ++level) {
            const int shift = 24 - 8 * level;
            if (level == 0)
                histogram_pass<DT, true, false, true>(cluster, g, S, rank, tid, slot0, prefix, shift, true, a.c, M,
                                                      key_k, sh, row_max, above);
            else
                histogram_pass<DT, true, false, false>(cluster, g, S, rank, tid, slot0, prefix, shift, false, a.c, M,
                                                       key_k, sh, row_max, above);
            if (level == 0) {
                // target mass: top_p of the mass of the top-k set (the whole row without top-k)
                const double want = ceil(static_cast<double>(a.top_p) * static_cast<double>(above));
                p_rem = static_cast<unsigned long long>(want);
                if (p_rem < 1) p_rem = 1;
                if (p_rem > above) p_rem = above;
            }
            if (warp == 0) decide<true>(sh, lane, 0u, p_rem);
            __syncthreads();
            prefix |= static_cast<uint32_t>(sh.bin) << shift;
            p_rem -= sh.mass_above;
            __syncthreads();
        }
        uint32_t key_p = prefix;
        if (DT == kBF16 && !(prefix & 0x80000000u)) key_p |= 0xffffu;
        if (above == 0 || !finite) key_p = 0;   // a row without mass: the nucleus drops nothing
        key_t = key_p > key_k ? key_p : key_k;
    }
    if (rank == 0 && tid == 0) a.thr[row] = key_t ? key_value(key_t) : neg_inf();
    if (kDraft) {
        draft_at_threshold<DT>(a, S, rank, row, tid, g, slot0, key_t ? key_value(key_t) : neg_inf());
        return;
    }
    if (a.stats && !kDraft) {
        // the mass of the kept set: one more pass (the descents above know it only in part)
        const bool finite = fabsf(row_max) <= kMaxLogit;
        const float M = finite ? __fmul_rn(row_max, a.c) : 0.f;
        unsigned long long kept = 0;
        stream_segment<DT>(g, rank * kWarps + warp, lane, slot0, [&](const float (&x)[ElemTraits<DT>::kEPV], int) {
#pragma unroll
            for (int j = 0; j < ElemTraits<DT>::kEPV; ++j) {
                if (order_key(x[j]) >= key_t) {
                    const float w = ex2_approx(fmaxf(__fmaf_rn(x[j], a.c, -M), kArgFloor));
                    kept += __float2ull_rz(w * kMassScale);
                }
            }
        });
        unsigned long long of_block = 0;
        block_prefix_u64(sh, kept, tid, of_block);
        if (tid == 0) sh.blk_above = of_block;
        cluster.sync();
        unsigned long long all = 0;
        for (int r = 0; r < S; ++r) all += cluster.map_shared_rank(&sh, r)->blk_above;
        if (rank == 0 && tid == 0) a.stats[row] = kept_stats(row_max, all, finite);
        cluster.sync();   // the peers have read this block's sum
    }
    // every pass ended with a cluster barrier after all remote reads: blocks may leave
}

}  // namespace svip
