// Truncation threshold of a logits row (top-k and nucleus / top-p).
//
// The kept set of a row is {i : l_i >= tau}: tau_k is the k-th largest logit, and inside that set
// tau is the largest logit value v for which the mass of {l_i >= v} reaches top_p of the mass of
// {l_i >= tau_k}; tokens tied with the last kept one are all kept.  The paper applies its length
// policy on top of samplers that truncate but does not define the truncation; these are the
// published definitions (top-k, nucleus sampling) read with a threshold so that the result does not
// depend on the order of equal logits.
//
// One cluster per row.  Top-k with a small k takes one pass over the row and the nucleus alone two, and a handful of candidates
// (see the candidate path below).  Otherwise, and where the candidates do not fit, the value is found by a radix descent over
// an order-preserving integer image of the logits, 8 bits per pass: every pass streams the row once (cp.async ring, as the other
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
constexpr int kCandPerBlock = 1024;      // top-k: candidates one of several blocks may collect (nucleus alone: kPoolCap)
constexpr int kSorted = 256;             // up to this many candidates are put in order, the keys by one warp
constexpr int kMaxGroups = 2048;         // groups of threads whose maxima give the bound of a top-k
constexpr int kOneWarp = 512;            // up to this many group maxima are searched by one warp
constexpr int kRetryTopK = 128;          // up to this k a second bound is tried where the candidates do not fit
constexpr int kStretches = 8;            // maxima that a thread keeps of the vectors it streams

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
    int groups;              // candidate path, top-k: log2 of the groups of threads per warp whose maxima bound the threshold
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
        struct {
            Candidate landing[kPoolCap];      // candidate path, block 0: the peers' candidates, one region per block (the
                                              // candidates of a block alone)
            union {
                struct {                      // top-k
                    uint16_t stretch_key[kStretches][kThreads];   // rows that do not fit the ring: see stream_maxima
                    union {
                        alignas(16) float group_max[kMaxGroups];  // group maxima of the whole cluster
                        Candidate cand[kCandPerBlock];            // then this block's elements at or above the bound
                    };
                };
                Candidate cand_alone[kPoolCap];   // nucleus alone: likewise
            };
        };
    };
    union {
        struct {
            unsigned long long blk_mass[256]; // this block's histogram, read by the peers
            uint32_t blk_cnt[256];
            uint32_t tot_cnt[256];            // the cluster's histogram
            unsigned long long tot_mass[256];
        };
        uint32_t vec_list[kPoolCap];          // nucleus alone: vectors with an element at or above the bound
        uint16_t stretch_list[kStretches * kThreads];   // top-k: stretches that may have one; room for every stretch of a block
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
    uint32_t n_vec;                       // how many of these there are (of vectors, may exceed the capacity)
    uint32_t n_cand;                      // how many candidates this block found (may exceed the capacity)
    uint32_t bound_key;                   // lower bound of the threshold
    uint32_t better[kMaxCluster];         // ... and a better one that each block finds, if they do not fit
    uint32_t top_key;
    int tied;                             // top-k: the bound is the largest group maximum, no better one exists
    // decision of a pass (written by warp 0)
    int bin;
    uint32_t cnt_above;
    unsigned long long mass_above;
};

// Block 0's working set while it finishes a row from its candidates; lives in the streaming ring, free by then.
struct PoolScratch {
    Candidate pool[kPoolCap];
    union {
        struct {                                         // up to kSorted candidates
            Candidate by_idx[kSorted];                   // candidates in index order ...
            unsigned long long mass_idx[kSorted];        // ... and their masses
            uint32_t key_t;                              // key of the threshold
            int unusable;                                // no finite mass in the row
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
        cn[j] = kByMass ? 0u : sh.tot_cnt[bin];
        ms[j] = kByMass ? sh.tot_mass[bin] : 0ull;
        csum += cn[j];
        msum += ms[j];
    }
    uint32_t cinc = csum;
    unsigned long long minc = msum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t cu = kByMass ? 0u : __shfl_up_sync(0xffffffffu, cinc, o);
        const unsigned long long mu = kByMass ? shfl_up_u64(minc, o) : 0ull;
        if (lane >= o) { cinc += cu; minc += mu; }
    }
    uint32_t cbefore = cinc - csum;              // digits above this lane's
    unsigned long long mbefore = minc - msum;
    int hit = -1;
    uint32_t c_at = 0;
    unsigned long long m_at = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bool reached = kByMass ? (mbefore + ms[j] >= p_rem) : (cbefore + cn[j] >= k_rem);
        if (hit < 0 && reached && (kByMass ? ms[j] > 0 : cn[j] > 0)) {
            hit = 255 - 8 * lane - j;
            c_at = cbefore;
            m_at = mbefore;
        }
        cbefore += cn[j];
        mbefore += ms[j];
    }
    const unsigned who = __ballot_sync(0xffffffffu, hit >= 0);
    if (who == 0) {
        // nothing reaches the target (an empty histogram): stay at the lowest digit
        if (lane == 0) { sh.bin = 0; sh.cnt_above = 0; sh.mass_above = 0; }
    } else if (lane == __ffs(who) - 1) {
        sh.bin = hit; sh.cnt_above = c_at; sh.mass_above = m_at;
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

__device__ __forceinline__ float weight_of_key(uint32_t key, float c, float M) {
    return ex2_approx(fmaxf(__fmaf_rn(key_value(key), c, -M), kArgFloor));
}
__device__ __forceinline__ unsigned long long mass_of_weight(float w) { return __float2ull_rz(w * kMassScale); }
__device__ __forceinline__ unsigned long long mass_of_key(uint32_t key, float c, float M) {
    return mass_of_weight(weight_of_key(key, c, M));
}

// ------------------------------------------------------------------ candidate path
//
// For a top-k with a small k (with or without the nucleus inside it) and for the nucleus alone: a lower bound t0 of
// the threshold from one pass over the row, the elements >= t0 from what the pass has left in the ring or from a second look,
// everything else from these candidates.
//   top-k    the maxima of disjoint groups of threads are distinct elements of the row, so the k-th largest of them
//            is a lower bound of tau_k.  With G groups about -G ln(1 - k/G) elements lie above it (G = 1.5 k: 1.65 k),
//            so the groups are made as large as that allows, which keeps the exchange and the search in it small.  The row
//            is read once: of rows that do not fit the ring the maxima of stretches of vectors are kept, and only the
//            stretches that reach the bound are fetched again.
//   nucleus  elements of mass below (1 - top_p) Z / V weigh less than (1 - top_p) Z together, so none of them is
//            in the nucleus, and neither with anything below Z in its place: the first pass takes maxima only, and the
//            masses of the threads' maxima stand for Z.  The second pass also sums the masses of all elements, in fixed
//            point and relative to the row's maximum, as the radix descent does: a cut must not depend on how many
//            blocks share the row, nor on which way the row goes (with Z summed in fp32 it did, for running masses within
//            1e-6 of top_p).
// A segment that fits the ring (small launches) is still in shared memory for the second look.  The blocks push
// their candidates into block 0 of the cluster, which puts up to kSorted of them in order and finds tau_k, the nucleus cut and
// the sample by scans of one warp over the masses; in more these are found by radix descents in shared memory.  It tells the other
// blocks whether they are needed again.  All masses are 2^-40 fixed point, so nothing depends on the order in which they are added or candidates arrive.
// Bound by the chain of exchanges for launches of up to about 100 rows, by the pass (nucleus: the two passes) over the rows above
// that.
// Rows of 152064 bf16, top-k 50 + top-p 0.9, against cluster barriers with remote reads and a counting finish in every
// block, and now: draft step of 16 rows 18.3 -> 8.1 us, 64 rows 21.5 -> 11.1, 256 rows 41.0 -> 18.9; threshold of 2304 rows
// 243 -> 124 us.  Top-p alone against the radix descent: 1040 rows 521 -> 97 us.  A top-k that reads its rows once, with one
// warp's search for the bound and one warp's sort, against two passes (of launches above 48 MB one and a half) and counting: draft
// step of 32 such rows 12.6 -> 8.4 us, threshold of 288 rows 24.4 -> 19.3, a round of 128 sequences of 256000
// fp32, top-k 100, 3 draft steps, 319 -> 265.

// Block-wide wait for an mbarrier of the exchange: one warp polls, the others sleep at the block barrier.
__device__ __forceinline__ void bar_wait(unsigned long long& bar, uint32_t parity, unsigned* status, int tid) {
    if (tid < 32 && !mbar_wait_bounded(smem_addr(&bar), parity) && tid == 0) atomicOr(status, SVIP_STATUS_WAIT_TIMEOUT);
    __syncthreads();
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
        if (!kByMass && tid < 256) sh.tot_cnt[tid] = 0;
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

// A bound (as an order key) that at least k of n <= 32 * kPer values reach, n >= k >= 1, and not many more than k.  By one warp,
// bit by bit below the bits that all of them share, the values in registers.  (Ranking all of them by comparing every pair in
// all warps took 3200 cycles for 192 values in the kernel, two blocks on an SM; this 1000 for 96.)
template <int kPer>
__device__ __forceinline__ uint32_t kth_bound(const float* values, int n, uint32_t k, int lane, uint32_t& top) {
    uint32_t key[kPer], low = 0xffffffffu;
    top = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = lane + 32 * j;
        key[j] = i < n ? order_key(values[i]) : 0u;
        top = max(top, key[j]);
        if (i < n) low = min(low, key[j]);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    low = __reduce_min_sync(0xffffffffu, low);
    if (top == low) return top;
    uint32_t step = 0x80000000u >> __clz(top ^ low);      // the highest bit in which they differ: clear in the lowest
    uint32_t bound = low & ~(2u * step - 1u);
#pragma unroll 1
    for (; step != 0; step >>= 1) {
        const uint32_t pivot = bound | step;
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) c += key[j] >= pivot ? 1u : 0u;
        c = __reduce_add_sync(0xffffffffu, c);
        if (c < k) continue;
        bound = pivot;
        if (c <= k + k / 8) break;
    }
    return bound;
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

// Sum over the lanes of a warp, modulo 2^64: 24, 24 and 16 bits apart, in 32 bits each.  All 64 bits: the weight of a row's
// largest logit is 2 to the rounding error of max * c, which is not near 1 where |max| / T is above some 10^8.
__device__ __forceinline__ unsigned long long warp_total_mass(unsigned long long v) {
    const uint32_t lo = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(v) & 0xffffffu);
    const uint32_t mid = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(v >> 24) & 0xffffffu);
    const uint32_t hi = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(v >> 48));
    return (static_cast<unsigned long long>(hi) << 48) + (static_cast<unsigned long long>(mid) << 24) + lo;
}

// A block barrier that the warps may reach in different places of the code.
__device__ __forceinline__ void block_meet() { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); }

// Sorts the 32 * kPer keys of a warp from the largest down (bitonic network); lane l ends up with places l * kPer ....
template <int kPer>
__device__ __forceinline__ void sort_down(uint32_t (&key)[kPer], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * kPer; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const bool down = ((lane * kPer + j) & size) == 0;
                if (stride >= kPer) {
                    const uint32_t other = __shfl_xor_sync(0xffffffffu, key[j], stride / kPer);
                    key[j] = ((lane & (stride / kPer)) == 0) == down ? max(key[j], other) : min(key[j], other);
                } else if ((j & stride) == 0) {
                    const uint32_t hi = max(key[j], key[j | stride]), lo = min(key[j], key[j | stride]);
                    key[j] = down ? hi : lo;
                    key[j | stride] = down ? lo : hi;
                }
            }
        }
    }
}

// Block 0, warp 0: the threshold of a row from its n <= 32 * kPer candidates in order of their keys, which stay in registers, the
// statistics, and (kDraft) the entropy; the sample waits at the block barrier for the threshold, which is left in ps.key_t.
// row_mass: mass of the whole row (nucleus alone).  A row whose maximum is not a number that masses can be taken against gets,
// in a draft step, a threshold only.
template <bool kDraft, bool kTopK, int kPer, class Tell>
__device__ __forceinline__ void finish_by_key(PoolScratch& ps, int n, const ThresholdArgs& a, bool use_p, unsigned long long row_mass,
                                              int row, int lane, Tell&& tell) {
    uint32_t key[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) key[j] = lane + 32 * j < n ? ps.pool[lane + 32 * j].key : 0u;
    sort_down<kPer>(key, lane);
    const float row_max = key_value(__shfl_sync(0xffffffffu, key[0], 0));      // the largest candidate is the largest logit of the row
    const bool finite = fabsf(row_max) <= kMaxLogit;
    const float M = finite ? __fmul_rn(row_max, a.c) : 0.f;
    if (!kDraft || finite) tell(kVerdictDone, 0u);
    uint32_t key_t = 0;
    if (kTopK) {
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if ((a.top_k - 1) % kPer == j) key_t = key[j];
        key_t = __shfl_sync(0xffffffffu, key_t, (a.top_k - 1) / kPer);
    }
    float w[kPer];       // the masses, before their conversion: half the registers
#pragma unroll
    for (int j = 0; j < kPer; ++j) w[j] = key[j] ? weight_of_key(key[j], a.c, M) : 0.f;
    if (use_p && finite) {
        unsigned long long sum = 0, kept = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const unsigned long long m = mass_of_weight(w[j]);
            sum += m;
            if (kTopK && key[j] >= key_t) kept += m;
        }
        const unsigned long long zk = kTopK ? warp_total_mass(kept) : row_mass;     // kTopK: of the candidates >= tau_k
        const unsigned long long incl = warp_scan_mass(sum, lane);
        if (zk > 0) {
            const unsigned long long want = nucleus_target(a.top_p, zk);
            unsigned long long cum = incl - sum;
            uint32_t at = 0, last = 0xffffffffu;       // key at which the sum is reached; lowest key
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                cum += mass_of_weight(w[j]);
                if (cum >= want) at = max(at, key[j]);
                if (key[j]) last = key[j];
            }
            const unsigned who = __ballot_sync(0xffffffffu, incl >= want);
            if (who) at = __shfl_sync(0xffffffffu, at, __ffs(who) - 1);
            else at = __reduce_min_sync(0xffffffffu, last);      // rounding at the very end of the candidates: all of them
            key_t = max(key_t, at);
        }
    }
    if (lane == 0) a.thr[row] = key_t ? key_value(key_t) : neg_inf();
    if (kDraft) {
        if (lane == 0) { ps.key_t = key_t; ps.unusable = !finite; }
        block_meet();
        if (!finite) return;
    } else if (!a.stats) {
        return;
    }
    unsigned long long z = 0;
    long long term = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        if (key[j] < key_t || key[j] == 0) continue;
        z += mass_of_weight(w[j]);
        if (kDraft) term += __float2ll_rz(w[j] * fmaxf(__fmaf_rn(key_value(key[j]), a.c, -M), kArgFloor) * kMassScale);
    }
    const unsigned long long zt = warp_total_mass(z);
    if (lane == 0 && a.stats) a.stats[row] = kept_stats(row_max, zt, finite);
    if (!kDraft) return;
    const long long aq = static_cast<long long>(warp_total_mass(static_cast<unsigned long long>(term)));
    if (lane == 0) {
        const float Z = static_cast<float>(static_cast<double>(zt) / 1099511627776.0);
        const float A = static_cast<float>(static_cast<double>(aq) / 1099511627776.0);
        const float H = fmaxf(kLn2 * (log2f(Z) - A / Z), 0.f);
        a.entropy[row] = H;
        a.stop[row] = __fsqrt_rn(H) > a.thresh ? 1 : 0;
    }
}

// Block 0, one warp: the sample from n <= kSorted candidates in index order, of which those with a key >= key_t are kept.  Lane l
// owns the places [l * per, (l + 1) * per).
__device__ __forceinline__ void sample_by_index(const PoolScratch& ps, int n, uint32_t key_t, float u, int32_t* token, int lane) {
    constexpr int kPer = kSorted / 32;
    const int per = (n + 31) / 32;
    const int lo = lane * per;
    const int mine = max(0, min(per, n - lo));
    unsigned long long sum = 0, cum[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (k < mine && ps.by_idx[lo + k].key >= key_t) sum += ps.mass_idx[lo + k];
        cum[k] = sum;
    }
    const unsigned long long incl = warp_scan_mass(sum, lane), before = incl - sum;
    const unsigned long long target = static_cast<unsigned long long>(static_cast<double>(u) * static_cast<double>(shfl_u64(incl, 31)));
    if (before <= target && target < incl) {      // exactly one lane: the target is less than the total
        int at = lo;
#pragma unroll
        for (int k = 0; k < kPer; ++k) at += k < mine && before + cum[k] <= target ? 1 : 0;
        *token = static_cast<int32_t>(ps.by_idx[at].idx);
    }
}

// Block 0 with all candidates of the cluster in ps.pool: finds the threshold and writes what it can.  Returns the
// verdict for the row (kVerdictDone, or kVerdictStream when the draft step has to be streamed at key_out), which
// `tell` passes on to the other blocks as soon as it is certain.  A chain of dependent steps.  Up to kSorted candidates: warp 0
// sorts the keys in registers and finds the threshold while the others put the candidates in index order by counting (80
// candidates: 3300 cycles for both orders by counting in all warps and 5200 for the rest in one warp that read its places anew in
// every step; 3200 in all now.  Draft step of 32 rows of 304 KB, top-k 50 + top-p 0.9, 10.0 -> 8.3 us, 8 rows of 64 KB fp32 8.6 -> 7.2).
template <int DT, bool kDraft, bool kTopK, class Tell>
__device__ __forceinline__ uint32_t finish_pool(SelectShared& sh, PoolScratch& ps, int n, const ThresholdArgs& a, bool use_p,
                                                unsigned long long row_mass, int row, int tid,
                                                uint32_t& key_out, Tell&& tell) {
    const int lane = tid & 31, warp = tid >> 5;
    if (n <= kSorted) {
        uint32_t verdict = kVerdictDone;
        if (warp == 0) {
            if (n <= 64) finish_by_key<kDraft, kTopK, 2>(ps, n, a, use_p, row_mass, row, lane, tell);
            else if (n <= 128) finish_by_key<kDraft, kTopK, 4>(ps, n, a, use_p, row_mass, row, lane, tell);
            else finish_by_key<kDraft, kTopK, kSorted / 32>(ps, n, a, use_p, row_mass, row, lane, tell);
        } else if (kDraft) {
            const float u = warp == 1 ? a.uniforms[row] : 0.f;
            const int i = (warp - 1) * 32 + lane;
            if (i - lane < n) {
                const Candidate me = i < n ? ps.pool[i] : Candidate{0u, 0u};
                const uint4* pairs = reinterpret_cast<const uint4*>(ps.pool);      // the one behind the last is a stand-in if n is odd
                uint32_t top = 0;
                int left = 0, left2 = 0;
#pragma unroll 4
                for (int j = 0; j < (n + 1) / 2; ++j) {
                    const uint4 o = pairs[j];
                    left += o.y < me.idx ? 1 : 0;
                    left2 += o.w < me.idx ? 1 : 0;
                    top = max(top, max(o.x, o.z));
                }
                if (i < n) {
                    const float row_max = key_value(top);
                    ps.by_idx[left + left2] = me;
                    ps.mass_idx[left + left2] = mass_of_key(me.key, a.c, fabsf(row_max) <= kMaxLogit ? __fmul_rn(row_max, a.c) : 0.f);
                }
            }
            block_meet();
            if (warp == 1 && !ps.unusable) sample_by_index(ps, n, ps.key_t, u, a.token + row, lane);
        }
        if (kDraft && ps.unusable) verdict = kVerdictStream;
        if (verdict == kVerdictStream) {
            key_out = ps.key_t;                        // what a row without finite mass is cut at
            if (warp == 0) tell(verdict, key_out);
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

// Where a block collects its candidates.
struct CollectInto {
    Candidate* cand;
    uint32_t cap;
};

// Element j of a vector.
template <int DT>
__device__ __forceinline__ float pick_element(const uint4& v, int j) {
    const int w = DT == kBF16 ? j >> 1 : j;
    const uint32_t word = w & 2 ? (w & 1 ? v.w : v.z) : (w & 1 ? v.y : v.x);
    return __uint_as_float(DT == kBF16 ? (j & 1 ? word & 0xffff0000u : word << 16) : word);
}

// The elements of a row at or above a bound, as they are found.
template <int DT>
struct Collector {
    static constexpr int EPV = ElemTraits<DT>::kEPV;
    const RowGeom& g;
    const CollectInto& to;
    SelectShared& sh;
    float bound;
    bool lowest;      // no bound: every element, -inf and NaN (which counts as -inf) among them
    __device__ __forceinline__ Collector(const RowGeom& g_, const CollectInto& to_, SelectShared& sh_, float bound_)
        : g(g_), to(to_), sh(sh_), bound(bound_), lowest(!(bound_ > neg_inf())) {}
    __device__ __forceinline__ bool above(float x) const { return x >= bound || lowest; }
    __device__ __forceinline__ void place(float x, uint32_t pos, int i) const {
        if (pos < to.cap) to.cand[pos] = Candidate{order_key(x), static_cast<uint32_t>(i)};
    }
    // A set that does not fit is of no use, and a flat row has tens of thousands of elements above the bound, each of which
    // would wait for its turn at the counter: collecting ends as soon as that is known, and a vector asks for all its places
    // at once (draft step with Gaussian logits, top-p 0.9: 1 row of 304 KB 39.3 -> 31.7 us, 384 rows of 64 KB 90 -> 70).
    __device__ __forceinline__ bool over() const { return *static_cast<volatile uint32_t*>(&sh.n_cand) > to.cap; }
    __device__ __forceinline__ void visit(const uint4& raw, int vi) const {
        float x[EPV];
        ElemTraits<DT>::unpack(raw, x);
        uint32_t hits = 0;
#pragma unroll
        for (int j = 0; j < EPV; ++j) hits |= above(x[j]) ? 1u << j : 0u;
        if (hits == 0 || over()) return;
        uint32_t pos = atomicAdd(&sh.n_cand, static_cast<uint32_t>(__popc(hits)));
        if ((hits & (hits - 1)) == 0) {        // mostly one
            const int j = __ffs(hits) - 1;
            place(pick_element<DT>(raw, j), pos, vi * EPV + j - g.pre);
        } else {
#pragma unroll
            for (int j = 0; j < EPV; ++j)
                if (hits >> j & 1u) place(x[j], pos++, vi * EPV + j - g.pre);
        }
    }
    // A vector that sticks out of the row; each(x) is told its elements.
    template <class F>
    __device__ __forceinline__ void edge(int vi, F&& each) const {
        float x[EPV];
        ElemTraits<DT>::unpack(ld_vec(g.base + vi), x);
#pragma unroll
        for (int j = 0; j < EPV; ++j) {
            const int i = vi * EPV + j - g.pre;
            if (i < 0 || i >= g.V) continue;
            each(x[j]);
            if (above(x[j])) place(x[j], atomicAdd(&sh.n_cand, 1u), i);
        }
    }
};

// How the vectors of a lane make up stretches, whose maxima are kept: `rounds` rounds of the ring (kStages vectors) each,
// `count` of them (at most kStretches).
struct Stretches {
    int rounds, count;
    __device__ __forceinline__ explicit Stretches(const RowGeom& g) {
        const int all = ((g.vps + 31) / 32 + kStages - 1) / kStages;
        rounds = (all + kStretches - 1) / kStretches;
        count = (all + rounds - 1) / rounds;
    }
};

// Pass 1 of a top-k: the largest logit of the thread's interior vectors.  Of rows that do not fit the ring, which would have
// to be read again for the candidates, the maximum of every stretch of vectors is kept (the upper half of its order key);
// only the few stretches that reach the bound are then fetched a second time, instead of the row.
template <int DT>
__device__ __forceinline__ float stream_maxima(const LaneSpan& s, uint32_t slot0, bool resident, const Stretches st,
                                               uint16_t (*keys)[kThreads]) {
    constexpr uint32_t kSlotStride = kThreads * 16;
    RawMax<DT> all, part;
    all.reset();
    part.reset();
    if (resident) {       // the vectors stay in the ring
        stream_interior(s, slot0, [&](const uint4& raw, int) { all.fold(raw); });
        return all.value();
    }
#pragma unroll
    for (int k = 0; k < kStages; ++k) {
        if (k < s.n) cp_async16(slot0 + k * kSlotStride, s.src + 32 * k);
        cp_async_commit();
    }
    uint16_t* at = &keys[0][threadIdx.x];
    int left = st.rounds;
    const auto flush = [&]() {
        *at = static_cast<uint16_t>(order_key(part.value()) >> 16);
        at += kThreads;
        all.fold(part);
        part.reset();
        left = st.rounds;
    };
    int it = 0;
    const int full = fewest_vectors(s);
    for (; it + kStages <= full; it += kStages) {
#pragma unroll
        for (int k = 0; k < kStages; ++k) {
            cp_async_wait<kStages - 1>();
            const uint4 raw = lds128(slot0 + k * kSlotStride);
            if (it + kStages + k < s.n) cp_async16(slot0 + k * kSlotStride, s.src + 32 * (it + kStages + k));
            cp_async_commit();
            part.fold(raw);
        }
        if (--left == 0) flush();
    }
    cp_async_wait<0>();
    if (it < s.n || left < st.rounds) {
        for (; it < s.n; ++it) part.fold(lds128(slot0 + (it & (kStages - 1)) * kSlotStride));
        flush();
    }
    for (; at < &keys[st.count][0]; at += kThreads) *at = 0;       // a lane with fewer
    return all.value();
}

// Pass 2 of a top-k: the elements at or above the bound (sh.bound_key).  `best`: what stream_maxima found.  `resident`: every
// segment of the row fits the ring and lies there (a property of the row, so the same in every warp: a block barrier depends
// on it).
template <int DT>
__device__ __forceinline__ void collect_top(const RowGeom& g, const LaneSpan& s, bool resident, const Stretches st, uint32_t slot0,
                                            float best, int rank, const CollectInto& to, SelectShared& sh) {
    const Collector<DT> c(g, to, sh, key_value(sh.bound_key));
    const int tid = threadIdx.x, lane = tid & 31;
    if (resident) {
        const unsigned hit = __ballot_sync(0xffffffffu, c.above(best));
        if (__popc(hit) > 8) {      // gathered: every lane looks through its own vectors
            revisit_interior(s, slot0, [&](const uint4& raw, int vi) { c.visit(raw, vi); }, [&]() { return c.over(); });
        } else {
            // the vectors of a lane that has something, side by side, four such lanes at a time
            for (unsigned left = hit; left;) {
                int src = -1;
#pragma unroll
                for (int q = 0; q < 32 / kStages; ++q) {
                    if (q == lane / kStages) src = __ffs(left) - 1;
                    left &= left - 1;
                }
                const int n = __shfl_sync(0xffffffffu, s.n, max(src, 0));
                const int k = lane % kStages;
                if (src >= 0 && k < n)
                    c.visit(lds128(slot0 + (src - lane) * 16 + k * (kThreads * 16)), s.vi0 - lane + src + 32 * k);
            }
        }
    } else {
        // Only threads whose largest element reaches the bound list stretches, since half a key does not tell: of logits that are
        // large against their spread, most stretches of a row agree with the bound in it (20 +- 0.01, 64 rows of 256000 fp32, top-k
        // 50: 17.1 us; with every thread's stretches listed 35, with a list of 1024 that is taken to mean too many candidates 215).
        const uint32_t cut = c.lowest ? 0u : sh.bound_key >> 16;
        const int vectors = st.rounds * kStages;
        if (c.above(best)) {
            for (int e = 0; e * vectors < s.n; ++e)
                if (sh.stretch_key[e][tid] >= cut) sh.stretch_list[atomicAdd(&sh.n_vec, 1u)] = static_cast<uint16_t>(e * kThreads + tid);
        }
        __syncthreads();
        // kStages threads per stretch, which take its vectors in turn; of bf16 rows two vectors of a thread are under way at a time
        // (of fp32 rows the registers for it have to be spilled: draft step of 256 rows of 1 MB 55.1 us, one at a time 52.0; bf16,
        // 288 rows of 304 KB: 20.5, one at a time 21.0).  Of a set that does not fit, a top-k still wants as many as there is room for
        // (see better_bound).
        const uint32_t items = sh.n_vec * kStages;
        const int inside = g.nvec - ((g.pre + g.V) % Collector<DT>::EPV != 0 ? 1 : 0);     // where a vector that sticks out begins
        for (int r = 0; r < st.rounds; ++r) {
            const auto vector_of = [&](uint32_t i) {      // which vector of the row, or -1
                if (i >= items) return -1;
                const uint32_t code = sh.stretch_list[i / kStages];
                const int t = static_cast<int>(code % kThreads);
                int lo, hi;
                seg_range(g, rank * kWarps + (t >> 5), lo, hi);
                const int first = lo == 0 && g.pre > 0 ? 1 : lo;        // as lane_span() has it
                const int vi = first + (t & 31) + 32 * (static_cast<int>(code / kThreads) * vectors + r * kStages + static_cast<int>(i % kStages));
                return vi < min(hi, inside) ? vi : -1;
            };
            constexpr int kAtOnce = DT == kBF16 ? 2 : 1;
            for (uint32_t i = tid; i < items && !c.over(); i += kAtOnce * kThreads) {
                int vi[kAtOnce];
                uint4 raw[kAtOnce];
#pragma unroll
                for (int q = 0; q < kAtOnce; ++q) {
                    vi[q] = vector_of(i + q * kThreads);
                    raw[q] = vi[q] >= 0 ? ld_vec(g.base + vi[q]) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int q = 0; q < kAtOnce; ++q)
                    if (vi[q] >= 0) c.visit(raw[q], vi[q]);
            }
        }
    }
    if (s.head) c.edge(0, [](float) {});
    if (s.tail) c.edge(g.nvec - 1, [](float) {});
}

// Pass 2 of the nucleus alone: the elements >= bound, and the mass of all elements of every warp's segment, which it leaves in
// sh.warp_above.
template <int DT>
__device__ __forceinline__ void collect_mass(const RowGeom& g, const LaneSpan& s, bool resident, uint32_t slot0, float bound,
                                             const CollectInto& to, SelectShared& sh, float scale, float row_max) {
    const Collector<DT> c(g, to, sh, bound);
    MassSum<DT> mass(scale, row_max);
    auto has = [&](const uint4& raw) {        // asked once per vector: it also counts its mass
        RawMax<DT> m;
        m.reset();
        m.fold(raw);
        const float top = m.value();
        mass.vector(raw, top);
        return c.above(top);
    };
    if (resident) {
        revisit_interior(s, slot0, [&](const uint4& raw, int vi) { if (has(raw)) c.visit(raw, vi); }, [&]() { return c.over(); });
    } else {
        // the streaming loop only lists the vectors, which are few, and all threads look at them afterwards: with the
        // elements looked at inside the unrolled loop, 2304 rows of 304 KB took 272 us instead of 174
        auto full = [&]() { return *static_cast<volatile uint32_t*>(&sh.n_vec) > kPoolCap; };
        stream_interior(s, slot0, [&](const uint4& raw, int vi) {
            if (has(raw) && !full()) {
                const uint32_t pos = atomicAdd(&sh.n_vec, 1u);
                if (pos < kPoolCap) sh.vec_list[pos] = static_cast<uint32_t>(vi);
            }
        }, full);
        __syncthreads();
        const uint32_t nv = sh.n_vec;
        if (nv <= kPoolCap) {
            for (uint32_t i = threadIdx.x; i < nv; i += kThreads) c.visit(ld_vec(g.base + sh.vec_list[i]), sh.vec_list[i]);
        } else {
            __syncthreads();
            if (threadIdx.x == 0) atomicAdd(&sh.n_cand, to.cap + 1);
        }
    }
    if (s.head) c.edge(0, [&](float x) { mass.one(x); });
    if (s.tail) c.edge(g.nvec - 1, [&](float x) { mass.one(x); });
    const unsigned long long m = warp_scan_mass(mass.sum, threadIdx.x & 31);
    if ((threadIdx.x & 31) == 31) sh.warp_above[threadIdx.x >> 5] = m;
}

// log2 of the groups of threads per warp whose maxima bound a top-k of a cluster of S blocks, if there are that many threads: in
// the cluster at least 3/2 k groups, which leave 1.65 to 2.1 k candidates (the search for the bound ends as soon as at most k/8
// more than k groups reach it); 4 k, which leave 1.15 to 1.35 k, where that mostly keeps the candidates within 128, of which a warp
// sorts four per lane and not eight (draft step of 32 rows of 304 KB, top-k 100: 11.6 -> 9.3 us).  Clusters of 3 and 6 come out at 768
// groups there from a k of 97 on, which are more than one warp searches: a descent gives the bound.
inline int choose_groups(int S, int k) {
    const long want = k > 64 && k <= 112 ? 4L * k : (3L * k + 1) / 2;
    int g = 0;
    while (g < 5 && (kWarps * S << g) < want) ++g;
    return g;
}

// The k-th largest of the maxima of groups of threads, 2^shift groups a warp (`best` is the thread's maximum), or somewhat
// less, left in sh.bound_key; the same in every block.  The first phase of bar_group has been opened, in all blocks.
__device__ __forceinline__ void group_bound(SelectShared& sh, float best, int shift, int S, int seg, int k, unsigned* status, int tid) {
    const int lane = tid & 31, width = 32 >> shift;
    for (int o = width >> 1; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    const int slot = (seg << shift) + (lane >> (5 - shift));
    const int n = (kWarps * S) << shift;
    const int first = lane & (width - 1);
    if (S == 1) {
        if (first == 0) sh.group_max[slot] = best;
        __syncthreads();
    } else {      // the threads of a group share the blocks to send to
        for (int r = first; r < S; r += width)
            push4(map_to_rank(smem_addr(&sh.group_max[slot]), r), map_to_rank(smem_addr(&sh.bar_group), r), __float_as_uint(best));
        if (tid < 32 && !mbar_wait_bounded(smem_addr(&sh.bar_group), 0) && tid == 0) atomicOr(status, SVIP_STATUS_WAIT_TIMEOUT);
        if (n > kOneWarp) __syncthreads();
    }
    if (n > kOneWarp) {       // of many values the upper 16 bits of the bound, by a descent
        const auto key_of = [&](int i) { return order_key(sh.group_max[i]); };
        const uint32_t key = pool_select<false>(sh, n, 0u, 32, 16, static_cast<uint32_t>(k), 0ull, tid, key_of, key_of);
        if (tid == 0) {
            sh.bound_key = key;
            sh.tied = 0;
        }
    } else if (tid < 32) {
        uint32_t top;
        const uint32_t key = n <= 128 ? kth_bound<4>(sh.group_max, n, static_cast<uint32_t>(k), lane, top)
                             : n <= 256 ? kth_bound<8>(sh.group_max, n, static_cast<uint32_t>(k), lane, top)
                                        : kth_bound<kOneWarp / 32>(sh.group_max, n, static_cast<uint32_t>(k), lane, top);
        if (lane == 0) {
            sh.bound_key = key;
            sh.tied = key == top;
        }
    }
    __syncthreads();
}

// A better bound for a top-k whose candidates do not fit; the same in every block.  The maxima of large groups bound next to
// nothing where the likely tokens are gathered in few warps (a vocabulary in order of frequency).  There every block that found
// too many elements takes the maxima of its threads, or of their stretches of vectors, as groups, stores what reaches
// the k-th largest of these (at least the first of them; a block alone whose row is in the ring goes by what it has stored, the 2048
// that came first), and any block with k elements stored takes their k-th largest: a
// bound for the row as well, and the blocks agree on the largest of these.  Rows of 50021 fp32 logits in order of frequency,
// top-k 50, against the maxima of the smallest groups of the cluster (few rows) or the k-th largest of what happened to be
// stored: 1 row 15.7 -> 13.3 us, 64 rows 22.4 -> 19.0, 300 rows 42.1 -> 36.6, 300 rows in reversed order 99.6 -> 35.9 (with
// the descent in place of the second attempt 123).  A block alone with its row in the ring, 600 rows of 32000 bf16: top-k 50 30.8 us,
// by the maxima of its threads first 49; top-k 100 39.5 and 90.  From a k of about 300 on those maxima say too little, and the attempt
// comes before the descent and not in its place (64 rows of 32000 bf16, top-k 300, 18.8 us without and 26.4 with it), hence the line
// at kRetryTopK, up to which it was seen to succeed.  A function of its own, because its code in line cost every top-k 3 %.
template <int DT>
__device__ __noinline__ uint32_t better_bound(SelectShared& sh, const CollectInto to, const RowGeom g, bool resident, uint32_t slot0,
                                              float best, int S, int rank, int k, unsigned* status) {
    const int tid = threadIdx.x;
    const uint32_t want = static_cast<uint32_t>(k);
    const uint32_t found = sh.n_cand;
    uint32_t bound = 0, stored = min(found, to.cap);
    if (found > to.cap && (S > 1 || !resident)) {
        const Stretches st(g);
        const int groups = resident ? kThreads : st.count * kThreads;
        if (resident) {
            __syncthreads();
            sh.group_max[tid] = best;       // where the candidates were
            stored = 0;
        }
        __syncthreads();
        if (groups >= k) {
            const auto key_of = [&](int i) {
                return resident ? order_key(sh.group_max[i]) : static_cast<uint32_t>((&sh.stretch_key[0][0])[i]) << 16;
            };
            bound = pool_select<false>(sh, groups, 0u, 32, 16, want, 0ull, tid, key_of, key_of);
        }
        if (bound > sh.bound_key) {
            __syncthreads();
            if (tid == 0) { sh.n_cand = 0; sh.n_vec = 0; sh.bound_key = bound; }
            __syncthreads();
            collect_top<DT>(g, lane_span<DT>(g, rank * kWarps + (tid >> 5), tid & 31), resident, st, slot0, best, rank, to, sh);
            __syncthreads();
            stored = min(sh.n_cand, to.cap);
        }
    }
    if (stored >= want) {
        const auto key_of = [&](int i) { return to.cand[i].key; };
        bound = max(bound, pool_select<false>(sh, static_cast<int>(stored), 0u, 32, 16, want, 0ull, tid, key_of, key_of));
    }
    if (S > 1) {
        if (tid == 0) {
            mbar_arrive_expect_tx(smem_addr(&sh.bar_group), static_cast<uint32_t>(S * 4));
            if (rank != 0) mbar_arrive_expect_tx(smem_addr(&sh.bar_verdict), 16);
        }
        if (tid < S) push4(map_to_rank(smem_addr(&sh.better[rank]), tid), map_to_rank(smem_addr(&sh.bar_group), tid), bound);
        bar_wait(sh.bar_group, 1, status, tid);
        for (int r = 0; r < S; ++r) bound = max(bound, sh.better[r]);
    }
    return bound;
}

// Barriers and counters of the path; needs no global memory, so it runs before the predecessor has finished.
__device__ __forceinline__ void candidate_open(SelectShared& sh, int S, int rank, int groups, bool use_k, int tid) {
    if (tid == 0) {
        if (S > 1) {
            mbar_init(smem_addr(&sh.ex.bar), 1);
            mbar_init(smem_addr(&sh.bar_group), 1);
            mbar_init(smem_addr(&sh.bar_verdict), 1);
            mbar_init(smem_addr(&sh.bar_pool), S);
            if (use_k) mbar_arrive_expect_tx(smem_addr(&sh.bar_group), static_cast<uint32_t>((kWarps * S * 4) << groups));
            else mbar_arrive_expect_tx(smem_addr(&sh.ex.bar), static_cast<uint32_t>(S * kWarps * sizeof(SegEntry)));
            if (rank != 0) mbar_arrive_expect_tx(smem_addr(&sh.bar_verdict), 16);   // block 0 gives the verdict
        }
        sh.n_cand = 0;
        sh.n_vec = 0;
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
    Candidate* const home = kTopK ? sh.cand : sh.cand_alone;
    const CollectInto to = S == 1 ? CollectInto{sh.landing, kPoolCap} : CollectInto{home, static_cast<uint32_t>(kTopK ? kCandPerBlock : kPoolCap)};
    const uint32_t region = kPoolCap / S;
    const bool resident = g.vps <= 32 * kStages;
    const Stretches stretches(g);
    // ---- pass 1: the largest logit of every thread, and from these the bound
    float best;
    if constexpr (kTopK) {
        best = stream_maxima<DT>(span, slot0, resident, stretches, sh.stretch_key);
    } else {
        RawMax<DT> m;
        m.reset();
        stream_interior(span, slot0, [&](const uint4& raw, int) { m.fold(raw); });
        best = m.value();
    }
    if (span.head || span.tail) {
        float x[EPV];
        if (span.head) { unpack_masked<DT>(ld_vec(g.base), 0, g, x); best = fmaxf(best, vec_max<EPV>(x)); }
        if (span.tail) { unpack_masked<DT>(ld_vec(g.base + g.nvec - 1), g.nvec - 1, g, x); best = fmaxf(best, vec_max<EPV>(x)); }
    }
    if constexpr (kTopK) {
        if (S > 1) cluster_wait();
        group_bound(sh, best, a.groups, S, seg, a.top_k, a.status, tid);
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
        }
        if (warp == 0) {       // one warp: in all of them these steps would get in each other's way
            if (S > 1 && !mbar_wait_bounded(smem_addr(&sh.ex.bar), 0) && lane == 0) atomicOr(a.status, SVIP_STATUS_WAIT_TIMEOUT);
            const Partial r = merge_entries<1>(LocalSegments{sh.ex.all}, S * kWarps, a.c, lane);
            // no element weighs more than 1, so the nucleus has at least top_p Z of them: a flat row does not fit
            const bool fits = fabsf(r.m) <= kMaxLogit && r.Z > 0.f && a.top_p * r.Z <= static_cast<float>(kPoolCap);
            // in log2 units, a little low for the roundings of the weights, and of the bound as a logit
            const float cut = log2f((1.f - a.top_p) * r.Z / static_cast<float>(g.V)) - 0.05f;
            if (lane == 0) {
                sh.blk_max = r.m;
                sh.bin = fits;
                sh.bound_key = order_key((__fmul_rn(r.m, a.c) + cut) / a.c - 5e-7f * fabsf(r.m));
            }
        }
        __syncthreads();
        row_max = sh.blk_max;       // what the radix descent needs first
        if (!sh.bin) return kVerdictDescend;   // in every block alike
    }
    uint32_t parity = 0;
    for (;;) {
        // ---- pass 2: the candidates
        pdl_launch_dependents();
        const uint32_t bound = sh.bound_key;
        if constexpr (kTopK) collect_top<DT>(g, span, resident, stretches, slot0, best, rank, to, sh);
        else collect_mass<DT>(g, span, resident, slot0, key_value(bound), to, sh, a.c, row_max);
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
                push8(map_to_rank(smem_addr(&sh.landing[rank * region + i]), 0), bar0, home[i].key, home[i].idx);
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
                verdict = kTopK && !fits && parity == 0 && !sh.tied && a.top_k <= kRetryTopK ? kVerdictRetry : kVerdictDescend;
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
                    const uint2 o = ld_remote8(map_to_rank(smem_addr(&home[t]), r));
                    scratch->pool[first + t] = Candidate{o.x, o.y};
                }
                if (tid == 0 && total < kPoolCap) scratch->pool[total] = Candidate{0u, 0xffffffffu};
                __syncthreads();
                return finish_pool<DT, kDraft, kTopK>(sh, *scratch, static_cast<int>(total), a, use_p, row_mass, row, tid,
                                                  key_out, tell);
            }
        }
        if (!kTopK || verdict != kVerdictRetry) return verdict;
        // ---- once more with a better bound
        __syncthreads();
        parity = 1;
        const uint32_t better = better_bound<DT>(sh, to, g, resident, slot0, best, S, rank, a.top_k, a.status);
        if (better <= bound) return kVerdictDescend;      // in every block alike
        __syncthreads();
        if (tid == 0) {
            sh.n_cand = 0;
            sh.n_vec = 0;
            sh.bound_key = better;
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
    RowGeom g = make_geom<DT>(rp, a.V, S * kWarps);
    const uint32_t slot0 = static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + tid * 16;
    const bool use_p = a.top_p < 1.0f;
    // a small k against the number of threads of the cluster, or the nucleus alone
    const bool by_candidates = kTopK ? a.top_k <= (S * kThreads) / 4 : use_p;
    const LaneSpan span = lane_span<DT>(g, rank * kWarps + warp, lane);
    if (by_candidates) candidate_open(sh, S, rank, a.groups, kTopK, tid);
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

    if (!kDraft) {
        // The geometry once more: kept across the candidate path it costs registers there, and few rows come here (threshold of 288
        // rows of 304 KB, top-k 50: 20.5 us, this way 19.3; the draft step does not gain).
        int again = row;
        asm volatile("" : "+r"(again));
        g = make_geom<DT>(static_cast<const char*>(a.logits) + static_cast<size_t>(again) * a.row_stride * ElemTraits<DT>::kBytes, a.V, S * kWarps);
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
