// Verification of a tree of draft candidates: several candidates per position, as when the length policy
// runs on top of a tree drafter (Section 3.3).  The paper states no accept rule for that setting; this is the
// published multi-candidate generalisation of Algorithms 2 and 4 (recursive rejection sampling): at a node with
// target distribution p, draft distribution q and candidates x_1..x_m,
//     p_1 = p;   accept x_i if r_i < min(1, p_i(x_i) / q(x_i));   else p_{i+1} = max(0, p_i - q) / S_i,
//     S_i = sum max(0, p_i - q);
// an accepted candidate becomes the current node; when none is accepted (or the node is a leaf) the next token is
// drawn from p_{m+1} (from p at a leaf) and the walk ends.  With one candidate per node it is svip_verify.
//
// One cluster per sequence.  The normalisers of every target row (and draft row) come from row_stats_kernel, as
// in the linear round.  The walk itself is a chain: every thread of the cluster takes the same decisions from the
// same bits (the two logits of the candidate, the normalisers, the masses S_i), and each rejection costs one pass
// over the node's two rows (from L2 after the first one) that sums max(0, p_i - q) per warp segment; the segment
// sums of the last pass are what the inverse CDF of the final draw needs, so the correction costs no further pass.
// Bound by the length of that chain, and the instructions of each of its links come from the instruction cache for
// the first time, so: what the decisions need besides the masses is fetched for all nodes at once before the walk starts,
// most of it while row_stats_kernel still runs; there is one copy of the loop over the rows, one vector at a time with the
// next one under way; and nothing of the walk lives in local memory.  64 trees of 14 nodes, 2 candidates a node, normalisers
// included: 32000 bf16 54.3 -> 36.3 us, 32000 fp32 77.6 -> 49.5; 32 trees of 152064 bf16 95.5 -> 55.1; 8 trees of
// 32000 bf16 27.8 -> 16.2 (four vectors of either row under way, the loop unrolled: 54 -> 41).
#pragma once

#include "svip_verify.cuh"

namespace svip {

constexpr int kTreeCache = 128;      // nodes whose tokens, draws and logits are fetched before the walk starts
constexpr int kMaxRejections = 16;   // candidates of one node that can be rejected before the rest is ignored

struct TreeArgs {
    const int32_t* tokens;    // [B, N]
    const int32_t* parent;    // [B, N]: -1 = child of the root, else a lower node index
    const void* q_logits;     // [B, N + 1] rows: root, then the nodes
    long q_row_stride;
    const float2* q_stats;    // per draft row (m, Z)
    const void* t_logits;
    long t_row_stride;
    const float2* p_stats;    // per target row (m, Z)
    int N, V;
    float c;
    const float* uniforms;    // [B, N + 1]: accept draw per node, then the final draw
    int32_t* n_accepted;      // [B]
    int32_t* path;            // [B, N]
    int32_t* next_token;      // [B]
    unsigned* status;
};

// Weights of the distribution after `nrej` rejections at a node, unnormalised: p for nrej == 0, else
// max(0, p_nrej - q) with p_1 = p and p_{i+1} = max(0, p_i - q) * rS[i].  Few members: registers are what the passes
// over the rows run short of.  Every operation is rounded by itself, so that of(), weights() and element() give the same
// number where a residual is at rounding level.
template <int DT>
struct TreeWeights {
    RowGeom gt;
    const char* qrow;
    float c, Mp, rZp, Mq, rZq;
    int nrej;
    const float* rS;            // shared memory: rS[i] = 1 / S_i, i = 1 .. nrej - 1 (entry 0 unused)
    struct Raw { uint4 t, q; };
    __device__ __forceinline__ float of(float p, float q) const {
        if (nrej == 0) return p;
        float r = p;
#pragma unroll 1
        for (int i = 1; i < nrej; ++i) r = __fmul_rn(fmaxf(__fsub_rn(r, q), 0.f), rS[i]);
        return fmaxf(__fsub_rn(r, q), 0.f);
    }
    // The draft row starts at the same 16-byte phase as the target row.
    __device__ __forceinline__ bool same_phase() const {
        return static_cast<int>(reinterpret_cast<uintptr_t>(qrow) & 15) == gt.pre * ElemTraits<DT>::kBytes;
    }
    __device__ __forceinline__ Raw load(int vi) const {
        Raw r;
        r.t = ld_vec(gt.base + vi);
        r.q = make_uint4(0, 0, 0, 0);
        if (nrej > 0 && same_phase())
            r.q = ld_vec(reinterpret_cast<const uint4*>(qrow - gt.pre * ElemTraits<DT>::kBytes) + vi);
        return r;
    }
    __device__ __forceinline__ void weights(int vi, const Raw& raw, float (&w)[ElemTraits<DT>::kEPV]) const {
        constexpr int EPV = ElemTraits<DT>::kEPV;
        unpack_masked<DT>(raw.t, vi, gt, w);
#pragma unroll
        for (int j = 0; j < EPV; ++j)      // NaN / -inf: no mass
            w[j] = __fmul_rn(ex2_approx(fmaxf(__fmaf_rn(w[j], c, -Mp), kArgFloor)), rZp);
        if (nrej == 0) return;
        float q[EPV];
        if (same_phase()) {
            unpack_masked<DT>(raw.q, vi, gt, q);
        } else {   // rows with different 16-byte phase: element loads
#pragma unroll
            for (int j = 0; j < EPV; ++j) {
                int i = vi * EPV + j - gt.pre;
                q[j] = (i >= 0 && i < gt.V) ? ElemTraits<DT>::load_one(qrow, i) : neg_inf();
            }
        }
#pragma unroll
        for (int j = 0; j < EPV; ++j) q[j] = __fmul_rn(ex2_approx(fmaxf(__fmaf_rn(q[j], c, -Mq), kArgFloor)), rZq);
#pragma unroll 1
        for (int i = 1; i < nrej; ++i) {
            const float s = rS[i];
#pragma unroll
            for (int j = 0; j < EPV; ++j) w[j] = __fmul_rn(fmaxf(__fsub_rn(w[j], q[j]), 0.f), s);
        }
#pragma unroll
        for (int j = 0; j < EPV; ++j) w[j] = fmaxf(__fsub_rn(w[j], q[j]), 0.f);
    }
    __device__ __forceinline__ float element(int vi, int j) const {
        const int i = vi * ElemTraits<DT>::kEPV + j - gt.pre;
        if (i < 0 || i >= gt.V) return 0.f;
        const char* trow = reinterpret_cast<const char*>(gt.base) + gt.pre * ElemTraits<DT>::kBytes;
        const float p = __fmul_rn(ex2_approx(fmaxf(__fmaf_rn(ElemTraits<DT>::load_one(trow, i), c, -Mp), kArgFloor)), rZp);
        float q = 0.f;
        if (nrej > 0) q = __fmul_rn(ex2_approx(fmaxf(__fmaf_rn(ElemTraits<DT>::load_one(qrow, i), c, -Mq), kArgFloor)), rZq);
        return of(p, q);
    }
};

// What the decision on node i needs: its parent, token and draw, and the logits of the token in the two rows of its
// parent.
struct TreeNode {
    int parent, token;
    float r, tv, dv;
};

template <int DT>
__device__ __forceinline__ TreeNode tree_node(const TreeArgs& a, int b, int i) {
    using E = ElemTraits<DT>;
    const size_t at = static_cast<size_t>(b) * a.N + i;
    TreeNode n;
    n.parent = __ldcg(a.parent + at);
    n.token = __ldcg(a.tokens + at);
    n.r = __ldcg(a.uniforms + static_cast<size_t>(b) * (a.N + 1) + i);
    n.tv = n.dv = 0.f;
    if (n.token >= 0 && n.token < a.V && n.parent >= -1 && n.parent < i) {
        const size_t row = static_cast<size_t>(b) * (a.N + 1) + n.parent + 1;
        n.tv = E::load_one_l2(static_cast<const char*>(a.t_logits) + row * a.t_row_stride * E::kBytes, n.token);
        n.dv = E::load_one_l2(static_cast<const char*>(a.q_logits) + row * a.q_row_stride * E::kBytes, n.token);
    }
    return n;
}

struct TreeShared {
    TreeNode node[kTreeCache];
    float2 ps[kTreeCache], qs[kTreeCache];    // (max, Z) of the target and draft rows: root, then the nodes
    float rS[kWarps][kMaxRejections];         // every warp keeps its own copy of what all of them compute
};

template <int DT>
__global__ void __launch_bounds__(kThreads, 2) verify_tree_kernel(TreeArgs a) {
    using E = ElemTraits<DT>;
    constexpr int EPV = E::kEPV;
    cg::cluster_group cluster = cg::this_cluster();
    const int S = cluster.dim_blocks().x;
    const int rank = cluster.block_rank();
    const int b = blockIdx.x / S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ RoundExchange ex;
    __shared__ ScanShared scan;
    __shared__ SegPick pick;
    __shared__ TreeShared sh;

    rounds_open(ex, S, tid);
    const int N = a.N;
    if (tid < N && tid < kTreeCache) sh.node[tid] = tree_node<DT>(a, b, tid);   // row_stats_kernel is the predecessor
    const float u_final = __ldcg(a.uniforms + static_cast<size_t>(b) * (N + 1) + N);
    pdl_wait();
    if (tid <= N && tid < kTreeCache) {
        const size_t row = static_cast<size_t>(b) * (N + 1) + tid;
        sh.ps[tid] = a.p_stats[row];
        sh.qs[tid] = a.q_stats[row];
    }
    int32_t* path = a.path + static_cast<size_t>(b) * N;
    const char* tl = static_cast<const char*>(a.t_logits);
    const char* ql = static_cast<const char*>(a.q_logits);
    const bool writer = rank == 0 && tid == 0;
    if (rank == 0)
        for (int i = tid; i < N; i += kThreads) path[i] = -1;
    __syncthreads();   // the -1 fill is in before thread 0 writes accepted nodes over it; sh is filled

    TreeWeights<DT> wf;
    wf.c = a.c;
    wf.rS = sh.rS[warp];
    int cur = -2, next = -1;         // the current node (-1: the root), and the one to go to
    int n_acc = 0, round = 0;
    int base = 0;                    // the children are looked for among 32 nodes at a time, in index order, from here ...
    unsigned kids = 0, bad = 0;      // ... those not yet tried, and the nodes whose parent is no earlier node
    bool malformed = false, drawn = false;   // drawn: pick holds the final draw of the current distribution
    while (true) {
        const auto stats = [&](const float2* cached, const float2* all) {
            return cur + 1 < kTreeCache ? cached[cur + 1] : all[static_cast<size_t>(b) * (N + 1) + cur + 1];
        };
        if (next != cur) {
            cur = next;
            const size_t row = static_cast<size_t>(b) * (N + 1) + cur + 1;
            wf.gt = make_geom<DT>(tl + row * a.t_row_stride * E::kBytes, a.V, S * kWarps);
            wf.qrow = ql + row * a.q_row_stride * E::kBytes;
            const float2 ps = stats(sh.ps, a.p_stats), qs = stats(sh.qs, a.q_stats);
            wf.Mp = __fmul_rn(ps.x, a.c);
            wf.rZp = 1.0f / ps.y;
            wf.Mq = __fmul_rn(qs.x, a.c);
            wf.rZq = 1.0f / qs.y;
            wf.nrej = 0;
            base = cur + 1 - 32;
            kids = bad = 0;
            drawn = false;
        }
        while (kids == 0 && base < N) {
            if (bad) malformed = true;
            base += 32;
            const int k = base + lane;
            int par = cur;
            if (k < N) par = k < kTreeCache ? sh.node[k].parent : __ldcg(a.parent + static_cast<size_t>(b) * N + k);
            kids = __ballot_sync(0xffffffffu, k < N && par == cur);
            bad = __ballot_sync(0xffffffffu, par < -1 || par >= k);
        }
        if (kids != 0 && wf.nrej >= kMaxRejections - 1) {     // the rest of the candidates is ignored
            malformed = true;
            kids = 0;
            base = N;
        }
        const bool last = kids == 0;      // no candidate accepted (or a leaf): the next token from this distribution
        if (last) {
            pdl_launch_dependents();
            if (drawn) break;
        } else {
            const int bit = __ffs(kids) - 1;
            kids &= kids - 1;
            const int i = base + bit;
            const TreeNode node = i < kTreeCache ? sh.node[i] : tree_node<DT>(a, b, i);
            bool acc = false;
            if (node.token >= 0 && node.token < a.V) {
                const bool q_zero = !(node.dv > neg_inf());
                if (wf.nrej == 0) {
                    // as in the linear round: the ratio from the difference of the two log2 arguments
                    acc = accept_test(node.tv, node.dv, stats(sh.ps, a.p_stats), stats(sh.qs, a.q_stats), a.c, node.r, false, false);
                } else {
                    // p_i(x) after the rejections so far; r < p_i / q without the division
                    const float p = ex2_approx(fmaxf(__fmaf_rn(node.tv, a.c, -wf.Mp), kArgFloor)) * wf.rZp;
                    const float q = q_zero ? 0.f : ex2_approx(fmaxf(__fmaf_rn(node.dv, a.c, -wf.Mq), kArgFloor)) * wf.rZq;
                    const float pi = wf.of(p, q) * wf.rS[wf.nrej];      // max(0, p_{i-1} - q) / S_{i-1}
                    acc = pi > 0.f && (q_zero || pi >= q || __fmul_rn(node.r, q) < pi);
                }
            }
            if (acc) {
                if (bad & ((1u << bit) - 1)) malformed = true;      // nodes ahead of this one
                if (writer) path[n_acc] = i;
                ++n_acc;
                next = i;
                continue;
            }
            wf.nrej += 1;
        }
        // The weights per warp segment, their total (after a rejection: S_i) and the segment that holds the final draw,
        // identical in every block of the cluster.
        int v_lo, v_hi;
        seg_range(wf.gt, rank * kWarps + warp, v_lo, v_hi);
        float mass = 0.f;
        typename TreeWeights<DT>::Raw next_raw = {};
        if (v_lo + lane < v_hi) next_raw = wf.load(v_lo + lane);
#pragma unroll 1
        for (int vi = v_lo + lane; vi < v_hi; vi += 32) {
            const typename TreeWeights<DT>::Raw raw = next_raw;
            if (vi + 32 < v_hi) next_raw = wf.load(vi + 32);
            float w[EPV];
            wf.weights(vi, raw, w);
#pragma unroll
            for (int j = 0; j < EPV; ++j) mass += w[j];
        }
        rounds_pick(ex, S, rank, round++, tid, warp_sum(mass), u_final, pick, a.status);
        if (last) break;
        drawn = pick.total > 0.f;
        if (drawn) {
            if (lane == 0) sh.rS[warp][wf.nrej] = 1.0f / pick.total;
            __syncwarp();
        } else {
            wf.nrej -= 1;      // no residual mass (rounding): the distribution stays as it was
        }
    }
    if (pick.total > 0.f) {
        if (pick.seg / kWarps == rank) {
            int v_lo, v_hi;
            seg_range(wf.gt, pick.seg, v_lo, v_hi);
            const int virt = fine_scan<EPV>(wf, v_lo, v_hi, pick.prefix, pick.target, scan, tid, lane, warp);
            if (tid == 0) a.next_token[b] = virt >= 0 ? virt - wf.gt.pre : 0;
        }
    } else if (writer) {
        atomicOr(a.status, SVIP_STATUS_NONFINITE_ROW);
        a.next_token[b] = 0;
    }
    if (writer) {
        a.n_accepted[b] = n_acc;
        if (malformed) atomicOr(a.status, SVIP_STATUS_BAD_TREE);
    }
}

// Greedy: a child is accepted iff its token is the argmax of the node's target row (Algorithm 3 at every
// node); otherwise that argmax is the next token (Algorithm 5).  One thread per sequence.
struct TreeGreedyArgs {
    const int32_t* tokens;
    const int32_t* parent;
    const int32_t* p_argmax;   // per target row
    int B, N;
    int32_t* n_accepted;
    int32_t* path;
    int32_t* next_token;
};

__global__ void __launch_bounds__(kPolicyThreads) verify_tree_greedy_kernel(TreeGreedyArgs a) {
    pdl_launch_dependents();
    pdl_wait();
    const int b = blockIdx.x * kPolicyThreads + threadIdx.x;
    if (b >= a.B) return;
    const int N = a.N;
    const int32_t* parent = a.parent + static_cast<size_t>(b) * N;
    const int32_t* tokens = a.tokens + static_cast<size_t>(b) * N;
    int32_t* path = a.path + static_cast<size_t>(b) * N;
    for (int i = 0; i < N; ++i) path[i] = -1;
    int cur = -1, n = 0;
    for (int step = 0; step <= N; ++step) {
        const int am = a.p_argmax[static_cast<size_t>(b) * (N + 1) + cur + 1];
        int taken = -1;
        for (int i = cur + 1; i < N && taken < 0; ++i)
            if (parent[i] == cur && tokens[i] == am) taken = i;
        if (taken < 0) { a.next_token[b] = am; break; }
        path[n++] = taken;
        cur = taken;
    }
    a.n_accepted[b] = n;
}

}  // namespace svip
