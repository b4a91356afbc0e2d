// Draft management around the attention: the next tree draft (Sec. 3.2.2, App. A.1), parallel tree pruning
// (Sec. 3.2.3), and the soft / sampled variants of the verification (App. A.2, App. B).
//
// All of them are one HBM-bound pass over rows of fp32 logits followed by a few dozen integer steps per sequence.  One
// kernel per call: a cluster per row scans it (see ss_rows.cuh) and leaves the row's result -- the k best entries, or
// the maximum with the softmax sums -- in its CTA 0; the CTA that finishes a sequence's last row does the sequence's
// tail, all nodes at once from their ancestor words.  The next draft has at most four rows per sequence, so one
// cluster takes the whole sequence and nothing goes through global memory.  Compiled without fast-math.
// Measured on a B200, before (chunks of 4096 logits, partial results and candidate lists through global memory, serial
// tails) and after: soft verification of 32 rows of 51200 logits 15.3 and 6.4 us, sampled verification of 64 rows of
// 32000 34.1 and 7.2 us, pruning over 1024 rows of 32000 126 and 31 us, the next draft of 16 sequences (64 rows of 32000) 15.6 and
// 5.3 us.  Pruning then 31.4 -> 28.4 with packed exponentials and without the sums that only the verification uses, 27.2 with owned rows
// asked for ahead.
#include <atomic>

#include "ss_draft_plan.h"
#include "ss_rows.cuh"

namespace ss {

// packed pairs of fp32 (one instruction for two values)
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr float kTinyExp = -200.f;                        // exp of it is 0 in fp32

// ---- the k best entries of a segment --------------------------------------------------------------------------------
// Pass 1 takes one maximum per thread.  The k-th largest warp maximum bounds the k-th best logit of the segment from
// below, and only a dozen logits or so reach that bound; the few threads that hold one find them (in
// the registers of pass 1 where the segment was one batch, else they read their logits again) and put them in a list, and each entry of the
// list counts how many are better.  Keeping a sorted list of k entries per thread costs 8 compare-and-swaps of 64-bit
// words per logit instead.  A logit for the list is read once more from memory, where it is in L2: picked out of the registers by an
// index, it takes the whole batch through a stack frame in local memory.  From HBM, before / after: sampled verification of 64 rows of 32000
// 9.4 / 7.2 us, 135 of 50257 16.3 / 12.0, 1024 of 8000 20.1 / 12.2, 1024 of 32000 40.2 / 30.3; 16 next drafts of four rows of 32000 8.6 / 5.3.
constexpr int kListCap = 512;
template <int NT>
struct TopKShared {
    static_assert(NT / 32 >= kMaxTopK, "the k-th largest warp maximum has to exist");
    unsigned long long part[kMaxClusterCtas * kMaxTopK];  // CTA 0 of a cluster: the lists of its CTAs, k entries each
    unsigned long long best[kMaxTopK];
    unsigned long long warp_best[NT / 32];
    unsigned long long list[kListCap];
    uint32_t warp_key[NT / 32];
    int n_list;
};
template <int NT>
struct ThreadMax {
    float v = -INFINITY;
    __device__ __forceinline__ void batch(const float4 (&q)[kRowVecs], int word) {
        #pragma unroll
        for (int k = 0; k < kRowVecs; ++k) v = fmaxf(v, fmaxf(fmaxf(q[k].x, q[k].y), fmaxf(q[k].z, q[k].w)));     // (a NaN is never the maximum)
    }
};
template <int NT>
struct Collect {
    const Segment& seg;
    TopKShared<NT>& s;
    float bound;
    __device__ __forceinline__ void batch(const float4 (&q)[kRowVecs], int word) {
        uint32_t hit = 0u;
        #pragma unroll
        for (int k = 0; k < kRowVecs; ++k)                // (a NaN is not below anything)
            hit |= ((q[k].x < bound ? 0u : 1u) | (q[k].y < bound ? 0u : 2u) | (q[k].z < bound ? 0u : 4u) | (q[k].w < bound ? 0u : 8u)) << (4 * k);
        static_assert(4 * kRowVecs <= 32, "a bit per logit");
        #pragma unroll 1
        for (; hit; hit &= hit - 1u) {
            const int j = __ffs(hit) - 1;
            const int at = word + (j >> 2) * 4 * NT + (j & 3);
            if (at < seg.skip || at >= seg.total) continue;
            const int p = atomicAdd(&s.n_list, 1);
            if (p < kListCap) s.list[p] = entry(order_key(seg.src[at]), seg.at + at);
        }
    }
};
// entry i of the distinct entries list[0 .. n) that has r better ones goes to best[r], r < k
__device__ __forceinline__ void rank_entry(const unsigned long long* list, int n, int i, int k, unsigned long long* best) {
    const unsigned long long e = list[i];
    int better = 0;
    #pragma unroll 4
    for (int j = 0; j < n; ++j) better += list[j] > e ? 1 : 0;
    if (better < k) best[better] = e;
}
// More candidates than the list holds (rows of equal logits, of -inf or of NaN): k passes over the segment, each for the
// best entry below the last, one logit at a time.
template <int NT>
static __device__ __noinline__ void select_by_passes(const Segment seg, int top_k, TopKShared<NT>& s) {
    unsigned long long below = ~0ull;
    for (int r = 0; r < top_k; ++r) {
        unsigned long long m = 0ull;
        for (int i = seg.skip + static_cast<int>(threadIdx.x); i < seg.total; i += NT) {
            const unsigned long long e = entry(order_key(seg.src[i]), seg.at + i);
            if (e < below && e > m) m = e;
        }
        m = warp_max_u64(m);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) s.warp_best[threadIdx.x >> 5] = m;
        __syncthreads();
        below = warp_max_u64(s.warp_best[threadIdx.x & (NT / 32 - 1)]);
        if (threadIdx.x == 0) s.best[r] = below;          // (0, no entry, once the segment is exhausted)
    }
}
// The k best entries of the segment in s.best, for every thread; q: the first batch of the segment
template <int NT>
__device__ __forceinline__ void segment_topk(const Segment& seg, int top_k, TopKShared<NT>& s, float4 (&q)[kRowVecs]) {
    constexpr int kWarps = NT / 32;
    const int lane = static_cast<int>(threadIdx.x) & 31, warp = static_cast<int>(threadIdx.x) >> 5;
    ThreadMax<NT> tm;
    scan_segment<NT>(seg, tm, q);
    const uint32_t wm = __reduce_max_sync(0xffffffffu, order_key(tm.v));
    if (lane == 0) s.warp_key[warp] = wm;
    if (threadIdx.x == 0) s.n_list = 0;
    if (threadIdx.x < kMaxTopK) s.best[threadIdx.x] = 0ull;
    __syncthreads();
    // the k-th largest warp maximum, equal ones in the order of their warps (every warp for itself)
    const uint32_t key = s.warp_key[lane & (kWarps - 1)];
    int before = 0;
    #pragma unroll
    for (int j = 0; j < kWarps; ++j) {
        const uint32_t o = __shfl_sync(0xffffffffu, key, j);
        before += (o > key || (o == key && j < (lane & (kWarps - 1)))) ? 1 : 0;
    }
    const float bound = key_value(__shfl_sync(0xffffffffu, key, __ffs(__ballot_sync(0xffffffffu, before == top_k - 1)) - 1));
    if (!(tm.v < bound)) {
        Collect<NT> collect{seg, s, bound};
        if (seg.total <= 4 * NT * kRowVecs) {
            collect.batch(q, 4 * static_cast<int>(threadIdx.x));
        } else {
            load_batch<NT>(seg, static_cast<int>(threadIdx.x), q);
            scan_segment<NT>(seg, collect, q);
        }
    }
    __syncthreads();
    const int n = s.n_list;
    if (n > kListCap) {
        select_by_passes<NT>(seg, top_k, s);
    } else {
        for (int i = static_cast<int>(threadIdx.x); i < n; i += NT) rank_entry(s.list, n, i, top_k, s.best);
    }
    __syncthreads();
}

// ---- softmax statistics: maximum (lowest index), Z = sum exp(x - m), W = sum (x - m) exp(x - m) ----------------------
struct Stats {
    unsigned long long best;      // entry of the maximum, 0: no comparable value
    float z, w;
};
// merges the lanes' statistics; every lane gets the result
static __device__ __noinline__ Stats warp_merge(Stats s) {
    const unsigned long long best = warp_max_u64(s.best);
    if (s.best != 0ull && s.best != best) {
        const float d = fmaxf(entry_value(s.best) - entry_value(best), kTinyExp), e = expf(d);
        s.w = (s.w + d * s.z) * e;
        s.z *= e;
    }
    #pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        s.z += __shfl_xor_sync(0xffffffffu, s.z, off);
        s.w += __shfl_xor_sync(0xffffffffu, s.w, off);
    }
    s.best = best;
    return s;
}
__device__ __forceinline__ Stats merge_two(const Stats& a, const Stats& b) {
    if (b.best == 0ull) return a;
    if (a.best == 0ull) return b;
    const bool first = a.best > b.best;
    Stats r = first ? a : b;
    const Stats& o = first ? b : a;
    const float d = fmaxf(entry_value(o.best) - entry_value(r.best), kTinyExp), e = expf(d);
    r.w += (o.w + d * o.z) * e;
    r.z += o.z * e;
    return r;
}
// exp(x - m) for pairs of logits: 2^t of t = (x - m) log2(e), and what t lost to rounding as a factor 1 + r ln(2).  Six packed
// operations, two clamps and two exponentials a pair: a third of what expf, the clamp and the sums take.  The clamp is for -inf
// and for NaN: they add nothing.  (exp(-100) is 0 with what is flushed to zero)
struct ExpPair {
    unsigned long long e, d;      // the exponentials; x - m
};
__device__ __forceinline__ ExpPair exp_pair(float x0, float x1, unsigned long long minus_m) {
    const unsigned long long log2e = pack2(1.44269502f, 1.44269502f), log2e_low = pack2(1.92596299e-8f, 1.92596299e-8f);
    const unsigned long long ln2 = pack2(0.693147182f, 0.693147182f), one = pack2(1.f, 1.f);
    float d0, d1;
    unpack2(add2(pack2(x0, x1), minus_m), d0, d1);
    const unsigned long long d = pack2(fmaxf(d0, -100.f), fmaxf(d1, -100.f));
    const unsigned long long t = mul2(d, log2e);
    const unsigned long long r = fma2(d, log2e_low, fma2(d, log2e, t ^ 0x8000000080000000ull));
    float t0, t1;
    unpack2(t, t0, t1);
    return {mul2(pack2(exp2_approx(t0), exp2_approx(t1)), fma2(r, ln2, one)), d};
}
// A thread's running statistics against its running maximum.  FULL: with the index of the maximum and W (pruning needs neither).
template <bool FULL>
struct RowStats {
    ArgMax am;
    unsigned long long z[2] = {0ull, 0ull}, w[2] = {0ull, 0ull};     // two pairs of partial sums each
    __device__ __forceinline__ void batch(const float4 (&q)[kRowVecs], int word) {
        const float m_old = am.v;
        if constexpr (FULL) {
            am.batch(q, word);
        } else {
            #pragma unroll
            for (int k = 0; k < kRowVecs; ++k) am.v = fmaxf(am.v, fmaxf(fmaxf(q[k].x, q[k].y), fmaxf(q[k].z, q[k].w)));     // (a NaN is never the maximum)
        }
        if (am.v > m_old) {
            const float d = fmaxf(m_old - am.v, kTinyExp), e = expf(d);
            #pragma unroll
            for (int j = 0; j < 2; ++j) {
                if constexpr (FULL) w[j] = mul2(fma2(pack2(d, d), z[j], w[j]), pack2(e, e));
                z[j] = mul2(z[j], pack2(e, e));
            }
        }
        const unsigned long long minus_m = pack2(-am.v, -am.v);
        #pragma unroll
        for (int k = 0; k < kRowVecs; ++k) {
            #pragma unroll
            for (int j = 0; j < 2; ++j) {
                const ExpPair p = j ? exp_pair(q[k].z, q[k].w, minus_m) : exp_pair(q[k].x, q[k].y, minus_m);
                z[j] = add2(z[j], p.e);
                if constexpr (FULL) w[j] = fma2(p.d, p.e, w[j]);
            }
        }
    }
    __device__ __forceinline__ Stats stats(const Segment& s) const {
        Stats st;
        st.best = am.best(s);
        float a, b;
        unpack2(add2(z[0], z[1]), a, b);
        st.z = a + b;
        unpack2(add2(w[0], w[1]), a, b);
        st.w = a + b;
        return st;
    }
};
// =============================================================================================================
// Next draft: the k best tokens of each of the gamma stream-logit rows of the last accepted node; tree of
// 1 + sum_g k^g nodes (cut after max_nodes), level by level, children of a node in rank order.  A cluster of
// gamma x n_cta CTAs per sequence.
struct DraftShape {
    int32_t parent[SS_MAX_NODES], depth[SS_MAX_NODES];
    int32_t child[SS_MAX_NODES];                          // which of the gamma x kMaxTopK best tokens the node carries
    int32_t total, bonus;
};
// The first SS_MAX_NODES threads work out the tree while the previous kernel drains, wait for that kernel, and leave the
// descriptor visible to the whole GPU: an attention call behind this kernel may read it before its own wait.  (1.3B step
// 161.6 us so, 163.0 with the release at the end of the kernel; alone, 16 drafts take 9.4 us, 9.0 with that.)
static __device__ __forceinline__ void write_shape(DraftShape& s, int gamma, int k, int max_nodes, const int32_t* bonus_token, ss_tree_desc* tree) {
    const int i = static_cast<int>(threadIdx.x);
    // level `dep` holds nodes [start, start + sz); node i there is child o % k of node prev_start + o / k
    int total = 1, par = -1, dep = 0, child = 0, start = 1, sz = k, prev_start = 0;
    #pragma unroll 1
    for (int lev = 1; lev <= gamma && start < max_nodes; ++lev) {
        if (i >= start && i < start + sz && i < max_nodes) {
            const int o = i - start;
            par = prev_start + o / k;
            child = (lev - 1) * kMaxTopK + o % k;
            dep = lev;
        }
        total = min(start + sz, max_nodes);
        prev_start = start; start += sz; sz *= k;
    }
    s.parent[i] = par; s.depth[i] = dep; s.child[i] = child;
    if (i == 0) s.total = total;
    asm volatile("bar.sync 1, 64;" ::: "memory");
    unsigned long long anc = 0ull;
    if (i < total) {
        #pragma unroll 1
        for (int a = i; a >= 0; a = s.parent[a]) anc |= 1ull << a;
    }
    wait_for_previous_kernel();
    if (i == 0) s.bonus = *bonus_token;
    tree->parent[i] = par;
    tree->depth[i] = dep;
    tree->anc_mask[i] = anc;
    if (i == 0) { tree->n_nodes = total; tree->gamma = gamma; tree->max_depth = s.depth[total - 1]; tree->reserved = 0; }
    __threadfence();
    asm volatile("bar.sync 1, 64;" ::: "memory");
}
static_assert(kDraftBatch == 4 * kDraftThreads * kRowVecs, "a batch of loads");
__global__ void __launch_bounds__(kDraftThreads, 2)
next_draft_kernel(const float* __restrict__ stream_logits, int n_rows, const int32_t* __restrict__ row_index,
                  const int32_t* __restrict__ bonus_token, int gamma, int vocab, int k, int max_nodes, int n_cta,
                  int32_t* __restrict__ draft_tokens, ss_tree_desc* __restrict__ trees) {
    const int rank = blockIdx.x, b = blockIdx.y;
    const int g = rank / n_cta, part = rank - g * n_cta;
    __shared__ TopKShared<kDraftThreads> s;
    __shared__ unsigned long long s_top[SS_MAX_GAMMA * kMaxTopK];
    __shared__ DraftShape s_shape;
    cluster_arrive();                                     // CTA 0 must have started before anyone stores to its shared memory
    // The shape of the tree does not depend on the logits: CTA 0 writes the descriptor before anything else, and the next kernel
    // may be scheduled once it is in memory.
    if (rank == 0 && threadIdx.x < SS_MAX_NODES) write_shape(s_shape, gamma, k, max_nodes, bonus_token + b, trees + b);
    wait_for_previous_kernel();
    if (rank != 0 || threadIdx.x == 0) release_next_kernel();
    int r = row_index ? row_index[b] : 0;
    r = min(max(r, 0), n_rows - 1);
    const Segment seg = make_segment(stream_logits, (static_cast<size_t>(b) * n_rows + r) * gamma + g, vocab, part, n_cta);
    float4 q[kRowVecs];
    load_first<kDraftThreads>(seg, q);
    segment_topk<kDraftThreads>(seg, k, s, q);
    const int i = static_cast<int>(threadIdx.x), warp = i >> 5, lane = i & 31;
    // the lists of a row lie one after another
    cluster_wait();                                       // (CTA 0 has started)
    if (i < k) cluster_store_u64(cluster_addr(s.part + rank * k + i, 0), s.best[i]);
    cluster_arrive();
    if (rank != 0) return;
    cluster_wait();
    if (warp < gamma) {                                   // one warp per stream
        const unsigned long long* list = s.part + warp * n_cta * k;
        for (int j = lane; j < n_cta * k; j += 32) rank_entry(list, n_cta * k, j, k, s_top + warp * kMaxTopK);
    }
    __syncthreads();
    if (i < max_nodes)
        draft_tokens[static_cast<size_t>(b) * max_nodes + i] =
            i == 0 ? s_shape.bonus : i < s_shape.total ? entry_index(s_top[s_shape.child[i]]) : -1;
}

// =============================================================================================================
// Row statistics of every node's logits, then per sequence either the pruning of the tree or the soft verification.
struct NodeTailArgs {
    float threshold, eps, delta;
    float* edge_prob;                 // [B][max_nodes]
    float* node_entropy;              // verification, may be null
    int32_t *new_index, *kept_nodes, *kept_tokens;     // pruning
    ss_tree_desc* pruned_trees;                         // pruning
    int32_t *accept_len, *accept_path, *last_node, *bonus_token;   // verification
};
// What a row leaves for the sequence's tail: which of its children's edges are ok, and its arg-max
struct RowOut {
    unsigned long long ok_children;
    int32_t argmax, pad;
};

// Pruning, after the edges are judged: a node survives when every edge of its root path is ok; survivors keep their
// order.  Node c's new index is the number of survivors before it.  Called by the first SS_MAX_NODES threads.
__device__ __forceinline__ void prune_tail(int T, int max_nodes, int b, unsigned long long ok, const TreeShared& tree, int gamma, const NodeTailArgs& ta) {
    const int i = static_cast<int>(threadIdx.x);
    unsigned long long keep = 0ull;
    int md = 0;
    for (int c = 0; c < T; ++c) {                         // (broadcast reads; every thread builds the same word)
        const bool kp = (tree.anc[c] & ~ok) == 0ull;
        keep |= kp ? 1ull << c : 0ull;
        md = kp ? max(md, tree.depth[c]) : md;
    }
    const int n = __popcll(keep);
    ss_tree_desc* out = ta.pruned_trees + b;
    const size_t row0 = static_cast<size_t>(b) * max_nodes;
    const bool live = i < T && ((keep >> i) & 1ull);
    const int at = __popcll(keep & ((1ull << i) - 1ull));          // new index of node i if it survives
    if (i < max_nodes) ta.new_index[row0 + i] = live ? at : -1;
    if (live) {
        const int p = i == 0 ? -1 : tree.parent[i];
        unsigned long long anc = 0ull;
        for (unsigned long long rest = tree.anc[i]; rest != 0ull; rest &= rest - 1ull)
            anc |= 1ull << __popcll(keep & ((rest & (0ull - rest)) - 1ull));
        out->parent[at] = p < 0 ? -1 : __popcll(keep & ((1ull << p) - 1ull));
        out->depth[at] = tree.depth[i];
        out->anc_mask[at] = anc;
        ta.kept_nodes[row0 + at] = i;
        ta.kept_tokens[row0 + at] = tree.tok[i];
    }
    if (i >= n) {
        out->parent[i] = -1;
        out->depth[i] = 0;
        out->anc_mask[i] = 0ull;
        if (i < max_nodes) { ta.kept_nodes[row0 + i] = -1; ta.kept_tokens[row0 + i] = -1; }
    }
    if (i == 0) { out->n_nodes = n; out->gamma = gamma; out->max_depth = md; out->reserved = 0; }
}

// SOFT: the verification, else the pruning; AHEAD: see RowsAhead
template <bool SOFT, int AHEAD>
__global__ void __launch_bounds__(kRowThreads, kRowBlocks)
node_stats_kernel(const float* __restrict__ logits, const int32_t* __restrict__ tokens, const ss_tree_desc* __restrict__ trees,
                  int max_nodes, int vocab, int n_cta, int slots, NodeTailArgs ta, int32_t* __restrict__ counters, RowOut* __restrict__ rows) {
    const int rank = blockIdx.x, t = blockIdx.y, b = blockIdx.z;
    __shared__ Stats s_part[kRowParts];
    __shared__ unsigned long long s_any[kRowThreads / 32];
    __shared__ bool s_none;
    __shared__ TreeShared s_tree;
    __shared__ float s_lse, s_bar;
    __shared__ uint32_t s_ok[2];
    __shared__ volatile int s_passed;
    if (n_cta > 1) cluster_arrive();
    const size_t row = static_cast<size_t>(b) * max_nodes + t;
    const Segment seg = make_segment(logits, row, vocab, rank, n_cta);
    ask_ahead<AHEAD>(seg, trees[b], t, slots, &s_passed);
    wait_for_previous_kernel();
    if (SOFT) release_next_kernel();                      // (pruning writes descriptors)
    if (AHEAD == kIfWaiting) wait_passed(&s_passed);
    float4 q[kRowVecs];
    if (AHEAD == kEveryRow) load_first<kRowThreads>(seg, q);    // (a row that no node owns is within the logits too)
    const int T = min(max(trees[b].n_nodes, 0), max_nodes);
    if (t >= max(T, 1)) {
        if (n_cta > 1) cluster_wait();
        return;
    }
    const int i = static_cast<int>(threadIdx.x);
    if (AHEAD != kEveryRow) load_first<kRowThreads>(seg, q);
    TreeRegs tree;
    tree.load(trees[b], tokens + static_cast<size_t>(b) * max_nodes, T);
    RowStats<SOFT> rs;
    scan_segment<kRowThreads>(seg, rs, q);
    tree.store(s_tree, T);
    // the logits of the node's children: on their way while the statistics are merged
    bool mine = false, legal = false;
    float child = 0.f;
    if (rank == 0 && i > 0 && i < T && tree.parent == t) {
        mine = true;
        legal = t < i && tree.tok >= 0 && tree.tok < vocab;
        if (legal) child = logits[row * vocab + tree.tok];
    }
    Stats st = warp_merge(rs.stats(seg));
    constexpr int kWarps = kRowThreads / 32;
    if (!hand_to_first(rank, n_cta, [&]() {
            if ((i & 31) == 0) {
                const uint32_t at = cluster_addr(&s_part[rank * kWarps + (i >> 5)], 0);
                cluster_store_u64(at, st.best);
                cluster_store_u64(at + 8, (static_cast<unsigned long long>(__float_as_uint(st.w)) << 32) | __float_as_uint(st.z));
            }
        }))
        return;
    if (i < 32) {
        Stats none;
        none.best = 0ull; none.z = 0.f; none.w = 0.f;
        const int n_part = n_cta * kWarps;
        st = warp_merge(merge_two(i < n_part ? s_part[i] : none, i + 32 < n_part ? s_part[i + 32] : none));
    }
    if (i == 0) {
        // log-sum-exp and entropy of the row, and the bar that its children's probabilities have to reach
        const float logz = logf(st.z);
        s_lse = entry_value(st.best) + logz;
        s_bar = ta.threshold;
        if (SOFT) {
            const float ent = logz - st.w / st.z;
            s_bar = fminf(ta.eps, ta.delta * expf(-ent));
            if (t < T && ta.node_entropy) ta.node_entropy[row] = ent;
        }
        if (t == 0 && T > 0) ta.edge_prob[row] = 1.f;     // the root
        s_none = st.best == 0ull;
    }
    __syncthreads();
    if (SOFT && s_none) st.best = best_of_any(logits, row, vocab, s_any);
    if (i < SS_MAX_NODES) {
        const float prob = legal ? expf(child - s_lse) : 0.f;
        if (mine) ta.edge_prob[static_cast<size_t>(b) * max_nodes + i] = prob;
        const uint32_t ok = __ballot_sync(0xffffffffu, legal && prob >= s_bar);
        if ((i & 31) == 0) s_ok[i >> 5] = ok;
        // a node whose parent is no node at all belongs to no row: row 0 looks after it
        if (t == 0 && i > 0 && i < T && (tree.parent < 0 || tree.parent >= T)) ta.edge_prob[static_cast<size_t>(b) * max_nodes + i] = 0.f;
    }
    __syncthreads();
    if (i == 0) {
        RowOut o;
        o.ok_children = (static_cast<unsigned long long>(s_ok[1]) << 32) | s_ok[0];
        o.argmax = entry_index(st.best);
        o.pad = 0;
        rows[row] = o;
    }
    if (!arrive_last(&counters[b], max(T, 1))) return;

    // ---- the sequence's tail: the first 64 threads -------------------------------------------------------------
    if (i >= SS_MAX_NODES) return;
    const RowOut* const mine_row = rows + static_cast<size_t>(b) * max_nodes + i;
    const unsigned long long okc = i < T ? __ldcg(&mine_row->ok_children) : 0ull;
    const int argmax = i < max(T, 1) ? __ldcg(&mine_row->argmax) : 0;
    __shared__ uint32_t s_all[2][2];
    __shared__ int32_t s_am[SS_MAX_NODES];
    if (i < T) s_tree.anc[i] = root_path(s_tree, i);      // (while the rows' results are on their way)
    s_am[i] = argmax;
    const uint32_t lo = __reduce_or_sync(0xffffffffu, static_cast<uint32_t>(okc));
    const uint32_t hi = __reduce_or_sync(0xffffffffu, static_cast<uint32_t>(okc >> 32));
    if ((i & 31) == 0) { s_all[i >> 5][0] = lo; s_all[i >> 5][1] = hi; }
    asm volatile("bar.sync 1, 64;" ::: "memory");
    const unsigned long long ok = 1ull | (static_cast<unsigned long long>(s_all[0][1] | s_all[1][1]) << 32) | (s_all[0][0] | s_all[1][0]);
    if (i == 0) counters[b] = 0;                          // leave the workspace ready for the next call
    if constexpr (!SOFT) {
        prune_tail(T, max_nodes, b, ok, s_tree, trees[b].gamma, ta);
    } else if (i < 32) {
        int len = 1;
        const int node = accept_path_of(s_tree, T, ok, ta.accept_path + static_cast<size_t>(b) * SS_PATH_STRIDE, &len);
        if (i == 0) {
            ta.accept_len[b] = len;
            ta.last_node[b] = node;
            ta.bonus_token[b] = s_am[node];
        }
    }
}

// =============================================================================================================
// Verification against tokens drawn from the softmax over each node's k largest logits (temperature 1).
__global__ void __launch_bounds__(kRowThreads, kRowBlocks)
sampled_verify_kernel(const float* __restrict__ logits, const int32_t* __restrict__ tokens, const ss_tree_desc* __restrict__ trees,
                      const float* __restrict__ uniforms, int max_nodes, int vocab, int k, int n_cta, int slots,
                      int32_t* __restrict__ accept_len, int32_t* __restrict__ accept_path, int32_t* __restrict__ last_node,
                      int32_t* __restrict__ bonus_token, int32_t* __restrict__ node_token, int32_t* __restrict__ counters,
                      int32_t* __restrict__ drawn) {
    const int rank = blockIdx.x, t = blockIdx.y, b = blockIdx.z;
    __shared__ TopKShared<kRowThreads> s;
    __shared__ TreeShared s_tree;
    __shared__ int32_t s_draw[SS_MAX_NODES];
    __shared__ volatile int s_passed;
    if (n_cta > 1) cluster_arrive();
    const size_t row = static_cast<size_t>(b) * max_nodes + t;
    const Segment seg = make_segment(logits, row, vocab, rank, n_cta);
    ask_ahead<kIfWaiting>(seg, trees[b], t, slots, &s_passed);
    wait_for_previous_kernel();
    release_next_kernel();
    wait_passed(&s_passed);
    const int T = min(max(trees[b].n_nodes, 0), max_nodes);
    if (t >= max(T, 1)) {
        if (n_cta > 1) cluster_wait();
        return;
    }
    float4 q[kRowVecs];
    load_first<kRowThreads>(seg, q);
    TreeRegs tree;
    tree.load(trees[b], tokens + static_cast<size_t>(b) * max_nodes, T);
    const float u = uniforms[row];
    segment_topk<kRowThreads>(seg, k, s, q);
    tree.store(s_tree, T);
    const int i = static_cast<int>(threadIdx.x);
    if (n_cta > 1) {
        if (!hand_to_first(rank, n_cta, [&]() { if (i < k) cluster_store_u64(cluster_addr(s.part + rank * k + i, 0), s.best[i]); })) return;
        if (i < n_cta * k) rank_entry(s.part, n_cta * k, i, k, s.best);
        __syncthreads();
    }
    if (i < 32) {
        // lane r holds the r-th best; every lane adds the probabilities up in rank order, as one thread would
        const unsigned long long top = i < k ? s.best[i] : 0ull;
        const float x0 = __shfl_sync(0xffffffffu, entry_value(top), 0);
        const float ex = i < k ? expf(entry_value(top) - x0) : 0.f;
        float z = 0.f, cdf = 0.f;
        #pragma unroll 1
        for (int r = 0; r < k; ++r) z += __shfl_sync(0xffffffffu, ex, r);
        int pick = k - 1;
        bool found = false;
        #pragma unroll 1
        for (int r = 0; r < k; ++r) {
            cdf += __shfl_sync(0xffffffffu, ex, r) / z;
            if (!found && cdf > u) { pick = r; found = true; }
        }
        const int token = __shfl_sync(0xffffffffu, entry_index(top), pick);
        if (i == 0) {
            drawn[row] = token;
            if (node_token && t < T) node_token[row] = token;
        }
    }
    if (!arrive_last(&counters[b], max(T, 1))) return;

    if (i < SS_MAX_NODES) {
        const int32_t token_i = i < max(T, 1) ? __ldcg(drawn + static_cast<size_t>(b) * max_nodes + i) : -1;
        if (i < T) s_tree.anc[i] = root_path(s_tree, i);
        s_draw[i] = token_i;
    }
    __syncthreads();
    if (i >= 32) return;
    const unsigned long long ok = matching_nodes(s_tree, T, s_draw);
    int len = 1;
    const int node = accept_path_of(s_tree, T, ok, accept_path + static_cast<size_t>(b) * SS_PATH_STRIDE, &len);
    if (i == 0) {
        accept_len[b] = len;
        last_node[b] = node;
        bonus_token[b] = s_draw[node];
        counters[b] = 0;
    }
}

// Whether the current device can hold a cluster of that many CTAs of the next draft (12 or 16): it takes a GPC with as many free places, which
// a partition of a GPU may not have.  Asked for once per device and size.
static bool draft_cluster_fits(int ctas) {
    static std::atomic<signed char> known[64][kMaxClusterCtas + 1];          // 0: not asked for yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    signed char k = known[dev][ctas].load(std::memory_order_relaxed);
    if (k == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctas, 1);
        cfg.blockDim = dim3(kDraftThreads);
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim = {static_cast<unsigned>(ctas), 1, 1};
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(next_draft_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, next_draft_kernel, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        known[dev][ctas].store(k = n > 0 ? 1 : -1, std::memory_order_relaxed);
    }
    return k > 0;
}

static size_t scan_workspace(int32_t batch, int32_t rows, int32_t vocab, size_t per_chunk) {
    if (batch < 1 || rows < 1 || vocab < 1) return 0;
    // (room for a partial result per 4096 logits, as callers have always been told; one result per row is used)
    const size_t n_chunks = (static_cast<size_t>(vocab) + 4095) / 4096;
    const size_t counters = (static_cast<size_t>(batch) * sizeof(int32_t) + 255) / 256 * 256;
    return kWsHeaderBytes + counters + static_cast<size_t>(batch) * rows * n_chunks * per_chunk;
}

}  // namespace ss

extern "C" size_t ss_next_draft_workspace_bytes(int32_t batch, int32_t gamma, int32_t vocab) {
    return ss::scan_workspace(batch, gamma < 1 ? 1 : gamma, vocab, ss::kMaxTopK * sizeof(unsigned long long));
}

extern "C" int32_t ss_next_draft(const float* stream_logits, int32_t n_rows, const int32_t* row_index, const int32_t* bonus_token,
                                 int32_t batch, int32_t gamma, int32_t vocab, int32_t top_k, int32_t max_nodes,
                                 int32_t* draft_tokens, ss_tree_desc* trees, void* workspace, size_t workspace_bytes, void* stream) {
    if (!stream_logits || !bonus_token || !draft_tokens || !trees || !workspace) return SS_ERR_INVALID_ARG;
    if (batch < 1 || batch > 65535 || n_rows < 1 || vocab < 1 || gamma < 1 || top_k < 1 || max_nodes < 1) return SS_ERR_INVALID_ARG;
    if (gamma > SS_MAX_GAMMA || top_k > SS_MAX_TOPK || top_k > vocab || max_nodes > SS_MAX_NODES) return SS_ERR_UNSUPPORTED;
    if (!ss::aligned16(stream_logits) || !ss::aligned16(workspace)) return SS_ERR_INVALID_ARG;
    if (workspace_bytes < ss_next_draft_workspace_bytes(batch, gamma, vocab)) return SS_ERR_WORKSPACE;
    const cudaError_t err = ss::launch_draft(batch, gamma, vocab, ss::draft_cluster_fits, [&](int n_cta) {
        const cudaError_t e = ss::launch_rows(ss::next_draft_kernel, dim3(gamma * n_cta, batch), dim3(ss::kDraftThreads), gamma * n_cta, true,
                                              static_cast<cudaStream_t>(stream), stream_logits, n_rows, row_index, bonus_token, gamma, vocab,
                                              top_k, max_nodes, n_cta, draft_tokens, trees);
        if (e != cudaSuccess && gamma * n_cta > ss::kPortableCtas) (void)cudaGetLastError();    // (there is a way out)
        return e;
    });
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}

extern "C" size_t ss_tree_prune_workspace_bytes(int32_t batch, int32_t max_nodes, int32_t vocab) {
    return ss::scan_workspace(batch, max_nodes, vocab, sizeof(ss::Stats));
}

template <bool SOFT>
static int32_t launch_node_stats(const float* logits, const int32_t* tokens, const ss_tree_desc* trees, int32_t batch,
                                 int32_t max_nodes, int32_t vocab, const ss::NodeTailArgs& ta, void* workspace, size_t workspace_bytes,
                                 void* stream) {
    if (!logits || !tokens || !trees || !workspace || !ta.edge_prob) return SS_ERR_INVALID_ARG;
    if (batch < 1 || batch > 65535 || max_nodes < 1 || vocab < 1) return SS_ERR_INVALID_ARG;
    if (max_nodes > SS_MAX_NODES) return SS_ERR_UNSUPPORTED;
    if (!ss::aligned16(logits) || !ss::aligned16(workspace)) return SS_ERR_INVALID_ARG;
    if (workspace_bytes < ss_tree_prune_workspace_bytes(batch, max_nodes, vocab)) return SS_ERR_WORKSPACE;
    const long long n_rows = static_cast<long long>(batch) * max_nodes;
    const int n_cta = ss::row_cluster(n_rows, vocab);
    char* ws = static_cast<char*>(workspace);
    const size_t counter_bytes = (static_cast<size_t>(batch) * sizeof(int32_t) + 255) / 256 * 256;
    const ss::RowsAhead ahead = ss::rows_ahead(n_rows, vocab, n_cta);
    const auto kernel = ahead == ss::kEveryRow    ? ss::node_stats_kernel<SOFT, ss::kEveryRow>
                        : ahead == ss::kOwnedRows ? ss::node_stats_kernel<SOFT, ss::kOwnedRows>
                                                  : ss::node_stats_kernel<SOFT, ss::kIfWaiting>;
    const cudaError_t err = ss::launch_rows(kernel, dim3(n_cta, max_nodes, batch), dim3(ss::kRowThreads), n_cta, true,
                                            static_cast<cudaStream_t>(stream), logits, tokens, trees, max_nodes, vocab, n_cta, ss::row_slots(), ta,
                                            reinterpret_cast<int32_t*>(ws + ss::kWsHeaderBytes),
                                            reinterpret_cast<ss::RowOut*>(ws + ss::kWsHeaderBytes + counter_bytes));
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}

extern "C" int32_t ss_tree_prune(const float* exit_logits, const int32_t* draft_tokens, const ss_tree_desc* trees, int32_t batch,
                                 int32_t max_nodes, int32_t vocab, float threshold, float* edge_prob, int32_t* new_index,
                                 int32_t* kept_nodes, int32_t* kept_tokens, ss_tree_desc* pruned_trees, void* workspace,
                                 size_t workspace_bytes, void* stream) {
    if (!new_index || !kept_nodes || !kept_tokens || !pruned_trees) return SS_ERR_INVALID_ARG;
    if (!(threshold == threshold)) return SS_ERR_INVALID_ARG;
    ss::NodeTailArgs ta = {};
    ta.threshold = threshold; ta.edge_prob = edge_prob;
    ta.new_index = new_index; ta.kept_nodes = kept_nodes; ta.kept_tokens = kept_tokens; ta.pruned_trees = pruned_trees;
    return launch_node_stats<false>(exit_logits, draft_tokens, trees, batch, max_nodes, vocab, ta, workspace, workspace_bytes, stream);
}

extern "C" int32_t ss_tree_verify_soft(const float* logits, const int32_t* draft_tokens, const ss_tree_desc* trees, int32_t batch,
                                       int32_t max_nodes, int32_t vocab, float eps, float delta, int32_t* accept_len,
                                       int32_t* accept_path, int32_t* last_node, int32_t* bonus_token, float* edge_prob,
                                       float* node_entropy, void* workspace, size_t workspace_bytes, void* stream) {
    if (!accept_len || !accept_path || !last_node || !bonus_token) return SS_ERR_INVALID_ARG;
    if (!(eps == eps) || !(delta == delta)) return SS_ERR_INVALID_ARG;
    ss::NodeTailArgs ta = {};
    ta.eps = eps; ta.delta = delta; ta.edge_prob = edge_prob; ta.node_entropy = node_entropy;
    ta.accept_len = accept_len; ta.accept_path = accept_path; ta.last_node = last_node; ta.bonus_token = bonus_token;
    return launch_node_stats<true>(logits, draft_tokens, trees, batch, max_nodes, vocab, ta, workspace, workspace_bytes, stream);
}

extern "C" size_t ss_tree_verify_sampled_workspace_bytes(int32_t batch, int32_t max_nodes, int32_t vocab) {
    return ss::scan_workspace(batch, max_nodes, vocab, ss::kMaxTopK * sizeof(unsigned long long));
}

extern "C" int32_t ss_tree_verify_sampled(const float* logits, const int32_t* draft_tokens, const ss_tree_desc* trees,
                                          const float* uniforms, int32_t batch, int32_t max_nodes, int32_t vocab, int32_t top_k,
                                          int32_t* accept_len, int32_t* accept_path, int32_t* last_node, int32_t* bonus_token,
                                          int32_t* node_token, void* workspace, size_t workspace_bytes, void* stream) {
    if (!logits || !draft_tokens || !trees || !uniforms || !accept_len || !accept_path || !last_node || !bonus_token || !workspace)
        return SS_ERR_INVALID_ARG;
    if (batch < 1 || batch > 65535 || max_nodes < 1 || vocab < 1 || top_k < 1) return SS_ERR_INVALID_ARG;
    if (max_nodes > SS_MAX_NODES || top_k > SS_MAX_TOPK || top_k > vocab) return SS_ERR_UNSUPPORTED;
    if (!ss::aligned16(logits) || !ss::aligned16(workspace)) return SS_ERR_INVALID_ARG;
    if (workspace_bytes < ss_tree_verify_sampled_workspace_bytes(batch, max_nodes, vocab)) return SS_ERR_WORKSPACE;
    const long long n_rows = static_cast<long long>(batch) * max_nodes;
    const int n_cta = ss::row_cluster(n_rows, vocab);
    char* ws = static_cast<char*>(workspace);
    const size_t counter_bytes = (static_cast<size_t>(batch) * sizeof(int32_t) + 255) / 256 * 256;
    const cudaError_t err = ss::launch_rows(ss::sampled_verify_kernel, dim3(n_cta, max_nodes, batch), dim3(ss::kRowThreads), n_cta, true,
                                            static_cast<cudaStream_t>(stream), logits, draft_tokens, trees, uniforms, max_nodes, vocab, top_k,
                                            n_cta, ss::row_slots(), accept_len, accept_path, last_node, bonus_token, node_token,
                                            reinterpret_cast<int32_t*>(ws + ss::kWsHeaderBytes),
                                            reinterpret_cast<int32_t*>(ws + ss::kWsHeaderBytes + counter_bytes));
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}
