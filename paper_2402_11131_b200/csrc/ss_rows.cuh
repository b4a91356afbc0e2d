// Scans over rows of fp32 logits, shared by the verification and the draft-management kernels.
//
// A row (one node's or one stream's logits) is scanned by a cluster of 1, 2, 4 or 8 CTAs, each taking a contiguous
// segment; the CTAs hand their partial result to CTA 0 of the cluster through distributed shared memory, so a row is
// finished without a trip through global memory.  What a sequence does with its rows' results runs in the CTA that
// finishes the sequence's last row (one arrival per row on a global counter, nobody waits).
//
// Order of logits.  Entries are ranked by an integer key that is monotone in the IEEE order of fp32 values, with
// -0 == +0 and every NaN below -inf, and equal keys by ascending index.  Compiled without fast-math: nothing is
// flushed or reassociated.
#pragma once
#include "ss_common.cuh"

namespace ss {

// 512 threads with eight 16-byte loads in flight each: 64 KB per CTA, two CTAs per SM, 19 MB over the GPU -- about
// twice what the HBM latency needs at full bandwidth, and a 16000-logit segment is one batch of loads.
constexpr int kRowThreads = 512;
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kRowVecs = 8;
constexpr int kMaxTopK = SS_MAX_TOPK;

__device__ __forceinline__ uint32_t order_key(float x) {
    if (x != x) return 0u;
    x += 0.0f;                                         // -0 -> +0
    const uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t key) {
    if (key == 0u) return __uint_as_float(0x7fc00000u);
    return __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
}
// larger = better: (key, lower index first); 0 = no entry
__device__ __forceinline__ unsigned long long entry(uint32_t key, int idx) {
    return (static_cast<unsigned long long>(key) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(idx));
}
__device__ __forceinline__ int entry_index(unsigned long long e) { return static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(e)); }
__device__ __forceinline__ uint32_t entry_key(unsigned long long e) { return static_cast<uint32_t>(e >> 32); }
__device__ __forceinline__ float entry_value(unsigned long long e) { return key_value(entry_key(e)); }

// maximum over the warp: two 32-bit reductions (the low words of the lanes that hold the largest high word)
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
    const uint32_t hi = static_cast<uint32_t>(v >> 32);
    const uint32_t top = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t low = __reduce_max_sync(0xffffffffu, hi == top ? static_cast<uint32_t>(v) : 0u);
    return (static_cast<unsigned long long>(top) << 32) | low;
}

// ---- the segment of a row that a CTA scans ----------------------------------------------------------------------
// Row `row` of a [rows][vocab] array whose base is 16-byte aligned; CTA `rank` of `n_cta` takes logits [lo, hi).
struct Segment {
    const float* base;
    size_t start;                 // first element of the row in the array
    int lo, hi;                   // logits of the row
};
__device__ __forceinline__ Segment make_segment(const float* base, size_t row, int vocab, int rank, int n_cta) {
    Segment s;
    s.base = base;
    s.start = row * static_cast<size_t>(vocab);
    const int per = ((vocab + n_cta - 1) / n_cta + 3) & ~3;
    s.lo = min(vocab, rank * per);
    s.hi = min(vocab, s.lo + per);
    return s;
}
// Calls f.batch(x, first) for batches of kRowVecs x 4 logits (first[v]: index in the row of x[4 v]; logits past the
// end read -inf) and f.one(x, index) for the up to six logits before the first and after the last 16-byte boundary.
// A thread meets its logits in ascending order of their index, except that the ones at the ends come last.
template <typename F>
__device__ __forceinline__ void scan_segment(const Segment& s, F& f) {
    const size_t e0 = s.start + s.lo, e1 = s.start + s.hi;
    const size_t v0 = (e0 + 3) >> 2, v1 = max(e1 >> 2, v0);
    const float4* vec = reinterpret_cast<const float4*>(s.base);
    const int n_vec = static_cast<int>(v1 - v0);
    const int at0 = static_cast<int>(v0 * 4 - s.start);                   // index in the row of the first vector
    for (int i = static_cast<int>(threadIdx.x); i < n_vec; i += kRowThreads * kRowVecs) {
        float x[4 * kRowVecs];
        int first[kRowVecs];
        #pragma unroll
        for (int v = 0; v < kRowVecs; ++v) {
            const int at = i + v * kRowThreads;
            float4 q = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (at < n_vec) q = __ldcs(vec + v0 + at);
            first[v] = at0 + 4 * at;
            x[4 * v] = q.x; x[4 * v + 1] = q.y; x[4 * v + 2] = q.z; x[4 * v + 3] = q.w;
        }
        f.batch(x, first);
    }
    // the ends: thread i < 3 the i-th logit before the first vector, threads 32.. those after the last
    const int head = static_cast<int>(min(v0 * 4, e1) - e0), tail0 = static_cast<int>(v1 * 4 - s.start);
    const int i = static_cast<int>(threadIdx.x);
    if (i < head) f.one(s.base[e0 + i], s.lo + i);
    if (i >= 32 && v1 * 4 >= e0 && tail0 + (i - 32) < s.hi && head < s.hi - s.lo) f.one(s.base[s.start + tail0 + (i - 32)], tail0 + (i - 32));
}

// ---- cluster plumbing --------------------------------------------------------------------------------------------
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of a shared-memory object of this CTA in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_store_u64(uint32_t addr, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// CTAs per row: more of them while the rows do not fill the SMs and a segment stays at a batch of loads or more (a
// shorter segment would leave threads without work and cost only the hand-over)
inline int row_cluster(long long rows, int vocab) {
    int c = 1;
    while (c < 8 && rows * c * 2 <= 2ll * sm_count() && vocab / (c * 2) >= kRowThreads * 4) c *= 2;
    return c;
}

// The first CTA of a row's cluster to see all rows of the sequence done returns true (every thread of it; it then sees
// what every other row's CTA wrote before its own call).  Word `counter` is zero between calls.
__device__ __forceinline__ bool arrive_last(int32_t* counter, int expected) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t prev;
        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(prev) : "l"(counter) : "memory");
        s_last = prev == expected - 1;
    }
    __syncthreads();
    return s_last;
}

// ---- arg-max of a row ---------------------------------------------------------------------------------------------
struct ArgMax {
    float v = -INFINITY;
    int i = 0x7fffffff;
    __device__ __forceinline__ void batch(const float (&x)[4 * kRowVecs], const int (&first)[kRowVecs]) {
        #pragma unroll
        for (int q = 0; q < 4 * kRowVecs; ++q)
            if (x[q] > v) { v = x[q]; i = first[q >> 2] + (q & 3); }
    }
    __device__ __forceinline__ void one(float x, int at) {
        if (x > v || (x == v && at < i)) { v = x; i = at; }
    }
};
// A thread's entry.  A thread that saw nothing above -inf does not know which of its logits are -inf and which are
// NaN; it counts as without an entry, and a row in which no thread has one is scanned again (entry_of_any).
__device__ __forceinline__ unsigned long long entry_of(const ArgMax& a) { return a.v > -INFINITY ? entry(order_key(a.v), a.i) : 0ull; }
struct AnyMax {
    unsigned long long e = 0ull;
    __device__ __forceinline__ void batch(const float (&x)[4 * kRowVecs], const int (&first)[kRowVecs]) {}
    __device__ __forceinline__ void one(float x, int at) {
        const unsigned long long n = entry(order_key(x), at);
        e = n > e ? n : e;
    }
};
// the best entry of a segment, one logit at a time (only for rows of -inf and NaN)
static __device__ __noinline__ unsigned long long entry_of_any(const Segment s) {
    AnyMax m;
    for (int i = s.lo + static_cast<int>(threadIdx.x); i < s.hi; i += kRowThreads) m.one(s.base[s.start + i], i);
    return m.e;
}
// maximum over the CTA, known to every thread of warp 0 (others: 0); `s_w` is a scratch array of kRowWarps words
__device__ __forceinline__ unsigned long long block_max(unsigned long long e, unsigned long long* s_w) {
    e = warp_max_u64(e);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x >= 32) return 0ull;
    return warp_max_u64(threadIdx.x < kRowWarps ? s_w[threadIdx.x] : 0ull);
}

// ---- the deepest accepted node ------------------------------------------------------------------------------------
// Tree arrays of a sequence in shared memory, loaded by the first SS_MAX_NODES threads
struct TreeShared {
    int32_t parent[SS_MAX_NODES], depth[SS_MAX_NODES], tok[SS_MAX_NODES];
    unsigned long long anc[SS_MAX_NODES];
};
// The arrays' entries of thread i < T, loaded before a row is scanned and put in shared memory after it (a store right
// after the load would hold up the thread's scan by a round trip to L2)
struct TreeRegs {
    int32_t parent, depth, tok;
    unsigned long long anc;
    __device__ __forceinline__ void load(const ss_tree_desc& tree, const int32_t* tokens, int T) {
        const int i = static_cast<int>(threadIdx.x);
        parent = -1; depth = 0; tok = -1; anc = 0ull;
        if (i < T) { parent = tree.parent[i]; depth = tree.depth[i]; anc = tree.anc_mask[i]; tok = tokens[i]; }
    }
    __device__ __forceinline__ void store(TreeShared& s, int T) const {
        const int i = static_cast<int>(threadIdx.x);
        if (i < T) { s.parent[i] = parent; s.depth[i] = depth; s.anc[i] = anc; s.tok[i] = tok; }
    }
};
// Bit c: node c's token is the one that `chosen` names for its parent (and bit 0, the root); one warp
__device__ __forceinline__ unsigned long long matching_nodes(const TreeShared& s, int T, const int32_t* chosen) {
    unsigned long long ok = 1ull;
    #pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = static_cast<int>(threadIdx.x & 31) + 32 * h;
        bool match = false;
        if (c > 0 && c < T) {
            const int p = s.parent[c];
            match = p >= 0 && p < c && s.tok[c] == chosen[p];
        }
        ok |= static_cast<unsigned long long>(__ballot_sync(0xffffffffu, match)) << (32 * h);
    }
    return ok;
}
// Called by the 32 lanes of one warp.  Bit c of `ok`: node c matches what its parent's row says (bit 0, the root, is
// set).  A node is valid when its whole root path is ok; the deepest valid node wins, the lowest index among equally
// deep ones.  Its root path is its ancestor word in ascending order (a parent's index is below its children's).
__device__ __forceinline__ int accept_path_of(const TreeShared& s, int T, unsigned long long ok, int32_t* path, int* len_out) {
    const int lane = static_cast<int>(threadIdx.x) & 31;
    uint32_t best = SS_MAX_NODES - 1;                     // the root: depth 0, node 0
    #pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c > 0 && c < T && (s.anc[c] & ~ok) == 0ull && s.depth[c] > 0)
            best = max(best, static_cast<uint32_t>(s.depth[c]) * SS_MAX_NODES + (SS_MAX_NODES - 1 - c));
    }
    best = __reduce_max_sync(0xffffffffu, best);
    const int node = SS_MAX_NODES - 1 - static_cast<int>(best & (SS_MAX_NODES - 1));
    const unsigned long long anc = node == 0 ? 1ull : s.anc[node];
    const int len = static_cast<int>(best / SS_MAX_NODES) + 1;
    #pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        if (i >= __popcll(anc)) path[i] = -1;
        if ((anc >> i) & 1ull) path[__popcll(anc & ((1ull << i) - 1ull))] = i;
    }
    *len_out = len;
    return node;
}

}  // namespace ss
