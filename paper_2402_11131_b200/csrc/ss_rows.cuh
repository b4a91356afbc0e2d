// Scans over rows of fp32 logits, shared by the verification and the draft-management kernels.
//
// A row (one node's or one stream's logits) is scanned by a cluster of 1, 2, 4 or 8 CTAs, each taking a contiguous
// segment; the CTAs hand their partial result to CTA 0 of the cluster through distributed shared memory, so a row is
// finished without a trip through global memory.  What a sequence does with its rows' results runs in the CTA that
// finishes the sequence's last row (one arrival per row on a global counter, nobody waits).
//
// The pass over a segment runs from registers, eight 16-byte loads per thread in flight.  Everything behind it is short:
// for one sequence these kernels are chains of latencies, in which most instructions execute once per CTA.  Measured and
// not kept: the segment staged in shared memory by bulk copies, one pass there for the maximum and one for the rest
// (1024 rows of 32000 logits: arg-max 35 us, softmax statistics 52 us, against 24 and 31 us before anything was asked for ahead).
//
// Order of logits.  Entries are ranked by an integer key that is monotone in the IEEE order of fp32 values, with
// -0 == +0 and every NaN below -inf, and equal keys by ascending index.  Compiled without fast-math: nothing is
// flushed or reassociated.
#pragma once
#include "ss_common.cuh"

namespace ss {

// Threads of a scan: 256 with eight 16-byte loads each in flight, four CTAs per SM (64 registers a thread): 128 KB in
// flight per SM.  Measured for 1024 rows of 32000 logits, arg-max / softmax statistics, before what is asked for ahead and the packed
// exponentials (21.6 / 27.2 us now): 23.6 / 31.2; four loads and six CTAs 28.2 / 36.6; 512 threads 25.1 / 36.1; two CTAs per row
// 27.5 / 39.1 (a CTA costs 4 us besides its loads).
constexpr int kRowThreads = 256;
constexpr int kRowVecs = 8;
constexpr int kRowBlocks = 4;         // CTAs per SM
constexpr int kRowParts = 64;         // partial results that CTA 0 of a cluster merges: 8 CTAs x 8 warps
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
// Row `row` of a [rows][vocab] array whose base is 16-byte aligned; CTA `rank` of `n_cta` takes logits [lo, hi).  Word
// i of `src` (16-byte aligned) is logit `at + i` of the row; the segment is words [skip, total).
struct Segment {
    const float* src;
    int at, skip, total;
};
__device__ __forceinline__ Segment make_segment(const float* base, size_t row, int vocab, int rank, int n_cta) {
    const int per = ((vocab + n_cta - 1) / n_cta + 3) & ~3;
    const int lo = min(vocab, rank * per), hi = min(vocab, lo + per);
    const float* first = base + row * static_cast<size_t>(vocab) + lo;
    Segment s;
    s.skip = static_cast<int>((reinterpret_cast<uintptr_t>(first) >> 2) & 3);
    s.src = first - s.skip;
    s.at = lo - s.skip;
    s.total = s.skip + hi - lo;
    return s;
}
// What a CTA asks for before the wait for the previous kernel: the first batch of its segment, on its way to L2.  No data reaches the SM,
// so it does not matter who writes the logits.  It pays where the previous kernel releases its successor early; behind one that does not,
// the wait is over at once.  Which CTAs ask (see rows_ahead for the sizes):
//   kEveryRow   all, whether a node owns their row or not
//   kOwnedRows  those of a row that a node owns by the tree's length as it stands before the wait.  The previous kernel may still be writing
//               it: a hint.  (Row t lies within the logits whatever it says.)
//   kIfWaiting  of those the ones that the GPU holds at once, by one thread and only if thread 32 is still in the wait (wait_passed) when the
//               length arrives: a prefetch that the loads meet costs 0.8 us (256 rows of 32000 in L2, 7.2 / 8.1)
// With kEveryRow the batch is also loaded beside the tree's length, with the others behind it.
enum RowsAhead { kEveryRow, kOwnedRows, kIfWaiting };
template <int AHEAD>
__device__ __forceinline__ void ask_ahead(const Segment& s, const ss_tree_desc& tree, int t, int slots, volatile int* passed) {
    constexpr int kBatchWords = 4 * kRowThreads * kRowVecs;
    if constexpr (AHEAD == kIfWaiting) {
        if (threadIdx.x != 0) return;
        *passed = 0;                                      // (later than thread 32's 1: it asks in vain)
        if (static_cast<int>((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) >= slots) return;
    }
    if constexpr (AHEAD != kEveryRow) {
        int n;
        asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(n) : "l"(&tree.n_nodes) : "memory");
        if (t >= max(n, 1)) return;
    }
    if constexpr (AHEAD == kIfWaiting) {
        const uint32_t bytes = static_cast<uint32_t>(min(s.total, kBatchWords)) / 4 * 16;
        if (*passed == 0 && bytes > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(s.src), "r"(bytes) : "memory");
    } else {
        static_assert(kRowThreads * 32 == kBatchWords, "a batch is a line of 32 logits to a thread");
        if (32 * static_cast<int>(threadIdx.x) < s.total) prefetch_l2(s.src + 32 * threadIdx.x);
    }
}
__device__ __forceinline__ void wait_passed(volatile int* passed) {
    if (threadIdx.x == 32) *passed = 1;
}
// Vector i of the segment (words 4 i .. 4 i + 3); words that are not the segment's read -inf.  The first and the last
// one are put together from single loads where they are not whole.
static __device__ __noinline__ float4 edge_vec(const float* src, int i, int skip, int total) {
    float4 q;
    q.x = 4 * i >= skip && 4 * i < total ? src[4 * i] : -INFINITY;
    q.y = 4 * i + 1 >= skip && 4 * i + 1 < total ? src[4 * i + 1] : -INFINITY;
    q.z = 4 * i + 2 >= skip && 4 * i + 2 < total ? src[4 * i + 2] : -INFINITY;
    q.w = 4 * i + 3 >= skip && 4 * i + 3 < total ? src[4 * i + 3] : -INFINITY;
    return q;
}
// A batch of a thread's vectors, from vector i on, those that are whole.  FIRST: the loads stay where they are written, so that they
// are on their way while what decides whether the row is scanned at all arrives (the length of the tree: a round trip to L2).
template <int NT, bool FIRST = false>
__device__ __forceinline__ void load_batch(const Segment& s, int i, float4 (&q)[kRowVecs]) {
    const int whole0 = s.skip ? 1 : 0, whole1 = s.total >> 2;                     // whole vectors: [whole0, whole1)
    const float4* vec = reinterpret_cast<const float4*>(s.src);
    #pragma unroll
    for (int v = 0; v < kRowVecs; ++v) {
        const int at = i + v * NT;
        q[v] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (at >= whole0 && at < whole1) {
            if constexpr (FIRST) asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(q[v].x), "=f"(q[v].y), "=f"(q[v].z), "=f"(q[v].w) : "l"(vec + at));
            else q[v] = __ldcs(vec + at);
        }
    }
}
template <int NT>
__device__ __forceinline__ void load_first(const Segment& s, float4 (&q)[kRowVecs]) { load_batch<NT, true>(s, static_cast<int>(threadIdx.x), q); }
// Calls f.batch(q, word) for batches of kRowVecs vectors, of which the first has been loaded; word: index of the first word of q[0],
// that of q[v] is v * 4 * NT further.  A thread meets its logits in ascending order.
template <int NT, typename F>
__device__ __forceinline__ void scan_segment(const Segment& s, F& f, float4 (&q)[kRowVecs]) {
    const int whole0 = s.skip ? 1 : 0, whole1 = s.total >> 2, n_vec = (s.total + 3) >> 2;
    for (int i = static_cast<int>(threadIdx.x); i < n_vec; i += NT * kRowVecs) {
        if (i >= NT * kRowVecs) load_batch<NT>(s, i, q);
        if (i < whole0 || (i + (kRowVecs - 1) * NT >= whole1 && (s.total & 3))) {
            #pragma unroll
            for (int v = 0; v < kRowVecs; ++v) {
                const int at = i + v * NT;
                if (at < n_vec && (at < whole0 || at >= whole1)) q[v] = edge_vec(s.src, at, s.skip, s.total);
            }
        }
        f.batch(q, 4 * i);
    }
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

// CTAs per row: more of them while the grid takes at most half of the GPU's slots -- the next kernel's CTAs then start in
// the other half and wait there, which hides its launch -- and a segment keeps two 16-byte loads per thread, a quarter of a batch.
// A segment of more than two batches is worth all slots: its batches of loads follow one another.  Measured against a
// line at a whole batch, greedy / soft / sampled: 16 rows of 51200 4.3 / 6.5 / 8.0 and 4.7 / 7.0 / 8.6 us, 32 of 51200 the same, 64 of 9000
// 4.8 / 7.5 / 9.0 and 4.3 / 6.6 / 7.6.  (For sampled verification alone, fewer CTAs per row were faster while its lists went through local
// memory; since they do not, more are: 64 rows of 32000, two CTAs and four 7.5 / 7.1 us, 32 of 51200 7.35 / 6.9.)
inline int row_cluster(long long rows, int vocab) {
    const long long slots = static_cast<long long>(kRowBlocks) * sm_count();
    int c = 1;
    while (c < 8 && vocab / (c * 2) >= kRowThreads * 8 && rows * c * 2 <= (vocab / c > 2 * kRowThreads * kRowVecs * 4 ? slots : slots / 2)) c *= 2;
    return c;
}
// kEveryRow on grids of at most half of the slots: at most a batch each for 296 CTAs, 9.7 MB, which little waits for.  64 rows of 32000,
// arg-max, loads behind the length / beside it and prefetched 5.2 / 4.5 us, 16 of them owned 4.25 / 4.2; 128 rows of 32000 6.8 / 6.1 (in L2
// 5.05 / 5.4) and, 32 owned, 5.45 / 5.45.  On larger grids it costs smaller trees more than it gives full ones: sixteen trees of 16 of 64 nodes, 32000 logits a row
// 11.9 us and 9.3 with owned rows only, 8000 logits 8.4 and 5.3.  kOwnedRows where the logits are too many to be in L2 (126 MB), 1024
// rows of 32000, kOwnedRows / kIfWaiting: 21.1 / 21.6 us, behind a kernel that does not release early 22.0 / 23.5; but 20000 logits (82 MB) that
// are in L2 10.8 / 9.4.
inline RowsAhead rows_ahead(long long rows, int vocab, int n_cta) {
    if (2 * rows * n_cta <= static_cast<long long>(kRowBlocks) * sm_count()) return kEveryRow;
    return rows * vocab > 25000000ll ? kOwnedRows : kIfWaiting;
}
inline int row_slots() { return kRowBlocks * sm_count(); }

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

// A partial result goes to the shared memory of the cluster's CTA 0; when this returns true (in CTA 0 only), all have
// arrived.  Every CTA of the cluster has called cluster_arrive() once, at its start; store(rank) stores.
template <typename F>
__device__ __forceinline__ bool hand_to_first(int rank, int n_cta, F&& store) {
    if (n_cta > 1) cluster_wait();                        // CTA 0 has started
    store();
    if (n_cta > 1) {
        cluster_arrive();
        if (rank != 0) return false;
        cluster_wait();
    } else {
        __syncthreads();
    }
    return true;
}

// ---- arg-max of a segment ----------------------------------------------------------------------------------------
struct ArgMax {
    float v = -INFINITY;
    int i = 0;
    template <int NT>
    __device__ __forceinline__ void take(const float4 (&q)[kRowVecs], int word) {
        #pragma unroll
        for (int k = 0; k < kRowVecs; ++k) {
            const int at = word + k * 4 * NT;
            if (q[k].x > v) { v = q[k].x; i = at; }
            if (q[k].y > v) { v = q[k].y; i = at + 1; }
            if (q[k].z > v) { v = q[k].z; i = at + 2; }
            if (q[k].w > v) { v = q[k].w; i = at + 3; }
        }
    }
    __device__ __forceinline__ void batch(const float4 (&q)[kRowVecs], int word) { take<kRowThreads>(q, word); }
    // A thread that met nothing above -inf has no entry: it does not know which of its logits are NaN
    __device__ __forceinline__ unsigned long long best(const Segment& s) const { return v > -INFINITY ? entry(order_key(v), s.at + i) : 0ull; }
};
// The best entry of a row of nothing but -inf and NaN (every thread of the CTA takes part; all get it)
static __device__ __noinline__ unsigned long long best_of_any(const float* base, size_t row, int vocab, unsigned long long* s_w) {
    unsigned long long e = 0ull;
    for (int i = static_cast<int>(threadIdx.x); i < vocab; i += kRowThreads) {
        const unsigned long long n = entry(order_key(base[row * static_cast<size_t>(vocab) + i]), i);
        e = n > e ? n : e;
    }
    e = warp_max_u64(e);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = e;
    __syncthreads();
    return warp_max_u64(s_w[threadIdx.x & (kRowThreads / 32 - 1)]);
}

// ---- the deepest accepted node ------------------------------------------------------------------------------------
// Tree arrays of a sequence in shared memory, loaded by the first SS_MAX_NODES threads (the ancestor words come last, from
// root_path, in the CTA that needs them)
struct TreeShared {
    int32_t parent[SS_MAX_NODES], depth[SS_MAX_NODES], tok[SS_MAX_NODES];
    unsigned long long anc[SS_MAX_NODES];
};
// The arrays' entries of thread i < T, loaded before a row is scanned and put in shared memory after it (a store right
// after the load would hold up the thread's scan by a round trip to L2)
struct TreeRegs {
    int32_t parent, depth, tok;
    __device__ __forceinline__ void load(const ss_tree_desc& tree, const int32_t* tokens, int T) {
        const int i = static_cast<int>(threadIdx.x);
        parent = -1; depth = 0; tok = -1;
        if (i < T) { parent = tree.parent[i]; depth = tree.depth[i]; tok = tokens[i]; }
    }
    __device__ __forceinline__ void store(TreeShared& s, int T) const {
        const int i = static_cast<int>(threadIdx.x);
        if (i < T) { s.parent[i] = parent; s.depth[i] = depth; s.tok[i] = tok; }
    }
};
// Ancestor word of node i from the parents (a verification needs no ancestor words in its descriptors).  The walk ends at a
// node whose parent is not below it: such a node is never ok, nor is anything behind it.
__device__ __forceinline__ unsigned long long root_path(const TreeShared& s, int i) {
    unsigned long long anc = 1ull << i;
    #pragma unroll 1
    for (int a = i, p = s.parent[i]; p >= 0 && p < a; a = p, p = s.parent[a]) anc |= 1ull << p;
    return anc;
}
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
