// Greedy tree verification (Sec. 3.2.2, App. A.1): per-node arg-max over the vocabulary, then the deepest node of the
// tree whose whole root path matches.
//
// HBM-bound in a batch (4*T*V bytes of logits per sequence, read once), a chain of latencies for one sequence.  One
// launch: a cluster per row (see ss_rows.cuh) finds the row's arg-max; the CTA that finishes a sequence's last row
// reads the T arg-maxes and picks the path from the ancestor words, all nodes at once.  Measured on a B200, before (a grid of
// 4096-logit chunks, one arrival per chunk, a serial walk) and after: 64 rows of 32000 logits 8.7 and 5.0 us, 1024 such
// rows 37.3 and 24.1 us; with the prefetch 21.6 (6.1 TB/s).
#include "ss_rows.cuh"

namespace ss {

template <int AHEAD>
__global__ void __launch_bounds__(kRowThreads, kRowBlocks)
tree_verify_kernel(const float* __restrict__ logits, const int32_t* __restrict__ tokens,
                   const ss_tree_desc* __restrict__ trees, int max_nodes, int vocab, int n_cta, int slots,
                   int32_t* __restrict__ accept_len, int32_t* __restrict__ accept_path,
                   int32_t* __restrict__ last_node, int32_t* __restrict__ bonus_token,
                   int32_t* __restrict__ node_argmax, int32_t* __restrict__ counters, int32_t* __restrict__ row_argmax) {
    const int rank = blockIdx.x, t = blockIdx.y, b = blockIdx.z;
    __shared__ unsigned long long s_part[kRowParts];
    __shared__ int32_t s_am[SS_MAX_NODES];
    __shared__ TreeShared s_tree;
    __shared__ volatile int s_passed;
    if (n_cta > 1) cluster_arrive();                      // CTA 0 must have started before anyone stores to its shared memory
    const Segment seg = make_segment(logits, static_cast<size_t>(b) * max_nodes + t, vocab, rank, n_cta);
    ask_ahead<AHEAD>(seg, trees[b], t, slots, &s_passed);
    wait_for_previous_kernel();
    release_next_kernel();
    if (AHEAD == kIfWaiting) wait_passed(&s_passed);
    float4 q[kRowVecs];
    if (AHEAD == kEveryRow) load_first<kRowThreads>(seg, q);    // (a row that no node owns is within the logits too)
    const int T = min(max(trees[b].n_nodes, 0), max_nodes);     // a descriptor is never trusted beyond the arrays' extent
    if (t >= max(T, 1)) {                                 // (the whole cluster: t is its row)
        if (n_cta > 1) cluster_wait();
        return;
    }
    if (AHEAD != kEveryRow) load_first<kRowThreads>(seg, q);
    TreeRegs tree;
    tree.load(trees[b], tokens + static_cast<size_t>(b) * max_nodes, T);
    ArgMax am;
    scan_segment<kRowThreads>(seg, am, q);
    tree.store(s_tree, T);
    unsigned long long best = warp_max_u64(am.best(seg));
    constexpr int kWarps = kRowThreads / 32;
    if (!hand_to_first(rank, n_cta, [&]() {
            if ((threadIdx.x & 31) == 0) cluster_store_u64(cluster_addr(&s_part[rank * kWarps + (threadIdx.x >> 5)], 0), best);
        }))
        return;
    const int lane = static_cast<int>(threadIdx.x) & 31, n_part = n_cta * kWarps;
    best = warp_max_u64(max(lane < n_part ? s_part[lane] : 0ull, lane + 32 < n_part ? s_part[lane + 32] : 0ull));
    if (best == 0ull) best = best_of_any(logits, static_cast<size_t>(b) * max_nodes + t, vocab, s_part);    // (CTA-uniform)
    if (threadIdx.x == 0) {
        const int i = entry_index(best);
        row_argmax[static_cast<size_t>(b) * max_nodes + t] = i;
        if (node_argmax && t < T) node_argmax[static_cast<size_t>(b) * max_nodes + t] = i;
    }
    if (!arrive_last(&counters[b], max(T, 1))) return;

    const int i = static_cast<int>(threadIdx.x);
    if (i < SS_MAX_NODES) {
        const int32_t am_i = i < max(T, 1) ? __ldcg(row_argmax + static_cast<size_t>(b) * max_nodes + i) : -1;
        if (i < T) s_tree.anc[i] = root_path(s_tree, i);  // (while the arg-max is on its way)
        s_am[i] = am_i;
    }
    __syncthreads();
    if (i >= 32) return;
    const unsigned long long ok = matching_nodes(s_tree, T, s_am);
    int len = 1;
    const int node = accept_path_of(s_tree, T, ok, accept_path + static_cast<size_t>(b) * SS_PATH_STRIDE, &len);
    if (i == 0) {
        accept_len[b] = len;
        last_node[b] = node;
        bonus_token[b] = s_am[node];
        counters[b] = 0;   // leave the workspace ready for the next call
    }
}

static cudaError_t launch_verify(const float* logits, const int32_t* tokens, const ss_tree_desc* trees, int batch, int max_nodes, int vocab,
                                 int32_t* accept_len, int32_t* accept_path, int32_t* last_node, int32_t* bonus_token, int32_t* node_argmax,
                                 char* ws, size_t counter_bytes, cudaStream_t stream, bool early) {
    const long long rows = static_cast<long long>(batch) * max_nodes;
    const int n_cta = row_cluster(rows, vocab);
    const RowsAhead ahead = rows_ahead(rows, vocab, n_cta);
    const auto kernel = ahead == kEveryRow ? tree_verify_kernel<kEveryRow> : ahead == kOwnedRows ? tree_verify_kernel<kOwnedRows> : tree_verify_kernel<kIfWaiting>;
    return launch_rows(kernel, dim3(n_cta, max_nodes, batch), dim3(kRowThreads), n_cta, early, stream, logits, tokens, trees, max_nodes, vocab,
                       n_cta, row_slots(), accept_len, accept_path, last_node, bonus_token, node_argmax,
                       reinterpret_cast<int32_t*>(ws + kWsHeaderBytes), reinterpret_cast<int32_t*>(ws + kWsHeaderBytes + counter_bytes));
}

}  // namespace ss

extern "C" size_t ss_tree_verify_workspace_bytes(int32_t batch, int32_t max_nodes, int32_t vocab) {
    if (batch < 1 || max_nodes < 1 || vocab < 1) return 0;
    // (room for an 8-byte entry per 4096 logits, as callers have always been told; an arg-max per row is used)
    const size_t n_chunks = (static_cast<size_t>(vocab) + 4095) / 4096;
    const size_t counters = (static_cast<size_t>(batch) * sizeof(int32_t) + 255) / 256 * 256;
    return ss::kWsHeaderBytes + counters + static_cast<size_t>(batch) * max_nodes * n_chunks * 8;
}

extern "C" int32_t ss_tree_verify(const float* logits, const int32_t* draft_tokens, const ss_tree_desc* trees,
                                  int32_t batch, int32_t max_nodes, int32_t vocab, int32_t* accept_len,
                                  int32_t* accept_path, int32_t* last_node, int32_t* bonus_token,
                                  int32_t* node_argmax, void* workspace, size_t workspace_bytes, void* stream) {
    if (!logits || !draft_tokens || !trees || !accept_len || !accept_path || !last_node || !bonus_token ||
        !workspace)
        return SS_ERR_INVALID_ARG;
    if (batch < 1 || max_nodes < 1 || vocab < 1 || batch > 65535) return SS_ERR_INVALID_ARG;
    if (max_nodes > SS_MAX_NODES) return SS_ERR_UNSUPPORTED;
    if (!ss::aligned16(logits) || !ss::aligned16(workspace)) return SS_ERR_INVALID_ARG;
    if (workspace_bytes < ss_tree_verify_workspace_bytes(batch, max_nodes, vocab)) return SS_ERR_WORKSPACE;
    const size_t counter_bytes = (static_cast<size_t>(batch) * sizeof(int32_t) + 255) / 256 * 256;
    const cudaError_t err = ss::launch_verify(logits, draft_tokens, trees, batch, max_nodes, vocab, accept_len, accept_path, last_node, bonus_token,
                                              node_argmax, static_cast<char*>(workspace), counter_bytes, static_cast<cudaStream_t>(stream), true);
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------------
// Verification without a caller-provided workspace.
//
// Some callers cannot hand this library scratch memory: code that runs where allocating device
// memory is not allowed (inside a region that forbids cudaMalloc, a plug-in that owns no allocator,
// a real-time loop whose memory was fixed at start-up).  For them the scratch of the verification
// kernel lives in this fixed device array, which every GPU that loads the library holds until the
// process exits.  All calls on a device share it, so calls that overlap on that device race.
namespace ss {

static __device__ __align__(256) unsigned char g_verify_static_scratch[SS_VERIFY_STATIC_SCRATCH_BYTES];

// Device address of the array, looked up once per device.  In host code the array's name is only a
// host-side handle, never a device address: the address must come from cudaGetSymbolAddress, taken
// with the device current.
static void* verify_static_scratch_ptr(int32_t* status) {
    static void* cached[64] = {nullptr};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        *status = SS_ERR_CUDA;
        return nullptr;
    }
    if (cached[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_verify_static_scratch) != cudaSuccess || p == nullptr) {
            *status = SS_ERR_CUDA;
            return nullptr;
        }
        cached[dev] = p;
    }
    *status = SS_OK;
    return cached[dev];
}

}  // namespace ss

extern "C" int32_t ss_tree_verify_static(const float* logits, const int32_t* draft_tokens,
                                         const ss_tree_desc* trees, int32_t batch, int32_t max_nodes,
                                         int32_t vocab, int32_t* accept_len, int32_t* accept_path,
                                         int32_t* last_node, int32_t* bonus_token, int32_t* node_argmax,
                                         void* stream) {
    if (!logits || !draft_tokens || !trees || !accept_len || !accept_path || !last_node || !bonus_token)
        return SS_ERR_INVALID_ARG;
    if (batch < 1 || max_nodes < 1 || vocab < 1 || batch > 65535) return SS_ERR_INVALID_ARG;
    if (max_nodes > SS_MAX_NODES) return SS_ERR_UNSUPPORTED;
    if (!ss::aligned16(logits)) return SS_ERR_INVALID_ARG;
    const size_t need = ss_tree_verify_workspace_bytes(batch, max_nodes, vocab);
    if (need == 0 || need > SS_VERIFY_STATIC_SCRATCH_BYTES) return SS_ERR_WORKSPACE;   // beyond the fixed scratch
    int32_t st = SS_OK;
    char* ws = static_cast<char*>(ss::verify_static_scratch_ptr(&st));
    if (ws == nullptr) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the array keeps the previous call's contents: the status word and the arrival counters must
    // start at zero (the rows' arg-maxes are rewritten before they are read)
    const size_t counter_bytes = (static_cast<size_t>(batch) * sizeof(int32_t) + 255) / 256 * 256;
    if (cudaMemsetAsync(ws, 0, ss::kWsHeaderBytes + counter_bytes, s) != cudaSuccess) return SS_ERR_CUDA;
    const cudaError_t err = ss::launch_verify(logits, draft_tokens, trees, batch, max_nodes, vocab, accept_len, accept_path, last_node, bonus_token,
                                              node_argmax, ws, counter_bytes, s, false);
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}
