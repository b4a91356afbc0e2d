// Tree-masked multi-stream attention on register-level MMAs, for layers with few rows or few keys (Eq. 1, Eq. 2; the rule
// is few_rows_block).  Included by ss_attention.cu after its helpers.
//
// What bounds such a layer.  16 rows against 528 keys of 64 dimensions are 4 MB for 32 heads: 0.7 us of HBM, and less of
// any other unit.  The layer is a chain of latencies -- the end of the previous kernel, the query rows, S, softmax and
// P V of a few tiles, the merge -- and a tile on tcgen05 costs four hand-overs between asynchronous units (S issued and
// committed, scores to registers, P to TMEM, P V issued and committed), about 1.2 us of an 8 us layer for each tile that
// is waited for.  With this few rows the register-level MMA (mma.sync, 950 FMA per cycle and SM measured) keeps up, and a
// warp that holds scores, P and O in registers hands nothing over.  Measured, us per plain layer of
// 32 heads, before (tcgen05) and after: 12 rows of 64, 512 keys 7.9 and 4.7; 27 rows of 80, 800 keys 9.1 and 7.4; sixteen
// sequences of 512 keys, 27 rows of 64, 40.8 and 20.9.
//
// A CTA takes half of an SM (113 KB of shared memory): under programmatic dependent launch the CTAs of the next layer
// sit beside those of this one with their first K/V tiles loaded, and what they may not read yet (query rows, this
// step's keys) on its way to L2.
//
// The rows of a head -- its main rows, then its stream rows -- are one block, or blocks of 32 or 64 that go to CTAs of their
// own; a block reads the cached slots and the stream keys of its own nodes.
// Eight warps: warp (team, g) takes rows 16 g .. 16 g + 15 and every (8 / RG)-th tile of 32 keys, RG = 1, 2, 4 groups of
// rows.  Every warp runs an online softmax of its own over its tiles (a reference per row, raised when a score exceeds it
// by more than 2^8; O is in registers, so raising costs a multiplication), so no two warps meet before the end, where
// the partial rows are combined through shared memory.  The warps themselves
// request the tile that takes a slot.
//
// Split heads (C > 1): the CTA's combined rows go to the workspace by bulk copy and each CTA combines its share of them
// as they arrive (publish_partial_rows, merge_partial_rows).  A head is split only when its tiles outweigh that merge.
#pragma once

namespace ss {

constexpr int kFwKeys = 32;                       // keys per tile
constexpr int kFwWarps = 8;
constexpr int kFwThreads = 32 * kFwWarps;
constexpr int kFwMaxRing = 12;
constexpr float kFwRaise = 8.f;                   // raise a reference when a score exceeds it by more than 2^8

template <int HD, int RG>
struct GeoF {
    static constexpr int kHalves = HD > 64 ? 2 : 1;               // 64-element boxes along head_dim
    static constexpr int kBoxBytes = kFwKeys * 128;               // one TMA box: 32 keys x 128 B
    static constexpr int kTileBytes = kHalves * kBoxBytes;        // a K tile or a V tile
    static constexpr int kRows = 16 * RG;
    static constexpr int kQHalf = kRows * 128;
    static constexpr int kQBytes = kHalves * kQHalf;
    static constexpr int kRing = HD > 64 ? 6 : 12;                // tiles in shared memory
    static constexpr int kDynSmem = kQBytes + 2 * kRing * kTileBytes;
    static constexpr int kKSteps = HD / 16;
    static constexpr int kPitch = HD + 4;                         // floats of a partial row: O, m, l, pad
    static constexpr size_t kCtaFloats = static_cast<size_t>(kRows) * kPitch;     // workspace of one CTA of a split block
    // teams of RG warps on different tiles = partials per row (16 rows at head_dim > 64: as many as there are slots)
    static constexpr int kTeams = RG == 1 && HD > 64 ? 6 : kFwWarps / RG;
    // A tile's slot held the tile kRing before it.  Where that was another team's, the team does not know that it has landed,
    // and a parity wait could take the phase before for the one awaited: such a team first waits for the request.
    static constexpr bool kForeign = kRing % kTeams != 0;
    static constexpr bool kQInRegs = HD <= 80;                    // (at 128 the fragments do not fit beside O)
    // The fragments of a step are loaded while the step before is multiplied.  32 rows of 80, 1024 keys 8.83 / 8.65 us; 16 heads 6.43 / 6.30;
    // but 16 rows of 64, 512 keys 4.67 / 4.88, 64 rows of 80, 250 keys 7.26 / 7.38, and at 128 neither way.
    static constexpr bool kAhead = HD == 80 && RG <= 2;
    static_assert(kQBytes % 1024 == 0, "swizzle atoms");
    static_assert(kDynSmem + 1024 <= (228 * 1024) / 2 - 1024, "two CTAs per SM");
    static_assert((kFwWarps * 16 + kRows) * kPitch * 4 <= kDynSmem, "shared memory holds the warps' partial rows and the CTA's");
};

struct CtrlF {
    unsigned long long full[kFwMaxRing];          // K and V of a tile in shared memory
    int done[kFwMaxRing];                         // warps that have read the slot's tile, over all its tiles
    int issued[kFwMaxRing];                       // last tile requested into the slot
    int abort, wait_limit;
};

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// a tile or a line on its way to L2: no data reaches the SM, so it may be asked for before the dependency wait whoever writes it
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ bool mbar_wait_warp_f(uint32_t bar, uint32_t parity, CtrlF* c, int* status) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait_limit_slow(bar, parity, &c->abort, &c->wait_limit, status));
}

// Visible keys x .. x + 31 of a row (Eq. 1 / Eq. 2 with the tree mask of App. A): the prefix and the node's root path, or
// the streams 1 .. stream of its own node.  Nothing past the end of the sequence's keys is ever visible.
__device__ __forceinline__ uint32_t low_bits(int n) { return n >= 32 ? ~0u : n <= 0 ? 0u : (1u << n) - 1u; }
__device__ __forceinline__ uint32_t visible32(bool cache, int x, int L, int gamma, const RowInfo& r, unsigned long long anc) {
    if (!r.valid) return 0u;
    if (cache) {
        const int np = L - x;                             // prefix keys from x on
        if (np > 0) return low_bits(np) | (np < 32 ? static_cast<uint32_t>(anc) << np : 0u);
        return static_cast<uint32_t>(anc >> min(-np, 63));
    }
    const int lo = r.node * gamma - x;
    return low_bits(lo + r.stream) & ~low_bits(lo);
}
// until tile t has been requested into its slot (which the tile before it has left)
__device__ __noinline__ bool wait_requested(CtrlF* c, int slot, int t, int* status) {
    const long long t0 = clock64();
    bool ok = true;
    while (*reinterpret_cast<volatile int*>(&c->issued[slot]) < t) {
        if (*reinterpret_cast<volatile int*>(&c->abort)) { ok = false; break; }
        if (clock64() - t0 > static_cast<long long>(*reinterpret_cast<volatile int*>(&c->wait_limit)) << 10) {
            *reinterpret_cast<volatile int*>(&c->abort) = 1;
            set_status(status, SS_ERR_DEVICE_TIMEOUT);
            ok = false;
            break;
        }
    }
    return __all_sync(0xffffffffu, ok);
}

// The CTA's share of its head's tiles: the cached slots [0, L+T) in tiles of kFwKeys, then the stream keys.
struct SpanF {
    int L, T, n_stream, slo;                      // the block's stream keys begin at slo
    int cache_tiles, j0, n;                       // tiles [j0, j0 + n) of the block
    __device__ __forceinline__ bool is_cache(int t) const { return j0 + t < cache_tiles; }
    __device__ __forceinline__ int first_key(int t) const { return j0 + t < cache_tiles ? (j0 + t) * kFwKeys : slo + (j0 + t - cache_tiles) * kFwKeys; }
    __device__ __forceinline__ int region(int t) const { return is_cache(t) ? L + T : n_stream; }
    __device__ __forceinline__ bool prefix_only(int t) const { return is_cache(t) && first_key(t) + kFwKeys <= L; }
};

// Tiles of a head up to which it is not split (what a split saves on the tiles has to outweigh the merge of the partial
// rows, about 2 us), and tiles per CTA that a split aims at.  Measured on plain layers of 32 heads, us: 12 rows of 64,
// 300 keys whole 4.4, split 5.2; 512 keys 5.0 and 5.8; 800 keys 6.5 and 5.5.  27 rows of 80, 512 keys: 4 tiles per CTA 7.0,
// 8 tiles 8.6.  12 rows of 128, 130 keys 4.3 and 5.9, 500 keys 8.4 and 6.4; 64 rows of 64, 130 keys 6.2 and 6.5, 400 keys 8.9 and 6.8; of
// 128, 100 keys 8.0 and 9.0, 200 keys 10.5 and 9.4.
__host__ __device__ constexpr int few_whole(int head_dim, int rows) {
    return rows == 16 ? (head_dim > 64 ? 8 : 20) : rows == 32 ? 6 : 8;
}
constexpr int kFwSplitTiles = 4;

template <int HD, int RG>
__global__ void __launch_bounds__(kFwThreads, 2) msa_attention_few_rows_kernel(const __grid_constant__ AttnArgs a) {
    using G = GeoF<HD, RG>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(16) CtrlF c;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int C = a.cluster;
    const int blk = static_cast<int>(blockIdx.x);
    const int rank = blk & (C - 1);
    const int pair = blk >> a.cluster_shift;               // (sequence, head); the row block is the grid's second index
    const int row0 = static_cast<int>(blockIdx.y) * G::kRows;
    int b = pair / a.n_heads;
    const int h = pair - b * a.n_heads;
    int* const status = a.status;
    const uint32_t q_base = smem_u32(smem_raw);            // [half][rows][128 B], 1024-byte aligned (checked below)
    const uint32_t ring = q_base + G::kQBytes;             // [slot][K, V][half][32 keys][128 B]

    // ---- prologue (see msa_attention_kernel: the same launch protocol) ------------------------------
    int L = 0, T = 0, cap = 0x7fffffff;
    long long slot0 = 0;
    const bool by_length = a.batch > 1 && a.batch <= 32;
    auto load_scalars = [&]() {
        if (by_length) {                                  // dispatched longest sequence first
            int len = -1;
            if (lane < a.batch) asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(len) : "l"(a.kv_len + lane) : "memory");
            int longer = 0;
            for (int o = 0; o < a.batch; ++o) {
                const int other = __shfl_sync(0xffffffffu, len, o);
                longer += (other > len || (other == len && o < lane)) ? 1 : 0;
            }
            b = __ffs(__ballot_sync(0xffffffffu, lane < a.batch && longer == b)) - 1;
        }
        asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(L) : "l"(a.kv_len + b) : "memory");
        asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(T) : "l"(&a.trees[b].n_nodes) : "memory");
        asm volatile("ld.global.cg.s64 %0, [%1];" : "=l"(slot0) : "l"(a.kv_start + b) : "memory");
        if (a.kv_capacity != nullptr) asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(cap) : "l"(a.kv_capacity + b) : "memory");
    };
    if (a.prefix_stable) load_scalars();
    if (tid < kFwMaxRing) {
        mbar_init(smem_u32(&c.full[tid]), 1);
        c.done[tid] = 0;
        c.issued[tid] = -1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (tid == 32) {
        c.abort = 0;
        c.wait_limit = static_cast<int>(kWaitCycles >> 10);
        tma_prefetch_desc(&a.tm_k); tma_prefetch_desc(&a.tm_v);
        if (a.gamma > 0) { tma_prefetch_desc(&a.tm_ks); tma_prefetch_desc(&a.tm_vs); }
    }
    // One thread waits for the previous kernel of the stream; only then may the next one be scheduled: two layers' CTAs
    // are on the GPU at most, and the slots of the one before are free, so all CTAs of a layer are resident at once.
    auto dependency_wait = [&]() {
        if (tid == 0) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
        __syncthreads();
    };
    if (!a.prefix_stable) {
        dependency_wait();
        load_scalars();
    } else {
        __syncthreads();                                   // the barriers are set up
    }
    const long long main_row0 = static_cast<long long>(b) * a.max_nodes, spec_row0 = main_row0 * a.gamma;
    T = min(max(T, 0), a.max_nodes);
    const bool over = L < 0 || L + T > cap, bad_smem = (q_base & 1023u) != 0u;       // (the latter never expected)
    const bool skip = over || bad_smem || T == 0;          // nothing read or written; the same in all CTAs of the head
    SpanF sp;
    sp.L = L; sp.T = T; sp.n_stream = T * a.gamma;
    // stream rows [r0, r1) of the block, numbered from the first stream row; they see stream keys from their first node's on
    const int r0 = max(row0 - a.tmax8, 0), r1 = min(row0 + G::kRows - a.tmax8, sp.n_stream);
    sp.slo = r1 > r0 ? ((r0 * a.gamma_magic) >> 16) * a.gamma : 0;
    const int own_streams = r1 > r0 ? r1 - sp.slo : 0;
    const bool any_row = row0 < T || r1 > r0;              // (a block without a row reads and writes nothing)
    sp.cache_tiles = (L + T + kFwKeys - 1) / kFwKeys;
    const int all_tiles = skip || !any_row ? 0 : sp.cache_tiles + (own_streams + kFwKeys - 1) / kFwKeys;
    // the CTAs that get tiles; the first ones take the odd tiles, so that the last has the masked ones
    int shift = 0;
    if (all_tiles > few_whole(HD, G::kRows))
        while (shift < a.cluster_shift && (all_tiles >> shift) > kFwSplitTiles) ++shift;
    const int ce = 1 << shift;
    // The others leave at once: the next layer's CTAs can have their place.  (CTA 0 of a head always waits for the previous
    // kernel, so this kernel never ends before that one.)
    if (rank > 0 && (rank >= ce || all_tiles == 0)) return;
    sp.j0 = (all_tiles * rank + ce - 1) >> shift;
    sp.n = ((all_tiles * (rank + 1) + ce - 1) >> shift) - sp.j0;

    // Requests tile t into slot st: a whole warp, each of 2 kHalves lanes one box (a box costs its thread 100 cycles)
    auto load_tile = [&](int t, int st) {
        const int x = sp.first_key(t);
        const bool cache = sp.is_cache(t);
        const uint32_t bar = smem_u32(&c.full[st]);
        if (lane == 0) {
            *reinterpret_cast<volatile int*>(&c.issued[st]) = t;
            mbar_expect_tx(bar, 2 * G::kTileBytes);
        }
        __syncwarp();
        if (lane < 2 * G::kHalves) {
            const int is_v = lane & 1, hh = lane >> 1;
            const CUtensorMap* const map = cache ? (is_v ? &a.tm_v : &a.tm_k) : (is_v ? &a.tm_vs : &a.tm_ks);
            tma_load_3d(ring + static_cast<uint32_t>(2 * st + is_v) * G::kTileBytes + static_cast<uint32_t>(hh) * G::kBoxBytes, map, hh * 64,
                        cache ? h * a.head_coord : h, static_cast<int>(cache ? slot0 + x : spec_row0 + x), bar);
        }
    };
    // 16-byte piece i of the query rows: row i / (HD / 8); rows that no node owns have none
    constexpr int kPieces = HD / 8;
    auto q_piece = [&](int i) -> const __nv_bfloat16* {
        const int lrow = i / kPieces, at = (i - lrow * kPieces) * 8, row = row0 + lrow;
        if (row < a.tmax8) return row < T ? a.q_main + ((main_row0 + row) * a.n_heads + h) * HD + at : nullptr;
        const int x = row - a.tmax8;
        return x < sp.n_stream ? a.q_spec + ((spec_row0 + x) * a.n_heads + h) * HD + at : nullptr;
    };
    // The first tiles need no hand-back (warp w requests tiles w and w + 8); before the dependency wait only those that
    // lie wholly inside the cached prefix.
    const int n_early = min(sp.n, G::kRing);
    if (a.prefix_stable) {
        for (int t = warp; t < n_early; t += kFwWarps) {
            if (sp.prefix_only(t)) {
                load_tile(t, t);
            } else if (lane < 2 * G::kHalves) {
                // what has to wait for the previous kernel comes to L2 meanwhile: this step's keys, and the query rows
                const bool cache = sp.is_cache(t);
                tma_prefetch_3d(cache ? ((lane & 1) ? &a.tm_v : &a.tm_k) : ((lane & 1) ? &a.tm_vs : &a.tm_ks), (lane >> 1) * 64,
                                cache ? h * a.head_coord : h, static_cast<int>((cache ? slot0 : spec_row0) + sp.first_key(t)));
            }
        }
        if (sp.n > 0) {
            for (int i = 8 * tid; i < G::kRows * kPieces; i += 8 * kFwThreads) {       // a line is 8 pieces
                const __nv_bfloat16* const p = q_piece(i);
                if (p != nullptr) prefetch_l2(p);
            }
        }
    }
    // a warp's rows and keys; everything that the promise covers is read before the wait
    const int rg = warp % RG, team = warp / RG, quad = lane & 3;
    RowInfo ri[2];
    unsigned long long anc[2] = {0ull, 0ull};
    #pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int row = row0 + 16 * rg + (lane >> 2) + 8 * e;
        ri[e].stream = 0;
        if (row < a.tmax8) {
            ri[e].valid = row < T; ri[e].node = row;
        } else {
            const int x = row - a.tmax8;
            ri[e].valid = x < sp.n_stream;
            ri[e].node = (x * a.gamma_magic) >> 16;
            ri[e].stream = x - ri[e].node * a.gamma + 1;
        }
        ri[e].valid = ri[e].valid && !skip;
        if (ri[e].valid && sp.n > 0) anc[e] = __ldcg(&a.trees[b].anc_mask[ri[e].node]);
    }
    if (a.prefix_stable) dependency_wait();
    if (sp.n > 0) {
        constexpr int kEach = (G::kRows * kPieces + kFwThreads - 1) / kFwThreads;
        uint4 q[kEach];
        // the caller may shorten the bound of the waits of a head of at most 64 rows (workspace word 1, units of 1024 cycles); asked for
        // with the query rows: behind them it would be a second round trip to L2 in every CTA's way
        int lim = 0;
        if (tid == 0) asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(lim) : "l"(a.status + 1) : "memory");
        #pragma unroll
        for (int k = 0; k < kEach; ++k) {
            const int i = tid + k * kFwThreads;
            const __nv_bfloat16* const p = i < G::kRows * kPieces ? q_piece(i) : nullptr;
            q[k] = make_uint4(0u, 0u, 0u, 0u);
            if (p != nullptr) q[k] = __ldcg(reinterpret_cast<const uint4*>(p));
        }
        for (int t = warp; t < n_early; t += kFwWarps)
            if (!a.prefix_stable || !sp.prefix_only(t)) load_tile(t, t);
        #pragma unroll
        for (int k = 0; k < kEach; ++k) {
            const int i = tid + k * kFwThreads;
            const int row = i / kPieces, pc = i - row * kPieces;
            if (a.scale_log2 < 0.f) { q[k].x ^= 0x80008000u; q[k].y ^= 0x80008000u; q[k].z ^= 0x80008000u; q[k].w ^= 0x80008000u; }   // |scale| below
            if (i < G::kRows * kPieces)
                st_shared_v4(q_base + (pc >> 3) * G::kQHalf + row * 128u + (static_cast<uint32_t>((pc ^ row) & 7) << 4), q[k].x, q[k].y, q[k].z, q[k].w);
        }
        if (tid == 0 && lim > 0 && gridDim.y * G::kRows <= 64) *reinterpret_cast<volatile int*>(&c.wait_limit) = lim;
    }
    if (tid == 0 && (over || bad_smem)) set_status(status, bad_smem ? SS_ERR_CUDA : SS_ERR_CAPACITY);
    __syncthreads();                                       // the query rows are in shared memory

    float m_ref[2] = {-INFINITY, -INFINITY}, l_part[2] = {0.f, 0.f};
    float o[HD / 8][4];
    #pragma unroll
    for (int i = 0; i < HD / 8; ++i) { o[i][0] = 0.f; o[i][1] = 0.f; o[i][2] = 0.f; o[i][3] = 0.f; }
    {
        const bool warp_active = __any_sync(0xffffffffu, ri[0].valid || ri[1].valid);
        // Matrix i / 8 of a four-matrix load: its row i % 8 (+ 8) and its 16-byte chunk (+ 1).  Offsets of the four chunk
        // pairs of a 128-byte row, the row included: K has its rows in the upper matrices, Q and V in the odd ones.
        const int mrow = lane & 7, odd = (lane >> 3) & 1, upper = lane >> 4;
        uint32_t off_k[4], off_v[4];
        #pragma unroll
        for (int j = 0; j < 4; ++j) {
            off_k[j] = static_cast<uint32_t>(mrow + 8 * upper) * 128u + (static_cast<uint32_t>((2 * j + odd) ^ mrow) << 4);
            off_v[j] = static_cast<uint32_t>(mrow + 8 * odd) * 128u + (static_cast<uint32_t>((2 * j + upper) ^ mrow) << 4);
        }
        const float scale = fabsf(a.scale_log2);
        const unsigned long long scale2 = pack_f32x2(scale, scale);
        auto load_q = [&](int ks, uint32_t (&f)[4]) { ldsm_x4(q_base + static_cast<uint32_t>(rg * 16 * 128) + off_v[ks & 3] + (ks >> 2) * G::kQHalf, f); };
        uint32_t qf[G::kQInRegs ? G::kKSteps : 1][4];
        if (G::kQInRegs && sp.n > 0) {
            #pragma unroll
            for (int ks = 0; ks < G::kKSteps; ++ks) load_q(ks, qf[G::kQInRegs ? ks : 0]);
        }
        int slot = team % G::kRing, round = team / G::kRing;
        #pragma unroll 1
        for (int t = team < G::kTeams ? team : sp.n; t < sp.n; t += G::kTeams) {
            if (G::kForeign && round > 0 && *reinterpret_cast<volatile int*>(&c.issued[slot]) < t && !wait_requested(&c, slot, t, status)) break;
            __syncwarp();
            if (!mbar_wait_warp_f(smem_u32(&c.full[slot]), static_cast<uint32_t>(round & 1), &c, status)) break;
            const uint32_t kt = ring + static_cast<uint32_t>(2 * slot) * G::kTileBytes, vt = kt + G::kTileBytes;
            const int x0 = sp.first_key(t);
            const bool cache = sp.is_cache(t);
            const bool masked = !cache || x0 + kFwKeys > L;
            if (warp_active) {
                // S: 16 rows x 32 keys, four chains of accumulation
                float s[4][4];
                #pragma unroll
                for (int n = 0; n < 4; ++n) { s[n][0] = 0.f; s[n][1] = 0.f; s[n][2] = 0.f; s[n][3] = 0.f; }
                uint32_t ka[4];
                #pragma unroll
                for (int j = 0; j < 4; ++j) ka[j] = kt + off_k[j];
                if constexpr (G::kAhead) {
                    uint32_t kf[2][2][4];
                    ldsm_x4(ka[0], kf[0][0]);
                    ldsm_x4(ka[0] + 16 * 128, kf[0][1]);
                    #pragma unroll
                    for (int ks = 0; ks < G::kKSteps; ++ks) {
                        if (ks + 1 < G::kKSteps) {
                            ldsm_x4(ka[(ks + 1) & 3] + ((ks + 1) >> 2) * G::kBoxBytes, kf[(ks + 1) & 1][0]);
                            ldsm_x4(ka[(ks + 1) & 3] + ((ks + 1) >> 2) * G::kBoxBytes + 16 * 128, kf[(ks + 1) & 1][1]);
                        }
                        const uint32_t (&f)[2][4] = kf[ks & 1];
                        mma_bf16(s[0], qf[ks], f[0][0], f[0][1]);
                        mma_bf16(s[1], qf[ks], f[0][2], f[0][3]);
                        mma_bf16(s[2], qf[ks], f[1][0], f[1][1]);
                        mma_bf16(s[3], qf[ks], f[1][2], f[1][3]);
                    }
                } else {
                    #pragma unroll
                    for (int ks = 0; ks < G::kKSteps; ++ks) {
                        uint32_t kf[2][4];
                        ldsm_x4(ka[ks & 3] + (ks >> 2) * G::kBoxBytes, kf[0]);
                        ldsm_x4(ka[ks & 3] + (ks >> 2) * G::kBoxBytes + 16 * 128, kf[1]);
                        if constexpr (!G::kQInRegs) load_q(ks, qf[0]);
                        const uint32_t (&qk)[4] = qf[G::kQInRegs ? ks : 0];
                        mma_bf16(s[0], qk, kf[0][0], kf[0][1]);
                        mma_bf16(s[1], qk, kf[0][2], kf[0][3]);
                        mma_bf16(s[2], qk, kf[1][0], kf[1][1]);
                        mma_bf16(s[3], qk, kf[1][2], kf[1][3]);
                    }
                }
                // s[n][2 e + i]: row e, key 8 n + 2 quad + i
                if (masked) {
                    const int nvk = sp.region(t) - x0;                            // valid keys (may exceed the tile)
                    const uint32_t vis0 = visible32(cache, x0, L, a.gamma, ri[0], anc[0]) >> (2 * quad), vis1 = visible32(cache, x0, L, a.gamma, ri[1], anc[1]) >> (2 * quad);
                    #pragma unroll
                    for (int n = 0; n < 4; ++n)
                        #pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            s[n][i] = ((vis0 >> (8 * n + i)) & 1u) ? s[n][i] : -INFINITY;
                            s[n][2 + i] = ((vis1 >> (8 * n + i)) & 1u) ? s[n][2 + i] : -INFINITY;
                        }
                    // V rows past the end of the sequence's keys may hold anything (even NaN patterns): the weight is 0 there,
                    // but 0 * NaN is NaN, so they are cleared (by every warp that reads them: all write the same)
                    if (nvk < kFwKeys) {
                        for (int i = lane; i < (kFwKeys - nvk) * 8 * G::kHalves; i += 32)
                            st_shared_v4(vt + static_cast<uint32_t>((i & 7) * 16) + static_cast<uint32_t>(nvk + (i >> 3) / G::kHalves) * 128u
                                         + static_cast<uint32_t>((i >> 3) % G::kHalves) * G::kBoxBytes, 0u, 0u, 0u, 0u);
                        __syncwarp();
                    }
                }
                float mx[2];
                #pragma unroll
                for (int e = 0; e < 2; ++e)
                    mx[e] = fmaxf(fmaxf(fmaxf(s[0][2 * e], s[0][2 * e + 1]), fmaxf(s[1][2 * e], s[1][2 * e + 1])),
                                  fmaxf(fmaxf(s[2][2 * e], s[2][2 * e + 1]), fmaxf(s[3][2 * e], s[3][2 * e + 1]))) * scale;
                // (a row that no node owns has zero queries and asks once at most)
                if (__any_sync(0xffffffffu, mx[0] > m_ref[0] + kFwRaise || mx[1] > m_ref[1] + kFwRaise)) {
                    float corr[2];
                    #pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], 1));
                        mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], 2));
                        const float m_new = fmaxf(m_ref[e], mx[e]);
                        corr[e] = m_new == m_ref[e] ? 1.f : exp2f(m_ref[e] - m_new);      // 0 when nothing was visible so far
                        m_ref[e] = m_new;
                        l_part[e] *= corr[e];
                    }
                    if (t != team) {                                              // (nothing accumulated before the first tile)
                        #pragma unroll
                        for (int i = 0; i < HD / 8; ++i) { o[i][0] *= corr[0]; o[i][1] *= corr[0]; o[i][2] *= corr[1]; o[i][3] *= corr[1]; }
                    }
                }
                // P as the A operand of P V: for keys 16 j ..: (row e, keys 16 j + 8 n + 2 quad ..) in word 2 n + e
                uint32_t pf[2][4];
                #pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float m = m_ref[e] == -INFINITY ? 0.f : m_ref[e];       // (no key seen so far: every weight is exp2(-inf) = 0)
                    const unsigned long long shift2 = pack_f32x2(-m, -m);
                    unsigned long long sum2 = pack_f32x2(0.f, 0.f);
                    #pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        float t0, t1;
                        unpack_f32x2(fma_f32x2(pack_f32x2(s[n][2 * e], s[n][2 * e + 1]), scale2, shift2), t0, t1);
                        const float e0 = exp2f(t0), e1 = exp2f(t1);
                        sum2 = add_f32x2(sum2, pack_f32x2(e0, e1));
                        pf[n >> 1][2 * (n & 1) + e] = pack_bf16(e0, e1);
                    }
                    float s0, s1;
                    unpack_f32x2(sum2, s0, s1);
                    l_part[e] += s0 + s1;
                }
                uint32_t va[4];
                #pragma unroll
                for (int j = 0; j < 4; ++j) va[j] = vt + off_v[j];
                if constexpr (G::kAhead) {
                    uint32_t vf[2][4];
                    ldsm_x4_t(va[0], vf[0]);
                    #pragma unroll
                    for (int i = 0; i < HD / 8; ++i) {                            // keys 16 j .., dimensions 16 d ..
                        const int j = i / (HD / 16), d = i % (HD / 16), jn = (i + 1) / (HD / 16), dn = (i + 1) % (HD / 16);
                        if (i + 1 < HD / 8) ldsm_x4_t(va[dn & 3] + 16 * 128 * jn + (dn >> 2) * G::kBoxBytes, vf[(i + 1) & 1]);
                        mma_bf16(o[2 * d], pf[j], vf[i & 1][0], vf[i & 1][1]);
                        mma_bf16(o[2 * d + 1], pf[j], vf[i & 1][2], vf[i & 1][3]);
                    }
                } else {
                    #pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        #pragma unroll
                        for (int d = 0; d < HD / 16; ++d) {
                            uint32_t vf[4];
                            ldsm_x4_t(va[d & 3] + 16 * 128 * j + (d >> 2) * G::kBoxBytes, vf);
                            mma_bf16(o[2 * d], pf[j], vf[0], vf[1]);
                            mma_bf16(o[2 * d + 1], pf[j], vf[2], vf[3]);
                        }
                    }
                }
            }
            // the last of the team's warps to have read the tile requests the one that takes its slot
            __syncwarp();
            if (t + G::kRing < sp.n) {
                int prev = 0;
                if (RG > 1) {
                    if (lane == 0) asm volatile("atom.acq_rel.cta.shared::cta.add.s32 %0, [%1], 1;" : "=r"(prev) : "r"(smem_u32(&c.done[slot])) : "memory");
                    prev = __shfl_sync(0xffffffffu, prev, 0);
                }
                if (RG == 1 || (prev & (RG - 1)) == RG - 1) load_tile(t + G::kRing, slot);
            }
            slot += G::kTeams;
            if (slot >= G::kRing) { slot -= G::kRing; ++round; }
        }
        #pragma unroll
        for (int e = 0; e < 2; ++e) {
            l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], 1);
            l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], 2);
        }
    }
    __syncthreads();  // every tile that was requested has been read: shared memory is free
    const bool aborted = *reinterpret_cast<volatile int*>(&c.abort) != 0;
    if (aborted && tid < kFwMaxRing && c.issued[tid] >= 0)     // a wait ran out: copies still in flight land first
        mbar_drain(smem_u32(&c.full[tid]), static_cast<uint32_t>((c.issued[tid] / G::kRing) & 1));

    // ======================================== epilogue ==========================================
    // The warps leave their partial rows (O, m, l) in shared memory; item i of the combination is four columns of the
    // i / (HD / 4)-th row.
    constexpr uint32_t RB = G::kPitch * 4;                                    // bytes of a partial row
    const uint32_t w_base = q_base, y_base = q_base + kFwWarps * 16 * RB;        // [8 warps][16 rows][pitch], then the CTA's rows
    const bool split = ce > 1;
    const bool live = sp.n > 0 && !aborted;                                   // CTA-uniform
    if (live && team < G::kTeams) {
        #pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (!ri[e].valid) continue;
            const uint32_t at = w_base + static_cast<uint32_t>(16 * warp + (lane >> 2) + 8 * e) * RB;
            #pragma unroll
            for (int i = 0; i < HD / 8; ++i) st_shared_v2(at + static_cast<uint32_t>(8 * i + 2 * quad) * 4u, __float_as_uint(o[i][2 * e]), __float_as_uint(o[i][2 * e + 1]));
            if (quad == 0) st_shared_v2(at + HD * 4u, __float_as_uint(m_ref[e]), __float_as_uint(l_part[e]));
        }
    }
    __syncthreads();
    if (!live) return;
    constexpr int kItems = HD / 4;
    // the block's rows that nodes own: main rows [row0, row0 + n_main), then stream rows [r0, r1)
    const int n_main = max(min(T - row0, G::kRows), 0), n_rows = n_main + max(r1 - r0, 0);
    // (one copy of the code for all of a thread's items, which runs once a layer: with the items of a thread unrolled, their loads in flight
    // together, layers take up to 0.25 us longer)
    #pragma unroll 1
    for (int i = tid; i < n_rows * kItems; i += kFwThreads) {
        const int rr = i / kItems, g4 = i - rr * kItems;
        RowInfo r;
        r.valid = true; r.node = row0 + rr; r.stream = 0;
        int row = rr;                                                         // in the block
        if (rr >= n_main) {
            const int xr = r0 + rr - n_main;
            r.node = (xr * a.gamma_magic) >> 16;
            r.stream = xr - r.node * a.gamma + 1;
            row = a.tmax8 + xr - row0;
        }
        // its row group's warp of every team holds the row: everything is asked for at once
        const uint32_t at = w_base + static_cast<uint32_t>(row) * RB;
        float2 ml[G::kTeams];
        float4 v[G::kTeams];
        #pragma unroll
        for (int p = 0; p < G::kTeams; ++p) {
            ml[p] = ld_shared_v2(at + static_cast<uint32_t>(G::kRows * p) * RB + HD * 4u);
            v[p] = ld_shared_v4(at + static_cast<uint32_t>(G::kRows * p) * RB + static_cast<uint32_t>(g4) * 16u);
        }
        float m = -INFINITY, l = 0.f;
        #pragma unroll
        for (int p = 0; p < G::kTeams; ++p) m = fmaxf(m, ml[p].x);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        #pragma unroll
        for (int p = 0; p < G::kTeams; ++p) {
            const float w = ml[p].x == -INFINITY ? 0.f : exp2f(ml[p].x - m);        // 0: saw no visible key
            l += w * ml[p].y;
            acc.x += w * v[p].x; acc.y += w * v[p].y; acc.z += w * v[p].z; acc.w += w * v[p].w;
        }
        if (!split) {
            const OutPtr dst = out_ptr<HD>(a, b, h, spec_row0, r);
            const float inv = 1.f / l;
            uint2 w;
            w.x = pack_bf16(acc.x * inv, acc.y * inv);
            w.y = pack_bf16(acc.z * inv, acc.w * inv);
            *reinterpret_cast<uint2*>(dst.o + g4 * 4) = w;
            if (dst.lse && g4 == 0) *dst.lse = (m + log2f(l)) * 0.6931471805599453f;
        } else {
            // (never +0: a word of a partial row that reads zero in the workspace has not arrived)
            const uint32_t y = y_base + static_cast<uint32_t>(row) * RB;
            st_shared_v4(y + static_cast<uint32_t>(g4) * 16u, never_plus_zero(__float_as_uint(acc.x)), never_plus_zero(__float_as_uint(acc.y)),
                         never_plus_zero(__float_as_uint(acc.z)), never_plus_zero(__float_as_uint(acc.w)));
            if (g4 == 0) st_shared_v4(y + HD * 4u, never_plus_zero(__float_as_uint(m)), never_plus_zero(__float_as_uint(l)), 0u, 0u);
        }
    }
    if (!split) return;
    fence_async_smem();                                                       // the copy engine reads these rows
    __syncthreads();
    Span rows;
    rows.T = T; rows.gamma = a.gamma; rows.tmax8 = a.tmax8; rows.n_stream = sp.n_stream; rows.spec_end = a.tmax8 + sp.n_stream;
    float* const part_group = a.partials + (static_cast<size_t>(blockIdx.y) * (gridDim.x >> a.cluster_shift) + pair) * C * G::kCtaFloats;
    const int share = G::kRows >> shift, first = rank * share;
    if (tid == 0) publish_partial_rows<HD>(rows, row0, G::kRows, y_base, part_group + static_cast<size_t>(rank) * G::kCtaFloats, first, share);
    // the other CTAs of the head were launched with this one and need nothing from it: the (bounded) wait is short
    const long long limit = static_cast<long long>(*reinterpret_cast<volatile int*>(&c.wait_limit)) << 10;
    if (!merge_partial_rows<HD>(a, rows, row0, b, h, spec_row0, ce, rank, y_base, part_group, G::kCtaFloats, first, share, tid, kFwThreads, limit, &c.abort)) {
        c.abort = 1;
        set_status(status, SS_ERR_DEVICE_TIMEOUT);
    }
    if (tid == 0) bulk_copies_read();
}

}  // namespace ss
