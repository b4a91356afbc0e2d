// Tree-masked multi-stream attention on tcgen05 for grids of more than one CTA per SM (Eq. 1, Eq. 2): batches, whose heads
// (64 query rows) or blocks of 128 rows (heads with more) need no split of their keys.  Included by ss_attention.cu after
// its helpers.
//
// What bounds such a layer: HBM for the keys (16 sequences x 32 heads of 256 to 4096 keys x 128: 88 us), and beside it what a CTA
// does one thing after another -- the end of the previous kernel, the query rows, and for each tile S, softmax, P V.  With
// one CTA per SM all of that is in the open.  So a CTA takes half of an SM (113 KB of shared memory, 256 TMEM columns, 320
// threads): one's chain passes under the other's tiles, and under programmatic dependent launch the first CTAs of the next
// layer wait with the first tiles of their prefix loaded.  Measured, us per
// layer, one CTA per SM (the kernels of the smaller grids) / this one: 64 rows, 16 sequences x 32 heads of 256 to 4096 keys x 128
// 112 / 97 (alone, 6.5 TB/s would be 88), of 2304 keys x 64 80 / 70, x 80 95 / 78; 320 rows, of 256 to 4096 keys x 128 322 / 288;
// 192 rows, of 1024 keys x 64 124 / 92.  With its MMAs in blocks of four (tc_mma_steps), of 512 to 4096 keys x 128 64 rows 102.8 -> 96.7, 320
// rows 288 -> 265.
//
//   S = Q K^T     A = the query rows, B = a K tile of 64 keys, both K-major in shared memory, N = 64
//   O += P V      A = P in TMEM, B = the V tile (MN-major), N = head_dim
//
// M = 64: rows 16 w .. 16 w + 15 of S, P and O lie in TMEM lanes 32 w .. 32 w + 15, so warp w of a team reads its rows
// whole with 16-lane loads (tcgen05.ld.16x256b: a thread gets two rows, 8 apart, and two of every eight columns), and P goes
// back by tcgen05.st.16x128b.  M = 128: a thread has a row.  Two teams of four warps take alternate tiles, each with a score
// buffer of its own; P goes over the scores it came from.  One warp issues all MMAs: S of tile t + 2 right behind P V of
// tile t, which reads the same buffer -- MMAs of a thread execute in the order of their issue -- so no barrier lies between them.
//
// Softmax with one reference per row: the maximum over the CTA's first tile, which team 0 leaves for team 1.  Any reference
// not absurdly far from the row's maximum gives the same result after normalisation, so nobody ever rescales the
// accumulator.  (The first tile shows every row a key: it holds prefix keys or the root.)  If a later tile's exponentials
// leave the range (a thread's sum to more than 2^60), the CTA lets everything in flight land, takes the exact maxima in a
// pass over its K tiles, and runs its tiles again against those.
#pragma once

namespace ss {

constexpr int kHfKeys = 64;                       // keys per tile
constexpr int kHfSoftmax = 256;                   // two teams of four warps
constexpr int kHfThreads = kHfSoftmax + 64;       // and the producer's and the MMA issuer's warps
constexpr int kHfMaxRing = 6;
constexpr float kHfLimit = 1152921504606846976.f; // 2^60

struct CtrlH {
    unsigned long long q_full, o_done;             // query rows in shared memory; the CTA's last P V complete
    unsigned long long k_full[kHfMaxRing], k_empty[kHfMaxRing], v_full[kHfMaxRing], v_empty[kHfMaxRing];
    unsigned long long s_full[2], p_full[2];       // score buffer: S complete / P written (4 warps)
    unsigned long long m_full[4];                  // the first tile's references of 16 rows
    unsigned long long drain;                      // start over: the issuer's last MMAs complete
    uint32_t row_ref[128];                         // the rows' references; start over: their exact maxima, as order keys
    uint32_t tmem_base;
    int wait_limit;                                // bound of every wait, in units of 1024 cycles
    int n_drains;                                  // completed phases of the drain barrier
    int abort;                                     // 1: a wait ran out of time; 2: a reference did not hold, start over
};

template <int HD, int M>
struct GeoH {
    static constexpr int kHalves = HD > 64 ? 2 : 1;               // 64-element boxes along head_dim
    static constexpr int kBoxBytes = kHfKeys * 128;               // one TMA box: 64 keys x 128 B
    static constexpr int kSlotBytes = kHalves * kBoxBytes;        // a K tile or a V tile
    static constexpr int kQHalfBytes = M * 128;
    static constexpr int kQBytes = kHalves * kQHalfBytes;         // the query rows
    // tiles in the K ring and in the V ring (a K slot is held until S is complete, a V slot until P V is)
    static constexpr int kRingK = HD > 64 ? (M == 64 ? 3 : 2) : 6, kRingV = HD > 64 ? 3 : 6;
    static constexpr int kDynSmem = kQBytes + (kRingK + kRingV) * kSlotBytes;
    static constexpr int kKSteps = HD / 16;
    static constexpr int kRows = M == 64 ? 2 : 1;                 // rows of a softmax thread
    static constexpr int kSplitCol = HD == 80 ? 48 : HD / 2;      // team 0 finishes columns [0, kSplitCol), team 1 the rest
    static constexpr uint32_t kTmemCols = 256;                    // O (128), two score buffers (64 each)
    static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(M >> 4) << 24);
    static constexpr uint32_t kIdescS = kIdesc | (static_cast<uint32_t>(kHfKeys >> 3) << 17);
    static constexpr uint32_t kIdescPV = kIdesc | (1u << 16) | (static_cast<uint32_t>(HD >> 3) << 17);
    static_assert(kDynSmem + static_cast<int>(sizeof(CtrlH)) <= (228 * 1024) / 2 - 1024, "two CTAs per SM");
    static_assert(kRingK <= kHfMaxRing && kRingV <= kHfMaxRing, "barriers");
};


// TMEM, 64 columns of 16 lanes: r[4 k + 2 e + i] of thread (4 r + q) is column 8 k + 2 q + i of lane r + 8 e
__device__ __forceinline__ void tmem_ld_rows64(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : SS_R16(r, 0), SS_R16(r, 16) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_rows16(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
// 32 columns of 16 lanes: r[2 k + e] is column 4 k + q of lane r + 8 e -- the 64 weights of a row as bf16 pairs
__device__ __forceinline__ void tmem_st_p64(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.16x128b.x8.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};"
                 ::SS_W16(r, 0), "r"(taddr) : "memory");
}
// order keys: unsigned integers in the order of the floats
__device__ __forceinline__ uint32_t max_key(float x) {
    const uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float max_of_key(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k ^ 0x80000000u) : ~k);
}
constexpr uint32_t kNoMax = 0x007fffffu;          // the key of -inf

// The CTA's tiles: the cached slots [0, L+T) in tiles of 64, then the stream keys [slo, shi) that its rows can see.
struct SpanH {
    int L, T, slo, shi;
    int cache_tiles, n;
    __device__ __forceinline__ bool is_cache(int t) const { return t < cache_tiles; }
    __device__ __forceinline__ int first_key(int t) const { return t < cache_tiles ? t * kHfKeys : slo + (t - cache_tiles) * kHfKeys; }
    __device__ __forceinline__ int end(int t) const { return t < cache_tiles ? L + T : shi; }
    __device__ __forceinline__ bool prefix_only(int t) const { return t < cache_tiles && (t + 1) * kHfKeys <= L; }
};

template <int HD, int M>
__global__ void __launch_bounds__(kHfThreads, 2) msa_attention_half_kernel(const __grid_constant__ AttnArgs a) {
    using G = GeoH<HD, M>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(16) CtrlH c;

    const int tid = threadIdx.x, warp = static_cast<int>(uniform(tid >> 5)), lane = tid & 31;
    const int rb = M == 64 ? 0 : static_cast<int>(blockIdx.x) % a.n_blocks;              // row block of the head
    const int pair = M == 64 ? static_cast<int>(blockIdx.x) : static_cast<int>(blockIdx.x) / a.n_blocks;
    int b = pair / a.n_heads;
    const int h = pair - b * a.n_heads;
    int* const status = a.status;
    const uint32_t q_base = smem_u32(smem_raw);            // [half][M rows][128 B], 1024-byte aligned (checked below)
    const uint32_t k_base = q_base + G::kQBytes, v_base = k_base + G::kRingK * G::kSlotBytes;   // [slot][half][64 keys][128 B]
    const bool is_softmax = warp < 8, producer = tid == kHfSoftmax;

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
    auto init_rings = [&]() {
        for (int s = 0; s < G::kRingK; ++s) { mbar_init(smem_u32(&c.k_full[s]), 1); mbar_init(smem_u32(&c.k_empty[s]), 1); }
        for (int s = 0; s < G::kRingV; ++s) { mbar_init(smem_u32(&c.v_full[s]), 1); mbar_init(smem_u32(&c.v_empty[s]), 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    };
    auto init_tiles = [&]() {
        for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&c.s_full[s]), 1); mbar_init(smem_u32(&c.p_full[s]), 4); }
        mbar_init(smem_u32(&c.o_done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    };
    if (producer) {
        mbar_init(smem_u32(&c.q_full), 1);
        init_rings();
        tma_prefetch_desc(&a.tm_k); tma_prefetch_desc(&a.tm_v); tma_prefetch_desc(&a.tm_qm);
        if (a.gamma > 0) { tma_prefetch_desc(M == 128 && rb > 0 ? &a.tm_qs1 : &a.tm_qs); tma_prefetch_desc(&a.tm_ks); tma_prefetch_desc(&a.tm_vs); }
    } else if (tid == 0) {
        c.abort = c.n_drains = 0;
        c.wait_limit = static_cast<int>(kWaitCycles >> 10);
        for (int s = 0; s < 4; ++s) mbar_init(smem_u32(&c.m_full[s]), 1);
        mbar_init(smem_u32(&c.drain), 1);
        init_tiles();
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c.tmem_base)), "r"(G::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // One thread waits for the previous kernel of the stream; only then may the next one be scheduled: two layers' CTAs
    // are on the GPU at most, and the slots of the one before are free, so all CTAs of a layer are resident at once.
    auto dependency_wait = [&]() {
        if (producer) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };
    if (!a.prefix_stable) {
        dependency_wait();
        load_scalars();
    }
    L = static_cast<int>(uniform(L));                       // (for the compiler: what follows from them is the same in all lanes)
    T = static_cast<int>(uniform(T));
    const long long spec_row0 = static_cast<long long>(b) * a.max_nodes * a.gamma;
    T = min(max(T, 0), a.max_nodes);
    const bool over = L < 0 || L + T > cap, bad_smem = (q_base & 1023u) != 0u;       // (the latter never expected)
    const bool skip = over || bad_smem || T == 0;          // nothing read or written; the same in all CTAs of the head
    const int n_stream = T * a.gamma, row0 = rb * M;
    SpanH sp;
    sp.L = L; sp.T = T;
    {
        // stream rows [x0, x1) of the block; row x = (node, stream) sees the stream keys node * gamma .. x
        const int x0 = max(row0, a.tmax8) - a.tmax8, x1 = min(row0 + M - a.tmax8, n_stream);
        const bool any = !skip && (row0 < T || x1 > x0);  // a block without a row reads nothing
        sp.slo = x1 > x0 ? x0 / a.gamma * a.gamma : 0;
        sp.shi = x1 > x0 ? x1 : 0;
        sp.cache_tiles = any ? (L + T + kHfKeys - 1) / kHfKeys : 0;
        sp.n = any ? sp.cache_tiles + (sp.shi - sp.slo + kHfKeys - 1) / kHfKeys : 0;
    }

    auto load_tile = [&](bool is_v, int t, int st) {
        const uint32_t bar = smem_u32(is_v ? &c.v_full[st] : &c.k_full[st]);
        mbar_expect_tx(bar, G::kSlotBytes);
        const uint32_t dst = (is_v ? v_base : k_base) + st * G::kSlotBytes;
        const int x = sp.first_key(t);
        #pragma unroll
        for (int hh = 0; hh < G::kHalves; ++hh) {
            if (sp.is_cache(t)) tma_load_3d(dst + hh * G::kBoxBytes, is_v ? &a.tm_v : &a.tm_k, hh * 64, h * a.head_coord, static_cast<int>(slot0 + x), bar);
            else tma_load_3d(dst + hh * G::kBoxBytes, is_v ? &a.tm_vs : &a.tm_ks, hh * 64, h, static_cast<int>(spec_row0 + x), bar);
        }
    };
    const bool with_spec = a.gamma > 0 && a.s0rows > 0;
    // the first tiles need no hand-back; before the dependency wait only those that lie wholly inside the cached prefix
    const int early_k = min(sp.n, G::kRingK), early_v = min(sp.n, G::kRingV);
    int n_pre = 0;
    if (a.prefix_stable) {
        if (producer) {
            for (; n_pre < early_v && sp.prefix_only(n_pre); ++n_pre) {
                if (n_pre < early_k) load_tile(false, n_pre, n_pre);
                load_tile(true, n_pre, n_pre);
            }
            // the query rows come to L2 meanwhile: nothing reaches the SM, whoever writes them
            if (sp.n > 0) {
                #pragma unroll
                for (int hh = 0; hh < G::kHalves; ++hh) {
                    if (rb > 0) tma_prefetch_3d(&a.tm_qs1, hh * 64, h, static_cast<int>(spec_row0 + row0 - a.tmax8));
                    else tma_prefetch_3d(&a.tm_qm, hh * 64, h, b * a.max_nodes);
                    if (rb == 0 && with_spec) tma_prefetch_3d(&a.tm_qs, hh * 64, h, static_cast<int>(spec_row0));
                }
            }
        }
        dependency_wait();
    }
    if (producer && (over || bad_smem)) set_status(status, bad_smem ? SS_ERR_CUDA : SS_ERR_CAPACITY);
    if (producer && sp.n > 0) {
        const uint32_t qbar = smem_u32(&c.q_full);
        mbar_expect_tx(qbar, G::kHalves * static_cast<uint32_t>(rb > 0 ? M : a.tmax8 + (with_spec ? a.s0rows : 0)) * 128u);
        #pragma unroll
        for (int hh = 0; hh < G::kHalves; ++hh) {
            const uint32_t dst = q_base + hh * G::kQHalfBytes;
            if (rb > 0) tma_load_3d(dst, &a.tm_qs1, hh * 64, h, static_cast<int>(spec_row0 + row0 - a.tmax8), qbar);
            else tma_load_3d(dst, &a.tm_qm, hh * 64, h, b * a.max_nodes, qbar);
            if (rb == 0 && with_spec) tma_load_3d(dst + a.tmax8 * 128u, &a.tm_qs, hh * 64, h, static_cast<int>(spec_row0), qbar);
        }
        for (int t = n_pre; t < early_v; ++t) {
            if (t < early_k) load_tile(false, t, t);
            load_tile(true, t, t);
        }
        if (M == 64) {
            // the caller may shorten the bound of the waits of a head of at most 64 rows (workspace word 1, units of 1024 cycles)
            int lim;
            asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(lim) : "l"(a.status + 1) : "memory");
            if (lim > 0) *reinterpret_cast<volatile int*>(&c.wait_limit) = lim;
        }
    }
    int n_k = early_k, n_v = early_v;                      // tiles requested so far (producer)
    // (producer) waits until every copy requested so far has landed
    auto land = [&]() {
        for (int s = 0; s < G::kRingK; ++s) if (n_k > s) mbar_drain(smem_u32(&c.k_full[s]), ((n_k - 1 - s) / G::kRingK) & 1);
        for (int s = 0; s < G::kRingV; ++s) if (n_v > s) mbar_drain(smem_u32(&c.v_full[s]), ((n_v - 1 - s) / G::kRingV) & 1);
    };
    const uint32_t tmem_o = c.tmem_base, tmem_s = tmem_o + 128;
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;

    // softmax threads.  M = 64: rows 16 (warp & 3) + lane / 4 (e = 0) and 8 further (1); of a tile keys 8 k + 2 quad + {0, 1}.
    // M = 128: row 32 (warp & 3) + lane.
    const int team = warp >> 2, quad = lane & 3, row_a = M == 64 ? 16 * (warp & 3) + (lane >> 2) : 32 * (warp & 3) + lane;
    RowInfo ri[G::kRows];
    unsigned long long anc[G::kRows];
    const float scale = a.scale_log2;                      // (a hidden score is -inf after scaling, whatever the sign)
    const uint32_t hidden = scale < 0.f ? 0x7f800000u : 0xff800000u;
    // reference; sums of the weights as rounded to bf16, and before
    float m_ref[G::kRows], l_part[G::kRows], l_exact[G::kRows];
    #pragma unroll
    for (int e = 0; e < G::kRows; ++e) { m_ref[e] = -INFINITY; l_part[e] = l_exact[e] = 0.f; anc[e] = 0ull; ri[e].valid = false; }
    bool warp_active = false, exact = false;               // exact: m_ref is the maximum over all of the CTA's keys
    if (is_softmax) {
        #pragma unroll
        for (int e = 0; e < G::kRows; ++e) {
            const int row = row0 + row_a + 8 * e;
            ri[e].stream = 0;
            if (row < a.tmax8) {
                ri[e].valid = row < T; ri[e].node = row;
            } else {
                const int x = row - a.tmax8;
                ri[e].valid = x < n_stream;
                ri[e].node = M == 64 ? (x * a.gamma_magic) >> 16 : a.gamma > 0 ? x / a.gamma : 0;
                ri[e].stream = x - ri[e].node * a.gamma + 1;
            }
            ri[e].valid = ri[e].valid && sp.n > 0;
            if (ri[e].valid) anc[e] = __ldcg(&a.trees[b].anc_mask[ri[e].node]);
            warp_active = warp_active || ri[e].valid;
        }
        warp_active = __any_sync(0xffffffffu, warp_active);
    }

    // The tile loops of all roles.  MAX: the pass that takes the rows' maxima only (no P, no V).
    auto run_tiles = [&](auto mode_tag, const int first_k, const int first_v) {
    constexpr bool kMax = decltype(mode_tag)::value;
    // (the outer branches are the same for all lanes of a warp, or the issuer's operands would not stay in uniform registers)
    if (warp == 8) {
        if (producer) {
            // K runs one tile ahead of V: a K slot comes back with S of its tile, a V slot only with P V
            auto request = [&](bool is_v, int& t) {
                if (t >= sp.n) return true;
                const int ring = is_v ? G::kRingV : G::kRingK, st = t % ring;
                if (t >= ring && !mbar_wait_limit(smem_u32(is_v ? &c.v_empty[st] : &c.k_empty[st]), (t / ring - 1) & 1, &c, status)) return false;
                load_tile(is_v, t, st);
                ++t;
                return true;
            };
            n_k = first_k;
            n_v = kMax ? sp.n : first_v;
            bool ok = request(false, n_k);
            while (ok && (n_k < sp.n || n_v < sp.n)) ok = request(false, n_k) && request(true, n_v);
            if (kMax) n_v = 0;
        }
    } else if (warp == 9) {
        bool ok = sp.n == 0 || mbar_wait_uniform(smem_u32(&c.q_full), 0, &c, status);
        if (!ok && lane == 0) mbar_drain(smem_u32(&c.q_full), 0);
        const uint64_t dq = desc_k_major(uniform(q_base));
        const uint32_t ut_o = uniform(tmem_o), ut_s = uniform(tmem_s);
        Ring rk, rv;
        rk.start(); rv.start();
        int ts = 0;                                       // next tile of S
        auto issue_s = [&]() {
            if (!mbar_wait_uniform(smem_u32(&c.k_full[rk.slot]), rk.round & 1, &c, status)) return false;
            tc_fence_after();
            const uint64_t dk = desc_k_major(uniform(k_base + rk.slot * G::kSlotBytes));
            const uint32_t sd = uniform(ut_s + (ts & 1) * kHfKeys);
            tc_mma_steps<4>(sd, dq, dk, G::kIdescS, 0u);
            if constexpr (G::kHalves == 2) tc_mma_steps<G::kKSteps - 4>(sd, dq + (G::kQHalfBytes >> 4), dk + (G::kBoxBytes >> 4), G::kIdescS, 1u);
            tc_commit_e(smem_u32(&c.s_full[ts & 1]));
            tc_commit_e(smem_u32(&c.k_empty[rk.slot]));
            rk.advance(G::kRingK);
            ++ts;
            return true;
        };
        if (ok && sp.n > 0) ok = issue_s();
        if (ok && sp.n > 1) ok = issue_s();
        for (int t = 0; ok && t < sp.n; ++t, rv.advance(G::kRingV)) {
            const int buf = t & 1;
            if (!kMax && !mbar_wait_uniform(smem_u32(&c.v_full[rv.slot]), rv.round & 1, &c, status)) break;
            if (!mbar_wait_uniform(smem_u32(&c.p_full[buf]), (t >> 1) & 1, &c, status)) break;
            tc_fence_after();
            if (!kMax) {
                const uint64_t dv = desc_mn_major(uniform(v_base + rv.slot * G::kSlotBytes), G::kBoxBytes);
                const uint32_t pa = uniform(ut_s + buf * kHfKeys);
                tc_mma_ts_steps(ut_o, pa, dv, G::kIdescPV, t > 0 ? 1u : 0u);
                tc_commit_e(smem_u32(&c.v_empty[rv.slot]));
                if (t == sp.n - 1) tc_commit_e(smem_u32(&c.o_done));
            }
            if (ts < sp.n && !issue_s()) break;           // S of tile t + 2 over the buffer that P V of tile t reads before it
        }
    } else {
        bool ok = true;
        if (!kMax && !exact && team == 1 && sp.n > 1) {
            ok = mbar_wait_limit_warp(smem_u32(&c.m_full[warp & 3]), 0, &c, status);
            #pragma unroll
            for (int e = 0; e < G::kRows; ++e) m_ref[e] = __uint_as_float(c.row_ref[row_a + 8 * e]);
        }
        #pragma unroll 1
        for (int t = team; ok && t < sp.n; t += 2) {
            if (!mbar_wait_limit_warp(smem_u32(&c.s_full[team]), (t >> 1) & 1, &c, status)) break;
            tc_fence_after();
            const int x0 = sp.first_key(t);
            const bool cache = sp.is_cache(t);
            const int nvk = min(kHfKeys, sp.end(t) - x0);
            const bool masked = !cache || x0 + kHfKeys > L;
            const uint32_t s_addr = tmem_s + lane_base + static_cast<uint32_t>(team * kHfKeys);
            // 32 scores at a time: M = 64 the thread's share of both its rows, M = 128 half of its row's 64
            constexpr int kPieces = M == 64 ? 1 : 2;
            uint32_t sr[32];
            auto load_scores = [&](int piece) {
                if constexpr (M == 64) tmem_ld_rows64(s_addr, sr);
                else tmem_ld32<0>(s_addr + 32u * piece, sr);
                tmem_wait_ld();
                if (masked) {
                    #pragma unroll
                    for (int e = 0; e < G::kRows; ++e) {
                        const unsigned long long vis = visible_mask(cache, x0, nvk, L, a.gamma, ri[e], anc[e]) >> (M == 64 ? 2 * quad : 32 * piece);
                        const uint32_t lo = static_cast<uint32_t>(vis);
                        if constexpr (M == 64) {
                            const uint32_t hi = static_cast<uint32_t>(vis >> 32);
                            #pragma unroll
                            for (int k = 0; k < 8; ++k)
                                #pragma unroll
                                for (int i = 0; i < 2; ++i)
                                    if (!(((k < 4 ? lo : hi) >> (8 * (k & 3) + i)) & 1u)) sr[4 * k + 2 * e + i] = hidden;
                        } else {
                            #pragma unroll
                            for (int i = 0; i < 32; ++i)
                                if (!((lo >> i) & 1u)) sr[i] = hidden;
                        }
                    }
                }
            };
            // score i of row e in the piece
            auto at = [](int e, int i) { return M == 64 ? 4 * (i >> 1) + 2 * e + (i & 1) : i; };
            constexpr int kPerRow = M == 64 ? 16 : 32;
            bool bad = false;
            if (warp_active) {
                if (kMax || (t == 0 && !exact)) {
                    #pragma unroll
                    for (int piece = kPieces - 1; piece >= 0; --piece) {
                        load_scores(piece);
                        #pragma unroll
                        for (int e = 0; e < G::kRows; ++e) {
                            float mx = -INFINITY;
                            #pragma unroll
                            for (int i = 0; i < kPerRow; i += 2) mx = fmaxf(mx, fmaxf(__uint_as_float(sr[at(e, i)]) * scale, __uint_as_float(sr[at(e, i + 1)]) * scale));
                            if constexpr (M == 64) {
                                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                            }
                            m_ref[e] = fmaxf(m_ref[e], mx);
                        }
                    }
                    if (!kMax) {
                        #pragma unroll
                        for (int e = 0; e < G::kRows; ++e) {
                            if (M == 128 || quad == 0) c.row_ref[row_a + 8 * e] = __float_as_uint(m_ref[e]);
                            // (a row without a key, an infinite score or a NaN: the exact maxima decide)
                            bad = bad || (ri[e].valid && !(m_ref[e] > -INFINITY && m_ref[e] < INFINITY));
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&c.m_full[warp & 3]));
                    }
                }
                if (!kMax) {
                    // P = exp2(S - m) as bf16, over the first half of the score columns.  Normalised by the sum of the rounded
                    // weights, so that their rounding cancels where one key dominates.
                    const unsigned long long scale2 = pack_f32x2(scale, scale);
                    #pragma unroll
                    for (int piece = 0; piece < kPieces; ++piece) {
                        if (M == 128 || t != 0 || exact) load_scores(piece);
                        uint32_t pk[16];
                        #pragma unroll
                        for (int e = 0; e < G::kRows; ++e) {
                            const float m = m_ref[e] > -INFINITY ? m_ref[e] : 0.f;
                            const unsigned long long shift2 = pack_f32x2(-m, -m);
                            unsigned long long sum2 = pack_f32x2(0.f, 0.f), exact2 = pack_f32x2(0.f, 0.f);
                            #pragma unroll
                            for (int i = 0; i < kPerRow; i += 2) {
                                float t0, t1;
                                unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sr[at(e, i)]), __uint_as_float(sr[at(e, i + 1)])), scale2, shift2), t0, t1);
                                const float e0 = exp2f(t0), e1 = exp2f(t1);
                                const uint32_t w = pack_bf16(e0, e1);
                                pk[M == 64 ? i + e : i >> 1] = w;
                                sum2 = add_f32x2(sum2, pack_f32x2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)));
                                exact2 = add_f32x2(exact2, pack_f32x2(e0, e1));
                            }
                            float s0, s1, y0, y1;
                            unpack_f32x2(sum2, s0, s1);
                            unpack_f32x2(exact2, y0, y1);
                            l_part[e] += s0 + s1;
                            l_exact[e] += y0 + y1;
                            bad = bad || (ri[e].valid && !(s0 + s1 <= kHfLimit));
                        }
                        if constexpr (M == 64) tmem_st_p64(s_addr, pk);
                        else tmem_st16<0>(s_addr + 16u * piece, pk);
                    }
                }
            } else if (!kMax && t == 0 && !exact) {
                if (lane == 0) mbar_arrive(smem_u32(&c.m_full[warp & 3]));
            }
            if (!kMax && !exact && __any_sync(0xffffffffu, bad)) {
                if (lane == 0) atomicCAS(&c.abort, 0, 2);             // every role leaves its loop and the CTA starts over
                break;
            }
            // V rows past the end of the sequence's keys may hold anything (even NaN patterns): P is 0 there, but 0 * NaN
            // is NaN, so they are cleared before P V reads them
            if (!kMax && nvk < kHfKeys) {
                const int vs = t % G::kRingV;
                if (!mbar_wait_limit_warp(smem_u32(&c.v_full[vs]), static_cast<uint32_t>((t / G::kRingV) & 1), &c, status)) break;
                constexpr int kRowPieces = G::kHalves * 8;            // 16-byte pieces of a V row
                for (int i = tid & 127; i < (kHfKeys - nvk) * kRowPieces; i += 128) {
                    const int vr = nvk + i / kRowPieces, pc = i % kRowPieces;
                    st_shared_v4(v_base + vs * G::kSlotBytes + (pc >> 3) * G::kBoxBytes + vr * 128u + (pc & 7) * 16u, 0u, 0u, 0u, 0u);
                }
                fence_async_smem();
            }
            if (warp_active) tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&c.p_full[team]));
        }
        // the last P V must be complete before the accumulator is read; products complete in issue order
        if (!kMax && sp.n > 0 && *reinterpret_cast<volatile int*>(&c.abort) == 0) {
            mbar_wait_limit_warp(smem_u32(&c.o_done), 0, &c, status);
            tc_fence_after();
        }
    }
    __syncwarp();     // the single-lane roles rejoin their warps
    };   // run_tiles

    run_tiles(std::false_type{}, early_k, early_v);
    if (__syncthreads_or(*reinterpret_cast<volatile int*>(&c.abort) == 2)) {
        // A reference did not hold.  Twice: what is in flight lands, the barriers are set up anew, the tiles run again --
        // first for the exact maxima, then against them.
        #pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (producer) {
                land();
                mbar_drain(smem_u32(&c.q_full), 0);
            } else if (warp == 9) {
                tc_commit_e(smem_u32(&c.drain));
                mbar_drain(smem_u32(&c.drain), static_cast<uint32_t>(pass));
            }
            __syncwarp();
            if (is_softmax) { tmem_wait_ld(); tmem_wait_st(); }
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (tid == 0) {
                for (int s = 0; s < G::kRingK; ++s) { mbar_inval(smem_u32(&c.k_full[s])); mbar_inval(smem_u32(&c.k_empty[s])); }
                for (int s = 0; s < G::kRingV; ++s) { mbar_inval(smem_u32(&c.v_full[s])); mbar_inval(smem_u32(&c.v_empty[s])); }
                for (int i = 0; i < 2; ++i) { mbar_inval(smem_u32(&c.s_full[i])); mbar_inval(smem_u32(&c.p_full[i])); }
                mbar_inval(smem_u32(&c.o_done));
                init_rings();
                init_tiles();
                c.abort = 0;
                c.n_drains = pass + 1;
                if (pass == 0) atomicAdd(a.status + 2, 1);            // diagnostics: blocks that started over
            }
            if (pass == 0 && tid < 128) c.row_ref[tid] = kNoMax;
            __syncthreads();
            if (pass == 0) {
                #pragma unroll
                for (int e = 0; e < G::kRows; ++e) { m_ref[e] = -INFINITY; l_part[e] = l_exact[e] = 0.f; }
                run_tiles(std::true_type{}, 0, 0);
                if (is_softmax && (M == 128 || quad == 0))
                    for (int e = 0; e < G::kRows; ++e) atomicMax(&c.row_ref[row_a + 8 * e], max_key(m_ref[e]));
                __syncthreads();
                if (is_softmax)
                    for (int e = 0; e < G::kRows; ++e) m_ref[e] = max_of_key(c.row_ref[row_a + 8 * e]);
                exact = true;
                if (*reinterpret_cast<volatile int*>(&c.abort) != 0) break;      // (a wait ran out)
            } else {
                run_tiles(std::false_type{}, 0, 0);
            }
        }
    }

    // ======================================== epilogue ==========================================
    // The rings are idle: every copy has landed and every MMA is complete.  The two threads that hold the same rows, one per
    // team, exchange their sums; then each finishes its team's columns of the rows.
    const bool aborted = __syncthreads_or(*reinterpret_cast<volatile int*>(&c.abort) != 0);
    if (aborted) {
        // A wait ran out.  Shared memory and TMEM are not given up before what is in flight has landed: copies (the producer may
        // have requested its last one long before another role gave up), MMAs with their commits, the softmax threads' stores.
        if (producer) {
            land();
            mbar_drain(smem_u32(&c.q_full), 0);
        } else if (warp == 9) {
            tc_commit_e(smem_u32(&c.drain));
            mbar_drain(smem_u32(&c.drain), static_cast<uint32_t>(*reinterpret_cast<volatile int*>(&c.n_drains) & 1));
        }
        __syncwarp();
        if (is_softmax) { tmem_wait_ld(); tmem_wait_st(); }
    }
    if (is_softmax && sp.n > 0 && !aborted) {
        const uint32_t x_base = k_base;                                       // [team][M rows] sums
        #pragma unroll
        for (int e = 0; e < G::kRows; ++e) {
            if constexpr (M == 64) {
                #pragma unroll
                for (int o = 1; o <= 2; o <<= 1) {
                    l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], o);
                    l_exact[e] += __shfl_xor_sync(0xffffffffu, l_exact[e], o);
                }
            }
            if (M == 128 || quad == 0) st_shared_v2(x_base + static_cast<uint32_t>(team * M + row_a + 8 * e) * 8u, __float_as_uint(l_part[e]), __float_as_uint(l_exact[e]));
        }
        named_barrier(1, kHfSoftmax);
        OutPtr dst[G::kRows];
        float inv[G::kRows];
        #pragma unroll
        for (int e = 0; e < G::kRows; ++e) {
            const float2 o = ld_shared_v2(x_base + static_cast<uint32_t>((team ^ 1) * M + row_a + 8 * e) * 8u);
            l_exact[e] += o.y;
            inv[e] = 1.f / (l_part[e] + o.x);
            dst[e] = out_ptr<HD>(a, b, h, spec_row0, ri[e]);
        }
        if (warp_active) {
            const int c_lo = team == 0 ? 0 : G::kSplitCol, c_hi = team == 0 ? G::kSplitCol : HD;
            #pragma unroll 1
            for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
                if constexpr (M == 64) {
                    uint32_t orr[8];
                    tmem_ld_rows16(tmem_o + lane_base + static_cast<uint32_t>(c0), orr);
                    tmem_wait_ld();
                    #pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        if (!ri[e].valid) continue;
                        #pragma unroll
                        for (int k = 0; k < 2; ++k)
                            *reinterpret_cast<uint32_t*>(dst[e].o + c0 + 8 * k + 2 * quad) =
                                pack_bf16(__uint_as_float(orr[4 * k + 2 * e]) * inv[e], __uint_as_float(orr[4 * k + 2 * e + 1]) * inv[e]);
                    }
                } else {
                    uint32_t orr[16];
                    tmem_ld16<0>(tmem_o + lane_base + static_cast<uint32_t>(c0), orr);
                    tmem_wait_ld();
                    float v[16];
                    #pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(orr[i]) * inv[0];
                    if (ri[0].valid) store_bf16x16(dst[0].o + c0, v);
                }
            }
            #pragma unroll
            for (int e = 0; e < G::kRows; ++e)
                if (ri[e].valid && (M == 128 || quad == 0) && team == 0 && dst[e].lse) *dst[e].lse = (m_ref[e] + log2f(l_exact[e])) * 0.6931471805599453f;
        }
    }
    tc_fence_before();
    __syncthreads();                                                          // TMEM is no longer read
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_o), "r"(G::kTmemCols) : "memory");
    }
}

}  // namespace ss
