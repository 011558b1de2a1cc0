// Multi-query decode attention over a paged bf16 KV cache on the tcgen05 tensor cores: each request contributes a
// short chunk of query rows (the pending token plus its k drafts) that attend to the cached prefix and, causally,
// to each other.  The keys of a request are cut into up to 16 splits ("split-K"), one CTA each; a CTA leaves an
// un-normalised partial output with its reference maximum and sum in global memory (a few MB that stay in L2),
// takes a ticket, and the last CTA of a (request, KV head, row group) to arrive merges the splits in split order
// and writes the result straight into the output projection's input format, so that a CTA that is not the last one
// leaves its SM to the next kernel at once.  Where all CTAs of a launch fit the device together and a group has many rows,
// the others stay for a moment and take a share of the rows; what they do not take the last one merges, so that no CTA's
// result depends on another one being on the device.
//
// One CTA = one KV head of one request x one key split x up to 112 query rows, where the rows are all (query head
// of the group, chunk row) pairs that share the KV head (GQA).  The keys are on the M side of the MMAs, the (few)
// query rows on the narrow N side:
//   S^T[128 keys x N rows] = K_tile[128 x hd] . Q^T[hd x N]          A = K rows from the cache, B = Q
//   O^T[hd x N rows]      += V_tile^T[hd x 128 keys] . P^T[128 x N]   A = V rows from the cache, B = P
//   L  [  * x N rows]      += 1[* x 128 keys] . P^T[128 x N]          the softmax denominators, by the same P
// with S^T (twice: two tiles in flight), O^T and L in tensor memory.  The cache stores, per page and
// head, the rows in 8-row groups of 8-element pieces ([slot/8][hd/8][slot%8][8]), which IS the operand order of
// both products (K-major for the first, MN-major for the second): a page lands in shared memory by one bulk copy
// and is read by the tensor cores as it is.  Q and P are fp32 values split into bf16 hi + lo terms (see
// attn_wide_q); K and V are the cache's bf16.
// Warps 0-7: one thread per key of a tile (= tensor-memory lane; warps w and w+4 share a lane quarter and take
// alternate 8-row column blocks): masking, exponentials relative to the score of the split's first key (any reference will
// do that keeps p in range; a row's maximum is only looked for when a score exceeds its reference by 2^40 and O^T has to
// be rescaled), P written back as the next MMA's B operand.  Warp 8: bulk copies of the K/V pages (a ring of three or four
// slots, K0 V0 K1 V1 ...; tiles of keys that were cached before this pass do not depend on the preceding QKV projection and
// are requested before the dependent-launch wait) and the MMA issue (one thread).  Every wait is bounded and raises the
// device error word, but for the shared merge's, which needs nobody to give up.
#pragma once
#include "common.cuh"
#include "layers.cuh"
#include "tcgen05.cuh"

namespace pipesd {

constexpr int kAttnWorkers = 256;           // threads of warps 0-7
constexpr int kAttnThreads = kAttnWorkers + 32;
constexpr int kAttnTile = 128;              // keys per tile = M of the MMAs
constexpr int kAttnMaxRows = 112;           // query rows per CTA (N of the MMAs; what fits beside the ring); more rows: more row groups
constexpr int kAttnMaxSplits = 16;          // key splits of one request
constexpr int kAttnMaxSlots = 4;            // tile slots of the K/V ring
constexpr int kAttnBigCols = kAttnMaxRows / 16;   // 8-row column blocks per worker warp of the large variant (the small one: 1, 16 rows)
constexpr int kAttnShortTail = 112;         // keys of the second tile up to which the third ring slot is cut down
constexpr int kAttnMergePolls = 128;        // looks a CTA takes at the ticket before it leaves its share of a merge to the last one
                                            // (0.3-0.5 us each; splits of one length end within a few us of each other)
constexpr float kAttnMaxExcess = 40.f;      // log2 units by which a score may exceed its row's reference: P, O^T and the
                                            // denominators stay below 2^60 and, next to a p of at least 1, lose nothing below

// Wait for a barrier phase.  Bounded by a try count (each try suspends for a hardware-chosen time; 2^22 of them take
// seconds), so that a protocol error cannot hang the GPU: the caller raises the error word and carries on.
__device__ __forceinline__ bool attn_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t it = 0; it < (1u << 22); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// The same for a whole warp: every lane waits, and the warp agrees on the outcome (the collective tensor-memory
// instructions that follow need a warp-uniform control flow).
__device__ __forceinline__ bool attn_wait_warp(uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, attn_wait(bar, parity));
}

__device__ __forceinline__ float fast_exp2(float x) {   // 2^x, relative error 2^-22; 2^-inf = 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One barrier of the worker warps that also tells whether any of their threads said yes.
__device__ __forceinline__ bool attn_workers_any(bool mine) {
    uint32_t any;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.aligned.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
        : "=r"(any)
        : "r"((uint32_t)mine), "n"(kAttnWorkers)
        : "memory");
    return any != 0;
}

// Shared-memory plan of one CTA with N query rows (a multiple of 16).  K and V tiles travel through a ring of three or four
// slots (attn_ring_bytes) in the order K0 V0 K1 V1 ...; a cut-down third one, where no CTA of the launch has more than two
// tiles and the second at most kAttnShortTail keys, still takes such a CTA's K/V in full before the first product starts.
template <int HD>
struct AttnSmem {
    static constexpr int kTileBytes = kAttnTile * HD * 2;            // one K or V tile
    static constexpr int kOnes = 256;                                 // 16 keys x 8 ones: the denominators' A operand
    __host__ __device__ static constexpr int q_bytes(int N) { return N * HD * 2; }          // hi or lo
    __host__ __device__ static constexpr int p_bytes(int N) { return kAttnTile * N * 2; }   // hi or lo
    __host__ __device__ static constexpr int small_bytes(int N) { return 8 * N * 4 + 128; } // warp maxima [4][N], horizon, reference
                                                                                            // maximum, factor, sums [N] each; barriers
    __host__ __device__ static constexpr size_t bytes(int N, int ring) {
        return (size_t)kOnes + ring + 2 * q_bytes(N) + 2 * p_bytes(N) + small_bytes(N);
    }
};

// An MMA of up to about 48 rows costs the same as one of 16 (fetch of the 128-row A operand, issue), so the hi and lo terms of
// Q, and of P, stand side by side as one operand of 2N rows -- half the MMAs, and the two halves of the result are added
// where it is read -- as long as the wider accumulators fit tensor memory: 8N columns up to 64 rows; up to 80 rows for P
// only, 6N; else the terms take turns, 4N.  (Batch of 16 at the 7b shape: 24 MMAs of 42 cycles per tile instead of 48.)
__host__ __device__ constexpr bool attn_wide_q(int N) { return N <= 64; }
__host__ __device__ constexpr bool attn_wide_p(int N) { return N <= 80; }
// Tensor-memory columns of a CTA with N query rows: S^T twice, O^T and L, as a power of two >= 32.
__host__ __device__ constexpr int attn_tmem_cols(int N) {
    int c = 32;
    while (c < 2 * N * (attn_wide_q(N) ? 2 : 1) + 2 * N * (attn_wide_p(N) ? 2 : 1)) c *= 2;
    return c;
}
// The ring: three slots of a tile (the third cut down where no split of the launch has more than two tiles, the second a
// short one), or four where that costs no resident CTA.  With three, the next K tile is only requested when the present
// V tile has been read, and its 3 us are waited for once per tile (8b shape, 17 rows: 3.9 us per tile).
static inline int attn_ring_bytes(int hd, int slots, bool short_tail) {
    const int tile = kAttnTile * hd * 2;
    return slots == 4 ? 4 * tile : 2 * tile + (short_tail ? kAttnShortTail * hd * 2 : tile);
}
static inline size_t attn_smem_bytes_raw(int hd, int N, int ring) {
    return hd == 128 ? AttnSmem<128>::bytes(N, ring) : AttnSmem<64>::bytes(N, ring);
}
constexpr int kAttnSmemMax = 227 * 1024;
static inline int attn_ring_slots(int hd, int N) {
    const size_t three = attn_smem_bytes_raw(hd, N, attn_ring_bytes(hd, 3, false)), four = attn_smem_bytes_raw(hd, N, attn_ring_bytes(hd, 4, false));
    const int cap = N > 16 ? 1 : 2;                              // CTAs per SM by registers
    auto per_sm = [&](size_t b) { const int n = (int)((size_t)(228 * 1024) / (b + 1024)); return n > cap ? cap : n; };
    return four <= (size_t)kAttnSmemMax && per_sm(four) >= per_sm(three) ? 4 : 3;
}
// Dynamic shared memory to ask for: the plan above, padded so that the CTAs an SM can hold never want more than the
// SM's 512 tensor-memory columns together (the allocation instruction blocks until its columns are free).
static inline size_t attn_smem_bytes(int hd, int N, bool short_tail) {
    const size_t need = attn_smem_bytes_raw(hd, N, attn_ring_bytes(hd, attn_ring_slots(hd, N), short_tail));
    const int max_ctas = 512 / attn_tmem_cols(N);
    const size_t floor_ = (size_t)kAttnSmemMax / (max_ctas + 1) + 1;
    return need > floor_ ? need : floor_;
}
static inline int attn_rows_n(int rows_per_kv_head) {    // N of a CTA that holds this many query rows
    const int r = rows_per_kv_head > kAttnMaxRows ? kAttnMaxRows : rows_per_kv_head;
    return (r + 15) / 16 * 16;
}

// Host: how one request's keys are split.  `units` = CTA groups that compete for the device per layer, counted in
// groups of this request's length: for a request verified alone its KV heads x row groups; in a batch the batch's
// (keys x groups) total divided by this request's keys.  slots[0 | 1] = CTAs of this kernel the device keeps resident
// at once for the request's row count with the whole | cut-down third ring slot.  As many splits as let all CTAs of the
// pass run in one wave (at most 16, at most one per 128 keys), then the fewest splits that leave each CTA the same
// number of 128-key tiles.  The plan fixes the order a row's keys are summed in: a function of the pass's composition
// and the device, the same every time that composition is verified.
struct AttnSplit { int splits, keys_per_split, short_tail; };
static inline AttnSplit attn_split_plan(int total_keys, int page_size, int units, const int* slots, int max_splits = kAttnMaxSplits) {
    auto chunk_of = [&](int s) {
        const int ch = (total_keys + s - 1) / s;
        return (ch + page_size - 1) / page_size * page_size;
    };
    auto tiles_of = [&](int s) { return (chunk_of(s) + kAttnTile - 1) / kAttnTile; };
    const int by_keys = (total_keys + kAttnTile - 1) / kAttnTile;
    AttnSplit p = {1, chunk_of(1), 0};
    for (int cls = 1; cls >= 0; --cls) {
        int s = slots[cls] / (units > 0 ? units : 1);
        s = s > max_splits ? max_splits : s;
        s = s > by_keys ? by_keys : s;
        s = s < 1 ? 1 : s;
        const int t = tiles_of(s);
        while (s > 1 && tiles_of(s - 1) == t) --s;
        p.splits = s;
        p.keys_per_split = chunk_of(s);
        p.short_tail = cls;
        if (cls == 0 || p.keys_per_split <= kAttnTile + kAttnShortTail) break;
    }
    return p;
}

// Per-CTA constants of the tile copies.
struct AttnCtx {
    const uint16_t* kbase;     // K block of page 0 for this layer and KV head
    const int32_t* bt;         // page ids of the request
    size_t page_stride;        // elements between consecutive pages of a layer
    size_t v_off;              // elements from a K block to the V block of the same page and head
    int page_size;
    int k0, k1;
};

// Issue (one warp) the copies of the K rows (kv = 0) or V rows (kv = 1) of one 128-key tile: the rows of a page that
// belong to one KV head are contiguous in the pool, already in operand order, so every page the tile touches is one
// bulk copy (lane l takes the l-th page), counted in bytes on the barrier.  Whole 8-row groups are copied: the rows
// of the last group at or beyond k1 are masked (K) or cleared (V) by the consumers.
// Inlined at its places: as a function of its own it made the kernel smaller and every pass slower (7b shape, 9 rows 3228 ->
// 3215 us, 17 rows 3916 -> 3883; 8b shape, 17 rows 5085 -> 5005; 7b shape, 2 rows and 1000 keys 2853 -> 2843).
template <int HD>
__device__ __forceinline__ void attn_issue_tile(const uint16_t* src0, const int32_t* bt, size_t page_stride, int page_size, int k1, uint32_t dst,
                                             uint32_t bar, int j0) {
    const int lane = threadIdx.x & 31;
    const int j1 = (min(j0 + kAttnTile, k1) + 7) & ~7;
    if (lane == 0) mbar_expect_tx(bar, (uint32_t)(j1 - j0) * (HD * 2));
    __syncwarp();
    const int pidx = j0 / page_size + lane;                                // page of the request
    const int js = max(j0, pidx * page_size), je = min(j1, (pidx + 1) * page_size);
    if (js < je) {
        const uint16_t* src = src0 + (size_t)bt[pidx] * page_stride + (size_t)(js - pidx * page_size) * HD;
        bulk_g2s(dst + (uint32_t)(js - j0) * (HD * 2), src, (uint32_t)(je - js) * (HD * 2), bar);
    }
}

struct AttnArgs {
    const float* q;            // [M][Hq*hd] rotated queries
    PassMeta meta;
    const uint16_t* kv_pool;
    int layer, n_pages, page_size, M, Hq, Hkv;
    int rows_cap;              // query rows per row group (kAttnMaxRows, or 16 for a batch whose requests have up to 32)
    int n_max;                 // N the launch's shared memory was sized for
    int ring, slots;           // bytes and slots of the K/V ring
    int share_merge;           // all CTAs of the launch fit the device together: the CTAs of a group merge its rows together
    int merge_polls;           // kAttnMergePolls, or the harness's limit
    int row_groups;
    float* o_part;             // partial results: [slot][hd], slot = it_part0 + ((kv head * R + row) * splits + split)
    float* m_part;             // [slot]
    float* l_part;             // [slot]
    int* tickets;              // [item][kv head][row group], zero between launches
    uint16_t* xf_out;          // the output projection's input: split-bf16 fragments, or (xd_tbs > 0) an xd array
    int xd_tbs;
    // Weights of the projections that follow (nullable): while this kernel runs, HBM carries little besides the K/V
    // it reads.  Once a CTA's own K/V tiles have all landed, its copy warp asks the L2 for this CTA's share of the
    // first pf_len[i] bytes at pf_ptr[i] (128-byte lines dealt over the whole grid).  Purely a hint.
    const unsigned char* pf_ptr[2];
    size_t pf_len[2];
    int* err;
};

// grid (max splits of the launch, n_kv_heads * row_groups, n_items), block 288.  CU = 1: launches of up to 16 query rows per
// CTA; the register bound is what lets two CTAs share an SM (a CTA's nine warps put three on one of the SM's four register
// partitions, 16K registers each, and two such triples must fit it).  CU = kAttnBigCols: more rows, one CTA per SM, and
// a worker's share of a tile's P, up to 56 values, stays in registers until the previous product is through.
template <int HD, int CU>
__global__ void __launch_bounds__(kAttnThreads, CU == 1 ? 3 : 1) attn_kernel(const AttnArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    using SM = AttnSmem<HD>;
    constexpr int HG = HD / 8;                                      // 8-element pieces of a row
    pdl_launch_dependents();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int item = a.meta.it_order[blockIdx.z];
    // per-request constants: independent loads, in flight together
    const int nsplit = a.meta.it_nsplit[item];
    const int rows = a.meta.it_rows[item];
    const int base = a.meta.it_base[item];
    const int chunk = a.meta.it_chunk[item];
    const int row0 = a.meta.it_row0[item];
    const int part0 = a.meta.it_part0[item];
    const int req_slot = a.meta.it_slot[item];
    const int sp = blockIdx.x;                                     // key split of this CTA
    if (sp >= nsplit) return;
    const int Hkv = a.Hkv, Hq = a.Hq;
    const int kvh = blockIdx.y % Hkv, rg = a.row_groups - 1 - blockIdx.y / Hkv;   // the latest rows see the most keys: first
    const int G = Hq / Hkv;
    const int R = G * rows;
    const int rho0 = rg * a.rows_cap;
    if (rho0 >= R) return;
    const int n_rows = min(a.rows_cap, R - rho0);
    const int N = (n_rows + 15) & ~15;
    if (N > a.n_max) return;
    const int NG = N / 8, NB = N / 16;
    const int total = base + rows;
    // query rows are numbered (chunk row, query head): a group's last row bounds the keys that any of its rows sees, so the
    // early groups of a prompt chunk stop short of the chunk's own later keys
    const int seen = min(total, base + (rho0 + n_rows - 1) / G + 1);
    AttnCtx c;
    c.k0 = min(sp * chunk, seen);
    c.k1 = min(c.k0 + chunk, seen);
    c.kbase = a.kv_pool + kv_index(a.layer, a.n_pages, 0, 0, Hkv, kvh, a.page_size, 0, HD, 0);
    c.page_stride = (size_t)2 * Hkv * a.page_size * HD;
    c.v_off = (size_t)Hkv * a.page_size * HD;
    c.page_size = a.page_size;
    c.bt = a.meta.block_tab + (size_t)req_slot * a.meta.max_pages;
    const int ntiles = c.k1 > c.k0 ? (c.k1 - c.k0 + kAttnTile - 1) / kAttnTile : 0;
    const size_t slot0 = (size_t)part0 + ((size_t)kvh * R + rho0) * nsplit;     // + row * nsplit + split
    const int KSo = (Hq * HD) / 16, NTo = xf_nt(a.M);

    // ---- shared memory: the ones come first (the tensor cores read a few KB past them, see below)
    unsigned char* ones = smem;
    unsigned char* ring = ones + SM::kOnes;                        // a.slots slots of a tile (of three, the last may be shorter)
    unsigned char* q_hi = ring + a.ring;
    unsigned char* q_lo = q_hi + SM::q_bytes(N);
    unsigned char* p_hi = q_lo + SM::q_bytes(N);
    float* wm = reinterpret_cast<float*>(p_hi + 2 * SM::p_bytes(N));   // [4][N] maxima of a tile per lane quarter
    int* hz = reinterpret_cast<int*>(wm + 4 * N);                  // [N] last visible key of a row
    float* m_ref = reinterpret_cast<float*>(hz + N);               // [N] reference score of a row
    float* alpha = m_ref + N;                                      // [N] rescale factor of a row for this tile
    float* Fl = alpha + N;                                         // [N] the CTA's partial denominators
    unsigned long long* bars = reinterpret_cast<unsigned long long*>(Fl + N);   // full[4], s_full[2], p_full, pv_done
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 8);
    unsigned* s_mine = reinterpret_cast<unsigned*>(tmem_slot + 1);
    const uint32_t bar_full = smem_u32(bars), bar_s = bar_full + 32, bar_p = bar_full + 48, bar_pv = bar_full + 56;
    const uint32_t tmem_cols = (uint32_t)attn_tmem_cols(N);
    const uint32_t ring_a = smem_u32(ring);
    const int slots = a.slots;
    // ring item i (K_t: 2t, V_t: 2t+1) lives in slot i % slots
    auto slot_of = [&](int i) { return slots == 4 ? i & 3 : i % 3; };
    auto turn_of = [&](int i) { return (uint32_t)(slots == 4 ? i >> 2 : i / 3) & 1u; };
    auto slot_addr = [&](int i) { return ring_a + (uint32_t)slot_of(i) * SM::kTileBytes; };

    auto issue_item = [&](int i) {
        attn_issue_tile<HD>(c.kbase + (i & 1 ? c.v_off : 0), c.bt, c.page_stride, c.page_size, c.k1, slot_addr(i), bar_full + 8 * slot_of(i),
                            c.k0 + (i >> 1) * kAttnTile);
    };

    bool ok = true;
    uint32_t tmem_held = 0;        // tensor memory to give back before leaving, if any (address 0 is a valid one)
    bool holds_tmem = false;
    // Tensor memory is released off the critical path: after the partial result has been announced.
    auto release_tmem = [&]() {
        if (holds_tmem && warp == 8) {
            tc_fence_after();
            tmem_dealloc(tmem_held, tmem_cols);
        }
    };
    if (ntiles > 0) {
        uint32_t tmem = 0;
        if (warp == 8) {
            // ---------------- barriers, the first three items of the ring, tensor memory
            if (lane == 0) {
                for (int i = 0; i < 8; ++i) mbar_init(bar_full + 8 * i, 1);
                fence_mbar_init();
            }
            __syncwarp();
            // Items made only of keys cached before this pass do not depend on the QKV projection that precedes this
            // kernel: they are requested now, the others after the dependency has resolved.
            const int early_tiles = base >= c.k1 ? ntiles : (base - c.k0) / kAttnTile;      // whole tiles below `base`
            const int first = min(2 * ntiles, slots);                                           // items requested up front
#pragma unroll 1
            for (int i = 0; i < first; ++i)
                if ((i >> 1) < early_tiles) issue_item(i);
            tmem_alloc(smem_u32(tmem_slot), tmem_cols);
            tc_fence_before();
            pdl_wait();
#pragma unroll 1
            for (int i = 0; i < first; ++i)
                if ((i >> 1) >= early_tiles) issue_item(i);
        } else {
            // operands that do not depend on the predecessor: the ones, the rows' horizons and initial state
            if (tid < SM::kOnes / 4) reinterpret_cast<uint32_t*>(ones)[tid] = 0x3F803F80u;
#pragma unroll 1
            for (int n = tid; n < N; n += kAttnWorkers) {
                const int rho = rho0 + n;
                // (a padding row has scores of 0; it sees every key, so that its reference is 0 too and nothing exceeds that)
                hz[n] = n < n_rows ? base + rho / G : 0x7fffffff;
                m_ref[n] = -INFINITY;
            }
            pdl_wait();
            // ---- stage Q (scaled by log2(e)/sqrt(hd)) as the K-major B operand, bf16 hi and lo terms:
            // piece (row n, k group g) at ((n/8) * HG + g) * 128 + (n%8) * 16.  Two pieces per thread and step, all
            // loads of a step in flight together.
            const float scale = rsqrtf((float)HD) * 1.4426950408889634f;   // scores in the log2 domain: p = 2^(s - m)
#pragma unroll 1
            for (int idx0 = tid; idx0 < N * HG; idx0 += 2 * kAttnWorkers) {
                float4 x[2][2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int idx = idx0 + u * kAttnWorkers, n = idx / HG, g = idx % HG;
                    x[u][0] = x[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (idx < N * HG && n < n_rows) {
                        const int rho = rho0 + n, gq = rho % G, r = rho / G;
                        const float4* qp = reinterpret_cast<const float4*>(a.q + ((size_t)(row0 + r) * Hq + kvh * G + gq) * HD + g * 8);
                        x[u][0] = qp[0];
                        x[u][1] = qp[1];
                    }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int idx = idx0 + u * kAttnWorkers, n = idx / HG, g = idx % HG;
                    if (idx >= N * HG) break;
                    const float v[8] = {x[u][0].x * scale, x[u][0].y * scale, x[u][0].z * scale, x[u][0].w * scale,
                                        x[u][1].x * scale, x[u][1].y * scale, x[u][1].z * scale, x[u][1].w * scale};
                    uint32_t h[4], l[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) split_bf16x2(v[2 * i], v[2 * i + 1], h[i], l[i]);
                    const uint32_t off = (uint32_t)(((n >> 3) * HG + g) * 128 + (n & 7) * 16);
                    *reinterpret_cast<uint4*>(q_hi + off) = make_uint4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<uint4*>(q_lo + off) = make_uint4(l[0], l[1], l[2], l[3]);
                }
            }
            fence_proxy_async_smem();      // the tensor cores read these through the asynchronous proxy
        }
        __syncthreads();                   // barriers, Q, ones and the tensor-memory base are in place
        tc_fence_after();
        tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
        const bool wide_q = attn_wide_q(N), wide_p = attn_wide_p(N);
        const int NS = wide_q ? 2 * N : N, NO = wide_p ? 2 * N : N;                                // columns of S^T / of O^T and L
        const uint32_t t_S = tmem, t_O = tmem + 2u * (uint32_t)NS, t_L = t_O + (uint32_t)NO;       // S^T twice, O^T, L

        if (warp == 8) {
            // ---------------- copies and MMA issue.  Ring item i may be requested once item i - slots has been read: a K tile
            // by the first product of its tile (s_full), a V tile by the second (pv_done).  The first product of tile t+1 is issued ahead of the second of tile t.
            const uint32_t idesc_qk = umma_idesc_bf16(128, NS, 0, 0), idesc_pv = umma_idesc_bf16(128, NO, 1, 1);
            const uint32_t qh = smem_u32(q_hi), ql = smem_u32(q_lo), ph = smem_u32(p_hi);
            // the denominators' A operand: 16 keys x 8 rows of ones; the other 120 rows of the MMA read whatever follows
            // in shared memory (the ring) and land in tensor-memory lanes that nobody reads
            const uint64_t ones_desc = umma_desc(smem_u32(ones), 128, 256);
            auto issue_qk = [&](int t) {       // S^T[t & 1] = K_t . Q^T
                const uint32_t d = t_S + (uint32_t)((t & 1) * NS);
                uint64_t kd = umma_desc(slot_addr(2 * t), 128, HG * 128), hd_ = umma_desc(qh, 128, HG * 128), ld_ = umma_desc(ql, 128, HG * 128);
#pragma unroll 4
                for (int kk = 0; kk < HD / 16; ++kk) {
                    umma_bf16(d, kd, hd_, idesc_qk, kk > 0);
                    if (!wide_q) umma_bf16(d, kd, ld_, idesc_qk, 1);
                    kd += 256 >> 4; hd_ += 256 >> 4; ld_ += 256 >> 4;
                }
                umma_commit(bar_s + 8 * (t & 1));
            };
            auto full_wait = [&](int i) { return attn_wait_warp(bar_full + 8 * slot_of(i), turn_of(i)); };
            auto request = [&](int i) {        // ring item i, if the split has it
                if ((i >> 1) < ntiles) issue_item(i);
            };
#pragma unroll 1
            for (int t = -1; t < ntiles && ok; ++t) {
                if (t + 1 < ntiles) {
                    ok = full_wait(2 * t + 2);                                           // K of tile t+1 has landed
                    // S^T[(t+1) & 1] was last read for tile t-1: free once P of tile t-1 was announced (seen below)
                    if (ok && elect_one()) { tc_fence_after(); issue_qk(t + 1); }
                }
                if (t < 0) continue;
                if (ok) ok = attn_wait_warp(bar_s + 8 * (t & 1), (uint32_t)(t >> 1) & 1u);   // K_t has been read
                if (ok) request(2 * t + slots);                                          // into K_t's slot
                if (ok) ok = attn_wait_warp(bar_p, (uint32_t)t & 1u);                    // P of tile t is written (and O^T rescaled)
                if (ok) ok = full_wait(2 * t + 1);                                       // V of tile t has landed
                if (ok && elect_one()) {
                    tc_fence_after();
                    const uint32_t va = slot_addr(2 * t + 1);
                    const int n_valid = min(kAttnTile, c.k1 - (c.k0 + t * kAttnTile));
                    const int n16 = (n_valid + 15) / 16;
                    // P: hi and lo row groups side by side, 2 * NG of them per key group
                    uint64_t vd = umma_desc(va, HG * 128, 128), pd = umma_desc(ph, 2 * NG * 128, 128);
                    uint32_t acc = t > 0 ? 1u : 0u;
#pragma unroll 2
                    for (int ks = 0; ks < n16; ++ks) {
                        umma_bf16(t_O, vd, pd, idesc_pv, acc);
                        umma_bf16(t_L, ones_desc, pd, idesc_pv, acc);
                        if (!wide_p) {
                            umma_bf16(t_O, vd, pd + (uint64_t)((NG * 128) >> 4), idesc_pv, 1);
                            umma_bf16(t_L, ones_desc, pd + (uint64_t)((NG * 128) >> 4), idesc_pv, 1);
                        }
                        vd += (2 * HG * 128) >> 4;
                        pd += (uint64_t)((4 * NG * 128) >> 4);
                        acc = 1u;
                    }
                    umma_commit(bar_pv);
                }
                if (ok && t == ntiles - 1) {
                    // every K/V tile of this CTA has landed and its last products are issued: hints for the weights
                    // of the projections that follow
                    const size_t n_thr = (size_t)gridDim.x * gridDim.y * gridDim.z * 32;
                    const size_t g = (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * 32 + lane;
#pragma unroll
                    for (int r = 0; r < 2; ++r)
                        if (a.pf_ptr[r] != nullptr)
                            for (size_t o = g * 128; o < a.pf_len[r]; o += n_thr * 128)
                                asm volatile("prefetch.global.L2 [%0];" ::"l"(a.pf_ptr[r] + o) : "memory");
                }
                if (ok && t + 2 < ntiles) {
                    ok = attn_wait_warp(bar_pv, (uint32_t)t & 1u);                       // V_t has been read
                    if (ok) request(2 * t + 1 + slots);                                  // into V_t's slot
                }
            }
            if (!ok && a.err && lane == 0) atomicExch(a.err, 3);
        } else {
            // ---------------- thread = key of the tile (tensor-memory lane 32 * quarter + lane); the two warps of a
            // lane quarter take alternate 8-row column blocks
            const int quarter = warp & 3, half = warp >> 2;
            const int kt = quarter * 32 + lane;                         // key within the tile
            const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
#pragma unroll 1
            for (int t = 0; t < ntiles; ++t) {
                const int j = c.k0 + t * kAttnTile + kt;                // this thread's key
                const int n_valid = min(kAttnTile, c.k1 - (c.k0 + t * kAttnTile));
                const uint32_t t_St = t_S + (uint32_t)((t & 1) * NS);
                if (ok) ok = attn_wait_warp(bar_s + 8 * (t & 1), (uint32_t)(t >> 1) & 1u);
                tc_fence_after();
                const bool need_mask = c.k0 + (t + 1) * kAttnTile - 1 > base || n_valid < kAttnTile;   // CTA-uniform
                // A row's reference: the score of the split's first key, if the row sees it (else it sees none of the split).
                // Softmax does not mind which: the largest p of the row is then at least 1, and no p may exceed
                // 2^kAttnMaxExcess, so that everything stays far inside the range of fp32 and of the bf16 terms.
                // eight columns of S^T: rows of Q's hi terms, and of its lo terms where they have columns of their own
                auto read_s = [&](uint32_t at, float (&s)[8]) {
                    float l[8];
                    tmem_ld8(at, s);
                    if (wide_q) tmem_ld8(at + (uint32_t)N, l);
                    tmem_ld_wait8(s);
                    if (wide_q) {
                        tmem_ld_wait8(l);
#pragma unroll
                        for (int i = 0; i < 8; ++i) s[i] += l[i];
                    }
                };
                if (t == 0) {
                    if (quarter == 0) {
#pragma unroll 1
                        for (int cu = half; cu < NG; cu += 2) {
                            float s[8];
                            read_s(t_St + cu * 8, s);
                            if (lane == 0) {
#pragma unroll
                                for (int i = 0; i < 8; ++i) m_ref[cu * 8 + i] = ok && j <= hz[cu * 8 + i] ? s[i] : -INFINITY;
                            }
                        }
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(kAttnWorkers) : "memory");
                }
                // ---- p = 2^(s - reference) as bf16 hi and lo terms, in registers: this part runs under the previous tile's
                // second product.  Done again, once, where some score exceeds its reference by too much.
#pragma unroll 1
                for (int again = 0;; ++again) {
                    bool over = false;
                    uint32_t hw[CU][4], lw[CU][4];
#pragma unroll
                    for (int q = 0; q < CU; ++q) {
                        const int cu = half + 2 * q;
                        if (cu < NG) {
                            float sc[8], mr[8];
                            read_s(t_St + lane_sel + cu * 8, sc);
                            *reinterpret_cast<float4*>(mr) = *reinterpret_cast<const float4*>(m_ref + cu * 8);
                            *reinterpret_cast<float4*>(mr + 4) = *reinterpret_cast<const float4*>(m_ref + cu * 8 + 4);
                            if (need_mask) {
#pragma unroll
                                for (int i = 0; i < 8; ++i)
                                    if (!(j < c.k1 && j <= hz[cu * 8 + i])) sc[i] = -INFINITY;
                            }
#pragma unroll
                            for (int i = 0; i < 8; i += 2) {
                                float p2[2];
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    over |= sc[i + e] > mr[i + e] + kAttnMaxExcess;
                                    p2[e] = (ok && mr[i + e] > -INFINITY) ? fast_exp2(sc[i + e] - mr[i + e]) : 0.f;    // masked: 2^-inf = 0
                                }
                                split_bf16x2(p2[0], p2[1], hw[q][i >> 1], lw[q][i >> 1]);
                            }
                        }
                    }
                    // the previous tile's second product has read P (and updated O^T, L): P may be overwritten
                    if (t > 0 && again == 0 && ok) ok = attn_wait_warp(bar_pv, (uint32_t)(t - 1) & 1u);
                    tc_fence_after();
                    // the MN-major B operand: piece (key group kg, row group g, key) at ((kg * 2 NG + g) * 8 + key % 8) * 16 holds
                    // 8 rows, their lo terms in row group NG + g
#pragma unroll
                    for (int q = 0; q < CU; ++q) {
                        const int cu = half + 2 * q;
                        if (cu < NG) {
                            const uint32_t off = (uint32_t)((((kt >> 3) * 2 * NG + cu) * 8 + (kt & 7)) * 16);
                            *reinterpret_cast<uint4*>(p_hi + off) = make_uint4(hw[q][0], hw[q][1], hw[q][2], hw[q][3]);
                            *reinterpret_cast<uint4*>(p_hi + off + NG * 128) = make_uint4(lw[q][0], lw[q][1], lw[q][2], lw[q][3]);
                        }
                    }
                    // V rows at and beyond the split's end must be finite (P is 0 there, but 0 * NaN is not): cleared, once
                    // the tile's V rows have landed (the copy may bring garbage rows of the last 8-row group)
                    if (n_valid < kAttnTile) {
                        if (ok) ok = attn_wait_warp(bar_full + 8 * slot_of(2 * t + 1), turn_of(2 * t + 1));
                        if (half == 0 && kt >= n_valid && kt < ((n_valid + 15) & ~15)) {
                            unsigned char* v_tile = ring + slot_of(2 * t + 1) * SM::kTileBytes;
#pragma unroll
                            for (int g = 0; g < HG; ++g)
                                *reinterpret_cast<uint4*>(v_tile + ((kt >> 3) * HG + g) * 128 + (kt & 7) * 16) = make_uint4(0, 0, 0, 0);
                        }
                    }
                    fence_proxy_async_smem();
                    tc_fence_before();
                    if (!attn_workers_any(over && ok && again == 0)) break;
                    // ---- rare: the rows' references move up to the tile's maxima (over the 32 keys of the warp, then over
                    // the lane quarters), what has been summed is rescaled, and P is written again
#pragma unroll 1
                    for (int cu = half; cu < NG; cu += 2) {
                        float s[8];
                        read_s(t_St + lane_sel + cu * 8, s);
                        float mine = -INFINITY;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float v = s[i];
                            if (need_mask && !(j < c.k1 && j <= hz[cu * 8 + i])) v = -INFINITY;
                            const float wmax = warp_max_redux(v);
                            if (lane == i) mine = wmax;
                        }
                        if (lane < 8) wm[quarter * N + cu * 8 + lane] = mine;
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(kAttnWorkers) : "memory");
                    if (tid < N) {
                        const float tmax = fmaxf(fmaxf(wm[tid], wm[N + tid]), fmaxf(wm[2 * N + tid], wm[3 * N + tid]));
                        const float m_old = m_ref[tid], m_new = fmaxf(m_old, tmax);
                        m_ref[tid] = m_new;
                        alpha[tid] = m_new > m_old ? fast_exp2(m_old - m_new) : 1.f;       // from -inf: nothing summed so far, 0
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(kAttnWorkers) : "memory");
                    if (t > 0) {
#pragma unroll 1
                        for (int cb = half; cb < 2 * NO / 16; cb += 2) {             // O^T and L: all columns from t_O
                            float o[16];
                            tmem_ld16(t_O + lane_sel + cb * 16, o);
                            tmem_ld_wait16(o);
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] *= alpha[(cb % NB) * 16 + i];
                            tmem_st16(t_O + lane_sel + cb * 16, o);
                        }
                        tmem_st_wait();
                    }
                }
                if (tid == 0) mbar_arrive(bar_p);
            }
            // ---- the CTA's partial result: O^T (thread = head dimension) and L (lanes 0-7 hold all rows' sums)
            if (ok) ok = attn_wait_warp(bar_pv, (uint32_t)(ntiles - 1) & 1u);
            tc_fence_after();
            // sixteen columns of O^T or L: the products with P's hi terms, and those with its lo terms where they are apart
            auto read_16 = [&](uint32_t at, float (&v)[16]) {
                tmem_ld16(at, v);
                tmem_ld_wait16(v);
                if (wide_p) {
                    float l[16];
                    tmem_ld16(at + (uint32_t)N, l);
                    tmem_ld_wait16(l);
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] += l[i];
                }
            };
            if (quarter == 0) {
                // the column blocks go to the two warps of the quarter the other way round than O^T's below, so that with
                // one block the denominators are stored by a warp that has no O^T columns to store
#pragma unroll 1
                for (int cb = half ^ 1; cb < NB; cb += 2) {
                    float l[16];
                    read_16(t_L + cb * 16, l);
                    if (lane == 0) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) Fl[cb * 16 + i] = ok ? l[i] : 0.f;
                    }
                    __syncwarp();
                    const int n = cb * 16 + lane;
                    if (nsplit > 1 && lane < 16 && n < n_rows) {         // lane = row: one store each
                        a.l_part[slot0 + (size_t)n * nsplit + sp] = Fl[n];
                        a.m_part[slot0 + (size_t)n * nsplit + sp] = m_ref[n];
                    }
                }
            }
            // nothing to merge: the rows are normalised and stored as the output projection's input.  Where a row lands
            // there (its token, its head's first k16 step) is worked out once per row, into the maxima's array
            uint32_t* otab = reinterpret_cast<uint32_t*>(wm);
            if (nsplit == 1 && tid < n_rows) {
                const int rho = rho0 + tid, gq = rho % G, r_in = rho / G;
                otab[tid] = act_index_row(row0 + r_in, ((kvh * G + gq) * HD) >> 4, KSo, NTo, a.xd_tbs);
            }
            const uint32_t ocol = act_index_col(kt, NTo, a.xd_tbs), olo = act_index_lo(a.xd_tbs);
            if (nsplit == 1) asm volatile("bar.sync 1, %0;" ::"n"(kAttnWorkers) : "memory");     // the sums and the table
#pragma unroll 1
            for (int cb = half; cb < NB; cb += 2) {
                float o[16];
                read_16(t_O + lane_sel + cb * 16, o);
                if (kt < HD) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int n = cb * 16 + i;
                        if (n < n_rows) {
                            const float v = ok ? o[i] : 0.f;
                            if (nsplit == 1) {
                                act_store_at(a.xf_out, otab[n] + ocol, olo, v / Fl[n]);
                            } else {
                                a.o_part[(slot0 + (size_t)n * nsplit + sp) * HD + kt] = v;
                            }
                        }
                    }
                }
            }
            if (!ok && a.err && lane == 0) atomicExch(a.err, 4);
            tc_fence_before();
        }
        __syncthreads();
        tmem_held = tmem;
        holds_tmem = true;
    } else {
        // empty split: contributes nothing (finite zeros, so the merge can read it unconditionally)
        pdl_wait();
#pragma unroll 1
        for (int i = tid; i < n_rows * HD; i += kAttnThreads) a.o_part[(slot0 + (size_t)(i / HD) * nsplit + sp) * HD + i % HD] = 0.f;
#pragma unroll 1
        for (int i = tid; i < n_rows; i += kAttnThreads) {
            a.m_part[slot0 + (size_t)i * nsplit + sp] = -INFINITY;
            a.l_part[slot0 + (size_t)i * nsplit + sp] = 0.f;
        }
        __syncthreads();
    }
    if (nsplit == 1) { release_tmem(); return; }

    // ---- merge of the splits, in split order, by the last CTA of this (request, KV head, row group) to arrive; or, where all
    // CTAs of the launch fit the device together and a group has more rows than one round of warps (nine) takes, by all CTAs
    // of the group, every nsplit-th row each (68 rows x 13 splits, 450 KB, take one SM 14 us).  Nobody depends on that: a CTA
    // that does not see all the others arrive within merge_polls looks, because other work holds the SMs they need, marks
    // its rows as not taken and leaves; the last one finds the marks in its ticket and merges those rows too.
    // (the barrier above orders the whole CTA's stores before thread 0's ticket, a release; the ticket or the poll is also an
    // acquire, and the barrier below orders it before everybody's loads of the other CTAs' partials)
    const bool share = a.share_merge && n_rows > kAttnThreads / 32;
    if (tid == 0) {
        // one byte of arrivals, one of departures (shared merges), 16 marks; zero again when the last is through
        unsigned* ticket = reinterpret_cast<unsigned*>(a.tickets) + ((size_t)item * Hkv + kvh) * a.row_groups + rg;
        auto ticket_add = [&](unsigned v) {
            unsigned t;
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(t) : "l"(ticket), "r"(v) : "memory");
            return t;
        };
        unsigned t = ticket_add(1u);
        const bool last = (t & 0xffu) == (unsigned)nsplit - 1u;
        unsigned mine = 0u;                                      // bit s: the rows of split s's share are this CTA's to merge
        if (!share) {
            mine = last ? 1u : 0u;
            if (last) *ticket = 0u;                              // self-cleaning: ready for the next launch
        } else {
            bool all = last;
            for (int it = 0; it < a.merge_polls && !all; ++it) {
                unsigned seen_t;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen_t) : "l"(ticket) : "memory");
                all = (seen_t & 0xffu) == (unsigned)nsplit;
            }
            if (last) mine = t >> 16;
            t = ticket_add(all ? 0x100u : 0x100u + (0x10000u << sp));
            // (a mark that comes after the last arrival is seen by nobody, and all partials are there)
            if ((t & 0xffu) == (unsigned)nsplit) mine |= 1u << sp;
            if (((t >> 8) & 0xffu) == (unsigned)nsplit - 1u) *ticket = 0u;
        }
        *s_mine = mine;
    }
    __syncthreads();
    release_tmem();
    const unsigned mine = *s_mine;
    if (mine == 0u) return;
    // warp = row, lane = four columns: one round covers nine rows.  All of a row's loads are issued before the first
    // use (one trip to the L2 for up to kMergeBatch splits): lane j fetches split j's maximum and denominator, every
    // lane its four columns of each split's numerator; the sums run in split order.
    constexpr int kMergeBatch = 10;
    const int rl_step = share ? nsplit : 1;
#pragma unroll 1
    for (unsigned left = mine; left != 0u; left &= left - 1u)    // shares to merge, one after the other
#pragma unroll 1
    for (int rl = (share ? __ffs(left) - 1 : 0) + warp * rl_step; rl < n_rows; rl += rl_step * (kAttnThreads / 32)) {
        const size_t sl0 = slot0 + (size_t)rl * nsplit;
        const float m_mine = lane < nsplit ? __ldcg(a.m_part + sl0 + lane) : -INFINITY;
        const float l_mine = lane < nsplit ? __ldcg(a.l_part + sl0 + lane) : 0.f;
        float4 ov[kMergeBatch];
#pragma unroll
        for (int j = 0; j < kMergeBatch; ++j)
            ov[j] = (j < nsplit && lane < HD / 4) ? __ldcg(reinterpret_cast<const float4*>(a.o_part + (sl0 + j) * HD) + lane)
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        const float m = warp_max_redux(m_mine);
        // an empty split, or one beyond the causal horizon, has no maximum and weighs nothing
        const float w_mine = (m_mine == -INFINITY) ? 0.f : exp2f(m_mine - m);
        const float wl_mine = w_mine * l_mine;
        float den = 0.f;
        float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < kMergeBatch; ++j) {
            const float w = __shfl_sync(0xffffffffu, w_mine, j);
            den += __shfl_sync(0xffffffffu, wl_mine, j);
            num.x += w * ov[j].x; num.y += w * ov[j].y; num.z += w * ov[j].z; num.w += w * ov[j].w;
        }
        for (int j = kMergeBatch; j < nsplit; ++j) {             // more splits than one batch holds: one by one
            const float w = __shfl_sync(0xffffffffu, w_mine, j);
            den += __shfl_sync(0xffffffffu, wl_mine, j);
            if (lane < HD / 4) {
                const float4 o = __ldcg(reinterpret_cast<const float4*>(a.o_part + (sl0 + j) * HD) + lane);
                num.x += w * o.x; num.y += w * o.y; num.z += w * o.z; num.w += w * o.w;
            }
        }
        if (lane < HD / 4) {
            const int rho = rho0 + rl, gq = rho % G, r_in = rho / G;
            const int dk = lane * 4;                                 // column within the head
            const float inv = 1.f / den;
            const uint32_t idx = act_index_row(row0 + r_in, ((kvh * G + gq) * HD) >> 4, KSo, NTo, a.xd_tbs) + act_index_col(dk, NTo, a.xd_tbs);
            uint32_t h[2], l[2];
            split_bf16x2(num.x * inv, num.y * inv, h[0], l[0]);
            split_bf16x2(num.z * inv, num.w * inv, h[1], l[1]);
            // columns dk, dk + 1 are neighbours in either layout; dk + 2 follows them in an xd array, one lane (16 bytes) on in
            // fragment order
            const uint32_t lo = act_index_lo(a.xd_tbs), next = a.xd_tbs > 0 ? 2 : 8;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                *reinterpret_cast<uint32_t*>(a.xf_out + idx + e * next) = h[e];
                *reinterpret_cast<uint32_t*>(a.xf_out + idx + e * next + lo) = l[e];
            }
        }
    }
}

}  // namespace pipesd
