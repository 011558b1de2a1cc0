// The whole layer stack of a pass of at most 32 rows as ONE persistent kernel: embedding, every layer's QKV projection,
// attention, output projection, gate/up and down projections, and the vocabulary projection, one CTA per SM.
//
// What bounds such a pass is the weights' stream from HBM, and what kept it from that bound were the dependencies: with
// a kernel per projection HBM stands still while a kernel reduces, stores, exits and the next one starts and fetches its
// activations.  Here every CTA has ONE copy stream that knows no phases: the weights of all projections and the cached
// K/V are requested in the order they will be used, as far ahead as the chip holds them: a ring of up to 192 KB of shared
// memory per SM, and, while a phase waits for its activations, another 192 KB of tensor memory, where weights are the MMA's
// A operand as well as in shared memory (56 MB in all, 7 us of HBM).  (Hints into the L2 beyond that gained nothing: an SM takes
// lines that a hint brought there in at 57 B/ns, those of HBM at 52.)
//
// Projections.  A CTA takes an equal, contiguous range of the matrix's (128-row block, k16 step) units, whatever their
// number: no last wave, no slices that do not divide.  Weights are the M side of tcgen05.mma (M = 128 rows, as they lie in
// the packed copy), the rows of the pass the N side: bf16 hi and lo terms side by side, one MMA of N = 16 per eight rows.
// One lane issues; the accumulator goes to registers after `flush` stages, where sums round to nearest (the tensor pipe
// truncates where it adds; see dense_chunk).  A row block that several CTAs share is exchanged through L2 as 16-byte words
// of three values and a phase number: a reader polls the data itself, one trip, no fence and no flag behind it.  The CTAs of a
// block finish a few rows of the pass each (sums in CTA order, epilogue): nobody finishes all.  The order of sums follows the
// weights' shape and the number of SMs alone.
// Between phases: one arrival counter, one look by one lane per CTA.
//
// Attention.  The keys of all (request, KV head) pairs form one line, cut into equal ranges, one per CTA; a range's parts
// (segments) run through the algorithm of attention.cuh (keys on the M side; S^T, O^T and denominators in tensor memory;
// exponentials relative to the segment's first key), K/V from the same copy stream, Q already in operand order.  A head whose keys are
// one CTA's is finished there; of others, partial results are exchanged like partial sums, each contributor merges every C-th row.
//
// What a phase costs beyond its stream (7b shape, 9 rows, us): look 0.5, activations 0.8, exchange and epilogue 2, release 1; the
// attention 12.  Every phase runs code that the one before it did not, so the hot paths are kept short and rolled: code that
// does not fit the instruction cache (32 to 64 KB, from how passes changed) cost more than anything it computed.
//
// Every wait is bounded; whoever gives up sets the CTA's abort flag and the device error word, and every role ends at its
// first wait that runs out, so that the kernel ends within seconds whatever went wrong.  The CTAs wait for one another: the
// launch is cooperative, so that all of them are on the device together or none is.
#pragma once
#include "attention.cuh"
#include "common.cuh"
#include "gemm.cuh"
#include "layers.cuh"
#include "tcgen05.cuh"

namespace pipesd {

constexpr int kStackThreads = 384;           // copies | activations | MMA | tables | 8 worker warps
constexpr int kStackWorkers = 256;
constexpr int kStackMaxCtas = 148;
constexpr int kStackSteps = 8;               // k16 steps per ring stage
constexpr int kStackSlot = kStackSteps * 4096;   // bytes of a ring slot: a stage of weights, or a K or V tile
constexpr int kStackMaxSlots = 6, kStackMinSlots = 3, kStackMaxActs = 8;
// Ring items on their way at once.  HBM is busy with two of 32 KB per SM (7.3 TB/s read alone; three 7.5, five 7.9), but a deeper queue
// serves some SMs before others (with five 44 SMs get 48 B/ns, 104 get 55, and a phase ends with the slowest: 7.0 TB/s), and
// everything else an SM fetches waits behind it (7b shape, 9 rows, us a pass: two 2850, three 2867, all 2960).
constexpr unsigned kStackInFlight = 2;
constexpr int kStackStaged = 6;              // stages of weights that tensor memory holds, beside the accumulators: columns 128..511
constexpr int kStackMaxN = 72;               // query rows per KV head and request
constexpr int kStackMaxSegs = 16, kStackMaxItems = 16;
constexpr int kStackSmemMax = 227 * 1024;
constexpr int kStackSyncBytes = 512;         // arrivals | base | phase number, a line each

enum StackKind { kStQkv = 0, kStAttn = 1, kStO = 2, kStGu = 3, kStDn = 4, kStLm = 5 };

struct StackGemm {
    const unsigned char* w;      // packed weights of layer 0
    const unsigned char* act;    // input, "xd" order with token blocks of T
    int N, KS, RB;
    int per;                     // k16 steps per CTA
    int flush;                   // stages per accumulator
};

struct StackArgs {
    StackGemm g[6];
    size_t layer_stride;         // bytes from one layer's weights (and gains) to the next's
    const float *n1, *n2, *final_norm;
    const uint16_t* emb;
    PassMeta meta;
    uint16_t* kv_pool;
    float *x, *cs, *sn, *logits, *ssq_a, *ssq_b;
    uint16_t *act_h, *act_attn, *act_ffn;
    uint16_t* qop;               // Q as the MMA's B operand: per (request, KV head) hi then lo terms of N rows
    size_t qop_bytes;
    uint4* ll;                   // exchange words
    size_t ll_ml;                // index of the attention's (reference, denominator) words
    int ll_rows;                 // rows of 128 words per CTA and shared row block
    unsigned* sync;
    int* err;
    int n_layers, d, Hq, Hkv, M, n_items, want_logits, n_pages, page_size, n_ssq;
    unsigned looks;              // kStackLooks, unless a harness asks for less
    int slots, acts;             // ring slots, activation slots
    int n_max, r_max, q_bufs, p_bufs;   // attention: N and rows per KV head of the largest request; buffers of Q and P
    float eps;
    double log_base;
};

struct StackSeg {
    int kvh, k0, k1, base, n_rows, N, row0, C, idx, ll0;
    unsigned q_off;              // elements
    const int32_t* bt;
};
struct StackItem { int base, rows, units, u0, N, row0, slot, rowsum; unsigned q0; };

// What a CTA does in a projection, the same in every layer.
struct StackGeo {
    int s, e, b, ks;             // its units, the row block and the k16 step they begin with
    int ring, flip, stages;      // its stages, as ring slots and turns further on, and their number
    int n_ent[2];                // groups of rows it finishes, per half of the workers
    int second;                  // the last row block of its range
};
struct StackEnt { int off, C, w, t, n; };       // words of the first contributor, contributors, first or last block, rows t .. t + n - 1

// Shared memory behind ring and scratch.
struct StackSmall {
    unsigned long long full_w[kStackMaxSlots], empty_w[kStackMaxSlots], full_a[kStackMaxActs], empty_a[kStackMaxActs], d_full[2], d_empty[2],
        q_full[2], q_empty[2], s_full[2], p_full, pv_done[2], phase, tables, last;
    uint32_t tmem;
    int go, abort;               // the launch has work to do; a role has given up
    unsigned base, epoch, issued_w, issued_a, issued_q;
    int n_seg, n_tiles;
    float rstd[32], red[8];
    long long kvoff[32];
    unsigned q_off[32];          // elements: the row's request's Q of KV head 0
    int q_N[32], q_r[32];        // N of its request; the row's number in it
    StackGeo geo[6];
    StackEnt ent[6][2][8];
    int snd[6][2][2][16];        // where the partial sums of a half's groups go (rows of 128 words): of the first, of the last block
    StackItem it[kStackMaxItems];
    StackSeg seg[kStackMaxSegs];
};

// How C CTAs that share a row block divide finishing it.  The two halves of the workers hold rows [0, h) and [h, M) of the
// pass, h = half_rows(M); up to three neighbouring rows of a half, a group, travel in one exchange word (as few as give every
// half of every CTA its own).  Groups are dealt to the CTAs in turn, a CTA's to its halves in turn.
__host__ __device__ inline int stack_half_rows(int M) { return (M + 1) / 2; }
__host__ __device__ inline int stack_group(int M, int C) { const int n = (M + 2 * C - 1) / (2 * C); return n > 3 ? 3 : n; }
__host__ __device__ inline int stack_half_groups(int M, int C) { const int g = stack_group(M, C); return (stack_half_rows(M) + g - 1) / g; }
// The most CTAs that share a row block of KS steps.
__host__ __device__ inline int stack_max_share(int KS, int per) { return (KS + per - 2) / per + 1; }

// k16 steps per CTA of a projection of RB row blocks, KS steps deep.
__host__ inline int stack_per(int KS, int RB, int ctas) {
    const int p = (int)(((long)RB * KS + ctas - 1) / ctas);
    return p > kStackSteps ? p : kStackSteps;
}

// Host and device: the sizes one launch needs.
struct StackPlan { int T, slots, acts, q_bufs, p_bufs, scratch; size_t smem; };
static inline bool stack_plan(StackPlan* p, int M, int hd, int n_max) {
    const int NT = xf_nt(M), act = NT * kStackSteps * 512;
    const int small = 256 + (int)((sizeof(StackSmall) + 127) / 128 * 128) + 8 * n_max * 4;    // with the ones in front
    const int attn = n_max * hd * 4 + n_max * 512 + 128;
    int scratch = 2 * act > attn ? 2 * act : attn;
    int slots = (kStackSmemMax - small - scratch) / kStackSlot;
    if (slots < kStackMinSlots) return false;
    if (slots > kStackMaxSlots) slots = kStackMaxSlots;
    scratch = (kStackSmemMax - small - slots * kStackSlot) / 128 * 128;
    p->T = 8 * NT;
    p->slots = slots;
    p->scratch = scratch;
    p->acts = scratch / act > kStackMaxActs ? kStackMaxActs : scratch / act;
    p->p_bufs = scratch >= attn + n_max * 512 ? 2 : 1;
    p->q_bufs = scratch >= attn + (p->p_bufs - 1) * n_max * 512 + n_max * hd * 4 ? 2 : 1;
    p->smem = kStackSmemMax;
    return true;
}
// Exchange words: per CTA and shared row block (two at most) stack_block_rows(...) rows of 128, one for each group it finishes and
// contributor; or partial attention results.
static inline int stack_block_rows(int rows, int KS, int RB, int ctas) {
    int best = 2;
    for (int C = stack_max_share(KS, stack_per(KS, RB, ctas)); C >= 2; --C) {
        const int n = (2 * stack_half_groups(rows, C) + C - 1) / C * C;
        best = n > best ? n : best;
    }
    return best;
}
static inline size_t stack_ll_rows(int rows, int Hq, int Hkv) {
    const int r = rows * (Hq / Hkv) < kStackMaxN ? rows * (Hq / Hkv) : kStackMaxN;
    return (size_t)kStackMaxCtas * r + (size_t)Hq * rows;
}

// ---- waits.  Bounded by counts (a try suspends for a hardware-chosen time, some 4 us: 2^18 of them take a second); a role gives up at its
// first wait that runs out, so that all of them are through within a few of these.
constexpr uint32_t kStackTries = 1u << 18;
__device__ __forceinline__ bool stack_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// A look that never suspends, the same for all lanes.
__device__ __forceinline__ bool stack_look(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return __all_sync(0xffffffffu, ok != 0u);
}
// (a converged warp, whose lanes have to leave with one answer: those that disagreed about a wait that runs out would go separate ways.
// A lane whose tries ran out therefore looks once more, behind the others' last tries: if one of those succeeded, the phase is over and
// this one does too; if none did, they are all here, and one's sight is the others'.  This costs nothing, and a vote behind every
// wait 0.5 %.  The limit is a constant: as an argument it cost 0.8 % of a pass (1b shape, 9 rows 796 -> 803 us, 7b shape 2634 -> 2646).)
__device__ __forceinline__ bool stack_wait(uint32_t bar, uint32_t parity) {
    bool done = false;
#pragma unroll 1
    for (uint32_t it = 0; it < kStackTries; ++it) {
        if (stack_try(bar, parity)) { done = true; break; }
    }
    if (!done) done = __any_sync(__activemask(), stack_try(bar, parity));
    return done;
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Looks that find nothing, a trip to the L2 each, before a reader of other CTAs' words gives up: seconds.
constexpr uint32_t kStackLooks = 1u << 22;
// (a converged warp: one lane looks, and its sight is the others' too)
__device__ __forceinline__ bool stack_arrived(const unsigned* ctr, unsigned target, const volatile int* abort_s, const int* err, int lane, uint32_t looks) {
    uint32_t it = 0;
#pragma unroll 1
    do {
        unsigned v = 0u;
        asm volatile("{\n .reg .pred q;\n setp.eq.s32 q, %2, 0;\n @q ld.acquire.gpu.global.u32 %0, [%1];\n}" : "+r"(v) : "l"(ctr), "r"(lane) : "memory");
        if ((int)(__shfl_sync(0xffffffffu, v, 0) - target) >= 0) return true;
        if ((it & 63u) == 63u && __any_sync(0xffffffffu, *abort_s || ld_relaxed(err) != 0)) return false;
    } while (++it < looks);
    return false;
}
// Orders what this thread has seen of other CTAs' ordinary stores before its later copies from global memory.
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
// Exchange words: three values and the phase number that vouches for them, 16 bytes written and read as one.  These, and ordinary
// accesses, where a condition holds, without a branch: a point that lanes meet again at costs more than the access.
__device__ __forceinline__ void ll_store_if(bool c, uint4* p, float x, float y, float z, unsigned epoch) {
    asm volatile("{\n .reg .pred q;\n .reg .b64 l, h;\n .reg .b128 w;\n setp.ne.u32 q, %5, 0;\n mov.b64 l, {%1, %2};\n mov.b64 h, {%3, %4};\n mov.b128 w, {l, h};\n"
                 " @q st.relaxed.gpu.global.b128 [%0], w;\n}" ::"l"(p), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(__float_as_uint(z)), "r"(epoch), "r"((uint32_t)c)
                 : "memory");
}
__device__ __forceinline__ void ll_load_if(bool c, uint4& v, const uint4* p) {
    asm volatile("{\n .reg .pred q;\n .reg .b64 l, h;\n .reg .b128 w;\n setp.ne.u32 q, %5, 0;\n mov.b64 l, {%0, %1};\n mov.b64 h, {%2, %3};\n mov.b128 w, {l, h};\n"
                 " @q ld.relaxed.gpu.global.b128 w, [%4];\n mov.b128 {l, h}, w;\n mov.b64 {%0, %1}, l;\n mov.b64 {%2, %3}, h;\n}"
                 : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(p), "r"((uint32_t)c) : "memory");
}
__device__ __forceinline__ void st_if(bool c, uint16_t* p, uint16_t v) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.global.b16 [%0], %1;\n}" ::"l"(p), "h"(v), "r"((uint32_t)c) : "memory");
}
__device__ __forceinline__ void st_if(bool c, float* p, float v) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.global.f32 [%0], %1;\n}" ::"l"(p), "f"(v), "r"((uint32_t)c) : "memory");
}
__device__ __forceinline__ float ld_if(bool c, const float* p) {             // from L2: other CTAs wrote it in this launch
    float v;
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n mov.f32 %0, 0f00000000;\n @q ld.global.cg.f32 %0, [%1];\n}" : "=f"(v) : "l"(p), "r"((uint32_t)c) : "memory");
    return v;
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* r) {
    uint32_t u[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]) : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = __uint_as_float(u[i]);
}

// What one lane of a converged warp issues, as predicated instructions: `go` is that lane's.  (A loop that one lane runs by itself
// pays a hundred cycles wherever branches meet again: with two waits, a stage of eight MMAs takes the issuer 658 cycles in a lane's
// own region, 440 in a converged warp; the MMAs themselves take 290.)
__device__ __forceinline__ void umma_bf16_if(uint32_t go, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
                 "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(go)
                 : "memory");
}
__device__ __forceinline__ void umma_bf16_ta_if(uint32_t go, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d_tmem),
                 "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(go)
                 : "memory");
}
__device__ __forceinline__ void umma_commit_if(uint32_t go, uint32_t bar) {
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar), "r"(go) : "memory");
}
__device__ __forceinline__ void tmem_copy_a_if(uint32_t go, uint32_t taddr, uint64_t desc) {
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q tcgen05.cp.cta_group::1.128x256b [%0], %1;\n}" ::"r"(taddr), "l"(desc), "r"(go) : "memory");
}
__device__ __forceinline__ void mbar_arrive_if(uint32_t go, uint32_t bar) {
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n @q mbarrier.arrive.shared::cta.b64 _, [%0];\n}" ::"r"(bar), "r"(go) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx_if(uint32_t go, uint32_t bar, uint32_t bytes) {
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(bar), "r"(bytes), "r"(go) : "memory");
}
// A copy whose bytes the barrier is told of first.
__device__ __forceinline__ void bulk_load_if(uint32_t go, uint32_t dst_smem, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %4, 0;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%3], %2;\n"
        " @q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n}" ::"r"(dst_smem), "l"(src), "r"(bytes), "r"(bar), "r"(go)
        : "memory");
}
__device__ __forceinline__ void bulk_load_hint_if(uint32_t go, uint32_t dst_smem, const void* src, uint32_t bytes, uint32_t bar, uint64_t pol) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%3], %2;\n"
        " @q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;\n}" ::"r"(dst_smem), "l"(src), "r"(bytes),
        "r"(bar), "l"(pol), "r"(go)
        : "memory");
}

// Position in a ring of n slots; `par`: parity of the turn.
struct StackRing {
    int slot;
    uint32_t par;
    __device__ __forceinline__ void step(int n) {
        if (++slot == n) { slot = 0; par ^= 1u; }
    }
    __device__ __forceinline__ void skip(int k, int n) {
        slot += k;
#pragma unroll 1
        while (slot >= n) { slot -= n; par ^= 1u; }
    }
};

// NT: groups of eight rows of the pass (1 to 4).  A constant, so that the MMA's descriptors differ by constants: the issuing warp's
// instructions are what a stage costs it.  (us a pass, with the waits' loops not unrolled, 125 KB of code instead of 170: 7b shape, 9
// rows 2844 -> 2794, 17 rows 3181 -> 3123; 8b shape, 17 rows 3910 -> 3862; 1b shape, 9 rows 888 -> 864.)
template <int NT, int HD>
__global__ void __launch_bounds__(kStackThreads, 1) layer_stack_kernel(const __grid_constant__ StackArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int HG = HD / 8;
    constexpr int kTile = kAttnTile * HD * 2;                 // bytes of a K or V tile
    constexpr int kPerTile = HD == 128 ? 2 : 1;               // ring slots a K/V tile pair takes
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = blockIdx.x, n_cta = gridDim.x;
    constexpr int T = 8 * NT;
    constexpr int act_stage = NT * kStackSteps * 512, act_step = NT * 512;
    unsigned char* ones = smem;
    unsigned char* ring = smem + 256;
    unsigned char* scratch = ring + a.slots * kStackSlot;
    const int small_bytes = (int)((sizeof(StackSmall) + 127) / 128 * 128);
    StackSmall& sm = *reinterpret_cast<StackSmall*>(smem + kStackSmemMax - small_bytes);
    float* wm = reinterpret_cast<float*>(smem + kStackSmemMax - small_bytes - 8 * a.n_max * 4);   // [4][N] maxima per lane quarter
    float* m_ref = wm + 4 * a.n_max;                          // [N] reference score
    float* alpha = m_ref + a.n_max;                           // [N] rescale factor
    const uint32_t ring_a = smem_u32(ring), scratch_a = smem_u32(scratch);
    const int q_bytes = a.n_max * HD * 4;
    unsigned char* p_op = scratch + a.q_bufs * q_bytes;       // P, hi and lo terms
    volatile int* abort_s = &sm.abort;
    const int n_phase = 5 * a.n_layers + (a.want_logits ? 1 : 0);

    if (tid == 0) {
        // an earlier launch gave up and the host has not seen it yet: its results are void, and so would be these
        sm.go = ld_relaxed(a.err) == 0;
        sm.abort = 0;
        sm.base = a.sync[32];
        sm.epoch = a.sync[64];
        sm.issued_w = sm.issued_a = sm.issued_q = 0;
        for (int i = 0; i < kStackMaxSlots; ++i) { mbar_init(smem_u32(&sm.full_w[i]), 1); mbar_init(smem_u32(&sm.empty_w[i]), 1); }
        for (int i = 0; i < kStackMaxActs; ++i) { mbar_init(smem_u32(&sm.full_a[i]), 1); mbar_init(smem_u32(&sm.empty_a[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sm.d_full[i]), 1);
            mbar_init(smem_u32(&sm.d_empty[i]), kStackWorkers / 32);
            mbar_init(smem_u32(&sm.q_full[i]), 1);
            mbar_init(smem_u32(&sm.q_empty[i]), 1);
            mbar_init(smem_u32(&sm.s_full[i]), 1);
            mbar_init(smem_u32(&sm.pv_done[i]), 1);
        }
        mbar_init(smem_u32(&sm.p_full), 1);
        mbar_init(smem_u32(&sm.phase), 1);
        mbar_init(smem_u32(&sm.tables), 1 + kStackWorkers / 32);
        mbar_init(smem_u32(&sm.last), 1);
        fence_mbar_init();
    }
    if (tid >= 64 && tid < 128) reinterpret_cast<uint32_t*>(ones)[tid - 64] = 0x3F803F80u;
    fence_proxy_async_smem();
    if (warp == 2) {
        tmem_alloc(smem_u32(&sm.tmem), 512);
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&sm.tmem);
    const unsigned base = sm.base, epoch0 = sm.epoch;
    unsigned* ctr = a.sync;
    auto give_up = [&](int code) {
        *abort_s = 1;
        atomicExch(a.err, code);
    };
    // units of a projection this CTA takes
    auto range = [&](const StackGemm& g, int& s, int& e) {
        s = min(cta * g.per, g.RB * g.KS);
        e = min(s + g.per, g.RB * g.KS);
    };
    // tensor-memory columns of the attention (the projections' accumulators, columns 0..127, are idle then)
    const uint32_t t_O = tmem + 4u * a.n_max, t_L = tmem + 6u * a.n_max;
    const bool wide_l = a.n_max <= 64;       // denominators of hi and lo terms in columns of their own

    // registers: 104 x 128 threads + 200 x 256, of the 168 x 384 the kernel is launched with
    const bool run = sm.go != 0;             // (the abort flag may be up by the time that a slow warp looks)
    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    if (warp == 0 && run) {
        // ---------------- the copy stream: weights and K/V
        StackRing r = {0, 1u};               // par: of the slot's `empty` phase to wait for
        unsigned issued = 0;
        bool ok = true;
        const uint64_t pol = l2_evict_first_policy();
        StackRing landed = {0, 0u};          // the item that has to be here before another is asked for
        auto slot_free = [&]() {
            ok = stack_wait(smem_u32(&sm.empty_w[r.slot]), r.par);
            if (ok && issued >= kStackInFlight) {
                ok = stack_wait(smem_u32(&sm.full_w[landed.slot]), landed.par);
                landed.step(a.slots);
            }
            return ok;
        };
        auto stream = [&](const StackGemm& g, const unsigned char* w) {
            int s, e;
            range(g, s, e);
            int ks = s % g.KS;
#pragma unroll 1
            while (s < e && ok) {
                const int n = min(min((ks | (kStackSteps - 1)) + 1, g.KS) - ks, e - s);
                if (!slot_free()) break;
                bulk_load_hint_if(lane == 0, ring_a + r.slot * kStackSlot, w + (size_t)s * 4096, (uint32_t)n * 4096u, smem_u32(&sm.full_w[r.slot]), pol);
                ++issued;
                r.step(a.slots);
                s += n;
                ks += n;
                if (ks == g.KS) ks = 0;
            }
        };
        auto stream_kv = [&](int l, unsigned target) {
            if (!stack_wait(smem_u32(&sm.tables), 0u)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            const size_t page_stride = (size_t)2 * a.Hkv * a.page_size * HD, v_off = (size_t)a.Hkv * a.page_size * HD;
            bool fresh = false;              // this layer's new rows are known to be in the cache
#pragma unroll 1
            for (int s = 0; s < sm.n_seg && ok; ++s) {
                const StackSeg& sg = sm.seg[s];
                const uint16_t* kb = a.kv_pool + kv_index(l, a.n_pages, 0, 0, a.Hkv, sg.kvh, a.page_size, 0, HD, 0);
                const int32_t* bt = sg.bt;
                const int k1 = sg.k1;
#pragma unroll 1
                for (int j0 = sg.k0; j0 < k1 && ok; j0 += kAttnTile) {
                    const int je = min(j0 + kAttnTile, k1), j1 = (je + 7) & ~7;
                    if (je > sg.base && !fresh) {
                        ok = stack_arrived(ctr, target, abort_s, a.err, lane, a.looks);
                        if (!ok) break;
                        fence_proxy_async_global();
                        fresh = true;
                    }
                    const int pidx = j0 / a.page_size + lane;
                    const int js = max(j0, pidx * a.page_size), jp = min(j1, (pidx + 1) * a.page_size);
                    const uint16_t* src = nullptr;
                    if (js < jp) src = kb + (size_t)bt[pidx] * page_stride + (size_t)(js - pidx * a.page_size) * HD;
#pragma unroll
                    for (int kv = 0; kv < 2; ++kv) {
                        if (kv == 0 || kPerTile == 2) {
                            if (!slot_free()) break;
                            mbar_expect_tx_if(lane == 0, smem_u32(&sm.full_w[r.slot]), (uint32_t)(j1 - j0) * (HD * 2) * (3 - kPerTile));
                            __syncwarp();
                        }
                        if (src != nullptr)
                            bulk_g2s(ring_a + r.slot * kStackSlot + (kPerTile == 1 ? kv * kTile : 0) + (uint32_t)(js - j0) * (HD * 2), src + kv * v_off,
                                     (uint32_t)(jp - js) * (HD * 2), smem_u32(&sm.full_w[r.slot]));
                        if (kv == 1 || kPerTile == 2) {
                            ++issued;
                            r.step(a.slots);
                        }
                    }
                }
            }
        };
        unsigned target = base + (unsigned)n_cta;
#pragma unroll 1
        for (int l = 0; l < a.n_layers && ok; ++l) {
#pragma unroll 1
            for (int kind = 0; kind < 5 && ok; ++kind, target += (unsigned)n_cta) {
                if (kind == kStAttn) stream_kv(l, target);
                else stream(a.g[kind], a.g[kind].w + (size_t)l * a.layer_stride);
            }
        }
        if (a.want_logits && ok) stream(a.g[kStLm], a.g[kStLm].w);
        if (!ok && lane == 0) give_up(11);
        if (lane == 0) sm.issued_w = issued;
    } else if (warp == 1 && run) {
        // ---------------- dependencies: one thread looks for the other CTAs' arrivals and fetches activations and Q
        {
            const uint32_t go = lane == 0;
            StackRing r = {0, 1u};
            unsigned issued = 0, q_n = 0, target = base + (unsigned)n_cta;
            bool ok = true;
#pragma unroll 1
            for (int p = 0; p < n_phase && ok; ++p, target += (unsigned)n_cta) {
                const int kind = p < 5 * a.n_layers ? p % 5 : (int)kStLm;
                // everything but the look itself comes before it: what follows it is on every phase's critical path
                if (p == 0) ok = stack_wait(smem_u32(&sm.tables), 0u);
                if (kind == kStAttn) {
                    ok = ok && stack_arrived(ctr, target, abort_s, a.err, lane, a.looks);
                    if (!ok) break;
                    fence_proxy_async_global();
#pragma unroll 1
                    for (int s = 0; s < sm.n_seg && ok; ++s, ++q_n) {
                        const StackSeg& sg = sm.seg[s];
                        const unsigned buf = a.q_bufs == 2 ? q_n & 1u : 0u, turn = a.q_bufs == 2 ? q_n >> 1 : q_n;
                        if (s == a.q_bufs) mbar_arrive_if(go, smem_u32(&sm.phase));
                        ok = stack_wait(smem_u32(&sm.q_empty[buf]), (turn & 1u) ^ 1u);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&sm.q_full[buf]), bytes = (uint32_t)(sg.N * HD * 4);
                        bulk_load_if(go, scratch_a + buf * q_bytes, a.qop + sg.q_off, bytes, bar);
                    }
                    if (sm.n_seg <= a.q_bufs) mbar_arrive_if(go, smem_u32(&sm.phase));
                } else {
                    const unsigned char* act = a.g[kind].act;
                    const int KS = a.g[kind].KS, e = sm.geo[kind].e;
                    int s = sm.geo[kind].s, ks = sm.geo[kind].ks;
                    bool told = false;
                    ok = ok && stack_wait(smem_u32(&sm.empty_a[r.slot]), r.par) && stack_arrived(ctr, target, abort_s, a.err, lane, a.looks);
                    if (!ok) break;
                    fence_proxy_async_global();
#pragma unroll 1
                    while (s < e) {
                        const int n = min(min((ks | (kStackSteps - 1)) + 1, KS) - ks, e - s);
                        const uint32_t bar = smem_u32(&sm.full_a[r.slot]);
                        bulk_load_if(go, scratch_a + r.slot * act_stage, act + (size_t)(ks * act_step), (uint32_t)(n * act_step), bar);
                        if (!told) { told = true; mbar_arrive_if(go, smem_u32(&sm.phase)); }
                        ++issued;
                        r.step(a.acts);
                        s += n;
                        ks += n;
                        if (ks == KS) ks = 0;
                        ok = stack_wait(smem_u32(&sm.empty_a[r.slot]), r.par);
                        if (!ok) break;
                    }
                    if (!told) mbar_arrive_if(go, smem_u32(&sm.phase));
                }
            }
            if (!ok && go) give_up(12);
            if (go) {
                sm.issued_a = issued;
                sm.issued_q = q_n;
            }
        }
    } else if (warp == 2 && run) {
        // ---------------- MMA issue (one lane's, by a converged warp)
        {
            const uint32_t go = elect_one();
            StackRing rw = {0, 0u}, ra = {0, 0u}, rd = {0, 1u};     // rd: accumulators, `empty` parity
            unsigned tile = 0, q_n = 0, staged = 0;                 // staged: weights' stages in tensor memory
            bool ok = true;
            constexpr uint32_t idesc = umma_idesc_bf16(128, 16 * NT, 0, 0);
            int put = 0, get = 0;                                   // their places, of kStackStaged
            auto staged_at = [&](int i) { return tmem + 512u - 64u * (uint32_t)(i + 1); };
            auto gemm = [&](const StackGemm& g, int room) -> bool {
                int s, e;
                range(g, s, e);
                int ks = s % g.KS;
                if (s >= e) return true;
                {
                    // The phase opens when its first activations land.  Until then the stages that the ring holds move on to
                    // tensor memory, as far as there is room, and the copy stream goes on into their slots: what is kept on
                    // the chip across a dependency doubles, to about 7 us of HBM.
                    const uint32_t first = smem_u32(&sm.full_a[ra.slot]);
                    if (!stack_wait(smem_u32(&sm.d_empty[rd.slot]), rd.par)) return false;
                    bool open = false;
                    // (looks, not tries: a try on either barrier would sleep through the other's news)
#pragma unroll 1
                    for (uint32_t it = 0; it < (1u << 24) && !open; ++it) {
                        open = stack_look(first, ra.par);
                        if ((it & 1023u) == 1023u && __any_sync(0xffffffffu, *abort_s)) return false;
                        if (!open && (int)staged < room && stack_look(smem_u32(&sm.full_w[rw.slot]), rw.par)) {
                            tc_fence_after();
                            const uint32_t to = staged_at(put);
                            const uint64_t wd = umma_desc(ring_a + rw.slot * kStackSlot, 128, 256);
#pragma unroll
                            for (int k = 0; k < kStackSteps; ++k) tmem_copy_a_if(go, to + 8 * k, wd + (uint64_t)(k * (4096 >> 4)));
                            umma_commit_if(go, smem_u32(&sm.empty_w[rw.slot]));
                            rw.step(a.slots);
                            ++staged;
                            if (++put == kStackStaged) put = 0;
                        }
                    }
                    if (!open) return false;
                }
                bool fresh = true;                       // the first accumulator and activations have been waited for
#pragma unroll 1
                while (s < e) {
                    const int end = min(g.KS, ks + (e - s));         // of this row block's steps here
#pragma unroll 1
                    while (ks < end) {
                        if (!fresh) if (!stack_wait(smem_u32(&sm.d_empty[rd.slot]), rd.par)) return false;
                        const uint32_t d = tmem + 64u * rd.slot;
                        uint32_t acc = 0u;
#pragma unroll 1
                        for (int f = 0; f < g.flush && ks < end; ++f) {
                            const int n = min((ks | (kStackSteps - 1)) + 1, end) - ks;
                            const uint64_t bd = umma_desc(scratch_a + ra.slot * act_stage, 128, 256);
                            constexpr uint64_t bs = act_step >> 4;
                            if (!fresh) if (!stack_wait(smem_u32(&sm.full_a[ra.slot]), ra.par)) return false;
                            fresh = false;
                            if (staged > 0) {
                                tc_fence_after();
                                const uint32_t at = staged_at(get);
                                --staged;
                                if (++get == kStackStaged) get = 0;
                                if (n == kStackSteps) {
#pragma unroll
                                    for (int k = 0; k < kStackSteps; ++k) umma_bf16_ta_if(go, d, at + 8 * k, bd + bs * k, idesc, k > 0 ? 1u : acc);
                                } else {
#pragma unroll 1
                                    for (int k = 0; k < n; ++k) umma_bf16_ta_if(go, d, at + 8 * k, bd + bs * k, idesc, k > 0 ? 1u : acc);
                                }
                            } else {
                                if (!stack_wait(smem_u32(&sm.full_w[rw.slot]), rw.par)) return false;
                                tc_fence_after();
                                const uint64_t wd = umma_desc(ring_a + rw.slot * kStackSlot, 128, 256);
                                if (n == kStackSteps) {
#pragma unroll
                                    for (int k = 0; k < kStackSteps; ++k) umma_bf16_if(go, d, wd + (uint64_t)(k * (4096 >> 4)), bd + bs * k, idesc, k > 0 ? 1u : acc);
                                } else {
#pragma unroll 1
                                    for (int k = 0; k < n; ++k) umma_bf16_if(go, d, wd + (uint64_t)(k * (4096 >> 4)), bd + bs * k, idesc, k > 0 ? 1u : acc);
                                }
                                umma_commit_if(go, smem_u32(&sm.empty_w[rw.slot]));
                                rw.step(a.slots);
                            }
                            acc = 1u;
                            umma_commit_if(go, smem_u32(&sm.empty_a[ra.slot]));
                            ra.step(a.acts);
                            ks += n;
                            s += n;
                        }
                        umma_commit_if(go, smem_u32(&sm.d_full[rd.slot]));
                        rd.step(2);
                    }
                    if (ks == g.KS) ks = 0;
                }
                return true;
            };
            auto attn = [&]() {
                ok = stack_wait(smem_u32(&sm.tables), 0u);
                if (!ok) return;
                const int n_tiles = sm.n_tiles;
                StackRing rk = rw, rv = rw;                          // K of the next first product, V of the next second one
                if (kPerTile == 2) rv.step(a.slots);
                int qs = 0, qj = sm.n_seg > 0 ? sm.seg[0].k0 : 0, ps = 0, pj = qj;
                const uint32_t ones_a = smem_u32(ones), p_a = smem_u32(p_op);
#pragma unroll 1
                for (int i = -1; i < n_tiles && ok; ++i) {
                    if (i + 1 < n_tiles) {
                        const StackSeg& sg = sm.seg[qs];
                        const unsigned buf = a.q_bufs == 2 ? q_n & 1u : 0u, turn = a.q_bufs == 2 ? q_n >> 1 : q_n;
                        if (qj == sg.k0) ok = stack_wait(smem_u32(&sm.q_full[buf]), turn & 1u);
                        if (ok) ok = stack_wait(smem_u32(&sm.full_w[rk.slot]), rk.par);
                        if (!ok) break;
                        tc_fence_after();
                        const unsigned sb = (tile + 1u + (unsigned)i) & 1u;
                        uint64_t kd = umma_desc(ring_a + rk.slot * kStackSlot, 128, HG * 128), qd = umma_desc(scratch_a + buf * q_bytes, 128, HG * 128);
                        const uint32_t id = umma_idesc_bf16(128, 2 * sg.N, 0, 0), d = tmem + sb * 2u * a.n_max;
#pragma unroll 1
                        for (int kk = 0; kk < HD / 16; ++kk) {
                            umma_bf16_if(go, d, kd, qd, id, kk > 0);
                            kd += 256 >> 4;
                            qd += 256 >> 4;
                        }
                        umma_commit_if(go, smem_u32(&sm.s_full[sb]));
                        if (kPerTile == 2) umma_commit_if(go, smem_u32(&sm.empty_w[rk.slot]));
                        rk.skip(kPerTile, a.slots);
                        qj += kAttnTile;
                        if (qj >= sg.k1) {
                            umma_commit_if(go, smem_u32(&sm.q_empty[buf]));
                            ++q_n;
                            ++qs;
                            if (qs < sm.n_seg) qj = sm.seg[qs].k0;
                        }
                    }
                    if (i < 0) continue;
                    const StackSeg& sg = sm.seg[ps];
                    ok = stack_wait(smem_u32(&sm.p_full), (tile + (unsigned)i) & 1u);
                    if (ok) ok = stack_wait(smem_u32(&sm.full_w[rv.slot]), rv.par);
                    if (!ok) break;
                    tc_fence_after();
                    const int NG = sg.N / 8, n16 = (min(kAttnTile, sg.k1 - pj) + 15) / 16, NL = (sg.N + 15) & ~15;
                    const uint32_t id = umma_idesc_bf16(128, 2 * sg.N, 1, 1), idl = wide_l ? id : umma_idesc_bf16(128, NL, 1, 1);
                    uint64_t vd = umma_desc(ring_a + rv.slot * kStackSlot + (kPerTile == 1 ? kTile : 0), HG * 128, 128);
                    uint64_t pd = umma_desc(p_a + (a.p_bufs == 2 ? ((tile + (unsigned)i) & 1u) * (uint32_t)(a.n_max * 512) : 0u), 2 * NG * 128, 128);
                    // the denominators' A operand: 16 keys x 8 rows of ones; the MMA's other 120 rows read whatever follows in
                    // shared memory and land in lanes nobody reads
                    const uint64_t od = umma_desc(ones_a, 128, 256);
                    uint32_t acc = pj > sg.k0 ? 1u : 0u;
#pragma unroll 1
                    for (int k = 0; k < n16; ++k) {
                        umma_bf16_if(go, t_O, vd, pd, id, acc);
                        umma_bf16_if(go, t_L, od, pd, idl, acc);
                        if (!wide_l) umma_bf16_if(go, t_L, od, pd + (uint64_t)((NG * 128) >> 4), idl, 1u);
                        vd += (2 * HG * 128) >> 4;
                        pd += (uint64_t)((4 * NG * 128) >> 4);
                        acc = 1u;
                    }
                    umma_commit_if(go, smem_u32(&sm.pv_done[(tile + (unsigned)i) & 1u]));
                    umma_commit_if(go, smem_u32(&sm.empty_w[rv.slot]));
                    rv.skip(kPerTile, a.slots);
                    pj += kAttnTile;
                    if (pj >= sg.k1) {
                        ++ps;
                        if (ps < sm.n_seg) pj = sm.seg[ps].k0;
                    }
                }
                tile += (unsigned)n_tiles;
                rw.skip(kPerTile * n_tiles, a.slots);
            };
            int n_done = 0;
            bool in_use = false;                                    // the attention's columns
#pragma unroll 1
            for (int p = 0; p < n_phase && ok; ++p, ++n_done) {
                const int kind = p < 5 * a.n_layers ? p % 5 : (int)kStLm;
                umma_commit_if(go, smem_u32(&sm.last));         // no MMA of an earlier phase reads tensor memory that stages move to
                ok = stack_wait(smem_u32(&sm.last), (uint32_t)p & 1u);
                if (!ok) continue;
                if (kind == kStAttn) {
                    attn();
                    if (sm.n_tiles > 0) {
                        put = get = 0;                                   // (none is staged across an attention with tiles)
                        in_use = true;
                    }
                    continue;
                }
                // weights to come before the next K/V tile; tensor memory beside the attention's columns while those are in use
                if (p == 0) ok = stack_wait(smem_u32(&sm.tables), 0u);
                int room = 0;
#pragma unroll 1
                for (int q = kind, i = p; q != kStAttn && i < n_phase; ++i) {
                    room += sm.geo[q].stages;
                    q = q == kStLm ? kStAttn : q == kStDn ? (i + 1 < 5 * a.n_layers ? kStQkv : kStLm) : q + 1;
                    if (q == kStAttn || (kind == kStQkv)) break;
                }
                // (until a phase of which this CTA has a part has opened: where it has none of the output projection, this role is
                // in the next phase while the workers are still in the attention)
                const int beside = in_use ? min((512 - 8 * a.n_max) / 64, kStackStaged) : kStackStaged;
                ok = gemm(a.g[kind], min(room, max(beside, 0)));
                if (sm.geo[kind].stages > 0) in_use = false;
            }
            if (!ok && go) give_up(13);
            // nothing of this CTA runs on the tensor cores when it leaves (one commit after the other: a wait for the newer one alone
            // would be satisfied by the phase before an older one that ran out)
            if (n_done > 0) stack_wait(smem_u32(&sm.last), (uint32_t)(n_done - 1) & 1u);
            umma_commit_if(go, smem_u32(&sm.last));
            stack_wait(smem_u32(&sm.last), (uint32_t)n_done & 1u);
        }
    } else if (warp == 3 && run) {
        // ---------------- tables, once: rows, requests, and this CTA's segments of the line of keys
        const int G = a.Hq / a.Hkv;
        int rows = 0, kb = 0;
        if (lane < a.n_items) { rows = a.meta.it_rows[lane]; kb = a.meta.it_base[lane]; }
        // Units of 16 keys per KV head, `per` of them a CTA's; at least 64 keys: shorter parts would only add partial results to
        // exchange.  If ranges up to a quarter longer let every range end with its head (so that a CTA has one part), heads are padded
        // to whole ranges: a second part costs a CTA two to three us, a tile 1.5.  (us a pass, 9 rows: 1b shape, 512 keys 866 -> 798, 7b
        // shape, 2048 keys 2836 -> 2798; 8b shape, 17 rows and 8192 keys 3892 -> 3713.)
        int units = (kb + rows + 15) / 16;
        int per = max((a.Hkv * (int)__reduce_add_sync(0xffffffffu, (unsigned)units) + n_cta - 1) / n_cta, 4);
#pragma unroll 1
        for (int longer = per; longer <= per + per / 4; ++longer) {
            if (a.Hkv * (int)__reduce_add_sync(0xffffffffu, (unsigned)((units + longer - 1) / longer)) > n_cta) continue;
            per = longer;
            units = (units + per - 1) / per * per;
            break;
        }
        const int N = (G * rows + 7) & ~7;
        int u0 = a.Hkv * units, q0 = a.Hkv * N * HD * 2, rs = a.Hkv * G * rows;      // inclusive sums over the items
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, u0, o), y = __shfl_up_sync(0xffffffffu, q0, o), z = __shfl_up_sync(0xffffffffu, rs, o);
            if (lane >= o) { u0 += x; q0 += y; rs += z; }
        }
        const int U = __shfl_sync(0xffffffffu, u0, 31);
        if (lane < a.n_items) {
            StackItem& it = sm.it[lane];
            it.base = kb; it.rows = rows; it.units = units; it.N = N;
            it.u0 = u0 - a.Hkv * units;
            it.q0 = (unsigned)(q0 - a.Hkv * N * HD * 2);
            it.rowsum = rs - a.Hkv * G * rows;
            it.row0 = a.meta.it_row0[lane];
            it.slot = a.meta.it_slot[lane];
        }
        __syncwarp();
        if (lane < a.M) {
            const int item = a.meta.row_item[lane], pos = a.meta.row_pos[lane];
            const int page = a.meta.block_tab[(size_t)sm.it[item].slot * a.meta.max_pages + pos / a.page_size];
            sm.kvoff[lane] = (long long)kv_index(0, a.n_pages, page, 0, a.Hkv, 0, a.page_size, pos % a.page_size, HD, 0);
            sm.q_off[lane] = sm.it[item].q0;
            sm.q_N[lane] = sm.it[item].N;
            sm.q_r[lane] = lane - sm.it[item].row0;
        }
        if (lane == 0) {
            int u = min(cta * per, U), n = 0, tiles = 0, i = 0;
            const int e = min(u + per, U);
            while (u < e && n < kStackMaxSegs) {
                while (i + 1 < a.n_items && u >= sm.it[i + 1].u0) ++i;
                const StackItem& it = sm.it[i];
                const int h = (u - it.u0) / it.units, off = u - it.u0 - h * it.units, len = min(it.units - off, e - u);
                const int hs = it.u0 + h * it.units, first = hs / per, last = (hs + it.units - 1) / per, R = G * it.rows;
                StackSeg& sg = sm.seg[n++];
                sg.kvh = h;
                sg.k0 = off * 16;
                sg.k1 = min((off + len) * 16, it.base + it.rows);
                sg.base = it.base;
                sg.n_rows = R;
                sg.N = it.N;
                sg.row0 = it.row0;
                sg.C = last - first + 1;
                sg.idx = cta - first;
                sg.ll0 = first * a.r_max + it.rowsum + h * R;
                sg.q_off = it.q0 + (unsigned)(h * it.N * HD * 2);
                sg.bt = a.meta.block_tab + (size_t)it.slot * a.meta.max_pages;
                tiles += (sg.k1 - sg.k0 + kAttnTile - 1) / kAttnTile;
                u += len;
            }
            // last first: a segment that ends with this pass's own keys then comes behind those that do not wait for them
            for (int k = 0; k < n / 2; ++k) {
                const StackSeg t = sm.seg[k];
                sm.seg[k] = sm.seg[n - 1 - k];
                sm.seg[n - 1 - k] = t;
            }
            sm.n_seg = n;
            sm.n_tiles = tiles;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.tables));
        asm volatile("bar.arrive 2, %0;" ::"n"(32 + kStackWorkers) : "memory");
    }
    } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    if (run) {
        // ---------------- workers: accumulators, epilogues, softmax, merges
        const int wt = tid - 128, quarter = warp & 3, half = (warp - 4) >> 2;
        const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
        const int G = a.Hq / a.Hkv;
        bool ok = true;
        auto sync_workers = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kStackWorkers) : "memory"); };
        uint32_t tries = kStackTries;         // one, once a wait has run out
        auto wait = [&](unsigned long long& bar, uint32_t parity) {
            bool done = false;
#pragma unroll 1
            for (uint32_t it = 0; it < tries; ++it) {
                if (stack_try(smem_u32(&bar), parity)) { done = true; break; }
            }
            if (!__all_sync(0xffffffffu, done)) {
                if (ok && lane == 0) give_up(14);
                tries = 1u;
                ok = false;
            }
        };
        // between two looks at other CTAs' words: false once it is time to give up (the whole warp)
        auto look_on = [&](uint32_t look) {
            if (ok && (look & 63u) == 63u && __any_sync(0xffffffffu, *abort_s || ld_relaxed(a.err) != 0 || look >= a.looks)) {
                ok = false;
                if (lane == 0) give_up(15);
            }
            return ok;
        };
        auto arrive_grid = [&]() {
            sync_workers();                   // (the fence between these stores and the copies that read them is the reader's)
            if (wt == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(ctr), "r"(1u) : "memory");
        };
        // one element of a projection's input: k-th column of row t
        auto act_put = [&](bool live, uint16_t* dst, int t, int k, float v) {
            uint16_t h, l;
            split_bf16(v, h, l);
            uint16_t* p = dst + (k >> 4) * (T * 32) + ((t >> 3) * 2 + ((k >> 3) & 1)) * 64 + (t & 7) * 8 + (k & 7);
            st_if(live, p, h);
            st_if(live, p + T * 16, l);
        };

        // ---- this CTA's part of the projections, one per warp
        if (warp - 4 < 6 && warp - 4 != kStAttn && a.g[warp - 4].KS > 0) {
            const int kind = warp - 4;
            const StackGemm& g = a.g[kind];
            const int KS = g.KS, per = g.per;
            int s, e;
            range(g, s, e);
            const int b0 = s / KS, b1 = s < e ? (e - 1) / KS : b0;
            StackGeo& geo = sm.geo[kind];
            int n0 = 0, n1 = 0;
#pragma unroll 1
            for (int w = 0; w < 2; ++w) {
                const int rb = w == 0 ? b0 : b1, first = rb * KS / per, C = (rb * KS + KS - 1) / per - first + 1;
                if (s >= e || C < 2 || (w == 1 && b1 == b0)) continue;
                const int gs = stack_group(a.M, C), nq = stack_half_groups(a.M, C), idx = cta - first, mh = stack_half_rows(a.M);
                // lane = group; for the first contributor the block may be the second of its two
                const int h = lane >= nq ? 1 : 0, q = lane - h * nq, t = h * mh + q * gs, n = min(gs, (h ? a.M : mh) - t);
                const int k = lane / C, o = lane - k * C, to = (first + o) * 2 + (o == 0 && first * per / KS != rb ? 1 : 0);
                const int at = to * a.ll_rows + k * C;
                const bool live = lane < 2 * nq && n > 0, mine = live && o == idx;
                if (lane < 2 * nq) sm.snd[kind][w][h][q] = at + idx;
                const unsigned m0 = __ballot_sync(0xffffffffu, mine && !(k & 1)), m1 = __ballot_sync(0xffffffffu, mine && (k & 1));
                if (mine) sm.ent[kind][k & 1][((k & 1) ? n1 : n0) + __popc(((k & 1) ? m1 : m0) & ((1u << lane) - 1u))] = StackEnt{at, C, w, t, n};
                n0 += __popc(m0);
                n1 += __popc(m1);
            }
            if (lane == 0) {
                int stages = 0;
                for (int i = s; i < e;) {
                    const int ks = i % KS, end = min(KS, ks + (e - i));
                    stages += (end - 1) / kStackSteps - ks / kStackSteps + 1;
                    i += end - ks;
                }
                geo = StackGeo{s, e, b0, s - b0 * KS, stages % a.slots, (stages / a.slots) & 1, stages, {n0, n1}, b1};
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.tables));
        // ---- embedding rows (a CTA's first is its only one where there are as many CTAs), rotary table, zeros behind the live rows
        // of Q
#pragma unroll 1
        for (int row = cta; row < a.M; row += n_cta) {
            const uint16_t* er = a.emb + (size_t)a.meta.row_tok[row] * a.d;
            float ss = 0.f;
#pragma unroll 1
            for (int e = wt * 4; e < a.d; e += kStackWorkers * 4) {
                const uint2 b = *reinterpret_cast<const uint2*>(er + e);
                const float4 v = make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u), __uint_as_float(b.y << 16),
                                             __uint_as_float(b.y & 0xffff0000u));
                *reinterpret_cast<float4*>(a.x + (size_t)row * a.d + e) = v;
                ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
                const float4 g = *reinterpret_cast<const float4*>(a.n1 + e);
                uint16_t* xd = a.act_h + act_index_row(row, e >> 4, a.d / 16, 0, T) + act_index_col(e & 15, 0, T);
                uint2 h, lo;
                split_bf16x2(v.x * g.x, v.y * g.y, h.x, lo.x);
                split_bf16x2(v.z * g.z, v.w * g.w, h.y, lo.y);
                *reinterpret_cast<uint2*>(xd) = h;
                *reinterpret_cast<uint2*>(xd + act_index_lo(T)) = lo;
            }
            ss = warp_sum(ss);
            if (row != cta) sync_workers();      // the row before has been summed
            if (lane == 0) sm.red[warp - 4] = ss;
            sync_workers();
#pragma unroll 1
            for (int i = wt; i < a.n_ssq; i += kStackWorkers) {
                float t = 0.f;
                if (i == 0) {
#pragma unroll
                    for (int w = 0; w < kStackWorkers / 32; ++w) t += sm.red[w];
                }
                a.ssq_a[(size_t)row * a.n_ssq + i] = t;
            }
        }
#pragma unroll 1
        for (int i = (n_cta - 1 - cta) * kStackWorkers + wt; i < a.M * (HD / 2); i += n_cta * kStackWorkers) {
            const double ang = (double)a.meta.row_pos[i / (HD / 2)] * exp(-2.0 * (double)(i % (HD / 2)) / (double)HD * a.log_base);
            double s, c;
            sincos(ang, &s, &c);
            a.cs[i] = (float)c;
            a.sn[i] = (float)s;
        }
#pragma unroll 1
        for (size_t i = (size_t)cta * kStackWorkers + wt; i < a.qop_bytes / 16; i += (size_t)n_cta * kStackWorkers)
            reinterpret_cast<uint4*>(a.qop)[i] = make_uint4(0u, 0u, 0u, 0u);
        arrive_grid();
        // (a barrier and not a wait that may run out: workers go on after one that did, and where they store follows from the tables)
        asm volatile("bar.sync 2, %0;" ::"n"(32 + kStackWorkers) : "memory");

        StackRing rw = {0, 0u}, rd = {0, 0u};
        unsigned tile = 0;
        const float q_scale = rsqrtf((float)HD) * 1.4426950408889634f;   // scores in the log2 domain: p = 2^(s - m)

        // ---- a projection
        auto gemm = [&](int kind, int l, unsigned epoch) {
            const StackGemm& g = a.g[kind];
            const int KS = g.KS;
            const bool normed = kind == kStQkv || kind == kStGu || kind == kStLm;
            if (normed) {
                const float* ssq = kind == kStGu ? a.ssq_b : a.ssq_a;
#pragma unroll 1
                for (int t = warp - 4; t < a.M; t += kStackWorkers / 32) {
                    float s = 0.f;
#pragma unroll 4
                    for (int i = lane; i < a.n_ssq; i += 32) s += __ldcg(ssq + (size_t)t * a.n_ssq + i);
                    s = warp_sum(s);
                    if (lane == 0) sm.rstd[t] = rsqrtf(s / (float)a.d + a.eps);
                }
                sync_workers();
            }
            const int in_tile = (quarter * 32 + lane) & 15;              // row of its 16-row tile
            struct Row { int rb, head, at; float gain; };                // a worker's row of a row block
            auto row_of = [&](int b) {
                const int pr = b * 128 + quarter * 32 + lane;
                Row r = {b, 0, 0, 0.f};
                if (kind == kStQkv) {
                    const int lr = qkv_logical_row(pr, HD), head = lr / HD, dim = lr % HD;
                    r.head = head;
                    if (head < a.Hq) {
                        const int kvh = head / G;
                        r.at = kvh << 16 | (head - kvh * G) << 8 | dim;
                    } else {
                        const int kv = head < a.Hq + a.Hkv ? 0 : 1, kvh = head - a.Hq - kv * a.Hkv;
                        r.at = (kv * a.Hkv + kvh) * a.page_size * HD + (int)kv_col_offset(dim);
                    }
                } else if (kind == kStO || kind == kStDn) {
                    const float* gp = kind == kStO ? reinterpret_cast<const float*>(reinterpret_cast<const char*>(a.n2) + (size_t)l * a.layer_stride)
                                      : l + 1 < a.n_layers ? reinterpret_cast<const float*>(reinterpret_cast<const char*>(a.n1) + (size_t)(l + 1) * a.layer_stride)
                                                           : a.final_norm;
                    r.gain = pr < g.N ? gp[pr] : 0.f;
                }
                return r;
            };
            // what the epilogue needs from memory besides the sum
            auto fetch = [&](bool want, const Row& r, int t, float& xa, float& xb) {
                if (kind == kStQkv) {
                    const int j = t * (HD / 2) + (qkv_logical_row(quarter * 32 + lane, HD) & (HD / 2 - 1));
                    xa = ld_if(want, a.cs + j);
                    xb = ld_if(want, a.sn + j);
                } else if (kind == kStO || kind == kStDn) {
                    const int pr = r.rb * 128 + quarter * 32 + lane;
                    xa = ld_if(want && pr < g.N, a.x + (size_t)t * a.d + pr);
                }
            };
            auto finish = [&](const Row& r, int t, float v, float xa, float xb) {
                const int pr = r.rb * 128 + quarter * 32 + lane;
                const bool live = pr < g.N;
                if (normed) v *= sm.rstd[t];
                if (kind == kStLm) {
                    st_if(live, a.logits + (size_t)t * g.N + pr, v);
                } else if (kind == kStO || kind == kStDn) {
                    xa = live ? xa + v : 0.f;
                    st_if(live, a.x + (size_t)t * a.d + pr, xa);
                    act_put(live, a.act_h, t, pr, xa * r.gain);
                    const float q = warp_sum(xa * xa);
                    st_if(lane == 0, (kind == kStO ? a.ssq_b : a.ssq_a) + t * a.n_ssq + r.rb * 4 + quarter, q);
                } else if (kind == kStGu) {
                    const float up = __shfl_xor_sync(0xffffffffu, v, 8);
                    act_put(live && in_tile < 8, a.act_ffn, t, gu_feature(pr), v / (1.f + expf(-v)) * up);
                } else {
                    const float partner = __shfl_xor_sync(0xffffffffu, v, 8);
                    const float turned = v * xa + (in_tile < 8 ? -partner : partner) * xb;
                    v = r.head < a.Hq + a.Hkv ? turned : v;
                    // queries: operand order of the scores' MMA, hi and lo terms
                    const int n = sm.q_r[t] * G + (r.at >> 8 & 255), N = sm.q_N[t], dim = r.at & 255;
                    const bool query = r.head < a.Hq;
                    uint16_t h, lo;
                    split_bf16(v * q_scale, h, lo);
                    uint16_t* p = a.qop + sm.q_off[t] + (r.at >> 16) * N * HD * 2 + ((n >> 3) * HG + (dim >> 3)) * 64 + (n & 7) * 8 + (dim & 7);
                    st_if(live && query, p, h);
                    st_if(live && query, p + N * HD, lo);
                    st_if(live && !query, a.kv_pool + (size_t)l * a.n_pages * 2 * a.Hkv * a.page_size * HD + (size_t)sm.kvoff[t] + r.at, f32_to_bf16_bits(v));
                }
            };

            const StackGeo& geo = sm.geo[kind];
            const int e = geo.e, n_ent = geo.n_ent[half], mh = stack_half_rows(a.M), t_half = half * mh, n_half = half ? a.M - mh : mh;
            int s = geo.s, b = geo.b, ks = geo.ks, i = 0;
            const StackEnt* ent = sm.ent[kind][half];
            const Row row0 = row_of(b), row1 = row_of(geo.second);
            auto row_sel = [&](int w) { return Row{w ? row1.rb : row0.rb, w ? row1.head : row0.head, w ? row1.at : row0.at, w ? row1.gain : row0.gain}; };
            // the first two groups' inputs are on their way before they are needed
            float xa[6], xb[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                xa[k] = xb[k] = 0.f;
                const int q = k / 3;
                fetch(q < n_ent && k - 3 * q < ent[q].n, row_sel(ent[q].w), ent[q].t + k - 3 * q, xa[k], xb[k]);
            }
            constexpr int kVals = 4 * NT > 6 ? 4 * NT : 6;
#pragma unroll 1
            for (;;) {
                // either a row block of which all K is here, or two groups of shared ones: rows t .. t + n - 1 of `row`, then of `rowb`
                float val[kVals];
                Row row, rowb;
                int t, n, tb = 0, nb = 0, gap = kVals;
                bool ready = false;
                if (s < e) {
                    const int end = min(KS, ks + (e - s));
                    const int stages = (end - 1) / kStackSteps - ks / kStackSteps + 1;
#pragma unroll
                    for (int k = 0; k < kVals; ++k) val[k] = 0.f;
#pragma unroll 1
                    for (int st = 0; st < stages; st += g.flush) {
                        wait(sm.d_full[rd.slot], rd.par);
                        tc_fence_after();
                        const uint32_t d = tmem + 64u * rd.slot + lane_sel + (uint32_t)t_half;
                        float hi[4 * NT], lo[4 * NT];
#pragma unroll
                        for (int k = 0; k < NT; ++k) {
                            tmem_ld4(d + 4 * k, hi + 4 * k);
                            tmem_ld4(d + 8 * NT + 4 * k, lo + 4 * k);
                        }
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int k = 0; k < 4 * NT; ++k) {
                            asm volatile("" : "+f"(hi[k]), "+f"(lo[k]));            // not read ahead of the wait
                            val[k] += hi[k] + lo[k];
                        }
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&sm.d_empty[rd.slot]));
                        rd.step(2);
                    }
                    const int len = end - ks;
                    const int w = s == geo.s ? 0 : 1, bb = b;
                    s += len;
                    ks = 0;
                    ++b;
                    if (len < KS) {
                        // a part of K: the groups go to the CTAs that finish them
                        const int first = bb * KS / g.per, gs = stack_group(a.M, (bb * KS + KS - 1) / g.per - first + 1);
                        const int* to = sm.snd[kind][w][half];
                        uint4* p = a.ll + quarter * 32 + lane;
                        if (gs == 1) {
#pragma unroll
                            for (int k = 0; k < 4 * NT; ++k) ll_store_if(k < n_half, p + (size_t)to[k] * 128, val[k], 0.f, 0.f, epoch);
                        } else if (gs == 2) {
#pragma unroll
                            for (int k = 0; k < 4 * NT; k += 2) ll_store_if(k < n_half, p + (size_t)to[k / 2] * 128, val[k], val[k + 1], 0.f, epoch);
                        } else {
#pragma unroll
                            for (int k = 0; k < 4 * NT; k += 3)
                                ll_store_if(k < n_half, p + (size_t)to[k / 3] * 128, val[k], k + 1 < 4 * NT ? val[k + 1 < 4 * NT ? k + 1 : 0] : 0.f,
                                            k + 2 < 4 * NT ? val[k + 2 < 4 * NT ? k + 2 : 0] : 0.f, epoch);
                        }
                        continue;
                    }
                    row = row_of(bb);
                    t = t_half;
                    n = n_half;
                } else if (i < n_ent) {
                    const StackEnt ea = ent[i], eb = i + 1 < n_ent ? ent[i + 1] : StackEnt{0, 0, 0, 0, 0};
                    const uint4* pa = a.ll + (size_t)ea.off * 128 + quarter * 32 + lane;
                    const uint4* pb = a.ll + (size_t)eb.off * 128 + quarter * 32 + lane;
#pragma unroll
                    for (int k = 0; k < kVals; ++k) val[k] = 0.f;
                    const int c_max = max(ea.C, eb.C);
#pragma unroll 1
                    for (int j0 = 0; j0 < c_max; j0 += 8, pa += 8 * 128, pb += 8 * 128) {
                        uint4 va[8], vb[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            va[u] = make_uint4(0u, 0u, 0u, j0 + u < ea.C ? ~epoch : epoch);
                            vb[u] = make_uint4(0u, 0u, 0u, j0 + u < eb.C ? ~epoch : epoch);
                        }
#pragma unroll 1
                        for (uint32_t look = 0;; ++look) {
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                ll_load_if(va[u].w != epoch, va[u], pa + u * 128);
                                ll_load_if(vb[u].w != epoch, vb[u], pb + u * 128);
                            }
                            bool stale = false;
#pragma unroll
                            for (int u = 0; u < 8; ++u) stale |= va[u].w != epoch || vb[u].w != epoch;
                            if (!__any_sync(0xffffffffu, stale)) break;
                            if (!look_on(look)) break;
                        }
                        // the partial sums in CTA order, as a tree of pairs (absent ones are zero)
                        auto sum8 = [](unsigned x0, unsigned x1, unsigned x2, unsigned x3, unsigned x4, unsigned x5, unsigned x6, unsigned x7) {
                            return ((__uint_as_float(x0) + __uint_as_float(x1)) + (__uint_as_float(x2) + __uint_as_float(x3))) +
                                   ((__uint_as_float(x4) + __uint_as_float(x5)) + (__uint_as_float(x6) + __uint_as_float(x7)));
                        };
                        val[0] += sum8(va[0].x, va[1].x, va[2].x, va[3].x, va[4].x, va[5].x, va[6].x, va[7].x);
                        val[1] += sum8(va[0].y, va[1].y, va[2].y, va[3].y, va[4].y, va[5].y, va[6].y, va[7].y);
                        val[2] += sum8(va[0].z, va[1].z, va[2].z, va[3].z, va[4].z, va[5].z, va[6].z, va[7].z);
                        val[3] += sum8(vb[0].x, vb[1].x, vb[2].x, vb[3].x, vb[4].x, vb[5].x, vb[6].x, vb[7].x);
                        val[4] += sum8(vb[0].y, vb[1].y, vb[2].y, vb[3].y, vb[4].y, vb[5].y, vb[6].y, vb[7].y);
                        val[5] += sum8(vb[0].z, vb[1].z, vb[2].z, vb[3].z, vb[4].z, vb[5].z, vb[6].z, vb[7].z);
                    }
                    row = row_sel(ea.w);
                    rowb = row_sel(eb.w);
                    t = ea.t;
                    n = ea.n;
                    tb = eb.t;
                    nb = eb.n;
                    gap = 3;
                    ready = i == 0;
                    i += 2;
                } else {
                    break;
                }
#pragma unroll 1
                for (int k = 0; n > 0; ++k) {
                    // (rows that nothing was fetched for: a row block that is this CTA's alone comes before the groups, whose inputs stay
                    // in xa, xb meanwhile)
                    float fa = xa[0], fb = xb[0];
                    if (!ready) fetch(true, row, t, fa, fb);
                    finish(row, t, val[0], fa, fb);
                    ++t;
                    int by = 1;
                    if (--n == 0 && gap == 3) {             // on to the second group
                        by = 3 - k;
                        gap = kVals;
                        row = rowb;
                        t = tb;
                        n = nb;
                    }
#pragma unroll 1
                    for (; by > 0; --by) {
#pragma unroll
                        for (int m = 0; m + 1 < kVals; ++m) val[m] = val[m + 1];
#pragma unroll
                        for (int m = 0; m < 5; ++m) { xa[m] = ready ? xa[m + 1] : xa[m]; xb[m] = ready ? xb[m + 1] : xb[m]; }
                    }
                }
            }
            rw.skip(geo.ring, a.slots);
            rw.par ^= (uint32_t)geo.flip;
        };

        // ---- attention: this CTA's segments, then its share of their merges
        auto attn = [&](unsigned epoch) {
            constexpr int kGroups = kStackWorkers / HD;
            const int kt = quarter * 32 + lane;                         // key within the tile; head dimension of O^T
            const int n_seg = sm.n_seg;
            auto product_done = [&](unsigned t) { wait(sm.pv_done[t & 1u], (t >> 1) & 1u); };       // second product of tile t
            StackRing rv = rw;                                          // V of the next tile
            if (kPerTile == 2 && n_seg > 0) rv.step(a.slots);
#pragma unroll 1
            for (int s = 0; s < n_seg; ++s) {
                const StackSeg& sg = sm.seg[s];
                const int N = sg.N, NG = N / 8, n_rows = sg.n_rows, k0 = sg.k0, k1 = sg.k1, kbase = sg.base;
                // eight columns of rows' hi terms and of their lo terms, N further on, added
                auto read_8 = [&](uint32_t at, float (&v)[8]) {
                    float lo[8];
                    tmem_ld8(at, v);
                    tmem_ld8(at + (uint32_t)N, lo);
                    tmem_ld_wait8(v);
                    tmem_ld_wait8(lo);
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] += lo[i];
                };
                // -inf where this thread's key is hidden from a row: rows are numbered (row of the request, query head), and a
                // row sees the keys up to its own
                auto hide = [&](float (&v)[8], int cu, int j) {
                    const int sees = j < k1 ? max(j - kbase, 0) * G : 0x7fffffff;         // the first row that sees key j
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] = cu * 8 + i >= sees ? v[i] : -INFINITY;
                };
#pragma unroll 1
                for (int j0 = k0; j0 < k1; j0 += kAttnTile, ++tile) {
                    const int j = j0 + kt, n_valid = min(kAttnTile, k1 - j0);
                    const uint32_t t_S = tmem + (tile & 1u) * 2u * a.n_max;
                    unsigned char* p_t = p_op + (a.p_bufs == 2 ? (tile & 1u) * (uint32_t)(a.n_max * 512) : 0u);
                    wait(sm.s_full[tile & 1u], (tile >> 1) & 1u);
                    tc_fence_after();
                    const bool need_mask = j0 + kAttnTile - 1 > kbase || n_valid < kAttnTile;
                    if (j0 == k0) {
                        // a row's reference: the score of the segment's first key; +inf, beside which every p is 0, where the row
                        // does not see that key (and so none).  A padding row's scores are 0, and it sees what the last row sees.
                        if (quarter == 0) {
#pragma unroll 1
                            for (int cu = half; cu < NG; cu += 2) {
                                float sc[8];
                                read_8(t_S + cu * 8, sc);
                                if (need_mask) hide(sc, cu, j0);
                                if (lane == 0) {
#pragma unroll
                                    for (int i = 0; i < 8; ++i) m_ref[cu * 8 + i] = sc[i] == -INFINITY ? INFINITY : sc[i];
                                }
                            }
                        }
                        sync_workers();
                    }
                    // the second product that read this place has: the tile before, or the one before that
                    if (j0 > k0 + (a.p_bufs - 1) * kAttnTile) product_done(tile - (unsigned)a.p_bufs);
                    tc_fence_after();
#pragma unroll 1
                    for (int again = 0;; ++again) {
                        float most = -INFINITY;
#pragma unroll 1
                        for (int cu = half; cu < NG; cu += 2) {
                            float sc[8], mr[8];
                            uint32_t hw[4], lw[4];
                            read_8(t_S + lane_sel + cu * 8, sc);
                            *reinterpret_cast<float4*>(mr) = *reinterpret_cast<const float4*>(m_ref + cu * 8);
                            *reinterpret_cast<float4*>(mr + 4) = *reinterpret_cast<const float4*>(m_ref + cu * 8 + 4);
                            if (need_mask) hide(sc, cu, j);
#pragma unroll
                            for (int i = 0; i < 8; i += 2) {
                                const float x0 = sc[i] - mr[i], x1 = sc[i + 1] - mr[i + 1];          // hidden: -inf, p = 0
                                most = fmaxf(most, fmaxf(x0, x1));
                                split_bf16x2(fast_exp2(x0), fast_exp2(x1), hw[i >> 1], lw[i >> 1]);
                            }
                            const uint32_t off = (uint32_t)((((kt >> 3) * 2 * NG + cu) * 8 + (kt & 7)) * 16);
                            *reinterpret_cast<uint4*>(p_t + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                            *reinterpret_cast<uint4*>(p_t + off + NG * 128) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                        }
                        // V rows at and beyond the segment's end must be finite (P is 0 there, but 0 * NaN is not): cleared once
                        // the tile's V rows have landed
                        if (n_valid < kAttnTile) {
                            wait(sm.full_w[rv.slot], rv.par);
                            if (half == 0 && kt >= n_valid && kt < ((n_valid + 15) & ~15)) {
                                unsigned char* v_tile = ring + rv.slot * kStackSlot + (kPerTile == 1 ? kTile : 0);
#pragma unroll 1
                                for (int gr = 0; gr < HG; ++gr)
                                    *reinterpret_cast<uint4*>(v_tile + ((kt >> 3) * HG + gr) * 128 + (kt & 7) * 16) = make_uint4(0, 0, 0, 0);
                            }
                        }
                        fence_proxy_async_smem();
                        tc_fence_before();
                        if (!attn_workers_any(most > kAttnMaxExcess && again == 0)) break;
                        // ---- rare: references move up to the tile's maxima, what has been summed is rescaled, P written again
                        if (a.p_bufs == 2 && j0 > k0) product_done(tile - 1u);           // O^T and L are at rest
#pragma unroll 1
                        for (int cu = half; cu < NG; cu += 2) {
                            float sc[8];
                            read_8(t_S + lane_sel + cu * 8, sc);
                            if (need_mask) hide(sc, cu, j);
                            float mine = -INFINITY;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const float wmax = warp_max_redux(sc[i]);
                                if (lane == i) mine = wmax;
                            }
                            if (lane < 8) wm[quarter * N + cu * 8 + lane] = mine;
                        }
                        sync_workers();
                        if (wt < N) {
                            const float tmax = fmaxf(fmaxf(wm[wt], wm[N + wt]), fmaxf(wm[2 * N + wt], wm[3 * N + wt]));
                            const float m_old = m_ref[wt];
                            const bool none = m_old == INFINITY || !(tmax > m_old);           // (a row that sees no key keeps seeing none)
                            m_ref[wt] = none ? m_old : tmax;
                            alpha[wt] = none ? 1.f : fast_exp2(m_old - tmax);
                        }
                        sync_workers();
                        if (j0 > k0) {
                            auto rescale = [&](uint32_t at, int cols) {                       // columns: rows' hi, then lo terms
#pragma unroll 1
                                for (int cb = half; cb < cols / 8; cb += 2) {
                                    float o[8];
                                    tmem_ld8(at + lane_sel + cb * 8, o);
                                    tmem_ld_wait8(o);
#pragma unroll
                                    for (int i = 0; i < 8; ++i) o[i] *= alpha[(cb % NG) * 8 + i];
                                    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(at + lane_sel + cb * 8),
                                                 "r"(__float_as_uint(o[0])), "r"(__float_as_uint(o[1])), "r"(__float_as_uint(o[2])),
                                                 "r"(__float_as_uint(o[3])), "r"(__float_as_uint(o[4])), "r"(__float_as_uint(o[5])),
                                                 "r"(__float_as_uint(o[6])), "r"(__float_as_uint(o[7]))
                                                 : "memory");
                                }
                            };
#pragma unroll 1
                            for (int z = 0; z < 2; ++z) rescale(z ? t_L : t_O, z == 0 || wide_l ? 2 * N : N);
                            tmem_st_wait();
                            tc_fence_before();
                            sync_workers();
                        }
                    }
                    if (wt == 0) mbar_arrive(smem_u32(&sm.p_full));
                    rv.skip(kPerTile, a.slots);
                }
                // ---- the result of this range: thread = head dimension of O^T; the denominators are the same in lanes 0-7 of L.  A head
                // whose keys are all here is finished; of others, the contributors exchange partial results.  (The reciprocal, as in the
                // merges, rounds 2^-24 of the value; the terms that are stored keep 2^-17.  Through the exchange, a head of one's own took its CTA a trip to the L2 per eight rows, four at 128 dimensions: prompts of 24 to
                // 32 tokens at d_model 512 to 1024 were up to 13 % slower than with a kernel per projection.)
                product_done(tile - 1u);
                tc_fence_after();
                const int ll_row = sg.ll0 + sg.idx * a.r_max;
                const bool alone = sg.C == 1, pairs = n_rows > kGroups * sg.C;
                if (quarter == 0) {
#pragma unroll 1
                    for (int cb = half; cb < NG; cb += 2) {
                        float o[8];
                        if (wide_l) {
                            read_8(t_L + cb * 8, o);
                        } else {
                            tmem_ld8(t_L + cb * 8, o);
                            tmem_ld_wait8(o);
                        }
                        float l = o[0];
#pragma unroll
                        for (int i = 1; i < 8; ++i) l = lane == i ? o[i] : l;                 // lane = row
                        const float m = lane < 8 ? m_ref[cb * 8 + lane] : 0.f;
                        if (alone && lane < 8) wm[cb * 8 + lane] = l;
                        ll_store_if(!alone && lane < 8 && cb * 8 + lane < n_rows, a.ll + a.ll_ml + ll_row + cb * 8 + lane, m == INFINITY ? -INFINITY : m, l, 0.f, epoch);
                    }
                }
                if (alone) sync_workers();
#pragma unroll 1
                for (int cb = half; cb < NG; cb += 2) {
                    float o[8];
                    read_8(t_O + lane_sel + cb * 8, o);
                    // rows in pairs where the merge takes them so
                    uint4* p = a.ll + (size_t)(ll_row + cb * 8) * HD + kt;
                    const int n = kt < HD ? n_rows - cb * 8 : 0;
                    if (alone) {
#pragma unroll 1
                        for (int i = 0; i < min(n, 8); ++i) {
                            const int r = cb * 8 + i;
                            act_put(true, a.act_attn, sg.row0 + r / G, (sg.kvh * G + r % G) * HD + kt, o[0] * (1.f / wm[r]));
#pragma unroll
                            for (int k = 0; k < 7; ++k) o[k] = o[k + 1];
                        }
                        __syncwarp();
                    } else if (pairs) {
#pragma unroll
                        for (int i = 0; i < 8; i += 2) ll_store_if(i < n, p + i / 2 * HD, o[i], o[i + 1], 0.f, epoch);
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; ++i) ll_store_if(i < n, p + i * HD, o[i], 0.f, 0.f, epoch);
                    }
                }
                tc_fence_before();
                sync_workers();                  // references and accumulators have been read: the next segment may begin
            }
            rw = rv;
            if (kPerTile == 2 && n_seg > 0) {    // the item after the last V
                rw.slot -= 1;
                if (rw.slot < 0) { rw.slot += a.slots; rw.par ^= 1u; }
            }
            // ---- merges: warp = 32 head dimensions of a row, or of two; lane j looks after contributor j's reference and denominator
            const int grp = wt / HD, dim = wt % HD;
#pragma unroll 1
            for (int s = 0; s < n_seg; ++s) {
                const StackSeg& sg = sm.seg[s];
                const int C = sg.C, gs = sg.n_rows > kGroups * C ? 2 : 1;
                if (C == 1) continue;
#pragma unroll 1
                for (int q = sg.idx + grp * C; q * gs < sg.n_rows; q += kGroups * C) {
                    // a row's words: of pair q, word q of its eight rows' block
                    const int r = q * gs, word = gs == 2 ? (q >> 2) * 8 + (q & 3) : q;
                    float m[2] = {-INFINITY, -INFINITY}, num[2] = {0.f, 0.f}, den[2] = {0.f, 0.f};
#pragma unroll 1
                    for (int j0 = 0; j0 < C; j0 += 32) {
                        const int nj = min(C - j0, 32);
                        const uint4* pm = a.ll + a.ll_ml + (size_t)(sg.ll0 + (j0 + lane) * a.r_max + r);
                        const uint4* po = a.ll + ((size_t)(sg.ll0 + j0 * a.r_max) + word) * HD + dim;
                        float w[2];
                        uint4 ml[2];
                        ml[0] = make_uint4(__float_as_uint(-INFINITY), 0u, 0u, lane < nj ? ~epoch : epoch);
                        ml[1] = make_uint4(__float_as_uint(-INFINITY), 0u, 0u, lane < nj && r + 1 < sg.n_rows && gs == 2 ? ~epoch : epoch);
#pragma unroll 1
                        for (int k0 = 0; k0 < nj; k0 += 8, po += 8 * (size_t)a.r_max * HD) {
                            uint4 v[8];
#pragma unroll
                            for (int u = 0; u < 8; ++u) v[u] = make_uint4(0u, 0u, 0u, k0 + u < nj ? ~epoch : epoch);
#pragma unroll 1
                            for (uint32_t look = 0;; ++look) {
                                ll_load_if(ml[0].w != epoch, ml[0], pm);
                                ll_load_if(ml[1].w != epoch, ml[1], pm + 1);
#pragma unroll
                                for (int u = 0; u < 8; ++u)
                                    ll_load_if(v[u].w != epoch, v[u], po + (size_t)u * a.r_max * HD);
                                bool stale = ml[0].w != epoch || ml[1].w != epoch;
#pragma unroll
                                for (int u = 0; u < 8; ++u) stale |= v[u].w != epoch;
                                if (!__any_sync(0xffffffffu, stale)) break;
                                if (!look_on(look)) break;
                            }
                            if (k0 == 0) {
                                // weights of these contributors; one beyond the row's horizon has no reference and weighs nothing
#pragma unroll
                                for (int z = 0; z < 2; ++z) {
                                    const float mj = __uint_as_float(ml[z].x), mb = fmaxf(m[z], warp_max_redux(mj));
                                    const float w0 = m[z] == -INFINITY ? 0.f : exp2f(m[z] - mb);
                                    w[z] = mj == -INFINITY ? 0.f : exp2f(mj - mb);
                                    m[z] = mb;
                                    num[z] *= w0;
                                    den[z] = den[z] * w0 + warp_sum(w[z] * __uint_as_float(ml[z].y));
                                }
                            }
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                num[0] += __shfl_sync(0xffffffffu, w[0], (k0 + u) & 31) * __uint_as_float(v[u].x);
                                num[1] += __shfl_sync(0xffffffffu, w[1], (k0 + u) & 31) * __uint_as_float(v[u].y);
                            }
                        }
                    }
#pragma unroll 1
                    for (int z = 0; z < gs && r + z < sg.n_rows; ++z) {
                        act_put(true, a.act_attn, sg.row0 + (r + z) / G, (sg.kvh * G + (r + z) % G) * HD + dim, num[0] * (1.f / den[0]));
                        num[0] = num[1];
                        den[0] = den[1];
                    }
                }
            }
        };

#pragma unroll 1
        for (int p = 0; p < n_phase; ++p) {
            const int l = p / 5, kind = l < a.n_layers ? p % 5 : (int)kStLm;
            wait(sm.phase, (uint32_t)p & 1u);
            const unsigned epoch = epoch0 + 1u + (unsigned)p;
            if (kind == kStAttn) attn(epoch);
            else gemm(kind, l, epoch);
            arrive_grid();
        }
        if (cta == 0 && wt == 0) {
            a.sync[32] = base + (unsigned)(n_phase + 1) * (unsigned)n_cta;
            a.sync[64] = epoch0 + 1u + (unsigned)n_phase;
        }
    }
    }
    __syncwarp();
    __syncthreads();
    if (sm.abort && tid == 0) {
        // let every copy already issued land before this CTA's shared memory is released
        const unsigned iw = sm.issued_w, ia = sm.issued_a, iq = sm.issued_q, nq = (unsigned)a.q_bufs;
        for (unsigned i = iw > (unsigned)a.slots ? iw - a.slots : 0u; i < iw; ++i) mbar_wait(smem_u32(&sm.full_w[i % a.slots]), (i / a.slots) & 1u);
        for (unsigned i = ia > (unsigned)a.acts ? ia - a.acts : 0u; i < ia; ++i) mbar_wait(smem_u32(&sm.full_a[i % a.acts]), (i / a.acts) & 1u);
        for (unsigned i = iq > nq ? iq - nq : 0u; i < iq; ++i) mbar_wait(smem_u32(&sm.q_full[i % nq]), (i / nq) & 1u);
    }
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace pipesd
