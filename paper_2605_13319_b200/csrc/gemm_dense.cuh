// Dense weight-streaming GEMM for passes of more than 32 rows (a batch of requests, a prompt chunk):
// y[M,N] = x[M,K] . W[N,K]^T on the tcgen05 tensor cores, with the same fused epilogues as the small-M kernel.
//
// A pair of CTAs (cta_group::2) = 256 rows of W x a block of up to 256 tokens x one K slice.  The weights are the M side of
// the MMA (128 rows from each CTA's shared memory), the tokens the N side (each CTA holds half of the block): activations
// arrive as split-bf16 hi and lo tiles in operand order ("xd" arrays, written by the producing kernel's epilogue), two
// MMAs per k16 step into one fp32 accumulator.
// What bounds it: the tensor pipe takes N/2 cycles per MMA, but every MMA fetches its operands from shared memory at 128 B
// per cycle (32 cycles for a CTA's 128 weight rows, N/4 for N tokens), and the copies into the ring need the same
// bandwidth.  One CTA alone with 128 x 256 tiles would want 352 cycles of shared memory per k16 step against 256 of math,
// and 20 KB of L2 per step; a pair halves the token side: 224 against 256 cycles, 12 KB.
// Sums: the tensor pipe truncates each accumulation, so a long K in one accumulator drifts (7b shape, layer 31's K after a
// 160-token prompt: relative L1 error 3.6e-3 with one accumulator over all of K, 2.6e-3 with the small-M kernel's slices).
// Every dense_chunk k16 steps the epilogue warps take the accumulator into registers and add there, rounding to nearest,
// while the MMAs go on in another accumulator: of two, or of four where tensor memory holds them (up to 64 tokens per CTA).
// K slices: where row pairs x token blocks leave SMs idle, S <= 4 pairs form a cluster and share K; the partial tiles cross
// the cluster through distributed shared memory (into the drained ring), each pair sums and finishes every S-th 16-token
// column block, slices in order.
// Warp 0: one lane of each CTA streams (weights, activations) into its ring (weights before the dependent-launch wait), by
// tensor copies of the pair (cta_group::2) whose bytes count on the EVEN CTA's barrier: that barrier alone tells the issuer
// that a stage has landed in both.  (A thread of the odd CTA that waits for its own copies and then arrives remotely is
// either unordered, if the arrival is relaxed, or slow: the release takes 600 cycles; 1024 rows x 12288 x 4096, us: relaxed
// 167, released by three threads in turn 181, this 167.)  Warp 1 of the even CTA: one lane issues the MMAs;
// tcgen05.commit frees a stage / hands an accumulator over in both CTAs.  Warp 2: tensor memory.  Warps 4-11: accumulators
// and epilogue (thread = weight row x half of the tokens, then token x weight rows).
#pragma once
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "gemm.cuh"
#include "tcgen05.cuh"

namespace pipesd {

constexpr int kDenseThreads = 384;
constexpr int kDenseMaxHalf = 128;        // tokens per CTA of a pair (half of a token block): a multiple of 16
constexpr int kDenseMaxSlices = 4;        // K slices: pairs per cluster (8 CTAs, the portable limit)
constexpr int kDenseMaxStages = 9;
constexpr int kDenseRow = 132;            // floats of a token's 128 results in shared memory: eight tokens on eight bank groups
constexpr int kDenseTail = 256 + 4 * 2 * kDenseMaxHalf;   // barriers, tensor-memory base | rstd
constexpr int kDenseSmem = 227 * 1024;    // the CTA has its SM to itself
constexpr int kDenseMaxAccs = 4;
static_assert(8 * (2 * kDenseMaxStages + 2 * kDenseMaxAccs) + 4 <= 256, "barriers and the tensor-memory slot fill the first 256 bytes of the tail");

// ---- "xd" activation arrays: the K-major B operand of tcgen05.mma, in global memory ---------------------------
// Blocks of `tbs` tokens (a multiple of 16), one per CTA of a pair.  Per (block, k16 step): the bf16 hi tile then the lo
// tile, tbs * 32 bytes each, cut into 8x8 core matrices: element (token t, k) of a tile at
// ((t / 8) * 2 + (k / 8) % 2) * 128 + (t % 8) * 16 + (k % 8) * 2.  A chunk of consecutive k16 steps of a block is one
// contiguous run.  (act_index_row / act_index_col and act_store_8, next to the fragment-order stores, write these.)
struct DensePlan {
    int tbs;      // tokens per CTA; a token block is 2 * tbs
    int n_tb;     // token blocks
    int S;        // K slices
};
// Host: token blocks and K slices of a GEMM of N output rows and depth K over M tokens.  pairs[S] = pairs of CTAs the device
// keeps resident at once in clusters of S pairs.  The model, in cycles of 1.9 GHz, is fitted to kernels timed alone (K =
// 4096 and 11008, cold weights): a k16 step costs 110 + 0.05 per token of the block (issue, hand-over of stages), or the
// tensor pipe's 1 per token, 1.3 with all SMs at it (the clock drops under the power cap), or the weights' stream from
// HBM (173 for 4 KB per SM at the copy peak, shared by the token blocks that read the same rows); a wave adds 7600 + 40
// per token (launch, first stages, epilogue), slices another 1500.  Measured against the model, us: 12288 x 4096, 306
// tokens in two blocks of 160: 67 (66), three of 128: 61 (58); 4096 x 11008, 48 tokens in three slices: 22.8 (21).
// A function of its arguments alone: producer and consumer derive the same plan.
static inline DensePlan dense_plan(int M, int N, int K, const int* pairs) {
    const int RBP = ((N + 127) / 128 + 1) / 2, KS = K / 16;
    const int lo = (M + 2 * kDenseMaxHalf - 1) / (2 * kDenseMaxHalf);
    DensePlan best = {kDenseMaxHalf, lo < 1 ? 1 : lo, 1};
    double best_cost = 1e300;
    for (int n = lo < 1 ? 1 : lo; n <= lo + 8; ++n) {
        const int tbs = ((M + 2 * n - 1) / (2 * n) + 15) / 16 * 16, tok = 2 * tbs;
        const int n_tb = (M + tok - 1) / tok;
        if (n_tb != n) continue;
        for (int S = 1; S <= kDenseMaxSlices && (S == 1 || KS / S >= 16); ++S) {
            const long units = (long)RBP * n_tb * S;
            const long waves = (units + pairs[S] - 1) / pairs[S];
            const double occ = (double)units / (waves * pairs[S]);
            const double step = std::max({110.0 + 0.05 * tok, tok * (1.0 + 0.3 * occ), 173.0 * occ / n_tb});
            const double cost = waves * ((KS + S - 1) / S * step + 7600.0 + 40.0 * tok + (S > 1 ? 1500.0 : 0.0));
            if (cost < best_cost * (1.0 - 1e-9)) { best_cost = cost; best = DensePlan{tbs, n_tb, S}; }
        }
    }
    return best;
}
// The same where only the results of rows first_row .. M-1 are wanted (a prompt's last rows): blocks for that many rows, or,
// if that is more, slices and block size of a pass of plan_rows rows (0: of this pass).
static inline DensePlan dense_plan_from(int M, int first_row, int plan_rows, int N, int K, const int* pairs) {
    DensePlan p = dense_plan(M - first_row > plan_rows ? M - first_row : plan_rows, N, K, pairs);
    p.n_tb = (M + 2 * p.tbs - 1) / (2 * p.tbs);
    return p;
}
// Host: k16 steps per accumulator: an eighth of K, as deep as the small-M kernel sums at the most slices it takes, so that a
// prompt's rows are as exact here as there; 8 at least and 32 at most.  (Logits of a 203-token prompt against 64 bits, mean
// over seeds: 1b shape, K = 2048, 3.6e-4 with 32 steps, 3.0e-4 with 16, 3.1e-4 with the small-M kernel; tiny shape, K = 256
// and 688, 4.0e-5 with 16 or 32, 3.0e-5 with 8, 3.1e-5 with the small-M kernel.  8 steps everywhere would cost a tenth to a
// third, as the accumulator changes hands more often.)
static inline int dense_chunk(int KS) { return KS >= 256 ? 32 : KS >= 128 ? 16 : 8; }
// Host: the ring.  As much of the shared memory as it gets.  A stage costs the issuer some 340 cycles of waiting and
// committing beside its MMAs, so small steps are taken eight at a time (4096 x 11008, 32 tokens per CTA, us: 94 with two
// steps a stage, 51.5 with four, 46.7 with eight; 80 tokens: 98, 70.3, 70.7; 64 tokens: 103, 63.1, 65.1).
struct DenseRing { int kc, stages; size_t smem; };
static inline DenseRing dense_ring(int tbs) {
    DenseRing r;
    r.kc = tbs <= 48 ? 8 : 4;
    const int stage = r.kc * (4096 + tbs * 64);
    const int s = (kDenseSmem - kDenseTail) / stage;
    r.stages = s > kDenseMaxStages ? kDenseMaxStages : s;
    r.smem = (size_t)r.stages * stage + kDenseTail;
    return r;
}
// Accumulators of 2 * tbs columns, taken in turn.  With two, the MMAs of a third chunk wait for the epilogue warps to have read
// the first: commit, loads and a releasing remote arrival, about the time of 16 steps at few tokens.
__host__ __device__ constexpr int dense_accs(int tbs) { return 2 * tbs * kDenseMaxAccs <= 512 ? kDenseMaxAccs : 2; }
__host__ __device__ constexpr int dense_tmem_cols(int tbs) {
    int c = 32;
    while (c < dense_accs(tbs) * 2 * tbs) c *= 2;
    return c;
}

// Packed weights and xd arrays as the copy engine sees them: rows of 1 KB, of which a run of k16 steps is a box.  Maps for
// boxes of 8 and 4 steps (the stages' sizes) and for single steps (the remainder of a slice).
struct RunMaps { CUtensorMap by8, by4, by1; };
struct DenseArgs {
    RunMaps w, t;       // weights, tokens (the input xd array)
    GemmArgs g;         // S = K slices; the mode's outputs as for the small-M kernel; W and xf are not read
    int kc;             // k16 steps per ring stage (g.stages stages)
    int chunk;          // k16 steps per accumulator, a multiple of kc
    int tbs_in;         // block size of the input array and of this launch
    int tbs_out;        // block size of the xd array this launch produces (kResid, kSwiglu)
    int tb0, n_tb;      // first token block of the launch, token blocks
    int out_row0;       // kPlain: the token whose result is row 0 of the output (earlier tokens are not stored)
};

// fp32 x[M][K] -> an xd array of blocks of tbs tokens (the component entry point; in a pass the producing kernels write it).
// One thread per (token, eight k).
__global__ void xd_format_kernel(const float* __restrict__ x, uint16_t* __restrict__ xd, int M, int K, int tbs) {
    const int KS = K / 16, per_tok = K / 8;
    const size_t n = (size_t)M * per_tok;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int tok = (int)(i / per_tok), k = 8 * (int)(i % per_tok);
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = x[(size_t)tok * K + k + e];
        act_store_8(xd + act_index_row(tok, k >> 4, KS, 0, tbs) + act_index_col(k & 15, 0, tbs), act_index_lo(tbs), v);
    }
}

// grid (2 * S * row pairs * n_tb), clusters of 2 * S: cluster rank = 2 * slice + CTA of the pair.  The token blocks of a
// row pair are neighbours in the launch order, so that they read its weights from HBM once.
template <int MODE>
__global__ void __launch_bounds__(kDenseThreads, 1) gemm_dense_kernel(const __grid_constant__ DenseArgs da) {
    const GemmArgs& a = da.g;
    extern __shared__ __align__(128) unsigned char smem[];
    const int TBS = da.tbs_in, NT = 2 * TBS;                           // tokens per CTA / per block
    const int KC = da.kc, CH = da.chunk, S = a.S;
    const int w_stage = KC * 4096, stage_bytes = w_stage + KC * TBS * 64;
    const int stages = a.stages;
    unsigned char* tail = smem + stages * stage_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);                // full[9], empty[9], acc_full[4], acc_empty[4]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 8 * (2 * kDenseMaxStages + 2 * kDenseMaxAccs));
    float* rstd_s = reinterpret_cast<float*>(tail + 256);              // [NT]
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kDenseMaxStages;
    const uint32_t acc_full = full0 + 16 * kDenseMaxStages, acc_empty = acc_full + 8 * kDenseMaxAccs;
    const int n_acc = dense_accs(TBS), acc_sh = n_acc == 4 ? 2 : 1;    // chunk ch: accumulator ch % n_acc, turn ch >> acc_sh
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int r = (int)(rank & 1), s = (int)(rank >> 1);
    const int cid = blockIdx.x / (2 * S);
    const int tb = da.tb0 + cid % da.n_tb, rbp = cid / da.n_tb;
    const int RB = (a.N + 127) / 128, rb = 2 * rbp + r;                // an odd RB: the last odd CTA computes a copy, stored by nobody
    const int KS = a.KS;
    const int ks0 = (int)(((long)KS * s) / S), ks1 = (int)(((long)KS * (s + 1)) / S);
    const int nks = ks1 - ks0;
    const int n_chunk = (nks + CH - 1) / CH;
    const int tok0 = tb * NT;
    const uint32_t tmem_cols = (uint32_t)dense_tmem_cols(TBS);

    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; ++i) {
            mbar_init(full0 + 8 * i, 1);                               // the even CTA's: bytes of both CTAs' copies (the odd one's is not used)
            mbar_init(empty0 + 8 * i, 1);
        }
        for (int i = 0; i < n_acc; ++i) {
            mbar_init(acc_full + 8 * i, 1);
            mbar_init(acc_empty + 8 * i, 16);                          // one arrival per epilogue warp of the pair
        }
        fence_mbar_init();
    }
    if (warp == 2) {
        tmem2_alloc(smem_u32(tmem_slot), tmem_cols);
        tc_fence_before();
    }
    if (threadIdx.x == 96) {
        tensor_map_prefetch(KC == 8 ? &da.w.by8 : &da.w.by4);
        tensor_map_prefetch(KC == 8 ? &da.t.by8 : &da.t.by4);
    }
    cluster_sync_all();                                                // barriers of all CTAs are in place
    pdl_launch_dependents();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

    // ring stages of KC steps, in the order all roles walk them (CH is a multiple of KC, so that only the slice's
    // last stage is shorter)
    const int n_stage = (nks + KC - 1) / KC;
    bool ok = true;
    if (warp == 0) {
        // ---------------- producer: lane 0 streams (weights, activations) into the ring
        if (lane == 0) {
            const int wrow = (min(rb, RB - 1) * KS + ks0) * 4, trow = ((2 * tb + r) * KS + ks0) * (TBS / 16);     // in rows of 1 KB
            const uint32_t lead_full = dsmem_addr(full0, rank & ~1u);
            auto steps = [&](int c) { return min(KC, nks - c * KC); };
            auto box = [](int left) { return left >= 8 ? 8 : left >= 4 ? 4 : 1; };                   // steps of the next copy
            // weights leave the L2 first, also where other token blocks read the same rows: those run at the same time (335 rows x
            // 28672 x 4096 in three blocks, us: 157 with the hint, 163 without)
            const uint64_t pol = l2_evict_first_policy();
            auto weights = [&](int c, int st) {
                const int kc = steps(c);
                const uint32_t dst = smem_base + st * stage_bytes, bar = lead_full + 8 * st;
                // the other CTA's bytes may count before this: the phase cannot complete without this arrival
                if (r == 0) mbar_expect_tx(full0 + 8 * st, 2u * (uint32_t)kc * (4096 + TBS * 64));
                for (int i = 0; i < kc;) {
                    const int n = box(kc - i);
                    const CUtensorMap* m = n == 8 ? &da.w.by8 : n == 4 ? &da.w.by4 : &da.w.by1;
                    tensor2_g2s_hint(dst + i * 4096, m, wrow + (c * KC + i) * 4, bar, pol);
                    i += n;
                }
            };
            auto tokens = [&](int c, int st) {
                const int kc = steps(c);
                const uint32_t dst = smem_base + st * stage_bytes + w_stage, bar = lead_full + 8 * st;
                for (int i = 0; i < kc;) {
                    const int n = box(kc - i);
                    const CUtensorMap* m = n == 8 ? &da.t.by8 : n == 4 ? &da.t.by4 : &da.t.by1;
                    tensor2_g2s(dst + i * (TBS * 64), m, trow + (c * KC + i) * (TBS / 16), bar);
                    i += n;
                }
            };
            // weights do not depend on the previous kernel: start them before the dependency wait
            const int pre = n_stage < stages ? n_stage : stages;
            for (int c = 0; c < pre; ++c) weights(c, c);
            pdl_wait();
            for (int c = 0; c < pre; ++c) tokens(c, c);
            int issued = pre, st = 0;
            uint32_t ph = 0;
            for (int c = pre; c < n_stage; ++c) {
                ok = mbar_wait(empty0 + 8 * st, ph);
                if (!ok) break;
                weights(c, st);
                tokens(c, st);
                issued = c + 1;
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
            if (!ok) {
                if (a.err) atomicExch(a.err, 6);
                // give up: let every copy already issued land before shared memory is released (the odd CTA's count here too,
                // and it stays for the even one at the cluster barrier below)
                if (r == 0)
                    for (int c = issued > stages ? issued - stages : 0; c < issued; ++c)
                        mbar_wait(full0 + 8 * (c % stages), (c / stages) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 1 && r == 0) {
        // ---------------- MMA issuer of the pair
        if (elect_one()) {
            const uint32_t idesc = umma_idesc_bf16(256, NT, 0, 0);
            const uint16_t mask = (uint16_t)(3u << rank);              // this CTA and its peer
            const uint32_t lo_step = (uint32_t)(TBS * 32) >> 4;        // hi tile -> lo tile, in descriptor units
            int st = 0;
            uint32_t ph = 0;
            for (int ch = 0; ch < n_chunk && ok; ++ch) {
                const int ac = ch & (n_acc - 1);
                if (ch >= n_acc) ok = mbar_wait_cluster(acc_empty + 8 * ac, (uint32_t)((ch >> acc_sh) - 1) & 1u);
                const uint32_t d = tmem + (uint32_t)(ac * NT);
                const int k_end = min(nks, (ch + 1) * CH);
                for (int k = ch * CH; k < k_end && ok; k += KC) {
                    ok = mbar_wait(full0 + 8 * st, ph);                // landed in both CTAs
                    if (!ok) break;
                    tc_fence_after();
                    uint64_t ad = umma_desc(smem_base + st * stage_bytes, 128, 256);
                    uint64_t bd = umma_desc(smem_base + st * stage_bytes + w_stage, 128, 256);
                    const int kc = min(KC, k_end - k);
                    uint32_t acc = k > ch * CH ? 1u : 0u;
                    for (int i = 0; i < kc; ++i) {
                        umma2_bf16(d, ad, bd, idesc, acc);
                        umma2_bf16(d, ad, bd + lo_step, idesc, 1u);
                        ad += 4096 >> 4;
                        bd += 2 * lo_step;
                        acc = 1u;
                    }
                    umma2_commit(empty0 + 8 * st, mask);               // the stage is free in both CTAs when these MMAs have read it
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
                if (ok) umma2_commit(acc_full + 8 * ac, mask);
            }
            if (!ok && a.err) atomicExch(a.err, 7);
        }
        __syncwarp();
    }
    if (warp < 4) {
        if (S > 1) { cluster_sync_all(); cluster_sync_all(); }
    } else {
        // ---------------- epilogue warps: thread = weight row (tensor-memory lane 32 * (warp % 4) + lane) x one CTA's tokens
        const int et = threadIdx.x - 128;                              // 0..255
        const int quarter = warp & 3, half = et >> 7;
        const int row = quarter * 32 + lane;                           // row within the block
        const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
        pdl_wait();
        if (a.ssq_in != nullptr) {
            for (int tl = et; tl < NT; tl += 256) {
                const int tok = tok0 + tl;
                float ss = 0.f;
                if (tok < a.M) {
#pragma unroll 8
                    for (int b = 0; b < a.n_ssq; ++b) ss += a.ssq_in[(size_t)b * a.M + tok];
                }
                rstd_s[tl] = rsqrtf(ss / (float)a.d_in + a.eps);
            }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        // ---- accumulators: chunk by chunk from tensor memory into registers
        const int ncb = TBS / 16;
        float acc[kDenseMaxHalf / 16][16];
#pragma unroll
        for (int cb = 0; cb < kDenseMaxHalf / 16; ++cb)
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[cb][i] = 0.f;
        const uint32_t lead_empty = dsmem_addr(acc_empty, rank & ~1u);
        for (int ch = 0; ch < n_chunk; ++ch) {
            const int ac = ch & (n_acc - 1);
            if (ok) ok = mbar_wait(acc_full + 8 * ac, (uint32_t)(ch >> acc_sh) & 1u);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            const uint32_t t = tmem + lane_sel + (uint32_t)(ac * NT + half * TBS);
#pragma unroll
            for (int cb = 0; cb < kDenseMaxHalf / 16; ++cb) {
                if (cb < ncb) {
                    float v[16];
                    tmem_ld16(t + cb * 16, v);
                    tmem_ld_wait16(v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[cb][i] += v[i];
                }
            }
            tc_fence_before();
            __syncwarp();
            // only where a later chunk waits for it: the releasing arrival costs 600 cycles
            if (lane == 0 && ch + n_acc < n_chunk) mbar_arrive_cluster(lead_empty + 8 * ac);
        }
        if (!ok && a.err && lane == 0) atomicExch(a.err, 9);
        __syncwarp();

        // ---- the sums leave the registers for the ring's place (the pair's MMAs are done, its copies consumed), token by
        // token: column block b (16 tokens) of the token block belongs to slice b % S of the same CTA of a pair, which
        // receives it as [b / S][slice][16 tokens][128 rows], a token padded to kDenseRow floats
        float* stage_s = reinterpret_cast<float*>(smem);
        if (S > 1) {
            cluster_sync_all();                                        // ... in every CTA of the cluster
#pragma unroll
            for (int cb = 0; cb < kDenseMaxHalf / 16; ++cb) {
                if (cb < ncb) {
                    const int b = half * ncb + cb;
                    const uint32_t dst = dsmem_addr(smem_base + (uint32_t)(((((b / S) * S + s) * 16) * kDenseRow + row) * 4), (uint32_t)((b % S) * 2 + r));
#pragma unroll
                    for (int i = 0; i < 16; ++i) dsmem_st_f32(dst + i * (kDenseRow * 4), acc[cb][i]);
                }
            }
            cluster_sync_all();
        } else {
#pragma unroll
            for (int cb = 0; cb < kDenseMaxHalf / 16; ++cb) {
                if (cb < ncb) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) stage_s[((half * ncb + cb) * 16 + i) * kDenseRow + row] = acc[cb][i];
                }
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");
        }

        // ---- the mode's arithmetic.  A warp takes eight tokens: lane = token (lane % 8) x two 16-row tiles (lane / 8 and
        // that + 4), so that a thread holds a tile's rotary pairs, gate/up pairs or a whole k16 step of the next GEMM's
        // input, and everything it loads and stores is in pieces of 16 bytes, eight lanes to a 128-byte line of an xd array.
        // (Thread = row and two-byte stores instead: 1024 tokens at the 7b shape, us, QKV 260, gate/up 356, O and down 113.)
        const int tk = lane & 7, tq = lane >> 3;
        const int half_hd = a.hd / 2;
        const int KS_out = (MODE == kSwiglu ? a.N / 2 : a.N) / 16;
        uint16_t* act_out = MODE == kSwiglu ? a.xf_act : a.xf_out;
        const uint32_t olo = act_index_lo(da.tbs_out);
        const int n_blk = (2 * ncb - s + S - 1) / S;                   // this slice's column blocks
#pragma unroll 1
        for (int it = warp - 4; it < 2 * n_blk; it += 8) {
            const int blk = it >> 1, tl16 = (it & 1) * 8 + tk;
            const int tl = (blk * S + s) * 16 + tl16, tok = tok0 + tl, tokc = min(tok, a.M - 1);
            const bool live = tok < a.M;
            // what the mode reads of global memory, for both tiles, in flight together
            float4 g0[2][4], g1[2][4];
            long long rk = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int pr0 = min(rb * 128 + (tq + 4 * h) * 16, a.N - 16);
                if (MODE == kResid) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        g0[h][j] = *reinterpret_cast<const float4*>(a.x + (size_t)tokc * a.N + pr0 + 4 * j);
                        g1[h][j] = *reinterpret_cast<const float4*>(a.gain_next + pr0 + 4 * j);
                    }
                } else if (MODE == kQkvRope) {
                    const size_t o = (size_t)tokc * half_hd + (pr0 % a.hd) / 2;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        g0[h][j] = *reinterpret_cast<const float4*>(a.cs + o + 4 * j);
                        g1[h][j] = *reinterpret_cast<const float4*>(a.sn + o + 4 * j);
                    }
                }
            }
            if (MODE == kQkvRope) rk = a.row_kvoff[tokc];
            const float scale = a.ssq_in != nullptr ? rstd_s[tl] : 1.f;
            float ss = 0.f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int tile = tq + 4 * h, pr0 = rb * 128 + tile * 16;
                const bool on = live && pr0 < a.N;                     // N is a multiple of 16
                float v[16];
                const float* sp = stage_s + (size_t)(blk * S * 16 + tl16) * kDenseRow + tile * 16;
#pragma unroll
                for (int j = 0; j < 4; ++j) *reinterpret_cast<float4*>(v + 4 * j) = *reinterpret_cast<const float4*>(sp + 4 * j);
#pragma unroll 1
                for (int q = 1; q < S; ++q) {                          // slices in order
                    sp += 16 * kDenseRow;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 p = *reinterpret_cast<const float4*>(sp + 4 * j);
                        v[4 * j] += p.x; v[4 * j + 1] += p.y; v[4 * j + 2] += p.z; v[4 * j + 3] += p.w;
                    }
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = ok ? v[i] * scale : 0.f;
                if (MODE == kPlain) {
                    if (on && tok >= da.out_row0) {
                        float4* op = reinterpret_cast<float4*>(a.out + (size_t)(tok - da.out_row0) * a.N + pr0);
#pragma unroll
                        for (int j = 0; j < 4; ++j) op[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    }
                } else if (MODE == kResid) {
                    if (on) {
                        float4* xp = reinterpret_cast<float4*>(a.x + (size_t)tok * a.N + pr0);
                        float y[16];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float4 n = make_float4(g0[h][j].x + v[4 * j], g0[h][j].y + v[4 * j + 1], g0[h][j].z + v[4 * j + 2], g0[h][j].w + v[4 * j + 3]);
                            xp[j] = n;
                            ss += n.x * n.x + n.y * n.y + n.z * n.z + n.w * n.w;
                            y[4 * j] = n.x * g1[h][j].x; y[4 * j + 1] = n.y * g1[h][j].y; y[4 * j + 2] = n.z * g1[h][j].z; y[4 * j + 3] = n.w * g1[h][j].w;
                        }
                        uint16_t* op = act_out + act_index_row(tok, pr0 >> 4, KS_out, 0, da.tbs_out);
                        act_store_8(op, olo, y);
                        act_store_8(op + 64, olo, y + 8);
                    }
                } else if (MODE == kSwiglu) {
                    if (on) {
                        const int f0 = gu_feature(pr0);
                        float y[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = v[i] / (1.f + expf(-v[i])) * v[i + 8];      // rows 0-7 gate, 8-15 up
                        act_store_8(act_out + act_index_row(tok, f0 >> 4, KS_out, 0, da.tbs_out) + (f0 & 8) * 8, olo, y);
                    }
                } else if (on) {                                       // kQkvRope: rows 0-7 are dims 8 tau .., rows 8-15 their partners
                    const int head = pr0 / a.hd, d0 = (pr0 % a.hd) / 2;
                    float lo8[8], hi8[8];
                    const float* c8 = reinterpret_cast<const float*>(g0[h]);
                    const float* s8 = reinterpret_cast<const float*>(g1[h]);
                    const bool rot = head < a.Hq + a.Hkv;              // v heads are not rotated
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        lo8[i] = rot ? v[i] * c8[i] - v[i + 8] * s8[i] : v[i];
                        hi8[i] = rot ? v[i + 8] * c8[i] + v[i] * s8[i] : v[i + 8];
                    }
                    if (head < a.Hq) {
                        float4* qp = reinterpret_cast<float4*>(a.q_out + ((size_t)tok * a.Hq + head) * a.hd + d0);
                        float4* qh = reinterpret_cast<float4*>(a.q_out + ((size_t)tok * a.Hq + head) * a.hd + half_hd + d0);
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            qp[j] = make_float4(lo8[4 * j], lo8[4 * j + 1], lo8[4 * j + 2], lo8[4 * j + 3]);
                            qh[j] = make_float4(hi8[4 * j], hi8[4 * j + 1], hi8[4 * j + 2], hi8[4 * j + 3]);
                        }
                    } else {
                        const int kv = head < a.Hq + a.Hkv ? 0 : 1;
                        const int kvh = kv ? head - a.Hq - a.Hkv : head - a.Hq;
                        const size_t per_head = (size_t)a.page_size * a.hd;
                        uint16_t* kp = a.kv_pool + (size_t)a.layer * a.n_pages * 2 * a.Hkv * per_head + (size_t)rk + ((size_t)kv * a.Hkv + kvh) * per_head;
                        *reinterpret_cast<uint4*>(kp + kv_col_offset(d0)) = bf16x8(lo8);
                        *reinterpret_cast<uint4*>(kp + kv_col_offset(half_hd + d0)) = bf16x8(hi8);
                    }
                }
            }
            if (MODE == kResid) {
                // sum of squares of the token's 128 new values: the lanes that share the token
                ss += __shfl_xor_sync(0xffffffffu, ss, 8);
                ss += __shfl_xor_sync(0xffffffffu, ss, 16);
                if (tq == 0 && live && rb < RB) a.ssq_out[(size_t)rb * a.M + tok] = ss;
            }
        }
        tc_fence_before();
    }
    __syncwarp();
    cluster_sync_all();                // nobody arrives on or reads from a CTA that has left
    if (warp == 2) {
        tc_fence_after();
        tmem2_dealloc(tmem, tmem_cols);
    }
}

}  // namespace pipesd
