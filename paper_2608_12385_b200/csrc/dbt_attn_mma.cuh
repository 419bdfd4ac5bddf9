// Grouped decode attention for a bf16 paged KV cache (sm_100a).
//
// The G primary query heads of a KV head and, in grouped mode, the G coupled branch heads
// (Q~_2 = Q_2 + a*Q_1) form one 16-row query tile, so every K/V page is fetched from HBM once
// and serves both paths (Section 4.1: "grouped or fused query execution lets the two paths
// share reads of the primary keys and values").  Keys 0..pos inclusive: the K_1,V_1 appended
// this step is already in its page.
//
// Work decomposition.  A (row, KV head) pair of u 64-token stages is cut into n ~ u / q equal
// segments (q: a target length chosen so that the segments fill one to three rounds of the
// grid); the segments of all pairs, in (row, KV head, segment) order with the rows by falling length,
// are dealt to a fixed grid of CTAs (two per SM), every second round backwards: the CTAs' shares then
// differ little however the lengths do, and the pairs of an incomplete last round are cut to fill it.
// (An equal share of all stages per CTA, cutting pairs at its borders, was measured: 16 % slower on 117
// ragged sequences, as every CTA pays for one more query build, fold and merge.)
// A CTA never straddles two pairs (the per-segment costs -- building the queries, folding the
// warps, the merge -- are then paid once per CTA for equal-length batches), and the split depends
// on the lengths only.  A segment's un-normalised partial (m, l, O) goes to the slot of its
// index, consecutive for one pair; the last segment of a pair to arrive merges them in segment
// order (in two levels above 8 segments), so the result does not depend on arrival order.
//
// Data movement: a producer warp walks the page table and brings 16-token pages in with one 4-D
// TMA box per page (K and V, 128B swizzle) into a shared-memory ring, 64 tokens per stage, ~190 KB
// in flight per SM, with the evict-first L2 hint.  Math: four consumer warps, one page each per
// stage, mma.sync m16n8k16 (bf16 in, fp32 accumulate), operands read with ldmatrix through the
// swizzle; with at most 8 query rows per KV head the products are taken transposed (keys on the
// M side).  Each warp keeps its own running (max, sum, O) and the four are folded in a fixed
// order at the end of a segment.  In decode steps the kernel also builds its queries and the
// new K,V row from the Q|K|V GEMM's split-K partials.  All waits are bounded.
#pragma once

#include <type_traits>

#include "dbt_fused.cuh"
#include "dbt_gemm_tc.cuh"
#include "dbt_gemm_prompt.cuh"

namespace dbt {

struct AttnParams {
    const float *Q;  // [rows][q_dim] fp32, post-RoPE, branch rows already coupled
    RowMap rm;
    int grouped;  // paths present: 0 or 1 = the primary alone, P >= 2 = the primary and P-1 decode branches
    int G, n_kv, num_pages, pt_stride;
    long long k_row0;  // first row of this layer's K plane in the pool's row numbering (the V plane is one plane further)
    const int32_t *page_table, *seq_len;
    float *part;        // [CTAs + pairs] segment partials: [16][DH] outputs, then [16][2] (m, l)
    int *tickets;       // [rows][n_kv] arrival counters (zero between launches)
    int *tickets2;      // [rows][n_kv][kAttMaxGroups] arrival counters of the segment groups
    __nv_bfloat16 *Ob;  // [rows][q_dim] attention output, hi plane (+ lo plane at lo_off)
    size_t lo_off;
    int *status;
    int evict_first;  // K/V pages carry the evict-first L2 hint (read once per step)
    // Decode steps take the Q|K|V GEMM's split-K partials directly (no kernel in between): each CTA
    // builds its pair's queries itself (1/rms, RoPE, Q~_2 = Q_2 + a*Q_1, Eq. asymattn), and the CTA that
    // owns the pair's last stage computes the new K_1, V_1 row, writes it to the pool for later steps
    // and patches it into the staged page.  qkv_P == nullptr: Q comes from `Q`, the cache is complete.
    const float *qkv_P;  // [nsplit][rows][q_dim | kv_dim | kv_dim]
    int qkv_nsplit;
    size_t qkv_stride;
    const float *ss;  // shares of sum(S^2) per row (nullptr: the GEMM input was already normalised)
    int ss_tiles, ss_ld, d_norm;
    float eps;
    const float *coup_a;
    const float2 *rope;
    __nv_bfloat16 *kpool, *vpool;  // this layer's K and V planes
    // Prompt chunks (Section 4.4 item 1, the primary path alone): pack > 0 packs `pack` consecutive positions of
    // a sequence (times the G heads of the KV head) into one 16-row query tile, each row with its own causal
    // limit; a chunk holds cn positions per sequence, nbk = ceil(cn / pack) tiles per sequence, one CTA pass per
    // (tile, KV head) over all its keys, no split.  Q rows and output rows are seq * cn + position.
    int pack, cn, nbk;
    // Rows of a boundary step that ride behind a prompt chunk (ride.K > 0; K rows per sequence, path-major queries in Q): they see
    // `ahead` positions more than seq_len says, the chunk's, and their outputs go to their places in the chunk.  The launch
    // starts beside the chunk's own attention and waits for that one at its end: it reads the Q|K|V kernel's queries, keys and
    // values without a wait of its own, so both prompt attention kernels let it in behind theirs (PromptAttnParams::let_in_late).
    RideRows ride;
    int ahead;
    const int *plan;   // the step's precomputed work split (embed_fused_kernel), or nullptr
    int plan_prewait;  // the plan may be read before the dependency wait
    // The producer does not wait for the kernel before (with plan_prewait): the pages it reads were written by earlier steps, which
    // are complete (the step's embedding kernel lets its dependents in only after its own wait), and the row that this step
    // adds to them is patched in shared memory.
    int early;
};

constexpr int kAttTile = 64;       // tokens per pipeline stage (4 pages)
constexpr int kAttWarps = 4;       // consumer warps, one page each
constexpr int kAttMaxItems = 256;  // rows per launch (prefill chunks and batches stay below)
constexpr int kAttMinUnits = 4;    // a CTA takes at least 4 tiles (256 tokens)
constexpr int kAttPauseAt = 1;     // the producer pauses after stage 1 (the second) until the queries are built
constexpr int kAttMaxSeg = 256;    // most segments a (sequence, KV head) pair is split into
constexpr int kAttGroup = 8;       // segments merged at once (one round of loads)
constexpr int kAttSingle = 16;     // up to this many segments, one CTA merges them all (two rounds of loads)
constexpr int kAttMaxGroups = kAttMaxSeg / kAttGroup;
constexpr unsigned kAttKeyMask = (1u << 24) - 1;  // keys of a row in the plan; its row index above
constexpr float kLog2e = 1.4426950408889634f;

// DEEP: one CTA per SM with a ring twice as deep instead of two CTAs per SM: the same bytes in flight per SM,
// half as many segments (fewer query builds, partials and merges).  (A second group of four consumer warps
// taking alternate stages of the deep ring was measured 1 % slower: the stream, not the consumers, sets the pace.)
template <int DH, bool DEEP = false>
struct AttCfg {
    static constexpr int kHalves = DH / 64;                 // 128-byte column groups per row
    static constexpr int kPageBytes = 16 * DH * 2;          // one page of K (or V) for one head
    static constexpr int kStageBytes = 2 * 4 * kPageBytes;  // K + V, 4 pages
    static constexpr int kStages = (DH == 128 ? 3 : 6) * (DEEP ? 2 : 1);  // 96 KB ring: two CTAs keep ~190 KB in flight per SM
    // scratch: one [16][DH + 8] fp32 slot (Q tile / warp fold; the padding keeps the fold's
    // fragment-shaped accesses off a single bank), m, l, flag, row tables
    static constexpr int kFoldStride = DH + 8;
    static constexpr int kScratchBytes = (16 * kFoldStride + 2 * 16 + 16 + 3 * kAttMaxItems + 12) * 4 + 2 * DH * 2 + 32;
    // room for the ring's barriers (two per stage, up to 12 stages) ahead of the scratch
    static constexpr int kBarBytes = 256;
    static_assert(2 * kStages * 8 <= kBarBytes, "the barriers must not reach into the scratch");
    static constexpr int kSmemBytes = kStages * kStageBytes + 1024 + kBarBytes + kScratchBytes;
};

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Transpose of an 8x8 matrix of 16-bit elements held one row pair per lane (the layout of an
// accumulator's 8x8 block packed to bf16).
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d_hint(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2, int c3,
                                                 uint64_t hint) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, "
        "%6}], [%2], %7;" ::"r"(dst),
        "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(hint)
        : "memory");
}
__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// The work split of one attention launch, computed by one warp from the keys nk[i] = keys | row << 24 of its rows in the
// order in which they are dealt (by falling length where the step's plan sorts them): cum[i] = stages of the rows before
// place i, segcum[i] = segments (per KV head) of the rows before place i.
// The same for every layer of a decode step, so a step computes it once (embed_fused_kernel) and the attention
// launches copy it; launches without a plan (prompt chunks) compute it themselves.
__device__ __forceinline__ void att_plan_warp(int lane, int items, int n_kv, int C0_arg, int min_units, int *cum, const unsigned *nk_s, int *segcum) {
    int running = 0, longest = 0;
    if (lane == 0) cum[0] = 0;
    for (int base = 0; base < items; base += 32) {
        int i = base + lane, u = 0;
        if (i < items) u = ((int)(nk_s[i] & kAttKeyMask) + kAttTile - 1) / kAttTile;
        int incl = u, mx = u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        longest = max(longest, mx);
        if (i < items) cum[i + 1] = running + incl;
        running += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    // Work split: a (row, KV head) pair of u stages is cut into n equal segments and CTA c takes
    // segments c, c + C0_arg, ...: a CTA never straddles two pairs, and the split depends on
    // the lengths only.  n = round or floor of u / q for a target segment length q = all stages /
    // (k * CTAs), k = 1..3 rounds; of these six candidates the one with the smallest estimated
    // time (rounds x (longest segment + a fixed per-segment cost of ~6 stages)) is taken, fewer
    // segments on ties.
    const int C0 = C0_arg, U0 = cum[items] * n_kv;
    auto seg_count = [&](int u, int q, int mode) {  // mode 0: round, 1: floor
        int n = mode == 0 ? (2 * u + q) / (2 * q) : u / q;
        return min(max(n, 1), min(max(u, 1), kAttMaxSeg));
    };
    int best_q = max((U0 + C0 - 1) / C0, min_units), best_mode = 0;
    int best_cost = -1, best_sg = 0;
    for (int cand = 0; cand < 6; cand++) {
        const int k = cand / 2 + 1, mode = cand & 1;
        const int q = max((U0 + k * C0 - 1) / (k * C0), min_units);
        int sg = 0, longest_seg = 0;
        for (int base = 0; base < items; base += 32) {
            int i = base + lane;
            if (i < items) {
                int u = cum[i + 1] - cum[i], n = seg_count(u, q, mode);
                sg += n;
                longest_seg = max(longest_seg, (u + n - 1) / n);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sg += __shfl_xor_sync(0xffffffffu, sg, o);
            longest_seg = max(longest_seg, __shfl_xor_sync(0xffffffffu, longest_seg, o));
        }
        sg *= n_kv;
        int rounds = (sg + C0 - 1) / C0, cost = rounds * (longest_seg + 6);
        if (best_cost < 0 || cost < best_cost || (cost == best_cost && sg < best_sg)) {
            best_cost = cost;
            best_q = q;
            best_mode = mode;
            best_sg = sg;
        }
        // the plain split fits one round, or every pair is already whole: take it (the common cases)
        if (cand == 0 && (rounds == 1 || sg == items * n_kv)) break;
    }
    // Whole pairs in several rounds: the rows of an incomplete last round are cut to fill it (936 equal pairs on 296 CTAs
    // would take four rounds for 3.16).
    const int pairs = items * n_kv, rem = pairs % C0;
    int tail0 = items, tail_n = 1;
    if (best_sg == pairs && pairs > C0 && rem > 0) {
        const int t0 = (pairs - rem + n_kv - 1) / n_kv;
        if (t0 < items && C0 / ((items - t0) * n_kv) > 1) {
            tail0 = t0;
            tail_n = min(C0 / ((items - t0) * n_kv), kAttGroup);
        }
    }
    int run2 = 0;
    if (lane == 0) segcum[0] = 0;
    for (int base = 0; base < items; base += 32) {
        int i = base + lane, n = 0;
        if (i < items) n = i >= tail0 ? max(1, min(tail_n, (cum[i + 1] - cum[i]) / min_units)) : seg_count(cum[i + 1] - cum[i], best_q, best_mode);
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (i < items) segcum[i + 1] = run2 + incl;
        run2 += __shfl_sync(0xffffffffu, incl, 31);
    }
}

constexpr int kAttPlanInts = 3 * kAttMaxItems + 2;  // cum [items + 1] | nk [items] | segcum [items + 1], at fixed offsets

// The shortest segment where the producers fill their rings before the queries exist (see AttnParams::early): three stages, and two
// where eight segments, one round of the merge's loads, still cover the pair.  One sequence of the 1B model (d_h 128, a ring of three)
// with 2 / 3 / 4 stages: context 700 592 / 609 / 617 us per step, context 2048 636 / 613 / 625.  Rings of six stages (d_h 64)
// want no longer ones: 2 and 3 / 4 and 6 stages, d 2048 at 700 positions 315 / 323 us and at 2048 323 / 328, d 512 with four
// sequences of 700 225 / 238; nor does d 3072 at d_h 128, 476 / 493.  In the 16-row form the same: 64 heads of 64 748 / 760 (700
// positions), 763 / 764 (2048), 48 of 128 939 / 949 and 966 / 965.
__device__ __forceinline__ int att_min_early(int stages) { return stages <= 2 * kAttGroup ? 2 : 3; }

// A decode step's plan (one position per sequence), by one block of at least 256 threads: rows by falling length.
__device__ __forceinline__ void att_plan_block(int B, const int32_t *seq_len, int n_kv, int C0, bool early, int *plan) {
    __shared__ int len[kAttMaxItems], cum[kAttMaxItems + 1], segcum[kAttMaxItems + 1];
    __shared__ unsigned nk[kAttMaxItems];
    __shared__ int min_units;
    const int i = threadIdx.x;
    if (i < B) len[i] = ld_mut(seq_len + i) + 1;
    __syncthreads();
    if (i < B) {
        int rank = 0;
        for (int j = 0; j < B; j++) rank += len[j] > len[i] || (len[j] == len[i] && j < i);
        nk[rank] = (unsigned)len[i] | (unsigned)i << 24;
        if (rank == 0) min_units = early ? att_min_early((len[i] + kAttTile - 1) / kAttTile) : kAttMinUnits;
    }
    __syncthreads();
    if (i < 32) att_plan_warp(i, B, n_kv, C0, min_units, cum, nk, segcum);
    __syncthreads();
    if (i <= B && i <= kAttMaxItems) {
        plan[i] = cum[i];
        plan[2 * kAttMaxItems + 1 + i] = segcum[i];
        if (i < B) plan[kAttMaxItems + 1 + i] = (int)nk[i];
    }
    if (i == 0 && B == kAttMaxItems) {  // (256 threads: the last place of 257)
        plan[B] = cum[B];
        plan[2 * kAttMaxItems + 1 + B] = segcum[B];
    }
}

// Eq. embeddings for the fused path: S^0 = RMSNorm(E[x]) and, for the first layer's Q|K|V GEMM,
// the input g_next * S^0 as two bf16 planes plus sum(S^0 ^2) per row (tile 0 carries the whole
// sum, the other tile slots are zeroed).  One block per row; with plan != nullptr (decode steps) one more block computes the
// step's attention work split, which needs the sequence lengths only (as a launch of its own it was one more link of the chain).
template <typename WT>
__global__ void __launch_bounds__(256) embed_fused_kernel(const int32_t *tokens, int n, int p0, RowMap rm,
                                                          const WT *__restrict__ E1, const WT *__restrict__ E2,
                                                          const float *__restrict__ g, float eps, int d, int V,
                                                          float *S, const float *__restrict__ g_next,
                                                          __nv_bfloat16 *Xb, size_t lo_off, float *ss_out, int ss_ld,
                                                          int ss_tiles, int *status, const int32_t *seq_len, int n_kv, int C0, int *plan,
                                                          int barrier, RideRows ride) {
    // barrier: the kernels of this step may rely on all earlier steps being complete, also before their own waits
    if (!barrier) pdl_launch_dependents();
    pdl_wait();
    if (barrier) pdl_launch_dependents();
    __shared__ float scratch[32];
    int r = blockIdx.x;
    if (plan && r == (int)gridDim.x - 1) {
        att_plan_block(rm.B, seq_len, n_kv, C0, barrier != 0, plan);
        return;
    }
    int path = r / rm.Bc();  // 0 primary; j >= 1: decode branch j with its own table E2[j-1] (Appendix C.1)
    int seq = rm.seq(r), off = rm.off(r);
    if (ride.K > 0 && r >= rm.Bc()) {  // behind a prompt chunk: the boundary step's rows, and rows of no sequence between
        if (r < ride.row0 || !ride.locate(r, path, seq)) return;
        off = rm.cn;
    }
    int tok = ld_mut(tokens + (size_t)seq * n + p0 + off);
    if (tok < 0 || tok >= V) {
        if (threadIdx.x == 0) report(status, kStatusBadToken, tok);
        tok = min(max(tok, 0), V - 1);
    }
    const WT *e = (path ? E2 + (size_t)(path - 1) * V * d : E1) + (size_t)tok * d;
    float ss = 0.f;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        float x = load1(e + i);
        ss += x * x;
    }
    ss = block_sum(ss, scratch);
    float inv = 1.f / sqrtf(ss / (float)d + eps), sq = 0.f;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        float s0 = g[i] * load1(e + i) * inv;
        S[(size_t)r * d + i] = s0;
        store_split(Xb, (size_t)r * d + i, lo_off, g_next[i] * s0);
        sq += s0 * s0;
    }
    sq = block_sum(sq, scratch);
    for (int t = threadIdx.x; t < ss_tiles; t += blockDim.x) ss_out[(size_t)t * ss_ld + r] = t == 0 ? sq : 0.f;
}

// Boundary step behind a chunk that its rows rode in: they leave for the decode kernels' places (path-major), with the last layer's
// input g * S and sum(S^2) as embed_fused_kernel leaves them; one more block computes the step's attention work split.
// (In place: the destinations, rows 0 .. K*B - 1, end before the first source, see ride_rows.)
__global__ void __launch_bounds__(256) ride_take_kernel(RideRows ride, float *S, const float *__restrict__ g, int d, __nv_bfloat16 *Xb, size_t lo_off,
                                                        float *ss_out, int ss_ld, int ss_tiles, const int32_t *seq_len, int n_kv, int C0,
                                                        int *plan, int early) {
    pdl_wait();
    pdl_launch_dependents();  // (behind the wait: see AttnParams::early)
    __shared__ float scratch[32];
    const int r = blockIdx.x;
    if (r == (int)gridDim.x - 1) {
        att_plan_block(ride.B, seq_len, n_kv, C0, early != 0, plan);
        return;
    }
    const float *src = S + (size_t)ride.row(r / ride.B, r % ride.B) * d;
    float sq = 0.f;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        const float x = __ldcg(src + i);
        S[(size_t)r * d + i] = x;
        store_split(Xb, (size_t)r * d + i, lo_off, g[i] * x);
        sq += x * x;
    }
    sq = block_sum(sq, scratch);
    for (int t = threadIdx.x; t < ss_tiles; t += blockDim.x) ss_out[(size_t)t * ss_ld + r] = t == 0 ? sq : 0.f;
}

template <int DH, bool NARROW, bool DEEP = false>
__global__ void __launch_bounds__(160, DEEP ? 1 : 2) attn_mma_kernel(const __grid_constant__ CUtensorMap tmKV, AttnParams p) {
    using Cfg = AttCfg<DH, DEEP>;
    constexpr int STAGES = Cfg::kStages, HALVES = Cfg::kHalves, KS = DH / 16, NB = DH / 8;
    extern __shared__ uint8_t smem_raw[];
    uint32_t raw = smem_u32(smem_raw);
    uint32_t tiles = (raw + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (tiles - raw);
    uint32_t bars = tiles + STAGES * Cfg::kStageBytes;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    constexpr int FS = Cfg::kFoldStride;
    float *sc_o = reinterpret_cast<float *>(gen + STAGES * Cfg::kStageBytes + Cfg::kBarBytes);  // [16][FS]
    float *sc_m = sc_o + 16 * FS;                                                   // [16]
    float *sc_l = sc_m + 16;                                                        // [16]
    int *flag = reinterpret_cast<int *>(sc_l + 16);                                 // [0] last?, [1] longest pair, [8..15] 1/rms per path
    int *cum = flag + 16;                // [items + 1] prefix of tiles per row
    unsigned *nk_s = reinterpret_cast<unsigned *>(cum + kAttMaxItems + 1);  // [items] visible keys per row | row << 24
    int *segcum = cum + 2 * kAttMaxItems + 1;   // [items + 1] prefix of segments per row (per KV head)
    __nv_bfloat16 *kv_new =  // [2][DH] this step's K, V row (16-byte aligned)
        reinterpret_cast<__nv_bfloat16 *>((reinterpret_cast<uintptr_t>(segcum + kAttMaxItems + 1) + 15) & ~(uintptr_t)15);

    DBT_TL_DECL;
    int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int items = p.rm.Bc(), Bc = items;
    const int P = p.grouped > 1 ? p.grouped : 1;  // query rows of a KV head: G heads of every path, path-major
    int nq_act = P * p.G, q_dim = p.n_kv * p.G * DH;
    const bool packed = p.pack > 0;
    if (packed) items = p.rm.B * p.nbk;
    // geometry of an item: its sequence, the keys visible to its last row, the positions it holds
    auto item_seq = [&](int i) { return packed ? i / p.nbk : p.rm.seq(i); };
    auto item_npos = [&](int i) { return packed ? min(p.pack, p.cn - (i % p.nbk) * p.pack) : 1; };
    auto item_row0 = [&](int i) { return packed ? (i / p.nbk) * p.cn + (i % p.nbk) * p.pack : i; };  // first Q / output row

    if (tid == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), kAttWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_launch_dependents();
    // A decode step's work split comes precomputed (the same for all its layers).  From the second layer on
    // it is read before the dependency wait: the kernel that wrote it finished long before any kernel that
    // could still be running now; in the first layer that kernel may still be running, so the wait comes first.
    const bool use_plan = p.plan != nullptr && !packed, riding = p.ride.K > 0;
    if (!riding && !(use_plan && p.plan_prewait)) pdl_wait();  // sequence lengths, Q and the freshly appended K/V come from earlier kernels of the step
    if (use_plan) {
        if (!p.plan_prewait) pdl_wait();
        for (int i = tid; i <= items; i += blockDim.x) {
            cum[i] = ld_mut(p.plan + i);
            segcum[i] = ld_mut(p.plan + 2 * kAttMaxItems + 1 + i);
            if (i < items) nk_s[i] = (unsigned)ld_mut(p.plan + kAttMaxItems + 1 + i);
        }
    } else if (warp == 0 && !packed) {
        for (int i = lane; i < items; i += 32)
            nk_s[i] = (unsigned)(ld_mut(p.seq_len + p.rm.seq(i)) + p.rm.off(i) + 1 + p.ahead) | (unsigned)i << 24;
        __syncwarp();
        att_plan_warp(lane, items, p.n_kv, (int)gridDim.x, kAttMinUnits, cum, nk_s, segcum);
    }
    __syncthreads();
    const int C = gridDim.x, Sg = packed ? items * p.n_kv : segcum[items] * p.n_kv;  // all segments, ordered (row, KV head, segment)
    if ((int)blockIdx.x >= Sg) return;  // (CTAs with work wait for the kernel before, so this one does not complete before it either way)
    // segment sidx -> its row and the keys it sees, KV head, stage range and the pair's segment count
    auto locate = [&](int sidx, int &item, int &nkeys, int &g, int &seg, int &n, int &ui, int &t0, int &t1) {
        if (packed) {  // one pass per (tile, KV head) over all its keys
            item = sidx / p.n_kv;
            nkeys = ld_mut(p.seq_len + item / p.nbk) + (item % p.nbk) * p.pack + item_npos(item);
            g = sidx % p.n_kv;
            seg = 0;
            n = 1;
            ui = (nkeys + kAttTile - 1) / kAttTile;
            t0 = 0;
            t1 = ui;
            return;
        }
        int lo = 0, hi = items - 1;
        while (lo < hi) {  // largest place whose first segment is <= sidx
            int mid = (lo + hi + 1) >> 1;
            if (segcum[mid] * p.n_kv <= sidx) lo = mid; else hi = mid - 1;
        }
        item = (int)(nk_s[lo] >> 24);
        nkeys = (int)(nk_s[lo] & kAttKeyMask);
        n = segcum[lo + 1] - segcum[lo];
        int rel = sidx - segcum[lo] * p.n_kv;
        g = rel / n;
        seg = rel % n;
        ui = cum[lo + 1] - cum[lo];
        t0 = (int)(((long long)seg * ui) / n);
        t1 = (int)(((long long)(seg + 1) * ui) / n);
    };
    // What the first queries and the new K, V row need besides the partials -- rotation, coupling, the page -- is requested before the
    // dependency wait: weights, a table and the plan (its positions), none of which this step's kernels write.
    float2 rope0 = make_float2(1.f, 0.f);
    float ca00 = 0.f, ca01 = 0.f;
    int page0 = 0;
    // (Not in the deep form: there it gained 0.5 % at 16 sequences of 2048 and lost 1 % at 8000.)
    const bool ahead = NARROW && !DEEP && use_plan && p.plan_prewait && p.qkv_P != nullptr;
    if (ahead && warp < kAttWarps) {
        constexpr int half = DH / 2;
        int item, nkeys, g, seg, n, ui, t0, t1;
        locate((int)blockIdx.x, item, nkeys, g, seg, n, ui, t0, t1);
        const int i = tid % half, o0 = (g * p.G + min(tid, p.G * half - 1) / half) * DH + i;
        rope0 = p.rope[(size_t)(nkeys - 1) * half + i];
        if (P > 1) {
            ca00 = p.coup_a[o0];
            ca01 = p.coup_a[o0 + half];
        }
        if (seg == n - 1 && tid < half) page0 = __ldg(p.page_table + (size_t)p.rm.seq(item) * p.pt_stride + ((nkeys - 1) >> 4));
    }
    if (use_plan && p.plan_prewait && !(p.early && warp == kAttWarps)) pdl_wait();
    DBT_TL_WAITED;
    // this CTA's segment of a round: every second round is dealt backwards
    auto dealt = [&](int round) { return round * C + ((round & 1) ? C - 1 - (int)blockIdx.x : (int)blockIdx.x); };

    if (warp == kAttWarps) {
        // ---- producer: walks the same segments as the consumers.  Lane 0 waits for the stage and
        // arms its barrier; up to four lanes then issue one box each (a page's K and V, both
        // 64-column pieces: 8 KB at d_h = 128), each after its own page-table lookup.
        if (lane == 0) tma_prefetch_desc(&tmKV);
        const uint64_t pol = l2_evict_first_policy();
        bool ok = true;
        int it = 0;
        // early: the ring is filled before the queries' loads go out.  (Asked of p.early at every stage instead, the deep form at d_h 64
        // streamed 7 % slower: 16 sequences of 6000 722 us per step, 707 now.)
        const int pause_at = p.early ? -1 : kAttPauseAt;
        for (int round = 0, sidx; ok && (sidx = dealt(round)) < Sg; round++) {
            int item, nkeys, g, seg, n, ui, t0, t1;
            locate(sidx, item, nkeys, g, seg, n, ui, t0, t1);
            int seq = item_seq(item), total_pages = (nkeys + 15) >> 4;
            // page ids 32 at a time (eight stages' worth, one coalesced load): a lookup per stage would put an
            // L2 round trip on every stage of this loop and cap a CTA at one stage per ~0.7 us
            int pt_base = -(1 << 30), my_page = 0;
            for (int t = t0; t < t1; t++, it++) {
                int s = it % STAGES;
                int p0 = t * 4, np = min(4, total_pages - p0);
                if (p0 + 4 > pt_base + 32) {
                    pt_base = p0;
                    my_page = p0 + lane < total_pages ? __ldg(p.page_table + (size_t)seq * p.pt_stride + p0 + lane) : 0;
                }
                if (lane == 0) {
                    if (it >= STAGES) ok = mbar_wait(empty_bar(s), ((it / STAGES) - 1) & 1);
                    if (ok) mbar_expect_tx(full_bar(s), (uint32_t)np * 2 * Cfg::kPageBytes);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                int page = __shfl_sync(0xffffffffu, my_page, (p0 - pt_base + lane) & 31);
                if (lane < np) {
                    if (page < 0 || page >= p.num_pages) {
                        report(p.status, kStatusBadPage, page);
                        page = 0;
                    }
                    int row = (int)(((long long)page * p.n_kv + g) * 16);
                    if (p.evict_first)
                        tma_load_4d_hint(tiles + s * Cfg::kStageBytes + lane * 2 * Cfg::kPageBytes, &tmKV, full_bar(s), 0, 0,
                                         (int)(p.k_row0 + row), 0, pol);
                    else
                        tma_load_4d(tiles + s * Cfg::kStageBytes + lane * 2 * Cfg::kPageBytes, &tmKV, full_bar(s), 0, 0,
                                    (int)(p.k_row0 + row), 0);
                }
                // After the first two stages the stream pauses until the consumers have their queries: their
                // few small loads would otherwise queue behind hundreds of CTAs' page traffic for several
                // microseconds, and nothing can be consumed before they return anyway.  (Letting the ring fill
                // at once instead, with the small loads issued first, was measured slower: the queries are ready
                // 0.8 us sooner but the stream then runs 10 % slower; pausing after one, two, four or six stages
                // gave 1.0446, 1.0384, 1.0420 and 1.0462 ms per step of the 1B model at batch 16.)
                if (it == pause_at || (it < pause_at && dealt(round + 1) >= Sg && t == t1 - 1)) asm volatile("bar.sync 2, 160;" ::: "memory");
            }
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 300);
        return;
    }

    // ---- consumers
    bool ok = true;
    int it = 0;
    const float qscale = kLog2e / sqrtf((float)DH);
    // The staged copy of the page that holds this step's position was read while the row was being
    // written: overwrite the row in shared memory with the values computed here (16-byte pieces,
    // lanes 0..15 the K row, lanes 16..31 the V row; DH = 64 uses half of each).
    auto patch_new_row = [&](uint32_t kpage, uint32_t vpage, int row) {
        int piece = lane & 15;
        if (piece < DH / 8) {
            int sg = row * HALVES + (piece >> 3);
            uint32_t dst = (lane < 16 ? kpage : vpage) + sg * 128 + (((piece & 7) ^ (sg & 7)) << 4);
            const uint4 v = *reinterpret_cast<const uint4 *>(kv_new + (lane < 16 ? 0 : DH) + piece * 8);
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
        }
        __syncwarp();
    };
    // A segment's last stage is written by ordinary stores too -- zeros behind the last key, the new row, in the narrow form the
    // warps' states -- and the next segment's pages then arrive in it by TMA, through the async proxy: every thread that wrote (each
    // comes here) orders its accesses before those ahead of the barrier arrival that gives the stage back.  Without a next
    // segment nothing arrives there any more.
    auto hand_over = [&](int round) {
        if (dealt(round + 1) < Sg) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };
    for (int round = 0, sidx; (sidx = dealt(round)) < Sg; round++) {
        int item, nkeys, g, seg, nseg, ui, t0, t1;
        locate(sidx, item, nkeys, g, seg, nseg, ui, t0, t1);
        if (packed) nq_act = item_npos(item) * p.G;  // rows: position-major, the G heads of each position

        // Query tile (16 rows x DH, fp32) into shared memory, then mma A fragments (bf16),
        // pre-scaled by log2(e)/sqrt(d_h).  Rows: G primary heads, then G coupled branch heads.
        consumer_sync();  // the previous segment is done with the scratch
        const bool owns_last = p.qkv_P != nullptr && seg == nseg - 1;  // this segment ends the pair
        if (p.qkv_P == nullptr) {
            for (int idx = tid; idx < 16 * DH / 4; idx += 128) {
                int q = idx / (DH / 4), c4 = idx % (DH / 4);
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (q < nq_act) {
                    int row = packed ? item_row0(item) + q / p.G : (q / p.G) * Bc + item;
                    int h = g * p.G + q % p.G;
                    v = __ldcg(reinterpret_cast<const float4 *>(p.Q + (size_t)row * q_dim + (size_t)h * DH) + c4);
                }
                reinterpret_cast<float4 *>(sc_o)[idx] = v;
            }
        } else {
            constexpr int half = DH / 2;
            const int kv_dim = p.n_kv * DH, ldp = q_dim + 2 * kv_dim, pos = nkeys - 1;
            const bool grp = P > 1;
            const int twin = grp ? Bc + item : item;  // the first branch's row travels with the primary's loads
            const size_t p1 = (size_t)item * ldp, p2 = (size_t)twin * ldp;
            // One round of loads: the first warp requests the norm shares of the pair's rows (lanes
            // 0..15 the primary row, 16..31 the first branch's) and hands 1/rms to the others through
            // shared memory; every thread requests the partials, the rotation and the coupling of its
            // outputs before anyone waits.  Further decode branches (Appendix C.1) follow in rounds of
            // their own.
            float myss = 0.f;
            if (p.ss && warp == 0)
                for (int t = lane & 15; t < p.ss_tiles; t += 16) myss += __ldcg(p.ss + (size_t)t * p.ss_ld + (lane < 16 ? item : twin));
            for (int idx = tid; idx < (16 - nq_act) * DH / 4; idx += 128)  // unused query rows
                reinterpret_cast<float4 *>(sc_o + (size_t)nq_act * DH)[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int nitems = p.G * half;
            const bool do_kv = owns_last && tid < half;
            float *rs_s = reinterpret_cast<float *>(flag + 8);  // [path]
            // the page of this step's position: requested with the first round of loads, used after it
            const bool pre = ahead && round == 0;
            const int page_new = pre ? page0 : do_kv ? __ldg(p.page_table + (size_t)p.rm.seq(item) * p.pt_stride + (pos >> 4)) : 0;
            float rs1 = 1.f, rs2 = 1.f, kvs[4] = {0.f, 0.f, 0.f, 0.f};
            float2 t_kv = make_float2(1.f, 0.f);
            for (int it0 = 0; it0 * 128 < nitems; it0++) {
                int idx = it0 * 128 + tid;
                bool act = idx < nitems;
                int j = act ? idx / half : 0, i = act ? idx % half : tid % half;
                int o0 = (g * p.G + j) * DH + i, o1 = o0 + half;
                const bool here = pre && it0 == 0;
                float2 t = here ? rope0 : p.rope[(size_t)pos * half + i];
                float ca0 = here ? ca00 : grp ? p.coup_a[o0] : 0.f, ca1 = here ? ca01 : grp ? p.coup_a[o1] : 0.f;
                const size_t offs[4] = {p1 + o0, p1 + o1, p2 + o0, p2 + o1};
                float sm[4] = {0.f, 0.f, 0.f, 0.f};
                if (act) {
                    if (NARROW && p.qkv_nsplit == 1) {  // (finished sums: the code of the general form alone is a microsecond of instruction misses)
#pragma unroll
                        for (int k = 0; k < 4; k++) sm[k] = __ldcg(p.qkv_P + offs[k]);
                    } else {
                        sum_splits_k<4, 12>(p.qkv_P, p.qkv_stride, p.qkv_nsplit, offs, sm);
                    }
                }
                if (it0 == 0) {
                    if (do_kv) {  // K_1 and V_1 of this step's token for this KV head (tid = rotation pair)
                        size_t ko = p1 + q_dim + (size_t)g * DH + tid, vo = ko + kv_dim;
                        const size_t koffs[4] = {ko, ko + half, vo, vo + half};
                        if (NARROW && p.qkv_nsplit == 1) {
#pragma unroll
                            for (int k = 0; k < 4; k++) kvs[k] = __ldcg(p.qkv_P + koffs[k]);
                        } else {
                            sum_splits_k<4, 12>(p.qkv_P, p.qkv_stride, p.qkv_nsplit, koffs, kvs);
                        }
                        t_kv = t;  // idx = tid < half in the first round: the same rotation pair
                    }
                    if (warp == 0) {
                        sc_m[lane] = myss;  // sc_m[0..15], sc_l[0..15] are contiguous
                        __syncwarp();
                        if ((lane & 15) == 0) {
                            float a = 0.f;
                            for (int k = 0; k < 16; k++) a += sc_m[lane + k];
                            rs_s[lane >> 4] = p.ss ? 1.f / sqrtf(a / (float)p.d_norm + p.eps) : 1.f;
                        }
                        for (int jp = 2; jp < P; jp++) {  // further branches: the whole warp per row
                            float a = 0.f;
                            if (p.ss)
                                for (int t2 = lane; t2 < p.ss_tiles; t2 += 32) a += __ldcg(p.ss + (size_t)t2 * p.ss_ld + jp * Bc + item);
                            sc_m[lane] = a;
                            __syncwarp();
                            if (lane == 0) {
                                float tot = 0.f;
                                for (int k = 0; k < 32; k++) tot += sc_m[k];
                                rs_s[jp] = p.ss ? 1.f / sqrtf(tot / (float)p.d_norm + p.eps) : 1.f;
                            }
                            __syncwarp();
                        }
                    }
                    DBT_TL_MARK(3);
                    consumer_sync();
                    rs1 = rs_s[0];
                    rs2 = rs_s[1];
                }
                if (act) {
                    float x0 = rs1 * sm[0], x1 = rs1 * sm[1];
                    float r0 = x0 * t.x - x1 * t.y, r1 = x1 * t.x + x0 * t.y;
                    sc_o[(size_t)j * DH + i] = r0;
                    sc_o[(size_t)j * DH + i + half] = r1;
                    if (grp) {
                        float y0 = rs2 * sm[2], y1 = rs2 * sm[3];
                        sc_o[(size_t)(p.G + j) * DH + i] = (y0 * t.x - y1 * t.y) + ca0 * r0;
                        sc_o[(size_t)(p.G + j) * DH + i + half] = (y1 * t.x + y0 * t.y) + ca1 * r1;
                    }
                    for (int jp = 2; jp < P; jp++) {  // Q~_j = Q_j + a * Q_1 for the further branches
                        const size_t pj = (size_t)(jp * Bc + item) * ldp;
                        const size_t offj[2] = {pj + o0, pj + o1};
                        float sj[2];
                        sum_splits_k<2, 12>(p.qkv_P, p.qkv_stride, p.qkv_nsplit, offj, sj);
                        const float rsj = rs_s[jp];
                        float y0 = rsj * sj[0], y1 = rsj * sj[1];
                        sc_o[(size_t)(jp * p.G + j) * DH + i] = (y0 * t.x - y1 * t.y) + ca0 * r0;
                        sc_o[(size_t)(jp * p.G + j) * DH + i + half] = (y1 * t.x + y0 * t.y) + ca1 * r1;
                    }
                }
            }
            if (do_kv) {
                // K_1 = RoPE(N_1 W_K), V_1 = N_1 W_V: to the staging row for the patch and to the pool
                int i = tid;
                float x0 = rs1 * kvs[0], x1 = rs1 * kvs[1];
                __nv_bfloat16 k0 = __float2bfloat16_rn(x0 * t_kv.x - x1 * t_kv.y), k1 = __float2bfloat16_rn(x1 * t_kv.x + x0 * t_kv.y);
                __nv_bfloat16 v0 = __float2bfloat16_rn(rs1 * kvs[2]), v1 = __float2bfloat16_rn(rs1 * kvs[3]);
                kv_new[i] = k0;
                kv_new[i + half] = k1;
                kv_new[DH + i] = v0;
                kv_new[DH + i + half] = v1;
                const int page = page_new;
                if (page < 0 || page >= p.num_pages) {
                    if (i == 0) report(p.status, kStatusBadPage, page);
                } else {
                    size_t base = (((size_t)page * p.n_kv + g) * 16 + (pos & 15)) * DH;
                    p.kpool[base + i] = k0;
                    p.kpool[base + i + half] = k1;
                    p.vpool[base + i] = v0;
                    p.vpool[base + i + half] = v1;
                }
            }
        }
        consumer_sync();
        if (round == 0) {
            if (!p.early) asm volatile("bar.arrive 2, 160;" ::: "memory");  // the producer may stream on
            DBT_TL_MARK(0);
        }
        // Output row of a path of the item.  (The 16-row form takes it from a base found once per segment: 8B, three ragged sequences of
        // up to 31867 positions with three paths 4688 -> 4667 us per step; the narrow form is 0.3 % slower that way.)
        const int orow = !NARROW && riding ? p.ride.row(0, item) : item, ostep = !NARROW && riding ? p.ride.spg : Bc;
        auto out_row = [&](int path) { return NARROW && riding ? p.ride.row(path, item) : orow + path * ostep; };
        int pair = item * p.n_kv + g;
        int first_slot = sidx - seg;  // the pair's segments occupy consecutive partial slots
        float *out = p.part + (size_t)sidx * 16 * (DH + 2);
        if constexpr (!NARROW) {
            uint32_t qa[KS][4];
            {
                int r0 = lane >> 2, c = (lane & 3) * 2;
                const float *q0 = sc_o + r0 * DH, *q1 = sc_o + (r0 + 8) * DH;
    #pragma unroll
                for (int ks = 0; ks < KS; ks++) {
                    int k = ks * 16 + c;
                    qa[ks][0] = pack_bf16(q0[k] * qscale, q0[k + 1] * qscale);
                    qa[ks][1] = pack_bf16(q1[k] * qscale, q1[k + 1] * qscale);
                    qa[ks][2] = pack_bf16(q0[k + 8] * qscale, q0[k + 9] * qscale);
                    qa[ks][3] = pack_bf16(q1[k + 8] * qscale, q1[k + 9] * qscale);
                }
            }
            consumer_sync();  // everyone has its fragments: the scratch is free again
            float o[NB][4];
    #pragma unroll
            for (int nb = 0; nb < NB; nb++) o[nb][0] = o[nb][1] = o[nb][2] = o[nb][3] = 0.f;
            float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};

            for (int t = t0; t < t1 && ok; t++, it++) {
                int s = it % STAGES;
                ok = mbar_wait(full_bar(s), (it / STAGES) & 1);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                int valid = min(16, nkeys - (t * kAttTile + warp * 16));  // valid tokens in this warp's page
                if (valid > 0) {
                    // a page's box: K then V, each [16 rows][DH], the 128-byte pieces of a row swizzled
                    uint32_t kpage = tiles + s * Cfg::kStageBytes + warp * 2 * Cfg::kPageBytes;
                    uint32_t vpage = kpage + Cfg::kPageBytes;
                    if (valid < 16) {
                        // stale slots past the end of the sequence: their scores are masked below, and
                        // their V rows are zeroed here so that 0 * garbage cannot produce a NaN
                        for (int idx = lane; idx < (16 - valid) * HALVES * 8; idx += 32) {
                            uint32_t a = vpage + valid * HALVES * 128 + idx * 16;
                            asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u) : "memory");
                        }
                        __syncwarp();
                    }
                    if (owns_last && t == ui - 1 && ((nkeys - 1) >> 4 & 3) == warp) patch_new_row(kpage, vpage, (nkeys - 1) & 15);
                // S = Q K^T for this warp's 16 tokens: two 8-token column blocks
                    float sacc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
                    {
                        int r = (lane & 7) + ((lane >> 4) << 3);  // token row this lane addresses
                        int cb = (lane >> 3) & 1;                 // which 8-dim chunk of the k-step
    #pragma unroll
                        for (int ks = 0; ks < KS; ks++) {
                            int chunk = ks * 2 + cb;  // 16-byte chunk index within the row
                            int sg = r * HALVES + (chunk >> 3);
                            uint32_t a = kpage + sg * 128 + (((chunk & 7) ^ (sg & 7)) << 4);
                            uint32_t kb[4];
                            ldsm_x4(a, kb);
                            mma_bf16(sacc[0], qa[ks], kb[0], kb[1]);
                            mma_bf16(sacc[1], qa[ks], kb[2], kb[3]);
                        }
                    }
                    // mask, online softmax (base 2), pack P as the A operand of P V
                    int col = (lane & 3) * 2;
                    float rmax[2] = {-INFINITY, -INFINITY};
                    // packed prompt tiles: the row of position pp sees the keys up to its own position only
                    int vrow[2] = {valid, valid};
                    if (packed) {
                        const int npos = nq_act / p.G, rem = nkeys - (t * kAttTile + warp * 16);
    #pragma unroll
                        for (int h = 0; h < 2; h++) vrow[h] = min(16, rem - max(npos - 1 - ((lane >> 2) + 8 * h) / p.G, 0));
                    }
    #pragma unroll
                    for (int nb = 0; nb < 2; nb++)
    #pragma unroll
                        for (int e = 0; e < 4; e++) {
                            int tk = nb * 8 + col + (e & 1);
                            if (tk >= vrow[e >> 1]) sacc[nb][e] = -INFINITY;
                            rmax[e >> 1] = fmaxf(rmax[e >> 1], sacc[nb][e]);
                        }
                    float corr[2], msub[2];
    #pragma unroll
                    for (int h = 0; h < 2; h++) {
                        rmax[h] = fmaxf(rmax[h], __shfl_xor_sync(0xffffffffu, rmax[h], 1));
                        rmax[h] = fmaxf(rmax[h], __shfl_xor_sync(0xffffffffu, rmax[h], 2));
                        float mnew = fmaxf(m_run[h], rmax[h]);
                        msub[h] = mnew == -INFINITY ? 0.f : mnew;
                        corr[h] = m_run[h] == -INFINITY ? 0.f : exp2f(m_run[h] - msub[h]);
                        m_run[h] = mnew;
                    }
                    float rsum[2] = {0.f, 0.f};
                    uint32_t pa[4];
    #pragma unroll
                    for (int nb = 0; nb < 2; nb++) {
                        float p0 = exp2f(sacc[nb][0] - msub[0]), p1 = exp2f(sacc[nb][1] - msub[0]);
                        float p2 = exp2f(sacc[nb][2] - msub[1]), p3 = exp2f(sacc[nb][3] - msub[1]);
                        rsum[0] += p0 + p1;
                        rsum[1] += p2 + p3;
                        pa[nb * 2 + 0] = pack_bf16(p0, p1);
                        pa[nb * 2 + 1] = pack_bf16(p2, p3);
                    }
    #pragma unroll
                    for (int h = 0; h < 2; h++) {
                        rsum[h] += __shfl_xor_sync(0xffffffffu, rsum[h], 1);
                        rsum[h] += __shfl_xor_sync(0xffffffffu, rsum[h], 2);
                        l_run[h] = l_run[h] * corr[h] + rsum[h];
                    }
    #pragma unroll
                    for (int nb = 0; nb < NB; nb++) {
                        o[nb][0] *= corr[0];
                        o[nb][1] *= corr[0];
                        o[nb][2] *= corr[1];
                        o[nb][3] *= corr[1];
                    }
                    // O += P V: V read transposed, two 8-dim column blocks per ldmatrix
                    {
                        int r = (lane & 7) + (((lane >> 3) & 1) << 3);  // token row
                        int cb = lane >> 4;                              // which of the two dim blocks
    #pragma unroll
                        for (int np = 0; np < NB / 2; np++) {
                            int chunk = np * 2 + cb;
                            int sg = r * HALVES + (chunk >> 3);
                            uint32_t a = vpage + sg * 128 + (((chunk & 7) ^ (sg & 7)) << 4);
                            uint32_t vb[4];
                            ldsm_x4_trans(a, vb);
                            mma_bf16(o[np * 2], pa, vb[0], vb[1]);
                            mma_bf16(o[np * 2 + 1], pa, vb[2], vb[3]);
                        }
                    }
                }
                // (the row's last stage may hold zeros and the new row: see hand_over)
                if (t + 1 == t1) hand_over(round);
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty_bar(s)) : "memory");
            }
            if (!ok) {
                // a ring that stopped filling stops for all four warps: every consumer leaves here
                if (lane == 0) report(p.status, kStatusWaitExpired, 310 + warp);
                return;
            }

            // ---- fold the four warps' states, (0+2) + (1+3), in registers through the one-slot
            // scratch; warp 0 then writes this segment's partial
            {
                int r0 = lane >> 2, c = (lane & 3) * 2;
                auto put = [&]() {
    #pragma unroll
                    for (int nb = 0; nb < NB; nb++) {
                        *reinterpret_cast<float2 *>(sc_o + (size_t)r0 * FS + nb * 8 + c) = make_float2(o[nb][0], o[nb][1]);
                        *reinterpret_cast<float2 *>(sc_o + (size_t)(r0 + 8) * FS + nb * 8 + c) = make_float2(o[nb][2], o[nb][3]);
                    }
                    if ((lane & 3) == 0) {
                        sc_m[r0] = m_run[0];
                        sc_m[r0 + 8] = m_run[1];
                        sc_l[r0] = l_run[0];
                        sc_l[r0 + 8] = l_run[1];
                    }
                };
                auto take = [&]() {  // this warp's state := this warp's state (+) the slot's state
    #pragma unroll
                    for (int h = 0; h < 2; h++) {
                        int r = r0 + 8 * h;
                        float mb = sc_m[r], lb = sc_l[r];
                        float M = fmaxf(m_run[h], mb);
                        float fa = m_run[h] == -INFINITY ? 0.f : exp2f(m_run[h] - M);
                        float fb = mb == -INFINITY ? 0.f : exp2f(mb - M);
                        l_run[h] = l_run[h] * fa + lb * fb;
                        m_run[h] = M;
    #pragma unroll
                        for (int nb = 0; nb < NB; nb++) {
                            float2 ob = *reinterpret_cast<const float2 *>(sc_o + (size_t)r * FS + nb * 8 + c);
                            o[nb][2 * h] = o[nb][2 * h] * fa + ob.x * fb;
                            o[nb][2 * h + 1] = o[nb][2 * h + 1] * fa + ob.y * fb;
                        }
                    }
                };
                for (int step = 0; step < 3; step++) {  // 2 -> 0, 3 -> 1, 1 -> 0
                    int src = step == 0 ? 2 : step == 1 ? 3 : 1, dst = step == 1 ? 1 : 0;
                    if (warp == src) put();
                    consumer_sync();
                    if (warp == dst) take();
                    consumer_sync();
                }
                if (warp == 0) {
    #pragma unroll
                    for (int h = 0; h < 2; h++) {
                        int q = r0 + 8 * h;
                        if (q < nq_act) {
                            if (nseg == 1) {
                                // the pair's only segment: normalise and write the head's output
                                int row = packed ? item_row0(item) + q / p.G : out_row(q / p.G);
                                int hq = g * p.G + q % p.G;
                                size_t ob = (size_t)row * q_dim + (size_t)hq * DH;
                                float inv = 1.f / l_run[h];
    #pragma unroll
                                for (int nb = 0; nb < NB; nb++)
    #pragma unroll
                                    for (int e = 0; e < 2; e++) {
                                        float x = o[nb][2 * h + e] * inv;
                                        __nv_bfloat16 hi = __float2bfloat16_rn(x);
                                        p.Ob[ob + nb * 8 + c + e] = hi;
                                        if (p.lo_off) p.Ob[ob + nb * 8 + c + e + p.lo_off] = __float2bfloat16_rn(x - __bfloat162float(hi));
                                    }
                            } else {
    #pragma unroll
                                for (int nb = 0; nb < NB; nb++)
                                    *reinterpret_cast<float2 *>(out + (size_t)q * DH + nb * 8 + c) =
                                        make_float2(o[nb][2 * h], o[nb][2 * h + 1]);
                                if ((lane & 3) == 0) {
                                    out[16 * DH + 2 * q] = m_run[h];  // base-2 units
                                    out[16 * DH + 2 * q + 1] = l_run[h];
                                }
                            }
                        }
                    }
                    if (nseg > 1) __threadfence();
                }
            }
        } else {
            // ---- narrow variant: at most 8 query rows per KV head.  The products are taken transposed,
            // S^T = K Q^T and O^T = V^T P^T, so that the 16 keys of a page fill the M side of
            // m16n8k16 and the (few) queries sit on the 8-wide N side: half the MMAs and half the
            // accumulators of the 16-query form.
            uint32_t qb[KS][2];
            {
                int n = lane >> 2, c = (lane & 3) * 2;
                const float *q0 = sc_o + n * DH;
#pragma unroll
                for (int ks = 0; ks < KS; ks++) {
                    int k = ks * 16 + c;
                    qb[ks][0] = pack_bf16(q0[k] * qscale, q0[k + 1] * qscale);
                    qb[ks][1] = pack_bf16(q0[k + 8] * qscale, q0[k + 9] * qscale);
                }
            }
            consumer_sync();  // everyone has its fragments: the scratch is free again
            constexpr int MB = DH / 16;  // 16-row blocks of O^T
            float o[MB][4];
#pragma unroll
            for (int mb = 0; mb < MB; mb++) o[mb][0] = o[mb][1] = o[mb][2] = o[mb][3] = 0.f;
            // per query column (2t, 2t+1): running max (same in the 8 lanes of a column) and this
            // lane's share of the running sum (reduced over the lanes once, after the loop)
            float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
            const int g8 = lane >> 2;

            for (int t = t0; t < t1 && ok; t++, it++) {
                int s = it % STAGES;
                ok = mbar_wait(full_bar(s), (it / STAGES) & 1);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                int valid = min(16, nkeys - (t * kAttTile + warp * 16));  // valid tokens in this warp's page
                if (valid > 0) {
                    uint32_t kpage = tiles + s * Cfg::kStageBytes + warp * 2 * Cfg::kPageBytes;
                    uint32_t vpage = kpage + Cfg::kPageBytes;
                    if (valid < 16) {
                        for (int idx = lane; idx < (16 - valid) * HALVES * 8; idx += 32) {
                            uint32_t a = vpage + valid * HALVES * 128 + idx * 16;
                            asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u) : "memory");
                        }
                        __syncwarp();
                    }
                    if (owns_last && t == ui - 1 && ((nkeys - 1) >> 4 & 3) == warp) patch_new_row(kpage, vpage, (nkeys - 1) & 15);
                    // S^T = K Q^T: K rows as the A operand
                    // (Two chains of products, added at the end, make a step of one sequence 0.3 to 0.6 % faster and none of 16
                    // sequences or more: 1B 626 / 629, 1036 / 1036, 117 ragged 2705 / 2701 us.  One keeps the sums' order.)
                    float sacc[4] = {0.f, 0.f, 0.f, 0.f};
                    {
                        int r = (lane & 7) + (((lane >> 3) & 1) << 3);  // key row this lane addresses
                        int cb = lane >> 4;                              // which 8-dim chunk of the k-step
#pragma unroll
                        for (int ks = 0; ks < KS; ks++) {
                            int chunk = ks * 2 + cb;
                            int sg = r * HALVES + (chunk >> 3);
                            uint32_t a = kpage + sg * 128 + (((chunk & 7) ^ (sg & 7)) << 4);
                            uint32_t ka[4];
                            ldsm_x4(a, ka);
                            mma_bf16(sacc, ka, qb[ks][0], qb[ks][1]);
                        }
                    }
                    // sacc: keys g8, g8+8 (rows) x queries 2t, 2t+1 (columns)
                    if (valid < 16) {
                        if (g8 >= valid) sacc[0] = sacc[1] = -INFINITY;
                        if (g8 + 8 >= valid) sacc[2] = sacc[3] = -INFINITY;
                    }
                    float rmax[2] = {fmaxf(sacc[0], sacc[2]), fmaxf(sacc[1], sacc[3])};
                    float corr[2], msub[2];
#pragma unroll
                    for (int j = 0; j < 2; j++) {
                        rmax[j] = fmaxf(rmax[j], __shfl_xor_sync(0xffffffffu, rmax[j], 4));
                        rmax[j] = fmaxf(rmax[j], __shfl_xor_sync(0xffffffffu, rmax[j], 8));
                        rmax[j] = fmaxf(rmax[j], __shfl_xor_sync(0xffffffffu, rmax[j], 16));
                        float mnew = fmaxf(m_run[j], rmax[j]);
                        msub[j] = mnew == -INFINITY ? 0.f : mnew;
                        corr[j] = m_run[j] == -INFINITY ? 0.f : exp2f(m_run[j] - msub[j]);
                        m_run[j] = mnew;
                    }
                    float p0 = exp2f(sacc[0] - msub[0]), p1 = exp2f(sacc[1] - msub[1]);
                    float p2 = exp2f(sacc[2] - msub[0]), p3 = exp2f(sacc[3] - msub[1]);
                    l_run[0] = l_run[0] * corr[0] + (p0 + p2);
                    l_run[1] = l_run[1] * corr[1] + (p1 + p3);
                    // P^T as the B operand of O^T += V^T P^T: transpose the two 8x8 blocks across the warp
                    uint32_t pb0 = movmatrix_trans(pack_bf16(p0, p1)), pb1 = movmatrix_trans(pack_bf16(p2, p3));
                    if (__any_sync(0xffffffffu, corr[0] != 1.f || corr[1] != 1.f)) {
#pragma unroll
                        for (int mb = 0; mb < MB; mb++) {
                            o[mb][0] *= corr[0];
                            o[mb][1] *= corr[1];
                            o[mb][2] *= corr[0];
                            o[mb][3] *= corr[1];
                        }
                    }
                    {
                        int r = (lane & 7) + ((lane >> 4) << 3);  // key row
                        int cb = (lane >> 3) & 1;                 // which 8-dim half of the 16-dim block
#pragma unroll
                        for (int mb = 0; mb < MB; mb++) {
                            int chunk = mb * 2 + cb;
                            int sg = r * HALVES + (chunk >> 3);
                            uint32_t a = vpage + sg * 128 + (((chunk & 7) ^ (sg & 7)) << 4);
                            uint32_t va[4];
                            ldsm_x4_trans(a, va);
                            mma_bf16(o[mb], va, pb0, pb1);
                        }
                    }
                }
                __syncwarp();
                // (the last stage is the fold's scratch first)
                if (lane == 0 && t + 1 < t1) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty_bar(s)) : "memory");
            }
            if (!ok) {
                if (lane == 0) report(p.status, kStatusWaitExpired, 310 + warp);
                return;
            }
#pragma unroll
            for (int j = 0; j < 2; j++) {  // the lanes' shares of the running sums
                l_run[j] += __shfl_xor_sync(0xffffffffu, l_run[j], 4);
                l_run[j] += __shfl_xor_sync(0xffffffffu, l_run[j], 8);
                l_run[j] += __shfl_xor_sync(0xffffffffu, l_run[j], 16);
            }
            if (round == 0) DBT_TL_MARK(1);
            // ---- fold the four warps' states.  Each leaves its own in its page of the last stage, which nobody else touches
            // ([8 queries][DH + 4], then (m, l) of each), and every thread adds four consecutive outputs of a query over the
            // four, as (0 + 2) + (1 + 3) like the 16-row form.  (Three rounds through one slot of scratch with six barriers, the outputs written by one warp in 4-byte
            // pieces, made a step of one sequence 3 % slower.)
            {
                constexpr int FN = DH + 4;
                static_assert((8 * FN + 16) * 4 <= 2 * Cfg::kPageBytes, "a warp's state fits its page");
                const int c = (lane & 3) * 2;
                float *last = reinterpret_cast<float *>(gen + (it - 1) % STAGES * Cfg::kStageBytes);
                constexpr int WS = 2 * Cfg::kPageBytes / 4;  // floats between two warps' states
                float *st = last + warp * WS;
                __syncwarp();
#pragma unroll
                for (int mb = 0; mb < MB; mb++) {
                    st[(size_t)c * FN + mb * 16 + g8] = o[mb][0];
                    st[(size_t)(c + 1) * FN + mb * 16 + g8] = o[mb][1];
                    st[(size_t)c * FN + mb * 16 + g8 + 8] = o[mb][2];
                    st[(size_t)(c + 1) * FN + mb * 16 + g8 + 8] = o[mb][3];
                }
                if (g8 == 0) {
                    *reinterpret_cast<float2 *>(st + 8 * FN + 2 * c) = make_float2(m_run[0], l_run[0]);
                    *reinterpret_cast<float2 *>(st + 8 * FN + 2 * c + 2) = make_float2(m_run[1], l_run[1]);
                }
                consumer_sync();
                constexpr int VQ = DH / 4;
                for (int idx = tid; idx < nq_act * VQ; idx += 128) {
                    const int q = idx / VQ, e = idx % VQ * 4;
                    float2 ml[kAttWarps];
                    float4 X[kAttWarps];
#pragma unroll
                    for (int w = 0; w < kAttWarps; w++) {
                        ml[w] = *reinterpret_cast<const float2 *>(last + w * WS + 8 * FN + 2 * q);
                        X[w] = *reinterpret_cast<const float4 *>(last + w * WS + q * FN + e);
                    }
                    // state a := state a (+) state b; which of the two products is rounded first is part of the result
                    auto take = [&](int a, int b) {
                        const float M = fmaxf(ml[a].x, ml[b].x);
                        const float fa = ml[a].x == -INFINITY ? 0.f : exp2f(ml[a].x - M), fb = ml[b].x == -INFINITY ? 0.f : exp2f(ml[b].x - M);
                        ml[a] = make_float2(M, fmaf(ml[b].y, fb, ml[a].y * fa));
                        X[a] = make_float4(fmaf(X[a].x, fa, X[b].x * fb), fmaf(X[a].y, fa, X[b].y * fb), fmaf(X[a].z, fa, X[b].z * fb),
                                           fmaf(X[a].w, fa, X[b].w * fb));
                    };
                    take(0, 2);
                    take(1, 3);
                    take(0, 1);
                    if (nseg == 1) {
                        // the pair's only segment: normalise and write the head's output
                        const int row = out_row(q / p.G), hq = g * p.G + q % p.G;
                        const float inv = 1.f / ml[0].y;
                        store_split4(p.Ob, (size_t)row * q_dim + (size_t)hq * DH + e, p.lo_off,
                                     make_float4(X[0].x * inv, X[0].y * inv, X[0].z * inv, X[0].w * inv));
                    } else {
                        *reinterpret_cast<float4 *>(out + (size_t)q * DH + e) = X[0];
                        if (e == 0) *reinterpret_cast<float2 *>(out + 16 * DH + 2 * q) = ml[0];  // base-2 units
                    }
                }
                if (nseg > 1) __threadfence();
                if (dealt(round + 1) < Sg) {  // the stage goes back to the producer
                    hand_over(round);
                    consumer_sync();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty_bar((it - 1) % STAGES)) : "memory");
                }
            }
        }
        // ---- merging a pair's segments.  Up to kAttSingle segments: the last one to arrive merges them
        // all, in segment order, and writes the output.  More: the segments form groups of kAttGroup;
        // the last arrival of a group merges it in place into the group's first slot, and the last
        // group to finish merges the group results: two short merges on several CTAs instead of one
        // long one on a single CTA (a pair of a 32k-token sequence has ~35 segments).
        // merge n partials at slots pbase + j * slot_stride; final: normalise and write the output,
        // else leave the merged (unnormalised) state in the first slot
        // A thread takes four consecutive outputs of up to two query rows, eight partials of each in flight: up to eight
        // query rows need one round of loads per eight partials.  (Two single outputs per thread took a round per 256
        // outputs: 5 us behind the last segment at 4 query rows, 9 at 8; now about 2.)
        // Four query rows at d_h 128 (or eight at 64) leave one such piece per thread: then sixteen partials of it.  (Eight, and the
        // second piece's idle arithmetic, made a primary-only step of two sequences of 9139 positions 12 us slower.)
        // The number of query rows is the step's, so the choice differs between a grouped and a primary-only step of the same
        // batch: both forms fold eight partials per common maximum, in the same order, and round alike.
        auto merge_rows = [&](auto pieces, float *pbase, int slot_stride, int n, bool final) {
            constexpr int A = decltype(pieces)::value, J = 16 / A;  // pieces of a thread, partials of each in flight
            const size_t sstr = (size_t)slot_stride * 16 * (DH + 2);
            constexpr int VQ = DH / 4;  // 16-byte pieces of a query row
            for (int idx0 = tid; idx0 < nq_act * VQ; idx0 += A * 128) {
                float M[A], L[A];
                float4 X[A];
                bool act[A];
                int ee[A], qq[A];
#pragma unroll
                for (int a = 0; a < A; a++) {
                    const int idx = idx0 + a * 128;
                    M[a] = -INFINITY, L[a] = 0.f, X[a] = make_float4(0.f, 0.f, 0.f, 0.f);
                    act[a] = idx < nq_act * VQ;
                    qq[a] = act[a] ? idx / VQ : 0;
                    ee[a] = act[a] ? idx % VQ * 4 : 0;
                }
                for (int sb = 0; sb < n; sb += J) {
                    float2 ml[A][J];
                    float4 ov[A][J];
#pragma unroll
                    for (int a = 0; a < A; a++)
#pragma unroll
                        for (int j = 0; j < J; j++) {
                            const bool on = act[a] && sb + j < n;
                            const float *pp = pbase + (size_t)(sb + j) * sstr;
                            ml[a][j] = on ? __ldcg(reinterpret_cast<const float2 *>(pp + 16 * DH) + qq[a]) : make_float2(-INFINITY, 0.f);
                            ov[a][j] = on ? ldcg4(pp + (size_t)qq[a] * DH + ee[a]) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                    for (int h = 0; h < J; h += 8) {  // eight at a time, however many are in flight
                        if (sb + h >= n) break;
#pragma unroll
                        for (int a = 0; a < A; a++) {
                            float Mn = M[a];
#pragma unroll
                            for (int j = h; j < h + 8; j++) Mn = fmaxf(Mn, ml[a][j].x);
                            const float sc = M[a] == -INFINITY ? 0.f : exp2f(M[a] - Mn);
                            L[a] *= sc;
                            X[a].x *= sc, X[a].y *= sc, X[a].z *= sc, X[a].w *= sc;
#pragma unroll
                            for (int j = h; j < h + 8; j++) {
                                const float f = ml[a][j].x == -INFINITY ? 0.f : exp2f(ml[a][j].x - Mn);
                                L[a] = fmaf(ml[a][j].y, f, L[a]);
                                X[a].x = fmaf(ov[a][j].x, f, X[a].x), X[a].y = fmaf(ov[a][j].y, f, X[a].y);
                                X[a].z = fmaf(ov[a][j].z, f, X[a].z), X[a].w = fmaf(ov[a][j].w, f, X[a].w);
                            }
                            M[a] = Mn;
                        }
                    }
                }
#pragma unroll
                for (int a = 0; a < A; a++) {
                    if (!act[a]) continue;
                    if (final) {
                        const int row = packed ? item_row0(item) + qq[a] / p.G : out_row(qq[a] / p.G);
                        const int h = g * p.G + qq[a] % p.G;
                        store_split4(p.Ob, (size_t)row * q_dim + (size_t)h * DH + ee[a], p.lo_off,
                                     make_float4(X[a].x / L[a], X[a].y / L[a], X[a].z / L[a], X[a].w / L[a]));
                    } else {
                        // this thread is the only reader of the first slot's elements (q, e..)
                        *reinterpret_cast<float4 *>(pbase + (size_t)qq[a] * DH + ee[a]) = X[a];
                        if (ee[a] == 0) {
                            sc_m[qq[a]] = M[a];
                            sc_l[qq[a]] = L[a];
                        }
                    }
                }
            }
            if (!final) {
                consumer_sync();  // every thread has read the first slot's (m, l): now they may change
                if (tid < nq_act) {
                    pbase[16 * DH + 2 * tid] = sc_m[tid];
                    pbase[16 * DH + 2 * tid + 1] = sc_l[tid];
                }
                __threadfence();
            }
        };
        auto merge = [&](float *pbase, int slot_stride, int n, bool final) {
            if (nq_act * (DH / 4) <= 128) merge_rows(std::integral_constant<int, 1>{}, pbase, slot_stride, n, final);
            else merge_rows(std::integral_constant<int, 2>{}, pbase, slot_stride, n, final);
        };
        auto arrive = [&](int *counter, int arrivals) {  // true in the CTA that arrives last
            consumer_sync();
            if (tid == 0) {
                int tkt = atomicAdd(counter, 1);
                int last = tkt == arrivals - 1;
                if (last) {
                    atomicExch(counter, 0);
                    __threadfence();
                }
                flag[0] = last;
            }
            consumer_sync();
            return flag[0] != 0;
        };
        if (nseg > 1) {
            float *slot0 = p.part + (size_t)first_slot * 16 * (DH + 2);
            if (nseg <= kAttSingle) {
                if (arrive(p.tickets + pair, nseg)) merge(slot0, 1, nseg, true);
            } else {
                int gi = seg / kAttGroup, ngroups = (nseg + kAttGroup - 1) / kAttGroup;
                int gs = min(kAttGroup, nseg - gi * kAttGroup);
                if (arrive(p.tickets2 + (size_t)pair * kAttMaxGroups + gi, gs)) {
                    merge(slot0 + (size_t)gi * kAttGroup * 16 * (DH + 2), 1, gs, false);
                    if (arrive(p.tickets + pair, ngroups)) merge(slot0, kAttGroup, ngroups, true);
                }
            }
        }
        if (round == 0) DBT_TL_MARK(2);
    }
    if (riding) pdl_wait();
#ifdef DBT_TL_ATT_ALL
    {  // every CTA leaves a record: mark 3 carries (SM id << 16 | block index)
        unsigned smid;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        tlx_[3] = ((unsigned long long)smid << 16) | blockIdx.x;
    }
    DBT_TL_END_IF(true, "attall");
#else
    DBT_TL_END("attentio");
#endif
}

// The K/V pool as a 4-D bf16 tensor (64 columns, 64-column piece of a row, row, K|V plane of a
// layer); rows = (layer, K|V, page, head, slot).  One box {64, d_h/64, 16, 2} brings a page's K and V
// of one KV head.  The row extent stops one plane short so that plane 1 of the last layer stays
// inside the allocation.
inline bool make_kv_page_map(CUtensorMap *map, const void *pool, uint64_t total_rows, uint64_t plane_rows, int head_dim) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || total_rows >= (1ull << 31) || total_rows <= plane_rows) return false;
    cuuint64_t dims[4] = {64, (cuuint64_t)head_dim / 64, total_rows - plane_rows, 2};
    cuuint64_t strides[3] = {128, (cuuint64_t)head_dim * 2, plane_rows * (cuuint64_t)head_dim * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)head_dim / 64, 16, 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(pool), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace dbt
