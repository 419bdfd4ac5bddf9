// GEMMs of a prompt chunk on pairs of SMs (tcgen05 cta_group::2), each with the elementwise work that follows it.
//
// A prompt chunk (Section 4.4 item 1: the primary path alone walks the prompt) is a dense contraction: up to 18944
// rows against every matrix of the layer.  Its bound is the tensor pipe, at twice the useful FLOPs because the
// activations are two bf16 planes (x = hi + lo, see dbt_gemm_tc.cuh).  What keeps the pipe busy here:
//   - a pair of CTAs (a cluster of two on neighbouring SMs) works on one 256-row x N-feature tile: one MMA of M = 256
//     reads 128 activation rows from each CTA and half of the weight tile from each, so a k-tile of 64 costs an SM
//     48 KB of shared-memory fill for 1024 cycles of MMA at N = 256 (a lone CTA with the same accumulators: 80 KB);
//   - persistent CTAs with two accumulators in tensor memory: the epilogue of one tile runs while the next tile's
//     MMAs are issued, and the TMA ring never drains between tiles;
//   - the rows are on the M side, so a thread of the epilogue holds one row and N / 2 consecutive features of it:
//     rotary pairs, gate / up pairs and a row's share of sum(S^2) meet in one thread, and the kernels that used to
//     follow each GEMM (residual, SwiGLU, rotation + cache append) and their fp32 partials are gone.
// Measured per layer and 2048 rows of the 1B model against one CTA per 256-row x 256-feature tile with the kernels in
// between: gate|up with SwiGLU 204 -> 122 us (1.55 PFLOP/s of tensor work), down + residual 86 + 15 -> 74, Q|K|V + rotation
// and append 61 + 25 -> 62, O + residual 41 + 15 -> 39.
//
// Few row tiles (decode steps of 129 to 256 stacked rows, short prompts) leave too few tiles for the chip: the contracted
// width of a tile is then split over 2 to 4 pairs of one cluster.  Each CTA owns a slice of the tile's columns, the others
// write their partial sums of it into its (by then idle) ring through distributed shared memory, and it adds them in split
// order and runs the epilogue of that slice: no partials in memory, no kernel to sum them.
//
// Roles: warp 0 TMA producer, warp 1 MMA issuer (of the pair's first CTA) and TMEM owner, warps 2..9 epilogue (two per
// TMEM lane quadrant, each taking half of the tile's columns).  Every wait is bounded: on expiry the CTA records
// kStatusWaitExpired, stops storing, waits (bounded) for the loads in flight, and still reaches the cluster barrier that the pair
// leaves by.
#pragma once

#include "dbt_gemm_tc.cuh"

namespace dbt {

enum PgMode {
    PG_STORE = 0,   // Y = acc (fp32 rows)
    PG_QKV = 1,     // 1/rms, RoPE on Q and K, Q out, K and V appended to the paged cache
    PG_RESID = 2,   // S += acc; the next GEMM's input g * S (two planes) and each row's share of sum(S^2)
    PG_GATEUP = 3,  // H = SiLU(rs * gate) * (rs * up), two planes
    PG_COMBINE = 4,  // PG_RESID behind an MoE layer's shared expert: the routed experts' rows join the residual too,
                     // S += acc + sum_j wts[r][j] Y[pos[r][j]] over the row's k selections (idx < 0: none)
};

constexpr int kPgM = 256;         // activation rows of a pair's tile
constexpr int kPgEpiWarps = 8;
constexpr int kPgThreads = 64 + 32 * kPgEpiWarps;
constexpr int kPgABytes = 2 * 128 * kTcK * 2;  // both planes of a CTA's 128 rows, one k-tile

struct PgSeg {
    int tile0;  // first feature tile of this matrix
    int n_out;  // its features (PG_GATEUP: of each of the two matrices)
    int col0;   // PG_STORE: its first column of P
};

// Rows of the boundary step that ride behind a chunk's own rows (RIDE): sequence b's K rows -- the primary's and its branches' at the
// position behind the chunk -- stand in one group of 32, row row0 + b / spg * 32 + path * spg + b % spg, so that one warp of an
// epilogue holds them and a branch reaches its primary row by a shuffle.
struct RideRows {
    int row0, spg, K, B;  // (K == 0: none)
    __host__ __device__ int row(int path, int b) const { return row0 + b / spg * 32 + path * spg + b % spg; }
    // the path and the sequence of a row; false: a row of no sequence
    __device__ bool locate(int r, int &path, int &b) const {
        const int q = r - row0, l = q & 31;
        path = l / spg;
        b = (q >> 5) * spg + l % spg;
        return path < K && b < B;
    }
};

struct PgParams {
    int K, R, m_tiles, tiles;  // tiles: m_tiles x feature tiles
    // Order of the tiles: groups of m_group row tiles, in a group feature tile by feature tile.  The pairs that run at
    // once then share about as many row tiles as weight tiles (9 x 8 of 74), whatever the chunk: with all 32 row tiles of
    // an 8192-row chunk side by side the 8B shape's gate|up re-read its 134 MB of activations from HBM (97 us per row tile).
    int m_group;
    int splits, kt_per_split;  // pairs per tile (1 to 4; a cluster is 2 * splits CTAs); k-tiles of each
    PgSeg seg[3];
    int nseg;
    int *status;
    // row factor 1/rms from the shares of sum(S^2) (nullptr: 1)
    const float *ss_in;
    int ss_tiles, ss_ld, d_norm;
    float eps;
    // PG_STORE
    float *P;
    int ldp;
    // PG_RESID
    float *S;
    const float *g_next;  // nullptr: 1
    __nv_bfloat16 *X;
    size_t x_lo;
    float *ss_out;  // [(feature tile * splits + split) * 2 + half][ss_ld]
    int d;
    // PG_COMBINE
    const float *Y;
    const int32_t *sel_idx, *sel_pos;
    const float *sel_wts;
    int kmax, k;
    // PG_GATEUP
    __nv_bfloat16 *H;
    size_t h_lo;
    int F;
    // PG_QKV: the segments are Q, K, V from number `first` on (1: K and V alone, the last layer of a chunk)
    int first;
    float *Q;
    __nv_bfloat16 *Qb;  // the prompt attention kernel's queries: bf16, times q_scale (nullptr: Q, fp32)
    float q_scale;
    int B, cn, dh, n_q, n_kv, num_pages, pt_stride;
    const float2 *rope;
    const int32_t *seq_len, *page_table;
    __nv_bfloat16 *kpool, *vpool;
    // RIDE: R counts the riding rows, `own` the chunk's
    RideRows ride;
    int own;
    const float *ride_coup;  // a, b or c (nullptr: no coupling)
    float *ride_q;           // PG_QKV: their queries, fp32, [path * B + sequence][q_dim]
};

template <int N>
struct PgCfg {
    static constexpr int kBBytes = N / 2 * kTcK * 2;  // this CTA's half of the weight tile
    static constexpr int kStageBytes = kPgABytes + kBBytes;
    static constexpr int kStages = N >= 128 ? 4 : 5;
    static constexpr int kStagingBytes = kPgEpiWarps * 4096;
    static constexpr int kAccStride = N > 128 ? 256 : N > 64 ? 128 : 64;  // TMEM columns between the two accumulators
    static constexpr int kTmemCols = 2 * kAccStride;
    static_assert((kTmemCols & (kTmemCols - 1)) == 0 && kTmemCols >= 32 && kTmemCols <= 512, "an allocation of tensor memory");
    static_assert(N % 32 == 0 && N <= 256, "N of a cta_group::2 MMA with M = 256");
    static constexpr int kSmemBytes = kStages * kStageBytes + kStagingBytes + 1024 + 256;
    static_assert(kSmemBytes <= 227 * 1024, "shared memory of one SM");
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The shared::cluster address of the same location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa_u32(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}
// The two halves of it: all threads arrive, and wait later.  The arrival orders no data (relaxed).
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// mbar_wait with cluster scope: the arrivals come from both CTAs of the pair.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, uint64_t limit = kWaitCycles) {
    uint32_t done = 0;
    long long t0 = 0;
    while (true) {
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        const long long t = clock64();
        if (t0 == 0) t0 = t;
        else if ((unsigned long long)(t - t0) > limit) return false;
    }
}
// Loads of a CTA pair: into this CTA's shared memory, completing on a barrier of either CTA (no multicast).
__device__ __forceinline__ void tma2_load_2d_hint(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, uint64_t hint) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, "
        "%4}], [%2], %5;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "l"(hint)
        : "memory");
}
__device__ __forceinline__ void tma2_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
// kind::f16, bf16 x bf16 -> fp32, K-major operands, M = 256 over the pair, N = n.
__host__ __device__ constexpr uint32_t umma2_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kPgM >> 4) << 24);
}
__device__ __forceinline__ void umma2_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
// Arrive on the barrier at this offset in both CTAs of the pair (mask: their ranks in the cluster) once the MMAs issued so
// far are done.
__device__ __forceinline__ void umma2_commit(uint32_t bar, uint32_t mask = 3) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((uint16_t)mask)
        : "memory");
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}
// Eight consecutive values as bf16 hi and lo pieces of 16 bytes.
__device__ __forceinline__ void split8(const float *v, uint4 &hi, uint4 &lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float a = v[2 * i], b = v[2 * i + 1];
        const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
        h[i] = *reinterpret_cast<const uint32_t *>(&p);
        l[i] = pack2(a - __low2float(p), b - __high2float(p));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Sixteen consecutive values as bf16.
__device__ __forceinline__ void store16(__nv_bfloat16 *dst, const float *x) {
#pragma unroll
    for (int i = 0; i < 2; i++)
        *reinterpret_cast<uint4 *>(dst + 8 * i) = make_uint4(pack2(x[8 * i], x[8 * i + 1]), pack2(x[8 * i + 2], x[8 * i + 3]),
                                                             pack2(x[8 * i + 4], x[8 * i + 5]), pack2(x[8 * i + 6], x[8 * i + 7]));
}

template <int N, int MODE, bool RIDE = false>
__global__ void __launch_bounds__(kPgThreads, 1)
gemm_prompt_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
                   const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmX, const PgParams p) {
    using Cfg = PgCfg<N>;
    DBT_TL_DECL;
    DBT_TL_SHARED;
    constexpr int STAGES = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (ring - raw);
    constexpr int kBarOff = STAGES * Cfg::kStageBytes + Cfg::kStagingBytes;
    const uint32_t bars = ring + kBarOff;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    auto acc_full = [&](int a) { return bars + 8u * (2 * STAGES + a); };
    auto acc_empty = [&](int a) { return bars + 8u * (2 * STAGES + 2 + a); };
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(gen + kBarOff + 8 * (2 * STAGES + 4));
    static_assert(8 * (2 * STAGES + 4) + 4 <= 256, "barrier area");

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // rank in the pair; the pair's first CTA; which part of the contracted width
    const int S = p.splits;
    const uint32_t crank = cluster_rank(), rank = crank & 1, lead = crank & ~1u, pair_mask = 3u << lead;
    const int split = (int)(crank >> 1);
    const int pair = blockIdx.x / (2 * S), npairs = gridDim.x / (2 * S);  // (splits > 1: one tile per cluster)
    const int kt0 = split * p.kt_per_split, nkt = min(p.kt_per_split, (p.K + kTcK - 1) / kTcK - kt0);

    if (tid == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; a++) {
            mbar_init(acc_full(a), 1);
            mbar_init(acc_empty(a), 2 * kPgEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                     "r"((uint32_t)Cfg::kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers exist before either signals the other's
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_holder;
    pdl_launch_dependents();

    const int n_tiles = p.tiles / p.m_tiles;
    auto tile_of = [&](int t, int &mt, int &nt) {
        const int per = p.m_group * n_tiles, gr = t / per, m0 = gr * p.m_group, in = t - gr * per, gm = min(p.m_group, p.m_tiles - m0);
        nt = in / gm;
        mt = m0 + in - nt * gm;
    };
    // feature tile -> matrix, first feature
    auto seg_of = [&](int nt) { return p.nseg > 2 && nt >= p.seg[2].tile0 ? 2 : p.nseg > 1 && nt >= p.seg[1].tile0 ? 1 : 0; };
    constexpr int kTileF = MODE == PG_GATEUP ? N / 2 : N;  // features of one tile (gate|up: N / 2 of each matrix)

    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer: this CTA's 128 rows of both planes and its half of the weight tile, completing on the
            // first CTA's barrier.  Weights do not depend on the kernel before: the first ring of them goes out early.
            tma_prefetch_desc(&tmW0);
            tma_prefetch_desc(&tmX);
            const uint64_t pol = l2_evict_first_policy();
            auto load_w = [&](int s, int nt, int kt) {
                const int sg = seg_of(nt);
                const int f0 = (nt - p.seg[sg].tile0) * kTileF;
                const CUtensorMap *tw;
                int row;
                if (MODE == PG_GATEUP) {  // first CTA: the gate rows, second CTA: the up rows of the same features
                    tw = rank == 0 ? &tmW0 : &tmW1;
                    row = f0;
                } else {
                    tw = sg == 0 ? &tmW0 : sg == 1 ? &tmW1 : &tmW2;
                    row = f0 + (int)rank * (N / 2);
                }
                tma2_load_2d_hint(ring + s * Cfg::kStageBytes + kPgABytes, tw, mapa_u32(full_bar(s), lead), kt * kTcK, row, pol);
            };
            auto load_x = [&](int s, int mt, int kt) {
                tma2_load_3d(ring + s * Cfg::kStageBytes, &tmX, mapa_u32(full_bar(s), lead), kt * kTcK, mt * kPgM + (int)rank * 128, 0);
            };
            const int npre = pair < p.tiles ? min(STAGES, nkt) : 0;
            int mt, nt;
            tile_of(pair, mt, nt);
            for (int i = 0; i < npre; i++) {
                if (rank == 0) mbar_expect_tx(full_bar(i), 2 * Cfg::kStageBytes);
                load_w(i, nt, kt0 + i);
            }
            pdl_wait();
            DBT_TL_WAITED;
            for (int i = 0; i < npre; i++) load_x(i, mt, kt0 + i);
            int it = 0;  // stages requested so far, over all tiles
            for (int t = pair; t < p.tiles && ok; t += npairs) {
                tile_of(t, mt, nt);
                for (int kt = 0; kt < nkt; kt++, it++) {
                    if (it < npre) continue;
                    const int s = it % STAGES;
                    if (it >= STAGES) ok = mbar_wait_cluster(empty_bar(s), ((it / STAGES) - 1) & 1);
                    if (!ok) break;
                    if (rank == 0) mbar_expect_tx(full_bar(s), 2 * Cfg::kStageBytes);
                    load_w(s, nt, kt0 + kt);
                    load_x(s, mt, kt0 + kt);
                }
            }
            DBT_TL_MARK(0);
            if (!ok) report(p.status, kStatusWaitExpired, 600);
            // The pair's last loads have landed before either CTA leaves, also where a wait ran out (they complete on the first CTA's
            // barriers; the second leaves by the cluster barrier).
            if (rank == 0)
                for (int j = max(0, it - STAGES); j < it; j++) mbar_wait_cluster(full_bar(j % STAGES), (j / STAGES) & 1, kWaitCycles / STAGES);
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // ---- MMA issuer of the pair
            constexpr uint32_t idesc = umma2_idesc(N);
            int it = 0, n_acc = 0;
            for (int t = pair; t < p.tiles && ok; t += npairs, n_acc++) {
                const int a = n_acc & 1;
                if (n_acc >= 2) ok = mbar_wait_cluster(acc_empty(a), ((n_acc >> 1) - 1) & 1);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem_base + a * Cfg::kAccStride;
                for (int kt = 0; kt < nkt; kt++, it++) {
                    const int s = it % STAGES;
                    ok = mbar_wait_cluster(full_bar(s), (it / STAGES) & 1);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t st = ring + s * Cfg::kStageBytes;
                    const uint64_t bdesc = umma_smem_desc(st + kPgABytes);
#pragma unroll
                    for (int part = 0; part < 2; part++) {
                        const uint64_t adesc = umma_smem_desc(st + part * (kPgABytes / 2));
#pragma unroll
                        for (int k = 0; k < kTcK / 16; k++) umma2_f16(acc, adesc + 2 * k, bdesc + 2 * k, idesc, (kt | part | k) != 0);
                    }
                    umma2_commit(empty_bar(s), pair_mask);
                }
                if (ok) umma2_commit(acc_full(a), pair_mask);
            }
            if (!ok) report(p.status, kStatusWaitExpired, 601);
        }
    }
    if (warp < 2) {
        if (S > 1) {  // the exchange's two barriers (acc_ready)
            __syncwarp();
            cluster_sync_all();
            cluster_sync_all();
        }
    } else {
        // ---- epilogue: TMEM lane = row, TMEM column = feature
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        float *stg = reinterpret_cast<float *>(gen + STAGES * Cfg::kStageBytes + (warp - 2) * 4096);
        pdl_wait();
        int n_acc = 0;
        for (int t = pair; t < p.tiles; t += npairs, n_acc++) {
            const int a = n_acc & 1;
            int mt, nt;
            tile_of(t, mt, nt);
            const int sg = seg_of(nt), f0 = (nt - p.seg[sg].tile0) * kTileF;
            const int row0 = mt * kPgM + (int)rank * 128 + quad * 32, row = row0 + lane;
            // riding rows: this warp's 32 rows are a group of them; the lane's path and sequence, the lane of its primary row
            const bool rides = RIDE && p.ride.K > 0 && row0 >= p.ride.row0;
            int path = 0, rb = 0;
            const bool on = !RIDE ? row < p.R : rides ? p.ride.locate(row, path, rb) : row < p.own;
            const int twin = rides ? lane % p.ride.spg : lane;
            // adds coup[f + i] times the primary row's value to a branch row's, of sixteen features
            auto couple = [&](float *x, int f, int n_feat) {
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const float y = __shfl_sync(0xffffffffu, x[i], twin), a = f + i < n_feat ? p.ride_coup[f + i] : 0.f;
                    if (path > 0) x[i] = fmaf(a, y, x[i]);
                }
            };
            float rs = 1.f;
            if (MODE == PG_QKV || MODE == PG_GATEUP || MODE == PG_STORE)
                rs = row_scale(p.ss_in, p.ss_tiles, p.ss_ld, on ? row : 0, p.d_norm, p.eps);
            const uint32_t tacc = lane_base + a * Cfg::kAccStride;
            auto acc_ready = [&] {
                bool r = mbar_wait_cluster(acc_full(a), (n_acc >> 1) & 1);
                ok = r = __all_sync(0xffffffffu, r);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                DBT_TL_SHARED_MARK(warp == 2 && lane == 0, 1);
                if (S > 1) {
                    // the slices that other CTAs own go to their rings, [source][4-column group][row][4]
                    cluster_sync_all();  // every pair's MMAs are done: the rings are idle
                    if (r) {
                        const int w = N / S;
#pragma unroll 1
                        for (int c = half * (N / 2); c < (half + 1) * (N / 2); c += 16) {
                            const int o = c / w;
                            if (o == split) continue;
                            uint32_t v[16];
                            __syncwarp();
                            tmem_ld16_issue(tacc + c, v);
                            tmem_ld_wait();
                            const int slot = split < o ? split : split - 1;
                            const uint32_t dst = mapa_u32(ring + (uint32_t)(((slot * w + c - o * w) * 128 + (quad * 32 + lane) * 4) * 4), (uint32_t)(2 * o) + rank);
#pragma unroll
                            for (int q = 0; q < 4; q++)
                                asm volatile("st.shared::cluster.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst + q * 128 * 16), "r"(v[4 * q]), "r"(v[4 * q + 1]),
                                             "r"(v[4 * q + 2]), "r"(v[4 * q + 3])
                                             : "memory");
                        }
                    }
                    __syncwarp();
                    cluster_sync_all();
                }
                DBT_TL_SHARED_MARK(warp == 2 && lane == 0, 2);
                return r;
            };
            // Adds the other splits' sums to 16 columns of this CTA's slice, in split order.
            auto add_peers = [&](uint32_t (&v)[16], int c) {
                const int w = N / S, lc = c - split * w;
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int k = 0; k < S; k++) {
                        float4 y = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]), __uint_as_float(v[4 * q + 2]),
                                               __uint_as_float(v[4 * q + 3]));
                        if (k != split)
                            y = *reinterpret_cast<const float4 *>(gen + (size_t)((((k < split ? k : k - 1) * w + lc + 4 * q) * 128 + (quad * 32 + lane) * 4) * 4));
                        x.x += y.x, x.y += y.y, x.z += y.z, x.w += y.w;
                    }
                    v[4 * q] = __float_as_uint(x.x), v[4 * q + 1] = __float_as_uint(x.y);
                    v[4 * q + 2] = __float_as_uint(x.z), v[4 * q + 3] = __float_as_uint(x.w);
                }
            };
            if constexpr (MODE == PG_STORE || MODE == PG_RESID || MODE == PG_COMBINE) {
                // Chunks of 32 columns go through a 4 KB staging tile of the warp (16-byte pieces, XOR-swizzled by row),
                // so that global memory sees 128-byte row pieces: lane l then holds columns 4 (l % 8) .. of row 4 i + l / 8.
                // What a chunk adds to the accumulator is requested a chunk ahead (the first before the accumulator is
                // there): the epilogue would otherwise wait for memory once per chunk, longer than the next tile's MMAs take.
                // PG_COMBINE has three times the rows in flight and takes them half a chunk at a time: with a whole chunk's 96
                // registers of them some spilled, and a spill waits for its load (9472 rows of the MoE model, K = 1408: 180 us, now
                // 132; 81 of it are left without the routed rows).  Fetching those rows into L2 a tile ahead made it 151.
                constexpr bool kResid = MODE != PG_STORE;
                constexpr int kPre = MODE == PG_COMBINE ? 2 : 0;  // selections whose rows are requested ahead
                constexpr int kAhead = MODE == PG_COMBINE ? 4 : 8;  // in groups of this many of a lane's eight rows
                const int c4 = (lane & 7) * 4, rsub = lane >> 3;
                float sq[8];
#pragma unroll
                for (int i = 0; i < 8; i++) sq[i] = 0.f;
                // this warp's columns: half of the CTA's slice, at least 32 (a slice of 32 leaves four warps without)
                const int wide = max(32, N / (2 * S)), cbase = split * (N / S) + half * wide, cend = half * wide < N / S ? wide : 0;
                int ps[kPre + 1];
                float wt[kPre + 1];
                if (MODE == PG_COMBINE) {  // this lane's own row's first selections
#pragma unroll
                    for (int j = 0; j < kPre; j++) {
                        const size_t o = (size_t)row * p.kmax + j;
                        const bool sel = on && j < p.k && __ldcg(p.sel_idx + o) >= 0;
                        ps[j] = sel ? __ldcg(p.sel_pos + o) : -1;
                        wt[j] = sel ? __ldcg(p.sel_wts + o) : 0.f;
                    }
                }
                float4 s4[kAhead], y4[kPre > 0 ? kPre : 1][kAhead];
                auto request = [&](int c, int i0) {
                    const int col = f0 + cbase + c + c4;
                    const bool con = col < p.seg[sg].n_out;
#pragma unroll
                    for (int i = 0; i < kAhead; i++) {
                        const int rl = (i0 + i) * 4 + rsub, r = row0 + rl;
                        s4[i] = con && r < p.R ? ldcg4(p.S + (size_t)r * p.d + col) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int j = 0; j < kPre; j++) {
                            const int q = __shfl_sync(0xffffffffu, ps[j], rl);
                            y4[j][i] = con && q >= 0 ? ldcg4(p.Y + (size_t)q * p.d + col) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    }
                };
                if (kResid && cend > 0) request(0, 0);
                if (!acc_ready()) break;
#pragma unroll 1
                for (int c = 0; c < cend; c += 32) {
                    const int col = f0 + cbase + c + c4;  // this lane's first column
                    const bool con = col < p.seg[sg].n_out;
                    uint32_t v[2][16];
                    __syncwarp();  // the staging tile has been read
                    tmem_ld16_issue(tacc + cbase + c, v[0]);
                    tmem_ld16_issue(tacc + cbase + c + 16, v[1]);
                    float4 gn = make_float4(1.f, 1.f, 1.f, 1.f);
                    if (kResid && p.g_next && con) gn = load_vec4(p.g_next + col);
                    tmem_ld_wait();
                    if (S > 1) {
                        add_peers(v[0], cbase + c);
                        add_peers(v[1], cbase + c + 16);
                    }
                    if constexpr (RIDE && MODE == PG_RESID) {
                        if (rides && p.ride_coup) {
#pragma unroll
                            for (int h = 0; h < 2; h++) couple(reinterpret_cast<float *>(v[h]), f0 + cbase + c + 16 * h, p.seg[sg].n_out);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        float4 x = make_float4(rs * __uint_as_float(v[j >> 2][(j & 3) * 4]), rs * __uint_as_float(v[j >> 2][(j & 3) * 4 + 1]),
                                               rs * __uint_as_float(v[j >> 2][(j & 3) * 4 + 2]), rs * __uint_as_float(v[j >> 2][(j & 3) * 4 + 3]));
                        *reinterpret_cast<float4 *>(stg + lane * 32 + ((j ^ (lane & 7)) << 2)) = x;
                    }
                    __syncwarp();
#pragma unroll
                    for (int i0 = 0; i0 < 8; i0 += kAhead) {
                        float4 add[kAhead];
                        if (kResid) {
#pragma unroll
                            for (int i = 0; i < kAhead; i++) {
                                float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                                for (int j = 0; j < kPre; j++) {
                                    const float g = __shfl_sync(0xffffffffu, wt[j], (i0 + i) * 4 + rsub);
                                    m.x = fmaf(g, y4[j][i].x, m.x), m.y = fmaf(g, y4[j][i].y, m.y);
                                    m.z = fmaf(g, y4[j][i].z, m.z), m.w = fmaf(g, y4[j][i].w, m.w);
                                }
                                add[i] = make_float4(s4[i].x + m.x, s4[i].y + m.y, s4[i].z + m.z, s4[i].w + m.w);
                            }
                            if (MODE == PG_COMBINE && p.k > kPre && con) {  // wider fan-outs: the further selections' rows
#pragma unroll
                                for (int i = 0; i < kAhead; i++) {
                                    const int r = row0 + (i0 + i) * 4 + rsub;
                                    if (r >= p.R) continue;
                                    for (int j = kPre; j < p.k; j++) {
                                        const size_t o = (size_t)r * p.kmax + j;
                                        if (__ldcg(p.sel_idx + o) < 0) continue;
                                        const float g = __ldcg(p.sel_wts + o);
                                        const float4 y = ldcg4(p.Y + (size_t)__ldcg(p.sel_pos + o) * p.d + col);
                                        add[i].x = fmaf(g, y.x, add[i].x), add[i].y = fmaf(g, y.y, add[i].y);
                                        add[i].z = fmaf(g, y.z, add[i].z), add[i].w = fmaf(g, y.w, add[i].w);
                                    }
                                }
                            }
                            if (i0 + kAhead < 8) request(c, i0 + kAhead);
                            else if (c + 32 < cend) request(c + 32, 0);
                        }
#pragma unroll
                        for (int i = 0; i < kAhead; i++) {
                            const int rl = (i0 + i) * 4 + rsub, r = row0 + rl;
                            float4 x = *reinterpret_cast<const float4 *>(stg + rl * 32 + (((lane & 7) ^ (rl & 7)) << 2));
                            if (!con || r >= p.R) continue;
                            if (MODE == PG_STORE) {
                                *reinterpret_cast<float4 *>(p.P + (size_t)r * p.ldp + p.seg[sg].col0 + col) = x;
                            } else {
                                const size_t o = (size_t)r * p.d + col;
                                x.x += add[i].x, x.y += add[i].y, x.z += add[i].z, x.w += add[i].w;
                                *reinterpret_cast<float4 *>(p.S + o) = x;
                                store_split4(p.X, o, p.x_lo, make_float4(gn.x * x.x, gn.y * x.y, gn.z * x.z, gn.w * x.w));
                                sq[i0 + i] += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
                            }
                        }
                    }
                }
                if (kResid) {
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        float q = sq[i];
                        q += __shfl_xor_sync(0xffffffffu, q, 1);
                        q += __shfl_xor_sync(0xffffffffu, q, 2);
                        q += __shfl_xor_sync(0xffffffffu, q, 4);
                        const int r = row0 + i * 4 + rsub;
                        if ((lane & 7) == 0 && r < p.R) p.ss_out[(size_t)((nt * S + split) * 2 + half) * p.ss_ld + r] = q;
                    }
                }
            } else if constexpr (MODE == PG_GATEUP) {
                if (!acc_ready()) break;
                const int fbase = half * (N / 4);
#pragma unroll 1
                for (int c = 0; c < N / 4; c += 16) {
                    uint32_t vg[16], vu[16];
                    __syncwarp();
                    tmem_ld16_issue(tacc + fbase + c, vg);
                    tmem_ld16_issue(tacc + N / 2 + fbase + c, vu);
                    tmem_ld_wait();
                    float h[16];
#pragma unroll
                    for (int i = 0; i < 16; i++) h[i] = silu(rs * __uint_as_float(vg[i])) * (rs * __uint_as_float(vu[i]));
                    if constexpr (RIDE)
                        if (rides) couple(h, f0 + fbase + c, p.F);
#pragma unroll
                    for (int q = 0; q < 2; q++) {  // F % 8 == 0: pieces of eight features are whole
                        const int f = f0 + fbase + c + q * 8;
                        if (on && f < p.F) {
                            uint4 hi, lo;
                            split8(h + q * 8, hi, lo);
                            const size_t o = (size_t)row * p.F + f;
                            *reinterpret_cast<uint4 *>(p.H + o) = hi;
                            *reinterpret_cast<uint4 *>(p.H + o + p.h_lo) = lo;
                        }
                    }
                }
            } else {
                if (!acc_ready()) break;
                // PG_QKV: the tile holds N / dh whole heads of one of Q, K, V; the two warps of a lane quadrant take the
                // first and the second half of every head's rotation pairs (i, i + dh / 2)
                const int hd = p.dh, hh2 = hd >> 1, span = hd >> 2, mat = sg + p.first;
                const int nh = mat == 0 ? p.n_q : p.n_kv;
                const int b = !on ? 0 : rides ? rb : row / p.cn, pos = ld_mut(p.seq_len + b) + (!on ? 0 : rides ? p.cn : row % p.cn);
                __nv_bfloat16 *kv = nullptr;
                if (mat != 0 && on && path == 0) {
                    const int page = p.page_table[(size_t)b * p.pt_stride + (pos >> 4)];
                    if (page < 0 || page >= p.num_pages) {
                        report(p.status, kStatusBadPage, page);
                    } else {
                        kv = (mat == 1 ? p.kpool : p.vpool) + ((size_t)page * p.n_kv * 16 + (pos & 15)) * hd;
                    }
                }
#pragma unroll 1
                for (int hc = split * (N / S) / hd; hc < (split + 1) * (N / S) / hd; hc++) {  // (N / splits holds whole heads)
                    const int head = f0 / hd + hc;
#pragma unroll 1
                    for (int j = 0; j < span; j += 16) {
                        const int i0 = half * span + j;  // rotation pairs i0 .. i0 + 15
                        uint32_t v0[16], v1[16];
                        __syncwarp();
                        tmem_ld16_issue(tacc + hc * hd + i0, v0);
                        tmem_ld16_issue(tacc + hc * hd + hh2 + i0, v1);
                        float4 cs[8];
                        if (mat != 2) {
                            const float4 *tab = reinterpret_cast<const float4 *>(p.rope + (size_t)pos * hh2 + i0);
#pragma unroll
                            for (int i = 0; i < 8; i++) cs[i] = tab[i];
                        }
                        tmem_ld_wait();
                        if (S > 1) {
                            add_peers(v0, hc * hd + i0);
                            add_peers(v1, hc * hd + hh2 + i0);
                        }
                        float x0[16], x1[16];
#pragma unroll
                        for (int i = 0; i < 16; i++) {
                            const float u = rs * __uint_as_float(v0[i]), w = rs * __uint_as_float(v1[i]);
                            if (mat != 2) {
                                const float cc = i & 1 ? cs[i >> 1].z : cs[i >> 1].x, sn = i & 1 ? cs[i >> 1].w : cs[i >> 1].y;
                                x0[i] = u * cc - w * sn;
                                x1[i] = w * cc + u * sn;
                            } else {
                                x0[i] = u;
                                x1[i] = w;
                            }
                        }
                        if (head >= nh) continue;
                        if (mat == 0) {
                            if constexpr (RIDE)
                                if (rides) {  // Q~_j = Q_j + a * Q_1
                                    couple(x0, head * hd + i0, p.n_q * hd);
                                    couple(x1, head * hd + hh2 + i0, p.n_q * hd);
                                    if (on) {
                                        float *q0 = p.ride_q + ((size_t)path * p.ride.B + rb) * p.n_q * hd + (size_t)head * hd + i0;
#pragma unroll
                                        for (int i = 0; i < 4; i++) {
                                            *reinterpret_cast<float4 *>(q0 + 4 * i) = make_float4(x0[4 * i], x0[4 * i + 1], x0[4 * i + 2], x0[4 * i + 3]);
                                            *reinterpret_cast<float4 *>(q0 + hh2 + 4 * i) = make_float4(x1[4 * i], x1[4 * i + 1], x1[4 * i + 2], x1[4 * i + 3]);
                                        }
                                    }
                                    continue;
                                }
                            if (on && p.Qb) {
                                __nv_bfloat16 *q0 = p.Qb + (size_t)row * p.n_q * hd + (size_t)head * hd + i0;
#pragma unroll
                                for (int i = 0; i < 16; i++) x0[i] *= p.q_scale, x1[i] *= p.q_scale;
                                store16(q0, x0);
                                store16(q0 + hh2, x1);
                            } else if (on) {
                                float *q0 = p.Q + (size_t)row * p.n_q * hd + (size_t)head * hd + i0;
#pragma unroll
                                for (int i = 0; i < 4; i++) {
                                    *reinterpret_cast<float4 *>(q0 + 4 * i) = make_float4(x0[4 * i], x0[4 * i + 1], x0[4 * i + 2], x0[4 * i + 3]);
                                    *reinterpret_cast<float4 *>(q0 + hh2 + 4 * i) =
                                        make_float4(x1[4 * i], x1[4 * i + 1], x1[4 * i + 2], x1[4 * i + 3]);
                                }
                            }
                        } else if (kv) {
                            __nv_bfloat16 *dst = kv + (size_t)head * 16 * hd + i0;
                            store16(dst, x0);
                            store16(dst + hh2, x1);
                        }
                    }
                }
            }
            DBT_TL_SHARED_MARK(warp == 2 && lane == 0, 3);
            // the accumulator may be overwritten: tell the pair's MMA issuer
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_u32(acc_empty(a), lead));
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 610 + warp);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();  // neither CTA leaves while the other may still signal its barriers
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Cfg::kTmemCols) : "memory");
    DBT_TL_SHARED_TAKE;
    DBT_TL_END("gemm_pg");
}

}  // namespace dbt
