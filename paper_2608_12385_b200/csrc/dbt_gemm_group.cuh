// Per-expert GEMMs of an MoE prompt chunk on pairs of SMs (tcgen05 cta_group::2).
//
// A chunk's rows, sorted by expert, are many short lists (a few dozen to a few hundred rows each), so here the weights
// take the M side -- a pair's tile is 256 weight rows -- and an expert's rows the N side, whose width follows the list:
// the list is cut into the fewest tiles of at most 256 rows, equally, rounded up to 32 (the step of N in an MMA of M = 256).  Little work is done for
// padding at any list length (with the rows on the M side every list would pay for a multiple of 256), and every
// expert's matrices are read once per row tile.  Otherwise as gemm_prompt_kernel: each CTA of the pair brings half of
// the weight tile and half of the rows (both planes), persistent CTAs walk the (expert, feature tile, row tile) units
// of the experts that have rows, two accumulators overlap one unit's epilogue with the next unit's MMAs.
//
// What bounds it: the tensor pipe from about 170 rows per expert on, the expert matrices' HBM stream below.  How many
// boxes a k-tile is cut into matters as much: with both planes' rows in 2 KB boxes of 16 rows (12 instructions per CTA and
// k-tile) gate|up of 9472 rows took 508 us with the tensor pipe 49 % busy, and each further box, even a prefetch, cost it
// about 37 cycles; one box of exactly the tile's rows of both planes (a tensor map per width, GgRowMaps): 384 us, 73 %; down
// 231 -> 192 us.  The ring holds as many stages as the widest tile allows: 1000 rows 2.19 -> 2.15 ms per 4 layers.
//
// Measured on the MoE model (64 experts x 1408, 2 per row), per layer and 2048 rows of a long prompt: gate|up with SwiGLU
// 269 + 31 -> 83 us (9472-row chunks), down 158 -> 41 us, against 64-row tiles on one SM in 2048-row chunks, which
// streamed every expert's matrices for 64 rows at a time.
//
//   GG_GATEUP: a CTA's 128 weight rows are 64 gate rows and the 64 up rows of the same features, so the gate and the up
//              value of an element sit 64 TMEM lanes apart; the two warps concerned swap halves of every 16 columns
//              through shared memory and each applies the SwiGLU to eight rows of 32 features.
//   GG_DOWN:   fp32 rows.
#pragma once

#include "dbt_gemm_prompt.cuh"

namespace dbt {

enum GgMode { GG_GATEUP = 0, GG_DOWN = 1 };

constexpr int kGgRingBytes = 4 * 3 * 16384;  // at the widest 4 stages of 128 weight rows and 128 rows of each plane
constexpr int kGgMaxStages = 8;  // a launch has as many stages, up to this, as its widest row tile leaves room for
constexpr int kGgMaxExperts = 1024;
constexpr int kGgScratchBytes = kPgEpiWarps * (2048 + 512);
constexpr int kGgSmemBytes = kGgRingBytes + kGgScratchBytes + (kGgMaxExperts + 2) * 4 + 1024 + 256;
static_assert(kGgSmemBytes <= 227 * 1024, "shared memory of one SM");

struct GgParams {
    int K, E, n_feat;           // contracted width; experts; features of one expert (GG_GATEUP: of each matrix)
    const int *cnt, *off;       // rows per expert, first sorted row
    const float *rs;            // GG_GATEUP: 1/rms per sorted row (nullptr: 1)
    __nv_bfloat16 *H;           // GG_GATEUP: [sorted row][n_feat], two planes
    size_t h_lo;
    float *Y;                   // GG_DOWN: [sorted row][n_feat]
    int *status;
};

__device__ __forceinline__ void tma2_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}

// The sorted rows as [plane][row][K]: map j brings a k-tile of 16 (j + 1) rows of both planes in one box.
struct GgRowMaps {
    CUtensorMap m[8];
};

// A unit of work: rows [row0, row0 + rows) of the sorted list against features f0.. of expert e; n: MMA width.
struct GgUnit {
    int e, f0, row0, rows, n;
};

template <int MODE>
__global__ void __launch_bounds__(kPgThreads, 1) __cluster_dims__(2, 1, 1)
gemm_group_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
                  const __grid_constant__ GgRowMaps tmX, const GgParams p) {
    constexpr int STAGES = kGgMaxStages;
    constexpr int kTileF = MODE == GG_GATEUP ? 128 : 256;  // features of a pair's tile
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (ring - raw);
    constexpr int kBarOff = kGgRingBytes + kGgScratchBytes;
    const uint32_t bars = ring + kBarOff;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    auto acc_full = [&](int a) { return bars + 8u * (2 * STAGES + a); };
    auto acc_empty = [&](int a) { return bars + 8u * (2 * STAGES + 2 + a); };
    auto swap_bar = [&](int i) { return bars + 8u * (2 * STAGES + 4 + i); };
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(gen + kBarOff + 8 * (2 * STAGES + 8));
    int *first = reinterpret_cast<int *>(gen + kBarOff + 256);  // first unit of each expert, [E] = all units, [E + 1] = the widest row tile

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int nkt = (p.K + kTcK - 1) / kTcK, nft = (p.n_feat + kTileF - 1) / kTileF;

    if (tid == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; a++) {
            mbar_init(acc_full(a), 1);
            mbar_init(acc_empty(a), 2 * kPgEpiWarps);
        }
        for (int i = 0; i < 4; i++) mbar_init(swap_bar(i), 2);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    pdl_wait();  // the row lists
    if (warp == 2) {
        int base = 0, widest = 32;
        for (int e0 = 0; e0 < p.E; e0 += 32) {
            const int e = e0 + lane, cnt = e < p.E ? ld_mut(p.cnt + e) : 0, rt = (cnt + 255) / 256, u = rt * nft;
            if (rt) widest = max(widest, ((cnt + rt - 1) / rt + 31) & ~31);
            int incl = u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (e < p.E) first[e] = base + incl - u;
            base += __shfl_sync(0xffffffffu, incl, 31);
        }
        widest = __reduce_max_sync(0xffffffffu, widest);
        if (lane == 0) first[p.E] = base, first[p.E + 1] = widest;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers exist before either signals the other's
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_holder;
    pdl_launch_dependents();

    const int units = first[p.E];
    const int slot = 16384 + first[p.E + 1] * 128, stages = min(STAGES, kGgRingBytes / slot);
    // Units in order of expert, feature tile, row tile: the row tiles that share a weight tile run side by side.
    auto unit_of = [&](int t) {
        int lo = 0, hi = p.E - 1;  // the last expert whose first unit is not past t
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        const int cnt = ld_mut(p.cnt + lo), rt = (cnt + 255) / 256, k = t - first[lo];
        const int per = ((cnt + rt - 1) / rt + 31) & ~31, r0 = (k % rt) * per;  // <= 256; a list of rt tiles never ends before its last one
        GgUnit u;
        u.e = lo;
        u.f0 = (k / rt) * kTileF;
        u.row0 = ld_mut(p.off + lo) + r0;
        u.rows = min(per, cnt - r0);
        u.n = per;
        return u;
    };

    bool ok = true;
    if (warp == 0) {
        // ---- TMA: lane 0 the rows (both planes), lanes 1, 2 the weight tile
        if (lane == 0) {
            tma_prefetch_desc(&tmW0);
        }
        int s = 0, ph = 1;
        for (int t = pair; t < units && ok; t += npairs) {
            const GgUnit u = unit_of(t);
            const CUtensorMap *mx = &tmX.m[u.n / 32 - 1];
            for (int kt = 0; kt < nkt; kt++) {
                if (lane == 0) {
                    ok = mbar_wait_cluster(empty_bar(s), ph);  // a fresh barrier's phase before the first is over
                    if (ok && rank == 0) mbar_expect_tx(full_bar(s), 2 * (16384 + u.n * 128));
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                const uint32_t st = ring + s * slot, bar = mapa_u32(full_bar(s), 0);
                if (lane == 0) tma2_load_3d(st + 16384, mx, bar, kt * kTcK, u.row0 + (int)rank * (u.n / 2), 0);
                if (MODE == GG_GATEUP) {
                    if (lane == 1) tma2_load_2d(st, &tmW0, bar, kt * kTcK, u.e * p.n_feat + u.f0 + (int)rank * 64);
                    if (lane == 2) tma2_load_2d(st + 8192, &tmW1, bar, kt * kTcK, u.e * p.n_feat + u.f0 + (int)rank * 64);
                } else {
                    if (lane == 1) tma2_load_2d(st, &tmW0, bar, kt * kTcK, u.e * p.n_feat + u.f0 + (int)rank * 128);
                }
                if (++s == stages) s = 0, ph ^= 1;
            }
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 700);
        // The pair's last loads have landed before either CTA leaves, see gemm_prompt_kernel.  (ph: parity of a stage's last fill; of a
        // stage that had none, that of the phase before a fresh barrier's first.)
        if (lane == 0 && rank == 0) {
            for (int j = 0; j < stages; j++) {
                mbar_wait_cluster(full_bar(s), ph, kWaitCycles / STAGES);
                if (++s == stages) s = 0, ph ^= 1;
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // ---- MMA issuer of the pair
            int s = 0, ph = 0, n_acc = 0;
            for (int t = pair; t < units && ok; t += npairs, n_acc++) {
                const GgUnit u = unit_of(t);
                const uint32_t idesc = umma2_idesc(u.n);
                const int a = n_acc & 1;
                if (n_acc >= 2) ok = mbar_wait_cluster(acc_empty(a), ((n_acc >> 1) - 1) & 1);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem_base + a * 256;
                for (int kt = 0; kt < nkt; kt++) {
                    ok = mbar_wait_cluster(full_bar(s), ph);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t st = ring + s * slot;
                    const uint64_t adesc = umma_smem_desc(st);
#pragma unroll
                    for (int part = 0; part < 2; part++) {
                        const uint64_t bdesc = umma_smem_desc(st + 16384 + part * u.n * 64);
#pragma unroll
                        for (int k = 0; k < kTcK / 16; k++) umma2_f16(acc, adesc + 2 * k, bdesc + 2 * k, idesc, (kt | part | k) != 0);
                    }
                    umma2_commit(empty_bar(s));
                    if (++s == stages) s = 0, ph ^= 1;
                }
                if (ok) umma2_commit(acc_full(a));
            }
            if (!ok) report(p.status, kStatusWaitExpired, 701);
        }
    } else {
        // ---- epilogue: TMEM lane = weight row, TMEM column = activation row; two warps per lane quadrant share the columns
        const int quad = warp & 3, half = (warp - 2) >> 2;
        float *xch = reinterpret_cast<float *>(gen + kGgRingBytes);          // [warp][2][8][32]
        float *rs_s = xch + kPgEpiWarps * 512 + (warp - 2) * 128;                       // this warp's rows' factors
        const int me = warp - 2, mate = half * 4 + (((quad ^ 2) + 2) & 3);              // the warp 64 lanes away, same columns
        int n_acc = 0, c_run = 0;
        for (int t = pair; t < units; t += npairs, n_acc++) {
            const GgUnit u = unit_of(t);
            const int a = n_acc & 1, cb = half * (u.n / 2), ncol = min(u.n / 2, u.rows - cb);  // this warp's columns: cb .. cb + ncol
            if (MODE == GG_GATEUP) {
                __syncwarp();
                for (int c = lane; c < u.n / 2; c += 32) rs_s[c] = p.rs && c < ncol ? ld_mut(p.rs + u.row0 + cb + c) : 1.f;
                __syncwarp();
            }
            ok = mbar_wait_cluster(acc_full(a), (n_acc >> 1) & 1);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t tacc = tmem_base + ((uint32_t)(quad * 32) << 16) + a * 256 + cb;
            if (MODE == GG_GATEUP) {
                const bool up = quad >= 2;
                const int f = u.f0 + (int)rank * 64 + (quad & 1) * 32 + lane;
#pragma unroll 1
                for (int c = 0; c < ncol; c += 16, c_run++) {
                    uint32_t v[16];
                    __syncwarp();
                    tmem_ld16_issue(tacc + c, v);
                    tmem_ld_wait();
                    float *out = xch + me * 512 + (c_run & 1) * 256, *in = xch + mate * 512 + (c_run & 1) * 256;
#pragma unroll
                    for (int i = 0; i < 8; i++) out[i * 32 + lane] = __uint_as_float(up ? v[i] : v[8 + i]);
                    __syncwarp();
                    const uint32_t sb = swap_bar(half * 2 + (quad & 1));
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sb) : "memory");
                    ok = mbar_wait(sb, c_run & 1);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const int c8 = c + (up ? 8 : 0);
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        const float rs = rs_s[c8 + i], other = rs * in[i * 32 + lane], mine = rs * __uint_as_float(up ? v[8 + i] : v[i]);
                        const float h = up ? silu(other) * mine : silu(mine) * other;
                        if (c8 + i < ncol && f < p.n_feat) store_split(p.H, (size_t)(u.row0 + cb + c8 + i) * p.n_feat + f, p.h_lo, h);
                    }
                }
            } else {
                const int f = u.f0 + (int)rank * 128 + quad * 32 + lane;
                float *y = p.Y + (size_t)(u.row0 + cb) * p.n_feat + f;
#pragma unroll 1
                for (int c = 0; c < ncol; c += 16) {
                    uint32_t v[16];
                    __syncwarp();
                    tmem_ld16_issue(tacc + c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; i++)
                        if (c + i < ncol && f < p.n_feat) y[(size_t)(c + i) * p.n_feat] = __uint_as_float(v[i]);
                }
            }
            if (!ok) break;
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_u32(acc_empty(a), 0));
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 710 + warp);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();  // neither CTA leaves while the other may still signal its barriers
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

}  // namespace dbt
