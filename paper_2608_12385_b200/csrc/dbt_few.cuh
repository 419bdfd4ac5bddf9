// Linear layers of bf16 dense decode steps at few stacked rows (K*B <= 8): five kernels per layer, no split-K.
//
// At so few rows a layer is bound by the latency of its dependent kernels, not by HBM (1B model, one sequence: 43 us per layer of the
// chain of split-K GEMMs for 15 us of streaming).  What shortens it here:
//   - a CTA owns 16 features (or 8 gate and the same 8 up features) over the whole contracted width, its eight warps share that
//     width and meet in shared memory, so that residual, couplings and SwiGLU are done where the sum ends and no kernel sums
//     partials (tcgen05 needs 128 features per tile: 16 tiles for a 2048-wide output, hence split-K there);
//   - the products are mma.sync m16n8k16 with the weights as A.  The order of the contracted width inside a product is free as
//     long as both operands agree, so a lane takes sixteen consecutive elements of a weight row and of a row as two 16-byte loads
//     from the staged tile.  The tensor pipe has 50 times the rate that these few columns need;
//   - weights come by TMA, 16 rows x 512 elements per stage, the first ring of them before the dependency wait; 1/rms is formed
//     by a warp of its own beside the products.
// The rows are the two bf16 planes x = hi + lo of the other chains.  Up to four rows, hi and lo share the eight columns of one
// product; up to eight take two products.
//
// One step, us, the split-K chain / here: 1B, context 2048, 1 and 2 sequences 735 / 640, 744 / 621; 4 paths of one 870 / 681; 3 of
// 1000 731 / 643; 4 of 2048 764 / 692; one of 64 positions 657 / 550; 8B, one of 2048 3367 / 2995; four of 32768 5747 / 5710.
// Tried: weights from global memory straight into registers (1B, one sequence: 920; the few scoreboards of a warp serialise the
// ring), or by cp.async (768); one CTA per SM with a ring of five (707 against 652); the next stage's fragments read while a
// stage is multiplied (+25); the following matrices requested into L2 during the attention launch (690 against 652) or a
// launch's own later stages before its wait (662 against 638): the requests delay the chain's small loads; the rows in four
// copies, so that the CTAs' reads of them spread over L2 (equal).
#pragma once

#include "dbt_attn_mma.cuh"

namespace dbt {

enum FewMode {
    FEW_STORE = 0,   // Y = rs * acc
    FEW_RESID = 1,   // S += acc (branch rows: + coup * acc of the primary row), the next input g * S, shares of sum(S^2)
    FEW_GATEUP = 2,  // H = SiLU(rs * gate) * (rs * up) (branch rows: + coup * H_1), two planes
};

constexpr int kFewRows = 8;       // most stacked rows
constexpr int kFewWarps = 8;      // they share the contracted width of a tile
constexpr int kFewThreads = (kFewWarps + 2) * 32;  // and the producer, and the warp that forms 1/rms
// Dynamic shared memory of a CTA: two of them per SM, or (launches of at most one CTA per SM) one.  What is in flight sets the rate of
// a stream: with 48, 64 and 80 KB of weights per CTA the gate|up launch of the 1B model moved its 46 MB at 3.6, 4.6 and 5.5 TB/s.
constexpr int kFewSmem = 101 * 1024, kFewSmemOne = 200 * 1024, kFewCtas = 2;
constexpr int kFewRowBytes = 48 * 1024;
constexpr int kFewMaxRing = 8;
constexpr int kFewStage = 64 * kFewWarps;  // elements of the contracted width of a stage: 64 (128 bytes of a row) per warp
constexpr int kFewColStride = 20; // floats between two columns of a warp's sums: the fragments' stores hit 32 banks

struct FewParams {
    int n_out[3], rows[3], tile0[3], col0[3], nseg;
    int tiles, K, R, Bc;
    const float *ss_in;  // shares of sum(S^2): [ss_tiles][kFewRows]; nullptr: rs = 1
    int ss_tiles, d_norm;
    float eps;
    const float *coup;  // FEW_RESID, FEW_GATEUP: c or b, nullptr: none
    float *Y;           // FEW_STORE
    int ldy;
    float *S;  // FEW_RESID
    const float *g_next;
    __nv_bfloat16 *Xn;
    size_t xn_lo;
    float *ss_out;  // [tile][kFewRows]
    int d;
    __nv_bfloat16 *H;  // FEW_GATEUP
    size_t h_lo;
    int F;
    int evict_first;
    int *status;
    int ring, x_resident;  // see few_layout
};

__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
// Eight 64-element columns of some weight rows (see make_few_weight_map).
__device__ __forceinline__ void tma_load_w(uint32_t dst, const CUtensorMap *map, uint32_t bar, int row, int col, uint64_t pol, bool hint) {
    if (!hint) return tma_load_3d(dst, map, bar, 0, row, col);
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(0), "r"(row), "r"(col), "l"(pol)
        : "memory");
}

// NR: room for 2, 4 or 8 rows over all paths.
template <int NR>
struct FewCfg {
    static constexpr int kWBytes = 16 * kFewStage * 2;      // a stage of sixteen weight rows
    static constexpr int kXBytes = 2 * NR * kFewStage * 2;  // and of the rows
};
// Shared memory of a CTA: the rows as a whole where they take at most kFewRowBytes (each CTA then reads them once, however many tiles it
// walks), and as many stages as fit beside them.
struct FewLayout {
    int resident, ring, bytes;
};
inline FewLayout few_layout(int NR, int TM, int K, bool single, int smem) {
    const int stages = (K + kFewStage - 1) / kFewStage, w = TM * 16 * kFewStage * 2, x = 2 * NR * kFewStage * 2;
    FewLayout l;
    l.resident = !single && stages * x <= kFewRowBytes;
    const int fixed = l.resident ? stages * x : 0, per = l.resident ? w : w + x;
    l.ring = (smem - 1024 - fixed) / per;
    l.ring = l.ring > kFewMaxRing ? kFewMaxRing : l.ring;
    l.bytes = fixed + l.ring * per + 1024;
    return l;
}

// TM: sixteens of weight rows per tile.  At eight rows a stage of them is as large as a stage of sixteen weight rows; two sixteens
// share it where the contracted width is long and that leaves enough tiles for the SMs.  One / two sixteens from 4096 elements on,
// us per step of four sequences: 8B at 2048 positions 3330 / 3146, at 32768 5695 / 5525, d 4096 F 11008 881 / 863, d 5120 F 27648
// 1305 / 1168, d 6144 F 16384 1060 / 983, d 8192 F 28672 1408 / 1309.  From 1024 elements on they would give 1 to 4 % more (1B 704 / 699,
// d 3072 556 / 532, d 3584 700 / 675); before long tiles were dealt equally they cost 1.5 % there, and the line has not moved.
template <int MODE, int NR, int TM>
__global__ void __launch_bounds__(kFewThreads, 2)
few_linear_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2,
                  const __grid_constant__ CUtensorMap tmX, const FewParams p) {
    using Cfg = FewCfg<NR>;
    constexpr bool FOUR = NR <= 4;
    constexpr int PL = FOUR ? 1 : 2, QS = TM == 1 ? 2 : 1;
    extern __shared__ uint8_t smem_raw[];
    constexpr int NB = TM == 1 ? 2 : 1;  // buffers of the warps' sums (two sixteens: two CTAs would not fit an SM with two)
    __shared__ float sums[NB][kFewWarps][TM][kFewRows * kFewColStride];
    __shared__ float fin[2][TM][kFewRows][16];
    __shared__ float rs_s[kFewRows];
    __shared__ int bad_s;  // a wait ran out: nothing is stored from here on
    __shared__ __align__(8) uint64_t bar_s[2 * kFewMaxRing + 1];
    DBT_TL_DECL;
    const int RING = p.ring;
    const bool xres = p.x_resident != 0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int stages = (p.K + kFewStage - 1) / kFewStage;  // of a tile
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, bars = smem_u32(bar_s);
    const uint32_t ring = base + (xres ? stages * Cfg::kXBytes : 0);
    const int stage_bytes = TM * Cfg::kWBytes + (xres ? 0 : Cfg::kXBytes);
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (kFewMaxRing + s); };
    const uint32_t x_bar = bars + 8u * (2 * kFewMaxRing);
    auto seg_of = [&](int tile) { return p.nseg > 2 && tile >= p.tile0[2] ? 2 : p.nseg > 1 && tile >= p.tile0[1] ? 1 : 0; };
    if (tid == 0) {
        for (int s = 0; s < RING; s++) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), kFewWarps);
        }
        mbar_init(x_bar, 1);
        bad_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_launch_dependents();

    if (warp == kFewWarps) {
        // ---- producer: a stage is 512 elements of the contracted width of the tile's sixteen weight rows (and of the rows, where they
        // are not resident), as eight 128-byte columns (a consumer warp each), 128B-swizzled.  The first ring of weights goes out
        // before the dependency wait.
        if (lane == 0) {
            tma_prefetch_desc(&tmW0);
            tma_prefetch_desc(&tmX);
            const uint64_t pol = l2_evict_first_policy();
            bool ok = true;
            auto load_w = [&](int s, int tile, int st) {
                const uint32_t dst = ring + s * stage_bytes;
                mbar_expect_tx(full_bar(s), stage_bytes);
                const int sg = seg_of(tile), row = (tile - p.tile0[sg]) * TM;
#pragma unroll
                for (int m = 0; m < TM; m++) {  // (rows past the matrix's last arrive as zeros)
                    if (MODE == FEW_GATEUP) {
                        tma_load_w(dst + m * Cfg::kWBytes, &tmW0, full_bar(s), (row + m) * 8, st * 8, pol, p.evict_first);
                        tma_load_w(dst + m * Cfg::kWBytes + Cfg::kWBytes / 2, &tmW1, full_bar(s), (row + m) * 8, st * 8, pol, p.evict_first);
                    } else {
                        tma_load_w(dst + m * Cfg::kWBytes, sg == 0 ? &tmW0 : sg == 1 ? &tmW1 : &tmW2, full_bar(s), (row + m) * 16, st * 8, pol,
                                   p.evict_first);
                    }
                }
            };
            auto load_x = [&](int s, int st) { tma_load_4d(ring + s * stage_bytes + TM * Cfg::kWBytes, &tmX, full_bar(s), 0, 0, st * 8, 0); };
            const int mine = (p.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, total = mine * stages, npre = min(RING, total);
            int tile = blockIdx.x, st = 0, i = 0;
            for (; i < npre; i++) {
                load_w(i, tile, st);
                if (++st == stages) st = 0, tile += gridDim.x;
            }
            pdl_wait();
            if (xres) {
                mbar_expect_tx(x_bar, stages * Cfg::kXBytes);
                for (int j = 0; j < stages; j++) tma_load_4d(base + j * Cfg::kXBytes, &tmX, x_bar, 0, 0, j * 8, 0);
            } else {
                for (int j = 0; j < npre; j++) load_x(j, j % stages);
            }
            int s = npre == RING ? 0 : npre, par = 0;
            for (; i < total; i++) {
                ok = mbar_wait(empty_bar(s), par);
                if (!ok) break;
                load_w(s, tile, st);
                if (!xres) load_x(s, st);
                if (++st == stages) st = 0, tile += gridDim.x;
                if (++s == RING) s = 0, par ^= 1;
            }
            if (!ok) report(p.status, kStatusWaitExpired, 700);
            // the loads have landed before the CTA leaves, also where a wait of the consumers ran out
            for (int j = max(0, i - RING); j < i; j++) mbar_wait(full_bar(j % RING), (j / RING) & 1, kWaitCycles / RING);
            if (xres) mbar_wait(x_bar, 0, kWaitCycles / RING);
        }
        return;
    }
    if (warp == kFewWarps + 1) {
        // ---- 1/rms of every row, beside the products that it scales: lane = (part, row)
        if (MODE == FEW_RESID) return;
        pdl_wait();
        float q = 0.f;
        if (p.ss_in) {
#pragma unroll 16
            for (int i = lane >> 3; i < p.ss_tiles; i += 4) q += __ldcg(p.ss_in + (size_t)i * kFewRows + (lane & 7));
        }
        q += __shfl_xor_sync(0xffffffffu, q, 8);
        q += __shfl_xor_sync(0xffffffffu, q, 16);
        if (lane < kFewRows) rs_s[lane] = p.ss_in ? 1.f / sqrtf(q / (float)p.d_norm + p.eps) : 1.f;
        __syncwarp();
        asm volatile("bar.arrive 3, %0;" ::"n"(32 + 128 * TM) : "memory");
        return;
    }

    // the epilogue's thread: feature ef, row er of sixteen `sub` of a tile
    const int sub = warp >> 2, etid = tid & 127;  // (four warps per sixteen)
    const int ef = MODE == FEW_GATEUP ? etid & 7 : etid & 15, er = MODE == FEW_GATEUP ? etid >> 3 : etid >> 4;
    float cp = 0.f, gn = 1.f, s_old = 0.f;
    auto load_vecs = [&](int tile) {
        if (MODE == FEW_RESID && er < kFewRows) {
            const int f = (tile * TM + sub) * 16 + ef;
            if (f < p.d) {
                gn = p.g_next ? p.g_next[f] : 1.f;
                cp = p.coup ? p.coup[f] : 0.f;
            }
        }
        const int h = (tile * TM + sub) * 8 + ef;
        if (MODE == FEW_GATEUP && er < kFewRows && h < p.F) cp = p.coup ? p.coup[h] : 0.f;
    };
    load_vecs(blockIdx.x);
    pdl_wait();
    DBT_TL_WAITED;
    auto load_s = [&](int tile) {
        const int f = (tile * TM + sub) * 16 + ef;
        if (MODE == FEW_RESID && er < p.R && f < p.d) s_old = __ldcg(p.S + (size_t)er * p.d + f);
    };
    load_s(blockIdx.x);
    int buf = 0, slot = 0, par = 0;
    // the rows' fragment: column g is row g's hi plane (at most four rows: rows 0..NR-1, their lo planes from column 4 on)
    const int xr = FOUR ? g & 3 : g;
    const bool xslot = xr < NR;
    // 16-byte piece c of a 128-byte row at offset o (a multiple of 128) behind a 1024-byte boundary
    auto piece = [&](uint32_t at, uint32_t o, int c) { return lds128(at + ((o + c * 16) ^ ((o >> 3) & 0x70))); };
    bool ok = !xres || mbar_wait(x_bar, 0);
    for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x, buf ^= 1) {
        float acc[TM][2][4];
#pragma unroll
        for (int m = 0; m < TM; m++)
#pragma unroll
            for (int i = 0; i < 8; i++) acc[m][i >> 2][i & 3] = 0.f;
        const int next = tile + (int)gridDim.x;
#pragma unroll 1
        for (int st = 0; st < stages; st += QS) {
            // two stages at a time (two sixteens: one): their fragments are read together, their products follow
            uint4 a[QS][TM][2][2], x[QS][2][PL];
            const int nst = min(QS, stages - st);
#pragma unroll
            for (int q = 0; q < QS; q++) {
                if (q >= nst) break;
                ok = ok && mbar_wait(full_bar(slot), par);
                if (tile == (int)blockIdx.x && st == 0 && q == 0) DBT_TL_MARK(0);
                // Lane t takes the row's sixteen elements 16 t .. 16 t + 15 of this warp's 64 as two 16-byte pieces: with the swizzle
                // no two lanes of a quarter warp meet in a bank.
                const uint32_t at = ring + slot * stage_bytes, xat = xres ? base + (st + q) * Cfg::kXBytes : at + TM * Cfg::kWBytes;
#pragma unroll
                for (int blk = 0; blk < 2; blk++) {
#pragma unroll
                    for (int mh = 0; mh < 2 * TM; mh++) {  // (gate|up: the gate rows' columns, then the up rows')
                        const int m = mh >> 1, h = mh & 1;
                        a[q][m][blk][h] = piece(at + m * Cfg::kWBytes, MODE == FEW_GATEUP ? h * (Cfg::kWBytes / 2) + warp * 1024 + g * 128 : warp * 2048 + (g + 8 * h) * 128, 2 * t + blk);
                    }
#pragma unroll
                    for (int pl = 0; pl < PL; pl++)
                        x[q][blk][pl] = xslot ? piece(xat, (((FOUR ? g >> 2 : pl) * 8 + warp) * NR + xr) * 128, 2 * t + blk) : make_uint4(0, 0, 0, 0);
                }
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty_bar(slot)) : "memory");
                if (++slot == RING) slot = 0, par ^= 1;
            }
#pragma unroll
            for (int q = 0; q < QS; q++) {
                if (q >= nst) break;
#pragma unroll
                for (int mb = 0; mb < 2 * TM; mb++) {
                    const int m = mb >> 1, blk = mb & 1;
                    const uint4 v = a[q][m][blk][0], w = a[q][m][blk][1];
                    const uint32_t fa[4] = {v.x, w.x, v.y, w.y}, fb[4] = {v.z, w.z, v.w, w.w};
#pragma unroll
                    for (int pl = 0; pl < PL; pl++) {
                        mma_bf16(acc[m][blk], fa, x[q][blk][pl].x, x[q][blk][pl].y);
                        mma_bf16(acc[m][blk], fb, x[q][blk][pl].z, x[q][blk][pl].w);
                    }
                }
            }
        }
        if (!ok && lane == 0) {
            report(p.status, kStatusWaitExpired, 701);
            bad_s = 1;
        }
        if (tile == (int)blockIdx.x) DBT_TL_MARK(1);
#pragma unroll
        for (int m = 0; m < TM; m++)  // [column][feature]
#pragma unroll
            for (int i = 0; i < 4; i++) sums[buf % NB][warp][m][(2 * t + (i & 1)) * kFewColStride + g + (i >> 1) * 8] = acc[m][0][i] + acc[m][1][i];
        asm volatile("bar.sync 2, 256;" ::: "memory");
        if (warp >= 4 * TM) continue;
        if (MODE != FEW_RESID && tile == (int)blockIdx.x) asm volatile("bar.sync 3, %0;" ::"n"(32 + 128 * TM) : "memory");  // 1/rms is there
        if (bad_s) continue;
        {
            const int f = etid & 15, r = etid >> 4;
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < kFewWarps; w++) {
                if (FOUR) {
                    if (r < 4) v += sums[buf % NB][w][sub][r * kFewColStride + f] + sums[buf % NB][w][sub][(r + 4) * kFewColStride + f];
                } else {
                    v += sums[buf % NB][w][sub][r * kFewColStride + f];
                }
            }
            if (NB == 1) asm volatile("bar.sync 2, 256;" ::: "memory");  // all have read: the next tile's sums may be written
            if (MODE == FEW_STORE) {
                const int sg = seg_of(tile), o = ((tile - p.tile0[sg]) * TM + sub) * 16 + f;
                if (r < min(p.rows[sg], p.R) && o < p.n_out[sg]) p.Y[(size_t)r * p.ldy + p.col0[sg] + o] = rs_s[r] * v;
                continue;
            }
            fin[buf][sub][r][f] = v;
        }
        if (TM == 1 || sub == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
        else asm volatile("bar.sync 4, 128;" ::: "memory");
        if (MODE == FEW_RESID) {
            const int o = (tile * TM + sub) * 16 + ef;
            const bool on = er < p.R && o < p.d;
            float s = 0.f;
            if (on) {
                s = s_old + fin[buf][sub][er][ef];
                if (er >= p.Bc && p.coup) s += cp * fin[buf][sub][er % p.Bc][ef];
                p.S[(size_t)er * p.d + o] = s;
                store_split(p.Xn, (size_t)er * p.d + o, p.xn_lo, gn * s);
            }
            float q = s * s;
#pragma unroll
            for (int i = 8; i > 0; i >>= 1) q += __shfl_xor_sync(0xffffffffu, q, i);
            if (ef == 0) p.ss_out[(size_t)(tile * TM + sub) * kFewRows + er] = q;
            if (next < p.tiles) {
                load_vecs(next);
                load_s(next);
            }
        } else {
            const int o = (tile * TM + sub) * 8 + ef;
            if (er < p.R && o < p.F) {
                const float rs = rs_s[er];
                float h = silu(rs * fin[buf][sub][er][ef]) * (rs * fin[buf][sub][er][8 + ef]);
                if (er >= p.Bc && p.coup) {
                    const int b = er % p.Bc;
                    h += cp * (silu(rs_s[b] * fin[buf][sub][b][ef]) * (rs_s[b] * fin[buf][sub][b][8 + ef]));
                }
                store_split(p.H, (size_t)er * p.F + o, p.h_lo, h);
            }
            if (next < p.tiles) load_vecs(next);
        }
    }
    DBT_TL_MARK(2);
    DBT_TL_END(MODE == FEW_STORE ? "few_stor" : MODE == FEW_RESID ? "few_resi" : "few_gate");
}

// A weight matrix [rows][K], K a multiple of 64, as (64 elements, row, 64-element column): a box is eight columns of box_rows rows.
inline bool make_few_weight_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t K, uint32_t box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || K % 64 != 0) return false;
    cuuint64_t dims[3] = {64, rows, K / 64};
    cuuint64_t strides[2] = {K * 2, 128};
    cuuint32_t box[3] = {64, box_rows, kFewWarps};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// Rows in two planes [2][plane_rows][K]: a box is eight columns of the first box_rows rows of both planes.
inline bool make_few_row_map(CUtensorMap *map, const void *base, uint64_t plane_rows, uint64_t K, uint32_t box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || K % 64 != 0) return false;
    cuuint64_t dims[4] = {64, plane_rows, K / 64, 2};
    cuuint64_t strides[3] = {K * 2, 128, plane_rows * K * 2};
    cuuint32_t box[4] = {64, box_rows, kFewWarps, 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace dbt
