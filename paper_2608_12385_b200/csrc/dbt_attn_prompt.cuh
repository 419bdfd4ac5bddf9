// Causal attention of a prompt chunk on the 5th-generation tensor cores, over the bf16 paged cache (Section 4.4
// item 1: the primary path alone walks the prompt and writes the cache; sm_100a).
//
// A CTA owns two query tiles of 128 rows -- 128 / G consecutive positions x the G heads of a KV head -- and streams the
// keys they may see in tiles of 128 (eight 16-token pages: a TMA box per page and K|V plane, laid out as 128-byte-swizzled
// groups of eight rows a fixed distance apart).  Per key tile: S = Q K^T into tensor memory, one thread per
// row takes the softmax of its 128 scores (no shuffle), writes P back over S as bf16, and O += P V takes P from tensor
// memory.  The two query tiles alternate: while the threads of one work on its scores the tensor cores run the other's
// products.  O stays in tensor memory; it is rescaled only when a row's maximum has grown by more than 2^8 since the
// scale in use was fixed (P then stays below 2^8, and P and O carry the same relative error as with the exact maximum).
//
// What bounds it: 4 x 128 x 128 x d_h FLOPs per (query tile, key tile) take 1024 cycles of the tensor pipe at d_h 128,
// the 16384 exponentials as many cycles of the special-function unit.
// Copy instructions count too: a page's 16 rows arrive as one 4 KB box at d_h 128 (two 2 KB boxes, one per 64 columns:
// one 8192-token prompt of the 1B model, 2 layers, 2.96 -> 2.92 ms).
// Measured per layer and 2048 rows: 1B model at 16 sequences of up to 2048 keys 112 -> 41 us; 8B shape, one sequence at 0..8192
// keys 644 -> 190 us (720 useful TFLOP/s) against warps of mma.sync m16n8k16 that shared the staged pages.
//
// Roles: warps 0..3 and 4..7 softmax of tile 0 and 1, warp 8 TMA, warp 9 MMA and TMEM owner.  All waits are bounded.
#pragma once

#include "dbt_attn_mma.cuh"

namespace dbt {

struct PromptAttnParams {
    int B, cn;       // sequences; positions per sequence in this chunk (their K, V are in the cache already)
    int G, n_kv, num_pages, pt_stride;
    long long k_row0, v_row0;  // first row of this layer's K and V planes in the pool's row numbering
    const int32_t *page_table, *seq_len;  // seq_len: positions before this chunk
    const __nv_bfloat16 *Q;  // attn_prompt_short_kernel: the queries that tmQ views
    __nv_bfloat16 *Ob;  // [B * cn][q_dim] attention output, hi plane (+ lo plane at lo_off)
    size_t lo_off;
    int *status;
    int let_in_late;  // the next launch starts behind this one's wait: it reads what the kernel before wrote without a wait of its own
    int nqb;  // query blocks per sequence: ceil(cn / (256 / G)); attn_prompt_short_kernel: ceil(cn / (128 / G))
};

constexpr int kPaThreads = 320;
constexpr int kPaKeys = 128;            // keys per tile
constexpr float kPaRescaleLog2 = 8.f;   // growth of a row's maximum (log2) that triggers a rescale of O

template <int DH>
struct PromptAttCfg {
    static constexpr int kHalves = DH / 64;
    static constexpr int kTileBytes = 128 * DH * 2;  // a query tile, or K or V of a key tile
    static constexpr int kStages = DH == 128 ? 2 : 4;
    static constexpr int kSmemBytes = 2 * kTileBytes + 2 * kStages * kTileBytes + 1024 + 256;
    static constexpr int kTmemCols = 512;
    static_assert(kSmemBytes <= 227 * 1024, "shared memory of one SM");
};

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
        "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
          "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
          "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t *r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
        "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]),
        "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]),
        "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 128B-swizzled operand of 8-row groups `group` bytes apart.  K-major (the keys): lbo unused.  MN-major (the values): 64
// elements of the non-contracted dimension per 128-byte row, the next 64 lbo bytes further, groups along the contraction.
__device__ __forceinline__ uint64_t umma_smem_desc_groups(uint32_t saddr, uint32_t group, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;
    d |= (uint64_t)(group >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// A from tensor memory (bf16, two per column), B from shared memory.
__device__ __forceinline__ void umma_f16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}

template <int DH>
__global__ void __launch_bounds__(kPaThreads, 1) attn_prompt_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                                    const __grid_constant__ CUtensorMap tmKV, const PromptAttnParams p) {
    using Cfg = PromptAttCfg<DH>;
    constexpr int STAGES = Cfg::kStages, HALVES = Cfg::kHalves, KS = DH / 16;
    constexpr uint32_t kHalfBytes = 128 * 128;       // queries: 128 rows of one 64-column piece
    constexpr uint32_t kGroup = HALVES * 1024;       // keys, values: 8 rows, their 64-column pieces one after the other
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t q_s = (raw + 1023u) & ~1023u, k_s = q_s + 2 * Cfg::kTileBytes, v_s = k_s + STAGES * Cfg::kTileBytes;
    const uint32_t bars = v_s + STAGES * Cfg::kTileBytes;
    auto k_full = [&](int s) { return bars + 8u * s; };
    auto k_empty = [&](int s) { return bars + 8u * (STAGES + s); };
    auto v_full = [&](int s) { return bars + 8u * (2 * STAGES + s); };
    auto v_empty = [&](int s) { return bars + 8u * (3 * STAGES + s); };
    const uint32_t q_full = bars + 8u * (4 * STAGES);
    auto s_full = [&](int i) { return bars + 8u * (4 * STAGES + 1 + i); };
    auto p_full = [&](int i) { return bars + 8u * (4 * STAGES + 3 + i); };
    auto o_full = [&](int i) { return bars + 8u * (4 * STAGES + 5 + i); };
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem_raw + (bars - raw) + 8 * (4 * STAGES + 7));
    static_assert(8 * (4 * STAGES + 7) + 4 <= 256, "barrier area");

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int PT = 128 / p.G, PB = 2 * PT;  // positions per tile, per block
    // block -> (query block, sequence, KV head): the last query blocks (most keys) are scheduled first
    const int per_j = p.B * p.n_kv;
    const int jb = p.nqb - 1 - (int)blockIdx.x / per_j, rest = (int)blockIdx.x % per_j;
    const int b = rest / p.n_kv, g = rest % p.n_kv;

    if (tid == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(k_full(s), 1);
            mbar_init(k_empty(s), 1);
            mbar_init(v_full(s), 1);
            mbar_init(v_empty(s), 1);
        }
        mbar_init(q_full, 1);
        for (int i = 0; i < 2; i++) {
            mbar_init(s_full(i), 1);
            mbar_init(p_full(i), 4);
            mbar_init(o_full(i), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                     "r"((uint32_t)Cfg::kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_holder;
    auto t_s = [&](int i) { return tmem + 128u * i; };
    auto t_o = [&](int i) { return tmem + 256u + (uint32_t)DH * i; };
    if (!p.let_in_late) pdl_launch_dependents();
    pdl_wait();  // the chunk's Q rows and its K, V rows in the cache come from the kernel before
    if (p.let_in_late) pdl_launch_dependents();

    const int len0 = ld_mut(p.seq_len + b);
    const int c0 = jb * PB;
    // keys visible to each tile's last position, and the tiles of keys that makes (0: the tile has no position)
    const int n_pos0 = max(0, min(PT, p.cn - c0)), n_pos1 = max(0, min(PT, p.cn - c0 - PT));
    const int keys0 = len0 + c0 + n_pos0, keys1 = n_pos1 > 0 ? len0 + c0 + PT + n_pos1 : 0;
    const int n_keys = max(keys0, keys1);
    const int T0 = (keys0 + kPaKeys - 1) / kPaKeys, T1 = (keys1 + kPaKeys - 1) / kPaKeys, T = max(T0, T1);

    bool ok = true;
    if (warp == 8) {
        // ---- TMA: lane l brings page l of the tile
        if (lane == 0) {
            tma_prefetch_desc(&tmQ);
            tma_prefetch_desc(&tmKV);
            mbar_expect_tx(q_full, 2 * Cfg::kTileBytes);
            for (int i = 0; i < 2; i++)
                for (int h = 0; h < HALVES; h++)  // rows past the chunk's last position are another sequence's, or zeros: never stored
                    tma_load_4d(q_s + i * Cfg::kTileBytes + h * kHalfBytes, &tmQ, q_full, 0, g * p.G, b * p.cn + c0 + i * PT, h);
        }
        __syncwarp();
        const int pages_total = (n_keys + 15) >> 4, my_pg = lane;
        const bool loads = my_pg < 8;
        int page = loads && my_pg < pages_total ? p.page_table[(size_t)b * p.pt_stride + my_pg] : 0;
        int nk = 0, nv = 0;  // tiles of keys, of values requested
        for (int t = 0; t < T && ok; t++) {
            const int s = t % STAGES, np = min(8, pages_total - t * 8);
            if (loads && my_pg < np && (page < 0 || page >= p.num_pages)) {
                report(p.status, kStatusBadPage, page);
                page = 0;
            }
            const int row = (int)(((long long)page * p.n_kv + g) * 16);
            const uint32_t off = s * Cfg::kTileBytes + my_pg * 2 * kGroup;
            const int nx = (t + 1) * 8 + my_pg;
            const int next_page = loads && nx < pages_total ? p.page_table[(size_t)b * p.pt_stride + nx] : 0;
            if (lane == 0) {
                if (t >= STAGES) ok = mbar_wait(k_empty(s), ((t / STAGES) - 1) & 1);
                if (ok) mbar_expect_tx(k_full(s), (uint32_t)np * HALVES * 2048);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (ok && loads && my_pg < np) tma_load_4d(k_s + off, &tmKV, k_full(s), 0, 0, 0, (int)((p.k_row0 + row) >> 3));
            nk += ok;
            if (lane == 0 && ok) {
                if (t >= STAGES) ok = mbar_wait(v_empty(s), ((t / STAGES) - 1) & 1);
                if (ok) mbar_expect_tx(v_full(s), (uint32_t)np * HALVES * 2048);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (ok && loads && my_pg < np) tma_load_4d(v_s + off, &tmKV, v_full(s), 0, 0, 0, (int)((p.v_row0 + row) >> 3));
            nv += ok;
            page = next_page;
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 400);
        // the last loads have landed before the CTA leaves, also where a wait ran out
        if (lane == 0) {
            mbar_wait(q_full, 0);
            for (int j = max(0, nk - STAGES); j < nk; j++) mbar_wait(k_full(j % STAGES), (j / STAGES) & 1, kWaitCycles / STAGES);
            for (int j = max(0, nv - STAGES); j < nv; j++) mbar_wait(v_full(j % STAGES), (j / STAGES) & 1, kWaitCycles / STAGES);
        }
    } else if (warp == 9) {
        // ---- MMA issuer (lane 0; the whole warp clears V rows behind the last key)
        constexpr uint32_t idesc_qk = umma_idesc(kPaKeys);
        constexpr uint32_t idesc_pv = umma_idesc(DH) | (1u << 16);  // B is MN-major
        auto wait = [&](uint32_t bar, int parity) {
            bool r = true;
            if (lane == 0) r = mbar_wait(bar, parity);
            r = __shfl_sync(0xffffffffu, r, 0);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            return r;
        };
        auto qk = [&](int i, int t) {
            if (lane != 0) return;
            const int s = t % STAGES;
#pragma unroll
            for (int k = 0; k < KS; k++) {
                const int h = k >> 2;
                umma_f16(t_s(i), umma_smem_desc(q_s + i * Cfg::kTileBytes + h * kHalfBytes) + 2 * (k & 3),
                         umma_smem_desc_groups(k_s + s * Cfg::kTileBytes + h * 1024, kGroup, 0) + 2 * (k & 3), idesc_qk, k != 0);
            }
            umma_commit(s_full(i));
        };
        const int Tn[2] = {T0, T1};
        ok = wait(q_full, 0) && wait(k_full(0), 0);
        if (ok) {
            for (int i = 0; i < 2; i++)
                if (Tn[i] > 0) qk(i, 0);
            if (lane == 0) umma_commit(k_empty(0));
        }
        for (int t = 0; t < T && ok; t++) {
            const int s = t % STAGES, par = (t / STAGES) & 1;
            if (t + 1 < T) ok = wait(k_full((t + 1) % STAGES), ((t + 1) / STAGES) & 1);
            ok = ok && wait(v_full(s), par);
            if (!ok) break;
            if (t == T - 1 && n_keys < T * kPaKeys) {
                // rows behind the last key hold stale memory: P is zero there, but 0 * NaN is not
                const int v0 = n_keys - t * kPaKeys;
                for (int h = 0; h < HALVES; h++)
                    for (int idx = v0 * 8 + lane; idx < kPaKeys * 8; idx += 32)
                        asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(v_s + s * Cfg::kTileBytes + (idx >> 6) * kGroup + h * 1024 + (idx & 63) * 16), "r"(0u)
                                     : "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
            }
            for (int i = 0; i < 2 && ok; i++) {
                if (t >= Tn[i]) continue;
                ok = wait(p_full(i), t & 1);
                if (!ok) break;
                if (lane == 0) {
                    const uint64_t vd = umma_smem_desc_groups(v_s + s * Cfg::kTileBytes, kGroup, 1024);
#pragma unroll
                    for (int k = 0; k < kPaKeys / 16; k++) umma_f16_ts(t_o(i), t_s(i) + 8 * k, vd + (2 * kGroup >> 4) * k, idesc_pv, (t | k) != 0);
                    if (t + 1 == Tn[i]) umma_commit(o_full(i));
                }
                if (t + 1 < Tn[i]) qk(i, t + 1);
            }
            if (lane == 0 && ok) {
                umma_commit(v_empty(s));
                if (t + 1 < T) umma_commit(k_empty((t + 1) % STAGES));
            }
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 410);
    } else {
        // ---- softmax of one query tile: thread = row
        const int i = warp >> 2, r = tid & 127, my_T = i ? T1 : T0;
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t ts = t_s(i) + lanes, to = t_o(i) + lanes;
        const int pos = c0 + i * PT + r / p.G;  // chunk position of this row
        const bool on = pos < p.cn;
        const int lim = len0 + min(pos, p.cn - 1) + 1;                             // keys this row sees
        const int lim_w = len0 + min(c0 + i * PT + (r & ~31) / p.G, p.cn - 1) + 1;  // keys the warp's first row sees
        float m_use = 0.f, l_run = 0.f;
        for (int t = 0; t < my_T; t++) {
            ok = mbar_wait(s_full(i), t & 1);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t v[128];
#pragma unroll
            for (int c = 0; c < 4; c++) tmem_ld32_issue(ts + 32 * c, v + 32 * c);
            tmem_ld_wait();
            const int vis = lim - t * kPaKeys;
            if ((t + 1) * kPaKeys > lim_w) {
#pragma unroll
                for (int c = 0; c < 128; c++)
                    if (c >= vis) v[c] = 0xff800000u;
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 128; c++) mx[c & 3] = fmaxf(mx[c & 3], __uint_as_float(v[c]));
            const float m_tile = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            if (t == 0) {
                m_use = m_tile;
            } else if (__any_sync(0xffffffffu, m_tile > m_use + kPaRescaleLog2)) {
                // s_full was signalled after the products of the tile before: O is at rest
                const float m_new = fmaxf(m_use, m_tile), corr = ex2_approx(m_use - m_new);
                m_use = m_new;
                l_run *= corr;
#pragma unroll 1
                for (int c = 0; c < DH; c += 32) {
                    uint32_t o[32];
                    tmem_ld32_issue(to + c, o);
                    tmem_ld_wait();
#pragma unroll
                    for (int k = 0; k < 32; k++) o[k] = __float_as_uint(__uint_as_float(o[k]) * corr);
                    tmem_st32(to + c, o);
                }
            }
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int h = 0; h < 2; h++) {
                uint32_t pk[32];
#pragma unroll
                for (int c = 0; c < 32; c++) {
                    const float a = ex2_approx(__uint_as_float(v[h * 64 + 2 * c]) - m_use), e = ex2_approx(__uint_as_float(v[h * 64 + 2 * c + 1]) - m_use);
                    sum[(2 * c) & 3] += a;
                    sum[(2 * c + 1) & 3] += e;
                    pk[c] = pack_bf16(a, e);
                }
                tmem_st32(ts + 32 * h, pk);
            }
            l_run += (sum[0] + sum[1]) + (sum[2] + sum[3]);
            tmem_st_wait();
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(p_full(i)) : "memory");
        }
        if (ok && my_T > 0) {
            ok = mbar_wait(o_full(i), 0);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (!ok && lane == 0) report(p.status, kStatusWaitExpired, 420 + warp);
        if (ok && my_T > 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const float inv = 1.f / l_run;
            const size_t o0 = ((size_t)b * p.cn + pos) * (size_t)(p.n_kv * p.G * DH) + (size_t)(g * p.G + r % p.G) * DH;
#pragma unroll 1
            for (int c = 0; c < DH; c += 32) {
                uint32_t o[32];
                __syncwarp();
                tmem_ld32_issue(to + c, o);
                tmem_ld_wait();
                if (!on) continue;
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const float x0 = __uint_as_float(o[q * 8 + 2 * e]) * inv, x1 = __uint_as_float(o[q * 8 + 2 * e + 1]) * inv;
                        const __nv_bfloat162 h2 = __floats2bfloat162_rn(x0, x1);
                        hi[e] = *reinterpret_cast<const uint32_t *>(&h2);
                        lo[e] = pack_bf16(x0 - __low2float(h2), x1 - __high2float(h2));
                    }
                    *reinterpret_cast<uint4 *>(p.Ob + o0 + c + q * 8) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4 *>(p.Ob + o0 + c + q * 8 + p.lo_off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 9)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)Cfg::kTmemCols) : "memory");
}

// ---- first chunks of at most 128 rows ----------------------------------------------------------------------
// There attn_prompt_kernel is its fixed part (tensor memory, a softmax of 128 scores per thread that runs once, cold, two store
// waits): 2 to 4 us per layer longer than warps of mma.sync m16n8k16 that share the staged pages.  A CTA holds 128 query rows --
// eight warps, each with the 16 / G consecutive positions x G heads of one m16 tile in registers -- and every warp runs the whole
// online softmax of its rows over the pages (one TMA box of K and V per page, 64 tokens per stage) up to its causal limit.
// Correct at any number of keys: a replayed capture may meet longer caches than the host saw.
// What bounds it: latency (first read of the lengths, page ids, pages, then a chain of page steps); a ring of six stages instead
// of three measured the same.  Prefill of 69 positions, 1B / 8B: 1.211 / 5.63 ms with attn_prompt_kernel, 1.180 / 5.54 here.
// short_prompt says where it is taken.
constexpr int kPsWarps = 8;  // consumer warps = query tiles per CTA

template <int DH>
struct PromptShortCfg {
    static constexpr int kPageBytes = 16 * DH * 2;
    static constexpr int kStageBytes = 2 * 4 * kPageBytes;
    static constexpr int kStages = 3;
    static constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 256;
};

template <int DH>
__global__ void __launch_bounds__((kPsWarps + 1) * 32, 1) attn_prompt_short_kernel(const __grid_constant__ CUtensorMap tmKV,
                                                                                  const PromptAttnParams p) {
    using Cfg = PromptShortCfg<DH>;
    constexpr int STAGES = Cfg::kStages, HALVES = DH / 64, KS = DH / 16, NB = DH / 8;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;
    const uint32_t bars = tiles + STAGES * Cfg::kStageBytes;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int PW = 16 / p.G, PB = kPsWarps * PW;  // positions per warp, per block
    // block -> (query block, sequence, KV head): the last query blocks (most keys) are scheduled first
    const int per_j = p.B * p.n_kv;
    const int jb = p.nqb - 1 - (int)blockIdx.x / per_j, rest = (int)blockIdx.x % per_j;
    const int b = rest / p.n_kv, g = rest % p.n_kv;
    if (tid == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), kPsWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (!p.let_in_late) pdl_launch_dependents();
    pdl_wait();  // the chunk's Q rows and its K, V rows in the cache come from the kernel before
    if (p.let_in_late) pdl_launch_dependents();
    const int len0 = ld_mut(p.seq_len + b);
    const int c0 = jb * PB, c_last = min(c0 + PB, p.cn) - 1;  // chunk positions of this block
    const int nkeys_max = len0 + c_last + 1;                  // keys visible to the block's last position
    const int T = (nkeys_max + kAttTile - 1) / kAttTile, total_pages = (nkeys_max + 15) >> 4;

    if (warp == kPsWarps) {
        // ---- producer: one box per page (K and V of this KV head), page ids fetched 32 at a time
        if (lane == 0) tma_prefetch_desc(&tmKV);
        bool ok = true;
        int pt_base = -(1 << 30), my_page = 0, t = 0;
        for (; t < T; t++) {
            const int s = t % STAGES, p0 = t * 4, np = min(4, total_pages - p0);
            if (p0 + 4 > pt_base + 32) {
                pt_base = p0;
                my_page = p0 + lane < total_pages ? p.page_table[(size_t)b * p.pt_stride + p0 + lane] : 0;
            }
            if (lane == 0) {
                if (t >= STAGES) ok = mbar_wait(empty_bar(s), ((t / STAGES) - 1) & 1);
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
                const int row = (int)(((long long)page * p.n_kv + g) * 16);
                tma_load_4d(tiles + s * Cfg::kStageBytes + lane * 2 * Cfg::kPageBytes, &tmKV, full_bar(s), 0, 0, (int)(p.k_row0 + row), 0);
            }
        }
        if (lane == 0) {
            if (!ok) report(p.status, kStatusWaitExpired, 440);
            // the last loads have landed before the CTA leaves, also where a wait ran out
            for (int j = max(0, t - STAGES); j < t; j++) mbar_wait(full_bar(j % STAGES), (j / STAGES) & 1, kWaitCycles / STAGES);
        }
        return;
    }

    // ---- consumers: warp w holds chunk positions cw0 .. cw0 + npos_w - 1 (x G heads) as one m16 tile
    const int q_dim = p.n_kv * p.G * DH;
    const int cw0 = c0 + warp * PW, npos_w = max(0, min(PW, p.cn - cw0));
    const int pos_last_w = len0 + cw0 + npos_w - 1;  // the last key this warp's rows may see
    const int r0 = lane >> 2, c = (lane & 3) * 2;
    uint32_t qa[KS][4];
    int pl[2];  // chunk position (relative to cw0) of this lane's two rows, clamped to the valid ones
    {
        const __nv_bfloat16 *qrow[2];
        bool on[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int r = r0 + 8 * h, pr = r / p.G;
            on[h] = pr < npos_w;
            pl[h] = min(pr, max(npos_w - 1, 0));
            qrow[h] = p.Q + (on[h] ? (size_t)(b * p.cn + cw0 + pr) * q_dim + (size_t)(g * p.G + r % p.G) * DH : 0);
        }
#pragma unroll
        for (int ks = 0; ks < KS; ks++) {
            const int k = ks * 16 + c;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                qa[ks][h] = on[h] ? __ldcg(reinterpret_cast<const uint32_t *>(qrow[h] + k)) : 0u;
                qa[ks][2 + h] = on[h] ? __ldcg(reinterpret_cast<const uint32_t *>(qrow[h] + k + 8)) : 0u;
            }
        }
    }
    float o[NB][4];
#pragma unroll
    for (int nb = 0; nb < NB; nb++) o[nb][0] = o[nb][1] = o[nb][2] = o[nb][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
    const int lim[2] = {len0 + cw0 + pl[0] + 1, len0 + cw0 + pl[1] + 1};  // keys visible to each of this lane's two rows

    bool ok = true;
    for (int t = 0; t < T; t++) {
        const int s = t % STAGES;
        ok = mbar_wait(full_bar(s), (t / STAGES) & 1);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (npos_w > 0) {
            for (int pg = 0; pg < 4; pg++) {
                const int key0 = t * kAttTile + pg * 16;
                if (key0 > pos_last_w) break;  // this page and the later ones lie behind the warp's causal limit
                const uint32_t kpage = tiles + s * Cfg::kStageBytes + pg * 2 * Cfg::kPageBytes;
                const uint32_t vpage = kpage + Cfg::kPageBytes;
                const int valid = min(16, nkeys_max - key0);
                if (valid < 16) {
                    // slots past the block's last key hold stale pool contents: their scores are masked below and their V rows
                    // zeroed, so that 0 * garbage is no NaN (every warp that reads the page writes the same zeros before)
                    for (int idx = lane; idx < (16 - valid) * HALVES * 8; idx += 32)
                        asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(vpage + valid * HALVES * 128 + idx * 16), "r"(0u) : "memory");
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                }
                // S = Q K^T for the page's 16 tokens: two 8-token column blocks
                float sacc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
                {
                    const int r = (lane & 7) + ((lane >> 4) << 3);  // token row this lane addresses
                    const int cb = (lane >> 3) & 1;                 // which 8-dim chunk of the k-step
#pragma unroll
                    for (int ks = 0; ks < KS; ks++) {
                        const int chunk = ks * 2 + cb, sg = r * HALVES + (chunk >> 3);
                        uint32_t kb[4];
                        ldsm_x4(kpage + sg * 128 + (((chunk & 7) ^ (sg & 7)) << 4), kb);
                        mma_bf16(sacc[0], qa[ks], kb[0], kb[1]);
                        mma_bf16(sacc[1], qa[ks], kb[2], kb[3]);
                    }
                }
                // causal mask per row, online softmax (base 2), P packed as the A operand of P V
                if (key0 + 16 > min(lim[0], lim[1])) {  // only pages that cross a row's limit need the mask
#pragma unroll
                    for (int nb = 0; nb < 2; nb++)
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            if (key0 + nb * 8 + c + (e & 1) >= lim[e >> 1]) sacc[nb][e] = -INFINITY;
                }
                float rmax[2] = {-INFINITY, -INFINITY}, corr[2], msub[2];
#pragma unroll
                for (int nb = 0; nb < 2; nb++)
#pragma unroll
                    for (int e = 0; e < 4; e++) rmax[e >> 1] = fmaxf(rmax[e >> 1], sacc[nb][e]);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    rmax[h] = fmaxf(rmax[h], __shfl_xor_sync(0xffffffffu, rmax[h], 1));
                    rmax[h] = fmaxf(rmax[h], __shfl_xor_sync(0xffffffffu, rmax[h], 2));
                    const float mnew = fmaxf(m_run[h], rmax[h]);
                    msub[h] = mnew == -INFINITY ? 0.f : mnew;
                    corr[h] = m_run[h] == -INFINITY ? 0.f : exp2f(m_run[h] - msub[h]);
                    m_run[h] = mnew;
                }
                float rsum[2] = {0.f, 0.f};
                uint32_t pa[4];
#pragma unroll
                for (int nb = 0; nb < 2; nb++) {
                    const float p0 = exp2f(sacc[nb][0] - msub[0]), p1 = exp2f(sacc[nb][1] - msub[0]);
                    const float p2 = exp2f(sacc[nb][2] - msub[1]), p3 = exp2f(sacc[nb][3] - msub[1]);
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
                if (__any_sync(0xffffffffu, corr[0] != 1.f || corr[1] != 1.f)) {
#pragma unroll
                    for (int nb = 0; nb < NB; nb++) {
                        o[nb][0] *= corr[0];
                        o[nb][1] *= corr[0];
                        o[nb][2] *= corr[1];
                        o[nb][3] *= corr[1];
                    }
                }
                // O += P V: V read transposed, two 8-dim column blocks per ldmatrix
                {
                    const int r = (lane & 7) + (((lane >> 3) & 1) << 3);  // token row
                    const int cb = lane >> 4;                             // which of the two dim blocks
#pragma unroll
                    for (int np = 0; np < NB / 2; np++) {
                        const int chunk = np * 2 + cb, sg = r * HALVES + (chunk >> 3);
                        uint32_t vb[4];
                        ldsm_x4_trans(vpage + sg * 128 + (((chunk & 7) ^ (sg & 7)) << 4), vb);
                        mma_bf16(o[np * 2], pa, vb[0], vb[1]);
                        mma_bf16(o[np * 2 + 1], pa, vb[2], vb[3]);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty_bar(s)) : "memory");
    }
    if (!ok) {
        if (lane == 0) report(p.status, kStatusWaitExpired, 450 + warp);
        return;
    }
    // ---- normalise and write the rows of this warp's positions (two bf16 planes)
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int r = r0 + 8 * h, pr = r / p.G;
        if (pr >= npos_w) continue;
        const size_t ob = (size_t)(b * p.cn + cw0 + pr) * q_dim + (size_t)(g * p.G + r % p.G) * DH + c;
        const float inv = 1.f / l_run[h];
#pragma unroll
        for (int nb = 0; nb < NB; nb++) {
            const float x0 = o[nb][2 * h] * inv, x1 = o[nb][2 * h + 1] * inv;
            const __nv_bfloat162 hi = __floats2bfloat162_rn(x0, x1);
            *reinterpret_cast<__nv_bfloat162 *>(p.Ob + ob + nb * 8) = hi;
            *reinterpret_cast<__nv_bfloat162 *>(p.Ob + ob + nb * 8 + p.lo_off) = __floats2bfloat162_rn(x0 - __low2float(hi), x1 - __high2float(hi));
        }
    }
}

// The chunk's queries [rows][n_q][DH] (bf16, scaled by log2(e) / sqrt(DH)): a box is 128 / G rows x G heads x 64 columns.
inline bool make_prompt_q_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t n_q, uint64_t dh, uint32_t G) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {64, n_q, rows, dh / 64};
    cuuint64_t strides[3] = {dh * 2, n_q * dh * 2, 128};
    cuuint32_t box[4] = {64, G, 128 / G, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// The pool as groups of 8 rows of one head: a box is a page's 16 rows as two groups, in each the 64-column pieces of the
// eight rows one after the other.
inline bool make_prompt_kv_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t dh) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {64, 8, dh / 64, rows / 8};
    cuuint64_t strides[3] = {dh * 2, 128, 8 * dh * 2};
    cuuint32_t box[4] = {64, 8, (cuuint32_t)(dh / 64), 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace dbt
