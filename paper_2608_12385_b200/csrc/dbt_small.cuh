// Decode steps of dense models on the CUDA cores at few rows (fp32 models; at most 32 stacked rows).
//
// Such a step is a chain of launches that each move a few hundred KB: its time is the number of links times what one
// takes from its dependency to its last store.  So there are five kernels per layer instead of nine, and each reads its
// weights before its dependency wait and does one round of dependent loads after it:
//   linear_small (Q|K|V)  the RMSNorm is applied in the same pass: every warp sums its rows' squares beside the products
//                         (y = (sum_k w g x) / rms, the factor comes out of the sum);
//   attn_small            rotation, the a coupling and the cache append happen where the queries are staged; a (sequence,
//                         KV head) pair is split over blocks by its own length and merged by the last one to arrive;
//   linear_small          O + residual; gate|up with the norm, SwiGLU and b; down with c and residual -- a warp keeps a
//                         feature of all rows, so a branch row finds its primary twin in the same warp.
// Measured on the tiny fp32 model (4 layers, batch 2, context 64..80), copies of the outputs included: 192 -> 126 us per step;
// with the cluster kernel behind each attention launch (its phases take 1.5, 3.1, 2.2 and 2.0 us) 90.
#pragma once

#include "dbt_fused.cuh"
#include "dbt_gemm_prompt.cuh"
#include "dbt_kernels.cuh"

namespace dbt {

constexpr int kSmallRows = 32;   // stacked rows at most: a lane per row in the epilogues
constexpr int kSmallWarps = 4;
constexpr int kSmallPre = 3;     // 256-element pieces of a weight row held in registers before the dependency wait

struct SmallLin {
    const void *W[3];
    float *Y[3];
    int n_out[3], rows[3];
    int nseg;
    const float *X;      // [rows][K]
    const float *g;      // norm gain (nullptr: X is taken as it is)
    float eps;
    int K, epi, Bc;
    const float *coup;   // b (SwiGLU), c (EPI_DOWN); nullptr: none
    float *S;            // EPI_RESID, EPI_DOWN
};

// The rows are read through L1, and only those that are there: every warp of the launch reads all of them, and straight from L2
// (with the last row in place of missing ones) the same few lines were asked for by all SMs at once.  fp32 models of 4 layers, per
// step at 64 positions: d 2048, 2 rows 1110 -> 482 us, 10 rows 2410 -> 1131 (the generic chain 631 and 1252); d 256, 9 rows
// 303 -> 191 (283).
template <typename WT, int RT, bool SWIGLU>
__global__ void __launch_bounds__(kSmallWarps * 32) linear_small_kernel(const SmallLin a) {
    pdl_launch_dependents();
    __shared__ float sh[kSmallWarps][kSmallRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, K = a.K;
    int f = blockIdx.x * kSmallWarps + warp, seg = 0;
    if (!SWIGLU)
        while (seg < a.nseg && f >= a.n_out[seg]) f -= a.n_out[seg++];
    const bool act = seg < a.nseg && f < a.n_out[seg];
    if (!act) seg = 0, f = 0;
    const int rows = act ? a.rows[seg] : 0, n_out = a.n_out[seg];
    const WT *w0 = reinterpret_cast<const WT *>(a.W[seg]) + (size_t)f * K;
    const WT *w1 = SWIGLU ? reinterpret_cast<const WT *>(a.W[1]) + (size_t)f * K : w0;
    float wa[kSmallPre][8], wb[SWIGLU ? kSmallPre : 1][8], gn[kSmallPre][8];
#pragma unroll
    for (int c = 0; c < kSmallPre; c++) {
        const int k = c * 256 + lane * 8;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            wa[c][i] = 0.f, gn[c][i] = 1.f;
            if (SWIGLU) wb[c][i] = 0.f;
        }
        if (k < K) {
            load8(w0 + k, wa[c]);
            if (SWIGLU) load8(w1 + k, wb[c]);
            if (a.g) load_vec8(a.g + k, gn[c]);
        }
    }
    const float cp = a.coup ? a.coup[f] : 0.f;
    pdl_wait();
    const bool resid = a.epi == EPI_RESID || a.epi == EPI_DOWN;
    const float s_in = resid && lane < rows ? __ldcg(a.S + (size_t)lane * n_out + f) : 0.f;
    for (int r0 = 0; r0 < rows; r0 += RT) {
        float acc[RT], up[SWIGLU ? RT : 1], ss[RT];
#pragma unroll
        for (int r = 0; r < RT; r++) {
            acc[r] = ss[r] = 0.f;
            if (SWIGLU) up[r] = 0.f;
        }
        auto piece = [&](const float (&wv)[8], const float (&uv)[8], const float (&gv)[8], int k) {
            float x[RT][8];
#pragma unroll
            for (int r = 0; r < RT; r++) {
                if (r0 + r < rows) {
                    load8(a.X + (size_t)(r0 + r) * K + k, x[r]);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; i++) x[r][i] = 0.f;
                }
            }
#pragma unroll
            for (int r = 0; r < RT; r++)
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const float xg = x[r][i] * gv[i];
                    acc[r] = fmaf(wv[i], xg, acc[r]);
                    if (SWIGLU) up[r] = fmaf(uv[i], xg, up[r]);
                    ss[r] = fmaf(x[r][i], x[r][i], ss[r]);
                }
        };
#pragma unroll
        for (int c = 0; c < kSmallPre; c++)
            if (c * 256 + lane * 8 < K) piece(wa[c], wb[SWIGLU ? c : 0], gn[c], c * 256 + lane * 8);
        for (int k = kSmallPre * 256 + lane * 8; k < K; k += 256) {
            float wv[8], uv[8], gv[8];
#pragma unroll
            for (int i = 0; i < 8; i++) gv[i] = 1.f, uv[i] = 0.f;
            load8(w0 + k, wv);
            if (SWIGLU) load8(w1 + k, uv);
            if (a.g) load_vec8(a.g + k, gv);
            piece(wv, uv, gv, k);
        }
#pragma unroll
        for (int r = 0; r < RT; r++) {
            float y = warp_sum(acc[r]), inv = 1.f;
            if (a.g) inv = 1.f / sqrtf(warp_sum(ss[r]) / (float)K + a.eps);
            y *= inv;
            if (SWIGLU) y = silu(y) * (inv * warp_sum(up[r]));
            if (lane == r && r0 + r < rows) sh[warp][r0 + r] = y;
        }
    }
    __syncwarp();
    if (lane < rows) {
        float y = sh[warp][lane];
        const size_t o = (size_t)lane * n_out + f;
        if (lane >= a.Bc && a.coup) y = fmaf(cp, sh[warp][lane % a.Bc], y);  // a branch row and its primary twin
        if (resid)
            a.S[o] = s_in + y;
        else
            a.Y[seg][o] = y;
    }
}

// Decode attention at few rows: one block per (sequence, KV head, split), 256 threads.
struct SmallAttn {
    const float *Q, *Kn, *Vn;  // this step's projections, before rotation
    int B, P, G, n_kv;         // P: residual paths present
    const float *coup_a;
    const float2 *rope;
    const int32_t *seq_len, *page_table;
    int pt_stride, num_pages;
    float *kpool, *vpool;
    float *part;               // [pair][split][NQ][DH + 2]
    int32_t *tickets;          // [pair], zero between launches
    float *O;
    int *status;
};
constexpr int kSaThreads = 256, kSaChunk = 256;  // keys per pass of a block
constexpr int kSaSplitKeys = 128;                // a split takes at least so many keys

template <int NQ, int DH>
__global__ void __launch_bounds__(kSaThreads) attn_small_kernel(const SmallAttn a) {
    constexpr int LPK = DH / 4, KPW = 32 / LPK, KPB = KPW * (kSaThreads / 32);  // lanes per key, keys per warp and block at once
    constexpr int NSUB = kSaThreads / LPK;                                      // key subsets of the P V pass
    __shared__ __align__(16) float qs[NQ][DH];
    __shared__ __align__(16) float sc[NQ][kSaChunk];
    __shared__ __align__(16) float red[kSaThreads / 32][NQ][DH];
    __shared__ float m_s[NQ], l_s[NQ], corr_s[NQ];
    __shared__ int last_s;
    __shared__ int page_s[kSaChunk / 16 + 1];  // the pass's pages: one load instead of one in front of every key
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x, g = blockIdx.y, sp = blockIdx.z, nsplit = gridDim.z;
    const int nq = a.P * a.G, q_dim = a.n_kv * a.G * DH, kv_dim = a.n_kv * DH, half = DH / 2;
    pdl_launch_dependents();
    DBT_TL_DECL;
    pdl_wait();
    DBT_TL_WAITED;
    const int pos = ld_mut(a.seq_len + b), nkeys = pos + 1;
    const int n_act = min(nsplit, (nkeys + kSaSplitKeys - 1) / kSaSplitKeys);  // by the sequence's own length
    if (sp >= n_act) return;
    const int pages = (nkeys + 15) >> 4, pps = (pages + n_act - 1) / n_act;
    const int jbeg = min(nkeys, sp * pps * 16), jend = min(nkeys, jbeg + pps * 16);
    const bool owns_new = pos >= jbeg && pos < jend;
    const int32_t *pt = a.page_table + (size_t)b * a.pt_stride;
    auto fetch_pages = [&](int j0) {  // jbeg, and with it every pass, starts on a page border
        if (tid < kSaChunk / 16 && j0 + tid * 16 < jend) {
            int page = pt[(j0 >> 4) + tid];
            if (page < 0 || page >= a.num_pages) {
                report(a.status, kStatusBadPage, page);
                page = -1;
            }
            page_s[tid] = page;
        }
    };
    fetch_pages(jbeg);
    // pool row of key j0 + j of this head (a bad page id was reported: the step runs on with page 0)
    auto row_of = [&](int j) { return (((size_t)max(page_s[j >> 4], 0) * a.n_kv + g) * 16 + (j & 15)) * DH; };
    // the new key and value: rotated, appended by the split that holds the position
    if (owns_new && tid < half) {
        const float2 t = a.rope[(size_t)pos * half + tid];
        const float *kn = a.Kn + (size_t)b * kv_dim + g * DH, *vn = a.Vn + (size_t)b * kv_dim + g * DH;
        const float x0 = __ldcg(kn + tid), x1 = __ldcg(kn + tid + half), v0 = __ldcg(vn + tid), v1 = __ldcg(vn + tid + half);
        const int page = pt[pos >> 4];
        if (page >= 0 && page < a.num_pages) {
            const size_t r = (((size_t)page * a.n_kv + g) * 16 + (pos & 15)) * DH;
            a.kpool[r + tid] = x0 * t.x - x1 * t.y;
            a.kpool[r + tid + half] = x1 * t.x + x0 * t.y;
            a.vpool[r + tid] = v0;
            a.vpool[r + tid + half] = v1;
        }
    }
    // queries: RoPE, Q~_j = Q_j + a * Q_1 (Eq. asymattn), scaled
    const float scale = 1.f / sqrtf((float)DH);
    for (int idx = tid; idx < NQ * half; idx += kSaThreads) {
        const int q = idx / half, i = idx % half;
        float r0 = 0.f, r1 = 0.f;
        if (q < nq) {
            const int path = q / a.G, h = g * a.G + q % a.G, o0 = h * DH + i, o1 = o0 + half;
            const float2 t = a.rope[(size_t)pos * half + i];
            const float *q1 = a.Q + (size_t)b * q_dim, *qj = a.Q + (size_t)(path * a.B + b) * q_dim;
            const float x0 = __ldcg(q1 + o0), x1 = __ldcg(q1 + o1), y0 = __ldcg(qj + o0), y1 = __ldcg(qj + o1);
            r0 = y0 * t.x - y1 * t.y;
            r1 = y1 * t.x + y0 * t.y;
            if (path) {
                r0 = fmaf(a.coup_a[o0], x0 * t.x - x1 * t.y, r0);
                r1 = fmaf(a.coup_a[o1], x1 * t.x + x0 * t.y, r1);
            }
        }
        qs[q][i] = r0 * scale;
        qs[q][i + half] = r1 * scale;
    }
    if (tid < NQ) {
        m_s[tid] = -INFINITY;
        l_s[tid] = 0.f;
    }
    DBT_TL_MARK(0);
    __syncthreads();  // (the appended row too: written by this block)
    const int dl = (lane % LPK) * 4, ksub = warp * KPW + lane / LPK;  // this thread's four dims; its key within KPB
    float o[NQ][4];
#pragma unroll
    for (int q = 0; q < NQ; q++) o[q][0] = o[q][1] = o[q][2] = o[q][3] = 0.f;
    for (int j0 = jbeg; j0 < jend; j0 += kSaChunk) {
        const int cnt = min(kSaChunk, jend - j0);
        if (j0 > jbeg) {
            fetch_pages(j0);
            __syncthreads();
        }
        constexpr int U = 4;  // keys in flight per lane group
        float4 vv[U];
#pragma unroll
        for (int u = 0; u < U; u++) {  // the first values travel with the first keys
            const int j = ksub + u * KPB;
            vv[u] = j < cnt ? ldcg4(a.vpool + row_of(j) + dl) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int k0 = 0; k0 < cnt; k0 += U * KPB) {
            float4 kk[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int j = k0 + ksub + u * KPB;
                kk[u] = j < cnt ? ldcg4(a.kpool + row_of(j) + dl) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int j = k0 + ksub + u * KPB;
#pragma unroll
                for (int q = 0; q < NQ; q++) {
                    const float4 w = *reinterpret_cast<const float4 *>(&qs[q][dl]);
                    float s = kk[u].x * w.x + kk[u].y * w.y + kk[u].z * w.z + kk[u].w * w.w;
#pragma unroll
                    for (int x = LPK / 2; x > 0; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
                    if (lane % LPK == 0 && j < cnt) sc[q][j] = s;
                }
            }
        }
        __syncthreads();
        for (int q = warp; q < NQ; q += kSaThreads / 32) {
            float mx = -INFINITY;
            for (int i = lane; i < cnt; i += 32) mx = fmaxf(mx, sc[q][i]);
            const float mold = m_s[q], mnew = fmaxf(mold, warp_max(mx));
            float s = 0.f;
            for (int i = lane; i < cnt; i += 32) {
                const float e = expf(sc[q][i] - mnew);
                sc[q][i] = e;
                s += e;
            }
            s = warp_sum(s);
            __syncwarp();
            if (lane == 0) {
                const float c = mold == -INFINITY ? 0.f : expf(mold - mnew);
                corr_s[q] = c;
                l_s[q] = l_s[q] * c + s;
                m_s[q] = mnew;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NQ; q++) {
            const float c = corr_s[q];
            o[q][0] *= c, o[q][1] *= c, o[q][2] *= c, o[q][3] *= c;
        }
        for (int k0 = 0; k0 < cnt; k0 += U * KPB) {
            if (k0 > 0) {
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int j = k0 + ksub + u * KPB;
                    vv[u] = j < cnt ? ldcg4(a.vpool + row_of(j) + dl) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int j = k0 + ksub + u * KPB;
                if (j < cnt) {
#pragma unroll
                    for (int q = 0; q < NQ; q++) {
                        const float pj = sc[q][j];
                        o[q][0] = fmaf(pj, vv[u].x, o[q][0]), o[q][1] = fmaf(pj, vv[u].y, o[q][1]);
                        o[q][2] = fmaf(pj, vv[u].z, o[q][2]), o[q][3] = fmaf(pj, vv[u].w, o[q][3]);
                    }
                }
            }
        }
        __syncthreads();  // the scores are free again
    }
    DBT_TL_MARK(1);
    // fold the key subsets: within a warp, then the warps in order
#pragma unroll
    for (int q = 0; q < NQ; q++) {
#pragma unroll
        for (int x = LPK; x < 32; x <<= 1)
#pragma unroll
            for (int e = 0; e < 4; e++) o[q][e] += __shfl_xor_sync(0xffffffffu, o[q][e], x);
        if (lane < LPK) *reinterpret_cast<float4 *>(&red[warp][q][dl]) = make_float4(o[q][0], o[q][1], o[q][2], o[q][3]);
    }
    __syncthreads();
    static_assert(NSUB == KPB, "a key subset per lane group");
    const size_t pair = (size_t)b * a.n_kv + g;
    float *part = a.part + (pair * nsplit + sp) * NQ * (DH + 2);
    for (int idx = tid; idx < nq * DH; idx += kSaThreads) {
        const int q = idx / DH, e = idx % DH;
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kSaThreads / 32; w++) t += red[w][q][e];
        if (n_act == 1)
            a.O[(size_t)((q / a.G) * a.B + b) * q_dim + (size_t)(g * a.G + q % a.G) * DH + e] = t / l_s[q];
        else
            part[(size_t)q * (DH + 2) + e] = t;
    }
    DBT_TL_END("attsmall");
    if (n_act == 1) return;
    if (tid < nq) {
        part[(size_t)tid * (DH + 2) + DH] = m_s[tid];
        part[(size_t)tid * (DH + 2) + DH + 1] = l_s[tid];
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const int tk = atomicAdd(a.tickets + pair, 1);
        last_s = tk == n_act - 1;
        if (last_s) atomicExch(a.tickets + pair, 0);
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    // the last split to arrive merges all of them, in split order
    const float *base = a.part + pair * nsplit * NQ * (DH + 2);
    for (int idx = tid; idx < nq * DH; idx += kSaThreads) {
        const int q = idx / DH, e = idx % DH;
        float M = -INFINITY, L = 0.f, t = 0.f;
        for (int s = 0; s < n_act; s++) M = fmaxf(M, __ldcg(base + ((size_t)s * NQ + q) * (DH + 2) + DH));
        for (int s = 0; s < n_act; s++) {
            const float *ps = base + ((size_t)s * NQ + q) * (DH + 2);
            const float w = expf(__ldcg(ps + DH) - M);
            L = fmaf(__ldcg(ps + DH + 1), w, L);
            t = fmaf(__ldcg(ps + e), w, t);
        }
        a.O[(size_t)((q / a.G) * a.B + b) * q_dim + (size_t)(g * a.G + q % a.G) * DH + e] = t / L;
    }
}

// Everything between two attention launches in one: O projection + residual, gate|up with norm, SwiGLU and b, down with c
// and residual, and the next layer's Q|K|V -- four dependent linear layers, which as launches of their own are four links of
// about 4.5 us each.  One cluster of 16 CTAs: each holds a sixteenth of every matrix in shared memory (bulk copies issued
// before the dependency wait, so they pass while the attention kernel runs) and sends what it computes to all 16 through
// distributed shared memory; between the layers each waits for the other slices' bytes instead of a kernel boundary.
// Taken where a layer's matrices fit the cluster's shared memory beside the rows (small_cluster_smem).
struct SmallMlp {
    const float *O, *wo, *g_mlp, *wg, *wu, *coup_b, *wd, *coup_c;
    const float *g_next, *w_next[3];  // the next layer's norm gain and Q, K, V matrices (g_next == nullptr: last layer)
    float *S, *y_next[3];
    int n_next[3], rows_next[3];
    int R, Bc, d, qd, F;
    float eps;
    int *status;
};
constexpr int kScCtas = 16, kScThreads = 512, kScMaxRows = 8, kScMaxSmem = 227 * 1024 - 256;  // (static shared memory beside it)

// Floats of one CTA's slices and row buffers.
struct SmallClusterLayout {
    int dO, Fs, qs;                           // features per CTA: O and down, gate (and up), next Q|K|V
    int wo, wg, wu, wd, wn, x, s, h, g1, g2, cb, cc, total;  // offsets
};
__host__ __device__ inline SmallClusterLayout small_cluster_layout(int R, int d, int qd, int F, int n_next) {
    SmallClusterLayout l;
    l.dO = d / kScCtas;
    l.Fs = F / kScCtas;
    l.qs = n_next / kScCtas;
    l.wo = 0;
    l.wg = l.wo + l.dO * qd;
    l.wu = l.wg + l.Fs * d;
    l.wd = l.wu + l.Fs * d;
    l.wn = l.wd + l.dO * F;
    l.x = l.wn + l.qs * d;
    l.s = l.x + R * (qd > d ? qd : d);
    l.h = l.s + R * d;
    l.g1 = l.h + R * F;
    l.g2 = l.g1 + d;
    l.cb = l.g2 + d;
    l.cc = l.cb + l.Fs;
    l.total = l.cc + l.dO;
    return l;
}
// Dynamic shared memory of a CTA; 0: the shape does not go this way.
inline size_t small_cluster_smem(int R, int d, int qd, int F, int n_next) {
    if (R > kScMaxRows || d > 256 || d % (4 * kScCtas) || F % (4 * kScCtas) || n_next % kScCtas || qd % 8) return 0;
    const size_t bytes = (size_t)small_cluster_layout(R, d, qd, F, n_next).total * 4;
    return bytes <= (size_t)kScMaxSmem ? bytes : 0;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const float *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes),
                 "r"(bar)
                 : "memory");
}
// Sixteen bytes into another CTA's shared memory, counted by its barrier.
__device__ __forceinline__ void st_async4(uint32_t addr, float4 v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(addr), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}

// The sums over the warp of RM (4 or 8) values per lane: lane l returns that of value l / (32 / RM).  A value halves with
// every exchange, 6 or 9 shuffles instead of 5 RM.
template <int RM>
__device__ __forceinline__ float warp_sum_rows(const float (&v)[RM]) {
    const int lane = threadIdx.x & 31;
    float t[RM];
#pragma unroll
    for (int r = 0; r < RM; r++) t[r] = v[r];
    int n = RM, o = 16;
#pragma unroll
    for (int step = 0; step < (RM == 8 ? 3 : 2); step++) {
        const bool up = lane & o;
#pragma unroll
        for (int r = 0; r < RM / 2; r++)
            if (r < n / 2) {
                const float keep = up ? t[r + n / 2] : t[r], give = up ? t[r] : t[r + n / 2];
                t[r] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        n /= 2;
        o /= 2;
    }
    float s = t[0];
#pragma unroll
    for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// w . x[row] over K (a multiple of 4) for the row of this lane (warp_sum_rows), by one warp, both in shared memory.
template <int RM>
__device__ __forceinline__ float sc_dot(const float *w, const float *x, int K, int R) {
    const int lane = threadIdx.x & 31;
    float acc[RM];
#pragma unroll
    for (int r = 0; r < RM; r++) acc[r] = 0.f;
    for (int k = lane * 4; k < K; k += 128) {
        const float4 a = *reinterpret_cast<const float4 *>(w + k);
#pragma unroll
        for (int r = 0; r < RM; r++) {
            const float4 b = *reinterpret_cast<const float4 *>(x + (size_t)min(r, R - 1) * K + k);
            acc[r] = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, acc[r]))));
        }
    }
    return warp_sum_rows<RM>(acc);
}

// Normalised rows in registers, for several features of one warp: g * S of all rows (at most 256 columns), and 1/rms of this
// lane's row, which the products are multiplied by.
// kGlobal: the rows lie in memory that the kernel before has written.
template <int RM, bool kGlobal = false>
struct ScRows {
    float4 x[RM][2];
    float inv;
    // norm = false: the rows as they are (g is not read)
    __device__ __forceinline__ void load(const float *S, const float *g, int K, int R, float eps, bool norm = true) {
        float ss[RM];
#pragma unroll
        for (int r = 0; r < RM; r++) ss[r] = 0.f;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = (threadIdx.x & 31) * 4 + u * 128;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f), gv = !norm ? make_float4(1.f, 1.f, 1.f, 1.f) : k < K ? load_vec4(g + k) : z;
#pragma unroll
            for (int r = 0; r < RM; r++) {
                const float *p = S + (size_t)min(r, R - 1) * K + k;
                const float4 v = k < K ? (kGlobal ? ldcg4(p) : *reinterpret_cast<const float4 *>(p)) : z;
                ss[r] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, ss[r]))));
                x[r][u] = make_float4(v.x * gv.x, v.y * gv.y, v.z * gv.z, v.w * gv.w);
            }
        }
        inv = norm ? 1.f / sqrtf(warp_sum_rows<RM>(ss) / (float)K + eps) : 1.f;
    }
    static __device__ __forceinline__ void weights(const float *w, int K, float4 (&a)[2]) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = (threadIdx.x & 31) * 4 + u * 128;
            a[u] = k < K ? *reinterpret_cast<const float4 *>(w + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __device__ __forceinline__ float dot(const float *w, int K) const {
        float4 a[2];
        weights(w, K, a);
        return dot(a);
    }
    __device__ __forceinline__ float dot(const float4 (&wa)[2]) const {
        float acc[RM];
#pragma unroll
        for (int r = 0; r < RM; r++) acc[r] = 0.f;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const float4 a = wa[u];
#pragma unroll
            for (int r = 0; r < RM; r++)
                acc[r] = fmaf(a.x, x[r][u].x, fmaf(a.y, x[r][u].y, fmaf(a.z, x[r][u].z, fmaf(a.w, x[r][u].w, acc[r]))));
        }
        return inv * warp_sum_rows<RM>(acc);
    }
};

template <int RM>
__global__ void __launch_bounds__(kScThreads, 1) small_mlp_kernel(const SmallMlp a) {
    DBT_TL_DECL;
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(8) unsigned long long bar_mem[7];  // four groups of weights, three exchanges
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, R = a.R;
    constexpr int NW = kScThreads / 32;
    const uint32_t rank = cluster_rank();
    const int n_next = a.n_next[0] + a.n_next[1] + a.n_next[2];
    const SmallClusterLayout l = small_cluster_layout(R, a.d, a.qd, a.F, n_next);
    auto bar = [&](int i) { return smem_u32(&bar_mem[i]); };
    if (tid == 0) {
        for (int i = 0; i < 7; i++) mbar_init(bar(i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // what the other 15 CTAs will send in the three exchanges
        mbar_expect_tx(bar(4), (kScCtas - 1) * R * l.dO * 4);
        mbar_expect_tx(bar(5), (kScCtas - 1) * R * l.Fs * 4);
        if (a.g_next) mbar_expect_tx(bar(6), (kScCtas - 1) * R * l.dO * 4);
        // this CTA's slice of every matrix: whole rows, contiguous in memory
        auto slice = [&](int off, const float *W, int f0, int nf, int K, int b) {
            if (nf > 0) bulk_load(smem_u32(sm + off), W + (size_t)f0 * K, (uint32_t)(nf * K * 4), bar(b));
        };
        mbar_expect_tx(bar(0), l.dO * a.qd * 4);
        slice(l.wo, a.wo, rank * l.dO, l.dO, a.qd, 0);
        mbar_expect_tx(bar(1), 2 * l.Fs * a.d * 4);
        slice(l.wg, a.wg, rank * l.Fs, l.Fs, a.d, 1);
        slice(l.wu, a.wu, rank * l.Fs, l.Fs, a.d, 1);
        mbar_expect_tx(bar(2), l.dO * a.F * 4);
        slice(l.wd, a.wd, rank * l.dO, l.dO, a.F, 2);
        if (a.g_next) {
            mbar_expect_tx(bar(3), l.qs * a.d * 4);
            int base = 0;
            for (int s = 0; s < 3; s++) {  // the slice may span two of Q, K, V
                const int lo = max((int)rank * l.qs, base), hi = min(((int)rank + 1) * l.qs, base + a.n_next[s]);
                if (hi > lo) slice(l.wn + (lo - (int)rank * l.qs) * a.d, a.w_next[s], lo - base, hi - lo, a.d, 3);
                base += a.n_next[s];
            }
        }
    }
    pdl_launch_dependents();
    const int f_o = rank * l.dO, f_h = rank * l.Fs;
    for (int i = tid; i < a.d; i += kScThreads) {  // gains and couplings come with the weights, before the wait
        sm[l.g1 + i] = a.g_mlp[i];
        if (a.g_next) sm[l.g2 + i] = a.g_next[i];
    }
    for (int i = tid; i < l.Fs; i += kScThreads) sm[l.cb + i] = a.coup_b[f_h + i];
    for (int i = tid; i < l.dO; i += kScThreads) sm[l.cc + i] = a.coup_c[f_o + i];
    __syncthreads();
    cluster_sync_all();  // every CTA of the cluster runs: its shared memory may be written
    pdl_wait();
    DBT_TL_WAITED;
    bool ok = true;
    for (int i = tid; i < R * a.qd / 4; i += kScThreads) *reinterpret_cast<float4 *>(sm + l.x + 4 * i) = ldcg4(a.O + 4 * i);
    // a lane's row in the sums over a warp, and the lane that writes it
    const int row = lane / (32 / RM);
    const bool writes = lane % (32 / RM) == 0 && row < R;
    const int twin = row >= a.Bc ? row % a.Bc * (32 / RM) : lane;  // lane of a branch row's primary twin
    // S of this warp's first O-projection feature, requested with the rows
    float s_in = warp < l.dO && writes ? __ldcg(a.S + (size_t)row * a.d + f_o + warp) : 0.f;
    __syncthreads();
    // Sends this CTA's slice [r][f0 .. f0 + n) of the rows at float offset off (row stride K) to all CTAs, warp w to CTA w, in
    // 16-byte pieces (single words were three times as slow), and waits for the bytes of the other slices: exchange e of three.
    static_assert(NW == kScCtas, "a warp per CTA");
    auto share = [&](int off, int K, int f0, int n, int e) {
        __syncthreads();
        const int pieces = n / 4;
        if (warp != (int)rank)
            for (int i = lane; i < R * pieces; i += 32) {
                const float *src = sm + off + i / pieces * K + f0 + 4 * (i % pieces);
                st_async4(mapa_u32(smem_u32(src), warp), *reinterpret_cast<const float4 *>(src), mapa_u32(bar(4 + e), warp));
            }
        ok = mbar_wait_cluster(bar(4 + e), 0) && ok;
    };
    DBT_TL_MARK(0);
    // O projection + residual
    ok = mbar_wait(bar(0), 0) && ok;
    for (int i = warp; i < l.dO; i += NW) {
        const float y = sc_dot<RM>(sm + l.wo + i * a.qd, sm + l.x, a.qd, R);
        if (i != warp) s_in = writes ? __ldcg(a.S + (size_t)row * a.d + f_o + i) : 0.f;
        if (writes) sm[l.s + row * a.d + f_o + i] = s_in + y;
    }
    share(l.s, a.d, f_o, l.dO, 0);
    DBT_TL_MARK(1);
    // gate | up, SwiGLU, b coupling
    ok = mbar_wait(bar(1), 0) && ok;
    ScRows<RM> xr;
    xr.load(sm + l.s, sm + l.g1, a.d, R, a.eps);
    for (int i = warp; i < l.Fs; i += NW) {
        const float *wg = sm + l.wg + i * a.d, *wu = sm + l.wu + i * a.d;
        const float gt = xr.dot(wg, a.d), up = xr.dot(wu, a.d);
        float h = silu(gt) * up;
        const float h1 = __shfl_sync(0xffffffffu, h, twin);
        if (row >= a.Bc) h = fmaf(sm[l.cb + i], h1, h);
        if (writes) sm[l.h + row * a.F + f_h + i] = h;
    }
    share(l.h, a.F, f_h, l.Fs, 1);
    if (!a.g_next) cluster_arrive();
    DBT_TL_MARK(2);
    // down, c coupling, residual
    ok = mbar_wait(bar(2), 0) && ok;
    for (int i = warp; i < l.dO; i += NW) {
        const int f = f_o + i;
        float mv = sc_dot<RM>(sm + l.wd + i * a.F, sm + l.h, a.F, R);
        const float m1 = __shfl_sync(0xffffffffu, mv, twin);
        if (row >= a.Bc) mv = fmaf(sm[l.cc + i], m1, mv);
        if (writes) {
            const float y = sm[l.s + row * a.d + f] + mv;
            sm[l.s + row * a.d + f] = y;
            if (ok) a.S[(size_t)row * a.d + f] = y;
        }
    }
    if (a.g_next) {
        share(l.s, a.d, f_o, l.dO, 2);
        cluster_arrive();
        DBT_TL_MARK(3);
        // the next layer's Q | K | V
        ok = mbar_wait(bar(3), 0) && ok;
        xr.load(sm + l.s, sm + l.g2, a.d, R, a.eps);
        for (int i = warp; i < l.qs; i += NW) {
            const float y = xr.dot(sm + l.wn + i * a.d, a.d);
            int f = rank * l.qs + i, s = 0;
            while (f >= a.n_next[s]) f -= a.n_next[s++];
            if (ok && writes && row < a.rows_next[s]) a.y_next[s][(size_t)row * a.n_next[s] + f] = y;
        }
    }
    if (!ok && lane == 0) report(a.status, kStatusWaitExpired, 800 + warp);
    // No CTA leaves before all have sent what they had to send (the arrivals stand behind the last exchange).  Where a wait ran out,
    // the bytes on their way here are waited for once more, so that none lands in the memory of a CTA that has gone.
    cluster_wait();
    if (!ok)
        for (int e = 0; e < (a.g_next ? 3 : 2); e++) mbar_wait_cluster(bar(4 + e), 0);
    DBT_TL_END("smlp");
}

// The shared output matrix at up to 8 rows and 256 columns: a warp takes four features, whose weights it requests before the
// dependency wait, and keeps the rows in registers (a warp per feature, 4096 of them, ran in waves: 17 us by events, now 7.5).
template <int RM>
__global__ void __launch_bounds__(256) logits_small_kernel(const SmallLin a) {
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, K = a.K, R = a.rows[0], V = a.n_out[0];
    const int f0 = (blockIdx.x * 8 + warp) * 4;
    const float *W = reinterpret_cast<const float *>(a.W[0]);
    typedef ScRows<RM, true> Rows;
    float4 w[4][2];
#pragma unroll
    for (int j = 0; j < 4; j++) Rows::weights(W + (size_t)min(f0 + j, V - 1) * K, K, w[j]);
    pdl_wait();
    Rows xr;
    xr.load(a.X, a.g, K, R, a.eps, a.g != nullptr);
    const int row = lane / (32 / RM), sub = lane % (32 / RM);
    float y[4];
#pragma unroll
    for (int j = 0; j < 4; j++) y[j] = xr.dot(w[j]);
#pragma unroll
    for (int j = 0; j < 4; j++)
        if (sub == j % (32 / RM) && row < R && f0 + j < V) a.Y[0][(size_t)row * V + f0 + j] = y[j];
}

}  // namespace dbt
