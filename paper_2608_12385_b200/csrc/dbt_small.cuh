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
// Measured on the tiny fp32 model (4 layers, batch 2, context 64..80): 192 -> 128 us per step, copies of the outputs included.
#pragma once

#include "dbt_fused.cuh"
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
            if (a.g) load8(a.g + k, gn[c]);
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
                const float *xp = a.X + (size_t)min(r0 + r, rows - 1) * K + k;
                const float4 x0 = ldcg4(xp), x1 = ldcg4(xp + 4);
                x[r][0] = x0.x, x[r][1] = x0.y, x[r][2] = x0.z, x[r][3] = x0.w;
                x[r][4] = x1.x, x[r][5] = x1.y, x[r][6] = x1.z, x[r][7] = x1.w;
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
            if (a.g) load8(a.g + k, gv);
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
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x, g = blockIdx.y, sp = blockIdx.z, nsplit = gridDim.z;
    const int nq = a.P * a.G, q_dim = a.n_kv * a.G * DH, kv_dim = a.n_kv * DH, half = DH / 2;
    pdl_launch_dependents();
    pdl_wait();
    const int pos = ld_mut(a.seq_len + b), nkeys = pos + 1;
    const int n_act = min(nsplit, (nkeys + kSaSplitKeys - 1) / kSaSplitKeys);  // by the sequence's own length
    if (sp >= n_act) return;
    const int pages = (nkeys + 15) >> 4, pps = (pages + n_act - 1) / n_act;
    const int jbeg = min(nkeys, sp * pps * 16), jend = min(nkeys, jbeg + pps * 16);
    const bool owns_new = pos >= jbeg && pos < jend;
    const int32_t *pt = a.page_table + (size_t)b * a.pt_stride;
    auto row_of = [&](int j) {  // pool row of key j of this head
        int page = pt[j >> 4];
        if (page < 0 || page >= a.num_pages) {
            report(a.status, kStatusBadPage, page);
            page = 0;
        }
        return (((size_t)page * a.n_kv + g) * 16 + (j & 15)) * DH;
    };
    // the new key and value: rotated, appended by the split that holds the position
    if (owns_new && tid < half) {
        const float2 t = a.rope[(size_t)pos * half + tid];
        const float *kn = a.Kn + (size_t)b * kv_dim + g * DH, *vn = a.Vn + (size_t)b * kv_dim + g * DH;
        const float x0 = __ldcg(kn + tid), x1 = __ldcg(kn + tid + half), v0 = __ldcg(vn + tid), v1 = __ldcg(vn + tid + half);
        const int page = pt[pos >> 4];
        if (page >= 0 && page < a.num_pages) {
            const size_t r = row_of(pos);
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
    __syncthreads();  // (the appended row too: written by this block)
    const int dl = (lane % LPK) * 4, ksub = warp * KPW + lane / LPK;  // this thread's four dims; its key within KPB
    float o[NQ][4];
#pragma unroll
    for (int q = 0; q < NQ; q++) o[q][0] = o[q][1] = o[q][2] = o[q][3] = 0.f;
    for (int j0 = jbeg; j0 < jend; j0 += kSaChunk) {
        const int cnt = min(kSaChunk, jend - j0);
        constexpr int U = 4;  // keys in flight per lane group
        float4 vv[U];
#pragma unroll
        for (int u = 0; u < U; u++) {  // the first values travel with the first keys
            const int j = ksub + u * KPB;
            vv[u] = j < cnt ? ldcg4(a.vpool + row_of(j0 + j) + dl) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int k0 = 0; k0 < cnt; k0 += U * KPB) {
            float4 kk[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int j = k0 + ksub + u * KPB;
                kk[u] = j < cnt ? ldcg4(a.kpool + row_of(j0 + j) + dl) : make_float4(0.f, 0.f, 0.f, 0.f);
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
                    vv[u] = j < cnt ? ldcg4(a.vpool + row_of(j0 + j) + dl) : make_float4(0.f, 0.f, 0.f, 0.f);
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

}  // namespace dbt
