// grad.cu -- reverse mode of ComputeAlgDist (per-sweep rescale form of Alg. 1)
// with respect to the undirected edge weights.
//
// Forward (sweep_kernels.cuh stores the frame s_t, rescaled iterate
// x_t = a_t s_t + b_t with a_t = 1/(max - min)(s_t), b_t = -a_t min(s_t) - 1/2,
// x_0 = s_0 = the Philox init):
//     y_t = M x_{t-1},  M = (1-omega) I + omega D^-1 W,   x_t = rescale(y_t),
//     rho_e = |x_k,i - x_k,j|.
// Given rhobar = dL/drho, backwards for t = k .. 1:
//     xbar_k,i   = sum_j c_ij (x_k,i - x_k,j),  c_ij = rhobar_e / rho_e (0 if rho_e = 0)
//     ybar_t     = a_t xbar_t + e_argmin a_t A_t - e_argmax a_t B_t,
//                  A_t = sum_i xbar_t,i (x_t,i - 1/2),  B_t = sum_i xbar_t,i (x_t,i + 1/2)
//                  (lowest-index argmin/argmax; ybar = 0 when max == min)
//     xbar_{t-1} = (1-omega) ybar_t + omega W (D^-1 ybar_t)        (W symmetric)
//     dL/dw_ij  += omega ybar_t,i . (x_{t-1,j} - avg_i) / D_i,   avg_i = D_i^-1 sum_l w_il x_{t-1,l}
// and in the stored frame x_{t-1,j} - avg_i = a_{t-1} (s_{t-1,j} - sigma_i) with
// sigma_i = D_i^-1 sum_l w_il s_{t-1,l}.  With U = D^-1 ybar_t the kernels keep,
// for the two entries p = (i, j), q = (j, i) of every edge,
//     G_p = sum_t (a_{t-1} U_i) . s_{t-1,j},   G_q = sum_t (a_{t-1} s_{t-1,i}) . U_j;
// both come from one visit of the edge's upper entry, which has row i in
// registers and fetches [U_j | s_j].  The sigma term needs no gather of its own:
// sum_t a_{t-1} U_i . sigma_i = C_i = D_i^-1 sum_l w_il G_il, taken once at the end, and
// dL/dw_e = omega (G_p - C_i + G_q - C_j).  All sums are in a fixed order (no
// floating-point atomics), G and C in FP64.
//
// Memory: the stored vectors after sweeps 0, c, 2c, ... (c = ceil(sqrt k)) are
// kept by the forward; each segment of c sweeps is recomputed from its
// checkpoint when the backward reaches it.
#include "sweep_kernels.cuh"

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>

struct ad_graph_s::Saved {
    int32_t R = 0, k = 0, c = 1;
    bool all = false;             // ckpt holds every iterate s_0 .. s_k (c = 1)
    double omega = 0.5;
    int32_t stride = 0, nchunks = 0, lpr = 1, cpl = 1;
    std::vector<void *> ckpt;     // stored vectors after sweep 0, c, 2c, ... (all: after every sweep)
    uint32_t *mm = nullptr;       // [2][k][stride] min then max slots of every sweep
    float *rho = nullptr;         // forward distances
};

namespace ad {

void free_saved(ad_graph_t g) {
    if (!g->saved) return;
    for (void *p : g->saved->ckpt) dfree(g, p);
    if (g->saved->mm) dfree(g, g->saved->mm);
    if (g->saved->rho) dfree(g, g->saved->rho);
    delete g->saved;
    g->saved = nullptr;
}

ad_status algebraic_distance_keep(ad_graph_t g, int32_t R, int32_t k, double omega, uint64_t seed, uint32_t stream_id,
                                  float *rho_dev, bool sqrt_checkpoints) {
    if (g->G != 1) return fail(AD_ERR_INVALID_ARG, "the reverse mode takes a single graph, not a batch");
    free_saved(g);
    auto *sv = new ad_graph_s::Saved();
    g->saved = sv;
    sv->R = R;
    sv->k = k;
    sv->omega = omega;
    const int V = 4;
    const int nch = (R + V - 1) / V;
    int p2 = 1;
    while (p2 < nch) p2 <<= 1;
    sv->nchunks = nch;
    sv->lpr = p2 < 32 ? p2 : 32;
    sv->cpl = p2 / sv->lpr;
    sv->stride = p2 * V;
    const size_t xbytes = ((size_t)g->n + 1) * sv->stride * sizeof(float);
    // every iterate s_0 .. s_k when they fit in half of the free memory (the
    // backward then recomputes nothing), else s_0, s_c, s_2c, ... with c = ceil(sqrt k)
    size_t free_b = 0, total_b = 0;
    const bool all = !sqrt_checkpoints && k > 0 && cudaMemGetInfo(&free_b, &total_b) == cudaSuccess &&
                     (size_t)(k + 1) * xbytes <= free_b / 2;
    int c = 1;
    if (!all)
        while ((int64_t)c * c < k) ++c;
    sv->c = c;
    sv->all = all;
    KeepSpec ks;
    ks.every = c;
    const int nck = all ? k + 1 : k > 0 ? (k + c - 1) / c : 1;
    for (int j = 0; j < nck; ++j) {
        void *p = nullptr;
        AD_TRY(dalloc(g, xbytes, &p));
        sv->ckpt.push_back(p);
    }
    ks.ckpt = sv->ckpt;
    AD_TRY(dalloc_t(g, 2 * (size_t)(k > 0 ? k : 1) * sv->stride, &sv->mm));
    ks.mm_copy = sv->mm;
    AD_TRY(algebraic_distance(g, R, k, omega, seed, stream_id, AD_STORAGE_FP32, 0, rho_dev, &ks));
    AD_TRY(dalloc_t(g, g->m + 1, &sv->rho));
    if (g->m > 0)
        AD_CUDA_TRY(cudaMemcpyAsync(sv->rho, rho_dev, g->m * sizeof(float), cudaMemcpyDeviceToDevice, g->stream));
    return AD_OK;
}

// ----------------------------------------------------------------------------
// Kernels (FP32 stored vectors)
// ----------------------------------------------------------------------------
struct BwArgs {
    const int64_t *rp;
    const int32_t *col;
    const float *w;
    const float *Dinv;
    const int64_t *eid;
    int32_t stride, nchunks, R;
    float omega;
    // distance backward
    const float *rho, *rhobar;
    const float *a_k;            // [stride] per-vector scale of the last iterate (device)
    // sweep backward
    const float *Z;              // rows [U_i | s_{t-1,i}], 2 * stride floats each
    const float *Ybar;           // ybar_t
    const float *a_prev;         // [stride] a_{t-1} (device; nullptr: 1, for t = 1)
    const float *Sk;             // stored s_k (distance backward input)
    const int64_t *upos, *eoff;
    float *xbar_out;
    double *G;                   // [m][2]: G_p and G_q of every edge
    float *part;                 // [n_big][2][stride]
    // plan
    const int32_t *big_row, *big_chunk, *medium_row, *small_row;
    uint32_t *big_counter;
    int64_t n_big, n_medium, n_small_rows, n_tasks, n_wide;
};

template <int CPL>
__device__ __forceinline__ void ld4(const float *base, int64_t row, int stride, int q, float *out) {
    const float4 f = __ldg(reinterpret_cast<const float4 *>(base + row * stride) + q);
    out[0] = f.x; out[1] = f.y; out[2] = f.z; out[3] = f.w;
}

// ---- distance backward: xbar_k from rhobar ----------------------------------
// One row (or chunk of a row) p in [p0, p1) processed by the warp (G groups
// over neighbours) or by one group (G = 1 group, gstride = 1):
// acc_a = sum c_p s_j, acc_b = sum c_p (scalar in slot 0)
template <int LPR, int CPL>
__device__ __forceinline__ void bw_gather(const BwArgs &a, int64_t p0, int64_t p1, int first, int gstride, int gl,
                                          float (&acc_a)[CPL * 4], float (&acc_b)[CPL * 4]) {
    for (int64_t p = p0 + first; p < p1; p += gstride) {
        const int32_t j = __ldg(a.col + p);
        {
            const int64_t e = a.eid[p];
            const float r = a.rho[e];
            const float cf = r > 0.f ? a.rhobar[e] / r : 0.f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int q = gl + c * LPR;
                if (q < a.nchunks) {
                    float s[4];
                    ld4<CPL>(a.Sk, j, a.stride, q, s);
#pragma unroll
                    for (int e4 = 0; e4 < 4; ++e4) acc_a[c * 4 + e4] = fmaf(cf, s[e4], acc_a[c * 4 + e4]);
                }
            }
            acc_b[0] += cf;
        }
    }
}

// xbar_k,i = a_k (sum_j c_ij s_i - sum_j c_ij s_j)
template <int LPR, int CPL>
__device__ __forceinline__ void bw_finish(const BwArgs &a, int64_t row, int gl, const float (&own)[CPL * 4],
                                          const float (&acc_a)[CPL * 4], const float (&acc_b)[CPL * 4]) {
    float *xo = a.xbar_out + row * (int64_t)a.stride;
    const float csum = acc_b[0];
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const int q = gl + c * LPR;
        if (q < a.nchunks) {
#pragma unroll
            for (int e4 = 0; e4 < 4; ++e4) {
                const int r = q * 4 + e4;
                xo[r] = (r < a.R ? __ldg(a.a_k + r) : 0.f) * (csum * own[c * 4 + e4] - acc_a[c * 4 + e4]);
            }
        }
    }
}

// a row of floats (pitch floats apart), the lane's chunks
template <int LPR, int CPL>
__device__ __forceinline__ void bw_row(const float *base, int64_t row, int pitch, int nchunks, int gl, float (&own)[CPL * 4]) {
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const int q = gl + c * LPR;
        if (q < nchunks) ld4<CPL>(base, row, pitch, q, own + c * 4);
        else {
#pragma unroll
            for (int e4 = 0; e4 < 4; ++e4) own[c * 4 + e4] = 0.f;
        }
    }
}

template <int LPR, int CPL>
__global__ void __launch_bounds__(256) k_bw(BwArgs a) {
    constexpr int E = CPL * 4, G = 32 / LPR;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int grp = lane / LPR, gl = lane % LPR;
    const int64_t W = (int64_t)gridDim.x * nwarps;
    for (int64_t task = (int64_t)blockIdx.x * nwarps + warp; task < a.n_tasks; task += W) {
        float acc_a[E], acc_b[E], own[E];
#pragma unroll
        for (int e = 0; e < E; ++e) { acc_a[e] = 0.f; acc_b[e] = 0.f; }
        if (task < a.n_big) {
            const int64_t row = a.big_row[task];
            const int32_t c = a.big_chunk[task];
            const int64_t rb = a.rp[row], re = a.rp[row + 1];
            const int64_t p0 = rb + (int64_t)c * kChunk, p1 = min(re, p0 + kChunk);
            bw_row<LPR, CPL>(a.Sk, row, a.stride, a.nchunks, gl, own);
            bw_gather<LPR, CPL>(a, p0, p1, grp, G, gl, acc_a, acc_b);
            reduce_groups<LPR, E>(acc_a);
            reduce_groups<LPR, E>(acc_b);
            float *part = a.part + task * (int64_t)2 * a.stride;
            if (grp == 0) {
#pragma unroll
                for (int cc = 0; cc < CPL; ++cc) {
                    const int q = gl + cc * LPR;
                    if (q < a.nchunks) {
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            __stcg(part + q * 4 + e4, acc_a[cc * 4 + e4]);
                            __stcg(part + a.stride + q * 4 + e4, acc_b[cc * 4 + e4]);
                        }
                    }
                }
                __threadfence();
            }
            __syncwarp();
            const int64_t t0 = task - c;
            const int32_t nchunk = (int32_t)((re - rb + kChunk - 1) / kChunk);
            uint32_t old = 0;
            if (lane == 0) old = atomicAdd(a.big_counter + t0, 1u);
            old = __shfl_sync(0xffffffffu, old, 0);
            if (old == (uint32_t)(nchunk - 1)) {
                __threadfence();
                if (grp == 0) {
                    float sa[E], sb[E];
#pragma unroll
                    for (int e = 0; e < E; ++e) { sa[e] = 0.f; sb[e] = 0.f; }
                    for (int32_t k2 = 0; k2 < nchunk; ++k2) {
                        const float *pp = a.part + (t0 + k2) * (int64_t)2 * a.stride;
#pragma unroll
                        for (int cc = 0; cc < CPL; ++cc) {
                            const int q = gl + cc * LPR;
                            if (q < a.nchunks) {
#pragma unroll
                                for (int e4 = 0; e4 < 4; ++e4) {
                                    sa[cc * 4 + e4] += __ldcg(pp + q * 4 + e4);
                                    sb[cc * 4 + e4] += __ldcg(pp + a.stride + q * 4 + e4);
                                }
                            }
                        }
                    }
                    bw_finish<LPR, CPL>(a, row, gl, own, sa, sb);
                }
                if (lane == 0) a.big_counter[t0] = 0u;
            }
        } else if (task < a.n_big + a.n_medium) {
            const int64_t row = a.medium_row[task - a.n_big];
            bw_row<LPR, CPL>(a.Sk, row, a.stride, a.nchunks, gl, own);
            bw_gather<LPR, CPL>(a, a.rp[row], a.rp[row + 1], grp, G, gl, acc_a, acc_b);
            reduce_groups<LPR, E>(acc_a);
            reduce_groups<LPR, E>(acc_b);
            if (grp == 0) bw_finish<LPR, CPL>(a, row, gl, own, acc_a, acc_b);
        } else {
            const int64_t si = (task - a.n_big - a.n_medium) * G + grp;
            if (si < a.n_small_rows) {
                const int64_t row = a.small_row[si];
                bw_row<LPR, CPL>(a.Sk, row, a.stride, a.nchunks, gl, own);
                bw_gather<LPR, CPL>(a, a.rp[row], a.rp[row + 1], 0, 1, gl, acc_a, acc_b);
                bw_finish<LPR, CPL>(a, row, gl, own, acc_a, acc_b);
            }
        }
    }
}

// ---- sweep backward ----------------------------------------------------------
// Per row: acc = sum_j w_ij U_j over all entries, and for the entries of its
// upper part the two dots of the edge.  Bound by the gathers: a lower entry
// fetches the U half of row j (stride floats), an upper one both halves, 1.5
// strides per entry on average where fetching [U | s] everywhere took 2; the sum of
// w s_j that this saves is recovered from G (top of the file).  Backward of R-MAT 22,
// R = 32, k = 30 with the streaming passes below: 214 -> 132 ms.
#ifndef AD_BW_MINB
#define AD_BW_MINB 3          // CTAs per SM (R-MAT 22, k = 30: backward 132 ms; 160 with 2, 166 with 4)
#endif
constexpr int kBwUB = 4;      // upper entries in flight per lane group (two row chunks each)

// the upper entries t = first, first + gstride, ... < len at q0, for a lane group;
// all 32 lanes call it.  au = a U_i, as = a s_i; Gp: accumulators of entry 0.
template <int LPR, int CPL>
__device__ __forceinline__ void bw_upper(const BwArgs &a, int64_t q0, int len, int first, int gstride, int gl,
                                         const float (&au)[CPL * 4], const float (&as)[CPL * 4], double *Gp,
                                         float (&acc)[CPL * 4]) {
    constexpr int UB = kBwUB, K = 2 * UB, NC = LPR < UB ? UB / LPR : 1;
    constexpr int NH = K / LPR > 0 ? K / LPR : 1;
    constexpr int WS = LPR > K ? LPR / K : 1;   // lanes that hold the same sum
    const int pitch = 2 * a.stride;
    int which = 0;                              // first of the sums this lane holds after group_sums
#pragma unroll
    for (int o = LPR / 2, c = K; o >= 1; o >>= 1)
        if (c > 1) {
            if (gl & o) which += c / 2;
            c >>= 1;
        }
    const bool writer = gl % WS == 0;
    const int maxlen = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(len - first, 0));
    int32_t cjn[NC];
    float wjn[NC];
    auto load_cols = [&](int b) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int l = i * LPR + gl, t = first + (b + l) * gstride;
            const bool ok = l < UB && t < len;
            cjn[i] = ok ? ld_stream(a.col + q0 + t) : 0;
            wjn[i] = ok ? (a.w ? ld_stream(a.w + q0 + t) : 1.f) : 0.f;
        }
    };
    load_cols(0);
    for (int b = 0; b * gstride < maxlen; b += UB) {
        int32_t cj[NC];
        float wj[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) { cj[i] = cjn[i]; wj[i] = wjn[i]; }
        load_cols(b + UB);
        double gold[NH];   // the accumulators this lane will add to, loaded with the rows
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int t = first + (b + (which + i) / 2) * gstride;
            gold[i] = writer && t < len ? __ldcg(Gp + 2 * (int64_t)t + (which + i) % 2) : 0.0;
        }
        float4 uu[UB][CPL], ss[UB][CPL];
        float wt[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int32_t j = __shfl_sync(0xffffffffu, cj[u / LPR], u % LPR, LPR);
            wt[u] = __shfl_sync(0xffffffffu, wj[u / LPR], u % LPR, LPR);
            const bool in = first + (b + u) * gstride < len;
            const float4 *z = reinterpret_cast<const float4 *>(a.Z + (int64_t)j * pitch);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int q = gl + c * LPR;
                const bool ok = in && q < a.nchunks;
                uu[u][c] = ok ? __ldg(z + q) : make_float4(0.f, 0.f, 0.f, 0.f);
                ss[u][c] = ok ? __ldg(z + a.stride / 4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        float dot[K];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            dot[2 * u] = 0.f;
            dot[2 * u + 1] = 0.f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const float uf[4] = {uu[u][c].x, uu[u][c].y, uu[u][c].z, uu[u][c].w};
                const float sf[4] = {ss[u][c].x, ss[u][c].y, ss[u][c].z, ss[u][c].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[c * 4 + e] = fmaf(wt[u], uf[e], acc[c * 4 + e]);
                    dot[2 * u] = fmaf(au[c * 4 + e], sf[e], dot[2 * u]);
                    dot[2 * u + 1] = fmaf(as[c * 4 + e], uf[e], dot[2 * u + 1]);
                }
            }
        }
        int w2 = 0;
        group_sums<LPR, K>(dot, gl, 0xffffffffu, w2);
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int t = first + (b + (which + i) / 2) * gstride;
            if (writer && t < len) Gp[2 * (int64_t)t + (which + i) % 2] = gold[i] + (double)dot[i];
        }
    }
}

// The part [p0, p0 + len) of a row whose upper entries start at `upos`, by the
// whole warp (WARP) or by a lane group per row; S: sum of w U_j (WARP: over all groups).
template <int LPR, int CPL, bool WARP>
__device__ __forceinline__ void bw_part(const BwArgs &a, const SweepArgs &ga, int64_t row, int64_t p0, int len, int lane,
                                        float (&S)[CPL * 4]) {
    constexpr int E = CPL * 4, G = 32 / LPR;
    const int gl = lane % LPR, grp = lane / LPR;
    const int64_t up = len > 0 ? a.upos[row] : 0;
    const int lower = len > 0 ? (int)min((int64_t)len, max((int64_t)0, up - p0)) : 0;
    team_gather<float, LPR, CPL, WARP ? G : 1, 1, AD_SWEEP_UB, false>(ga, p0, lower, lane, S);
    float au[E], as[E], acc[E];
    bw_row<LPR, CPL>(a.Z, row, 2 * a.stride, a.nchunks, gl, au);
    bw_row<LPR, CPL>(a.Z + a.stride, row, 2 * a.stride, a.nchunks, gl, as);
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = (gl + c * LPR) * 4 + e;
            const float av = r < a.R ? (a.a_prev ? __ldg(a.a_prev + r) : 1.f) : 0.f;
            au[c * 4 + e] *= av;
            as[c * 4 + e] *= av;
            acc[c * 4 + e] = 0.f;
        }
    const int64_t q0 = p0 + lower;
    double *Gp = a.G + 2 * (len > lower ? a.eoff[row] + (q0 - up) : 0);
    bw_upper<LPR, CPL>(a, q0, len - lower, WARP ? grp : 0, WARP ? G : 1, gl, au, as, Gp, acc);
    if (WARP) reduce_groups<LPR, E>(acc);
#pragma unroll
    for (int e = 0; e < E; ++e) S[e] += acc[e];
}

// xbar_{t-1,i} = (1 - omega) ybar_i + omega sum_j w_ij U_j
template <int LPR, int CPL>
__device__ __forceinline__ void bw_store(const BwArgs &a, int64_t row, int gl, const float (&S)[CPL * 4]) {
    const float om = a.omega, om1 = 1.f - a.omega;
    float4 *xo = reinterpret_cast<float4 *>(a.xbar_out + row * (int64_t)a.stride);
    const float4 *yb = reinterpret_cast<const float4 *>(a.Ybar + row * (int64_t)a.stride);
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const int q = gl + c * LPR;
        if (q < a.nchunks) {
            const float4 y = __ldg(yb + q);
            xo[q] = make_float4(fmaf(om1, y.x, om * S[c * 4]), fmaf(om1, y.y, om * S[c * 4 + 1]),
                                fmaf(om1, y.z, om * S[c * 4 + 2]), fmaf(om1, y.w, om * S[c * 4 + 3]));
        }
    }
}

template <int LPR, int CPL>
__global__ void __launch_bounds__(256, AD_BW_MINB) k_bw_sweep(BwArgs a) {
    constexpr int E = CPL * 4, G = 32 / LPR;
    const int lane = threadIdx.x & 31, grp = lane / LPR, gl = lane % LPR;
    SweepArgs ga;                       // what team_gather reads: U_j is the first half of row j of Z
    ga.col = a.col;
    ga.w = a.w;
    ga.x_in = a.Z;
    ga.stride = 2 * a.stride;
    ga.nchunks = a.nchunks;
    const uint32_t n_big = (uint32_t)a.n_big, n_wide = (uint32_t)a.n_wide;
    const uint32_t n_rows = (uint32_t)(a.n_medium - a.n_wide + a.n_small_rows);   // rows of one lane group
    const TaskIter it = task_iter(n_big + n_wide + (n_rows + G - 1) / G, 0);
    for (uint32_t task = it.t; task < it.t_end; task += it.step) {
        float S[E];
        if (task < n_big) {
            // ---- a chunk of a high-degree row; the last chunk adds the partial sums in order
            const int64_t row = a.big_row[task];
            const int32_t c = a.big_chunk[task];
            const int64_t rb = a.rp[row], re = a.rp[row + 1];
            const int64_t p0 = rb + (int64_t)c * kChunk;
            bw_part<LPR, CPL, true>(a, ga, row, p0, (int)(min(re, p0 + kChunk) - p0), lane, S);
            float4 *part = reinterpret_cast<float4 *>(a.part + task * (int64_t)a.stride);
            if (grp == 0) {
#pragma unroll
                for (int cc = 0; cc < CPL; ++cc)
                    if (gl + cc * LPR < a.nchunks)
                        __stcg(part + gl + cc * LPR, make_float4(S[cc * 4], S[cc * 4 + 1], S[cc * 4 + 2], S[cc * 4 + 3]));
                __threadfence();
            }
            __syncwarp();
            const uint32_t t0 = task - c;
            const int32_t nchunk = (int32_t)((re - rb + kChunk - 1) / kChunk);
            uint32_t old = 0;
            if (lane == 0) old = atomicAdd(a.big_counter + t0, 1u);
            old = __shfl_sync(0xffffffffu, old, 0);
            if (old == (uint32_t)(nchunk - 1)) {
                __threadfence();
                SweepArgs pa;
                pa.part = a.part;
                pa.stride = a.stride;
                pa.nchunks = a.nchunks;
                sum_partials<float, LPR, CPL>(pa, t0, nchunk, grp, gl, S);
                if (grp == 0) bw_store<LPR, CPL>(a, row, gl, S);
                if (lane == 0) a.big_counter[t0] = 0u;
            }
        } else if (task < n_big + n_wide) {
            const int64_t row = a.medium_row[task - n_big];
            const int64_t p0 = a.rp[row];
            bw_part<LPR, CPL, true>(a, ga, row, p0, (int)(a.rp[row + 1] - p0), lane, S);
            if (grp == 0) bw_store<LPR, CPL>(a, row, gl, S);
        } else {
            // ---- G rows of about the same degree, one per lane group
            const uint32_t i = (task - n_big - n_wide) * G + grp, med = (uint32_t)a.n_medium - n_wide;
            const bool have = i < n_rows;
            const int64_t row = !have ? 0 : i < med ? a.medium_row[n_wide + i] : a.small_row[i - med];
            const int64_t p0 = have ? a.rp[row] : 0;
            bw_part<LPR, CPL, false>(a, ga, row, p0, have ? (int)(a.rp[row + 1] - p0) : 0, lane, S);
            if (have) bw_store<LPR, CPL>(a, row, gl, S);
        }
    }
}

// C_i = D_i^-1 sum_l w_il G_il in FP64: a warp per chunk or row, a lane per
// low-degree row; chunks leave their sums in partC, added in order by k_bw_c_big.
__device__ __forceinline__ double bw_entry_g(const double *G, const int64_t *eid, const float *w, int64_t p, bool upper) {
    return (w ? (double)w[p] : 1.0) * G[2 * eid[p] + (upper ? 0 : 1)];
}
__global__ void k_bw_c(BwArgs a, const double *D, double *C, double *partC) {
    const int lane = threadIdx.x & 31;
    const int64_t W = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t n_tasks = a.n_big + a.n_medium + (a.n_small_rows + 31) / 32;
    for (int64_t task = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); task < n_tasks; task += W) {
        if (task < a.n_big + a.n_medium) {
            const bool big = task < a.n_big;
            const int64_t row = big ? a.big_row[task] : a.medium_row[task - a.n_big];
            const int64_t p0 = a.rp[row] + (big ? (int64_t)a.big_chunk[task] * kChunk : 0);
            const int64_t p1 = big ? min(a.rp[row + 1], p0 + kChunk) : a.rp[row + 1], up = a.upos[row];
            double s = 0.0;
            for (int64_t p = p0 + lane; p < p1; p += 32) s += bw_entry_g(a.G, a.eid, a.w, p, p >= up);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) {
                if (big) partC[task] = s;
                else C[row] = s / D[row];
            }
        } else {
            const int64_t i = (task - a.n_big - a.n_medium) * 32 + lane;
            if (i < a.n_small_rows) {
                const int64_t row = a.small_row[i], up = a.upos[row];
                double s = 0.0;
                for (int64_t p = a.rp[row]; p < a.rp[row + 1]; ++p) s += bw_entry_g(a.G, a.eid, a.w, p, p >= up);
                C[row] = s / D[row];
            }
        }
    }
}
__global__ void k_bw_c_big(BwArgs a, const double *D, double *C, const double *partC) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.n_big; t += (int64_t)gridDim.x * blockDim.x) {
        if (a.big_chunk[t] != 0) continue;
        const int64_t row = a.big_row[t];
        double s = 0.0;
        for (int64_t u = t; u < a.n_big && a.big_row[u] == row; ++u) s += partC[u];
        C[row] = s / D[row];
    }
}

// per-block partial sums of A = sum xbar (x - 1/2) and B = sum xbar (x + 1/2),
// x = a (s - lo) - 1/2, and the lowest-index argmin / argmax of each vector
// of the stored iterate (active rows).  A streaming pass over two blocks: a
// thread takes one 16-byte chunk of every so many rows.  Products in FP32 (FP64
// runs on a very narrow pipe on this part), each thread's running sums compensated
// (Kahan), the threads' sums combined in FP64.  B = A + sum xbar.
constexpr int kRedBlocks = 1216;      // 8 per SM: the per-thread sums are latency bound
__device__ __forceinline__ void kahan_add(float &sum, float &comp, float x) {
    const float y = x - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

__global__ void __launch_bounds__(256) k_bw_partial(const float *xbar, const float *S, const int64_t *rp, int64_t n,
                                                    int32_t stride, int32_t R, const uint32_t *mn, const uint32_t *mx,
                                                    const float *a_t, double *partA, double *partB,
                                                    unsigned long long *amin, unsigned long long *amax) {
    __shared__ double sA[4][256], sX[4][256];
    const int nq = stride / 4, q = threadIdx.x & (nq - 1);   // stride is a power of two, at most 256
    const int per = blockDim.x / nq, sub = threadIdx.x / nq;
    float accA[4], cA[4], accX[4], cX[4], lo[4], hi[4], ar[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        accA[e] = cA[e] = accX[e] = cX[e] = 0.f;
        const int r = 4 * q + e;
        lo[e] = r < R ? ord2f(mn[r]) : 0.f;
        hi[e] = r < R ? ord2f(mx[r]) : 0.f;
        ar[e] = r < R ? a_t[r] : 0.f;
    }
    if (4 * q < R)
        for (int64_t i = (int64_t)blockIdx.x * per + sub; i < n; i += (int64_t)gridDim.x * per) {
            if (rp[i + 1] == rp[i]) continue;
            const float4 xb4 = __ldg(reinterpret_cast<const float4 *>(xbar + i * stride) + q);
            const float4 s4 = __ldg(reinterpret_cast<const float4 *>(S + i * stride) + q);
            const float xb[4] = {xb4.x, xb4.y, xb4.z, xb4.w}, sv[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (4 * q + e >= R) break;
                // the lowest-index argmin / argmax of the vector (the rescale's sub-gradient points)
                if (sv[e] == lo[e]) atomicMin(amin + 4 * q + e, (unsigned long long)i);
                if (sv[e] == hi[e]) atomicMin(amax + 4 * q + e, (unsigned long long)i);
                const float xv = ar[e] * (sv[e] - lo[e]) - 0.5f;
                kahan_add(accA[e], cA[e], xb[e] * (xv - 0.5f));
                kahan_add(accX[e], cX[e], xb[e]);
            }
        }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        sA[e][threadIdx.x] = (double)accA[e] - (double)cA[e];
        sX[e][threadIdx.x] = (double)accX[e] - (double)cX[e];
    }
    __syncthreads();
    if (threadIdx.x < R) {
        const int e = threadIdx.x & 3, qq = threadIdx.x >> 2;
        double tA = 0.0, tX = 0.0;
        for (int s2 = 0; s2 < per; ++s2) { tA += sA[e][s2 * nq + qq]; tX += sX[e][s2 * nq + qq]; }
        partA[(int64_t)blockIdx.x * R + threadIdx.x] = tA;
        partB[(int64_t)blockIdx.x * R + threadIdx.x] = tA + tX;
    }
}

// one warp per vector r: the lanes sum every 32nd block's partial, then a butterfly
__global__ void k_bw_reduce(const double *partA, const double *partB, int nblocks, int32_t R, double *A, double *B) {
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < R; r += blockDim.x >> 5) {
        double tA = 0.0, tB = 0.0;
        for (int b = lane; b < nblocks; b += 32) {
            tA += partA[(int64_t)b * R + r];
            tB += partB[(int64_t)b * R + r];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            tA += __shfl_xor_sync(0xffffffffu, tA, o);
            tB += __shfl_xor_sync(0xffffffffu, tB, o);
        }
        if (lane == 0) {
            A[r] = tA;
            B[r] = tB;
        }
    }
}

// ybar = a xbar (+ a A at the argmin, - a B at the argmax); U = D^-1 ybar, written
// with a copy of s_{t-1} into the rows of Z (the adjoint gather reads both).  A
// streaming pass, one 16-byte chunk per thread; rows of degree 0 are never read
// by anything and are left out.  a * xbar in FP32 is the correctly rounded
// product, i.e. what FP64 then rounding gives; FP64 only at the two corrected
// entries of each vector.
__global__ void __launch_bounds__(256) k_bw_ybar(const float *xbar, const int64_t *rp, const float *Dinv, int64_t n,
                                                 int32_t qshift, int32_t R, const float *a_t, const double *A,
                                                 const double *B, const unsigned long long *amin,
                                                 const unsigned long long *amax, float *ybar, const float *S, float *Z) {
    const int64_t total = n << qshift;
    const int nq = 1 << qshift;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t >> qshift;
        const int q = (int)(t & (nq - 1));
        if (4 * q >= R || rp[i + 1] == rp[i]) continue;
        const float4 xb4 = __ldg(reinterpret_cast<const float4 *>(xbar) + t);
        const float4 s4 = __ldg(reinterpret_cast<const float4 *>(S) + t);
        const float dinv = __ldg(Dinv + i);
        const float xb[4] = {xb4.x, xb4.y, xb4.z, xb4.w};
        float yb[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = 4 * q + e;
            yb[e] = 0.f;
            if (r < R) {
                const float ar = __ldg(a_t + r);
                if (ar > 0.f) {
                    yb[e] = ar * xb[e];
                    const bool lo_i = (unsigned long long)i == __ldg(amin + r), hi_i = (unsigned long long)i == __ldg(amax + r);
                    if (lo_i || hi_i) {
                        double v = (double)ar * xb[e];
                        if (lo_i) v += (double)ar * A[r];
                        if (hi_i) v -= (double)ar * B[r];
                        yb[e] = (float)v;
                    }
                }
            }
        }
        reinterpret_cast<float4 *>(ybar)[t] = make_float4(yb[0], yb[1], yb[2], yb[3]);
        float4 *z = reinterpret_cast<float4 *>(Z) + (i << (qshift + 1)) + q;   // U and s_{t-1} side by side
        z[0] = make_float4(yb[0] * dinv, yb[1] * dinv, yb[2] * dinv, yb[3] * dinv);
        z[nq] = s4;
    }
}

__global__ void k_scale_from_mm(const uint32_t *mn, const uint32_t *mx, int32_t stride, float *a) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= stride) return;
    const float lo = ord2f(mn[r]), hi = ord2f(mx[r]);   // the forward sweeps' scale, bit for bit
    a[r] = hi > lo ? 1.f / (hi - lo) : 0.f;
}

// dL/dw_e = omega (G_p - C_i + G_q - C_j); a thread per CSR entry, the upper ones write
__global__ void k_edge_grad(const int32_t *col, const int32_t *erow, const int64_t *upos, const int64_t *eoff, int64_t nnz,
                            const double *G, const double *C, double omega, float *wbar) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = erow[p], j = col[p];
        if (j <= i) continue;
        const int64_t e = eoff[i] + (p - upos[i]);
        wbar[e] = (float)(omega * ((G[2 * e] - C[i]) + (G[2 * e + 1] - C[j])));
    }
}

template <int LPR, int CPL>
static ad_status launch_bw(ad_graph_t g, const BwArgs &a, bool sweep) {
    int per_sm = 0;
    if (sweep) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bw_sweep<LPR, CPL>, 256, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bw<LPR, CPL>, 256, 0);
    int64_t blocks = (int64_t)(per_sm > 0 ? per_sm : 1) * g->num_sms;
    const int64_t need = (a.n_tasks + 7) / 8;
    if (blocks > need) blocks = need > 0 ? need : 1;
    if (sweep) AD_LAUNCH((k_bw_sweep<LPR, CPL>), (int)blocks, 256, 0, g->stream, a);
    else AD_LAUNCH((k_bw<LPR, CPL>), (int)blocks, 256, 0, g->stream, a);
    return AD_OK;
}

static ad_status dispatch_bw(ad_graph_t g, int lpr, int cpl, const BwArgs &a, bool sweep) {
    switch (lpr * 100 + cpl) {
        case 101: return launch_bw<1, 1>(g, a, sweep);
        case 201: return launch_bw<2, 1>(g, a, sweep);
        case 401: return launch_bw<4, 1>(g, a, sweep);
        case 801: return launch_bw<8, 1>(g, a, sweep);
        case 1601: return launch_bw<16, 1>(g, a, sweep);
        case 3201: return launch_bw<32, 1>(g, a, sweep);
        case 3202: return launch_bw<32, 2>(g, a, sweep);
        default: return fail(AD_ERR_INVALID_ARG, "unsupported R for the reverse mode");
    }
}

static void fill_bw_plan(BwArgs &a, const RowPlan &p) {
    a.big_row = p.big_row; a.big_chunk = p.big_chunk; a.medium_row = p.medium_row; a.small_row = p.small_row;
    a.big_counter = p.big_counter;
    a.n_big = p.n_big; a.n_medium = p.n_medium; a.n_small_rows = p.n_small_rows;
    a.n_wide = p.n_wide;
    a.n_tasks = p.tasks();
}

ad_status backward(ad_graph_t g, const float *rhobar_dev, float *wbar_dev) {
    auto *sv = g->saved;
    const int32_t R = sv->R, k = sv->k, c = sv->c, stride = sv->stride;
    const int64_t n = g->n, nnz = g->nnz;
    AD_TRY(ensure_mirror(g));
    RowPlan *plan = nullptr;
    AD_TRY(get_row_plan(g, 32 / sv->lpr, false, &plan));
    // buffers
    std::vector<float *> seg(c + 1, nullptr);
    if (!sv->all)   // (with every iterate kept, seg points into the kept iterates)
        for (int u = 1; u <= c; ++u) AD_TRY(dalloc_t(g, (n + 1) * stride, &seg[u]));
    float *xbar = nullptr, *xbar2 = nullptr, *ybar = nullptr, *part = nullptr;
    float *a_t = nullptr, *a_p = nullptr, *a_k = nullptr;   // scales of sweep t, t - 1 and k
    double *G = nullptr, *C = nullptr, *partC = nullptr, *partA = nullptr, *partB = nullptr, *A = nullptr, *B = nullptr;
    unsigned long long *amin = nullptr, *amax = nullptr;
    uint32_t *scratch_mm = nullptr;
    AD_TRY(dalloc_t(g, (n + 1) * stride, &xbar));
    AD_TRY(dalloc_t(g, (n + 1) * stride, &xbar2));
    AD_TRY(dalloc_t(g, (n + 1) * stride, &ybar));
    // rows [U_j | s_{t-1,j}] side by side, so that the adjoint gather fetches one
    // contiguous 2 * stride row per entry (measured at R-MAT 22: 2% faster backward)
    float *Z = nullptr;
    AD_TRY(dalloc_t(g, (n + 1) * 2 * (size_t)stride, &Z));
    AD_TRY(dalloc_t(g, (size_t)std::max<int64_t>(plan->n_big, 1) * 2 * stride, &part));
    AD_TRY(dalloc_t(g, 2 * (size_t)g->m + 2, &G));
    AD_TRY(dalloc_t(g, n + 1, &C));
    AD_TRY(dalloc_t(g, (size_t)std::max<int64_t>(plan->n_big, 1), &partC));
    AD_TRY(dalloc_t(g, (size_t)kRedBlocks * stride, &partA));
    AD_TRY(dalloc_t(g, (size_t)kRedBlocks * stride, &partB));
    AD_TRY(dalloc_t(g, stride, &A));
    AD_TRY(dalloc_t(g, stride, &B));
    AD_TRY(dalloc_t(g, stride, &amin));
    AD_TRY(dalloc_t(g, stride, &amax));
    AD_TRY(dalloc_t(g, stride, &a_t));
    AD_TRY(dalloc_t(g, stride, &a_p));
    AD_TRY(dalloc_t(g, stride, &a_k));
    AD_TRY(dalloc_t(g, 2 * stride, &scratch_mm));
    AD_CUDA_TRY(cudaMemsetAsync(G, 0, 2 * (size_t)g->m * sizeof(double), g->stream));
    const uint32_t *mm_min = sv->mm, *mm_max = sv->mm + (size_t)k * stride;
    int qshift = 0;   // stride / 4 = 1 << qshift (a power of two)
    while ((4 << qshift) < stride) ++qshift;
    auto slot_min = [&](int t) { return mm_min + (size_t)(t - 1) * stride; };   // min/max of s_t, t >= 1
    auto slot_max = [&](int t) { return mm_max + (size_t)(t - 1) * stride; };

    BwArgs a;
    memset(&a, 0, sizeof(a));
    a.rp = g->rp; a.col = g->col; a.w = g->w; a.Dinv = g->Dinv; a.eid = g->eid;
    a.stride = stride; a.nchunks = sv->nchunks; a.R = R; a.omega = (float)sv->omega;
    a.rho = sv->rho; a.rhobar = rhobar_dev;
    a.upos = g->upos; a.eoff = g->eoff;
    a.G = G; a.part = part;
    fill_bw_plan(a, *plan);

    const int nseg = k > 0 ? (k + c - 1) / c : 0;
    if (k == 0) {
        // rho of the raw init: xbar_0 = sum c_ij (x_i - x_j); weights do not enter
        AD_CUDA_TRY(cudaMemsetAsync(wbar_dev, 0, g->m * sizeof(float), g->stream));
        return AD_OK;
    }
    bool have_xbar = false;
    for (int j = nseg - 1; j >= 0; --j) {
        const int t0 = j * c, len = std::min(c, k - t0);
        seg[0] = static_cast<float *>(sv->ckpt[j]);
        for (int u = 1; u <= len; ++u) {
            const int t = t0 + u;   // produce s_t from s_{t-1}
            if (sv->all) {          // kept by the forward: the same values the sweep would give
                seg[u] = static_cast<float *>(sv->ckpt[t]);
                continue;
            }
            AD_CUDA_TRY(cudaMemsetAsync(scratch_mm, 0xff, stride * sizeof(uint32_t), g->stream));
            AD_CUDA_TRY(cudaMemsetAsync(scratch_mm + stride, 0, stride * sizeof(uint32_t), g->stream));
            AD_TRY(sweep_step(g, AD_STORAGE_FP32, R, sv->omega, seg[u - 1], seg[u], t >= 2 ? slot_min(t - 1) : nullptr,
                              t >= 2 ? slot_max(t - 1) : nullptr, scratch_mm, scratch_mm + stride));
        }
        if (!have_xbar) {   // distance backward on s_k
            AD_LAUNCH(k_scale_from_mm, 1, 256, 0, g->stream, slot_min(k), slot_max(k), stride, a_k);
            a.a_k = a_k;
            a.Sk = seg[len];
            a.xbar_out = xbar;
            AD_TRY(dispatch_bw(g, sv->lpr, sv->cpl, a, false));
            have_xbar = true;
        }
        for (int u = len; u >= 1; --u) {
            const int t = t0 + u;
            const float *St = seg[u], *Sp = seg[u - 1];
            // rescale adjoint of sweep t
            AD_LAUNCH(k_scale_from_mm, 1, 256, 0, g->stream, slot_min(t), slot_max(t), stride, a_t);
            AD_CUDA_TRY(cudaMemsetAsync(amin, 0xff, stride * sizeof(unsigned long long), g->stream));
            AD_CUDA_TRY(cudaMemsetAsync(amax, 0xff, stride * sizeof(unsigned long long), g->stream));
            AD_LAUNCH(k_bw_partial, kRedBlocks, 256, 0, g->stream, xbar, St, g->rp, n, stride, R, slot_min(t),
                      slot_max(t), a_t, partA, partB, amin, amax);
            AD_LAUNCH(k_bw_reduce, 1, 1024, 0, g->stream, partA, partB, kRedBlocks, R, A, B);
            AD_LAUNCH(k_bw_ybar, g->num_sms * 16, 256, 0, g->stream, xbar, g->rp, g->Dinv, n, qshift, R, a_t, A, B, amin,
                      amax, ybar, Sp, Z);
            // sweep adjoint + weight terms
            if (t >= 2) {
                AD_LAUNCH(k_scale_from_mm, 1, 256, 0, g->stream, slot_min(t - 1), slot_max(t - 1), stride, a_p);
                a.a_prev = a_p;
            } else {
                a.a_prev = nullptr;
            }
            a.Z = Z;
            a.Ybar = ybar;
            a.xbar_out = xbar2;
            AD_TRY(dispatch_bw(g, sv->lpr, sv->cpl, a, true));
            std::swap(xbar, xbar2);
        }
    }
    AD_LAUNCH(k_bw_c, g->num_sms * 8, 256, 0, g->stream, a, g->D, C, partC);
    if (a.n_big > 0) AD_LAUNCH(k_bw_c_big, g->num_sms, 256, 0, g->stream, a, g->D, C, partC);
    AD_LAUNCH(k_edge_grad, g->num_sms * 16, 256, 0, g->stream, g->col, g->erow, g->upos, g->eoff, nnz, G, C, sv->omega,
              wbar_dev);
    AD_CUDA_TRY(cudaStreamSynchronize(g->stream));
    if (!sv->all)
        for (int u = 1; u <= c; ++u) dfree(g, seg[u]);
    for (void *p : {(void *)xbar, (void *)xbar2, (void *)ybar, (void *)Z, (void *)part, (void *)G, (void *)C, (void *)partC,
                    (void *)partA, (void *)partB, (void *)A, (void *)B, (void *)amin, (void *)amax, (void *)a_t, (void *)a_p, (void *)a_k,
                    (void *)scratch_mm})
        dfree(g, p);
    return AD_OK;
}

}  // namespace ad

extern "C" ad_status ad_algebraic_distance_backward(ad_graph_t g, const float *rho_bar, float *w_bar) {
    using namespace ad;
    if (!g) return fail(AD_ERR_INVALID_ARG, "NULL graph");
    if (!g->saved) return fail(AD_ERR_STATE, "no kept state: run ad_algebraic_distance with AD_DIST_KEEP_STATE first");
    if (g->m > 0 && (!rho_bar || !w_bar)) return fail(AD_ERR_INVALID_ARG, "NULL rho_bar or w_bar");
    float *rb = nullptr, *wb = nullptr;
    AD_TRY(dalloc_t(g, g->m + 1, &rb));
    AD_TRY(dalloc_t(g, g->m + 1, &wb));
    AD_TRY(copy_in(g, rb, rho_bar, g->m * sizeof(float)));
    ad_status st = backward(g, rb, wb);
    if (st == AD_OK) st = copy_out(g, w_bar, wb, g->m * sizeof(float));
    if (st == AD_OK) st = cudaStreamSynchronize(g->stream) == cudaSuccess ? AD_OK : fail(AD_ERR_CUDA, "sync");
    dfree(g, rb);
    dfree(g, wb);
    return st;
}
