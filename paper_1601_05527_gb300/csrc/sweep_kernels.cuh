// sweep_kernels.cuh -- kernels of ComputeAlgDist (Alg. 1) on sm_103a: Philox
// init, JOR sweeps with the per-sweep rescale fused into the epilogue, and the
// per-edge distance.  Instantiated once per storage type (sweep_<type>.cu).
//
// Data layout: the R test vectors of vertex i form row i of X[n][stride]
// (stride = lanes_per_row * chunks_per_lane * V elements, 16-byte chunks,
// V = 4 FP32 or 8 16-bit values).  A lane group of LPR lanes owns one row at a
// time; lane gl of the group holds chunks gl, gl + LPR, ... of the row.
//
// Stored frame.  The iterate of Alg. 1 after sweep t is x_t = rescale(M x_{t-1}),
// M = (1-omega) I + omega D^-1 W, rescale mapping [min, max] of each vector
// onto [-1/2, 1/2].  M commutes with adding a constant vector and with scaling,
// and rescale ignores both, so the kernels store
//     s_t = a_{t-1} (M s_{t-1} - s_{t-1}[anchor]),   a_{t-1} = 1 / (max - min)(s_{t-1}),
// which differs from x_t by a per-vector shift only: the same rescaled values,
// the same distances rho = a_t |s_i - s_j|.  The anchor is the vertex of
// largest weighted degree of each graph.  Its value lies inside the bulk of
// the smoothed vector, so the stored values are deviations around zero instead
// of a common offset plus small deviations -- which is what lets 16-bit
// storage resolve the small distances of well-mixed graphs.  Each sweep
// reduces min/max of what it stores; the next launch turns them into a.
#pragma once
#include "ad_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

// Tuning parameters (compile-time; the defaults are the measured choice on GB300).
#ifndef AD_SWEEP_UB
#define AD_SWEEP_UB 8          // independent row loads in flight per lane (FP32 storage)
#endif
#ifndef AD_SWEEP_UB16
#define AD_SWEEP_UB16 4        // ... for the 16-bit storage formats
#endif
#ifndef AD_SWEEP_UBS
#define AD_SWEEP_UBS 4         // ... of a low-degree row
#endif
#ifndef AD_SWEEP_MINB
#define AD_SWEEP_MINB 4        // resident CTAs per SM requested from ptxas for the FP32 sweep
#endif
#ifndef AD_SWEEP_MINB16
#define AD_SWEEP_MINB16 5      // ... for the 16-bit storage formats
#endif
#ifndef AD_DIST_UB
#define AD_DIST_UB 4           // distance: edges of one lane group in flight
#endif
#ifndef AD_DIST_MINB
#define AD_DIST_MINB 4         // ... for the distance pass
#endif
#ifndef AD_MAX_LPR
#define AD_MAX_LPR 32          // most lanes that share one row (more chunks go to each lane beyond it)
#endif
#ifndef AD_COL_STREAM
#define AD_COL_STREAM 1        // 1: read column indices with the streaming (evict-first) hint
#endif

namespace ad {

template <typename T>
__device__ __forceinline__ T ld_stream(const T *p) {
#if AD_COL_STREAM
    return __ldcs(p);
#else
    return __ldg(p);
#endif
}

struct SweepArgs {
    const int64_t *rp;
    const int32_t *col;
    const float *w;        // nullable
    const float *Dinv;
    const double *D;
    const int64_t *upos;   // distance: first upper entry
    const int64_t *eoff;   // distance: edge id of that entry
    const void *x_in;
    void *x_out;
    float *part;           // [n_big][stride] partial sums of big rows
    const uint32_t *mm_prev_min, *mm_prev_max;  // nullptr at t = 0
    uint32_t *mm_min, *mm_max;                  // this sweep's min/max
    float *rho;            // distance output
    // plan
    const int32_t *big_row, *big_chunk, *medium_row, *small_row;
    uint32_t *big_counter;
    int64_t n_big, n_medium, n_small_rows;
    int64_t n_wide;        // sweep: the first n_wide medium rows take a whole warp each, the others share warps
    int64_t n_tasks;       // distance: tasks of the plan; sweep: an upper bound (the kernel counts its own)
    int32_t stride;        // elements per row
    int32_t nchunks;       // valid 16-byte chunks per row (ceil(R / V))
    int32_t R;
    float omega;
    int32_t normalize;
    // batches: graph gph owns rows [voff[gph], voff[gph+1]); min/max slots are
    // [G][stride] per sweep.  Batched launches give each warp a contiguous
    // block of tasks so that consecutive rows mostly share one graph.
    const int64_t *voff;
    int32_t G;
    int32_t blocked;
    const int32_t *anchor;   // [G] vertex whose previous value is subtracted (the stored frame's centre)
    float *ac;               // [G][2][stride]: scale a and centre c of this sweep (k_scale_center)
};

__device__ __forceinline__ int graph_of(const int64_t *voff, int G, int64_t row) {
    int lo = 0, hi = G;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(voff + mid) <= row) lo = mid; else hi = mid;
    }
    return lo;
}

// graph_of with the vertex range of the last graph found kept: the rows a
// lane group visits in a batch mostly lie in one graph, so most lookups are
// one comparison instead of a binary search
struct GraphCache {
    int64_t lo = 0, hi = -1;
    int g = 0;
    __device__ __forceinline__ int of(const int64_t *voff, int G, int64_t row) {
        if (row >= lo && row < hi) return g;
        g = graph_of(voff, G, row);
        lo = __ldg(voff + g);
        hi = __ldg(voff + g + 1);
        return g;
    }
};

// task index range of warp `wid` among `W` warps: [t, t_end) stepping `step`
// (there are at most n < 2^31 tasks)
struct TaskIter {
    uint32_t t, t_end, step;
};
__device__ __forceinline__ TaskIter task_iter(uint32_t n_tasks, int blocked) {
    TaskIter it;
    const uint32_t nw = blockDim.x >> 5, warp = threadIdx.x >> 5;
    if (blocked) {
        // a contiguous range of tasks per CTA, the CTA's warps interleaved inside
        // it: a batch's lanes then meet few graphs (each change of graph flushes
        // the min/max), and the CTA's warps share neighbouring rows
        const uint32_t per = (n_tasks + gridDim.x - 1) / gridDim.x;
        it.t = min(n_tasks, blockIdx.x * per) + warp;
        it.t_end = min(n_tasks, blockIdx.x * per + per);
        it.step = nw;
    } else {
        it.t = blockIdx.x * nw + warp;
        it.t_end = n_tasks;
        it.step = gridDim.x * nw;
    }
    return it;
}

// ----------------------------------------------------------------------------
// Init: x[i][r] = rand(-0.5, 0.5) from Philox, counter (i, r/4, stream), i the
// vertex id inside its graph.  One thread per (row, quad of vectors); rows of
// degree 0 are skipped.
// ----------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void init_rows(const int64_t *__restrict__ rp, int64_t n, int32_t stride, uint32_t seed_lo,
                                          uint32_t seed_hi, uint32_t stream_id, const int64_t *voff, int G,
                                          T *__restrict__ x) {
    const int32_t quads = stride / 4;
    const int64_t total = n * quads;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / quads;
        const int32_t q = (int32_t)(t - i * quads);
        if (rp[i + 1] == rp[i]) continue;
        const int64_t li = G > 1 ? i - voff[graph_of(voff, G, i)] : i;   // id inside its graph
        uint4 c = make_uint4((uint32_t)((uint64_t)li), (uint32_t)((uint64_t)li >> 32), (uint32_t)q, stream_id);
        uint4 u = philox4x32_10(c, make_uint2(seed_lo, seed_hi));
        float v[4] = {unit_centered(u.x), unit_centered(u.y), unit_centered(u.z), unit_centered(u.w)};
        T *dst = x + i * stride + 4 * q;
        if constexpr (sizeof(T) == 4) {
            *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
            uint2 p = make_uint2(Store<T>::pack2(v[0], v[1]), Store<T>::pack2(v[2], v[3]));
            *reinterpret_cast<uint2 *>(dst) = p;
        }
    }
}

template <typename T>
__global__ void k_init(const int64_t *__restrict__ rp, int64_t n, int32_t stride, uint32_t seed_lo,
                       uint32_t seed_hi, uint32_t stream_id, const int64_t *voff, int G, T *__restrict__ x) {
    init_rows<T>(rp, n, stride, seed_lo, seed_hi, stream_id, voff, G, x);
}

// ----------------------------------------------------------------------------
// Helpers for the lane-group kernels
// ----------------------------------------------------------------------------
// Two FP32 additions (or fused multiply-adds) in one packed instruction; each
// half is rounded as the scalar operation would be, so sums are unchanged.
__device__ __forceinline__ void add_f32x2(float &a0, float &a1, float b0, float b1) {
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\t"
        "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}
__device__ __forceinline__ void fma_f32x2(float &a0, float &a1, float w, float b0, float b1) {
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tmov.b64 z, {%4, %4};\n\t"
        "fma.rn.f32x2 x, z, y, x;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1), "f"(w));
}
// acc[e] += f[e] (W: acc[e] = fmaf(w, f[e], acc[e])) for an even count of values
template <int N, bool W>
__device__ __forceinline__ void accumulate(float *acc, const float *f, float w) {
#pragma unroll
    for (int e = 0; e < N; e += 2) {
        if (W) fma_f32x2(acc[e], acc[e + 1], w, f[e], f[e + 1]);
        else add_f32x2(acc[e], acc[e + 1], f[e], f[e + 1]);
    }
}
// Loads of the test-vector block.  Separate launches read it through the
// read-only path; a persistent launch (k_relax) rewrites it between sweeps, so
// there it is read coherently from L2, and the per-sweep scale and centre come
// from shared memory.
template <bool P>
__device__ __forceinline__ uint4 ldx(const uint4 *p) { return P ? __ldcg(p) : __ldg(p); }
// scale and centre of the frame: shared memory (single graphs) or global memory (batches)
__device__ __forceinline__ float4 ldac(const float *p) { return *reinterpret_cast<const float4 *>(p); }

template <typename T, int LPR, int CPL>
struct Lane {
    static constexpr int V = Store<T>::V;
    static constexpr int E = CPL * V;       // elements held by one lane
    static constexpr int G = 32 / LPR;      // groups per warp
};

// Gather-accumulate of CSR rows by teams of lanes.  The sweep is bound by these
// gathers (a row of 16-byte chunks per CSR entry, from L2): what counts is how many
// are in flight and how few instructions stand between them.  Rows of 9 .. 127
// entries share a warp, so that their epilogues run side by side and no butterfly
// over nearly empty groups is needed; from 128 on a row fills a warp by itself.
// Against a warp per medium row with the min/max in registers (one sweep, GB300):
// R-MAT 20, R = 32, FP32 410 -> 303 us (FP16 349 -> 264 us), Barabasi-Albert 200K,
// R = 10, weighted 68 -> 39 us.  The order in which the
// entries of a row are added is fixed: entry t of a row (of a chunk of a long
// row) belongs to residue t mod MOD, the entries of one residue are added in
// order, and the MOD sums are added as a binary tree over adjacent residues.
// How many lanes share that work is free: a team is MOD / RES sub-groups of
// LPR lanes, sub-group s holding the RES residues s RES .. s RES + RES - 1 in
// RES accumulators per lane, and a warp holds RPW teams, a row each.
//   MOD = G, RES = 1   the whole warp on one row (chunks, rows of many entries)
//   MOD = G, RES > 1   several rows per warp: no butterfly over idle groups, and
//                      the epilogue of a row runs beside those of the others
//   MOD = 1, RES = 1   one lane group per row, added one after the other
template <int LPR, int MOD, int RES>
struct Team {
    static constexpr int Q = MOD / RES;         // sub-groups of a team
    static constexpr int TL = LPR * Q;          // lanes of a team
    static constexpr int RPW = 32 / TL;         // teams (rows) per warp
    static constexpr int NL = LPR > 4 ? LPR : 4;   // entries per sub-group and batch
    static constexpr int NC = NL / LPR;         // column indices a lane loads per batch
    static constexpr int BT = NL / RES * MOD;   // entries per team and batch
};

// One batch of a team's row: its NL entries per sub-group, at most UB row loads
// issued before any is used.  FULL: every entry of the batch exists on every
// lane of the warp; otherwise the entries at or past `left` are left out.
template <typename T, int LPR, int CPL, int MOD, int RES, int UB0, bool W, bool P, bool FULL>
__device__ __forceinline__ void gather_batch(const uint4 *const (&xl)[CPL], uint32_t row_q, const int32_t *cj,
                                             const float *wj, int sub, int left, int maxleft,
                                             float (&acc)[RES][CPL * Store<T>::V]) {
    using TM = Team<LPR, MOD, RES>;
    constexpr int V = Store<T>::V, NL = TM::NL, NC = TM::NC;
    constexpr int UB1 = UB0 / CPL > 0 ? UB0 / CPL : 1;
    constexpr int UB = UB1 < NL ? UB1 : NL;
    // Unrolled, but for eight rounds (16-bit storage, a row over the whole warp): the
    // code of the four places that gather outgrows the instruction cache there (a sweep
    // of R-MAT 18, R = 256, rolled: Q16 617 -> 452 us, BF16 372 -> 337 us; 64
    // Watts-Strogatz graphs, BF16: 657 -> 676 us).
    constexpr int ROUNDS = NL / UB < 8 ? NL / UB : 1;
#pragma unroll ROUNDS
    for (int l0 = 0; l0 < NL; l0 += UB) {
        if (!FULL && (l0 / RES) * MOD >= maxleft) break;   // warp-uniform
        uint4 v[UB][CPL];
        float wt[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int l = l0 + u;
            const int32_t nb = __shfl_sync(0xffffffffu, cj[NC == 1 ? 0 : l / LPR], l % LPR, LPR);
            if (W) wt[u] = __shfl_sync(0xffffffffu, wj[NC == 1 ? 0 : l / LPR], l % LPR, LPR);
            const bool ok = FULL || (l / RES) * MOD + sub * RES + l % RES < left;
#pragma unroll
            for (int c = 0; c < CPL; ++c)
                v[u][c] = ok ? ldx<P>(xl[c] + (uint64_t)(uint32_t)nb * row_q) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < UB; ++u)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                float f[V];
                Store<T>::unpack(v[u][c], f);
                accumulate<V, W>(acc[u % RES] + c * V, f, W ? wt[u] : 1.f);
            }
    }
}

// The sum of a team's row: entries p0 .. p0 + d - 1, d the same on all lanes of
// a team (0: no row); all 32 lanes call it.  The next batch's column indices
// (and weights) are loaded before the current batch is used.  Every lane of
// sub-group 0 (for RES = MOD of every one) ends with the row's sum.
template <typename T, int LPR, int CPL, int MOD, int RES, int UB, bool W, bool P>
__device__ __forceinline__ void team_gather_w(const SweepArgs &a, int64_t p0, int d, int lane, float (&S)[CPL * Store<T>::V]) {
    using TM = Team<LPR, MOD, RES>;
    constexpr int V = Store<T>::V, E = CPL * V, NC = TM::NC;
    const int gl = lane % LPR, sub = lane % TM::TL / LPR;
    const uint32_t row_q = (uint32_t)(a.stride / V);
    const uint4 *xl[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c)   // a lane past the row's chunks reads the last one again: its sums are not used
        xl[c] = reinterpret_cast<const uint4 *>(a.x_in) + min(gl + c * LPR, a.nchunks - 1);
    int maxd = d, mind = d;
    if (TM::RPW > 1) {
        maxd = __reduce_max_sync(0xffffffffu, d);
        mind = __reduce_min_sync(0xffffffffu, d);
    }
    float acc[RES][E];
#pragma unroll
    for (int r = 0; r < RES; ++r)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[r][e] = 0.f;
    int32_t cjn[NC], off[NC];
    float wjn[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const int l = i * LPR + gl;
        off[i] = (l / RES) * MOD + sub * RES + l % RES;
        cjn[i] = 0;
        wjn[i] = 0.f;
        if (off[i] < d) {
            cjn[i] = ld_stream(a.col + p0 + off[i]);
            if (W) wjn[i] = ld_stream(a.w + p0 + off[i]);
        }
    }
    for (int b = 0; b < maxd; b += TM::BT) {
        int32_t cj[NC];
        float wj[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            cj[i] = cjn[i];
            wj[i] = wjn[i];
            const int t = b + TM::BT + off[i];
            if (t < d) {
                cjn[i] = ld_stream(a.col + p0 + t);
                if (W) wjn[i] = ld_stream(a.w + p0 + t);
            }
        }
        if (b + TM::BT <= mind) gather_batch<T, LPR, CPL, MOD, RES, UB, W, P, true>(xl, row_q, cj, wj, sub, 0, 0, acc);
        else gather_batch<T, LPR, CPL, MOD, RES, UB, W, P, false>(xl, row_q, cj, wj, sub, d - b, maxd - b, acc);
    }
    // the tree over the residues: inside the lane, then over the sub-groups
#pragma unroll
    for (int o = 1; o < RES; o <<= 1)
#pragma unroll
        for (int r = 0; r + o < RES; r += 2 * o)
#pragma unroll
            for (int e = 0; e < E; ++e) acc[r][e] += acc[r + o][e];
#pragma unroll
    for (int e = 0; e < E; ++e) S[e] = acc[0][e];
#pragma unroll
    for (int o = LPR; o < TM::TL; o <<= 1)
#pragma unroll
        for (int e = 0; e < E; ++e) S[e] += __shfl_xor_sync(0xffffffffu, S[e], o);
}

template <typename T, int LPR, int CPL, int MOD, int RES, int UB, bool P>
__device__ __forceinline__ void team_gather(const SweepArgs &a, int64_t p0, int d, int lane, float (&S)[CPL * Store<T>::V]) {
    if (!a.w) {   // the weighted loop reads a.w: it is reached only with weights present
        team_gather_w<T, LPR, CPL, MOD, RES, UB, false, P>(a, p0, d, lane, S);
        return;
    }
    team_gather_w<T, LPR, CPL, MOD, RES, UB, true, P>(a, p0, d, lane, S);
}

// Residues per lane of the rows that share a warp: 16 sums a lane, that is four
// accumulators of one FP32 chunk (four rows per warp for up to eight lanes per row),
// two where a lane holds eight values (16-bit storage, or two FP32 chunks), one where
// it holds 16: 64 (16-bit: 48) registers hold no more beside the loads in flight.
// Measured at R-MAT 20, R = 32, FP32: 303 us with four, 323 with two.
constexpr int kTeamRes = 4;
template <typename T, int LPR, int CPL>
constexpr int team_res() {
    constexpr int G = 32 / LPR, want = kTeamRes * 4 / (Store<T>::V * CPL);
    return G < want ? G : want;
}

// Sum over the G groups of a warp (butterfly: every group ends with the total).
template <int LPR, int E>
__device__ __forceinline__ void reduce_groups(float (&acc)[E]) {
#pragma unroll
    for (int off = LPR; off < 32; off <<= 1)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], off);
}

// Epilogue of a row: z = (1-omega) s_i + omega Dinv_i S, store a (z - c), track min/max.
template <typename T, int LPR, int CPL, bool P = false>
__device__ __forceinline__ void load_own(const SweepArgs &a, int64_t row, int gl, uint4 (&own)[CPL]) {
    const uint4 *X = reinterpret_cast<const uint4 *>(a.x_in);
    const int64_t row_q = a.stride / Store<T>::V;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const int q = gl + c * LPR;
        own[c] = q < a.nchunks ? ldx<P>(X + row * row_q + q) : make_uint4(0, 0, 0, 0);
    }
}

// Running minimum / maximum of a vector in shared memory, as plain floats: the
// bit patterns of non-negative floats order like integers, those of negative
// ones like unsigned integers reversed.
__device__ __forceinline__ void smem_min(float *p, float f) {
    if (__float_as_int(f) >= 0) atomicMin(reinterpret_cast<int *>(p), __float_as_int(f));
    else atomicMax(reinterpret_cast<unsigned int *>(p), __float_as_uint(f));
}
__device__ __forceinline__ void smem_max(float *p, float f) {
    if (__float_as_int(f) >= 0) atomicMax(reinterpret_cast<int *>(p), __float_as_int(f));
    else atomicMin(reinterpret_cast<unsigned int *>(p), __float_as_uint(f));
}

// The min/max of the stored values of one graph that a warp has met.
//
// Single graphs: one copy per CTA in shared memory, mm[0 .. stride) the minima,
// then the maxima.  A CTA sees thousands of rows; one that stays inside the bounds
// met so far -- nearly every row -- only reads them (one wavefront for all rows of
// a warp), and no lane keeps them in registers, which the gathers need.
template <typename T>
struct SharedExtremes {
    static constexpr int V = Store<T>::V;
    float *mm;

    // the values o of chunk number q of a row (chunk slot c of the lane), stored as v
    __device__ __forceinline__ void add(const SweepArgs &a, int c, int q, const float (&o)[V], const uint4 &v) {
#pragma unroll
        for (int e4 = 0; e4 < V / 4; ++e4) {
            const float4 lo = ldac(mm + q * V + 4 * e4), hi = ldac(mm + a.stride + q * V + 4 * e4);
            const float *oo = o + 4 * e4;
            if (oo[0] < lo.x || oo[1] < lo.y || oo[2] < lo.z || oo[3] < lo.w || oo[0] > hi.x || oo[1] > hi.y ||
                oo[2] > hi.z || oo[3] > hi.w) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    smem_min(mm + q * V + 4 * e4 + j, oo[j]);
                    smem_max(mm + a.stride + q * V + 4 * e4 + j, oo[j]);
                }
            }
        }
    }
};

// Batches: in registers, as the lane's 16-byte chunks are stored (two values to a
// word for the 16-bit formats: eight registers a chunk), merged over the lane groups
// when the warp moves to another graph.  A warp meets a graph for a few tasks only,
// in which most rows set new bounds: with a copy per warp in shared memory the
// conflicting atomics took 43% of the L1 pipe (64 Watts-Strogatz graphs of 2,000 to
// 20,000 vertices, BF16, R = 16: 78 -> 58 us a sweep in registers; 1,000 graphs of
// 1,000 vertices: 112 -> 77 us, FP32 122 -> 108 us).
template <typename T, int LPR, int CPL>
struct RegisterExtremes {
    using S = Store<T>;
    static constexpr int V = S::V;
    uint4 mn[CPL], mx[CPL];

    __device__ __forceinline__ static uint4 min4(const uint4 &x, const uint4 &y) {
        return make_uint4(S::min_word(x.x, y.x), S::min_word(x.y, y.y), S::min_word(x.z, y.z), S::min_word(x.w, y.w));
    }
    __device__ __forceinline__ static uint4 max4(const uint4 &x, const uint4 &y) {
        return make_uint4(S::max_word(x.x, y.x), S::max_word(x.y, y.y), S::max_word(x.z, y.z), S::max_word(x.w, y.w));
    }
    __device__ __forceinline__ static uint4 shfl_xor4(const uint4 &x, int o) {
        return make_uint4(__shfl_xor_sync(0xffffffffu, x.x, o), __shfl_xor_sync(0xffffffffu, x.y, o),
                          __shfl_xor_sync(0xffffffffu, x.z, o), __shfl_xor_sync(0xffffffffu, x.w, o));
    }
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            mn[c] = make_uint4(S::kMinInit, S::kMinInit, S::kMinInit, S::kMinInit);
            mx[c] = make_uint4(S::kMaxInit, S::kMaxInit, S::kMaxInit, S::kMaxInit);
        }
    }
    __device__ __forceinline__ void add(const SweepArgs &a, int c, int q, const float (&o)[V], const uint4 &v) {
        mn[c] = min4(mn[c], v);
        mx[c] = max4(mx[c], v);
    }
    // merge into the global slots of graph g; all 32 lanes
    __device__ __forceinline__ void flush(const SweepArgs &a, int g, int lane) {
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                mn[c] = min4(mn[c], shfl_xor4(mn[c], o));
                mx[c] = max4(mx[c], shfl_xor4(mx[c], o));
            }
        uint32_t *gmin = a.mm_min + (size_t)g * a.stride, *gmax = a.mm_max + (size_t)g * a.stride;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int q = lane + c * LPR;
            if (lane < LPR && q < a.nchunks) {
                float lo[V], hi[V];
                S::unpack(mn[c], lo);
                S::unpack(mx[c], hi);
#pragma unroll
                for (int e = 0; e < V; ++e)
                    if (lo[e] <= hi[e]) {   // (no row: not so)
                        atomicMin(gmin + q * V + e, f2ord(lo[e]));
                        atomicMax(gmax + q * V + e, f2ord(hi[e]));
                    }
            }
        }
    }
};

// in: the row is of the graph that x describes; otherwise its values go to the global slots
template <typename T, int LPR, int CPL, bool P, typename X>
__device__ __forceinline__ void row_epilogue(const SweepArgs &a, int64_t row, int gl, const uint4 (&own)[CPL],
                                             const float (&S)[CPL * Store<T>::V], const float *acg, X &x, bool in,
                                             uint32_t *gmin, uint32_t *gmax) {
    constexpr int V = Store<T>::V;
    uint4 *Y = reinterpret_cast<uint4 *>(a.x_out);
    const int64_t row_q = a.stride / V;
    const float dinv = __ldg(a.Dinv + row);
    const float om = a.omega, om1 = 1.f - a.omega;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const int q = gl + c * LPR;
        if (q < a.nchunks) {
            float y[V], o[V];
            Store<T>::unpack(own[c], y);
#pragma unroll
            for (int e4 = 0; e4 < V / 4; ++e4) {   // scale and centre of the row's graph
                const float4 av = ldac(acg + q * V + 4 * e4);
                const float4 cv = ldac(acg + a.stride + q * V + 4 * e4);
                const float A[4] = {av.x, av.y, av.z, av.w}, C[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int e = 4 * e4 + j;
                    const float z = fmaf(om1, y[e], om * (S[c * V + e] * dinv));
                    o[e] = Store<T>::round(A[j] * (z - C[j]));
                }
            }
            const uint4 v = Store<T>::pack(o);
            Y[row * row_q + q] = v;
            if (in) {
                x.add(a, c, q, o, v);
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    atomicMin(gmin + q * V + e, f2ord(o[e]));
                    atomicMax(gmax + q * V + e, f2ord(o[e]));
                }
            }
        }
    }
}

// Scale a = 1 / (max - min) of the previous sweep's stored values for the
// lane's elements (1 before the first sweep, 0 for a vector with max == min).
template <typename T, int LPR, int CPL, bool P = false>
__device__ __forceinline__ void load_scale(const uint32_t *pmin, const uint32_t *pmax, int gl,
                                           float (&A)[CPL * Store<T>::V]) {
    // pmin / pmax point at the slots of the row's graph (nullptr: no rescale yet)
    constexpr int V = Store<T>::V;
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const int r = (gl + c * LPR) * V + e;
            float av = 1.f;
            if (pmin) {   // FP32 on purpose: FP64 division runs on a very narrow pipe on this part
                const float lo = ord2f(P ? __ldcg(pmin + r) : pmin[r]), hi = ord2f(P ? __ldcg(pmax + r) : pmax[r]);
                av = hi > lo ? 1.f / (hi - lo) : 0.f;
            }
            A[c * V + e] = av;
        }
}

// Scale a = 1 / (max - min) of the previous sweep's stored values (1 before the
// first sweep, 0 for a vector with max == min) and centre c of the stored frame
// (the previous values of the graph's anchor vertex) of one graph, written to
// A[0 .. stride) and A[stride .. 2 stride).  One thread per 16-byte chunk.
template <typename T, bool P>
__device__ __forceinline__ void scale_center(const uint32_t *pmin, const uint32_t *pmax, const void *x_in, int32_t anchor,
                                             int32_t stride, float *A) {
    constexpr int V = Store<T>::V;
    const uint4 *xa = reinterpret_cast<const uint4 *>(x_in) + (int64_t)anchor * (stride / V);
    for (int q = threadIdx.x; q < stride / V; q += blockDim.x) {
        float f[V];
        Store<T>::unpack(ldx<P>(xa + q), f);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const int r = q * V + e;
            float av = 1.f;
            if (pmin) {   // FP32 on purpose: FP64 division runs on a very narrow pipe on this part
                const float lo = ord2f(P ? __ldcg(pmin + r) : pmin[r]), hi = ord2f(P ? __ldcg(pmax + r) : pmax[r]);
                av = hi > lo ? 1.f / (hi - lo) : 0.f;
            }
            A[r] = av;
            A[stride + r] = f[e];
        }
    }
}

// The same for every graph of a batch (block g), which the sweep then reads from
// one cached line per graph; a single graph's sweep computes its own in shared memory.
template <typename T>
__global__ void k_scale_center(const uint32_t *pmin, const uint32_t *pmax, const void *x_in, const int32_t *anchor,
                               int32_t stride, float *ac) {
    const size_t g = blockIdx.x;
    scale_center<T, false>(pmin ? pmin + g * stride : nullptr, pmax ? pmax + g * stride : nullptr, x_in, anchor[g], stride,
                           ac + g * 2 * stride);
}

// ----------------------------------------------------------------------------
// The graph a warp of a batch is in: its vertex range and min/max, which go to
// the global slots when the warp moves to another graph (tasks are ordered by
// vertex, so a warp meets few).  A row of yet another graph in the same warp (at
// the border of two graphs) goes to the global slots directly.
// ----------------------------------------------------------------------------
template <typename T, int LPR, int CPL>
struct WarpGraph {
    int g = -1;
    int32_t lo = 0, hi = 0;   // vertices of graph g
    RegisterExtremes<T, LPR, CPL> x;

    __device__ __forceinline__ void flush(const SweepArgs &a, int lane) {
        if (g >= 0) x.flush(a, g, lane);
    }
    // all 32 lanes; have: the lane has a row.  True: the row is in graph g.
    __device__ __forceinline__ bool enter(const SweepArgs &a, int lane, bool have, int32_t row) {
        if (__any_sync(0xffffffffu, have && !(row >= lo && row < hi))) {
            flush(a, lane);
            const int last = __reduce_max_sync(0xffffffffu, have ? row : -1);
            g = graph_of(a.voff, a.G, last);
            lo = (int32_t)__ldg(a.voff + g);
            hi = (int32_t)__ldg(a.voff + g + 1);
            x.reset();
        }
        return row >= lo && row < hi;
    }
};

// ----------------------------------------------------------------------------
// One JOR sweep (Alg. 1 inner loop) over all rows of degree > 0.
// ----------------------------------------------------------------------------
// Sum of the partial rows of one high-degree row (its chunks t0 .. t0 +
// nchunk - 1): group g adds partials g, g + G, ... in order, then the groups'
// sums are added (once per high-degree row).
template <typename T, int LPR, int CPL>
__device__ __forceinline__ void sum_partials(const SweepArgs &a, int64_t t0, int32_t nchunk, int grp, int gl, float (&S)[CPL * Store<T>::V]) {
    constexpr int V = Store<T>::V, E = CPL * V, G = 32 / LPR;
#pragma unroll
    for (int e = 0; e < E; ++e) S[e] = 0.f;
    for (int32_t cc2 = grp; cc2 < nchunk; cc2 += G) {
        const float4 *pp = reinterpret_cast<const float4 *>(a.part + (t0 + cc2) * (int64_t)a.stride);
#pragma unroll
        for (int cc = 0; cc < CPL; ++cc) {
            const int q = gl + cc * LPR;
            if (q < a.nchunks) {
#pragma unroll
                for (int e4 = 0; e4 < V / 4; ++e4) {
                    const float4 f = __ldcg(pp + (q * V) / 4 + e4);
                    S[cc * V + 4 * e4 + 0] += f.x;
                    S[cc * V + 4 * e4 + 1] += f.y;
                    S[cc * V + 4 * e4 + 2] += f.z;
                    S[cc * V + 4 * e4 + 3] += f.w;
                }
            }
        }
    }
    reduce_groups<LPR, E>(S);
}

// Registers against warps, one sweep of R-MAT 20, R = 32: FP32 with eight loads in
// flight at 3 / 4 CTAs per SM 343 / 303 us, with four at 4 / 5 CTAs 326 / 339 us;
// FP16 with four at 3 / 4 / 5 CTAs 314 / 275 / 264 us.
template <typename T>
constexpr int sweep_minb() { return sizeof(T) == 4 ? AD_SWEEP_MINB : AD_SWEEP_MINB16; }
// Row loads in flight per lane.  The 48 registers of the 16-bit formats hold four
// loads (16) beside the 16 sums of a lane; with eight the compiler spills up to ten
// times as much (a sweep of R-MAT 18: FP16, R = 256 475 -> 398 us with four, Q16,
// R = 40 186 -> 167 us).  Up to R = 32 a batch has four entries a lane either way.
template <typename T>
constexpr int sweep_loads() { return sizeof(T) == 4 ? AD_SWEEP_UB : AD_SWEEP_UB16; }

// The tasks of one sweep on this CTA, then the CTA's min/max to the sweep's
// slots.  P: inside the persistent launch.  B: a batch of graphs.  acs: scale and
// centre of a single graph in shared memory (batches read them from a.ac); mm:
// its min/max copy, initialised (batches have none).
template <typename T, int LPR, int CPL, bool P, bool B>
__device__ __forceinline__ void sweep_tasks(const SweepArgs &a, const float *acs, float *mm) {
    using L = Lane<T, LPR, CPL>;
    constexpr int V = L::V, E = L::E, G = L::G, RES = team_res<T, LPR, CPL>();
    constexpr int UB = sweep_loads<T>(), UBS = AD_SWEEP_UBS;
    using TM = Team<LPR, G, RES>;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, gl = lane % LPR;

    WarpGraph<T, LPR, CPL> wg;   // batches
    if (B) wg.x.reset();
    SharedExtremes<T> cta{mm};   // single graphs
    // epilogue of the lanes with a row (writer: the lane stores a part of it)
    auto finish = [&](int32_t row, bool have, bool writer, const uint4 (&own)[CPL], const float (&S)[E]) {
        if (B) {
            const bool in = wg.enter(a, lane, have, row);
            if (writer) {
                const int g = in ? wg.g : graph_of(a.voff, a.G, row);
                row_epilogue<T, LPR, CPL, P>(a, row, gl, own, S, a.ac + (size_t)g * 2 * a.stride, wg.x, in,
                                             a.mm_min + (size_t)g * a.stride, a.mm_max + (size_t)g * a.stride);
            }
        } else if (writer) {
            row_epilogue<T, LPR, CPL, P>(a, row, gl, own, S, acs, cta, true, nullptr, nullptr);
        }
    };

    const uint32_t n_big = (uint32_t)a.n_big, n_wide = (uint32_t)a.n_wide;
    const uint32_t team_tasks = ((uint32_t)a.n_medium - n_wide + TM::RPW - 1) / TM::RPW;
    const uint32_t n_tasks = n_big + n_wide + team_tasks + ((uint32_t)a.n_small_rows + G - 1) / G;
    const TaskIter it = task_iter(n_tasks, B ? 1 : 0);
    for (uint32_t task = it.t; task < it.t_end; task += it.step) {
        float S[E];
        if (task < n_big) {
            // ---- a chunk of a high-degree row; the last chunk combines
            const int32_t row = a.big_row[task];
            const int32_t c = a.big_chunk[task];
            const int64_t rb = a.rp[row], re = a.rp[row + 1];
            const int64_t p0 = rb + (int64_t)c * kChunk, p1 = min(re, p0 + kChunk);
            team_gather<T, LPR, CPL, G, 1, UB, P>(a, p0, (int)(p1 - p0), lane, S);
            float *part = a.part + task * (int64_t)a.stride;
            if (grp == 0) {
#pragma unroll
                for (int cc = 0; cc < CPL; ++cc) {
                    const int q = gl + cc * LPR;
                    if (q < a.nchunks) {
#pragma unroll
                        for (int e4 = 0; e4 < V / 4; ++e4)
                            __stcg(reinterpret_cast<float4 *>(part + q * V) + e4,
                                   make_float4(S[cc * V + 4 * e4], S[cc * V + 4 * e4 + 1], S[cc * V + 4 * e4 + 2],
                                               S[cc * V + 4 * e4 + 3]));
                    }
                }
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
                // group g sums partials g, g + G, ... (fixed order); then the groups' sums are added
                uint4 own[CPL];
                load_own<T, LPR, CPL, P>(a, row, gl, own);
                sum_partials<T, LPR, CPL>(a, t0, nchunk, grp, gl, S);
                finish(row, true, grp == 0, own, S);
                if (lane == 0) a.big_counter[t0] = 0u;
            }
        } else if (task < n_big + n_wide) {
            // ---- one row, whole warp
            const int32_t row = a.medium_row[task - n_big];
            uint4 own[CPL];
            load_own<T, LPR, CPL, P>(a, row, gl, own);
            const int64_t p0 = a.rp[row];
            team_gather<T, LPR, CPL, G, 1, UB, P>(a, p0, (int)(a.rp[row + 1] - p0), lane, S);
            finish(row, true, grp == 0, own, S);
        } else if (task < n_big + n_wide + team_tasks) {
            // ---- RPW rows of about the same degree, one per team
            const uint32_t mi = n_wide + (task - n_big - n_wide) * TM::RPW + lane / TM::TL;
            const bool have = mi < (uint32_t)a.n_medium;
            const int32_t row = have ? a.medium_row[mi] : 0;
            const int64_t p0 = have ? a.rp[row] : 0;
            const int d = have ? (int)(a.rp[row + 1] - p0) : 0;
            uint4 own[CPL];
            load_own<T, LPR, CPL, P>(a, row, gl, own);
            team_gather<T, LPR, CPL, G, RES, UB, P>(a, p0, d, lane, S);
            finish(row, have, have && lane % TM::TL < LPR, own, S);
        } else {
            // ---- G low-degree rows, one per lane group
            const uint32_t si = (task - n_big - n_wide - team_tasks) * G + grp;
            const bool have = si < (uint32_t)a.n_small_rows;
            const int32_t row = have ? a.small_row[si] : 0;
            const int64_t p0 = have ? a.rp[row] : 0;
            const int d = have ? (int)(a.rp[row + 1] - p0) : 0;
            uint4 own[CPL];
            load_own<T, LPR, CPL, P>(a, row, gl, own);
            team_gather<T, LPR, CPL, 1, 1, UBS, P>(a, p0, d, lane, S);
            finish(row, have, have, own, S);
        }
    }
    if (B) {
        wg.flush(a, lane);
        return;
    }
    __syncthreads();
    for (int r = threadIdx.x; r < a.nchunks * V; r += blockDim.x)
        if (mm[r] <= mm[a.stride + r]) {
            atomicMin(a.mm_min + r, f2ord(mm[r]));
            atomicMax(a.mm_max + r, f2ord(mm[a.stride + r]));
        }
}

// Shared memory of a sweep of a single graph: [2][stride] scale and centre, then
// [2][stride] min/max.  Batches use none.
__host__ __device__ constexpr size_t sweep_smem(int stride, bool batch) {
    return batch ? 0 : (size_t)4 * stride * sizeof(float);
}

__device__ __forceinline__ void reset_minmax(int32_t stride, float *mm) {
    for (int r = threadIdx.x; r < stride; r += blockDim.x) {
        mm[r] = INFINITY;
        mm[stride + r] = -INFINITY;
    }
}

template <typename T, int LPR, int CPL, bool B>
__global__ void __launch_bounds__(256, sweep_minb<T>()) k_sweep(SweepArgs a) {
    extern __shared__ __align__(16) float sm[];   // sweep_smem()
    float *mm = sm + 2 * a.stride;
    if (!B) {
        scale_center<T, false>(a.mm_prev_min, a.mm_prev_max, a.x_in, __ldg(a.anchor), a.stride, sm);
        reset_minmax(a.stride, mm);
        __syncthreads();
    }
    sweep_tasks<T, LPR, CPL, false, B>(a, sm, mm);
}

// ----------------------------------------------------------------------------
// Edge distance: for every upper entry (i, j > i) of the CSR, edge id e =
// eoff[i] + (p - upos[i]), rho_e = sqrt(sum_r a_r^2 (y_i^r - y_j^r)^2).
// A lane group handles one edge; its lanes hold different chunks of R.
// ----------------------------------------------------------------------------
// Sums of K values over the LPR lanes of a group, transposed: each exchange
// halves the values a lane holds, so K sums take about LPR shuffles in total
// instead of K * log2(LPR).  Afterwards lane gl holds in s[0 .. NH) the sums of
// values which .. which + NH - 1 (NH = max(1, K / LPR)); when LPR > K the lanes
// that differ only in their low bits hold the same sums.
template <int LPR, int K>
__device__ __forceinline__ void group_sums(float (&s)[K], int gl, unsigned gmask, int &which) {
    static_assert(K >= 1 && (K & (K - 1)) == 0, "the transposed sums halve K: K must be a power of two");
    which = 0;
#pragma unroll
    for (int o = LPR / 2, c = K; o >= 1; o >>= 1) {
        if (c > 1) {
            const bool upper = (gl & o) != 0;
#pragma unroll
            for (int i = 0; i < K / 2; ++i) {
                if (i < c / 2) {
                    const float send = upper ? s[i] : s[i + c / 2];
                    const float keep = upper ? s[i + c / 2] : s[i];
                    s[i] = keep + __shfl_xor_sync(gmask, send, o);
                }
            }
            if (upper) which += c / 2;
            c >>= 1;
        } else {
            s[0] += __shfl_xor_sync(gmask, s[0], o);
        }
    }
}

template <typename T, int LPR, int CPL, bool P>
__device__ __forceinline__ void edge_rows(const SweepArgs &a, int64_t row, int64_t p0, int64_t p1, int step,
                                          int first, int gl, unsigned gmask, const float (&A2)[CPL * Store<T>::V]) {
    constexpr int V = Store<T>::V, E = CPL * V;
    // edges of one group in flight: a power of two (group_sums halves it)
    constexpr int UB = AD_DIST_UB;
    const uint4 *X = reinterpret_cast<const uint4 *>(a.x_in);
    const int64_t row_q = a.stride / V;
    float yi[E];
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const int q = gl + c * LPR;
        if (q < a.nchunks) Store<T>::unpack(ldx<P>(X + row * row_q + q), yi + c * V);
        else {
#pragma unroll
            for (int e = 0; e < V; ++e) yi[c * V + e] = 0.f;
        }
    }
    const int64_t ebase = a.eoff[row] - a.upos[row];
    const double Di = a.normalize ? a.D[row] : 0.0;
    // the lanes of one group share p, so the group-masked reduction below is uniform
    for (int64_t pb = p0 + first; pb < p1; pb += (int64_t)step * UB) {
        int32_t jn[UB];
        uint4 v[UB][CPL];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int64_t p = pb + (int64_t)u * step;
            jn[u] = p < p1 ? ld_stream(a.col + p) : 0;
        }
#pragma unroll
        for (int u = 0; u < UB; ++u)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int q = gl + c * LPR;
                v[u][c] = (pb + (int64_t)u * step < p1 && q < a.nchunks) ? ldx<P>(X + (int64_t)jn[u] * row_q + q)
                                                                          : make_uint4(0, 0, 0, 0);
            }
        float s[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            s[u] = 0.f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                float yj[V];
                Store<T>::unpack(v[u][c], yj);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const float d = yi[c * V + e] - yj[e];
                    s[u] = fmaf(A2[c * V + e] * d, d, s[u]);
                }
            }
        }
        int which = 0;
        group_sums<LPR, UB>(s, gl, gmask, which);
        constexpr int NH = UB / LPR > 0 ? UB / LPR : 1;
        constexpr int WS = LPR > UB ? LPR / UB : 1;   // lanes per edge that hold the same sum
        const bool writer = gl % WS == 0;
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            int32_t jw = 0;
#pragma unroll
            for (int u = 0; u < UB; ++u) jw = (u == which + i) ? jn[u] : jw;
            const int64_t p = pb + (int64_t)(which + i) * step;
            if (writer && p < p1) {
                float rho = sqrtf(s[i]);
                if (a.normalize) rho = (float)((double)rho * sqrt(Di * a.D[jw]));
                a.rho[ebase + p] = rho;
            }
        }
    }
}

template <typename T, int LPR, int CPL, bool P>
__device__ __forceinline__ void distance_tasks(const SweepArgs &a) {
    using L = Lane<T, LPR, CPL>;
    constexpr int V = L::V, E = L::E, G = L::G;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, gl = lane % LPR;
    const unsigned gmask = LPR == 32 ? 0xffffffffu : (((1u << LPR) - 1u) << (grp * LPR));
    float A[E], A2[E];
    int cg = -1;
    // squared scale of the last rescale of graph g; padded vectors r >= R excluded
    auto enter = [&](int g) {
        if (g == cg) return;
        cg = g;
        load_scale<T, LPR, CPL, P>(a.mm_prev_min ? a.mm_prev_min + (size_t)g * a.stride : nullptr,
                                a.mm_prev_max ? a.mm_prev_max + (size_t)g * a.stride : nullptr, gl, A);
#pragma unroll
        for (int c = 0; c < CPL; ++c)
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int r = (gl + c * LPR) * V + e;
                A2[c * V + e] = (r < a.R) ? A[c * V + e] * A[c * V + e] : 0.f;
            }
    };
    GraphCache gcache;
    auto row_graph = [&](int64_t row) { return a.G > 1 ? gcache.of(a.voff, a.G, row) : 0; };
    const TaskIter it = task_iter((uint32_t)a.n_tasks, a.blocked);
    for (int64_t task = it.t; task < it.t_end; task += it.step) {
        if (task < a.n_big) {
            const int64_t row = a.big_row[task];
            const int32_t c = a.big_chunk[task];
            const int64_t ub = a.upos[row], ue = a.rp[row + 1];
            const int64_t p0 = ub + (int64_t)c * kChunk, p1 = min(ue, p0 + kChunk);
            enter(row_graph(row));
            edge_rows<T, LPR, CPL, P>(a, row, p0, p1, G, grp, gl, gmask, A2);
        } else if (task < a.n_big + a.n_medium) {
            const int64_t row = a.medium_row[task - a.n_big];
            enter(row_graph(row));
            edge_rows<T, LPR, CPL, P>(a, row, a.upos[row], a.rp[row + 1], G, grp, gl, gmask, A2);
        } else {
            const int64_t si = (task - a.n_big - a.n_medium) * G + grp;
            if (si < a.n_small_rows) {
                const int64_t row = a.small_row[si];
                enter(row_graph(row));
                edge_rows<T, LPR, CPL, P>(a, row, a.upos[row], a.rp[row + 1], 1, 0, gl, gmask, A2);
            }
        }
    }
}

template <typename T, int LPR, int CPL>
__global__ void __launch_bounds__(256, AD_DIST_MINB) k_distance(SweepArgs a) {
    distance_tasks<T, LPR, CPL, false>(a);
}

// ----------------------------------------------------------------------------
// Persistent relaxation: the whole of Alg. 1 for a single graph in one
// cooperative launch -- init, k sweeps, each followed by a grid-wide barrier
// (the next sweep's rescale needs every CTA's min/max), and the distances.
// The barrier is a counter that every CTA increments and then polls with an
// acquire load, at most kBarrierPolls times; a CTA that runs out writes
// AD_ERR_TIMEOUT to *err and returns, and the others stop at their next
// barrier once they see the error.
// ----------------------------------------------------------------------------
#ifndef AD_BARRIER_POLLS
#define AD_BARRIER_POLLS (1u << 25)   // with the 32 ns back-off and the loads: a few seconds
#endif

struct RelaxArgs {
    SweepArgs s;            // sweep plan and constant fields (x_in / x_out / slots set per sweep)
    SweepArgs d;            // distance plan
    int64_t n;              // vertices
    int32_t k;
    void *x0, *x1;
    uint32_t *mm_min, *mm_max;   // [k][stride]
    uint32_t seed_lo, seed_hi, stream_id;
    unsigned int *bar;      // [kBarrierSlots] arrival counters, zero before the launch
    int *err;               // zero before the launch
    unsigned int polls;     // barrier poll limit
    unsigned int extra;     // arrivals the barrier waits for beyond the grid (0; > 0 only to test the limit)
};

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add_u32(unsigned int *p, unsigned int v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// Arrivals are spread over kBarrierSlots counters (CTA b adds to slot b mod
// kBarrierSlots) so that they do not queue on one address; warp 0 of every
// CTA sums the slots with acquire loads until the total reaches the target.
constexpr int kBarrierSlots = 32;

// false: the barrier timed out here or elsewhere (every thread of the CTA gets the same answer)
__device__ __forceinline__ bool grid_barrier(const RelaxArgs &r, unsigned int phase) {
    __syncthreads();
    __shared__ int ok_s;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        if (lane == 0) red_release_add_u32(r.bar + (blockIdx.x % kBarrierSlots), 1u);
        const unsigned int target = (gridDim.x + r.extra) * phase;
        int ok = 1;
        unsigned int polls = 0;
        for (;;) {
            unsigned int v = ld_acquire_u32(r.bar + lane);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (v >= target) break;
            if (*(volatile int *)r.err != 0) { ok = 0; break; }
            if (++polls > r.polls) {
                if (lane == 0) atomicCAS(r.err, 0, (int)AD_ERR_TIMEOUT);
                ok = 0;
                break;
            }
            __nanosleep(32);
        }
        if (lane == 0) ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

template <typename T, int LPR, int CPL>
__global__ void __launch_bounds__(256, sweep_minb<T>()) k_relax(RelaxArgs r) {
    constexpr int V = Store<T>::V;
    extern __shared__ __align__(16) float sm[];   // sweep_smem()
    float *mm = sm + 2 * r.s.stride;
    // x0 <- rand(-0.5, 0.5) on every row of degree > 0
    init_rows<T>(r.s.rp, r.n, r.s.stride, r.seed_lo, r.seed_hi, r.stream_id, r.s.voff, 1, static_cast<T *>(r.x0));
    if (!grid_barrier(r, 1)) return;
    for (int32_t t = 0; t < r.k; ++t) {
        SweepArgs a = r.s;
        a.x_in = (t & 1) ? r.x1 : r.x0;
        a.x_out = (t & 1) ? r.x0 : r.x1;
        a.mm_prev_min = t > 0 ? r.mm_min + (size_t)(t - 1) * a.stride : nullptr;
        a.mm_prev_max = t > 0 ? r.mm_max + (size_t)(t - 1) * a.stride : nullptr;
        a.mm_min = r.mm_min + (size_t)t * a.stride;
        a.mm_max = r.mm_max + (size_t)t * a.stride;
        scale_center<T, true>(a.mm_prev_min, a.mm_prev_max, a.x_in, __ldg(a.anchor), a.stride, sm);
        reset_minmax(a.stride, mm);
        __syncthreads();
        sweep_tasks<T, LPR, CPL, true, false>(a, sm, mm);
        if (!grid_barrier(r, (unsigned int)t + 2)) return;
    }
    SweepArgs d = r.d;
    d.x_in = (r.k & 1) ? r.x1 : r.x0;
    d.mm_prev_min = r.k > 0 ? r.mm_min + (size_t)(r.k - 1) * d.stride : nullptr;
    d.mm_prev_max = r.k > 0 ? r.mm_max + (size_t)(r.k - 1) * d.stride : nullptr;
    distance_tasks<T, LPR, CPL, true>(d);
}

struct Config {
    int lpr, cpl, V, stride, nchunks;
    int per_sm = 0;   // sweep CTAs per SM (0: as many as fit)
};


template <typename T, int LPR, int CPL>
ad_status launch_sweep(ad_graph_t g, const SweepArgs &a, int blocks, size_t smem) {
    if (a.G > 1) {
        AD_LAUNCH(k_scale_center<T>, a.G, 32, 0, g->stream, a.mm_prev_min, a.mm_prev_max, a.x_in, a.anchor, a.stride,
                  a.ac);
        AD_LAUNCH((k_sweep<T, LPR, CPL, true>), blocks, 256, smem, g->stream, a);
    } else {
        AD_LAUNCH((k_sweep<T, LPR, CPL, false>), blocks, 256, smem, g->stream, a);
    }
    return AD_OK;
}
template <typename T, int LPR, int CPL>
ad_status launch_distance(ad_graph_t g, const SweepArgs &a, int blocks) {
    AD_LAUNCH((k_distance<T, LPR, CPL>), blocks, 256, 0, g->stream, a);
    return AD_OK;
}
template <typename T, int LPR, int CPL>
int blocks_for(bool sweep, bool batch, size_t smem) {
    int per_sm = 0;
    if (sweep && batch)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep<T, LPR, CPL, true>, 256, smem);
    else if (sweep)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep<T, LPR, CPL, false>, 256, smem);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_distance<T, LPR, CPL>, 256, 0);
    return per_sm > 0 ? per_sm : 1;
}

// f(lanes per row, chunks per lane) for a sweep or distance shape, as constants
template <typename F>
ad_status with_shape(const Config &cf, F f) {
    using std::integral_constant;
    switch (cf.lpr * 100 + cf.cpl) {
        case 101: return f(integral_constant<int, 1>{}, integral_constant<int, 1>{});
        case 201: return f(integral_constant<int, 2>{}, integral_constant<int, 1>{});
        case 401: return f(integral_constant<int, 4>{}, integral_constant<int, 1>{});
        case 801: return f(integral_constant<int, 8>{}, integral_constant<int, 1>{});
        case 1601: return f(integral_constant<int, 16>{}, integral_constant<int, 1>{});
        case 3201: return f(integral_constant<int, 32>{}, integral_constant<int, 1>{});
        case 3202: return f(integral_constant<int, 32>{}, integral_constant<int, 2>{});
        // fewer lanes per row, more chunks per lane: the alternative shapes the autotuner tries
        case 102: return f(integral_constant<int, 1>{}, integral_constant<int, 2>{});
        case 202: return f(integral_constant<int, 2>{}, integral_constant<int, 2>{});
        case 402: return f(integral_constant<int, 4>{}, integral_constant<int, 2>{});
        case 802: return f(integral_constant<int, 8>{}, integral_constant<int, 2>{});
        case 1602: return f(integral_constant<int, 16>{}, integral_constant<int, 2>{});
        default: return fail(AD_ERR_INVALID_ARG, "unsupported R / storage combination");
    }
}

template <typename T>
ad_status dispatch(ad_graph_t g, const Config &cf, bool sweep, const SweepArgs &a, int64_t n_tasks,
                          size_t smem) {
    // persistent grid: every SM full, but no more warps than tasks
    return with_shape(cf, [&](auto lpr_c, auto cpl_c) -> ad_status {
        constexpr int LPR = decltype(lpr_c)::value, CPL = decltype(cpl_c)::value;
        int per_sm = blocks_for<T, LPR, CPL>(sweep, a.G > 1, smem);
        if (sweep && cf.per_sm > 0 && cf.per_sm < per_sm) per_sm = cf.per_sm;
        int64_t blocks = (int64_t)per_sm * g->num_sms;
        const int64_t need = (n_tasks + 7) / 8;
        if (blocks > need) blocks = need > 0 ? need : 1;
        return sweep ? launch_sweep<T, LPR, CPL>(g, a, (int)blocks, smem)
                     : launch_distance<T, LPR, CPL>(g, a, (int)blocks);
    });
}

// CTAs of the sweep that fit on an SM
template <typename T>
ad_status sweep_ctas(const Config &cf, bool batch, int *per_sm) {
    return with_shape(cf, [&](auto lpr_c, auto cpl_c) -> ad_status {
        *per_sm = blocks_for<T, decltype(lpr_c)::value, decltype(cpl_c)::value>(true, batch, sweep_smem(cf.stride, batch));
        return AD_OK;
    });
}

// Persistent launch of k_relax: every CTA co-resident (cooperative launch),
// as many as fit or as the larger of the two plans can use.
template <typename T, int LPR, int CPL>
ad_status launch_relax(ad_graph_t g, const Config &cf, RelaxArgs &r) {
    const size_t smem = sweep_smem(r.s.stride, false);
    int per_sm = 0;
    AD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_relax<T, LPR, CPL>, 256, smem));
    if (per_sm < 1) return fail(AD_ERR_CUDA, "the persistent relaxation kernel does not fit on an SM");
    if (cf.per_sm > 0 && cf.per_sm < per_sm) per_sm = cf.per_sm;
    int64_t blocks = (int64_t)per_sm * g->num_sms;
    const int64_t need = (std::max(r.s.n_tasks, r.d.n_tasks) + 7) / 8;
    if (blocks > need) blocks = need > 0 ? need : 1;
    void *args[] = {&r};
    ::ad::g_launches.fetch_add(1, std::memory_order_relaxed);
    AD_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_relax<T, LPR, CPL>, dim3((unsigned)blocks), dim3(256), args,
                                            smem, g->stream));
    return AD_OK;
}

template <typename T>
ad_status relax_dispatch(ad_graph_t g, const Config &cf, RelaxArgs &r) {
    using std::integral_constant;
    auto run = [&](auto lpr_c, auto cpl_c) -> ad_status {
        return launch_relax<T, decltype(lpr_c)::value, decltype(cpl_c)::value>(g, cf, r);
    };
    switch (cf.lpr * 100 + cf.cpl) {
        case 101: return run(integral_constant<int, 1>{}, integral_constant<int, 1>{});
        case 201: return run(integral_constant<int, 2>{}, integral_constant<int, 1>{});
        case 401: return run(integral_constant<int, 4>{}, integral_constant<int, 1>{});
        case 801: return run(integral_constant<int, 8>{}, integral_constant<int, 1>{});
        case 1601: return run(integral_constant<int, 16>{}, integral_constant<int, 1>{});
        case 3201: return run(integral_constant<int, 32>{}, integral_constant<int, 1>{});
        case 3202: return run(integral_constant<int, 32>{}, integral_constant<int, 2>{});
        default: return fail(AD_ERR_INVALID_ARG, "the persistent relaxation takes the natural lane shapes only");
    }
}

// one instantiation per storage type, each in its own translation unit
ad_status dispatch_f32(ad_graph_t g, const Config &cf, bool sweep, const SweepArgs &a, int64_t n_tasks, size_t smem);
ad_status dispatch_bf16(ad_graph_t g, const Config &cf, bool sweep, const SweepArgs &a, int64_t n_tasks, size_t smem);
ad_status dispatch_f16(ad_graph_t g, const Config &cf, bool sweep, const SweepArgs &a, int64_t n_tasks, size_t smem);
ad_status dispatch_q16(ad_graph_t g, const Config &cf, bool sweep, const SweepArgs &a, int64_t n_tasks, size_t smem);
ad_status ctas_f32(const Config &cf, bool batch, int *per_sm);
ad_status ctas_bf16(const Config &cf, bool batch, int *per_sm);
ad_status ctas_f16(const Config &cf, bool batch, int *per_sm);
ad_status ctas_q16(const Config &cf, bool batch, int *per_sm);
ad_status relax_f32(ad_graph_t g, const Config &cf, RelaxArgs &r);
ad_status relax_bf16(ad_graph_t g, const Config &cf, RelaxArgs &r);
ad_status relax_f16(ad_graph_t g, const Config &cf, RelaxArgs &r);
ad_status relax_q16(ad_graph_t g, const Config &cf, RelaxArgs &r);
ad_status launch_init(ad_graph_t g, ad_storage storage, int blocks, int32_t stride, uint64_t seed, uint32_t stream_id,
                      void *x);

}  // namespace ad
