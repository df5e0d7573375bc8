// HOT iteration kernels for sm_103a (GB300).
//
// One iteration of Algorithm 2 (arXiv 2408.00598) on a batch of instances is
// three launches in FP32 bulk mode:
//   k_vec32   -- slab totals and cross-slab row sums of the state (inputs of
//                the marginals that Prop. 3 needs);
//   k_alpha32 -- Prop. 3: the right-hand side R of eq. (update:y) from the
//                slab sums, its closed-form solution y-bar, and the per-slab
//                broadcast vectors alpha/beta of A^T y-bar; elementwise over
//                the pieces, in chunks;
//   k_sweep   -- Steps 2-4 fused into one streaming pass over the flow state:
//                x-bar, z-bar = Pi_+(...), the Halpern update, and the slab
//                row/column sums of the new state (the A v products of the
//                next iteration); on check iterations also the KKT partial
//                sums of eq. (kkt_res).
// FP64 mode runs the same solve as k_vec, k_marg (instance-wide vectors, one
// CTA per instance) and k_alpha, in FP64.
// A block of K iterations ends with the KKT check, the restart rule, and the
// restart itself (new anchor), see launch_block_end.  Small instances run the
// same steps inside one kernel (hot_group.cu).
//
// FP32 bulk mode stores the anchor u (= v0 - sigma g0) and the delta d in FP32
// and forms every element from small quantities (see hot_internal.h):
// g - v/sigma = -(dA) - (u + d)/sigma with dA = A^T(y-bar - y0), and
// x-bar = u + d + sigma dA.  The reduced cost g = c - A^T y-bar itself (needed
// where z-bar = 0, i.e. on the support of the plan, where it tends to 0) is an
// unevaluated float pair: A^T y-bar is split per slab row/column into a hi
// part on the exact grid 2^-E of the scaled cost, so c - alpha_hi - beta_hi is
// exact in FP32, plus an FP32 lo part.  FP64 arithmetic runs at a small
// fraction of the FP32 rate on this part, so the per-iteration sums and the
// Prop. 3 solve use double-float pairs (two FP32 values, about 48 bits);
// FP64 is left to once-per-cycle work (restart, anchor sums).
#include "hot_internal.h"
#include "hot_block.cuh"

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

namespace hot {

// Stages of the FP32 sweep pipeline: each holds one pass of P rows
// (one float4 of u and one of the delta per thread).
constexpr int kStages = 4;
constexpr int kStageBytes = 2 * kThreads * 16;
// k_sweep32 dynamic shared memory: the pass ring, plus on check iterations
// the x-bar row partials, column partials and per-warp row pairs
constexpr int kSweepSmem = kStages * kStageBytes;
constexpr int kSweepSmemChk = kSweepSmem + (kRowSmemBytes + 256 * 4) + kThreads * 4 * 4 + (kThreads / 32) * kMaxTR * 8;

struct TileCtx {
    int inst, slab, band;
};

// Resolve tile t of the batch; returns false (block-uniform) if the instance
// is not running.
__device__ __forceinline__ bool resolve_tile(const WorkDev* __restrict__ W, int t, TileCtx& tc, int* s_tile) {
    if (threadIdx.x == 0) {
        const int i = find_inst(W->pre_tile, W->ninst, t);
        s_tile[0] = i;
        s_tile[1] = t - W->pre_tile[i];
        s_tile[2] = W->inst[i].ctl->status;
        s_tile[3] = W->inst[i].ctl->restart_pending;
    }
    __syncthreads();
    tc.inst = s_tile[0];
    g_tile_slab(W->inst[tc.inst], s_tile[1], tc.slab, tc.band);
    return true;
}

// Programmatic dependent launch: the kernels of the iteration chain are
// launched with programmatic stream serialisation, so the launch of a kernel
// is prepared while its predecessor runs.  Each one first waits for the
// predecessor grid to complete and its memory to be visible (everything
// below then sees stream order).  No kernel triggers its successor early:
// CTAs placed ahead of time and left waiting cost more than they saved.
__device__ __forceinline__ void pdl_enter() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// ----------------------------------------------------------------- k_vec --
// T1[j] = sum_k rowsum(f1 slab j)[k] (j < n), T2[k] = sum_j rowsum(f2 slab k)[j]
// (k < m), P1[k] = sum_j rowsum(f1 slab j)[k], P2[j] = sum_k rowsum(f2 slab k)[j];
// row sums are those of u + d (the slab sums of u are kept separately).  One
// warp per output; outputs at vecs[which * L + index], L = max(m, n).
__global__ void __launch_bounds__(kThreads) k_vec(const WorkDev* __restrict__ W) {
    pdl_enter();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ninst = W->ninst;
    const int nitems = W->pre_vec[ninst];
    for (int base = blockIdx.x * (kThreads / 32); base < nitems; base += gridDim.x * (kThreads / 32)) {
        const int item = base + warp;
        if (item >= nitems) continue;
        const int i = find_inst(W->pre_vec, ninst, item);
        const HotInst& I = W->inst[i];
        if (I.ctl->status != ST_RUNNING) continue;
        const int m = I.m, n = I.n, L = g_L(I);
        int q = item - W->pre_vec[i];
        int which;
        if (q < n) which = 0;
        else if ((q -= n) < m) which = 1;
        else if ((q -= m) < m) which = 2;
        else {
            q -= m;
            which = 3;
        }
        const double* __restrict__ rs = I.rs;
        const double* __restrict__ rs0 = I.rs0;
        const size_t f2 = (size_t)n * m;               // first row of the f2 half
        double acc = 0.0;
        if (which == 0) {                              // T1[j]: f1 slab j, its m rows
            for (int t = lane; t < m; t += 32) acc += rs[(size_t)q * m + t] + rs0[(size_t)q * m + t];
        } else if (which == 1) {                       // T2[k]: f2 slab k, its n rows
            for (int t = lane; t < n; t += 32) acc += rs[f2 + (size_t)q * n + t] + rs0[f2 + (size_t)q * n + t];
        } else if (which == 2) {                       // P1[k]: row k of every f1 slab
            for (int t = lane; t < n; t += 32) acc += rs[(size_t)t * m + q] + rs0[(size_t)t * m + q];
        } else {                                       // P2[j]: row j of every f2 slab
            for (int t = lane; t < m; t += 32) acc += rs[f2 + (size_t)t * n + q] + rs0[f2 + (size_t)t * n + q];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) I.vecs[which * L + q] = acc;
    }
}

__global__ void __launch_bounds__(kThreads) k_marg(const WorkDev* __restrict__ W) {
    pdl_enter();
    extern __shared__ double sv[];                   // 7 L: T1 T2 P1 P2 colmu1 rowmu2, then s
    __shared__ double s_red[4 * 32];
    const int ninst = W->ninst;
    for (int inst = blockIdx.x; inst < ninst; inst += gridDim.x) {
        const HotInst& I = W->inst[inst];
        if (I.grp || I.ctl->status != ST_RUNNING) continue;     // block-uniform
        const int L = g_L(I);
        for (int q = threadIdx.x; q < 4 * L; q += blockDim.x) sv[q] = I.vecs[q];
        marg64(I, recip64(I.m, I.n, I.ctl->sigma), I.cs_part, I.mvec, sv, s_red);
        __syncthreads();
    }
}

// Per-slab entries of dy = A^T-pieces of y-bar - y0.  The anchor part of R
// (row sums and column totals of u) is precomputed once per cycle by
// k_anchor; here only the delta's sums enter.
template <bool CHECK>
__global__ void __launch_bounds__(kThreads) k_alpha(const WorkDev* __restrict__ W) {
    pdl_enter();
    __shared__ double s_red[4 * 32];
    __shared__ float s_max[32];
    __shared__ int s_t[4];
    const int ninst = W->ninst;
    const int nslab = W->pre_slab[ninst];
    for (int t = blockIdx.x; t < nslab; t += gridDim.x) {
        if (threadIdx.x == 0) {
            const int i = find_inst(W->pre_slab, ninst, t);
            s_t[0] = i;
            s_t[1] = t - W->pre_slab[i];
            s_t[2] = W->inst[i].ctl->status;
        }
        __syncthreads();
        if (s_t[2] != ST_RUNNING) {
            __syncthreads();
            continue;
        }
        const HotInst& I = W->inst[s_t[0]];
        const int slab = s_t[1], Ls = g_side(I, slab);
        const size_t o = 2 * g_row(I, slab);
        pieces64<CHECK>(I, recip64(I.m, I.n, I.ctl->sigma), slab, 0, Ls, true, I.rs, I.cs_part, I.mvec, I.ab64 + o, I.dab64 + o, s_red, s_max);
        __syncthreads();
    }
}

// ------------------------------------------------------- k_vec32/k_alpha32 --
// FP32 bulk mode.  The same Prop. 3 solve as k_vec/k_marg/k_alpha, with the
// per-iteration arithmetic on double-float pairs: FP64 throughput on this
// part is a small fraction of FP32, and pairs carry about 48 bits, far more
// than the FP32 row and column partial sums they combine.
//
// k_vec32: T1, T2, P1, P2 of u + d.  A work item is one CTA: for T1/T2 (sums
// along contiguous rows) 8 outputs, one warp each; for P1/P2 (sums down the
// columns of the row-sum matrices) 32 columns x kVecRows rows, one column per
// lane and kVecRows / 8 rows per warp, combined in a fixed order into one
// partial per row block (k_alpha32 adds the partials).  Every lane issues
// its loads before it adds, so an item costs about one L2 round trip.
// SINGLE (a batch of one instance): the CTA that finishes the instance's last
// item also forms its Prop. 3 stage (k_stage32's work), which saves a kernel
// on the single-instance path; batches of many instances launch k_stage32,
// since there every item would pay the count's atomic and barriers.
template <bool SINGLE>
__global__ void __launch_bounds__(kThreads) k_vec32(const WorkDev* __restrict__ W, int j) {
    pdl_enter();
    constexpr int kW = kThreads / 32;
    constexpr int kRW = kVecRows / kW;               // rows per warp in a P item
    __shared__ float2 s_p[kThreads];
    __shared__ float2 s_red[SINGLE ? 2 * 32 : 1];
    __shared__ int s_t[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ninst = W->ninst;
    const int nitems = W->pre_vec[ninst];
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        if (threadIdx.x == 0) {
            const int i = find_inst(W->pre_vec, ninst, it);
            s_t[0] = i;
            s_t[1] = it - W->pre_vec[i];
            s_t[2] = W->inst[i].ctl->status;
        }
        __syncthreads();
        if (s_t[2] == ST_RUNNING) {
            const HotInst I = W->inst[s_t[0]];
            const int m = I.m, n = I.n, L = g_L(I);
            const int t1 = (n + 7) / 8, t2 = (m + 7) / 8;
            const int c1 = (m + 31) / 32, r1 = (n + kVecRows - 1) / kVecRows;   // P1: columns k, rows j
            const int c2 = (n + 31) / 32, r2 = (m + kVecRows - 1) / kVecRows;   // P2: columns j, rows k
            const size_t f2 = (size_t)n * m;                 // first row of the f2 half
            int item = s_t[1];
            const float2* __restrict__ rs = I.rs2;           // row sums of u + d
            if (item < t1 + t2) {
                // T1[j]: the m rows of f1 slab j; T2[k]: the n rows of f2 slab k
                const int which = item < t1 ? 0 : 1;
                const int q = (which ? item - t1 : item) * 8 + warp;
                const int cnt = which ? m : n, len = which ? n : m;
                if (q < cnt) {                                // warp-uniform
                    const float2* row = rs + (which ? f2 + (size_t)q * n : (size_t)q * m);
                    DF acc{0.f, 0.f};
                    for (int t0 = 0; t0 < len; t0 += 8 * 32) {
                        float2 v[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int t = t0 + u * 32 + lane;
                            v[u] = t < len ? row[t] : make_float2(0.f, 0.f);
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u) acc = df_add(acc, df_ld(v[u]));
                    }
                    acc = warp_sum_df(acc);
                    if (lane == 0) I.vec2[which * L + q] = df_st(acc);
                    if (lane == 0) s_p[warp] = df_st(acc);
                } else if (lane == 0) {
                    s_p[warp] = make_float2(0.f, 0.f);
                }
                // the item's total, for the half totals F1, F2 of the stage
                __syncthreads();
                if (threadIdx.x == 0) {
                    DF tot = df_ld(s_p[0]);
                    for (int w = 1; w < kW; ++w) tot = df_add(tot, df_ld(s_p[w]));
                    I.vec2[(size_t)(2 + r1 + r2) * L + item] = df_st(tot);
                }
            } else {
                item -= t1 + t2;
                // P1[k] = sum_j rs(f1 slab j)[k]; P2[j] = sum_k rs(f2 slab k)[j]:
                // 32 columns x kVecRows rows per item, one partial per row block
                const int which = item < c1 * r1 ? 0 : 1;
                if (which) item -= c1 * r1;
                const int ncol = which ? n : m, nrow = which ? m : n, nc = which ? c2 : c1;
                const int part = item / nc;
                const int q = (item - part * nc) * 32 + lane;
                const int t0 = part * kVecRows + warp * kRW;
                float2 v[kRW];
#pragma unroll
                for (int u = 0; u < kRW; ++u) {
                    const int t = t0 + u;
                    const size_t idx = which ? f2 + (size_t)t * n + q : (size_t)t * m + q;
                    v[u] = (q < ncol && t < nrow) ? rs[idx] : make_float2(0.f, 0.f);
                }
                DF acc{0.f, 0.f};
#pragma unroll
                for (int u = 0; u < kRW; ++u) acc = df_add(acc, df_ld(v[u]));
                s_p[threadIdx.x] = df_st(acc);
                __syncthreads();
                if (warp == 0 && q < ncol) {
                    DF tot = df_ld(s_p[lane]);
                    for (int w = 1; w < kW; ++w) tot = df_add(tot, df_ld(s_p[w * 32 + lane]));
                    I.vec2[(size_t)(2 + (which ? r1 : 0) + part) * L + q] = df_st(tot);
                }
            }
            if constexpr (SINGLE) {
                // The barrier orders this CTA's writes of the item before thread
                // 0's fence, which makes them visible device-wide before the
                // count (the pattern of a grid-wide barrier); the last CTA reads
                // the others' through L2 (__ldcg in stage_in).
                __syncthreads();
                if (threadIdx.x == 0) {
                    __threadfence();
                    const unsigned int done = atomicAdd(I.vcount, 1u) + 1u;
                    s_t[3] = done == (unsigned int)vec32_items_dev(m, n);
                    if (s_t[3]) __threadfence();
                }
                __syncthreads();
                if (s_t[3]) {
                    alpha32_stage(I, I.stg2, s_red);
                    if (threadIdx.x == 0) {
                        *I.vcount = 0u;                           // for the next launch
                        *I.p32 = make_p32(I.ctl->sigma, I.ctl->k + j, I.h, I.gadmm, I.relax);
                    }
                }
            }
        }
        __syncthreads();
    }
}

// k_stage32: the instance-wide Prop. 3 stage (alpha32_stage) from k_vec32's
// sums, one CTA per instance, and the element constants of the iteration.
// (A kernel of its own: forming it in the CTA that finishes an instance's
// last k_vec32 item cost every item an atomic and a barrier, which batches of
// many small instances paid many times over.)
__global__ void __launch_bounds__(kThreads) k_stage32(const WorkDev* __restrict__ W, int j) {
    pdl_enter();
    __shared__ float2 s_red[2 * 32];
    const int ninst = W->ninst;
    for (int i = blockIdx.x; i < ninst; i += gridDim.x) {
        const HotInst I = W->inst[i];
        if (I.grp || I.ctl->status != ST_RUNNING) continue;   // block-uniform
        alpha32_stage(I, I.stg2, s_red);
        if (threadIdx.x == 0) *I.p32 = make_p32(I.ctl->sigma, I.ctl->k + j, I.h, I.gadmm, I.relax);
        __syncthreads();
    }
}

// k_alpha32: the pieces of y-bar - y0 (pairs, kept for the restart), their
// FP32 split for the sweep, and on check iterations the partial sums of
// <b, y>, of <c, A^T(y-bar - y0)> and max |A^T y|.  An instance's 4mn pieces
// are cut into chunks of kAlphaChunk (kAPT per thread, consecutive threads on
// consecutive pieces); a CTA takes chunks in a grid-stride loop and loads the
// inputs of all its pieces of a chunk before it computes any.  The
// instance-wide O(m + n) stage of Prop. 3 comes from k_stage32 (stg2), so a
// piece is a few loads and double-float operations.  The descriptor is copied
// into registers: the stores below cannot then force reloads of its fields.
// Per-chunk partial sums sit at the chunk's index (dobj_part, cD_part;
// k_check adds them in order).
template <bool CHECK>
__global__ void __launch_bounds__(kThreads, 2) k_alpha32(const WorkDev* __restrict__ W, int j) {
    pdl_enter();
    __shared__ float2 s_red[2 * 32];
    __shared__ float s_max[32];
    const int ninst = W->ninst;
    const int nchunk = W->pre_achunk[ninst];
    const int tid = threadIdx.x;
    for (int c = blockIdx.x; c < nchunk; c += gridDim.x) {
        // every thread resolves the chunk itself (uniform, no barrier)
        const int inst = find_inst(W->pre_achunk, ninst, c);
        const HotInst I = W->inst[inst];
        const int m = I.m, n = I.n;
        const int cl = c - W->pre_achunk[inst];
        const int npieces = 4 * m * n;
        // every input is loaded before the status is known (the instance's
        // memory is valid either way), so the chunk costs one round trip less
        int ps[kAPT], pi[kAPT];
        PieceIn pin[kAPT];
#pragma unroll
        for (int u = 0; u < kAPT; ++u) {
            const int q = cl * kAlphaChunk + u * kThreads + tid;
            ps[u] = -1;
            if (q < npieces) {
                piece_slab(I, q, ps[u], pi[u]);
                pin[u] = piece_in(I, ps[u], pi[u], CHECK);
            }
        }
        const PieceK K = piece_consts(I, *I.cyc);
        if (I.ctl->status != ST_RUNNING) continue;
        float2* __restrict__ dab2 = I.dab2;
        float4* __restrict__ ab32 = I.ab32;
        float ymax = 0.f;
        DF dob{0.f, 0.f};
        // <c, A^T(y-bar - y0)>: the cost is separable, so a slab contributes
        // sum_r dalpha_r C(r) + sum_c dbeta_c C(c), C(x) = sum_y (X_x - X_y)^2
        DF cdd{0.f, 0.f};
#pragma unroll
        for (int u = 0; u < kAPT; ++u) {
            if (ps[u] < 0) continue;
            const int slab = ps[u], idx = pi[u];
            const int Ls = slab < n ? m : n;
            const PieceIn& a = pin[u];
            bool zero;
            const DF dv = piece_dv(I, K, slab, idx, a, zero);
            const bool col = idx >= Ls;
            const size_t o = 2 * g_row(I, slab) + idx;
            if (CHECK) dab2[o] = df_st(dv);          // read at the block's end only
            ab32[o] = piece_pack(a, dv, K, I.coord_real);
            if (CHECK) {
                const DF full = df_add(DF{a.a0.x, a.a0.y}, dv);
                ymax = fmaxf(ymax, fabsf(full.hi));
                const float2* csum = I.csum2 + g_xbase(I, slab);
                cdd = df_add(cdd, df_mul(dv, df_ld(csum[col ? idx - Ls : idx])));
                if (col && !zero) dob = df_add(dob, df_mul(df_ld(a.mu), full));
            }
        }
        if (CHECK) {
            DF red[2] = {dob, cdd};
            block_sum_df<2>(red, s_red);
            const float bm = block_max(ymax, s_max);
            if (tid == 0) {
                reinterpret_cast<float2*>(I.dobj_part)[cl] = df_st(red[0]);
                reinterpret_cast<float2*>(I.cD_part)[cl] = df_st(red[1]);
                atomicMax(&I.ctl->ymax_bits, __float_as_uint(bm));
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_anchor(const WorkDev* __restrict__ W) {
    pdl_enter();
    __shared__ int s_t[4];
    const int ninst = W->ninst;
    const int nslab = W->pre_slab[ninst];
    int any = 0;
    for (int i = threadIdx.x; i < ninst; i += blockDim.x) {
        const HotCtl* C = W->inst[i].ctl;
        any |= (!W->inst[i].grp && C->status == ST_RUNNING && C->restart_pending != 0);
    }
    if (!__syncthreads_or(any)) return;
    for (int t = blockIdx.x; t < nslab; t += gridDim.x) {
        if (threadIdx.x == 0) {
            const int i = find_inst(W->pre_slab, ninst, t);
            s_t[0] = i;
            s_t[1] = t - W->pre_slab[i];
            s_t[2] = (W->inst[i].ctl->status == ST_RUNNING) && W->inst[i].ctl->restart_pending;
        }
        __syncthreads();
        if (s_t[2]) anchor_slab(W->inst[s_t[0]], s_t[1], W->inst[s_t[0]].ctl->sigma);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kThreads) k_anchor_one(HotInst I, double sigma) {
    for (int slab = blockIdx.x; slab < g_nslab(I); slab += gridDim.x) anchor_slab(I, slab, sigma);
}

// --------------------------------------------------------------- k_sweep --
// FP64 mode: Steps 2-4 of Algorithm 2, tiles in a grid-stride loop
// (sweep64_tile, hot_block.cuh).
template <bool CHECK>
__global__ void __launch_bounds__(kThreads, 2) k_sweep64(const WorkDev* __restrict__ W, int j) {
    pdl_enter();
    __shared__ Sweep64Smem sm;
    __shared__ int s_tile[4];
    __shared__ P64 s_p64;
    const int ninst = W->ninst;
    const int ntiles = W->pre_tile[ninst];
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        TileCtx tc;
        resolve_tile(W, t, tc, s_tile);
        if (s_tile[2] != ST_RUNNING) {
            __syncthreads();
            continue;
        }
        const HotInst& I = W->inst[tc.inst];
        if (threadIdx.x == 0) s_p64 = make_p64(I.ctl->sigma, I.ctl->k + j, I.h, I.gadmm, I.relax);
        __syncthreads();
        const size_t o = 2 * g_row(I, tc.slab);
        sweep64_tile<CHECK>(I, tc.slab, tc.band, (const double*)((j & 1) ? I.d1 : I.d0),
                            (double*)((j & 1) ? I.d0 : I.d1), s_p64, I.ab64 + o, I.dab64 + o, I.rs, I.cs_part, sm);
        __syncthreads();
    }
}

// -------------------------------------------------------------- k_sweep32 --
// FP32 bulk mode: Steps 2-4 of Algorithm 2 as one streaming pass over the
// flow state.  A CTA takes the tiles blockIdx.x, blockIdx.x + G, ... (TR rows
// of one slab each) and streams their passes (P rows: every thread one float4
// of u and one of the delta) through a kStages-deep cp.async ring that is not
// drained between tiles, so the next tile's loads are in flight while the
// current tile's row and column sums are reduced.  The rows' alpha pieces
// travel in the group of each tile's first pass into a ring of their own, and
// the first threads leave each tile's descriptor (128 bytes) in a third ring for the
// compute side.
//
// The scaled cost is separable, h (x_r - x_c)^2 = h x_r^2 + h x_c^2 - 2 h x_r x_c
// (x the bin coordinates of the slab's half, integers in FP32 mode), so the
// grid part of the reduced cost is Gh = (A_r + B_c) - 2 h x_r x_c with
// A_r = h x_r^2 - alpha_hi (per row) and B_c = h x_c^2 - beta_hi (per column):
// every term is an integer multiple of 2^-E, so Gh is exact in FP32.  The
// coordinates travel in the w component of the alpha/beta pieces (k_alpha32),
// so the sweep reads no coordinate array.  A tile's offsets in the per-slab
// arrays are resolved once, by the issue side, into its descriptor.
// Zeros in place of a tile's delta: a tile spans TR * pitch <= kMaxTileElems
// floats (checked when the instance is created); zero-initialised at module load.
__device__ __align__(16) float g_zero_tile[kMaxTileElems];

__global__ void __launch_bounds__(kThreads) k_tile_table(const WorkDev* __restrict__ W, int ntiles) {
    const int t = blockIdx.x * kThreads + threadIdx.x;
    if (t >= ntiles) return;
    SweepTile d{};
    const int i = find_inst(W->pre_tile, W->ninst, t);
    const HotInst& I = W->inst[i];
    d.inst = i;
    g_tile_slab(I, t - W->pre_tile[i], d.slab, d.band);
    d.S = g_side(I, d.slab);
    const int pitch = g_pitch(I, d.slab);
    d.NC = pitch / 4;
    d.P = kThreads / d.NC;
    d.r0 = d.band * I.TR;
    d.r1 = min(d.S, d.r0 + I.TR);
    d.npass = (d.r1 - d.r0 + d.P - 1) / d.P;
    d.row = (int)g_row(I, d.slab);
    d.tile = g_tile(I, d.slab, d.band);
    d.colp = (int)g_colp(I, d.slab, d.band);
    d.elem = (long long)g_elem(I, d.slab);
    d.ctl = I.ctl;
    const size_t first = (size_t)d.elem + (size_t)d.r0 * pitch;
    d.u = (const float*)I.u + first;
    d.d0 = (const float*)I.d0 + first;
    d.d1 = (const float*)I.d1 + first;
    d.ab = I.ab32 + 2 * (size_t)d.row + d.r0;
    d.p32 = I.p32;
    W->tiles[t] = d;
}

// PAD: some slab side of the batch is not a multiple of 4, so a thread's
// last column group may reach into the pad columns, which are masked (a
// variant of its own: the masks cost the unpadded sweep registers).
// FIRST (the first iteration of a block, never a check): a tile whose delta
// is known to be zero copies it from the zero tile (a variant of its own, so
// the other iterations' sweep carries none of it).
template <bool CHECK, bool PAD, bool FIRST = false>
__global__ void __launch_bounds__(kThreads, CHECK ? 2 : 3) k_sweep32(const WorkDev* __restrict__ W, int j) {
    pdl_enter();
    constexpr int NV = 4;
    constexpr int kW = kThreads / 32;
    constexpr int kRowN = kRowSmemBytes / sizeof(float) + 256;
    __shared__ __align__(16) float s_row[kRowN];
    __shared__ __align__(16) float s_col[kThreads * NV];
    __shared__ __align__(16) float4 s_alpha[kStages][kMaxTR];
    __shared__ __align__(16) float2 s_rdf[kW][kMaxTR];            // per-warp row partial pairs
    // descriptors of the tiles in flight: the issue side starts tiles up to kStages
    // ahead of the one being computed, so twice as many slots are never reused early
    __shared__ SweepTile s_td[2 * kStages];
    __shared__ float2 s_red[kNK * 32];
    // dynamic: the pass ring [kStages][2][kThreads] float4, then (check
    // iterations) the x-bar row and column partials
    extern __shared__ float4 s_stage[];
    float* s_xrow = reinterpret_cast<float*>(s_stage + kStages * 2 * kThreads);
    float* s_xcol = s_xrow + kRowN;
    float2 (*s_xdf)[kMaxTR] = reinterpret_cast<float2 (*)[kMaxTR]>(s_xcol + kThreads * NV);
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x;
    const int ntiles = W->pre_tile[W->ninst];

    // ---- issue side: every thread walks the same tile sequence
    struct Cur {
        const float* u;            // this thread's source of the next pass (u)
        const float* d;            // and of the delta
        const float4* a;           // alpha piece of this thread's row of the tile (tid < tile rows)
        int step;                  // P rows, in floats
        int mine;                  // passes of the tile left in which this thread copies a row
        int left, it, ik;          // passes left, tile, tiles started
        bool acopy;                // the next pass is the tile's first and this thread copies an alpha piece
    } c;
    // a state larger than L2: odd iterations take the tiles in reverse order,
    // so a sweep starts on the tiles whose state the previous sweep touched
    // last (still in L2)
    const bool rev = (j & 1) && W->alternate;
    auto at = [&](int t) { return W->tiles + (rev ? ntiles - 1 - t : t); };
    auto set_tile = [&](int t) {
        // tiles of an instance that is not running are passed over
        while (t < ntiles && at(t)->ctl->status != ST_RUNNING) t += G;
        c.it = t;
        if (t < ntiles) {
            const SweepTile* d = at(t);
            // the next tile's descriptor on its way into L1
            if (t + G < ntiles) asm volatile("prefetch.global.L1 [%0];\n" ::"l"(at(t + G)));
            const int NC = d->NC, P = d->P;
            const int ro = tid / NC, cg = tid - ro * NC;
            const int sp = PAD ? (d->S + 3) & ~3 : d->S;   // row pitch (without padded slabs, the side)
            const int base = ro * sp + cg * NV;
            const bool dz = FIRST && d->ctl->dzero;
            c.u = d->u + base;
            // a delta known to be zero (first iteration after an FP32 restart,
            // which stores none) is copied from a zero tile: L2 hits, no HBM read
            c.d = dz ? g_zero_tile + base : ((j & 1) ? d->d1 : d->d0) + base;
            const int nr = d->r1 - d->r0;
            c.a = d->ab + tid;
            c.step = P * sp;
            // rows ro, ro + P, ... below nr (threads past P rows copy nothing)
            c.mine = ro < P && ro < nr ? (nr - ro + P - 1) / P : 0;
            c.left = d->npass;
            c.acopy = tid < nr;
            if (tid < (int)(sizeof(SweepTile) / 16))
                reinterpret_cast<float4*>(&s_td[c.ik % (2 * kStages)])[tid] = reinterpret_cast<const float4*>(d)[tid];
        }
    };
    c.ik = 0;
    unsigned long long pol_ef;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(pol_ef));
    set_tile(blockIdx.x);
    // one commit group per call: the copies of global pass n (ring slot n % kStages)
    auto issue = [&](int n) {
        if (c.it < ntiles) {
            if (c.mine > 0) {
                float4* su = s_stage + (size_t)(n % kStages) * 2 * kThreads + tid;
                cp_async16_ef(su, c.u, pol_ef);
                cp_async16_ef(su + kThreads, c.d, pol_ef);
                --c.mine;
            }
            if (c.acopy) {
                cp_async16(&s_alpha[c.ik % kStages][tid], c.a);
                c.acopy = false;
            }
            c.u += c.step;
            c.d += c.step;
            if (--c.left == 0) {
                ++c.ik;
                set_tile(c.it + G);
            }
        }
        cp_async_commit();
    };
#pragma unroll 1
    for (int q = 0; q < kStages - 1; ++q) issue(q);

    // ---- compute side
    // per column of this thread: B_c = h x_c^2 - beta_hi (exact), beta_lo,
    // dbeta, x_c; loaded for the next tile during the current tile's epilogue
    float4 bq[NV];
    P32 p;
    auto load_cols = [&](const SweepTile& d) {
        const int ro = tid / d.NC, c0 = (tid - ro * d.NC) * NV;
        p = *d.p32;
        const float4* ab = d.ab - d.r0 + d.S;
#pragma unroll
        for (int e = 0; e < NV; ++e)
            bq[e] = ro < d.P && (!PAD || c0 + e < d.S) ? ab[c0 + e] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    bool have = false;                           // bq, p hold the current tile's values
    int n = 0;                                   // global index of the next pass to compute
    for (int ck = 0;; ++ck) {
        // the tile's alpha pieces and its descriptor: group n (its first pass)
        // and the first threads' store, both complete before this barrier
        cp_async_wait<kStages - 2>();
        __syncthreads();
        // the issue side has started every tile this CTA still has (it runs ahead)
        if (c.it >= ntiles && ck >= c.ik) break;
        const SweepTile& dc = s_td[ck % (2 * kStages)];
        if (!have) load_cols(dc);
        const HotInst& I = W->inst[dc.inst];
        const int S = dc.S, Sp = PAD ? (dc.S + 3) & ~3 : dc.S, NC = dc.NC, P = dc.P;
        const int r0 = dc.r0, nr = dc.r1 - dc.r0;
        const int ro = tid / NC, cg = tid - ro * NC;
        const bool active = ro < P;
        const int c0 = cg * NV;
        const int nval = PAD ? S - c0 : NV;       // columns of this thread's group inside the slab (pad after)
        const int cr = PAD ? I.coord_real : 0;    // real-valued coordinates (general variant only)
        const float h = p.h;
        if (!cr) {
#pragma unroll
            for (int e = 0; e < NV; ++e) {
                const float cf = bq[e].w;                      // column coordinate x_c
                bq[e] = make_float4(fmaf(cf * cf, h, -bq[e].x), bq[e].y, bq[e].z, cf);
            }
        }
        const float4* sa = s_alpha[ck % kStages];
        float* __restrict__ dout = (float*)((j & 1) ? I.d0 : I.d1) + dc.elem + ((size_t)r0 + ro) * Sp + c0;
        const int ostep = P * Sp;
        float* srow = s_row + ro * (NC + 1) + cg;
        float* sxrow = s_xrow + (CHECK ? ro * (NC + 1) + cg : 0);
        const int rstep = P * (NC + 1);
        float cacc[NV], xacc[NV];
#pragma unroll
        for (int e = 0; e < NV; ++e) cacc[e] = xacc[e] = 0.f;
        // KKT partials: FP32 chains of at most 64 terms per thread and tile
        // (a tile has TR * S / 1024 <= 16 passes), summed over the CTA in pairs.
        // The objective's share <c, d> is not formed here: it only reports the
        // value, so the pass that ends an instance forms it once (MODE 2)
        float k32[kNK - 1] = {0.f, 0.f, 0.f, 0.f};
        int rr = ro;                              // this thread's row, relative to r0
#pragma unroll 1
        for (int q = 0; q < dc.npass; ++q, ++n) {
            issue(n + kStages - 1);
            cp_async_wait<kStages - 1>();         // this thread's pass-n copies are in
            if (active && rr < nr) {
                const float4* su = s_stage + (size_t)(n % kStages) * 2 * kThreads + tid;
                const float4 U = su[0], D = su[kThreads];
                const float uu[NV] = {U.x, U.y, U.z, U.w};
                const float dd[NV] = {D.x, D.y, D.z, D.w};
                const float4 a = sa[rr];
                const float rf = a.w;                         // row coordinate x_r
                const float Ar = fmaf(rf * rf, h, -a.x);      // h x_r^2 - alpha_hi (exact)
                const float m2hr = -2.f * h * rf;             // exact
                float out[NV], xo[NV];
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    const float4 b = bq[e];
                    float Gh, Gl;
                    if (PAD && cr) {
                        reduced_cost(a, b, h, 1, Gh, Gl);          // pieces h x^2 - alpha, h x^2 - beta as pairs
                    } else {
                        Gh = fmaf(m2hr, b.w, Ar + b.x);            // h (x_r-x_c)^2 - alpha_hi - beta_hi
                        Gl = -(a.y + b.y);
                    }
                    const float Dv = a.z + b.z;                  // A^T (y-bar - y0)
                    const float s = uu[e] + dd[e];
                    const float w = fmaf(-s, p.sih, -Dv);        // g - v/sigma
                    const float mg = -(Gh + Gl);                 // -g
                    const float r = fmaxf(w, mg);                // z-bar - g
                    out[e] = !PAD || e < nval ? fmaf(p.trs, r, p.rho * dd[e]) : 0.f;   // pad columns stay 0
                    if constexpr (CHECK) {
                        xo[e] = 0.f;
                        if (!PAD || e < nval) {
                            const float zb = (w > mg) ? ((Gh + Gl) + w) : 0.f;
                            const float xb = fmaf(p.sf, Dv, s);
                            xo[e] = xb;
                            const float mn = fminf(xb, zb);
                            k32[0] = fmaf(r, r, k32[0]);
                            k32[1] = fmaf(mn, mn, k32[1]);
                            k32[2] = fmaf(xb, xb, k32[2]);
                            k32[3] = fmaf(zb, zb, k32[3]);
                            xacc[e] += xb;
                        }
                    }
                    cacc[e] += out[e];
                }
                __stcs(reinterpret_cast<float4*>(dout), make_float4(out[0], out[1], out[2], out[3]));
                *srow = (out[0] + out[1]) + (out[2] + out[3]);
                if constexpr (CHECK) *sxrow = (xo[0] + xo[1]) + (xo[2] + xo[3]);
            }
            dout += ostep;
            srow += rstep;
            if constexpr (CHECK) sxrow += rstep;
            rr += P;
        }
        // ---- tile epilogue: column and row sums as double-float pairs
        if (active) {
            *reinterpret_cast<float4*>(&s_col[ro * Sp + c0]) = make_float4(cacc[0], cacc[1], cacc[2], cacc[3]);
            if constexpr (CHECK)
                *reinterpret_cast<float4*>(&s_xcol[ro * Sp + c0]) = make_float4(xacc[0], xacc[1], xacc[2], xacc[3]);
        }
        __syncthreads();
        // the next tile's column values (the first threads stored its descriptor while
        // issuing its first pass, before this barrier); the loads complete
        // under the reductions below
        have = !(c.it >= ntiles && ck + 1 >= c.ik);
        if (have) load_cols(s_td[(ck + 1) % (2 * kStages)]);
        const size_t cbase = dc.colp;
        // rows: warp w sums partials [w NC/8, (w+1) NC/8) of rows lane, lane + 32, ...
        // (row stride NC + 1 keeps the lanes on distinct banks), then the 8
        // pairs of each row are combined in warp order
        {
            const int w0 = (warp * NC) / kW, w1 = ((warp + 1) * NC) / kW;
            for (int r = lane; r < nr; r += 32) {
                DF a{0.f, 0.f}, x{0.f, 0.f};
                for (int cc = w0; cc < w1; ++cc) {
                    a = df_add(a, s_row[r * (NC + 1) + cc]);
                    if constexpr (CHECK) x = df_add(x, s_xrow[r * (NC + 1) + cc]);
                }
                s_rdf[warp][r] = df_st(a);
                if constexpr (CHECK) s_xdf[warp][r] = df_st(x);
            }
        }
        if constexpr (CHECK) {
            DF kd[kNK - 1];
#pragma unroll
            for (int qq = 0; qq < kNK - 1; ++qq) kd[qq] = DF{k32[qq], 0.f};
            block_sum_df<kNK - 1>(kd, s_red);    // its barriers also publish s_rdf
            if (tid == 0) {
                float2* o = reinterpret_cast<float2*>(I.tile_kkt) + (size_t)dc.tile * kNK;
#pragma unroll
                for (int qq = 0; qq < kNK - 1; ++qq) o[qq] = df_st(kd[qq]);
            }
        } else {
            __syncthreads();
        }
        // rows on the first warps, columns on the last: side by side up to sides of 128
        for (int r = tid; r < nr; r += kThreads) {
            const float2 u0 = I.rs02[dc.row + r0 + r];          // row sum of u
            DF a = df_ld(s_rdf[0][r]), x{0.f, 0.f};
            if constexpr (CHECK) x = df_ld(s_xdf[0][r]);
#pragma unroll
            for (int w = 1; w < kW; ++w) {
                a = df_add(a, df_ld(s_rdf[w][r]));
                if constexpr (CHECK) x = df_add(x, df_ld(s_xdf[w][r]));
            }
            a = df_add(a, df_ld(u0));
            I.rs2[dc.row + r0 + r] = df_st(a);
            if constexpr (CHECK) I.xrs[dc.row + r0 + r] = df_val(x);
        }
        for (int cc = kThreads - 1 - tid; cc < S; cc += kThreads) {
            DF a{0.f, 0.f}, x{0.f, 0.f};
            for (int qq = 0; qq < P; ++qq) {
                a = df_add(a, s_col[qq * Sp + cc]);
                if constexpr (CHECK) x = df_add(x, s_xcol[qq * Sp + cc]);
            }
            I.cs32[cbase + cc] = df_f(a);
            if constexpr (CHECK) I.xcs_part[cbase + cc] = df_val(x);
        }
    }
    cp_async_wait<0>();
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kThreads, 3) k_restart(const WorkDev* __restrict__ W) {
    pdl_enter();
    extern __shared__ float4 s_ring[];               // FP32 mode: restart_ring<MODE>() passes in flight
    __shared__ double s_row[MODE == 1 ? kRowSmemBytes / 8 * 2 : 1];
    __shared__ double s_col[MODE == 1 ? kThreads * 4 : 1];
    __shared__ double s_red[2 * 32];
    __shared__ int s_tile[4];
    const int ninst = W->ninst;
    const int ntiles = W->pre_tile[ninst];
    // most blocks end without a restart: leave at once unless some instance needs this pass
    int any = 0;
    for (int i = threadIdx.x; i < ninst; i += blockDim.x) {
        const HotCtl* C = W->inst[i].ctl;
        any |= !W->inst[i].grp && ((MODE == 2) ? (C->just_finished != 0) : (C->status == ST_RUNNING && C->restart_pending != 0));
    }
    if (!__syncthreads_or(any)) return;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        TileCtx tc;
        resolve_tile(W, t, tc, s_tile);
        const HotInst& I = W->inst[tc.inst];
        bool go;
        if (MODE == 2) go = I.ctl->just_finished != 0;
        else go = (s_tile[2] == ST_RUNNING) && (s_tile[3] != 0);
        if (go) restart_tile<T, MODE, kRestartSlots>(I, tc.slab, tc.band, s_row, s_col, s_red, s_ring);
        __syncthreads();
    }
}

// Initial point w0 = 0 of a new instance: v0 = 0 and y0 = 0, so
// u = v0 - sigma0 (c - A^T y0) = -sigma0 c, with its sums in FP64.  The cost is
// the same in every slab of a half: k_init forms the first slab of each, and
// k_init_copy repeats it (FP64 arithmetic on every element, at a 64th of the
// FP32 rate, took most of the set-up).  d = 0 and x_r = z_r = 0 are not stored:
// the first sweep takes the delta as zero (HotCtl::dzero; FP64 mode clears d0)
// and the first restart the reference point (restart_tile).  256 x 256: 549 us,
// 537 MB written -> 45 + 25 us, 134 MB.  One launch per instance (descriptor by value).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_init(HotInst I, double sigma0) {
    using V = VecT<T>;
    constexpr int NV = V::N;
    __shared__ double s_row[kRowSmemBytes / 8 * 2];
    __shared__ double s_col[kThreads * 4];
    __shared__ double s_red[32];
    const int TR = I.TR;
    for (int t = blockIdx.x; t < I.nb1 + I.nb2; t += gridDim.x) {
        const int slab = t < I.nb1 ? 0 : I.n, band = t < I.nb1 ? t : t - I.nb1;
        const int S = g_side(I, slab), Sp = g_pitch(I, slab);   // this slab's side and row pitch
        const int NC = Sp / NV;
        const int P = kThreads / NC;
        const int cg = threadIdx.x % NC, ro = threadIdx.x / NC;
        const bool active = ro < P;
        const int c0 = cg * NV;
        const int r0 = band * TR, r1 = min(S, r0 + TR);
        const size_t off = g_elem(I, slab);
        DF cuf{0.f, 0.f};
        double ccol[NV];
        DF fcol[NV];
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            ccol[e] = 0.0;
            fcol[e] = DF{0.f, 0.f};
        }
        if (active) {
            for (int r = r0 + ro; r < r1; r += P) {
                T uu[NV];
                DF rsf{0.f, 0.f};
                double rs = 0.0;
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    const int xb0 = g_xbase(I, slab);
                    const bool v = c0 + e < S;                 // pad columns: 0
                    const double dc = v ? I.X64[xb0 + r] - I.X64[xb0 + c0 + e] : 0.0;
                    uu[e] = v ? (T)(-sigma0 * (dc * dc * I.h)) : T(0);
                    if constexpr (std::is_same<T, float>::value) {
                        rsf = df_add(rsf, (float)uu[e]);
                        fcol[e] = df_add(fcol[e], (float)uu[e]);
                        if (I.coord_real) {                                     // <c, u> with the FP32 positions
                            const float* X32 = I.X32 + xb0;
                            if (v) cuf = df_add(cuf, cost_times(cost_pair(X32[r], X32[c0 + e]), (float)uu[e]));
                        } else {
                            const float cq = (float)(dc * dc), p = cq * (float)uu[e];
                            cuf = df_add(cuf, DF{p, fmaf(cq, (float)uu[e], -p)});   // <c, u>
                        }
                    } else {
                        rs += (double)uu[e];
                        ccol[e] += (double)uu[e];
                    }
                }
                if constexpr (std::is_same<T, float>::value) rs = df_val(rsf);
                V::st((T*)I.u + off + (size_t)r * Sp + c0, uu);
                s_row[(r - r0) * NC + cg] = rs;
            }
        }
        if constexpr (std::is_same<T, float>::value)
#pragma unroll
            for (int e = 0; e < NV; ++e) ccol[e] = df_val(fcol[e]);
        __syncthreads();
        if (active)
#pragma unroll
            for (int e = 0; e < NV; ++e) s_col[ro * Sp + c0 + e] = ccol[e];
        __syncthreads();
        const size_t cbase = g_colp(I, slab, band);
        for (int c = threadIdx.x; c < S; c += blockDim.x) I.cs0_part[cbase + c] = sum_f64_strided(s_col + c, P, Sp);
        for (int rr = threadIdx.x; rr < r1 - r0; rr += blockDim.x)
            I.rs0[g_row(I, slab) + r0 + rr] = sum_f64_strided(s_row + rr * NC, NC, 1);
        if constexpr (std::is_same<T, float>::value) {
            DF cu[1] = {cuf};
            block_sum_df<1>(cu, reinterpret_cast<float2*>(s_red));
            if (threadIdx.x == 0) reinterpret_cast<float2*>(I.cu_part)[g_tile(I, slab, band)] = df_st(cu[0]);
        }
        __syncthreads();
    }
}

// The first slab of each half (k_init) repeated into the others: blockIdx.y the
// slab, blockIdx.x a part of it; the slab's sums with part 0.
constexpr int kCopyPart = 16;               // 16-byte words per thread
template <typename T>
__global__ void __launch_bounds__(kThreads) k_init_copy(HotInst I) {
    const int slab = blockIdx.y, first = slab < I.n ? 0 : I.n;
    if (slab == first) return;
    const int S = g_side(I, slab), nb = g_nb(I, slab);
    const size_t words = (size_t)S * g_pitch(I, slab) * sizeof(T) / 16;
    const float4* __restrict__ src = reinterpret_cast<const float4*>((const T*)I.u + g_elem(I, first));
    float4* __restrict__ dst = reinterpret_cast<float4*>((T*)I.u + g_elem(I, slab));
    const size_t q0 = (size_t)blockIdx.x * kThreads * kCopyPart + threadIdx.x;
#pragma unroll 4
    for (int u = 0; u < kCopyPart; ++u) {
        const size_t q = q0 + (size_t)u * kThreads;
        if (q < words) __stcs(dst + q, src[q]);
    }
    if (blockIdx.x == 0) {
        for (int q = threadIdx.x; q < S; q += kThreads) I.rs0[g_row(I, slab) + q] = I.rs0[g_row(I, first) + q];
        for (int q = threadIdx.x; q < S * nb; q += kThreads)
            I.cs0_part[g_colp(I, slab, 0) + q] = I.cs0_part[g_colp(I, first, 0) + q];
        for (int q = threadIdx.x; q < nb; q += kThreads) I.cu_part[g_tile(I, slab, q)] = I.cu_part[g_tile(I, first, q)];
    }
}

// --------------------------------------------------------------- k_kkt1 --
// Partial sums of ||A x-bar - b||^2 from the x-bar slab sums.  F32 (FP32 bulk
// mode): the partials are double-float pairs, like every per-block partial of
// that mode (tile KKT sums, <c, u>, <b, y>, the restart norms): GB300 runs FP64
// at a small fraction of the FP32 rate, and FP64 block reductions dominated
// these small kernels.  FP64 mode keeps FP64 throughout.

template <bool F32>
__global__ void __launch_bounds__(kThreads) k_kkt1(const WorkDev* __restrict__ W) {
    pdl_enter();
    __shared__ double s_red[kNK * 32];
    __shared__ int s_t[3];
    const int ninst = W->ninst;
    const int nchunks = W->pre_k1[ninst];
    for (int t = blockIdx.x; t < nchunks; t += gridDim.x) {
        if (threadIdx.x == 0) {
            const int i = find_inst(W->pre_k1, ninst, t);
            s_t[0] = i;
            s_t[1] = t - W->pre_k1[i];
            s_t[2] = W->inst[i].ctl->status;
        }
        __syncthreads();
        if (s_t[2] != ST_RUNNING) {
            __syncthreads();
            continue;
        }
        const HotInst& I = W->inst[s_t[0]];
        if (s_t[1] < I.n_k1) residual_chunk<F32>(I, s_t[1], s_red);
        else tile_chunk(I, s_t[1] - I.n_k1, reinterpret_cast<float2*>(s_red));
        __syncthreads();
    }
}

// --------------------------------------------------------------- k_check --
// Stopping rule eq. (kkt_res) and the restart rule, one CTA per instance.
template <bool F32>
__global__ void __launch_bounds__(kThreads) k_check(const WorkDev* __restrict__ W, int K, double a1, double a2,
                                                    double a3) {
    pdl_enter();
    __shared__ double s_red[8 * 32];
    const int ninst = W->ninst;
    for (int i = blockIdx.x; i < ninst; i += gridDim.x) {
        const HotInst& I = W->inst[i];
        if (I.grp || I.ctl->status != ST_RUNNING) continue;   // block-uniform
        check_instance<F32>(I, W, i, K, a1, a2, a3, s_red);
        __syncthreads();
    }
}

template <bool F32>
__global__ void __launch_bounds__(kThreads) k_restart_sigma(const WorkDev* __restrict__ W) {
    pdl_enter();
    __shared__ double s_red[2 * 32];
    const int ninst = W->ninst;
    for (int i = blockIdx.x; i < ninst; i += gridDim.x) {
        const HotInst& I = W->inst[i];
        if (I.grp || I.ctl->status != ST_RUNNING || !I.ctl->restart_pending) continue;
        sigma_instance<F32>(I, s_red);
        __syncthreads();
    }
}

// End of a block: an FP32 instance that finished in it adds the <c, d> share
// of its final check iteration (per-tile pairs from the restart pass MODE 2,
// summed in tile order) to its objective; every instance's flags reset.
// One CTA per instance.
__global__ void __launch_bounds__(kThreads) k_block_end(const WorkDev* __restrict__ W) {
    pdl_enter();
    __shared__ float2 s_red[32];
    const int ninst = W->ninst;
    for (int i = blockIdx.x; i < ninst; i += gridDim.x) {
        const HotInst& I = W->inst[i];
        if (I.grp) continue;
        end_instance(I, s_red);
        __syncthreads();
    }
}

// ------------------------------------------------------------- launchers --

// SM count x resident CTAs per SM (at most cap) of one kernel at kThreads
template <typename F>
static int occ_grid(F kernel, int sms, size_t dyn_smem, int cap) {
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kThreads, dyn_smem) != cudaSuccess || per < 1)
        per = 1;
    return sms * (per < cap ? per : cap);
}

LaunchDims make_launch_dims(int device, int fp64) {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (sms <= 0) sms = 1;
    LaunchDims d;
    if (fp64) {
        d.grid_tile = occ_grid(k_sweep64<false>, sms, 0, 8);
        d.grid_tile_chk = occ_grid(k_sweep64<true>, sms, 0, 8);
        d.grid_rst = std::min(occ_grid(k_restart<double, 0>, sms, 0, 8), occ_grid(k_restart<double, 1>, sms, 0, 8));
        d.grid_slab = occ_grid(k_alpha<true>, sms, 0, 4);
        d.grid_alpha = d.grid_slab;
        d.grid_vec = occ_grid(k_vec, sms, 0, 4);
        d.grid_vec1 = d.grid_vec;
    } else {
        d.grid_tile = occ_grid(k_sweep32<false, false>, sms, kSweepSmem, 8);
        d.grid_tile_chk = occ_grid(k_sweep32<true, false>, sms, kSweepSmemChk, 8);
        d.grid_rst = std::min(occ_grid(k_restart<float, 0>, sms, restart_ring(0), 8),
                              occ_grid(k_restart<float, 1>, sms, restart_ring(1), 8));
        d.grid_slab = occ_grid(k_anchor, sms, 0, 4);
        d.grid_alpha = occ_grid(k_alpha32<true>, sms, 0, 2);
        d.grid_vec = occ_grid(k_vec32<false>, sms, 0, 4);
        d.grid_vec1 = occ_grid(k_vec32<true>, sms, 0, 4);
    }
    d.grid_k1 = occ_grid(k_kkt1<true>, sms, 0, 6);
    d.grid_inst = sms * 2;
    return d;
}

int sweep_grid(int fp64) {
    static std::atomic<int> cache[2][64];    // per precision and device ordinal; 0 = not yet queried
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 0;
    std::atomic<int>& c = cache[fp64 ? 1 : 0][dev];
    if (c.load() == 0) c.store(make_launch_dims(dev, fp64).grid_tile);
    return c.load();
}

void launch_tile_table(const WorkDev* w, int ntiles, cudaStream_t st) {
    if (ntiles > 0) k_tile_table<<<(ntiles + kThreads - 1) / kThreads, kThreads, 0, st>>>(w, ntiles);
}

void launch_init(const HotInst& I, double sigma0, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int L = g_L(I), Lp = (L + 3) & ~3;
    const size_t words = (size_t)L * Lp * (I.fp64 ? 8 : 4) / 16;               // of the larger slab
    const dim3 copy((unsigned)((words + kThreads * kCopyPart - 1) / (kThreads * kCopyPart)), (unsigned)g_nslab(I));
    if (I.fp64) {
        k_init<double><<<I.nb1 + I.nb2, kThreads, 0, st>>>(I, sigma0);
        k_init_copy<double><<<copy, kThreads, 0, st>>>(I);
        cudaMemsetAsync(I.d0, 0, g_state_len(I) * sizeof(double), st);
    } else {
        k_init<float><<<I.nb1 + I.nb2, kThreads, 0, st>>>(I, sigma0);
        k_init_copy<float><<<copy, kThreads, 0, st>>>(I);
    }
    k_anchor_one<<<g_nslab(I) < sms * 4 ? g_nslab(I) : sms * 4, kThreads, 0, st>>>(I, sigma0);
}

cudaError_t kernels_init(int device) {
    (void)device;
    cudaError_t e = cudaFuncSetAttribute(k_sweep32<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep32<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmemChk);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep32<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep32<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmemChk);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep32<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep32<false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_restart<float, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)restart_ring(0));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_restart<float, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)restart_ring(1));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_restart<float, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)restart_ring(2));
    if (e == cudaSuccess) e = group_init();
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_marg, cudaFuncAttributeMaxDynamicSharedMemorySize, 7 * kMaxS * 8);
    return e;
}

// One launch of the chain (cudaLaunchKernelEx keeps every call site in one form),
// programmatically dependent on the previous kernel (pdl_enter in every kernel).
template <typename... KArgs, typename... Args>
static void launch(const LaunchDims&, void (*k)(KArgs...), int grid, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, args...);
}

void launch_solve_kernels(const WorkDev* w, const LaunchDims& ld, int fp64, int j, bool check, bool single,
                          cudaStream_t st) {
    if (fp64) {
        launch(ld, k_vec, ld.grid_vec, 0, st, w);
        launch(ld, k_marg, ld.grid_inst, 7 * kMaxS * 8, st, w);
        launch(ld, check ? k_alpha<true> : k_alpha<false>, ld.grid_slab, 0, st, w);
    } else {
        if (single) {
            launch(ld, k_vec32<true>, ld.grid_vec1, 0, st, w, j);
        } else {
            launch(ld, k_vec32<false>, ld.grid_vec, 0, st, w, j);
            launch(ld, k_stage32, ld.grid_inst, 0, st, w, j);
        }
        launch(ld, check ? k_alpha32<true> : k_alpha32<false>, ld.grid_alpha, 0, st, w, j);
    }
}

void launch_sweep(const WorkDev* w, const LaunchDims& ld, int fp64, int j, bool check, bool pad, cudaStream_t st) {
    if (fp64)
        launch(ld, check ? k_sweep64<true> : k_sweep64<false>, check ? ld.grid_tile_chk : ld.grid_tile, 0, st, w, j);
    else if (check)
        launch(ld, pad ? k_sweep32<true, true> : k_sweep32<true, false>, ld.grid_tile_chk, kSweepSmemChk, st, w, j);
    else if (j == 0)
        launch(ld, pad ? k_sweep32<false, true, true> : k_sweep32<false, false, true>, ld.grid_tile, kSweepSmem, st, w, j);
    else
        launch(ld, pad ? k_sweep32<false, true> : k_sweep32<false, false>, ld.grid_tile, kSweepSmem, st, w, j);
}

void launch_block_end(const WorkDev* w, const LaunchDims& ld, int fp64, int K, double a1, double a2, double a3,
                      cudaStream_t st) {
    if (fp64) {
        launch(ld, k_kkt1<false>, ld.grid_k1, 0, st, w);
        launch(ld, k_check<false>, ld.grid_inst, 0, st, w, K, a1, a2, a3);
        launch(ld, k_restart<double, 0>, ld.grid_rst, 0, st, w);
        launch(ld, k_restart_sigma<false>, ld.grid_inst, 0, st, w);
        launch(ld, k_restart<double, 1>, ld.grid_rst, 0, st, w);
        launch(ld, k_anchor, ld.grid_slab, 0, st, w);
        launch(ld, k_restart<double, 2>, ld.grid_rst, 0, st, w);
    } else {
        launch(ld, k_kkt1<true>, ld.grid_k1, 0, st, w);
        launch(ld, k_check<true>, ld.grid_inst, 0, st, w, K, a1, a2, a3);
        launch(ld, k_restart<float, 0>, ld.grid_rst, restart_ring(0), st, w);
        launch(ld, k_restart_sigma<true>, ld.grid_inst, 0, st, w);
        launch(ld, k_restart<float, 1>, ld.grid_rst, restart_ring(1), st, w);
        launch(ld, k_anchor, ld.grid_slab, 0, st, w);
        launch(ld, k_restart<float, 2>, ld.grid_rst, restart_ring(2), st, w);
    }
    launch(ld, k_block_end, ld.grid_inst, 0, st, w);
}

}  // namespace hot
