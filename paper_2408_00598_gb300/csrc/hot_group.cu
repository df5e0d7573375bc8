// Check blocks (K iterations of Algorithm 2, arXiv 2408.00598, and the stopping
// and restart rules) of small instances in one kernel: k_group32 (FP32 bulk
// mode), k_group64.
//
// The chain k_vec32 -> k_alpha32 -> k_sweep32 costs three launch boundaries per
// iteration, about 20 us on small grids whose sweep itself takes one or two, and
// eight more per block.  Here a group of CTAs takes an instance through its
// blocks with two waits per iteration:
//   A  slab sums: T and P of each slab (a warp per sum) from the row sums;
//      wait
//   B  every CTA forms the O(m + n) stage of Prop. 3 for itself (the same bits
//      in every CTA), then for each of its tiles the pieces of A^T y-bar (in
//      shared memory), Steps 2-4, and the tile's row and column sums;
//      wait
// and the block end (hot_block.cuh) with waits in place of its launches.  A CTA
// owns the same tiles throughout, so the flow state needs no exchange: only the
// row sums (2mn), column partials and slab sums go through L2.  The first
// tile's state is copied to shared memory while the sums and the second wait
// run, every further tile's under the sums of the one before.  Every sum that
// feeds the iterates is formed in the order of the chain (hot_dev.cuh, k_vec32,
// k_sweep32), so an instance's iterates do not depend on which of the two ran,
// nor on the size of its group.
//
// Bound by latency: an iteration of a 32 x 32 pair takes 19,400 cycles, the two
// waits 3,000 each with the CTAs' skew, slab sums 1,900, stage 3,000, pieces 2,000,
// sweep and sums 3,000.  us per iteration of a solve (block ends included), chain
// -> group: 32 x 32 24.6 -> 11.3, 64 x 64 24.7 -> 12.1, 128 x 128 31.8 -> 21.7,
// 192 x 192 58.3 -> 56.0.
//
// The groups of one launch are independent.  The grid is launched
// cooperatively, so that the CTAs of a group are resident together; it has the
// CTAs that plan_groups gave work, so that a small instance leaves the rest of
// the device to other contexts and to the caller's kernels.  Every wait is
// bounded and sets W->err when it runs out.

#include <atomic>

#include "hot_block.cuh"

namespace hot {

namespace {

constexpr int kW = kThreads / 32;
constexpr int kRowN = kRowSmemBytes / sizeof(float) + 256;
constexpr int kRing = 4;                  // passes of state in flight (one float4 of u and of d per thread each)

// Geometry of a tile; offsets fit 32 bits (sides up to kMaxGroupSide).
struct GTile {
    int slab, band, r0, nr;
    int row, colp, elem;          // g_row, g_colp, first element of row r0
    int tile;
};
__device__ __forceinline__ GTile gtile(const HotInst& I, int t) {
    GTile g;
    g_tile_slab(I, t, g.slab, g.band);
    const int S = g_side(I, g.slab);
    g.r0 = g.band * I.TR;
    g.nr = min(S, g.r0 + I.TR) - g.r0;
    g.row = (int)g_row(I, g.slab);
    g.colp = (int)g_colp(I, g.slab, g.band);
    g.elem = (int)g_elem(I, g.slab) + g.r0 * g_pitch(I, g.slab);
    g.tile = t;
    return g;
}
struct GroupSmem {
    float row[kRowN];
    float xrow[kRowN];
    float col[kThreads * 4];
    float xcol[kThreads * 4];
    float2 rdf[kW][kMaxTR];
    float4 st[kRing][2][kThreads];        // the state's passes in flight: u, delta
    float4 alpha[kMaxTR];
    float4 beta[kMaxGroupSide];
    // T and P of every slab, replaced in place by the stage's vectors:
    // (mvA, sy) of column j at j, (mvS, sp) of row k at n + k
    float4 vec[2 * kMaxGroupSide];
    float2 mar[2 * kMaxGroupSide];        // column totals of mu (cm2), row totals of nu (rm2)
    float2 red[8 * 32];                   // block sums, up to eight at once (check_instance)
    HotInst I;
    CycleK C;
    GTile tile[kTileTable];
    StageK K;
    PieceK PK;
    DF F[2];                              // half totals
    DF sm1, sm2;                          // the marginals' sums
    P32 p[64];                            // of every iteration of the block (check_every <= 64)
    int dead;                             // a wait of this CTA ran out
    int polls;                            // polls of a wait before it gives up (WorkDev::polls)
    // buffers of the block end
    __device__ double* rows() { return reinterpret_cast<double*>(row); }      // row and xrow
    __device__ double* cols() { return reinterpret_cast<double*>(col); }      // col and xcol
    __device__ double* reds() { return reinterpret_cast<double*>(red); }
    __device__ float4* ring() { return &st[0][0][0]; }                       // kRing slots of two arrays
};

// All CTAs of the group have arrived for the `epoch`-th time in this launch
// (the last CTA to leave clears the counter).  One thread per CTA arrives with a release
// and polls with an acquire: 2,300 cycles with 32 CTAs, 2,800 with 304 (a flag
// per CTA polled by whole warps took 2,000 and 8,200: the polls hold up the
// arrivals).  The barrier at the top orders the CTA's writes before thread 0's
// arrival, the one at the end the other CTAs' writes before this CTA's reads
// (through L2, __ldcg).  Without the __syncwarp the first warp stayed split
// after the poll, and what it runs alone next (group_stage) took three times
// as long.
template <typename S>
__device__ __forceinline__ bool group_wait(S& s, int G, unsigned epoch, int* err) {
    __syncthreads();
    if (G == 1) return true;
    if (threadIdx.x == 0) {
        unsigned* count = s.I.gcount;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(count) : "memory");
        unsigned v;
        int left = s.polls;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(count) : "memory");
        } while (v < epoch * (unsigned)G && --left > 0);
        if (left <= 0) {
            s.dead = 1;
            atomicExch(err, 1);
        }
    }
    __syncwarp();                                // the polling thread rejoins its warp
    __syncthreads();
    return s.dead == 0;
}

// What a thread needs of a half (f1 or f2): side, row pitch, column groups,
// rows per pass, and the thread's row and column group of a pass.
struct Half {
    int S, Sp, NC, P, ro, cg;
};
__device__ __forceinline__ Half half_of(int side) {
    Half h;
    h.S = side;
    h.Sp = (side + 3) & ~3;
    h.NC = h.Sp / 4;
    h.P = kThreads / h.NC;
    h.ro = (int)threadIdx.x / h.NC;
    h.cg = (int)threadIdx.x - h.ro * h.NC;
    return h;
}

// T or P of slab q (k_vec32's sums, in its order), one warp: T, the total of
// the slab's row sums (lane-strided, then the shuffle tree), or P, the column
// sum across the other half's slabs: P2[j] for f1 slab j, P1[k] for f2 slab k,
// in blocks of kVecRows rows, each block in eight runs of eight rows.  Valid
// in lane 0.
__device__ __forceinline__ DF slab_sum(const HotInst& I, const float2* __restrict__ rs, int q, bool cross, int lane) {
    const int m = I.m, n = I.n, h2 = n * m;               // h2: first row of the f2 half
    const bool f1 = q < n;
    const int len = f1 ? m : n;
    int at, step, left;                                   // this lane's terms: at, at + step, ... (left of them)
    if (cross) {
        const int c0 = (lane >> 3) * kVecRows + (lane & 7) * 8;
        step = f1 ? n : m;
        at = (f1 ? h2 + q : q - n) + c0 * step;
        left = len - c0;                                  // f1 slab j: m rows k; f2 slab k: n rows j
    } else {
        step = 32;
        at = (f1 ? q * m : h2 + (q - n) * n) + lane;
        left = (len - lane + 31) >> 5;
    }
    float2 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = u < left ? __ldcg(rs + at + u * step) : make_float2(0.f, 0.f);
    DF c{0.f, 0.f}, b{0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 8; ++u) c = df_add(c, df_ld(v[u]));
    if (!cross) {
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) c = df_add(c, df_shfl_down(c, o));
        return c;
    }
#pragma unroll 1
    for (int u = 0; u < 8; ++u)                           // the block's eight runs, in order
        b = df_add(b, DF{__shfl_sync(0xffffffffu, c.hi, (lane & ~7) + u), __shfl_sync(0xffffffffu, c.lo, (lane & ~7) + u)});
    c = DF{0.f, 0.f};
#pragma unroll 1
    for (int u = 0; u * kVecRows < len; ++u)
        c = df_add(c, DF{__shfl_sync(0xffffffffu, b.hi, 8 * u), __shfl_sync(0xffffffffu, b.lo, 8 * u)});
    return c;
}

// Half total F1 (half 0: the f1 slabs' T) or F2 by one warp each, in the order
// of k_vec32's item totals and alpha32_stage's block sum: the items of 8 slabs
// left to right, the shuffle tree over 32 items (the f2 items after the f1
// ones), then the warps' totals.
__device__ __forceinline__ void group_half_total(GroupSmem& s, int half, int lane) {
    const int m = s.I.m, n = s.I.n;
    const int t1 = (n + 7) / 8, t2 = (m + 7) / 8;                 // t1 + t2 <= 64
    const int cnt = half ? m : n;
    const float4* tp = s.vec + (half ? n : 0);
    DF F{0.f, 0.f};
#pragma unroll 1
    for (int q = lane; q - lane < t1 + t2; q += 32) {
        const int item = half ? q - t1 : q;
        const int s0 = item * 8;
        float2 v[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const bool in = item >= 0 && s0 + w < cnt;
            const float4 t = in ? tp[s0 + w] : make_float4(0.f, 0.f, 0.f, 0.f);
            v[w] = make_float2(t.x, t.y);
        }
        DF a = df_ld(v[0]);
#pragma unroll
        for (int w = 1; w < 8; ++w) a = df_add(a, df_ld(v[w]));
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) a = df_add(a, df_shfl_down(a, o));
        F = df_add(F, a);
    }
    if (lane == 0) s.F[half] = F;
}

// The stage's scalars, by one warp.
__device__ __forceinline__ void group_stage(GroupSmem& s, float kdl, int lane) {
    const int m = s.I.m, n = s.I.n;
    const float4 last = s.vec[n + m - 1];
    const StageK K = stage_scalars(m, n, s.C, s.sm1, s.sm2, s.F[0], s.F[1], DF{last.x, last.y}, DF{last.z, last.w},
                                   df_ld(s.mar[n + m - 1]), kdl);
    if (lane == 0) s.K = K;
}

// The stage's vectors, one entry per thread.
__device__ __forceinline__ void group_vectors(GroupSmem& s) {
    const int m = s.I.m, n = s.I.n;
    const StageK& K = s.K;
#pragma unroll 1
    for (int q = threadIdx.x; q < m + n; q += kThreads) {
        const float4 t = s.vec[q];
        const DF T{t.x, t.y}, P{t.z, t.w};
        const bool col = q < n, last = q == n + m - 1;
                const DF c = df_ld(s.mar[q]);
        // column: a_j, bb_j; row: (T2 - P1)/sigma, r3_k
        const DF A = df_mul(col ? df_sub(P, T) : df_sub(T, P), K.is);
        DF B = df_mul(df_sub(c, T), K.is);
        if (last) B = df_sub(B, K.drop);
        const DF Bi = df_mul(B, col ? K.imin : K.in);       // bb_j (1/m + 1/n); r3_k / n
        const DF e = df_add(A, col ? df_neg(B) : B);    // a_j - bb_j; e_k
        const DF f = df_mul(df_add(e, col ? K.T3in : K.cst), col ? K.in : K.imn);   // sy_j + yasum; s_k
        DF x, y;
        if (col) {
            x = df_sub(df_mul(A, K.in), Bi);                   // mvA_j
            y = df_sub(f, K.yasum);                            // sy_j
        } else {
            const DF ya = df_add(df_neg(df_mul(df_add(f, K.dsiw), last ? K.dl : K.im)), K.tin);
            x = df_sub(df_add(Bi, K.T3in2), df_mul(ya, (float)(m + n)));   // mvS_k
            y = df_sub(f, df_mul(ya, (float)n));                  // sp_k
        }
        s.vec[q] = make_float4(x.hi, x.lo, y.hi, y.lo);
    }
}

// The inputs of one piece of a tile that do not wait for the stage: item < nr
// is the alpha piece of row r0 + item, item >= nr the beta piece of column
// item - nr.
struct PieceLd {
    float2 a0, x, y;              // y: a column's first two bands until piece_finish sums them
    float2 z;                     // and the next two
    float xc;
};
__device__ __forceinline__ PieceLd piece_load(const HotInst& I, const GTile& g, int S, int item,
                                              const float2* __restrict__ rs, const float* __restrict__ cs) {
    PieceLd p;
    const int m = I.m, n = I.n;
    const bool f1 = g.slab < n, row = item < g.nr;
    const int e = row ? g.r0 + item : item - g.nr;
    p.a0 = I.ab0_32[2 * g.row + (row ? 0 : S) + e];
    p.xc = I.X32[(f1 ? 0 : m) + e];
    if (row) {
        const int j = f1 ? g.slab : e, k = f1 ? e : g.slab - n;
        p.x = __ldcg(rs + n * m + k * n + j);
        p.y = __ldcg(rs + j * m + k);
    } else {
        const int nb = f1 ? I.nb1 : I.nb2;
        const float* c = cs + (g.colp - g.band * S) + e;
        p.y.x = __ldcg(c);
        p.y.y = nb > 1 ? __ldcg(c + S) : 0.f;
        p.z.x = nb > 2 ? __ldcg(c + 2 * S) : 0.f;
        p.z.y = nb > 3 ? __ldcg(c + 3 * S) : 0.f;
        p.x = I.K2[g.row + e];
    }
    return p;
}
// The piece itself (piece_dv and piece_pack), into shared memory; the pair and
// the float4 also go to global memory on check iterations (the restart and the
// objective read them there).
__device__ __forceinline__ void piece_finish(GroupSmem& s, const GTile& g, int S, int item, const PieceLd& p,
                                             const float* __restrict__ cs, bool out) {
    const HotInst& I = s.I;
    const PieceK& K = s.PK;
    const int n = I.n;
    const bool f1 = g.slab < n, row = item < g.nr;
    const int e = row ? g.r0 + item : item - g.nr;
    const float4 own = s.vec[g.slab];                            // of the slab itself
    const float4 oth = s.vec[row ? (f1 ? n + e : e) : g.slab];
    const float4 vj = f1 ? own : oth, vk = f1 ? oth : own;
    float kd = 0.f;                                              // the column's total over its bands, left to right
    if (!row) {
        const int nb = f1 ? I.nb1 : I.nb2;
        kd = __fadd_rn(kd, p.y.x);
        if (nb > 1) kd = __fadd_rn(kd, p.y.y);
        if (nb > 2) kd = __fadd_rn(kd, p.z.x);
        if (nb > 3) kd = __fadd_rn(kd, p.z.y);
#pragma unroll 1
        for (int b = 4; b < nb; ++b) kd = __fadd_rn(kd, __ldcg(cs + (g.colp + (b - g.band) * S) + e));
    }
    // row: R1 / sigma, then + mvA_j + mvS_k, over m + n; column: K2 - kd / (sigma side) + colc
    DF q = df_mul(row ? df_sub(df_ld(p.x), df_ld(p.y)) : DF{kd, 0.f}, row ? K.is : f1 ? K.isim : K.isin);
    DF dv{0.f, 0.f};                                             // the dropped row's piece stays 0
    if (row) {
        q = df_add(df_add(q, DF{vj.x, vj.y}), DF{vk.x, vk.y});
        dv = df_mul(q, K.imn);
        if (!f1) dv = df_neg(dv);
    } else if (g.slab != n + I.m - 1 || e != n - 1) {
        const DF colc = df_mul(DF{own.z, own.w}, f1 ? df_neg(K.im) : K.in);
        dv = df_add(df_sub(df_ld(p.x), q), colc);
    }
    PieceIn a;
    a.a0 = p.a0;
    a.xc = p.xc;
    const float4 w = piece_pack(a, dv, K, I.coord_real);
    if (row) s.alpha[item] = w;
    else s.beta[e] = w;
    if (out && (row || g.band == 0)) {
        const int o = 2 * g.row + (row ? 0 : S) + e;
        I.dab2[o] = df_st(dv);
        I.ab32[o] = w;
    }
}

// Asynchronous copies of the state into the ring: pass slot c of a tile into
// st[c % kRing], a commit group per pass.  A thread reads back only what it
// copied, so its own wait_group is enough; no registers are held meanwhile
// (spilled registers are costly here: an acquire drops the L1 lines they
// sit in).
__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_pass(GroupSmem& s, int c, bool v, int o, const float* __restrict__ u,
                                          const float* din) {
    if (v) {
        copy16(&s.st[c][0][threadIdx.x], u + o);
        if (din) copy16(&s.st[c][1][threadIdx.x], din + o);
        else s.st[c][1][threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ int tile_off(const GTile& g, const Half& hf) { return g.elem + hf.ro * hf.Sp + hf.cg * 4; }
// the first kRing passes of a tile
__device__ __forceinline__ void copy_tile(GroupSmem& s, const GTile& g, const Half& hf, const float* __restrict__ u,
                                          const float* din) {
    int rr = hf.ro < hf.P ? hf.ro : g.nr, o = tile_off(g, hf);
#pragma unroll 1
    for (int c = 0; c < kRing; ++c) {
        copy_pass(s, c, rr < g.nr, o, u, din);
        rr += hf.P;
        o += hf.P * hf.Sp;
    }
}

// block_sum_df in rolled loops (the same order): the code of this kernel has
// to stay in the instruction caches.
__device__ __forceinline__ void group_block_sum(DF (&v)[kNK - 1], float2* sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < kNK - 1; ++q) v[q] = df_add(v[q], df_shfl_down(v[q], o));
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < kNK - 1; ++q) sh[q * 32 + warp] = df_st(v[q]);
    __syncthreads();
    if (warp < kNK - 1) {                            // a warp per sum
        DF x = lane < kW ? df_ld(sh[warp * 32 + lane]) : DF{0.f, 0.f};
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) x = df_add(x, df_shfl_down(x, o));
        __syncwarp();
        if (lane == 0) sh[warp * 32] = df_st(x);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kNK - 1; ++q) v[q] = df_ld(sh[q * 32]);
    __syncthreads();
}

// Steps 2-4 on one tile (k_sweep32's arithmetic and sums).  The tile's first
// passes are in the ring; din = nullptr: the delta is zero.  `between`
// runs after the state's last use and before the sums: it loads what the next
// tile needs, under the sums' latency.
template <bool CHECK, bool PAD, typename F>
__device__ __forceinline__ void group_sweep(GroupSmem& s, const GTile& g, const Half& hf, const P32& p,
                                            const float* __restrict__ u, const float* din, float* dout,
                                            float2* __restrict__ rs_out, float* __restrict__ cs_out, F between) {
    const HotInst& I = s.I;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int S = hf.S, Sp = hf.Sp, NC = hf.NC, P = hf.P, nr = g.nr;
    const int ro = hf.ro;
    const bool active = ro < P;
    const int c0 = hf.cg * 4;
    const int nval = PAD ? S - c0 : 4;
    const int cr = PAD ? I.coord_real : 0;
    const float h = p.h;
    float4 bq[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        bq[e] = active && (!PAD || c0 + e < S) ? s.beta[c0 + e] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (!cr) {
            const float cf = bq[e].w;
            bq[e] = make_float4(fmaf(cf * cf, h, -bq[e].x), bq[e].y, bq[e].z, cf);
        }
    }
    float cacc[4], xacc[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) cacc[e] = xacc[e] = 0.f;
    float k32[kNK - 1] = {0.f, 0.f, 0.f, 0.f};
    const int step = P * Sp, rstep = P * (NC + 1);
    int at = tile_off(g, hf);                         // this thread's element of the pass
    int sr = ro * (NC + 1) + hf.cg;                   // and its row partial
    int rr = active ? ro : nr;
    const int npass = (nr + P - 1) / P;
    // this thread's row of the tile (rows below) and its row sum of u
    const int r = tid;
    const float2 r0 = r < nr ? I.rs02[g.row + g.r0 + r] : make_float2(0.f, 0.f);
#pragma unroll 1
    for (int q = 0; q < npass; ++q) {
            asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 1) : "memory");
            const int c = q % kRing;
            if (rr < nr) {
                const float4 Uq = s.st[c][0][tid], Dq = s.st[c][1][tid];
                const float uu[4] = {Uq.x, Uq.y, Uq.z, Uq.w};
                const float dd[4] = {Dq.x, Dq.y, Dq.z, Dq.w};
                const float4 a = s.alpha[rr];
                const float rf = a.w;
                const float Ar = fmaf(rf * rf, h, -a.x);
                const float m2hr = -2.f * h * rf;
                float out[4], xo[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float4 b = bq[e];
                    float Gh, Gl;
                    if (PAD && cr) {
                        reduced_cost(a, b, h, 1, Gh, Gl);
                    } else {
                        Gh = fmaf(m2hr, b.w, Ar + b.x);
                        Gl = -(a.y + b.y);
                    }
                    const float Dv = a.z + b.z;
                    const float sv = uu[e] + dd[e];
                    const float w = fmaf(-sv, p.sih, -Dv);
                    const float mg = -(Gh + Gl);
                    const float r = fmaxf(w, mg);
                    out[e] = !PAD || e < nval ? fmaf(p.trs, r, p.rho * dd[e]) : 0.f;
                    if constexpr (CHECK) {
                        xo[e] = 0.f;
                        if (!PAD || e < nval) {
                            const float zb = (w > mg) ? ((Gh + Gl) + w) : 0.f;
                            const float xb = fmaf(p.sf, Dv, sv);
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
                *reinterpret_cast<float4*>(dout + at) = make_float4(out[0], out[1], out[2], out[3]);
                s.row[sr] = (out[0] + out[1]) + (out[2] + out[3]);
                if constexpr (CHECK) s.xrow[sr] = (xo[0] + xo[1]) + (xo[2] + xo[3]);
            }
            copy_pass(s, c, rr + kRing * P < nr, at + kRing * step, u, din);   // into the slot just read
            rr += P;
            at += step;
            sr += rstep;
    }
    if (active) {
        *reinterpret_cast<float4*>(&s.col[ro * Sp + c0]) = make_float4(cacc[0], cacc[1], cacc[2], cacc[3]);
        if constexpr (CHECK)
            *reinterpret_cast<float4*>(&s.xcol[ro * Sp + c0]) = make_float4(xacc[0], xacc[1], xacc[2], xacc[3]);
    }
    between();
    __syncthreads();
    {
        const int w0 = (warp * NC) / kW, w1 = ((warp + 1) * NC) / kW;
#pragma unroll 1
        for (int t = lane; t < nr; t += 32) {
            DF a{0.f, 0.f};
#pragma unroll 1
            for (int cc = w0; cc < w1; ++cc) a = df_add(a, s.row[t * (NC + 1) + cc]);
            s.rdf[warp][t] = df_st(a);
        }
    }
    if constexpr (CHECK) {
        DF kd[kNK - 1];
#pragma unroll
        for (int qq = 0; qq < kNK - 1; ++qq) kd[qq] = DF{k32[qq], 0.f};
        group_block_sum(kd, s.red);                  // its barriers also publish rdf
        if (tid == 0) {
            float2* o = reinterpret_cast<float2*>(I.tile_kkt) + g.tile * kNK;
#pragma unroll
            for (int qq = 0; qq < kNK - 1; ++qq) o[qq] = df_st(kd[qq]);
        }
    } else {
        __syncthreads();
    }
    // rows on the first warps, columns on the last: side by side up to sides of 128
    if (r < nr) {
        float2 v[kW];
#pragma unroll
        for (int w = 0; w < kW; ++w) v[w] = s.rdf[w][r];
        DF a = df_ld(v[0]);
#pragma unroll
        for (int w = 1; w < kW; ++w) a = df_add(a, df_ld(v[w]));
        a = df_add(a, df_ld(r0));
        __stcg(rs_out + g.row + g.r0 + r, df_st(a));
    }
    if (const int cc = kThreads - 1 - tid; cc < S) {
        DF a{0.f, 0.f}, x{0.f, 0.f};
#pragma unroll 4
        for (int qq = 0; qq < P; ++qq) {
            a = df_add(a, s.col[qq * Sp + cc]);
            if constexpr (CHECK) x = df_add(x, s.xcol[qq * Sp + cc]);
        }
        __stcg(cs_out + g.colp + cc, df_f(a));
        if constexpr (CHECK) I.xcs_part[g.colp + cc] = df_val(x);
    }
    if constexpr (CHECK) {
        // the row sums of x-bar, in the same order, through the same buffer
        __syncthreads();
        const int w0 = (warp * NC) / kW, w1 = ((warp + 1) * NC) / kW;
#pragma unroll 1
        for (int t = lane; t < nr; t += 32) {
            DF x{0.f, 0.f};
#pragma unroll 1
            for (int cc = w0; cc < w1; ++cc) x = df_add(x, s.xrow[t * (NC + 1) + cc]);
            s.rdf[warp][t] = df_st(x);
        }
        __syncthreads();
        if (r < nr) {
            DF x = df_ld(s.rdf[0][r]);
#pragma unroll 1
            for (int w = 1; w < kW; ++w) x = df_add(x, df_ld(s.rdf[w][r]));
            I.xrs[g.row + g.r0 + r] = df_val(x);
        }
    }
}

// The end of a check block (the kernels k_kkt1 ... k_block_end of the chain),
// shared out over the group's CTAs.  Returns true when the instance goes on.
// Out of line: its code is large and runs once in K iterations.
struct BlockRule {
    int K;
    double a1, a2, a3;
};
template <typename T, typename S>
__device__ __noinline__ bool group_block_end(S& s, const WorkDev* W, int inst, int rank, int G,
                                             unsigned& epoch, BlockRule rule) {
    const HotInst& I = s.I;
    constexpr bool F32 = std::is_same<T, float>::value;
    double* s_row = s.rows();
    double* s_col = s.cols();
    double* s_red = s.reds();
    const int nt = g_ntiles(I);
    if (!group_wait(s, G, ++epoch, W->err)) return false;
#pragma unroll 1
    for (int c = rank; c < I.n_k1 + (F32 ? I.n_achunk + I.n_kc : 0); c += G) {
        if (c < I.n_k1) residual_chunk<F32>(I, c, s_red);
        else if (c < I.n_k1 + I.n_achunk) objective_chunk(I, c - I.n_k1, reinterpret_cast<float2*>(s_red), reinterpret_cast<float*>(s_col));
        else tile_chunk(I, c - I.n_k1 - I.n_achunk, reinterpret_cast<float2*>(s_red));
        __syncthreads();
    }
    if (!group_wait(s, G, ++epoch, W->err)) return false;
    if (rank == 0) check_instance<F32>(I, W, inst, rule.K, rule.a1, rule.a2, rule.a3, s_red);
    if (!group_wait(s, G, ++epoch, W->err)) return false;
    const int status = __ldcg(&I.ctl->status), restart = __ldcg(&I.ctl->restart_pending);
    auto tiles = [&](auto mode) {
#pragma unroll 1
        for (int t = rank; t < nt; t += G) {
            int slab, band;
            g_tile_slab(I, t, slab, band);
            restart_tile<T, decltype(mode)::value, decltype(mode)::value == 0 ? kRing / 2 : kRing>(I, slab, band, s_row, s_col,
                                                                                                s_red, s.ring());
            __syncthreads();
        }
    };
    if (status != ST_RUNNING) {
        tiles(std::integral_constant<int, 2>());             // x-bar and <c, d> of the final iteration
        if (!group_wait(s, G, ++epoch, W->err)) return false;
        if (rank == 0) end_instance(I, reinterpret_cast<float2*>(s_red));
        return false;
    }
    if (!restart) return true;
    tiles(std::integral_constant<int, 0>());
    if (!group_wait(s, G, ++epoch, W->err)) return false;
    if (rank == 0) sigma_instance<F32>(I, s_red);
    if (!group_wait(s, G, ++epoch, W->err)) return false;
    tiles(std::integral_constant<int, 1>());
    if (!group_wait(s, G, ++epoch, W->err)) return false;
    const double sigma = __ldcg(&I.ctl->sigma);
#pragma unroll 1
    for (int slab = rank; slab < g_nslab(I); slab += G) anchor_slab(I, slab, sigma);
    if (rank == 0 && threadIdx.x == 0) I.ctl->restart_pending = 0;   // read by every CTA before the waits above
    return group_wait(s, G, ++epoch, W->err);
}

template <bool PAD>
__device__ __forceinline__ void group_instance(GroupSmem& s, const WorkDev* __restrict__ W, int inst, int rank, int G,
                                               int blocks, BlockRule rule) {
    const HotInst& I = s.I;
    const int K = rule.K;
    int* err = W->err;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ns = I.m + I.n, nt = g_ntiles(I);
    const int nq = (nt - rank + G - 1) / G;            // tiles of this CTA: rank, rank + G, ... (at most kTileTable)
    const float* u = (const float*)I.u;
    float* d0 = (float*)I.d0;
    float* d1 = (float*)I.d1;
    const Half h1 = half_of(I.m), h2 = half_of(I.n);
    if (tid == 64) {
        s.sm1 = df_from(I.sum_mu1);
        s.sm2 = df_from(I.sum_mu2);
    }
#pragma unroll 1
    for (int q = tid; q < ns; q += kThreads) s.mar[q] = q < I.n ? I.cm2[q] : I.rm2[q - I.n];
    unsigned epoch = 0;
#pragma unroll 1
  for (int blk = 0; blk < blocks; ++blk) {
    const bool dz = __ldcg(&I.ctl->dzero) != 0;
    if (tid < K) s.p[tid] = make_p32(__ldcg(&I.ctl->sigma), __ldcg(&I.ctl->k) + tid, I.h, I.gadmm, I.relax);
    if (tid >= 128 && tid - 128 < nq) s.tile[tid - 128] = gtile(I, rank + (tid - 128) * G);
#pragma unroll 1
    for (int q = tid; q < (int)(sizeof(CycleK) / 8); q += kThreads)
        reinterpret_cast<double*>(&s.C)[q] = __ldcg(reinterpret_cast<const double*>(I.cyc) + q);
    __syncthreads();
    if (tid == 96) s.PK = piece_consts(I, s.C);        // read after the first wait
#pragma unroll 1
    for (int it = 0; it < K; ++it) {
        // iteration it reads the delta of it - 1: d0 at the block's start, then
        // d1 in place; the check iteration leaves d1 for the restart and writes d0
        const bool check = it == K - 1;
        const float* din = it == 0 ? (dz ? nullptr : d0) : d1;
        float* dout = check ? d0 : d1;
        const float2* rs = it & 1 ? I.rs2b : I.rs2;
        float2* rs_out = it & 1 ? I.rs2 : I.rs2b;
        const float* cs = it & 1 ? I.cs32b : I.cs32;
        float* cs_out = it & 1 ? I.cs32 : I.cs32b;
        PieceLd pl = {};
        if (it > 0 && !group_wait(s, G, ++epoch, err)) return;
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
            const GTile& g = s.tile[q];
            const Half& hf = g.slab < I.n ? h1 : h2;
            if (q == 0) {
                copy_tile(s, g, hf, u, din);                  // arrives under the sums and the second wait
                // A: slab sums (T and P of slab w as two jobs, on the last warps first)
#pragma unroll 1
                for (int w = rank + G * (kW - 1 - warp); w < 2 * ns; w += G * kW) {
                    const bool cross = w >= ns;
                    const int slab = cross ? w - ns : w;
                    const DF v = slab_sum(I, rs, slab, cross, lane);
                    if (lane == 0) __stcg(reinterpret_cast<float2*>(I.tp + slab) + (cross ? 1 : 0), df_st(v));
                }
                if (tid < g.nr + hf.S) pl = piece_load(I, g, hf.S, tid, rs, cs);   // arrives under the wait
                float kdl = 0.f;
                if (warp == 0) {
                    const float* c = cs + g_colp(I, ns - 1, 0) + (I.n - 1);
#pragma unroll 1
                    for (int b = 0; b < I.nb2; ++b) kdl = __fadd_rn(kdl, __ldcg(c + b * I.n));
                }
                if (!group_wait(s, G, ++epoch, err)) return;
                // B: the stage
#pragma unroll 1
                for (int w = tid; w < ns; w += kThreads) s.vec[w] = __ldcg(I.tp + w);
                __syncthreads();
                if (warp < 2) group_half_total(s, warp, lane);
                __syncthreads();
                if (warp == 0) group_stage(s, kdl, lane);
                __syncthreads();
                group_vectors(s);
                __syncthreads();
            }
#pragma unroll 1
            for (int item = tid; item < g.nr + hf.S; item += kThreads) {
                if (item != tid) pl = piece_load(I, g, hf.S, item, rs, cs);
                piece_finish(s, g, hf.S, item, pl, cs, check);
            }
            __syncthreads();
            auto between = [&]() {
                const int qn = q + 1;
                if (qn == nq) return;
                const GTile& gn = s.tile[qn];
                const Half& hn = gn.slab < I.n ? h1 : h2;
                copy_tile(s, gn, hn, u, din);
                if (tid < gn.nr + hn.S) pl = piece_load(I, gn, hn.S, tid, rs, cs);
            };
            if (check)
                group_sweep<true, PAD>(s, g, hf, s.p[it], u, din, dout, rs_out, cs_out, between);
            else
                group_sweep<false, PAD>(s, g, hf, s.p[it], u, din, dout, rs_out, cs_out, between);
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (!group_block_end<float>(s, W, inst, rank, G, epoch, rule)) return;
  }
}

// The entries of one CTA: each names an instance, the CTA's rank in its group
// and the group's size.  run(s, entry) takes the instance through its blocks.
template <typename S, typename F>
__device__ __forceinline__ void group_entries(S& s, const WorkDev* __restrict__ W, F run) {
    const int tid = threadIdx.x;
    const int e0 = W->gstart[blockIdx.x], e1 = W->gstart[blockIdx.x + 1];
    if (tid == 0) {
        s.dead = __ldcg(W->err);                       // set in an earlier launch: nothing more is done
        s.polls = W->polls;
    }
#pragma unroll 1
    for (int e = e0; e < e1; ++e) {
        const int4 ge = W->gent[e];                    // instance, rank, group size
        __syncthreads();
        if (s.dead) return;                            // its state is lost; no later entry would be waited for
        const HotInst* src = W->inst + ge.x;
#pragma unroll 1
        for (int q = tid; q < (int)(sizeof(HotInst) / 8); q += kThreads)
            reinterpret_cast<double*>(&s.I)[q] = reinterpret_cast<const double*>(src)[q];
        __syncthreads();
        if (s.I.ctl->status != ST_RUNNING) continue;   // the same for the whole group
        if (ge.y == 0 && tid == 0 && s.I.ctl->total == 0) s.I.ctl->t_start = clock_ns();
        run(ge);
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        if (ge.z > 1 && tid == 0 && s.dead == 0) {
            // the last CTA to leave (all have left their waits) clears the counters for the next launch
            __threadfence();
            if (atomicAdd(s.I.gcount + 1, 1u) == (unsigned)ge.z - 1u) {
                s.I.gcount[0] = 0u;
                s.I.gcount[1] = 0u;
            }
        }
    }
}

template <bool PAD>
__global__ void __launch_bounds__(kThreads, 2) k_group32(const WorkDev* __restrict__ W, int blocks, BlockRule rule) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    GroupSmem& s = *reinterpret_cast<GroupSmem*>(s_raw);
    group_entries(s, W, [&](int4 ge) { group_instance<PAD>(s, W, ge.x, ge.y, ge.z, blocks, rule); });
}

// -------------------------------------------------------------- k_group64 --
// The same for FP64 mode: slab sums (k_vec's), wait, the vectors of Prop. 3 in
// every CTA (marg64), then per tile the pieces (pieces64) and the sweep
// (sweep64_tile), wait; the block end.  The arithmetic and its order are the
// chain's (k_vec, k_marg, k_alpha, k_sweep64).  us per iteration of a solve,
// chain -> group: 16 x 16 27.6 -> 15.4, 64 x 64 58 -> 31, 96 x 96 80 -> 70; bound by
// FP64 latency (about 60 cycles an operation, 440 a conversion) and the waits.
struct Group64Smem {
    Sweep64Smem sw;
    double red[8 * 32];
    double sv[7 * kMaxGroupSide64];        // T1 T2 P1 P2, then the work vectors of marg64
    double mv[4 * kMaxGroupSide64];
    double ab[2 * kMaxGroupSide64], dab[2 * kMaxGroupSide64];   // pieces of the tile's slab
    float mx[32];
    HotInst I;
    Recip64 R;
    P64 p[64];
    int dead, polls;
    __device__ double* rows() { return sw.row; }             // row and xrow
    __device__ double* cols() { return sw.col; }             // col and xcol
    __device__ double* reds() { return red; }
    __device__ float4* ring() { return nullptr; }            // FP32 mode only
};

// T1[j], T2[k], P1[k], P2[j] (k_vec's order), one warp; valid in lane 0.
__device__ __forceinline__ double vec64(const HotInst& I, const double* __restrict__ rs, int q, int lane, int& out) {
    const int m = I.m, n = I.n, L = g_L(I), f2 = n * m;      // f2: first row of the f2 half
    int at, step, len;
    if (q < n) {                                             // T1[j]: f1 slab j, its m rows
        at = q * m, step = 1, len = m, out = q;
    } else if ((q -= n) < m) {                               // T2[k]: f2 slab k, its n rows
        at = f2 + q * n, step = 1, len = n, out = L + q;
    } else if ((q -= m) < m) {                               // P1[k]: row k of every f1 slab
        at = q, step = m, len = n, out = 2 * L + q;
    } else {                                                 // P2[j]: row j of every f2 slab
        q -= m;
        at = f2 + q, step = n, len = m, out = 3 * L + q;
    }
    double acc = 0.0;
#pragma unroll 4
    for (int t = lane; t < len; t += 32) acc += __ldcg(rs + at + t * step) + I.rs0[at + t * step];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    return acc;
}

__device__ __forceinline__ void group_instance64(Group64Smem& s, const WorkDev* __restrict__ W, int inst, int rank,
                                                 int G, int blocks, BlockRule rule) {
    const HotInst& I = s.I;
    const int K = rule.K;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int L = g_L(I), nv = 2 * (I.m + I.n), nt = g_ntiles(I);
    unsigned epoch = 0;
#pragma unroll 1
    for (int blk = 0; blk < blocks; ++blk) {
        const double sigma = __ldcg(&I.ctl->sigma);
        if (tid < K) s.p[tid] = make_p64(sigma, __ldcg(&I.ctl->k) + tid, I.h, I.gadmm, I.relax);
        if (tid == kThreads - 1) s.R = recip64(I.m, I.n, sigma);
        __syncthreads();
#pragma unroll 1
        for (int it = 0; it < K; ++it) {
            const bool check = it == K - 1;
            const double* din = (const double*)(it & 1 ? I.d1 : I.d0);
            double* dout = (double*)(it & 1 ? I.d0 : I.d1);
            const double* rs = it & 1 ? I.rsb : I.rs;
            double* rs_out = it & 1 ? I.rs : I.rsb;
            const double* cs = it & 1 ? I.cs_partb : I.cs_part;
            double* cs_out = it & 1 ? I.cs_part : I.cs_partb;
            if (it > 0 && !group_wait(s, G, ++epoch, W->err)) return;
#pragma unroll 1
            for (int q = rank + G * warp; q < nv; q += G * kW) {
                int out = 0;
                const double v = vec64(I, rs, q, lane, out);
                if (lane == 0) __stcg(I.vecs + out, v);
            }
            if (!group_wait(s, G, ++epoch, W->err)) return;
#pragma unroll 1
            for (int q = tid; q < 4 * L; q += kThreads) s.sv[q] = __ldcg(I.vecs + q);
            marg64(I, s.R, cs, s.mv, s.sv, s.red);
            __syncthreads();
#pragma unroll 1
            for (int t = rank; t < nt; t += G) {
                int slab, band;
                g_tile_slab(I, t, slab, band);
                const int S = g_side(I, slab), r0 = band * I.TR, nr = min(S, r0 + I.TR) - r0;
                const size_t o = 2 * g_row(I, slab);
                if (check) {
                    pieces64<true>(I, s.R, slab, r0, nr, band == 0, rs, cs, s.mv, s.ab, s.dab, s.red, s.mx);
                    __syncthreads();
                    // the block end reads the pieces in global memory
                    for (int q = tid; q < 2 * S; q += kThreads)
                        if (q >= S ? band == 0 : q >= r0 && q < r0 + nr) {
                            I.ab64[o + q] = s.ab[q];
                            I.dab64[o + q] = s.dab[q];
                        }
                    sweep64_tile<true>(I, slab, band, din, dout, s.p[it], s.ab, s.dab, rs_out, cs_out, s.sw);
                } else {
                    pieces64<false>(I, s.R, slab, r0, nr, band == 0, rs, cs, s.mv, s.ab, s.dab, s.red, s.mx);
                    __syncthreads();
                    sweep64_tile<false>(I, slab, band, din, dout, s.p[it], s.ab, s.dab, rs_out, cs_out, s.sw);
                }
                __syncthreads();
            }
        }
        if (!group_block_end<double>(s, W, inst, rank, G, epoch, rule)) return;
    }
}

__global__ void __launch_bounds__(kThreads, 2) k_group64(const WorkDev* __restrict__ W, int blocks, BlockRule rule) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    Group64Smem& s = *reinterpret_cast<Group64Smem*>(s_raw);
    group_entries(s, W, [&](int4 ge) { group_instance64(s, W, ge.x, ge.y, ge.z, blocks, rule); });
}

}  // namespace

static_assert(sizeof(HotInst) % 8 == 0 && sizeof(CycleK) % 8 == 0, "descriptors are copied in 8-byte words");

cudaError_t group_init() {
    cudaError_t e =
        cudaFuncSetAttribute(k_group32<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GroupSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_group32<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GroupSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_group64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Group64Smem));
    return e;
}

int group_grid(int fp64) {
    static std::atomic<int> cache[2][64];    // per precision and device ordinal; 0 = not yet queried
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::atomic<int>& c = cache[fp64 ? 1 : 0][dev];
    if (c.load() == 0) {
        int sms = 0, a = 0, b = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (group_init() != cudaSuccess) return 0;
        cudaError_t e = fp64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_group64, kThreads, sizeof(Group64Smem))
                             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_group32<false>, kThreads, sizeof(GroupSmem));
        b = a;
        if (e == cudaSuccess && !fp64)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_group32<true>, kThreads, sizeof(GroupSmem));
        if (e != cudaSuccess) return 0;
        c.store(sms * (a < b ? a : b));
    }
    return c.load();
}

cudaError_t launch_group(const WorkDev* w, int grid, int fp64, int K, int blocks, double a1, double a2, double a3, bool pad,
                         cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = fp64 ? sizeof(Group64Smem) : sizeof(GroupSmem);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;       // the CTAs of a group wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const BlockRule rule{K, a1, a2, a3};
    return cudaLaunchKernelEx(&cfg, fp64 ? k_group64 : pad ? k_group32<true> : k_group32<false>, w, blocks, rule);
}

}  // namespace hot
