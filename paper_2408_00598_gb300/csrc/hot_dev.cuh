// Device functions that the HOT kernels share: block sums, the element math of
// Steps 2-3 of Algorithm 2 (arXiv 2408.00598), and the Prop. 3 pieces of FP32
// bulk mode (hot_kernels.cu runs them as a chain of kernels, hot_group.cu inside
// one kernel per check block; the results are the same bit for bit, so every sum
// that feeds the iterates has one order, given here).
#pragma once

#include "hot_df.cuh"
#include "hot_internal.h"

#include <cstdint>
#include <type_traits>

namespace hot {

// ---------------------------------------------------------------- helpers --

// the device's clock in nanoseconds
__device__ __forceinline__ unsigned long long clock_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;\n" : "=l"(t));
    return t;
}

__device__ __forceinline__ int find_inst(const int* __restrict__ pre, int n, int t) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sh) {
    // deterministic: fixed shuffle tree, then warp partials summed in order
#pragma unroll
    for (int q = 0; q < NV; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sh[q * 32 + warp] = v[q];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            double x = lane < nw ? sh[q * 32 + lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            v[q] = x;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sh[q * 32] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = sh[q * 32];
    __syncthreads();
}

// block_sum when only the first n threads hold values: up to a warp of them the
// other warps' sums are zeros, so the first warp's is the result (the same bits)
template <int NV>
__device__ __forceinline__ void block_sum_first(double (&v)[NV], int n, double* sh) {
    if (n > 32) {
        block_sum<NV>(v, sh);
        return;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
        if (threadIdx.x == 0)
#pragma unroll
            for (int q = 0; q < NV; ++q) sh[q] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = sh[q];
}

__device__ __forceinline__ float block_max(float v, float* sh) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    float r = 0.f;
    if (threadIdx.x == 0)
        for (int q = 0; q < nw; ++q) r = fmaxf(r, sh[q]);
    __syncthreads();
    return r;  // valid in thread 0
}

__device__ __forceinline__ double sum_f64_strided(const double* p, int count, int stride) {
    double acc = 0.0;
    for (int q = 0; q < count; ++q) acc += p[q * stride];
    return acc;
}

// Column total over a slab's bands: init + p[0] + p[stride] + ... (nb terms,
// added left to right in band order), the loads issued four at a time so that
// nb bands cost about nb / 4 round trips instead of nb.
template <typename T>
__device__ __forceinline__ T sum_bands(const T* p, size_t stride, int nb, T init = T(0)) {
    T acc = init;
    for (int b0 = 0; b0 < nb; b0 += 4) {
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = b0 + u < nb ? p[(size_t)(b0 + u) * stride] : T(0);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (b0 + u < nb) acc += v[u];
    }
    return acc;
}

// deterministic block sum of NV pairs; every thread receives the totals
template <int NV>
__device__ __forceinline__ void block_sum_df(DF (&v)[NV], float2* sh) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = warp_sum_df(v[q]);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sh[q * 32 + warp] = df_st(v[q]);
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            DF x = lane < nw ? df_ld(sh[q * 32 + lane]) : DF{0.f, 0.f};
            x = warp_sum_df(x);
            if (lane == 0) sh[q * 32] = df_st(x);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = df_ld(sh[q * 32]);
    __syncthreads();
}


// ------------------------------------------------------ per-tile parameters --

struct P64 {
    double is, s, rho, trs, h;
};

// Step 4 on the delta d = v - v0 of v = x + sigma z, with v-bar - v = sigma r:
//   Halpern (Algorithm 2): d' = rho_k d + 2 rho_k sigma r, rho_k = (k+1)/(k+2);
//   generalized ADMM:      d' = d + rho sigma r          (w' = (1-rho) w + rho w-bar).
// Both are d' = rho d + trs r.
__device__ __forceinline__ P32 make_p32(double sigma, int k, double h, int gadmm = 0, double relax = 1.0) {
    P32 p{};
    p.sih = (float)(1.0 / sigma);
    p.sf = (float)sigma;
    const double rho = gadmm ? 1.0 : (k + 1.0) / (k + 2.0);
    p.rho = (float)rho;
    p.trs = (float)(gadmm ? relax * sigma : 2.0 * rho * sigma);
    p.h = (float)h;
    return p;
}
__device__ __forceinline__ P64 make_p64(double sigma, int k, double h, int gadmm = 0, double relax = 1.0) {
    P64 p;
    p.is = 1.0 / sigma;
    p.s = sigma;
    p.rho = gadmm ? 1.0 : (k + 1.0) / (k + 2.0);
    p.trs = gadmm ? relax * sigma : 2.0 * p.rho * sigma;
    p.h = h;
    return p;
}

// (x_r - x_c)^2 of two FP32 coordinates as a pair (the difference exact by a
// two-sum, its square by fma), and a product with an FP32 value as a pair:
// the objective's parts in FP32 mode with real-valued coordinates.
__device__ __forceinline__ DF cost_pair(float xr, float xc) {
    const float d = xr - xc;
    const float bv = d - xr;
    const float de = (xr - (d - bv)) + (-xc - bv);          // two-sum error of xr + (-xc)
    const float c = d * d;
    return DF{c, fmaf(d, d, -c) + 2.f * d * de};
}
__device__ __forceinline__ DF cost_times(DF c, float v) {
    const float p = c.hi * v;
    return DF{p, fmaf(c.hi, v, -p) + c.lo * v};
}

// The reduced cost g = c - alpha_r - beta_c of an element as an unevaluated
// pair (Gh, Gl), from its row piece a and column piece b.  Integer
// coordinates: Gh = h (x_r - x_c)^2 - alpha_hi - beta_hi is exact on the grid
// 2^-E, Gl = -(alpha_lo + beta_lo).  Real coordinates (pieces P_r, Q_c as
// pairs): g = P_r + Q_c - 2 h x_r x_c by two exact two-sums and the product's
// fma error.
__device__ __forceinline__ void reduced_cost(const float4& a, const float4& b, float h, int coord_real, float& Gh,
                                             float& Gl) {
    const float m2hr = -2.f * h * a.w;                       // exact
    if (coord_real) {
        // every rounding named (see hot_df.cuh)
        const float t = __fadd_rn(a.x, b.x);
        const float tb = __fsub_rn(t, a.x);
        const float te = __fadd_rn(__fsub_rn(a.x, __fsub_rn(t, tb)), __fsub_rn(b.x, tb));   // two-sum error of P_hi + Q_hi
        const float ph = __fmul_rn(m2hr, b.w);
        const float pe = fmaf(m2hr, b.w, -ph);               // exact error of the product
        Gh = __fadd_rn(t, ph);
        const float sb = __fsub_rn(Gh, t);
        const float se = __fadd_rn(__fsub_rn(t, __fsub_rn(Gh, sb)), __fsub_rn(ph, sb));      // two-sum error of t + ph
        Gl = __fadd_rn(se, __fadd_rn(__fadd_rn(te, pe), __fadd_rn(a.y, b.y)));
    } else {
        Gh = fmaf(m2hr, b.w, fmaf(a.w * a.w, h, -a.x) + fmaf(b.w * b.w, h, -b.x));
        Gl = -(a.y + b.y);
    }
}

// Element math of Steps 2-3.  Inputs: anchor u, delta d, cost cq = (r-c)^2
// (unscaled integer), the slab row/column pieces of A^T y-bar (hi, lo) and of
// dA = A^T(y-bar - y0).  Outputs: w = g - v/sigma, mg = -g and
// r = z-bar - g = max(-g, g - v/sigma), the dual residual entry.
struct E32 {
    float Gh, Gl, D, s, w, mg, r;
};
__device__ __forceinline__ E32 elem32(float u, float d, float cq, const float4& a, const float4& b, const P32& p,
                                      int coord_real = 0) {
    E32 e;
    if (coord_real) {
        reduced_cost(a, b, p.h, 1, e.Gh, e.Gl);
    } else {
        e.Gh = fmaf(cq, p.h, -a.x) - b.x;   // exact: every term is on the grid 2^-E
        e.Gl = -(a.y + b.y);
    }
    e.D = a.z + b.z;                        // A^T (y-bar - y0)
    e.s = u + d;
    e.w = fmaf(-e.s, p.sih, -e.D);          // g - v/sigma
    e.mg = -(e.Gh + e.Gl);                  // -g
    e.r = fmaxf(e.w, e.mg);
    return e;
}
// x-bar = v - sigma g = u + d + sigma dA and z-bar = max(0, 2g - v/sigma).
__device__ __forceinline__ void xz32(const E32& e, const P32& p, float& xb, float& zb) {
    zb = (e.w > e.mg) ? ((e.Gh + e.Gl) + e.w) : 0.f;
    xb = fmaf(p.sf, e.D, e.s);
}

struct E64 {
    double g, D, s, w, r;
};
__device__ __forceinline__ E64 elem64(double u, double d, double cq, double a, double b, double da, double db,
                                      const P64& p) {
    E64 e;
    e.g = cq * p.h - a - b;
    e.D = da + db;
    e.s = u + d;
    e.w = -e.D - e.s * p.is;
    e.r = fmax(e.w, -e.g);
    return e;
}
__device__ __forceinline__ void xz64(const E64& e, const P64& p, double& xb, double& zb) {
    zb = (e.w > -e.g) ? (e.g + e.w) : 0.0;
    xb = e.s + p.s * e.D;
}

template <typename T> struct VecT;
template <> struct VecT<float> {
    using type = float4;
    static constexpr int N = 4;
    __device__ static void ld(const float* p, float (&x)[4]) {
        const float4 t = __ldcs(reinterpret_cast<const float4*>(p));
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    }
    __device__ static void st(float* p, const float (&x)[4]) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(x[0], x[1], x[2], x[3]));
    }
};
template <> struct VecT<double> {
    using type = double2;
    static constexpr int N = 2;
    __device__ static void ld(const double* p, double (&x)[2]) {
        const double2 t = __ldcs(reinterpret_cast<const double2*>(p));
        x[0] = t.x; x[1] = t.y;
    }
    __device__ static void st(double* p, const double (&x)[2]) {
        __stcs(reinterpret_cast<double2*>(p), make_double2(x[0], x[1]));
    }
};

// Asynchronous global -> shared copies (16 B per thread, cached in L2 only).
// A thread waits only for its own copies (cp.async.wait_group), so a pipeline
// in which every thread reads back only what it copied needs no barrier.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16_ef(void* smem, const void* gmem, unsigned long long pol) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "l"(pol) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Rows of a P partial (see k_vec32): P1 and P2 are formed from partial sums over
// blocks of this many rows.
constexpr int kVecRows = 64;

// Pieces of A^T(y-bar - y0) in FP32 mode: per slab its row pieces (alpha),
// then its column pieces (beta), slab after slab as in ab32, 4mn per instance.
// The inputs of one piece, loaded in one round before any is computed:
//   row piece e of f1 slab j (k = e) or f2 slab k (j = e): the row sums of
//     u + d of f2 slab k row j (x) and of f1 slab j row k (y);
//   column piece e: the sigma-scaled anchor constant K2 (x), the column total
//     of the delta over the slab's bands (y.x) and on check iterations the
//     marginal entry (mu).
struct PieceIn {
    float2 a0;            // anchor piece (hi, lo)
    float2 x, y, mu;
    float2 s0, s1;        // the stage entries the piece uses (k_stage32): row pieces mvA_j, mvS_k; column pieces sy_j or sp_k
    float xc;             // bin coordinate of the piece's row or column
};
__device__ __forceinline__ void piece_slab(const HotInst& I, int q, int& slab, int& idx) {
    const int m = I.m, n = I.n;
    const int h1 = 2 * m * n;                     // pieces of the f1 half: n slabs of 2m
    if (q < h1) {
        slab = q / (2 * m);
        idx = q - slab * 2 * m;
    } else {
        const int r = q - h1, t = r / (2 * n);
        slab = n + t;
        idx = r - t * 2 * n;
    }
}
__device__ __forceinline__ PieceIn piece_in(const HotInst& I, int slab, int idx, bool check) {
    const int m = I.m, n = I.n;
    const bool f1 = slab < n;
    const int Ls = f1 ? m : n;
    PieceIn p;
    p.a0 = I.ab0_32[2 * g_row(I, slab) + idx];
    p.mu = make_float2(0.f, 0.f);
    p.xc = I.X32[g_xbase(I, slab) + (idx < Ls ? idx : idx - Ls)];
    const int L = g_L(I);
    const float2* __restrict__ sq = I.stg2;
    if (idx < Ls) {
        const float2* __restrict__ rs = I.rs2;
        const int j = f1 ? slab : idx, k = f1 ? idx : slab - n;
        p.x = rs[(size_t)n * m + (size_t)k * n + j];
        p.y = rs[(size_t)j * m + k];
        p.s0 = sq[j];                 // mvA_j
        p.s1 = sq[L + k];             // mvS_k
    } else {
        p.s0 = f1 ? sq[2 * L + slab] : sq[3 * L + slab - n];   // sy_j / sp_k
        p.s1 = make_float2(0.f, 0.f);
        const int e = idx - Ls, nb = f1 ? I.nb1 : I.nb2;
        p.x = I.K2[g_row(I, slab) + e];
        float kd = 0.f;
        kd += sum_bands(I.cs32 + g_colp(I, slab, 0) + e, (size_t)Ls, nb);
        p.y = make_float2(kd, 0.f);
        if (check) p.mu = f1 ? I.mu1f[(size_t)e * n + slab] : I.mu2f[(size_t)(slab - n) * n + e];
    }
    return p;
}

// Constants of the piece formula for the current cycle (from CycleK) and the
// cost grid 2^-E.
struct PieceK {
    DF is, imn, im, in, isim, isin;
    float grid, igrid;
};
__device__ __forceinline__ PieceK piece_consts(const HotInst& I, const CycleK& C) {
    PieceK K;
    K.is = df_ld(C.is);
    K.imn = df_ld(C.imn);
    K.im = df_ld(C.im);
    K.in = df_ld(C.in);
    K.isim = df_ld(C.isim);
    K.isin = df_ld(C.isin);
    K.igrid = (float)I.h;
    K.grid = 1.0f / K.igrid;                 // powers of two: exact
    return K;
}

// Piece idx of slab s of A^T(y-bar - y0) from its inputs and the stage sq of
// k_vec32 (Prop. 3): row pieces (idx < side) are y1(k, j) on f1 slab j row k
// and -y1(k, j) on f2 slab k row j, with
//   y1(k, j) = (R1(k, j) + mvA_j + mvS_k) / (m + n),
//   R1(k, j) = -(rowsum f1 slab j [k] - rowsum f2 slab k [j]) / sigma;
// column pieces are y2(i, j) on f1 slab j and y3(k, l) on f2 slab k (y3(m, n) = 0,
// the row dropped by eq. 7-8).  *zero is set for that last piece.
__device__ __forceinline__ DF piece_dv(const HotInst& I, const PieceK& K, int slab, int idx, const PieceIn& a,
                                      bool& zero) {
    const int m = I.m, n = I.n;
    const bool f1 = slab < n;
    const int Ls = f1 ? m : n;
    zero = false;
    if (idx < Ls) {
        const DF R1 = df_mul(df_sub(df_ld(a.x), df_ld(a.y)), K.is);
        const DF y1 = df_mul(df_add(df_add(R1, df_ld(a.s0)), df_ld(a.s1)), K.imn);
        return f1 ? y1 : df_neg(y1);
    }
    const int e = idx - Ls;
    zero = !f1 && slab == n + m - 1 && e == n - 1;
    if (zero) return DF{0.f, 0.f};
    const DF colc = f1 ? df_mul(df_ld(a.s0), df_neg(K.im)) : df_mul(df_ld(a.s0), K.in);
    const DF isc = f1 ? K.isim : K.isin;
    return df_add(df_sub(df_ld(a.x), df_mul(isc, a.y.x)), colc);
}

// The float4 the sweep reads for a piece: the full piece A^T y-bar = anchor +
// dv split into a part on the cost grid 2^-E (hi, so that c - hi_r - hi_c is
// exact in FP32) and an FP32 remainder, then dv itself, then the bin
// coordinate of the piece's row or column.  With real-valued coordinates
// (coord_real) the first two are instead the pair h x^2 - (anchor + dv), the
// piece's share of the separable cost h (x_r - x_c)^2 = h x_r^2 + h x_c^2 -
// 2 h x_r x_c less the piece itself (x^2 exact as a pair by fma; h a power of 2).
__device__ __forceinline__ float4 piece_pack(const PieceIn& a, DF dv, const PieceK& K, int coord_real) {
    const float df = df_f(dv);
    if (coord_real) {
        const float x2 = a.xc * a.xc;
        const DF hx2{x2 * K.igrid, fmaf(a.xc, a.xc, -x2) * K.igrid};
        const DF P = df_sub(hx2, df_add(DF{a.a0.x, a.a0.y}, dv));
        return make_float4(P.hi, P.lo, df, a.xc);
    }
    const float dh = rintf(df * K.grid) * K.igrid;
    return make_float4(a.a0.x + dh, a.a0.y + (df - dh), df, a.xc);
}


// The instance-wide O(m + n) stage of Prop. 3: from T1, T2, P1, P2 (k_vec32)
// the vectors
//   mvA_j = a_j/n - (1/m + 1/n) bb_j      (column part of y1-hat), j < n
//   mvS_k = r3_k/n + T3/n^2 - (m+n) y1a_k (row part of y1, times m+n), k < m
//   sy_j  = sum_k y1(k, j)                (for y2)
//   sp_k  = sum_j y1(k, j)                (for y3)
// into rows 0-3 of sq (mvA at j, mvS at k, sy at j, sp at k), with
//   a_j = (P2_j - T1_j)/sigma, bb_j = (colmu1_j - T1_j)/sigma,
//   r3_k = (rowmu2_k - T2_k)/sigma (less the dropped (m, n) entry's share at k = m-1),
//   e_k = (T2_k - P1_k)/sigma + r3_k,  s_k = (e_k + cst)/(m+n).
// Every global scalar is fixed by the two half totals F1 = sum_j T1_j = sum_k P1_k
// and F2 = sum_k T2_k = sum_j P2_j (the state summed over the f1 and f2 slabs)
// and the k = m-1 entries:
//   sum a = (F2 - F1)/sigma,  sum bb = (sum mu1 - F1)/sigma,
//   T3 = sum r3 = (sum mu2 - F2)/sigma - (dropped entry),
//   sum d_k e_k = (1/m) ((F2 - F1)/sigma + T3) + (d_last - 1/m) e_{m-1}
// (d the diagonal of W-hat: 1/m, ..., 1/m, d_last).  F1 and F2 come from the
// per-item totals of k_vec32's T items (one block reduction); every thread
// loads the k = m-1 entries itself, so the only barrier is that reduction's.
struct StageIn {
    DF T1, P2, cm;        // column quantities at j = q < n (P2 summed over its row blocks)
    DF T2, P1, rm;        // row quantities at k = q < m (P1 summed over its row blocks)
};
// sum of the row-block partials at column q of rows first, first + 1, ...
__device__ __forceinline__ DF sum_partials(const float2* __restrict__ v, int L, int first, int count, int q) {
    DF acc{0.f, 0.f};
    for (int b0 = 0; b0 < count; b0 += 4) {
        float2 pp[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            pp[u] = b0 + u < count ? __ldcg(v + (size_t)(first + b0 + u) * L + q) : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = df_add(acc, df_ld(pp[u]));
    }
    return acc;
}
__device__ __forceinline__ StageIn stage_in(const HotInst& I, int q) {
    const int m = I.m, n = I.n, L = g_L(I);
    const float2* __restrict__ v = I.vec2;
    const int r1 = (n + kVecRows - 1) / kVecRows, r2 = (m + kVecRows - 1) / kVecRows;
    StageIn s{};
    if (q < n) {
        s.T1 = df_ld(__ldcg(v + q));
        s.P2 = sum_partials(v, L, 2 + r1, r2, q);
        s.cm = df_ld(I.cm2[q]);
    }
    if (q < m) {
        s.T2 = df_ld(__ldcg(v + L + q));
        s.P1 = sum_partials(v, L, 2, r1, q);
        s.rm = df_ld(I.rm2[q]);
    }
    return s;
}

// The scalars of the stage and the constants its per-index parts use.
struct StageK {
    DF is, im, in, imn, imin, dl;             // CycleK's, as pairs
    DF drop, cst, dsiw, tin, yasum, T3in, T3in2;
    float mpn, fn;
};
// From the half totals F1, F2, the entries T2, P1 (and rm) at k = m - 1, and
// the delta's column total kdl of the dropped (m, n) row of eq. (7).
__device__ __forceinline__ StageK stage_scalars(int m, int n, const CycleK& C, DF sum_mu1, DF sum_mu2, DF F1,
                                                DF F2, DF T2l, DF P1l, DF rml, float kdl) {
    StageK K;
    K.is = df_ld(C.is);
    K.im = df_ld(C.im);
    K.in = df_ld(C.in);
    K.imn = df_ld(C.imn);
    K.imin = df_ld(C.imin);
    K.dl = df_ld(C.dl);
    const DF sumd = df_ld(C.sumd), iw = df_ld(C.iw);
    // the dropped (m, n) row of eq. (7): column n-1 of the last f2 slab
    K.drop = df_mul(df_add(df_ld(C.mk), -kdl), K.is);
    const DF dF = df_mul(df_sub(F2, F1), K.is);
    const DF suma = dF;
    const DF sumbb = df_mul(df_sub(sum_mu1, F1), K.is);
    const DF T3 = df_sub(df_mul(df_sub(sum_mu2, F2), K.is), K.drop);
    const DF R3l = df_sub(df_mul(df_sub(rml, T2l), K.is), K.drop);
    const DF el = df_add(df_mul(df_sub(T2l, P1l), K.is), R3l);
    const DF sde = df_add(df_mul(df_add(dF, T3), K.im), df_mul(el, df_sub(K.dl, K.im)));     // sum d_k e_k
    K.cst = df_add(df_sub(df_mul(suma, K.in), df_mul(sumbb, K.imin)), df_mul(T3, K.in));
    const DF ds = df_mul(df_add(sde, df_mul(K.cst, sumd)), K.imn);                          // sum d_k s_k
    K.dsiw = df_mul(ds, iw);
    const DF tsum = df_neg(df_add(ds, df_mul(K.dsiw, sumd)));                            // 1^T W-hat s
    K.tin = df_mul(tsum, K.in);
    K.yasum = df_add(tsum, df_mul(K.tin, (float)m));                                   // 1^T y1a over k < m
    K.T3in = df_mul(T3, K.in);
    K.T3in2 = df_mul(K.T3in, K.in);
    K.mpn = (float)(m + n);
    K.fn = (float)n;
    return K;
}
__device__ __forceinline__ DF stage_mvA(const StageK& K, DF T1, DF P2, DF cm) {
    const DF A = df_mul(df_sub(P2, T1), K.is);                                           // a_j
    const DF B = df_mul(df_sub(cm, T1), K.is);                                           // bb_j
    return df_sub(df_mul(A, K.in), df_mul(B, K.imin));
}
__device__ __forceinline__ DF stage_sy(const StageK& K, DF T1, DF P2, DF cm) {
    const DF A = df_mul(df_sub(P2, T1), K.is);
    const DF B = df_mul(df_sub(cm, T1), K.is);
    return df_sub(df_mul(df_add(df_sub(A, B), K.T3in), K.in), K.yasum);
}
// mvS_k and sp_k; last: k = m - 1
__device__ __forceinline__ void stage_row(const StageK& K, DF T2, DF P1, DF rm, bool last, DF& mvS, DF& sp) {
    DF R3 = df_mul(df_sub(rm, T2), K.is);                                                // r3_k
    if (last) R3 = df_sub(R3, K.drop);
    const DF e = df_add(df_mul(df_sub(T2, P1), K.is), R3);
    const DF sk = df_mul(df_add(e, K.cst), K.imn);                                       // s_k
    const DF ya = df_add(df_neg(df_mul(df_add(sk, K.dsiw), last ? K.dl : K.im)), K.tin); // y1a_k
    mvS = df_sub(df_add(df_mul(R3, K.in), K.T3in2), df_mul(ya, K.mpn));
    sp = df_sub(sk, df_mul(ya, K.fn));
}

// Every thread of the calling CTA takes part; the results are stored to sq
// (global) by the thread of each index.
__device__ __forceinline__ void alpha32_stage(const HotInst& I, float2* __restrict__ sq, float2* s_red) {
    const int m = I.m, n = I.n, L = g_L(I);
    const CycleK C = *I.cyc;
    const float2* __restrict__ v = I.vec2;
    const int r1 = (n + kVecRows - 1) / kVecRows, r2 = (m + kVecRows - 1) / kVecRows;
    const int t1 = (n + 7) / 8, t2 = (m + 7) / 8;        // T items of k_vec32
    const float2* __restrict__ tp = v + (size_t)(2 + r1 + r2) * L;
    // F1, F2 from the T items' totals (t1 + t2 <= L <= 4 * kThreads)
    DF red[2] = {DF{0.f, 0.f}, DF{0.f, 0.f}};
    for (int q = threadIdx.x; q < t1 + t2; q += blockDim.x) {
        const DF x = df_ld(__ldcg(tp + q));
        if (q < t1) red[0] = df_add(red[0], x);
        else red[1] = df_add(red[1], x);
    }
    // the k = m-1 entries (every thread), and the entries of this thread's first index
    const StageIn last = stage_in(I, m - 1);
    const int sl = g_nslab(I) - 1;
    const float kdl = sum_bands(I.cs32 + g_colp(I, sl, 0) + (n - 1), (size_t)n, I.nb2);
    const StageIn own = stage_in(I, threadIdx.x);
    block_sum_df<2>(red, s_red);
    const StageK K = stage_scalars(m, n, C, df_from(I.sum_mu1), df_from(I.sum_mu2), red[0], red[1], last.T2, last.P1, last.rm, kdl);
    const int top = m > n ? m : n;
    for (int q = threadIdx.x; q < top; q += blockDim.x) {
        const StageIn s = q == (int)threadIdx.x ? own : stage_in(I, q);
        if (q < n) {
            sq[0 * (size_t)L + q] = df_st(stage_mvA(K, s.T1, s.P2, s.cm));
            sq[2 * (size_t)L + q] = df_st(stage_sy(K, s.T1, s.P2, s.cm));
        }
        if (q < m) {
            DF mvS, sp;
            stage_row(K, s.T2, s.P1, s.rm, q == m - 1, mvS, sp);
            sq[1 * (size_t)L + q] = df_st(mvS);
            sq[3 * (size_t)L + q] = df_st(sp);
        }
    }
}

// ---------------------------------------------------------- k_marg/k_alpha --
// Prop. 3 on R' = (b - A(u + d))/sigma, the right-hand side whose solution is
// dy = y-bar - y0: with v = sigma g0 + u + d, the right-hand side of
// eq. (update:y) is R = b/sigma - A(v/sigma - c) = AA^T y0 + R'.  R' comes
// from the slab sums of u + d.  With j < n and k < m:
//   a_j = sum_k R1(k,j), bb_j = sum_i R2(i,j), r3_k = sum_l R3(k,l), T3 = sum r3,
//   y1-hat(k,j) = (R1(k,j) + a_j/n - (1/m+1/n) bb_j + r3_k/n + T3/n^2)/(m+n),
//   s_k = sum_j y1-hat(k,j),  t = W-hat s,  y1^a = t + (1^T t / n) 1,
//   y1 = y1-hat - y1^a,  y2(i,j) = (R2(i,j) - sum_k y1(k,j))/m,
//   y3(k,l) = (R3(k,l) + sum_j y1(k,j))/n.
// marg64 (one CTA) forms the O(m + n) vectors shared by all
// slabs, at mv[w * L + index], L = max(m, n):
//   w = 0: a_j / n - (1/m + 1/n) bb_j        (column part of y1-hat), j < n
//   w = 1: r3_k / n + T3 / n^2 - (m+n) y1^a_k (row part of y1, times m+n), k < m
//   w = 2: sum_k y1(k,j)                      (for y2), j < n
//   w = 3: sum_j y1(k,j)                      (for y3), k < m
// pieces64 then forms the slab's entries with products only
// (FP64 division is slow on this part; reciprocals are taken once).
// Reciprocals of a cycle (FP64 divisions take hundreds of cycles here: formed
// once by the caller).
struct Recip64 {
    double is, im, in_, imn, dl, iw;
};
__device__ __forceinline__ Recip64 recip64(int mi, int ni, double sigma) {
    const double m = mi, n = ni;
    Recip64 r;
    r.is = 1.0 / sigma;
    r.in_ = 1.0 / n;
    r.im = 1.0 / m;
    r.imn = 1.0 / (m + n);
    r.dl = (1.0 - r.in_) / (m + 1.0);
    r.iw = 1.0 / (r.im - r.dl);                    // 1/w, w = 1/m - (1-1/n)/(m+1)
    return r;
}

// The O(m + n) vectors mv of Prop. 3 in FP64 from T1, T2, P1, P2 (the first four
// of the 7 L doubles sv); cs: column partials of the delta.  One CTA.
__device__ __forceinline__ void marg64(const HotInst& I, const Recip64& R, const double* cs, double* mv, double* sv,
                                       double* s_red) {
    const int mi = I.m, ni = I.n, L = g_L(I);
    const double m = mi, n = ni;
    const double is = R.is, in_ = R.in_, im = R.im, imn = R.imn, dl = R.dl, iw = R.iw;
    double* T1 = sv;
    double* T2 = sv + L;
    double* P1 = sv + 2 * L;
    double* P2 = sv + 3 * L;
    double* cm = sv + 4 * L;
    double* rm = sv + 5 * L;
    double* ss = sv + 6 * L;
    for (int q = threadIdx.x; q < ni; q += blockDim.x) cm[q] = I.colmu1[q];
    for (int q = threadIdx.x; q < mi; q += blockDim.x) rm[q] = I.rowmu2[q];
    // the dropped (m, n) row of eq. (7): column n-1 of the last f2 slab
    const int sl = g_nslab(I) - 1;
    const double kap_last =
        sum_bands(cs + g_colp(I, sl, 0) + (ni - 1), (size_t)ni, I.nb2, I.kapa[g_row(I, sl) + (ni - 1)]);
    const double mu_last = I.mu2[(size_t)(mi - 1) * ni + (ni - 1)];
    __syncthreads();
    auto A_ = [&](int j) { return -(T1[j] - P2[j]) * is; };
    auto B_ = [&](int j) { return (cm[j] - T1[j]) * is; };
    auto R3_ = [&](int k) {
        double r = (rm[k] - T2[k]) * is;
        if (k == mi - 1) r -= (mu_last - kap_last) * is;
        return r;
    };
    double red[3] = {0.0, 0.0, 0.0}, one[1];
    for (int j = threadIdx.x; j < ni; j += blockDim.x) {
        red[0] += A_(j);
        red[1] += B_(j);
    }
    for (int k = threadIdx.x; k < mi; k += blockDim.x) red[2] += R3_(k);
    block_sum_first<3>(red, L, s_red);
    const double Asum = red[0], Bsum = red[1], T3 = red[2];
    one[0] = 0.0;
    for (int k = threadIdx.x; k < mi; k += blockDim.x) {
        const double rowR1 = -(P1[k] - T2[k]) * is;
        const double s = (rowR1 + Asum * in_ - (im + in_) * Bsum + R3_(k) + T3 * in_) * imn;   // s_k
        ss[k] = s;
        one[0] += (k == mi - 1 ? dl : im) * s;
    }
    block_sum_first<1>(one, L, s_red);
    const double ds = one[0];
    one[0] = 0.0;
    for (int k = threadIdx.x; k < mi; k += blockDim.x) {
        const double dq = (k == mi - 1 ? dl : im);
        one[0] += -dq * ss[k] - dq * ds * iw;       // 1^T W-hat s
    }
    block_sum_first<1>(one, L, s_red);
    const double tsum = one[0];
    const double yasum = tsum + m * tsum * in_;    // 1^T y1^a over k < m
    for (int k = threadIdx.x; k < mi; k += blockDim.x) {
        const double dq = (k == mi - 1 ? dl : im);
        const double ya = -dq * ss[k] - dq * ds * iw + tsum * in_;   // y1^a_k
        mv[L + k] = R3_(k) * in_ + T3 * in_ * in_ - (m + n) * ya;
        mv[3 * L + k] = ss[k] - n * ya;
    }
    for (int j = threadIdx.x; j < ni; j += blockDim.x) {
        const double aq = A_(j), bq = B_(j);
        mv[j] = aq * in_ - (im + in_) * bq;
        mv[2 * L + j] = (aq - bq + T3 * in_) * in_ - yasum;
    }
}

// The slab's pieces, in FP64: entries of dy = y-bar - y0 (dab) and of y-bar
// itself (ab) for its rows [r0, r0 + nr) and, with cols, its columns (from the
// slab's side on).  rs, cs: row sums and column partials of the delta; mv: the
// vectors of marg64.  The anchor part of R (row sums and column totals of u) is
// formed once per cycle by k_anchor.  CHECK: the slab's share of <b, y> (when it
// has the columns) and max |A^T y|.
template <bool CHECK>
__device__ __forceinline__ void pieces64(const HotInst& I, const Recip64& R, int slab, int r0, int nr, bool first,
                                         const double* __restrict__ rs, const double* __restrict__ cs,
                                         const double* __restrict__ mv, double* ab, double* dab, double* s_red,
                                         float* s_max) {
    const int mi = I.m, ni = I.n, L = g_L(I), Ls = g_side(I, slab), nb = g_nb(I, slab);
    const double is = R.is, im = R.im, in_ = R.in_, imn = R.imn;
    const double* __restrict__ R1a = I.R1a + g_row(I, slab);
    const double* __restrict__ kapa = I.kapa + g_row(I, slab);
    const double* __restrict__ ab0 = I.ab0 + 2 * g_row(I, slab);
    const size_t f2 = (size_t)ni * mi;            // first row of the f2 half
    const bool f1 = slab < ni;
    float ymax = 0.f;
    double dob = 0.0;
    // idx < Ls: alpha (row) entries, idx >= Ls: beta (column) entries; returns the full piece
    auto put = [&](int idx, double dv) -> double {
        dab[idx] = dv;
        const double full = ab0[idx] + dv;
        ab[idx] = full;
        if (CHECK) ymax = fmaxf(ymax, fabsf((float)full));
        return full;
    };
    for (int r = r0 + (int)threadIdx.x; r < r0 + nr; r += kThreads) {
        const int j = f1 ? slab : r, k = f1 ? r : slab - ni;
        const double R1 = R1a[r] - (__ldcg(rs + (size_t)j * mi + k) - __ldcg(rs + f2 + (size_t)k * ni + j)) * is;
        const double y1 = (R1 + mv[j] + mv[L + k]) * imn;              // y1(k, j)
        put(r, f1 ? y1 : -y1);                                         // A2 = -1_n^T kron I_M
    }
    const double sy = f1 ? mv[2 * L + slab] : mv[3 * L + slab - ni];
    for (int c = threadIdx.x; c < Ls; c += kThreads) {
        if (!f1 && slab == ni + mi - 1 && c == ni - 1) {
            put(Ls + c, 0.0);                                          // no row: y3(m, n) = 0
            continue;
        }
        double kd = 0.0;                                               // column total of the delta over the bands
        for (int b = 0; b < nb; ++b) kd += __ldcg(cs + g_colp(I, slab, 0) + (size_t)b * Ls + c);
        const double kap = kapa[c] + kd;
        const double mu = f1 ? I.mu1[(size_t)c * ni + slab] : I.mu2[(size_t)(slab - ni) * ni + c];
        const double full = f1 ? put(Ls + c, ((mu - kap) * is - sy) * im)       // y2(i, j)
                               : put(Ls + c, ((mu - kap) * is + sy) * in_);     // y3(k, l)
        if (CHECK) dob += mu * full;                                   // <b, y>: mu1 . y2, mu2 . y3
    }
    if (CHECK) {
        double red[1] = {dob};
        block_sum<1>(red, s_red);
        const float bm = block_max(ymax, s_max);
        if (threadIdx.x == 0) {
            if (first) I.dobj_part[slab] = red[0];
            atomicMax(&I.ctl->ymax_bits, __float_as_uint(bm));
        }
    }
}

}  // namespace hot
