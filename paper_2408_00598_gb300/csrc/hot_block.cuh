// Device functions of one CTA that hot_kernels.cu launches as kernels and
// hot_group.cu calls inside its kernels: the FP64 sweep of a tile, and the end of
// a check block (the KKT partial sums, the stopping and restart rules, the
// sigma update, the restart passes over the state, and the anchor constants of
// the new cycle).
#pragma once

#include "hot_dev.cuh"

namespace hot {

// ----------------------------------------------------------- FP64 sweep --
constexpr int kMaxTR64 = 64;               // FP64 tiles: TR <= side and TR * (longer row pitch) <= 4096
struct Sweep64Smem {
    double row[kRowSmemBytes / 8 + 256];
    double xrow[kRowSmemBytes / 8 + 256];
    double col[kThreads * 2];
    double xcol[kThreads * 2];
    double red[kNK * 32];
    double3 a[kMaxTR64];                   // per row: alpha, scaled x, dalpha
};

// a > b for doubles, on the integer pipe (FP64 comparisons run at a 64th of the
// FP32 rate, like all FP64 instructions here).  A NaN sorts by its sign bit, beyond
// the infinities: which of z-bar - g's two values stays is then arbitrary, but a
// NaN among the pieces or the state is also in x-bar = u + d + sigma D, whose
// objective the check tests (HOT_NUMERIC).
__device__ __forceinline__ bool gt64(double a, double b) {
    long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    x ^= (x >> 63) & 0x7fffffffffffffffLL;
    y ^= (y >> 63) & 0x7fffffffffffffffLL;
    return x > y;
}

// -a on the integer pipe, for the same reason
__device__ __forceinline__ double neg64(double a) {
    return __hiloint2double(__double2hiint(a) ^ 0x80000000, __double2loint(a));
}

// Steps 2-4 of Algorithm 2 on one tile (TR rows of a slab) in FP64, and the
// tile's row and column sums.  ab, dab: the slab's pieces, rows then columns.
// Bound: the FP64 pipe (2 lanes per clock and SM).  An element takes 9.5 FP64
// instructions (about 13 before): the cost h (x_r - x_c)^2 enters the reduced
// cost by one fma of the difference t, with x times 2^floor(e / 2), h = 2^e, and
// for odd e one factor doubled in its exponent; comparisons run on integers.
// (The separable form h x_r^2 - alpha + h x_c^2 - beta - 2 h x_r x_c takes 8.5, but its
// error is relative to the largest cost instead of the element's.)  FP64 pipe
// 81 % busy.  One sweep: 128 x 128 125 -> 97 us, 256 x 256 947 -> 692 us; on check
// iterations 224 -> 196 and 1,748 -> 1,456 us.
template <bool CHECK>
__device__ __forceinline__ void sweep64_tile(const HotInst& I, int slab, int band, const double* __restrict__ din_,
                                             double* __restrict__ dout_, const P64& p, const double* __restrict__ ab,
                                             const double* __restrict__ dab, double* __restrict__ rs_out,
                                             double* __restrict__ cs_out, Sweep64Smem& s) {
    constexpr int NV = 2;
    const int S = g_side(I, slab), Sp = g_pitch(I, slab), TR = I.TR;       // this slab's side and row pitch
    const int NC = Sp / NV;
    const int P = kThreads / NC;
    const int tid = threadIdx.x;
    const int cg = tid % NC, ro = tid / NC;
    const bool active = ro < P;
    const int r0 = band * TR, nr = min(S, r0 + TR) - r0;
    const size_t off = g_elem(I, slab) + (size_t)r0 * Sp;
    const double* __restrict__ u = (const double*)I.u + off;
    const double* __restrict__ din = din_ + off;
    double* __restrict__ dout = dout_ + off;
    const double* __restrict__ X = I.X64 + g_xbase(I, slab);               // bin coordinates of this half
    const int he = (__double2hiint(p.h) >> 20) - 1023;                     // h = 2^he
    const int odd = (he & 1) << 20;
    const double sc = __hiloint2double(((he >> 1) + 1023) << 20, 0);       // h = sc^2, or 2 sc^2 for odd he
    if (tid < nr) s.a[tid] = make_double3(ab[r0 + tid], X[r0 + tid] * sc, dab[r0 + tid]);
    const int c0 = cg * NV;
    const int nval = S - c0;                                               // columns inside the slab (pad after)
    double B[NV], db[NV], xc[NV], cacc[NV], xacc[NV];
#pragma unroll
    for (int e = 0; e < NV; ++e) {
        const bool v = active && e < nval;
        xc[e] = v ? X[c0 + e] * sc : 0.0;
        B[e] = v ? ab[S + c0 + e] : 0.0;
        db[e] = v ? dab[S + c0 + e] : 0.0;
        cacc[e] = xacc[e] = 0.0;
    }
    double k64[kNK] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const double nis = -p.is, rho = p.rho, trs = p.trs, sg = p.s;
    double un[NV] = {0.0, 0.0}, dn[NV] = {0.0, 0.0};
    if (active && ro < nr) {                                               // in flight across the barrier
        VecT<double>::ld(u + (size_t)ro * Sp + c0, un);
        VecT<double>::ld(din + (size_t)ro * Sp + c0, dn);
    }
    __syncthreads();
    if (active) {
        for (int r = ro; r < nr; r += P) {
            const double uu[NV] = {un[0], un[1]}, dd[NV] = {dn[0], dn[1]};
            if (r + P < nr) {                                              // the next row's loads
                VecT<double>::ld(u + (size_t)(r + P) * Sp + c0, un);
                VecT<double>::ld(din + (size_t)(r + P) * Sp + c0, dn);
            }
            const double3 a = s.a[r];
            double out[NV], xo[NV];
#pragma unroll
            for (int e = 0; e < NV; ++e) {
                const double t = a.y - xc[e];
                const double t2 = __hiloint2double(__double2hiint(t) + odd, __double2loint(t));
                const double g = fma(t2, t, -a.x) - B[e];                  // c - A^T y-bar
                const double D = a.z + db[e];                              // A^T (y-bar - y0)
                const double sv = uu[e] + dd[e];
                const double w = fma(nis, sv, -D);                         // g - v / sigma
                const double mg = neg64(g);
                const bool pos = gt64(w, mg);                              // z-bar > 0
                const double r_ = pos ? w : mg;                            // z-bar - g
                out[e] = fma(trs, r_, rho * dd[e]);
                xo[e] = 0.0;
                if (e >= nval) {
                    out[e] = 0.0;                                          // pad columns stay 0
                    continue;
                }
                if constexpr (CHECK) {
                    const double zb = pos ? g + w : 0.0, xb = fma(sg, D, sv);
                    const double mn = gt64(xb, zb) ? zb : xb;
                    const double dx = X[r0 + r] - X[c0 + e];
                    xo[e] = xb;
                    k64[0] = fma(r_, r_, k64[0]);
                    k64[1] = fma(mn, mn, k64[1]);
                    k64[2] = fma(xb, xb, k64[2]);
                    k64[3] = fma(zb, zb, k64[3]);
                    k64[4] = fma(dx * dx, xb, k64[4]);
                    xacc[e] += xb;
                }
                cacc[e] += out[e];
            }
            VecT<double>::st(dout + (size_t)r * Sp + c0, out);
            s.row[r * (NC + 1) + cg] = out[0] + out[1];
            if constexpr (CHECK) s.xrow[r * (NC + 1) + cg] = xo[0] + xo[1];
        }
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            s.col[ro * Sp + c0 + e] = cacc[e];
            if constexpr (CHECK) s.xcol[ro * Sp + c0 + e] = xacc[e];
        }
    }
    __syncthreads();
    const size_t cbase = g_colp(I, slab, band), rbase = g_row(I, slab) + r0;
    if (P < 16) {
        for (int c = tid; c < S; c += kThreads) {
            cs_out[cbase + c] = sum_f64_strided(s.col + c, P, Sp);
            if constexpr (CHECK) I.xcs_part[cbase + c] = sum_f64_strided(s.xcol + c, P, Sp);
        }
    } else {
        // short rows, many partials per column (sides up to 32): eight lanes per
        // column, as for the rows below (0.8 us of an iteration of 16 x 16)
        for (int q = tid; q < ((S * 8 + 31) & ~31); q += kThreads) {       // whole warps
            const int c = q >> 3, l = q & 7;
            double acc = 0.0, xac = 0.0;
            for (int p_ = l; c < S && p_ < P; p_ += 8) {
                acc += s.col[p_ * Sp + c];
                if constexpr (CHECK) xac += s.xcol[p_ * Sp + c];
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                acc += __shfl_down_sync(0xffffffffu, acc, o, 8);
                if constexpr (CHECK) xac += __shfl_down_sync(0xffffffffu, xac, o, 8);
            }
            if (l == 0 && c < S) {
                cs_out[cbase + c] = acc;
                if constexpr (CHECK) I.xcs_part[cbase + c] = xac;
            }
        }
    }
    // rows: eight lanes per row, each every eighth partial, then the lanes' sums
    // (one thread per row was a chain of NC dependent adds on one warp)
    for (int q = tid; q < ((nr * 8 + 31) & ~31); q += kThreads) {
        const int r = q >> 3, l = q & 7;
        double acc = 0.0, xac = 0.0;
        if (r < nr)
            for (int c = l; c < NC; c += 8) {
                acc += s.row[r * (NC + 1) + c];
                if constexpr (CHECK) xac += s.xrow[r * (NC + 1) + c];
            }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            acc += __shfl_down_sync(0xffffffffu, acc, o, 8);
            if constexpr (CHECK) xac += __shfl_down_sync(0xffffffffu, xac, o, 8);
        }
        if (l == 0 && r < nr) {
            rs_out[rbase + r] = acc;
            if constexpr (CHECK) I.xrs[rbase + r] = xac;
        }
    }
    if constexpr (CHECK) {
        block_sum<kNK>(k64, s.red);
        if (tid == 0) {
            double* o = I.tile_kkt + (size_t)g_tile(I, slab, band) * kNK;
#pragma unroll
            for (int q = 0; q < kNK; ++q) o[q] = k64[q];
        }
    }
}

// Once per cycle (after a restart, and at the start): the anchor parts of the
// right-hand side, per slab: R1a along the slab's rows and the column totals
// of u.  One CTA per slab.
__device__ __forceinline__ void anchor_slab(const HotInst& I, int slab, double sigma) {
    const int mi = I.m, ni = I.n, Ls = g_side(I, slab), nb = g_nb(I, slab);
    const double is = 1.0 / sigma;
    const size_t f2 = (size_t)ni * mi;                // first row of the f2 half
    if (!I.fp64 && slab == 0 && threadIdx.x == 0) {
        const double m = mi, n = ni;
        const double dl = (1.0 - 1.0 / n) / (m + 1.0);
        CycleK& K = *I.cyc;
        K.is = df_st(df_from(is));
        K.in = df_st(df_from(1.0 / n));
        K.im = df_st(df_from(1.0 / m));
        K.imn = df_st(df_from(1.0 / (m + n)));
        K.imin = df_st(df_from(1.0 / m + 1.0 / n));
        K.iw = df_st(df_from(1.0 / (1.0 / m - dl)));       // 1/w, w = 1/m - (1-1/n)/(m+1)
        K.dl = df_st(df_from(dl));
        K.sumd = df_st(df_from((mi - 1) / m + dl));
        K.isim = df_st(df_from(is / m));
        K.isin = df_st(df_from(is / n));
    }
    const bool last = slab == g_nslab(I) - 1;
    const size_t ro = g_row(I, slab);
    for (int q = threadIdx.x; q < Ls; q += blockDim.x) {
        // f1 slab j: rows k, R1(k, j); f2 slab k: rows j, R1(k, j)
        const int j = slab < ni ? slab : q;
        const int k = slab < ni ? q : slab - ni;
        I.R1a[ro + q] = -(I.rs0[(size_t)j * mi + k] - I.rs0[f2 + (size_t)k * ni + j]) * is;
        double kap = 0.0;
        kap += sum_bands(I.cs0_part + g_colp(I, slab, 0) + q, (size_t)Ls, nb);
        I.kapa[ro + q] = kap;
        if (!I.fp64) {
            // pairs for the FP32-mode solve: the row sums of u (also those of
            // u + d, d = 0 at the anchor); K2 is the sigma-scaled anchor part
            // of y2 (f1 slab j, column i) resp. y3 (f2 slab k, column l)
            const float2 r0 = df_st(df_from(I.rs0[ro + q]));
            I.rs02[ro + q] = r0;
            I.rs2[ro + q] = r0;
            if (last && q == ni - 1) I.cyc->mk = df_st(df_from(I.mu2[(size_t)(mi - 1) * ni + (ni - 1)] - kap));
            double k2;
            if (slab < ni) k2 = (I.mu1[(size_t)q * ni + slab] - kap) * is / mi;
            else if (last && q == ni - 1) k2 = 0.0;
            else k2 = (I.mu2[(size_t)(slab - ni) * ni + q] - kap) * is / ni;
            I.K2[ro + q] = df_st(df_from(k2));
        }
    }
}

// ---------------------------------------------------------- restart tiles --
// MODE 0: partial ||x-bar - x_r||^2, ||z-bar - z_r||^2 of the check iteration.
// MODE 1: restart at the check iteration: anchor and iterate <- w-bar, i.e.
//         v0 = x-bar + sigma_new z-bar and y0 = y-bar, stored as
//         u = v0 - sigma_new g-bar = x-bar + sigma_new r (r = z-bar - g-bar);
//         (x_r, z_r) = (x-bar, z-bar); delta = 0; FP64 slab sums of u;
//         A^T y0 pieces <- those of y-bar.
// MODE 2: x-bar of the final check iteration into x_r (the solution), and
//         (FP32 mode) the tile's share of <c, d> of that iteration, which
//         completes the reported objective (k_block_end).
// The check iteration (index K-1, odd) read delta buffer d1.
// FP32 mode streams the state through a ring of SLOTS passes per thread in
// shared memory (u and d; MODE 0 also x_r and z_r), a commit group per pass:
// more bytes in flight than registers can hold beside the double-float sums.
// 512 x 512: MODE 0 1,052 -> 886 us (4.8 TB/s of its 16 B per variable, now bound by
// the issue of its pair sums, 73 %), MODE 2 639 us, MODE 1 1,532 us: its epilogue
// adds a row's partials in one chain, whose order the iterates depend on.
constexpr int kRestartSlots = 4;
__host__ __device__ constexpr size_t restart_ring(int mode) {
    return (size_t)kRestartSlots * (mode == 0 ? 4 : 2) * kThreads * sizeof(float4);
}
template <typename T, int MODE, int SLOTS>
__device__ __forceinline__ void restart_tile(const HotInst& I, int slab, int band, double* s_row, double* s_col,
                                             double* s_red, float4* s_ring) {
    using V = VecT<T>;
    constexpr int NV = V::N;
    constexpr bool F32 = std::is_same<T, float>::value;
    const int S = g_side(I, slab), Sp = g_pitch(I, slab), TR = I.TR;   // this slab's side and row pitch
    const int NC = Sp / NV;
    const int P = kThreads / NC;
    const int cg = threadIdx.x % NC, ro = threadIdx.x / NC;
    const bool active = ro < P;
    const int r0 = band * TR, r1 = min(S, r0 + TR);
    const size_t off = g_elem(I, slab);
    T* u = (T*)I.u + off;
    const T* d1 = (const T*)I.d1 + off;
    T* d0 = (T*)I.d0 + off;
    T* xr = (T*)I.xr + off;
    T* zr = (T*)I.zr + off;
    // x-bar, z-bar need the check iteration's sigma; MODE 1 runs after
    // k_restart_sigma has replaced it (kept in sigma_old)
    const double sig_old = (MODE == 1) ? I.ctl->sigma_old : I.ctl->sigma;
    const double sig_new = I.ctl->sigma;
    const bool origin = I.ctl->restarts == 0;        // MODE 0: the reference point is still w0 = 0 (not stored)
    const int c0 = cg * NV;
    const int nval = S - c0;                         // columns inside the slab (pad columns after)
    const int cr = F32 ? I.coord_real : 0;           // real-valued coordinates: the cost term in pairs
    const int xb0 = g_xbase(I, slab);                // bin coordinates of this slab's half
    // sums that feed later iterations: FP64 (FP64 mode) or double-float (FP32 mode)
    double racc[2] = {0.0, 0.0};
    DF fr[2] = {DF{0.f, 0.f}, DF{0.f, 0.f}};
    double ccol[NV];
    DF fcol[NV];
#pragma unroll
    for (int e = 0; e < NV; ++e) {
        ccol[e] = 0.0;
        fcol[e] = DF{0.f, 0.f};
    }
    if (active) {
        // loop invariants of the tile, read once: the check iteration's
        // constants, this thread's column pieces and column coordinates, and
        // the arrays behind restrict-qualified locals (the stores below then
        // force no reloads of the descriptor)
        const P32 p32 = make_p32(sig_old, 0, I.h);
        const P64 p64 = make_p64(sig_old, 0, I.h);
        const float4* __restrict__ ab32 = F32 ? I.ab32 + 2 * g_row(I, slab) : nullptr;
        const double* __restrict__ ab64 = F32 ? nullptr : I.ab64 + 2 * g_row(I, slab);
        const double* __restrict__ dab64 = F32 ? nullptr : I.dab64 + 2 * g_row(I, slab);
        const float* __restrict__ X32 = I.X32 + xb0;
        const double* __restrict__ X64 = I.X64 + xb0;
        float4 bq[NV];
        T xc[NV], bb[NV], db[NV];
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            const bool v = e < nval;
            if constexpr (F32) {
                bq[e] = v ? ab32[S + c0 + e] : make_float4(0.f, 0.f, 0.f, 0.f);
                xc[e] = v ? X32[c0 + e] : 0.f;
            } else {
                bb[e] = v ? ab64[S + c0 + e] : 0.0;
                db[e] = v ? dab64[S + c0 + e] : 0.0;
                xc[e] = v ? X64[c0 + e] : 0.0;
            }
        }
        const float fsig = (float)sig_new;
        constexpr int NA = MODE == 0 ? 4 : 2;            // arrays in a slot
        float4* ring = s_ring + threadIdx.x;
        unsigned long long pol = 0;
        if constexpr (F32) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(pol));
        auto issue = [&](int q, int r) {                 // row r into slot q % SLOTS
            if constexpr (F32) {
                if (r < r1) {
                    const size_t o = (size_t)r * Sp + c0;
                    float4* p = ring + (q % SLOTS) * NA * kThreads;
                    cp_async16_ef(p, (const float*)u + o, pol);
                    cp_async16_ef(p + kThreads, (const float*)d1 + o, pol);
                    if (MODE == 0 && !origin) {
                        cp_async16_ef(p + 2 * kThreads, (const float*)xr + o, pol);
                        cp_async16_ef(p + 3 * kThreads, (const float*)zr + o, pol);
                    }
                }
                cp_async_commit();
            }
        };
#pragma unroll 1
        for (int q = 0; q < SLOTS - 1; ++q) issue(q, r0 + ro + q * P);
        int q = 0;
#pragma unroll 1
        for (int r = r0 + ro; r < r1; r += P, ++q) {
            T uu[NV], dd[NV], xbv[NV], zbv[NV], rv[NV];
            const float4* slot = ring + (q % SLOTS) * NA * kThreads;
            if constexpr (F32) {
                issue(q + SLOTS - 1, r + (SLOTS - 1) * P);
                cp_async_wait<SLOTS - 1>();
                const float4 a = slot[0], b = slot[kThreads];
                uu[0] = a.x, uu[1] = a.y, uu[2] = a.z, uu[3] = a.w;
                dd[0] = b.x, dd[1] = b.y, dd[2] = b.z, dd[3] = b.w;
            } else {
                V::ld(u + (size_t)r * Sp + c0, uu);
                V::ld(d1 + (size_t)r * Sp + c0, dd);
            }
            if constexpr (F32) {
                const float4 a = ab32[r];
                const float xrow = X32[r];
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    const float dc = xrow - xc[e];
                    const E32 el = elem32(uu[e], dd[e], dc * dc, a, bq[e], p32, cr);
                    xz32(el, p32, xbv[e], zbv[e]);
                    rv[e] = el.r;
                }
            } else {
                const double a = ab64[r], da = dab64[r];
                const double xrow = X64[r];
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    const double dc = xrow - xc[e];
                    const E64 el = elem64(uu[e], dd[e], dc * dc, a, bb[e], da, db[e], p64);
                    xz64(el, p64, xbv[e], zbv[e]);
                    rv[e] = el.r;
                }
            }
#pragma unroll
            for (int e = 0; e < NV; ++e)
                if (e >= nval) xbv[e] = zbv[e] = rv[e] = T(0);   // pad columns: zero in every array
            if constexpr (MODE == 0) {
                T xo[NV], zo[NV];
                if (origin) {
#pragma unroll
                    for (int e = 0; e < NV; ++e) xo[e] = zo[e] = T(0);
                } else if constexpr (F32) {
                    const float4 a = slot[2 * kThreads], b = slot[3 * kThreads];
                    xo[0] = a.x, xo[1] = a.y, xo[2] = a.z, xo[3] = a.w;
                    zo[0] = b.x, zo[1] = b.y, zo[2] = b.z, zo[3] = b.w;
                } else {
                    V::ld(xr + (size_t)r * Sp + c0, xo);
                    V::ld(zr + (size_t)r * Sp + c0, zo);
                }
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    if constexpr (F32) {
                        // (a - b)^2: the difference is exact to rounding, its square
                        // split by fma
                        const float dx = xbv[e] - xo[e], dz = zbv[e] - zo[e];
                        fr[0] = df_dot(fr[0], dx, dx);
                        fr[1] = df_dot(fr[1], dz, dz);
                    } else {
                        const double dx = xbv[e] - xo[e], dz = zbv[e] - zo[e];
                        racc[0] += dx * dx;
                        racc[1] += dz * dz;
                    }
                }
            } else if constexpr (MODE == 1) {
                // the slab sums of u enter every later right-hand side of Prop. 3,
                // where they cancel against b: FP64-level accuracy is needed
                T nu_[NV], zero[NV];
                DF rsf{0.f, 0.f};
                double rsd = 0.0;
                (void)rsd;
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    if constexpr (F32) nu_[e] = fmaf(fsig, rv[e], xbv[e]);
                    else nu_[e] = xbv[e] + sig_new * rv[e];
                    zero[e] = T(0);
                    if constexpr (F32) {
                        rsf = df_add(rsf, (float)nu_[e]);
                        fcol[e] = df_add(fcol[e], (float)nu_[e]);
                        // <c, u>: (r-c)^2 u exactly as a pair (the integer cost is exact in FP32)
                        if (cr) {
                            fr[0] = df_add(fr[0], cost_times(cost_pair(X32[r], xc[e]), (float)nu_[e]));
                        } else {
                            const float dc = X32[r] - xc[e];
                            fr[0] = df_dot(fr[0], dc * dc, (float)nu_[e]);
                        }
                    } else {
                        rsd += nu_[e];
                        ccol[e] += nu_[e];
                    }
                }
                V::st(u + (size_t)r * Sp + c0, nu_);
                V::st(xr + (size_t)r * Sp + c0, xbv);
                V::st(zr + (size_t)r * Sp + c0, zbv);
                if constexpr (!F32) V::st(d0 + (size_t)r * Sp + c0, zero);   // FP32: dzero instead
                if constexpr (F32) reinterpret_cast<float2*>(s_row)[(r - r0) * NC + cg] = df_st(rsf);
                else s_row[(r - r0) * NC + cg] = rsd;
            } else {
                V::st(xr + (size_t)r * Sp + c0, xbv);
                if constexpr (F32) {
                    // <c, d> of the final check iteration: (r-c)^2 d exactly as a pair
                    // (real-valued coordinates: the cost itself as a pair)
#pragma unroll
                    for (int e = 0; e < NV; ++e) {
                        if (e >= nval) continue;
                        if (cr) {
                            fr[0] = df_add(fr[0], cost_times(cost_pair(X32[r], xc[e]), (float)dd[e]));
                        } else {
                            const float dc = X32[r] - xc[e];
                            fr[0] = df_dot(fr[0], dc * dc, (float)dd[e]);
                        }
                    }
                }
            }
        }
    }
    // FP32 mode: the tile's sums as double-float pairs (GB300 runs FP64 at a
    // small fraction of the FP32 rate); FP64 mode: FP64
    if constexpr (MODE == 0) {
        if constexpr (F32) {
            block_sum_df<2>(fr, reinterpret_cast<float2*>(s_red));
            if (threadIdx.x == 0) {
                float2* o = reinterpret_cast<float2*>(I.rst_part) + (size_t)g_tile(I, slab, band) * 2;
                o[0] = df_st(fr[0]);
                o[1] = df_st(fr[1]);
            }
        } else {
            block_sum<2>(racc, s_red);
            if (threadIdx.x == 0) {
                double* o = I.rst_part + (size_t)g_tile(I, slab, band) * 2;
                o[0] = racc[0];
                o[1] = racc[1];
            }
        }
    } else if constexpr (MODE == 2) {
        if constexpr (F32) {
            DF cd[1] = {fr[0]};                           // <c, d> of this thread's share
            block_sum_df<1>(cd, reinterpret_cast<float2*>(s_red));
            if (threadIdx.x == 0)
                reinterpret_cast<float2*>(I.tile_kkt)[(size_t)g_tile(I, slab, band) * kNK + kNK - 1] = df_st(cd[0]);
        }
    } else if constexpr (MODE == 1) {
        if constexpr (F32) {
            DF cu[1] = {fr[0]};                           // <c, u> of this thread's share
            block_sum_df<1>(cu, reinterpret_cast<float2*>(s_red));
            if (threadIdx.x == 0) reinterpret_cast<float2*>(I.cu_part)[g_tile(I, slab, band)] = df_st(cu[0]);
        }
        __syncthreads();
        if (active)
#pragma unroll
            for (int e = 0; e < NV; ++e) {
                if constexpr (F32) reinterpret_cast<float2*>(s_col)[ro * Sp + c0 + e] = df_st(fcol[e]);
                else s_col[ro * Sp + c0 + e] = ccol[e];
            }
        __syncthreads();
        const size_t cbase = g_colp(I, slab, band);
        for (int c = threadIdx.x; c < S; c += blockDim.x) {
            if constexpr (F32) {
                const float2* sc = reinterpret_cast<const float2*>(s_col) + c;
                DF a{0.f, 0.f};
                for (int q = 0; q < P; ++q) a = df_add(a, df_ld(sc[(size_t)q * Sp]));
                I.cs0_part[cbase + c] = df_val(a);
            } else {
                I.cs0_part[cbase + c] = sum_f64_strided(s_col + c, P, Sp);
            }
            I.cs_part[cbase + c] = 0.0;
            I.cs32[cbase + c] = 0.f;
        }
        // y0 <- y-bar: A^T y0 pieces of this tile's rows (and, for band 0, columns)
        const size_t o = 2 * g_row(I, slab);
        const double ih = 1.0 / I.h;                         // a power of two: exact
        auto set_anchor = [&](int idx) {
            const double a0 = I.ab0[o + idx] + (F32 ? df_val(df_ld(I.dab2[o + idx])) : I.dab64[o + idx]);
            I.ab0[o + idx] = a0;
            if (I.ab0_32) {
                // integer coordinates: hi on the grid 2^-E (the reduced cost is then
                // exact in FP32); real ones form it in pairs and take a plain
                // double-float split, whose lo part keeps 2^-24 of hi, not of 2^-E
                const double hi = I.coord_real ? (double)(float)a0 : rint(a0 * ih) * I.h;
                I.ab0_32[o + idx] = make_float2((float)hi, (float)(a0 - hi));
            }
        };
        for (int rr = threadIdx.x; rr < r1 - r0; rr += blockDim.x) {
            if constexpr (F32) {
                const float2* sr = reinterpret_cast<const float2*>(s_row) + (size_t)rr * NC;
                DF a{0.f, 0.f};
                for (int q = 0; q < NC; ++q) a = df_add(a, df_ld(sr[q]));
                I.rs0[g_row(I, slab) + r0 + rr] = df_val(a);
            } else {
                I.rs0[g_row(I, slab) + r0 + rr] = sum_f64_strided(s_row + rr * NC, NC, 1);
            }
            if (!F32) I.rs[g_row(I, slab) + r0 + rr] = 0.0;      // FP32: k_anchor resets rs2
            set_anchor(r0 + rr);
        }
        if (band == 0)
            for (int c = threadIdx.x; c < S; c += blockDim.x) set_anchor(S + c);
    }
}

// Chunk cl of the objective's parts of the check iteration, for an instance
// that k_group32 runs (k_alpha32<true> forms them in the chain): partial <b, y>
// and <c, A^T(y-bar - y0)> and max |A^T y|, from the pairs in dab2, in
// k_alpha32's order.
__device__ __forceinline__ void objective_chunk(const HotInst& I, int cl, float2* s_red, float* s_max) {
    const int m = I.m, n = I.n, npieces = 4 * m * n;
    float ymax = 0.f;
    DF dob{0.f, 0.f}, cdd{0.f, 0.f};
#pragma unroll
    for (int u = 0; u < kAPT; ++u) {
        const int q = cl * kAlphaChunk + u * kThreads + (int)threadIdx.x;
        if (q >= npieces) continue;
        int slab, idx;
        piece_slab(I, q, slab, idx);
        const bool f1 = slab < n;
        const int Ls = f1 ? m : n;
        const size_t o = 2 * g_row(I, slab) + idx;
        const float2 a0 = I.ab0_32[o];
        const DF dv = df_ld(I.dab2[o]);
        const bool col = idx >= Ls;
        const bool zero = !f1 && slab == n + m - 1 && idx - Ls == n - 1;
        const DF full = df_add(DF{a0.x, a0.y}, dv);
        ymax = fmaxf(ymax, fabsf(full.hi));
        const int e = col ? idx - Ls : idx;
        cdd = df_add(cdd, df_mul(dv, df_ld(I.csum2[g_xbase(I, slab) + e])));
        if (col && !zero) {
            const float2 mu = f1 ? I.mu1f[(size_t)e * n + slab] : I.mu2f[(size_t)(slab - n) * n + e];
            dob = df_add(dob, df_mul(df_ld(mu), full));
        }
    }
    DF red[2] = {dob, cdd};
    block_sum_df<2>(red, s_red);
    const float bm = block_max(ymax, s_max);
    if (threadIdx.x == 0) {
        reinterpret_cast<float2*>(I.dobj_part)[cl] = df_st(red[0]);
        reinterpret_cast<float2*>(I.cD_part)[cl] = df_st(red[1]);
        atomicMax(&I.ctl->ymax_bits, __float_as_uint(bm));
    }
}

// Chunk `chunk` (kThreads rows) of the partial sums of ||A x-bar - b||^2 from the
// x-bar slab sums.
template <bool F32>
__device__ __forceinline__ void residual_chunk(const HotInst& I, int chunk, double* s_red) {
    const int m = I.m, n = I.n;
    const int MN = m * n;
    const int q = chunk * kThreads + threadIdx.x;
    double res = 0.0;
    if (q < 3 * MN - 1) {
        if (q < MN) {                                  // conservation rows (k, j)
            const int j = q / m, k = q % m;
            res = I.xrs[(size_t)j * m + k] - I.xrs[(size_t)MN + (size_t)k * n + j];
        } else if (q < 2 * MN) {                       // mu1 rows (i, j)
            const int j = (q - MN) / m, i = (q - MN) % m;
            double kap = 0.0;
            kap += sum_bands(I.xcs_part + g_colp(I, j, 0) + i, (size_t)m, I.nb1);
            res = kap - I.mu1[(size_t)i * n + j];
        } else {                                       // mu2 rows (k, l), the last one dropped
            const int k = (q - 2 * MN) / n, l = (q - 2 * MN) % n;
            double kap = 0.0;
            kap += sum_bands(I.xcs_part + g_colp(I, n + k, 0) + l, (size_t)n, I.nb2);
            res = kap - I.mu2[(size_t)k * n + l];
        }
    }
    if constexpr (F32) {
        const DF r = df_from(res);
        DF v[1] = {df_mul(r, r)};
        block_sum_df<1>(v, reinterpret_cast<float2*>(s_red));
        if (threadIdx.x == 0) reinterpret_cast<float2*>(I.k1_part)[chunk] = df_st(v[0]);
    } else {
        double v[1] = {res * res};
        block_sum<1>(v, s_red);
        if (threadIdx.x == 0) I.k1_part[chunk] = v[0];
    }
}

// Chunk `chunk` (kThreads tiles) of the check sweep's KKT sums and of <c, u>
// (FP32 mode): one pair each, so that k_check, a single CTA, adds few (512 x 512,
// 16,384 tiles: 24 us; 20 us at 256 x 256 before, 11 now).
__device__ __forceinline__ void tile_chunk(const HotInst& I, int chunk, float2* s_red) {
    const int t = chunk * kThreads + (int)threadIdx.x;
    const bool in = t < g_ntiles(I);
    const float2* tk = reinterpret_cast<const float2*>(I.tile_kkt) + (size_t)t * kNK;
    const float2 z = make_float2(0.f, 0.f);
    DF v[kNK];
#pragma unroll
    for (int e = 0; e < kNK - 1; ++e) v[e] = df_ld(in ? tk[e] : z);
    v[kNK - 1] = df_ld(in ? reinterpret_cast<const float2*>(I.cu_part)[t] : z);
    block_sum_df<kNK>(v, s_red);
    if (threadIdx.x == 0)
#pragma unroll
        for (int e = 0; e < kNK; ++e) I.kc_part[chunk * kNK + e] = df_st(v[e]);
}

// Sum of count pairs p[0], p[stride], ... of this thread's share (q = threadIdx.x,
// q + blockDim.x, ...), the loads issued four at a time.
__device__ __forceinline__ DF sum_pairs(const float2* __restrict__ p, int count, int stride) {
    DF acc{0.f, 0.f};
    for (int q0 = threadIdx.x; q0 < count; q0 += 4 * blockDim.x) {
        float2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u * blockDim.x;
            v[u] = q < count ? p[(size_t)q * stride] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = df_add(acc, df_ld(v[u]));
    }
    return acc;
}

// Stopping rule eq. (kkt_res) and the restart rule of instance i, one CTA.
template <bool F32>
__device__ __forceinline__ void check_instance(const HotInst& I, const WorkDev* W, int i, int K, double a1, double a2,
                                               double a3, double* s_red) {
    HotCtl* C = I.ctl;
    const int ntile = g_ntiles(I), nslab = g_nslab(I);
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if constexpr (F32) {
        // eight sums of pairs, a warp each: the check sweep's KKT sums (0-3) and
        // <c, u> (7) per chunk of tiles, k_alpha32's <c, A^T(y-bar - y0)> (4) and
        // <b, y> (6) per chunk, and the ||A x - b||^2 chunks (5); the objective's
        // <c, d> share is added when the instance ends.  (Short code: it runs
        // once a block, from cold instruction caches, while the grid waits.)
        float2* sh = reinterpret_cast<float2*>(s_red);
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const bool tile = w < 4 || w == 7;
        const float2* p = tile ? I.kc_part + (w < 4 ? w : 4)
                               : reinterpret_cast<const float2*>(w == 4 ? I.cD_part : w == 5 ? I.k1_part : I.dobj_part);
        const int count = tile ? I.n_kc : w == 5 ? I.n_k1 : I.n_achunk, stride = tile ? kNK : 1;
        DF acc{0.f, 0.f};
#pragma unroll 1
        for (int q0 = lane; q0 < count; q0 += 4 * 32) {
            float2 t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                t[u] = q0 + u * 32 < count ? p[(size_t)(q0 + u * 32) * stride] : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc = df_add(acc, df_ld(t[u]));
        }
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) acc = df_add(acc, df_shfl_down(acc, o));
        if (lane == 0) sh[w] = df_st(acc);
        __syncthreads();
        const double mine = df_val(df_ld(sh[threadIdx.x & 7])) * ((threadIdx.x & 7) == 4 ? C->sigma : 1.0);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __shfl_sync(0xffffffffu, mine, e);
    } else {
        for (int q = threadIdx.x; q < ntile; q += blockDim.x)
            for (int e = 0; e < kNK; ++e) v[e] += I.tile_kkt[(size_t)q * kNK + e];
        for (int q = threadIdx.x; q < I.n_k1; q += blockDim.x) v[5] += I.k1_part[q];
        // partial sums of <b, y>: one per slab
        for (int q = threadIdx.x; q < nslab; q += blockDim.x) v[6] += I.dobj_part[q];
        block_sum<8>(v, s_red);
    }
    // FP32 mode: <c, x-bar> = <c, u> + <c, d> + sigma <c, A^T(y-bar - y0)>
    // from exact per-tile and per-slab parts (the per-element x-bar is
    // rounded where u + d nearly cancels); <c, d> joins at the end
    // (restart pass MODE 2, k_block_end)
    if (threadIdx.x >= 32) return;
    // the roots and quotients side by side in the first warp: one square root
    // and one division of FP64 instead of seven and three
    const int lane = threadIdx.x;
    const double root = sqrt(lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2] : lane == 3 ? v[3] : lane == 4 ? v[5] : C->sigma);
    auto from = [](double x, int l) { return __shfl_sync(0xffffffffu, x, l); };
    const double nr = from(root, 0), nmn = from(root, 1), nx = from(root, 2), nz = from(root, 3), nax = from(root, 4),
                 nsig = from(root, 5);
    const double quot = (lane == 0 ? nr : lane == 1 ? nmn : nax) /
                        (lane == 0 ? 1.0 + I.norm_c : lane == 1 ? 1.0 + nx + nz : 1.0 + I.norm_b);
    const double rel_dual = from(quot, 0), rel_comp = from(quot, 1), rel_primal = from(quot, 2);
    if (lane == 0) {
        const double cx = v[4] + v[7], dob = v[6];
        const double scale = 1.0 / I.h;
        const double rel = fmax(rel_dual, fmax(rel_comp, rel_primal));
        const double absk = fmax(nr, fmax(nmn, nax));      // Table VI
        C->abs_kkt = absk;
        C->rel_dual = rel_dual;
        C->rel_comp = rel_comp;
        C->rel_primal = rel_primal;
        C->rel_kkt = rel;
        C->pobj = cx;                 // sum (r-c)^2 x-bar: unscaled <c, x-bar>
        C->dzero = 0;                 // this block's first sweep has read it
        C->dobj = dob * scale;
        const long long total = C->total + K;
        const int kcheck = C->k + K - 1;
        C->total = total;
        int fin = 0;
        if (!(rel == rel) || isinf(rel) || !(cx == cx) || isinf(cx)) {
            C->status = ST_NUMERIC;
            fin = 1;
        } else if (C->cancel) {
            C->status = ST_CANCELLED;
            fin = 1;
        } else if ((I.stop_abs ? absk : rel) <= C->tol) {
            C->status = ST_CONVERGED;
            fin = 1;
        } else if (total >= C->max_iter) {
            C->status = ST_CAPPED;
            fin = 1;
        } else {
            const double r = nsig * nr;     // ||w - w-bar||_M = sqrt(sigma) ||z-bar - g||
            C->res_norm = r;
            if (C->r0 < 0.0) C->r0 = r;
            const bool rs = (r <= a1 * C->r0) || (C->rprev >= 0.0 && r <= a2 * C->r0 && r > C->rprev) ||
                            ((double)kcheck >= a3 * (double)total);
            C->rprev = r;
            if (rs) C->restart_pending = 1;
            else C->k = C->k + K;
        }
        if (fin) {
            C->t_end = clock_ns();
            C->just_finished = 1;
            atomicSub(W->n_running, 1);
        }
        W->st_out[i] = C->status;
    }
}

// Sigma update at a restart: sigma <- sqrt(sigma ||x-bar - x_r|| / ||z-bar - z_r||) on the grid 2^(j/16).
template <bool F32>
__device__ __forceinline__ void sigma_instance(const HotInst& I, double* s_red) {
    HotCtl* C = I.ctl;
    const int ntile = g_ntiles(I);
    double v[2] = {0.0, 0.0};
    if constexpr (F32) {
        const float2* rp = reinterpret_cast<const float2*>(I.rst_part);
        DF w[2] = {sum_pairs(rp, ntile, 2), sum_pairs(rp + 1, ntile, 2)};
        block_sum_df<2>(w, reinterpret_cast<float2*>(s_red));
        v[0] = df_val(w[0]);
        v[1] = df_val(w[1]);
    } else {
        for (int q = threadIdx.x; q < ntile; q += blockDim.x) {
            v[0] += I.rst_part[(size_t)q * 2];
            v[1] += I.rst_part[(size_t)q * 2 + 1];
        }
        block_sum<2>(v, s_red);
    }
    if (threadIdx.x == 0) {
        const double dx = sqrt(v[0]), dz = sqrt(v[1]);
        const double old = C->sigma;
        C->dx2 = v[0];
        C->dz2 = v[1];
        C->sigma_old = old;
        // geometric mean of the old sigma and the movement ratio, rounded
        // to the grid 2^(j/16) (so rounding noise in dx, dz does not move it)
        if (dx > 0.0 && dz > 0.0 && isfinite(dx / dz)) C->sigma = exp2(rint(log2(sqrt(old * (dx / dz))) * 16.0) / 16.0);
        C->k = 0;
        C->r0 = -1.0;
        C->rprev = -1.0;
        C->restarts += 1;
        if constexpr (F32) C->dzero = 1;   // MODE 1 stores no zero delta; the next first sweep reads none
    }
}

// End of a block of one instance: an FP32 instance that finished in it adds the
// <c, d> share of its final check iteration (per-tile pairs from the restart
// pass MODE 2, summed in tile order) to its objective; the flags reset.
__device__ __forceinline__ void end_instance(const HotInst& I, float2* s_red) {
    HotCtl* C = I.ctl;
    if (C->just_finished && !I.fp64) {                    // block-uniform
        DF cd[1] = {sum_pairs(reinterpret_cast<const float2*>(I.tile_kkt) + (kNK - 1), g_ntiles(I), kNK)};
        block_sum_df<1>(cd, s_red);
        if (threadIdx.x == 0) C->pobj += df_val(cd[0]);
    }
    if (threadIdx.x == 0) {
        C->restart_pending = 0;
        C->just_finished = 0;
    }
}

}  // namespace hot
