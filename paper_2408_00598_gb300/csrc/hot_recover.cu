// Algorithm 1 of arXiv 2408.00598 on the GPU: the transport plan from the
// reduced-model flows, one intermediate node (k, j) per warp ("parallelise the
// (k, j) loop", Remark after Prop. 1).
//
// For node (k, j), Algorithm 1's inner loops (i = 1..m, then l = 1..n, move
// min(f1_{i,k,j}, f2_{k,j,l}) and subtract it from both) are the north-west-
// corner coupling of the sources a_i = f1_{i,k,j} with the sinks
// b_l = f2_{k,j,l}: with exclusive prefix sums A_i, B_l, the mass moved from i
// to l is the overlap of [A_i, A_{i+1}) and [B_l, B_{l+1}), and mass beyond
// min(sum a, sum b) is left unassigned exactly as the sequential loop leaves
// it.  In FP64 mode each lane takes a set of sources i, finds its first sink by
// binary search and walks forward; FP32 mode merges the ends of the two
// sides.  Entries are written in (node, i, l) order.
// Flows are clipped at 0 first (an approximate solution may have small
// negative entries).  In the slab layout both a and b are contiguous rows:
// a = row k of f1 slab j (m sources i), b = row j of f2 slab k (n sinks l).
// A plan entry runs from source bin (i, j), index i n + j of mu, to target bin
// (k, l), index k n + l of nu.
#include "hot_engine.h"
#include "hot_df.cuh"

namespace hot {

constexpr int kRecWarps = 8;

// k_recover_df's arrays in shared memory have one unused entry after every
// eight: its lanes work on runs of consecutive entries (eight at a side of
// 256), which would otherwise start in the same banks.
__host__ __device__ constexpr int pidx(int i) { return i + (i >> 3); }
// shared memory of one warp in k_recover_df, in floats: the pairs A (m + 1) and
// B (n + 1) and the entries' indices (16 bits each), to an even count
__host__ __device__ constexpr size_t recover_df_words(int m, int n) {
    return (2 * ((size_t)pidx(m) + 1) + 2 * ((size_t)pidx(n) + 1) + (m + 1) / 2 + (n + 1) / 2 + 1) & ~(size_t)1;
}
// longest walk (m + n - 1 merge steps) whose directions fit 32 bits per lane
constexpr int kPathSteps = 32 * 32;
// the same for k_recover, in doubles
__host__ __device__ constexpr size_t recover_words(int m, int n) { return 2 * ((size_t)m + n) + 2; }

// first entries of f1 row k of slab j and of f2 row j of slab k; a slab's
// rows are stored at a pitch of its side rounded up to a multiple of 4
__host__ __device__ constexpr int row_pitch(int side) { return (side + 3) & ~3; }
__device__ __forceinline__ size_t node_row_a(int m, int k, int j) { return ((size_t)j * m + k) * row_pitch(m); }
__device__ __forceinline__ size_t node_row_b(int m, int n, int k, int j) {
    return (size_t)n * m * row_pitch(m) + ((size_t)k * n + j) * row_pitch(n);
}

template <typename T>
__device__ __forceinline__ void load_node(const T* __restrict__ x, int m, int n, int k, int j, double* a, double* b,
                                          double* A, double* B) {
    const int lane = threadIdx.x & 31;
    const T* ra = x + node_row_a(m, k, j);
    const T* rb = x + node_row_b(m, n, k, j);
    for (int t = lane; t < m; t += 32) a[t] = fmax((double)ra[t], 0.0);
    for (int t = lane; t < n; t += 32) b[t] = fmax((double)rb[t], 0.0);
    __syncwarp();
    // exclusive prefix sums, sequential per 32-chunk with a warp scan (FP64);
    // a tree scan's partial sums need not be ordered to the last bit, so a
    // running maximum keeps A and B non-decreasing (the walk relies on it)
    double carryA = 0.0, carryB = 0.0, runA = 0.0, runB = 0.0;
    const int L = m > n ? m : n;
    for (int base = 0; base < L; base += 32) {
        const int t = base + lane;
        double va = t < m ? a[t] : 0.0, vb = t < n ? b[t] : 0.0;
        double sa = va, sb = vb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double ya = __shfl_up_sync(0xffffffffu, sa, o);
            const double yb = __shfl_up_sync(0xffffffffu, sb, o);
            if (lane >= o) {
                sa += ya;
                sb += yb;
            }
        }
        double ea = fmax(carryA + sa - va, runA), eb = fmax(carryB + sb - vb, runB);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double ya = __shfl_up_sync(0xffffffffu, ea, o);
            const double yb = __shfl_up_sync(0xffffffffu, eb, o);
            if (lane >= o) {
                ea = fmax(ea, ya);
                eb = fmax(eb, yb);
            }
        }
        if (t < m) A[t] = ea;
        if (t < n) B[t] = eb;
        runA = __shfl_sync(0xffffffffu, ea, 31);
        runB = __shfl_sync(0xffffffffu, eb, 31);
        carryA += __shfl_sync(0xffffffffu, sa, 31);
        carryB += __shfl_sync(0xffffffffu, sb, 31);
    }
    if (lane == 0) {
        A[m] = fmax(carryA, runA);
        B[n] = fmax(carryB, runB);
    }
    __syncwarp();
}

// number of sinks (of n) overlapping source i (and optionally write them)
__device__ __forceinline__ int node_source(int n, int i, const double* A, const double* B, const double* a,
                                           const double* b, int32_t* src, int32_t* dst, double* mass, size_t pos,
                                           int src_id, int node_k) {
    if (!(a[i] > 0.0)) return 0;             // the loops move nothing out of an empty source
    const double lo = A[i];
    const double hi = fmin(A[i + 1], B[n]);
    if (!(hi > lo)) return 0;
    // first l with B[l+1] > lo
    int l0 = 0, l1 = n - 1;
    while (l0 < l1) {
        const int mid = (l0 + l1) >> 1;
        if (B[mid + 1] > lo) l1 = mid; else l0 = mid + 1;
    }
    int cnt = 0;
    for (int l = l0; l < n && B[l] < hi; ++l) {
        const double p = fmin(hi, B[l + 1]) - fmax(lo, B[l]);
        if (p > 0.0 && b[l] > 0.0) {
            if (src) {
                src[pos + cnt] = src_id;
                dst[pos + cnt] = node_k * n + l;
                mass[pos + cnt] = p;
            }
            ++cnt;
        }
    }
    return cnt;
}

template <typename T>
__global__ void __launch_bounds__(kRecWarps * 32) k_recover(const T* __restrict__ x, int m, int n, int count_only,
                                                            int* __restrict__ counts,
                                                            const long long* __restrict__ offs,
                                                            int32_t* __restrict__ src, int32_t* __restrict__ dst,
                                                            double* __restrict__ mass, double* __restrict__ marg1,
                                                            double* __restrict__ marg2) {
    extern __shared__ double sh[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = blockDim.x >> 5;
    double* a = sh + (size_t)warp * recover_words(m, n);
    double* b = a + m;
    double* A = b + n;
    double* B = A + m + 1;
    const int nodes = m * n;
    for (int node = blockIdx.x * nw + warp; node < nodes; node += gridDim.x * nw) {
        const int k = node / n, j = node % n;    // k-major node order
        load_node(x, m, n, k, j, a, b, A, B);
        if (count_only) {
            int c = 0;
            for (int i = lane; i < m; i += 32) c += node_source(n, i, A, B, a, b, nullptr, nullptr, nullptr, 0, 0, k);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
            if (lane == 0) counts[node] = c;
            // marginals of the plan: source (i, j) gets min(a_i, max(0, Btot - A_i)),
            // target (k, l) gets min(b_l, max(0, Atot - B_l))
            for (int t = lane; t < m; t += 32) {
                const double ga = fmin(a[t], fmax(0.0, B[n] - A[t]));
                if (ga > 0.0) atomicAdd(&marg1[(size_t)t * n + j], ga);
            }
            for (int t = lane; t < n; t += 32) {
                const double gb = fmin(b[t], fmax(0.0, A[m] - B[t]));
                if (gb > 0.0) atomicAdd(&marg2[(size_t)k * n + t], gb);
            }
        } else {
            long long pos = offs[node];
            for (int base = 0; base < m; base += 32) {
                const int i = base + lane;
                int c = 0;
                if (i < m) c = node_source(n, i, A, B, a, b, nullptr, nullptr, nullptr, 0, 0, k);
                int incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (i < m && c > 0)
                    node_source(n, i, A, B, a, b, src, dst, mass, (size_t)(pos + incl - c), i * n + j, k);
                pos += __shfl_sync(0xffffffffu, incl, 31);
            }
        }
        __syncwarp();
    }
}

// FP32 bulk mode: the same node procedure with the prefix sums, comparisons
// and overlaps of the FP32 flows in double-float pairs (FP64 arithmetic runs
// at a small fraction of the FP32 rate on this part; a pair holds the sum of
// FP32 values to about 48 bits, as a running FP64 sum of them does).
__device__ __forceinline__ bool df_lt(DF a, DF b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ DF df_min(DF a, DF b) { return df_lt(b, a) ? b : a; }
__device__ __forceinline__ DF df_max(DF a, DF b) { return df_lt(a, b) ? b : a; }
__device__ __forceinline__ bool df_pos(DF a) { return a.hi > 0.f || (a.hi == 0.f && a.lo > 0.f); }
__device__ __forceinline__ DF df_shfl_up(DF a, int o) {
    return DF{__shfl_up_sync(0xffffffffu, a.hi, o), __shfl_up_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ DF df_shfl(DF a, int l) {
    return DF{__shfl_sync(0xffffffffu, a.hi, l), __shfl_sync(0xffffffffu, a.lo, l)};
}

// One side of a node: the places of the positive flows of ra[0, m) into ix, in
// order (a converged solution has about a third; the others hold no mass and
// take no entry), and their exclusive prefix sums into A (which first holds the
// flows themselves), the total into A[count].  A lane takes a run of consecutive entries: its own prefix
// sums first, then a warp scan of the runs' totals, then the sums shifted by
// the run's offset.  Prefix sums of positive entries never decrease, but sums
// rounded in different orders could by an ulp; the offsets pass through a
// running maximum and a run's sums are kept between its offset and the next,
// since the merge below relies on the order.  Returns the count.
__device__ __forceinline__ int load_side_df(const float* __restrict__ ra, int m, unsigned short* ix, float2* A) {
    const int lane = threadIdx.x & 31;
    int cnt = 0;
    for (int base = 0; base < m; base += 128) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = base + u * 32 + lane;
            v[u] = t < m ? __ldg(ra + t) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned mask = __ballot_sync(0xffffffffu, v[u] > 0.f);
            if (v[u] > 0.f) {
                const int at = cnt + __popc(mask & ((1u << lane) - 1u));
                A[pidx(at)].x = v[u];
                ix[at] = (unsigned short)(base + u * 32 + lane);
            }
            cnt += __popc(mask);
        }
    }
    __syncwarp();
    const int per = (cnt + 31) >> 5, i0 = min(cnt, lane * per), i1 = min(cnt, i0 + per);
    DF s{0.f, 0.f};
    for (int i = i0; i < i1; ++i) {
        const float v = A[pidx(i)].x;
        A[pidx(i)] = df_st(s);
        s = df_add(s, v);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const DF y = df_shfl_up(s, o);
        if (lane >= o) s = df_add(s, y);
    }
    DF off = df_shfl_up(s, 1);
    if (lane == 0) off = DF{0.f, 0.f};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const DF y = df_shfl_up(off, o);
        if (lane >= o) off = df_max(off, y);
    }
    const DF total = df_max(df_shfl(s, 31), df_shfl(off, 31));
    DF next = DF{__shfl_down_sync(0xffffffffu, off.hi, 1), __shfl_down_sync(0xffffffffu, off.lo, 1)};
    if (lane == 31) next = total;
    DF prev = off;
    for (int i = i0; i < i1; ++i) {
        prev = df_min(df_max(df_add(off, df_ld(A[pidx(i)])), prev), next);
        A[pidx(i)] = df_st(prev);
    }
    if (lane == 0) A[pidx(cnt)] = df_st(total);
    __syncwarp();
    return cnt;
}

// A pair as a double (df_val).  The conversions are written out in integers
// for normal numbers: FP64 instructions run at a 64th of the FP32 rate here, and
// the conversions would be two of the three.
__device__ __forceinline__ double f2d(float x) {
    const unsigned u = __float_as_uint(x), ex = (u >> 23) & 0xffu;
    if (ex == 0u || ex == 255u) return ex == 0u && (u << 1) == 0u ? 0.0 : (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double df_dbl(DF a) { return a.lo == 0.f ? f2d(a.hi) : f2d(a.hi) + f2d(a.lo); }

// Adds a side's share of the plan's marginals: min(a_t, max(0, other - A_t)),
// other the other side's total; the flows a are read again (ra).
__device__ __forceinline__ void side_marginal(double* __restrict__ marg, int cnt, const float* __restrict__ ra,
                                              const unsigned short* ix, const float2* A, DF other) {
    for (int t = threadIdx.x & 31; t < cnt; t += 32) {
        const int i = ix[t];
        const float a = __ldg(ra + i);
        double g = f2d(a);                                   // all of it, up to the entry that `other` cuts
        if (df_lt(other, df_ld(A[pidx(t + 1)]))) {
            DF r = df_sub(other, df_ld(A[pidx(t)]));
            if (!df_pos(r)) r = DF{0.f, 0.f};
            g = df_dbl(df_min(DF{a, 0.f}, r));
        }
        if (g > 0.0) atomicAdd(marg + i, g);
    }
}

// The node's coupling as a merge of the source ends A[1..m] with the sink
// ends B[1..n] (ties: source first).  After the first d merged ends the walk
// stands at source p, sink q = d - p; the step from there moves the overlap
// min(A[p+1], B[q+1]) - max(A[p], B[q]) from source p to sink q (an entry
// when positive and both the source and the sink hold mass) and passes the
// nearer end, which is the next step's max(A[p], B[q]).  These are the pairs
// and masses of the north-west-corner loops of Algorithm 1, in (i, l) order.
// A lane takes a contiguous range of steps and finds its start by a binary
// search on the merge diagonal (merge path), so a node costs about log2(m + n)
// + (m + n)/32 steps per lane.
__device__ __forceinline__ int merge_split(const float2* A, const float2* B, int m, int n, int d) {
    int lo = d - n > 0 ? d - n : 0, hi = d < m ? d : m;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        // source end mid + 1 is among the first d ends iff it is <= sink end d - mid
        if (!df_lt(df_ld(B[pidx(d - mid)]), df_ld(A[pidx(mid + 1)]))) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// A lane's steps [d0, d1): bit t of the result is set where step d0 + t passes a
// source's end (steps past the end of a side: 0).  COUNT: the entries are counted
// into c.
template <bool COUNT, class BITS>
__device__ __forceinline__ BITS merge_walk(const float2* A, const float2* B, int ca, int cb, int d0, int d1, int& c) {
    BITS bits = 0;
    if (d0 >= d1) return bits;
    int p = merge_split(A, B, ca, cb, d0), q = d0 - p;
    if (p >= ca || q >= cb) return bits;
    DF ae = df_ld(A[pidx(p + 1)]), be = df_ld(B[pidx(q + 1)]);
    DF prev = COUNT ? df_max(df_ld(A[pidx(p)]), df_ld(B[pidx(q)])) : DF{0.f, 0.f};
    BITS bit = 1;
    for (int d = d0; d < d1 && p < ca && q < cb; ++d, bit <<= 1) {
        const bool sf = !df_lt(be, ae);                  // source p ends first (or both end)
        if (COUNT) {
            const DF end = sf ? ae : be;
            if (df_pos(df_sub(end, prev))) ++c;
            prev = end;
        }
        if (sf) bits |= bit;
        p += sf;
        q += !sf;
        const DF nx = df_ld(sf ? A[pidx(p + 1 < ca ? p + 1 : ca)] : B[pidx(q + 1 < cb ? q + 1 : cb)]);
        if (sf) ae = nx;
        else be = nx;
    }
    return bits;
}

// One node (k, j) per warp.  FILL = false: the node's entry count and the
// plan's marginals.  FILL = true: its entries, 32 merge steps at a time:
// consecutive lanes form consecutive steps' overlaps and write the entries next
// to each other.  (A lane writing its own run put a partial 32-byte sector per
// entry and array into L2.)  Where step d stands follows from the directions of
// the steps before it: p is the number of sources among them.  PATH: the count
// leaves them in `path`, 32 bits per lane and node, and the fill reads those
// 128 bytes; otherwise (walks of more than kPathSteps, or no memory for `path`)
// the fill walks again.  Nothing is written when the plan exceeds cap.
// Bound: instruction issue (79 % of cycles).  256 x 256, a converged pair (11.6 M
// entries): count 172 us, fill 169 us; the whole call 1.32 ms with the walk over
// all m + n ends, 0.46 ms with both kernels walking and one CTA scanning, 0.41 ms
// now; 512 x 512 (71 M) 10.0 -> 3.3 -> 2.7 ms.
template <bool FILL, bool PATH>
__global__ void __launch_bounds__(kRecWarps * 32) k_recover_df(const float* __restrict__ x, int m, int n,
                                                               int* __restrict__ counts, unsigned* __restrict__ path,
                                                               const long long* __restrict__ offs,
                                                               const unsigned long long* __restrict__ total,
                                                               unsigned long long cap, int32_t* __restrict__ src,
                                                               int32_t* __restrict__ dst, double* __restrict__ mass,
                                                               double* __restrict__ marg1,
                                                               double* __restrict__ marg2) {
    using Bits = std::conditional_t<PATH, unsigned, unsigned long long>;
    if (FILL && *total > cap) return;
    extern __shared__ float4 shdf[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = blockDim.x >> 5;
    float2* A = reinterpret_cast<float2*>(reinterpret_cast<float*>(shdf) + (size_t)warp * recover_df_words(m, n));
    float2* B = A + pidx(m) + 1;
    unsigned short* ia = reinterpret_cast<unsigned short*>(B + pidx(n) + 1);
    unsigned short* ib = ia + ((m + 1) & ~1);
    const int nodes = m * n;
    for (int r = blockIdx.x * nw + warp; r < nodes; r += gridDim.x * nw) {
        // warps at work together take different k and j: their sums go to different marginals
        const int j = r % n, k = (r / n + j) % m;
        const int node = k * n + j;
        const float* ra = x + node_row_a(m, k, j);
        const float* rb = x + node_row_b(m, n, k, j);
        Bits bits = 0;
        if (FILL && PATH) bits = path[(size_t)node * 32 + lane];
        const int ca = load_side_df(ra, m, ia, A);
        const int cb = load_side_df(rb, n, ib, B);
        const int steps = ca && cb ? ca + cb - 1 : 0;    // every step stands inside both sides until one ends
        const int span = (steps + 31) >> 5;              // merge steps per lane
        int c = 0;
        if (!FILL || !PATH) {
            const int d0 = min(steps, lane * span), d1 = min(steps, d0 + span);
            bits = merge_walk<!FILL, Bits>(A, B, ca, cb, d0, d1, c);
        }
        if (!FILL) {
            if (PATH) path[(size_t)node * 32 + lane] = (unsigned)bits;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
            if (lane == 0) counts[node] = c;
            // marg1 is kept as [j][i]
            const DF At = df_ld(A[pidx(ca)]), Bt = df_ld(B[pidx(cb)]);
            side_marginal(marg1 + (size_t)j * m, ca, ra, ia, A, Bt);
            side_marginal(marg2 + (size_t)k * n, cb, rb, ib, B, At);
        } else {
            const int own = __popcll(bits);              // sources passed before a lane's steps
            int before = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, before, o);
                if (lane >= o) before += y;
            }
            before -= own;
            const float inv = 1.f / (float)span;
            size_t pos = (size_t)offs[node];
            DF last{0.f, 0.f};                           // the end passed before this round's first step
            for (int base = 0; base < steps; base += 32) {
                const int d = base + lane;
                const int w = (int)(((float)d + 0.5f) * inv);    // d / span: at least 0.5 / 64 from the next integer
                const Bits ahead = __shfl_sync(0xffffffffu, bits, w & 31) & (((Bits)1 << ((d - w * span) & 63)) - 1);
                const int pp = __shfl_sync(0xffffffffu, before, w & 31) + __popcll(ahead), qq = d - pp;
                const bool in = d < steps && pp < ca && qq < cb;
                DF end{0.f, 0.f};
                if (in) end = df_min(df_ld(A[pidx(pp + 1)]), df_ld(B[pidx(qq + 1)]));
                DF prev = df_shfl_up(end, 1);
                if (lane == 0) prev = last;
                last = df_shfl(end, 31);
                const DF ov = df_sub(end, prev);
                const bool out = in && df_pos(ov);
                const unsigned mask = __ballot_sync(0xffffffffu, out);
                const size_t o = pos + __popc(mask & ((1u << lane) - 1u));
                if (out && o < cap) {
                    src[o] = ia[pp] * n + j;
                    dst[o] = k * n + ib[qq];
                    mass[o] = df_dbl(ov);
                }
                pos += __popc(mask);
            }
        }
        __syncwarp();
    }
}

// Exclusive scan of n counts into offsets: each CTA adds up all counts before
// its segment, then scans the segment, a count per thread and step.  The sums are
// read from L2 once per CTA, which costs less than a second launch.  65,536
// counts: 131 -> 12 us (29 on one CTA, whose loads' latency bound it).
constexpr int kScanCtas = 64;
__global__ void __launch_bounds__(1024) k_scan(const int* __restrict__ counts, long long* __restrict__ offs, int n,
                                               unsigned long long* __restrict__ total) {
    __shared__ long long s_w[32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int seg = ((n + kScanCtas - 1) / kScanCtas + 1023) & ~1023;
    const int s0 = min(n, (int)blockIdx.x * seg), s1 = min(n, s0 + seg);
    long long sum = 0;
#pragma unroll 8
    for (int t = tid; t < s0; t += 1024) sum += counts[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_w[warp] = sum;
    __syncthreads();
    long long carry = 0;
    for (int w = 0; w < 32; ++w) carry += s_w[w];
    for (int base = s0; base < s1; base += 1024) {
        const int t = base + tid;
        const int v = t < s1 ? counts[t] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();                                 // s_w has been read
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        long long at = carry + incl - v;
        for (int w = 0; w < 32; ++w) {
            const long long x = s_w[w];
            if (w < warp) at += x;
            carry += x;
        }
        if (t < s1) offs[t] = at;
    }
    if (blockIdx.x == kScanCtas - 1 && tid == 0) *total = (unsigned long long)carry;
}

// L1 distances of the plan's marginals to mu1 and mu2 (blockIdx.y: which):
// partial sums per CTA, added in order by the CTA that finishes last.
// t1: marg1 is stored [j][i] (k_recover_df) instead of [i][j].
constexpr int kL1Ctas = 64;
__global__ void __launch_bounds__(256) k_marg_l1(const double* __restrict__ marg, const double* __restrict__ mu1,
                                                 const double* __restrict__ mu2, int m, int n, int t1,
                                                 double* __restrict__ part, unsigned int* __restrict__ done,
                                                 double* __restrict__ out) {
    __shared__ double s[256];
    __shared__ int s_last;
    const int which = blockIdx.y, M = m * n;
    const double* mg = marg + (size_t)which * M;
    const double* mu = which ? mu2 : mu1;
    double acc = 0.0;
    for (int t = blockIdx.x * 256 + threadIdx.x; t < M; t += kL1Ctas * 256)
        acc += fabs(mg[t] - mu[!which && t1 ? (t % m) * n + t / m : t]);
    auto block = [&](double v) {
        s[threadIdx.x] = v;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < (unsigned)o) s[threadIdx.x] += s[threadIdx.x + o];
            __syncthreads();
        }
        return s[0];
    };
    const double tot = block(acc);
    if (threadIdx.x == 0) {
        part[which * kL1Ctas + blockIdx.x] = tot;
        __threadfence();
        s_last = atomicAdd(done + which, 1u) == kL1Ctas - 1;
        __threadfence();
    }
    __syncthreads();
    if (s_last) {
        const double v = threadIdx.x < kL1Ctas ? __ldcg(part + which * kL1Ctas + threadIdx.x) : 0.0;
        __syncthreads();
        const double all = block(v);
        if (threadIdx.x == 0) out[which] = all;
    }
}

// x-bar from the slab layout into the paper's vec order (eq. 4-6):
// f1_{i,k,j} at i + m k + m^2 j (same as slab j, row k, col i);
// f2_{k,j,l} at n m^2 + k + m j + m n l (slab n + k, row j, col l); the
// slab rows sit at their padded pitch.
// f1 rows keep their order (a warp per row); f2 is transposed in k and l for
// each j, in 32 x 32 blocks through shared memory, so that both sides are read
// and written in whole lines.  256 x 256: 151 -> 84 us (f2 was read with the
// stride of a slab), 403 MB, 0.72 of the measured copy bandwidth.
template <typename T>
__global__ void __launch_bounds__(256) k_export(const T* __restrict__ x, int m, int n, double* __restrict__ out) {
    __shared__ T tile[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t mp = row_pitch(m), np = row_pitch(n);
    const size_t half = (size_t)m * m * n, half_p = (size_t)n * m * mp;
    // f1: rows (j, k), eight per step and CTA
    const int rows = n * m, rsteps = (rows + 7) / 8;
    const int kt = (m + 31) / 32, lt = (n + 31) / 32;
    const long long items = (long long)rsteps + (long long)n * kt * lt;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        if (it < rsteps) {
            const int r = (int)it * 8 + warp;
            if (r < rows) {
                const T* row = x + (size_t)r * mp;
                double* o = out + (size_t)r * m;
#pragma unroll 4
                for (int i = lane; i < m; i += 32) o[i] = (double)__ldcs(row + i);
            }
        } else {
            const int q = (int)(it - rsteps);
            const int j = q / (kt * lt), k0 = (q / lt) % kt * 32, l0 = q % lt * 32;
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + warp + 8 * u, l = l0 + lane;
                if (k < m && l < n) tile[warp + 8 * u][lane] = __ldcs(x + half_p + ((size_t)k * n + j) * np + l);
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int l = l0 + warp + 8 * u, k = k0 + lane;
                if (k < m && l < n) out[half + (size_t)l * m * n + (size_t)j * m + k] = (double)tile[lane][warp + 8 * u];
            }
        }
    }
}

int export_flows(Inst* I, double* x, int space, cudaStream_t st) {
    const int m = I->m, n = I->n;
    const size_t V = (size_t)m * n * (m + n);
    int dev = 0, sms = 0;
    HOT_CK(cudaGetDevice(&dev));
    HOT_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    double* dst = x;
    double* tmp = nullptr;
    if (space == HOT_SPACE_HOST) {
        HOT_CK(cudaMallocAsync(&tmp, V * 8, st));
        dst = tmp;
    }
    const int grid = sms * 8;
    if (I->fp64) k_export<double><<<grid, 256, 0, st>>>((const double*)I->desc.xr, m, n, dst);
    else k_export<float><<<grid, 256, 0, st>>>((const float*)I->desc.xr, m, n, dst);
    HOT_CK(cudaGetLastError());
    if (tmp) {
        HOT_CK(cudaMemcpyAsync(x, tmp, V * 8, cudaMemcpyDeviceToHost, st));
        cudaFreeAsync(tmp, st);
    }
    HOT_CK(cudaStreamSynchronize(st));
    return HOT_OK;
}

int recover_plan(Ctx* ctx, Inst* I, int32_t* src, int32_t* dst, double* mass, int space, size_t cap, size_t* nnz,
                 double* marg_l1, cudaStream_t st) {
    const int m = I->m, n = I->n;
    const int nodes = m * n;
    // one scratch allocation: offsets, marginals, L1 partials, total, L1, L1 counters, counts
    const size_t o_marg = sizeof(long long) * nodes, o_part = o_marg + sizeof(double) * 2 * nodes,
                 o_tot = o_part + sizeof(double) * 2 * kL1Ctas, o_l1 = o_tot + 8, o_done = o_l1 + 16,
                 o_cnt = o_done + 8, bytes = o_cnt + sizeof(int) * nodes;
    // and the merge directions that the count leaves for the fill (k_recover_df)
    const bool want = cap > 0 || src || dst || mass;
    const size_t o_path = (bytes + 127) & ~(size_t)127;
    bool keep = want && !I->fp64 && m + n - 1 <= kPathSteps;
    char* scr = nullptr;
    if (keep && cudaMallocAsync((void**)&scr, o_path + sizeof(unsigned) * 32 * nodes, st) != cudaSuccess) {
        cudaGetLastError();
        keep = false;
    }
    if (!keep) HOT_CK(cudaMallocAsync((void**)&scr, bytes, st));
    unsigned* path = keep ? (unsigned*)(scr + o_path) : nullptr;
    long long* offs = (long long*)scr;
    double* marg = (double*)(scr + o_marg);
    unsigned long long* dtot = (unsigned long long*)(scr + o_tot);
    double* l1 = (double*)(scr + o_l1);
    unsigned int* done = (unsigned int*)(scr + o_done);
    int* counts = (int*)(scr + o_cnt);
    int32_t *ds = src, *dd = dst;
    double* dm = mass;
    bool staged = false;
    auto finish = [&](int rc) {
        if (staged) {
            if (ds) cudaFreeAsync(ds, st);
            if (dd) cudaFreeAsync(dd, st);
            if (dm) cudaFreeAsync(dm, st);
        }
        cudaFreeAsync(scr, st);
        return rc;
    };
    auto failed = [&](cudaError_t e, const char* what) {
        if (e == cudaSuccess) return false;
        set_error(std::string(what) + ": " + cudaGetErrorString(e));
        return true;
    };
    // warps per CTA (each has its own part of the shared memory): up to
    // kRecWarps, fewer where that leaves more of them resident on an SM
    auto warps_for = [](size_t per) {
        int best = 1, most = 0;
        for (int w = kRecWarps; w >= 1; --w) {
            if (w * per > 200 * 1024) continue;
            const int res = std::min(48, (int)((227 * 1024) / (w * per + 1024)) * w);
            if (res > most) {
                most = res;
                best = w;
            }
        }
        return best;
    };
    const size_t per = I->fp64 ? recover_words(m, n) * sizeof(double) : recover_df_words(m, n) * sizeof(float);
    const int nw = warps_for(per);
    const size_t shm = (size_t)nw * per;
    const auto count_df = keep ? k_recover_df<false, true> : k_recover_df<false, false>;
    const auto fill_df = keep ? k_recover_df<true, true> : k_recover_df<true, false>;
    cudaError_t e = cudaFuncSetAttribute(count_df, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fill_df, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_recover<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    int sms = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    if (e == cudaSuccess) e = cudaMemsetAsync(marg, 0, o_cnt - o_marg, st);
    if (failed(e, "plan recovery")) return finish(HOT_ECUDA);
    const int grid = std::max(1, std::min((nodes + nw - 1) / nw, sms * (64 / nw)));
    if (I->fp64)
        k_recover<double><<<grid, nw * 32, shm, st>>>((const double*)I->desc.xr, m, n, 1, counts, nullptr,
                                                              nullptr, nullptr, nullptr, marg, marg + nodes);
    else
        count_df<<<grid, nw * 32, shm, st>>>((const float*)I->desc.xr, m, n, counts, path, nullptr, nullptr, 0, nullptr,
                                             nullptr, nullptr, marg, marg + nodes);
    k_scan<<<kScanCtas, 1024, 0, st>>>(counts, offs, nodes, dtot);
    if (marg_l1)
        // marginals against mu1 (row-major (i, j)) and mu2 (row-major (k, l))
        k_marg_l1<<<dim3(kL1Ctas, 2), 256, 0, st>>>(marg, I->desc.mu1, I->desc.mu2, m, n, I->fp64 ? 0 : 1,
                                                    (double*)(scr + o_part), done, l1);
    auto fill = [&](size_t room) {
        if (I->fp64)
            k_recover<double><<<grid, nw * 32, shm, st>>>((const double*)I->desc.xr, m, n, 0, counts, offs, ds, dd, dm,
                                                          nullptr, nullptr);
        else
            fill_df<<<grid, nw * 32, shm, st>>>((const float*)I->desc.xr, m, n, counts, path, offs, dtot, room, ds, dd, dm,
                                                nullptr, nullptr);
    };
    // device outputs of an FP32 solution: the fill runs behind the count without
    // a look at the total (it writes nothing when the plan does not fit)
    const bool ahead = want && !I->fp64 && space == HOT_SPACE_DEVICE && cap > 0;
    if (ahead) fill(cap);
    unsigned long long tot = 0;
    double hl1[2] = {0.0, 0.0};
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&tot, dtot, sizeof(tot), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && marg_l1) e = cudaMemcpyAsync(hl1, l1, sizeof(hl1), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (failed(e, "plan recovery")) return finish(HOT_ECUDA);
    *nnz = (size_t)tot;
    if (marg_l1) {
        marg_l1[0] = hl1[0];
        marg_l1[1] = hl1[1];
    }
    if (!want) return finish(HOT_OK);
    if (cap < tot) {
        set_error("output capacity " + std::to_string(cap) + " < plan size " + std::to_string(tot));
        return finish(HOT_EINVAL);
    }
    if (ahead || tot == 0) return finish(HOT_OK);
    if (space == HOT_SPACE_HOST) {
        staged = true;
        ds = dd = nullptr;
        dm = nullptr;
        e = cudaMallocAsync((void**)&ds, sizeof(int32_t) * tot, st);
        if (e == cudaSuccess) e = cudaMallocAsync((void**)&dd, sizeof(int32_t) * tot, st);
        if (e == cudaSuccess) e = cudaMallocAsync((void**)&dm, sizeof(double) * tot, st);
        if (failed(e, "device allocation for the plan")) return finish(HOT_ENOMEM);
    }
    fill(tot);
    e = cudaGetLastError();
    if (space == HOT_SPACE_HOST) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(src, ds, sizeof(int32_t) * tot, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dst, dd, sizeof(int32_t) * tot, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(mass, dm, sizeof(double) * tot, cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (failed(e, "plan recovery")) return finish(HOT_ECUDA);
    return finish(HOT_OK);
}

}  // namespace hot
