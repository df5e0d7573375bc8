// Consumers of a recovered transport plan: the barycentric projection used
// by colour transfer (Sec. IV-B and App. G of arXiv 2408.00598).
//
// A plan is a list of entries (s, t, pi) in device memory (Algorithm 1's
// output from hot_recover_plan).  Source bin s is sent to
//     T(s) = sum_t pi(s, t) y_t / sum_t pi(s, t),
// y_t a D-vector per target bin.  One streaming pass accumulates numerator
// and weight per source, runs of one source in registers and those sums with
// FP64 atomic adds in L2 (the entries of one
// source are spread over the m nodes (k, j) it ships through, so a segmented
// sum would need an m-fold partial array); a second pass divides.  The order
// of the atomic adds is not fixed, so results are reproducible to rounding
// (about 1e-16 relative per entry), not bit for bit.
#include "hot_internal.h"
#include "hot_engine.h"

#include <string>
#include <type_traits>

namespace hot {

namespace {

constexpr int kBaryMaxD = 8;

// A thread takes kRun consecutive entries and adds up those of one source
// before it goes on to the next (Algorithm 1 writes a source's entries of a node
// one after the other); the finished sums of a warp are then added to global
// memory with consecutive lanes on consecutive components, so that the D
// doubles of a source go to L2 as one or two sectors instead of D.  Bound: FP64
// atomic adds at L2 (about 170 G/s).  12.6 M entries, D = 3, 1.4 per source
// and node: 0.31 -> 0.21 ms.
// The dimension is a template argument: FP64 instructions that a predicate
// switches off still pass through the pipe, which runs at a 64th of the FP32 rate.
constexpr int kRun = 8;
template <int D>
__global__ void __launch_bounds__(256) k_bary_acc(const int* __restrict__ src, const int* __restrict__ dst,
                                                  const double* __restrict__ mass, size_t nnz,
                                                  const double* __restrict__ y, int ndst,
                                                  double* __restrict__ num, double* __restrict__ w, int nsrc,
                                                  int* __restrict__ bad) {
    __shared__ double s_num[8][32 * D];
    __shared__ int s_src[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t warps = (size_t)gridDim.x * (blockDim.x >> 5);
    int nbad = 0;
    for (size_t base = ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * 32 * kRun; base < nnz;
         base += warps * 32 * kRun) {
        const size_t e0 = base + (size_t)lane * kRun;
        double acc[D], aw = 0.0;
        int cur = -1;                                        // the source being added up
#pragma unroll
        for (int d = 0; d < D; ++d) acc[d] = 0.0;
#pragma unroll 1
        for (int t = 0; t <= kRun; ++t) {
            const size_t e = e0 + t;
            int s = -1, q = 0;
            double p = 0.0;
            if (t < kRun && e < nnz) {
                s = src[e];
                q = dst[e];
                p = mass[e];
                if (s < 0 || s >= nsrc || q < 0 || q >= ndst) {   // reported, never dereferenced
                    ++nbad;
                    s = cur;                                 // stays with the open sum, adds nothing
                    q = -1;
                }
            }
            const bool flush = cur >= 0 && (s != cur);
            const unsigned mask = __ballot_sync(0xffffffffu, flush);
            if (mask) {
                const int cnt = __popc(mask), at = __popc(mask & ((1u << lane) - 1u));
                if (flush) {
                    atomicAdd(&w[cur], aw);
                    s_src[warp][at] = cur;
#pragma unroll
                    for (int d = 0; d < D; ++d)
                        s_num[warp][at * D + d] = acc[d];
                }
                __syncwarp();
                for (int c = lane; c < cnt * D; c += 32) {
                    const int f = c / D;
                    atomicAdd(&num[(size_t)s_src[warp][f] * D + (c - f * D)], s_num[warp][c]);
                }
                __syncwarp();
            }
            if (s != cur) {
                cur = s;
                aw = 0.0;
#pragma unroll
                for (int d = 0; d < D; ++d) acc[d] = 0.0;
            }
            if (s >= 0 && q >= 0) {
                aw += p;
#pragma unroll
                for (int d = 0; d < D; ++d)
                    acc[d] += p * y[(size_t)q * D + d];
            }
        }
    }
    if (nbad) atomicAdd(bad, nbad);
}

__global__ void __launch_bounds__(256) k_bary_div(double* __restrict__ num, const double* __restrict__ w, int nsrc,
                                                  int D) {
    const size_t n = (size_t)nsrc * D;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
        const double ws = w[q / D];
        num[q] = ws > 0.0 ? num[q] / ws : 0.0;
    }
}

}  // namespace

int barycentric_map(const int* src, const int* dst, const double* mass, size_t nnz, const double* y, int ndst,
                    int D, double* out, double* weight, int nsrc, cudaStream_t st) {
    if (D < 1 || D > kBaryMaxD || nsrc < 0 || ndst < 0) {
        set_error("barycentric map: D must be in [1, 8] and the bin counts non-negative");
        return HOT_EINVAL;
    }
    if ((nnz > 0 && (!src || !dst || !mass || !y)) || (nsrc > 0 && (!out || !weight))) {
        set_error("barycentric map: null pointer");
        return HOT_EINVAL;
    }
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
    int* d_bad = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&d_bad, sizeof(int), st);
    if (e != cudaSuccess) {
        set_error(std::string("barycentric map: ") + cudaGetErrorString(e));
        return HOT_ENOMEM;
    }
    int h_bad = 0;
    e = cudaMemsetAsync(d_bad, 0, sizeof(int), st);
    if (e == cudaSuccess && nsrc > 0) e = cudaMemsetAsync(out, 0, (size_t)nsrc * D * sizeof(double), st);
    if (e == cudaSuccess && nsrc > 0) e = cudaMemsetAsync(weight, 0, (size_t)nsrc * sizeof(double), st);
    if (e == cudaSuccess && nnz > 0) {
        auto launch = [&](auto dim) {
            k_bary_acc<decltype(dim)::value>
                <<<sms * 8, 256, 0, st>>>(src, dst, mass, nnz, y, ndst, out, weight, nsrc, d_bad);
        };
        switch (D) {
            case 1: launch(std::integral_constant<int, 1>()); break;
            case 2: launch(std::integral_constant<int, 2>()); break;
            case 3: launch(std::integral_constant<int, 3>()); break;
            case 4: launch(std::integral_constant<int, 4>()); break;
            case 5: launch(std::integral_constant<int, 5>()); break;
            case 6: launch(std::integral_constant<int, 6>()); break;
            case 7: launch(std::integral_constant<int, 7>()); break;
            default: launch(std::integral_constant<int, 8>()); break;
        }
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && nsrc > 0) {
        k_bary_div<<<sms * 4, 256, 0, st>>>(out, weight, nsrc, D);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFreeAsync(d_bad, st);
    if (e != cudaSuccess) {
        set_error(std::string("barycentric map failed on the device: ") + cudaGetErrorString(e));
        return HOT_ECUDA;
    }
    if (h_bad) {
        set_error("barycentric map: " + std::to_string(h_bad) + " entries with a bin index out of range (skipped)");
        return HOT_EINVAL;
    }
    return HOT_OK;
}

}  // namespace hot
