// Single device functions of the library on given inputs, for test_gpu_device_functions.py.
#include "hot_block.cuh"

using namespace hot;

namespace {

__global__ void __launch_bounds__(kThreads) k_sweep(HotInst I, P64 p, const double* ab, const double* dab, double* out,
                                                    double* rs, double* cs) {
    __shared__ Sweep64Smem sm;
    sweep64_tile<false>(I, 0, 0, (const double*)I.d0, out, p, ab, dab, rs, cs, sm);
}

// one sum of products per thread
__global__ void k_dot(const float* x, const float* y, int terms, int sums, float* hi, float* lo) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= sums) return;
    DF a{0.f, 0.f};
    for (int q = 0; q < terms; ++q) a = df_dot(a, x[t * terms + q], y[t * terms + q]);
    hi[t] = a.hi;
    lo[t] = a.lo;
}

}  // namespace

// The reduced costs g = h (X_r - X_c)^2 - alpha_r - beta_c of one S x S tile as the FP64 sweep forms them:
// with u = d = 0, A^T(y-bar - y0) = 0 and unit constants its new delta is max(0, -g).  ab: alpha, then beta.
extern "C" int probe_sweep64(int S, double h, const double* X, const double* ab, double* out) {
    const int Sp = (S + 3) & ~3;
    const size_t state = (size_t)S * Sp;
    double* d = nullptr;
    const size_t words = 3 * state + 2 * S + 2 * S + 2 * S + 4 * S;
    if (cudaMalloc(&d, words * 8) != cudaSuccess) return 1;
    cudaMemset(d, 0, words * 8);
    double *u = d, *d0 = u + state, *o = d0 + state, *x = o + state, *pc = x + 2 * S, *dp = pc + 2 * S, *sums = dp + 2 * S;
    cudaMemcpy(x, X, S * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(x + S, X, S * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(pc, ab, 2 * S * 8, cudaMemcpyHostToDevice);
    HotInst I{};
    I.m = I.n = I.TR = S;
    I.mp = I.np = Sp;
    I.nb1 = I.nb2 = 1;
    I.h = h;
    I.u = u;
    I.d0 = d0;
    I.X64 = x;
    P64 p{};
    p.is = p.s = p.trs = 1.0;
    p.h = h;
    k_sweep<<<1, kThreads>>>(I, p, pc, dp, o, sums, sums + S);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy2D(out, S * 8, o, Sp * 8, S * 8, S, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}

// sums[t] = sum over q of x[t][q] y[t][q], as a pair
extern "C" int probe_dot(const float* x, const float* y, int terms, int sums, float* hi, float* lo) {
    const size_t N = (size_t)terms * sums;
    float* d = nullptr;
    if (cudaMalloc(&d, (2 * N + 2 * sums) * 4) != cudaSuccess) return 1;
    float *dx = d, *dy = d + N, *dh = dy + N, *dl = dh + sums;
    cudaMemcpy(dx, x, N * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(dy, y, N * 4, cudaMemcpyHostToDevice);
    k_dot<<<(sums + 127) / 128, 128>>>(dx, dy, terms, sums, dh, dl);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(hi, dh, sums * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(lo, dl, sums * 4, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
