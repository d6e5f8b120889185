// Device and host functions of the kernels' headers, callable one at a time.
#include <vector>

#include "cgks_kernels.cuh"

using namespace cgks;

namespace {
// A device array, filled from host memory or with zeros
template <typename T> struct Array {
    T* p = nullptr;
    Array(size_t n, const T* from = nullptr)
    {
        if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess) { p = nullptr; return; }
        if (from) cudaMemcpy(p, from, n * sizeof(T), cudaMemcpyHostToDevice);
        else cudaMemset(p, 0, n * sizeof(T));
    }
    ~Array() { cudaFree(p); }
};
}  // namespace

extern "C" long long unit_fr_nrow(int dir, int na, int nb) { return fr_nrow(dir, na, nb); }
extern "C" int unit_descriptor_bytes() { return (int)sizeof(Work); }

// The stage-1 update of an nx x ny periodic mesh with spacing h
// (order 5, FP32 bulk): averages W [4][ny nx], x-face flux sums fx [ny (nx + 1)][4]
// (the integral to dt/2), all else zero -> W* as hi and lo [4][ny nx].
extern "C" int unit_stage1_averages(int nx, int ny, double h, const double* W, const float* fx, float* hi, float* lo)
{
    constexpr int M = 2, NP = 12 + 8 * M;
    const size_t P = (size_t)nx * ny, nfx = (size_t)ny * (nx + 1), nfy = (size_t)nx * (ny + 1);
    std::vector<float> f0((NP + 4) * P, 0.0f), fo(nfx * (2 * M + 2) * 4, 0.0f);
    for (size_t e = 0; e < 4 * P; ++e) {
        f0[e] = (float)W[e];
        f0[NP * P + e] = (float)(W[e] - (double)f0[e]);
    }
    // the face sums come after the two interface states of the M points
    for (size_t e = 0; e < 4 * nfx; ++e) fo[2 * M * nfx * 4 + e] = fx[e];
    Array<double> S0(NP * P), ACC((4 + 8 * M) * P), scal(64);
    Array<float> F0(f0.size(), f0.data()), F1(f0.size()), X(fo.size(), fo.data()), Y(nfy * (2 * M + 2) * 4);
    if (!S0.p || !ACC.p || !scal.p || !F0.p || !F1.p || !X.p || !Y.p) return 1;
    cudaMemcpy(S0.p, W, 4 * P * sizeof(double), cudaMemcpyHostToDevice);
    Work w = {};
    Mesh& g = w.m0;
    g.nx = nx; g.ny = ny; g.order = 5; g.plane = (long long)P;
    g.dx = g.dy = h; g.idx = g.idy = 1.0 / h;
    g.idxf = g.idyf = (float)g.idx;
    g.idxlo = g.idylo = (float)(g.idx - (double)g.idxf);
    g.gamma = 1.4;
    g.S0 = S0.p; g.F0 = F0.p; g.F1 = F1.p; g.ACC = ACC.p;
    g.FO[0] = X.p; g.FO[1] = Y.p;
    g.dt = scal.p; g.tn = scal.p + 1; g.dtf = (float*)(scal.p + 2);
    g.status = (unsigned*)(scal.p + 3); g.bad = (long long*)(scal.p + 4);
    w.n = 1;
    w.total = (long long)P;
    k_update2<M, float, 1, true><<<(int)((P + 255) / 256), 256>>>(w);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    cudaMemcpy(hi, F1.p, 4 * P * sizeof(float), cudaMemcpyDeviceToHost);
    cudaMemcpy(lo, F1.p + NP * P, 4 * P * sizeof(float), cudaMemcpyDeviceToHost);
    return 0;
}

// recip and recip_sqrt of floats
__global__ void k_reciprocals(const float* x, float* r, float* q, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = recip(x[i]);
    q[i] = recip_sqrt(x[i]);
}
extern "C" int unit_reciprocals(const float* x, float* r, float* q, int n)
{
    Array<float> X(n, x), A(n), B(n);
    if (!X.p || !A.p || !B.p) return 1;
    k_reciprocals<<<(n + 255) / 256, 256>>>(X.p, A.p, B.p, n);
    return cudaMemcpy(r, A.p, n * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess ||
           cudaMemcpy(q, B.p, n * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess;
}
