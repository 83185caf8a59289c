// Evaluates the device functions of the library that stand in for CUDA's own
// division and tanh, so that a test can bound their errors.
#include "fpd_device.cuh"

namespace {

__global__ void k_recip(const double *x, double *y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = fpd::recip(x[i]);
}

// out[i] = phi_f32, plain[i] = the same profile by sqrtf and tanhf
__global__ void k_phi(const float *dx, const float *dy, float a, float inv_xi, float rcut2, float *out, float *plain,
                      int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = fpd::phi_f32(dx[i], dy[i], a, inv_xi, rcut2);
    const float r2 = dx[i] * dx[i] + dy[i] * dy[i];
    plain[i] = r2 < rcut2 ? 0.5f * (tanhf((a - sqrtf(r2)) * inv_xi) + 1.0f) : 0.0f;
}

struct Buffer {
    void *p = nullptr;
    explicit Buffer(size_t bytes) { if (cudaMalloc(&p, bytes) != cudaSuccess) p = nullptr; }
    ~Buffer() { cudaFree(p); }
};

}  // namespace

extern "C" int recip_f64(const double *x, double *y, int n) {
    const size_t b = n * sizeof(double);
    Buffer in(b), out(b);
    if (!in.p || !out.p) return 1;
    cudaMemcpy(in.p, x, b, cudaMemcpyHostToDevice);
    k_recip<<<(n + 255) / 256, 256>>>((const double *)in.p, (double *)out.p, n);
    return cudaMemcpy(y, out.p, b, cudaMemcpyDeviceToHost) != cudaSuccess;
}

extern "C" int phi_f32(const float *dx, const float *dy, float a, float inv_xi, float rcut2, float *out, float *plain,
                       int n) {
    const size_t b = n * sizeof(float);
    Buffer x(b), y(b), o(b), q(b);
    if (!x.p || !y.p || !o.p || !q.p) return 1;
    cudaMemcpy(x.p, dx, b, cudaMemcpyHostToDevice);
    cudaMemcpy(y.p, dy, b, cudaMemcpyHostToDevice);
    k_phi<<<(n + 255) / 256, 256>>>((const float *)x.p, (const float *)y.p, a, inv_xi, rcut2, (float *)o.p,
                                    (float *)q.p, n);
    return cudaMemcpy(out, o.p, b, cudaMemcpyDeviceToHost) != cudaSuccess ||
           cudaMemcpy(plain, q.p, b, cudaMemcpyDeviceToHost) != cudaSuccess;
}
