// Device build of recip64 (lbm_collide64.cuh) for the GPU test that compares it
// with the division.  Test infrastructure only.
#include "../paper_2212_07494_gb300/csrc/lbm_collide64.cuh"

__global__ void k_recip(const double *in, double *out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = lbm::recip64(in[i]);
}

extern "C" int device_recip64(const double *in, double *out, int n) {
    k_recip<<<(n + 255) / 256, 256>>>(in, out, n);
    return (int)cudaDeviceSynchronize();
}
