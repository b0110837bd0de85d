// The arithmetic headers of the update kernel, element by element (test_gpu_arithmetic.py).
#include "fdlb_weno.cuh"

template <typename T>
__global__ void k_faces(const T* v, int n, T* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fdlb::weno_face(v[5 * i], v[5 * i + 1], v[5 * i + 2], v[5 * i + 3], v[5 * i + 4]);
}

extern "C" int faces32(const float* v, int n, float* out) {
    k_faces<<<(n + 255) / 256, 256>>>(v, n, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" int faces64(const double* v, int n, double* out) {
    k_faces<<<(n + 255) / 256, 256>>>(v, n, out);
    return (int)cudaDeviceSynchronize();
}
