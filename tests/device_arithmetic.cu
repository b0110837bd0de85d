// The arithmetic headers of the update kernel, element by element (test_gpu_arithmetic.py).
#include "fdlb_round.cuh"
#include "fdlb_weno.cuh"

template <typename T>
__global__ void k_faces(const T* v, int n, T* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fdlb::weno_face(v[5 * i], v[5 * i + 1], v[5 * i + 2], v[5 * i + 3], v[5 * i + 4]);
}

// How many of the 2^24 random numbers round base + inc to each of two values, and to anything else.
__global__ void k_round(float base, float inc, float lo, float hi, unsigned long long* count) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    const float x = fdlb::sr_add(base, inc, j << 8 | 0x5a);
    atomicAdd(count + (x == lo ? 0 : x == hi ? 1 : 2), 1ull);
}

extern "C" int rounding(float base, float inc, float lo, float hi, unsigned long long* count) {
    k_round<<<(1 << 24) / 256, 256>>>(base, inc, lo, hi, count);
    return (int)cudaDeviceSynchronize();
}
extern "C" int faces32(const float* v, int n, float* out) {
    k_faces<<<(n + 255) / 256, 256>>>(v, n, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" int faces64(const double* v, int n, double* out) {
    k_faces<<<(n + 255) / 256, 256>>>(v, n, out);
    return (int)cudaDeviceSynchronize();
}
