// The limiter of the sweeps on arrays, for test_gpu_limiter: out = the half slope of
// the sweeps with upwind owners, ref = the one with the divide.
#include "../paper_2208_09132_gb300/csrc/pack.cuh"

template <typename T>
__global__ void k_limiter(const T* s1, const T* s2, T* out, T* ref, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = cdg::vanleer1(s1[i], s2[i]);
    ref[i] = cdg::Num<T>::vanleer(s1[i], s2[i]);
}
extern "C" int limiter_f64(const double* s1, const double* s2, double* out, double* ref, int n) {
    k_limiter<double><<<(n + 255) / 256, 256>>>(s1, s2, out, ref, n);
    return (int)cudaDeviceSynchronize();
}
