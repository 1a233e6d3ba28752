// Basis-independent velocity moments int phi~ v_h on each sub-tet (Eq. vis3).
#include "dev.cuh"

namespace stdg {

__global__ void k_moments(int N, int Ng, FxBlocks Mij, const double* __restrict__ V,
                          double dt, double* __restrict__ U) {
  const int j = blockIdx.x;
  const int Nst = N * Ng;
  const size_t NN = (size_t)N * N;
  for (int o = threadIdx.x; o < 2 * 3 * Nst; o += blockDim.x) {
    const int s = o / (3 * Nst), rem = o % (3 * Nst), c = rem / Nst, ta = (rem % Nst) / N, k = rem % N;
    const double* v = V + (size_t)j * 3 * Nst + c * Nst + ta * N;
    double acc = 0.0;
    for (int ll = 0; ll < N; ++ll) acc = fma(fx_entry(Mij, NN, (size_t)j * 2 + s, k * N + ll, N), v[ll], acc);
    U[(size_t)j * 6 * Nst + o] = dt * acc;
  }
}

cudaError_t launch_moments(int nf, int N, int Ng, const FxBlocks& Mij, const double* V, double dt,
                           double* U, cudaStream_t st) {
  if (nf > 0) k_moments<<<nf, 128, 0, st>>>(N, Ng, Mij, V, dt, U);
  return cudaGetLastError();
}

}  // namespace stdg
